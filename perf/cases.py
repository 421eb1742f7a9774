"""The work that users of this framework have it do, as measurable cases.

A case is one pass of a program's main loop through the public entry points:
time steps of one lattice in each state form and scheme, a window of a run to
the terminal velocity (steps, then observables), a whole short run from host
fields, a snapshot (initial discs, steps, fields read back), an ensemble
advancing together, and training and asking the surrogate network.

    listed()            the cases that are always measured
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs and handles, as a program has them before the call
    run(state)          one pass; its outputs
    work(case)          bytes and operations that the pass cannot do without
    exact(case, seed)   the same outputs in 64 bits, in plain torch and numpy

State outputs are views of the handle's own device buffers: the planes of
include/lbm.h ("Device data layout") that hold the state after an even number
of steps.
"""
import math

import numpy as np
import torch

from paper_2207_09431_gb300 import inputs, lbm

GRIDS = {"mixed": ((100, 200), (150, 300), (200, 400), (300, 600)), "small": ((100, 200),)}
NODE_STEPS_MOST = 2048 * 4096 * 20  # node updates of the largest case


def listed():
    return [
        # the smallest lattice that the tests and the smoke run use: launches and latency
        dict(name="steps_64x128", kind="lattice", nx=64, ny=128, steps=64, density_ratio=100.0),
        # a window of the run to the terminal velocity on the paper's lattice: steps, then observables
        dict(name="window_200x400", kind="lattice", nx=200, ny=400, steps=200, density_ratio=100.0, observe=True),
        # the benchmark's end-to-end run: host fields up, steps, observables back
        dict(name="run_2048x4096", kind="lattice", nx=2048, ny=4096, steps=20, density_ratio=1000.0, upload=True,
             observe=True),
        # the state held as C (collapse_h), variable mobility, a ragged lattice, from host fields
        dict(name="collapsed_517x1031", kind="lattice", nx=517, ny=1031, steps=40, density_ratio=100.0, collapse_h=1,
             mobility=1, upload=True),
        # FP16 storage of g
        dict(name="fp16_1024x2048", kind="lattice", nx=1024, ny=2048, steps=20, density_ratio=1000.0, collapse_h=1,
             storage=1),
        # three components, fully periodic, the paper's Sec. 3.1 size
        dict(name="three_256x256", kind="three", nx=256, steps=64, mobility=1),
        # the mixed difference scheme on the paper's lattice (the stability comparison)
        dict(name="mixed_200x400", kind="lattice", nx=200, ny=400, steps=64, density_ratio=100.0, fd_scheme=1),
        # velocity inlet and convective outlet on the paper's channel
        dict(name="channel_240x60", kind="channel", nx=240, ny=60, steps=64),
        # a parameter study: cases of several sizes in persistent launches
        dict(name="ensemble_48_mixed", kind="ensemble", cases=48, grids="mixed", steps=64, persistent=True),
        # the surrogate's training set: many small cases, one launch per step
        dict(name="ensemble_256_100x200", kind="ensemble", cases=256, grids="small", steps=32, persistent=False),
        # a plotted run: discs set up by the library, steps, observables, fields read back
        dict(name="snapshot_400x800", kind="snapshot", nx=400, ny=800, steps=16, density_ratio=100.0),
        # the surrogate: training, then terminal states of a parameter study
        dict(name="surrogate_512x40", kind="surrogate", members=5, rows=512, batch=128, epochs=40, ask=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("lattice",) * 4 + ("three", "mixed", "channel", "ensemble", "snapshot", "surrogate"))
    if kind == "lattice":
        nx = _log_int(rng, 48, 2048)
        ny = _log_int(rng, max(96, nx), 2 * nx + 1)
        steps = 2 * _log_int(rng, 8, 100)
        steps = max(2, min(steps, NODE_STEPS_MOST // (nx * ny) // 2 * 2))
        form = rng.choice(("populations", "populations", "collapsed", "fp16"))
        upload = rng.random() < 0.3
        case = dict(kind="lattice", nx=nx, ny=ny, steps=steps, density_ratio=1000.0 if upload and nx >= 400 else 100.0)
        if form != "populations":
            case["collapse_h"] = 1
        if form == "fp16":
            case["storage"] = 1
        if upload:
            case["upload"] = True
            if case["density_ratio"] == 100.0 and rng.random() < 0.5:
                case["mobility"] = 1
        if rng.random() < 0.5:
            case["observe"] = True
        return case
    if kind == "three":
        nx = _log_int(rng, 128, 1024)
        case = dict(kind="three", nx=nx, steps=2 * _log_int(rng, 8, 40), mobility=rng.choice((0, 1)))
        if rng.random() < 0.3:
            case["collapse_h"] = 1
        return case
    if kind == "mixed":
        nx = _log_int(rng, 48, 800)
        return dict(kind="lattice", nx=nx, ny=_log_int(rng, max(96, nx), 2 * nx + 1), steps=2 * _log_int(rng, 5, 32),
                    density_ratio=100.0, fd_scheme=1)
    if kind == "channel":
        ny = _log_int(rng, 16, 120)
        return dict(kind="channel", nx=4 * ny + rng.randint(0, 7), ny=ny, steps=2 * _log_int(rng, 5, 40))
    if kind == "ensemble":
        count, grids = _log_int(rng, 4, 200), rng.choice(("mixed", "small"))
        nodes = count * sum(nx * ny for nx, ny in GRIDS[grids]) // len(GRIDS[grids])
        steps = max(2, min(2 * _log_int(rng, 4, 32), NODE_STEPS_MOST * 2 // 3 // nodes // 2 * 2))
        return dict(kind="ensemble", cases=count, grids=grids, steps=steps, persistent=rng.random() < 0.5)
    if kind == "snapshot":
        nx = _log_int(rng, 48, 700)
        return dict(kind="snapshot", nx=nx, ny=_log_int(rng, max(96, nx), 2 * nx + 1), steps=2 * _log_int(rng, 2, 16),
                    density_ratio=100.0)
    rows = _log_int(rng, 40, 1200)
    return dict(kind="surrogate", members=rng.randint(1, 8), rows=rows, batch=_log_int(rng, 16, 512),
                epochs=_log_int(rng, 4, 30), ask=_log_int(rng, 1, 512))


# ------------------------------------------------------------------- inputs

FIELDS = ("C1", "rho", "p", "ux", "uy")  # what a snapshot reads back


def _bubble(case, seed):
    """(params, discs) of a rising bubble, R = nx / 8, its place, shear thinning
    and tension by seed: at density ratio 1000 the bandwidth sweep's set-up,
    else that of the ensemble."""
    r = np.random.default_rng([seed, 17])
    nx, ny, ratio = case["nx"], case["ny"], case["density_ratio"]
    R = nx / 8.0
    d = 2.0 * R
    n, vary = float(r.uniform(-0.05, 0.05)), float(r.uniform(0.9, 1.1))
    if ratio < 1000.0:
        physics = dict(n=0.75 + 3.0 * n, k=1.667e-2, sigma=(1.0 - 1.0 / ratio) * 1e-5 * d * vary, gravity=1e-4 / d)
    else:
        physics = dict(n=0.7 + n, k=1.667e-2, sigma=(1.0 - 1.0 / ratio) * 2e-7 * d * d * vary, gravity=2e-6)
    p = inputs.rising_bubble_params(nx, ny, density_ratio=ratio, mobility=case.get("mobility", 0), **physics)
    p.update(collapse_h=case.get("collapse_h", 0), storage=case.get("storage", 0), fd_scheme=case.get("fd_scheme", 0))
    centre = (nx / 2.0 + float(r.uniform(-0.1, 0.1)) * nx, 0.3 * ny + float(r.uniform(-0.02, 0.02)) * ny)
    return p, [(centre[0], centre[1], R, 3)]


def _swirl(p, seed, amplitude=1e-3):
    """A smooth divergence-free velocity that vanishes through the walls."""
    x = 2.0 * np.pi * (np.arange(p["nx"]) / p["nx"] + np.random.default_rng([seed, 5]).uniform())[None, :]
    y = np.pi * ((np.arange(p["ny"]) + 0.5) / p["ny"])[:, None]
    ux = amplitude * np.sin(2.0 * y) * np.cos(x)
    return dict(ux=inputs.round_to_fp32(ux),
                uy=inputs.round_to_fp32(amplitude * 2.0 * p["ny"] / p["nx"] * np.sin(y) ** 2 * np.sin(x)))


def _lattice_inputs(case, seed):
    """(params, C, velocities) of one lattice."""
    if case["kind"] == "three":
        p, discs = inputs.three_comp_case(case["nx"], mobility=case["mobility"], seed=seed)
        p["collapse_h"] = case.get("collapse_h", 0)
    elif case["kind"] == "channel":
        r = np.random.default_rng([seed, 17])
        p, C, ux = inputs.open_channel_case(float(r.uniform(0.6, 1.2)), ny=case["ny"], nx=case["nx"],
                                            u_in=float(r.uniform(0.03, 0.05)))
        y = (np.arange(case["ny"]) + 0.5) / case["ny"]
        x = np.arange(case["nx"]) / case["nx"]
        ux = ux * (1.0 + 0.2 * np.sin(2.0 * np.pi * (x[None, :] + r.uniform())) * (y * (1.0 - y))[:, None])
        return p, C, dict(ux=inputs.round_to_fp32(ux))
    else:
        p, discs = _bubble(case, seed)
    C = inputs.bubble_fields(p["nx"], p["ny"], p["ncomp"], p["xi"], discs, seed=seed, noise=1e-8,
                             periodic_y=bool(p["periodic_y"]))
    moving = case["kind"] == "lattice" and case["density_ratio"] < 1000.0
    return p, inputs.round_to_fp32(C), _swirl(p, seed) if moving else {}


def _ensemble_inputs(case, seed):
    """[(params, C, velocities)] of an ensemble at the density ratio and mobility
    of the surrogate's training set, the grids in turn."""
    out, grids = [], GRIDS[case["grids"]]
    for i in range(case["cases"]):
        p, discs, _ = inputs.ensemble_cases(1, seed=1000 * seed + 7919 * i, grids=(grids[i % len(grids)],))[0]
        C = inputs.bubble_fields(p["nx"], p["ny"], 2, p["xi"], discs, seed=i, noise=1e-8)
        out.append((p, inputs.round_to_fp32(C), _swirl(p, 1000 * seed + i)))
    return out


def _surrogate_inputs(case, seed):
    """(initial weights, X, Y, X asked): the features of seeded rising-bubble
    cases and smooth terminal states of them."""
    r = np.random.default_rng([seed, 29])

    def features(n):
        nn, eo, lm = r.uniform(0.4, 1.0, n), r.uniform(1.0, 100.0, n), r.uniform(-3.0, 1.0, n)
        return np.stack([nn, eo, lm, np.full(n, 100.0), 0.25 * lm + 1.5 * nn - 0.75 * np.log10(eo) + 2.0], axis=1)

    X = features(case["rows"])
    Y = np.stack([-7.0 + 0.4 * np.log(X[:, 1]) - 0.3 * X[:, 2] * X[:, 0], 1.0 + 0.9 * X[:, 2] - 0.5 * X[:, 0] ** 2], axis=1)
    Y = Y + 0.01 * r.standard_normal(Y.shape)
    return inputs.mlp_init(case["members"], seed=seed % 1000), X, Y, features(case["ask"])


# ---------------------------------------------------- device state as outputs

def _state_views(arena, base, p):
    """The buffers of a handle at byte `base` of its arena that hold the state
    after an even number of steps since lbm_set_fields (include/lbm.h), with
    the padding columns."""
    nx, ny, nh = p["nx"], p["ny"], p["ncomp"] - 1
    pitch = -(-nx // 32) * 32
    plane = -(-(4 * ny * pitch) // 256) * 64  # floats per plane
    hp = nh if p.get("collapse_h") else 9 * nh
    blocks = (ny, pitch // 32)

    def view(first, count):
        return arena[base + 4 * first:base + 4 * (first + count)].view(torch.float32)

    out = {}
    if p.get("storage"):
        out["g"] = view(0, 9 * ny * pitch // 2).view(torch.float16).view(*blocks, 9, 32)
        out["p0"] = view(9 * plane // 2, ny * pitch).view(ny, pitch)
    else:
        out["g"] = view(0, 9 * ny * pitch).view(*blocks, 9, 32)
    if p.get("collapse_h"):
        out["C"] = view(18 * plane, nh * plane).view(nh, plane)[:, :ny * pitch].view(nh, ny, pitch)
    else:
        out["h"] = view(18 * plane, 9 * nh * ny * pitch).view(*blocks, 9 * nh, 32)
    out["tau"] = view(18 * plane + 2 * hp * plane, ny * pitch).view(ny, pitch)
    return out


def _without_padding(views, nx):
    """The columns x < nx of _state_views: whole blocks of 32 and the rest of the last one."""
    out = {}
    for k, v in views.items():
        if k in ("g", "h"):
            out[k] = v[:, :nx // 32]
            if nx % 32:
                out[k + "_last"] = v[:, nx // 32, :, :nx % 32]
        else:
            out[k] = v[..., :nx]
    return {k: v for k, v in out.items() if v.numel()}


def prepare(case, seed):
    stream = torch.cuda.Stream()
    kind = case["kind"]
    if kind == "ensemble":
        cases = _ensemble_inputs(case, seed)
        batch = lbm.Batch([p for p, _, _ in cases], stream=stream)
        if case["persistent"]:
            batch.set_persistent(True)
        views, base = [], 0
        for i, (p, C, u) in enumerate(cases):
            batch.case(i).set_fields(C, **u)
            views.append(_state_views(batch.arena, base, p))
            base += -(-lbm.lbm_required_bytes(p) // 256) * 256
        batch.autotune(reps=2)
        return dict(case=case, batch=batch, stream=stream, views=views)
    if kind == "surrogate":
        w, X, Y, asked = _surrogate_inputs(case, seed)
        net = lbm.Surrogate(w, max_batch=512, max_rows=2048, stream=stream)
        return dict(case=case, net=net, X=X, Y=Y, asked=asked, seed=seed % 1000)
    if kind == "snapshot":
        p, discs = _bubble(case, seed)
        return dict(case=case, lat=lbm.Lattice(p, stream=stream), discs=discs, seed=seed)
    p, C, u = _lattice_inputs(case, seed)
    lat = lbm.Lattice(p, stream=stream)
    state = dict(case=case, lat=lat, views=_without_padding(_state_views(lat.arena, 0, p), p["nx"]))
    if case.get("upload"):  # the program's fields, in page-locked memory
        state["fields"] = {k: torch.from_numpy(v).pin_memory().numpy() for k, v in dict(u, C=C).items()}
    else:
        lat.set_fields(C, **u)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ensemble":
        state["batch"].step(case["steps"])
        with torch.cuda.stream(state["stream"]):  # every case's state in one tensor, as a program stores an ensemble
            return {k: torch.cat([v[k].reshape(-1) for v in state["views"]]) for k in ("g", "h", "tau")}
    if kind == "surrogate":
        net = state["net"]
        loss = net.train(state["X"], state["Y"], case["epochs"], case["batch"], 2e-3, seed=state["seed"])
        mean, spread, outside = net.predict(state["asked"])
        return dict(loss=loss, weights=[net.weights(m) for m in range(case["members"])], mean=mean, spread=spread,
                    outside=outside)
    lat = state["lat"]
    if kind == "snapshot":
        lat.init_bubbles(state["discs"], seed=state["seed"], noise=1e-8)
        lat.step(case["steps"])
        return dict(observables=lat.observables(), fields={f: lat.field(f) for f in FIELDS})
    if case.get("upload"):
        lat.set_fields(**state["fields"])
    lat.step(case["steps"])
    out = dict(state["views"])
    if case.get("observe"):
        out["observables"] = lat.observables()
    return out


# --------------------------------------------------------------------- work

STEP_FLOPS = {2: 500.0, 3: 900.0}  # additions and multiplications of one node update (Sec. 2.2-2.3)


def _step_bytes(case, ncomp):
    """State of one node, read once and written once."""
    nh = ncomp - 1
    if case.get("storage"):
        return 2.0 * (18 + 4 + 4 * nh + 4)
    return 8.0 * (9 + (nh if case.get("collapse_h") else 9 * nh) + 1)


def work(case):
    kind = case["kind"]
    if kind == "surrogate":
        params = 5 * 128 + 128 + 2 * (128 * 128 + 128) + 128 * 2 + 2
        batch = min(case["batch"], case["rows"])
        rows = case["rows"] // batch * batch * case["epochs"]
        return {"bytes": case["members"] * params * 4.0 * 3 + (case["rows"] * 7 + case["ask"] * 9) * 8.0,
                "flops": case["members"] * params * (6.0 * rows + 2.0 * case["ask"])}
    if kind == "ensemble":
        grids = GRIDS[case["grids"]]
        nodes = sum(grids[i % len(grids)][0] * grids[i % len(grids)][1] for i in range(case["cases"]))
        return {"bytes": nodes * 152.0 * case["steps"], "flops": nodes * STEP_FLOPS[2] * case["steps"]}
    ncomp = 3 if kind == "three" else 2
    nodes = case["nx"] * case.get("ny", case["nx"])
    moved = nodes * _step_bytes(case, ncomp) * case["steps"]
    if case.get("upload"):
        moved += nodes * (8.0 * (ncomp - 1) + 0.5 * _step_bytes(case, ncomp))
    if case.get("observe") or kind == "snapshot":
        moved += nodes * 0.5 * _step_bytes(case, ncomp)
    if kind == "snapshot":
        moved += nodes * (0.5 * _step_bytes(case, ncomp) + 8.0 * len(FIELDS))
    return {"bytes": moved, "flops": nodes * STEP_FLOPS[ncomp] * case["steps"]}


# -------------------------------------------- the same in 64 bits, plain torch

_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_W = (4.0 / 9.0,) + (1.0 / 9.0,) * 4 + (1.0 / 36.0,) * 4
_BACK = (0, 3, 4, 1, 2, 7, 8, 5, 6)


class _Reference:
    """The step of arXiv 2207.09431 (Sec. 2) on FP64 tensors (..., ny, nx);
    lattices of one shape may share a leading dimension, their parameters then
    have that dimension too."""

    def __init__(self, cases, C, ux=None, uy=None):
        p = cases[0]
        self.p, self.dev = p, "cuda" if torch.cuda.is_available() else "cpu"
        self.nx, self.ny, self.nh = p["nx"], p["ny"], p["ncomp"] - 1
        self.periodic, self.open = bool(p.get("periodic_y", 0)), bool(p.get("open_x", 0))

        def par(f):
            return torch.tensor([float(f(q)) for q in cases], dtype=torch.float64, device=self.dev).view(-1, 1, 1)

        self.rho = [par(lambda q, i=i: q["rho"][i]) for i in range(3)]
        self.tau_i = [par(lambda q, i=i: q["tau"][i]) for i in range(3)]
        s12, s13, s23 = (par(lambda q, k=k: q.get(k, 1e-3)) for k in ("sigma12", "sigma13", "sigma23"))
        self.s12, self.s13, self.s23 = s12, s13, s23
        self.S = [s12 + s13 - s23, s12 + s23 - s13, s13 + s23 - s12]
        self.ST = 3.0 / sum(1.0 / s for s in self.S)
        self.lam, self.xi = par(lambda q: q.get("Lambda", 0.0)), par(lambda q: q.get("xi", 4.0))
        self.D0, self.grav = par(lambda q: q.get("D0", 4.0 / 300.0)), par(lambda q: q.get("gravity", 0.0))
        self.n, self.k = par(lambda q: q["pl_n"]), par(lambda q: q["pl_k"])
        self.tmin, self.tmax = par(lambda q: q["tau_min"]), par(lambda q: q["tau_max"])
        self.fx = par(lambda q: q.get("force_x", 0.0))
        self.scheme, self.mobility = p.get("fd_scheme", 0), p.get("mobility", 0)
        # rows and columns seen by stencils of reach two
        y, x = np.arange(-2, self.ny + 2), np.arange(-2, self.nx + 2)
        y = y % self.ny if self.periodic else np.where(y < 0, -1 - y, np.where(y >= self.ny, 2 * self.ny - 1 - y, y))
        x = np.where(x < 0, -1 - x, np.where(x >= self.nx, 2 * self.nx - 1 - x, x)) if self.open else x % self.nx
        self.iy, self.ix = torch.from_numpy(y).to(self.dev), torch.from_numpy(x).to(self.dev)
        C = torch.as_tensor(np.asarray(C), dtype=torch.float64, device=self.dev)  # (nh, lattices, ny, nx)
        z = torch.zeros_like(C[0])
        u = tuple(z if v is None else z + torch.as_tensor(v, dtype=torch.float64, device=self.dev) for v in (ux, uy))
        F = self.fields([C[i] for i in range(self.nh)], p=z, u=u)
        G, self.g, heq, _, _, _ = self.equilibria(F)
        self.h = heq
        self.tau = self.relaxation(F, torch.zeros_like(z))

    def pad(self, X):
        return X.index_select(-2, self.iy).index_select(-1, self.ix)

    def at(self, Xp, dx, dy):
        return Xp[..., 2 + dy:2 + dy + self.ny, 2 + dx:2 + dx + self.nx]

    def stencil(self, X, want_lap=False):
        """(pair of gradients, Laplacian or None, directional derivative of every direction)."""
        Xp = self.pad(X)
        v = [self.at(Xp, _EX[a], _EY[a]) for a in range(9)]
        gx = 3.0 * sum(_W[a] * _EX[a] * v[a] for a in range(1, 9) if _EX[a])
        gy = 3.0 * sum(_W[a] * _EY[a] * v[a] for a in range(1, 9) if _EY[a])
        lap = 6.0 * sum(_W[a] * (v[a] - v[0]) for a in range(1, 9)) if want_lap else None
        d = [torch.zeros_like(X)]
        for a in range(1, 9):
            if self.scheme == 0:
                d.append(0.5 * (v[a] - v[_BACK[a]]))
            else:
                far = self.at(Xp, 2 * _EX[a], 2 * _EY[a])
                d.append(0.25 * (5.0 * v[a] - far - 3.0 * v[0] - v[_BACK[a]]))
        return (gx, gy), lap, d

    def fields(self, Ct, g=None, p=None, u=None):
        C = list(Ct) + ([torch.zeros_like(Ct[0])] if self.nh == 1 else [])
        C.append(1.0 - C[0] - C[1])
        w = [c.clamp(0.0, 1.0) for c in C]
        total = w[0] + w[1] + w[2]
        w = [c / total for c in w]
        rho = w[0] * self.rho[0] + w[1] * self.rho[1] + w[2] * self.rho[2]
        st = [self.stencil(c, True) for c in C[:2]]
        gC = [s[0] for s in st] + [tuple(-(st[0][0][k] + st[1][0][k]) for k in (0, 1))]
        lap = [st[0][1], st[1][1], -(st[0][1] + st[1][1])]
        dC = [st[0][2], st[1][2], [-(a + b) for a, b in zip(st[0][2], st[1][2])]]
        C1, C2, C3 = C
        S, L = self.S, self.lam
        mix = S[0] * C1 + S[1] * C2 + S[2] * C3
        e = [2 * self.s12 * C1 * C2 ** 2 + 2 * self.s13 * C1 * C3 ** 2 + C2 * C3 * (mix + S[0] * C1)
             + 2 * L * C1 * C2 ** 2 * C3 ** 2,
             2 * self.s12 * C1 ** 2 * C2 + 2 * self.s23 * C2 * C3 ** 2 + C1 * C3 * (mix + S[1] * C2)
             + 2 * L * C1 ** 2 * C2 * C3 ** 2,
             2 * self.s13 * C1 ** 2 * C3 + 2 * self.s23 * C2 ** 2 * C3 + C1 * C2 * (mix + S[2] * C3)
             + 2 * L * C1 ** 2 * C2 ** 2 * C3]
        mu = [4.0 * self.ST / self.xi * sum((e[i] - e[j]) / S[j] for j in range(3) if j != i)
              - 0.75 * self.xi * S[i] * lap[i] for i in range(3)]
        (rx, ry), _, drho = self.stencil(rho)
        Fs = [sum(mu[i] * gC[i][k] for i in range(3)) for k in (0, 1)]
        Fb = [self.fx + torch.zeros_like(rho), -rho * self.grav]
        if g is not None:
            m = [sum(e_[a] * g[a] for a in range(9) if e_[a]) for e_ in (_EX, _EY)]
            u = tuple((3.0 * m[k] + 0.5 * (Fs[k] + Fb[k])) / rho for k in (0, 1))
            p = sum(g) + (u[0] * rx + u[1] * ry) / 6.0
        return dict(C=C, w=w, rho=rho, gC=gC, dC=dC, mu=mu, grho=(rx, ry), drho=drho, Fs=Fs, Fb=Fb, u=u, p=p)

    @staticmethod
    def gamma(a, ux, uy):
        eu = _EX[a] * ux + _EY[a] * uy
        return _W[a] * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))

    def equilibria(self, F):
        ux, uy = F["u"]
        (px, py), _, dp = self.stencil(F["p"])
        G, geq, heq, phig, phih = [], [], [], [], []
        uFs, u_rho = ux * F["Fs"][0] + uy * F["Fs"][1], ux * F["grho"][0] + uy * F["grho"][1]
        u_p = ux * px + uy * py
        for a in range(9):
            Ga = self.gamma(a, ux, uy)
            eF = sum(F["mu"][i] * F["dC"][i][a] for i in range(3)) - uFs + (_EX[a] - ux) * F["Fb"][0] \
                + (_EY[a] - uy) * F["Fb"][1]
            pg = (F["drho"][a] - u_rho) / 3.0 * (Ga - _W[a]) + eF * Ga
            G.append(Ga)
            phig.append(pg)
            geq.append(_W[a] * F["p"] + F["rho"] / 3.0 * (Ga - _W[a]) - 0.5 * pg)
            for i in range(self.nh):
                eC = F["dC"][i][a] - (ux * F["gC"][i][0] + uy * F["gC"][i][1])
                ph = (eC - 3.0 * F["C"][i] / F["rho"] * (dp[a] - u_p - eF)) * Ga
                phih.append((i, a, ph))
                heq.append((i, a, F["C"][i] * Ga - 0.5 * ph))
        order = lambda q: [[v for i, _, v in q if i == j] for j in range(self.nh)]  # noqa: E731
        return G, geq, order(heq), phig, order(phih), dp

    def relaxation(self, F, shear):
        t = (self.k * shear ** (self.n - 1.0)) * 3.0 / F["rho"] if self.p.get("powerlaw") else self.tau_i[0] + 0.0 * shear
        if self.p.get("powerlaw"):
            t = torch.where(shear > 0, t, torch.where(self.n < 1, torch.inf, torch.where(self.n > 1, 0.0, t)))
            t = torch.minimum(torch.maximum(t, self.tmin), self.tmax)
        return F["w"][0] * t + F["w"][1] * self.tau_i[1] + F["w"][2] * self.tau_i[2]

    def step(self):
        F = self.fields([sum(h) for h in self.h], g=self.g)
        G, geq, heq, phig, phih, _ = self.equilibria(F)
        fac = 3.0 * 2.0 * self.tau / (2.0 * self.tau + 1.0)
        ne = [fac * (self.g[a] - geq[a]) for a in range(9)]
        P = [sum(e1[a] * e2[a] * ne[a] for a in range(9) if e1[a] * e2[a])
             for e1, e2 in ((_EX, _EX), (_EY, _EY), (_EX, _EY))]
        D = [-q / (2.0 * self.tau * F["rho"] / 3.0) for q in P]
        tau = self.relaxation(F, torch.sqrt(2.0 * (D[0] ** 2 + D[1] ** 2 + 2.0 * D[2] ** 2)))
        src = []
        for i in range(self.nh):
            (mx, my), lapmu, _ = self.stencil(F["mu"][i], True)
            d = self.D0 / self.S[i]
            if self.mobility:
                c, raw = F["C"][i].clamp(0.0, 1.0), F["C"][i]
                inside = (raw >= 0) & (raw <= 1)
                src.append(d * c * (1.0 - c) * lapmu + torch.where(
                    inside, d * (1.0 - 2.0 * raw) * (F["gC"][i][0] * mx + F["gC"][i][1] * my), 0.0))
            else:
                src.append(d * lapmu)
        gp = [self.g[a] - (self.g[a] - geq[a]) / (tau + 0.5) + phig[a] for a in range(9)]
        hp = [[heq[i][a] + phih[i][a] + 0.5 * src[i] * G[a] for a in range(9)] for i in range(self.nh)]
        old_g, old_h = self.g, self.h
        self.g = self.stream(gp)
        self.h = [self.stream(hp[i]) for i in range(self.nh)]
        if self.open:
            self.boundaries(F, gp, old_g, old_h)
        for i in range(self.nh):
            for a in range(9):
                new = self.h[i][a] + 0.5 * src[i] * G[a]
                if self.open and _EX[a] == -1:  # the outlet's entering h follow its own rule
                    new[..., -1] = torch.where(self.enters[a], self.h[i][a][..., -1], new[..., -1])
                self.h[i][a] = new
        if self.open:
            self.outlet(F, old_g, old_h)
        self.tau = tau

    def stream(self, f):
        out = []
        for a in range(9):
            v = torch.roll(f[a], (_EY[a], _EX[a]), (-2, -1))
            if not self.periodic and _EY[a]:
                row = 0 if _EY[a] == 1 else self.ny - 1
                v[..., row, :] = f[_BACK[a]][..., row, :]
            out.append(v)
        return out

    def boundaries(self, F, gp, old_g, old_h):
        """What enters at x = 0: equilibrium at (u_in, 0) plus column 0's non-equilibrium part, and c_in."""
        u_in = torch.tensor(float(self.p["u_in"]), dtype=torch.float64, device=self.dev)
        y = torch.arange(self.ny, device=self.dev)
        self.enters = {}
        ux, uy = F["u"]
        for a in range(9):
            if not _EX[a]:
                continue
            sy = y - _EY[a]
            ok = torch.ones_like(sy, dtype=torch.bool) if self.periodic else (sy >= 0) & (sy < self.ny)
            self.enters[a] = ok
            sy = sy % self.ny
            if _EX[a] == 1:
                c = lambda X: X[..., 0].index_select(-1, sy)  # noqa: E731
                Gin = self.gamma(a, u_in, 0.0 * u_in)
                base = _W[a] * c(F["p"])
                eq_in = base + c(F["rho"]) / 3.0 * (Gin - _W[a])
                eq_0 = base + c(F["rho"]) / 3.0 * (self.gamma(a, c(ux), c(uy)) - _W[a])
                self.g[a][..., 0] = torch.where(ok, eq_in + c(gp[a]) - eq_0, self.g[a][..., 0])
                for i in range(self.nh):
                    self.h[i][a][..., 0] = torch.where(ok, self.p["c_in"][i] * Gin, self.h[i][a][..., 0])

    def outlet(self, F, old_g, old_h):
        """What enters at x = nx - 1: the convective condition, then the shift to zero pressure."""
        U = F["u"][0][..., -1].clamp(0.0, 1.0)
        wsum = 0.0
        for a in range(9):
            if _EX[a] != -1:
                continue
            ok = self.enters[a]
            wsum = wsum + _W[a] * ok
            for f, old in [(self.g, old_g)] + [(self.h[i], old_h[i]) for i in range(self.nh)]:
                new = (old[a][..., -1] + U * f[a][..., -2]) / (1.0 + U)
                f[a][..., -1] = torch.where(ok, new, f[a][..., -1])
        p0 = sum(self.g[a][..., -1] for a in range(9))
        for a in range(9):
            if _EX[a] == -1:
                self.g[a][..., -1] -= torch.where(self.enters[a], p0 * _W[a] / wsum, 0.0)

    # ---- outputs

    def macro(self):
        return self.fields([sum(h) for h in self.h], g=self.g)

    def views(self, b, p):
        """Lattice b's state as _state_views lays it out."""
        pitch = -(-self.nx // 32) * 32

        def padded(v):
            return torch.nn.functional.pad(v, (0, pitch - self.nx))

        def blocks(planes):  # (q, ny, nx) -> (ny, pitch / 32, q, 32)
            v = padded(planes)
            return v.view(v.shape[0], self.ny, pitch // 32, 32).permute(1, 2, 0, 3).contiguous()

        g = torch.stack([v[b] for v in self.g])
        h = torch.stack([torch.stack([v[b] for v in hi]) for hi in self.h])
        out = {}
        if p.get("storage"):
            P0 = g.sum(0)
            scale = 2.0 ** (14 - math.ceil(math.log2(max(p["rho"]))))
            w = torch.tensor(_W, dtype=torch.float64, device=self.dev).view(9, 1, 1)
            out["g"], out["p0"] = blocks((g - w * P0) * scale), padded(P0)
        else:
            out["g"] = blocks(g)
        if p.get("collapse_h"):
            out["C"] = padded(h.sum(1))
        else:
            out["h"] = blocks(h.reshape(-1, self.ny, self.nx))
        out["tau"] = padded(self.tau[b])
        return out

    def observables(self, p, step):
        """The sums of Sec. 3.1 and Eq. 37-44 for one two-component lattice; None
        for the sideways velocity, which cancels to rounding where the bubble
        starts from rest."""
        F = self.macro()
        C, u = [c[0] for c in F["C"]], [v[0] for v in F["u"]]
        x = torch.arange(self.nx, dtype=torch.float64, device=self.dev)[None, :]
        y = torch.arange(self.ny, dtype=torch.float64, device=self.dev)[:, None]
        cg = C[2]
        raw = [float(v.sum()) for v in C] + [float(torch.where(v > 0.5, v, 0.0).sum()) for v in C]
        raw += [float(v.sum()) for v in (cg, cg * x, cg * y, cg * u[0], cg * u[1])]
        yy, xx = torch.nonzero(cg > 0.5, as_tuple=True)
        raw += [float(v) for v in (xx.min(), xx.max(), yy.min(), yy.max())] if xx.numel() else [-1.0] * 4
        A, U = raw[6], raw[10] / raw[6]
        d = 2.0 * math.sqrt(A / math.pi)
        rl, rg, g, s = p["rho"][0], p["rho"][2], p["gravity"], p["sigma13"]
        n, k = p["pl_n"], p["pl_k"]
        return dict(step=step, mass=raw[:3], mass_thr=raw[3:6], area=A, centroid=[raw[7] / A, raw[8] / A],
                    velocity=[None, U], rise_velocity=U, y_integrated=raw[8] / A, d_eq=d,
                    aspect_E=(raw[14] - raw[13] + 1.0) / (raw[12] - raw[11] + 1.0),
                    drag_coefficient=4.0 * d * g * (rl - rg) / (3.0 * rl * U * U),
                    Re=rl * abs(U) ** (2.0 - n) * d ** n / k, Eo=(rl - rg) * g * d * d / s,
                    Mo=g * (rl - rg) / (rl * rl * s ** 3) * (k * (abs(U) / d) ** (n - 1.0)) ** 4,
                    raw=raw[:9] + [None] + raw[10:])


def _split_mix(seed, counters):
    """SplitMix64 outputs at the given counters of a stream."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (counters.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _exact_discs(p, discs, seed, noise):
    """C_1 of the initial discs with their noise (Eq. 42)."""
    nx, ny = p["nx"], p["ny"]
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    gas = np.zeros((ny, nx))
    for cx, cy, R, _ in discs:
        dx = np.abs(x - cx)
        dx = np.where(dx > 0.5 * nx, nx - dx, dx)
        gas += 0.5 - 0.5 * np.tanh((np.sqrt(dx ** 2 + (y - cy) ** 2) - R) / (0.5 * p["xi"]))
    z = _split_mix(seed, np.arange(2 * nx * ny, 3 * nx * ny))
    gas += noise * (2.0 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53).reshape(ny, nx) - 1.0)
    return (1.0 - gas)[None]


def _bf16(t):
    return t.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _exact_surrogate(case, seed):
    """Training and answers of the 5-128-128-128-2 network in 64 bits; its
    definition takes the operands of every product in BF16."""
    w0, X, Y, asked = _surrogate_inputs(case, seed)
    rows, batch = case["rows"], min(case["batch"], case["rows"])
    sizes = (5, 128, 128, 128, 2)
    mx, my = X.mean(0), Y.mean(0)
    vx, vy = (X * X).mean(0) - mx * mx, (Y * Y).mean(0) - my * my
    sx, sy = np.where(vx > 1e-24, np.sqrt(np.maximum(vx, 0)), 1.0), np.where(vy > 1e-24, np.sqrt(np.maximum(vy, 0)), 1.0)
    xs, ys = torch.from_numpy((X - mx) / sx), torch.from_numpy((Y - my) / sy)

    def layers(w):
        out, o = [], 0
        for i, j in zip(sizes, sizes[1:]):
            out.append((w[o:o + i * j].view(j, i), w[o + i * j:o + i * j + j]))
            o += i * j + j
        return out

    def forward(w, x):
        acts = [x]
        for l, (W, b) in enumerate(layers(w)):
            z = _bf16(acts[-1]) @ _bf16(W).T + b
            acts.append(torch.tanh(z) if l < 3 else z)
        return acts

    weights, answers, loss = [], [], 0.0
    for mem in range(case["members"]):
        w = torch.from_numpy(w0[mem]).clone()
        m, v, t = torch.zeros_like(w), torch.zeros_like(w), 0
        s0 = (seed % 1000 + 0x1234567 * (mem + 1)) % 2 ** 64
        draws = case["epochs"] * (rows - 1) if batch < rows else 0
        z = [int(q) for q in _split_mix(s0, np.arange(draws))] if draws else []
        at = 0
        for _ in range(case["epochs"]):
            perm = list(range(rows))
            if batch < rows:
                for r in range(rows - 1, 0, -1):
                    j = z[at] % (r + 1)
                    at += 1
                    perm[r], perm[j] = perm[j], perm[r]
            for b0 in range(0, rows - batch + 1, batch):
                idx = torch.tensor(perm[b0:b0 + batch])
                T = ys[idx]
                acts = forward(w, xs[idx])
                loss = float(0.5 * ((acts[-1] - T) ** 2).sum() / batch)
                dz = (acts[-1] - T) / batch
                grads = []
                for l in range(3, -1, -1):
                    W, _ = layers(w)[l]
                    grads = [(_bf16(dz).T @ _bf16(acts[l])).reshape(-1), dz.sum(0)] + grads
                    if l:
                        dz = (_bf16(dz) @ _bf16(W)) * (1.0 - acts[l] ** 2)
                g = torch.cat(grads)
                t += 1
                m = 0.9 * m + 0.1 * g
                v = 0.999 * v + 0.001 * g * g
                w = w - 2e-3 * (m / (1.0 - 0.9 ** t)) / (torch.sqrt(v / (1.0 - 0.999 ** t)) + 1e-8)
        weights.append(w.numpy())
        answers.append(forward(w, torch.from_numpy((asked - mx) / sx))[-1].numpy() * sy + my)
    a = np.stack(answers)
    mean = a.mean(0)
    return dict(loss=loss, weights=weights, mean=mean, spread=np.abs(a - mean).max(0),
                outside=((asked < X.min(0)) | (asked > X.max(0))).any(1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        return _exact_surrogate(case, seed)
    if kind == "ensemble":
        cases = _ensemble_inputs(case, seed)
        views = [None] * len(cases)
        for grid in GRIDS[case["grids"]]:
            at = [i for i, (p, _, _) in enumerate(cases) if (p["nx"], p["ny"]) == grid]
            for part in (at[k:k + 64] for k in range(0, len(at), 64)):
                ref = _Reference([cases[i][0] for i in part], np.stack([cases[i][1][0] for i in part])[None],
                                 **{k: np.stack([cases[i][2][k] for i in part]) for k in ("ux", "uy")})
                for _ in range(case["steps"]):
                    ref.step()
                for b, i in enumerate(part):
                    views[i] = ref.views(b, cases[i][0])
        return {k: torch.cat([v[k].reshape(-1) for v in views]) for k in ("g", "h", "tau")}
    if kind == "snapshot":
        p, discs = _bubble(case, seed)
        ref = _Reference([p], _exact_discs(p, discs, seed, 1e-8)[:, None])
    else:
        p, C, u = _lattice_inputs(case, seed)
        ref = _Reference([p], np.asarray(C)[:, None], **u)
    for _ in range(case["steps"]):
        ref.step()
    if kind == "snapshot":
        F = ref.macro()
        return dict(observables=ref.observables(p, case["steps"]),
                    fields=dict(C1=F["C"][0][0], rho=F["rho"][0], p=F["p"][0], ux=F["u"][0][0], uy=F["u"][1][0]))
    out = _without_padding(ref.views(0, p), p["nx"])
    if kind == "lattice" and not u:
        out["tau"] = None  # where a fluid is still at rest, its viscosity is that of the rounding's strain rate
    if case.get("observe"):
        out["observables"] = ref.observables(p, case["steps"])
    return out
