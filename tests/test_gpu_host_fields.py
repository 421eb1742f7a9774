"""Fields in and out: set-up from host fields around the edges of the upload chunks,
discs set up on the device, and fields converted on the device.

Tolerances: the initial state against the oracle by the rule of tests/test_gpu_parity.py
(max(1e-5, 3 x the deviation of the oracle's FP32 build)); discs and density against
FP64 numpy to one FP32 unit of the value (the same FP64 expression, rounded to FP32;
a last-place difference of the FP64 value can move that rounding by one unit)."""
import numpy as np
import pytest

import oracle
from paper_2207_09431_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_09431_gb300 import lbm as _lbm

    _lbm.load_library()
    return _lbm


def relerr(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-12 * b.size))


@pytest.mark.parametrize("nx,ny", [(33, 63), (32, 64), (40, 65), (31, 67), (65, 130)])
@pytest.mark.parametrize("periodic_y", [0, 1])
@pytest.mark.parametrize("extra", [{}, {"fd_scheme": 1}, {"ncomp": 3}])
@pytest.mark.parametrize("given", [(), ("p",), ("p", "ux", "uy")])
def test_initial_state_at_chunk_edges(lbm, nx, ny, periodic_y, extra, given):
    p, _ = inputs.small_case()
    p = dict(p, nx=nx, ny=ny, periodic_y=periodic_y)
    p.update(extra)
    discs = [(nx / 2, 2.0, 8.0, 3)] + ([(nx / 3, ny / 2, 6.0, 2)] if p["ncomp"] == 3 else [])
    C = inputs.round_to_fp32(inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=1, noise=1e-4,
                                                  periodic_y=bool(periodic_y)))
    r = np.random.default_rng(ny)
    f = {k: inputs.round_to_fp32((1e-5 if k == "p" else 1e-3) * r.normal(size=(ny, nx))) for k in given}
    lat, orc, o32 = lbm.Lattice(p), oracle.Oracle(p), oracle.Oracle(p, "f32")
    for o in (lat, orc, o32):
        o.set_fields(C, **f)
    for name in ("g", "h", "tau"):
        ref = orc.field(name)
        assert relerr(lat.field(name), ref) <= max(1e-5, 3.0 * relerr(o32.field(name), ref)), name


@pytest.mark.parametrize("nx,ny,count", [(1, 3, 1), (31, 9, 0), (33, 40, 16), (64, 65, 17), (50, 70, 33), (200, 130, 1)])
@pytest.mark.parametrize("ncomp,periodic_y,noise", [(2, 0, 1e-6), (2, 1, 0.0), (3, 1, 1e-3)])
def test_discs_match_the_host_profile(lbm, nx, ny, count, ncomp, periodic_y, noise):
    p, _ = inputs.small_case()
    p = dict(p, nx=nx, ny=ny, ncomp=ncomp, periodic_y=periodic_y)
    r = np.random.default_rng(count)
    discs = [(float(r.uniform(0, nx)), float(r.uniform(0, ny)), float(r.uniform(1, 12)),
              3 if ncomp == 2 or i % 2 else 2) for i in range(count)]
    want = inputs.bubble_fields(nx, ny, ncomp, p["xi"], discs, seed=11, noise=noise, periodic_y=bool(periodic_y))
    a, b = lbm.Lattice(dict(p, collapse_h=1)), lbm.Lattice(dict(p, collapse_h=1))  # the state holds C itself
    a.init_bubbles(discs, seed=11, noise=noise)
    b.set_fields(want)
    for name in ("C1", "C2")[:ncomp - 1]:
        x, y = a.field(name), b.field(name)
        assert np.max(np.abs(x - y)) <= 2.0 ** -23 * max(1.0, np.max(np.abs(want)))


@pytest.mark.parametrize("nx,ny", [(5, 3), (32, 8), (33, 41)])
@pytest.mark.parametrize("form", ["populations", "fp16", "three"])
def test_fields_are_one_state(lbm, nx, ny, form):
    p, _ = inputs.small_case()
    p = dict(p, nx=nx, ny=ny)
    if form == "fp16":
        p.update(collapse_h=1, storage=1)
    if form == "three":
        p["ncomp"] = 3
    discs = [(nx / 2, ny / 2, 4.0, 3)] + ([(1.0, 1.0, 2.0, 2)] if form == "three" else [])
    lat = lbm.Lattice(p)
    lat.set_fields(inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=1, noise=1e-3))
    for _ in range(2):  # both buffers
        lat.step(1)
        c = [lat.field(f"C{i}") for i in (1, 2, 3)]
        assert np.array_equal(c[2], (np.float32(1) - c[0].astype(np.float32) - c[1].astype(np.float32)).astype(float))
        w = [np.clip(v, 0.0, 1.0) for v in c]
        rho = (w[0] * p["rho"][0] + w[1] * p["rho"][1] + w[2] * p["rho"][2]) / (w[0] + w[1] + w[2])
        assert np.allclose(lat.field("rho"), rho, rtol=1e-14, atol=0)
        if form != "fp16":
            h = lat.field("h").astype(np.float32)
            for i in range(p["ncomp"] - 1):
                s = np.zeros((ny, nx), np.float32)
                for a in range(9):
                    s = s + h[i, a]
                assert np.array_equal(s.astype(float), c[i])
        before = lat.field("g"), lat.field("tau")
        assert np.array_equal(before[0], lat.field("g")) and np.array_equal(before[1], lat.field("tau"))
