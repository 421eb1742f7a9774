"""Batches whose work is shared out in equal lists (several pieces per CTA) against the
same cases on lattices of their own, bit for bit, whichever configuration the
autotuner picks: many cases, few, and ragged ones, one launch per step and persistent."""
import numpy as np
import pytest

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


def case(nx, ny, i, form):
    p, _ = inputs.small_case(mobility=i % 2)
    p = dict(p, nx=nx, ny=ny, periodic_y=i % 3 == 2, pl_n=0.6 + 0.05 * (i % 5))
    if form in ("collapsed", "fp16"):
        p["collapse_h"] = 1
    if form == "fp16":
        p["storage"] = 1
    discs = [(nx / 2, ny / 3, min(nx, ny) / 6 + 2, 3)]
    if form == "three":
        p["ncomp"] = 3
        discs.append((nx / 4, ny / 1.5, 4.0, 2))
    C = inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=i, noise=1e-5, periodic_y=bool(p["periodic_y"]))
    u = 1e-3 * np.random.default_rng(i).normal(size=(ny, nx))
    return p, C, u


@pytest.mark.parametrize("shapes", [[(100, 200)] * 60, [(150, 300), (33, 45), (200, 400), (7, 500), (300, 60)],
                                    [(20, 3)], [(16, 8), (3, 3)], [(101, 97)] * 5 + [(58, 640)] * 30])
@pytest.mark.parametrize("form", ["populations", "collapsed", "fp16", "three"])
@pytest.mark.parametrize("persistent", [False, True])
def test_shared_work_equals_single_lattices(lbm, shapes, form, persistent):
    if form == "fp16" and not persistent:
        pytest.skip("per-step FP16 batches are not tuned")
    cases = [case(nx, ny, i, form) for i, (nx, ny) in enumerate(shapes)]
    batch = lbm.Batch([p for p, _, _ in cases])
    batch.set_persistent(persistent)
    for i, (p, C, u) in enumerate(cases):
        batch.case(i).set_fields(C, ux=u, uy=-u)
    batch.autotune(reps=1)
    batch.step(5)
    if len(cases) > 4:
        batch.set_active(2, False)  # another list
    batch.step(18)
    for i in sorted({0, 1, 2, len(cases) - 1} & set(range(len(cases)))):
        p, C, u = cases[i]
        lat = lbm.Lattice(p)
        lat.set_fields(C, ux=u, uy=-u)
        lat.step(5 if i == 2 and len(cases) > 4 else 23)
        for f in ("g", "tau", "C1"):
            assert np.array_equal(batch.case(i).field(f), lat.field(f)), (i, f)
