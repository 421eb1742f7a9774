"""FP16 batches with one launch per step are tuned and run to their end like the others: the
cases of a tuned batch against the same cases on lattices of their own, bit for bit."""
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


@pytest.mark.parametrize("ncomp", [2, 3])
@pytest.mark.parametrize("shapes", [[(20, 3)], [(100, 200)] * 12, [(33, 45), (150, 90), (7, 300)]])
def test_fp16_batches_are_tuned(lbm, ncomp, shapes):
    cases = []
    for i, (nx, ny) in enumerate(shapes):
        p, _ = inputs.small_case(mobility=i % 2)
        p = dict(p, nx=nx, ny=ny, ncomp=ncomp, collapse_h=1, storage=1)
        discs = [(nx / 2, ny / 3, min(nx, ny) / 6 + 2, 3)] + ([(nx / 4, ny / 1.5, 3.0, 2)] if ncomp == 3 else [])
        cases.append((p, inputs.bubble_fields(nx, ny, ncomp, p["xi"], discs, seed=i, noise=1e-5)))
    batch = lbm.Batch([p for p, _ in cases])
    for i, (_, C) in enumerate(cases):
        batch.case(i).set_fields(C)
    assert batch.autotune(reps=1) >= 0
    batch.step(19)
    for i, (p, C) in enumerate(cases):
        lat = lbm.Lattice(p)
        lat.set_fields(C)
        lat.step(19)
        for f in ("g", "tau", "C1"):
            assert np.array_equal(batch.case(i).field(f), lat.field(f)), (i, f)
    outcomes = batch.run(window=10, max_steps=20)
    assert len(outcomes) == len(cases)
