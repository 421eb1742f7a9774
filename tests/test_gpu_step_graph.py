"""Repeated runs on a created stream, where one captured graph serves both buffers, against
direct launches: the same bits for even and odd runs and runs around the graph's length."""
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


@pytest.mark.parametrize("runs", [(34, 34, 34), (17, 17, 17, 17), (16, 17, 18, 33), (49, 32, 1, 64), (20, 3, 20)])
@pytest.mark.parametrize("fd_scheme", [0, 1])
def test_repeated_runs_equal_direct_launches(lbm, runs, fd_scheme):
    import torch

    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=50, ny=37, fd_scheme=fd_scheme)
    C = inputs.bubble_fields(50, 37, 2, p["xi"], [(25, 12, 7.0, 3)], seed=3, noise=1e-5)
    direct, replay = lbm.Lattice(p), lbm.Lattice(p, stream=torch.cuda.Stream())
    for lat in (direct, replay):
        lat.set_fields(C)
    for n in runs:
        for lat in (direct, replay):
            lat.step(n)
        for f in ("g", "h", "tau", "shear"):
            assert np.array_equal(replay.field(f), direct.field(f)), (n, f)
