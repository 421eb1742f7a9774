"""Calls of few and many steps on a created stream, where runs of 16 and of 4 steps are captured at different
times on small and large lattices and replayed from either buffer, against direct launches: the same bits,
also where the launch configuration or the state changes between calls."""
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


@pytest.mark.parametrize("nx,ny", [(50, 37), (230, 201)])  # either side of the small lattices' rule (45000 nodes)
@pytest.mark.parametrize("runs", [(5,) * 7, (4, 5, 8, 5, 9, 5, 3, 6), (10, 40, 10, 7, 64), (13, 20, 5, 17, 5, 18, 16),
                                  (7, 33, 5, 12, 34, 5, 5)])
@pytest.mark.parametrize("change", [None, "configuration", "state"])
@pytest.mark.parametrize("extra", [{}, {"fd_scheme": 1}, {"ncomp": 3}])
def test_runs_equal_direct_launches(lbm, nx, ny, runs, change, extra):
    import torch

    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, **extra)
    C = inputs.bubble_fields(nx, ny, p.get("ncomp", 2), p["xi"], [(nx / 2, ny / 3, 7.0, 3)], seed=3, noise=1e-5)
    direct, replay = lbm.Lattice(p), lbm.Lattice(p, stream=torch.cuda.Stream())
    for lat in (direct, replay):
        lat.set_fields(C)
    for k, n in enumerate(runs):
        for lat in (direct, replay):
            if change == "state" and k == 3:
                lat.set_fields(C)
            if change == "configuration" and k % 2:
                lbm.lbm_set_kernel_config(lat.h, (3 * k) % lbm.lbm_kernel_config_count(lat.h))
            lat.step(n)
        for f in ("g", "h", "tau", "shear", "SV"):
            assert np.array_equal(replay.field(f), direct.field(f)), (k, n, f)
