"""The one-per-SM tiles of three components (32 x 12, 32 x 14) against the row sweep, bit
for bit, at the edges of their tiles, and the sizes around which the first configuration changes."""
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


@pytest.mark.parametrize("nx,ny", [(1, 3), (32, 12), (33, 13), (31, 14), (40, 15), (65, 28), (180, 180), (200, 200), (255, 256),
                                   (264, 264), (300, 300)])
@pytest.mark.parametrize("collapse_h", [0, 1])
@pytest.mark.parametrize("periodic_y", [0, 1])
def test_tiles_equal_the_sweep(lbm, nx, ny, collapse_h, periodic_y):
    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, ncomp=3, collapse_h=collapse_h, periodic_y=periodic_y)
    discs = [(nx / 2, ny / 3, 4.0, 3), (nx / 3, ny / 2, 3.0, 2)]
    C = inputs.bubble_fields(nx, ny, 3, p["xi"], discs, seed=nx, noise=1e-5, periodic_y=bool(periodic_y))
    u = 1e-3 * np.random.default_rng(ny).normal(size=(ny, nx))

    def fields(config):
        lat = lbm.Lattice(p)
        if config is not None:
            lbm.lbm_set_kernel_config(lat.h, config)
        lat.set_fields(C, ux=u, uy=-u)
        lat.step(5)
        return [lat.field(f) for f in ("g", "tau", "C1", "C2", "shear")]

    want = fields(0)
    lat = lbm.Lattice(p)
    for config in range(lbm.lbm_kernel_config_count(lat.h)):
        lbm.lbm_set_kernel_config(lat.h, config)
        if any(s in lbm.lbm_kernel_name(lat.h, 0) for s in ("[32x12/480/1]", "[32x14/544/1]")):
            for a, b in zip(fields(config), want):
                assert np.array_equal(a, b), config
    for a, b in zip(fields(None), want):
        assert np.array_equal(a, b)
