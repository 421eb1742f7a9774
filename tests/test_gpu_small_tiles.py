"""The small-tile launch configurations and the size rule that picks a handle's
first configuration: the same fields, bit for bit, as the row sweep (configuration
0) at the edges of the tiles, walls and periodic, every state form."""
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


def fields(lbm, p, C, config, u):
    lat = lbm.Lattice(p)
    if config is not None:
        lbm.lbm_set_kernel_config(lat.h, config)
    lat.set_fields(C, ux=u, uy=-u)
    lat.step(5)
    return [lat.field(f) for f in ("g", "tau", "C1", "shear") + (() if p.get("collapse_h") else ("h",))]


@pytest.mark.parametrize("nx,ny", [(1, 3), (15, 5), (16, 4), (17, 7), (32, 8), (33, 9), (50, 31)])
@pytest.mark.parametrize("form", ["populations", "collapsed", "fp16", "three"])
def test_small_tiles_equal_the_sweep(lbm, nx, ny, form):
    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, periodic_y=nx % 2)
    if form in ("collapsed", "fp16"):
        p["collapse_h"] = 1
    if form == "fp16":
        p["storage"] = 1
    discs = [(nx / 2, ny / 3, 4.0, 3)]
    if form == "three":
        p["ncomp"] = 3
        discs.append((nx / 3, ny / 2, 3.0, 2))
    C = inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=nx, noise=1e-5)
    u = 1e-3 * np.random.default_rng(ny).normal(size=(ny, nx))
    n = lbm.lbm_kernel_config_count(lbm.Lattice(p).h)
    want = fields(lbm, p, C, 0, u)
    for config in [None] + list(range(n - (2 if form == "three" else 3), n)):
        for a, b in zip(fields(lbm, p, C, config, u), want):
            assert np.array_equal(a, b), (config, nx, ny)


@pytest.mark.parametrize("nx,ny", [(64, 128), (100, 200), (150, 300), (200, 400), (300, 600), (2, 3000), (3000, 3)])
def test_first_configuration_steps_like_the_sweep(lbm, nx, ny):
    p, _ = inputs.small_case()
    p = dict(p, nx=nx, ny=ny)
    C = inputs.bubble_fields(nx, ny, 2, p["xi"], [(nx / 2, ny / 3, 12.0, 3)], seed=1, noise=1e-6)
    u = 1e-3 * np.random.default_rng(2).normal(size=(ny, nx))
    for a, b in zip(fields(lbm, p, C, None, u), fields(lbm, p, C, 0, u)):
        assert np.array_equal(a, b)
