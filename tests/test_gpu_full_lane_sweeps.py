"""Row sweeps of three, six and eight rows per pipeline step, and of 18 to 90 columns, against the
64-column sweep of two rows, bit for bit, at the edges of their strips and segments."""
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


@pytest.mark.parametrize("nx,ny", [(1, 3), (18, 8), (19, 9), (25, 5), (26, 6), (27, 7), (42, 4), (59, 3), (90, 12), (91, 13),
                                   (181, 37), (300, 599)])
@pytest.mark.parametrize("form", ["populations", "collapsed", "fp16", "three"])
@pytest.mark.parametrize("periodic_y", [0, 1])
def test_shapes_equal_the_two_row_sweep(lbm, nx, ny, form, periodic_y):
    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, periodic_y=periodic_y)
    if form in ("collapsed", "fp16"):
        p["collapse_h"] = 1
    if form == "fp16":
        p["storage"] = 1
    discs = [(nx / 2, ny / 3, 4.0, 3)]
    if form == "three":
        p["ncomp"] = 3
        discs.append((nx / 3, ny / 2, 3.0, 2))
    C = inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=nx, noise=1e-5, periodic_y=bool(periodic_y))
    u = 1e-3 * np.random.default_rng(ny).normal(size=(ny, nx))

    def fields(config):
        lat = lbm.Lattice(p)
        if config is not None:
            lbm.lbm_set_kernel_config(lat.h, config)
        lat.set_fields(C, ux=u, uy=-u)
        lat.step(5)
        return [lat.field(f) for f in ("g", "tau", "C1", "shear")]

    names, want = [], fields(0)
    lat = lbm.Lattice(p)
    for config in range(lbm.lbm_kernel_config_count(lat.h)):
        lbm.lbm_set_kernel_config(lat.h, config)
        names.append(lbm.lbm_kernel_name(lat.h, 0))
    shapes = ("26x6",) if form == "three" else ("90x2", "58x3", "42x4", "18x8", "26x6")
    for shape in shapes:
        config = [i for i, n in enumerate(names) if f"[{shape}/192/" in n]
        for a, b in zip(fields(config[0]), want):
            assert np.array_equal(a, b), shape
    for a, b in zip(fields(None), want):  # the configuration a handle starts with
        assert np.array_equal(a, b)
