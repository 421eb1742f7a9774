"""lbm_observables at the edges of its 32 x 8 tiles, every state form, against FP64
sums of the fields that lbm_get_field returns.

Tolerances: the sums are FP64 sums of the same FP32 C (compensated runs), so masses and
centroid sums agree to 1e-11 of the sum of magnitudes; the velocity in the sums and in the
fields is the same FP32 expression, in which the compiler may fuse a product differently: a
few units of 2^-23 of its terms, taken as 1e-5 of the sum of magnitudes."""
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


@pytest.mark.parametrize("nx,ny", [(4, 3), (31, 9), (32, 8), (33, 7), (64, 16), (100, 57), (400, 700)])
@pytest.mark.parametrize("form,gas", [("populations", 3), ("collapsed", 3), ("fp16", 3), ("three", 3), ("three", 2),
                                      ("open", 3)])
def test_observables_at_tile_edges(lbm, nx, ny, form, gas):
    p, _ = inputs.small_case()
    p = dict(p, nx=nx, ny=ny, gravity=1e-6, gas_comp=gas)
    if form in ("collapsed", "fp16"):
        p.update(collapse_h=1, periodic_y=1)
    if form == "fp16":
        p["storage"] = 1
    if form == "three":
        p["ncomp"] = 3
    if form == "open":
        p.update(open_x=1, u_in=0.01)
    discs = [(nx * 0.6, ny * 0.4, min(nx, ny) / 4 + 1, 3)] + ([(nx * 0.2, ny * 0.7, 3.0, 2)] if form == "three" else [])
    C = inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=3, noise=1e-4)
    u = 1e-3 * np.random.default_rng(nx).normal(size=(ny, nx))
    lat = lbm.Lattice(p)
    lat.set_fields(C, ux=u, uy=0.01 - u)
    lat.step(1)
    raw = np.array(lat.observables()["raw"])
    c = [lat.field(f"C{i}") for i in (1, 2, 3)]
    cg, ux, uy = c[gas - 1], lat.field("ux"), lat.field("uy")
    x, y = np.meshgrid(np.arange(nx, dtype=float), np.arange(ny, dtype=float))
    terms = c + [np.where(v > 0.5, v, 0.0) for v in c] + [cg, cg * x, cg * y, cg * ux, cg * uy]
    for i, t in enumerate(terms):
        tol = (1e-5 if i >= 9 else 1e-11) * np.abs(t).sum() + 1e-30
        assert abs(raw[i] - t.sum()) <= tol, (i, raw[i], t.sum())
    yy, xx = np.nonzero(cg > 0.5)
    want = [xx.min(), xx.max(), yy.min(), yy.max()] if xx.size else [-1] * 4
    assert raw[11:].tolist() == [float(v) for v in want]
