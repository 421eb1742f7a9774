"""Values that are not finite come out as the formulas give them: a NaN or an infinity is not
hidden, and one in a place stays there."""
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


@pytest.mark.parametrize("ncomp,component", [(2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_density_of_a_node_that_is_not_finite(lbm, ncomp, component, bad):
    p, _ = inputs.small_case()
    p = dict(p, nx=40, ny=33, ncomp=ncomp, collapse_h=1)  # the state holds C itself
    C = inputs.bubble_fields(40, 33, ncomp, p["xi"], [(20, 12, 7.0, 3)])
    C[component, 5, 6] = C[component, 14, 20] = bad
    lat = lbm.Lattice(p)
    lat.set_fields(C)
    c = [lat.field(f"C{i}") for i in (1, 2, 3)]
    w = [np.clip(v, 0.0, 1.0) for v in c]  # keeps NaN
    want = (w[0] * p["rho"][0] + w[1] * p["rho"][1] + w[2] * p["rho"][2]) / (w[0] + w[1] + w[2])
    got = lat.field("rho")
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.isnan(want).any() == np.isnan(bad)
    assert np.allclose(got, want, rtol=1e-14, atol=0, equal_nan=True)


@pytest.mark.parametrize("rows", [5, 16, 17, 130])
def test_gradients_with_a_weight_that_is_infinite(lbm, rows):
    # a saturated unit (tanh = 1) leaves finite gradients, however many places of a 16-row tile are empty;
    # tolerance of tests/test_gpu_surrogate.py
    from oracle import mlp

    w = inputs.mlp_init(1, seed=3)
    w[0, 0] = np.inf
    r = np.random.default_rng(rows)
    X, T = np.abs(r.normal(size=(rows, 5))) + 0.1, r.normal(size=(rows, 2))
    Y, loss, g = lbm.Surrogate(w, max_batch=rows, max_rows=rows).forward_backward(0, X, T)
    params = inputs.mlp_unflatten(w[0])
    Yo, cache = mlp.forward(params, X)
    go = inputs.mlp_flatten(mlp.backward(params, cache, Yo, T))
    assert np.isfinite(go).all() and np.isfinite(g).all() and np.isfinite(loss)
    assert np.linalg.norm(Y - Yo) <= 1e-3 * np.linalg.norm(Yo)
    assert np.linalg.norm(g - go) <= 1e-3 * np.linalg.norm(go)
