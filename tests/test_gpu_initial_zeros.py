"""Initial populations where nothing acts (one phase, no gravity) are +0, as w p + rho cs^2 (Gamma - w)
- Phi / 2 with every term zero gives them: the same bits with the velocity left out or given as zero."""
import numpy as np
import pytest

from paper_2207_09431_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [{}, {"collapse_h": 1}, {"fd_scheme": 1}, {"ncomp": 3}])
def test_no_negative_zeros_at_rest(extra):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_09431_gb300 import lbm

    p, _ = inputs.small_case()
    p = dict(p, nx=50, ny=70, gravity=0.0, **extra)
    C = inputs.bubble_fields(50, 70, p.get("ncomp", 2), p["xi"], [(25, 30, 8.0, 3)])
    rest, given = lbm.Lattice(p), lbm.Lattice(p)
    rest.set_fields(C)
    given.set_fields(C, ux=np.zeros((70, 50)))
    g = rest.field("g")
    assert (g == 0).sum() > 1000 and not np.signbit(g[g == 0]).any()
    assert g.tobytes() == given.field("g").tobytes()
