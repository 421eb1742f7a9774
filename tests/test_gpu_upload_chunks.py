"""Large page-locked fields go up in row chunks beside the set-up, others whole: the same bits everywhere."""
import numpy as np
import pytest

from paper_2207_09431_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periodic_y", [0, 1])
@pytest.mark.parametrize("extra", [{}, {"collapse_h": 1, "storage": 1}, {"fd_scheme": 1}, {"ncomp": 3}])
@pytest.mark.parametrize("given", [(), ("p", "ux", "uy"), ("uy",)])
def test_chunks_equal_one_upload(periodic_y, extra, given):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_09431_gb300 import lbm

    nx, ny = (2101, 2003) if extra.get("ncomp", 2) == 2 else (1050, 2003)  # C of just over 32 MB, ragged chunks
    p, _ = inputs.small_case()
    p = dict(p, nx=nx, ny=ny, periodic_y=periodic_y, **extra)
    r = np.random.default_rng(1)
    C = r.uniform(0.0, 0.5, size=(p.get("ncomp", 2) - 1, ny, nx))
    assert C.nbytes >= 32 << 20
    f = {k: 1e-3 * r.normal(size=(ny, nx)) for k in given}
    whole, chunks = lbm.Lattice(p), lbm.Lattice(p)
    whole.set_fields(C, **f)
    pinned = {k: torch.from_numpy(v).pin_memory() for k, v in dict(f, C=C).items()}
    chunks.set_fields(**{k: v.numpy() for k, v in pinned.items()})
    torch.cuda.synchronize()
    assert torch.equal(whole.arena, chunks.arena)  # state, staged fields and all
