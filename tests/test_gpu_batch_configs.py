"""Every launch configuration of a batch, selected one after the other (shared lists with several pieces a
CTA and empty items among them), against the same cases on lattices of their own, bit for bit."""
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


def case(nx, ny, i, form):
    p, _ = inputs.small_case(mobility=i % 2)
    p = dict(p, nx=nx, ny=ny, periodic_y=i % 3 == 2, pl_n=0.6 + 0.05 * (i % 5))
    if form in ("collapsed", "fp16"):
        p["collapse_h"] = 1
    if form == "fp16":
        p["storage"] = 1
    discs = [(nx / 2, ny / 3, min(nx, ny) / 6 + 2, 3)]
    if form == "three":
        p["ncomp"] = 3
        discs.append((nx / 4, ny / 1.5, 4.0, 2))
    C = inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], discs, seed=i, noise=1e-5, periodic_y=bool(p["periodic_y"]))
    u = 1e-3 * np.random.default_rng(i).normal(size=(ny, nx))
    return p, C, u


# one share a strip and less; more strips than CTA slots, so that a share has several pieces (of several cases);
# shares of unequal numbers of pieces, padded with empty items
SHAPES = [[(20, 3), (101, 97)], [(33, 12)] * 700, [(58, 640)] * 20 + [(7, 20), (150, 33)] * 150]


@pytest.mark.parametrize("shapes", range(len(SHAPES)))
@pytest.mark.parametrize("form", ["populations", "collapsed", "fp16", "three"])
@pytest.mark.parametrize("persistent", [False, True])
def test_every_configuration_equals_single_lattices(lbm, shapes, form, persistent):
    cases = [case(nx, ny, i, form) for i, (nx, ny) in enumerate(SHAPES[shapes])]
    watched = sorted({0, 1, len(cases) // 2, len(cases) - 2, len(cases) - 1})
    want = {}
    for i in watched:
        p, C, u = cases[i]
        lat = lbm.Lattice(p)
        lat.set_fields(C, ux=u, uy=-u)
        lat.step(19)
        want[i] = {f: lat.field(f) for f in ("g", "tau", "C1")}
    batch = lbm.Batch([p for p, _, _ in cases])
    batch.set_persistent(persistent)
    count = lbm.lbm_batch_kernel_config_count(batch.b)
    assert count >= 2
    for config in range(count):
        for i, (_, C, u) in enumerate(cases):
            batch.case(i).set_fields(C, ux=u, uy=-u)
        lbm.lbm_batch_set_kernel_config(batch.b, config)
        batch.step(19)
        for i in watched:
            for f, v in want[i].items():
                assert np.array_equal(batch.case(i).field(f), v), (config, i, f)
    for config in (-1, count):
        with pytest.raises(lbm.LbmError):
            lbm.lbm_batch_set_kernel_config(batch.b, config)
