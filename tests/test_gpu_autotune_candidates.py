"""lbm_autotune chooses among the configurations that suit the lattice's size, and values stay the same bits."""
import re

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


@pytest.mark.parametrize("nx,ny", [(3, 3), (64, 40), (98, 98), (180, 180), (200, 200), (256, 256), (300, 400), (700, 500)])
@pytest.mark.parametrize("form", ["populations", "collapsed", "fp16", "three"])
def test_chosen_configuration_suits_the_size(lbm, nx, ny, form):
    import torch

    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, collapse_h=int(form in ("collapsed", "fp16")), storage=int(form == "fp16"),
             ncomp=3 if form == "three" else 2)
    C = inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], [(nx / 2, ny / 3, min(nx, ny) / 6, 3)], seed=1, noise=1e-5)
    tuned, plain = lbm.Lattice(p), lbm.Lattice(p)
    for lat in (tuned, plain):
        lat.set_fields(C)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def tiles(tx, ty):
        return -(-nx // tx) * -(-ny // ty)

    for lat, name in ((tuned, tuned.autotune(reps=2)), (plain, lbm.lbm_kernel_name(plain.h, 0))):
        tile = re.match(r"k_step_fused\[(\d+)x(\d+)/\d+/(\d)\]", name)
        if tile and name not in [f"k_step_fused[{n}]" for n in ("32x8/352/3", "32x8/448/2", "32x16/640/2", "64x8/704/1",
                                                                 "32x8/352/2")]:
            tx, ty, per_sm = map(int, tile.groups())
            assert tiles(tx, ty) <= per_sm * sms, name
        if form == "three" and tiles(16, 8) <= 2 * sms or form != "three" and tiles(16, 4) <= sms:
            assert tile, name
    for lat in (tuned, plain):
        lat.step(5)
    for f in ("g", "tau", "C1"):
        assert np.array_equal(tuned.field(f), plain.field(f))
