"""lbm_get_field into new and old memory, at any address: every value, and nothing beside the array."""
import ctypes
import mmap

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


@pytest.mark.parametrize("nx,ny", [(1, 3), (31, 9), (64, 128), (129, 131), (300, 400)])
@pytest.mark.parametrize("form", ["populations", "fp16", "three"])
def test_new_memory_is_filled_and_nothing_else(lbm, nx, ny, form):
    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, collapse_h=int(form == "fp16"), storage=int(form == "fp16"), ncomp=3 if form == "three" else 2)
    lat = lbm.Lattice(p)
    lat.set_fields(inputs.bubble_fields(nx, ny, p["ncomp"], p["xi"], [(nx / 2, ny / 3, 5.0, 3)], seed=1, noise=1e-4))
    lat.step(3)
    library = lbm.load_library()
    for name in ("C1", "C3", "rho", "ux", "mu1", "tau", "g", "SV") + (() if form == "fp16" else ("h",)):
        want = lat.field(name)
        for before in (0, 1, 511, 8190):  # doubles before the array: page boundaries anywhere in it
            memory = mmap.mmap(-1, 8 * (before + want.size + 9))
            values = np.frombuffer(memory, dtype=np.float64)
            array = values[before:before + want.size]
            if before:
                values[before - 1] = -7.5
            values[before + want.size] = -8.5
            at = array.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
            assert library.lbm_get_field(lat.h, lbm.FIELD_IDS[name], at, want.size) == 0
            assert np.array_equal(array, want.ravel()), name
            assert values[before + want.size] == -8.5 and (not before or values[before - 1] == -7.5)
            assert not values[before + want.size + 1:].any() and not values[:max(0, before - 1)].any()
            del values, array


@pytest.mark.parametrize("nx,ny", [(8, 320), (8, 321), (64, 40), (41, 64), (64, 64), (64, 65), (128, 64), (91, 91)])
@pytest.mark.parametrize("ncomp", [2, 3])
def test_small_fields_equal_the_stored_state(lbm, nx, ny, ncomp):
    """Either side of the sizes that are converted on the host, against the arena's own planes (include/lbm.h)."""
    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, ncomp=ncomp)
    lat = lbm.Lattice(p)
    lat.set_fields(inputs.bubble_fields(nx, ny, ncomp, p["xi"], [(nx / 2, ny / 3, 3.0, 3)], seed=1, noise=1e-4))
    pitch, nh = (nx + 31) // 32 * 32, ncomp - 1
    plane = (ny * pitch * 4 + 255) // 256 * 64
    for steps in (0, 2):  # buffer 0 holds the state after an even number of steps
        lat.step(steps)
        words = lat.arena.cpu().numpy().view(np.float32)

        def populations(first, nq):
            v = words[first:first + nq * ny * pitch].reshape(ny, pitch // 32, nq, 32)
            return v.transpose(2, 0, 1, 3).reshape(nq, ny, pitch)[:, :, :nx].astype(np.float64)

        assert np.array_equal(lat.field("g"), populations(0, 9))
        assert np.array_equal(lat.field("h").reshape(9 * nh, ny, nx), populations(18 * plane, 9 * nh))
        tau = words[(18 + 18 * nh) * plane:][:ny * pitch].reshape(ny, pitch)[:, :nx]
        assert np.array_equal(lat.field("tau"), tau.astype(np.float64))
