"""The two-kernel step (mixed difference scheme, open x) at the edges of its 32 x 4
tiles, against the FP64 oracle.

Tolerance: the rule of tests/test_gpu_parity.py, per field max(1e-5, 3 x the deviation
of the oracle's FP32 build on the same case), for its reason (FP32 arithmetic of
the same operations in the same order)."""
import numpy as np
import pytest

import oracle
from paper_2207_09431_gb300 import inputs

pytestmark = pytest.mark.gpu
FIELDS = ("C1", "p", "ux", "uy", "tau", "g", "h")


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_09431_gb300 import lbm as _lbm

    _lbm.load_library()
    return _lbm


def relerr(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-12 * b.size))


def swirl(nx, ny):
    x = 2.0 * np.pi * (np.arange(nx) + 0.3) / nx
    y = np.pi * (np.arange(ny) + 0.5) / ny
    ux = 2e-3 * np.sin(2.0 * y)[:, None] * np.cos(x)[None, :]
    uy = 2e-3 * (np.sin(y) ** 2)[:, None] * np.sin(x)[None, :]
    return inputs.round_to_fp32(ux), inputs.round_to_fp32(uy)


def check(lbm, p, C, steps, **fields):
    lat, orc, o32 = lbm.Lattice(p), oracle.Oracle(p), oracle.Oracle(p, "f32")
    for o in (lat, orc, o32):
        o.set_fields(C, **fields)
        o.step(steps)
    bad = {}
    for name in FIELDS:
        ref = orc.field(name)
        err, floor = relerr(lat.field(name), ref), relerr(o32.field(name), ref)
        if not err <= max(1e-5, 3.0 * floor):
            bad[name] = (err, floor)
    assert not bad, bad


@pytest.mark.parametrize("nx,ny", [(3, 3), (2, 9), (31, 4), (32, 5), (33, 7), (38, 10), (64, 8), (65, 41), (96, 3)])
@pytest.mark.parametrize("ncomp,periodic_y", [(2, 0), (2, 1), (3, 1)])
def test_mixed_scheme_at_tile_edges(lbm, nx, ny, ncomp, periodic_y):
    p, _ = inputs.small_case(mobility=1)
    p = dict(p, nx=nx, ny=ny, ncomp=ncomp, periodic_y=periodic_y, fd_scheme=1)
    discs = [(nx / 2, ny / 3, 3.0, 3)] + ([(nx / 4, ny / 2, 2.0, 2)] if ncomp == 3 else [])
    C = inputs.round_to_fp32(inputs.bubble_fields(nx, ny, ncomp, p["xi"], discs, seed=nx, noise=1e-6,
                                                  periodic_y=bool(periodic_y)))
    ux, uy = swirl(nx, ny)
    check(lbm, p, C, 7, ux=ux, uy=uy)


@pytest.mark.parametrize("nx,ny", [(4, 3), (5, 8), (32, 4), (33, 9), (34, 5), (65, 12)])
@pytest.mark.parametrize("fd_scheme,periodic_y", [(0, 0), (1, 0), (0, 1)])
def test_open_ends_at_tile_edges(lbm, nx, ny, fd_scheme, periodic_y):
    p, _, ux = inputs.open_channel_case(0.7, ny=ny, nx=nx, u_in=0.03)
    p = dict(p, rho=(1.0, 1.0, 0.1), tau=(0.8, 0.8, 0.5), gravity=1e-6, gas_comp=3, fd_scheme=fd_scheme,
             periodic_y=periodic_y)
    C = inputs.round_to_fp32(inputs.bubble_fields(nx, ny, 2, 4.0, [(2.0, ny / 2, 3.0, 3)], seed=nx, noise=1e-6,
                                                  periodic_y=bool(periodic_y)))
    check(lbm, p, C, 7, ux=inputs.round_to_fp32(ux))
