"""The tile shape that small FP32 grids take (16 x 16 cells, one per thread) gives the bits of the 32 x 32 tile
(HLBM_FP32_TILE=4) on every boundary kind, at grids of one cell, below, at and above one tile, and FP64 walls on each of the
three tile shapes agree with the oracle-checked FP64 form to rounding (same formulas, tile shape only: exact equality)."""
import numpy as np
import pytest

from paper_2002_03644_gb300 import inputs
from test_gpu_parity import _env, hl  # noqa: F401

pytestmark = pytest.mark.gpu

STATE = np.array([[1.02, 0.08, 0.01, 0.21], [0.98, 0.05, -0.02, 0.19], [1.01, 0.06, 0.03, 0.2], [0.99, 0.07, 0.0, 0.205]])


@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 2, 2, 1), (0, 0, 3, 3), (3, 3, 1, 2)])
@pytest.mark.parametrize("nx,ny", [(2, 2), (15, 17), (16, 16), (33, 48), (150, 70)])
@pytest.mark.parametrize("sigma,phi", [(0.0, 0), (0.6, 1)])
def test_small_tile_gives_the_bits_of_the_large_one(hl, bc, nx, ny, sigma, phi):  # noqa: F811
    case = inputs.random_smooth(nx, ny, seed=3, amp=0.03, u0=(0.05, -0.02), theta0=0.2, mu=2e-3, sigma=sigma, bc=bc, bc_state=STATE)
    case.phi_mode = phi
    out = []
    for env in ({}, {"HLBM_FP32_TILE": 4}):
        with _env(HLBM_MARCH=-1, HLBM_FP32_TMA=-1, **env):
            s = hl.Solver(nx, ny, precision=1, **case.params())
            s.init(*case.fields())
            s.step(7)
            out.append(s.populations())
            s.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("nx,ny", [(90, 90), (96, 200)])
def test_fp64_wall_tiles_are_the_same_function(hl, nx, ny):  # noqa: F811
    """A periodic flow is the same whether a row is cut into tiles of 8 or 16: a case twice as wide, of two copies side by
    side, takes the next tile shape and must repeat the narrow one's columns (within rounding that the compiler may choose)."""
    case = inputs.random_smooth(nx, ny, seed=4, amp=0.03, u0=(0.05, 0.0), theta0=0.2, mu=2e-3, sigma=0.5, bc=(0, 0, 3, 3), bc_state=STATE)
    out = []
    for k in (1, 4):
        s = hl.Solver(k * nx, ny, precision=0, **case.params())
        s.init(*[np.ascontiguousarray(np.tile(f, (1, k))) for f in case.fields()])
        s.step(7)
        out.append(s.populations())
        s.close()
    assert np.abs(out[1][:, :, :nx] - out[0]).max() <= 1e-13
