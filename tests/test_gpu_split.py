"""The two-pass FP64 step (the FP64 default without wall sides) against the tiled FP64 kernel (HLBM_MARCH=-1), which computes
the same formulas with IEEE divisions and recomputed halos: every boundary kind and corner, both Phi forms, sigma = 0 and > 0,
the ablations, zero viscosity, and grids of one cell, one column, one row and around the 32-column blocks.

Grids up to 768^2 derive the level macros from F (13-plane checkpoints), larger ones keep them: one such grid is among them.

Tolerance: the two differ by roundings of 2^-53 relative per operation.  A step chains about 30 operations on values of the
fields' scale and 8 steps follow each other, with at most second differences in between (factor 4): 8 * 30 * 4 * 2^-53 = 1e-13;
1e-12 of the field's scale is asserted (s and a1 at their own scale, where a1 is a difference of velocities of relative size
0.01: 1e-10)."""
import numpy as np
import pytest

from paper_2002_03644_gb300 import inputs
from test_gpu_parity import BCS, _env, hl  # noqa: F401

pytestmark = pytest.mark.gpu

STATE = np.array([[1.02, 0.08, 0.01, 0.21], [0.98, 0.05, -0.02, 0.19], [1.01, 0.06, 0.03, 0.2], [0.99, 0.07, 0.0, 0.205]])


def run(hl, case, steps, **env):  # noqa: F811
    with _env(**env):
        s = hl.Solver(case.nx, case.ny, precision=0, **case.params())
    s.init(*case.fields())
    s.step(steps)
    m = s.macros()
    m["F"] = s.populations()
    s.close()
    return m


def compare(a, b):
    for k in b:
        tol = (1e-10 if k == "a1" else 1e-12) * max(float(np.abs(b[k]).max()), 1e-6)
        assert float(np.abs(a[k] - b[k]).max()) <= tol, k


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("kw", [dict(sigma=0.0), dict(sigma=0.5), dict(sigma=0.0, mu=0.0), dict(sigma=0.7, ablation=3)],
                         ids=["sigma0", "sigma", "inviscid", "ablation"])
@pytest.mark.parametrize("phi", [0, 1])
def test_two_passes_equal_the_tiled_kernel(hl, bc, kw, phi):  # noqa: F811
    ablation = kw.get("ablation", 0)
    kw = {k: v for k, v in kw.items() if k != "ablation"}
    case = inputs.random_smooth(45, 37, seed=8, amp=0.04, u0=(0.06, -0.03), theta0=0.2, bc=bc, bc_state=STATE,
                                **dict(dict(mu=3e-3), **kw))
    case.phi_mode, case.ablation = phi, ablation
    compare(run(hl, case, 8), run(hl, case, 8, HLBM_MARCH=-1))


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (2, 100), (31, 9), (32, 8), (33, 7), (400, 4), (65, 300), (769, 768)])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 2, 2, 1)])
def test_two_passes_at_the_edges_of_a_block(hl, nx, ny, bc):  # noqa: F811
    case = inputs.random_smooth(nx, ny, seed=9, amp=0.03, u0=(-0.05, 0.04), theta0=0.2, mu=2e-3, sigma=0.4, bc=bc, bc_state=STATE)
    compare(run(hl, case, 8), run(hl, case, 8, HLBM_MARCH=-1))
