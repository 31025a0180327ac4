"""A NaN in the entropy of one cell spreads through the two-pass FP64 step as far as through the kernels that compare doubles
(the tiled one on small grids, the marching one, which also keeps the level's values, on large ones): a limited slope beside
it is 0, not NaN.  The state is set from a checkpoint, so that the populations around the cell are finite."""
import numpy as np
import pytest

from paper_2002_03644_gb300 import inputs
from test_gpu_parity import _env, hl  # noqa: F401

pytestmark = pytest.mark.gpu

PLANE_S = 9


@pytest.mark.parametrize("u0", [(0.06, 0.03), (-0.06, -0.03)])
@pytest.mark.parametrize("nx,ny,march", [(45, 37, -1), (800, 760, 0)])
def test_nan_spreads_no_further_than_by_comparison(hl, nx, ny, march, u0):  # noqa: F811
    case = inputs.random_smooth(nx, ny, seed=8, amp=0.01, u0=u0, theta0=0.2, mu=1e-3)
    pitch = (nx + 31) // 32 * 32
    out = []
    for env in ({}, {"HLBM_MARCH": march}):
        with _env(**env):
            s = hl.Solver(nx, ny, precision=0, **case.params())
        s.init(*case.fields())
        blob = s.state()
        planes = 13 if march < 0 else 17
        state = blob[-planes * pitch * ny * 8:].view(np.float64).reshape(planes, ny, pitch)
        state[PLANE_S, ny // 2, nx // 2] = np.nan
        s.set_state(blob)
        masks = []
        for _ in range(3):
            s.step(1)
            m = s.macros()
            masks.append({k: np.isnan(v) for k, v in m.items()})
        out.append(masks)
        s.close()
    for a, b in zip(*out):
        for k in a:
            assert b[k].any() and np.array_equal(a[k], b[k]), k
