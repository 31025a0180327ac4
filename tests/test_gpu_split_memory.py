"""What an FP64 handle without wall sides holds between calls: the planes that the two passes of a step hand to each other lie
in the state copy that is not current and in the staging buffer, so a handle takes 2 x 17 planes of state and 9 of staging, no
more than the marching kernel's; and a run resumed from a checkpoint, which rebuilds them, continues bitwise."""
import numpy as np
import pytest

from paper_2002_03644_gb300 import inputs
from test_gpu_parity import _env, hl  # noqa: F401
from test_gpu_split import STATE, compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2048, 2048), (768, 768)])
def test_memory_of_a_handle(hl, nx, ny):  # noqa: F811
    import torch
    small = inputs.uniform(32, 32)
    hl.Solver(32, 32, precision=0, **small.params()).close()  # what the first handle of a process loads
    before = torch.cuda.mem_get_info()[0]
    s = hl.Solver(nx, ny, precision=0, **small.params())
    used = before - torch.cuda.mem_get_info()[0]
    s.close()
    # three large allocations and the small ones, each rounded up to 2 MB
    assert used <= 43 * nx * ny * 8 + 8 * 2 ** 21


@pytest.mark.parametrize("nx,ny", [(45, 37), (769, 768)])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 2, 2, 1)])
@pytest.mark.parametrize("sigma,phi", [(0.0, 0), (0.4, 1)])
def test_resumed_run_continues_bitwise(hl, nx, ny, bc, sigma, phi):  # noqa: F811
    case = inputs.random_smooth(nx, ny, seed=9, amp=0.03, u0=(-0.05, 0.04), theta0=0.2, mu=2e-3, sigma=sigma, bc=bc, bc_state=STATE)
    case.phi_mode = phi
    a = hl.Solver(nx, ny, precision=0, **case.params())
    a.init(*case.fields())
    a.step(5)
    blob = a.state()
    b = hl.Solver(nx, ny, precision=0, **case.params())
    b.init(*[np.roll(f, 3, axis=1) for f in case.fields()])
    b.step(2)
    b.set_state(blob)
    a.macros()  # reading the fields between two steps changes nothing
    for s in (a, b):
        s.step(4)
    assert np.array_equal(a.state(), b.state())
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny,march", [(769, 768, -1), (45, 37, 0)])
def test_checkpoint_of_another_kernel(hl, nx, ny, march):  # noqa: F811
    """13 planes into a handle whose own checkpoints hold 17, and 17 into one of 13."""
    case = inputs.random_smooth(nx, ny, seed=9, amp=0.03, u0=(-0.05, 0.04), theta0=0.2, mu=2e-3, sigma=0.4, bc=(1, 2, 2, 1), bc_state=STATE)
    with _env(HLBM_MARCH=march):
        a = hl.Solver(nx, ny, precision=0, **case.params())
    b = hl.Solver(nx, ny, precision=0, **case.params())
    a.init(*case.fields())
    a.step(3)
    assert a.state().size != hl.hlbm_state_bytes(b.h)
    b.set_state(a.state())
    out = []
    for s in (b, a):
        s.step(5)
        m = s.macros()
        m["F"] = s.populations()
        out.append(m)
        s.close()
    compare(*out)
