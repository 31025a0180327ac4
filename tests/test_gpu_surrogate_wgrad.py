"""The surrogate's gradients over channel counts, image widths and batch sizes at the edges of the weight-gradient kernel:
results of 1 to 4 blocks of 16 channels each way, widths that divide into its stages of 64 pixels and that do not, images
smaller than a stage, and pixel counts just below and above one chunk of 16384.

Tolerance: as in test_gpu_surrogate.py, element by element within 1e-2 of the tensor's largest element against the reference
with the same BF16 roundings.  What remains is FP32 summation (up to 16384 products in one chain of tensor-core additions,
each truncated to 24 bits: 1024 steps of 2^-24, 6e-5) and BF16 roundings flipped by it."""
import numpy as np
import pytest

from oracle import surrogate_oracle as S
from test_gpu_surrogate import env, unpack  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,shape", [
    ((4, 16, 4), (1, 1, 1)),
    ((3, 33, 20, 3), (2, 5, 7)),
    ((4, 48, 48, 4), (1, 8, 96)),
    ((4, 32, 64, 48, 4), (2, 3, 128)),
    ((20, 64, 16, 20), (1, 64, 33)),
    ((4, 64, 64, 4), (1, 63, 260)),
    ((4, 64, 64, 4), (1, 64, 256)),
    ((4, 64, 64, 4), (1, 65, 256)),
], ids=lambda v: "x".join(map(str, v)))
def test_gradients_at_the_edges_of_the_weight_gradient_kernel(env, widths, shape):  # noqa: F811
    torch, hlbm, surrogate = env
    B, H, W = shape
    sur = surrogate.Surrogate(widths, H, W, batch_max=B, seed=4)
    params = unpack(widths, sur.params())
    rng = np.random.default_rng(6)
    x = rng.normal(size=(B, H, W, widths[0])).astype(np.float32)
    t = (x + 0.1 * rng.normal(size=x.shape)).astype(np.float32)
    sur.forward(torch.from_numpy(x).cuda())
    hlbm.hlbm_sur_backward(sur.s, torch.from_numpy(t).cuda())
    g = sur.grads().astype(np.float64)
    sur.synchronize()
    sur.close()
    y, cache = S.forward_bf16(params, x.transpose(0, 3, 1, 2).astype(np.float64))
    o = 0
    for l, (dw, db) in enumerate(S.backward_bf16(cache, y, t.transpose(0, 3, 1, 2).astype(np.float64))):
        for name, ref in (("dW", dw), ("db", db)):
            err = float(np.abs(g[o:o + ref.size].reshape(ref.shape) - ref).max() / np.abs(ref).max())
            assert err < 1e-2, (name, l, err)
            o += ref.size
