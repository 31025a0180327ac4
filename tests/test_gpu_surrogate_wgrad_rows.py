"""The surrogate's gradients on images whose rows are several segments of 256 columns, where the kernel with all taps per CTA
takes halo columns from the neighbouring segment and a chunk may end in one segment and begin in the next: on either side of
the number of chunks from which it is taken, heights of one row and below a chunk's 64, and a width (384) that is no multiple
of a segment.  Tolerance and reference as in test_gpu_surrogate_wgrad.py."""
import pytest

from test_gpu_surrogate import env  # noqa: F401
from test_gpu_surrogate_wgrad import test_gradients_at_the_edges_of_the_weight_gradient_kernel as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,shape", [
    ((4, 64, 64, 4), (1, 1, 512)),
    ((4, 64, 48, 4), (3, 21, 768)),
    ((4, 64, 64, 4), (2, 33, 1280)),
    ((4, 64, 64, 4), (1, 65, 384)),
    ((20, 64, 20), (1, 500, 512)),
    ((20, 64, 20), (1, 512, 512)),
    ((4, 32, 16, 4), (2, 511, 512)),
    ((4, 32, 16, 4), (2, 512, 512)),
], ids=lambda v: "x".join(map(str, v)))
def test_gradients_over_several_segments(env, widths, shape):  # noqa: F811
    check(env, widths, shape)
