"""G_H of the tensor-core kernel at its edges, with the tolerance of the gradient tests: one chunk of channels and several tiles
per block, slices of inputs, signs of W that stay in shared memory (up to 65536 / N channels) and that do not (256 inputs, 257 and 512 channels)."""
import pytest

from test_gpu_backward import B, ctx, run_case  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,d_in,d_out", [(1, 0, 4, 1), (127, 500, 64, 64), (40000, 60000, 60, 5), (39000, 60000, 256, 64), (19000, 60000, 128, 130),
                                            (20000, 60000, 260, 70), (300, 2000, 516, 256), (300, 2000, 256, 257), (30000, 60000, 256, 512), (20100, 60000, 132, 300), (9600, 30000, 64, 512)])
def test_input_gradient(B, ctx, n, m, d_in, d_out):  # noqa: F811
    run_case(B, ctx, n, m, d_in, d_out, seed=d_in + d_out)
