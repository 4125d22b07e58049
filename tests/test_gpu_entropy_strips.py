"""Strip widths of the entropy bins at the column counts where they change, against the oracle."""
import pytest

from test_gpu_entropy import activations, check, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 8, 9, 16, 17, 24, 25, 32, 33])
@pytest.mark.parametrize("n,M", [(1025, 100), (40000, 1750), (3000, 3500)])
def test_strip_widths(ctx, n, d, M):  # noqa: F811
    check(ctx, activations(n, d, n + d), M)


@pytest.mark.parametrize("d,M", [(17, 200), (25, 1750), (32, 64)])
def test_one_wide_strip(ctx, d, M):  # noqa: F811
    check(ctx, activations(1 << 20, d, d), M)
