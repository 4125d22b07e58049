"""Graphs of about as many rows as the short-row aggregation has warps (148 x 32, and 148 x 24 for bytes): one row per warp below."""
import pytest

from test_gpu_short_rows import ctx, test_hidden_and_narrow_layers as check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,d_out", [(300, 8), (300, 64), (300, 100), (90, 130)])
@pytest.mark.parametrize("n,e,seed", [(4736, 15000, 21), (4737, 15000, 22), (3552, 20000, 23), (3553, 20000, 24)])
def test_rows_around_the_number_of_warps(ctx, n, e, seed, d_in, d_out):  # noqa: F811
    check(ctx, n, e, seed, d_in, d_out)
