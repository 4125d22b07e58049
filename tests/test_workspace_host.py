"""What bigcn_workspace_bytes() counts for the order that aggregates the packed bits first; host functions only."""
import ctypes

import pytest

N, NNZ = 2449029, 126149029


@pytest.fixture(scope="module")
def workspace():
    from paper_2210_13149_b200 import binding, build
    build.build()
    lib = binding.load()
    return lambda n, nnz, dims: lib.bigcn_workspace_bytes(n, nnz, (ctypes.c_int32 * len(dims))(*dims), len(dims) - 1, 0)


def buffers(n, dims):
    """The two packed buffers and the contraction's rows, each within 256 bytes, and the counter."""
    stride = max((d + 127) // 128 * 16 for d in dims[:-1])
    return 2 * n * (stride + 4) + n * max((d + 3) // 4 * 16 for d in dims[1:]) + 8 * 256


@pytest.mark.parametrize("dims", [[1000, 16], [500, 64], [1280, 128], [600, 32, 7], [100, 30]])
def test_layers_that_contract_first_ask_for_no_more_than_their_rows(workspace, dims):
    n, nnz = (20_000_000, 60_000_000) if dims == [1280, 128] else (N, NNZ)
    assert workspace(n, nnz, dims) <= buffers(n, dims)


@pytest.mark.parametrize("dims,inputs", [([100, 256], 100), ([256, 256], 256), ([100, 256, 256, 47], 256), ([64, 64], 64)])
def test_layers_that_may_aggregate_first_get_room_for_their_sums(workspace, dims, inputs):
    assert workspace(N, NNZ, dims) >= N * 512 * -(-inputs // 128) + N * 16 + 2 * N * 20


@pytest.mark.parametrize("n,nnz,dims", [(2500, 6500, [257, 47]), (400, 5400, [602, 200]), (60000, 210000, [33, 256])])
def test_small_graphs_have_room_for_either_order(workspace, n, nnz, dims):
    assert workspace(n, nnz, dims) >= n * 512 * -(-dims[0] // 128) + n * 16


@pytest.mark.parametrize("d_out,least", [(33, 5 << 20), (48, 5 << 20), (49, 4 << 20), (64, 4 << 20)])
def test_grouped_rows_get_room_for_their_parts_and_the_plan(workspace, d_out, least):
    """From the first graph that takes them by default on: a record of 16 bytes per group (at least one per 128 entries), two rows of sums
    per unit of work (at most 2,048 entries)."""
    n, dims = 100_000, [700, 100, d_out]
    with_parts, without = workspace(n, least, dims), workspace(n, least - 1, dims)
    assert with_parts - without >= least // 128 * 16 + least // 2048 * 2 * 48 * 4
