"""Forwards whose last layer takes its byte rows as grouped products by default, in the workspace that bigcn_workspace_bytes() asks for and
in one a kilobyte smaller: the parts' room is missed by the last layer alone."""
import pytest
import torch

from paper_2210_13149_b200 import synth

pytestmark = pytest.mark.gpu


def forward(n, nnz_per_node, dims, short, order=0):
    """(kernels launched, the logits)"""
    from paper_2210_13149_b200 import binding as B
    ctx = B.BiGCN(0)
    ctx.set_option(B.OPT_ORDER, order)
    gen = torch.Generator(device="cuda").manual_seed(3)
    rowptr = torch.arange(n + 1, device="cuda") * nnz_per_node
    cols = torch.randint(0, n, (n, nnz_per_node), device="cuda", generator=gen, dtype=torch.int32).sort(1).values.reshape(-1)
    G = B.make_graph(rowptr, cols, torch.full((cols.numel(),), 1.0 / nnz_per_node, device="cuda"))
    layers = ctx.prepare_layers(synth.weights(dims, 5, "cuda"))
    bits, beta = ctx.pack_features(torch.randn((n, dims[0]), device="cuda", generator=gen))
    size = ctx.workspace_bytes(n, G.nnz, dims) - short
    ctx.workspace = None
    ctx.workspace_bytes = lambda *a: size
    before = ctx.launch_count()
    logits = ctx.forward_packed(G, layers, bits, beta)
    ctx.sync_check()
    assert ctx.workspace.numel() == size
    launches = ctx.launch_count() - before
    ctx.close()
    return launches, logits


def test_one_layer():
    full, logits = forward(110_000, 50, [100, 47], 0)
    short, streamed = forward(110_000, 50, [100, 47], 1024)
    assert (full, short) == (3, 2)                                       # contraction, the graph's plan, aggregation
    assert (logits - streamed).abs().max() <= 1e-5 * logits.abs().max()


def test_only_the_grouped_rows_ask_for_the_plan():
    """The first layer contracts first, the last is too large to get room for its packed bits' sums unasked."""
    full, logits = forward(150_000, 41, [700, 100, 47], 0)
    short, streamed = forward(150_000, 41, [700, 100, 47], 1024)
    assert (full, short) == (5, 4)
    assert (logits - streamed).abs().max() <= 1e-5 * logits.abs().max()


def test_a_layer_that_aggregates_the_packed_bits_before_one_with_grouped_rows():
    dims = [100, 184, 47]
    full, logits = forward(110_000, 50, dims, 0)
    short, streamed = forward(110_000, 50, dims, 1024)
    # the plan, aggregation and products of the bits; contraction and aggregation, with the same plan where grouped
    assert (full, short) == (5, 5)
    assert forward(110_000, 50, dims, 1024, order=1)[0] == 4
    assert (logits - streamed).abs().max() <= 1e-5 * logits.abs().max()


def test_several_layers_share_the_plan():
    """Every layer's rows as grouped products, by option: the graph's plan is made once; against the streams, up to sign flips of hidden sums
    at their threshold."""
    from paper_2210_13149_b200 import binding as B
    n, dims = 3000, [100, 47, 64, 33]
    rowptr, cols = synth.power_law_graph(n, 90_000, 3, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(4)
    X = torch.randn((n, dims[0]), device="cuda", generator=gen)
    got = {}
    for option in (2, 0):
        ctx = B.BiGCN(0)
        ctx.set_option(B.OPT_ORDER, 1)
        ctx.set_option(B.OPT_BYTE_AGGREGATION, option)
        G = ctx.normalize_adjacency(rowptr, cols)
        layers = ctx.prepare_layers(synth.weights(dims, 5, "cuda"))
        bits, beta = ctx.pack_features(X)
        before = ctx.launch_count()
        got[option] = ctx.forward_packed(G, layers, bits, beta)
        ctx.sync_check()
        assert ctx.launch_count() - before == (7 if option else 6)
        ctx.close()
    same = ((got[2] - got[0]).abs() <= 1e-4 + 1e-5 * got[0].abs()).all(1)
    assert same.float().mean() > 0.95
