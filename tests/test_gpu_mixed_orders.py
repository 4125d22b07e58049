"""Forwards whose layers run in both orders: the plan of the graph, made once and shared by the layers that aggregate the packed
bits first, has to outlive the layers that contract first."""
import numpy as np
import pytest
import torch

import oracle
from paper_2210_13149_b200 import synth
from parity_util import assert_close, bits_from_dev, bits_to_dev, dev, device_graph

pytestmark = pytest.mark.gpu


def up(x):
    return (x + 255) // 256 * 256


# The first layer (more than 1,280 inputs) and the last (more than 256 outputs) contract first, the middle one aggregates the
# bits first.  Their order-one scratch, of the widest output, is larger than the middle layer's; with 200 and 160 columns
# the first layer's aggregation takes its rows from a counter that it keeps there, with 64 it does not.
@pytest.mark.parametrize("dims", [(1433, 200, 64, 349), (1433, 160, 200, 512), (1433, 64, 64, 349), (1290, 200, 256, 340)])
@pytest.mark.parametrize("n,e", [(3000, 20000), (2500, 60000)])
@pytest.mark.parametrize("small_workspace", [False, True])
def test_forward_with_layers_of_both_orders(dims, n, e, small_workspace):
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(n + dims[1])
    g = oracle.normalize_adjacency(n, *synth.edge_list(*synth.power_law_graph(n, e, n)))
    G = device_graph(B, g)
    W = [(rng.standard_normal((a, b)) * a ** -0.5).astype(np.float32) for a, b in zip(dims[:-1], dims[1:])]
    ctx = B.BiGCN(0)
    ctx.set_option(B.OPT_ORDER, 2)
    layers = ctx.prepare_layers([dev(w) for w in W])
    bits, beta = ctx.pack_features(dev(rng.standard_normal((n, dims[0])).astype(np.float32)))
    # one call per layer: each makes its own plan
    x = (bits, beta)
    for l in range(2):
        before = ctx.launch_count()
        out = ctx.layer_forward(G, layers[l], *x, want_h=False, next_layer=layers[l + 1])
        assert ctx.launch_count() - before == (2 if l == 0 else 3), "not the orders under test"
        x = (out["next_bits"], out["next_beta"])
    want = ctx.layer_forward(G, layers[2], *x)["h"]
    assert_close(want, oracle.layer_forward_packed(g, oracle.Layer(W[2]), bits_from_dev(x[0]), x[1].cpu().numpy()).H_out)
    if small_workspace:                                     # room for the contraction's rows but not for P and a plan behind them
        stride = max(B.packed_stride_words(d) for d in dims[:-1])
        size = up(n * max((d + 3) // 4 * 4 for d in dims[1:]) * 4) + 256 + 2 * (up(n * stride * 4) + up(n * 4))
        assert size < ctx.workspace_bytes(n, g.nnz, dims)
        ctx.workspace = torch.empty(size, dtype=torch.uint8, device="cuda")
        ctx._check(ctx.lib.bigcn_set_workspace(ctx.h, B._ptr(ctx.workspace), size))
        ctx.ensure_workspace = lambda nbytes: None
    ctx.workspace.fill_(0x55)
    before = ctx.launch_count()
    got = ctx.forward_packed(G, layers, bits, beta)
    ctx.sync_check()
    assert ctx.launch_count() - before == 7                 # 2 + (plan, two products) + 2
    assert torch.equal(got, want)
    ctx.close()
