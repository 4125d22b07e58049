"""Rounding of the weight gradients against 64 bits."""
import pytest
import torch

from paper_2210_13149_b200 import synth

pytestmark = pytest.mark.gpu


# The longest fp32 accumulation of a part decides: ceil(n / parts) nodes in steps of 16 nodes and three terms, each cut to 2^-23 of
# the sum so far at worst, half of it on average over a sum that grows evenly, and half of that in the mean: steps / 4 *
# 2^-23 of a part, and no more of the whole.  Parts (slabs, or accumulators of one): four for every multiprocessor and 128 x
# 128 weights.
@pytest.mark.parametrize("n,mean,d_in,d_out", [(100000, 20, 64, 64), (100000, 20, 100, 90), (600000, 10, 64, 128), (100000, 20, 300, 200),
                                               (250000, 6, 128, 40)])
def test_weight_gradient_keeps_short_accumulations(n, mean, d_in, d_out):
    from paper_2210_13149_b200 import binding as B
    ctx = B.BiGCN(0)
    G = ctx.normalize_adjacency(*synth.power_law_graph(n, n * mean, 3, device="cuda"))
    W = synth.weights([d_in, d_out], 5, "cuda")[0]
    layer = ctx.prepare_layers([W])[0]
    gen = torch.Generator(device="cuda").manual_seed(7)
    X = torch.randn((n, d_in), device="cuda", generator=gen)
    bits, beta = ctx.pack_features(X)
    g = torch.randn((n, d_out), device="cuda", generator=gen) * 0.02 + 0.01
    _, got = ctx.layer_backward(G, layer, W, bits, beta, g, want_g_in=False)
    ctx.sync_check()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), G.rowptr[1:] - G.rowptr[:-1])
    gz = torch.zeros((n, d_out), dtype=torch.float64, device="cuda")
    for a in range(0, d_out, 16):
        gz[:, a:a + 16].index_add_(0, rows, G.val.double()[:, None] * g[:, a:a + 16].double()[G.colidx.long()])
    gwt = torch.zeros((d_in, d_out), dtype=torch.float64, device="cuda")
    for a in range(0, n, 50000):
        gwt += (torch.where(X[a:a + 50000] >= 0, 1.0, -1.0).double() * beta[a:a + 50000].double()[:, None]).t() @ gz[a:a + 50000]
    signs = torch.where(W >= 0, 1.0, -1.0).double()
    want = signs * ((gwt * signs).sum(0) / d_in)[None, :] + layer.alpha.double()[None, :] * gwt * (W.abs() < 1)
    parts = 4 * torch.cuda.get_device_properties(0).multi_processor_count // (-(-d_in // 128) * -(-d_out // 128))
    steps = -(-n // parts) / 16 * 3
    error = float((got.double() - want).norm() / want.norm())
    assert error <= steps / 4 * 2.0 ** -23, (error, steps)
    ctx.close()
