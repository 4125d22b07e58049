"""The aggregation of short rows in registers (spmm_rows_kernel) against the oracle: hidden layers (bits and beta), last
layers of one vector per row, and the gradients' fp32 rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2210_13149_b200 import synth
from parity_util import ATOL, RTOL, assert_close, bits_from_dev, bits_to_dev, dev, device_graph, flip_report

pytestmark = pytest.mark.gpu

# one row; no entries at all; fewer rows than a set; short rows, rows just above the 64 entries of a lane group, hub rows
GRAPHS = [(1, 0, 1), (40, 0, 2), (33, 120, 3), (700, 2000, 4), (900, 60000, 5), (15000, 60000, 6), (13000, 900000, 7)]


@pytest.fixture()
def ctx():
    from paper_2210_13149_b200 import binding
    c = binding.BiGCN(0)
    c.set_option(binding.OPT_ORDER, 1)
    yield c
    c.sync_check()
    c.close()


# fp16 rows of 1, 2, 4, 8 and 16 vectors, full and ragged; bytes (d_in <= 127, more than 128 columns); int16 (d_in > 2048)
@pytest.mark.parametrize("d_in,d_out", [(300, 1), (300, 8), (300, 9), (300, 31), (300, 32), (300, 57), (300, 64), (300, 128), (90, 130), (90, 256), (2100, 40)])
@pytest.mark.parametrize("n,e,seed", GRAPHS)
def test_hidden_and_narrow_layers(ctx, n, e, seed, d_in, d_out):
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(seed + d_out)
    g = oracle.normalize_adjacency(n, *synth.edge_list(*synth.power_law_graph(n, e, seed)))
    H = rng.standard_normal((n, d_in)).astype(np.float32)
    W = (rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)
    t = oracle.layer_forward(g, oracle.Layer(W), H)
    shift, scale = oracle.col_stats(t.H_out)
    G, layer = device_graph(B, g), B.make_layer(d_in, d_out, bits_to_dev(t.bitsT), dev(t.alpha))
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)), dev(shift), dev(scale))
    out = ctx.layer_forward(G, layer, bits_to_dev(t.bits), dev(t.beta), want_h=False, next_layer=nxt)
    F, beta = oracle.binarize_rows(t.H_out, shift, scale)
    flips, bad, _ = flip_report(bits_from_dev(out["next_bits"]), F, t.H_out, shift)
    assert bad == 0, "%d of %d flips away from the threshold" % (bad, flips)
    np.testing.assert_allclose(out["next_beta"].cpu().numpy(), beta, rtol=10 * RTOL, atol=ATOL * float(scale.max()))
    assert_close(ctx.layer_forward(G, layer, bits_to_dev(t.bits), dev(t.beta))["h"], t.H_out, "H'")
    assert_close(ctx.forward_packed(G, [layer], bits_to_dev(t.bits), dev(t.beta)), t.H_out, "logits")


@pytest.mark.parametrize("d_out", [1, 4, 13, 32, 64])
@pytest.mark.parametrize("n,e,seed", GRAPHS)
def test_gradient_rows(ctx, n, e, seed, d_out):
    """fp32 rows of 1 to 16 vectors; the bound is that of the gradient tests: fp32 sums against double."""
    from paper_2210_13149_b200 import binding as B
    d_in = 24
    rng = np.random.default_rng(seed * 10 + d_out)
    g = oracle.normalize_adjacency(n, *synth.edge_list(*synth.power_law_graph(n, e, seed)))
    W = (rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    g_out = (rng.standard_normal((n, d_out)) * 0.02).astype(np.float32)
    want = oracle.layer_backward(g, W, F, beta, g_out)
    bitsT, alpha = ctx.pack_weights(dev(W))
    _, g_w = ctx.layer_backward(device_graph(B, g), B.make_layer(d_in, d_out, bitsT, alpha), dev(W), bits_to_dev(oracle.pack_rows(F)), dev(beta), dev(g_out))
    ref = want.G_W
    got = g_w.cpu().numpy()
    assert np.all(np.abs(got - ref) <= 1e-4 * np.abs(ref) + 2e-6 * np.abs(ref).max())
