"""The layer with the aggregation of the packed bits before the contraction (BIGCN_OPT_ORDER = 2) against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2210_13149_b200 import synth
from parity_util import RTOL, ATOL, assert_close, bits_from_dev, bits_to_dev, dev, device_graph, flip_report

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    from paper_2210_13149_b200 import binding
    c = binding.BiGCN(0)
    c.set_option(binding.OPT_ORDER, 2)
    yield c
    c.sync_check()
    c.close()


def graph(n, e, seed):
    return oracle.normalize_adjacency(n, *synth.edge_list(*synth.power_law_graph(n, e, seed)))


# one row; rows on either side of a tile of 32; no edges; hub rows of several pieces, units and read-backs; every slice
# width (64, 128, 256 columns and their combinations), a last slice of one column, the widest layers
SHAPES = [(1, 0, 1, 1), (31, 60, 64, 64), (33, 200, 65, 3), (200, 0, 128, 128), (500, 6000, 129, 129), (700, 9000, 256, 256),
          (2500, 4000, 257, 47), (3000, 900000, 100, 256), (4000, 1500000, 256, 41), (400, 5000, 602, 200),
          (2000, 700000, 512, 256), (300, 3000, 1280, 128), (60000, 150000, 33, 256)]


@pytest.mark.parametrize("n,e,d_in,d_out", SHAPES)
def test_bits_first_against_oracle(ctx, n, e, d_in, d_out):
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(n + d_in * 7 + d_out)
    g = graph(n, e, 11 + n)
    H = rng.standard_normal((n, d_in)).astype(np.float32)
    W = (rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)
    t = oracle.layer_forward(g, oracle.Layer(W), H)
    shift, scale = oracle.col_stats(t.H_out)
    G, layer = device_graph(B, g), B.make_layer(d_in, d_out, bits_to_dev(t.bitsT), dev(t.alpha))
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)), dev(shift), dev(scale))
    before = ctx.launch_count()
    out = ctx.layer_forward(G, layer, bits_to_dev(t.bits), dev(t.beta), want_h=True, next_layer=nxt)
    assert ctx.launch_count() - before == 3 + (d_in > 256 and 0 < d_in % 256 <= 128), "not the kernels under test"
    only = ctx.layer_forward(G, layer, bits_to_dev(t.bits), dev(t.beta), want_h=False, next_layer=nxt)
    assert_close(out["h"], t.H_out, "H'")
    F, beta = oracle.binarize_rows(t.H_out, shift, scale)
    for o in (out, only):
        flips, bad, _ = flip_report(bits_from_dev(o["next_bits"]), F, t.H_out, shift)
        assert bad == 0, "%d of %d flips away from the threshold" % (bad, flips)
        np.testing.assert_allclose(o["next_beta"].cpu().numpy(), beta, rtol=10 * RTOL, atol=ATOL * float(scale.max()))


@pytest.mark.parametrize("span", [0, 12, 40])
@pytest.mark.parametrize("n,e", [(600, 24000), (600, 150000)])
def test_bits_first_signed_edge_values_of_wide_range(ctx, n, e, span):
    """Edge values of both signs over 2^-span .. 2^span.  A weight is rounded to 2^-22 of the largest of its row in rows of
    up to 128 entries (2^-26 of its piece's in longer ones) and P to 2^-29 of the row's sum of |w|; the contraction adds up
    d_in such values, hence the bound."""
    from paper_2210_13149_b200 import binding as B
    d_in, d_out = 200, 256
    rng = np.random.default_rng(5 + span)
    g = graph(n, e, 31)
    g.val[:] = (g.val * np.exp2(rng.integers(-span, span + 1, g.val.shape)) * rng.choice([-1.0, 1.0], g.val.shape)).astype(np.float32)
    H = rng.standard_normal((n, d_in)).astype(np.float32)
    W = (rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)
    t = oracle.layer_forward(g, oracle.Layer(W), H)
    out = ctx.layer_forward(device_graph(B, g), B.make_layer(d_in, d_out, bits_to_dev(t.bitsT), dev(t.alpha)), bits_to_dev(t.bits), dev(t.beta))
    deg = np.diff(g.rowptr)
    w = np.abs(g.val) * t.beta[g.colidx]
    wsum = np.add.reduceat(w, g.rowptr[:-1].astype(np.int64))
    wmax = np.maximum.reduceat(w, g.rowptr[:-1].astype(np.int64))
    unit = np.where(deg <= 128, 2.0 ** -22 * wmax, 2.0 ** -26 * wmax) * deg + 2.0 ** -21 * wsum
    assert np.all(np.abs(out["h"].cpu().numpy() - t.H_out) <= unit[:, None] * d_in * np.abs(t.alpha)[None, :] + 1e-30)


# the node's own term: one and several tiles, mostly empty rows, one and two blocks of 128 output columns, more tiles than
# a block's buffers hold
@pytest.mark.parametrize("n,e,d_in,d_out", [(1, 0, 5, 1), (33, 60, 64, 7), (300, 200, 64, 200), (500, 6000, 300, 129),
                                             (4200, 50000, 127, 256), (30000, 60000, 40, 128)])
def test_bits_first_sage_layer(ctx, n, e, d_in, d_out):
    from paper_2210_13149_b200 import binding as B
    from test_gpu_sage import check_sage_layer
    check_sage_layer(ctx, 0, n, e, d_in, d_out)
    rng = np.random.default_rng(n)
    G = ctx.mean_adjacency(*(t.cuda() for t in synth.power_law_graph(n, e, 3)))
    own, nbr = ctx.prepare_layers([dev((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)) for _ in range(2)])
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)))
    bits, beta = ctx.pack_features(dev(rng.standard_normal((n, d_in)).astype(np.float32)))
    both, only = (ctx.sage_layer_forward(G, own, nbr, bits, beta, want_h=h, next_layer=nxt) for h in (True, False))
    assert torch.equal(both["next_bits"], only["next_bits"]) and torch.equal(both["next_beta"], only["next_beta"])
