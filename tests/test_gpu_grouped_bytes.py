"""Byte rows of 33..64 columns as grouped integer products (spmm_bytes.cu) against the oracle: BIGCN_OPT_BYTE_AGGREGATION = 2 takes them
there whatever the graph.  Graphs: one row; isolated nodes; pairs of rows and rows on either side of a group of 128 entries; hub rows of
several pieces, scales and units of work.  Columns: three and four products, the last of one column; rows of 48 bytes, of 64, and with
the node factor in their tail; plain and half-dot bytes."""
import numpy as np
import pytest
import torch
from scipy.sparse import csr_matrix

import oracle
from paper_2210_13149_b200 import synth
from parity_util import ATOL, RTOL, assert_close, bits_from_dev, bits_to_dev, dev, device_graph, flip_report
from test_gpu_sage import check_sage_layer

pytestmark = pytest.mark.gpu

GRAPHS = [(1, 0, 1), (70, 0, 2), (129, 4000, 3), (900, 60000, 4), (3000, 900000, 5), (24000, 400000, 6)]


@pytest.fixture()
def ctx():
    from paper_2210_13149_b200 import binding
    c = binding.BiGCN(0)
    c.set_option(binding.OPT_ORDER, 1)
    c.set_option(binding.OPT_BYTE_AGGREGATION, 2)
    c.ensure_workspace(1 << 28)
    yield c
    c.sync_check()
    c.close()


@pytest.mark.parametrize("fmt", [3, 5])
@pytest.mark.parametrize("d_out", [33, 47, 48, 49, 60, 61, 64])
@pytest.mark.parametrize("n,e,seed", GRAPHS)
def test_layers(ctx, n, e, seed, d_out, fmt):
    from paper_2210_13149_b200 import binding as B
    d_in = 127 if fmt == 3 else (128 if d_out % 2 else 255)
    ctx.set_option(B.OPT_ZETA_FORMAT, fmt)
    rng = np.random.default_rng(seed + d_out)
    g = oracle.normalize_adjacency(n, *synth.edge_list(*synth.power_law_graph(n, e, seed)))
    H = rng.standard_normal((n, d_in)).astype(np.float32)
    t = oracle.layer_forward(g, oracle.Layer((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)), H)
    shift, scale = oracle.col_stats(t.H_out)
    G, layer = device_graph(B, g), B.make_layer(d_in, d_out, bits_to_dev(t.bitsT), dev(t.alpha))
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)), dev(shift), dev(scale))
    out = ctx.layer_forward(G, layer, bits_to_dev(t.bits), dev(t.beta), want_h=True, next_layer=nxt)
    assert_close(out["h"], t.H_out, "H'")
    F, beta = oracle.binarize_rows(t.H_out, shift, scale)
    flips, bad, _ = flip_report(bits_from_dev(out["next_bits"]), F, t.H_out, shift)
    assert bad == 0, "%d of %d flips away from the threshold" % (bad, flips)
    np.testing.assert_allclose(out["next_beta"].cpu().numpy(), beta, rtol=10 * RTOL, atol=ATOL * float(scale.max()))
    assert_close(ctx.forward_packed(G, [layer], bits_to_dev(t.bits), dev(t.beta)), t.H_out, "logits")


def weighted(rng, lens, n, make):
    rowptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    return rowptr, cols, np.concatenate([make(k) for k in lens]).astype(np.float32)


@pytest.mark.parametrize("entries", [1, 31, 64, 65, 128, 129, 480, 481, 2000, 4500])
@pytest.mark.parametrize("weights", ["both signs, wide", "largest first", "largest last", "not finite", "tiny"])
def test_any_weights(ctx, entries, weights):
    """No less precise than the literal fp32 order (BIGCN_OPT_ZETA_FORMAT = 1); weights without a fixed point are summed as written."""
    from paper_2210_13149_b200 import binding as B
    n, d_in, d_out = 5000, 200, 47
    rng = np.random.default_rng(entries)
    lens = np.where(np.arange(n) % 50 == 7, entries, np.arange(n) % 3)

    def make(k):
        w = 0.5 + rng.random(k)
        if weights == "both signs, wide":
            w *= np.exp2(rng.uniform(-12, 0, k)) * rng.choice([-1.0, 1.0], k)
        elif weights in ("largest first", "largest last") and k:
            w[0 if weights == "largest first" else -1] = 1e4
        elif weights == "not finite" and k:
            w[rng.integers(k)] = rng.choice([np.inf, np.nan, 1e38])
        elif weights == "tiny":
            w *= 2.0 ** -110
        return w

    rowptr, cols, val = weighted(rng, lens, n, make)
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    signs, alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    G, layer = B.make_graph(dev(rowptr), dev(cols), dev(val)), B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(signs)), dev(alpha))
    row = np.repeat(np.arange(n), lens)
    dots = F.astype(np.float64) @ signs.astype(np.float64)
    with np.errstate(over="ignore", invalid="ignore"):
        w = (val * beta[cols]).astype(np.float64)                              # the fp32 product every order starts from
        exact = csr_matrix((w, cols, rowptr), shape=(n, n)) @ dots * alpha.astype(np.float64)
        unit = np.bincount(row, np.abs(w), n)[:, None] * alpha.astype(np.float64)[None, :] * d_in ** 0.5
    got = {}
    for fmt in (5, 1):
        ctx.set_option(B.OPT_ZETA_FORMAT, fmt)
        got[fmt] = ctx.forward_packed(G, [layer], bits_to_dev(oracle.pack_rows(F)), dev(beta)).cpu().numpy().astype(np.float64)
    finite = np.isfinite(exact).all(1) & (np.abs(exact) < 1e37).all(1)
    assert not np.isfinite(got[5][~np.isfinite(exact).all(1)]).all(1).any()
    rms = {f: np.sqrt(np.mean(((h[finite] - exact[finite]) / np.maximum(unit[finite], 1e-300)) ** 2)) for f, h in got.items()}
    assert rms[5] <= rms[1] * 1.05 + 2.0 ** -30


@pytest.mark.parametrize("entries", [100, 128, 129, 480, 481, 2000])
@pytest.mark.parametrize("where", ["first", "last"])
@pytest.mark.parametrize("d_in,d_out,fmt", [(126, 47, 3), (200, 47, 5), (200, 64, 5)])
def test_columns_in_which_the_largest_weight_meets_a_dot_of_zero(ctx, entries, where, d_in, d_out, fmt):
    """Single sums against what the digits of weights a thousand times smaller leave of them."""
    from paper_2210_13149_b200 import binding as B
    n, rows = 4000, 40
    rng = np.random.default_rng(entries + d_in)
    lens = np.where(np.arange(n) < rows, entries, 1)
    make = lambda k: np.where(np.arange(k) == (0 if where == "first" else k - 1), 1.0, (0.5 + rng.random(k)) * 2.0 ** -10)
    rowptr, cols, val = weighted(rng, lens, n, make)
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    signs, alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    ctx.set_option(B.OPT_ZETA_FORMAT, fmt)
    G, layer = B.make_graph(dev(rowptr), dev(cols), dev(val)), B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(signs)), dev(alpha))
    h = ctx.layer_forward(G, layer, bits_to_dev(oracle.pack_rows(F)), dev(beta))["h"].cpu().numpy().astype(np.float64)
    dots = F.astype(np.float64) @ signs.astype(np.float64)
    w = (val * beta[cols]).astype(np.float64)                                  # the fp32 product every order starts from
    seen = 0
    for r in range(rows):
        a, b = rowptr[r], rowptr[r + 1]
        top = cols[a if where == "first" else b - 1]
        zero = dots[top] == 0
        terms = w[a:b, None] * dots[cols[a:b]][:, zero]
        # A weight is off by 2^-30 of its row's largest, 2^-27 of its scale's where a row has several pieces; sums of pieces are fp32 (three
        # roundings each), and so are the three sums of half-dot bytes, each as large as sum |w|, in which the largest weight cancels.
        off = 2.0 ** (-30 if entries <= 128 else -27) * w[a:b].max() * np.abs(dots[cols[a:b]][:, zero]).sum(0)
        fp32 = sum(np.abs(terms[i:i + 128]).sum(0) for i in range(0, b - a, 128)) + (0 if fmt == 3 else 4 * w[a:b].sum())
        assert np.all(np.abs(h[r, zero] - terms.sum(0) * alpha[zero]) <= alpha[zero] * (off + 2.0 ** -22 * fp32))
        seen += zero.sum()
    assert seen > 20


@pytest.mark.parametrize("d_in,d_out", [(127, 33), (255, 47), (128, 60), (200, 64)])
def test_sage_layers(ctx, d_in, d_out):
    """The neighbours' term with the node's own added at a row's end."""
    check_sage_layer(ctx, 0, 33000, 400000, d_in, d_out)
