"""Weights without a common fixed point in the packed-bit order: NaN, infinities, and magnitudes far from 1, in rows of every length,
against the layer's definition in NumPy."""
import numpy as np
import pytest
import torch

import oracle
from paper_2210_13149_b200 import synth
from parity_util import bits_from_dev, bits_to_dev, dev

pytestmark = pytest.mark.gpu

# which nodes' factors: some of everything, or all of one magnitude (the smallest: below 2^-126 their weights are denormal)
FACTORS = {"mixed": (np.nan, np.inf, -np.inf, 1e33, 1e-33, 0.0), "tiny": (1e-30,), "small": (3e-26,), "huge": (1e34,), "large": (1e29,), "zero": (0.0,)}


# rows of a few entries; hub rows of several pieces and units; one and two blocks of 128 output columns
@pytest.mark.parametrize("kind", list(FACTORS))
@pytest.mark.parametrize("n,e,d_in,d_out", [(700, 2500, 60, 100), (900, 60000, 130, 256), (1500, 100000, 300, 40)])
@pytest.mark.parametrize("own_term", [False, True])
def test_weights_without_a_fixed_point(kind, n, e, d_in, d_out, own_term):
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(n + d_in)
    src, dst = synth.edge_list(*synth.power_law_graph(n, e, 3))
    g = oracle.mean_adjacency(n, src, dst) if own_term else oracle.normalize_adjacency(n, src, dst)
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    values = FACTORS[kind]
    for i, v in enumerate(values):                                             # "mixed" leaves most nodes and rows as they are
        rows = rng.choice(n, 2, replace=False) if kind == "mixed" else np.arange(n)
        beta[rows] = np.float32(v) * (rng.random(len(rows)).astype(np.float32) + np.float32(0.5))
    signs, alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    own_signs, own_alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    # the definition, entry by entry: a product with a dot of 0 is kept, for inf * 0
    dots = (F.astype(np.int32) @ signs.astype(np.int32)).astype(np.float64)
    rows = np.repeat(np.arange(n), np.diff(g.rowptr))
    with np.errstate(all="ignore"):
        w = (g.val * beta[g.colidx]).astype(np.float64)
        want, size = np.zeros((n, d_out)), np.zeros((n, 1))
        np.add.at(want, rows, w[:, None] * dots[g.colidx])
        np.add.at(size, rows[np.isfinite(w)], np.abs(w[np.isfinite(w)])[:, None])
        want, size = want * alpha, size * alpha * d_in
        if own_term:
            t = (beta[:, None] * own_alpha[None, :]).astype(np.float64) * (F.astype(np.int32) @ own_signs.astype(np.int32))
            want, size = want + t, size + np.where(np.isfinite(t), np.abs(t), 0)
    assert kind != "mixed" or (np.isnan(want).any() and np.isinf(want).any() and np.isfinite(want).any())

    ctx = B.BiGCN(0)
    ctx.set_option(B.OPT_ORDER, 2)
    G = B.make_graph(dev(g.rowptr), dev(g.colidx), dev(g.val))
    nbr = B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(signs)), dev(alpha))
    own = B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(own_signs)), dev(own_alpha))
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)))
    bits, beta_dev = bits_to_dev(oracle.pack_rows(F)), dev(beta)
    run = (lambda h: ctx.sage_layer_forward(G, own, nbr, bits, beta_dev, want_h=h, next_layer=nxt)) if own_term else \
          (lambda h: ctx.layer_forward(G, nbr, bits, beta_dev, want_h=h, next_layer=nxt))
    both, only = run(True), run(False)
    ctx.sync_check()
    ctx.close()
    h = both["h"].cpu().numpy()
    finite = np.isfinite(want)
    np.testing.assert_array_equal(np.where(finite, 0, h), np.where(finite, 0, want))      # NaN and the signs of infinities
    # Finite sums: fp32 sums of up to a thousand terms, or fixed point to 2^-30 of sum |w| in each of d_in columns; denormal
    # products are off by 2^-150 each.
    terms = np.diff(g.rowptr).max() + 1
    bound = np.broadcast_to(size, want.shape) * 2e-6 + terms * d_in * 2.0 ** -149
    assert np.all(np.abs(np.where(finite, h - np.where(finite, want, 0), 0)) <= bound)
    for out in (both, only):
        got = oracle.unpack_rows(bits_from_dev(out["next_bits"]), d_out) > 0
        clear = ~finite | (np.abs(np.where(finite, want, 0)) > bound)
        with np.errstate(invalid="ignore"):
            assert np.array_equal(got[clear], (want >= 0)[clear])
            l1 = np.abs(want).mean(1)
        got_beta = out["next_beta"].cpu().numpy()
        ok = np.isfinite(l1)
        np.testing.assert_array_equal(np.where(ok, 0, got_beta), np.where(ok, 0, l1))
        assert np.all(np.abs(got_beta[ok] - l1[ok]) <= bound[ok].max(1) + 1e-5 * l1[ok])
