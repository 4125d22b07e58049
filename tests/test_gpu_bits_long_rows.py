"""Rows of many pieces in the packed-bit order: pieces that share a scale and one read-back, against 64 bits."""
import numpy as np
import pytest

import oracle
from parity_util import bits_to_dev, dev

pytestmark = pytest.mark.gpu


# on either side of 384 entries and of a unit of work (2,048 entries and rows); rows over several units
@pytest.mark.parametrize("entries", [384, 385, 1300, 2044, 2600, 5000])
@pytest.mark.parametrize("weights", ["even", "largest first", "growing"])
@pytest.mark.parametrize("d_in,d_out", [(200, 130), (60, 40)])
def test_long_rows_against_64_bits(entries, weights, d_in, d_out):
    """No less precise than the order that contracts first, whose fp32 sums round every addition."""
    from paper_2210_13149_b200 import binding as B
    n, rows = 6000, 96
    rng = np.random.default_rng(entries + d_in)
    lens = np.where(np.arange(n) < rows, entries, 1)
    rowptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    val = (0.5 + rng.random(len(cols))).astype(np.float32)
    for r in range(rows):
        a, b = rowptr[r], rowptr[r + 1]
        if weights == "largest first":
            val[a] = 1e4
        elif weights == "growing":
            val[a:b] *= np.float32(2.0) ** np.linspace(-12, 0, b - a).astype(np.float32)
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    signs, alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    G, layer = B.make_graph(dev(rowptr), dev(cols), dev(val)), B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(signs)), dev(alpha))
    w = (val * beta[cols]).astype(np.float64)                                  # the fp32 product both orders start from
    dots = F.astype(np.float64) @ signs.astype(np.float64)
    exact = np.stack([w[rowptr[r]:rowptr[r + 1]] @ dots[cols[rowptr[r]:rowptr[r + 1]]] for r in range(rows)]) * alpha.astype(np.float64)
    rms = {}
    for order in (1, 2):
        ctx = B.BiGCN(0)
        ctx.set_option(B.OPT_ORDER, order)
        h = ctx.layer_forward(G, layer, bits_to_dev(oracle.pack_rows(F)), dev(beta))["h"]
        ctx.sync_check()
        rms[order] = np.sqrt(((h.cpu().numpy()[:rows] - exact) ** 2).mean())
        ctx.close()
    assert rms[2] <= rms[1] * 1.05
