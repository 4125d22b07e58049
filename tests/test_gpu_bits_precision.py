"""Rounding of the packed-bit order against 64 bits, on rows in which one weight outweighs all others together."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import bits_to_dev, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entries", [2, 40, 65, 128])
@pytest.mark.parametrize("share", [1e-3, 1e-6])
def test_rows_with_one_large_weight(entries, share):
    """A weight is rounded to 2^-30 of the row's sum of |w| at most, P is exact, and H' is rounded to fp32 three times (its high
    half, the sum of its halves, the product with the scale).  Independent errors: rms no larger than
    sum |w| alpha sqrt(d_in) (2^-30 sqrt(entries) + 2^-24 sqrt(3)).  And no larger than the other order's."""
    from paper_2210_13149_b200 import binding as B
    n, d_in, d_out = 512, 200, 256
    rng = np.random.default_rng(entries)
    cols = np.stack([np.sort(rng.choice(n, entries, replace=False)) for _ in range(n)]).astype(np.int32)
    val = (share * (0.5 + rng.random((n, entries)))).astype(np.float32)
    val[np.arange(n), rng.integers(0, entries, n)] = 1.0
    G = B.make_graph(dev(np.arange(n + 1, dtype=np.int64) * entries), dev(cols.reshape(-1)), dev(val.reshape(-1)))
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    signs, alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    layer = B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(signs)), dev(alpha))
    w = (val * beta[cols]).astype(np.float64)                                  # the fp32 product both orders start from
    dots = F.astype(np.float64) @ signs.astype(np.float64)
    exact = np.einsum("ne,nej->nj", w, dots[cols]) * alpha.astype(np.float64)
    unit = np.abs(w).sum(1)[:, None] * alpha[None, :] * d_in ** 0.5
    rms = {}
    for order in (1, 2):
        ctx = B.BiGCN(0)
        ctx.set_option(B.OPT_ORDER, order)
        h = ctx.layer_forward(G, layer, bits_to_dev(oracle.pack_rows(F)), dev(beta))["h"]
        ctx.sync_check()
        rms[order] = np.sqrt((((h.cpu().numpy() - exact) / unit) ** 2).mean())
        ctx.close()
    assert rms[2] <= 2.0 ** -30 * entries ** 0.5 + 2.0 ** -24 * 3 ** 0.5
    assert rms[2] <= rms[1] * 1.05
