"""Bi-GraphSAGE layers of 33..48 outputs on the lane-per-entry stream (the default for these sizes): edge values of either sign, and
factors that are not finite, against the layer's definition in NumPy.  Rows of a few entries, of several passes, and hub rows that a
block splits; plain and half-dot bytes, odd and even inputs."""
import numpy as np
import pytest
import torch
from scipy.sparse import csr_matrix

import oracle
from parity_util import bits_from_dev, bits_to_dev, dev

pytestmark = pytest.mark.gpu

N = 33000


@pytest.mark.parametrize("values", ["both signs", "not finite"])
@pytest.mark.parametrize("d_in,d_out", [(90, 33), (127, 47), (128, 48), (201, 40), (256, 47)])
@pytest.mark.parametrize("long_rows", [False, True])
def test_edge_values(values, d_in, d_out, long_rows):
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(d_in + d_out)
    lens = np.where(np.arange(N) % 5000 == 7, 3000, np.arange(N) % 61)                   # 30 on average, hub rows of 3,000
    rowptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    cols = np.concatenate([np.sort(rng.choice(N, k, replace=False)) for k in lens]).astype(np.int32)
    val = ((0.5 + rng.random(len(cols))) * rng.choice([-1, 1], len(cols))).astype(np.float32)
    F, beta = oracle.binarize_rows(rng.standard_normal((N, d_in)).astype(np.float32))
    if values == "not finite":
        beta[rng.choice(N, 40, replace=False)] = np.inf
        beta[rng.choice(N, 3, replace=False)] = np.nan
    (nbr, a_nbr), (own, a_own) = (oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)) for _ in range(2))
    dots = [F.astype(np.float64) @ s.astype(np.float64) for s in (nbr, own)]
    with np.errstate(invalid="ignore"):
        w = (val * beta[cols]).astype(np.float64)
        want = np.empty((N, d_out))
        for r in range(N):                                                               # entry by entry: a product with a dot of 0 is kept, for inf * 0
            a, b = rowptr[r], rowptr[r + 1]
            want[r] = (w[a:b, None] * dots[0][cols[a:b]]).sum(0)
        want = want * a_nbr + (beta[:, None] * a_own[None, :]).astype(np.float64) * dots[1]
        size = csr_matrix((np.where(np.isfinite(w), np.abs(w), 0), cols, rowptr), shape=(N, N)) @ np.ones(N)
    finite = np.isfinite(want)
    assert values == "both signs" or (np.isinf(want).any() and np.isnan(want).any())

    ctx = B.BiGCN(0)
    if long_rows:
        ctx.set_option(B.OPT_LONG_ROW, 512)                                              # hub rows are split over a block
    G = B.make_graph(dev(rowptr), dev(cols), dev(val))
    layers = [B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(s)), dev(a)) for s, a in ((own, a_own), (nbr, a_nbr))]
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)))
    bits, beta_dev = bits_to_dev(oracle.pack_rows(F)), dev(beta)
    ctx.set_option(B.OPT_ORDER, 1)
    outs = [ctx.sage_layer_forward(G, *layers, bits, beta_dev), ctx.sage_layer_forward(G, *layers, bits, beta_dev, want_h=True, next_layer=nxt)]
    ctx.sync_check()
    ctx.close()
    # fp32 sums of up to 3,000 products, each rounding within 2^-24 of the sums so far
    size = size * a_nbr.max() + np.where(np.isfinite(beta), beta, 0) * a_own.max()
    bound = np.broadcast_to(size[:, None] * d_in * 2e-6 + 1e-6, want.shape)
    for out in outs:
        h = out["h"].cpu().numpy()
        np.testing.assert_array_equal(np.where(finite, 0, h), np.where(finite, 0, want))   # NaN and the signs of infinities
        assert np.all(np.abs(np.where(finite, h - np.where(finite, want, 0), 0)) <= bound)
    sign = oracle.unpack_rows(bits_from_dev(outs[1]["next_bits"]), d_out) > 0
    clear = ~finite | (np.abs(np.where(finite, want, 0)) > bound)
    with np.errstate(invalid="ignore"):
        np.testing.assert_array_equal(sign[clear], (want >= 0)[clear])
