"""Infinite node factors in layers whose width is no multiple of a vector: the padding columns of a row stay out of the next layer's
scale.  Odd widths of the input, so that no dot is 0; against the layer's definition in NumPy."""
import numpy as np
import pytest
import torch

import oracle
from paper_2210_13149_b200 import synth
from parity_util import ATOL, RTOL, bits_from_dev, bits_to_dev, dev

pytestmark = pytest.mark.gpu


# rows of 16-bit integers and of fp32; the last on a graph whose hub rows are split over a block
@pytest.mark.parametrize("n,e,d_in,d_out,fmt", [(300, 900, 201, 5, 0), (300, 900, 201, 60, 0), (300, 900, 33, 251, 4), (300, 900, 33, 30, 2),
                                               (300, 900, 33, 30, 1), (4000, 90000, 201, 60, 0)])
@pytest.mark.parametrize("own_term", [False, True])
def test_infinite_factors(n, e, d_in, d_out, fmt, own_term):
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(n + d_in + d_out)
    src, dst = synth.edge_list(*synth.power_law_graph(n - 1, e, 7))                      # node n - 1 has no neighbour
    g = oracle.mean_adjacency(n, src, dst) if own_term else oracle.normalize_adjacency(n, src, dst)
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    beta[[int(np.diff(g.rowptr)[:-1].argmin()), n - 1]] = np.inf
    nbr, own = (oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32)) for _ in range(2))
    rows = np.repeat(np.arange(n), np.diff(g.rowptr))
    with np.errstate(invalid="ignore"):
        want = np.zeros((n, d_out))
        np.add.at(want, rows, (g.val * beta[g.colidx]).astype(np.float64)[:, None] * (F.astype(np.float64) @ nbr[0])[g.colidx])
        want *= nbr[1]
        if own_term:
            want += (beta[:, None] * own[1][None, :]).astype(np.float64) * (F.astype(np.float64) @ own[0])
        l1 = np.abs(want).mean(1)
    assert np.isinf(l1[n - 1]) and not np.isnan(l1).any()

    ctx = B.BiGCN(0)
    ctx.set_option(B.OPT_ORDER, 1)
    ctx.set_option(B.OPT_ZETA_FORMAT, fmt)
    G = B.make_graph(dev(g.rowptr), dev(g.colidx), dev(g.val))
    layer, self_layer = (B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(s)), dev(a)) for s, a in (nbr, own))
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), dev(np.ones(1, np.float32)))
    bits, beta_dev = bits_to_dev(oracle.pack_rows(F)), dev(beta)
    for want_h in (True, False):
        out = ctx.sage_layer_forward(G, self_layer, layer, bits, beta_dev, want_h=want_h, next_layer=nxt) if own_term else \
              ctx.layer_forward(G, layer, bits, beta_dev, want_h=want_h, next_layer=nxt)
        got = out["next_beta"].cpu().numpy()
        np.testing.assert_array_equal(np.isinf(got), np.isinf(l1))
        assert not np.isnan(got).any()
        np.testing.assert_allclose(got[np.isfinite(l1)], l1[np.isfinite(l1)], rtol=RTOL, atol=ATOL)
        sign = oracle.unpack_rows(bits_from_dev(out["next_bits"]), d_out) > 0
        np.testing.assert_array_equal(sign[np.isinf(want)], (want > 0)[np.isinf(want)])
        if want_h:
            h = out["h"].cpu().numpy()
            np.testing.assert_array_equal(np.where(np.isinf(want), h, 0), np.where(np.isinf(want), want, 0))
    ctx.sync_check()
    ctx.close()
