"""Bi-GraphSAGE layers of 33..64 outputs against the oracle under the tolerance of the other layers.  Where sage_lane_pays() says so, the
neighbours of a layer of 33..48 outputs are byte rows for the lane-per-entry stream, with the node's own term added at a row's end: plain
bytes up to 127 inputs, half-dot bytes with the node factor in the rows' tail from 2^20 outputs on; elsewhere, and for 49..64 outputs,
16-bit rows."""
import numpy as np
import pytest

import oracle
from paper_2210_13149_b200 import synth
from parity_util import assert_close, bits_to_dev, dev
from test_gpu_sage import check_sage_layer, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

# (nodes, pairs): tensor-core contraction (2^20 outputs and more) with byte rows; bit-count contraction below that
SIZES = [(33000, 330000), (600, 9000)]


@pytest.mark.parametrize("n,e", SIZES)
@pytest.mark.parametrize("d_in,d_out", [(90, 33), (127, 47), (128, 48), (200, 49), (256, 47), (255, 60), (256, 61), (100, 64)])
def test_narrow_sage_layers(ctx, n, e, d_in, d_out):  # noqa: F811
    check_sage_layer(ctx, 0, n, e, d_in, d_out)


@pytest.mark.parametrize("n,e", SIZES + [(3000, 900000)])           # the last: hub rows, taken by a block
@pytest.mark.parametrize("d_in,d_out", [(256, 47), (256, 60), (100, 64), (200, 33)])
def test_narrow_sage_logits(ctx, n, e, d_in, d_out):  # noqa: F811
    from paper_2210_13149_b200 import binding as B
    rng = np.random.default_rng(n + d_out)
    g = oracle.mean_adjacency(n, *synth.edge_list(*synth.power_law_graph(n, e, 300 + n)))
    H = rng.standard_normal((n, d_in)).astype(np.float32)
    W = [(rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32) for _ in range(2)]
    t = oracle.sage_layer_forward(g, oracle.SageLayer(*W), H)
    G = B.make_graph(dev(g.rowptr), dev(g.colidx), dev(g.val), dev(g.dinv))
    out = ctx.sage_layer_forward(G, B.make_layer(d_in, d_out, bits_to_dev(t.bitsT_self), dev(t.alpha_self)),
                                 B.make_layer(d_in, d_out, bits_to_dev(t.bitsT_nbr), dev(t.alpha_nbr)), bits_to_dev(t.bits), dev(t.beta))
    assert_close(out["h"], t.H_out, "logits")


# byte rows: plain ones on a dense graph, half-dot ones; their hub rows are split over a block
BYTE_ROWS = [(3000, 900000, 100, 47), (3000, 900000, 127, 33), (24000, 800000, 256, 47), (24000, 800000, 255, 48), (32700, 1000000, 128, 33)]


@pytest.mark.parametrize("n,e,d_in,d_out", BYTE_ROWS)
def test_narrow_sage_logits_of_split_rows(ctx, n, e, d_in, d_out):  # noqa: F811
    rows = np.diff(synth.power_law_graph(n, e, 300 + n)[0].numpy())
    mean = rows.sum() // n
    assert mean >= 20 and (d_in <= 127 or n * d_out >= 1 << 20)                # byte rows
    assert n <= 32768 and rows.max() > max(128, 4 * (mean + 1), rows.sum() // 3552)   # the default length from which H' splits a row
    test_narrow_sage_logits(ctx, n, e, d_in, d_out)


@pytest.mark.parametrize("n,e,d_in,d_out", BYTE_ROWS)
def test_narrow_sage_layers_of_split_rows(ctx, n, e, d_in, d_out):  # noqa: F811
    assert synth.power_law_graph(n, e, 200 + n)[1].numel() >= 30 * n           # byte rows where a next layer follows, too
    check_sage_layer(ctx, 0, n, e, d_in, d_out)
