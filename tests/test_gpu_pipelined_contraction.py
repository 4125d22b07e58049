"""The pipelined contraction of layers of more than 256 inputs: the same integers as the bit-count pipe, so the same H'."""
import pytest
import torch

from paper_2210_13149_b200 import synth

pytestmark = pytest.mark.gpu


# one row; the edges of a tile; enough tiles that every block goes round its operand tiles and both accumulators several times, with a
# ragged last tile.  Widths: 64, 128 and 256 channels, ragged and in two slices; panels with two, three and four operand tiles; an odd
# number of 128-position pieces; the widest panel of each width that is covered and the first that is not
@pytest.mark.parametrize("n", [1, 128, 129, 60001])
@pytest.mark.parametrize("d_in,d_out", [(257, 256), (300, 400), (384, 130), (500, 256), (512, 512), (513, 256), (602, 41), (1000, 100),
                                        (1024, 128), (1025, 128), (2048, 64), (2049, 64)])
def test_pipelined_contraction_equals_the_bit_count_pipe(n, d_in, d_out):
    from paper_2210_13149_b200 import binding as B
    ctx = B.BiGCN(0)
    G = ctx.normalize_adjacency(*(t.cuda() for t in synth.power_law_graph(n, 2 * n, n)))
    gen = torch.Generator(device="cuda").manual_seed(d_in + d_out)
    X = torch.randn((n, d_in), device="cuda", generator=gen)
    W = torch.randn((d_in, d_out), device="cuda", generator=gen)
    X[0] = W[:, 0]                                              # dot = d_in, the largest there is
    bits, beta = ctx.pack_features(X)
    layer = ctx.prepare_layers([W])[0]
    for fmt in (B.ZETA_AUTO, B.ZETA_F32, B.ZETA_I16):
        ctx.set_option(B.OPT_ZETA_FORMAT, fmt)
        ctx.set_option(B.OPT_CONTRACTION, 1)
        want = ctx.layer_forward(G, layer, bits, beta)["h"]
        ctx.set_option(B.OPT_CONTRACTION, 2)
        got = ctx.layer_forward(G, layer, bits, beta)["h"]
        ctx.sync_check()
        assert torch.equal(got, want)
    ctx.close()
