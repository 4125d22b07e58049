"""The tensor-core contraction of layers of more than 256 inputs: the same integers as the bit-count pipe, so the same H'."""
import numpy as np
import pytest
import torch

from paper_2210_13149_b200 import synth

pytestmark = pytest.mark.gpu


# d_in: one word, one piece and one chunk past 256, an odd number of pieces, dots beyond what a half's 511 trick holds,
# int16 dots; panels that stay in shared memory with one tile per multiprocessor, with several, and that do not; rows at
# the edges of a tile; 64, 128 and more channels, ragged
@pytest.mark.parametrize("n", [1, 127, 129, 5000])
@pytest.mark.parametrize("d_in,d_out", [(257, 1), (289, 64), (384, 65), (500, 256), (602, 200), (640, 129), (1433, 64),
                                        (2048, 300), (2049, 47), (3703, 64), (3703, 130)])
def test_wide_contraction_equals_the_bit_count_pipe(n, d_in, d_out):
    from paper_2210_13149_b200 import binding as B
    ctx = B.BiGCN(0)
    G = ctx.normalize_adjacency(*(t.cuda() for t in synth.power_law_graph(n, 4 * n, n)))
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


# between one slice and two per multiprocessor, and on either side: two blocks with a whole panel, a panel in chunks, three slices of 128
@pytest.mark.parametrize("n,d_in,d_out", [(18944, 1000, 128), (18945, 1000, 128), (37888, 300, 41), (37889, 300, 41), (25000, 1433, 64),
                                          (12601, 300, 300), (12545, 1000, 256)])
def test_one_wave_of_the_wide_contraction(n, d_in, d_out):
    test_wide_contraction_equals_the_bit_count_pipe(n, d_in, d_out)
