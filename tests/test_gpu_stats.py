"""bigcn_stats: the times of a layer's two products under the names they have in either order."""
import pytest
import torch

from paper_2210_13149_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2])
def test_both_products_of_a_layer_are_timed(order):
    from paper_2210_13149_b200 import binding as B
    ctx = B.BiGCN(0)
    ctx.set_option(B.OPT_ORDER, order)
    n, dims = 300000, (256, 256, 256, 40)
    G = ctx.normalize_adjacency(*synth.power_law_graph(n, 3000000, 1, device="cuda"))
    layers = ctx.prepare_layers(synth.weights(dims, 2, "cuda"))
    X = torch.randn((n, dims[0]), device="cuda")
    ctx.ensure_workspace(1 << 30)                                        # room for either order in every layer
    for _ in range(3):
        logits, st = ctx.forward(G, layers, X, stats=True)
    assert st.launches == (7 if order == 1 else 8)                       # pack, two per layer; pack, plan, two per layer
    for l in range(3):
        # neither product of a layer of these sizes takes less than a thirtieth of the other: 77 M multiply-adds per input
        # column against 3.3 M gathered rows
        assert st.ms_gemm[l] > st.ms_spmm[l] / 30 > 0 and st.ms_spmm[l] > st.ms_gemm[l] / 30
    assert st.ms_pack + sum(st.ms_gemm[:3]) + sum(st.ms_spmm[:3]) == pytest.approx(st.ms_total, rel=0.02)
    ctx.close()
