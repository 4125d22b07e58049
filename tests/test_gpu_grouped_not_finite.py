"""Grouped byte rows whose weights have no fixed point: results against the layer's definition in NumPy, and what one such weight beside a
hub row costs."""
import numpy as np
import pytest
import torch

import oracle
from parity_util import bits_to_dev, dev

pytestmark = pytest.mark.gpu


# rows of a group, on either side of one, of several pieces, scales and units of work; pairs of rows (of 0..60 entries) around them
@pytest.mark.parametrize("entries", [1, 64, 128, 129, 480, 700, 5000])
@pytest.mark.parametrize("d_in,d_out,fmt", [(127, 33, 3), (200, 47, 5), (201, 64, 5)])
@pytest.mark.parametrize("where", ["one", "some", "tiny"])
def test_weights_without_a_fixed_point(entries, d_in, d_out, fmt, where):
    from paper_2210_13149_b200 import binding as B
    n = 6000
    rng = np.random.default_rng(entries + d_out)
    lens = np.where(np.arange(n) % 100 == 7, entries, np.arange(n) % 61)
    rowptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    val = ((0.5 + rng.random(len(cols))) * rng.choice([-1, 1], len(cols))).astype(np.float32)
    if where == "tiny":                                                          # the row's other entries too, or some of its pieces only
        for r in range(7, n, 200):
            val[rowptr[r]:rowptr[r + 1]] *= np.float32(2.0 ** -110)
        val[rowptr[107]:rowptr[107] + entries // 2] *= np.float32(2.0 ** -110)
    else:
        for r in range(7, n, 100):
            at = rng.choice(np.arange(rowptr[r], rowptr[r + 1]), 1 if where == "one" else min(entries, 3), replace=False)
            val[at] = rng.choice([np.inf, -np.inf, np.nan, 1e34], len(at))
        val[rng.choice(len(val), 60, replace=False)] = np.inf                    # in rows of a pair
    F, beta = oracle.binarize_rows(rng.standard_normal((n, d_in)).astype(np.float32))
    signs, alpha = oracle.binarize_cols((rng.standard_normal((d_in, d_out)) * d_in ** -0.5).astype(np.float32))
    dots = F.astype(np.float64) @ signs.astype(np.float64)
    with np.errstate(invalid="ignore"):
        w = (val * beta[cols]).astype(np.float64)
        # entry by entry: a product with a dot of 0 is kept, for inf * 0
        want = np.stack([(w[a:b, None] * dots[cols[a:b]]).sum(0) for a, b in zip(rowptr, rowptr[1:])]) * alpha
        size = np.array([np.abs(w[a:b][np.isfinite(w[a:b])]).sum() for a, b in zip(rowptr, rowptr[1:])]) * alpha.max() * d_in
    ctx = B.BiGCN(0)
    ctx.set_option(B.OPT_ORDER, 1)
    ctx.set_option(B.OPT_BYTE_AGGREGATION, 2)
    ctx.set_option(B.OPT_ZETA_FORMAT, fmt)
    ctx.ensure_workspace(1 << 28)
    G, layer = B.make_graph(dev(rowptr), dev(cols), dev(val)), B.make_layer(d_in, d_out, bits_to_dev(oracle.pack_cols(signs)), dev(alpha))
    h = ctx.layer_forward(G, layer, bits_to_dev(oracle.pack_rows(F)), dev(beta))["h"].cpu().numpy()
    ctx.sync_check()
    ctx.close()
    finite = np.isfinite(want)
    np.testing.assert_array_equal(np.where(finite, 0, h), np.where(finite, 0, want))    # NaN and the signs of infinities
    assert np.all(np.abs(np.where(finite, h - np.where(finite, want, 0), 0)) <= size[:, None] * 2e-6)


def test_one_weight_beside_a_hub_row():
    """A graph of 200,000 nodes with a row of 100,000 entries, one of them NaN: the launch takes no more than three times as long."""
    from paper_2210_13149_b200 import binding as B
    n, hub = 200_000, 100_000
    gen = torch.Generator(device="cuda").manual_seed(1)
    lens = torch.full((n,), 60, device="cuda", dtype=torch.int64)
    lens[777] = hub
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = lens.cumsum(0)
    cols = torch.randint(0, n, (int(rowptr[-1]),), device="cuda", generator=gen, dtype=torch.int32)
    val = torch.rand(cols.numel(), device="cuda", generator=gen) / 60
    ctx = B.BiGCN(0)
    bits, beta = ctx.pack_features(torch.randn((n, 256), device="cuda", generator=gen))
    layer = ctx.prepare_layers([torch.randn((256, 47), device="cuda", generator=gen)])[0]
    took = []
    for bad in (False, True):
        v = val.clone()
        if bad:
            v[int(rowptr[777]) + 5] = float("nan")
        G = B.make_graph(rowptr, cols, v)
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            h = ctx.layer_forward(G, layer, bits, beta)["h"]
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        took.append(sorted(times)[3])
        assert bool(torch.isnan(h[777]).all()) == bad and not bool(torch.isnan(h[776]).any())
    ctx.close()
    assert took[1] < 3 * took[0], took
