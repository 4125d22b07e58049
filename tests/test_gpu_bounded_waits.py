"""A wait that runs out inside the second product of a layer on packed bits: every block still ends, the status is reported, and
the device stays usable.  In a process of its own, because the reported flag stays up."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Layers of one and of two blocks of 128 output columns, whose waiting groups are four and eight warps, with the bits alone and
# with H', with and without a node's own term; 40 tiles and more to a block, 1 to 5 chunks of inputs to a tile.  With a
# few tries some of the warps of a group meet the end of their tries while others see the barrier complete.
CHILD = """
import torch
from paper_2210_13149_b200 import binding as B, synth
ctx = B.BiGCN(0)
ctx.set_option(B.OPT_ORDER, 2)
n = 200000
ctx.ensure_workspace(2 << 30)           # room for this order in every case from the first call on
pattern = synth.power_law_graph(n, 300000, 1, device="cuda")
G, M = ctx.normalize_adjacency(*pattern), ctx.mean_adjacency(*pattern)
cases = []
for d_in, d_out in ((64, 128), (100, 256), (600, 200)):
    own, nbr = ctx.prepare_layers([torch.randn((d_in, d_out), device="cuda") for _ in range(2)])
    nxt = B.make_layer(d_out, 1, torch.zeros((1, 16), dtype=torch.int32, device="cuda"), torch.ones(1, device="cuda"))
    bits, beta = ctx.pack_features(torch.randn((n, d_in), device="cuda"))
    for h in (False, True):
        cases.append(lambda a=(G, own, bits, beta), k=dict(want_h=h, next_layer=nxt): ctx.layer_forward(*a, **k))
        if d_in < 600:
            cases.append(lambda a=(M, own, nbr, bits, beta), k=dict(want_h=h, next_layer=nxt): ctx.sage_layer_forward(*a, **k))
want = [f()["next_bits"] for f in cases]
ctx.sync_check()
for tries in (1, 2, 3):
    ctx.set_option(B.OPT_WAIT_TRIES, tries)
    for f in cases:
        f()
    torch.cuda.synchronize()
try:
    ctx.sync_check()
    print("no wait ran out")
except B.BigcnError as e:
    print("status", e.status, e)
ctx.set_option(B.OPT_WAIT_TRIES, 0)
assert all(torch.equal(f()["next_bits"], w) for f, w in zip(cases, want))
print("usable")
"""


def test_a_wait_that_runs_out_ends_every_block_and_is_reported():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "status 8" in r.stdout and "a bounded wait ran out (layer kernel on packed bits)" in r.stdout, r.stdout
    assert r.stdout.endswith("usable\n")
