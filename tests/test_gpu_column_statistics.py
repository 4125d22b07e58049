"""Column statistics of one kernel whose last block of a column group adds the chunks up, against numpy in 64 bits."""
import numpy as np
import pytest

from parity_util import dev

pytestmark = pytest.mark.gpu


# one block and several per column group; rows on either side of a chunk of 64; one column, ragged and many groups (above 444 one chunk each)
@pytest.mark.parametrize("n,d", [(1, 1), (64, 33), (65, 33), (129, 600), (20000, 500), (70000, 7), (130, 20000)])
def test_column_statistics(n, d):
    from paper_2210_13149_b200 import binding as B
    H = np.random.default_rng(n + d).standard_normal((n, d)).astype(np.float32) * 3 + 100
    mean, var = H.astype(np.float64).mean(0), H.astype(np.float64).var(0)
    ctx = B.BiGCN(0)
    for _ in range(2):                                                         # the second call finds the counters as the first did
        shift, scale = ctx.col_stats(dev(H))
        np.testing.assert_allclose(shift.cpu().numpy(), mean, rtol=1e-7)       # one rounding of a sum in 64 bits
        np.testing.assert_allclose(scale.cpu().numpy(), 1 / np.sqrt(var + np.float64(np.float32(1e-5))), rtol=2e-7)
    ctx.sync_check()
    ctx.close()
