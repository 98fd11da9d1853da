"""The sum of the training gradients over blocks of rows adds pairs of pairs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    from paper_2110_14734_gb300 import build
    build.build()
    from paper_2110_14734_gb300 import pdw1
    return pdw1


# 16 rows (a block's tile) repeated 2^k times: every block has the same sums, in
# which the mean over all rows only scales by a power of two, so that adding pairs of
# equal numbers rounds nothing and gives the gradients of the 16 rows bit for bit.
# One after the other, three equal numbers already round.
@pytest.mark.parametrize("times", [2, 4, 64, 128])
def test_equal_blocks_add_up_exactly(pd, times):
    rng = np.random.default_rng(4)
    p = (0.1 * rng.standard_normal(pd.WS_NPARAMS)).astype(np.float32)
    x = rng.standard_normal((16, pd.WS_NFEAT)).astype(np.float32)
    t = rng.standard_normal(16).astype(np.float32)
    m = (rng.random(16) < 0.8).astype(np.float32)
    c = pd.pd_create(0)
    try:
        pd.pd_ws_set_params(c, p)
        loss, g = pd.pd_ws_grad(c, x, t, m)
        loss_n, g_n = pd.pd_ws_grad(c, np.tile(x, (times, 1)), np.tile(t, times), np.tile(m, times))
    finally:
        c.close()
    assert np.array_equal(g, g_n) and loss == loss_n
