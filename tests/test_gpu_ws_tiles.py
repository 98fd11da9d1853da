"""The warm-start network at row counts around its tiles (16 rows a block, 152
blocks), against 64 bits.  The tolerance: sums of at most 128 float32 products per
unit and layer, of n rows per gradient, each rounded once (2^-24), over three
layers: 2^-24 (3 * 128 + n) relative to the sum of magnitudes, which the largest
entry's magnitude times a few bounds; 1e-5 of the norm covers it tenfold at these
sizes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    from paper_2110_14734_gb300 import build
    build.build()
    from paper_2110_14734_gb300 import pdw1
    return pdw1


@pytest.mark.parametrize("n", [1, 15, 16, 17, 100, 2432, 2433, 5000])
def test_forward_and_gradients(pd, n):
    rng = np.random.default_rng(n)
    p = (0.1 * rng.standard_normal(pd.WS_NPARAMS)).astype(np.float32)
    f = rng.standard_normal((n, pd.WS_NFEAT)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    m = (rng.random(n) < 0.8).astype(np.float32)
    c = pd.pd_create(0)
    try:
        pd.pd_ws_set_params(c, p)
        y = pd.pd_ws_forward(c, f)
        loss, g = pd.pd_ws_grad(c, f, t, m)
        again = pd.pd_ws_grad(c, f, t, m)
    finally:
        c.close()
    assert again[0] == loss and np.array_equal(again[1], g)  # sums in a fixed order
    bf = lambda a: torch.from_numpy(a).bfloat16().double()  # noqa: E731
    w1, b1, w2, b2, w3, b3 = torch.split(torch.from_numpy(p), [72 * 128, 128, 128 * 128, 128, 128, 1])
    leaves = [bf(w1.numpy()).view(72, 128), b1.double(), bf(w2.numpy()).view(128, 128), b2.double(), bf(w3.numpy()),
              b3.double()]
    for x in leaves:
        x.requires_grad_(True)
    h = torch.relu(bf(f) @ leaves[0] + leaves[1])
    h = torch.relu(h @ leaves[2] + leaves[3])
    ye = h @ leaves[4] + leaves[5]
    le = (torch.from_numpy(m).double() * (ye - torch.from_numpy(t).double()) ** 2).sum() / n
    le.backward()
    ge = torch.cat([x.grad.reshape(-1) for x in leaves]).numpy()
    assert np.linalg.norm(y - ye.detach().numpy()) <= 1e-5 * np.linalg.norm(ye.detach().numpy())
    assert abs(loss - le.item()) <= 1e-5 * max(le.item(), 1e-3)
    assert np.linalg.norm(g - ge) <= 1e-5 * np.linalg.norm(ge) + 1e-30
