"""Condensation and lower bounds around the sizes where their form changes: one
block up to 8,192 points, tiles of 4,096 keys above; one launch of the lower
bounds up to 8,192 nodes.  Against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2110_14734_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    from paper_2110_14734_gb300 import build
    build.build()
    from paper_2110_14734_gb300 import pdw1
    return pdw1


@pytest.fixture(scope="module")
def ctx(pd):
    c = pd.pd_create(0)
    yield c
    c.close()


def _diagram(kind, n, seed):
    if kind == "u8":  # many duplicates, about half below the diagonal's other side
        return np.random.default_rng(seed).integers(0, 256, (n, 2)).astype(np.uint8)
    if kind == "far":  # both signs, wide keys
        return np.random.default_rng(seed).uniform(-500, 500, (n, 2)).astype(np.float32)
    if kind == "line":  # one birth: the key's x part is empty
        return np.stack([np.full(n, 0.25), 0.25 + synth.mixture_f32(n, seed)[:, 0]], 1).astype(np.float32)
    return synth.mixture_f32(n, seed)


SIZES = [(1, 0), (0, 1), (1, 1), (33, 31), (1023, 1025), (4096, 4095), (4096, 4096), (8193, 0), (4097, 4096),
         (6000, 6288), (6144, 6145), (20000, 30000)]


@pytest.mark.parametrize("kind", ["f32", "u8", "far", "line"])
@pytest.mark.parametrize("na,nb", SIZES)
def test_condense_and_bounds_match_oracle(pd, ctx, kind, na, nb):
    A, B = _diagram(kind, na, 3 * na + nb), _diagram(kind, nb, 3 * na + nb + 1)
    dt = "u8" if kind == "u8" else "f32"
    k = oracle.default_shift(dt)
    hats = [oracle.condense0(*oracle.quantize(x, dt, k)) for x in (A, B)]
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    for G, P, seed in ((1, 0, 0), (300, 1, 7), (1 << 22, 9000, 3)):
        exp = oracle.condense_delta(*hats, G, P, seed)
        got = pd.pd_condense(ctx, dA, dB, G, P, pd.opts(seed=seed))
        assert got["n_nodes"] == len(exp["X"])
        for a in ("X", "Y", "cntA", "cntB"):
            np.testing.assert_array_equal(got[a].cpu().numpy(), exp[a])
        np.testing.assert_array_equal(got["morton"].cpu().numpy().view(np.uint64), exp["code"])
    if len(hats[0][0]) * len(hats[1][0]) < 3e8:
        for kappa, tau in ((1, 0), (0, 5000), (1, 77)):
            LA, LB = oracle.rwmd(*hats, kappa=kappa, tau=tau)[:2]
            got = pd.pd_rwmd_lower_bound(ctx, dA, dB, pd.opts(diag_kappa=kappa, diag_tau=tau))
            assert got == (LA, LB, max(LA, LB))


@pytest.mark.parametrize("n", [5, 5000, 9000])
def test_bad_and_empty_points(pd, ctx, n):
    A = synth.mixture_f32(n, n)
    on = A.copy()
    on[:, 1] = on[:, 0]  # every point on the diagonal
    assert pd.pd_condense(ctx, on, on)["n_nodes"] == 0
    assert pd.pd_rwmd_lower_bound(ctx, on, on[:0]) == (0, 0, 0)
    for bad in (np.nan, np.inf, -np.inf, 600.0):
        X = A.copy()
        X[n // 2, 1] = bad
        with pytest.raises(pd.PDError) as e:
            pd.pd_condense(ctx, X, A)
        assert e.value.status == pd.PD_EINVAL
    assert pd.pd_condense(ctx, A, on)["n_nodes"] > 0  # the context stays usable


# quantisation in single precision (a power of two scales a float exactly) up to
# k = 127 and in double above: ties, denormals, both forms of the stage
@pytest.mark.parametrize("k", [0, 1, 20, 100, 127, 128, 140])
@pytest.mark.parametrize("n", [500, 9000])
def test_quantised_coordinates_are_the_rounded_products(pd, ctx, k, n):
    rng = np.random.default_rng(k)
    q = rng.integers(-4000, 4000, (n, 2)) / 2.0  # whole numbers and ties
    q[: n // 4] += rng.uniform(-0.5, 0.5, (n // 4, 2))
    q[n // 4 : n // 3] *= 60000
    with np.errstate(under="ignore"):
        A = (q * 2.0 ** -k).astype(np.float32)
    exp = np.rint(A.astype(np.float64) * 2.0 ** k).astype(np.int64)
    exp = np.unique(exp[exp[:, 0] != exp[:, 1]], axis=0)
    got = pd.pd_condense(ctx, torch.from_numpy(A).cuda(), torch.from_numpy(A[:0]).cuda(), 1, 0, pd.opts(coord_shift=k))
    at = np.unique(np.stack([got["X"].cpu().numpy(), got["Y"].cpu().numpy()], 1), axis=0)
    np.testing.assert_array_equal(at, exp)


@pytest.mark.parametrize("v,k", [(np.inf, 20), (np.nan, 20), (3e38, 20), (1.0, 29), (1.0, 127), (2.0, 128)])
def test_coordinates_past_the_limit_stay_rejected(pd, ctx, v, k):
    A = torch.tensor([[0.0, v]], dtype=torch.float32).cuda()
    with pytest.raises(pd.PDError) as e:
        pd.pd_condense(ctx, A, A[:0], 1, 0, pd.opts(coord_shift=k))
    assert e.value.status == pd.PD_EINVAL
