"""The 64-bit simplex kernel's forms of an instance and the waves that mix them
with the 32-bit kernel's.  Optima are integers: equality with the 32-bit kernel,
closed forms or single solves."""
import numpy as np
import pytest
import torch

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


def _circulant(n, k, cost, supply, seed=0):
    """Network of n nodes with arcs to the same k distances from every node."""
    d = np.random.default_rng(seed).choice(n - 1, k, replace=False) + 1
    a = dict(row_ptr=k * np.arange(n + 1), head=np.sort((np.arange(n)[:, None] + d) % n, 1).reshape(-1).astype(np.int32),
             cost=np.broadcast_to(np.asarray(cost, np.int64), (n * k,)).copy(), supply=np.asarray(supply, np.int64))
    return {x: torch.from_numpy(v).cuda() for x, v in a.items()}


# arc lists around whole chunks (64) and pricing blocks, which may end inside the
# list, at its padding or among the artificial arcs
@pytest.mark.parametrize("n,k", [(16, 3), (64, 1), (64, 63), (1024, 8), (1025, 8), (2049, 5)])
@pytest.mark.parametrize("block", [0, 1, 8, 1000])
def test_packed_lists(pd, ctx, n, k, block):
    rng = np.random.default_rng(n * k)
    sup = rng.integers(-5, 6, n)
    sup[-1] -= sup.sum()
    net = _circulant(n, k, rng.integers(0, 1000, n * k), sup, n * k)

    def solve(**kw):
        try:
            return pd.pd_mcf_solve(ctx, net, pd.opts(**kw))[0]
        except pd.PDError as e:
            return e.status

    assert solve(ns_smem=0, ns_block=block) == solve(ns_block=block) == solve()


# One look at every arc (no supplies: the start is optimal).  0.60 ms; 1.46 with
# the ends' form looked up arc by arc, 1.14 with tails and heads apart.
def test_packed_lists_are_priced_at_their_rate(pd, ctx):
    n, k = 9000, 222
    net = _circulant(n, k, 1 << 26, np.zeros(n))
    ms = [pd.pd_mcf_solve(ctx, net)[1]["ns_kernel_ms"] for _ in range(5)]
    assert min(ms) < 1.1, ms


# 46,337 x 46,337 arcs and the nodes just fit 31-bit arc ids; rows padded to 46,344 would not
def test_largest_matrix_is_taken(pd, ctx):
    n = 46337
    at = np.random.default_rng(3).permutation(1 << 17)[: 2 * n]
    pts = np.stack([at // 512, at // 512 + 1 + at % 512], 1).astype(np.float32) / 64
    A, B = (torch.from_numpy(np.ascontiguousarray(p)).cuda() for p in (pts[:n], pts[n:]))
    c = pd.pd_create(0)
    try:
        with pytest.raises(pd.PDError) as e:  # one pivot is enough to see that it was taken
            pd.pd_w1_approx(c, A, B, 0.5, pd.opts(condense=0, ns_transport=2, warm_start=0, max_rounds=1))
    finally:
        c.close()
    assert e.value.status == pd.PD_ETIMEOUT


def _u(n, seed, scale=1.0):
    return torch.from_numpy((synth.uniform_exp(n, seed) * scale).astype(np.float32)).cuda()


# a wave of every form at once: matrices of the three layouts, of half an SM, for
# the 64-bit kernel, and one-sided pairs (arc lists); twice, the second time from
# the captured graph
def test_a_wave_of_all_forms(pd, ctx):
    def mixture(n, seed):
        return torch.from_numpy(synth.mixture_f32(n, seed)).cuda()

    none = _u(40, 1)[:0]
    pairs = [(mixture(9000, 1), mixture(9000, 2)), (_u(200, 3), none), (mixture(6000, 1), mixture(6000, 2)),
             (_u(400, 5, 100.0), _u(300, 6, 100.0)), (none, _u(90, 7)), (_u(2600, 8), _u(2500, 9))]
    pairs += [(_u(300 + i, 20 + i), _u(280, 60 + i)) for i in range(4)] * 40
    o = pd.opts(ns_transport=2, batch_slots=len(pairs))
    exp = [pd.pd_w1_approx(ctx, a, b, 0.1, pd.opts(ns_transport=2, warm_start=0))["opt_quanta"] for a, b in pairs[:10]]
    for _ in range(2):
        got = pd.pd_w1_approx_batch(ctx, [a for a, _ in pairs], [b for _, b in pairs], 0.1, o)
        assert [r["opt_quanta"] for r in got] == exp[:6] + exp[6:] * 40


# Pairs for the two kernels take the device's time together, not one after the
# other: 40 instances on 152 SMs, about 75 ms for each kernel alone.
def test_a_mixed_wave_overlaps(pd, ctx):
    far = [(_u(1500, i, 100.0), _u(1500, 50 + i, 100.0)) for i in range(4)] * 5
    near = [(_u(6000, i), _u(6000, 50 + i)) for i in range(4)] * 5

    def ms(pairs):
        return min(max(r["ns_kernel_ms"] for r in pd.pd_w1_approx_batch(ctx, [a for a, _ in pairs], [b for _, b in pairs], 0.1))
                   for _ in range(3))

    apart = ms(far), ms(near)
    assert min(apart) > 40
    assert ms(far + near) < max(apart) + 0.5 * min(apart), apart


# cost matrices on the layouts with more nodes (N + 2 up to 13,040 and 23,664, then
# the 64-bit kernel), rows from every alignment of the sinks' potentials, either
# side the longer one, cold and from a start.  At s = 2,000 no two nodes of the
# 128 x 256 lattice are separated before they are leaves: every arc of the matrix is
# one of the network and the certificate holds.
@pytest.mark.parametrize("na,nb", [(57, 12981), (58, 12981), (61, 13500), (64, 14001), (59, 23603), (60, 23603),
                                   (13500, 62)])
def test_large_matrices(pd, ctx, na, nb):
    at = np.random.default_rng(na * nb).permutation(1 << 15)[: na + nb]
    pts = np.stack([at // 256, at // 256 + 1 + at % 256], 1).astype(np.float32) / 64
    A, B = (torch.from_numpy(np.ascontiguousarray(p)).cuda() for p in (pts[:na], pts[na:]))
    kw = dict(condense=0, ns_transport=2, s_override=2000)
    exp = pd.pd_w1_approx(ctx, A, B, 0.1, pd.opts(warm_start=0, ns_smem=0, **kw))
    for start in (0, 3, 4):
        got = pd.pd_w1_approx(ctx, A, B, 0.1, pd.opts(warm_start=start, **kw))
        assert got["cert_failures"] == exp["cert_failures"] == 0
        assert got["opt_quanta"] == exp["opt_quanta"]


def _grid(side, top):
    """A square grid, arcs both ways between neighbours, costs up to top."""
    rng = np.random.default_rng(side)
    n = side * side
    u = np.arange(n)
    r, d = u[u % side < side - 1], u[u < n - side]
    t, h = np.r_[r, r + 1, d, d + side], np.r_[r + 1, r, d + side, d]
    o = np.lexsort((h, t))
    sup = np.zeros(n, np.int64)
    at = rng.permutation(n)[: n // 4 * 2]
    k = len(at) // 2
    sup[at[:k]] = rng.integers(1, 9, k)
    sup[at[k:]] = -sup[at[:k]]
    a = dict(row_ptr=np.r_[0, np.cumsum(np.bincount(t, minlength=n))], head=h[o].astype(np.int32),
             cost=rng.integers(1, top + 1, len(t))[o], supply=sup)
    return {x: torch.from_numpy(v).cuda() for x, v in a.items()}


# Routes of more than 32 bits of cost: the 32-bit kernel's tree, from each of its
# layouts, is where the 64-bit kernel goes on.
@pytest.mark.parametrize("side", [30, 100, 130])
def test_a_handed_back_tree_goes_on(pd, ctx, side):
    big = _grid(side, 1 << 25)
    opt, r = pd.pd_mcf_solve(ctx, big)
    exp = pd.pd_mcf_solve(ctx, big, pd.opts(ns_smem=0))[0]
    assert opt == exp and opt == pd.pd_mcf_solve(ctx, big, pd.opts(max_rounds=r["pivots"]))[0]
    with pytest.raises(pd.PDError) as e:  # pivots of both kernels count
        pd.pd_mcf_solve(ctx, big, pd.opts(max_rounds=r["pivots"] - 1))
    assert e.value.status == pd.PD_ETIMEOUT


# ... which takes 1.7 times as long as a solve that fits, and 4.2 times from a cold start
def test_a_handed_back_solve_is_not_done_twice(pd, ctx):
    ms = [min(pd.pd_mcf_solve(ctx, _grid(30, top))[1]["ns_kernel_ms"] for _ in range(4)) for top in (1 << 25, 1 << 10)]
    assert ms[0] < 2.8 * ms[1], ms


# Lists of more nodes than the 32-bit kernel holds stay in order: 174,644 pivots
# (2.9 s), spread over the pricing blocks 274,555 (5.0 s).
def test_large_lists_stay_in_order(pd, ctx):
    A, B = (torch.from_numpy(synth.gaussian_pd(15000, s)).cuda() for s in (1000, 1001))
    r = pd.pd_w1_approx(ctx, A, B, 0.1, pd.opts(s_override=9, ns_transport=0, warm_start=0))
    assert r["n_nodes"] > 23663 and r["n_arcs"] > 1 << 22
    assert r["pivots"] < 220000
