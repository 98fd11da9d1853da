"""The 32-bit simplex kernel against the 64-bit one (ns_smem = 0 runs that one
on any instance) and against closed forms: edges of its three layouts, matrix
rows around the padding, paths longer than its lists, and the instances that it
has to hand back to the 64-bit kernel.  Optima are integers: equality."""
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


def _net(n, tails, heads, cost, supply):
    order = np.lexsort((heads, tails))
    tails, heads, cost = (np.asarray(x)[order] for x in (tails, heads, cost))
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, tails + 1, 1)
    a = dict(row_ptr=np.cumsum(rp), head=heads.astype(np.int32), cost=cost.astype(np.int64),
             supply=np.asarray(supply, np.int64))
    return {k: torch.from_numpy(v).cuda() for k, v in a.items()}


def _chain(n, cost, supply):
    """Both directions of a line of n nodes."""
    u = np.arange(n - 1)
    return _net(n, np.r_[u, u + 1], np.r_[u + 1, u], np.r_[cost, cost], supply)


def _chain_opt(cost, supply):
    return int(np.sum(np.abs(np.cumsum(supply)[:-1]) * np.asarray(cost, np.int64)))


# a shortest route above the 32-bit kernel's artificial cost, potentials above
# its limit, and costs above what it takes at all
@pytest.mark.parametrize("n,c", [(3, 1 << 25), (40, 1 << 25), (40, (1 << 25) + 1), (2000, (1 << 20) + 3)])
def test_costs_beyond_32_bits_reach_the_64_bit_kernel(pd, ctx, n, c):
    cost = np.full(n - 1, c, np.int64)
    sup = np.zeros(n, np.int64)
    sup[0], sup[-1] = 3, -3
    net = _chain(n, cost, sup)
    assert pd.pd_mcf_solve(ctx, net)[0] == _chain_opt(cost, sup)
    assert pd.pd_mcf_solve_noalloc(net) == _chain_opt(cost, sup)


def test_infeasible_stays_infeasible(pd, ctx):
    for c in (7, 1 << 25):  # two components that each lack balance
        net = _net(40, [0, 1, 20], [1, 0, 21], [c] * 3, [5] + [0] * 38 + [-5])
        with pytest.raises(pd.PDError) as e:
            pd.pd_mcf_solve(ctx, net)
        assert e.value.status == pd.PD_EINFEASIBLE


# tree paths past the register forms (32, 64, 128 nodes) and the listed ones (1024)
@pytest.mark.parametrize("n", [2, 31, 66, 131, 1030, 3001, 7823])
def test_long_paths(pd, ctx, n):
    rng = np.random.default_rng(n)
    cost = rng.integers(0, 50, n - 1)
    sup = rng.integers(-9, 10, n)
    sup[-1] -= sup.sum()
    net = _chain(n, cost, sup)
    assert pd.pd_mcf_solve(ctx, net)[0] == _chain_opt(cost, sup)
    one = np.zeros(n, np.int64)
    one[0], one[-1] = 1, -1  # a single path through the whole line
    net["supply"] = torch.from_numpy(one).cuda()
    assert pd.pd_mcf_solve(ctx, net)[0] == _chain_opt(cost, one)


# nodes + root around the capacities of the layouts (7824, 13040, 23664) and the
# limit of 16-bit node ids
@pytest.mark.parametrize("n", [7823, 7824, 13039, 13040, 23663, 23664])
def test_layout_edges(pd, ctx, n):
    rng = np.random.default_rng(n)
    side = int(np.sqrt(n))
    u = np.arange(n)
    hop = np.unique(np.r_[1, rng.integers(2, side, 3)])  # a line and three strides: connected both ways
    t = np.concatenate([np.r_[u[:-h], u[h:]] for h in hop])
    h = np.concatenate([np.r_[u[h:], u[:-h]] for h in hop])
    cost = rng.integers(1, 1000, len(t))
    sup = np.zeros(n, np.int64)
    at = rng.choice(n, 600, replace=False)
    sup[at] = np.r_[np.full(300, 2), np.full(300, -2)]
    net = _net(n, t, h, cost, sup)
    assert pd.pd_mcf_solve(ctx, net)[0] == pd.pd_mcf_solve(ctx, net, pd.opts(ns_smem=0))[0]


# rows of the cost matrix around the padding to eight columns, one-sided and
# unequal diagrams (arcs of the diagonal node), and blocks smaller than a step
@pytest.mark.parametrize("na,nb", [(1, 1), (1, 0), (0, 3), (2, 7), (8, 8), (9, 17), (30, 31), (33, 64), (257, 63)])
def test_small_and_ragged_pairs(pd, ctx, na, nb):
    A = torch.from_numpy(synth.mixture_f32(max(na, 1), 7 * na + nb)[:na]).cuda()
    B = torch.from_numpy(synth.mixture_f32(max(nb, 1), 7 * na + nb + 1)[:nb]).cuda()
    for kw in (dict(), dict(diag_kappa=0, diag_tau=20000), dict(ns_block=1)):
        got = pd.pd_w1_approx(ctx, A, B, 0.5, pd.opts(**kw))
        exp = pd.pd_w1_approx(ctx, A, B, 0.5, pd.opts(ns_smem=0, **kw))
        assert got["opt_quanta"] == exp["opt_quanta"]


# a batch whose pairs go to different kernels: coordinates far beyond 32-bit
# potentials beside ordinary ones, one-sided pairs, and a wave larger than the slots
def test_mixed_batch(pd, ctx):
    small = [torch.from_numpy(synth.uniform_exp(n, 50 + n)).cuda() for n in (40, 90, 300)]
    far = [torch.from_numpy((synth.uniform_exp(n, n) * 100).astype(np.float32)).cuda() for n in (60, 80)]
    none = small[0][:0]
    As, Bs = [small[0], far[0], small[2], none, small[1]], [small[1], far[1], small[0], small[2], none]
    for kw in (dict(), dict(batch_slots=2)):
        got = pd.pd_w1_approx_batch(ctx, As, Bs, 0.5, pd.opts(**kw))
        for r, a, b in zip(got, As, Bs):
            assert r["opt_quanta"] == pd.pd_w1_approx(ctx, a, b, 0.5, pd.opts(ns_smem=0))["opt_quanta"]


# caps take effect where they did: the pivot cap, and a status per call
def test_pivot_cap(pd, ctx):
    A, B = (torch.from_numpy(synth.uniform_exp(300, s)).cuda() for s in (1, 2))
    full = pd.pd_w1_approx(ctx, A, B, 0.5)["opt_quanta"]
    with pytest.raises(pd.PDError) as e:
        pd.pd_w1_approx(ctx, A, B, 0.5, pd.opts(max_rounds=3))
    assert e.value.status == pd.PD_ETIMEOUT
    assert pd.pd_w1_approx(ctx, A, B, 0.5)["opt_quanta"] == full


def _grid_pair(nodes, seed):
    """Two disjoint diagrams of `nodes` points in all on a lattice of 4,096 places."""
    rng = np.random.default_rng(seed)
    at = rng.permutation(4096)[:nodes]
    pts = np.stack([at // 64, at // 64 + 1 + at % 64], 1).astype(np.float32) / 64
    k = nodes // 2 + int(rng.integers(-40, 41))
    return tuple(torch.from_numpy(np.ascontiguousarray(p)).cuda() for p in (pts[:k], pts[k:]))


# around the sizes up to which an instance takes half an SM by itself, and up
# to which half an SM holds it (more such pairs than SMs)
@pytest.mark.parametrize("nodes", [1277, 1278, 1279, 1280, 1281])
def test_small_instances_on_half_an_sm(pd, ctx, nodes):
    A, B = _grid_pair(nodes, nodes)
    got = pd.pd_w1_approx(ctx, A, B, 0.01, pd.opts(warm_start=0))
    assert got["opt_quanta"] == pd.pd_w1_approx(ctx, A, B, 0.01, pd.opts(ns_smem=0))["opt_quanta"]


def test_two_instances_per_sm(pd, ctx):
    pairs = [_grid_pair(n, n) for n in (3708, 3709, 3710, 3711, 3712, 3713, 700)]
    exp = [pd.pd_w1_approx(ctx, a, b, 0.01, pd.opts(ns_smem=0))["opt_quanta"] for a, b in pairs]
    many = [i for i in range(4) for _ in range(40)] + list(range(4, len(pairs)))  # 160 that surely fit, then the edge
    got = pd.pd_w1_approx_batch(ctx, [pairs[i][0] for i in many], [pairs[i][1] for i in many], 0.01)
    assert [r["opt_quanta"] for r in got] == [exp[i] for i in many]


# arc lists around the size from which their chunks are spread over the pricing
# blocks, with and without a part chunk: assignment problems
@pytest.mark.parametrize("k", [2047, 2048, 2050])
def test_spread_arc_lists(pd, ctx, k):
    from scipy.optimize import linear_sum_assignment
    cost = np.random.default_rng(k).integers(0, 1 << 20, (k, k))
    u, v = np.divmod(np.arange(k * k), k)
    net = _net(2 * k, u, v + k, cost.reshape(-1), np.r_[np.ones(k, np.int64), -np.ones(k, np.int64)])
    assert pd.pd_mcf_solve(ctx, net)[0] == cost[linear_sum_assignment(cost)].sum()
