"""Calls under memory caps of their context that they had always been content
with (the least ones found by bisection, plus a hundredth): scratch that only
saves time gives way."""
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


def _both(pd, cap, call):
    """The call's results without a cap and with it."""
    out = []
    for bytes_ in (0, cap + cap // 100):
        c = pd.pd_create(0, bytes_)
        try:
            out.append(call(c))
        finally:
            c.close()
    return out


# the warm-start network's rows, and its gradients' partial sums: another number
# of blocks adds in another order, each addition rounded once (2^-24), at most 160
# of them and 8 more in pairs
@pytest.mark.parametrize("n,grad,forward", [(16, 634877, 411646), (500, 2277367, 492542), (2048, 7536611, 712701),
                                            (5000, 17235902, 1150971), (20000, 19791796, 3375091)])
def test_network_rows(pd, n, grad, forward):
    rng = np.random.default_rng(n)
    p = (0.1 * rng.standard_normal(pd.WS_NPARAMS)).astype(np.float32)
    x = rng.standard_normal((n, pd.WS_NFEAT)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)

    def run(f):
        def call(c):
            pd.pd_ws_set_params(c, p)
            return f(c)
        return call

    a, b = _both(pd, forward, run(lambda c: pd.pd_ws_forward(c, x)))
    assert np.array_equal(a, b)
    (la, a), (lb, b) = _both(pd, grad, run(lambda c: pd.pd_ws_grad(c, x, t)))
    assert abs(la - lb) <= 1e-5 * la and np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(a)


def _mixture(n):
    return [torch.from_numpy(synth.mixture_f32(n, s)).cuda() for s in (1, 2)]


# the WSPD walk's room for pairs handed on
@pytest.mark.parametrize("n,s,cap", [(300, 1, 279551), (300, 8, 923644), (5000, 1, 6471655)])
def test_network_of_nodes(pd, n, s, cap):
    c = pd.pd_create(0)
    nodes = pd.pd_condense(c, *_mixture(n), 1, 0)
    c.close()
    a, b = _both(pd, cap, lambda c: pd.pd_wspd_sparsify(c, nodes, s))
    assert all(torch.equal(a[k], b[k]) for k in ("row_ptr", "head", "cost", "supply"))


@pytest.mark.parametrize("tree,cap", [(0, 461822), (1, 449534)])
def test_network_size(pd, tree, cap):
    a, b = _both(pd, cap, lambda c: pd.pd_w1_sparsify_count(c, *_mixture(300), 0.5, pd.opts(tree=tree))["n_arcs"])
    assert a == b


# the long sort's counts and tile states, kept while the next stage takes its own
@pytest.mark.parametrize("n,cap", [(5000, 638973), (100000, 17366974)])
def test_bounds(pd, n, cap):
    a, b = _both(pd, cap, lambda c: tuple(pd.pd_rwmd_lower_bound(c, *_mixture(n))))
    assert a == b
