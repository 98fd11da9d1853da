"""The warps' walk over the WSPD's pairs against the oracle's sequential
enumeration, where it can go wrong: fewer pairs than lanes, chunks that end
inside a warp, stacks near their end (points on a line of doubling gaps give the
longest split paths), pairs handed on between launches, coordinates near the
limit (64-bit distances overflow) and thresholds beyond 64 bits.  Integers:
equality."""
import numpy as np
import pytest
import torch

import oracle

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


def _spread(v):
    x = np.asarray(v, np.uint64)
    for s, m in ((16, 0x0000FFFF0000FFFF), (8, 0x00FF00FF00FF00FF), (4, 0x0F0F0F0F0F0F0F0F), (2, 0x3333333333333333),
                 (1, 0x5555555555555555)):
        x = (x | (x << np.uint64(s))) & np.uint64(m)
    return x


def _nodes(X, Y):
    code = _spread(np.asarray(X, np.int64) - np.min(X)) | _spread(np.asarray(Y, np.int64) - np.min(Y)) << np.uint64(1)
    code, at = np.unique(code, return_index=True)
    X, Y = np.asarray(X, np.int32)[at], np.asarray(Y, np.int32)[at]
    A = 1 + np.arange(len(X), dtype=np.int64) % 3
    B = np.arange(len(X), dtype=np.int64) % 2
    return dict(X=X, Y=Y, cntA=A, cntB=B, code=code)


def _cases():
    rng = np.random.default_rng(5)
    g = np.int64(1) << np.arange(29)
    lim = (1 << 30) - 1
    yield "two", _nodes([0, 5], [0, 9])
    yield "three", _nodes([0, 5, 6], [0, 9, 9])
    yield "doubling", _nodes(np.r_[g, -g, np.zeros(29, np.int64), 7 * g[:25]], np.r_[g, g, g, -3 * g[:25]])
    yield "grid", _nodes(np.repeat(np.arange(40), 40), np.tile(np.arange(40), 40))
    yield "cloud", _nodes(rng.integers(0, 1 << 20, 1500), rng.integers(0, 1 << 20, 1500))
    # exact costs around squares, below and above where the float root alone is enough
    d = np.array([0, 2896308, 2896309, (1 << 22) - 1, 1 << 22, (1 << 22) + 1, (1 << 26) + 3, (1 << 29) + 1, lim - 1, lim])
    yield "squares", _nodes(np.r_[d, d], np.r_[0 * d, d % 2 + 1])
    yield "limits", _nodes(np.r_[rng.integers(-lim, lim, 120), -lim, lim], np.r_[rng.integers(-lim, lim, 120), -lim, lim])


@pytest.mark.parametrize("s", [1, 40, 4000000])
@pytest.mark.parametrize("name,nodes", list(_cases()), ids=lambda v: v if isinstance(v, str) else "")
def test_network_and_count_match_oracle(pd, ctx, name, nodes, s):
    d = {k: torch.from_numpy(np.ascontiguousarray(nodes[k])).cuda() for k in ("X", "Y", "cntA", "cntB")}
    d["morton"] = torch.from_numpy(nodes["code"].view(np.int64)).cuda()
    tree = oracle.radix_tree(nodes)
    exp = oracle.build_network(nodes, *oracle.wspd(nodes, tree, s))
    got = pd.pd_wspd_sparsify(ctx, d, s)
    for k in ("row_ptr", "head", "cost", "supply"):
        np.testing.assert_array_equal(got[k].cpu().numpy(), exp[k])
    assert pd.pd_wspd_count(ctx, d, s, 0) == got["n_arcs"] == int(exp["row_ptr"][-1])
    assert pd.pd_wspd_count(ctx, d, s, 1) == pd.pd_wspd_sparsify_tree(ctx, d, s, 1)[0]["n_arcs"]


# lattices with holes: counting stops at pairs of nodes below which only leaves
# can be separated; spacings and s on both sides of where that is looked for
@pytest.mark.parametrize("step,side,keep", [(1, 50, 0.6), (7, 40, 0.9), (1 << 20, 30, 0.8), (1 << 25, 20, 1.0)])
@pytest.mark.parametrize("s", [1, 4, 9, 40, 327])
def test_lattice_counts_match_oracle(pd, ctx, step, side, keep, s):
    rng = np.random.default_rng(side)
    X, Y = np.divmod(np.flatnonzero(rng.random(side * side) < keep), side)
    nodes = _nodes(step * X, step * Y)
    exp = oracle.build_network(nodes, *oracle.wspd(nodes, oracle.radix_tree(nodes), s))
    d = {k: torch.from_numpy(np.ascontiguousarray(nodes[k])).cuda() for k in ("X", "Y", "cntA", "cntB")}
    d["morton"] = torch.from_numpy(nodes["code"].view(np.int64)).cuda()
    assert pd.pd_wspd_count(ctx, d, s, 0) == int(exp["row_ptr"][-1])
