"""The tuner's choices hold for the kernel and the form of arcs that they were
measured on, in a context and in the cache file."""
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


def _pair(scale=1.0):
    return [torch.from_numpy((synth.uniform_exp(400, s) * scale).astype(np.float32)).cuda() for s in (1, 2)]


def _list(cls):
    """An arc list of about 1.4 * 2^cls arcs and nodes."""
    n = 1000
    k = int(1.4 * 2 ** cls / n) - 1
    rng = np.random.default_rng(1)
    d = rng.choice(n - 2, k - 1, replace=False) + 2
    head = np.sort((np.arange(n)[:, None] + np.r_[1, d]) % n, 1).reshape(-1).astype(np.int32)
    sup = rng.integers(-9, 10, n)
    sup[-1] -= sup.sum()
    a = dict(row_ptr=k * np.arange(n + 1), head=head, cost=rng.integers(1, 1000, n * k), supply=sup)
    return {x: torch.from_numpy(v).cuda() for x, v in a.items()}


def _path(r):
    return r["opt_quanta"], r["pivots"], r["arcs_priced"]


@pytest.fixture(scope="module")
def line(pd, tmp_path_factory):
    """The fields of the cache line of the pair's matrix."""
    cache = str(tmp_path_factory.mktemp("tune") / "tune.txt")
    c = pd.pd_create(0)
    try:
        t = pd.pd_autotune(c, [_pair()[0]], [_pair()[1]], 0.5, pd.opts(ns_transport=2), cache_path=cache)
    finally:
        c.close()
    assert t["from_cache"] == 0 and t["ns_walk"] == 0  # a kernel that does not walk
    return open(cache).read().split()


def test_a_matrix_leaves_other_forms_alone(pd, line, tmp_path):
    cache = tmp_path / "tune.txt"
    cache.write_text(" ".join(line[:-2] + ["4096", "32"]) + "\n")
    net = _list(int(line[-3]))
    o = pd.opts(ns_transport=2, warm_start=0)
    got = []
    for path in (None, str(cache)):
        c = pd.pd_create(0)
        try:
            if path:
                t = pd.pd_autotune(c, [_pair()[0]], [_pair()[1]], 0.5, o, cache_path=path)
                assert (t["from_cache"], t["ns_block"], t["ns_walk"]) == (1, 4096, 32)
            got.append([_path(pd.pd_w1_approx(c, *_pair(), 0.5, o)), _path(pd.pd_w1_approx(c, *_pair(100.0), 0.5, o)),
                        _path(pd.pd_mcf_solve(c, net)[1])])
        finally:
            c.close()
    assert got[0][0][0] == got[1][0][0] and got[0][0] != got[1][0]  # the block is used where it belongs
    assert got[0][1:] == got[1][1:]  # a 64-bit matrix and an arc list of the class


def test_lines_without_a_form_are_not_taken(pd, line, tmp_path):
    cache = tmp_path / "tune.txt"
    other = ["Some_GPU 99 %s 8192 8" % line[-3], "Some_GPU 99 f3 %s 8192 8" % line[-3]]
    cache.write_text("\n".join(other + [" ".join(line[:2] + [line[-3], "4096", "32"])]) + "\n")
    c = pd.pd_create(0)
    try:
        t = pd.pd_autotune(c, [_pair()[0]], [_pair()[1]], 0.5, pd.opts(ns_transport=2), cache_path=str(cache))
    finally:
        c.close()
    assert t["from_cache"] == 0 and t["pairs"] == 1
    lines = cache.read_text().splitlines()
    assert lines[:2] == other and len(lines) == 3 and lines[2].split()[:4] == line[:4]


def test_both_kernels_are_tuned(pd, tmp_path):
    cache = str(tmp_path / "tune.txt")
    A, B = zip(_pair(), _pair(100.0))
    c = pd.pd_create(0)
    try:
        t = pd.pd_autotune(c, A, B, 0.5, pd.opts(ns_transport=2), cache_path=cache)
        assert t["pairs"] == 2 and t["ns_block"] == pd.pd_tuned_block(c, 1 << t["size_class"])
    finally:
        c.close()
    forms = [x.split()[2] for x in open(cache)]
    assert sorted(forms) == ["f1", "f3"]
