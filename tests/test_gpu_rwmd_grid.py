"""The lower bounds' grid search on diagrams that crowd: clusters of the two sides
on the same places, next to each other and far apart, cells with thousands of
nodes beside empty ones, lattices.  Against the oracle's brute force: equality."""
import time

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


def _clusters(n, seed, centres, far, spread):
    r = np.random.default_rng(seed)
    c = np.random.default_rng(centres[0]).random((centres[1], 2)) * far
    p = c[r.integers(0, len(c), n)] + r.standard_normal((n, 2)) * spread
    p.sort(1)
    p[:, 1] += 1e-3
    return p.astype(np.float32)


KINDS = {
    "same": lambda n, s: _clusters(n, s, (7, 3), 200.0, 1e-3),
    "apart": lambda n, s: _clusters(n, s, (s, 3), 200.0, 1e-3),
    "many apart": lambda n, s: _clusters(n, s, (s, 40), 100.0, 1e-2),
    "loose": lambda n, s: _clusters(n, s, (s, 400), 100.0, 0.5),
    "shifted": lambda n, s: synth.mixture_f32(n, s) + np.float32(40 * s),
    "line": lambda n, s: np.stack([np.zeros(n), np.linspace(1e-3, 300, n) + s * 1e-4], 1).astype(np.float32),
}


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_crowded_diagrams(pd, kind):
    A, B = (KINDS[kind](n, s) for n, s in ((20000, 1), (19000, 2)))
    qa, qb = oracle.quantize(A, "f32", 20), oracle.quantize(B, "f32", 20)
    Ah, Bh = oracle.condense0(*qa), oracle.condense0(*qb)
    assert len(Ah[0]) * len(Bh[0]) >= 1 << 28
    c = pd.pd_create(0)
    try:
        for kappa, tau in ((1, 0), (0, 1 << 24)):
            got = pd.pd_rwmd_lower_bound(c, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(),
                                         pd.opts(diag_kappa=kappa, diag_tau=tau))
            assert got == oracle.rwmd(Ah, Bh, kappa, tau)
    finally:
        c.close()


# 3.2 ms; 8.3 where most queries end unfinished and go to the all-pairs scan
def test_clusters_apart_are_within_reach(pd):
    A, B = (torch.from_numpy(_clusters(100000, s, (s, 40), 200.0, 1e-3)).cuda() for s in (1, 2))
    c = pd.pd_create(0)
    ms = []
    try:
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            pd.pd_rwmd_lower_bound(c, A, B)
            ms.append(1e3 * (time.perf_counter() - t))
    finally:
        c.close()
    assert min(ms) < 5.5, ms
