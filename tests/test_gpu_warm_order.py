"""The warm start's candidate lists and their order on the device: sizes around
the 32 columns of a block and the rows its threads share, all arcs at once up to
2^18 and lists above, many equal reduced costs (lattices).  A start changes no
optimum: equality with the cold solve."""
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


@pytest.mark.parametrize("kind", ["mixture", "lattice"])
@pytest.mark.parametrize("na,nb", [(1, 40), (31, 33), (33, 8200), (8200, 33), (513, 511), (512, 512), (700, 640)])
def test_started_solve_has_the_cold_optimum(pd, ctx, kind, na, nb):
    def diagram(n, seed):
        if kind == "mixture":
            return synth.mixture_f32(n, seed)
        at = np.random.default_rng(seed).permutation(1 << 15)[:n]
        return (np.stack([at // 256, at // 256 + 1 + at % 256], 1) / 64).astype(np.float32)

    A, B = (torch.from_numpy(np.ascontiguousarray(diagram(n, s))).cuda() for n, s in ((na, na), (nb, nb + 1)))
    kw = dict(ns_transport=2, condense=0)
    cold = pd.pd_w1_approx(ctx, A, B, 0.5, pd.opts(warm_start=0, **kw))["opt_quanta"]
    for ws in (2, 3, 4):
        assert pd.pd_w1_approx(ctx, A, B, 0.5, pd.opts(warm_start=ws, **kw))["opt_quanta"] == cold
