"""Stages whose scratch is larger than it has to be fall back to less of it under
a context's memory cap: the network's first guess at its arcs, the sorts' tile
states, the lower bounds' grid, the walk's hand-over buffers.  From the least cap
that still works upwards the results are those without a cap."""
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


def _run(pd, call, cap):
    ctx = pd.pd_create(0, cap)
    try:
        return call(ctx)
    except pd.PDError as e:
        assert e.status == pd.PD_ENOMEM
        return None
    finally:
        ctx.close()


def _calls(pd):
    A, B = (torch.from_numpy(synth.mixture_f32(20000, s)).cuda() for s in (1, 2))
    ctx = pd.pd_create(0)
    nodes = pd.pd_condense(ctx, A, B, 1, 0)
    ctx.close()

    def flat(d):
        return tuple(tuple(d[k].cpu().tolist()) if torch.is_tensor(d[k]) else d[k] for k in sorted(d))

    return {"condense": lambda c: flat(pd.pd_condense(c, A, B, 3, 0)),
            "bounds": lambda c: tuple(pd.pd_rwmd_lower_bound(c, A, B)),
            "network": lambda c: flat(pd.pd_wspd_sparsify(c, nodes, 1)),
            "count": lambda c: pd.pd_w1_sparsify_count(c, A, B, 0.5)["n_arcs"]}


@pytest.mark.parametrize("name", ["condense", "bounds", "network", "count"])
def test_results_do_not_depend_on_the_cap(pd, name):
    call = _calls(pd)[name]
    exp = _run(pd, call, 0)
    lo, hi = 1 << 20, 1 << 28
    assert _run(pd, call, lo) is None and _run(pd, call, hi) == exp
    while hi - lo > lo // 16:  # every size on the way is one of the forms, or refused
        mid = (lo + hi) // 2
        got = _run(pd, call, mid)
        assert got is None or got == exp
        lo, hi = (mid, hi) if got is None else (lo, mid)
