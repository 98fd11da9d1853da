"""The long radix sort where a tile does not wait for the counts of the tiles
before it but counts their digits itself: sizes around whole tiles (4,096 keys),
few and many digits, with and without values.  Against numpy's stable sort:
equality."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SORT = "_ZN2pd8sort_u64EPNS_3CtxERPmS3_RPjS5_liP11CUstream_sti"  # pd::sort_u64(..., stream, polls)


@pytest.fixture(scope="module")
def pd():
    from paper_2110_14734_gb300 import build
    build.build()
    from paper_2110_14734_gb300 import pdw1
    return pdw1


@pytest.mark.parametrize("n", [8193, 12287, 12288, 12289, 700001])
@pytest.mark.parametrize("bits", [3, 16, 37])
@pytest.mark.parametrize("values", [False, True])
@pytest.mark.parametrize("polls", [0, 4096])
def test_sort_never_depends_on_the_wait(pd, n, bits, values, polls):
    sort = getattr(pd._lib, SORT)
    sort.restype = ctypes.c_int
    keys = np.random.default_rng(n + bits).integers(0, 1 << bits, n)
    order = np.argsort(keys, kind="stable")
    k = [torch.from_numpy(keys).cuda(), torch.full((n,), -1, dtype=torch.int64, device="cuda")]
    v = [torch.arange(n, dtype=torch.int32, device="cuda"), torch.full((n,), -1, dtype=torch.int32, device="cuda")]
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in k] + [ctypes.c_void_p(t.data_ptr() if values else None) for t in v]
    c = pd.pd_create(0)
    try:
        torch.cuda.synchronize()
        assert sort(c.ptr, *[ctypes.byref(p) for p in ptr], ctypes.c_int64(n), ctypes.c_int(bits), None,
                    ctypes.c_int(polls)) == pd.PD_OK
        torch.cuda.synchronize()
    finally:
        c.close()
    at = [t.data_ptr() for t in k].index(ptr[0].value)
    assert np.array_equal(k[at].cpu().numpy(), keys[order])
    if values:
        at = [t.data_ptr() for t in v].index(ptr[2].value)
        assert np.array_equal(v[at].cpu().numpy(), order)
