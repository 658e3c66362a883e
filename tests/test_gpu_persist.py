"""The persisting L2 area: reserved while a portfolio created with
ART_FLAG_L2_PERSIST lives, then as it was found, unless the caller has set a limit
of its own since."""
import ctypes

import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu

LIMIT = 0x06  # CU_LIMIT_PERSISTING_L2_CACHE_SIZE


def _limit(cu):
    v = ctypes.c_size_t()
    assert cu.cuCtxGetLimit(ctypes.byref(v), LIMIT) == 0
    return v.value


def test_persisting_limit_comes_back():
    cu = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    w = workloads.random_case(3, catalogue=100, n_elt=3, n_layers=1, n_trials=8, dense_k=4, max_elts_per_layer=3)
    found = _limit(cu)
    try:
        p = art.portfolio_from_workload(w, flags=art.ART_FLAG_L2_PERSIST)
        q = art.portfolio_from_workload(w, flags=art.ART_FLAG_L2_PERSIST)
        reserved = _limit(cu)
        assert reserved > found
        p.close()
        assert _limit(cu) == reserved
        q.close()
        assert _limit(cu) == found
        # the caller's own limit, set while a portfolio lives, stays
        p = art.portfolio_from_workload(w, flags=art.ART_FLAG_L2_PERSIST)
        assert cu.cuCtxSetLimit(LIMIT, ctypes.c_size_t(8 << 20)) == 0
        mine = _limit(cu)
        assert mine != reserved
        p.close()
        assert _limit(cu) == mine
    finally:
        cu.cuCtxSetLimit(LIMIT, ctypes.c_size_t(found))
