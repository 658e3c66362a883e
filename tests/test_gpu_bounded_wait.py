"""A kernel's wait for its own copies is bounded: when it runs out, every lane
of the warp gives up together and the status says so. The wait here is for a
copy that nobody requested, with limits of microseconds."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit_us", [0, 1, 50])
def test_wait_gives_up_and_reports(limit_us):
    w = workloads.random_case(3, catalogue=100, n_elt=3, n_layers=1, n_trials=40, dense_k=8, max_elts_per_layer=3)
    p = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER, variant=art.ART_VARIANT_SKIP)
    try:
        disagree = torch.zeros(1, dtype=torch.int32, device="cuda")
        f = art.lib().art_test_wait
        f.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p]
        stream = torch.cuda.current_stream().cuda_stream or None
        assert f(p.handle, 1000 * limit_us, disagree.data_ptr(), stream) == art.ART_OK
        assert art.art_get_device_status(p) == art.ART_ETIMEOUT
        assert disagree.item() == 0
        # the status was read and cleared; the next call is not affected
        ids = torch.from_numpy(np.ascontiguousarray(w.yet.event_ids)).cuda()
        y = torch.empty((1, 40), dtype=torch.float64, device="cuda")
        art.art_run_ylt(p, 40, ids, None, 8, y)
        assert art.art_get_device_status(p) == art.ART_OK
    finally:
        p.close()
