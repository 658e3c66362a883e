"""Payouts under a caller's capture: the caller's graph holds kernels only (a
graph with allocation nodes cannot be a child graph, nor run twice at once),
and its replays give the results of a plain call."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu

MEM_ALLOC, MEM_FREE = 10, 11  # CUgraphNodeType


def test_captured_payouts_allocate_nothing():
    cu = ctypes.CDLL("libcuda.so.1")
    T, K, C = 4000, 256, 20_000
    w = workloads.random_case(9, catalogue=C, n_elt=6, n_layers=1, n_trials=T, dense_k=K, max_elts_per_layer=6,
                              nnz_frac=0.1)
    p = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER)
    try:
        ids = torch.from_numpy(np.ascontiguousarray(w.yet.event_ids)).cuda()
        out = [torch.zeros(T * K, dtype=torch.float64, device="cuda"), torch.zeros(T, dtype=torch.int32, device="cuda"),
               torch.zeros(T, dtype=torch.float64, device="cuda")]
        art.art_run_payouts(p, 0, T, ids, None, K, *out)
        want = [t.cpu().numpy().copy() for t in out]
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        h, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
        assert cu.cuStreamBeginCapture_v2(h, 1) == 0  # thread-local
        art.art_run_payouts(p, 0, T, ids, None, K, *out, stream=stream)
        assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
        n = ctypes.c_size_t()
        assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0 and n.value > 0
        nodes = (ctypes.c_void_p * n.value)()
        assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
        kinds = []
        for node in nodes:
            kind = ctypes.c_int()
            assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
            kinds.append(kind.value)
        assert not {MEM_ALLOC, MEM_FREE} & set(kinds)
        ex = ctypes.c_void_p()
        assert cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)) == 0
        for _ in range(2):
            for t in out:
                t.fill_(-5)
            torch.cuda.synchronize()
            assert cu.cuGraphLaunch(ex, h) == 0
            stream.synchronize()
            # FP64 running sums against exact ones: an ulp of the running sum per event
            gross = float(want[2].max()) + float(w.portfolio.agg_ret[0])
            for t, v in zip(out, want):
                np.testing.assert_allclose(t.cpu().numpy(), v, rtol=1e-12, atol=K * 2.3e-16 * gross)
        cu.cuGraphExecDestroy(ex)
        cu.cuGraphDestroy(graph)
    finally:
        p.close()
