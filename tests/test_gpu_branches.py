"""Branches that only unusual inputs reach: table builds over events with more
losses than a block evaluates ahead, and the adjoint over ids in host memory,
which it reads one by one."""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz", [0.2, 0.45, 0.6, 0.9])
@pytest.mark.parametrize("fp64", [False, True])
def test_tile_builds_of_dense_tables(nnz, fp64):
    """24 ELTs: 128 events hold 614 to 2,765 losses, below and above the 1,536 and
    2,048 that the builds of several groups evaluate ahead. The same tables, and
    so the same YLT, as the builds from the per-layer tables."""
    n_layers, C, T, K = 17, 3001, 300, 200
    w = workloads.random_case(13, catalogue=C, n_elt=24, n_layers=n_layers, n_trials=T, dense_k=K, max_elts_per_layer=9,
                              nnz_frac=nnz)
    p = w.portfolio
    for j in range(n_layers):  # ascending lists: both builds sum in this order
        a, b = p.layer_elt_off[j], p.layer_elt_off[j + 1]
        p.layer_elt_ids[a:b] = np.sort(p.layer_elt_ids[a:b])
    p.occ_ret[:], p.occ_lim[:] = 1e5, 5e6
    ids = torch.from_numpy(np.ascontiguousarray(w.yet.event_ids)).cuda()
    base = art.ART_LAYOUT_LAYER | (art.ART_LAYOUT_OCC64 if fp64 else 0)
    got = []
    for layouts in (base, base | art.ART_LAYOUT_SPARSE):
        h = art.portfolio_from_workload(w, layouts=layouts, variant=art.ART_VARIANT_FP64 if fp64 else art.ART_VARIANT_SKIP)
        try:
            y = torch.full((n_layers, T), -1.0, dtype=torch.float64, device="cuda")
            art.art_run_ylt(h, T, ids, None, K, y)
            assert art.art_get_device_status(h) == art.ART_OK
            got.append(y.cpu().numpy())
        finally:
            h.close()
    assert got[0].max() > 0
    np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("n_elt,per,nnz", [(8, 4, 0.1), (24, 24, 0.5)])  # records, table rows
def test_adjoint_over_ids_in_host_memory(ragged, n_elt, per, nnz):
    T, K, C, L = 400, 132, 2000, 3
    w = workloads.random_case(3, catalogue=C, n_elt=n_elt, n_layers=L, n_trials=1, dense_k=4, max_elts_per_layer=per,
                              nnz_frac=nnz)
    rng = np.random.default_rng(5)
    lengths = rng.integers(0, 2 * K, T) if ragged else np.full(T, K)
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    ids = torch.from_numpy(rng.integers(0, C, int(off[-1]), dtype=np.int32))
    dev, pinned = ids.cuda(), ids.pin_memory()
    d_off = torch.from_numpy(off).cuda() if ragged else None
    g = torch.from_numpy(rng.uniform(0.5, 1.5, (L, T))).cuda()
    p = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP | art.ART_LAYOUT_SPARSE,
                                    variant=art.ART_VARIANT_SKIP)
    try:
        y = torch.empty((L, T), dtype=torch.float64, device="cuda")
        br = torch.empty((L, T), dtype=torch.uint8, device="cuda")
        art.art_run_ylt(p, T, dev, d_off, 0 if ragged else K, y, br)
        outs = []
        stream = torch.cuda.current_stream().cuda_stream or None
        for ptr in (dev.data_ptr(), pinned.data_ptr()):
            gt = torch.full((L, 4), -1.0, dtype=torch.float64, device="cuda")
            gm = torch.full((n_elt,), -1.0, dtype=torch.float64, device="cuda")
            rc = art.lib().art_run_ylt_backward(p.handle, T, ptr, None if d_off is None else d_off.data_ptr(),
                                                0 if ragged else K, br.data_ptr(), g.data_ptr(), gt.data_ptr(),
                                                gm.data_ptr(), stream)
            assert rc == art.ART_OK and art.art_get_device_status(p) == art.ART_OK
            outs.append((gt.cpu().numpy(), gm.cpu().numpy()))
        np.testing.assert_array_equal(outs[0][0], outs[1][0])
        np.testing.assert_array_equal(outs[0][1], outs[1][1])
    finally:
        p.close()
