"""The group adjoint where events hold many losses: by table rows, by records
with events evaluated from their row, and both in one call (they share the
call's scratch), against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


def _check(w, layouts, lengths, seed):
    rng = np.random.default_rng(seed)
    L, E, C, T = w.portfolio.n_layers, w.portfolio.n_elt, w.portfolio.catalogue_size, lengths.size
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    ids = rng.integers(0, C, size=int(off[-1]), dtype=np.int32)
    w.yet = workloads.YET(n_trials=T, event_ids=ids, trial_off=off)
    s = oracle.ylt(w.oracle_problem(), want_sum=True)[2]
    w.portfolio.agg_ret[:] = np.median(s, axis=1) * 0.5 + 1.0
    w.portfolio.agg_lim[:] = np.median(s, axis=1) + 1.0
    g = rng.uniform(0.5, 1.5, size=(L, T))
    ot, om, _, _ = oracle.grad(w.oracle_problem(), g)
    p = art.portfolio_from_workload(w, layouts=layouts, variant=art.ART_VARIANT_SKIP)
    try:
        d_ids, d_off = torch.from_numpy(ids).cuda(), torch.from_numpy(off).cuda()
        y = torch.empty((L, T), dtype=torch.float64, device="cuda")
        br = torch.empty((L, T), dtype=torch.uint8, device="cuda")
        art.art_run_ylt(p, T, d_ids, d_off, 0, y, br)
        gt = torch.empty((L, 4), dtype=torch.float64, device="cuda")
        gm = torch.empty(E, dtype=torch.float64, device="cuda")
        art.art_run_ylt_backward(p, T, d_ids, d_off, 0, br, torch.from_numpy(g).cuda(), gt, gm)
        assert art.art_get_device_status(p) == art.ART_OK
    finally:
        p.close()
    # weights and products are FP32 (2^-24 each), the sums compensated
    np.testing.assert_allclose(gt.cpu().numpy(), ot, rtol=1e-6, atol=1e-6 * np.abs(ot).max())
    np.testing.assert_allclose(gm.cpu().numpy(), om, rtol=2e-6, atol=1e-6 * np.abs(om).max())


LENGTHS = np.array([0, 1, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 1000] * 3 + [300] * 40)


# losses per event below and above the line between records and rows, row widths 4 to 32
@pytest.mark.parametrize("n_elt,n_layers,per,nnz", [(4, 1, 4, 0.9), (8, 1, 8, 0.12), (8, 1, 8, 0.9), (16, 2, 16, 0.08),
                                                    (16, 8, 8, 0.14), (16, 8, 8, 0.3), (24, 1, 24, 0.07), (24, 3, 24, 0.4),
                                                    (32, 1, 32, 0.07), (32, 5, 32, 0.15)])
@pytest.mark.parametrize("csr", [False, True])
def test_dense_groups(n_elt, n_layers, per, nnz, csr):
    w = workloads.random_case(71 + n_elt, catalogue=3001, n_elt=n_elt, n_layers=n_layers, n_trials=1, dense_k=4,
                              max_elts_per_layer=per, nnz_frac=nnz, mult_range=(0.8, 1.2))
    layouts = art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP | (art.ART_LAYOUT_SPARSE if csr else 0)
    _check(w, layouts, np.random.default_rng(n_elt).permutation(LENGTHS), n_elt)


def test_dense_and_sparse_groups_in_one_call():
    """Groups of 32 ELTs each, every second one dense."""
    w = workloads.random_case(5, catalogue=2999, n_elt=96, n_layers=3, n_trials=1, dense_k=4, max_elts_per_layer=32,
                              nnz_frac=0.5, mult_range=(0.8, 1.2))
    p = w.portfolio
    p.layer_elt_off = np.array([0, 32, 64, 96], np.int32)
    p.layer_elt_ids = np.arange(96, dtype=np.int32)
    keep = np.random.default_rng(3).random((32, 2999)) < 0.04
    p.elt_losses[32:64] *= keep
    for layouts in (art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP,
                    art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP | art.ART_LAYOUT_SPARSE):
        _check(w, layouts, LENGTHS, 9)
