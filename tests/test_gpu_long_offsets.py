"""A CSR trial of more events than the passes' 32-bit positions hold counts as
empty and is reported; its neighbours are not affected. (No id of such a trial
is read, so the id array need not hold it.)"""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,layouts,n_layers", [
    (art.ART_VARIANT_SKIP, art.ART_LAYOUT_LAYER, 1), (art.ART_VARIANT_SKIP, art.ART_LAYOUT_LAYER, 5),
    (art.ART_VARIANT_FP64, art.ART_LAYOUT_LAYER | art.ART_LAYOUT_OCC64, 3)])
@pytest.mark.parametrize("length", [0xfffff001, 0xffffffff, 1 << 32, (1 << 32) + 5, 1 << 40])
def test_trial_longer_than_the_positions(variant, layouts, n_layers, length):
    w = workloads.random_case(4, catalogue=500, n_elt=8, n_layers=n_layers, n_trials=1, dense_k=4, max_elts_per_layer=4,
                              nnz_frac=0.5)
    # covers of 50 times their retention: whole-number tables, and so the passes
    # that hold positions in 32 bits (the others would read the ids)
    w.portfolio.occ_ret[:], w.portfolio.occ_lim[:] = 1e5, 5e6
    ids = torch.from_numpy(np.random.default_rng(1).integers(0, 500, 64, dtype=np.int32)).cuda()
    p = art.portfolio_from_workload(w, layouts=layouts, variant=variant)
    try:
        want = torch.zeros((n_layers, 2), dtype=torch.float64, device="cuda")
        art.art_run_ylt(p, 2, ids, torch.tensor([0, 10, 33], dtype=torch.int64, device="cuda"), 0, want)
        assert art.art_get_device_status(p) == art.ART_OK
        off = torch.tensor([0, 10, 33, 33 + length, 33 + length], dtype=torch.int64, device="cuda")
        y = torch.full((n_layers, 4), -1.0, dtype=torch.float64, device="cuda")
        art.art_run_ylt(p, 4, ids, off, 0, y)
        assert art.art_get_device_status(p) == art.ART_EINVAL
        np.testing.assert_array_equal(y[:, :2].cpu().numpy(), want.cpu().numpy())
        assert torch.all(y[:, 2:] == 0.0)
    finally:
        p.close()
