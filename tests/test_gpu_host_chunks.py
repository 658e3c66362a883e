"""Host buffers that go to the device in chunks of trials: every chunk takes
the tables that were built for the call, wherever the chunk's ids were staged
(a ragged chunk's id pointer is shifted back by its first index, so it may
point outside every allocation)."""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,layouts", [
    ("ART_VARIANT_SKIP", art.ART_LAYOUT_LAYER),
    ("ART_VARIANT_FP64", art.ART_LAYOUT_LAYER | art.ART_LAYOUT_OCC64),
    ("ART_VARIANT_AUTO", art.ART_LAYOUT_LAYER | art.ART_LAYOUT_SPARSE),
])
def test_ragged_chunks_equal_the_device_call(variant, layouts):
    n_layers, T = 9, 120_000  # two occurrence groups: staged; 180 million ids: eleven chunks
    w = workloads.random_case(5, catalogue=5000, n_elt=12, n_layers=n_layers, n_trials=1, dense_k=4,
                              max_elts_per_layer=6, nnz_frac=0.2)
    rng = np.random.default_rng(1)
    off = np.concatenate([[0], np.cumsum(rng.integers(1200, 1800, T))]).astype(np.int64)
    ids = rng.integers(0, 5000, int(off[-1]), dtype=np.int32)
    p = art.portfolio_from_workload(w, layouts=layouts, variant=getattr(art, variant))
    try:
        host = np.zeros((n_layers, T))
        art.art_run_ylt_host(p, T, ids, off, 0, host)
        dev = torch.zeros((n_layers, T), dtype=torch.float64, device="cuda")
        art.art_run_ylt(p, T, torch.from_numpy(ids).cuda(), torch.from_numpy(off).cuda(), 0, dev)
        np.testing.assert_array_equal(host, dev.cpu().numpy())  # the same whole-number sums
    finally:
        p.close()
