"""What the library keeps between calls is bounded and comes back: by
art_release_scratch where no portfolio ever lived, and with the last portfolio."""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _metrics(y):
    L, n = y.shape
    out = [torch.empty(s, dtype=torch.float64, device="cuda") for s in (L, (L, 1), (L, 1))]
    art.art_metrics(y, n, L, [0.99], *out)


def test_release_scratch_after_metrics_only():
    y = torch.rand((64, 1_000_000), dtype=torch.float64, device="cuda")
    _metrics(y[:1])  # module loading is not scratch
    art.art_release_scratch()
    before = _free()
    for _ in range(3):
        _metrics(y)  # 64 lists of 125,000 places: 64 MB
    kept = before - _free()
    assert 32 << 20 <= kept <= 300 << 20
    art.art_release_scratch()
    assert before - _free() <= 4 << 20
    _metrics(y)  # and it is taken again when needed
    art.art_release_scratch()


def test_last_portfolio_gives_scratch_back():
    y = torch.rand((64, 1_000_000), dtype=torch.float64, device="cuda")
    w = workloads.random_case(3, catalogue=100, n_elt=3, n_layers=1, n_trials=8, dense_k=4, max_elts_per_layer=3)
    _metrics(y[:1])
    art.art_release_scratch()
    art.portfolio_from_workload(w).close()
    torch.cuda.empty_cache()
    before = _free()
    p, q = art.portfolio_from_workload(w), art.portfolio_from_workload(w)
    torch.cuda.empty_cache()
    _metrics(y)
    torch.cuda.synchronize()
    p.close()
    assert before - _free() >= 32 << 20  # another portfolio lives
    q.close()
    assert before - _free() <= 8 << 20
