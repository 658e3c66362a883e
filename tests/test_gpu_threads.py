"""Calls from several host threads at once, each on its own stream: sizes that
differ from thread to thread, so that no thread's launch depends on a limit that
another sets."""
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu


def _run_all(works):
    errors = []

    def guarded(f):
        try:
            f()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(repr(e))

    threads = [threading.Thread(target=guarded, args=(f,)) for f in works]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]


def test_metrics_of_different_lengths():
    def work(n, n_p):
        probs = [0.99, 0.9, 0.95, 0.97, 0.5, 0.8, 0.995, 0.75][:n_p]
        stream = torch.cuda.Stream()
        y = np.random.default_rng(n).lognormal(10.0, 1.0, (3, n))
        dev = torch.from_numpy(y).cuda()
        torch.cuda.synchronize()
        mean = torch.empty(3, dtype=torch.float64, device="cuda")
        pml = torch.empty((3, n_p), dtype=torch.float64, device="cuda")
        tvar = torch.empty((3, n_p), dtype=torch.float64, device="cuda")
        for _ in range(2000):
            art.art_metrics(dev, n, 3, probs, mean, pml, tvar, stream=stream)
        stream.synchronize()
        np.testing.assert_array_equal(pml.cpu().numpy(), oracle.metrics(y, probs)[1])

    # rows that fit shared memory (of several sizes), lists, and the general path with 5 to 8 probabilities
    _run_all([lambda n=n, q=q: work(n, q) for n, q in [(50, 1), (1000, 1), (26_000, 2), (60_000, 1), (60_001, 7), (60_002, 8)]])


def test_portfolios_of_different_catalogues():
    def work(catalogue):
        stream = torch.cuda.Stream()
        w = workloads.random_case(catalogue, catalogue=catalogue, n_elt=8, n_layers=2, n_trials=64, dense_k=256,
                                  max_elts_per_layer=4, nnz_frac=0.1)
        p = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER | art.ART_LAYOUT_OCC64)
        ids = torch.from_numpy(np.ascontiguousarray(w.yet.event_ids)).cuda()
        y = torch.empty((2, 64), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ref, gross, _ = oracle.ylt(w.oracle_problem())
        for variant in (art.ART_VARIANT_SKIP, art.ART_VARIANT_FP64):
            art.art_set_variant(p, variant)
            for _ in range(1000):
                art.art_run_ylt(p, 64, ids, None, 256, y, stream=stream)
            stream.synchronize()
            assert np.all(np.abs(y.cpu().numpy() - ref) <= 1e-6 * gross + 1e-9)
        p.close()

    _run_all([lambda c=c: work(c) for c in (100, 20_000, 300_000, 1_200_000)])
