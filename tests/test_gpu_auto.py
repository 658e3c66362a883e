"""The default variant's choice between the passes over whole-number tables and
the sparse variant, and the payouts' between their table and the evaluation by
event: whichever is taken, by the host or on the device, the results are its own
in full, and the choice is near the better one in time. The bounds on time are
wide (a choice gone wrong costs three to twenty times)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu

LAYOUTS = art.ART_LAYOUT_LAYER | art.ART_LAYOUT_SPARSE


def _case(n_layers, catalogue, nnz, seed=7):
    return workloads.random_case(seed, catalogue=catalogue, n_elt=24, n_layers=n_layers, n_trials=1, dense_k=4,
                                 max_elts_per_layer=8, nnz_frac=nnz)


def _yet(rng, catalogue, lengths, room):
    """A CSR YET on the device, its ids at the start of a buffer of `room` ids."""
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    ids = rng.integers(0, catalogue, size=int(off[-1]), dtype=np.int32)
    buf = torch.zeros(max(room, ids.size), dtype=torch.int32, device="cuda")
    buf[:ids.size].copy_(torch.from_numpy(ids))
    return ids, off, buf[:ids.size], torch.from_numpy(off).cuda()


@pytest.mark.parametrize("n_layers,catalogue,trials,k", [(20, 300_000, 3000, 6), (20, 300_000, 6000, 900),
                                                         (9, 2000, 700, 40), (70, 50_000, 2000, 300)])
@pytest.mark.parametrize("room", [0, 1 << 26])
def test_default_variant_runs_one_form_in_full(n_layers, catalogue, trials, k, room):
    w = _case(n_layers, catalogue, 0.02)
    rng = np.random.default_rng(k)
    ids, off, dev, doff = _yet(rng, catalogue, rng.integers(0, 2 * k, trials), room)
    got = {}
    for name in ("AUTO", "SKIP", "SPARSE", "GRAPH"):
        variant = art.ART_VARIANT_AUTO if name == "GRAPH" else getattr(art, "ART_VARIANT_" + name)
        p = art.portfolio_from_workload(w, layouts=LAYOUTS, variant=variant, flags=art.ART_FLAG_GRAPH if name == "GRAPH" else 0)
        try:
            y = torch.full((n_layers, trials), -1.0, dtype=torch.float64, device="cuda")
            br = torch.full((n_layers, trials), 9, dtype=torch.uint8, device="cuda")
            for _ in range(2):
                art.art_run_ylt(p, trials, dev, doff, 0, y, br)
            assert art.art_get_device_status(p) == art.ART_OK
            got[name] = y.cpu().numpy(), br.cpu().numpy()
        finally:
            p.close()
    for name in ("AUTO", "GRAPH"):
        assert any(np.array_equal(got[name][0], got[f][0]) and np.array_equal(got[name][1], got[f][1])
                   for f in ("SKIP", "SPARSE"))


@pytest.mark.parametrize("trials,k", [(500, 7), (4000, 30), (3000, 400)])
@pytest.mark.parametrize("room", [0, 1 << 26])
def test_payouts_run_one_form_in_full(trials, k, room):
    catalogue = 150_000
    w = _case(2, catalogue, 0.05)
    rng = np.random.default_rng(k)
    lengths = rng.integers(0, 2 * k, trials)
    ids, off, dev, doff = _yet(rng, catalogue, lengths, room)
    w.yet = workloads.YET(n_trials=trials, event_ids=ids, trial_off=off)
    ref, gross, _ = oracle.ylt(w.oracle_problem())
    p = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER)
    try:
        pay = torch.full((ids.size,), -7.0, dtype=torch.float64, device="cuda")
        ex = torch.full((trials,), -9, dtype=torch.int32, device="cuda")
        y = torch.full((trials,), -1.0, dtype=torch.float64, device="cuda")
        art.art_run_payouts(p, 1, trials, dev, doff, 0, pay, ex, y)
        assert art.art_get_device_status(p) == art.ART_OK
        tol = 1e-6 * gross[1] + 1e-9  # FP32 occurrence losses against the FP64 oracle, as everywhere
        assert np.all(np.abs(y.cpu().numpy() - ref[1]) <= tol)
        sums = np.add.reduceat(np.append(pay.cpu().numpy(), 0.0), off[:-1].clip(max=ids.size))
        sums[lengths == 0] = 0.0
        assert np.all(np.abs(sums - ref[1]) <= 2 * tol)
        assert torch.all(pay >= 0) and torch.all(ex >= -1) and np.all(ex.cpu().numpy() < np.maximum(lengths, 1))
    finally:
        p.close()


def _time_us(f, reps=5):
    for _ in range(3):
        f()
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            f()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 1e3 / reps)
    return min(times)


@pytest.mark.parametrize("n_layers,nnz,trials,k", [(64, 0.02, 20_000, 10), (64, 0.02, 200_000, 12), (64, 0.02, 50_000, 600),
                                                   (400, 1e-4, 20_000, 600), (16, 1e-4, 50_000, 600)])
@pytest.mark.parametrize("room", [0, 1 << 26])
def test_default_variant_is_near_the_faster_form(n_layers, nnz, trials, k, room):
    catalogue = 1_000_000
    w = _case(n_layers, catalogue, nnz)
    rng = np.random.default_rng(k)
    _, off, dev, doff = _yet(rng, catalogue, rng.integers(k // 2, 2 * k, trials), room)
    p = art.portfolio_from_workload(w, layouts=LAYOUTS)
    try:
        y = torch.empty((n_layers, trials), dtype=torch.float64, device="cuda")
        t = {}
        for v in ("SKIP", "SPARSE", "AUTO"):
            art.art_set_variant(p, getattr(art, "ART_VARIANT_" + v))
            t[v] = _time_us(lambda: art.art_run_ylt(p, trials, dev, doff, 0, y))
        # half as long again, and a few microseconds per empty launch of the form not taken
        assert t["AUTO"] <= 1.5 * min(t["SKIP"], t["SPARSE"]) + 20.0 + 5.0 * ((n_layers + 7) // 8), t
    finally:
        p.close()


def test_payouts_of_a_few_long_trials():
    """One warp per trial: evaluated event by event one trial of 400,000 events
    takes about 19 ms, over the table of whole losses about 2."""
    w = _case(1, 1_000_000, 0.02)
    ids = torch.from_numpy(np.random.default_rng(2).integers(0, 1_000_000, 400_000, dtype=np.int32)).cuda()
    p = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER)
    try:
        pay = torch.empty(400_000, dtype=torch.float64, device="cuda")
        assert _time_us(lambda: art.art_run_payouts(p, 0, 1, ids, None, 400_000, pay)) <= 8000.0
    finally:
        p.close()
