"""The one-read metrics (sample, pass, finish) against a full sort in FP64:
sizes around the rows that fit shared memory, distributions that make the
sample's threshold, the tie key and the lists go each way, misaligned rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1308_2572_gb300 import art

pytestmark = pytest.mark.gpu


def _rows(n, rng):
    ln = rng.lognormal(15.0, 2.0, n)
    rows = [ln, np.where(ln > np.median(ln), ln, 0.0),             # half the trials without a loss
            np.minimum(ln, np.quantile(ln, 0.7)),                  # capped in 30% of trials
            np.minimum(ln, np.quantile(ln, 0.9995)),               # capped in fewer than k
            np.full(n, 4.0e7), np.zeros(n),                        # constant
            np.where(np.arange(n) == n // 3, 1e300, ln),           # one loss far above any sample
            np.where(rng.random(n) < 0.002, ln, 0.0),              # fewer losses than k at 0.99
            np.floor(ln / 1e6) * 1e6,                              # heavy ties everywhere
            np.sort(ln), 1e-310 * rng.integers(0, 1000, n),        # ordered; subnormal
            np.where(rng.random(n) < 0.4, 3.0, np.where(rng.random(n) < 0.5, 2.0, 5.0))]  # the second value repeats
    return np.stack(rows)


@pytest.mark.parametrize("n", [1, 2, 33, 1000, 26624, 26625, 50_003, 300_001])
def test_metrics_match_a_full_sort(n):
    rng = np.random.default_rng(n)
    y = _rows(n, rng)
    dev = torch.from_numpy(y).cuda()
    for probs in ([0.99], [0.95, 0.999], [0.9, 0.99, 0.996], [0.5, 0.97]):
        L, n_p = y.shape[0], len(probs)
        om, op, ot = oracle.metrics(y, probs)
        outs = []
        for fn in (art.art_metrics, art.art_metrics_noalloc, art.art_metrics):
            mean = torch.full((L,), -1.0, dtype=torch.float64, device="cuda")
            pml = torch.full((L, n_p), -1.0, dtype=torch.float64, device="cuda")
            tvar = torch.full((L, n_p), -1.0, dtype=torch.float64, device="cuda")
            fn(dev, n, L, probs, mean, pml, tvar)
            outs.append([t.cpu().numpy() for t in (mean, pml, tvar)])
        for got in outs:
            np.testing.assert_array_equal(got[1], op)  # selected exactly
            # one or two roundings against the oracle's sequential FP64 sums
            np.testing.assert_allclose(got[0], om, rtol=1e-12, atol=1e-320)
            np.testing.assert_allclose(got[2], ot, rtol=1e-12, atol=1e-320)
        for a, b in zip(outs[0], outs[2]):
            np.testing.assert_array_equal(a, b)  # repeatable bits


@pytest.mark.parametrize("n", [26_625, 60_000, 300_001])
def test_losses_below_the_normal_range(n):
    """Losses whose high word is 0 (below 2^-1042), beside trials without a
    loss and beside ordinary ones: selected and summed as any other."""
    rng = np.random.default_rng(n)
    tiny = 5e-324 * rng.integers(1, 1 << 31, n)
    ln = rng.lognormal(15.0, 2.0, n)
    y = np.stack([np.where(np.arange(n) % 50 == 0, tiny, 0.0), np.where(rng.random(n) < 0.004, tiny, 0.0), tiny,
                  np.where(rng.random(n) < 0.3, ln, tiny), np.where(rng.random(n) < 0.001, ln, 0.0) + (np.arange(n) == 7) * 5e-324])
    dev = torch.from_numpy(y).cuda()
    for probs in ([0.99], [0.96, 0.999]):
        L, n_p = y.shape[0], len(probs)
        om, op, ot = oracle.metrics(y, probs)
        mean = torch.full((L,), -1.0, dtype=torch.float64, device="cuda")
        pml = torch.full((L, n_p), -1.0, dtype=torch.float64, device="cuda")
        tvar = torch.full((L, n_p), -1.0, dtype=torch.float64, device="cuda")
        art.art_metrics(dev, n, L, probs, mean, pml, tvar)
        np.testing.assert_array_equal(pml.cpu().numpy(), op)
        # the oracle's sums are exact here or round as above; a subnormal quotient rounds to its unit
        np.testing.assert_allclose(mean.cpu().numpy(), om, rtol=1e-12, atol=1e-323)
        np.testing.assert_allclose(tvar.cpu().numpy(), ot, rtol=1e-12, atol=1e-323)


def _atom_rows(n, rng):
    """Rows whose sample threshold falls on a value that repeats (a layer whose
    events mostly pay their full limit), with other values around it."""
    ln = rng.lognormal(15.0, 1.0, n)
    pick = rng.random(n)
    count = rng.poisson(0.2, n)
    rows = [5e6 * count, 5e6 * rng.poisson(0.6, n), 5e6 * rng.poisson(3.0, n), 5e6 * np.minimum(count, 2),
            5e6 * count + np.where(pick < 0.01, ln, 0.0),                      # losses between the multiples
            np.where(pick < 0.3, 7e6, ln),                                    # one atom inside the losses
            np.where(pick < 0.2, 7e6, np.where(pick < 0.4, 7e6 * (1 + 2.0 ** -40), 0.0)),  # two atoms in one bin
            np.where(pick < 0.2, 7e6, np.where(pick < 0.4, 7e6 * (1 + 2.0 ** -18), 0.0)),
            np.where(pick < 0.15, 7e6, np.where(pick < 0.16, ln, 0.0)),        # an atom and few others
            np.where(pick < 0.5, 7e6, 0.0) + (np.arange(n) == 5) * 1e7,        # the largest is no tie
            np.where(pick < 0.2, 1e-320, 0.0), np.where(pick < 0.2, 1e-320, ln)]  # subnormal atom
    return np.stack(rows)


@pytest.mark.parametrize("n", [12_288, 12_289, 26_625, 50_003, 300_001])
def test_repeating_values_at_the_threshold(n):
    rng = np.random.default_rng(n)
    y = _atom_rows(n, rng)
    dev = torch.from_numpy(y).cuda()
    for probs in ([0.99], [0.955], [0.99, 0.996, 0.999], [0.951, 0.98, 0.9999]):
        L, n_p = y.shape[0], len(probs)
        om, op, ot = oracle.metrics(y, probs)
        for fn in (art.art_metrics, art.art_metrics_noalloc):
            mean = torch.full((L,), -1.0, dtype=torch.float64, device="cuda")
            pml = torch.full((L, n_p), -1.0, dtype=torch.float64, device="cuda")
            tvar = torch.full((L, n_p), -1.0, dtype=torch.float64, device="cuda")
            fn(dev, n, L, probs, mean, pml, tvar)
            np.testing.assert_array_equal(pml.cpu().numpy(), op)
            # one or two roundings against the oracle's sequential FP64 sums; subnormal units
            np.testing.assert_allclose(mean.cpu().numpy(), om, rtol=1e-12, atol=1e-323)
            np.testing.assert_allclose(tvar.cpu().numpy(), ot, rtol=1e-12, atol=1e-323)


def test_repeating_values_take_no_longer():
    """Full limits only (0, 1, 2, ... times one), where the list would overflow,
    against losses that do not repeat; and few layers of long lists against
    ranks that no list serves. Wide bounds: a wrong form takes 3 to 60 times."""
    def time_us(y, probs):
        L, n = y.shape
        out = [torch.empty(s, dtype=torch.float64, device="cuda") for s in (L, (L, len(probs)), (L, len(probs)))]
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            art.art_metrics(y, n, L, probs, *out)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return min(times)

    g = torch.Generator(device="cuda").manual_seed(3)
    for L, n in [(1, 1_000_000), (64, 300_000)]:
        plain = torch.exp(15.0 + torch.randn((L, n), generator=g, device="cuda")).double()
        atoms = torch.poisson(torch.full((L, n), 0.2, device="cuda"), generator=g).double() * 5e6
        probs = [0.99, 0.996, 0.999]
        assert time_us(atoms, probs) <= 4.0 * time_us(plain, probs)
    long = torch.exp(15.0 + torch.randn((1, 30_000_000), generator=g, device="cuda")).double()
    probs = [0.951, 0.97, 0.99]
    assert time_us(long, probs) <= 2.5 * time_us(long, [0.9] + probs[1:])
