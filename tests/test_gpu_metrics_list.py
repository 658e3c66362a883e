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
