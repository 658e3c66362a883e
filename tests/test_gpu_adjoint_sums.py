"""The adjoint's column sums over many short trials: each trial's FP32 partials
go into the compensated pair, so the error does not grow with the trials."""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_trials,k", [(8_000_000, 1), (2_000_000, 5)])
def test_many_short_trials(n_trials, k):
    C, E, g = 64, 3, 0.75
    rng = np.random.default_rng(k)
    losses = rng.uniform(1e5, 1e6, (E, C)).astype(np.float32)
    losses[:, ::4] = 0.0
    ids = rng.integers(0, C, n_trials * k, dtype=np.int32)
    one, inf = np.ones(E, np.float32), np.full(E, np.inf, np.float32)
    # every loss is on its middle branch, as is every trial with a loss
    p = art.art_create_portfolio(C, torch.from_numpy(losses).cuda(), one, 0 * one, inf, [0, E], np.arange(E),
                                 [[1.0, 1e9, 0.5, 1e12]], layouts=art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP,
                                 variant=art.ART_VARIANT_SKIP)
    try:
        dev = torch.from_numpy(ids).cuda()
        y = torch.empty((1, n_trials), dtype=torch.float64, device="cuda")
        br = torch.empty((1, n_trials), dtype=torch.uint8, device="cuda")
        art.art_run_ylt(p, n_trials, dev, None, k, y, br)
        gt = torch.empty((1, 4), dtype=torch.float64, device="cuda")
        gm = torch.empty(E, dtype=torch.float64, device="cuda")
        w = torch.full((1, n_trials), g, dtype=torch.float64, device="cuda")
        art.art_run_ylt_backward(p, n_trials, dev, None, k, br, w, gt, gm)
        assert art.art_get_device_status(p) == art.ART_OK
        want = g * losses.astype(np.float64) @ np.bincount(ids, minlength=C)
        # g is exact in FP32; a term's product rounds once (2^-24), as does a lane's sum of a
        # second event; the fold over the lanes rounds at most five times, each at random over
        # millions of trials: 2^-24 and as much again for what does not cancel
        np.testing.assert_allclose(gm.cpu().numpy(), want, rtol=2.0 ** -23)
    finally:
        p.close()
