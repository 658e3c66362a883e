"""Calls that find no room for their tables take the forms that need less: the
group adjoint 8 bytes per catalogue event instead of 32, the payouts none."""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art

pytestmark = pytest.mark.gpu


def _fill(leave):
    """Tensors that take the device's free memory but for about `leave` bytes."""
    held = []
    for step in (1 << 32, 1 << 28, 1 << 25):
        while True:
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            n = (free - leave) // step
            if n <= 0:
                break
            held.append(torch.empty(n * step, dtype=torch.uint8, device="cuda"))
    return held


def test_adjoint_and_payouts_without_room():
    C, T, K = 100_000_000, 500, 400
    g = torch.Generator(device="cuda").manual_seed(1)
    losses = torch.zeros((2, C), dtype=torch.float32, device="cuda")
    at = torch.randint(0, C, (C // 10,), generator=g, device="cuda")
    losses[0, at] = 1e5 + 1e6 * torch.rand(at.numel(), generator=g, device="cuda")
    losses[1, at[::2]] = 2e5
    one, inf = np.ones(2, np.float32), np.full(2, np.inf, np.float32)
    p = art.art_create_portfolio(C, losses, one, 0 * one, inf, [0, 2], [0, 1], [[1e5, 5e6, 1e6, 2.4e8]],
                                 layouts=art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP, variant=art.ART_VARIANT_SKIP)
    held = []
    try:
        del losses
        ids = at[torch.randint(0, at.numel(), (T * K,), generator=g, device="cuda")].int()
        del at
        y = torch.empty((1, T), dtype=torch.float64, device="cuda")
        br = torch.empty((1, T), dtype=torch.uint8, device="cuda")
        w = torch.rand((1, T), generator=g, device="cuda", dtype=torch.float64)
        gt, gm = torch.empty((1, 4), dtype=torch.float64, device="cuda"), torch.empty(2, dtype=torch.float64, device="cuda")
        long = ids.repeat(100)  # 20,000,000 events: the table of whole losses pays
        pay = torch.empty(long.numel(), dtype=torch.float64, device="cuda")
        ex = torch.empty(100 * T, dtype=torch.int32, device="cuda")
        yl = torch.empty(100 * T, dtype=torch.float64, device="cuda")
        art.art_run_ylt(p, T, ids, None, K, y, br)

        def run():
            art.art_run_ylt_backward(p, T, ids, None, K, br, w, gt, gm)
            return gt.cpu().numpy().copy(), gm.cpu().numpy().copy()

        def payouts():
            art.art_run_payouts(p, 0, 100 * T, long, None, K, pay, ex, yl)
            assert art.art_get_device_status(p) == art.ART_OK
            return yl.cpu().numpy().copy(), ex.cpu().numpy().copy()

        want, want_pay = run(), payouts()
        assert np.abs(want[1]).min() > 0 and want_pay[0].max() > 0
        torch.cuda.empty_cache()
        art.art_release_scratch()
        held = _fill(1600 << 20)  # 3.2 GB of records do not fit, 0.8 GB of masks do
        got = run()
        # the terms' counts and sums are formed alike; columns round in another order (FP32 terms)
        np.testing.assert_allclose(got[0], want[0], rtol=1e-6)
        np.testing.assert_allclose(got[1], want[1], rtol=1e-6)
        art.art_release_scratch()
        held += _fill(250 << 20)  # nor do 400 MB of whole losses
        got_pay = payouts()
        np.testing.assert_allclose(got_pay[0], want_pay[0], rtol=1e-12, atol=1e-4)
        assert np.mean(got_pay[1] != want_pay[1]) < 1e-3  # an exact tie at the limit may round
    finally:
        held.clear()
        torch.cuda.empty_cache()
        p.close()
        art.art_release_scratch()
