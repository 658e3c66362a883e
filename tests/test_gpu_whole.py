"""The passes over occurrence tables of whole numbers (skip variant, payouts):
sums are exact, so the YLT equals the FP64 sum of the FP32 occurrence losses
(every partial sum is a multiple of one unit below 2^53) bit for bit, at the
edges of chunks, vectors, layers per group and alignments of the id array."""
import numpy as np
import pytest
import torch

from paper_1308_2572_gb300 import art, workloads

pytestmark = pytest.mark.gpu

# around a warp's vector (4), a half chunk (128) and a chunk (256) of ids
LENGTHS = [0, 1, 3, 4, 5, 31, 127, 128, 129, 252, 255, 256, 257, 260, 511, 513, 1000, 2049]


def _case(n_layers, catalogue, seed=5, unlimited=False):
    rng = np.random.default_rng(seed)
    w = workloads.random_case(seed, catalogue=catalogue, n_elt=12, n_layers=n_layers, n_trials=1, dense_k=4,
                              max_elts_per_layer=6, nnz_frac=0.2)
    p = w.portfolio
    if unlimited:
        p.occ_lim[0] = np.inf
        p.elt_lim[:] = np.inf  # nothing bounds the first layer's losses: its group keeps FP32 tables
    return w, rng


def _occ_losses(p):
    """o[j][i] in FP32 as the library forms them (m = 1), widened to FP64."""
    out = np.zeros((p.n_layers, p.catalogue_size))
    for j in range(p.n_layers):
        x = np.zeros(p.catalogue_size, np.float32)
        for e in p.layer_elt_ids[p.layer_elt_off[j]:p.layer_elt_off[j + 1]]:
            f = np.minimum(np.maximum(p.elt_losses[e] - p.elt_ded[e], np.float32(0)), p.elt_lim[e])
            x = x + f.astype(np.float32)
        o = np.minimum(np.maximum(x - np.float32(p.occ_ret[j]), np.float32(0)), np.float32(p.occ_lim[j]))
        out[j] = o.astype(np.float64)
    return out


def _yet(rng, catalogue, lengths, shift):
    """A ragged YET whose id array starts `shift` ids past a 16-byte boundary."""
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    ids = rng.integers(0, catalogue, size=int(off[-1]), dtype=np.int32)
    buf = torch.zeros(ids.size + 8, dtype=torch.int32, device="cuda")
    dev = buf[shift:shift + ids.size]
    dev.copy_(torch.from_numpy(ids))
    return ids, off, dev, torch.from_numpy(off).cuda()


def _expected(o, p, ids, off):
    s = np.stack([np.add.reduceat(np.append(o[j][ids], 0.0), off[:-1].clip(max=max(0, ids.size))) for j in range(len(o))])
    s[:, np.diff(off) == 0] = 0.0
    return np.minimum(np.maximum(s - p.agg_ret[:, None], 0.0), p.agg_lim[:, None])


# catalogues whose bitmap fits, folds once and needs more than one fold
@pytest.mark.parametrize("n_layers,catalogue", [(1, 97), (2, 5000), (3, 5000), (8, 97), (9, 5000), (17, 5000),
                                                (1, 1_999_999), (8, 1_999_999), (1, 4_000_037), (3, 4_000_037)])
def test_skip_sums_are_exact(n_layers, catalogue):
    w, rng = _case(n_layers, catalogue)
    p = w.portfolio
    o = _occ_losses(p)
    lengths = np.array(LENGTHS * 4 + [1000] * 90)
    rng.shuffle(lengths)
    port = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER, variant=art.ART_VARIANT_SKIP)
    try:
        for shift in range(4):
            ids, off, dev, doff = _yet(rng, catalogue, lengths, shift)
            want = _expected(o, p, ids, off)
            y = torch.full((n_layers, lengths.size), -1.0, dtype=torch.float64, device="cuda")
            br = torch.full((n_layers, lengths.size), 9, dtype=torch.uint8, device="cuda")
            art.art_run_ylt(port, lengths.size, dev, doff, 0, y, br)
            assert art.art_get_device_status(port) == art.ART_OK
            np.testing.assert_array_equal(y.cpu().numpy(), want)
            s = want + 0.0
            b = br.cpu().numpy()
            assert np.all(b[s == 0] == 0) and np.all((b == 1) == ((s > 0) & (s < p.agg_lim[:, None])))
        for k in (1, 4, 6, 256, 1000):  # dense
            t = 61
            ids = rng.integers(0, catalogue, size=t * k, dtype=np.int32)
            y = torch.full((n_layers, t), -1.0, dtype=torch.float64, device="cuda")
            art.art_run_ylt(port, t, torch.from_numpy(ids).cuda(), None, k, y)
            np.testing.assert_array_equal(y.cpu().numpy(), _expected(o, p, ids, np.arange(t + 1) * k))
        # ids outside the catalogue count as no loss and are reported
        ids, off, dev, doff = _yet(rng, catalogue, lengths, 1)
        bad = ids.copy()
        bad[::97] = np.where(np.arange(bad[::97].size) % 2 == 0, catalogue, -5)
        dev.copy_(torch.from_numpy(bad))
        art.art_run_ylt(port, lengths.size, dev, doff, 0, torch.empty((n_layers, lengths.size), dtype=torch.float64, device="cuda"))
        assert art.art_get_device_status(port) == art.ART_EID_RANGE
    finally:
        port.close()


@pytest.mark.parametrize("n_layers", [1, 8])
def test_long_trials(n_layers):
    """Trials of more than 2^20 events: the lanes' counts outgrow the short
    reduction."""
    w, rng = _case(n_layers, 97, seed=41)
    p = w.portfolio
    p.agg_ret[:] *= 1e4
    p.agg_lim[:] *= 1e5
    o = _occ_losses(p)
    k = (1 << 20) + 1237
    ids = rng.integers(0, 97, size=3 * k, dtype=np.int32)
    port = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER, variant=art.ART_VARIANT_SKIP)
    try:
        y = torch.empty((n_layers, 3), dtype=torch.float64, device="cuda")
        art.art_run_ylt(port, 3, torch.from_numpy(ids).cuda(), None, k, y)
        # the FP64 sum of whole numbers of one unit: exact below 2^53 units
        np.testing.assert_array_equal(y.cpu().numpy(), _expected(o, p, ids, np.arange(4) * k))
    finally:
        port.close()


@pytest.mark.parametrize("variant", ["ART_VARIANT_SKIP", "ART_VARIANT_FP64", "ART_VARIANT_AUTO"])
def test_captured_call_takes_new_occurrence_terms(variant):
    """A call captured by the caller and replayed after art_update_terms builds
    its tables from the terms as they are then, whatever their units."""
    w, rng = _case(17, 5000, seed=3)
    p = w.portfolio
    ids = torch.from_numpy(rng.integers(0, 5000, size=400 * 100, dtype=np.int32)).cuda()
    port = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER | art.ART_LAYOUT_SPARSE | art.ART_LAYOUT_OCC64,
                                       variant=getattr(art, variant))
    try:
        y = torch.zeros((17, 400), dtype=torch.float64, device="cuda")
        want = torch.zeros_like(y)
        art.art_run_ylt(port, 400, ids, None, 100, y)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            art.art_run_ylt(port, 400, ids, None, 100, y)
        m, d, l, t = art.art_get_terms(port)
        t2 = t.copy()
        t2[:, 0] *= 37.0
        t2[:, 1] = np.where(np.arange(17) % 2 == 0, t[:, 1] * 900.0, np.inf)
        for terms in (t, t2, t):
            art.art_update_terms(port, terms=terms)
            y.fill_(-1.0)
            g.replay()
            art.art_run_ylt(port, 400, ids, None, 100, want)
            torch.cuda.synchronize()
            np.testing.assert_allclose(y.cpu().numpy(), want.cpu().numpy(), rtol=1e-11, atol=1e-9)
    finally:
        port.close()


def test_unbounded_losses_keep_the_fp32_tables():
    """A group with a layer whose losses are not bounded takes the compensated
    pass; the other groups' results stay exact."""
    w, rng = _case(9, 5000, unlimited=True)
    p = w.portfolio
    o = _occ_losses(p)
    lengths = np.array(LENGTHS * 3)
    ids, off, dev, doff = _yet(rng, 5000, lengths, 3)
    port = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER, variant=art.ART_VARIANT_SKIP)
    try:
        y = torch.empty((9, lengths.size), dtype=torch.float64, device="cuda")
        art.art_run_ylt(port, lengths.size, dev, doff, 0, y)
        want = _expected(o, p, ids, off)
        got = y.cpu().numpy()
        np.testing.assert_array_equal(got[8], want[8])
        # the compensated sums: an error of order n u^2 of the sum
        np.testing.assert_allclose(got, want, rtol=1e-11, atol=1e-11 * float(o.max()))
    finally:
        port.close()


@pytest.mark.parametrize("n_layers,catalogue,csr", [(1, 97, True), (2, 5000, True), (3, 5000, False), (4, 1_999_999, True),
                                                    (5, 5000, True), (17, 5000, True), (17, 97, False)])
def test_all_fp64_rounds_once(n_layers, catalogue, csr):
    """The all-FP64 variant over whole-number tables: the exact sum of the
    FP64 occurrence losses, rounded once, then the aggregate terms."""
    import math
    w, rng = _case(n_layers, catalogue, seed=23)
    p = w.portfolio
    o = np.zeros((n_layers, catalogue))
    for j in range(n_layers):
        x = np.zeros(catalogue)
        for e in p.layer_elt_ids[p.layer_elt_off[j]:p.layer_elt_off[j + 1]]:
            x += np.minimum(np.maximum(p.elt_losses[e].astype(np.float64) - float(p.elt_ded[e]), 0.0), float(p.elt_lim[e]))
        o[j] = np.minimum(np.maximum(x - p.occ_ret[j], 0.0), p.occ_lim[j])
    lengths = np.array(LENGTHS * 2 + [300] * 40)
    rng.shuffle(lengths)
    layouts = art.ART_LAYOUT_LAYER | art.ART_LAYOUT_OCC64 | (art.ART_LAYOUT_SPARSE if csr else 0)
    port = art.portfolio_from_workload(w, layouts=layouts, variant=art.ART_VARIANT_FP64)
    try:
        for shift in (0, 3):
            ids, off, dev, doff = _yet(rng, catalogue, lengths, shift)
            y = torch.full((n_layers, lengths.size), -1.0, dtype=torch.float64, device="cuda")
            art.art_run_ylt(port, lengths.size, dev, doff, 0, y)
            assert art.art_get_device_status(port) == art.ART_OK
            s = np.array([[math.fsum(o[j][ids[off[t]:off[t + 1]]]) for t in range(lengths.size)] for j in range(n_layers)])
            want = np.minimum(np.maximum(s - p.agg_ret[:, None], 0.0), p.agg_lim[:, None])
            np.testing.assert_array_equal(y.cpu().numpy(), want)
    finally:
        port.close()


@pytest.mark.parametrize("catalogue", [97, 1_999_999])
def test_payouts_are_exact(catalogue):
    w, rng = _case(2, catalogue, seed=11)
    p = w.portfolio
    o = _occ_losses(p)
    lengths = np.array(LENGTHS * 4 + [1000] * (1100 if catalogue > 1000 else 60))
    rng.shuffle(lengths)
    port = art.portfolio_from_workload(w, layouts=art.ART_LAYOUT_LAYER)
    try:
        for j, shift, pshift in [(0, 0, 0), (1, 1, 1), (0, 3, 0), (1, 2, 3)]:
            ids, off, dev, doff = _yet(rng, catalogue, lengths, shift)
            buf = torch.full((ids.size + 8,), -7.0, dtype=torch.float64, device="cuda")
            pay = buf[pshift:pshift + ids.size]
            ex = torch.full((lengths.size,), -9, dtype=torch.int32, device="cuda")
            y = torch.full((lengths.size,), -1.0, dtype=torch.float64, device="cuda")
            art.art_run_payouts(port, j, lengths.size, dev, doff, 0, pay, ex, y)
            assert art.art_get_device_status(port) == art.ART_OK
            np.testing.assert_array_equal(y.cpu().numpy(), _expected(o[j:j + 1], _Layer(p, j), ids, off)[0])
            got, exh = pay.cpu().numpy(), ex.cpu().numpy()
            assert torch.all(buf[:pshift] == -7.0) and torch.all(buf[pshift + ids.size:] == -7.0)
            for t in range(lengths.size):
                c = np.cumsum(o[j][ids[off[t]:off[t + 1]]])
                a = np.minimum(np.maximum(c - p.agg_ret[j], 0.0), p.agg_lim[j])
                full = np.nonzero(c - p.agg_ret[j] >= p.agg_lim[j])[0]
                assert exh[t] == (full[0] if full.size else -1)
                # a payout of the exact difference against one of rounded values: an ulp of each
                np.testing.assert_allclose(got[off[t]:off[t + 1]], np.diff(np.concatenate([[0.0], a])), rtol=0,
                                           atol=4e-16 * max(1.0, float(c[-1]) if c.size else 1.0))
    finally:
        port.close()


class _Layer:
    def __init__(self, p, j):
        self.agg_ret, self.agg_lim = p.agg_ret[j:j + 1], p.agg_lim[j:j + 1]


@pytest.mark.parametrize("n_elt,n_layers,per,nnz", [(3, 1, 3, 0.3), (8, 2, 8, 0.1), (16, 8, 8, 0.02), (16, 8, 16, 0.5),
                                                    (24, 5, 12, 0.2), (32, 4, 32, 0.3), (40, 9, 20, 0.1)])
def test_adjoint_records(n_elt, n_layers, per, nnz):
    """The group adjoint against the FP64 oracle at the edges of its records:
    one to 32 columns, events with up to three columns on their middle branch
    and with more (evaluated from their row), records from the CSR and from
    the table rows (the same bits), ragged trials of 0 to 2,049 events."""
    import oracle
    w = workloads.random_case(31 + n_elt, catalogue=3001, n_elt=n_elt, n_layers=n_layers, n_trials=1, dense_k=4,
                              max_elts_per_layer=per, nnz_frac=nnz, mult_range=(0.8, 1.2))
    rng = np.random.default_rng(n_elt)
    lengths = np.array(LENGTHS * 3 + [700] * 60)
    rng.shuffle(lengths)
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    ids = rng.integers(0, 3001, size=int(off[-1]), dtype=np.int32)
    w.yet = workloads.YET(n_trials=lengths.size, event_ids=ids, trial_off=off)
    s = oracle.ylt(w.oracle_problem(), want_sum=True)[2]
    w.portfolio.agg_ret[:] = np.median(s, axis=1) * 0.5 + 1.0
    w.portfolio.agg_lim[:] = np.median(s, axis=1) + 1.0
    g = rng.uniform(0.5, 1.5, size=(n_layers, lengths.size))
    ot, om, _, _ = oracle.grad(w.oracle_problem(), g)
    outs = []
    for layouts in (art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP,
                    art.ART_LAYOUT_LAYER | art.ART_LAYOUT_GROUP | art.ART_LAYOUT_SPARSE):
        p = art.portfolio_from_workload(w, layouts=layouts, variant=art.ART_VARIANT_SKIP)
        try:
            d_ids, d_off = torch.from_numpy(ids).cuda(), torch.from_numpy(off).cuda()
            y = torch.empty((n_layers, lengths.size), dtype=torch.float64, device="cuda")
            br = torch.empty((n_layers, lengths.size), dtype=torch.uint8, device="cuda")
            art.art_run_ylt(p, lengths.size, d_ids, d_off, 0, y, br)
            gt = torch.empty((n_layers, 4), dtype=torch.float64, device="cuda")
            gm = torch.empty(n_elt, dtype=torch.float64, device="cuda")
            art.art_run_ylt_backward(p, lengths.size, d_ids, d_off, 0, br, torch.from_numpy(g).cuda(), gt, gm)
            assert art.art_get_device_status(p) == art.ART_OK
            outs.append((gt.cpu().numpy(), gm.cpu().numpy()))
        finally:
            p.close()
    np.testing.assert_array_equal(outs[0][0], outs[1][0])
    np.testing.assert_array_equal(outs[0][1], outs[1][1])
    # weights and products are FP32 (2^-24 each), the sums compensated
    np.testing.assert_allclose(outs[1][0], ot, rtol=1e-6, atol=1e-6 * np.abs(ot).max())
    np.testing.assert_allclose(outs[1][1], om, rtol=2e-6, atol=1e-6 * np.abs(om).max())
