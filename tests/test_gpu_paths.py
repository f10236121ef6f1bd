"""The forms a call can take, at the sizes where each begins and ends: against the
general form (bit-identical where both run the same arithmetic), the oracle or
numpy in 64 bits.  Tolerances are those of the neighbouring tests (rho 1e-4 of
max(rho, 1); an FP32 transform 4e-7 log2 N ||x||)."""
import threading

import numpy as np
import pytest

import oracle
import workloads
from mfgb_testutil import RHO_TOL, oracle_rho_series, oracle_segment, gpu_rho_series, rho_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_4175_gb300 import build
    build.build()
    import paper_0906_4175_gb300 as m
    oracle.build()
    return m


def _segment(mf, lg, fs=4096.0, seed=5):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = 70.0 * torch.randn(1 << lg, dtype=torch.float32, device="cuda", generator=g)   # loudest rho about 4 .. 7
    return mf.Segment(x, fs)


def _run(mf, bank, segs, thr, cap=1 << 20):
    out = [x.cpu().numpy().copy() for x in mf.filter_bank(bank, segs, thr, trig_cap=cap)]
    return out[0].view(np.uint8), out[1][:min(int(out[2][0]), cap)].view(np.uint8), int(out[2][0])


def _masses(n, seed=1):
    m = np.random.default_rng(seed).uniform(1.0, 6.0, (n, 2))
    return m[:, 0].copy(), m[:, 1].copy()


# rows per warp (row lengths 128, 256, 512) and the deferred peaks of every row
# length, whose rule is 2^26 samples in a batch: one template below and above it
@pytest.mark.parametrize("lg,n", [(13, 3), (14, 5), (15, 33), (16, 1), (16, 1025), (17, 7), (18, 255), (18, 257),
                                  (19, 129), (20, 63), (20, 65), (21, 33), (22, 17)])
def test_rows_and_tiles_agree(mf, monkeypatch, lg, n):
    bank, seg = mf.Bank(*_masses(n)), _segment(mf, lg)
    monkeypatch.setenv("MFGB_SPLIT_ALT", "0")
    a = _run(mf, bank, [seg], 4.75)
    monkeypatch.setenv("MFGB_P2ROWS", "0")
    b = _run(mf, bank, [seg], 4.75)
    assert bank.check() == 0 and a[2] == b[2]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def test_rows_of_the_1024_by_512_split(mf, monkeypatch):
    bank, seg = mf.Bank(*_masses(130)), _segment(mf, 19)
    monkeypatch.setenv("MFGB_SPLIT_ALT", "1")
    a = _run(mf, bank, [seg], 4.75)
    monkeypatch.setenv("MFGB_P2ROWS", "0")
    b = _run(mf, bank, [seg], 4.75)
    assert a[2] == b[2] and np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


# the units and anchors of a small bank in one launch (stage profiling keeps the
# two launches), below and above the limit of eight blocks per SM
@pytest.mark.parametrize("lg,n", [(10, 3), (13, 75), (16, 16), (16, 1300), (20, 5)])
def test_merged_units_and_anchors(mf, lg, n):
    bank, seg = mf.Bank(*_masses(n)), _segment(mf, lg)
    a = _run(mf, bank, [seg, seg], 4.5)
    bank.profile(True)
    b = _run(mf, bank, [seg, seg], 4.5)
    bank.profile(False)
    assert a[2] == b[2] and np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


# every sample a trigger: up to 16384 records by rank, then tiles of 4096
@pytest.mark.parametrize("lg,n,segs", [(10, 1, 1), (10, 8, 1), (10, 4, 2), (10, 9, 1), (11, 5, 3), (14, 9, 2),
                                       (10, 16, 1), (10, 17, 1)])
def test_trigger_order(mf, lg, n, segs):
    N = 1 << lg
    bank = mf.Bank(*_masses(n))
    ss = [_segment(mf, lg, seed=7 + i) for i in range(segs)]
    _, trig, nt = mf.filter_bank(bank, ss, 0.0, trig_cap=n * segs * N)
    assert bank.check() == 0
    t = mf.triggers_to_numpy(trig, nt)
    assert t.size == n * segs * N
    i = np.arange(t.size)
    assert np.array_equal(t["tmpl"], i // (segs * N)) and np.array_equal(t["seg"], i // N % segs)
    assert np.array_equal(t["j"], i % N)
    for s in range(segs):   # the records travelled with their keys
        one = mf.triggers_to_numpy(*mf.filter_bank(bank, [ss[s]], 0.0, trig_cap=n * N)[1:])
        assert np.array_equal(t["rho"].reshape(n, segs, N)[:, s].ravel(), one["rho"])
        assert np.array_equal(t["z_im"].reshape(n, segs, N)[:, s].ravel(), one["z_im"])


# short segments share launches (16 at most, four waves of tiles): as each alone,
# with longer segments between them, one wave of tiles and one tile more, and
# trigger keys of more than 32 bits
@pytest.mark.parametrize("lgs,n,thr", [((10, 11, 12, 13, 14, 15, 16), 3, 4.0), ((12, 13, 13, 14), 75, 4.5),
                                       ((13, 17, 10, 20, 16), 5, 4.5), ((13, 13), 304, 4.75), ((13, 13), 305, 4.75),
                                       ((16, 16, 15), 38, 4.75), ((14,) * 9, 152, 4.75), ((10,) * 33, 2, 3.5),
                                       ((20,) + (10,) * 1024, 3, 4.0)])
def test_short_segments_together(mf, lgs, n, thr):
    bank = mf.Bank(*_masses(n))
    pool = {}
    for i, lg in enumerate(lgs):
        if (lg, i % 5) not in pool:
            pool[lg, i % 5] = _segment(mf, lg, seed=i % 5)
    segs = [pool[lg, i % 5] for i, lg in enumerate(lgs)]
    peaks, trig, nt = mf.filter_bank(bank, segs, thr, trig_cap=1 << 20)
    assert bank.check() == 0
    peaks, trig = peaks.cpu().numpy().view(np.uint8).reshape(n, len(segs), -1), mf.triggers_to_numpy(trig, nt)
    key = (trig["tmpl"].astype(np.int64) * len(segs) + trig["seg"]) << 22 | trig["j"]
    assert np.all(np.diff(key) > 0)
    one, alone = mf.Bank(*_masses(n)), {}
    for i, s in enumerate(segs):
        if id(s) not in alone:
            p1, t1, n1 = mf.filter_bank(one, [s], thr, trig_cap=1 << 20)
            alone[id(s)] = p1.cpu().numpy().view(np.uint8).reshape(n, -1).copy(), mf.triggers_to_numpy(t1, n1).copy()
        p1, t1 = alone[id(s)]
        mine = trig[trig["seg"] == i]
        assert np.array_equal(peaks[:, i], p1) and mine.size == t1.size
        for f in ("tmpl", "j", "rho", "z_re", "z_im"):
            assert np.array_equal(mine[f], t1[f]), f


# a capture whose workspace was made by calls on single segments takes them one by one
def test_short_segments_in_a_capture(mf):
    import torch
    bank, segs = mf.Bank(*_masses(20)), [_segment(mf, lg) for lg in (12, 15, 13)]
    ref = _run(mf, mf.Bank(*_masses(20)), segs, 4.25)
    for warm in ([[s] for s in segs], [segs]):
        for w in warm:
            mf.filter_bank(bank, w, 4.25, trig_cap=1 << 20)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            out = mf.filter_bank(bank, segs, 4.25, trig_cap=1 << 20)
        for _ in range(2):
            g.replay()
            torch.cuda.synchronize()
            nt = int(out[2][0])
            assert nt == ref[2] and np.array_equal(out[0].cpu().numpy().view(np.uint8), ref[0])
            assert np.array_equal(out[1][:nt].cpu().numpy().view(np.uint8), ref[1])


def test_trigger_overflow_of_both_sorts(mf):
    bank, seg = mf.Bank(*_masses(9)), _segment(mf, 12)
    full = mf.triggers_to_numpy(*mf.filter_bank(bank, [seg], 0.0, trig_cap=9 << 12)[1:])
    ids = full["tmpl"].astype(np.int64) << 12 | full["j"]
    for cap in (1, 8192, 8193, 20000):
        _, trig, nt = mf.filter_bank(bank, [seg], 0.0, trig_cap=cap)
        assert bank.check() == mf.MF_EOVERFLOW if hasattr(mf, "MF_EOVERFLOW") else bank.check() != 0
        assert int(nt.item()) == full.size
        t = mf.triggers_to_numpy(trig, nt)
        k = t["tmpl"].astype(np.int64) << 12 | t["j"]
        assert k.size == cap and np.all(np.diff(k) > 0)
        assert np.array_equal(t["rho"], full["rho"][np.searchsorted(ids, k)])


# one CTA up to 8192 triggers (of a capacity below or above that), then tiles
@pytest.mark.parametrize("n,cap,W", [(1, 1, 3), (33, 64, 0), (1024, 8192, 5), (8191, 9000, 40), (8192, 8192, 3),
                                     (8193, 8193, 3), (40000, 60000, 0), (40000, 40000, 100), (30000, 30000, 1 << 20)])
def test_cluster_sizes(mf, n, cap, W):
    import torch
    rng = np.random.default_rng(n + W)
    key = np.sort(rng.choice(61 * 3 * 50000, n, replace=False))
    a = np.zeros(n, dtype=[("tmpl", "i4"), ("seg", "i4"), ("j", "i4"), ("rho", "f4"), ("z_re", "f4"), ("z_im", "f4")])
    a["tmpl"], a["seg"], a["j"] = key // 150000, key // 50000 % 3, key % 50000
    a["rho"] = rng.choice([6.0, 6.5, 7.25, 9.0], n)
    a["z_re"] = rng.standard_normal(n).astype(np.float32)
    buf = np.zeros((cap, 6), dtype=np.float32)
    buf[:n] = np.ascontiguousarray(a).view(np.float32).reshape(-1, 6)
    ev, n_ev = mf.cluster_triggers(torch.from_numpy(buf).cuda(), torch.tensor([n], device="cuda"), 61, 3, 50000, W)
    got = mf.events_to_numpy(ev, n_ev)
    o = np.zeros(n, dtype=oracle.TRIG_DTYPE)
    for f in a.dtype.names:
        o[f] = a[f]
    ref = oracle.cluster(o, W)
    assert int(n_ev.item()) == ref.size
    for f in ("tmpl", "seg", "j", "n_trig", "n_tmpl"):
        assert np.array_equal(got[f], ref[f]), f
    assert np.array_equal(got["rho"], ref["rho"].astype(np.float32))
    assert np.array_equal(got["z_re"], ref["z_re"].astype(np.float32))


# Eq. (5): single samples against the series, over the row lengths, p, the sizes
# of the segment table (1, 16, 256) and more rows than blocks; both are FP32 sums
# of the same terms in another order, held to the tolerance of the chi^2 tests
@pytest.mark.parametrize("lg,p,n_seg", [(10, 1, 1), (12, 3, 2), (14, 16, 17), (16, 64, 1), (18, 16, 16), (21, 8, 1)])
def test_chisq_points_and_series(mf, lg, p, n_seg):
    import torch
    N, n = 1 << lg, 3
    bank = mf.Bank(*_masses(n, seed=4), f_low=60.0)
    segs = [_segment(mf, lg, seed=20 + i) for i in range(n_seg)]
    rng = np.random.default_rng(lg)
    rows = np.stack([rng.integers(0, n, 200), rng.integers(0, n_seg, 200), rng.integers(0, N, 200)], 1).astype(np.int32)
    got = mf.chisq_points(bank, segs, torch.from_numpy(rows).cuda(), p=p).cpu().numpy().astype(np.float64)
    for s in range(n_seg):
        chi = mf.chisq_series(bank, segs[s], list(range(n)), p=p)[0].cpu().numpy().astype(np.float64)
        rho = gpu_rho_series(mf, bank, segs[s], n, N)[0] if lg <= 18 else None
        for (t, sg, j), g in zip(rows, got):
            if sg == s:
                r2 = rho[t, j] ** 2 if rho is not None else 40.0
                assert abs(g - chi[t, j]) <= 2e-4 * (chi[t, j] + 2.0 * r2) + 1e-4, (t, s, j, g, chi[t, j])


@pytest.mark.parametrize("lg", [10, 13, 16, 17, 18, 21])
def test_chisq_series_batches_agree(mf, lg):
    """A list of one template and the same template inside a longer list."""
    bank, seg = mf.Bank(*_masses(7, seed=4), f_low=60.0), _segment(mf, lg)
    a, ea = mf.chisq_series(bank, seg, [5, 0, 6, 2], p=5)
    for i, t in enumerate((5, 0, 6, 2)):
        b, eb = mf.chisq_series(bank, seg, [t], p=5)
        assert np.array_equal(a[i].cpu().numpy(), b[0].cpu().numpy())
        assert np.array_equal(ea[i].cpu().numpy(), eb[0].cpu().numpy())


# the phase at 64-bit accuracy between anchors 1, 2, .. 256 bins apart (short to
# long segments, light and heavy banks), columns sharing a record or not
@pytest.mark.parametrize("lg,fs,f_low,m_lo,m_hi", [(10, 4096.0, 40.0, 1.2, 12.0), (12, 1024.0, 30.0, 1.2, 3.0),
                                                   (13, 2048.0, 55.0, 8.0, 17.0), (16, 2048.0, 40.0, 1.2, 1.6),
                                                   (16, 4096.0, 30.0, 1.0, 9.0), (18, 4096.0, 40.0, 1.0, 3.0),
                                                   (20, 4096.0, 40.0, 1.0, 3.0)])
def test_phase_fp64_anchor_spacings(mf, lg, fs, f_low, m_lo, m_hi):
    import torch
    wl = workloads.small(seed=300 + lg, N=1 << lg, fs=fs, n_templates=3, m_lo=m_lo, m_hi=m_hi)
    s32, s64 = oracle_segment(wl.segments[0], f_low)
    seg = mf.Segment(torch.from_numpy(s32).cuda(), fs)
    bank = mf.Bank(wl.m1, wl.m2, f_low=f_low, phase_mode=mf.MF_PHASE_FP64)
    rho, z, _ = gpu_rho_series(mf, bank, seg, 3, 1 << lg)
    for t, r in enumerate(oracle_rho_series(wl.m1, wl.m2, s64, fs, f_low)):
        assert rho_err(rho[t], r["rho"]).max() <= RHO_TOL
        assert (np.abs(z[t] - r["z"]) / r["sigma"]).max() <= RHO_TOL


# one kernel for 4096 .. 16384 points: fewer, as many and more sequences than CTAs, an
# odd one in the last pair, complex64 arrays on an 8-byte boundary, in place
@pytest.mark.parametrize("lg,batch", [(12, 1), (12, 607), (12, 611), (13, 305), (14, 151), (14, 154)])
@pytest.mark.parametrize("sign", [-1, 1])
def test_fft_of_one_kernel(mf, lg, batch, sign):
    import torch
    N = 1 << lg
    rng = np.random.default_rng([lg, batch])
    x = (rng.standard_normal((batch, N)) + 1j * rng.standard_normal((batch, N))).astype(np.complex64)
    buf = torch.zeros(batch * N + 1, dtype=torch.complex64, device="cuda")
    t = buf[1:].view(batch, N)
    t.copy_(torch.from_numpy(x))
    out = mf.fft(t, sign=sign).cpu().numpy()
    mf.fft(t, sign=sign, out=t)
    assert np.array_equal(out.view(np.uint64), t.cpu().numpy().view(np.uint64))
    assert buf[0].item() == 0
    x = x.astype(np.complex128)
    ref = np.fft.fft(x, axis=-1) if sign < 0 else np.fft.ifft(x, axis=-1) * N
    tol = 4e-7 * lg * np.linalg.norm(x, axis=-1, keepdims=True)
    assert np.all(np.abs(out - ref) <= tol)


# W from the one-sequence-per-CTA transform (to 2^17 samples) and the long one: the
# filter of new samples equals that of a new segment, every bin of the split included
@pytest.mark.parametrize("lg", [10, 12, 15, 17, 18])
def test_refresh_equals_upload(mf, lg):
    import torch
    g = torch.Generator(device="cuda").manual_seed(lg)
    a, b = (torch.randn(1 << lg, dtype=torch.float32, device="cuda", generator=g) for _ in range(2))
    bank, seg = mf.Bank(*_masses(2)), mf.Segment(a, 1024.0)
    seg.refresh(b)
    x, y = _run(mf, bank, [seg], 2.0), _run(mf, bank, [mf.Segment(b, 1024.0)], 2.0)
    assert x[2] == y[2] and np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])


def test_scratch_of_threads_and_streams(mf):
    """chi^2 series of two banks on two threads and streams share the scratch
    pool; every call's result is that of the call alone."""
    import torch
    work = [(mf.Bank(*_masses(6, seed=s)), _segment(mf, lg, seed=s)) for s, lg in ((1, 16), (2, 18))]
    torch.cuda.synchronize()
    alone = [mf.chisq_series(b, g, list(range(6)), p=8)[0].clone() for b, g in work]
    torch.cuda.synchronize()
    bad = []

    def go(i):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(8):
                got = mf.chisq_series(*work[i], list(range(6)), p=8)[0]
                st.synchronize()
                if not torch.equal(got, alone[i]):
                    bad.append(i)

    th = [threading.Thread(target=go, args=(i,)) for i in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad


# bands that end below fs/8 (the leading-row form of the staged pass 1): whole and
# mixed batches against one CTA per tile, which forms every row
@pytest.mark.parametrize("lg,fs,m", [(16, 16384.0, 3.0), (17, 4096.0, 20.0), (18, 4096.0, 10.0), (19, 4096.0, 16.0),
                                     (20, 4096.0, 5.0), (20, 8192.0, 8.0), (21, 4096.0, 30.0)])
def test_leading_bands(mf, monkeypatch, lg, fs, m):
    r = np.random.default_rng(lg)
    m1, m2 = r.uniform(0.3 * m, 1.5 * m, (2, 21))
    bank, seg = mf.Bank(m1, m2), _segment(mf, lg, fs)
    a = _run(mf, bank, [seg], 4.75)
    monkeypatch.setenv("MFGB_P1PF", "0")
    b = _run(mf, bank, [seg], 4.75)
    assert bank.check() == 0 and a[2] == b[2]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


# chi^2 tiles in clusters of four and two and alone (at most one wave of two blocks
# per SM, two sub-bands or more per block): one template, whose tiles are few,
# against the same template among many
@pytest.mark.parametrize("lg,p,n", [(10, 3, 400), (10, 7, 80), (12, 16, 200), (14, 2, 3), (14, 6, 30), (14, 7, 30),
                                    (14, 16, 170), (16, 16, 20), (16, 64, 12), (17, 9, 9), (18, 16, 12)])
def test_chisq_tiles_in_clusters(mf, lg, p, n):
    bank, seg = mf.Bank(*_masses(n)), _segment(mf, lg)
    many = mf.chisq_series(bank, seg, list(range(n)), p=p)[0].cpu().numpy()
    assert bank.check() == 0
    for t in {0, n // 2, n - 1}:
        one = mf.chisq_series(bank, seg, [t], p=p)[0].cpu().numpy()[0]
        # both are FP32 sums of p + 1 squares of size rho^2 <= chi^2 + rho^2 terms
        assert np.max(np.abs(one - many[t])) <= 1e-4 * max(1.0, float(np.max(many[t])))


# clustering and the chi^2 of single samples allocate scratch in stream order, in a
# capture as allocation nodes of the graph
def test_events_in_a_capture(mf):
    import torch
    bank, seg = mf.Bank(*_masses(12)), _segment(mf, 16)
    loudest = float(mf.filter_bank(bank, [seg], 1e9, trig_cap=1 << 16)[0].view(-1, 4)[:, 0].max())
    _, trig, nt = mf.filter_bank(bank, [seg], 0.75 * loudest, trig_cap=1 << 16)
    ev, n_ev = mf.cluster_triggers(trig, nt, bank.n, 1, seg.N, 40)
    n = int(n_ev.item())
    assert n > 1
    rows = ev[:n].clone()
    chi = mf.chisq_points(bank, [seg], rows, p=8)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ev2, n2 = mf.cluster_triggers(trig, nt, bank.n, 1, seg.N, 40)
        chi2 = mf.chisq_points(bank, [seg], rows, p=8)
    for _ in range(3):
        g.replay()
        torch.cuda.synchronize()
        assert int(n2.item()) == n and torch.equal(ev2[:n].view(torch.int32), ev[:n].view(torch.int32))
        assert torch.equal(chi2, chi)
