"""Performance cases of the matched-filter library: what a user's program has it do, at the sizes it is used at.

Each case is one call, or one short sequence of calls, of the package's public entry points on device
data that the program already holds (bank, segments, output buffers).  Inputs are made here from the
seed with plain torch: Gaussian noise coloured by the initial-LIGO PSD from f_low up, with loud
injections of 2PN templates, as 32-bit samples.  ``exact`` evaluates the same equations in 64 bits with
torch and numpy alone.

Kinds:
  search  refresh every segment with its samples, then filter the bank over all of them (a search step);
  bank    filter a bank over segments that are already conditioned;
  chisq   the chi^2 series of a list of templates;
  events  triggers -> events -> chi^2 at every event;
  refine  rho^2 of trigger rows at continuous (m1, m2, t) and its gradient;
  fft     a batched complex transform.
"""
import math

import numpy as np
import torch

import paper_0906_4175_gb300 as mf

MSUN_S = 4.925490947e-6   # G Msun / c^3 in seconds
F0 = 150.0                # the PSD's knee


def _mass(case, rng):
    """Template masses: uniform in [m_lo, m_hi], total mass at most m_tot."""
    n, lo, hi, tot = case["templates"], case["m_lo"], case["m_hi"], case["m_tot"]
    m = np.empty((0, 2))
    while len(m) < n:
        c = rng.uniform(lo, hi, size=(2 * n + 16, 2))
        m = np.concatenate([m, c[c.sum(1) <= tot]])
    return m[:n, 0].copy(), m[:n, 1].copy()


def listed():
    return [
        # One short segment against a handful of templates (the 16-template, 32 s workload): a low-latency
        # search step, where launches and latency count.
        dict(name="search_tiny", kind="search", log2n="16", fs=2048.0, f_low=40.0, templates=16, m_lo=1.2, m_hi=1.6,
             m_tot=35.0, threshold=6.0, phase="anchor", cap=1 << 20),
        # Several short segments at once, at a low sample rate: a ragged bank on the shortest transforms.
        dict(name="search_short", kind="search", log2n="12,13,13,14", fs=1024.0, f_low=40.0, templates=75, m_lo=1.2,
             m_hi=3.0, m_tot=35.0, threshold=6.0, phase="anchor", cap=1 << 20),
        # The flagship search step: 1024 templates over one 256 s segment at 4096 Hz.
        dict(name="search_scale", kind="search", log2n="20", fs=4096.0, f_low=40.0, templates=1024, m_lo=1.0, m_hi=3.0,
             m_tot=35.0, threshold=6.0, phase="anchor", cap=1 << 20),
        # A wide-mass bank over segments of four lengths in one call (the largest case).
        dict(name="bank_uneven", kind="bank", log2n="18,18,19,19,20,20,21,21", fs=4096.0, f_low=40.0, templates=4096,
             m_lo=1.0, m_hi=34.0, m_tot=35.0, threshold=6.0, phase="anchor", cap=1 << 22),
        # The paper's longest transforms: 4 x 2^20 points.
        dict(name="bank_long", kind="bank", log2n="22", fs=4096.0, f_low=40.0, templates=128, m_lo=1.0, m_hi=3.0,
             m_tot=35.0, threshold=6.0, phase="anchor", cap=1 << 20),
        # The phase evaluated in 64 bits at every bin: the accuracy option of the bank.
        dict(name="bank_phase64", kind="bank", log2n="18", fs=4096.0, f_low=40.0, templates=250, m_lo=1.0, m_hi=3.0,
             m_tot=35.0, threshold=6.0, phase="fp64", cap=1 << 20),
        # The chi^2 series the paper moved to its GPU: 64 templates, p = 16, every sample of 256 s.
        dict(name="chisq_scale", kind="chisq", log2n="20", fs=4096.0, f_low=40.0, templates=64, m_lo=1.0, m_hi=3.0,
             m_tot=35.0, p=16),
        # The same on a 32 s segment at 2048 Hz: the chi^2 step of the low-latency search.
        dict(name="chisq_short", kind="chisq", log2n="16", fs=2048.0, f_low=40.0, templates=16, m_lo=1.2, m_hi=1.6,
             m_tot=35.0, p=16),
        # Post-processing of a search: about 5000 triggers into events, chi^2 at each event.
        dict(name="events_scale", kind="events", log2n="20", fs=4096.0, f_low=40.0, templates=1024, m_lo=1.0, m_hi=3.0,
             m_tot=35.0, p=16, clusters=9, triggers=5000, window=4096, cap=1 << 20),
        # Gradient refinement of 256 coarse triggers spread over 32 segments.
        dict(name="refine_bank", kind="refine", log2n=",".join(["20"] * 32), fs=4096.0, f_low=40.0, rows=256, m_lo=1.0,
             m_hi=20.0, m_tot=40.0),
        # The paper's transform benchmark at 2^20 points (inverse), and a forward one of short transforms.
        dict(name="fft_long", kind="fft", log2=20, batch=64, sign=1),
        dict(name="fft_short", kind="fft", log2=14, batch=1000, sign=-1),
    ]


def draw(rng):
    kind = rng.choice(["search", "search", "bank", "chisq", "events", "refine", "fft", "fft"])
    lu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    if kind == "fft":
        lg = rng.randint(10, 22)
        return dict(kind="fft", log2=lg, batch=lu(1, max(2, (1 << 27) >> lg)), sign=rng.choice([-1, 1]))
    fs = rng.choice([1024.0, 2048.0, 4096.0])
    f_low = rng.choice([30.0, 40.0, 40.0, 55.0])
    lo, hi = rng.choice([(1.2, 1.6), (1.0, 3.0), (1.0, 34.0)])
    case = dict(kind=kind, fs=fs, f_low=f_low, m_lo=lo, m_hi=hi, m_tot=35.0)
    if kind in ("search", "bank"):
        n_seg = rng.choice([1, 1, 2, 3, 8])
        logs = [rng.randint(12, 22) if n_seg == 1 else rng.randint(12, 21) for _ in range(n_seg)]
        total = sum(1 << g for g in logs)
        phase = rng.choice(["anchor"] * 5 + ["fp64"])
        most = max(1, min(4096, ((1 << 33) if phase == "anchor" else (1 << 30)) // total))
        return dict(case, log2n=",".join(map(str, logs)), templates=lu(1, most), threshold=round(rng.uniform(5.5, 8.0), 2),
                    phase=phase, cap=1 << (23 if hi > 3 else 20))
    if kind == "chisq":
        lg = rng.randint(12, 21)
        return dict(case, log2n=str(lg), templates=lu(1, max(2, min(256, (1 << 27) >> lg))), p=rng.choice([4, 8, 16]))
    if kind == "events":
        lg, clusters = rng.randint(14, 20), lu(1, 64)
        return dict(case, log2n=str(lg), templates=lu(16, 1024), p=rng.choice([8, 16]), clusters=clusters,
                    triggers=lu(100, 50000), window=lu(16, min(4096, (1 << lg) // (3 * clusters))), cap=1 << 20)
    n_seg = rng.choice([1, 4, 16])
    return dict(case, kind="refine", log2n=",".join([str(rng.randint(14, 20))] * n_seg), rows=lu(1, 512))


# ---- the equations in 64 bits, with torch alone ------------------------------------------------------

def _psd(N, fs):
    """Eq. (2) on bins 0..N/2 (infinite at 0)."""
    x = torch.arange(N // 2 + 1, dtype=torch.float64, device="cuda") * (fs / N) / F0
    S = (4.49 * x) ** -56.0 + 0.16 * x ** -4.52 + 0.52 + 0.32 * x * x
    S[0] = math.inf
    return S


def _coeffs(m1, m2):
    """Psi = -pi/4 + sum_p c_p f^(-p/3), p = 1, 2, 3, 5 (numbers or tensors), f_isco and A = Mc^(5/6)."""
    M = m1 + m2
    eta = m1 * m2 / (M * M)
    v1 = (math.pi * MSUN_S * M) ** (1.0 / 3.0)
    pre = 3.0 / (128.0 * eta)
    a2 = 3715.0 / 756.0 + 55.0 * eta / 9.0
    a4 = 15293365.0 / 508032.0 + 27145.0 * eta / 504.0 + 3085.0 * eta * eta / 72.0
    c = (pre * a4 / v1, pre * (-16.0 * math.pi) / v1 ** 2, pre * a2 / v1 ** 3, pre / v1 ** 5)
    return c, 1.0 / (6.0 * math.sqrt(6.0) * math.pi * MSUN_S * M), (eta ** 0.6 * M) ** (5.0 / 6.0)


def _band(N, fs, f_low, f_isco):
    lo = max(1, math.ceil(f_low * N / fs))
    hi = min(math.floor(min(f_isco, 0.5 * fs) * N / fs) + 1, N // 2)
    return lo, max(lo, hi)


def _psi(c, f):
    u = f ** (-1.0 / 3.0)
    u2 = u * u
    return -math.pi / 4.0 + c[0] * u + c[1] * u2 + c[2] * u2 * u + c[3] * u2 * u2 * u


def _template(m1, m2, N, fs, f_low):
    """(k_lo, k_hi, h~ on the band without its amplitude constant, A)."""
    c, f_isco, A = _coeffs(m1, m2)
    lo, hi = _band(N, fs, f_low, f_isco)
    f = torch.arange(lo, hi, dtype=torch.float64, device="cuda") * (fs / N)
    return lo, hi, torch.polar(f ** (-7.0 / 6.0), -_psi(c, f)), A


def _samples(case, seed):
    """Every segment's samples (float32, cuda) and its injections as (m1, m2, snr, j0)."""
    rng = np.random.default_rng([seed, 1])
    out = []
    for i, lg in enumerate(int(v) for v in case["log2n"].split(",")):
        N, fs = 1 << lg, case["fs"]
        gen = torch.Generator(device="cuda").manual_seed(seed * 1000 + i)
        S = _psd(N, fs)
        lo = max(1, math.ceil(case["f_low"] * N / fs))
        g = torch.randn(N // 2 + 1, 2, dtype=torch.float64, device="cuda", generator=gen)
        st = torch.zeros(N // 2 + 1, dtype=torch.complex128, device="cuda")
        st[lo:N // 2] = torch.view_as_complex(g)[lo:N // 2] * torch.sqrt(N / fs * S[lo:N // 2] / 4)
        inj = []
        # a heavy template rings in thousands of others for seconds: two injections per segment of a wide bank
        for _ in range(1 if lg < 18 else 2 if case["m_hi"] > 3 and case["kind"] != "refine" else 8):
            m1, m2 = rng.uniform(case["m_lo"], case["m_hi"], size=2)
            if m1 + m2 > case["m_tot"]:
                m1, m2 = m1 / 2, m2 / 2
            snr, j0, phi = rng.uniform(8.0, 20.0), int(rng.integers(0, N)), rng.uniform(0, 2 * math.pi)
            a, b, h, _ = _template(m1, m2, N, fs, case["f_low"])
            if b <= a:
                continue
            sig = torch.sqrt(4 * fs / N * (h.abs() ** 2 / S[a:b]).sum())
            k = torch.arange(a, b, dtype=torch.int64, device="cuda")
            turn = (k * j0 % N).to(torch.float64) / N
            st[a:b] += snr / sig * h * torch.polar(torch.ones_like(turn), phi - 2 * math.pi * turn)
            inj.append((m1, m2, snr, j0))
        s = torch.fft.irfft(st * fs, n=N)
        out.append((s.to(torch.float32), inj))
    return out


def _triggers(case, seed):
    """Sorted trigger records (int32 words [n, 6]): samples around a few times, over many templates."""
    rng = np.random.default_rng([seed, 2])
    N, n, c = 1 << int(case["log2n"]), case["triggers"], case["clusters"]
    at = ((np.arange(c) + rng.uniform(0.4, 0.6, c)) * N / c).astype(np.int64)
    which = np.arange(n) % c
    j = at[which] + np.clip(np.rint(rng.normal(0, case["window"] / 10.0, n)), -0.4 * case["window"], 0.4 * case["window"])
    j = j.astype(np.int64)
    t = rng.integers(0, case["templates"], n)
    _, keep = np.unique(t * N + j, return_index=True)
    t, j = t[keep], j[keep]
    rho = (6.0 + rng.exponential(1.5, len(t))).astype(np.float32)
    ph = rng.uniform(0, 2 * math.pi, len(t))
    rec = np.zeros((len(t), 6), dtype=np.int32)
    rec[:, 0], rec[:, 2] = t, j
    rec[:, 3] = rho.view(np.int32)
    rec[:, 4] = (rho * np.cos(ph)).astype(np.float32).view(np.int32)
    rec[:, 5] = (rho * np.sin(ph)).astype(np.float32).view(np.int32)
    return rec


def _theta(case, seed, segs):
    """Rows (m1, m2, t) near injections, and each row's segment."""
    rng = np.random.default_rng([seed, 3])
    rows, where = [], []
    for i in range(case["rows"]):
        s = i % len(segs)
        N = segs[s][0].numel()
        inj = segs[s][1]
        m1, m2, _, j0 = inj[(i // len(segs)) % len(inj)]
        e = rng.normal(0, 2e-3, 2)
        rows.append((m1 * (1 + e[0]), m2 * (1 + e[1]), ((N - j0) % N) / case["fs"] + rng.normal(0, 2e-4)))
        where.append(s)
    return torch.tensor(rows, dtype=torch.float64, device="cuda"), torch.tensor(where, dtype=torch.int32, device="cuda")


# ---- the cases ---------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "fft":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(case["batch"], 1 << case["log2"], dtype=torch.complex64, device="cuda", generator=gen)
        return dict(kind=kind, x=x, y=torch.empty_like(x), sign=case["sign"])
    data = _samples(case, seed)
    segs = [mf.Segment(s, case["fs"]) for s, _ in data]
    st = dict(kind=kind, segs=segs, samples=[s for s, _ in data])
    if kind == "refine":
        st["theta"], st["row_seg"] = _theta(case, seed, data)
        st["f_low"] = case["f_low"]
        st["theta"].requires_grad_(True)
        return st
    phase = mf.MF_PHASE_FP64 if case.get("phase") == "fp64" else mf.MF_PHASE_ANCHOR
    m1, m2 = _mass(case, np.random.default_rng([seed, 4]))
    st["bank"] = mf.Bank(m1, m2, f_low=case["f_low"], phase_mode=phase)
    if kind in ("search", "bank"):
        n = case["templates"] * len(segs)
        peaks = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
        trig = torch.zeros((case["cap"], 6), dtype=torch.float32, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        st.update(out=(peaks, trig, count), threshold=case["threshold"], cap=case["cap"])
        st["views"] = dict(peak_rho=peaks[:, 0], peak_j=peaks.view(torch.int32)[:, 1], peak_z=peaks[:, 2:],
                           trig_at=trig.view(torch.int32)[:, :3], trig_rho=trig[:, 3], trig_z=trig[:, 4:], n_trig=count)
    elif kind == "chisq":
        st.update(tmpl=torch.arange(case["templates"], dtype=torch.int32, device="cuda"), p=case["p"])
    else:
        rec = _triggers(case, seed)
        trig = torch.zeros((case["cap"], 6), dtype=torch.int32, device="cuda")
        trig[:len(rec)] = torch.from_numpy(rec).cuda()
        st.update(trig=trig.view(torch.float32), n_trig=torch.tensor([len(rec)], dtype=torch.int64, device="cuda"),
                  templates=case["templates"], window=case["window"], p=case["p"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "fft":
        return mf.fft(st["x"], sign=st["sign"], out=st["y"])
    if kind in ("search", "bank"):
        if kind == "search":
            for seg, s in zip(st["segs"], st["samples"]):
                seg.refresh(s)
        mf.filter_bank(st["bank"], st["segs"], st["threshold"], trig_cap=st["cap"], out=st["out"])
        return st["views"]
    if kind == "chisq":
        chisq, edges = mf.chisq_series(st["bank"], st["segs"][0], st["tmpl"], p=st["p"])
        return dict(chisq=chisq, edges=edges)
    if kind == "events":
        ev, n_ev = mf.cluster_triggers(st["trig"], st["n_trig"], st["templates"], 1, st["segs"][0].N, st["window"])
        found = ev[:int(n_ev.item())]
        chisq = mf.chisq_points(st["bank"], st["segs"], found, p=st["p"])
        words = found.view(torch.int32)
        return dict(at=words[:, :3], rho=found[:, 3], z=found[:, 4:6], size=words[:, 6:], chisq=chisq)
    rho2 = mf.RefineFn.apply(st["theta"], st["segs"], None, st["f_low"], st["row_seg"])
    grad, = torch.autograd.grad(rho2.sum(), st["theta"])
    return dict(rho2=rho2.detach(), grad=grad)


def work(case):
    if case["kind"] == "fft":
        n = case["batch"] << case["log2"]
        return dict(bytes=16 * n, flops=5 * n * case["log2"])
    ns = [1 << int(v) for v in case["log2n"].split(",")]
    data = sum((4 if case["kind"] == "search" else 8) * (N if case["kind"] == "search" else N // 2) for N in ns)
    if case["kind"] in ("search", "bank"):
        fft = sum(5 * N * math.log2(N) for N in ns)
        return dict(bytes=data + case["templates"] * len(ns) * 16, flops=case["templates"] * fft)
    if case["kind"] == "chisq":
        N, n, p = ns[0], case["templates"], case["p"]
        return dict(bytes=data + 4 * n * N + 8 * n * (p + 1), flops=n * ((p + 1) * 5 * N * math.log2(N) + 3 * p * N))
    if case["kind"] == "events":
        return dict(bytes=data + 24 * case["triggers"] + 36 * case["clusters"], flops=case["clusters"] * 20 * ns[0] // 2)
    return dict(bytes=data + case["rows"] * 56, flops=case["rows"] * 40 * ns[0] // 2)


# ---- what run() returns, in 64 bits ------------------------------------------------------------------

def _spectrum(s, fs):
    """conj(s~_k)/S_k with s~ = dt DFT(s), and S."""
    N = s.numel()
    S = _psd(N, fs)
    return torch.fft.rfft(s.to(torch.float64)).conj() / fs / S, S


def _z(h, Y, lo, hi, N, fs):
    X = torch.zeros(N, dtype=torch.complex128, device="cuda")
    X[lo:hi] = h * Y[lo:hi]
    return torch.fft.ifft(X) * (4 * fs)      # 4 df N ifft


def _exact_filter(case, seed):
    rng = np.random.default_rng([seed, 4])
    m1, m2 = _mass(case, rng)
    data = [(s, *_spectrum(s, case["fs"])) for s, _ in _samples(case, seed)]
    n_seg, cap, thr = len(data), case["cap"], case["threshold"]
    n = case["templates"] * n_seg
    rho_p, z_p = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, 2, dtype=torch.float64, device="cuda")
    rho_t, z_t, at = [], [], []
    for g, (s, Y, S) in enumerate(data):
        N = s.numel()
        fs = case["fs"]
        for t in range(case["templates"]):
            lo, hi, h, A = _template(m1[t], m2[t], N, fs, case["f_low"])
            if hi <= lo:
                continue
            z = _z(h, Y, lo, hi, N, fs)
            sig = torch.sqrt(4 * fs / N * (h.abs() ** 2 / S[lo:hi]).sum())
            rho = z.abs() / sig
            top = rho.argmax()
            i = t * n_seg + g
            rho_p[i] = rho[top]
            z_p[i] = torch.view_as_real(z[top]) * A
            j = (rho > thr).nonzero().flatten()
            rho_t.append(rho[j])
            z_t.append(torch.view_as_real(z[j]) * A)
            at.append(i * (1 << 23) + j)
    order = torch.cat(at).argsort()[:cap]
    tr, tz = torch.zeros(cap, dtype=torch.float64, device="cuda"), torch.zeros(cap, 2, dtype=torch.float64, device="cuda")
    tr[:len(order)] = torch.cat(rho_t)[order]
    tz[:len(order)] = torch.cat(z_t)[order]
    return dict(peak_rho=rho_p, peak_j=None, peak_z=z_p, trig_at=None, trig_rho=tr, trig_z=tz, n_trig=None)


def _edges(h, S, lo, hi, p):
    """Sub-band edges: the smallest bins at which the running |h|^2/S reaches l/p of its total."""
    c = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), (h.abs() ** 2 / S[lo:hi]).cumsum(0)])
    want = torch.arange(1, p, dtype=torch.float64, device="cuda") / p * c[-1]
    return [lo] + (torch.searchsorted(c, want) + lo).tolist() + [hi], c[-1]


def _exact_chisq(case, seed):
    m1, m2 = _mass(case, np.random.default_rng([seed, 4]))
    s = _samples(case, seed)[0][0]
    N, fs, p = s.numel(), case["fs"], case["p"]
    Y, S = _spectrum(s, fs)
    out = torch.zeros(case["templates"], N, dtype=torch.float64, device="cuda")
    for t in range(case["templates"]):
        lo, hi, h, _ = _template(m1[t], m2[t], N, fs, case["f_low"])
        if hi <= lo:
            continue
        e, tot = _edges(h, S, lo, hi, p)
        z = _z(h, Y, lo, hi, N, fs)
        for a, b in zip(e, e[1:]):
            out[t] += (_z(h[a - lo:b - lo], Y, a, b, N, fs) - z / p).abs() ** 2
        out[t] *= p / (4 * fs / N * tot)
    return dict(chisq=out, edges=None)


def _clusters(rows, window):
    """Single linkage of rows sorted by (group, j): the index ranges of its clusters."""
    cut = np.flatnonzero((np.diff(rows[:, 0]) != 0) | (np.diff(rows[:, 1]) > window)) + 1
    return np.split(np.arange(len(rows)), cut)


def _exact_events(case, seed):
    rec = _triggers(case, seed)
    rho = np.ascontiguousarray(rec[:, 3]).view(np.float32)
    loud = lambda c: min(c, key=lambda i: (-rho[i], rec[i, 2], rec[i, 0]))  # noqa: E731
    first = np.array([loud(c) for c in _clusters(rec[:, [0, 2]], case["window"])])
    first = first[np.lexsort((rec[first, 0], rec[first, 2]))]
    two = np.stack([np.zeros(len(first), dtype=np.int64), rec[first, 2]], 1)
    found = [loud(first[c]) for c in _clusters(two, case["window"])]
    found = np.array(sorted(found, key=lambda i: rec[i, 2]))
    m1, m2 = _mass(case, np.random.default_rng([seed, 4]))
    s = _samples(case, seed)[0][0]
    N, fs, p = s.numel(), case["fs"], case["p"]
    Y, S = _spectrum(s, fs)
    chisq = torch.zeros(len(found), dtype=torch.float64, device="cuda")
    for n, i in enumerate(found):
        t, j = rec[i, 0], int(rec[i, 2])
        lo, hi, h, _ = _template(m1[t], m2[t], N, fs, case["f_low"])
        e, tot = _edges(h, S, lo, hi, p)
        k = torch.arange(lo, hi, dtype=torch.int64, device="cuda")
        x = h * Y[lo:hi] * torch.polar(torch.ones(hi - lo, dtype=torch.float64, device="cuda"),
                                       2 * math.pi * (k * j % N).to(torch.float64) / N) * (4 * fs / N)
        z = x.sum()
        chisq[n] = sum((x[a - lo:b - lo].sum() - z / p).abs() ** 2 for a, b in zip(e, e[1:])) * p / (4 * fs / N * tot)
    f = np.ascontiguousarray(rec[found, 3:]).view(np.float32).astype(np.float64)
    return dict(at=None, rho=torch.from_numpy(f[:, 0].copy()), z=torch.from_numpy(f[:, 1:].copy()), size=None, chisq=chisq)


def _exact_refine(case, seed):
    data = _samples(case, seed)
    theta, row_seg = _theta(case, seed, data)
    spec = [_spectrum(s, case["fs"]) for s, _ in data]
    obj = torch.zeros(case["rows"], dtype=torch.float64, device="cuda")
    grad = torch.zeros(case["rows"], 3, dtype=torch.float64, device="cuda")
    for i, g in enumerate(row_seg.tolist()):
        Y, S = spec[g]
        N, fs = data[g][0].numel(), case["fs"]
        th = theta[i].clone().requires_grad_(True)
        c, f_isco, _ = _coeffs(th[0], th[1])
        lo, hi = _band(N, fs, case["f_low"], float(f_isco.detach()))
        f = torch.arange(lo, hi, dtype=torch.float64, device="cuda") * (fs / N)
        amp = f ** (-7.0 / 6.0)
        z = (torch.polar(amp, 2 * math.pi * f * th[2] - _psi(c, f)) * Y[lo:hi]).sum() * (4 * fs / N)
        rho2 = (z.real ** 2 + z.imag ** 2) / (4 * fs / N * (amp * amp / S[lo:hi]).sum())
        grad[i], = torch.autograd.grad(rho2, th)
        obj[i] = rho2.detach()
    return dict(rho2=obj, grad=grad)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fft":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(case["batch"], 1 << case["log2"], dtype=torch.complex64, device="cuda", generator=gen)
        out = torch.empty_like(x, dtype=torch.complex128)
        for b in range(case["batch"]):
            v = x[b].to(torch.complex128)
            out[b] = torch.fft.fft(v) if case["sign"] < 0 else torch.fft.ifft(v) * v.numel()
        return out
    if kind in ("search", "bank"):
        if kind == "bank" and case["templates"] * sum(1 << int(v) for v in case["log2n"].split(",")) > 1 << 33:
            return None       # over 20 s of 64-bit transforms
        return _exact_filter(case, seed)
    return {"chisq": _exact_chisq, "events": _exact_events, "refine": _exact_refine}[kind](case, seed)
