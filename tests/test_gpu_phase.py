"""The phase of MF_PHASE_FP64, in turns mod 1, against the Sec. 1.1 formula in
extended precision at every bin of the band.

Tolerance: the value is rounded once, to FP32 in [-1/4, 1/4] (half an ulp there:
2^-27 = 7.5e-9); before that the 64-bit sum is good to 4e-10, and the FP64
rounding of the template's constants (a few 1e-16 of up to 1e4 turns) is within
5e-11.  FP64 at every bin rounded to FP32 in [-1/2, 1/2], which
this mode must not fall behind, is off by up to 2^-26 = 1.5e-8."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -27 + 4e-10 + 5e-11
LD = np.longdouble


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_4175_gb300 import build
    build.build()
    import paper_0906_4175_gb300 as m
    return m


def _psi(m1, m2, f):
    pi = LD("3.14159265358979323846264338327950288")
    m1, m2 = LD(m1), LD(m2)
    M = m1 + m2
    eta = m1 * m2 / (M * M)
    v = np.cbrt(pi * M * LD(oracle.MSUN_S) * f)
    v = v - (v * v * v - pi * M * LD(oracle.MSUN_S) * f) / (3 * v * v)
    a2 = LD(3715) / 756 + 55 * eta / 9
    a4 = LD(15293365) / 508032 + 27145 * eta / 504 + 3085 * eta * eta / 72
    series = 1 + v * v * (a2 + v * (-16 * pi + v * a4))
    return (-pi / 4 + 3 / (128 * eta * v ** 5) * series) / (2 * pi)


@pytest.mark.parametrize("lg,fs,f_low,m_lo,m_hi", [(10, 4096.0, 40.0, 1.2, 12.0), (12, 1024.0, 30.0, 1.2, 3.0),
                                                   (16, 4096.0, 30.0, 1.0, 9.0), (18, 4096.0, 40.0, 1.0, 34.0),
                                                   (18, 2048.0, 10.0, 1.0, 3.0), (20, 4096.0, 40.0, 5.0, 34.0),
                                                   (22, 16384.0, 15.0, 1.0, 3.0)])
def test_phase_at_every_bin(mf, lg, fs, f_low, m_lo, m_hi):
    import torch
    N = 1 << lg
    m = np.random.default_rng(lg).uniform(m_lo, m_hi, (2, 2))
    bank = mf.Bank(m[0], m[1], f_low=f_low, phase_mode=mf.MF_PHASE_FP64)
    seg = mf.Segment(torch.randn(N, device="cuda", dtype=torch.float32), fs)
    out = torch.empty(N // 2, dtype=torch.float64, device="cuda")
    for t in range(2):
        mf._native.check(mf._native.lib().mf_debug_phase(bank.handle, seg.handle, t, out.data_ptr(), None))
        lo, hi = oracle.band(N, fs, f_low, oracle.f_isco(m[0][t], m[1][t]))
        k = np.arange(lo, hi)
        if k.size > 200000:     # the lowest bins, where the phase turns fastest, and a sample
            k = np.concatenate([k[:100000], np.sort(np.random.default_rng(1).choice(k[100000:], 100000, replace=False))])
        err = LD(1) * out.cpu().numpy()[k] - _psi(m[0][t], m[1][t], k * (LD(fs) / N))
        err = np.abs(err - np.rint(err)).astype(np.float64)
        assert err.max() <= TOL, (t, err.max())
        assert np.sqrt(np.mean(err ** 2)) <= TOL / np.sqrt(3)
