"""Bounded device waits that run out: the caller must be able to see it.  The
waits are given a limit they cannot keep; nothing is withheld and nothing
faults, the CTAs give up and return."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_4175_gb300 import build
    build.build()
    import paper_0906_4175_gb300 as m
    return m


@pytest.mark.parametrize("n", [8193, 60000])
def test_clustering_that_gives_up_says_so(mf, n):
    """More than 8192 triggers: the CTAs without a tile of the first step wait
    for the others'.  n_events must not read as a count, also when it held one
    before, and the next call must work."""
    import torch
    a = np.zeros(n, dtype=mf.TRIG_DTYPE)
    a["j"] = 10 * np.arange(n)
    a["rho"] = np.random.default_rng(n).choice([6.0, 7.0, 8.5], n)
    trig = torch.from_numpy(a.view(np.float32).reshape(-1, 6)).cuda()
    nt = torch.tensor([n], device="cuda")
    ev, n_ev = mf.cluster_triggers(trig, nt, 1, 1, 1 << 20, 3)
    assert int(n_ev.item()) == n
    L = mf._native.lib()
    L.mf_debug_cluster_spin(1)
    try:
        bad, n_bad = mf.cluster_triggers(trig, nt, 1, 1, 1 << 20, 3)
        torch.cuda.synchronize()
    finally:
        L.mf_debug_cluster_spin(0)
    assert int(n_bad.item()) == -1
    with pytest.raises(mf.MFError) as e:
        mf.events_to_numpy(bad, n_bad)
    assert e.value.code == mf.MF_ETIMEOUT
    ev2, n_ev = mf.cluster_triggers(trig, nt, 1, 1, 1 << 20, 3)
    assert int(n_ev.item()) == n and torch.equal(ev2.view(torch.int32), ev.view(torch.int32))


@pytest.mark.parametrize("lg", [16, 17, 18, 19, 21, 22])
def test_chisq_reports_waits_at_every_length(mf, lg):
    """The staged first pass needs a place for the status of a wait that runs
    out, and refuses to start without one; a new bank's first call has it."""
    import torch
    bank = mf.Bank([1.4, 2.0], [1.3, 1.7])
    seg = mf.Segment(torch.randn(1 << lg, dtype=torch.float32, device="cuda"), 4096.0)
    chi, _ = mf.chisq_series(bank, seg, [0, 1], p=2)
    assert bank.check() == 0 and bool(torch.isfinite(chi).all())
