"""Scratch that outlives a call: what the library's pool keeps, and when it goes
back to the system.  Handles are counted per process, so each case runs in a
process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes, gc
import numpy as np, torch
from paper_0906_4175_gb300 import build
build.build()
import paper_0906_4175_gb300 as mf
L = mf._native.lib()
MB = 1 << 20

def reserved():
    torch.cuda.synchronize()
    v = ctypes.c_int64()
    assert L.mf_debug_scratch_reserved(ctypes.byref(v)) == 0
    return v.value

def bank(n=4):
    m = np.random.default_rng(1).uniform(1.2, 3.0, n)
    return mf.Bank(m, m[::-1].copy())

def segment(lg=16, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return mf.Segment(torch.randn(1 << lg, dtype=torch.float32, device="cuda", generator=g), 4096.0)
"""


def _child(body):
    env = dict(os.environ, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", PRELUDE + body], capture_output=True, text=True, timeout=300, env=env)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("order", ["b a c", "a c b", "a b c", "c b a"])
def test_scratch_is_kept_while_a_handle_lives(order):
    """One bank and two segments, destroyed in several orders: the pool keeps
    the chi^2 series' scratch until the last of them is gone, twice over."""
    _child("""
for cycle in range(2):
    h = {"b": bank(), "a": segment(seed=2), "c": segment(seed=3)}
    mf.chisq_series(h["b"], h["a"], [0, 1, 2, 3], p=16)     # 4 x 17 exchanges of 512 KB
    for name in %r.split():
        assert reserved() >= 32 * MB, (cycle, name, reserved())
        h[name].close()
    assert reserved() == 0, (cycle, reserved())
""" % order)


def test_release_of_scratch_without_handles():
    """A program that only transforms makes no handle: its scratch goes back
    when it asks, and later calls work as before."""
    _child("""
x = torch.randn(8, 1 << 20, dtype=torch.complex64, device="cuda")     # exchange of 64 MB
y = mf.fft(x)
assert reserved() >= 64 * MB
mf.release_scratch()
assert reserved() == 0
assert torch.equal(mf.fft(x), y)
torch.cuda.synchronize()
mf.release_scratch()
assert reserved() == 0
""")


def test_kept_scratch_makes_room():
    """A bank's workspace that fits only without what the pool keeps."""
    _child("""
b, s = bank(8), segment(20)
ref = mf.filter_bank(bank(8), [s], 4.0, trig_cap=1 << 12)
mf.chisq_series(b, s, list(range(8)), p=8)              # 72 exchanges of 8 MB
held = reserved()
assert held >= 512 * MB
L.mf_debug_alloc_limit(held + 32 * MB)                  # the workspace's exchange is 64 MB
got = mf.filter_bank(b, [s], 4.0, trig_cap=1 << 12)
L.mf_debug_alloc_limit(-1)
n = int(ref[2].item())
assert b.check() == 0 and int(got[2].item()) == n
assert torch.equal(got[0], ref[0]) and torch.equal(got[1][:n], ref[1][:n])
assert reserved() == 0
""")


def test_a_refused_allocation_leaves_no_error_behind():
    """MF_ENOMEM from one call; the next one's launches are its own."""
    _child("""
b, s = bank(), segment()
_, trig, nt = mf.filter_bank(b, [s], 3.0, trig_cap=1 << 14)
for refused in (lambda: mf.filter_bank(b, [s], 3.0, trig_cap=1 << 20), lambda: mf.chisq_series(b, s, [0, 1], p=8),
                lambda: mf.synth_segment(np.zeros(1 << 20), 1 << 20, 4096.0)):
    L.mf_debug_alloc_limit(1 << 16)
    try:
        refused()
        raise SystemExit("not refused")
    except mf.MFError as e:
        assert e.code == mf._native.MF_ENOMEM, e
    L.mf_debug_alloc_limit(-1)
    mf.cluster_triggers(trig, nt, b.n, 1, s.N, 40)
    torch.cuda.synchronize()
""")


GRAPH = """
def loud(lg, seed):     # loudest rho about 4 .. 7
    g = torch.Generator(device="cuda").manual_seed(seed)
    return mf.Segment(70.0 * torch.randn(1 << lg, dtype=torch.float32, device="cuda", generator=g), 4096.0)

def run(b, segs):
    return mf.filter_bank(b, segs, 3.5, trig_cap=1 << 16)

def host(out):
    torch.cuda.synchronize()
    n = int(out[2].item())
    return n, out[0].cpu().numpy().tobytes(), out[1][:n].cpu().numpy().tobytes()

def alone_allocates_nothing(call):
    # the hook fails the next allocation, whoever makes it: still armed afterwards
    L.mf_debug_fail_alloc(0)
    out = call()
    try:
        bank()
        raise SystemExit("the call allocated")
    except mf.MFError as e:
        assert e.code == mf._native.MF_ENOMEM
    finally:
        L.mf_debug_fail_alloc(-1)
    return out
"""


@pytest.mark.parametrize("captured", ["[s[0]]", "s[:2]", "s"])
def test_calls_after_a_capture_keep_its_workspace(captured):
    """A graph of short segments, captured after calls on single ones: eager
    calls on several allocate nothing, so its replays stay valid."""
    _child(GRAPH + """
s = [loud(lg, lg) for lg in (15, 12, 13)]
ref = host(run(bank(20), s))
assert 0 < ref[0] <= 1 << 16
b = bank(20)
for one in s:
    run(b, [one])
part = %s
want = host(run(bank(20), part))
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    out = run(b, part)
for _ in range(2):
    assert host(alone_allocates_nothing(lambda: run(b, s))) == ref
    out[0].zero_(); out[1].zero_()
    g.replay()
    assert host(out) == want
assert b.check() == 0
""" % captured)


def test_no_room_for_segments_together():
    """The grouped workspace cannot be had: one after the other, in the one that
    is there, and later calls do not try again."""
    _child(GRAPH + """
s = [loud(lg, lg) for lg in (15, 12, 13)]
ref = host(run(bank(20), s))
assert 0 < ref[0] <= 1 << 16
for k in range(13):                  # every allocation of the larger workspace
    b = bank(20)
    for one in s:
        run(b, [one])
    torch.cuda.synchronize()
    L.mf_debug_fail_alloc(k)
    assert host(run(b, s)) == ref, k
    L.mf_debug_fail_alloc(-1)
    assert host(alone_allocates_nothing(lambda: run(b, s))) == ref, k
    assert b.check() == 0
""")


@pytest.mark.parametrize("cond", ["fp64", "fp32"])
def test_refresh_keeps_one_exchange(cond):
    """The first refresh of a segment of 2^22 samples keeps its exchange of 32 MB
    and nothing else; FP32 conditioning forms the spectrum in the weights' place."""
    _child("""
s, other = segment(22), segment(22, seed=2)
x = torch.randn(1 << 22, dtype=torch.float32, device="cuda")
for one in (other, s):
    one.set_conditioning("%s")
other.refresh(x)                    # the kernels are loaded
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
s.refresh(x)
torch.cuda.synchronize()
assert free - torch.cuda.mem_get_info()[0] <= 34 * MB
b = bank()
one = [t.cpu() for t in mf.filter_bank(b, [s], 0.1, trig_cap=1 << 10)]
s.refresh(x)
two = [t.cpu() for t in mf.filter_bank(b, [s], 0.1, trig_cap=1 << 10)]
assert torch.equal(one[0].view(torch.int32), two[0].view(torch.int32)) and torch.equal(one[2], two[2])
""" % cond)
