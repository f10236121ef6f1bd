"""The chi^2 series of a template is that template's alone: the same bits by
itself and in any list, however many CTAs share its tiles."""
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


def _case(mf, lg, n):
    import torch
    m = np.random.default_rng(lg).uniform(1.0, 6.0, (2, n))
    g = torch.Generator(device="cuda").manual_seed(lg)
    x = 70.0 * torch.randn(1 << lg, dtype=torch.float32, device="cuda", generator=g)
    return mf.Bank(m[0], m[1]), mf.Segment(x, 4096.0)


# lists long enough for one CTA per tile; shorter ones take clusters of two (from
# p = 3) and four (from p = 7) at each length; p + 1 not a multiple of the groups
@pytest.mark.parametrize("lg,n", [(10, 400), (11, 400), (12, 320), (13, 320), (14, 170), (15, 80), (16, 42), (17, 22),
                                  (18, 12), (19, 5), (21, 3)])
@pytest.mark.parametrize("p", [1, 2, 3, 6, 7, 16])
def test_same_bits_in_every_list(mf, lg, n, p):
    bank, seg = _case(mf, lg, n)
    many = mf.chisq_series(bank, seg, list(range(n)), p=p)[0].cpu().numpy().view(np.uint32)
    assert bank.check() == 0
    for k in sorted({1, max(1, n // 5), n // 2}):
        some = mf.chisq_series(bank, seg, list(range(n - k, n)), p=p)[0].cpu().numpy().view(np.uint32)
        assert np.array_equal(some, many[n - k:]), k


# the allocation limits leave room for some of the templates' p + 1 exchanges, for
# one template's, and for one band of one template's (1024-point rows need p + 1)
@pytest.mark.parametrize("lg,p", [(10, 1), (12, 16), (13, 2), (14, 3), (15, 7), (16, 6), (17, 16), (18, 5), (19, 4), (21, 8),
                                  (22, 3)])
def test_little_memory(mf, lg, p):
    import torch
    n = 3 if lg > 18 else 7
    bank, seg = _case(mf, lg, n)
    want, edges = (x.cpu().numpy() for x in mf.chisq_series(bank, seg, list(range(n)), p=p))
    L = mf._native.lib()
    one = 8 * seg.N * (p + 1)
    for limit in (3 * one, one + (1 << 16), 20 * seg.N + (1 << 16)):
        L.mf_debug_alloc_limit(limit)
        try:
            if lg in (19, 20) and limit < one:
                with pytest.raises(mf.MFError) as e:
                    mf.chisq_series(bank, seg, list(range(n)), p=p)
                assert e.value.code == mf._native.MF_ENOMEM
                continue
            got, ge = (x.cpu().numpy() for x in mf.chisq_series(bank, seg, list(range(n)), p=p))
        finally:
            L.mf_debug_alloc_limit(-1)
        assert bank.check() == 0
        assert np.array_equal(ge, edges) and np.array_equal(got.view(np.uint32), want.view(np.uint32)), limit
