"""mf_autotune times only schedules that the bank's phase form has."""
import json

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


@pytest.mark.parametrize("phase", ["MF_PHASE_FP64", "MF_PHASE_FP32"])
def test_no_persistent_candidate_without_its_phase(mf, tmp_path, phase):
    """Five exchange budgets times the rows and per-tile forms of pass 2: the
    persistent scheduler would run the per-batch path under another name."""
    import torch
    bank = mf.Bank([1.4, 2.0, 1.2], [1.3, 1.7, 1.2], phase_mode=getattr(mf, phase))
    seg = mf.Segment(70.0 * torch.randn(1 << 14, dtype=torch.float32, device="cuda"), 4096.0)
    before = [x.cpu().numpy().copy() for x in mf.filter_bank(bank, [seg], 3.5, trig_cap=1 << 16)]
    cache = tmp_path / "tuned.json"
    mf.autotune(bank, [seg], 3.5, repeats=1, cache_path=str(cache))
    tuned = json.loads(cache.read_text())
    assert tuned["scheduler"] == "batch" and tuned["candidates"] == 10
    after = [x.cpu().numpy() for x in mf.filter_bank(bank, [seg], 3.5, trig_cap=1 << 16)]
    n = int(before[2][0])
    assert n == int(after[2][0]) and np.array_equal(before[0].view(np.uint8), after[0].view(np.uint8))
    assert np.array_equal(before[1][:n].view(np.uint8), after[1][:n].view(np.uint8))
