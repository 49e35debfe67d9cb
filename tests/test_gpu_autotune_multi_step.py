"""The autotuners and the multi-step kernel: the time they report is that of the way a long call then
takes, that way stays the multi-step kernel where it is faster (FP32 64^3 x 8: by a third), and a batch made from
a level whose shape was set keeps to that shape."""
import pytest
import torch

from paper_2608_23786_gb300 import Ensemble, mclbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)


def _ms(stream, call, n):
    call()
    a, z = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    a.record(stream)
    call()
    z.record(stream)
    z.synchronize()
    return a.elapsed_time(z) / n


@pytest.mark.parametrize("pattern", ["pull", "aa"])
def test_the_context_tuner_reports_what_a_long_call_takes(pattern):
    e = Ensemble(64, 8, Re=800.0, Ma=0.025, pattern=pattern).init()
    best = mclbm.mclbm_autotune(e.ctx, 2)[3]
    assert e.steps_taken == 0
    before = mclbm.mclbm_get_step_launches(e.ctx)[1]
    ms = _ms(e.stream, lambda: e.step(48), 48)
    assert mclbm.mclbm_get_step_launches(e.ctx)[1] == before + 96
    assert best <= 1.2 * ms  # a launch per step takes 1.4 times as long
    ref = Ensemble(64, 8, Re=800.0, Ma=0.025, pattern=pattern).init()
    for _ in range(96):
        ref.step(1)
    assert torch.equal(e.populations(7), ref.populations(7))


def test_the_batch_tuner_reports_what_a_long_call_takes():
    s = torch.cuda.Stream()
    lev = [Ensemble(16 << k, M, Re=200.0 * 4**k, Ma=0.05 / 2**k, stream=s).init() for k, M in enumerate((8, 4, 4))]
    b = mclbm.mclbm_batch_create([e.ctx for e in lev], [1, 4, 16])
    try:
        best = mclbm.mclbm_batch_autotune(b, 1)[3]
        before = mclbm.mclbm_get_step_launches(lev[2].ctx)[1]
        ms = _ms(s, lambda: mclbm.mclbm_batch_step(b, 8), 8)
        assert mclbm.mclbm_get_step_launches(lev[2].ctx)[1] == before + 2 * 8 * 16
        assert best <= 1.2 * ms
    finally:
        mclbm.mclbm_batch_destroy(b)


def test_a_batch_takes_the_shape_that_was_set_on_its_first_level():
    s = torch.cuda.Stream()
    lev = [Ensemble(32, 4, Re=400.0, Ma=0.05, stream=s).init() for _ in range(2)]
    mclbm.mclbm_set_launch(lev[0].ctx, 2, 128, 2)
    b = mclbm.mclbm_batch_create([e.ctx for e in lev], [1, 16])
    try:
        mclbm.mclbm_batch_step(b, 2)
        assert mclbm.mclbm_get_step_launches(lev[1].ctx) == (0, 0)
        ref = Ensemble(32, 4, Re=400.0, Ma=0.05).init()
        for _ in range(32):
            ref.step(1)
        assert torch.equal(lev[1].populations(3), ref.populations(3))
    finally:
        mclbm.mclbm_batch_destroy(b)
