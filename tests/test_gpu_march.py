"""Calls of several steps on FP32 and (small) FP16 and FP64 storage (one launch of the multi-step kernel) against the same steps
taken one call at a time (a launch per step): the same bits, for both streaming patterns, one and
several tiles per plane, several planes per tile, windows and whole lattices in L2, even and odd
step counts and a state at an odd step."""
import pytest
import torch

from paper_2608_23786_gb300 import Ensemble, mclbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)


def _pair(N, M, precision="fp32", **kw):
    return [Ensemble(N, M, Re=12.5 * N, Ma=1.6 / max(N, 32), precision=precision, **kw).init() for _ in range(2)]


def _same(a, b):
    mclbm.mclbm_device_status(a.ctx)
    assert a.steps_taken == b.steps_taken
    for m in sorted({0, a.M // 2, a.M - 1}):
        assert torch.equal(a.populations(m), b.populations(m)), m


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("N,M,steps", [(8, 1, 12), (8, 131, 12), (8, 600, 5), (16, 3, 13), (32, 7, 17),
                                       (32, 12, 5), (64, 1, 6), (64, 9, 23), (128, 2, 7), (256, 1, 5)])
def test_several_steps_equal_single_steps(N, M, steps, pattern, lattice):
    a, b = _pair(N, M, pattern=pattern, lattice=lattice)
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    _same(a, b)


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("N,M,steps", [(8, 1, 7), (16, 3, 6), (32, 4, 8), (32, 7, 9), (64, 2, 6), (64, 3, 13),
                                       (128, 1, 12)])
def test_fp16_several_steps_equal_single_steps(N, M, steps, pattern, lattice):
    a, b = _pair(N, M, "fp16", pattern=pattern, lattice=lattice)
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    _same(a, b)


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("N,M,steps", [(8, 1, 16), (8, 131, 9), (16, 3, 17), (32, 1, 17), (32, 5, 8), (32, 16, 8)])
def test_fp64_several_steps_equal_single_steps(N, M, steps, pattern, lattice):
    a, b = _pair(N, M, "fp64", pattern=pattern, lattice=lattice)
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    _same(a, b)


@pytest.mark.parametrize("pattern", ["pull", "aa"])
def test_from_an_odd_step_and_in_turn_with_single_steps(pattern):
    a, b = _pair(64, 6, pattern=pattern)
    for n in (1, 5, 2, 1, 8):
        a.step(n)
    for _ in range(17):
        b.step(1)
    _same(a, b)


def test_a_chosen_shape_keeps_a_launch_per_step():
    a, b = _pair(32, 20)
    mclbm.mclbm_set_launch(b.ctx, 1, 128, 0)
    _same(a.step(14), b.step(14))


@pytest.mark.parametrize("precision,macro", [("fp32", 1), ("fp32", 3), ("fp16", 6)])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
def test_batch_level_by_level_equals_single_steps(precision, macro, pattern):
    """Levels that the multi-step kernel serves, and one (the coarsest, a few steps) that it does not."""
    pairs = [_pair(16 << k, M, precision, pattern=pattern) for k, M in enumerate((6, 3, 2))]
    b = mclbm.mclbm_batch_create([a.ctx for a, _ in pairs], [1, 4, 16])
    try:
        mclbm.mclbm_batch_step(b, macro)
        mclbm.mclbm_batch_step(b, 1)
        assert mclbm.mclbm_batch_macro_steps(b) == macro + 1
        for (x, y), sub in zip(pairs, (1, 4, 16)):
            for _ in range(sub * (macro + 1)):
                y.step(1)
            _same(x, y)
    finally:
        mclbm.mclbm_batch_destroy(b)
