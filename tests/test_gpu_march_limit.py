"""Which steps run in the multi-step kernel (the context counts them), calls split into several launches
(mclbm_set_step_limit) against one launch and against a launch per step, bit for bit, in every mode of the
kernel: in place under AA, in place in a pull lattice, and through the states of the adjoint's segments."""
import numpy as np
import pytest
import torch

import ensemble_inputs as gen
from paper_2608_23786_gb300 import Ensemble, mclbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)
    mclbm.load(build_if_missing=True, lattice=27)


def _ensemble(N, M, precision, pattern, lattice, limit=0):
    e = Ensemble(N, M, Re=12.5 * N, Ma=1.6 / max(N, 32), precision=precision, pattern=pattern, lattice=lattice).init()
    mclbm.mclbm_set_step_limit(e.ctx, limit)
    return e


def _same(a, b):
    mclbm.mclbm_device_status(a.ctx)
    assert a.steps_taken == b.steps_taken
    for m in sorted({0, a.M // 2, a.M - 1}):
        assert torch.equal(a.populations(m), b.populations(m)), m


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("precision,N,M,steps", [("fp32", 32, 7, 29), ("fp32", 64, 9, 29), ("fp16", 32, 4, 29),
                                                 ("fp64", 32, 2, 29)])
def test_split_calls_give_the_same_bits(precision, N, M, steps, pattern, lattice):
    one, split, single = (_ensemble(N, M, precision, pattern, lattice, k) for k in (0, 8, 1))
    for e in (one, split, single):
        e.step(steps)
    whole = steps & ~1 if pattern == "pull" else steps
    assert mclbm.mclbm_get_step_launches(one.ctx) == (1, whole)
    rest = steps - 24  # a launch of one step is none of the multi-step kernel's
    assert mclbm.mclbm_get_step_launches(split.ctx) == (4, 24 + (rest & ~1 if pattern == "pull" else rest))
    assert mclbm.mclbm_get_step_launches(single.ctx) == (0, 0)
    _same(split, one)
    _same(single, one)


@pytest.mark.parametrize("precision,N,M,served", [("fp32", 8, 1, 12), ("fp32", 32, 7, 6), ("fp32", 64, 2, 3),
                                                  ("fp16", 32, 1, 6), ("fp64", 32, 1, 16), ("fp64", 32, 2, 8)])
def test_short_calls_and_chosen_shapes_are_single_launches(precision, N, M, served):
    e = _ensemble(N, M, precision, "aa", 19)
    e.step(served - 1)
    assert mclbm.mclbm_get_step_launches(e.ctx) == (0, 0)
    e.step(served)
    assert mclbm.mclbm_get_step_launches(e.ctx) == (1, served)
    for parity in (0, 1):
        kind, vec, block = mclbm.mclbm_get_launch_parity(e.ctx, parity)
        mclbm.mclbm_set_launch_parity(e.ctx, parity, vec, block, kind)
    e.step(served)
    assert mclbm.mclbm_get_step_launches(e.ctx) == (1, served)


def test_a_long_call_is_several_launches():
    """160,000 steps of about 14 us: a launch lasts about a second."""
    e = _ensemble(8, 1, "fp64", "aa", 19)
    e.step(160000)
    launches, steps = mclbm.mclbm_get_step_launches(e.ctx)
    assert steps == 160000 and 3 <= launches <= 5
    mclbm.mclbm_device_status(e.ctx)


def _gradient(N, M, precision, lattice, steps, ckpt, limit):
    e = Ensemble(N, M, Re=200.0, Ma=0.05, precision=precision, lattice=lattice).init(gen.draw_params(5, M))
    mclbm.mclbm_set_step_limit(e.ctx, limit)
    need = mclbm.mclbm_grad_required_bytes(e.ctx, steps, ckpt)
    buf = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    J, G = mclbm.mclbm_grad(e.ctx, 0, steps, ckpt, (buf.data_ptr() + 255) // 256 * 256, need, M)
    return J, G, mclbm.mclbm_get_step_launches(e.ctx), e


# segments that the multi-step kernel takes (20 steps and more on small ensembles), two nodes per thread,
# four, and the D3Q27 run ahead in shared memory
@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("precision,N,M", [("fp32", 16, 3), ("fp32", 32, 5), ("fp32", 64, 2), ("fp16", 16, 3),
                                           ("fp16", 32, 5), ("fp64", 16, 3), ("fp64", 32, 2)])
def test_trajectories_give_the_gradient_of_single_launches(precision, N, M, lattice):
    steps, ckpt = 45, 20
    J1, G1, none, e1 = _gradient(N, M, precision, lattice, steps, ckpt, 1)
    assert none == (0, 0)
    for limit in (0, 6):
        J, G, (launches, taken), e = _gradient(N, M, precision, lattice, steps, ckpt, limit)
        # forward to 40 (the last, short segment keeps its 4 states) and the 19 states of two segments again
        assert launches >= 4 and taken >= 40 + 2 * 18
        assert np.array_equal(J, J1) and np.array_equal(G, G1)
        assert np.isfinite(G).all() and np.abs(G).max() > 0
        _same(e, e1)


@pytest.mark.parametrize("pattern", ["pull", "aa"])
def test_fp64_batch_level_by_level_equals_single_steps(pattern):
    pairs = [[_ensemble(8 << k, M, "fp64", pattern, 19) for _ in range(2)] for k, M in enumerate((4, 3, 2))]
    b = mclbm.mclbm_batch_create([a.ctx for a, _ in pairs], [1, 4, 16])
    try:
        mclbm.mclbm_batch_step(b, 2)
        assert mclbm.mclbm_get_step_launches(pairs[2][0].ctx) == (1, 32)
        mclbm.mclbm_set_step_limit(pairs[2][0].ctx, 1)  # the level with the work: sub-steps in one launch again
        mclbm.mclbm_batch_step(b, 1)
        assert mclbm.mclbm_get_step_launches(pairs[2][0].ctx) == (1, 32)
        for (x, y), sub in zip(pairs, (1, 4, 16)):
            for _ in range(3 * sub):
                y.step(1)
            _same(x, y)
    finally:
        mclbm.mclbm_batch_destroy(b)


@pytest.mark.parametrize("pattern", ["pull", "aa"])
@pytest.mark.parametrize("precision,M,by_level", [("fp32", 1, False), ("fp32", 64, True), ("fp64", 4, True)])
def test_small_levels_keep_a_launch_per_sub_step(precision, M, by_level, pattern):
    """Levels too small to be worth a launch of their own (8^3, 16^3, 32^3 of one sample, FP32) stay in one
    launch per sub-step; either way the levels end in the bits of single steps."""
    stream = torch.cuda.Stream()
    pairs = [[Ensemble(8 << k, M, Re=100.0 * 4**k, Ma=0.05 / 2**k, precision=precision, pattern=pattern, stream=stream).init()
              for _ in range(2)] for k in range(3)]
    b = mclbm.mclbm_batch_create([a.ctx for a, _ in pairs], [1, 4, 16])
    try:
        for _ in range(2):
            mclbm.mclbm_batch_step(b, 2)
        assert (mclbm.mclbm_get_step_launches(pairs[2][0].ctx)[0] > 0) == by_level
        for (x, y), sub in zip(pairs, (1, 4, 16)):
            for _ in range(4 * sub):
                y.step(1)
            _same(x, y)
    finally:
        mclbm.mclbm_batch_destroy(b)
