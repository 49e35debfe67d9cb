"""A bounded device wait that gave up (the wait self-test stands in for the stepper's) is reported by
every call that returns results of the context, not by mclbm_device_status alone, and an initialisation or
a load clears it."""
import os

import numpy as np
import pytest
import torch

from paper_2608_23786_gb300 import Ensemble, mclbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)


def _ensemble(seed=1):
    return Ensemble(16, 3, Re=200.0, Ma=0.05, precision="fp32", seed=seed).init().step(14)


def _status(call):
    try:
        call()
    except mclbm.MclbmError as e:
        return e.status
    return "OK"


READERS = {
    "energy": lambda e, o: e.energy(),
    "enstrophy": lambda e, o: e.energy(enstrophy=True),
    "energy_mean_var": lambda e, o: e.energy_mean_var(),
    "spectrum": lambda e, o: e.spectrum(),
    "sf_trace": lambda e, o: e.sf_trace(),
    "sf_axes": lambda e, o: e.sf_axes(4),
    "w1": lambda e, o: e.w1(o),
    "w1_as_other": lambda e, o: o.w1(e),
    "check_finite": lambda e, o: e.check_finite(),
    "device_status": lambda e, o: mclbm.mclbm_device_status(e.ctx),
}


@pytest.mark.parametrize("name", READERS)
def test_readers_report_a_wait_that_gave_up(name):
    read, other, ens = READERS[name], _ensemble(2), _ensemble()
    assert _status(lambda: read(ens, other)) == "OK"
    mclbm.mclbm_selftest_timeout(ens.ctx)
    assert _status(lambda: read(ens, other)) == "TIMEOUT"
    assert "wait" in mclbm.mclbm_last_error()
    ens.init().step(14)
    assert _status(lambda: read(ens, other)) == "OK"
    assert _status(lambda: other.energy()) == "OK"


def test_save_writes_no_file_of_such_a_state_and_load_clears_it(tmp_path):
    ens = _ensemble()
    good, bad = (os.path.join(tmp_path, f) for f in ("good", "bad"))
    mclbm.mclbm_save(ens.ctx, good)
    f = ens.populations(2).clone()
    mclbm.mclbm_selftest_timeout(ens.ctx)
    assert _status(lambda: mclbm.mclbm_save(ens.ctx, bad)) == "TIMEOUT"
    assert not os.path.exists(bad)
    mclbm.mclbm_load(ens.ctx, good)
    assert _status(lambda: ens.energy()) == "OK" and torch.equal(ens.populations(2), f)


def test_gradient_reports_it():
    """A word set after the initialisation, as a wait of the forward run would leave it."""
    ens = Ensemble(8, 2, Re=100.0, Ma=0.05, precision="fp32").init()
    need = mclbm.mclbm_grad_required_bytes(ens.ctx, 16, 8)
    buf = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    ptr = (buf.data_ptr() + 255) // 256 * 256
    J, G = mclbm.mclbm_grad(ens.ctx, 0, 16, 8, ptr, need, 2)
    assert np.isfinite(J).all() and np.isfinite(G).all()
    ens.init()
    mclbm.mclbm_selftest_timeout(ens.ctx)
    assert _status(lambda: mclbm.mclbm_grad(ens.ctx, 0, 16, 8, ptr, need, 2)) == "TIMEOUT"


@pytest.mark.parametrize("lattice,N,M,pattern", [(19, 32, 7, "pull"), (19, 64, 9, "aa"), (27, 64, 2, "pull")])
def test_a_launch_that_finds_the_word_set_ends_and_is_reported(lattice, N, M, pattern):
    """The multi-step kernel's ways out: with the error word set its warps leave at their first long
    wait, in whatever part of the work; the call ends, the state is reported, and the next run is whole."""
    mclbm.load(build_if_missing=True, lattice=lattice)
    make = lambda: Ensemble(N, M, Re=12.5 * N, Ma=1.6 / 64, pattern=pattern, lattice=lattice).init()  # noqa: E731
    ref, ens = make(), make()
    mclbm.mclbm_set_step_limit(ref.ctx, 1)
    ref.step(40)
    mclbm.mclbm_selftest_timeout(ens.ctx)
    ens.step(40)
    assert _status(lambda: ens.energy()) == "TIMEOUT"
    ens.init().step(40)
    assert _status(lambda: ens.energy()) == "OK"
    assert mclbm.mclbm_get_step_launches(ens.ctx) == (2, 80)
    assert all(torch.equal(ens.populations(m), ref.populations(m)) for m in range(M))
