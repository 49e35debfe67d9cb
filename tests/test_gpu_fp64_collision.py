"""The FP64 collision on strongly non-equilibrium states (populations up to 30% off the weights, at
three density scales) against the oracle's, one step.  Bound: the update is f - omega Ds - beta Dh with
|beta| below about 5 here and some 50 roundings per value, 5 * 50 * 1.1e-16 < 3e-14 of the largest
population; 1e-12 relative per population is the repository's FP64 bound."""
import numpy as np
import pytest
import torch

import ensemble_inputs as gen
import oracle
from gpu_helpers import lib_populations, oracle_to_lib
from paper_2608_23786_gb300 import Ensemble, mclbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("N,M", [(8, 1), (16, 2)])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e3])
def test_one_step_from_a_random_state(lattice, N, M, scale):
    mclbm.load(build_if_missing=True, lattice=lattice)
    _, w, _ = oracle.lattice(lattice)
    f = scale * w[None, :, None, None, None] * (1 + 0.3 * gen.uniform(17 + N, (M, lattice, N, N, N)))
    ens = Ensemble(N, M, Re=100.0, Ma=0.05, precision="fp64", lattice=lattice).init()
    for m in range(M):
        ens.set_populations(torch.from_numpy(oracle_to_lib(f[m]).copy()), m)
    ens.step(1)
    ref = np.ascontiguousarray(f)
    oracle.run(ref, oracle.units(N, 100.0, 0.05)["omega"], 1)
    got = lib_populations(ens)
    assert np.max(np.abs(got - ref) / (scale * w[None, :, None, None, None])) <= 1e-12
