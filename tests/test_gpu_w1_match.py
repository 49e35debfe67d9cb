"""The warp assignment kernel of the two-point W1 at the edges of its column counts per lane (L = 32,
64, 128, 256 atoms per side) and just beyond, equal and repeated atoms, against the oracle's
assignment.  Tolerance: the plan is optimal for costs from FP32 atoms (relative error ~1e-7 per
cost) and its cost is summed in FP64, so each pair is within 2e-6 of the exact optimum."""
import pytest
import torch

import ensemble_inputs as gen
from oracle import stats
from paper_2608_23786_gb300 import mclbm

pytestmark = pytest.mark.gpu
pytest.importorskip("scipy")

RTOL = 2e-6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)


def _gpu(ua, ub, vector):
    G = ua.shape[1]
    da, db = (torch.as_tensor(u, device="cuda").contiguous() for u in (ua, ub))
    nb = mclbm.mclbm_w1_2pt_work_bytes(ua.shape[0], ub.shape[0], G, vector)
    work = torch.empty(nb, dtype=torch.uint8, device="cuda")
    per = torch.empty(G * (G + 1) // 2 * (1 if vector else 3), dtype=torch.float64, device="cuda")
    W = mclbm.mclbm_w1_2pt(da.data_ptr(), ua.shape[0], db.data_ptr(), ub.shape[0], G, vector, work.data_ptr(), nb,
                           torch.cuda.current_stream().cuda_stream, per.data_ptr())
    return W, per.cpu().numpy()


@pytest.mark.parametrize("MA,MB", [(1, 1), (2, 2), (31, 31), (32, 32), (33, 33), (64, 64), (65, 65), (128, 128),
                                   (129, 129), (256, 256), (257, 257), (96, 32), (85, 255)])
@pytest.mark.parametrize("vector", [1, 0])
def test_edges_of_the_warp_kernel(MA, MB, vector):
    ua = gen.uniform(300 + MA, (MA, 2, 3))
    ub = gen.uniform(700 + MB, (MB, 2, 3)) * 1.2 + 0.05
    W, per = _gpu(ua, ub, vector)
    Wref, Dref = stats.w1_two_point(ua, ub, vector=bool(vector), per_pair=True)
    scale = abs(Dref).max()
    assert (abs(per - Dref.ravel()) <= RTOL * abs(Dref.ravel()) + 1e-14 * scale).all()
    assert abs(W - Wref) <= RTOL * Wref


def test_coinciding_atoms_cost_nothing():
    ua = gen.uniform(9, (70, 2, 3))
    ua[35:] = ua[:35]  # every atom twice
    W, per = _gpu(ua, ua[::-1].copy(), 1)
    assert W == 0.0 and (per == 0.0).all()
