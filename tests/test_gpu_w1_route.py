"""Two-point W1 of unequal sample counts with lcm <= 256 on both sides of the line between the warp
kernel (atoms repeated) and the block solver (nothing repeated), which depends on the counts and on the
number of problems: the same values, against the oracle's transport linear program.  Tolerance: as in
the other two-point tests, 2e-6 relative per pair (costs from FP32 atoms, summed in FP64)."""
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


# atoms repeated: always; always; from 171 (20, 16), 300 (64, 96), 534 (100, 40) and 2100 problems on (10, 7);
# never; never.  15 problems, 45 by components, and 630, 1890 by components; 2145 and 6435.
@pytest.mark.parametrize("MA,MB", [(50, 100), (24, 36), (20, 16), (64, 96), (100, 40), (10, 7), (12, 11), (16, 15)])
@pytest.mark.parametrize("G", [1, 5, 35, 65])
def test_both_routes_against_the_oracle(MA, MB, G):
    ua = gen.uniform(900 + MA, (MA, G, 3))
    ub = gen.uniform(950 + MB, (MB, G, 3)) * 1.2 + 0.05
    few = min(G, 4)
    for vector in (1, 0):
        _, per = _gpu(ua, ub, vector)
        _, Dref = stats.w1_two_point(ua[:, :few], ub[:, :few], vector=bool(vector), per_pair=True)
        got = per.reshape(-1, 1 if vector else 3)
        ref = Dref.reshape(-1, 1 if vector else 3)
        for i in range(few):
            for j in range(i, few):
                a, b = got[stats.pair_index(i, j, G)], ref[stats.pair_index(i, j, few)]
                assert (abs(a - b) <= RTOL * abs(b) + 1e-14 * abs(ref).max()).all(), (i, j, vector)
