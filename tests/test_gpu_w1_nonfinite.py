"""Two-point W1 of fields that hold a NaN or an infinity: NONFINITE for every solver (the warp kernel at
each of its column counts, the block solver for equal and unequal counts), the pairs that do not touch
the bad point keep their values, and the next call with finite fields works."""
import numpy as np
import pytest
import torch

import ensemble_inputs as gen
from paper_2608_23786_gb300 import mclbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)


def _call(ua, ub, vector):
    G = ua.shape[1]
    da, db = (torch.as_tensor(u, device="cuda").contiguous() for u in (ua, ub))
    nb = mclbm.mclbm_w1_2pt_work_bytes(ua.shape[0], ub.shape[0], G, vector)
    work = torch.empty(nb, dtype=torch.uint8, device="cuda")
    per = torch.zeros(G * (G + 1) // 2 * (1 if vector else 3), dtype=torch.float64, device="cuda")
    status = "OK"
    try:
        mclbm.mclbm_w1_2pt(da.data_ptr(), ua.shape[0], db.data_ptr(), ub.shape[0], G, vector, work.data_ptr(), nb,
                           torch.cuda.current_stream().cuda_stream, per.data_ptr())
    except mclbm.MclbmError as e:
        status = e.status
    return status, per.cpu().numpy()


@pytest.mark.parametrize("MA,MB", [(8, 8), (40, 40), (64, 32), (100, 100), (200, 200), (257, 257), (16, 15), (30, 7)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("side", [0, 1])
def test_nonfinite_atoms_are_reported(MA, MB, bad, side):
    G, point = 3, 1
    u = [gen.uniform(400 + MA, (MA, G, 3)), gen.uniform(500 + MB, (MB, G, 3)) + 0.1]
    for vector in (1, 0):
        status, clean = _call(u[0], u[1], vector)
        assert status == "OK" and np.isfinite(clean).all()
        v = [a.copy() for a in u]
        v[side][-1, point, 2] = bad
        status, per = _call(v[0], v[1], vector)
        assert status == "NONFINITE"
        touched = np.array([point in (i, j) for i in range(G) for j in range(i, G)])
        if vector:
            assert not np.isfinite(per[touched]).any()
            assert (per[~touched] == clean[~touched]).all()
        else:  # only the bad component
            per, ref = per.reshape(-1, 3), clean.reshape(-1, 3)
            assert not np.isfinite(per[touched, 2]).any()
            assert (per[~touched] == ref[~touched]).all() and (per[:, :2] == ref[:, :2]).all()
