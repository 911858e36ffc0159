"""The batched solver's default launch shape when there are more problems than
SMs (256 threads at floor(1/eps) > 20, else by the largest problem), against
the oracle on the largest problem and a few others."""
import numpy as np
import pytest

import oracle
from paper_2203_03732_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [0.05, 0.04, 0.003])
@pytest.mark.parametrize("n_max", [701, 1300])
def test_more_problems_than_sms(n_max, eps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as prot
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = np.array([5 + i % 40 for i in range(sms)] + [n_max, 300], np.int32)
    mats = [W.assignment_euclid_2d(int(n), 200 + i) for i, n in enumerate(sizes)]
    got = prot.assign_batched(torch.from_numpy(np.concatenate([m.ravel() for m in mats])).cuda(), sizes, eps)
    off = np.concatenate([[0], np.cumsum(sizes)])
    for i in (0, 1, 39, len(sizes) - 2, len(sizes) - 1):
        ref = oracle.assign(mats[i], eps)
        for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
            assert np.array_equal(got[k][off[i]:off[i + 1]].cpu().numpy(), ref[k]), (i, k)
        assert abs(float(got["costs"][i]) - ref["cost"]) <= 1e-12 * abs(ref["cost"])
