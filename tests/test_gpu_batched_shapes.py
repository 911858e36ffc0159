"""The batched solver's default launch shapes (threads per CTA by the largest
problem) against the oracle, problem by problem."""
import numpy as np
import pytest

import oracle
from paper_2203_03732_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def prot():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as P
    return P


@pytest.mark.parametrize("n_max", [300, 401, 701])
def test_default_batched_shapes(prot, n_max):
    """Default launch shapes by the largest problem (128, 256, 512 threads)."""
    import torch
    sizes = np.array([n_max, 1, 2, 31, 64, 257, 300, n_max // 2], np.int32)
    mats = [W.assignment_euclid_2d(int(n), 70 + i) for i, n in enumerate(sizes)]
    got = prot.assign_batched(torch.from_numpy(np.concatenate([m.ravel() for m in mats])).cuda(), sizes, 0.02)
    off = 0
    for i, n in enumerate(sizes):
        ref = oracle.assign(mats[i], 0.02)
        for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
            assert np.array_equal(got[k][off:off + n].cpu().numpy(), ref[k]), (i, k)
        off += int(n)
