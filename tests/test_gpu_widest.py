"""The widest problems a single solve takes: 89,808 columns, limited by the
key copy in shared memory.  One column more is refused."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N_COLS = 89808


@pytest.fixture(scope="module")
def prot():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as P
    return P


@pytest.mark.parametrize("rule,mode", [("lowest", oracle.MODE_EVICT_RESUME), ("offset", oracle.MODE_OFFSET)])
@pytest.mark.parametrize("eps", [0.1, 0.003])
def test_widest_accepted(prot, rule, mode, eps):
    import torch
    C = np.random.default_rng(3).random((5, N_COLS)).astype(np.float32)
    got = prot.assign(torch.from_numpy(C).cuda(), eps, rule=rule)
    ref = oracle.assign(C, eps, mode=mode)
    for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


def test_next_size_refused(prot):
    import torch
    with pytest.raises(prot.PrError, match=f"max {N_COLS}") as e:
        prot.assign(torch.zeros((1, N_COLS + 1), device="cuda"), 0.1)
    assert e.value.status == -1
