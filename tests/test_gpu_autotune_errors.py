"""The launch-shape autotuner on batches with invalid costs: it reports the
error instead of a shape timed on stopped solves, and nothing is remembered."""
import ctypes
import os

import numpy as np
import pytest

from paper_2203_03732_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = np.array([40, 33], np.int32)


@pytest.fixture
def prot(tmp_path, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as P
    monkeypatch.setenv("PROT_TUNE_CACHE", str(tmp_path / "tune.json"))
    return P


def packed():
    import torch
    mats = [W.assignment_euclid_2d(int(n), 3) for n in SIZES]
    mats[1][5, 6] = 1.25
    return torch.from_numpy(np.concatenate([m.ravel() for m in mats])).cuda()


def test_entry_point_reports_the_error(prot):
    import torch
    from paper_2203_03732_gb300 import _lib
    L = _lib.load()
    C = packed()
    n_ptr = SIZES.ctypes.data_as(ctypes.c_void_p)
    out = prot._batched_outputs(torch, C.device, SIZES)
    ws = prot.Workspace().get(L.pr_assign_batched_workspace(len(SIZES), n_ptr))
    best, ms = _lib.PrBatchedTune(), ctypes.c_float()
    rc = L.pr_assign_batched_autotune(None, None, 0, 0, C.data_ptr(), _lib.PR_F64, len(SIZES), n_ptr, 0.1,
                                      out["row_to_col"].data_ptr(), out["col_to_row"].data_ptr(),
                                      out["y_row"].data_ptr(), out["y_col"].data_ptr(), out["costs"].data_ptr(),
                                      out["phases"].data_ptr(), ctypes.byref(best), ctypes.byref(ms), ws.data_ptr(),
                                      ws.numel(), None)
    assert rc == _lib.PR_ERR_INVALID


def test_nothing_is_remembered(prot):
    import torch
    C = packed()
    with pytest.raises(prot.PrError) as e:
        prot.assign_batched(C, SIZES, 0.1, tune="auto")
    assert e.value.status == -1
    got = prot.assign_batched(C, SIZES, 0.1, tune="auto", sync=False)
    assert torch.isnan(got["costs"]).all()
    X, Y = (torch.from_numpy(x).cuda() for x in W.cloud_pairs_normal(2, 50, 3, seed=1))
    X[0, 3, 1] = float("inf")
    assert torch.isnan(prot.assignment_loss(X, Y, 0.1)).all()
    assert not os.path.exists(os.environ["PROT_TUNE_CACHE"])
