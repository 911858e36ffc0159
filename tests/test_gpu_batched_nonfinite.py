"""Batched costs from points with coordinates that make a distance NaN or
infinite: the call reports PR_ERR_INVALID, and an asynchronous loss over such
clouds, and its gradients, are NaN."""
import numpy as np
import pytest

from paper_2203_03732_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# a problem larger than the bad one runs before it on the same CTA's memory;
# 33 and 45 columns leave padding columns beside real ones
SIZES = np.array([90, 33, 45], np.int32)


@pytest.fixture(scope="module")
def prot():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as P
    return P


def clouds(dim, bad):
    XA, XB = (x.copy() for x in W.points_uniform(int(SIZES.sum()), int(SIZES.sum()), dim, 5, dtype=np.float32))
    first, last = int(SIZES[0]), int(SIZES[:2].sum())
    if bad == "one nan":
        XB[first + 7, dim - 1] = np.nan
    elif bad == "all nan":
        XB[first:last] = np.nan
    elif bad == "inf":
        XA[first + 3, 0] = np.inf
    else:  # finite, but the squared distance overflows
        XA[first + 3, 0] = 3e38
    return XA, XB


@pytest.mark.parametrize("dim", [2, 3, 5])
@pytest.mark.parametrize("bad", ["one nan", "all nan", "inf", "overflow"])
@pytest.mark.parametrize("metric,eps", [("sqeuclidean", 0.1), ("euclidean", 0.005), ("sqeuclidean", 0.003)])
def test_reported(prot, dim, bad, metric, eps):
    import torch
    XA, XB = (torch.from_numpy(x).cuda() for x in clouds(dim, bad))
    with pytest.raises(prot.PrError) as e:
        prot.assign_batched_points(XA, XB, SIZES, eps, metric=metric)
    assert e.value.status == -1
    got = prot.assign_batched_points(XA, XB, SIZES, eps, metric=metric, sync=False)
    with pytest.raises(prot.PrError):
        prot.ws_status()
    assert torch.isnan(got["costs"]).all()


@pytest.mark.parametrize("dim", [2, 3, 4])
def test_loss_and_gradients_are_nan(prot, tmp_path, monkeypatch, dim):
    import torch
    monkeypatch.setenv("PROT_TUNE_CACHE", str(tmp_path / "tune.json"))
    X, Y = (torch.from_numpy(x).cuda() for x in W.cloud_pairs_normal(3, 70, dim, seed=2))
    prot.assignment_loss(X, Y, 0.1)  # finite clouds first: the launch shape is known below
    X[1, 4, 0] = float("nan")
    X.requires_grad_(True)
    Y.requires_grad_(True)
    loss = prot.assignment_loss(X, Y, 0.1)
    gX, gY = torch.autograd.grad(loss.sum(), (X, Y))
    assert torch.isnan(loss).all() and torch.isnan(gX).all() and torch.isnan(gY).all()


def test_unsolved_problems_have_indices_in_range(prot):
    """After an error an asynchronous caller may still index with the mates."""
    import torch
    XA, XB = (torch.from_numpy(x).cuda() for x in clouds(3, "one nan"))
    got = prot.assign_batched_points(XA, XB, SIZES, 0.1, sync=False)
    off = 0
    for n in SIZES:
        want = torch.arange(int(n), dtype=torch.int32, device="cuda")
        for k in ("row_to_col", "col_to_row"):
            assert torch.equal(got[k][off:off + int(n)], want), k
        off += int(n)
