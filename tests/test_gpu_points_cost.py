"""The cost of a points solve, bit for bit: 1024 strided partial sums and a
halving tree, at row counts whose last partial row ends inside a warp, with
another solve's partial sums left in the workspace."""
import numpy as np
import pytest

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


def matched_cost(A, B, mate, squared):
    d = np.zeros(len(B))
    for k in range(B.shape[1]):
        t = B[:, k].astype(np.float64) - A[mate, k].astype(np.float64)
        d = d + t * t
    if not squared:
        d = np.sqrt(d)
    part = np.zeros(1024)
    for s in range(0, len(d), 1024):
        c = d[s:s + 1024]
        part[:len(c)] = part[:len(c)] + c
    w = 512
    while w:
        part[:w] = part[:w] + part[w:2 * w]
        w //= 2
    return part[0]


@pytest.mark.parametrize("n", [2049, 2064, 3071, 4097])
@pytest.mark.parametrize("metric", ["euclidean", "sqeuclidean"])
def test_cost_bits(prot, n, metric):
    import torch
    ws = prot.Workspace()
    for seed in range(6):
        A, B = W.points_uniform(n, n, 2, 100 + seed, dtype=np.float32)
        B = B * np.float32(1 + seed)  # another scale: stale sums would show
        got = prot.assign_points(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), 0.2, metric=metric, ws=ws)
        want = matched_cost(A, B, got["row_to_col"].cpu().numpy(), metric == "sqeuclidean")
        assert float(got["cost"]) == want
