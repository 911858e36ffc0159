"""Which form runs a solve by default: one CTA from the start or not, seen in
loop_ctas, and the sizes around the take-overs (test_cta_choice.py holds the
rule itself).  Results against the oracle each time."""
import numpy as np
import pytest

import oracle
from paper_2203_03732_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("row_to_col", "col_to_row", "y_row", "y_col")


@pytest.fixture(scope="module")
def prot():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as P
    return P


def solve(prot, C, eps):
    import torch
    got = prot.assign(torch.from_numpy(C).cuda(), eps)
    ref = oracle.assign(C, eps, mode=oracle.MODE_EVICT_RESUME)
    for k in KEYS:
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    assert got["stats"]["cells_examined"] == ref["stats"]["scanned"]
    return got["stats"]


@pytest.mark.parametrize("nB,nA,eps,one", [
    (384, 384, 0.01, True), (385, 385, 0.01, False), (64, 8000, 0.005, True), (64, 8000, 0.003, False),
    (300, 7000, 0.01, False), (300, 7000, 0.1, True), (384, 8000, 0.003, False), (384, 512, 0.003, True),
    (384, 513, 0.003, False), (200, 1000, 0.02, True), (201, 1000, 0.02, False)])
def test_one_cta_from_the_start(prot, nB, nA, eps, one):
    assert (solve(prot, W.assignment_euclid_2d(nB, 9, n_a=nA), eps)["loop_ctas"] == 1) == one


@pytest.mark.parametrize("nB,nA,eps,squared", [
    (1536, 1536, 0.1, True), (1537, 1537, 0.1, True),   # the largest taken over inside a phase, and the next
    (500, 600, 0.01, False), (3000, 3000, 0.01, False), (6399, 6399, 0.01, False),  # at 64 free rows (T = 5, 30, 63)
    (700, 8000, 0.003, False), (700, 8192, 0.003, False)])  # rows of 16,000 bytes; more columns than one CTA's state holds
def test_around_the_take_overs(prot, nB, nA, eps, squared):
    A, B = W.points_uniform(nA, nB, 2, 23)
    assert solve(prot, W.pairwise_cost(A, B, squared=squared), eps)["loop_ctas"] > 1


@pytest.mark.parametrize("nB,nA", [(4096, 4096), (4097, 4100)])
@pytest.mark.parametrize("eps", [0.1, 0.05, 0.04])
def test_phase_loop_with_and_without_fast_rounds(prot, nB, nA, eps):
    """floor(1/eps) <= 20 and more than 4096 rows: the loop without them."""
    solve(prot, W.assignment_euclid_2d(nB, 31, n_a=nA), eps)
