"""The one-CTA solver of small problems and its take-over from the grid, against
the oracle: matching, duals, cost, phase and round counts and entries examined,
at the limits of its storage types, row counts and round numbers."""
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


def check(prot, C, eps, ctas=None):
    import torch
    got = prot.assign(torch.from_numpy(C).cuda(), eps)
    ref = oracle.assign(C, eps, mode=oracle.MODE_EVICT_RESUME)
    for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    st = got["stats"]
    for k in ("phases", "rounds", "free_at_stop", "threshold"):
        assert st[k] == ref["stats"][k], k
    assert st["cells_examined"] == ref["stats"]["scanned"]
    # FP64 sums of at most 2500 costs in [0, 1] in another order
    assert abs(float(got["cost"]) - ref["cost"]) <= 2500 * 2.0 ** -53 * ref["cost"]
    if ctas is not None:
        assert st["loop_ctas"] == ctas


# floor(1/eps) 100 (bytes, plain add), 142 (bytes with carries), 333 (16 bits)
@pytest.mark.parametrize("form", ["solo", "hand"])
@pytest.mark.parametrize("nB,nA", [(1, 1), (31, 32), (33, 33), (500, 545), (1000, 1000)])
@pytest.mark.parametrize("eps", [0.01, 0.007, 0.003])
def test_forms_and_storage_types(prot, monkeypatch, form, nB, nA, eps):
    monkeypatch.setenv("PR_PHASE_MODE", form)
    check(prot, W.assignment_euclid_2d(nB, 300 + nB, n_a=nA), eps, 1 if form == "solo" else None)


@pytest.mark.parametrize("n", [256, 257, 512, 513, 2500])
@pytest.mark.parametrize("eps", [0.05, 0.01])
def test_default_choice_around_its_limits(prot, n, eps):
    """The sizes on either side of the choice between one CTA, the grid with a
    take-over, and (eps = 0.05 at the largest) the grid alone."""
    check(prot, W.assignment_euclid_2d(n, 40 + n), eps)


@pytest.mark.parametrize("form", ["solo", "hand"])
def test_rounds_past_their_16_bit_numbers(prot, monkeypatch, form):
    """84,334 phases: the round numbers are renewed on the way."""
    monkeypatch.setenv("PR_PHASE_MODE", form)
    check(prot, W.assignment_euclid_2d(33, 3), 5e-5)


@pytest.mark.parametrize("eps", [0.75, 0.3])
def test_crowded_rounds(prot, monkeypatch, eps):
    """Most edges admissible: rounds of many rows that lose the same column
    (a lane per row), then rounds of few."""
    monkeypatch.setenv("PR_PHASE_MODE", "solo")
    g = np.random.default_rng(5)
    check(prot, g.random((700, 731)), eps, 1)
    check(prot, np.round(g.random((300, 300)) * 4) / 4, eps, 1)


@pytest.mark.parametrize("nB,nA,eps", [(400, 400, 0.1), (1000, 1000, 0.1), (1000, 1010, 0.3), (1024, 1024, 0.05)])
@pytest.mark.parametrize("squared", [True, False])
def test_take_over_inside_a_phase(prot, nB, nA, eps, squared):
    """One phase of many rounds (squared distances: over a hundred): the grid
    runs its first 16 rounds, one CTA the rest, with the keys, won columns,
    losers and queued rows of the unfinished phase."""
    A, B = W.points_uniform(nA, nB, 2, 17 + nB)
    check(prot, W.pairwise_cost(A, B, squared=squared), eps)


@pytest.mark.parametrize("form", ["solo", "hand"])
@pytest.mark.parametrize("nB,nA,eps", [(33, 33, 5e-5), (300, 300, 0.003), (500, 545, 0.007), (900, 900, 0.01)])
def test_sequential_greedy_on_one_cta(prot, monkeypatch, form, nB, nA, eps):
    """Every storage type, and phase tags past 2^16 (84,000 phases)."""
    import torch
    monkeypatch.setenv("PR_PHASE_MODE", form)
    C = W.assignment_euclid_2d(nB, 3 if nB == 33 else 500 + nB, n_a=nA)
    got = prot.assign(torch.from_numpy(C).cuda(), eps, rule="sequential")
    ref = oracle.assign(C, eps, mode=oracle.MODE_SEQUENTIAL)
    for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    assert got["stats"]["phases"] == ref["stats"]["phases"]
    assert got["stats"]["free_at_stop"] == ref["stats"]["free_at_stop"]
