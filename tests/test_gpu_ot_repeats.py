"""Transport solves repeat: grants to empty lists, evictions and columns shared
by many proposers give the oracle's duals and plan on every one of several
solves in the same workspace."""
import numpy as np
import pytest

from oracle import ot as O
from paper_2203_03732_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nB,nA,eps", [(90, 33, 0.1), (33, 400, 0.05)])
def test_every_solve_gives_the_oracles_plan(nB, nA, eps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    import paper_2203_03732_gb300 as prot
    C, nu, mu = W.ot_euclid_2d(nB, nA, 7)
    ref = O.ot(C, nu, mu, eps)
    Ct, nut, mut = (torch.from_numpy(x).cuda() for x in (C, nu, mu))
    ws = prot.Workspace()
    for _ in range(20):
        r = prot.ot(Ct, nut, mut, eps, ws=ws)
        dense = np.zeros((nB, nA))
        dense[r["plan_row"].cpu().numpy(), r["plan_col"].cpu().numpy()] = r["plan_mass"].cpu().numpy()
        assert np.array_equal(dense, ref["mass"])
        assert np.array_equal(r["y_sup"].cpu().numpy(), ref["F"])
        assert np.array_equal(r["dem_lo"].cpu().numpy(), ref["clo"])
        assert np.array_equal(r["dem_hi"].cpu().numpy(), ref["chi"])
