"""Rounding in groups of columns: rows on every alignment, widths around the
kernels' chunks, costs on and next to multiples of eps, and points of every
kernel form (2-D, 3-D, any dimension; scales near the ends of FP32), against
the oracle.  Duals and matching of a solve change with any rounded cost."""
import numpy as np
import pytest

import oracle
from oracle import points as OP

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


KEYS = ("row_to_col", "col_to_row", "y_row", "y_col")


def near_multiples(shape, eps, dtype, seed):
    """A third of the costs on a multiple of eps or one ulp beside it, with 0,
    -0.0, 1 and a subnormal among them; the rest uniform."""
    g = np.random.default_rng(seed)
    C = g.random(shape).astype(dtype)
    k = (g.integers(0, int(1 / eps) + 1, shape) * eps).astype(dtype)
    side = g.integers(-1, 2, shape)
    k = np.where(side < 0, np.nextafter(k, dtype(0)), np.where(side > 0, np.nextafter(k, dtype(2)), k))
    C = np.clip(np.where(g.random(shape) < 1 / 3, k, C), 0, 1).astype(dtype)
    C[0, :4] = [0.0, -0.0, 1.0, np.finfo(dtype).tiny / 4]
    return C


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("shift,cols", [(0, 512), (0, 128), (1, 127), (1, 513), (2, 257), (3, 1023)])
@pytest.mark.parametrize("eps", [0.01, 0.003])
def test_rows_on_every_alignment(prot, dtype, shift, cols, eps):
    import torch
    rows = 60
    wide = near_multiples((rows, cols + shift), eps, dtype, cols + shift)
    got = prot.assign(torch.from_numpy(wide).cuda()[:, shift:], eps)
    ref = oracle.assign(np.ascontiguousarray(wide[:, shift:]), eps)
    for k in KEYS:
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("eps", [0.01, 0.003])
def test_packed_problems_on_every_alignment(prot, dtype, eps):
    import torch
    sizes = np.array([5, 127, 3, 129, 64, 1, 255, 31], np.int32)
    mats = [near_multiples((n, n), eps, dtype, 10 + n) if n > 3 else np.full((n, n), 0.5, dtype) for n in sizes]
    got = prot.assign_batched(torch.from_numpy(np.concatenate([m.ravel() for m in mats])).cuda(), sizes, eps)
    off = 0
    for m, n in zip(mats, sizes):
        ref = oracle.assign(m, eps)
        for k in KEYS:
            assert np.array_equal(got[k][off:off + n].cpu().numpy(), ref[k]), (n, k)
        off += int(n)


@pytest.mark.parametrize("dim", [1, 2, 3, 4])
@pytest.mark.parametrize("squared", [True, False])
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e15])
@pytest.mark.parametrize("eps", [0.1, 0.003])
def test_points_of_every_form(prot, dim, squared, scale, eps):
    """Coordinates on a coarse lattice (distances repeat, many costs land on
    multiples of eps) and off it; scales whose squared distances leave the
    estimate's range take the exact way."""
    import torch
    g = np.random.default_rng(dim)
    n, m = 61, 77
    X = np.round(g.random((n + m, dim)) * 20) / 20
    X[::2] += 1e-3 * g.random((len(X[::2]), dim))
    X = (X * scale).astype(np.float32)
    XB, XA = np.ascontiguousarray(X[:n]), np.ascontiguousarray(X[n:])
    metric = "sqeuclidean" if squared else "euclidean"
    ref = OP.assign_points(XA, XB, eps, squared)
    got = prot.assign_points(torch.from_numpy(XA).cuda(), torch.from_numpy(XB).cuda(), eps, metric=metric)
    for k in KEYS:
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    sizes = np.array([n, 9, m - 16], np.int32)  # B = first points, A = last points of the same pool
    A, B = X[-int(sizes.sum()):], X[:int(sizes.sum())]
    got = prot.assign_batched_points(torch.from_numpy(np.ascontiguousarray(A)).cuda(),
                                     torch.from_numpy(np.ascontiguousarray(B)).cuda(), sizes, eps, metric=metric)
    off = 0
    for n_i in sizes:
        ref = OP.assign_points(np.ascontiguousarray(A[off:off + n_i]), np.ascontiguousarray(B[off:off + n_i]), eps,
                               squared)
        for k in KEYS:
            assert np.array_equal(got[k][off:off + n_i].cpu().numpy(), ref[k]), (n_i, k)
        off += int(n_i)
