"""Rounding of matrices full of exact zeros and ones, with tiny and negative
zero costs among them, against the oracle; and every cost outside [0, 1] is
reported, wherever it lies in a group of columns."""
import numpy as np
import pytest

import oracle

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


def same(got, ref, off=0):
    for k in KEYS:
        n = len(ref[k])
        assert np.array_equal(got[k][off:off + n].cpu().numpy(), ref[k]), k


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("eps", [0.3, 0.1, 0.01, 0.003, 1 / 32766.5])
@pytest.mark.parametrize("cols", [96, 101])
def test_zeros_and_ones(prot, dtype, eps, cols):
    import torch
    g = np.random.default_rng(8)
    C = g.random((40, cols))
    w = g.random((40, cols))
    C = np.where(w < 0.3, 0.0, np.where(w < 0.6, 1.0, C)).astype(dtype)
    tiny = np.finfo(dtype).tiny
    special = np.array([-0.0, tiny, tiny / 4, 2.0 ** -126, 2.0 ** -127, 2.0 ** -128, eps / 4, eps, 1 - 2.0 ** -24],
                       dtype)
    C[w > 0.9] = special[g.integers(0, len(special), int((w > 0.9).sum()))]
    got = prot.assign(torch.from_numpy(C).cuda(), eps)
    same(got, oracle.assign(C, eps))
    sizes = np.array([40, 33, 5], np.int32)
    mats = [np.ascontiguousarray(C[:n, :n]) for n in sizes]
    got = prot.assign_batched(torch.from_numpy(np.concatenate([m.ravel() for m in mats])).cuda(), sizes, eps)
    off = 0
    for n, m in zip(sizes, mats):
        same(got, oracle.assign(m, eps), off)
        off += int(n)


def outside(dtype):
    one, zero = dtype(1), dtype(0)
    neg_nan = np.array([-1], np.int32 if dtype == np.float32 else np.int64).view(dtype)[0]
    return [np.nextafter(one, dtype(2)), dtype(1.5), np.nextafter(zero, dtype(-1)), dtype(-1e-30), dtype(-1),
            dtype(np.nan), neg_nan, dtype(np.inf), dtype(-np.inf)]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("which", range(9))
def test_costs_outside_the_range_are_reported(prot, dtype, which):
    import torch
    base = torch.from_numpy(np.random.default_rng(2).random((20, 35)).astype(dtype)).cuda()
    for aligned in (True, False):
        for col in list(range(8)) + [33, 34]:
            C = base.clone() if aligned else torch.cat([base[:, :1], base], 1)[:, 1:]
            C[7, col] = float(outside(dtype)[which]) if which != 6 else torch.from_numpy(
                np.array([outside(dtype)[which]])).cuda()[0]
            with pytest.raises(prot.PrError) as e:
                prot.assign(C, 0.1)
            assert e.value.status == -1, (aligned, col)
