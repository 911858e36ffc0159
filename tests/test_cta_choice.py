"""The rule that gives a solve, or its last part, to one CTA (cta_choice.cuh),
compiled with the host compiler: its lines, and that no CTA takes over rows
which the grid's CTAs keep to themselves."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_03732_gb300", "csrc")

SRC = """
#include "cta_choice.cuh"
extern "C" void choose(int seq, int n_rows, int n_cols, int row_bytes, int T, int K, int ctas, const char *mode,
                       int *out) {
    const prot::CtaChoice c = prot::choose_cta(seq, n_rows, n_cols, row_bytes, T, K, ctas, mode);
    out[0] = c.solo; out[1] = c.hand; out[2] = c.mid;
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("choice")
    (d / "c.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "c.cpp"), "-o", str(d / "c.so")],
                   check=True)
    L = ctypes.CDLL(str(d / "c.so"))

    def f(n_rows, n_cols, eps, ctas=152, seq=False, mode=None):
        K = int(1 / eps)
        row_bytes = (n_cols + 31) // 32 * 32 * (1 if K <= 252 else 2)
        out = (ctypes.c_int * 3)()
        L.choose(int(seq), n_rows, n_cols, row_bytes, int(eps * n_rows), K, ctas, mode, out)
        return dict(solo=bool(out[0]), hand=out[1], mid=bool(out[2]))
    return f


def test_rows_kept_by_the_grids_ctas_are_never_taken_over(choose):
    """More than 256 rows per CTA: CTAs keep rows that are in no pool."""
    assert choose(6000, 6000, 0.005, ctas=152)["hand"] == 43
    assert choose(6000, 6000, 0.005, ctas=24)["hand"] == 43  # 250 rows per CTA
    assert choose(6000, 6000, 0.005, ctas=20) == dict(solo=False, hand=0, mid=False)
    assert choose(1500, 1500, 0.1, ctas=6)["mid"]
    assert choose(1500, 1500, 0.1, ctas=5) == dict(solo=False, hand=0, mid=False)
    assert choose(6000, 6000, 0.005, ctas=20, mode=b"hand")["hand"] == 0
    assert choose(300, 300, 0.01, seq=True, mode=b"solo") == dict(solo=False, hand=64, mid=False)
    # the sequential rule's ring holds every row
    assert choose(6000, 6000, 0.003, ctas=20, seq=True)["hand"] == choose(6000, 6000, 0.003, seq=True)["hand"]


def test_lines_of_the_rule(choose):
    assert choose(384, 384, 0.01)["solo"] and not choose(385, 385, 0.01)["solo"]
    assert not choose(300, 300, 0.01, seq=True)["solo"]
    assert choose(1000, 1000, 0.01)["hand"] == 64 and choose(6400, 6400, 0.01)["hand"] == 0  # T = 64
    assert choose(1536, 1536, 0.05)["mid"] and not choose(1537, 1537, 0.05)["mid"]
    assert not choose(1536, 1536, 0.04)["mid"]  # floor(1/eps) > 20
    assert choose(300, 300, 0.1, mode=b"grid") == dict(solo=False, hand=0, mid=False)
    assert choose(4000, 4000, 0.01, mode=b"solo")["solo"]


@pytest.mark.parametrize("n_rows,n_cols,eps,solo", [
    (64, 8000, 0.005, True), (64, 8000, 0.003, False), (32, 8000, 0.003, True),  # 512 KB of rounded costs
    (384, 8000, 0.05, True), (384, 8000, 0.04, False), (65, 8000, 0.02, True), (200, 8000, 0.02, True),
    (201, 8000, 0.02, False), (65, 8000, 0.01, False), (384, 8000, 0.003, False), (300, 7000, 0.01, False),
    (384, 512, 0.01, True), (384, 513, 0.01, False), (300, 450, 0.003, True), (300, 600, 0.003, False)])
def test_one_cta_from_the_start(choose, n_rows, n_cols, eps, solo):
    """Wide problems whose crowded phases one SM would scan alone go to the grid."""
    assert choose(n_rows, n_cols, eps)["solo"] == solo
