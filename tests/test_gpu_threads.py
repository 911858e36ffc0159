"""Solves from several threads at once, each with a workspace and a stream of
its own: the launch limits found on the first call and the kernels' shared-
memory limits are the same for every thread."""
import subprocess
import sys
import os
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# a fresh process: the first calls of the library come from four threads
SRC = textwrap.dedent("""
    import threading
    import numpy as np
    import torch
    import oracle
    import paper_2203_03732_gb300 as prot
    g = np.random.default_rng(4)
    # keys of the sequential rule: 96 bytes, 70,016 and 140,032 bytes of shared memory
    cases = [(40, 96, 0.05), (3, 70016, 0.05), (3, 70016, 0.003), (500, 500, 0.02)]
    mats = [g.random((b, a)).astype(np.float32) for b, a, _ in cases]
    refs = [oracle.assign(C, e, mode=oracle.MODE_SEQUENTIAL) for C, (_, _, e) in zip(mats, cases)]
    data = [torch.from_numpy(C).cuda() for C in mats]
    torch.cuda.synchronize()
    bad = []
    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(30):
                    got = prot.assign(data[i], cases[i][2], rule="sequential")
                    for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
                        assert np.array_equal(got[k].cpu().numpy(), refs[i][k]), (i, k)
        except Exception as e:
            bad.append((i, repr(e)))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(cases))]
    for t in threads: t.start()
    for t in threads: t.join()
    assert not bad, bad
    print("ok")
""")


def test_first_calls_from_four_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", SRC], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stderr[-2000:]
