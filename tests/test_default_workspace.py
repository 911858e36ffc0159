"""Calls without a workspace of their own: which default workspace they get
(no GPU: streams are stand-ins, nothing is allocated), and, on a GPU, solves
enqueued on two streams and from two threads."""
import threading
import types

import numpy as np
import pytest

import oracle
from paper_2203_03732_gb300 import workloads as W

torch = pytest.importorskip("torch")
import paper_2203_03732_gb300 as prot


@pytest.fixture
def streams(monkeypatch):
    """set(handle) makes `handle` the current stream of the device."""
    cur = types.SimpleNamespace(handle=0)
    cap = types.SimpleNamespace(on=False)
    monkeypatch.setattr(prot, "_raw_stream", lambda *a: cur.handle)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: cap.on)
    monkeypatch.setattr(prot, "_default_ws", threading.local())
    monkeypatch.setattr(prot, "_last_default_ws", {})

    def set_(handle, capturing=False):
        cur.handle, cap.on = handle, capturing
    return set_


def default():
    return prot._workspace(torch.device("cuda", 0))


def test_one_workspace_per_stream(streams):
    a = default()
    streams(7)
    b = default()
    assert a is not b and default() is b
    streams(0)
    assert default() is a


def test_one_workspace_per_thread(streams):
    got = {}
    t = threading.Thread(target=lambda: got.update(ws=default()))
    t.start()
    t.join()
    assert got["ws"] is not default()


def test_captured_calls_share_none(streams):
    eager = default()
    streams(0, capturing=True)
    a, b = default(), default()
    assert a is not eager and a is not b
    streams(0)
    assert default() is eager


def test_kept_workspaces_are_bounded(streams):
    first = default()
    for h in range(1, 40):
        streams(h)
        last = default()
    assert len(prot._default_ws.by_stream) == prot._DEFAULT_WS_PER_THREAD
    assert default() is last
    streams(0)
    assert default() is not first


def test_status_workspace(streams):
    a = default()
    streams(5)
    b = default()
    assert prot._status_workspace(torch) is b
    streams(0)
    assert prot._status_workspace(torch) is a
    streams(9)  # no call on this stream: the thread's last
    assert prot._status_workspace(torch) is b
    got = {}
    t = threading.Thread(target=lambda: got.update(ws=prot._status_workspace(torch)))
    t.start()
    t.join()
    assert got["ws"] is b  # another thread without calls: any thread's last


def problems():
    out = []
    for i, (n, eps) in enumerate([(300, 0.01), (1200, 0.01), (2500, 0.05), (500, 0.003)]):
        C = W.assignment_euclid_2d(n, 60 + i)
        out.append((C, eps, oracle.assign(C, eps)))
    return out


def check(got, refs):
    for g, (_, _, ref) in zip(got, refs):
        for k in ("row_to_col", "col_to_row", "y_row", "y_col"):
            assert np.array_equal(g[k].cpu().numpy(), ref[k]), k


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_03732_gb300 import build
    build.build()


@pytest.mark.gpu
def test_solves_on_two_streams(gpu):
    refs = problems()
    data = [torch.from_numpy(C).cuda() for C, _, _ in refs]
    torch.cuda.synchronize()
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(3):
        got = []
        for i, (C, (_, eps, _)) in enumerate(zip(data, refs)):
            with torch.cuda.stream(s[i % 2]):
                got.append(prot.assign(C, eps, sync=False))
        for st in s:
            with torch.cuda.stream(st):
                prot.ws_status()
        check(got, refs)


@pytest.mark.gpu
def test_solves_from_two_threads_on_one_stream(gpu):
    refs = problems()
    data = [torch.from_numpy(C).cuda() for C, _, _ in refs]
    torch.cuda.synchronize()
    got = [[None] * len(refs) for _ in range(2)]

    def work(t):
        for i in range(len(refs)):
            j = (i + t) % len(refs)
            got[t][j] = prot.assign(data[j], refs[j][1], sync=False)
    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for g in got:
        check(g, refs)


@pytest.mark.gpu
def test_one_workspace_on_two_streams_in_turn(gpu):
    """A workspace that moves to another stream and then grows."""
    refs = problems()
    data = [torch.from_numpy(C).cuda() for C, _, _ in refs]
    ws = prot.Workspace()
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for i, (C, (_, eps, _)) in enumerate(zip(data, refs)):
        s[i % 2].wait_stream(s[(i + 1) % 2])
        s[i % 2].wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s[i % 2]):
            got.append(prot.assign(C, eps, ws=ws, sync=False))
    prot.ws_status(ws)
    check(got, refs)
