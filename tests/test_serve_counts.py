"""The server's counts of requests on the CPU, with fakes in place of handles
and of the CUDA calls: peak_running is the number of requests that were admitted
and not finished at the same time."""
import contextlib
import threading
import types

import numpy as np
import pytest

pytest.importorskip("torch")
from paper_1807_04638_gb300 import serve  # noqa: E402


class FakeArray:
    def to(self, *a, **k):
        return self

    def double(self):
        return self

    cpu = double

    def numpy(self):
        return np.zeros(1)


class FakeHandle:
    dtype = stream = _h = None

    def __init__(self, register):
        self.lddmm_register = lambda *a: register()

    def close(self):
        pass


@pytest.fixture
def make_server(monkeypatch):
    monkeypatch.setattr(serve.N, "workspace_bytes", lambda n, *a: n[0])
    monkeypatch.setattr(serve, "_key", lambda n, *a: tuple(n))
    null = lambda *a, **k: contextlib.nullcontext()
    torch = types.SimpleNamespace(cuda=types.SimpleNamespace(device=null, stream=null),
                                  from_numpy=lambda a: FakeArray(), zeros=lambda *a, **k: FakeArray())

    def make(register, budget=1e9, slots=4):
        srv = serve.Server(budget_bytes=budget, max_inflight=slots)
        srv.torch = torch
        srv._make_handle = lambda req: FakeHandle(register)
        return srv

    return make


def requests(sizes, gap=0.0):
    return [serve.Request(rid=i, I0=np.zeros((m, 1, 1)), I1=np.zeros((m, 1, 1)), params=None, arrival=gap * i)
            for i, m in enumerate(sizes)]


def test_requests_one_after_another_count_once(make_server):
    """Each request ends long before the next arrives."""
    srv = make_server(lambda: {"status": "ok"})
    res = srv.run_trace(requests([8, 8, 16], gap=0.2))
    assert [r.status for r in res] == ["ok"] * 3
    assert all(a.finished < b.admitted for a, b in zip(res, res[1:]))
    assert srv.peak_running == 1 and srv.running == 0


def test_requests_that_run_together_are_counted(make_server):
    together = threading.Barrier(3, timeout=20)

    def register():
        together.wait()
        return {"status": "ok"}

    srv = make_server(register)
    res = srv.run_trace(requests([8, 8, 16]))
    assert [r.status for r in res] == ["ok"] * 3
    assert srv.peak_running == 3 and srv.running == 0 and srv.inflight == 0


def test_a_request_that_waits_for_memory_or_is_refused_is_not_counted(make_server):
    """Room for one handle at a time, and one request that never fits."""
    srv = make_server(lambda: {"status": "ok"}, budget=10)
    res = srv.run_trace(requests([8, 9, 7, 11]))
    assert [r.status for r in res[:3]] == ["ok"] * 3 and "budget" in res[3].status
    assert srv.peak_running == 1 and srv.running == 0 and srv.inflight == 0
