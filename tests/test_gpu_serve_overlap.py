"""Requests that arrive together run at the same time on the device: by the
server's count and by the times of their results."""
import pytest

import test_gpu_serve

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_requests_that_arrive_together_overlap():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_04638_gb300 as pkg
    from paper_1807_04638_gb300.serve import Server
    reqs = test_gpu_serve.make_requests(pkg, test_gpu_serve.SPECS[:4])
    for r in reqs:
        r.arrival = 0.0
    srv = Server(budget_bytes=64e9, max_inflight=4)
    try:
        res = srv.run_trace(reqs)
    finally:
        srv.close()
    assert all(r.status == "LDDMM_OK" for r in res), [r.status for r in res]
    # admitted before the first one ends
    assert max(r.admitted for r in res) < min(r.finished for r in res)
    assert srv.peak_running == 4 and srv.running == 0
