"""Stepping one handle while another thread captures its own stream in global
mode: the steps run, the capture stays valid, and so does what it holds. The
handle captures its graphs meanwhile: the first ones, or the chain of a long run."""
import threading

import pytest

from paper_1904_12553_gb300 import Solver, workloads as W
from test_parity_gpu import _gpu  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("before", [1, 6])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_steps_beside_a_capture(before, precision):
    w = W.random_smooth(3, 3, 64, 48, precision=precision, amp_u=0.01)
    s = Solver(w.params, stream=torch.cuda.Stream())
    s.init(w.c0, w.u0)
    s.step(before)
    torch.cuda.synchronize()
    x = torch.zeros(8, device="cuda")
    graph, failed = torch.cuda.CUDAGraph(), []
    ready, go_on = threading.Event(), threading.Event()

    def capture():
        try:
            with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="global"):
                x.add_(1)
                ready.set()
                go_on.wait(60)
                x.add_(1)
        except Exception as e:
            failed.append(e)
            ready.set()

    t = threading.Thread(target=capture)
    t.start()
    assert ready.wait(60)
    try:
        s.step(400)
    finally:
        go_on.set()
        t.join()
    assert not failed, failed
    assert s.steps_taken == before + 400
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 8
    r = Solver(w.params)
    r.init(w.c0, w.u0)
    r.step(before + 400)
    a, b = s.moments(), r.moments()
    for k in a:
        assert (a[k] == b[k]).all(), k
    s.close()
    r.close()
