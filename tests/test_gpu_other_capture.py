"""Calls of a long-running context while another thread captures a stream of its
own in the global mode, which an event query of any thread would end: within 5000
unread passes the stage times ask whether their first event pairs have finished."""
import threading

import pytest

from synth import cfg_tiny, make_system

pytestmark = pytest.mark.gpu


def test_capture_of_another_thread_stays_valid():
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1902_03837_gb300 import chi0 as lib
    s = make_system(cfg_tiny(seed=5, freqs=(0.1j,), eta=0.0))
    mine = torch.cuda.Stream()
    ctx = lib.Chi0.for_system(s, stream=mine.cuda_stream)
    ctx.load_system(s)
    ctx.compute_rho(0)
    ctx.synchronize()
    x = torch.arange(1000.0, device="cuda")
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    begun, finish, failed = threading.Event(), threading.Event(), []
    graph = torch.cuda.CUDAGraph()

    def capture():
        try:
            with torch.cuda.graph(graph, capture_error_mode="global"):
                begun.set()
                finish.wait(60)
                y.add_(x)
        except RuntimeError as e:
            failed.append(e)
            begun.set()

    t = threading.Thread(target=capture)
    t.start()
    begun.wait(60)
    for _ in range(5000):
        ctx.compute_rho(0)
    finish.set()
    t.join()
    assert not failed, failed
    graph.replay()
    graph.replay()
    ctx.synchronize()
    torch.cuda.synchronize()
    assert torch.equal(y, 2 * x)
    ctx.close()
