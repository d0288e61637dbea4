"""gs_free_graph beside other work: a launch in flight finishes first, and a
capture that another thread is recording goes on."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_mod():
    import torch
    assert torch.cuda.is_available()
    return torch


@pytest.fixture
def graph(torch_mod):
    import paper_2607_06604_gb300 as gs
    X = np.random.default_rng(0).integers(0, 100_000, size=(6000, 3)).astype(np.int32)
    return gs, gs.gs_build_graph(X, 100_000, np.array([0, 3000, 6000, 9000], dtype=np.int64))


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_other_thread_captures(torch_mod, graph, mode):
    torch, (gs, g) = torch_mod, graph
    gs.gs_count_3pcf(g)
    t = torch.zeros(4, device="cuda")
    side, recorded = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        recorded.capture_begin(capture_error_mode=mode)
        t += 1
        other = threading.Thread(target=lambda: gs.gs_free_graph(g))
        other.start()
        other.join()
        t += 1
        recorded.capture_end()
    recorded.replay()
    torch.cuda.synchronize()
    assert t.tolist() == [2.0] * 4


def test_work_in_flight_finishes_first(torch_mod, graph):
    """Work on another stream (here none that uses the graph) is done when the
    graph is given back."""
    torch, (gs, g) = torch_mod, graph
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)
    assert not side.query()
    gs.gs_free_graph(g)
    assert side.query()
