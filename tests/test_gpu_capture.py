"""Stream capture beside the library's own threads (needs a GPU: -m gpu)."""
import threading

import numpy as np
import pytest

import oracle
from paper_2307_04890_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()
    oracle.build_oracle()


def dev(u, v, t):
    f = lambda x, d: torch.from_numpy(np.ascontiguousarray(x, dtype=d).view(np.int32 if d == np.uint32 else d)).cuda()  # noqa: E731
    return f(u, np.uint32), f(v, np.uint32), f(t, np.int64)


def test_a_thread_that_scheduled_ends_while_another_captures():
    """The pinned memory of an ending thread is released without an effect on a capture
    that forbids unsafe calls in all threads."""
    events = dev(*synth.uniform_events(500, 3000, t_range=900, seed=1))
    scheduled, end = threading.Event(), threading.Event()

    def work():
        plan = tn.Plan(*events, 500)
        plan.destroy()
        torch.cuda.synchronize()
        scheduled.set()
        end.wait()

    thread = threading.Thread(target=work)
    thread.start()
    scheduled.wait()
    x = torch.zeros(1000, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x.add_(1)
        end.set()
        thread.join()
        x.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, torch.full_like(x, 2))
