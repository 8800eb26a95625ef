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


def check_replays(graph, S, ref):
    for _ in range(2):
        S.fill_(-1)
        graph.launch()
        torch.cuda.synchronize()
        assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)


@pytest.mark.parametrize("slabs", [(64, 64), (32, 4)])
def test_replayed_content_ids(slabs):
    """Graphs whose launch allocates content ids: one or two jobs of it."""
    n = 3000
    streams = [synth.powerlaw_bursty(n, 60_000, seed=k) for k in range(2)]
    plans = [tn.Plan(*dev(*s), n, slab_words=w, window_events=2480) for s, w in zip(streams, slabs)]
    mats = [torch.empty((n, tn.tn_row_words(n)), dtype=torch.int64, device="cuda") for _ in plans]
    graph = tn.BatchGraph(plans, mats)
    for S, (u, v, t) in zip(mats, streams):
        check_replays(graph, S, oracle.component_matrix(u, v, t, n))
    assert all(p.status() == 0 for p in plans)
    graph.destroy()


def test_no_room_for_replayed_content_ids():
    """Content ids that a direct call would do without are not recorded in a graph."""
    n, m = 10_000_000, 700_000
    rng = np.random.default_rng(1)
    hot = rng.integers(0, n, 500)
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    u[::3], v[::3] = rng.choice(hot, len(u[::3])), rng.choice(hot, len(v[::3]))
    t = np.arange(m)
    src = np.unique(hot)[:128].astype(np.uint32)
    S = torch.empty((n, tn.tn_row_words(128)), dtype=torch.int64, device="cuda")
    plan = tn.Plan(*dev(u, v, t), n, slab_words=64, window_events=2480)
    sources = torch.from_numpy(src.view(np.int32)).cuda()
    plan.apply(S, ncols=128, src=sources, init=True)
    ref = S.clone()
    tn.tn_init_matrix(S, n, 128, src=sources)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.cuda.mem_get_info()[0] - (250 << 20)  # the ids are 320 MB
    filler = torch.empty(room, dtype=torch.uint8, device="cuda")
    try:
        graph = tn.BatchGraph([plan], [S], ncols=[128], init=False)
        graph.launch()
        torch.cuda.synchronize()
        graph.destroy()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert plan.status() == 0 and torch.equal(S, ref)
