"""Schedules at the edges of the planner's units (needs a GPU: -m gpu): chunks of
16 events, packs of 64 levels and 2,030 ops, timestamp groups around the 48
events above which the whole CTA takes them unchecked, local ids that are the
node ids (networks of at most two nodes per window event), windows stretched by a
group into the second pass, and batches large enough to be copied into buffers of
their exact size.  Bit for bit against the oracle."""
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


def check(u, v, t, n, directed=False, **options):
    du, dv = (torch.from_numpy(np.ascontiguousarray(x, dtype=np.uint32).view(np.int32)).cuda() for x in (u, v))
    dt = torch.from_numpy(np.ascontiguousarray(t, dtype=np.int64)).cuda()
    plan = tn.Plan(du, dv, dt, n, directed=directed, **options)
    S = torch.full((n, tn.tn_row_words(n)), -1, dtype=torch.int64, device="cuda")
    plan.apply(S, init=True)
    assert plan.status() == 0
    stats = plan.stats()
    plan.destroy()
    ref = (oracle.component_matrix_directed if directed else oracle.component_matrix)(u, v, t, n)
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)
    return stats


SHAPES = [dict(window_events=2600), dict(window_events=2600, slab_words=2, smem_rows=1), dict(window_events=2600, resident_words=1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("m", [1, 15, 16, 17, 63, 64, 65, 2029, 2030, 2031, 5001])
def test_one_level_per_event_and_one_level_for_all(m, shape):
    """A star (every event its own level) and a matching (all events one level)."""
    rng = np.random.default_rng(m)
    leaves = rng.integers(1, 200, m)
    check(np.zeros(m, int), leaves, np.arange(m), 200, **shape)
    n = 2 * m
    ids = rng.permutation(n)
    st = check(ids[:m], ids[m:], np.arange(m), n, **shape)
    assert st["ops"] == m and st["levels"] == -(-m // 2600)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("group", [2, 16, 17, 47, 48, 49, 127, 128, 129, 400])
def test_groups_with_and_without_shared_nodes(group, directed):
    """Groups of one size whose events share no node, with one pair that shares one
    at either end of the group, self-loops and duplicates among them."""
    rng = np.random.default_rng(group)
    n, us, vs, ts = 2 * group + 10, [], [], []
    for g in range(24):
        ids = rng.permutation(n)[: 2 * group]
        a, b = ids[:group].copy(), ids[group:].copy()
        if g % 4 == 1:
            a[-1] = b[0]
        elif g % 4 == 2:
            b[-1], a[0] = a[0], b[1]
        elif g % 4 == 3:
            a[0], b[-1] = b[0], a[-1]  # two self-loops
            if group > 2:
                a[1], b[1] = a[2], b[2]
        us.append(a)
        vs.append(b)
        ts.append(np.full(group, g))
    u, v, t = np.concatenate(us), np.concatenate(vs), np.concatenate(ts)
    for window in (40, 700, 2600):
        check(u, v, t, n, directed=directed, window_events=window)
        check(u, v, t, n, directed=directed, window_events=window, slab_words=8, smem_rows=1)


@pytest.mark.parametrize("events", [2600, 2664, 2665, 6000, 20_000])
def test_windows_stretched_by_a_group(events):
    """One group longer than the window: first pass, second pass, global memory."""
    rng = np.random.default_rng(events)
    n = 900
    u, v = rng.integers(0, n, events + 500), rng.integers(0, n, events + 500)
    t = np.concatenate([np.arange(100), np.full(events, 200), 201 + np.arange(400)])
    check(u, v, t, n, window_events=2600)


@pytest.mark.parametrize("extra", [-1, 0])
@pytest.mark.parametrize("shape", [dict(), dict(window_events=2600), dict(resident_words=1, window_events=2600)])
def test_exact_buffers(shape, extra):
    """Around the batch size from which the schedule is copied into exact buffers,
    with groups whose multi-source updates name source lists and saved rows."""
    m, n = (1 << 20) + extra, 300
    rng = np.random.default_rng(5)
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    t = np.sort(rng.integers(0, m // 3, m))
    check(u, v, t, n, **shape)


def test_plans_of_many_threads():
    """Threads that schedule at the same time, each on its own stream, with refused
    batches in between: every thread gets the counters of its own plan."""
    from concurrent.futures import ThreadPoolExecutor

    n = 600
    batches = [synth.uniform_events(n, 700 + 911 * k, t_range=300, seed=k) for k in range(8)]
    refs = [oracle.component_matrix(u, v, t, n) for u, v, t in batches]

    def work(k):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            u, v = (torch.from_numpy(np.ascontiguousarray(x, dtype=np.uint32).view(np.int32)).cuda() for x in batches[k][:2])
            t = torch.from_numpy(np.ascontiguousarray(batches[k][2], dtype=np.int64)).cuda()
            back = t.flip(0).contiguous()
            for _ in range(6):
                with pytest.raises(tn.TnError):
                    tn.Plan(u, v, back, n, stream=stream)
                plan = tn.Plan(u, v, t, n, stream=stream)
                S = torch.empty((n, tn.tn_row_words(n)), dtype=torch.int64, device="cuda")
                plan.apply(S, init=True, stream=stream)
                stats = plan.stats()
                assert stats["windows"] == -(-len(batches[k][0]) // 1280)
                stream.synchronize()
                assert plan.status() == 0
                assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : refs[k].shape[1]], refs[k])
                plan.destroy(stream=stream)
        return True

    with ThreadPoolExecutor(8) as pool:
        assert all(pool.map(work, range(8)))
