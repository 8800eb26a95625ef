"""Which form a plan takes (needs a GPU: -m gpu): row buffers that the options name,
windows kept as shared-memory records or run as tiles.  Results bit for bit against the
oracle in every form."""
import json

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


def applied(events, n, directed=False, **options):
    plan = tn.Plan(*dev(*events), n, directed=directed, **options)
    S = torch.full((n, tn.tn_row_words(n)), -1, dtype=torch.int64, device="cuda")
    plan.apply(S, init=True)
    assert plan.status() == 0
    ref = (oracle.component_matrix_directed if directed else oracle.component_matrix)(*events, n)
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)
    return plan


def stream_launch(run, tmp_path):
    """The launch (grid, block) of the one streaming kernel that `run` launches."""
    for _ in range(2):  # (a process's first session may start too late for its kernels)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            run()
            torch.cuda.synchronize()
    prof.export_chrome_trace(str(tmp_path / "trace.json"))
    trace = json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
    launches = [e["args"] for e in trace if "stream_kernel" in e.get("name", "") and "block" in e.get("args", {})]
    if not launches:
        pytest.skip("no kernel records from the profiler")
    assert len(launches) == 1
    return launches[0]


@pytest.mark.parametrize("rows,threads", [(640, 160), (0, 416)])
def test_row_buffer_of_an_open_width(rows, threads, tmp_path):
    """An 80 KB row buffer gives two CTAs of 4 consumer warps per SM also where the slab
    width is left open and no window fits the buffer."""
    n, m = 3000, 20_000
    u, v, _ = synth.uniform_events(n, m, t_range=m, seed=3)
    options = dict(smem_rows=rows) if rows else dict(window_events=2100)
    plan = applied((u, v, np.arange(m) // 1000), n, slab_words=0, **options)
    assert plan.stats()["local_windows"] == 0
    S = torch.empty((n, tn.tn_row_words(n)), dtype=torch.int64, device="cuda")
    assert stream_launch(lambda: plan.apply(S, init=True), tmp_path)["block"][0] == threads


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("windows,ties", [(10, 1), (70, 1), (70, 3), (1050, 3)])
def test_a_short_last_window(windows, ties, directed):
    """Windows of 1,000 events whose rows do not fit the row buffer, and a last one of 9
    events (at most one window in 64: as a tile, so that the plan's rows are tracked),
    below and above the batch size from which schedules are copied."""
    n, m = 20_000, 1000 * windows + 9
    u, v, _ = synth.uniform_events(n, m, t_range=m, seed=windows)
    t = np.arange(m) // ties
    t[-9:] = t[-10] + 1 + np.arange(9) // 3  # 1,000 is no multiple of 3: the last window starts with the first of these
    v[-2] = u[-3]
    plan = applied((u, v, t), n, directed=directed, slab_words=16, window_events=1000)
    stats = plan.stats()
    assert stats["windows"] == windows + 1 and stats["local_windows"] == (1 if windows < 64 else 0)
    whole = tn.Plan(*dev(u, v, t), n, directed=directed, slab_words=16, window_events=1000, smem_rows=1).stats()
    assert (stats["ops"], stats["levels"]) == (whole["ops"], whole["levels"])
    if windows > 64:  # the counters are those of a plan that never had a record
        assert all(stats[k] == whole[k] for k in ("items", "aux", "temps"))


def hubs(n, m, h, ties, seed):
    """Every event joins one of h hubs and any other node; `ties` events a timestamp."""
    rng = np.random.default_rng(seed)
    ends = np.stack([rng.integers(0, h, m), rng.integers(h, n, m)])
    u, v = np.where(rng.random(m) < 0.5, ends, ends[::-1])
    return u, v, np.arange(m) // ties


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("stream", ["hubs", "bursty", "open"])
def test_short_levels_become_records(stream, directed):
    """Open options: streams of short levels, without ties, with large timestamp groups,
    and of a network whose rows would fit a resident CTA but for its saved rows."""
    if stream == "hubs":
        n, events = 26_000, hubs(26_000, 60_000, 32, 1, 1)
    elif stream == "bursty":
        n = 26_000
        events = synth.powerlaw_bursty(n, 100_000, seed=3)
    else:
        n = tn.tn_resident_max_rows(1)
        events = hubs(n, 60_000, 1, 64, 2)
    stats = applied(events, n, directed=directed).stats()
    assert stats["levels"] >= 256 and 0 < stats["local_windows"] <= stats["windows"] == -(-len(events[0]) // 640)


@pytest.mark.parametrize("slab,h,records", [(24, 32, True), (32, 32, True), (32, 300, False), (64, 32, False)])
def test_short_levels_in_wide_slabs(slab, h, records):
    """Records where most windows fit the row buffer, else the tiles stay as they were."""
    n = 60_000
    stats = applied(hubs(n, 60_000, h, 1, h), n, slab_words=slab).stats()
    assert stats["levels"] >= 256 and (stats["local_windows"] > 0) == records
    assert stats["windows"] == -(-60_000 // (640 if records else 1280))


def test_long_levels_stay_tiles():
    n = 26_000
    stats = applied(synth.er_poisson(n, 200_000, seed=3), n).stats()
    assert stats["levels"] >= 256 and stats["local_windows"] == 0


@pytest.mark.parametrize("n,h,ties,records", [(24_000, 1, 64, True), (24_000, 12, 300, True), (24_000, 500, 1, False)])
def test_resident_networks_around_hubs(n, h, ties, records):
    """Open options, rows that fit resident CTAs: long source lists in every level are
    walked as records, streams without them stay resident."""
    stats = applied(hubs(n, 100_000, h, ties, n + h), n).stats()
    assert stats["levels"] >= 256 and (stats["local_windows"] > 0) == records


@pytest.mark.parametrize("n,m,replicas,ncols", [(2000, 40_000, 3, 0), (30_000, 60_000, 1, 0), (30_000, 60_000, 2, 1500)])
def test_autotune_times_a_plan_without_options(n, m, replicas, ncols):
    events = dev(*synth.activity_driven(n, m, seed=n))
    first = tn.tn_autotune(*events, n, replicas=replicas, ncols=ncols)
    assert 0 < first["open_ms"] < float("inf") and 0 < first["best_ms"] < float("inf")
    again = tn.tn_autotune(*events, n, replicas=replicas, ncols=ncols)
    assert again["cached"] and again["open_ms"] == first["open_ms"]


@pytest.mark.parametrize("directed", [False, True])
def test_batches_of_small_networks(directed, tmp_path):
    """Ten networks of short levels: resident CTAs would make five waves, so the launch
    takes their record schedules (8 CTAs each).  One network alone is resident."""
    n, copies = 8000, 5
    streams = [synth.powerlaw_bursty(n, 300_000, seed=k) for k in (0, 2)]
    plans = [tn.Plan(*dev(*s), n, directed=directed) for s in streams]
    assert all(p.stats()["levels"] >= 8192 and p.stats()["local_windows"] == 0 for p in plans)
    refs = [(oracle.component_matrix_directed if directed else oracle.component_matrix)(*s, n) for s in streams]
    mats = [torch.empty((n, tn.tn_row_words(n)), dtype=torch.int64, device="cuda") for _ in range(2 * copies)]

    def check():
        for k, S in enumerate(mats):
            got = S.cpu().numpy().view(np.uint64)
            assert np.array_equal(got[:, : refs[k % 2].shape[1]], refs[k % 2])
            S.fill_(-1)

    tn.tn_plan_apply_batch(plans * copies, mats)
    check()
    graph = tn.BatchGraph(plans * copies, mats)
    for _ in range(2):
        graph.launch()
        check()
    graph.destroy()
    assert all(p.status() == 0 for p in plans)
    for k in range(2):
        plans[k].apply(mats[k], init=True)
        assert np.array_equal(mats[k].cpu().numpy().view(np.uint64)[:, : refs[k].shape[1]], refs[k])
    assert stream_launch(lambda: plans[0].apply(mats[0], init=True), tmp_path)["grid"][0] == 125
    assert stream_launch(lambda: tn.tn_plan_apply_batch(plans * copies, mats), tmp_path)["grid"][0] == 2 * copies * 8


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("n,h,ties", [(26_000, 32, 1), (26_000, 8, 64), (20_000, 1, 64)])
def test_columns_and_sketches_around_hubs(n, h, ties, directed):
    """Few columns and sketches of streams of short levels: narrow records, with the
    maximum as well."""
    u, v, t = hubs(n, 60_000, h, ties, h)
    events = dev(u, v, t)
    src = np.random.default_rng(h).integers(0, n, 700).astype(np.uint32)
    S = tn.tn_component_columns(*events, n, torch.from_numpy(src.view(np.int32)).cuda(), directed=directed)
    ref = oracle.component_matrix_directed(u, v, t, n, src=src) if directed else oracle.component_matrix(u, v, t, n, src=src)
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)
    for p in (4, 10, 13):
        R = tn.tn_hll_sketches(*events, n, p, 5, directed=directed)
        assert np.array_equal(R.cpu().numpy()[:, : 1 << p], oracle.hll_sketches(u, v, t, n, p, 5, directed=directed))
