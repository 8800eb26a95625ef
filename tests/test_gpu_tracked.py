"""Tracked rows (needs a GPU: -m gpu): marks and content ids must never skip an update
that changes something.  Streams that saturate and are then disturbed by late nodes,
that fall into components, tie-heavy ones with multi-source updates and saved rows,
directed ones, batches that continue from unknown content, sketches (maximum instead
of OR), and networks too large for a mark per row.  Bit for bit against the oracle."""
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


def late_nodes(n, m, seed, ties):
    """Uniform events among growing sets of nodes: after each quiet stretch new nodes
    join, and a tenth of the nodes forms components of two and three."""
    rng = np.random.default_rng(seed)
    small = n // 10
    main = np.arange(small, n)
    us, vs = [], []
    for k, share in enumerate((0.5, 0.7, 0.9, 0.99, 1.0)):
        nodes = main[: max(2, int(len(main) * share))]
        u = rng.choice(nodes, m // 5)
        v = rng.choice(nodes, m // 5)
        pair = rng.random(m // 5) < 0.15
        x = rng.integers(0, max(1, small // 3), m // 5) * 3
        u[pair], v[pair] = x[pair], (x + rng.integers(1, 3, m // 5))[pair]
        us.append(u)
        vs.append(v)
    u, v = np.concatenate(us), np.concatenate(vs)
    t = np.arange(len(u)) if ties == 1 else np.sort(rng.integers(0, len(u) // ties, len(u)))
    return u, v, t


STREAMS = {
    "late": lambda: (700, *late_nodes(700, 60_000, 1, 1)),
    "late-ties": lambda: (900, *late_nodes(900, 60_000, 2, 40)),
    "bursty": lambda: (3000, *synth.powerlaw_bursty(3000, 90_000, seed=3)),
    "er": lambda: (1300, *synth.er_poisson(1300, 70_000, seed=4)),
    "sparse": lambda: (5000, *synth.activity_driven(5000, 12_000, seed=5)),
}


@pytest.mark.parametrize("slab", [2, 8, 16, 32, 64])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("name", sorted(STREAMS))
def test_matrix(name, directed, slab):
    n, u, v, t = STREAMS[name]()
    plan = tn.Plan(*dev(u, v, t), n, slab_words=slab, window_events=2480, directed=directed)
    assert plan.stats()["local_windows"] == 0
    S = torch.full((n, tn.tn_row_words(n)), -1, dtype=torch.int64, device="cuda")
    plan.apply(S, init=True)
    plan.apply(S)  # again, from content the application does not know
    assert plan.status() == 0
    once = (oracle.component_matrix_directed if directed else oracle.component_matrix)(u, v, t, n)
    if directed:
        ref = oracle.component_matrix_directed(np.concatenate((u, u)), np.concatenate((v, v)), np.concatenate((t, t + int(t[-1]) + 1)), n)
    else:
        ref = oracle.apply_events(u, v, t, n, once.copy())
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)
    plan.apply(S, init=True)
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], once)


@pytest.mark.parametrize("slab", [16, 64])
@pytest.mark.parametrize("n", [300_000, 500_000, 1_000_000, 2_500_000])
def test_columns_of_large_networks(n, slab):
    """A mark per row, per two, per four rows, none; ids.  Sources with their own
    activity, so that most of the stream does not reach them."""
    rng = np.random.default_rng(n)
    m = 60_000
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    hot = rng.integers(0, n, 3000)
    pick = rng.random(m) < 0.6
    u[pick], v[pick] = rng.choice(hot, m)[pick], rng.choice(hot, m)[pick]
    t = np.sort(rng.integers(0, 8_000, m))
    src = rng.choice(hot, 130).astype(np.uint32)
    plan = tn.Plan(*dev(u, v, t), n, slab_words=slab, window_events=2480)
    S = torch.full((n, tn.tn_row_words(len(src))), -1, dtype=torch.int64, device="cuda")
    plan.apply(S, ncols=len(src), src=torch.from_numpy(src.view(np.int32)).cuda(), init=True)
    assert plan.status() == 0
    ref = oracle.component_matrix(u, v, t, n, src=src)
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)


@pytest.mark.parametrize("p", [5, 9])
@pytest.mark.parametrize("reverse", [False, True])
def test_sketches(p, reverse):
    n, u, v, t = STREAMS["late-ties"]()
    R = tn.tn_hll_sketches(*dev(u, v, t), n, p, 11, reverse=reverse)
    assert np.array_equal(R.cpu().numpy()[:, : 1 << p], oracle.hll_sketches(u, v, t, n, p, 11, reverse=reverse))


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("shape", [dict(), dict(resident_words=1), dict(resident_words=2, window_events=700)])
@pytest.mark.parametrize("stream", ["late", "late-ties", "er", "bridge"])
def test_settled_networks(stream, shape, directed):
    """Long batches of small networks: resident CTAs skip packs that change nothing and
    stop once every row equals its component's.  `bridge`: two halves settle, one late
    event joins them, and another one at the very end adds a node."""
    n = 900
    if stream == "er":
        u, v, t = synth.er_poisson(n, 200_000, seed=8)
    elif stream == "bridge":
        rng = np.random.default_rng(9)
        m, half = 200_000, n // 2
        side = rng.integers(0, 2, m) * half
        u, v = side + rng.integers(0, half - 1, m), side + rng.integers(0, half - 1, m)
        u[m // 2], v[m // 2] = 3, half + 5
        u[-1], v[-1] = n - 1, 0
        t = np.arange(m)
    else:
        u, v, t = late_nodes(n, 200_000, 10, 1 if stream == "late" else 30)
    plan = tn.Plan(*dev(u, v, t), n, directed=directed, **shape)
    S = torch.full((n, tn.tn_row_words(n)), -1, dtype=torch.int64, device="cuda")
    ref = (oracle.component_matrix_directed if directed else oracle.component_matrix)(u, v, t, n)
    for _ in range(2):
        plan.apply(S, init=True)
        assert plan.status() == 0
        got = S.cpu().numpy().view(np.uint64)
        assert np.array_equal(got[:, : ref.shape[1]], ref) and not got[:, ref.shape[1]:].any()


@pytest.mark.parametrize("words", [1, 2])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("sources", [1, 3, 4, 5, 8, 9, 2500])
def test_resident_levels_of_many_ops_and_sources(sources, directed, words):
    """Star groups of `sources` edges, so many at once that a level has more ops than
    the CTA has threads, between groups of disjoint pairs; a 2,500-edge star keeps its
    source list outside the packs."""
    n = 6000
    rng = np.random.default_rng(sources)
    us, vs, ts = [], [], []
    for step in range(6):
        nodes = rng.permutation(n)
        if step % 2:
            u, v = nodes[: n // 2], nodes[n // 2 :]
        else:
            stars = min(1200, n // (sources + 1))
            hub, leaf = nodes[:stars], nodes[stars : stars * (sources + 1)]
            u, v = leaf, np.repeat(hub, sources)
        us.append(u)
        vs.append(v)
        ts.append(np.full(len(u), step))
    u, v, t = np.concatenate(us), np.concatenate(vs), np.concatenate(ts)
    plan = tn.Plan(*dev(u, v, t), n, resident_words=words, window_events=2480, directed=directed)
    S = torch.empty((n, tn.tn_row_words(n)), dtype=torch.int64, device="cuda")
    plan.apply(S, init=True)
    assert plan.status() == 0
    ref = (oracle.component_matrix_directed if directed else oracle.component_matrix)(u, v, t, n)
    assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)
