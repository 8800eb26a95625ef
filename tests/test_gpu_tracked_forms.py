"""Tracked rows in the launches that the general tests do not reach (needs a GPU: -m gpu):
sketches (byte-wise maximum) of networks too large for resident CTAs, the early stop of
column slabs, and open plans of different widths in one launch.  Bit for bit against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2307_04890_gb300 import synth
from test_gpu_tracked import dev, late_nodes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()
    oracle.build_oracle()


@pytest.mark.parametrize("p,ties,reverse", [(4, 1, False), (10, 30, False), (10, 1, True), (6, 30, True)])
def test_sketches_of_large_networks(p, ties, reverse):
    """Marks with the maximum: 2-word slabs above the resident limit, tiles at any level
    length from 64 events a node on.  Rows settle, their content becomes the reference,
    late nodes disturb it; PULLs and saved rows with ties."""
    n = tn.tn_resident_max_rows(1) + 72
    u, v, t = late_nodes(n, 64 * n, p, ties)
    R = tn.tn_hll_sketches(*dev(u, v, t), n, p, 11, reverse=reverse)
    assert np.array_equal(R.cpu().numpy()[:, : 1 << p], oracle.hll_sketches(u, v, t, n, p, 11, reverse=reverse))


@pytest.mark.parametrize("slab", [2, 16])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("stream", ["late", "late-ties", "bridge"])
def test_settled_column_slabs(stream, directed, slab):
    """Long batches (component labels): a CTA stops once every row equals its
    component's, not before a stream disturbed after settling has settled again."""
    n, m = 900, 200_000
    if stream == "bridge":
        rng = np.random.default_rng(9)
        half = n // 2
        side = rng.integers(0, 2, m) * half
        u, v = side + rng.integers(0, half - 1, m), side + rng.integers(0, half - 1, m)
        u[m // 2], v[m // 2] = 3, half + 5
        u[-1], v[-1] = n - 1, 0
        t = np.arange(m)
    else:
        u, v, t = late_nodes(n, m, 10, 1 if stream == "late" else 30)
    plan = tn.Plan(*dev(u, v, t), n, directed=directed, slab_words=slab, window_events=2480)
    assert plan.stats()["local_windows"] == 0
    S = torch.full((n, tn.tn_row_words(n)), -1, dtype=torch.int64, device="cuda")
    ref = (oracle.component_matrix_directed if directed else oracle.component_matrix)(u, v, t, n)
    for _ in range(2):
        plan.apply(S, init=True)
        assert plan.status() == 0
        got = S.cpu().numpy().view(np.uint64)
        assert np.array_equal(got[:, : ref.shape[1]], ref) and not got[:, ref.shape[1]:].any()


def test_open_widths_in_one_launch():
    """Two networks above the resident limit and a few columns of a third: three widths,
    chosen together."""
    jobs = []
    for n, m, nsrc, seed in ((60_000, 40_000, 0, 1), (26_000, 30_000, 0, 2), (30_000, 30_000, 200, 3)):
        u, v, t = synth.er_poisson(n, m, seed=seed)
        src = np.random.default_rng(seed).integers(0, n, nsrc).astype(np.uint32) if nsrc else None
        jobs.append((n, u, v, t, src))
    plans = [tn.Plan(*dev(u, v, t), n) for n, u, v, t, _ in jobs]
    assert all(p.stats()["local_windows"] == 0 for p in plans)
    ncols = [n if src is None else len(src) for n, _, _, _, src in jobs]
    mats = [torch.full((n, tn.tn_row_words(c)), -1, dtype=torch.int64, device="cuda") for (n, *_), c in zip(jobs, ncols)]
    srcs = [None if src is None else torch.from_numpy(src.view(np.int32)).cuda() for *_, src in jobs]
    tn.tn_plan_apply_batch(plans, mats, ncols=ncols, init=True, srcs=srcs)
    for p, S, (n, u, v, t, src) in zip(plans, mats, jobs):
        assert p.status() == 0
        ref = oracle.component_matrix(u, v, t, n) if src is None else oracle.component_matrix(u, v, t, n, src=src)
        assert np.array_equal(S.cpu().numpy().view(np.uint64)[:, : ref.shape[1]], ref)
