"""Workloads of temporal out-components and network hashing on one GPU.

Each case is a call sequence of the public API on the kind of event stream it is
used for: whole component matrices from small to large networks, sampled source
columns, the hashed estimate, HyperLogLog sketches, events arriving in batches,
host arrays, and the serving engine.  Event streams are drawn on the GPU from the
seed with the statistics of ``paper_2307_04890_gb300.synth`` (uniform pairs with
ties, activity-driven, bursty power-law links, Erdos-Renyi with Poisson links);
event times of Poisson streams are sorted uniform draws, which is the same process
given its number of events.  As in the id spaces of real networks, about 2 % of the
ids of the uniform and activity-driven streams have no event: they stay isolated.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2307_04890_gb300 as tn

MASK64 = (1 << 64) - 1


def listed():
    return [
        # the smallest network of the project's configurations: ties at every other
        # timestamp, one call from events to sizes; latency and launches count
        dict(name="matrix-uniform-small", kind="matrix", events="uniform", n=1000, m=20_000, t_range=10_000),
        # the paper's Erdos-Renyi sweep: few nodes, many events, one call
        dict(name="matrix-er", kind="matrix", events="er", n=10_000, m=10_000_000),
        # a sparse stream (a few events per node, odd sizes): most rows stay short
        dict(name="matrix-activity-sparse", kind="matrix", events="activity", n=123_457, m=300_007),
        # the activity-driven configuration: a plan with default options, applied, then sizes
        dict(name="plan-activity", kind="plan", events="activity", n=100_000, m=10_000_000, slab_words=0),
        # the bursty power-law configuration (large tie groups) with the wide slabs it is tuned to
        dict(name="plan-bursty", kind="plan", events="bursty", n=500_000, m=25_000_000, slab_words=64),
        # the out-components of a sample of sources only, directed events
        dict(name="columns-directed", kind="columns", events="activity", n=200_003, m=3_000_000, nsrc=5_000, directed=True),
        # network hashing end to end at the hashed configuration's sizes: proxies and sampled
        # exact columns in one batch, fused estimates, error statistics
        dict(name="hashed-sampled", kind="hashed", events="activity", n=1_000_000, m=5_000_000, k=16_384, R=8, nsrc=65_536),
        # network hashing of the paper's sweep: n_s = 0.3 n super-nodes, 5 replicas, every source
        dict(name="hashed-er", kind="hashed", events="er", n=5_000, m=100_000, k=1_500, R=5, nsrc=0),
        # the whole exact path from host arrays to host sizes
        dict(name="host-bursty", kind="host", events="bursty", n=20_011, m=500_009),
        # events arriving in batches cut anywhere, nodes joining half way, sizes after every batch
        dict(name="online-activity", kind="online", events="activity", n=20_000, m=2_000_000, batches=7, grow=2_500),
        # HyperLogLog sketches over the reversed sequence and their size estimates
        dict(name="hll-reversed", kind="hll", events="uniform", n=20_000, m=500_000, t_range=2_000, p=10, reverse=True),
        # a burst of requests of mixed sizes to a running server, four batches each
        dict(name="serving-mixed", kind="serving", jobs=32, n_lo=1_000, n_hi=20_000, m_lo=10_000, m_hi=300_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matrix", "matrix", "plan", "plan", "columns", "hashed", "host", "online", "hll", "serving"])
    if kind == "serving":
        return dict(kind=kind, jobs=rng.randint(8, 32), n_lo=1_000, n_hi=_log_int(rng, 2_000, 20_000), m_lo=10_000,
                    m_hi=_log_int(rng, 20_000, 300_000))
    if kind == "hashed":
        n = _log_int(rng, 500, 500_000)
        R = rng.randint(2, 8)
        every = n <= 20_000 and rng.random() < 0.5
        return dict(kind=kind, events=rng.choice(["activity", "er"]), n=n, m=_log_int(rng, 10_000, 5_000_000),
                    k=_log_int(rng, max(30, n // 100), min(16_384, int(0.5 * n))), R=R,
                    nsrc=0 if every else min(n, _log_int(rng, 16, 30_000)))
    if kind == "hll":
        m = _log_int(rng, 10_000, 500_000)
        return dict(kind=kind, events="uniform", n=_log_int(rng, 500, 20_000), m=m, t_range=_log_int(rng, 500, 3_000),
                    p=rng.randint(4, 11), reverse=rng.random() < 0.5)
    top = {"matrix": 200_000, "plan": 200_000, "columns": 400_000, "host": 50_000, "online": 50_000}[kind]
    n = _log_int(rng, 500, top)
    m = _log_int(rng, 5_000, min(10_000_000, 1_000_000_000_000 // n, {"host": 2_000_000, "online": 2_000_000}.get(kind, 10_000_000)))
    case = dict(kind=kind, events=rng.choice(["uniform", "activity", "bursty", "er"]), n=n, m=m)
    if case["events"] == "uniform":
        case["t_range"] = _log_int(rng, 100, 2 * m)
    if kind == "plan":
        case["slab_words"] = rng.choice([0, 0, 8, 16, 32, 64])
    elif kind == "columns":
        case["nsrc"] = _log_int(rng, 50, min(n, 20_000))
        case["directed"] = rng.random() < 0.5
    elif kind == "online":
        case["batches"] = rng.randint(2, 9)
        case["grow"] = rng.choice([0, 64, 3_000])
    return case


# ---------------------------------------------------------------------------
# event streams, on the GPU (integer sums only: the same events for the same seed)
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _other(g, u, n):
    """A uniform partner different from u."""
    return (u + torch.randint(1, n, u.shape, generator=g, device="cuda")) % n


def _present(g, n):
    """The ids that take part in events, in random order."""
    return torch.randperm(n, generator=g, device="cuda")[:max(2, n - n // 50)]


def _uniform(g, n, m, t_range):
    ids = _present(g, n)
    n = ids.numel()
    u = torch.randint(0, n, (m,), generator=g, device="cuda")
    return ids[u], ids[_other(g, u, n)], torch.randint(0, t_range, (m,), generator=g, device="cuda").sort().values


def _activity(g, n, m):
    ids = _present(g, n)
    n = ids.numel()
    a = _rand(g, n)
    e = 1.0 - 2.1
    a = ((1e-3 ** e + a * (1.0 - 1e-3 ** e)) ** (1.0 / e)).cpu().numpy()
    cdf = torch.from_numpy(np.cumsum(a) / a.sum()).cuda()
    u = torch.searchsorted(cdf, _rand(g, m), right=True).clamp_(max=n - 1)
    t = (_rand(g, m) * (m / a.sum() * 1e6)).long().sort().values
    return ids[u], ids[_other(g, u, n)], t


def _er(g, n, m):
    pairs = n * (n - 1) // 2
    links = n + int(np.random.default_rng(int(torch.randint(0, 1 << 31, (1,), generator=g, device="cuda"))).normal() * math.sqrt(n))
    links = max(1, min(pairs, links))
    a = torch.randint(0, n, (2 * links + 64,), generator=g, device="cuda")
    b = _other(g, a, n)
    key = torch.unique(torch.minimum(a, b) * n + torch.maximum(a, b))
    key = key[torch.randperm(key.numel(), generator=g, device="cuda")[:links]]
    pick = key[torch.randint(0, key.numel(), (m,), generator=g, device="cuda")]
    t = (_rand(g, m) * (m / key.numel() * 1e6)).long().sort().values
    return pick // n, pick % n, t


def _bursty(g, n, m):
    k_max = int(n ** (1.0 / 1.5))
    pmf = np.arange(1, k_max + 1, dtype=np.float64) ** -2.5
    cdf = torch.from_numpy(np.cumsum(pmf) / pmf.sum()).cuda()
    deg = torch.searchsorted(cdf, _rand(g, n), right=True).clamp_(max=k_max - 1) + 1
    stubs = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    stubs = stubs[torch.randperm(stubs.numel(), generator=g, device="cuda")]
    a, b = stubs[0:stubs.numel() // 2 * 2:2], stubs[1::2]
    key = torch.unique((torch.minimum(a, b) * n + torch.maximum(a, b))[a != b])
    ea, eb = key // n, key % n
    horizon = 1.2 * 180_000.0 * m / key.numel()  # milliseconds; the mean gap of a link is 180 s
    while True:
        now = torch.zeros(key.numel(), dtype=torch.int64, device="cuda")
        alive = torch.arange(key.numel(), device="cuda")
        times, owners, count = [], [], 0
        while alive.numel():
            gaps = (60_000.0 / (1.0 - _rand(g, alive.numel(), 16)) ** (1.0 / 1.5)).clamp_(max=1e12).long()
            at = now[:, None] + torch.cumsum(gaps, 1)
            inside = at <= horizon
            times.append(at[inside])
            owners.append(alive[:, None].expand_as(at)[inside])
            count += times[-1].numel()
            keep = inside[:, -1]
            alive, now = alive[keep], at[keep, -1]
        if count >= m:
            break
        horizon *= 1.5
    t, order = torch.sort(torch.cat(times), stable=True)
    o = torch.cat(owners)[order[:m]]
    return ea[o], eb[o], t[:m] // 1000


def _events(case, g):
    n, m = case["n"], case["m"]
    if case["events"] == "uniform":
        u, v, t = _uniform(g, n, m, case["t_range"])
    else:
        u, v, t = {"activity": _activity, "er": _er, "bursty": _bursty}[case["events"]](g, n, m)
    return u.int().contiguous(), v.int().contiguous(), t.contiguous()


def _hash_seed(seed):
    return (seed * 0x9E3779B1 + 0x7F4A7C15) & 0xFFFFFFFF


def _cuts(m, parts, seed):
    """Batch bounds anywhere in the stream, also inside groups of equal timestamps."""
    inner = np.sort(np.random.default_rng(seed).integers(1, m, size=parts - 1)).tolist() if parts > 1 else []
    return [0, *inner, m]


class _RunningServer:
    """A server with the options it is deployed with; closed with its state."""

    def __init__(self):
        self.server = tn.Server(max_active=32, workers=16)
        self.next_id = 0

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "serving":
        rng, sizes = np.random.default_rng(seed), np.random.default_rng(case["jobs"])
        jobs = []
        for _ in range(case["jobs"]):
            n = int(np.exp(sizes.uniform(np.log(case["n_lo"]), np.log(case["n_hi"]))))
            m = int(np.exp(sizes.uniform(np.log(case["m_lo"]), np.log(case["m_hi"]))))
            ids = rng.permutation(n)[:n - n // 50].astype(np.uint32)
            u = rng.integers(0, len(ids), m)
            v = (u + rng.integers(1, len(ids), m)) % len(ids)
            t = np.sort(rng.integers(0, m, m))
            jobs.append((n, ids[u], ids[v], t, np.array([0, m // 4, m // 2, 3 * m // 4, m], np.uint64)))
        return dict(case=case, jobs=jobs, running=_RunningServer())
    u, v, t = _events(case, g)
    state = dict(case=case, u=u, v=v, t=t)
    if kind == "host":
        return dict(case=case, u=u.cpu().numpy().view(np.uint32), v=v.cpu().numpy().view(np.uint32), t=t.cpu().numpy())
    if kind == "plan":
        state["S"] = torch.empty((case["n"], tn.tn_row_words(case["n"])), dtype=torch.int64, device="cuda")
    if kind in ("columns", "hashed") and case["nsrc"]:
        state["src"] = torch.randperm(case["n"], generator=g, device="cuda")[:case["nsrc"]].int().sort().values
    if kind == "hashed":
        nsrc = case["nsrc"] or case["n"]
        state["P"] = torch.empty((case["R"], case["k"], tn.tn_row_words(case["k"])), dtype=torch.int64, device="cuda")
        state["S"] = torch.empty((case["n"], tn.tn_row_words(nsrc)), dtype=torch.int64, device="cuda")
    if kind in ("hashed", "hll"):
        state["seed"] = _hash_seed(seed)
    if kind == "online":
        state["cuts"] = _cuts(case["m"], case["batches"], seed)
    return state


def _run_hashed(s, case):
    n, k, R, src = case["n"], case["k"], case["R"], s.get("src")
    nsrc = case["nsrc"] or n
    H, pu, pv = tn.tn_hash_proxy(s["u"], s["v"], n, k, R, s["seed"])
    plans = [tn.Plan(pu[j], pv[j], s["t"], k) for j in range(R)]
    plans.append(tn.Plan(s["u"], s["v"], s["t"], n))
    tn.tn_plan_apply_batch(plans, [s["P"][j] for j in range(R)] + [s["S"]], ncols=[k] * R + [nsrc], init=True,
                           srcs=[None] * R + [src])
    est = tn.tn_hash_estimate(s["P"], R, k, H, n, src=src)
    exact, _, _ = tn.tn_out_sizes(s["S"], n, nsrc)
    err = tn.tn_error_stats(est, exact, n)
    for p in plans:
        p.destroy()
    return dict(H=H, P=s["P"], S=s["S"], est=est, exact=exact, err=err)


def _run_online(s, case):
    n, sizes = case["n"], []
    with tn.Online(n) as o:
        for b, (a, e) in enumerate(zip(s["cuts"][:-1], s["cuts"][1:])):
            if b == case["batches"] // 2 and case["grow"]:
                n += case["grow"]
                o.grow(n)
            o.push(s["u"][a:e], s["v"][a:e], s["t"][a:e])
            sizes.append(tn.tn_out_sizes(o.matrix(), n, n)[0])
        o.flush()
        S = o.matrix().clone()
        return dict(S=S, sizes=sizes, final=tn.tn_out_sizes(S, n, n, argmax=True)[0::2])


def _run_serving(s, case):
    r = s["running"]
    first = r.next_id
    for n, u, v, t, cuts in s["jobs"]:
        r.server.submit(r.next_id, n, u, v, t, cuts)
        r.next_id += 1
    left = len(s["jobs"])
    while left:
        left -= len(r.server.poll(wait_ms=1000))
    done = [r.server.results.pop(first + i) for i in range(len(s["jobs"]))]
    return dict(sizes=np.concatenate([d[0] for d in done]).astype(np.int64), argmax=np.array([d[1] for d in done]))


def run(s):
    case = s["case"]
    kind, n = case["kind"], case.get("n")
    if kind == "matrix":
        S = tn.tn_component_matrix(s["u"], s["v"], s["t"], n)
        return (S, *tn.tn_out_sizes(S, n, n, in_sizes=True, argmax=True))
    if kind == "plan":
        plan = tn.Plan(s["u"], s["v"], s["t"], n, slab_words=case["slab_words"])
        plan.apply(s["S"], init=True)
        out, _, best = tn.tn_out_sizes(s["S"], n, n, argmax=True)
        plan.destroy()
        return s["S"], out, best
    if kind == "columns":
        S = tn.tn_component_columns(s["u"], s["v"], s["t"], n, s["src"], directed=case["directed"])
        return S, tn.tn_out_sizes(S, n, case["nsrc"])[0]
    if kind == "host":
        return tn.tn_out_component_sizes_host(s["u"], s["v"], s["t"], n)
    if kind == "hll":
        R = tn.tn_hll_sketches(s["u"], s["v"], s["t"], n, case["p"], s["seed"], reverse=case["reverse"])
        return R, tn.tn_hll_estimate(R, n, case["p"])
    return {"hashed": _run_hashed, "online": _run_online, "serving": _run_serving}[kind](s, case)


def work(case):
    """Events in once (endpoints and time), results out once."""
    kind = case["kind"]
    if kind == "serving":
        jobs, n, m = case["jobs"], math.sqrt(case["n_lo"] * case["n_hi"]), math.sqrt(case["m_lo"] * case["m_hi"])
        return {"bytes": jobs * (16 * m + 4 * n), "flops": 0}
    n, m = case["n"], case["m"]
    words = lambda c: 16 * ((c + 1023) // 1024)  # noqa: E731
    out = {
        "matrix": lambda: n * words(n) * 8 + 8 * n + 4,
        "plan": lambda: n * words(n) * 8 + 4 * n + 4,
        "columns": lambda: n * words(case["nsrc"]) * 8 + 8 * case["nsrc"],
        "host": lambda: 4 * n + 4,
        "online": lambda: (n + case["grow"]) * words(n + case["grow"]) * 8 + 4 * (n + case["grow"]) * (case["batches"] + 1),
        "hll": lambda: n * max(128, 1 << case["p"]) + 8 * n,
        "hashed": lambda: 4 * case["R"] * n + 8 * case["R"] * case["k"] * words(case["k"])
        + 8 * n * words(case["nsrc"] or n) + 8 * (case["nsrc"] or n),
    }[kind]()
    return {"bytes": 16 * m + out, "flops": 0}


# ---------------------------------------------------------------------------
# the floating-point results in 64 bits, by plain torch and numpy
# ---------------------------------------------------------------------------
def _splitmix(state):
    """Output of one SplitMix64 step from each state (uint64 array)."""
    z = state + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _exact_hll(case, seed):
    u, v, t = _events(case, _generator(seed))
    n, p = case["n"], case["p"]
    h = _splitmix(np.uint64(_hash_seed(seed)) ^ np.arange(n, dtype=np.uint64))
    reg = (h >> np.uint64(64 - p)).astype(np.int64)
    rank = [64 - p + 1 if not x else 64 - int(x).bit_length() + 1 for x in (h << np.uint64(p))]
    M = torch.zeros((n, 1 << p), device="cuda")
    M[torch.arange(n, device="cuda"), torch.from_numpy(reg).cuda()] = torch.tensor(rank, dtype=torch.float32, device="cuda")
    ends = torch.unique_consecutive(t, return_counts=True)[1].cumsum(0).tolist()
    groups = list(zip([0, *ends[:-1]], ends))
    for a, e in groups[::-1] if case["reverse"] else groups:
        x, y = u[a:e].long(), v[a:e].long()
        M.index_reduce_(0, torch.cat((x, y)), torch.cat((M[y], M[x])), "amax")
    s = 1 << p
    alpha = {16: 0.673, 32: 0.697, 64: 0.709}.get(s, 0.7213 / (1.0 + 1.079 / s))
    est = alpha * s * s / torch.exp2(-M.double()).sum(1)
    zeros = (M == 0).sum(1).double()
    small = (est <= 2.5 * s) & (zeros > 0)
    return None, torch.where(small, s * torch.log(s / zeros.clamp(min=1.0)), est)


def _component_rows(u, v, t, n):
    """Component matrix as n Python integers (bit c of row i: i reached from c)."""
    S = [1 << i for i in range(n)]
    ends = np.flatnonzero(np.append(t[1:] != t[:-1], True)) + 1
    a = 0
    for e in ends.tolist():
        if e == a + 1:
            x, y = u[a], v[a]
            S[x] = S[y] = S[x] | S[y]
        else:
            old = {x: S[x] for x in (*u[a:e], *v[a:e])}
            for x, y in zip(u[a:e], v[a:e]):
                S[x] |= old[y]
                S[y] |= old[x]
        a = e
    return S


def _columns(S, n):
    raw = b"".join(x.to_bytes((n + 7) // 8, "little") for x in S)
    return np.unpackbits(np.frombuffer(raw, np.uint8).reshape(n, -1), axis=1, bitorder="little")[:, :n]


def _hash(seed, j, n, k):
    p, state = (1 << 61) - 1, seed ^ j

    def step(s):
        s = (s + 0x9E3779B97F4A7C15) & MASK64
        z = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & MASK64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK64
        return s, z ^ (z >> 31)

    state = step(state)[1]
    A = []
    for _ in range(12):
        state, hi = step(state)
        state, lo = step(state)
        A.append((((hi % 2147483647) << 32) + lo % 2147483647) % p)
    cubic = lambda c, x: (((c[0] * x + c[1]) * x + c[2]) * x + c[3]) % p  # noqa: E731
    return [(cubic(A[:4], x & 0xFFFF) ^ cubic(A[4:8], x >> 16) ^ cubic(A[8:], (x & 0xFFFF) + (x >> 16))) % k for x in range(n)]


def _exact_hashed(case, seed):
    n, m, k, R = case["n"], case["m"], case["k"], case["R"]
    if n > 6_000 or m * R > 1_000_000:
        return None  # minutes in plain Python
    g = _generator(seed)
    u, v, t = (x.cpu().numpy() for x in _events(case, g))
    src = np.arange(n)
    if case["nsrc"]:
        src = np.sort(torch.randperm(n, generator=g, device="cuda")[:case["nsrc"]].cpu().numpy())
    exact = _columns(_component_rows(u.tolist(), v.tolist(), t, n), n)[:, src].sum(0, dtype=np.int64)
    hit = np.ones((n, len(src)), np.uint8)
    for j in range(R):
        h = np.array(_hash(_hash_seed(seed), j, n, k))
        P = _columns(_component_rows(h[u].tolist(), h[v].tolist(), t, k), k)
        hit &= P[h][:, h[src]]
    est = hit.sum(0, dtype=np.int64)
    d = np.abs(est - exact)
    rel = d / exact
    w1 = int(np.abs(np.sort(est) - np.sort(exact)).sum())
    c = len(src)
    err = dict(count=c, sum_abs=int(d.sum()), max_abs=int(d.max()), w1_num=w1, rel_sum=math.fsum(rel), max_rel=float(rel.max()),
               mean_abs=int(d.sum()) / c, mean_rel=math.fsum(rel) / c, w1=w1 / c)
    return dict(H=None, P=None, S=None, est=est, exact=exact, err=err)


def exact(case, seed):
    if case["kind"] == "hll":
        return _exact_hll(case, seed)
    if case["kind"] == "hashed":
        return _exact_hashed(case, seed)
    return None  # bits and counts: the same integers or wrong
