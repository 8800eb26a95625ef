// Scheduling of an event batch for the streaming kernel.
//
// Algorithm 1 (Section 3.1) is a strict sequence of row updates, but two
// events that share no node commute, and the columns of the matrix are
// independent.  The schedule groups the updates into "levels": inside a level
// no two updates conflict, so the streaming kernel can issue all of a level's
// row loads at once and only needs a barrier between levels.
//
// Equal timestamps (Section 2.1: adjacency needs dt > 0) are applied as one
// snapshot.  A group whose events share no node is a set of ordinary updates
// (EVENT: r = S[u] | S[v] into both rows).  Inside any other group G with node
// counts c(x) (occurrences of x in G):
//   * an event whose two ends both occur once in G is an ordinary update;
//   * a node y occurring once, whose partner x occurs several times, gets
//     ONEWAY: S[y] |= S[x] at level L (x is not written at level L);
//   * a node x occurring several times gets one PULL at level L+1:
//     S[x] |= OR of its partners' rows, where a partner y occurring once is
//     read from S[y] (already y_old | x_old: the extra x_old is harmless) and a
//     partner z occurring several times is read from a saved copy of z's old
//     row (COPY at level L into a temporary slot).
// This reproduces S_new[x] = S_old[x] | OR_{(x,y) in G} S_old[y] exactly.
// Directed events x -> y write only y: a lone event is ONEWAY y |= x, a group
// that shares nodes becomes one PULL per receiver, a sender that also receives
// in the group being read from its saved old row.
//
// The batch is cut into windows of about `window_events` events, never inside
// a timestamp group.  Each window is scheduled independently by one CTA
// (levels restart at every window, which acts as one extra barrier):
//   1. node ids of the window are compacted through a hash table;
//   2. groups of up to kPairGroup events are checked for shared nodes, pair by
//      pair, by all threads;
//   3. one warp walks the window in time order, 16 events (32 endpoints) at a
//      time, and assigns levels (level of an update = 1 + last level at which
//      any of its rows was touched); a group that shares nodes is scheduled on
//      the way, a large one by the whole CTA;
//   4. the window's updates are counting-sorted by level into packs that the
//      streaming kernel copies whole (tn_internal.cuh describes the layout).
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "tn_internal.cuh"

namespace tn {

constexpr int kPlanThreads = 512;
constexpr int kPlanThreadsSmall = 256;  // windows of up to 1,024 events
// Default window of plans that name a row buffer: its rows fit a record.
constexpr uint32_t kRecordWindow = 640;
constexpr uint32_t kDefaultSlab = 16;
constexpr uint32_t kRowBufferBytes = 160 * 1024;  // default shared-memory row buffer, slabs of up to 16 words
constexpr uint32_t kRowBufferWide = 192 * 1024;   // default (and largest) row buffer for wider slabs
constexpr uint32_t kEmpty = 0xFFFFFFFFu;
// Windows of up to this many events may become shared-memory records.
constexpr uint32_t kRecordEvents = 2048;
// Records are kept if more than one window in this many is one.
constexpr uint64_t kTileShare = 64;
// Groups of at least this many events go to the whole CTA unchecked: comparing
// their events pair by pair would cost more than the group's own phases (bursty
// n = 20,011, 500,009 events, groups of 107: plan 0.21 ms at 128, 0.18 ms at 48;
// uniform and activity-driven batches take the same time with both).
constexpr uint32_t kPairGroup = 48;
// Groups that share nodes and are no longer than this stay with the warp that walks
// the window: the CTA's barriers would take longer than the group (2.5 us each).
constexpr uint32_t kWarpGroup = 48;
// Default window of tiles.  Larger windows have fewer levels per event, each of
// which costs every CTA a barrier and a memory latency, but are scheduled by one CTA
// each and are stretched by large timestamp groups; 2,000 ops are one pack.  Schedule
// and apply at 1,280, 2,000, 2,480, 5,000 events: activity-driven n = 10^5, m = 10^7, 16
// words, 1.3 + 25.1, 1.3 + 23.2, 1.9 + 23.2, 1.8 + 20.7 ms; ER n = 10^4, m = 10^7, resident,
// 1.2 + 0.7, 1.2 + 0.6, 1.7 + 0.6, 1.5 + 0.6; bursty n = 2 10^5, m = 5 10^6, 32 words, 1.0 +
// 88.0, 1.0 + 91.6, 1.3 + 92.7, 2.1 + 91.0 (windows of two groups leave shared memory).  Short
// batches gain more from a short schedule: n = 1,000, 20,000 uniform events, resident,
// 94 + 65 us at 1,280, 114 + 62 at 2,000, 125 + 65 at 2,480.
static uint32_t default_window(uint64_t m) { return m < (1u << 16) ? 1280u : 2000u; }
// Room of the first pass's arena behind the target: a window is stretched by the
// rest of its last timestamp group (2,400 events at the largest default window: two
// CTAs per SM).
static uint64_t window_slack(uint32_t window) { return window < 320 ? 64 : window / 5; }
// Batches of at least this many events are copied into buffers of their exact size (8
// to 12 bytes per event); below it the staging buffers (44 to 53 bytes) are kept, except
// by plans made without a host wait: an online state with its own update stream keeps up
// to kOnlineFlight of them, and the serving engine charges a job for exact ones.
constexpr uint64_t kCompactEvents = 1ull << 20;
// Batches whose rows may all settle well before the end: component labels (three
// launches), for the forms that use them.
constexpr uint64_t kLabelEvents = 1ull << 17, kLabelFactor = 40;

// event flags of a window
constexpr uint8_t kFlagStart = 1;   // first event of its timestamp group
constexpr uint8_t kFlagHard = 2;    // on a group's first event: the group shares nodes
constexpr uint8_t kFlagDir = 4;     // directed event outside such a group: one ONEWAY
constexpr uint8_t kFlagNoop = 8;
constexpr uint8_t kFlagIso = 16;
constexpr uint8_t kFlagShA = 32;
constexpr uint8_t kFlagShB = 64;

__host__ __device__ inline uint64_t hash_slots(uint64_t E) { return ((3 * E + 31) / 32) * 32; }

// Arena of a window of E events, indices of type I (uint16_t in shared memory,
// uint32_t for windows scheduled in global memory).  The scratch part holds in
// turn the hash table (keys, ids), the node state (occurrences, last level,
// run) and the level bounds, pack table and last writers.
template <typename I>
__host__ __device__ inline uint64_t scratch_words(uint64_t E)
{
    const uint64_t H = hash_slots(E);
    uint64_t b = H * (4 + sizeof(I));
    const uint64_t state = 2 * E * (4 + 2 * sizeof(I));
    if (state > b) b = state;
    if (b < 16 * E) b = 16 * E;
    return (b + 3) / 4 + 64;
}

template <typename I>
__host__ __device__ inline uint64_t arena_bytes(uint64_t E)
{
    return (8 * ((E + 15) / 16) + 4 * (scratch_words<I>(E) + 3 * E) + sizeof(I) * 6 * E + E + 15) & ~15ull;
}

template <typename I>
struct Arena {
    uint32_t *rowsg;    // [2E] global id of every local row id
    uint32_t *run_lev;  // [E] fill counter, then level, of every PULL
    uint32_t *scratch;
    I *lu, *lv, *evl, *run_node, *run_aux, *run_temp;  // [E] each
    uint8_t *flg;       // [E]
    uint2 *chunk;       // [ceil(E / 16)] chunks of the level walk
    __device__ Arena(uint8_t *p, uint32_t E)
    {
        chunk = reinterpret_cast<uint2 *>(p);
        rowsg = reinterpret_cast<uint32_t *>(chunk + (E + 15) / 16);
        run_lev = rowsg + 2 * (uint64_t)E;
        scratch = run_lev + E;
        lu = reinterpret_cast<I *>(scratch + scratch_words<I>(E));
        lv = lu + E;
        evl = lv + E;
        run_node = evl + E;
        run_aux = run_node + E;
        run_temp = run_aux + E;
        flg = reinterpret_cast<uint8_t *>(run_temp + E);
    }
};

// Counters of a plan (device, one copy to the host per synchronisation).
struct PlanCounters {
    unsigned long long error;       // bit 0: id out of range, bit 1: time order
    unsigned long long late;        // windows left to the second pass
    unsigned long long arena;       // arena bytes of those scheduled in global memory
    unsigned long long big;         // how many of them are
    unsigned long long blob8, naux, list_words, items, ops, levels, local, temps;
    unsigned long long blob_used, aux_used;  // allocation of the exact buffers
    long long t_first, t_last;
    unsigned long long chain; // sum over the levels of tiles of their longest source list
    unsigned long long done;  // CTAs of the first pass
};

// device head of a plan: counters, status word, time bounds
struct PlanHead {
    PlanCounters cnt;
    int64_t tbounds[2];
    int32_t status;
    int32_t pad;
};

struct PlanArgs {
    Mail *mail;  // of the waiting thread, or nullptr
    uint32_t mail_seq;
    const uint32_t *u, *v;
    const int64_t *t;
    uint64_t m;
    uint32_t n;
    const int64_t *t_after;
    uint32_t window;     // target events per window
    uint32_t directed;   // 1: events are u -> v (only S[v] is updated)
    uint32_t nw;         // number of windows
    uint32_t first_max;  // largest window of the first pass (its shared-memory arena)
    uint32_t smem_max;   // largest window scheduled in shared memory
    uint32_t dcap;       // row slots of a local window
    uint32_t unit8;      // staging units (8 bytes) per event
    uint32_t chain;      // 1: count the longest source lists
    uint64_t *wstart;    // [nw + 1]
    uint32_t *naux_w;    // [nw] source-list entries of every window
    WinDesc *desc;       // [nw]
    uint2 *blob;         // window w: units blob_base(w) ...
    uint32_t *aux;       // window w: words 3 * s_w ...
    uint32_t *late_list; // [nw] windows of the second pass
    uint64_t *late_off;  // [nw] their arena offsets (kSmemArena: in shared memory)
    uint8_t *late_arena;
    PlanCounters *cnt;
    int64_t *tbounds;
};
constexpr uint64_t kSmemArena = ~0ull;

// Staging region of window w, starting at event s: 4 units per event hold 3 ops
// and the pack headers (at most one pack of 18 units per 64 levels or 2,030
// ops, and a window has at most one level per event), 5 units a record (10
// words per event); an even unit, so packs are 16-byte aligned.
__host__ __device__ inline uint64_t blob_base(uint64_t s, uint64_t w, uint32_t unit8)
{
    return ((unit8 * s + 1) & ~1ull) + 64 * w;
}

// ---------------------------------------------------------------------------
// validation (Section 2.1: nodes in [0, n), events time-ordered) and windows
// ---------------------------------------------------------------------------
// window w starts at the first timestamp-group start at or after w * window
__device__ inline uint64_t window_start(const PlanArgs &a, uint64_t w)
{
    uint64_t s = w * (uint64_t)a.window;
    if (w == 0) return 0;
    if (w >= a.nw || s >= a.m) return a.m;
    const int64_t key = a.t[s];
    if (key != a.t[s - 1]) return s;
    // first index with t > key: gallop, then binary search
    uint64_t lo = s, step = 1;
    while (lo + step < a.m && a.t[lo + step] <= key) {
        lo += step;
        step *= 2;
    }
    uint64_t hi = lo + step < a.m ? lo + step : a.m;  // t[lo] <= key, hi past it or the end
    while (lo + 1 < hi) {
        const uint64_t mid = lo + (hi - lo) / 2;
        if (a.t[mid] > key) hi = mid;
        else lo = mid;
    }
    return hi;
}

__global__ void inspect_kernel(PlanArgs a)
{
    const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, nt = (uint64_t)gridDim.x * blockDim.x;
    uint32_t bad = 0;
    for (uint64_t e = tid; e < a.m; e += nt) {
        if (a.u[e] >= a.n || a.v[e] >= a.n) bad |= 1u;
        if (e > 0 && a.t[e] < a.t[e - 1]) bad |= 2u;
    }
    if (tid == 0) {
        if (a.t_after && !(a.t[0] > *a.t_after)) bad |= 2u;
        a.cnt->t_first = a.tbounds[0] = a.t[0];
        a.cnt->t_last = a.tbounds[1] = a.t[a.m - 1];
        a.wstart[a.nw] = a.m;
    }
    if (bad) atomicOr(&a.cnt->error, (unsigned long long)bad);
    for (uint64_t w = tid; w < a.nw; w += nt) {
        const uint64_t s = window_start(a, w), e = window_start(a, w + 1);
        a.wstart[w] = s;
        if (e <= s || e - s <= a.first_max) continue;  // (e < s only in unordered input, refused as a whole)
        const uint64_t E = e - s;
        const unsigned long long slot = atomicAdd(&a.cnt->late, 1ull);
        a.late_list[slot] = (uint32_t)w;
        a.late_off[slot] = kSmemArena;
        if (E > a.smem_max) {
            atomicAdd(&a.cnt->big, 1ull);
            a.late_off[slot] = atomicAdd(&a.cnt->arena, (unsigned long long)arena_bytes<uint32_t>(E));
        }
    }
}

// ---------------------------------------------------------------------------
// per-window scheduler
// ---------------------------------------------------------------------------
__device__ inline uint32_t hslot(uint32_t key, uint32_t H)
{
    return (uint32_t)(((uint64_t)(key * 0x9E3779B1u) * H) >> 32);
}

__device__ inline void hinsert(uint32_t *hkey, uint32_t H, uint32_t key)
{
    uint32_t s = hslot(key, H);
    for (uint32_t probe = 0; probe < H; ++probe) {  // the table always has free slots
        uint32_t cur = hkey[s];
        if (cur == key) return;
        if (cur == kEmpty) {
            uint32_t prev = atomicCAS(&hkey[s], kEmpty, key);
            if (prev == kEmpty || prev == key) return;
        }
        s = (s + 1 == H) ? 0 : s + 1;
    }
}

template <typename I>
__device__ inline uint32_t hlookup(const uint32_t *hkey, const I *hval, uint32_t H, uint32_t key)
{
    uint32_t s = hslot(key, H);
    for (uint32_t probe = 0; probe < H && hkey[s] != key; ++probe) s = (s + 1 == H) ? 0 : s + 1;
    return hval[s];
}

// Appends of a warp to one counter per level: the lanes of one level take
// consecutive positions with a single shared-memory atomic.  All lanes call it.
__device__ inline uint32_t level_append(uint32_t *lh, uint32_t level, bool act)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t same = __match_any_sync(0xffffffffu, act ? level : 0xffffffffu);
    const uint32_t leader = __ffs(same) - 1;
    uint32_t base = 0;
    if (act && lane == leader) base = atomicAdd(&lh[level], (uint32_t)__popc(same));
    return __shfl_sync(0xffffffffu, base, leader) + __popc(same & ((1u << lane) - 1u));
}

// Scan state shared by the threads of a window's CTA: runs, source-list words,
// saved rows, largest level, next event, end of the group handed over.
enum { kScRuns = 0, kScAux, kScTemp, kScMaxlev, kScNext, kScEnd, kScCount };

// The snapshot rule for one timestamp group [i, g1), with every thread of the CTA
// or (kWarp) with one warp.  The numbering of runs and slots, the order of ops inside a level and
// of sources inside a PULL list are unspecified; none of them changes the
// result.  In an undirected group, nodes that occur once take part in exactly
// one event, so a lone event (both ends once) touches no other event's rows and
// gets its level at once; the other events share one level L = 1 + the latest
// level of their nodes, with the PULLs at L + 1.  Phases are separated by
// barriers, so a run's and a slot's number are final before anyone reads them.
template <typename I, bool kWarp>
__device__ __forceinline__ void schedule_group(uint32_t i, uint32_t g1, bool directed, const Arena<I> &A, uint32_t *ncnt, I *nlev,
                               I *nrun, uint32_t *auxw, uint32_t *sc)
{
    constexpr I kNone = (I)~(I)0, kClaim = (I)(kNone - 1);
    __shared__ uint32_t Lc, any, run0;
    const uint32_t T = kWarp ? 32u : blockDim.x, tid = kWarp ? threadIdx.x & 31u : threadIdx.x;
    auto phase_end = [] {
        if (kWarp) __syncwarp();
        else __syncthreads();
    };
    for (uint32_t j = i + tid; j < g1; j += T) {
        const uint32_t x = A.lu[j], y = A.lv[j];
        ncnt[x] = 0;
        ncnt[y] = 0;
        nrun[x] = kNone;
        nrun[y] = kNone;
    }
    if (tid == 0) {
        Lc = 0;
        any = 0;
        run0 = sc[kScRuns];
    }
    phase_end();
    for (uint32_t j = i + tid; j < g1; j += T) {
        const uint32_t x = A.lu[j], y = A.lv[j];
        if (x == y) continue;
        if (!directed) atomicAdd(&ncnt[x], 1u);
        atomicAdd(&ncnt[y], 1u);
    }
    phase_end();
    // roles; lone events' levels; one run (PULL) per node occurring several
    // times (directed: per receiver)
    auto claim_run = [&](uint32_t x) {
        if (atomicCAS(&nrun[x], kNone, kClaim) != kNone) return;
        const uint32_t r = atomicAdd(&sc[kScRuns], 1u);
        const uint32_t b = atomicAdd(&sc[kScAux], 1u + ncnt[x]);
        A.run_node[r] = (I)x;
        A.run_aux[r] = (I)b;
        A.run_lev[r] = 0;  // fill counter until the level is known
        A.run_temp[r] = kNone;
        auxw[b] = ncnt[x];
        nrun[x] = (I)r;
    };
    for (uint32_t j = i + tid; j < g1; j += T) {
        const uint32_t x = A.lu[j], y = A.lv[j];
        if (x == y) {
            A.flg[j] = kFlagNoop;
            continue;
        }
        const bool sx = directed || ncnt[x] > 1, sy = directed || ncnt[y] > 1;
        const uint32_t lev = max((uint32_t)nlev[x], (uint32_t)nlev[y]);
        if (!sx && !sy) {
            nlev[x] = (I)(lev + 1);
            nlev[y] = (I)(lev + 1);
            A.evl[j] = (I)(lev + 1);
            A.flg[j] = kFlagIso;
            atomicMax(&sc[kScMaxlev], lev + 1);
            continue;
        }
        atomicMax(&Lc, lev);
        any = 1;
        A.flg[j] = (sx ? kFlagShA : 0u) | (sy ? kFlagShB : 0u);
        if (sx && !directed) claim_run(x);
        if (sy) claim_run(y);
    }
    phase_end();
    // saved rows: a node with a run that another run reads is read from a copy
    // of its old row
    auto claim_temp = [&](uint32_t r) {
        if (atomicCAS(&A.run_temp[r], kNone, kClaim) == kNone) A.run_temp[r] = (I)atomicAdd(&sc[kScTemp], 1u);
    };
    for (uint32_t j = i + tid; j < g1; j += T)
        if (A.flg[j] == (kFlagShA | kFlagShB)) {
            if (nrun[A.lu[j]] != kNone) claim_temp(nrun[A.lu[j]]);
            if (!directed) claim_temp(nrun[A.lv[j]]);
        }
    phase_end();
    // source lists (entries: local row ids, or temp references)
    auto add_source = [&](uint32_t node, uint32_t from) {
        const uint32_t r = nrun[node];
        const uint32_t f = nrun[from];
        const uint32_t ref = f != kNone ? kTempRef | A.run_temp[f] : from;
        auxw[A.run_aux[r] + 1u + atomicAdd(&A.run_lev[r], 1u)] = ref;
    };
    for (uint32_t j = i + tid; j < g1; j += T) {
        const uint32_t f = A.flg[j];
        if (f & (kFlagNoop | kFlagIso)) continue;
        const uint32_t x = A.lu[j], y = A.lv[j];
        if ((f & kFlagShA) && !directed) add_source(x, y);
        if (f & kFlagShB) add_source(y, x);
    }
    phase_end();
    // levels of the shared part: ONEWAY / COPY at L, PULL at L + 1
    if (any) {
        const uint32_t L = Lc + 1;
        for (uint32_t j = i + tid; j < g1; j += T) {
            if (A.flg[j] & (kFlagNoop | kFlagIso)) continue;
            A.evl[j] = (I)L;
            nlev[A.lu[j]] = (I)(L + 1);
            nlev[A.lv[j]] = (I)(L + 1);
        }
        for (uint32_t r = run0 + tid; r < sc[kScRuns]; r += T) A.run_lev[r] = L;
        if (tid == 0) atomicMax(&sc[kScMaxlev], L + 1);
    }
    phase_end();
}

// Chunks of 16 events (32 endpoints: lane 2k + side holds one endpoint of event
// k), prepared by all warps: their events' flags, and per chunk the lanes that take
// part (no self-loops), whether a node occurs twice, whether a group that shares
// nodes begins in it.
constexpr uint32_t kChunkTwice = 1u, kChunkHard = 2u;

template <typename I>
__device__ __forceinline__ void prepare_chunks(uint32_t E, bool directed, const Arena<I> &A)
{
    const uint32_t lane = threadIdx.x & 31u, side = lane & 1u;
    const I *mine = side ? A.lv : A.lu;
    for (uint32_t c = threadIdx.x >> 5; 16 * c < E; c += blockDim.x >> 5) {
        const uint32_t e = 16 * c + (lane >> 1);
        const uint32_t x = e < E ? (uint32_t)mine[e] : 0u, f = e < E ? (uint32_t)A.flg[e] : 0u;
        const uint32_t other = __shfl_xor_sync(0xffffffffu, x, 1);
        const bool live = e < E && x != other;
        const uint32_t same = __match_any_sync(0xffffffffu, live ? x : 0x80000000u | lane);
        const bool twice = __any_sync(0xffffffffu, same & (same - 1u)), hard = __any_sync(0xffffffffu, f & kFlagHard);
        const uint32_t lanes = __ballot_sync(0xffffffffu, live);
        if (e < E && !side) A.flg[e] = (uint8_t)(f | (!live ? kFlagNoop : directed ? kFlagDir : kFlagIso));
        if (lane == 0) A.chunk[c] = make_uint2(lanes, (twice ? kChunkTwice : 0u) | (hard ? kChunkHard : 0u));
    }
}

// Levels of the events from sc[kScNext] up to the next group that shares nodes,
// by warp 0.  Each event's level needs only its two nodes' last levels, so a chunk
// without repeated nodes takes one round: a shared-memory read, a shuffle, a write.
// In a chunk with repeated nodes an event waits until the earlier events on its
// nodes are done.  One warp's walk is bound by the number of dependent
// instructions, so everything else about a chunk is prepared by all warps (550
// cycles a chunk before, 770 with a match in every chunk).
template <typename I>
__device__ __forceinline__ void scan_levels(uint32_t E, const Arena<I> &A, I *nlev, uint32_t *sc)
{
    const uint32_t lane = threadIdx.x & 31u, side = lane & 1u;
    const I *mine = side ? A.lv : A.lu;
    const uint32_t first = sc[kScNext];
    uint32_t c = first >> 4, top = 0, end = E;
    const uint32_t chunks = (E + 15u) >> 4;
    // events before `first` are done
    uint32_t keep = 0xffffffffu << (2u * (first & 15u));
    auto load = [&](uint32_t k) {
        const uint32_t e = 16 * k + (lane >> 1);
        return e < E ? (uint32_t)mine[e] : 0u;
    };
    uint32_t x = load(c);
    uint2 info = c < chunks ? A.chunk[c] : make_uint2(0u, 0u);
    for (; c < chunks; ++c) {
        const uint32_t node = x, e = 16 * c + (lane >> 1), what = info.y;
        uint32_t lanes = info.x & keep, stop = 16u;
        keep = 0xffffffffu;
        x = load(c + 1);
        if (c + 1 < chunks) info = A.chunk[c + 1];
        if (what & kChunkHard) {  // the first such group at or behind `first` ends the walk
            const uint32_t hard = __ballot_sync(0xffffffffu, e >= first && e < E && (A.flg[e] & kFlagHard));
            if (hard) {
                stop = (__ffs(hard) - 1) >> 1;
                lanes &= (1u << (2u * stop)) - 1u;
            }
        }
        const bool live = (lanes >> lane) & 1u;
        uint32_t lev = 0;
        if (!(what & kChunkTwice)) {
            lev = live ? (uint32_t)nlev[node] : 0u;
            lev = max(lev, __shfl_xor_sync(0xffffffffu, lev, 1)) + 1u;
            if (live) nlev[node] = (I)lev;
        } else {
            const uint32_t same = __match_any_sync(0xffffffffu, live ? node : 0x80000000u | lane);
            const uint32_t before = same & ((1u << lane) - 1u);
            uint32_t pending = lanes;
            while (pending) {
                const uint32_t ready = __ballot_sync(0xffffffffu, ((pending >> lane) & 1u) && !(before & pending));
                const uint32_t both = ready & (((ready & 0x55555555u) << 1) | ((ready >> 1) & 0x55555555u));
                const bool go = (both >> lane) & 1u;
                uint32_t l = go ? (uint32_t)nlev[node] : 0u;
                l = max(l, __shfl_xor_sync(0xffffffffu, l, 1)) + 1u;
                if (go) {
                    nlev[node] = (I)l;
                    lev = l;
                }
                __syncwarp();
                pending &= ~both;
            }
        }
        __syncwarp();
        if (live) {
            A.evl[e] = (I)lev;  // (both endpoints' lanes write the same level)
            top = max(top, lev);
        }
        if (stop < 16u) {
            end = 16 * c + stop;
            break;
        }
    }
    __syncwarp();
    top = __reduce_max_sync(0xffffffffu, top);
    const uint32_t next = end < E ? end : E;
    // end of the group at `next`
    uint32_t g1 = next + 1;
    if (next < E) {
        for (;;) {
            const uint32_t e = g1 + lane;
            const uint32_t starts = __ballot_sync(0xffffffffu, e >= E || (A.flg[e] & kFlagStart));
            if (starts) {
                g1 += __ffs(starts) - 1;
                break;
            }
            g1 += 32u;
        }
        if (g1 > E) g1 = E;
    }
    if (lane == 0) {
        sc[kScNext] = next;
        sc[kScEnd] = g1;
        if (top > sc[kScMaxlev]) sc[kScMaxlev] = top;
    }
}

// kTiles: a window that was scheduled as a record, again as tiles.
template <typename I, bool kTiles = false>
__device__ __forceinline__ void schedule_window(const PlanArgs &a, uint32_t w, uint8_t *arena)
{
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t tot;
    __shared__ uint32_t sc[kScCount];
    __shared__ uint32_t res[3];  // packs, units, lists outside the packs

    const uint64_t s = a.wstart[w];
    const uint32_t E = (uint32_t)(a.wstart[w + 1] - s);
    const uint32_t T = blockDim.x, tid = threadIdx.x, lane = tid & 31u;
    WinDesc *desc = a.desc + w;
    const uint32_t record_units = kTiles ? desc->pack[0] : 0u;  // (overwritten below, by thread 0 at the earliest)
    if (E == 0) {
        if (tid == 0) {
            *desc = WinDesc{};
            a.naux_w[w] = 0;
        }
        return;
    }
    const Arena<I> A(arena, E);
    const uint32_t *U = a.u + s, *V = a.v + s;
    const int64_t *Tt = a.t + s;

    // 1. local row ids 0..D-1: the node ids themselves in a network of at most
    //    2E nodes (unless the window may become a record, whose rows are
    //    gathered), else compacted through a hash table.  The endpoints wait in
    //    rowsg until it is filled.
    const bool direct = a.unit8 < 5 && a.n <= 2 * (uint64_t)E;
    uint32_t D;
    for (uint32_t i0 = 0; i0 < E; i0 += 4 * T) {
        uint32_t uu[4], vv[4];
        int64_t ta[4], tb[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t i = i0 + q * T + tid;
            const bool in = i < E;
            uu[q] = in ? U[i] : 0u;
            vv[q] = in ? V[i] : 0u;
            ta[q] = in ? Tt[i] : 0;
            tb[q] = in && i ? Tt[i - 1] : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t i = i0 + q * T + tid;
            if (i >= E) continue;
            A.flg[i] = (i == 0 || ta[q] != tb[q]) ? kFlagStart : 0;
            if (direct) {
                A.lu[i] = (I)uu[q];
                A.lv[i] = (I)vv[q];
            } else {
                A.rowsg[i] = uu[q];
                A.rowsg[E + i] = vv[q];
            }
        }
    }
    if (tid < kScCount) sc[tid] = 0;
    if (direct) {
        D = a.n;
        for (uint32_t i = tid; i < D; i += T) A.rowsg[i] = i;
        __syncthreads();
    } else {
        const uint32_t H = (uint32_t)hash_slots(E);
        uint32_t *hkey = A.scratch;
        I *hval = reinterpret_cast<I *>(A.scratch + H);
        for (uint32_t i = tid; i < H; i += T) hkey[i] = kEmpty;
        __syncthreads();
        for (uint32_t i = tid; i < 2 * E; i += T) hinsert(hkey, H, A.rowsg[i]);
        __syncthreads();
        for (uint32_t i = tid; i < H; i += T) hval[i] = hkey[i] != kEmpty ? 1 : 0;
        __syncthreads();
        D = block_excl_scan_array(hval, H, warp_sums, &tot);
        for (uint32_t i = tid; i < 2 * E; i += T) A.lu[i] = (I)hlookup(hkey, hval, H, A.rowsg[i]);  // lu, then lv
        __syncthreads();
        for (uint32_t i = tid; i < H; i += T)
            if (hkey[i] != kEmpty) A.rowsg[hval[i]] = hkey[i];
        __syncthreads();
    }
    uint32_t *ncnt = A.scratch;
    I *nlev = reinterpret_cast<I *>(A.scratch + 2 * (uint64_t)E), *nrun = nlev + 2 * (uint64_t)E;
    for (uint32_t i = tid; i < D; i += T) nlev[i] = 0;

    // 2. groups that share nodes (marked on their first event)
    for (uint32_t i = tid; i < E; i += T) {
        const uint32_t x = A.lu[i], y = A.lv[i];
        bool shared = false;
        uint32_t j = i + 1;
        for (; j < E && j - i < kPairGroup && !(A.flg[j] & kFlagStart) && !shared; ++j) {
            const uint32_t p = A.lu[j], q = A.lv[j];
            shared = x != y && p != q && (x == p || x == q || y == p || y == q);
        }
        if (!shared) {
            if (j - i >= kPairGroup && (A.flg[i] & kFlagStart)) A.flg[i] = kFlagStart | kFlagHard;
            continue;
        }
        uint32_t g = i;
        while (!(A.flg[g] & kFlagStart) && i - g < kPairGroup) --g;  // (a larger group is marked by its first event)
        if (A.flg[g] & kFlagStart) A.flg[g] = kFlagStart | kFlagHard;
    }
    __syncthreads();

    // 3. levels in time order
    prepare_chunks(E, a.directed != 0, A);
    __syncthreads();
    uint32_t *auxw = a.aux + 3 * s;
    for (;;) {
        if (tid < 32) {
            for (;;) {
                scan_levels(E, A, nlev, sc);
                __syncwarp();
                const uint32_t i = sc[kScNext], g1 = sc[kScEnd];
                if (i >= E || g1 - i > kWarpGroup) break;
                schedule_group<I, true>(i, g1, a.directed != 0, A, ncnt, nlev, nrun, auxw, sc);
                if (lane == 0) sc[kScNext] = g1;
                __syncwarp();
            }
        }
        __syncthreads();
        const uint32_t next = sc[kScNext], end = sc[kScEnd];
        if (next >= E) break;
        schedule_group<I, false>(next, end, a.directed != 0, A, ncnt, nlev, nrun, auxw, sc);
        if (tid == 0) sc[kScNext] = end;
        __syncthreads();
    }
    const uint32_t maxlev = sc[kScMaxlev], naux = sc[kScAux], ntemp = sc[kScTemp], nruns = sc[kScRuns];
    __syncthreads();

    // 4. counting sort of the updates by level (levels 1..maxlev -> 0..maxlev-1)
    uint32_t *lh = A.scratch;  // node state is dead
    for (uint32_t j = tid; j < maxlev + 1; j += T) lh[j] = 0;
    __syncthreads();
    // an event is one op: EVENT, a directed ONEWAY, or the ONEWAY of its end that occurs once
    auto has_op = [&](uint32_t i) {
        const uint32_t f = i < E ? (uint32_t)A.flg[i] : (uint32_t)kFlagNoop;
        return !(f & kFlagNoop) && (f & (kFlagShA | kFlagShB)) != (kFlagShA | kFlagShB);
    };
    for (uint32_t i0 = 0; i0 < E; i0 += T) {
        const uint32_t i = i0 + tid;
        const bool act = has_op(i);
        level_append(lh, act ? A.evl[i] - 1u : 0u, act);
    }
    for (uint32_t r = tid; r < nruns; r += T) {
        const uint32_t L = A.run_lev[r];
        atomicAdd(&lh[L], 1u);  // PULL at level L+1 -> index L
        if (A.run_temp[r] != (I)~(I)0) atomicAdd(&lh[L - 1], 1u);
    }
    __syncthreads();
    const uint32_t nops = block_excl_scan_array(lh, maxlev + 1, warp_sums, &tot);

    // 5. mode: the window's rows and saved rows fit the streaming kernel's
    //    shared-memory row buffer, and its record fits one staging buffer
    const uint32_t rec_words = 4 + D + (maxlev + 1) + nops + naux;
    const uint32_t rec_words_pad = (rec_words + 3u) & ~3u;
    const bool local = !kTiles && E <= kRecordEvents && a.unit8 >= 5 && D + ntemp <= a.dcap && rec_words_pad <= kRecordWords;
    const uint64_t region = blob_base(s, w, a.unit8);

    if (local) {
        // record: header | rows[D] | lvl[maxlev+1] | ops[nops] | aux[naux] | pad
        uint32_t *pack = reinterpret_cast<uint32_t *>(a.blob + region);
        uint32_t *rec = pack + 4;
        uint32_t *rrows = rec + 4, *rlvl = rrows + D, *rops = rlvl + maxlev + 1, *raux = rops + nops;
        if (tid == 0) {
            pack[0] = nops;
            pack[1] = (kPackLocal | kPackWindow) << 16;
            pack[2] = pack[3] = 0;
            rec[0] = D;
            rec[1] = ntemp;
            rec[2] = maxlev;
            rec[3] = nops;
        }
        for (uint32_t d = tid; d < D; d += T) rrows[d] = A.rowsg[d];
        for (uint32_t j = tid; j < maxlev + 1; j += T) rlvl[j] = lh[j];
        for (uint32_t k = rec_words + tid; k < rec_words_pad; k += T) rec[k] = 0;
        for (uint32_t r = tid; r < nruns; r += T) {
            const uint32_t b = A.run_aux[r], c = auxw[b];
            raux[b] = c;
            for (uint32_t q = 1; q <= c; ++q) {
                const uint32_t ref = auxw[b + q];
                raux[b + q] = (ref & kTempRef) ? D + (ref & ~kTempRef) : ref;
            }
        }
        __syncthreads();
        for (uint32_t i0 = 0; i0 < E; i0 += T) {
            const uint32_t i = i0 + tid;
            const bool act = has_op(i);
            const uint32_t pos = level_append(lh, act ? A.evl[i] - 1u : 0u, act);
            if (!act) continue;
            const uint32_t f = A.flg[i], x = A.lu[i], y = A.lv[i];
            rops[pos] = (f & kFlagIso) ? local_op(kEvent, x, y)
                        : ((f & kFlagDir) || (f & kFlagShA)) ? local_op(kOneway, y, x)  // y |= x
                                                             : local_op(kOneway, x, y);
        }
        for (uint32_t r = tid; r < nruns; r += T) {
            const uint32_t L = A.run_lev[r];
            rops[atomicAdd(&lh[L], 1u)] = local_op(kPull, A.run_node[r], A.run_aux[r]);
            if (A.run_temp[r] != (I)~(I)0)
                rops[atomicAdd(&lh[L - 1], 1u)] = local_op(kCopy, D + A.run_temp[r], A.run_node[r]);
        }
        // last write of every row: ops are in level order and a level writes a
        // row at most once, so it is the op with the highest index writing it
        uint32_t *lastw = A.scratch + maxlev + 2;  // lh holds scratch[0 .. maxlev]
        for (uint32_t d = tid; d < D; d += T) lastw[d] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < nops; i += T) {
            const uint32_t op = rops[i], kind = op >> kKindShift;
            if (kind == kCopy) continue;  // writes a saved copy, not a row
            atomicMax(&lastw[(op >> kLocalBits) & kLocalMask], i + 1);
            if (kind == kEvent) atomicMax(&lastw[op & kLocalMask], i + 1);
        }
        __syncthreads();
        for (uint32_t i = tid; i < nops; i += T) {
            uint32_t op = rops[i];
            const uint32_t kind = op >> kKindShift;
            if (kind == kCopy) continue;
            if (lastw[(op >> kLocalBits) & kLocalMask] == i + 1) op |= kLastA;
            if (kind == kEvent && lastw[op & kLocalMask] == i + 1) op |= kLastB;
            rops[i] = op;
        }
        if (tid == 0) {
            res[0] = nops ? 1u : 0u;
            res[1] = 2 + rec_words_pad / 2;
            WinDesc d{};
            d.off = region;
            d.npacks = res[0];
            d.pack[0] = res[1];
            *desc = d;
            a.naux_w[w] = 0;
        }
    } else {
        // packs: as many whole levels as fit with the source lists of their PULLs;
        // a level whose lists do not fit keeps them in the plan's list buffer, and
        // one with more ops than a pack holds is cut.  Warp 0 cuts the packs and
        // writes their headers.
        uint32_t *la = A.scratch + maxlev + 2;  // list words of the levels before
        uint32_t *lm = la + maxlev + 2;         // longest list of the level (a.chain)
        uint32_t *pq = lm + maxlev + 2;         // per pack: first op, its unit, next free list word (0: none), spare
        const bool chain = a.chain && nruns;
        for (uint32_t j = tid; j < maxlev + 1; j += T) {
            la[j] = 0;
            if (chain) lm[j] = 0;
        }
        __syncthreads();
        for (uint32_t r = tid; r < nruns; r += T) {
            const uint32_t c = auxw[A.run_aux[r]];
            atomicAdd(&la[A.run_lev[r]], 1u + c);
            if (chain) atomicMax(&lm[A.run_lev[r]], c);
        }
        __syncthreads();
        if (chain && tid >= T - 32) {  // (the last warp: warp 0 cuts the packs)
            uint32_t sum = 0;
            for (uint32_t j = lane; j < maxlev + 1; j += 32) sum += lm[j];
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (lane == 0 && sum) atomicAdd(&a.cnt->chain, (unsigned long long)sum);
        }
        block_excl_scan_array(la, maxlev + 1, warp_sums, &tot);
        if (tid < 32) {
            uint32_t p = 0, l = 0, q = 0, unit = 0, outside = 0;
            while (q < nops) {
                uint32_t rel[2], list[2], with[2], fit[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t j = l + 1 + lane + 32 * h;
                    rel[h] = j <= maxlev ? lh[j] - q : 0x10000000u;
                    list[h] = j <= maxlev ? la[j] - la[l] : 0u;
                    with[h] = __popc(__ballot_sync(0xffffffffu, rel[h] + (list[h] + 1) / 2 <= kPackOps));
                    fit[h] = __popc(__ballot_sync(0xffffffffu, rel[h] <= kPackOps));
                }
                const uint32_t kw = with[0] + (with[0] == 32u ? with[1] : 0u);
                // levels whose lists stay outside: one at a time, or a part of one
                const uint32_t k = kw ? kw : fit[0] ? 1u : 0u;
                const uint32_t last = k ? lh[l + k] - q : kPackOps;
                const uint32_t words = kw ? la[l + k] - la[l] : 0u;
                uint32_t *hdr = reinterpret_cast<uint32_t *>(a.blob + region + unit);
                uint16_t *seg = reinterpret_cast<uint16_t *>(hdr + 4);
                if (lane == 0) {
                    hdr[0] = last;
                    hdr[1] = (k ? k : 1u) | (q == 0 ? kPackWindow << 16 : 0u) | (nruns ? kPackTies << 16 : 0u);
                    hdr[2] = hdr[3] = 0;
                    pq[4 * p] = q;
                    pq[4 * p + 1] = unit + kPackHead;
                    pq[4 * p + 2] = kw ? 2 * (kPackHead + last) : 0u;
                    if (!k) seg[0] = (uint16_t)last;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (lane + 32 * h < k) seg[lane + 32 * h] = (uint16_t)rel[h];
                if (!kw) outside = 1;
                unit += (kPackHead + last + (words + 1) / 2 + 1u) & ~1u;
                q += last;
                l += k;
                ++p;
            }
            if (lane == 0) {
                res[0] = p;
                res[1] = unit;
                res[2] = outside;
            }
        }
        __syncthreads();
        const uint32_t np = res[0];
        uint2 *ops = a.blob + region;
        auto pack_of = [&](uint32_t pos) -> uint32_t {
            uint32_t lo = 0, hi = np;
            while (lo + 1 < hi) {
                const uint32_t mid = (lo + hi) / 2;
                if (pq[4 * mid] <= pos) lo = mid;
                else hi = mid;
            }
            return lo;
        };
        auto place = [&](uint32_t pos) -> uint2 * {
            const uint32_t p = pack_of(pos);
            return ops + pq[4 * p + 1] + (pos - pq[4 * p]);
        };
        for (uint32_t i0 = 0; i0 < E; i0 += T) {
            const uint32_t i = i0 + tid;
            const bool act = has_op(i);
            const uint32_t pos = level_append(lh, act ? A.evl[i] - 1u : 0u, act);
            if (!act) continue;
            const uint32_t f = A.flg[i], x = A.rowsg[A.lu[i]], y = A.rowsg[A.lv[i]];
            *place(pos) = (f & kFlagIso) ? make_uint2(op_a(kEvent, x), y)
                          : ((f & kFlagDir) || (f & kFlagShA)) ? make_uint2(op_a(kOneway, y), x)  // y |= x
                                                               : make_uint2(op_a(kOneway, x), y);
        }
        for (uint32_t r = tid; r < nruns; r += T) {
            const uint32_t L = A.run_lev[r], xg = A.rowsg[A.run_node[r]], b = A.run_aux[r], c = auxw[b];
            const uint32_t pos = atomicAdd(&lh[L], 1u), p = pack_of(pos);
            uint32_t *list = auxw + b;
            uint32_t where = kOutsideList + (uint32_t)(3 * s) + b;
            if (pq[4 * p + 2]) {
                where = atomicAdd(&pq[4 * p + 2], 1u + c);
                list = reinterpret_cast<uint32_t *>(ops + pq[4 * p + 1] - kPackHead) + where;
                list[0] = c;
            }
            for (uint32_t q = 1; q <= c; ++q) {  // lists name rows by node id
                const uint32_t ref = auxw[b + q];
                list[q] = (ref & kTempRef) ? ref : A.rowsg[ref];
            }
            ops[pq[4 * p + 1] + (pos - pq[4 * p])] = make_uint2(op_a(kPull, xg), where);
            if (A.run_temp[r] != (I)~(I)0)
                *place(atomicAdd(&lh[L - 1], 1u)) = make_uint2(op_a(kCopy, A.run_temp[r]), xg);
        }
        // pack sizes: the first kDescPacks in the descriptor, all of them behind
        // the packs when there are more
        for (uint32_t p = tid; p < np; p += T) {
            const uint32_t b = pq[4 * p + 1] - kPackHead, e = p + 1 < np ? pq[4 * p + 5] - kPackHead : res[1];
            if (p < kDescPacks) desc->pack[p] = e - b;
            if (np > kDescPacks) reinterpret_cast<uint32_t *>(ops + res[1])[p] = e - b;
        }
        if (tid == 0) {
            desc->off = region;
            desc->npacks = np;
            desc->tab = res[1];
            a.naux_w[w] = res[2] ? naux : 0u;
            if (res[2]) atomicAdd(&a.cnt->list_words, (unsigned long long)naux);
        }
    }
    if (tid == 0) {
        PlanCounters *c = a.cnt;
        const uint32_t units = res[1] + (res[0] > kDescPacks ? (res[0] + 1) / 2 : 0u);
        atomicAdd(&c->blob8, (unsigned long long)((units + 1) & ~1u) - record_units);
        atomicAdd(&c->items, (unsigned long long)res[0] - (kTiles ? 1u : 0u));
        if (kTiles) {  // (a record, counted once already)
            atomicAdd(&c->local, ~0ull);
        } else {
            atomicAdd(&c->ops, (unsigned long long)nops);
            atomicAdd(&c->levels, (unsigned long long)maxlev);
        }
        if (local) {
            atomicAdd(&c->local, 1ull);
        } else {
            if (naux) atomicAdd(&c->naux, (unsigned long long)naux);
            if (ntemp) atomicMax(&c->temps, (unsigned long long)ntemp);
        }
    }
}

// First pass: every window that fits the arena of this launch.  What bounds it
// is latency: the level walk of one warp per window (about 100 cycles per 16
// events) between phases of scattered shared-memory accesses.  Small windows
// leave room for several CTAs per SM; 512 threads shorten the parallel phases of
// large ones.  tn_plan_create on 10^7 activity-driven events (n = 10^5, windows of
// 2,000): 1.27 ms; windows of 640: 1.16 ms; with one thread walking each window event by event (137 us a
// window) and three host waits 3.4 ms.  20,000 uniform events: 0.09 ms (0.34).
__global__ void __launch_bounds__(kPlanThreads) schedule_first_kernel(PlanArgs a)
{
    extern __shared__ __align__(16) uint8_t smem_arena[];
    const uint32_t w = blockIdx.x;
    // refused input: window bounds may not be ordered; too large: second pass
    if (!a.cnt->error && a.wstart[w + 1] - a.wstart[w] <= a.first_max) schedule_window<uint16_t>(a, w, smem_arena);
    if (!a.mail) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&a.cnt->done, 1ull) == gridDim.x - 1) {
            __threadfence();
            mail_send(a.mail, a.mail_seq, a.cnt);
        }
    }
}

// Second pass: windows stretched by a large timestamp group, in all of shared
// memory or, above that, in global memory.
__global__ void __launch_bounds__(kPlanThreads) schedule_late_kernel(PlanArgs a)
{
    extern __shared__ __align__(16) uint8_t smem_arena[];
    const uint32_t w = a.late_list[blockIdx.x];
    const uint64_t off = a.late_off[blockIdx.x];
    if (off == kSmemArena) schedule_window<uint16_t>(a, w, smem_arena);
    else schedule_window<uint32_t>(a, w, a.late_arena + off);
}

// The few records of a plan of tiles, as tiles: records keep no track of rows, so one
// of them would have every update of the plan executed.  A tile's descriptor has
// tab > 0.
__global__ void __launch_bounds__(kPlanThreads) schedule_tiles_kernel(PlanArgs a)
{
    extern __shared__ __align__(16) uint8_t smem_arena[];
    const WinDesc *desc = a.desc + blockIdx.x;
    if (desc->npacks == 0 || desc->tab != 0) return;
    schedule_window<uint16_t, true>(a, blockIdx.x, smem_arena);
}

// Copies the plan into a buffer of its exact size: what a finished plan needs of the
// head, and every window (in no particular order: descriptors name offsets) with its
// PULL lists.
__global__ void compact_kernel(PlanArgs a, PlanHead *head, WinDesc *to_desc, uint2 *blob, uint32_t *aux)
{
    __shared__ unsigned long long base[2];
    const uint32_t w = blockIdx.x;
    const WinDesc *desc = a.desc + w;
    const uint32_t np = desc->npacks;
    if (threadIdx.x == 0) {
        if (w == 0) {
            head->tbounds[0] = a.tbounds[0];
            head->tbounds[1] = a.tbounds[1];
            head->status = 0;
        }
        to_desc[w] = *desc;
    }
    if (np == 0) return;
    const uint64_t src = desc->off;
    const uint32_t naux = a.naux_w[w];
    uint32_t units = 0;
    if (np > kDescPacks) units = desc->tab + (np + 1) / 2;
    else
        for (uint32_t p = 0; p < np; ++p) units += desc->pack[p];
    units = (units + 1) & ~1u;
    if (threadIdx.x == 0) {
        base[0] = atomicAdd(&a.cnt->blob_used, (unsigned long long)units);
        base[1] = naux ? atomicAdd(&a.cnt->aux_used, (unsigned long long)naux) : 0ull;
    }
    __syncthreads();
    const uint64_t dst = base[0];
    const uint4 *from = reinterpret_cast<const uint4 *>(a.blob + src);
    uint4 *to = reinterpret_cast<uint4 *>(blob + dst);
    for (uint32_t k = threadIdx.x; k < units / 2; k += blockDim.x) to[k] = from[k];
    if (threadIdx.x == 0) to_desc[w].off = dst;
    if (naux == 0) return;
    const uint64_t s3 = 3 * a.wstart[w];
    for (uint32_t k = threadIdx.x; k < naux; k += blockDim.x) aux[base[1] + k] = a.aux[s3 + k];
    __syncthreads();
    const uint32_t *table = reinterpret_cast<const uint32_t *>(a.blob + src + desc->tab);
    uint32_t u0 = 0;
    for (uint32_t p = 0; p < np; ++p) {
        const uint32_t n8 = np > kDescPacks ? table[p] : desc->pack[p];
        const uint32_t nops = a.blob[src + u0].x;
        uint2 *ops = blob + dst + u0 + kPackHead;
        for (uint32_t k = threadIdx.x; k < nops; k += blockDim.x)
            if ((ops[k].x >> kKindShift) == kPull && ops[k].y >= kOutsideList) ops[k].y = (uint32_t)(ops[k].y - s3 + base[1]);
        u0 += n8;
    }
}

// ---------------------------------------------------------------------------
// connected components of the batch's events (long batches): once every row equals
// its component's root row, no event can change anything any more, and a CTA stops
// reading the schedule.  Lock-free union by smaller
// id; a parent read from a stale cache line is still an ancestor, and a failed
// compare-and-swap returns the true one.  10^7 events on 10^4 nodes: 0.03 ms.
// ---------------------------------------------------------------------------
__global__ void label_init_kernel(uint32_t *parent, uint32_t n)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) parent[i] = i;
}

__device__ inline uint32_t label_root(const uint32_t *parent, uint32_t x)
{
    for (uint32_t p = parent[x]; p != x; p = parent[x]) x = p;  // ids fall along a path
    return x;
}

__global__ void label_union_kernel(const uint32_t *u, const uint32_t *v, uint64_t m, uint32_t *parent)
{
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < m; e += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t x = label_root(parent, u[e]), y = label_root(parent, v[e]);
        while (x != y) {
            if (x < y) {
                const uint32_t z = x;
                x = y;
                y = z;
            }
            const uint32_t was = atomicCAS(&parent[x], x, y);  // x > y: paths keep falling
            if (was == x) break;
            x = label_root(parent, was);
            y = label_root(parent, y);
        }
        // short paths for the events that follow
        if (parent[u[e]] != y) atomicMin(&parent[u[e]], y);
        if (parent[v[e]] != y) atomicMin(&parent[v[e]], y);
    }
}

__global__ void label_flatten_kernel(uint32_t *parent, uint32_t n)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t x = i;
        for (uint32_t p = *(volatile uint32_t *)&parent[x]; p != x; p = *(volatile uint32_t *)&parent[x]) x = p;
        parent[i] = x;
    }
}

template <typename F>
static uint32_t largest_window(uint64_t budget, F bytes)
{
    uint32_t E = 64;
    while (bytes(E + 64) <= budget) E += 64;
    return E;
}

// largest window whose arena fits shared memory
static uint32_t smem_max_events()
{
    static uint32_t cached = 0;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (cached) return cached;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // (static shared memory of the kernels: at most 1 KB)
    cached = largest_window((uint64_t)optin - 1024, [](uint64_t E) { return arena_bytes<uint16_t>(E); });
    return cached;
}

template <typename T>
static cudaError_t alloc_async(T **p, uint64_t count, cudaStream_t st)
{
    *p = nullptr;
    if (count == 0) return cudaSuccess;
    return cudaMallocAsync((void **)p, count * sizeof(T), st);
}

}  // namespace tn

using namespace tn;

static void free_plan_buffers(tn_plan *p, cudaStream_t st)
{
    if (p->batch_plan) {
        free_plan_buffers(p->batch_plan, st);
        free(p->batch_plan);
    }
    if (p->d_mem) cudaFreeAsync(p->d_mem, st);
    if (p->d_label) cudaFreeAsync(p->d_label, st);
}

// Whether a schedule made for tiles is walked faster as records, in shared memory:
// one of short levels, over rows that mostly do not settle.  A level costs a CTA 0.27 us
// there, 0.85 us (8 words) to 1.5 us (32 words) in tiles, which win by the rows that they
// need not move.  Apply, tiles and records:
//  - without ties.  Streams around 96 hubs (60 ops a level), n = 6 10^4: 6 events a node
//    7.6 and 4.5 ms, 24 events a node 28.2 and 17.4, 50 events a node (every row settles)
//    28.8 and 35.3; 256 hubs (119), n = 2 10^5: 11.7 and 7.2; activity-driven, n =
//    2.6 10^4 (122): 2.1 and 2.1, n = 6 10^4 (202): 9.4 and 11.3.  In narrow slabs (few
//    columns) records gain, 5,000 columns, 2 words: activity-driven n = 2.6 10^4 (128) 2.1
//    and 1.4, n = 6 10^4 (218) 3.5 and 2.9, n = 10^5 (293) 2.7 and 2.8.  64 hubs (44), n =
//    10^5, 32 words 63.3 and 18.7.
//  - large timestamp groups that share nodes.  Bursty n = 2.6 10^4, m = 10^6 (81): 21.0
//    and 15.5 ms; n = 10^5, m = 5 10^6 (306): 90.1 and 62.2; n = 1.2 10^5, m = 10^6
//    (424): 14.5 and 14.6; n = 2 10^5, m = 5 10^6 (645): 92 and 137.
// Resident CTAs walk a level in 0.1 us (rows of two words 0.12, in packs with ties 0.17
// and 0.2), but one thread combines a PULL's sources (27 or 36 ns each, all others wait
// at the level's barrier), every wave of CTAs walks all levels, and 16-word records of
// such a network take one wave.  Levels of settled rows are not walked: from about 11
// events a node on, with long source lists from about 24.  Apply (estimate) around one
// hub, n = 24,000, m = 200,000:
//   groups of 3, 8, 64 events: resident 75.3 (78.9), 41.3 (41.8), 19.0 (19.5) ms, records
//   45.5 (40.5), 15.4 (16.5), 4.3 (4.3); no groups 59.9 (60.3), 54.3 (55.6); 30 events a
//   node in groups of 4: 97.8 (114), records 108 (107); n = 12,000, groups of 8, 64: 16.1
//   (17.2), 7.3 (8.5), records 15.3 (16.5), 4.3 (4.3).  Bursty n = 20,011, m = 500,009:
//   6.1, records 7.1 (6.3).  The margin covers the error.  Sketches (byte-wise maximum)
//   pay 42 ns a source, and 39 in records: one hub, groups of 64, n = 20,000, m = 300,000,
//   p = 10 14.9, records 16.5; p = 12 (four waves) 28.5 and 17.6.
// From kRecordLevels levels on: below, the second schedule takes as long as it saves.
constexpr uint64_t kRecordLevels = 256;
static bool records_over_tiles(const tn_plan *p, uint32_t slab)
{
    if (16 * p->aux > p->ops) return p->ops < 400 * p->levels && p->m < 64ull * p->n;
    const uint64_t limit = slab < kDefaultSlab ? 256 : 72 + p->n / 1024;
    return p->ops < (limit < 256 ? limit : 256) * p->levels && p->m < 32ull * p->n;
}

static bool records_faster(const tn_plan *p, uint64_t chain, const PlanUse &use, uint32_t slab)
{
    if (p->levels < kRecordLevels) return false;
    const uint32_t ncols = use.ncols ? use.ncols : p->n, rw = p->auto_form ? resident_form(p, ncols) : 0u;
    if (rw) {
        const double L = (double)p->levels, ops = (double)p->ops, waves = (double)resident_waves(p, ncols, rw);
        const double level = rw == 1 ? (p->aux ? 170.0 : 100.0) : (p->aux ? 200.0 : 120.0);
        const double source = (use.max ? 42.0 : 27.0) * (rw == 1 ? 1.0 : 1.33);
        const double per_event = (double)p->n / (double)p->m;
        const double walked = 11.0 * per_event < 1.0 ? 11.0 * per_event : 1.0, listed = 24.0 * per_event < 1.0 ? 24.0 * per_event : 1.0;
        const double resident = waves * (walked * (level * L + 0.5 * ops) + listed * source * (double)chain);
        return resident > 1.25 * (270.0 * L + (3.5 + 0.27 * slab) * ops + (use.max ? 39.0 : 5.0) * (double)chain);
    }
    return records_over_tiles(p, slab);
}

// Resident plans that may be launched with others keep a record schedule beside their
// own, for launches of so many networks that column slabs are due: from this many
// levels (times the waves of CTAs that walk them) on, where it costs 5 to 7 % of applying
// the plan once (n = 20,000, m = 300,000, bursty: 0.2 of 4.2 ms) and six such networks in
// one launch take 4.9 ms instead of 10.1 as tiles.
constexpr uint64_t kBatchLevels = 8192;

// wait_end: return only once the plan's device buffers are written (else they
// may be written by work enqueued on `stream`, which later users must follow).
// as_records: a plan of open options whose windows are to be records.
static tn_status plan_create_impl(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                                  const int64_t *t_after, const tn_plan_options *opt, void *stream,
                                  tn_plan **plan_out, bool wait_end, const PlanUse &use, bool as_records = false)
{
    if (!plan_out) return TN_EINVAL;
    *plan_out = nullptr;
    if (!u || !v || !t || m == 0 || n == 0 || n >= (1u << 30) || m >= (1ull << 30)) return TN_EINVAL;
    uint32_t sw = kDefaultSlab, window = 0, rows = 0, wave = 0, resident = 0;
    if (opt) {
        for (int i = 0; i < 2; ++i)
            if (opt->reserved[i]) return TN_EINVAL;
        if (opt->directed > 1) return TN_EINVAL;
        if (opt->slab_words) sw = opt->slab_words;
        if (opt->window_events) window = opt->window_events;
        rows = opt->smem_rows;
        wave = opt->wave_ctas;
        resident = opt->resident_words;
    }
    if (sw < 2 || sw > kMaxSlabWords || (sw & 1u)) return TN_EINVAL;  // even: whole 16-byte chunks
    // records of a column subset or of sketches: as many CTAs as one wave holds
    uint32_t record_slab = sw;
    if (use.ncols && use.ncols != n && !wave && (!opt || !opt->slab_words))
        while (record_slab > 2 && (use.ncols + 63ull) / 64 <= (uint64_t)multiprocessors() * (record_slab / 2)) record_slab /= 2;
    if (as_records) sw = record_slab;
    // everything but the window left open: no records, and the form is chosen when
    // the plan is applied.  Networks of the same size whose slab width is given keep
    // record windows unless the batch is long enough for rows to settle: their levels
    // are short and deep (bursty n = 20,011, 500,009 events, 16 words: 6.6 ms, 11.4 ms
    // in tiles).
    const bool auto_form = !as_records && (!opt || (!opt->slab_words && !rows && !wave && !resident)) && n <= resident_max_rows(1);
    const bool auto_window = window == 0 && !resident;
    if (!window) window = rows || as_records || (n <= resident_max_rows(1) && !auto_form && m < 64ull * n) ? kRecordWindow : default_window(m);
    const bool records = !auto_form && !(auto_window && window != kRecordWindow);
    if (window < 32) window = 32;
    if (resident) {
        // the resident-slab form keeps every row in shared memory: no row
        // buffer, and every window becomes level-ordered packs of node-id ops
        if ((resident != 1 && resident != 2) || opt->slab_words || opt->smem_rows || wave)
            return TN_EINVAL;
        if (n > resident_max_rows(resident)) return TN_EINVAL;
        rows = 1;
    }
    const bool rows_given = rows != 0;
    if (rows == 0) rows = (sw <= 16 ? kRowBufferBytes : kRowBufferWide) / (sw * 8);
    if (rows > kLocalSlotLimit) rows = kLocalSlotLimit;
    if ((uint64_t)rows * sw * 8 > kRowBufferWide) return TN_EINVAL;  // row buffer must fit the kernel's shared memory
    cudaStream_t st = (cudaStream_t)stream;
    tn_internal_keep_pool();

    PlanArgs a;
    memset(&a, 0, sizeof(a));
    a.u = u;
    a.v = v;
    a.t = t;
    a.m = m;
    a.n = n;
    a.t_after = t_after;
    a.window = window;
    a.directed = opt ? opt->directed : 0u;
    a.nw = (uint32_t)((m + window - 1) / window);
    a.smem_max = smem_max_events();
    const uint64_t first_max = window + window_slack(window) < m ? window + window_slack(window) : m;
    a.first_max = first_max < a.smem_max ? (uint32_t)first_max : a.smem_max;
    a.dcap = rows;
    a.chain = auto_form;
    a.unit8 = window <= kRecordEvents && rows > 1 && records ? 5 : 4;

    tn_plan *p = (tn_plan *)calloc(1, sizeof(tn_plan));
    if (!p) return TN_ENOMEM;
    cudaGetDevice(&p->device);
    p->m = m;
    p->n = n;
    p->windows = a.nw;
    p->slab_words = sw;
    p->wave_ctas = wave;
    p->dcap = rows;
    p->buffer_bytes = rows_given ? rows * sw * 8 : kRowBufferWide;
    p->resident = resident;
    p->auto_form = auto_form;
    p->auto_slab = !resident && !wave && (!opt || !opt->slab_words);

    tn_status rc = TN_OK;
    PlanCounters host;
    memset(&host, 0, sizeof(host));
    const auto part = [](uint64_t bytes) { return (bytes + 255) & ~255ull; };
    bool must_wait = false;
    const bool compact = m >= kCompactEvents || !wait_end;
    const uint64_t blocks = (m + 1023) / 1024;
    cudaError_t err = cudaSuccess;

#define TN_STEP(expr)                  \
    do {                               \
        err = (expr);                  \
        if (err != cudaSuccess) goto fail; \
    } while (0)

    {
        // head, window bounds, second-pass offsets and list, source-list counts,
        // windows, packs and lists: one buffer
        const uint64_t at_bounds = part(sizeof(PlanHead)), at_win = at_bounds + part(8 * (3ull * a.nw + 2));
        const uint64_t at_blob = at_win + part(sizeof(WinDesc) * (uint64_t)a.nw);
        const uint64_t blob_bytes = part(8 * (blob_base(m, a.nw, a.unit8) + 64)), aux_bytes = 12 * m;
        uint8_t *mem = nullptr;
        TN_STEP(alloc_async(&mem, at_blob + blob_bytes + aux_bytes, st));
        p->d_mem = mem;
        p->d_head = reinterpret_cast<PlanHead *>(mem);
        a.wstart = reinterpret_cast<uint64_t *>(mem + at_bounds);
        p->d_win = reinterpret_cast<WinDesc *>(mem + at_win);
        p->d_blob = reinterpret_cast<uint2 *>(mem + at_blob);
        p->d_aux = reinterpret_cast<uint32_t *>(mem + at_blob + blob_bytes);
    }
    p->d_status = &p->d_head->status;
    p->d_tbounds = p->d_head->tbounds;
    a.cnt = &p->d_head->cnt;
    a.tbounds = p->d_head->tbounds;
    TN_STEP(cudaMemsetAsync(p->d_head, 0, sizeof(PlanHead), st));
    a.late_off = a.wstart + a.nw + 1;
    a.late_list = reinterpret_cast<uint32_t *>(a.late_off + a.nw);
    a.naux_w = a.late_list + a.nw;
    a.desc = p->d_win;
    a.blob = p->d_blob;
    a.aux = p->d_aux;
    TN_STEP(tn_internal_allow_max_dyn_smem((const void *)schedule_first_kernel));
    // Counters by mailbox where a call's latency counts (20,000 events: 146 us with
    // sizes, 133 us with the mailbox; 32 serving jobs on 16 threads: 15.0 and 11.8 ms);
    // batches that are compacted wait for their copies anyway (ER, 10^7 events: 16 us
    // more for the 5,000 CTAs' count).
    if (m < kCompactEvents) a.mail = mail_open(st, &a.mail_seq);
    tn_internal_count_launches(2);
    inspect_kernel<<<(unsigned)(blocks < 1216 ? blocks : 1216), 256, 0, st>>>(a);
    schedule_first_kernel<<<a.nw, a.first_max > 1024 ? kPlanThreads : kPlanThreadsSmall, arena_bytes<uint16_t>(a.first_max), st>>>(a);
    TN_STEP(cudaGetLastError());
    if (a.mail) {
        TN_STEP(mail_wait(a.mail, a.mail_seq, st));
        memcpy(&host, a.mail->word, sizeof(host));
    } else {
        TN_STEP(cudaMemcpyAsync(&host, a.cnt, sizeof(host), cudaMemcpyDeviceToHost, st));
        TN_STEP(tn_internal_stream_wait(st));
    }
    if (host.error & 1ull) {
        rc = TN_ERANGE;
        goto done;
    }
    if (host.error & 2ull) {
        rc = TN_EORDER;
        goto done;
    }
    if (host.late) {
        const uint32_t late = (uint32_t)host.late;
        TN_STEP(alloc_async(&a.late_arena, host.arena, st));
        TN_STEP(tn_internal_allow_max_dyn_smem((const void *)schedule_late_kernel));
        tn_internal_count_launches(1);
        schedule_late_kernel<<<late, kPlanThreads, arena_bytes<uint16_t>(a.smem_max), st>>>(a);
        TN_STEP(cudaGetLastError());
        TN_STEP(cudaMemcpyAsync(&host, a.cnt, sizeof(host), cudaMemcpyDeviceToHost, st));
        TN_STEP(tn_internal_stream_wait(st));
    }
    // Records among many more tiles: 1 of 1,001 windows (2,000 events, the last one short)
    // takes 25.3 ms to apply, all as tiles 19.9 ms (activity-driven, n = 10^5, m = 2 10^6,
    // 16 words).  With a tenth of the windows as records, every update executed, some
    // streams are faster than as tiles (bursty n = 1.2 10^5, m = 3 10^6: 42.7 ms, 51.3).
    if (host.local && kTileShare * host.local <= a.nw && !wave && tracked_slab(sw, (uint64_t)rows * sw * 8)) {
        TN_STEP(tn_internal_allow_max_dyn_smem((const void *)schedule_tiles_kernel));
        tn_internal_count_launches(1);
        schedule_tiles_kernel<<<a.nw, kPlanThreads, arena_bytes<uint16_t>(kRecordEvents), st>>>(a);
        TN_STEP(cudaGetLastError());
        TN_STEP(cudaMemcpyAsync(&host, a.cnt, sizeof(host), cudaMemcpyDeviceToHost, st));
        TN_STEP(tn_internal_stream_wait(st));
    }
    p->t_first = host.t_first;
    p->t_last = host.t_last;
    p->items = host.items;
    p->blob8 = host.blob8;
    p->aux = host.naux;
    p->temps = host.temps;
    p->levels = host.levels;
    p->ops = host.ops;
    p->local_windows = host.local;
    p->big_windows = host.big;
    if (auto_window && window != kRecordWindow && sw <= 32 && records_faster(p, host.chain, use, record_slab)) {
        tn_plan *q = nullptr;
        rc = plan_create_impl(u, v, t, m, n, t_after, opt, stream, &q, wait_end, use, true);
        // in wide slabs the row buffer may hold too few rows for most windows (256 hubs,
        // n = 6 10^4, 32 words: none, 25.0 ms in windows of 640, 20.6 ms as they were)
        if (rc == TN_OK && (sw <= 16 || 2 * q->local_windows >= q->windows)) {
            free_plan_buffers(p, st);
            if (a.late_arena) cudaFreeAsync(a.late_arena, st);
            free(p);
            *plan_out = q;
            return TN_OK;
        }
        if (q) {
            free_plan_buffers(q, st);
            free(q);
        } else if (rc != TN_OK) {
            cudaGetLastError();  // (no memory for a second schedule: the first one stands)
            rc = TN_OK;
        }
    }
    if (resident && !resident_fits(n, p->temps, resident)) {  // saved rows of the tie groups do not fit
        rc = TN_EINVAL;
        goto done;
    }
    if ((resident || p->auto_slab || sw <= 16) && !wave && !p->local_windows && m >= kLabelEvents && m >= kLabelFactor * n) {
        TN_STEP(alloc_async(&p->d_label, n, st));
        const unsigned nb = (n + 255) / 256;
        tn_internal_count_launches(3);
        label_init_kernel<<<nb, 256, 0, st>>>(p->d_label, n);
        label_union_kernel<<<(unsigned)(blocks < 1216 ? blocks : 1216), 256, 0, st>>>(u, v, m, p->d_label);
        label_flatten_kernel<<<nb, 256, 0, st>>>(p->d_label, n);
        TN_STEP(cudaGetLastError());
        must_wait = true;
    }
    if (compact) {
        must_wait = true;
        const uint64_t at_win = part(sizeof(PlanHead)), at_blob = at_win + part(sizeof(WinDesc) * (uint64_t)a.nw);
        const uint64_t at_lists = at_blob + 8 * (p->blob8 + 2);
        uint8_t *exact = nullptr;
        TN_STEP(alloc_async(&exact, at_lists + 4 * host.list_words, st));
        PlanHead *head = reinterpret_cast<PlanHead *>(exact);
        WinDesc *win = reinterpret_cast<WinDesc *>(exact + at_win);
        uint2 *blob = reinterpret_cast<uint2 *>(exact + at_blob);
        uint32_t *aux = reinterpret_cast<uint32_t *>(exact + at_lists);
        tn_internal_count_launches(1);
        compact_kernel<<<a.nw, 256, 0, st>>>(a, head, win, blob, aux);
        cudaFreeAsync(p->d_mem, st);
        p->d_mem = exact;
        p->d_head = head;
        p->d_win = win;
        p->d_blob = blob;
        p->d_aux = aux;
        p->d_status = &head->status;
        p->d_tbounds = head->tbounds;
        TN_STEP(cudaGetLastError());
    }
    if (p->auto_form && !use.ncols && records_over_tiles(p, kDefaultSlab)) {
        const uint32_t alone = resident_form(p, n);
        if (alone && p->levels * resident_waves(p, n, alone) >= kBatchLevels) {
            // (without memory for it, the plan does without)
            if (plan_create_impl(u, v, t, m, n, nullptr, opt, stream, &p->batch_plan, false, PlanUse{n, false}, true) == TN_OK)
                p->batch_plan->d_status = p->d_status;
            else
                cudaGetLastError();
            must_wait = true;
        }
    }
    // the plan is complete, and its events are read, when this call returns
    if (must_wait && wait_end) TN_STEP(tn_internal_stream_wait(st));
    goto done;

fail:
    tn_internal_set_cuda_error(err);
    rc = err == cudaErrorMemoryAllocation ? TN_ENOMEM : TN_ECUDA;
done:
    if (a.late_arena) cudaFreeAsync(a.late_arena, st);
    if (rc != TN_OK) {
        free_plan_buffers(p, st);
        free(p);
        return rc;
    }
    *plan_out = p;
    return TN_OK;
#undef TN_STEP
}

extern "C" tn_status tn_plan_create(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m,
                                    uint32_t n, const int64_t *t_after, const tn_plan_options *opt,
                                    void *stream, tn_plan **plan_out)
{
    return plan_create_impl(u, v, t, m, n, t_after, opt, stream, plan_out, true, PlanUse{0, false});
}

tn_status tn::plan_create_for(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                              const int64_t *t_after, const tn_plan_options *opt, const PlanUse &use, void *stream,
                              tn_plan **plan_out)
{
    return plan_create_impl(u, v, t, m, n, t_after, opt, stream, plan_out, true, use);
}

tn_status tn::plan_create_ordered(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                                  const tn_plan_options *opt, cudaStream_t stream, tn_plan **plan_out)
{
    return plan_create_impl(u, v, t, m, n, nullptr, opt, stream, plan_out, false, PlanUse{n, false});
}

extern "C" tn_status tn_plan_destroy(tn_plan *p, void *stream)
{
    if (!p) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    free_plan_buffers(p, st);
    free(p);
    return TN_OK;
}

tn_status tn::plan_use_status(tn_plan *p, int32_t *status, cudaStream_t st)
{
    if (!p || !status) return TN_EINVAL;
    (void)st;
    p->d_status = status;
    if (p->batch_plan) p->batch_plan->d_status = status;
    return TN_OK;
}

extern "C" tn_status tn_plan_get_stats(const tn_plan *p, tn_plan_stats *s)
{
    if (!p || !s) return TN_EINVAL;
    memset(s, 0, sizeof(*s));
    s->events = p->m;
    s->windows = p->windows;
    s->levels = p->levels;
    s->ops = p->ops;
    s->aux = p->aux;
    s->temps = p->temps;
    s->big_windows = p->big_windows;
    s->local_windows = p->local_windows;
    s->items = p->items;
    s->t_first = p->t_first;
    s->t_last = p->t_last;
    return TN_OK;
}

extern "C" tn_status tn_plan_status(tn_plan *p, void *stream)
{
    if (!p) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int32_t h = 0;
    TN_CUDA_TRY(cudaMemcpyAsync(&h, p->d_status, sizeof(h), cudaMemcpyDeviceToHost, st));
    TN_CUDA_TRY(cudaMemsetAsync(p->d_status, 0, sizeof(int32_t), st));
    TN_CUDA_TRY(tn_internal_stream_wait(st));
    return (tn_status)h;
}
