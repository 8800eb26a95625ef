// Column-slab streaming of a scheduled event batch into component matrices.
//
// Algorithm 1 (Section 3.1) updates whole rows, but bit column j of the matrix
// (the out-component of source j) evolves independently of every other column.
// Each CTA therefore owns a slab of `sw` consecutive 64-bit words of every row
// (64*sw source columns, 2 <= sw <= 128) and streams the whole level-ordered
// schedule over it:
//   * a producer warp copies the schedule, pack by pack, into a ring of shared
//     memory stages with bulk asynchronous copies (cp.async.bulk, completion on
//     an mbarrier), so the ops are read from L2/HBM once per CTA and without
//     occupying the consumer threads;
//   * consumer warps (12 when the CTA holds its SM alone, 4 when two CTAs share
//     an SM) apply a pack: a window whose rows fit the shared-memory row
//     buffer (a record) is gathered, updated level by level in shared
//     memory and written through at each row's last write; a tile of ops on
//     rows in HBM (a level of a tile pack) runs through a private per-thread ring of
//     cp.async copies, with hub PULLs as L2 OR-reductions.  A named
//     barrier orders one level's stores before the next level's loads.
// All waits are bounded (TN_ETIMEOUT).  The barrier before a pack is a reduction
// (bar.red.or) of every consumer's stop condition, so all consumers leave the
// loop at the same barrier and none can be left waiting on it.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "tn_internal.cuh"

namespace tn {

// Consumer warps per CTA, chosen at launch: 12 when a CTA's row buffer leaves
// no room for a second CTA on the SM, 4 when two CTAs share an SM (both then
// fit in the register file).  The producer is one more warp.
constexpr int kWarpsAlone = 12;
constexpr int kWarpsShared = 4;
constexpr int kMaxThreads = 32 * kWarpsAlone + 32;
constexpr int kStages = 2;
constexpr uint32_t kStageShift = 1;
constexpr size_t kSlabHead = (size_t)kStages * kStageBytes + 64;  // stages, barriers
constexpr int kMaxPlans = 24;  // networks per launch
constexpr int kMaxJobs = 2 * kMaxPlans;  // a network spread over a wave has CTAs of two widths

struct Job {
    const uint2 *blob;
    const WinDesc *win;
    const uint32_t *aux;
    uint64_t *S;
    uint64_t ld;    // row stride in words
    uint64_t *tmp;  // saved-row slots of global windows, ld words each
    int32_t *status;
    uint64_t w_begin;  // first row word of the job's first CTA
    uint32_t sw;    // slab words per CTA (even, 2..kMaxSlabWords)
    uint32_t cpr;   // 16-byte chunks of a row segment = sw / 2
    uint32_t nwin;  // windows of the schedule
    uint32_t cta_begin;
    uint32_t dcap;  // row slots of the shared-memory row buffer
    uint32_t track;       // TrackMode of a column slab
    uint32_t *ids;        // content ids of the rows, then of the saved rows
    uint32_t pitch;       // ids per row, one per CTA
    uint32_t mark_words;  // 32-bit words of the marks (0: every op is executed)
    uint32_t mark_shift;  // 2^mark_shift rows per mark
    uint32_t mark_init;   // S starts as the identity (1) or the source columns (2); 0: unknown content
    const uint32_t *src;
    uint32_t ncols;
    // resident-slab form (rw > 0): each CTA keeps rw words of every row in shared memory
    uint32_t rw;     // words of every row per CTA (1 or 2), 0 = column-slab form
    uint32_t res_threads;  // consumer threads of a resident CTA
    const uint32_t *label; // component of every node, or NULL
    uint32_t identity;     // resident: S starts as the identity (and is not read)
    uint32_t rows;   // rows of the matrix (node count of the plan)
    uint32_t ntemp;  // saved-row slots of the plan's tie groups
};

struct JobList {
    Job job[kMaxJobs];
    uint32_t count;
    uint32_t smem_bytes;  // dynamic shared memory of the launch
};

__device__ inline uint32_t find_job(const JobList &jl, uint32_t cta)
{
    uint32_t j = 0;
    while (j + 1 < jl.count && jl.job[j + 1].cta_begin <= cta) ++j;
    return j;
}

// The ring of schedule packs: `nst` (a power of two) stages of kStageBytes in
// shared memory and their full / empty barriers.  Behind the last pack comes a
// stage whose header says kPackEnd.
struct PackRing {
    uint8_t *stage;
    uint64_t *full, *empty;
    uint32_t mask, shift;  // of nst
    __device__ uint8_t *at(uint32_t q) const { return stage + (size_t)(q & mask) * kStageBytes; }
    __device__ bool wait_full(uint32_t q) const { return mbar_wait_bounded(&full[q & mask], (q >> shift) & 1u); }
    // false on a timeout, or once the consumers have set `stop`
    __device__ bool wait_empty(uint32_t q, volatile uint32_t *stop) const
    {
        if (q <= mask) return true;
        for (uint32_t i = 0; i < kWaitPolls && *stop == 0; ++i)
            if (mbar_try_wait(&empty[q & mask], ((q >> shift) - 1u) & 1u)) return true;
        return false;
    }
};

// Producer warp: one bulk copy per pack.  Lane k holds the descriptor of window
// w0 + k; the next 32 descriptors are loaded one batch ahead.
__device__ void produce_packs(const Job &J, const PackRing &ring, volatile uint32_t *abort_flag)
{
    const uint32_t lane = threadIdx.x & 31u, nwin = J.nwin;
    const uint4 *win = reinterpret_cast<const uint4 *>(J.win);
    const uint4 none = make_uint4(0u, 0u, 0u, 0u);
    uint32_t q = 0;
    bool ok = true;
    uint4 na = lane < nwin ? __ldg(win + 2 * lane) : none, nb = lane < nwin ? __ldg(win + 2 * lane + 1) : none;
    for (uint32_t w0 = 0; w0 < nwin && ok; w0 += 32) {
        const uint4 da = na, db = nb;
        const uint32_t ahead = w0 + 32 + lane;
        if (ahead < nwin) {
            na = __ldg(win + 2 * (uint64_t)ahead);
            nb = __ldg(win + 2 * (uint64_t)ahead + 1);
        }
        const uint32_t count = nwin - w0 < 32 ? nwin - w0 : 32u;
        for (uint32_t k = 0; k < count && ok; ++k) {
            const uint32_t lo = __shfl_sync(0xffffffffu, da.x, k), hi = __shfl_sync(0xffffffffu, da.y, k);
            const uint32_t np = __shfl_sync(0xffffffffu, da.z, k), tab = __shfl_sync(0xffffffffu, da.w, k);
            const uint32_t p0 = __shfl_sync(0xffffffffu, db.x, k), p1 = __shfl_sync(0xffffffffu, db.y, k);
            const uint32_t p2 = __shfl_sync(0xffffffffu, db.z, k), p3 = __shfl_sync(0xffffffffu, db.w, k);
            const uint2 *src = J.blob + (((uint64_t)hi << 32) | lo);
            const uint32_t *table = reinterpret_cast<const uint32_t *>(src + tab);
            if (lane == 0) {
                for (uint32_t p = 0; p < np; ++p) {
                    const uint32_t n8 = np > kDescPacks ? __ldg(table + p) : p == 0 ? p0 : p == 1 ? p1 : p == 2 ? p2 : p3;
                    if (!ring.wait_empty(q, abort_flag)) {
                        ok = false;
                        break;
                    }
                    uint64_t *bar = &ring.full[q & ring.mask];
                    mbar_arrive_expect_tx(bar, n8 * 8u);
                    bulk_g2s(ring.at(q), src, n8 * 8u, bar);
                    src += n8;
                    ++q;
                }
            }
            ok = __shfl_sync(0xffffffffu, (int)ok, 0);
        }
    }
    if (lane == 0) {
        if (ok && ring.wait_empty(q, abort_flag)) {
            reinterpret_cast<uint32_t *>(ring.at(q))[1] = kPackEnd << 16;
            mbar_arrive(&ring.full[q & ring.mask]);
            ++q;
        } else if (*abort_flag == 0) {  // (consumers that stop early need no more packs)
            record_status(J.status, TN_ETIMEOUT);
            *abort_flag = 1;
        }
        // no bulk copy may still be writing this CTA's shared memory at exit
        for (uint32_t c = q > ring.mask + 1 ? q - ring.mask - 1 : 0; c < q; ++c) ring.wait_full(c);
    }
}

// A consumer thread's place in the slab: `cpr` consecutive threads share one row
// segment (one 16-byte chunk each) and `stride` row segments are handled at once.
struct Lane {
    uint32_t chunk, lane0, stride, cpr;
    uint64_t col;  // first word of this thread's chunk
    uint8_t *base; // this thread's chunk of row 0
    uint32_t pitch;  // bytes per row (below 2^28: one multiply-add per row address)
    const uint32_t *pack;  // the pack being applied (source lists)
    bool active;   // chunk inside the matrix and thread inside the row groups
};

// consumer threads of this launch (all warps but the producer)
__device__ inline uint32_t consumers() { return blockDim.x - 32u; }

__device__ inline Lane make_lane(const Job &J, uint32_t ct, uint64_t w0)
{
    Lane L;
    L.cpr = J.cpr;
    L.chunk = ct % L.cpr;
    L.lane0 = ct / L.cpr;
    L.stride = consumers() / L.cpr;
    L.col = w0 + 2ull * L.chunk;
    L.base = reinterpret_cast<uint8_t *>(J.S + L.col);
    L.pitch = (uint32_t)(8 * J.ld);
    L.active = L.lane0 < L.stride && L.col < J.ld;
    return L;
}

__device__ inline uint64_t *row_of(const Lane &L, uint32_t row)
{
    return reinterpret_cast<uint64_t *>(L.base + (uint64_t)row * L.pitch);
}

// Source list of a PULL: its count, then its references.
__device__ inline const uint32_t *source_list(const uint32_t *aux, const uint32_t *pack, uint32_t b)
{
    return b < kOutsideList ? pack + b : aux + (b - kOutsideList);
}

__device__ inline uint64_t *row_ptr(const Job &J, uint32_t ref, uint64_t col)
{
    if (ref & kTempRef) return J.tmp + (uint64_t)(ref & ~kTempRef) * J.ld + col;
    return J.S + (uint64_t)ref * J.ld + col;
}

__device__ inline void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"r"(consumers()) : "memory"); }
__device__ inline void consumers_sync(uint32_t count) { asm volatile("bar.sync 1, %0;" ::"r"(count) : "memory"); }

// Barrier of the consumer warps (named barrier 1) that also ORs a predicate
// across them, so that every consumer takes the same decision to stop.
__device__ inline bool consumers_sync_or(bool p, uint32_t count)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred ip, op;\n\t"
        "setp.ne.u32 ip, %1, 0;\n\t"
        "bar.red.or.pred op, 1, %2, ip;\n\t"
        "selp.u32 %0, 1, 0, op;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(count)
        : "memory");
    return r != 0;
}

__device__ inline bool consumers_sync_or(bool p) { return consumers_sync_or(p, consumers()); }

__device__ inline void cp_async16(void *smem_dst, const void *gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(smem_dst)), "l"(gmem_src) : "memory");
}

__device__ inline void cp_async16(uint32_t smem_dst, const void *gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}

__device__ inline void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ inline u64x2 lds16(const u64x2 *p)
{
    u64x2 r;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(r.x), "=l"(r.y) : "r"(smem_addr(p)) : "memory");
    return r;
}

__device__ inline u64x2 lds16(uint32_t a)
{
    u64x2 r;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(r.x), "=l"(r.y) : "r"(a) : "memory");
    return r;
}

__device__ inline void sts16(u64x2 *p, u64x2 v)
{
    asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(smem_addr(p)), "l"(v.x), "l"(v.y) : "memory");
}

// ---------------------------------------------------------------------------
// global tile: ops name rows by node id and read/write the matrix directly
// ---------------------------------------------------------------------------
// PULL: S[x] |= OR of the listed source rows (aux[b] = count, then refs)
template <bool kMax>
__device__ inline void apply_pull(const Job &J, uint32_t x, uint32_t b, const Lane &L)
{
    const uint64_t col = L.col;
    uint64_t *pd = J.S + (uint64_t)x * J.ld + col;
    u64x2 acc = ld_row16(pd);
    const uint32_t *list = source_list(J.aux, L.pack, b);
    const uint32_t c = list[0];
    for (uint32_t i = 0; i < c; i += 8) {
        uint32_t ref[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) ref[k] = (i + k < c) ? list[1 + i + k] : kNoRef;
        u64x2 r[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            r[k] = (ref[k] != kNoRef) ? ld_row16(row_ptr(J, ref[k], col)) : u64x2{0, 0};
#pragma unroll
        for (int k = 0; k < 8; ++k) acc = combine16<kMax>(acc, r[k]);
    }
    st_row16(pd, acc);
}

// Direct form, for row buffers too small to stage a chunk: four ops in flight per thread.
template <bool kMax>
__device__ inline void apply_tile_direct(const Job &J, const uint2 *ops, uint32_t count, const Lane &L)
{
    if (!L.active) return;  // partial last slab, or a thread outside the row groups
    const uint64_t col = L.col;
    const uint32_t stride = L.stride;
    for (uint32_t o = L.lane0; o < count; o += 4 * stride) {
        uint2 op[4];
        bool live[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t idx = o + k * stride;
            live[k] = idx < count;
            op[k] = live[k] ? ops[idx] : make_uint2(0u, 0u);
        }
        // loads of all four ops first (they are independent inside a level)
        u64x2 ra[4], rb[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t kind = op[k].x >> kKindShift;
            if (!live[k] || kind == kPull) continue;
            if (kind != kCopy) ra[k] = ld_row16(J.S + (uint64_t)(op[k].x & kIdMask) * J.ld + col);
            rb[k] = ld_row16(J.S + (uint64_t)op[k].y * J.ld + col);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t kind = op[k].x >> kKindShift;
            if (!live[k] || kind == kPull) continue;
            const uint64_t ia = (uint64_t)(op[k].x & kIdMask) * J.ld + col;
            if (kind == kCopy) {
                st_row16(J.tmp + ia, rb[k]);
            } else {
                const u64x2 r = combine16<kMax>(ra[k], rb[k]);
                st_row16(J.S + ia, r);
                if (kind == kEvent) st_row16(J.S + (uint64_t)op[k].y * J.ld + col, r);
            }
        }
    }
    // multi-source updates of tie groups (hub rows) in a second pass
    for (uint32_t o = L.lane0; o < count; o += stride) {
        const uint2 op = ops[o];
        if ((op.x >> kKindShift) == kPull) apply_pull<kMax>(J, op.x & kIdMask, op.y, L);
    }
}

// Ops of one level are independent.  Each consumer thread takes the ops
// lane0, lane0 + stride, ... of the tile and runs them through a private ring
// of kRing op slots in shared memory (two row chunks per op): the copies of
// the op kRing - 1 places ahead are issued (cp.async, one commit group per op)
// before the current op's rows are read back, combined and stored from
// registers.  A thread reads only the slots it filled itself, so no barrier is
// needed inside a tile; the item loop's barrier orders one level's stores
// before the next level's loads.
constexpr int kRing = 8;

__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ inline void cp_async_wait_group()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ inline void red_or16(uint64_t *p, u64x2 v)
{
    asm volatile("red.global.or.b64 [%0], %1;" ::"l"(p), "l"(v.x) : "memory");
    asm volatile("red.global.or.b64 [%0], %1;" ::"l"(p + 1), "l"(v.y) : "memory");
}

// The thread's PULLs, S[x] |= OR of the listed source rows, as a flat sequence
// of (x, source) pairs through the same private ring: a source chunk is copied
// in kRing - 1 pairs ahead, then ORed into row x by a reduction at L2
// (red.global.or), so x is never loaded and the pairs of one PULL need no
// order among themselves (OR is associative and commutative).  Rows written
// by a PULL are read by no other op of the same level.
struct PullCursor {
    uint32_t o, q, c;  // op index, next source (0-based), source count
};

__device__ inline void pull_cursor_seek(PullCursor &cur, const Job &J, const uint2 *ops, uint32_t count,
                                        const Lane &L)
{
    const uint32_t stride = L.stride;
    while (cur.o < count && cur.q >= cur.c) {
        cur.o += stride;
        while (cur.o < count && (ops[cur.o].x >> kKindShift) != kPull) cur.o += stride;
        cur.q = 0;
        cur.c = cur.o < count ? source_list(J.aux, L.pack, ops[cur.o].y)[0] : 0u;
    }
}

__device__ inline void apply_pulls_ring(const Job &J, const uint2 *ops, uint32_t count, u64x2 *mine, const Lane &L)
{
    const uint32_t cpr = L.cpr, stride = L.stride;
    const uint64_t col = L.col;
    PullCursor in{L.lane0, 0u, 0u};
    while (in.o < count && (ops[in.o].x >> kKindShift) != kPull) in.o += stride;
    if (in.o >= count) return;
    in.c = source_list(J.aux, L.pack, ops[in.o].y)[0];
    pull_cursor_seek(in, J, ops, count, L);
    PullCursor out = in;
    uint32_t issued = 0, done = 0;
    auto issue = [&]() {
        if (in.o >= count) return;
        const uint32_t ref = source_list(J.aux, L.pack, ops[in.o].y)[1 + in.q];
        const uint32_t q = L.lane0 + (issued % kRing) * stride;
        cp_async16(mine + (2 * q) * cpr, row_ptr(J, ref, col));
        ++issued;
        ++in.q;
        pull_cursor_seek(in, J, ops, count, L);
    };
#pragma unroll 1
    for (uint32_t k = 0; k < kRing - 1; ++k) {
        issue();
        cp_async_commit();
    }
#pragma unroll 1
    while (done < issued) {
        issue();
        cp_async_commit();
        cp_async_wait_group<kRing - 1>();  // pair `done` has landed
        const uint32_t q = L.lane0 + (done % kRing) * stride;
        red_or16(J.S + (uint64_t)(ops[out.o].x & kIdMask) * J.ld + col, lds16(mine + (2 * q) * cpr));
        ++done;
        ++out.q;
        pull_cursor_seek(out, J, ops, count, L);
    }
    cp_async_wait_group<0>();
}

template <bool kMax>
__device__ inline void apply_tile(const Job &J, const uint2 *ops, uint32_t count, u64x2 *buf, uint32_t dcap,
                                  const Lane &L)
{
    const uint32_t cpr = L.cpr, stride = L.stride;
    const uint64_t col = L.col;
    if (dcap < 2u * kRing * stride) {
        apply_tile_direct<kMax>(J, ops, count, L);
        return;
    }
    if (!L.active) return;
    u64x2 *mine = buf + L.chunk;
    const uint32_t nk = count > L.lane0 ? (count - L.lane0 + stride - 1) / stride : 0;
    // ring slot r of this thread holds its op's rows in slots 2q, 2q + 1, q = lane0 + r * stride
    auto issue = [&](uint32_t k) {
        const uint2 op = ops[L.lane0 + k * stride];
        const uint32_t kind = op.x >> kKindShift;
        const uint32_t q = L.lane0 + (k % kRing) * stride;
        if (kind != kPull) {
            if (kind != kCopy) cp_async16(mine + (2 * q) * cpr, J.S + (uint64_t)(op.x & kIdMask) * J.ld + col);
            cp_async16(mine + (2 * q + 1) * cpr, J.S + (uint64_t)op.y * J.ld + col);
        }
    };
#pragma unroll 1
    for (uint32_t k = 0; k < kRing - 1; ++k) {
        if (k < nk) issue(k);
        cp_async_commit();
    }
#pragma unroll 1
    for (uint32_t k = 0; k < nk; ++k) {
        if (k + kRing - 1 < nk) issue(k + kRing - 1);
        cp_async_commit();
        cp_async_wait_group<kRing - 1>();  // op k's copies have landed
        const uint2 op = ops[L.lane0 + k * stride];
        const uint32_t kind = op.x >> kKindShift;
        if (kind == kPull) continue;
        const uint32_t q = L.lane0 + (k % kRing) * stride;
        const uint64_t ia = (uint64_t)(op.x & kIdMask) * J.ld + col;
        const u64x2 rb = lds16(mine + (2 * q + 1) * cpr);
        if (kind == kCopy) {
            st_row16(J.tmp + ia, rb);
        } else {
            const u64x2 r = combine16<kMax>(lds16(mine + (2 * q) * cpr), rb);
            st_row16(J.S + ia, r);
            if (kind == kEvent) st_row16(J.S + (uint64_t)op.y * J.ld + col, r);
        }
    }
    cp_async_wait_group<0>();
    // multi-source updates of tie groups (hub rows) in a second pass
    if (kMax) {
        for (uint32_t o = L.lane0; o < count; o += stride) {
            const uint2 op = ops[o];
            if ((op.x >> kKindShift) == kPull) apply_pull<kMax>(J, op.x & kIdMask, op.y, L);
        }
    } else {
        apply_pulls_ring(J, ops, count, mine, L);
    }
}

// ---------------------------------------------------------------------------
// tracked rows: updates that cannot change anything are not made
//
// Early in a stream most row segments of a slab are still zero; later most
// events meet rows that already hold the same content.  A CTA keeps what it
// needs to know about its rows, skips the ops that this shows to change nothing
// without touching the matrix, and stores only chunks that change.  Every
// skipped update is one that would write what is there; nothing is carried over
// between applications.  Two forms:
//
// Marks (slabs of up to 16 words): one reference content C (16 bytes per thread)
// and one bit per row in shared memory, "this row's segment equals C".  An op is
// skipped when all its rows are marked; marked rows are not loaded; a row is
// marked when its result equals C.  C starts as zero (all rows but the sources'
// marked, when the application initialises S).  When most ops are executed all
// the same, the marks are dropped; when at least half of the executed updates
// find both rows equal, the largest such content becomes the new C.  When a bit
// per row does not fit, a bit stands for 2^shift consecutive rows, for C = zero
// only (rows never return to zero).
//
// Ids (wider slabs): a content id per row in global memory; rows with equal ids
// hold equal segments (the reverse need not be known).  An op is skipped when
// its rows' ids are equal.  A row that took over the other's content takes its
// id, rows found equal take the smaller id, new content gets an id no row has had
// (one per op).  Id 0 is the zero segment, which is never loaded.
// ids[row][cta]: the CTAs of a matrix run the same ops at about the same time, so
// the eight ids of a sector are read from DRAM once.
//
// Ids find nearly every update that changes nothing, but each level waits for
// them (an L2 access under load, about 2 us); marks cost two shared-memory reads
// and find what is zero or in the main component's final state.  Executed share
// (simulated, n = 10^5, 50 events per node, 64 words): bursty 0.24 by ids, 0.53
// by marks; activity-driven 0.19 and 0.20.  Measured, stream kernel: bursty n =
// 5 10^5, m = 2.5 10^7, 64 words 543 ms by ids, 1,037 by marks, 765 with every op
// executed (1,085 with every chunk stored as well); activity-driven n = 10^5, m =
// 10^7, 16 words 38.5, 25.0, 90.2 and 119 ms.
// ---------------------------------------------------------------------------
constexpr uint32_t kMarkWords = 16;  // widest slab whose rows are marked
constexpr uint32_t kMarkShift = 2;   // at most 4 rows per bit

extern __shared__ __align__(128) uint8_t dyn_smem[];  // dynamic shared memory of the streaming kernel

// Shared memory behind the row buffer (byte offset `at`): listed ops of all
// warps (12 x 192 or 4 x 576): uint4 {op.x, row b, a, b}, a and b = 0 for rows
// whose content is known (C, or zero), else their ids or 1 | their indices |
// statistics [3][4] (marks: per window, ops, executed, sampled updates, of these
// equal rows; ids: executed flags of three packs) | key of the largest candidate: size << 10 | row
// group | (marks) candidates, 16 bytes per consumer | mark bits of the rows, then
// of the saved rows.
constexpr uint32_t kListOps = 2304;
constexpr uint32_t kIdBytes = 18 * kListOps + 64;
constexpr uint32_t kMarkBytes = kIdBytes + 16 * 32 * kWarpsAlone;

enum TrackMode : int { kNoTrack = 0, kMarks = 1, kIds = 2 };

struct Track {
    uint32_t at;
    uint32_t slot;    // this warp's first list entry
    uint32_t rows;    // first saved row
    // ids
    uint32_t *ids;    // this CTA's id of row 0
    uint32_t pitch;   // ids per row
    uint32_t fresh;   // the id that op 0 of the current segment may take
    // marks
    uint32_t shift;   // 2^shift rows per bit
    u64x2 c;          // this thread's chunk of C (ids: zero)
    uint32_t c_size;  // size of C
    bool on;          // marks are valid
    bool want;        // this window looks for a candidate
    bool quiet;       // the last window executed nothing
    uint32_t best_size;               // of this row group's candidate
    bool settled;     // nothing changed in the last window, as far as it was counted
    bool sample;      // this window counts equal rows (every fourth, and those that look for a candidate)
    uint32_t n_ops, n_live;    // of this window, this warp
    uint32_t n_seen, n_equal;  // sampled updates, of equal rows, this thread
    __device__ uint4 *list() const { return reinterpret_cast<uint4 *>(dyn_smem + at) + slot; }
    __device__ uint16_t *index() const { return reinterpret_cast<uint16_t *>(dyn_smem + at + 16 * kListOps) + slot; }
    __device__ uint32_t *stat(uint32_t q) const { return reinterpret_cast<uint32_t *>(dyn_smem + at + 18 * kListOps) + 4 * (q % 3u); }
    __device__ uint32_t *key() const { return reinterpret_cast<uint32_t *>(dyn_smem + at + 18 * kListOps) + 12; }
    __device__ u64x2 *cand(uint32_t i) const { return reinterpret_cast<u64x2 *>(dyn_smem + at + kIdBytes) + i; }
    __device__ uint32_t *bits() const { return reinterpret_cast<uint32_t *>(dyn_smem + at + kMarkBytes); }
    __device__ uint32_t *id_ptr(uint32_t ref) const
    {
        return ids + (uint64_t)((ref & kTempRef) ? rows + (ref & ~kTempRef) : ref) * pitch;
    }
    __device__ uint32_t id(uint32_t ref) const
    {
        uint32_t x;
        asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(x) : "l"(id_ptr(ref)) : "memory");
        return x;
    }
    // saved rows have a bit each, behind the rows' bits
    __device__ uint32_t bit_of(uint32_t ref) const
    {
        return (ref & kTempRef) ? (rows >> shift) + 1u + (ref & ~kTempRef) : ref >> shift;
    }
    __device__ bool marked(uint32_t ref) const
    {
        const uint32_t i = bit_of(ref);
        return (bits()[i >> 5] >> (i & 31u)) & 1u;
    }
    __device__ void mark(uint32_t ref) const
    {
        const uint32_t i = bit_of(ref);
        if (shift == 0 || (ref & kTempRef)) atomicOr(bits() + (i >> 5), 1u << (i & 31u));
    }
    __device__ void unmark(uint32_t ref) const
    {
        const uint32_t i = bit_of(ref);
        atomicAnd(bits() + (i >> 5), ~(1u << (i & 31u)));
    }
};

__device__ inline bool same16(u64x2 a, u64x2 b) { return a.x == b.x && a.y == b.y; }

// Ids: whether an op is to be executed; `e` becomes its list entry.  A PULL whose
// sources that differ from its row all share one id is the ONEWAY update from
// any of them.
__device__ inline bool id_live(const Job &J, const Track &T, uint2 op, const uint32_t *pack, uint4 &e)
{
    const uint32_t kind = op.x >> kKindShift, a = op.x & kIdMask;
    if (kind == kCopy) {
        e = make_uint4(op.x, op.y, 0u, T.id(op.y));
        return true;
    }
    if (kind != kPull) {
        const uint32_t ia = T.id(a), ib = T.id(op.y);
        e = make_uint4(op.x, op.y, ia, ib);
        return ia != ib && !(kind == kOneway && ib == 0);
    }
    const uint32_t ia = T.id(a);
    const uint32_t *list = source_list(J.aux, pack, op.y);
    const uint32_t c = list[0];
    uint32_t found = 0, from = 0, fid = 0;
    for (uint32_t i = 0; i < c && found < 2; i += 8) {  // eight independent loads at a time
        uint32_t ref[8], sid[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) ref[k] = list[1 + (i + k < c ? i + k : i)];
#pragma unroll
        for (int k = 0; k < 8; ++k) sid[k] = T.id(ref[k]);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (sid[k] == ia || sid[k] == 0 || (found && sid[k] == fid)) continue;
            ++found;
            from = ref[k];
            fid = sid[k];
        }
    }
    if (found == 0) return false;
    e = found == 1 ? make_uint4(op_a(kOneway, a), from, ia, fid) : make_uint4(op.x, op.y, ia, 0u);
    return true;
}

// Marks: likewise.  A COPY of a marked row marks the saved row instead.
__device__ inline bool mark_live(const Job &J, const Track &T, uint2 op, const uint32_t *pack, uint4 &e)
{
    const uint32_t kind = op.x >> kKindShift, a = op.x & kIdMask;
    e = make_uint4(op.x, op.y, 1u, 1u);
    if (kind == kCopy) {
        if (T.marked(op.y)) {
            T.mark(kTempRef | a);
            return false;
        }
        if (T.marked(kTempRef | a)) T.unmark(kTempRef | a);
        return true;
    }
    const bool ma = T.marked(a);
    e.z = !ma;
    if (kind != kPull) {
        const bool mb = T.marked(op.y);
        e.w = !mb;
        return !(ma && mb);
    }
    if (!ma) return true;
    const uint32_t *list = source_list(J.aux, pack, op.y);
    const uint32_t c = list[0];
    bool live = false;
    for (uint32_t i = 0; i < c && !live; i += 8) {  // eight independent loads at a time
        uint32_t ref[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) ref[k] = list[1 + (i + k < c ? i + k : i)];
#pragma unroll
        for (int k = 0; k < 8; ++k) live |= !T.marked(ref[k]);
    }
    return live;
}

// Size of a row group's content (cpr lanes, one chunk each): bits, or the sum of
// the registers of a sketch; below 2^22.
template <bool kMax>
__device__ inline uint32_t content_size(u64x2 r, uint32_t cpr, uint32_t group_mask)
{
    uint32_t n;
    if (kMax) {
        n = __vsadu4((uint32_t)r.x, 0u) + __vsadu4((uint32_t)(r.x >> 32), 0u) + __vsadu4((uint32_t)r.y, 0u) +
            __vsadu4((uint32_t)(r.y >> 32), 0u);
    } else {
        n = __popcll(r.x) + __popcll(r.y);
    }
    for (uint32_t d = 1; d < cpr; d <<= 1) n += __shfl_xor_sync(group_mask, n, d);
    return n;
}

// What one executed EVENT, ONEWAY or COPY (entry e, rows' chunks ra, rb) writes:
// the chunks that change, and what the CTA knows about its rows.  `i` is its list
// position.  All lanes of the warp call it (lanes without an op with a PULL entry).
template <bool kMax, int kMode>
__device__ inline void track_update(const Job &J, Track &T, const Lane &L, uint32_t group_mask, uint4 e, u64x2 ra,
                                    u64x2 rb, uint32_t i)
{
    const bool active = L.active;
    const uint32_t kind = e.x >> kKindShift, a = e.x & kIdMask, ref = e.y;
    const bool update = kind == kEvent || kind == kOneway;
    const u64x2 r = combine16<kMax>(ra, rb);
    const bool new_a = active && update && !same16(r, ra), new_b = active && update && !same16(r, rb);
    if (new_a) st_row16(row_of(L, a), r);
    if (new_b && kind == kEvent) st_row16(row_of(L, ref), r);
    if (kind == kCopy && active) st_row16(J.tmp + (uint64_t)a * J.ld + L.col, rb);
    if (kMode == kIds) {
        const bool any_a = (__ballot_sync(0xffffffffu, new_a) & group_mask) != 0;
        const bool any_b = (__ballot_sync(0xffffffffu, new_b) & group_mask) != 0;
        if (L.chunk == 0) {
            const uint32_t ia = e.z, ib = e.w;
            if (update) {
                const uint32_t fresh = T.fresh + T.index()[i];
                const uint32_t id = any_a && any_b ? fresh : any_a ? ib : any_b ? ia : min(ia, ib);
                if (id != ia) *T.id_ptr(a) = id;
                if (kind == kEvent && id != ib) *T.id_ptr(ref) = id;
            } else if (kind == kCopy) {
                *T.id_ptr(kTempRef | a) = ib;
            }
        }
        return;
    }
    if (kMode == kMarks) {
        const uint32_t other = __ballot_sync(0xffffffffu, active && !same16(r, T.c));
        if (update && L.chunk == 0) {
            const bool all = !(other & group_mask);
            if (all != (e.z == 0)) {
                if (all) T.mark(a);
                else T.unmark(a);
            }
            if (kind == kEvent && all != (e.w == 0)) {
                if (all) T.mark(ref);
                else T.unmark(ref);
            }
        }
    }
    if (!T.sample) return;
    const uint32_t differ = __ballot_sync(0xffffffffu, new_a || new_b);
    const bool equal = update && !(differ & group_mask);
    T.n_seen += update;
    T.n_equal += equal;
    if (T.want && equal) {
        const uint32_t size = content_size<kMax>(active ? r : u64x2{0, 0}, L.cpr, group_mask);
        if (size > T.best_size) {
            T.best_size = size;
            *T.cand(L.lane0 * L.cpr + L.chunk) = r;
        }
    }
}

// Entry of this row group's k-th op: this warp's list, or, with kNoTrack, the ops
// first, first + step, ... themselves; a PULL of no row past the end.
template <int kMode>
__device__ inline uint4 track_entry(const Track &T, const uint2 *ops, uint32_t cnt, uint32_t i)
{
    if (i >= cnt) return make_uint4(op_a(kPull, kIdMask), 0u, 0u, 0u);
    if (kMode != kNoTrack) return T.list()[i];
    const uint2 op = ops[i];
    return make_uint4(op.x, op.y, 1u, 1u);
}

template <int kMode>
__device__ inline uint64_t *track_row_b(const Job &J, const Lane &L, uint32_t ref)
{
    if (kMode == kIds) return row_ptr(J, ref, L.col);  // (a PULL run as ONEWAY may read a saved row)
    return row_of(L, ref);
}

// Up to two ops per row group, one after the other, loaded straight into
// registers, a PULL's sources (the first eight) together with its row: one memory
// latency instead of a copy ring's start and drain.  Levels of tie-heavy streams
// are that short (hubs chain every timestamp group to the one before).
template <bool kMax, int kMode>
__device__ void track_short(const Job &J, Track &T, const uint2 *ops, uint32_t cnt, uint32_t first, uint32_t step,
                            uint32_t rounds, const Lane &L, uint32_t group_mask)
{
    const u64x2 zero{0, 0}, known = kMode == kMarks ? T.c : zero;
    const bool active = L.active;
#pragma unroll 1
    for (uint32_t k = 0; k < rounds; ++k) {
        const uint32_t i = first + k * step;
        const uint4 e = track_entry<kMode>(T, ops, cnt, i);
        const uint32_t kind = e.x >> kKindShift, a = e.x & kIdMask;
        const bool pull = kind == kPull && a != kIdMask;
        u64x2 ra = known, rb = known, acc = zero, r[8];
        if (active && kind != kPull) {
            if (e.z != 0 && kind != kCopy) ra = ld_row16(row_of(L, a));
            if (e.w != 0) rb = ld_row16(track_row_b<kMode>(J, L, e.y));
        }
        if (pull) {
            const uint32_t *list = source_list(J.aux, L.pack, e.y);
            const uint32_t c = list[0];
            if (active && e.z != 0) ra = ld_row16(row_of(L, a));
            for (uint32_t q = 0; q < c; q += 8) {
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    r[h] = zero;
                    if (q + h >= c) continue;
                    const uint32_t ref = list[1 + q + h];
                    if (kMode == kMarks && T.marked(ref)) r[h] = known;
                    else if (active) r[h] = ld_row16(row_ptr(J, ref, L.col));
                }
#pragma unroll
                for (int h = 0; h < 8; ++h) acc = combine16<kMax>(acc, r[h]);
            }
        }
        track_update<kMax, kMode>(J, T, L, group_mask, e, ra, rb, i);
        if (!__any_sync(0xffffffffu, pull)) continue;
        acc = combine16<kMax>(acc, ra);
        const bool new_a = active && pull && !same16(acc, ra);
        if (new_a) st_row16(row_of(L, a), acc);
        if (kMode == kMarks) {
            const uint32_t other = __ballot_sync(0xffffffffu, active && !same16(acc, T.c));
            const bool all = !(other & group_mask);
            if (pull && L.chunk == 0 && all != (e.z == 0)) {
                if (all) T.mark(a);
                else T.unmark(a);
            }
        } else if (kMode == kIds) {
            const bool any = (__ballot_sync(0xffffffffu, new_a) & group_mask) != 0;
            if (any && L.chunk == 0) *T.id_ptr(a) = T.fresh + T.index()[i];
        }
    }
}

// The ops of a segment through the private copy ring of every row group (kRing op
// slots of two chunks, as apply_tile).  Steps of two ops, the copies of the step
// kRing / 2 - 1 places ahead issued before the current step's rows are read back;
// ops are fetched a step before they are needed, so that no copy waits for a
// shared-memory load.  (One op per step, fetched where it is used, every op
// executed: 126 ms instead of 90 ms for 10^7 activity-driven events at n = 10^5.)
template <bool kMax, int kMode>
__device__ bool track_ring(const Job &J, Track &T, const uint2 *ops, uint32_t cnt, uint32_t first, uint32_t step,
                           uint32_t rounds, u64x2 *buf, const Lane &L, uint32_t group_mask)
{
    const uint32_t cpr = L.cpr;
    const bool active = L.active;
    // slot i of this thread: two chunks; cpr * stride = the consumer threads
    const uint32_t slot0 = smem_addr(buf + L.chunk + 2 * L.lane0 * cpr), slot_step = 32 * consumers(), second = 16 * cpr;
    bool pulls = false;
    auto entry = [&](uint32_t k) -> uint4 { return track_entry<kMode>(T, ops, cnt, first + k * step); };
    uint4 in[2], out[2];  // entries of the next copies and of the next updates
    auto issue = [&](uint32_t k) {
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t slot = slot0 + ((k + h) % kRing) * slot_step, kind = in[h].x >> kKindShift;
            if (active && kind != kPull) {
                if (in[h].z != 0 && kind != kCopy)
                    cp_async16(slot, row_of(L, in[h].x & kIdMask));
                if (in[h].w != 0) cp_async16(slot + second, track_row_b<kMode>(J, L, in[h].y));
            }
            in[h] = entry(k + 2 + h);
        }
        cp_async_commit();
    };
#pragma unroll
    for (uint32_t h = 0; h < 2; ++h) out[h] = in[h] = entry(h);
#pragma unroll 1
    for (uint32_t k = 0; k < kRing - 2; k += 2) issue(k);
#pragma unroll 1
    for (uint32_t k = 0; k < rounds; k += 2) {
        issue(k + kRing - 2);
        cp_async_wait_group<kRing / 2 - 1>();  // this step's copies have landed
        u64x2 ra[2], rb[2];
        const u64x2 known = kMode == kMarks ? T.c : u64x2{0, 0};
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t slot = slot0 + ((k + h) % kRing) * slot_step;
            ra[h] = kMode == kNoTrack || out[h].z != 0 ? lds16(slot) : known;
            rb[h] = kMode == kNoTrack || out[h].w != 0 ? lds16(slot + second) : known;
        }
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            track_update<kMax, kMode>(J, T, L, group_mask, out[h], ra[h], rb[h], first + (k + h) * step);
            pulls |= (out[h].x >> kKindShift) == kPull && (out[h].x & kIdMask) != kIdMask;
            out[h] = entry(k + 2 + h);
        }
    }
    cp_async_wait_group<0>();
    return pulls;
}

// Listed PULLs, x |= every source.  Marks: marked sources stand for C and are not
// loaded.  Ids: at least two sources differ from x; the result is new content.
template <bool kMax, int kMode>
__device__ void track_pulls(const Job &J, Track &T, uint32_t cnt, const Lane &L, uint32_t group_mask)
{
    const uint32_t per = 32u / L.cpr, g = (threadIdx.x & 31u) / L.cpr;
    const u64x2 zero{0, 0};
    for (uint32_t i = g; i < cnt; i += per) {
        const uint4 e = T.list()[i];
        if ((e.x >> kKindShift) != kPull) continue;
        const uint32_t *list = source_list(J.aux, L.pack, e.y);
        const uint32_t x = e.x & kIdMask, c = list[0];
        uint64_t *px = J.S + (uint64_t)x * J.ld + L.col;
        u64x2 old = zero, acc = zero;
        if (kMode == kMarks) old = e.z == 0 ? T.c : L.active ? ld_row16(px) : zero;
        for (uint32_t q = 0; q < c; q += 8) {
            uint32_t ref[8];
            u64x2 r[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) ref[k] = list[1 + (q + k < c ? q + k : q)];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (kMode == kMarks && T.marked(ref[k])) r[k] = T.c;
                else r[k] = L.active ? ld_row16(row_ptr(J, ref[k], L.col)) : zero;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) acc = combine16<kMax>(acc, r[k]);
        }
        if (kMode == kMarks) {
            acc = combine16<kMax>(acc, old);
            if (L.active && !same16(acc, old)) st_row16(px, acc);
            const bool all = __all_sync(group_mask, !L.active || same16(acc, T.c));
            if (L.chunk == 0 && all != (e.z == 0)) {
                if (all) T.mark(x);
                else T.unmark(x);
            }
        } else {
            if (L.active) {
                if (kMax) st_row16(px, combine16<kMax>(ld_row16(px), acc));
                else red_or16(px, acc);
            }
            if (L.chunk == 0) *T.id_ptr(x) = T.fresh + T.index()[i];
        }
    }
}

// One segment with marks or ids (cpr a power of two up to 32: a row group is part
// of a warp): every warp lists the ops of its share that are to be executed,
// then its row groups run them.  Whether there were any.
template <bool kMax, int kMode>
__device__ bool track_tile(const Job &J, Track &T, const uint2 *ops, uint32_t count, u64x2 *buf, const Lane &L,
                           uint32_t group_mask)
{
    const uint32_t lane = threadIdx.x & 31u, warp = (threadIdx.x >> 5) - 1u, warps = consumers() >> 5, per = 32u / L.cpr;
    uint32_t cnt = 0;
    // op i belongs to warp i mod warps: short levels spread over all warps
    for (uint32_t b = 0; b + warp < count; b += warps * 32u) {
        const uint32_t i = b + lane * warps + warp;
        uint4 e;
        const bool live = i < count && (kMode == kIds ? id_live(J, T, ops[i], L.pack, e) : mark_live(J, T, ops[i], L.pack, e));
        const uint32_t m = __ballot_sync(0xffffffffu, live);
        if (live) {
            const uint32_t to = cnt + __popc(m & ((1u << lane) - 1u));
            T.list()[to] = e;
            if (kMode == kIds) T.index()[to] = (uint16_t)i;
        }
        cnt += __popc(m);
    }
    __syncwarp();
    if (kMode == kMarks) {
        T.n_ops += (count - min(count, warp) + warps - 1) / warps;
        T.n_live += cnt;
    }
    if (cnt == 0) return false;
    const uint32_t rounds = (cnt + per - 1) / per;
    if (rounds <= 2)
        track_short<kMax, kMode>(J, T, ops, cnt, lane / L.cpr, per, rounds, L, group_mask);
    else if (__any_sync(0xffffffffu, track_ring<kMax, kMode>(J, T, ops, cnt, lane / L.cpr, per, rounds, buf, L, group_mask)))
        track_pulls<kMax, kMode>(J, T, cnt, L, group_mask);
    return true;
}

// One segment with every op executed.
template <bool kMax>
__device__ void whole_tile(const Job &J, Track &T, const uint2 *ops, uint32_t count, u64x2 *buf, const Lane &L,
                           uint32_t group_mask)
{
    const uint32_t before = ((threadIdx.x >> 5) - 1u) * (32u / L.cpr);  // row groups of the warps before this one
    if (count <= before) return;
    const uint32_t rounds = (count - before + L.stride - 1) / L.stride;
    if (rounds <= 2) {
        track_short<kMax, kNoTrack>(J, T, ops, count, L.lane0, L.stride, rounds, L, group_mask);
        return;
    }
    const bool pulls = track_ring<kMax, kNoTrack>(J, T, ops, count, L.lane0, L.stride, rounds, buf, L, group_mask);
    if (!pulls || !L.active) return;
    // multi-source updates of tie groups (hub rows) in a second pass
    if (kMax) {
        for (uint32_t o = L.lane0; o < count; o += L.stride) {
            const uint2 op = ops[o];
            if ((op.x >> kKindShift) == kPull) apply_pull<kMax>(J, op.x & kIdMask, op.y, L);
        }
    } else {
        apply_pulls_ring(J, ops, count, buf + L.chunk, L);
    }
}

// Marks of a freshly initialised S: every row whose segment is zero.
__device__ void mark_init(const Job &J, Track &T, uint64_t w0, uint32_t ct)
{
    const uint32_t nbits = (T.rows >> T.shift) + 1u, full = nbits / 32u;
    for (uint32_t i = ct; i < J.mark_words; i += consumers())
        T.bits()[i] = J.mark_init == 0 || i > full ? 0u : i < full ? 0xffffffffu : (1u << (nbits & 31u)) - 1u;
    if (ct < 13) T.stat(0)[ct] = 0;  // and the key
    consumers_sync();
    if (J.mark_init == 0 || J.mark_words == 0) return;
    const uint64_t c0 = 64 * w0, c1 = 64 * (w0 + J.sw) < J.ncols ? 64 * (w0 + J.sw) : J.ncols;
    for (uint64_t c = c0 + ct; c < c1; c += consumers()) {
        const uint32_t x = J.mark_init == 1 ? (uint32_t)c : __ldg(J.src + c);
        if (x < T.rows) T.unmark(x);
    }
    consumers_sync();
}

// Marks, end of a window (before the next one's first barrier): statistics.
// Every lane of a row group has counted its sampled updates.
__device__ inline void mark_count(Track &T, uint32_t win)
{
    uint32_t seen = 0, equal = 0;
    if (T.sample) {
        seen = __reduce_add_sync(0xffffffffu, T.n_seen);
        equal = __reduce_add_sync(0xffffffffu, T.n_equal);
    }
    uint32_t *stat = T.stat(win);
    if ((threadIdx.x & 31u) == 0) {
        if (T.n_ops) atomicAdd(&stat[0], T.n_ops);
        if (T.n_live) atomicAdd(&stat[1], T.n_live);
        if (seen) atomicAdd(&stat[2], seen);
        if (equal) atomicAdd(&stat[3], equal);
    }
    T.n_ops = T.n_live = T.n_seen = T.n_equal = 0;
}

// Marks, at a window's first pack, all consumers: read the last window's
// statistics and choose how the next one is run.  `win` counts windows.
__device__ inline void mark_window(const Job &J, Track &T, uint32_t win, const Lane &L, uint32_t ct)
{
    uint32_t *prev = T.stat(win + 2u), *next = T.stat(win + 1u);
    const uint32_t ops = *(volatile uint32_t *)&prev[0], live = *(volatile uint32_t *)&prev[1],
                   seen = *(volatile uint32_t *)&prev[2], equal = *(volatile uint32_t *)&prev[3];
    if (ct < 4) next[ct] = 0;  // read last two windows ago
    T.quiet = T.on && live == 0;
    T.settled = seen ? equal == seen : T.quiet;
    T.sample = (win & 3u) == 0;
    if (T.want) {
        if (L.chunk == 0 && T.best_size) atomicMax(T.key(), T.best_size << 10 | L.lane0);
        consumers_sync();
        const uint32_t key = *(volatile uint32_t *)T.key();
        T.want = false;
        T.best_size = 0;
        if (key != 0 && (!T.on || (key >> 10) > T.c_size)) {
            T.c = *T.cand((key & 1023u) * L.cpr + L.chunk);
            T.c_size = key >> 10;
            T.on = true;
            T.quiet = false;
            for (uint32_t i = ct; i < J.mark_words; i += consumers()) T.bits()[i] = 0;
        }
        consumers_sync();
        if (ct == 0) *T.key() = 0;
        return;
    }
    if (T.shift == 0 && seen && 2 * equal >= seen && (!T.on || 8 * live >= ops)) T.want = T.sample = true;
    else if (T.on && seen && 2 * live > ops) T.on = false;  // too few rows are marked: the checks do not pay
}

// Ids at the start: every row its own, or, in a matrix initialised by this
// application, 0 but for the rows whose source column lies in the CTA's slab.
__global__ void init_ids_kernel(uint32_t *ids, uint64_t rows, uint32_t pitch, uint32_t sw, bool zero, bool identity)
{
    const uint64_t total = rows * pitch / 4;  // pitch is a multiple of 8
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < total; p += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t row = 4 * p / pitch;
        const uint32_t cta = (uint32_t)(4 * p - row * pitch), own = (uint32_t)(row / 64 / sw);
        const uint32_t other = zero ? 0u : (uint32_t)row + 1u, mine = identity ? (uint32_t)row + 1u : other;
        reinterpret_cast<uint4 *>(ids)[p] = make_uint4(own == cta ? mine : other, own == cta + 1 ? mine : other,
                                                       own == cta + 2 ? mine : other, own == cta + 3 ? mine : other);
    }
}

__global__ void init_source_ids_kernel(uint32_t *ids, uint32_t pitch, uint32_t sw, const uint32_t *src, uint32_t nsrc,
                                       uint32_t rows)
{
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nsrc; c += gridDim.x * blockDim.x)
        if (src[c] < rows) ids[(uint64_t)src[c] * pitch + c / 64 / sw] = src[c] + 1u;
}

// ---------------------------------------------------------------------------
// local record: the window's rows are gathered into shared memory, its levels
// are applied there, and every written row goes back to the matrix from the op
// that writes it for the last time (rows that are only read are not stored)
// ---------------------------------------------------------------------------
template <bool kMax>
__device__ inline void apply_record(const Job &J, const uint32_t *rec, u64x2 *buf, const Lane &L)
{
    const uint32_t D = rec[0], nlev = rec[2], nops = rec[3];
    const uint32_t *rows = rec + 4, *lvl = rows + D, *ops = lvl + nlev + 1, *aux = ops + nops;
    const uint32_t cpr = L.cpr, lane0 = L.lane0, stride = L.stride;
    const uint64_t col = L.col;
    const bool active = L.active;
    u64x2 *mine = buf + L.chunk;  // slot q of this chunk lives at buf[q * cpr + chunk]

    if (active) {
        uint32_t d = lane0;
        for (; d + 3 * stride < D; d += 4 * stride) {
            uint32_t r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] = rows[d + k * stride];
#pragma unroll
            for (int k = 0; k < 4; ++k) cp_async16(mine + (d + k * stride) * cpr, J.S + (uint64_t)r[k] * J.ld + col);
        }
        for (; d < D; d += stride) cp_async16(mine + d * cpr, J.S + (uint64_t)rows[d] * J.ld + col);
    }
    cp_async_wait_all();
    consumers_sync();
    for (uint32_t l = 0; l < nlev; ++l) {
        if (active) {
            const uint32_t e = lvl[l + 1];
            // two ops per step: the ops of one level touch distinct rows, so
            // both ops' loads can be issued before either op's stores
            for (uint32_t o = lvl[l] + lane0; o < e; o += 2 * stride) {
                uint32_t op[2];
                bool live[2];
                u64x2 x[2], y[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t idx = o + k * stride;
                    live[k] = idx < e;
                    op[k] = live[k] ? ops[idx] : (kPull << kKindShift);
                    const uint32_t kind = op[k] >> kKindShift, a = (op[k] >> kLocalBits) & kLocalMask,
                                   b = op[k] & kLocalMask;
                    if (kind != kPull) {
                        x[k] = lds16(mine + a * cpr);
                        y[k] = lds16(mine + b * cpr);
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t kind = op[k] >> kKindShift, a = (op[k] >> kLocalBits) & kLocalMask,
                                   b = op[k] & kLocalMask;
                    // a row's last write in the window also goes to the matrix (write-through)
                    if (kind == kEvent) {
                        const u64x2 r = combine16<kMax>(x[k], y[k]);
                        sts16(mine + a * cpr, r);
                        sts16(mine + b * cpr, r);
                        if (op[k] & kLastA) st_row16(J.S + (uint64_t)rows[a] * J.ld + col, r);
                        if (op[k] & kLastB) st_row16(J.S + (uint64_t)rows[b] * J.ld + col, r);
                    } else if (kind == kOneway) {
                        const u64x2 r = combine16<kMax>(x[k], y[k]);
                        sts16(mine + a * cpr, r);
                        if (op[k] & kLastA) st_row16(J.S + (uint64_t)rows[a] * J.ld + col, r);
                    } else if (kind == kCopy) {
                        sts16(mine + a * cpr, y[k]);
                    } else if (live[k]) {
                        u64x2 acc = lds16(mine + a * cpr);
                        const uint32_t c = aux[b];
                        for (uint32_t q = 1; q <= c; ++q) acc = combine16<kMax>(acc, lds16(mine + aux[b + q] * cpr));
                        sts16(mine + a * cpr, acc);
                        if (op[k] & kLastA) st_row16(J.S + (uint64_t)rows[a] * J.ld + col, acc);
                    }
                }
            }
        }
        consumers_sync();
    }
    // no write-back pass: every written row was stored at its last write
}

// ---------------------------------------------------------------------------
// resident slab: for a network small enough that rw words of EVERY row fit in
// shared memory, the CTA loads its slab of the matrix once, applies the whole
// schedule there and stores it once; only the schedule streams from L2/HBM.
// The plan holds tile packs only (node-id ops).  Consumers take one op each of
// the current segment (its ops are independent), fetch their op of the next
// segment beside it, and meet at a named barrier; a level costs its barrier and
// about 60 instructions (resident_levels; larger ones also the bank conflicts of
// random rows: 0.12 us for 93 ops, 0.18 us for 319).
// Once a pack changes nothing, the next one is checked as a whole without its
// level barriers (if no op changes a row as the rows stand, none does), and after
// a run of such packs the rows are compared with their component's root rows: when
// all are equal, nothing that is left of the schedule can change a row, and the
// CTA stops.  ER n = 10^4, m = 10^7 (the giant component settles in the first few
// per cent): 21.0 ms with every level walked, 8.2 ms with packs checked, 0.47 ms.
// Shared memory: barriers | rows[rows] | saved rows[ntemp] | ring.
// ---------------------------------------------------------------------------
constexpr uint32_t kResidentMaxStages = 8;
constexpr uint32_t kResidentHead = 128;  // the ring's barriers
constexpr uint32_t kResidentMinStages = 2;
// Consumer threads of a resident CTA (the rest exit): enough for a level of
// average size, since every level's barrier waits for all of them.
constexpr uint32_t kResidentConsumers = 256;
// Most waves of open plans in one launch; beyond, column slabs.  Batches of networks,
// resident and column slabs: ER n = 8,000 (5 waves) 1.09, 1.81 ms, n = 20,000 (9, 13 waves)
// 2.84, 3.06 and 4.08, 3.17; activity-driven n = 16,384 (11 waves) 4.9, 5.4; bursty n =
// 20,000 (5, 7, 9 waves) 5.8, 7.8 and 8.65, 8.57 and 11.1, 9.8.  With records kept for
// that launch: bursty n = 8,000 (3, 5 waves) 3.0, 3.0 and 4.6, 3.1; activity-driven n =
// 8,000 (7 waves) 2.4, 2.3.
constexpr uint64_t kResidentWaves = 11, kResidentTieWaves = 7;

template <int RW>
struct alignas(RW == 1 ? 8 : 16) RRow {
    uint64_t w[RW];
};

__host__ __device__ inline uint64_t resident_rows_bytes(uint64_t rows, uint64_t temps, uint32_t rw)
{
    return ((rows + temps) * 8ull * rw + 127ull) & ~127ull;
}

template <bool kMax, int RW>
__device__ inline RRow<RW> rcombine(RRow<RW> a, const RRow<RW> &b)
{
#pragma unroll
    for (int k = 0; k < RW; ++k) a.w[k] = kMax ? max8x8(a.w[k], b.w[k]) : (a.w[k] | b.w[k]);
    return a;
}

template <int RW>
__device__ inline RRow<RW> ld_rrow(const uint64_t *p)
{
    RRow<RW> r;
    if (RW == 1) {
        asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(r.w[0]) : "l"(p) : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < RW; k += 2) {
            const u64x2 x = ld_row16(p + k);
            r.w[k] = x.x;
            r.w[k + 1] = x.y;
        }
    }
    return r;
}

template <int RW>
__device__ inline void st_rrow(uint64_t *p, const RRow<RW> &r)
{
    if (RW == 1) {
        asm volatile("st.global.u64 [%0], %1;" ::"l"(p), "l"(r.w[0]) : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < RW; k += 2) st_row16(p + k, u64x2{r.w[k], r.w[k + 1]});
    }
}

// Rows of the resident slab by 32-bit shared-memory address.
template <int RW>
__device__ inline RRow<RW> lds_rrow(uint32_t a)
{
    RRow<RW> r;
    if (RW == 1) {
        asm volatile("ld.shared.u64 %0, [%1];" : "=l"(r.w[0]) : "r"(a) : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < RW; k += 2)
            asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(r.w[k]), "=l"(r.w[k + 1]) : "r"(a + 8u * k) : "memory");
    }
    return r;
}

template <int RW>
__device__ inline void sts_rrow(uint32_t a, const RRow<RW> &r)
{
    if (RW == 1) {
        asm volatile("st.shared.u64 [%0], %1;" ::"r"(a), "l"(r.w[0]) : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < RW; k += 2)
            asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(a + 8u * k), "l"(r.w[k]), "l"(r.w[k + 1]) : "memory");
    }
}

__device__ inline uint2 lds_op(uint32_t a)
{
    uint2 r;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "r"(a) : "memory");
    return r;
}

__device__ inline uint32_t lds_u16(uint32_t a)
{
    uint16_t r;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(r) : "r"(a) : "memory");
    return r;
}

__device__ inline uint32_t lds_u32(uint32_t a)
{
    uint32_t r;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(a) : "memory");
    return r;
}

template <int RW>
__device__ inline bool same_row(const RRow<RW> &a, const RRow<RW> &b)
{
    bool same = true;
#pragma unroll
    for (int k = 0; k < RW; ++k) same = same && a.w[k] == b.w[k];
    return same;
}

// Whether an op on rows (shared address rb, node ids; saved rows: tb, temp ids)
// would change a row as the rows stand.
template <bool kMax, int RW>
__device__ inline bool resident_live(uint2 op, uint32_t rb, uint32_t tb, const uint32_t *aux, const uint32_t *pack)
{
    constexpr uint32_t kRowB = 8u * RW;
    const uint32_t kind = op.x >> kKindShift;
    const RRow<RW> x = lds_rrow<RW>(rb + (op.x & kIdMask) * kRowB);
    if (kind != kPull) {
        const RRow<RW> y = lds_rrow<RW>(rb + op.y * kRowB);
        return !same_row<RW>(kind == kEvent ? y : rcombine<kMax, RW>(x, y), x);
    }
    const uint32_t *list = source_list(aux, pack, op.y);
    for (uint32_t q = 1; q <= list[0]; ++q) {
        const uint32_t ref = list[q];
        const RRow<RW> y = lds_rrow<RW>((ref & kTempRef) ? tb + (ref & ~kTempRef) * kRowB : rb + ref * kRowB);
        if (!same_row<RW>(rcombine<kMax, RW>(x, y), x)) return true;
    }
    return false;
}

// One thread's op of a level, with everything worked out before the level's barrier:
// r = [la] | [lb] (PULL: and its sources) goes to sa and, for an EVENT, to lb.
// EVENT and ONEWAY: la = sa; PULL: la = lb = sa; COPY: la = lb; no op: row 0.
struct ResOp {
    uint32_t la, lb, sa;
    bool store, both;
    uint32_t list, c, ref[4];  // PULL: source list, number of sources (else 0), the first ones
};

// Word b of a source list, in the pack at shared address packa or outside it.
__device__ inline uint32_t list_word(const uint32_t *aux, uint32_t packa, uint32_t b)
{
    return b < kOutsideList ? lds_u32(packa + 4u * b) : __ldg(aux + (b - kOutsideList));
}

template <int RW, bool kTies, bool kAhead>
__device__ __forceinline__ ResOp res_decode(uint2 op, bool act, uint32_t rb, uint32_t tb, const uint32_t *aux,
                                            uint32_t packa)
{
    constexpr uint32_t kRowB = 8u * RW;
    const uint32_t kind = op.x >> kKindShift;
    ResOp o;
    o.store = act;
    o.both = act && kind == kEvent;
    if (!kTies) {
        o.sa = o.la = act ? rb + (op.x & kIdMask) * kRowB : rb;
        o.lb = act ? rb + op.y * kRowB : rb;
        return o;
    }
    const bool pull = act && kind == kPull, copy = act && kind == kCopy;
    o.sa = (copy ? tb : rb) + (act ? op.x & kIdMask : 0u) * kRowB;
    o.lb = pull ? o.sa : act ? rb + op.y * kRowB : rb;
    o.la = copy ? o.lb : o.sa;
    o.list = op.y;
    o.c = 0;
    if (pull) {
        o.c = list_word(aux, packa, op.y);
        if (!kAhead) return o;
        if (op.y < kOutsideList) {  // (words behind the list's end stay unused)
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k)
                o.ref[k] = lds_u32(packa + 4u * (op.y + 1 + k < kStageBytes / 4 ? op.y + 1 + k : op.y));
        } else {
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) o.ref[k] = k < o.c ? list_word(aux, packa, op.y + 1 + k) : 0u;
        }
    }
    return o;
}

// Stores the result of an op; whether a row changed.
template <int RW>
__device__ __forceinline__ uint64_t res_store(const ResOp &o, const RRow<RW> &x, const RRow<RW> &y, const RRow<RW> &r)
{
    if (o.store) sts_rrow<RW>(o.sa, r);
    if (o.both) sts_rrow<RW>(o.lb, r);
    uint64_t diff = 0;
#pragma unroll
    for (int w = 0; w < RW; ++w) diff |= (r.w[w] ^ x.w[w]) | (o.both ? r.w[w] ^ y.w[w] : 0ull);
    return o.store ? diff : 0ull;
}

// r combined with the `c` sources at word b of a list.
template <bool kMax, int RW>
__device__ __noinline__ RRow<RW> resident_sources(RRow<RW> r, uint32_t b, uint32_t c, uint32_t rb, uint32_t tb,
                                                  const uint32_t *aux, uint32_t packa)
{
    constexpr uint32_t kRowB = 8u * RW;
    for (uint32_t q = 0; q < c; q += 4) {  // four independent loads at a time
        RRow<RW> z[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t ref = list_word(aux, packa, b + (q + j < c ? q + j : q));
            z[j] = lds_rrow<RW>((ref & kTempRef ? tb : rb) + (ref & ~kTempRef) * kRowB);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) r = rcombine<kMax, RW>(r, z[j]);
    }
    return r;
}

// Ops i, i + C, ..., K of them, of a level that ends at e.
template <int K, bool kMax, int RW, bool kTies>
__device__ __forceinline__ uint64_t resident_round(uint32_t opa, uint32_t i, uint32_t e, uint32_t C, uint32_t rb,
                                                   uint32_t tb, const uint32_t *aux, uint32_t packa)
{
    uint2 op[K];
    ResOp o[K];
    RRow<RW> x[K], y[K];
    uint64_t diff = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) op[k] = lds_op(opa + (i + k * C < e ? i + k * C : i) * 8u);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        o[k] = res_decode<RW, kTies, false>(op[k], i + k * C < e, rb, tb, aux, packa);
        x[k] = lds_rrow<RW>(o[k].la);
        y[k] = lds_rrow<RW>(o[k].lb);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        RRow<RW> r = rcombine<kMax, RW>(x[k], y[k]);
        if (kTies && o[k].c) r = resident_sources<kMax, RW>(r, o[k].list + 1, o[k].c, rb, tb, aux, packa);
        diff |= res_store<RW>(o[k], x[k], y[k], r);
    }
    return diff;
}

// The ops of a level behind the consumers' first ones, from op `first` on.  Out of
// line, as the sources above: rare, and the level loop stays short.
template <bool kMax, int RW, bool kTies>
__device__ __noinline__ uint64_t resident_more(uint32_t opa, uint32_t first, uint32_t e, uint32_t ct, uint32_t C,
                                               uint32_t rb, uint32_t tb, const uint32_t *aux, uint32_t packa)
{
    uint64_t diff = 0;
    for (; first + C < e; first += 2 * C)
        if (first + ct < e) diff |= resident_round<2, kMax, RW, kTies>(opa, first + ct, e, C, rb, tb, aux, packa);
    for (; first < e; first += C)
        if (first + ct < e) diff |= resident_round<1, kMax, RW, kTies>(opa, first + ct, e, C, rb, tb, aux, packa);
    return diff;
}

// The levels of one pack; whether a row changed.  The chain of a level runs from
// barrier to barrier through the rows' load, one combine and the store, all without
// a branch; the next level's op is decoded while the rows load, and the one after
// it fetched.  Bound by the instructions of one warp's chain and, with 8 warps, by
// issue slots.  A level of 93 ops, 256 threads: 307 cycles with ops decoded behind
// the barrier and conditional stores, 219 now (449 and 317 with the code for ties);
// warps that skip what they have no op for take 270 (the branch is longer than the
// skipped part).  Bursty n = 20,011, 500,009 events: 6.46 ms, 5.30 ms now.
template <bool kMax, int RW, bool kTies>
__device__ __forceinline__ bool resident_levels(uint32_t opa, uint32_t sega, uint32_t nseg, uint32_t rb, uint32_t tb,
                                                const uint32_t *aux, uint32_t ct, uint32_t C)
{
    constexpr uint32_t kRowB = 8u * RW;
    const uint32_t packa = opa - kPackHead * 8u;
    // (ops and ends behind the pack's last are inside the stage and unused)
    auto fetch = [&](uint32_t i) { return lds_op(opa + (i + ct < kPackOps ? i + ct : 0u) * 8u); };
    uint64_t diff = 0;
    uint32_t b = 0, e = lds_u16(sega), e1 = lds_u16(sega + 2u);
    uint2 next = fetch(e);
    ResOp o = res_decode<RW, kTies, true>(fetch(0), ct < e, rb, tb, aux, packa);
    for (uint32_t k = 1;; ++k) {
        const RRow<RW> x = lds_rrow<RW>(o.la), y = lds_rrow<RW>(o.lb);
        const uint32_t e2 = lds_u16(sega + 2u * (k + 1));
        const uint2 after = fetch(e1);
        const ResOp on = res_decode<RW, kTies, true>(next, e + ct < e1 && k < nseg, rb, tb, aux, packa);
        RRow<RW> r = rcombine<kMax, RW>(x, y);
        if (kTies && o.c) {
            RRow<RW> z[4];  // four independent loads
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t ref = (uint32_t)j < o.c ? o.ref[j] : o.ref[0];
                z[j] = lds_rrow<RW>((ref & kTempRef ? tb : rb) + (ref & ~kTempRef) * kRowB);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) r = rcombine<kMax, RW>(r, z[j]);
            if (o.c > 4) r = resident_sources<kMax, RW>(r, o.list + 5, o.c - 4, rb, tb, aux, packa);
        }
        diff |= res_store<RW>(o, x, y, r);
        if (e - b > C) diff |= resident_more<kMax, RW, kTies>(opa, b + C, e, ct, C, rb, tb, aux, packa);
        if (k >= nseg) break;
        consumers_sync(C);
        b = e;
        e = e1;
        e1 = e2;
        next = after;
        o = on;
    }
    return diff != 0;
}

template <bool kMax, int RW>
__device__ void resident_slab(const Job &J, uint32_t smem_bytes, uint8_t *smem, uint32_t cta)
{
    __shared__ int32_t r_gate;
    __shared__ uint32_t r_abort, r_ran[3];
    using Row = RRow<RW>;
    // the job's fields in registers (the barriers' memory clobbers would reload them)
    const uint32_t *const aux = J.aux;
    int32_t *const status = J.status;
    uint64_t *const S = J.S;
    const uint64_t ld = J.ld;
    const uint32_t rows = J.rows;
    Row *R = reinterpret_cast<Row *>(smem + kResidentHead);
    const uint32_t rb = smem_addr(R), tb = rb + rows * 8u * RW;  // rows, then saved rows
    const uint32_t ring_off = kResidentHead + (uint32_t)resident_rows_bytes(rows, J.ntemp, RW);
    // a power of two of stages (at least kResidentMinStages by the plan's check)
    const uint32_t fit = (smem_bytes - ring_off) / kStageBytes;
    uint32_t nst = kResidentMaxStages;
    while (nst > fit) nst >>= 1;
    PackRing ring;
    ring.full = reinterpret_cast<uint64_t *>(smem);
    ring.empty = ring.full + kResidentMaxStages;
    ring.stage = smem + ring_off;
    ring.mask = nst - 1;
    ring.shift = __ffs(nst) - 1;
    const uint64_t w0 = J.w_begin + (uint64_t)cta * RW;
    const uint32_t C = consumers() < J.res_threads ? consumers() : J.res_threads;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    if (threadIdx.x == 0) {
        r_gate = *(volatile int32_t *)status;  // an earlier error gates this job
        r_abort = 0;
        r_ran[0] = r_ran[1] = r_ran[2] = 1;
        for (uint32_t s = 0; s < nst; ++s) {
            mbar_init(&ring.full[s], 1);
            mbar_init(&ring.empty[s], C / 32u);
        }
        fence_mbar_init();
    }
    __syncthreads();
    if (r_gate != 0) return;
    if (warp == 0) {
        produce_packs(J, ring, &r_abort);
        return;
    }
    // ---------------- consumers ----------------
    const uint32_t ct = threadIdx.x - 32;
    if (ct >= C) return;  // small levels keep few warps busy: the others leave
    if (J.identity) {  // one bit per row of this slab, nothing to read
        for (uint32_t i = ct; i < rows; i += C) {
            Row r{};
            if (i / 64 - w0 < RW && i / 64 >= w0) r.w[i / 64 - w0] = 1ull << (i % 64);
            R[i] = r;
        }
    } else {
        uint32_t i = ct;
        for (; i + 3 * C < rows; i += 4 * C) {
            Row r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] = ld_rrow<RW>(S + (uint64_t)(i + k * C) * ld + w0);
#pragma unroll
            for (int k = 0; k < 4; ++k) R[i + k * C] = r[k];
        }
        for (; i < rows; i += C) R[i] = ld_rrow<RW>(S + (uint64_t)i * ld + w0);
    }
    uint32_t skipped = 0, check = 2;  // packs skipped in a row; at this many the rows are compared
    for (uint32_t q = 0;; ++q) {
        const bool ready = ring.wait_full(q);
        if (!ready && ct == 0) record_status(status, TN_ETIMEOUT);
        const uint32_t *head = reinterpret_cast<const uint32_t *>(ring.at(q));
        const bool stop = !ready || *(volatile uint32_t *)&r_abort != 0 || ((head[1] >> 16) & kPackEnd);
        // orders the previous pack's (or the loads') stores before this pack's
        // loads, and agrees on stopping
        if (consumers_sync_or(stop, C)) {
            if (!ready || *(volatile uint32_t *)&r_abort != 0) return;
            break;
        }
        const uint16_t *seg = reinterpret_cast<const uint16_t *>(head + 4);
        uint32_t nseg = head[1] & 0xFFFFu;
        const uint32_t nops = head[0], opa = smem_addr(head) + kPackHead * 8u;
        if (*(volatile uint32_t *)&r_ran[(q + 2u) % 3u] == 0) {
            // the last pack changed nothing: look at all levels of this one at
            // once, first the ops on rows (saved rows are written on the way),
            // then the PULLs; if none changes a row as they stand, none does
            const bool ties = (head[1] >> 16) & kPackTies;
            bool live = false;
            for (uint32_t o0 = ct; o0 < nops && !live; o0 += 4 * C) {
                // four ops of independent loads; past the end, op 0 again
                uint2 op[4];
                RRow<RW> x[4], y[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) op[k] = lds_op(opa + (o0 + k * C < nops ? o0 + k * C : 0u) * 8u);
                if (ties) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t kind = op[k].x >> kKindShift;
                        if (kind == kCopy)
                            sts_rrow<RW>(tb + (op[k].x & kIdMask) * (8u * RW), lds_rrow<RW>(rb + op[k].y * (8u * RW)));
                        else if (kind != kPull) live |= resident_live<kMax, RW>(op[k], rb, tb, aux, head);
                    }
                    continue;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[k] = lds_rrow<RW>(rb + (op[k].x & kIdMask) * (8u * RW));
                    y[k] = lds_rrow<RW>(rb + op[k].y * (8u * RW));
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    live |= !same_row<RW>((op[k].x >> kKindShift) == kEvent ? y[k] : rcombine<kMax, RW>(x[k], y[k]), x[k]);
            }
            live = consumers_sync_or(live, C);
            if (!live && ties) {
                for (uint32_t o = ct; o < nops && !live; o += C) {
                    const uint2 op = lds_op(opa + o * 8u);
                    if ((op.x >> kKindShift) == kPull) live = resident_live<kMax, RW>(op, rb, tb, aux, head);
                }
                live = consumers_sync_or(live, C);
            }
            if (!live) {
                nseg = 0;
                if (J.label && ++skipped == check) {
                    // every row equal to its component's root row: nothing that is
                    // left of the schedule can change a row
                    bool differ = false;
                    for (uint32_t i = ct; i < rows && !differ; i += C)
                        differ = !same_row<RW>(R[i], R[__ldg(J.label + i)]);
                    if (!consumers_sync_or(differ, C)) {
                        if (ct == 0) r_abort = 1;
                        break;
                    }
                    check *= 2;
                }
            } else {
                skipped = 0;
            }
        }
        if (ct == 0) r_ran[(q + 1u) % 3u] = 0;  // read one pack ago, set in the next one
        bool changed = false;
        const uint32_t sega = smem_addr(seg);
        if (nseg == 0) {
        } else if ((head[1] >> 16) & kPackTies) {
            changed = resident_levels<kMax, RW, true>(opa, sega, nseg, rb, tb, aux, ct, C);
        } else {
            changed = resident_levels<kMax, RW, false>(opa, sega, nseg, rb, tb, aux, ct, C);
        }
        changed = __any_sync(0xffffffffu, changed);
        if (lane == 0) {
            if (changed) r_ran[q % 3u] = 1;
            mbar_arrive(&ring.empty[q & ring.mask]);
        }
    }
    for (uint32_t i = ct; i < rows; i += C) st_rrow<RW>(S + (uint64_t)i * ld + w0, R[i]);
    if (J.identity && (w0 + RW) * 64 >= J.ncols) {  // the padding behind the last slab
        const uint32_t pad = (uint32_t)(ld - (w0 + RW));
        for (uint64_t k = ct; pad && k < (uint64_t)rows * pad; k += C)
            S[k / pad * ld + w0 + RW + k % pad] = 0ull;
    }
}

// The next pack of the ring, once every consumer is done with the one before
// (level barrier: its stores are ordered before this pack's loads).  All
// consumers agree on stopping; false = stop.
__device__ inline bool next_pack(const Job &J, const PackRing &ring, uint32_t q, const uint32_t *abort_flag, bool ready)
{
    if (!ready && threadIdx.x == 32) record_status(J.status, TN_ETIMEOUT);
    const uint32_t meta = reinterpret_cast<const uint32_t *>(ring.at(q))[1];
    const bool stop = !ready || *(volatile const uint32_t *)abort_flag != 0 || ((meta >> 16) & kPackEnd);
    return !consumers_sync_or(stop);
}

// Consumers of a column slab in a plan with records, or whose slab width does not
// divide a warp into row groups, or whose row buffer is too small for copy rings.
template <bool kMax>
__device__ void consume_plain(const Job &J, const PackRing &ring, const uint32_t *abort_flag, u64x2 *rowbuf, Lane L,
                              uint32_t ct)
{
    for (uint32_t q = 0;; ++q) {
        if (!next_pack(J, ring, q, abort_flag, ring.wait_full(q))) return;
        const uint32_t *head = reinterpret_cast<const uint32_t *>(ring.at(q));
        const uint32_t nseg = head[1] & 0xFFFFu;
        L.pack = head;
        if ((head[1] >> 16) & kPackLocal) {
            apply_record<kMax>(J, head + 4, rowbuf, L);
        } else {
            const uint16_t *seg = reinterpret_cast<const uint16_t *>(head + 4);
            const uint2 *ops = reinterpret_cast<const uint2 *>(head) + kPackHead;
            for (uint32_t k = 0, b = 0; k < nseg; ++k) {
                const uint32_t e = seg[k];
                if (e == b) continue;
                if (b) consumers_sync();
                apply_tile<kMax>(J, ops + b, e - b, rowbuf, J.dcap, L);
                b = e;
            }
        }
        __syncwarp();
        if ((ct & 31u) == 0) mbar_arrive(&ring.empty[q & ring.mask]);
    }
}

// Whether some row of the slab, in this thread's share, differs from its
// component's root row.  If none does, nothing that is left of the schedule can
// change a row.  Reads the slab once at most (n = 10^5: 12.8 MB per CTA).
__device__ inline bool rows_differ(const Job &J, const Lane &L)
{
    if (!L.active) return false;
    uint32_t have = kNoRef;
    u64x2 root{0, 0};
    for (uint32_t i = L.lane0; i < J.rows; i += 4 * L.stride) {
        u64x2 r[4];
        uint32_t lab[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t row = i + k * L.stride < J.rows ? i + k * L.stride : i;
            lab[k] = __ldg(J.label + row);
            r[k] = ld_row16(row_of(L, row));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (lab[k] != have) {
                have = lab[k];
                root = ld_row16(row_of(L, have));
            }
            if (!same16(r[k], root)) return true;
        }
    }
    return false;
}

// Consumers of a column slab with tracked rows (tiles only).  While nothing is
// executed, the next pack is looked at as a whole, without its level barriers:
// if none of its ops is to be executed, no row changes between its levels either.
template <bool kMax, int kMode>
__device__ void consume_tracked(const Job &J, const PackRing &ring, const uint32_t *abort_flag, u64x2 *rowbuf,
                                uint64_t w0, uint32_t cta, Lane L, uint32_t ct)
{
    Track T;
    T.at = (uint32_t)(kSlabHead + (size_t)J.dcap * J.sw * 8);
    T.slot = (ct >> 5) * (kListOps / (consumers() >> 5));
    T.rows = J.rows;
    T.c = u64x2{0, 0};
    T.want = T.quiet = T.on = T.settled = false;
    T.best_size = T.n_ops = T.n_live = T.n_seen = T.n_equal = T.c_size = T.shift = T.fresh = 0;
    T.sample = kMode == kMarks;
    if (kMode == kIds) {
        T.ids = J.ids + cta;
        T.pitch = J.pitch;
        if (ct < 3) *T.stat(ct) = 1;
    } else {
        T.on = J.mark_words != 0;
        T.shift = J.mark_shift;
        mark_init(J, T, w0, ct);
        if (!T.on) T.shift = 1;  // no marks at all: no candidates either
    }
    const uint32_t g = (ct & 31u) / L.cpr;
    const uint32_t group_mask = L.cpr == 32 ? 0xffffffffu : ((1u << L.cpr) - 1u) << (g * L.cpr);
    uint32_t settled = 0, check = 2;  // windows that changed nothing; at this many the rows are compared
    uint32_t win = 0, first = J.rows + 1u;  // ids 1..rows are the rows' own
    for (uint32_t q = 0;; ++q) {
        const bool ready = __all_sync(0xffffffffu, ring.wait_full(q));
        const uint32_t *head = reinterpret_cast<const uint32_t *>(ring.at(q));
        const bool starts = kMode == kMarks && q && ready && ((head[1] >> 16) & kPackWindow);
        if (starts) mark_count(T, win);  // of the window that ends here, read behind the barrier
        if (!next_pack(J, ring, q, abort_flag, ready)) return;
        if (starts) {
            mark_window(J, T, ++win, L, ct);
            if (J.label && T.settled && ++settled == check) {
                if (!consumers_sync_or(rows_differ(J, L))) {
                    if (ct == 0) *const_cast<volatile uint32_t *>(abort_flag) = 1;
                    return;
                }
                check *= 2;
            }
        }
        const uint16_t *seg = reinterpret_cast<const uint16_t *>(head + 4);
        const uint2 *ops = reinterpret_cast<const uint2 *>(head) + kPackHead;
        const uint32_t nops = head[0];
        uint32_t nseg = head[1] & 0xFFFFu;
        L.pack = head;
        if (kMode == kIds) {
            T.quiet = *(volatile uint32_t *)T.stat(q + 2) == 0;  // the last pack executed nothing
            if (ct == 0) *T.stat(q + 1) = 0;                     // read one pack ago, set in the next one
        }
        if (T.quiet) {
            bool live = false;
            uint4 e;
            for (uint32_t i = ct; i < nops && !live; i += consumers())
                live = kMode == kIds ? id_live(J, T, ops[i], L.pack, e) : mark_live(J, T, ops[i], L.pack, e);
            if (!consumers_sync_or(live)) {
                nseg = 0;
                if (kMode == kMarks && ct == 0) T.n_ops += nops;
            }
        }
        bool ran = false;
        for (uint32_t k = 0, b = 0; k < nseg; ++k) {
            const uint32_t e = seg[k];
            if (e == b) continue;
            if (b) consumers_sync();
            T.fresh = first + b;
            if (kMode == kIds || T.on) ran |= track_tile<kMax, kMode>(J, T, ops + b, e - b, rowbuf, L, group_mask);
            else whole_tile<kMax>(J, T, ops + b, e - b, rowbuf, L, group_mask);
            b = e;
        }
        if (kMode == kIds && ran && (ct & 31u) == 0) *T.stat(q) = 1;
        first += nops;
        __syncwarp();
        if ((ct & 31u) == 0) mbar_arrive(&ring.empty[q & ring.mask]);
    }
}

template <bool kMax>
__global__ void __launch_bounds__(kMaxThreads) stream_kernel(const __grid_constant__ JobList jl)
{
    uint8_t *const smem = dyn_smem;
    __shared__ uint32_t producer_abort;
    __shared__ int32_t gate;

    const Job &J = jl.job[find_job(jl, blockIdx.x)];
    if (J.rw) {
        const uint32_t cta = blockIdx.x - J.cta_begin;
        if (J.rw == 1) resident_slab<kMax, 1>(J, jl.smem_bytes, smem, cta);
        else resident_slab<kMax, 2>(J, jl.smem_bytes, smem, cta);
        return;
    }
    PackRing ring;  // kStages stages, then the barriers and the row buffer
    ring.stage = smem;
    ring.full = reinterpret_cast<uint64_t *>(smem + (size_t)kStages * kStageBytes);
    ring.empty = ring.full + kStages;
    ring.mask = kStages - 1;
    ring.shift = kStageShift;
    u64x2 *rowbuf = reinterpret_cast<u64x2 *>(smem + kSlabHead);
    const uint64_t w0 = J.w_begin + (uint64_t)(blockIdx.x - J.cta_begin) * J.sw;
    const uint32_t warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        gate = *(volatile int32_t *)J.status;  // an earlier error gates this job
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&ring.full[s], 1);
            mbar_init(&ring.empty[s], consumers() / 32u);
        }
        producer_abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (gate != 0) return;
    if (warp == 0) {
        produce_packs(J, ring, &producer_abort);
        return;
    }
    const uint32_t ct = threadIdx.x - 32;
    const Lane L = make_lane(J, ct, w0);
    const uint32_t cta = blockIdx.x - J.cta_begin;
    if (J.track == kIds) consume_tracked<kMax, kIds>(J, ring, &producer_abort, rowbuf, w0, cta, L, ct);
    else if (J.track == kMarks) consume_tracked<kMax, kMarks>(J, ring, &producer_abort, rowbuf, w0, cta, L, ct);
    else consume_plain<kMax>(J, ring, &producer_abort, rowbuf, L, ct);
}

// Self-test of the bounded waits: one thread waits on an mbarrier that nothing
// ever completes, through the same bounded wait the streaming kernel uses, and
// records TN_ETIMEOUT when the wait gives up.
__global__ void wait_selftest_kernel(int32_t *status)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    fence_mbar_init();
    if (!mbar_wait_bounded(&bar, 0)) record_status(status, TN_ETIMEOUT);
}

// S <- identity (full matrix) -- Algorithm 1, first line; one row per warp step
__global__ void init_identity_kernel(uint64_t *S, uint32_t n_rows, uint64_t ld, const int32_t *status)
{
    if (*(volatile const int32_t *)status != 0) return;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t r = blockIdx.x * (uint64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < n_rows; r += warps) {
        uint64_t *row = S + r * ld;
        const uint64_t diag = r >> 6;
        for (uint64_t w = 2 * lane; w < ld; w += 64) {
            u64x2 z{w == diag ? (1ull << (r & 63)) : 0ull, w + 1 == diag ? (1ull << (r & 63)) : 0ull};
            st_row16(row + w, z);
        }
    }
}

__global__ void zero_kernel(uint64_t *S, uint64_t total, const int32_t *status)
{
    if (*(volatile const int32_t *)status != 0) return;
    for (uint64_t i = 2 * (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x); i < total;
         i += 2 * (uint64_t)gridDim.x * blockDim.x)
        st_row16(S + i, u64x2{0ull, 0ull});
}

// column c of the matrix starts as the single source src[c]; ids >= n_rows
// are skipped and reported as TN_ERANGE
__global__ void init_sources_kernel(uint64_t *S, uint64_t ld, const uint32_t *src, uint32_t nsrc, uint32_t n_rows,
                                    int32_t *status)
{
    if (*(volatile const int32_t *)status != 0) return;
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nsrc; c += gridDim.x * blockDim.x) {
        const uint32_t x = src[c];
        if (x >= n_rows) {
            record_status(status, TN_ERANGE);
            continue;
        }
        atomicOr((unsigned long long *)(S + (uint64_t)x * ld + (c >> 6)), 1ull << (c & 63));
    }
}

__global__ void check_ids_kernel(const uint32_t *ids, uint32_t count, uint32_t n, int32_t *status)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        if (ids[i] >= n) record_status(status, TN_ERANGE);
}

// Validating check that every source id is a node id (< n).
static tn_status validate_sources(const uint32_t *src, uint32_t nsrc, uint32_t n, cudaStream_t st)
{
    int32_t *d = nullptr, h = 0;
    TN_CUDA_TRY(cudaMallocAsync((void **)&d, sizeof(int32_t), st));
    TN_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof(int32_t), st));
    tn_internal_count_launches(1);
    check_ids_kernel<<<(nsrc + 255) / 256 < 1024 ? (nsrc + 255) / 256 : 1024, 256, 0, st>>>(src, nsrc, n, d);
    TN_CUDA_TRY(cudaGetLastError());
    TN_CUDA_TRY(cudaMemcpyAsync(&h, d, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    TN_CUDA_TRY(cudaFreeAsync(d, st));
    TN_CUDA_TRY(cudaStreamSynchronize(st));
    return (tn_status)h;
}

// batch order check (streaming, Section 3.5): the batch must start after t_last
__global__ void order_gate_kernel(const int64_t *tb, const int64_t *t_last, int32_t *status)
{
    if (*t_last >= tb[0]) record_status(status, TN_EORDER);
}

__global__ void set_t_last_kernel(const int64_t *tb, int64_t *t_last, const int32_t *status)
{
    if (*(volatile const int32_t *)status == 0) *t_last = tb[1];
}

// Column slabs of one matrix of `ld` row words: ceil(ld / sw) CTAs of sw
// words, or -- with wave > 0 -- exactly max(wave, ceil(ld / sw)) CTAs of two
// widths that differ by one unit (16 words when sw is a multiple of 16 and the
// row holds that many units, else 2 words): the wider ones first.
struct SlabSplit {
    uint64_t w_begin;
    uint32_t sw, ctas;
};

static int split_slabs(uint64_t ld, uint32_t sw, uint32_t wave, SlabSplit out[2])
{
    const uint64_t plain = (ld + sw - 1) / sw;
    if (wave == 0 || ld == 0) {
        out[0] = SlabSplit{0, sw, (uint32_t)plain};
        return 1;
    }
    const uint64_t C = wave > plain ? wave : plain;
    const uint32_t unit = (sw % 16 == 0 && ld / 16 >= C) ? 16u : 2u;
    const uint64_t units = ld / unit;  // ld is a multiple of 16
    if (units <= C) {  // no more CTAs than units: one unit each
        out[0] = SlabSplit{0, unit, (uint32_t)units};
        return 1;
    }
    const uint64_t q = units / C, r = units % C;
    int k = 0;
    if (r) out[k++] = SlabSplit{0, (uint32_t)((q + 1) * unit), (uint32_t)r};
    out[k++] = SlabSplit{r * (q + 1) * unit, (uint32_t)(q * unit), (uint32_t)(C - r)};
    return k;
}

// Dynamic shared memory the streaming kernel can use on the current device
// (the opt-in maximum minus its static shared memory), cached per device.
static uint32_t stream_smem_limit()
{
    static std::mutex mu;
    static uint32_t cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (!cached[dev]) {
        int optin = 0;
        cudaFuncAttributes fa;
        if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, (const void *)stream_kernel<false>) != cudaSuccess)
            return 0;
        cached[dev] = (uint32_t)(optin - (int)fa.sharedSizeBytes);
    }
    return cached[dev];
}

int multiprocessors()
{
    static std::mutex mu;
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    std::lock_guard<std::mutex> lock(mu);
    if (!cached[dev] && cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        cached[dev] = 0;
    return cached[dev] > 0 ? cached[dev] : 1;
}

// dynamic shared memory of a CTA that leaves room for a second one on its SM
constexpr uint64_t kHalfSmSmem = 112 * 1024;

// Row slots of the copy rings of 12 consumer warps.
static uint32_t ring_slots(uint32_t words) { return 2u * kRing * (32u * kWarpsAlone / (words / 2)); }

bool tracked_slab(uint32_t words, uint64_t bytes)
{
    const uint32_t cpr = words / 2;
    return !(cpr & (cpr - 1)) && cpr <= 32 && bytes / (8 * words) >= ring_slots(words);
}

bool resident_fits(uint64_t rows, uint64_t temps, uint32_t words)
{
    if (words != 1 && words != 2) return false;
    return kResidentHead + resident_rows_bytes(rows, temps, words) + (uint64_t)kResidentMinStages * kStageBytes <=
           stream_smem_limit();
}

uint32_t resident_max_rows(uint32_t words)
{
    if (words != 1 && words != 2) return 0;
    const uint64_t lim = stream_smem_limit();
    const uint64_t fixed = kResidentHead + (uint64_t)kResidentMinStages * kStageBytes;
    if (lim <= fixed) return 0;
    return (uint32_t)(((lim - fixed) & ~127ull) / (8ull * words));
}

static int grid_for(uint64_t work)
{
    uint64_t g = (work + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 8192 ? 8192 : g));
}


// Slab widths of the plans of a launch that leave them open: the narrowest that
// keep the launch's CTAs within one wave (a CTA fills an SM, and every CTA walks
// its whole schedule), at most 64 words; the largest matrices, whose rows come
// from DRAM, are narrowed first.  Stream kernel: 5,000 directed columns (79 words),
// m = 3 10^6: 24.1 ms at 16 words (5 CTAs), 13.4 ms at 2 (40); ER n = 4 10^4, m = 5
// 10^6: 27.8 ms at 16 words (40), 21.2 ms at 8 (79), 34.7 ms at 4 (157, two waves);
// bursty n = 2 10^5, m = 5 10^6: 136 ms at 16 (196, two waves), 91 ms at 32 (98), 144
// ms at 64 (49); 8 proxies of 16,384 nodes with 65,536 columns of n = 10^6, m = 5
// 10^6: 46 ms at 32 and 16 words (128), 58 ms at 16 and 16 (192), 115 ms at 32 and 32.
static void open_slab_words(const tn_plan *const *plans, const uint32_t *ncols, const uint32_t *rw, uint32_t count,
                            uint32_t *sw)
{
    uint64_t ctas = 0, words[kMaxPlans];
    uint32_t open[kMaxPlans], n_open = 0;
    for (uint32_t i = 0; i < count; ++i) {
        words[i] = ((uint64_t)ncols[i] + 63) / 64;
        sw[i] = plans[i]->slab_words;
        if (!rw[i] && plans[i]->auto_slab && !plans[i]->local_windows) {
            sw[i] = 64;
            uint32_t at = n_open++;  // in falling order of matrix size
            for (; at > 0 && plans[open[at - 1]]->n * words[open[at - 1]] < plans[i]->n * words[i]; --at)
                open[at] = open[at - 1];
            open[at] = i;
        }
        const uint32_t w = rw[i] ? rw[i] : sw[i];
        ctas += (words[i] + w - 1) / w;
    }
    const uint64_t sms = (uint64_t)multiprocessors();
    for (bool more = n_open > 0; more;) {
        more = false;
        for (uint32_t k = 0; k < n_open; ++k) {
            const uint32_t i = open[k], half = sw[i] / 2;
            if (half < 2) continue;
            const uint64_t then = ctas - (words[i] + sw[i] - 1) / sw[i] + (words[i] + half - 1) / half;
            if (then > sms) continue;
            ctas = then;
            sw[i] = half;
            more = true;
        }
    }
}

// Waves of `ctas` resident CTAs of `rows` bytes of rows.  In a launch of such CTAs alone
// two share an SM if they fit beside the smallest ring (the launch then gives them one),
// at the same speed, since a level's latency bounds each.
static uint64_t resident_waves_of(uint64_t ctas, uint64_t rows, bool alone)
{
    const bool pair = alone && kResidentHead + rows + (uint64_t)kResidentMinStages * kStageBytes <= kHalfSmSmem;
    const uint64_t slots = (uint64_t)multiprocessors() * (pair ? 2 : 1);
    return (ctas + slots - 1) / slots;
}

// Form of every plan of a launch: words of a row per resident CTA, or 0 for column
// slabs.  Plans that leave the form open take the resident one if their rows fit
// and the batch touches enough of them to pay for loading and storing all rows (n =
// 20,000: 2,500 events of distinct nodes 0.15 ms, in tiles 0.05; 5,000 events 0.155,
// 0.125), while the launch's resident CTAs make at most kResidentWaves waves, or
// kResidentTieWaves of plans with large groups that share nodes; of one and two words
// the one with fewer waves, and where both have as many, one word (3 activity-driven
// networks of n = 8,000, two waves each, 0.68 and 0.91 ms), but two where that needs no
// second CTA on an SM (five ER networks of 1,500 nodes and one of 5,000 0.197 and 0.189).
static void choose_forms(const tn_plan *const *plans, const uint32_t *ncols, uint32_t count, uint32_t *rw)
{
    uint64_t ctas[3] = {0, 0, 0}, rows[3] = {0, 0, 0};
    bool two = true, alone = true;
    auto fits = [&](const tn_plan *p, uint32_t w) {
        return p->auto_form && 4 * p->ops >= p->n && resident_fits(p->n, p->temps, w);
    };
    for (uint32_t i = 0; i < count; ++i) {
        rw[i] = plans[i]->resident;
        if (rw[i]) continue;
        if (!fits(plans[i], 1)) {
            alone = false;
            continue;
        }
        two = two && fits(plans[i], 2);
        for (uint32_t w = 1; w <= 2; ++w) {
            ctas[w] += ((ncols[i] + 63ull) / 64 + w - 1) / w;
            const uint64_t bytes = resident_rows_bytes(plans[i]->n, plans[i]->temps, w);
            if (bytes > rows[w]) rows[w] = bytes;
        }
    }
    if (!ctas[1]) return;
    const uint64_t one = resident_waves_of(ctas[1], rows[1], alone), other = resident_waves_of(ctas[2], rows[2], alone);
    const uint32_t w = two && (other < one || (other == 1 && ctas[1] > (uint64_t)multiprocessors())) ? 2 : 1;
    const uint64_t waves = w == 2 ? other : one;
    for (uint32_t i = 0; i < count; ++i) {
        const bool ties = 16 * plans[i]->aux > plans[i]->ops;
        const uint64_t most = plans[i]->batch_plan ? (ties ? 3 : 7) : ties ? kResidentTieWaves : kResidentWaves;
        if (!rw[i] && fits(plans[i], 1) && waves <= most) rw[i] = w;
    }
}

uint32_t resident_form(const tn_plan *p, uint32_t ncols)
{
    uint32_t rw = 0;
    choose_forms(&p, &ncols, 1, &rw);
    return rw;
}

uint64_t resident_waves(const tn_plan *p, uint32_t ncols, uint32_t words)
{
    return resident_waves_of(((ncols + 63ull) / 64 + words - 1) / words, resident_rows_bytes(p->n, p->temps, words), true);
}

// Whether content ids of `bytes` may be allocated on `st`.  A call learns from the
// allocation itself that there is no room; a capture only records it, and the graph's
// launch would fail instead.  `held`: bytes of the launch's earlier ids; half of the
// free memory is left for what the caller allocates before the graph runs.
static bool ids_allowed(cudaStream_t st, uint64_t bytes, uint64_t held)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (capture == cudaStreamCaptureStatusNone) return true;
    size_t free_b = 0, total_b = 0;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t err = cudaMemGetInfo(&free_b, &total_b);
    cudaThreadExchangeStreamCaptureMode(&mode);
    return err == cudaSuccess && bytes + held <= free_b / 2;
}

tn_status apply_jobs(const tn_plan *const *plans, uint64_t *const *S, const uint32_t *ncols,
                     const uint32_t *const *src, int64_t *const *t_last, uint32_t count, uint32_t flags,
                     cudaStream_t st)
{
    // host-side argument checks
    for (uint32_t i = 0; i < count; ++i) {
        const tn_plan *p = plans[i];
        if (!p || !S[i] || ncols[i] == 0) return TN_EINVAL;
        // the identity initialisation needs one column per node
        if ((flags & TN_INIT_IDENTITY) && !src[i] && ncols[i] != p->n) return TN_EINVAL;
    }
    const size_t smem_base = kSlabHead;
    const size_t smem_limit = stream_smem_limit();
    if ((flags & kApplyMax) || !smem_limit)
        for (uint32_t i = 0; i < count; ++i)
            if (plans[i]->resident) return TN_EINVAL;
    uint64_t *tmps[kMaxPlans];
    uint32_t *idbuf[kMaxPlans];
    uint64_t ids_held = 0;
    for (uint32_t base = 0; base < count; base += kMaxPlans) {
        const uint32_t nj = count - base < (uint32_t)kMaxPlans ? count - base : (uint32_t)kMaxPlans;
        JobList jl;
        memset(&jl, 0, sizeof(jl));
        jl.count = 0;
        uint32_t ctas = 0;
        size_t smem = smem_base;
        uint32_t rws[kMaxPlans];
        choose_forms(plans + base, ncols + base, nj, rws);
        const tn_plan *used[kMaxPlans];  // the schedule applied
        for (uint32_t j = 0; j < nj; ++j) {
            const tn_plan *p = plans[base + j];
            used[j] = !rws[j] && p->batch_plan ? p->batch_plan : p;
        }
        uint32_t sws[kMaxPlans];
        open_slab_words(used, ncols + base, rws, nj, sws);
        for (uint32_t j = 0; j < nj; ++j) {
            const uint32_t i = base + j;
            const tn_plan *p = used[j];
            const uint64_t ld = tn_row_words(ncols[i]);
            tmps[j] = nullptr;
            idbuf[j] = nullptr;
            if (rws[j]) continue;  // second pass below
            if (t_last && t_last[i]) {
                tn_internal_count_launches(1);
                order_gate_kernel<<<1, 1, 0, st>>>(p->d_tbounds, t_last[i], p->d_status);
            }
            if (flags & TN_INIT_IDENTITY) {
                if (!src[i]) {
                    tn_internal_count_launches(1);
                    init_identity_kernel<<<grid_for(p->n * 32ull), 256, 0, st>>>(S[i], p->n, ld, p->d_status);
                } else {
                    tn_internal_count_launches(1);
                    zero_kernel<<<grid_for(p->n * ld / 2), 256, 0, st>>>(S[i], (uint64_t)p->n * ld, p->d_status);
                    tn_internal_count_launches(1);
                    init_sources_kernel<<<grid_for(ncols[i]), 256, 0, st>>>(S[i], ld, src[i], ncols[i], p->n,
                                                                            p->d_status);
                }
            }
            if (p->temps) TN_CUDA_TRY(cudaMallocAsync((void **)&tmps[j], p->temps * ld * sizeof(uint64_t), st));
            // Row buffer of the launch: records use all of the plan's; tiles only
            // the copy rings of 12 consumer warps.
            const bool open = p->auto_slab && !p->local_windows;
            const uint32_t sw = sws[j];
            // words that hold columns (the rest of the row is zero padding and stays so)
            const uint64_t wide = open ? (((uint64_t)ncols[i] + 63) / 64 + 1) & ~1ull : ld;
            uint32_t dcap = open ? p->buffer_bytes / (8 * sw) : p->dcap;
            const uint32_t ring_rows = ring_slots(sw);
            if (p->local_windows == 0 && dcap > ring_rows) dcap = ring_rows;
            size_t need = smem_base + (size_t)dcap * sw * 8;
            // Tracked rows: tile windows only (records do not keep track), row groups
            // that are whole parts of a warp, and copy rings that fit.  Wide slabs
            // by ids, if the ops pay for setting the ids up (4 bytes per row and
            // CTA against 512 to 2,048 bytes per op and CTA); others by marks, a
            // row or, where that does not fit, up to 4 rows per mark.
            const uint32_t nct = (uint32_t)((wide + sw - 1) / sw);
            const uint64_t rows = (uint64_t)p->n + p->temps;
            const bool zero = (flags & TN_INIT_IDENTITY) != 0;
            uint32_t track = kNoTrack, mark_words = 0, mark_shift = 0, *ids = nullptr;
            const uint32_t pitch = (nct + 7u) & ~7u;
            if (!p->local_windows && tracked_slab(sw, (uint64_t)dcap * sw * 8) && !p->wave_ctas &&
                need + kMarkBytes <= smem_limit) {
                track = kMarks;
                if (sw > kMarkWords && 16 * p->ops >= p->n && rows + p->ops < 0xFFFFFFF0ull &&
                    ids_allowed(st, rows * pitch * 4, ids_held)) {
                    if (cudaMallocAsync((void **)&ids, rows * pitch * 4, st) == cudaSuccess) {
                        track = kIds;
                        ids_held += rows * pitch * 4;
                        tn_internal_count_launches(1);
                        init_ids_kernel<<<grid_for(rows * pitch / 4), 256, 0, st>>>(ids, rows, pitch, sw,
                                                                                   zero, zero && !src[i]);
                        if (zero && src[i]) {
                            tn_internal_count_launches(1);
                            init_source_ids_kernel<<<grid_for(ncols[i]), 256, 0, st>>>(ids, pitch, sw,
                                                                                      src[i], ncols[i], p->n);
                        }
                    } else {
                        cudaGetLastError();  // no room for ids: marks
                        ids = nullptr;
                    }
                }
                if (track == kMarks) {
                    for (;; ++mark_shift) {
                        mark_words = (uint32_t)((((uint64_t)p->n >> mark_shift) + 1 + p->temps + 31) / 32);
                        if (need + kMarkBytes + 4ull * mark_words <= smem_limit || mark_shift == kMarkShift) break;
                    }
                    if (need + kMarkBytes + 4ull * mark_words > smem_limit || (mark_shift && !zero)) mark_words = 0;
                }
                need += (track == kIds ? kIdBytes : kMarkBytes) + 4ull * mark_words;
            }
            idbuf[j] = ids;
            if (need > smem) smem = need;
            SlabSplit sp[2];
            const int parts = split_slabs(wide, sw, p->wave_ctas, sp);
            for (int k = 0; k < parts; ++k) {
                Job &J = jl.job[jl.count++];
                J.blob = p->d_blob;
                J.win = p->d_win;
                J.aux = p->d_aux;
                J.nwin = (uint32_t)p->windows;
                J.S = S[i];
                J.ld = ld;
                J.tmp = tmps[j];
                J.status = p->d_status;
                J.w_begin = sp[k].w_begin;
                J.sw = sp[k].sw;
                J.cpr = sp[k].sw / 2;
                J.dcap = dcap;
                J.track = track;
                J.ids = ids;
                J.pitch = pitch;
                J.mark_words = mark_words;
                J.mark_shift = mark_shift;
                J.mark_init = !zero ? 0u : src[i] ? 2u : 1u;
                J.src = src[i];
                J.ncols = ncols[i];
                J.rows = p->n;
                J.label = p->d_label;
                J.cta_begin = ctas;
                ctas += sp[k].ctas;
            }
        }
        // resident-slab jobs after the column-slab ones: their CTAs are short,
        // and the long column-slab CTAs are dispatched first.  Their schedule
        // ring has 8 stages (one CTA of 12 consumer warps per SM) while the
        // resident CTAs fit one wave; beyond that 4, or 2 if only that lets two
        // CTAs share an SM
        uint64_t res_ctas = 0, rb_max = 0;
        for (uint32_t j = 0; j < nj; ++j) {
            const tn_plan *p = plans[base + j];
            if (!rws[j]) continue;
            res_ctas += ((ncols[base + j] + 63) / 64 + rws[j] - 1) / rws[j];
            const uint64_t rb = kResidentHead + resident_rows_bytes(p->n, p->temps, rws[j]);
            if (rb > rb_max) rb_max = rb;
        }
        uint64_t stages = kResidentMaxStages;
        if (res_ctas > (uint64_t)multiprocessors()) {
            stages = 4;
            if (smem <= kHalfSmSmem && rb_max + 4ull * kStageBytes > kHalfSmSmem &&
                rb_max + 2ull * kStageBytes <= kHalfSmSmem)
                stages = 2;
        }
        for (uint32_t j = 0; j < nj; ++j) {
            const uint32_t i = base + j;
            const tn_plan *p = plans[i];
            if (!rws[j]) continue;
            const uint64_t ld = tn_row_words(ncols[i]);
            if (t_last && t_last[i]) {
                tn_internal_count_launches(1);
                order_gate_kernel<<<1, 1, 0, st>>>(p->d_tbounds, t_last[i], p->d_status);
            }
            // a single matrix's CTAs start from the identity by themselves (one launch
            // less on the path of a small network, and S is not read)
            const bool own_identity = (flags & TN_INIT_IDENTITY) && !src[i] && count == 1;
            if (flags & TN_INIT_IDENTITY) {
                if (!src[i]) {
                    if (!own_identity) {
                        tn_internal_count_launches(1);
                        init_identity_kernel<<<grid_for(p->n * 32ull), 256, 0, st>>>(S[i], p->n, ld, p->d_status);
                    }
                } else {
                    tn_internal_count_launches(1);
                    zero_kernel<<<grid_for(p->n * ld / 2), 256, 0, st>>>(S[i], (uint64_t)p->n * ld, p->d_status);
                    tn_internal_count_launches(1);
                    init_sources_kernel<<<grid_for(ncols[i]), 256, 0, st>>>(S[i], ld, src[i], ncols[i], p->n,
                                                                            p->d_status);
                }
            }
            // words holding columns (the rest of the row is zero padding and stays so)
            const uint64_t used = (ncols[i] + 63) / 64;
            const uint32_t rw = rws[j];
            const uint64_t rb = kResidentHead + resident_rows_bytes(p->n, p->temps, rw);
            uint64_t need = rb + stages * kStageBytes;
            if (need > smem_limit) need = smem_limit;
            if (rb + (uint64_t)kResidentMinStages * kStageBytes > smem_limit) return TN_EINVAL;
            if (need > smem) smem = need;
            Job &J = jl.job[jl.count++];
            J.blob = p->d_blob;
            J.win = p->d_win;
            J.aux = p->d_aux;
            J.nwin = (uint32_t)p->windows;
            J.S = S[i];
            J.ld = ld;
            J.tmp = nullptr;
            J.status = p->d_status;
            J.w_begin = 0;
            J.sw = rw;
            J.cpr = 0;
            J.dcap = 0;
            J.rw = rw;
            J.res_threads = p->ops > kResidentConsumers * p->levels ? 32u * kWarpsAlone : kResidentConsumers;
            J.identity = own_identity;
            J.label = p->d_label;
            J.ncols = ncols[i];
            J.rows = p->n;
            J.ntemp = (uint32_t)p->temps;
            J.cta_begin = ctas;
            ctas += (uint32_t)((used + rw - 1) / rw);
        }
        jl.smem_bytes = (uint32_t)smem;
        TN_CUDA_TRY(cudaGetLastError());
        if (ctas) {
            tn_internal_count_launches(1);
            const void *kernel = (flags & kApplyMax) ? (const void *)stream_kernel<true> : (const void *)stream_kernel<false>;
            TN_CUDA_TRY(tn_internal_allow_max_dyn_smem(kernel));
            // 4 consumer warps if two CTAs of that size fit on an SM, else 12
            int pair = 0;
            const int shared_threads = 32 * kWarpsShared + 32;
            TN_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pair, kernel, shared_threads, smem));
            const int threads = pair >= 2 ? shared_threads : kMaxThreads;
            if (flags & kApplyMax)
                stream_kernel<true><<<ctas, threads, smem, st>>>(jl);
            else
                stream_kernel<false><<<ctas, threads, smem, st>>>(jl);
        }
        TN_CUDA_TRY(cudaGetLastError());
        for (uint32_t j = 0; j < nj; ++j) {
            const uint32_t i = base + j;
            if (t_last && t_last[i]) {
                tn_internal_count_launches(1);
                set_t_last_kernel<<<1, 1, 0, st>>>(plans[i]->d_tbounds, t_last[i], plans[i]->d_status);
            }
            if (tmps[j]) TN_CUDA_TRY(cudaFreeAsync(tmps[j], st));
            if (idbuf[j]) TN_CUDA_TRY(cudaFreeAsync(idbuf[j], st));
        }
        TN_CUDA_TRY(cudaGetLastError());
    }
    return TN_OK;
}

}  // namespace tn

using namespace tn;

extern "C" tn_status tn_plan_apply(const tn_plan *plan, uint64_t *S, uint32_t ncols, const uint32_t *src,
                                   int64_t *t_last, uint32_t flags, void *stream)
{
    if (!plan || !S || (flags & ~TN_INIT_IDENTITY)) return TN_EINVAL;
    return apply_jobs(&plan, &S, &ncols, &src, &t_last, 1, flags, (cudaStream_t)stream);
}

extern "C" tn_status tn_plan_apply_batch(const tn_plan *const *plans, uint64_t *const *S, const uint32_t *ncols,
                                         const uint32_t *const *src, uint32_t count, uint32_t flags, void *stream)
{
    if (!plans || !S || !ncols || count == 0 || (flags & ~TN_INIT_IDENTITY)) return TN_EINVAL;
    if (src) return apply_jobs(plans, S, ncols, src, nullptr, count, flags, (cudaStream_t)stream);
    const uint32_t **none = (const uint32_t **)calloc(count, sizeof(uint32_t *));
    if (!none) return TN_ENOMEM;
    tn_status rc = apply_jobs(plans, S, ncols, none, nullptr, count, flags, (cudaStream_t)stream);
    free(none);
    return rc;
}

// reversed sequence (Section 3.4): event m-1-e becomes event e and its time is
// complemented (~t = -t - 1 keeps equal times equal and the order non-decreasing)
// Directed events are also turned around (u -> v becomes v -> u), so that in
// both modes row i ends as the out-component of i.
__global__ void reverse_events_kernel(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m,
                                      bool turn, uint32_t *ru, uint32_t *rv, int64_t *rt)
{
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < m; e += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = m - 1 - e;
        ru[e] = turn ? v[s] : u[s];
        rv[e] = turn ? u[s] : v[s];
        rt[e] = ~t[s];
    }
}

static tn_status one_shot(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                          const uint32_t *src, uint32_t ncols, uint64_t *S, int64_t *t_last, uint32_t flags,
                          void *stream);

tn_status tn::reversed_events(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, bool turn,
                              uint32_t **ru, uint32_t **rv, int64_t **rt, cudaStream_t st)
{
    *ru = nullptr;
    *rv = nullptr;
    *rt = nullptr;
    TN_CUDA_TRY(cudaMallocAsync((void **)ru, m * 4, st));
    TN_CUDA_TRY(cudaMallocAsync((void **)rv, m * 4, st));
    TN_CUDA_TRY(cudaMallocAsync((void **)rt, m * 8, st));
    tn_internal_count_launches(1);
    reverse_events_kernel<<<grid_for(m), 256, 0, st>>>(u, v, t, m, turn, *ru, *rv, *rt);
    TN_CUDA_TRY(cudaGetLastError());
    return TN_OK;
}

// TN_REVERSE: the same path over the reversed sequence, from the identity
static tn_status one_shot_reversed(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                                   const uint32_t *src, uint32_t ncols, uint64_t *S, int64_t *t_last,
                                   uint32_t flags, void *stream)
{
    if (t_last || !(flags & TN_INIT_IDENTITY)) return TN_EINVAL;  // not a streaming mode
    if (m == 0) return one_shot(u, v, t, m, n, src, ncols, S, nullptr, flags & ~TN_REVERSE, stream);
    if (!u || !v || !t || m >= (1ull << 30)) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t *ru = nullptr, *rv = nullptr;
    int64_t *rt = nullptr;
    const tn_status rr = reversed_events(u, v, t, m, (flags & TN_DIRECTED) != 0, &ru, &rv, &rt, st);
    if (rr != TN_OK) return rr;
    const tn_status rc = one_shot(ru, rv, rt, m, n, src, ncols, S, nullptr, flags & ~TN_REVERSE, stream);
    cudaFreeAsync(ru, st);
    cudaFreeAsync(rv, st);
    cudaFreeAsync(rt, st);
    return rc;
}

static tn_status one_shot(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                          const uint32_t *src, uint32_t ncols, uint64_t *S, int64_t *t_last, uint32_t flags,
                          void *stream)
{
    if (!S || n == 0 || n >= (1u << 30) || (flags & ~(TN_INIT_IDENTITY | TN_REVERSE | TN_DIRECTED))) return TN_EINVAL;
    if (flags & TN_REVERSE) return one_shot_reversed(u, v, t, m, n, src, ncols, S, t_last, flags, stream);
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t ld = tn_row_words(ncols);
    if (src && (flags & TN_INIT_IDENTITY)) {
        const tn_status rc = validate_sources(src, ncols, n, st);
        if (rc != TN_OK) return rc;
    }
    if (m == 0) {
        if (flags & TN_INIT_IDENTITY) {
            int32_t *zero = nullptr;
            TN_CUDA_TRY(cudaMallocAsync((void **)&zero, sizeof(int32_t), st));
            TN_CUDA_TRY(cudaMemsetAsync(zero, 0, sizeof(int32_t), st));
            if (!src) {
                tn_internal_count_launches(1);
                init_identity_kernel<<<grid_for(n * 32ull), 256, 0, st>>>(S, n, ld, zero);
            } else {
                tn_internal_count_launches(1);
                zero_kernel<<<grid_for(n * ld / 2), 256, 0, st>>>(S, (uint64_t)n * ld, zero);
                tn_internal_count_launches(1);
                init_sources_kernel<<<grid_for(ncols), 256, 0, st>>>(S, ld, src, ncols, n, zero);
            }
            TN_CUDA_TRY(cudaFreeAsync(zero, st));
            TN_CUDA_TRY(cudaGetLastError());
        }
        return TN_OK;
    }
    tn_plan_options opt;
    memset(&opt, 0, sizeof(opt));
    opt.directed = (flags & TN_DIRECTED) ? 1u : 0u;
    tn_plan *plan = nullptr;
    tn_status rc = plan_create_for(u, v, t, m, n, t_last, &opt, PlanUse{ncols, false}, stream, &plan);
    if (rc != TN_OK) return rc;
    flags &= ~TN_DIRECTED;
    rc = apply_jobs((const tn_plan *const *)&plan, &S, &ncols, &src, &t_last, 1, flags, st);
    tn_plan_destroy(plan, stream);
    return rc;
}

extern "C" tn_status tn_component_matrix(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m,
                                         uint32_t n, uint64_t *S, int64_t *t_last, uint32_t flags, void *stream)
{
    return one_shot(u, v, t, m, n, nullptr, n, S, t_last, flags, stream);
}

extern "C" tn_status tn_component_columns(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m,
                                          uint32_t n, const uint32_t *src, uint32_t nsrc, uint64_t *S,
                                          int64_t *t_last, uint32_t flags, void *stream)
{
    if (!src || nsrc == 0) return TN_EINVAL;
    return one_shot(u, v, t, m, n, src, nsrc, S, t_last, flags, stream);
}

extern "C" tn_status tn_init_matrix(uint64_t *S, uint32_t n_rows, uint32_t ncols, const uint32_t *src, void *stream)
{
    if (!S || n_rows == 0 || ncols == 0 || n_rows >= (1u << 30)) return TN_EINVAL;
    if (!src && ncols != n_rows) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (src) {
        const tn_status rc = validate_sources(src, ncols, n_rows, st);
        if (rc != TN_OK) return rc;
    }
    const uint64_t ld = tn_row_words(ncols);
    int32_t *zero = nullptr;
    TN_CUDA_TRY(cudaMallocAsync((void **)&zero, sizeof(int32_t), st));
    TN_CUDA_TRY(cudaMemsetAsync(zero, 0, sizeof(int32_t), st));
    if (!src) {
        tn_internal_count_launches(1);
        init_identity_kernel<<<grid_for(n_rows * 32ull), 256, 0, st>>>(S, n_rows, ld, zero);
    } else {
        tn_internal_count_launches(2);
        zero_kernel<<<grid_for(n_rows * ld / 2), 256, 0, st>>>(S, (uint64_t)n_rows * ld, zero);
        init_sources_kernel<<<grid_for(ncols), 256, 0, st>>>(S, ld, src, ncols, n_rows, zero);
    }
    TN_CUDA_TRY(cudaGetLastError());
    TN_CUDA_TRY(cudaFreeAsync(zero, st));
    return TN_OK;
}

extern "C" tn_status tn_selftest_wait_timeout(void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    int32_t *d = nullptr, h = 0;
    TN_CUDA_TRY(cudaMallocAsync((void **)&d, sizeof(int32_t), st));
    TN_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof(int32_t), st));
    tn_internal_count_launches(1);
    wait_selftest_kernel<<<1, 32, 0, st>>>(d);
    TN_CUDA_TRY(cudaGetLastError());
    TN_CUDA_TRY(cudaMemcpyAsync(&h, d, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    TN_CUDA_TRY(cudaFreeAsync(d, st));
    TN_CUDA_TRY(cudaStreamSynchronize(st));
    return (tn_status)h;
}

extern "C" uint32_t tn_resident_max_rows(uint32_t resident_words) { return tn::resident_max_rows(resident_words); }
