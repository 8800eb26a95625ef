// Internal helpers shared by the libtn translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tn.h"

#define TN_CUDA_TRY(expr)                                   \
    do {                                                    \
        cudaError_t err_ = (expr);                          \
        if (err_ != cudaSuccess) {                          \
            tn_internal_set_cuda_error(err_);               \
            return err_ == cudaErrorMemoryAllocation ? TN_ENOMEM : TN_ECUDA; \
        }                                                   \
    } while (0)

void tn_internal_set_cuda_error(cudaError_t err);
// Keeps memory freed to the current device's stream-ordered pool cached for
// reuse instead of returning it to the driver at every synchronisation.
void tn_internal_keep_pool(void);
// Raises a kernel's dynamic shared-memory limit to everything the device allows
// beside the kernel's static shared memory.  Always the same value for a given
// kernel, so concurrent callers (threads, streams) cannot undo each other.
cudaError_t tn_internal_allow_max_dyn_smem(const void *kernel);
// Adds `count` to the process-wide kernel launch counter (tn_kernel_launches).
void tn_internal_count_launches(uint64_t count);
// Waits on the host for the work enqueued on `stream` so far, sleeping rather
// than spinning (an event with blocking synchronisation, one per host thread
// and device): many threads waiting at once (the serving engine's workers)
// then leave the host cores to the threads that have work.
cudaError_t tn_internal_stream_wait(cudaStream_t stream);

namespace tn {
// A few counters from a kernel's last CTA to the host thread that waits for them, in
// pinned host memory of that thread: the words, then the call's number in `seq`.  A
// copy back and an event cost two driver calls (which threads of one process take in
// turn) and the wake-up of a blocked thread instead.
constexpr uint32_t kMailWords = 24;
struct Mail {
    uint64_t word[kMailWords];
    uint32_t seq, pad;
};
// This thread's mailbox and a new number for a launch on `stream`; nullptr if there is
// none (no pinned memory, or the stream is being captured: copy back and wait then).
Mail *mail_open(cudaStream_t stream, uint32_t *seq);
// Waits until the kernel has written `seq`: polls for a while, then blocks until the
// stream's work is done.  Every opened mailbox is waited for before its thread goes on.
cudaError_t mail_wait(const Mail *mail, uint32_t seq, cudaStream_t stream);

// By one thread of the last CTA, behind a fence for what it has read.
template <typename T>
__device__ inline void mail_send(Mail *mail, uint32_t seq, const T *from)
{
    static_assert(sizeof(T) % 8 == 0 && sizeof(T) / 8 <= kMailWords, "mailbox too small");
    const volatile uint64_t *w = reinterpret_cast<const volatile uint64_t *>(from);
    uint64_t x[sizeof(T) / 8];
#pragma unroll
    for (uint32_t k = 0; k < sizeof(T) / 8; ++k) x[k] = w[k];
#pragma unroll
    for (uint32_t k = 0; k < sizeof(T) / 8; ++k) *(volatile uint64_t *)&mail->word[k] = x[k];
    __threadfence_system();
    *(volatile uint32_t *)&mail->seq = seq;
}
}  // namespace tn

namespace tn {

// Bounded device-side waits: a wait that has not completed after this many
// polls (each poll suspends for up to ~1 us) records TN_ETIMEOUT and gives up.
constexpr uint32_t kWaitPolls = 1u << 22;

// Op encoding of the row-update schedule (see tn_plan.cu).
//   a: bits 31..30 = kind, bits 29..0 = destination node / temp id
//   b: EVENT / ONEWAY / COPY: source node id;  PULL: its source list: count c, then
// c source references (bit 31 set = temp slot, else node id), at word b of the
// pack, or, from kOutsideList on, at word b - kOutsideList of the plan's list
// buffer (the lists of one level did not fit a pack).
enum OpKind : uint32_t { kEvent = 0u, kOneway = 1u, kCopy = 2u, kPull = 3u };
constexpr uint32_t kKindShift = 30;
constexpr uint32_t kIdMask = (1u << 30) - 1u;
constexpr uint32_t kTempRef = 1u << 31;
constexpr uint32_t kNoRef = 0xFFFFFFFFu;  // empty slot in a batch of source references
constexpr uint32_t kOutsideList = 8192;

__host__ __device__ inline uint32_t op_a(uint32_t kind, uint32_t id) { return (kind << kKindShift) | id; }

// Packs of the streaming kernel: what one stage of its shared-memory ring
// holds, copied whole.  A window of the schedule is a run of consecutive packs
// (16-byte aligned, sizes in 8-byte units).
//   tile pack: uint32 ops, uint32 segments | flags << 16, 8 spare bytes,
//     uint16 end[64] (op offsets where its segments end), then the ops as uint2
//     (node ids), then the source lists of its PULLs.  A segment is a level, or a part of one
//     when the level does not fit a pack; ops of one segment never conflict.
//   record pack (kPackLocal; a window whose rows fit the kernel's shared-memory
//     row buffer): 16 bytes like the above, then uint32 words D, T, nlev, nops |
//     rows[D] (node ids) | lvl[nlev + 1] (op offsets) | ops[nops] | aux[...] |
//     zero padding to 16 B.
//     Rows are named by local slots: 0..D-1 the window's rows, D..D+T-1 saved
//     copies.  op = kind << 30 | la << 29 | lb << 28 | a << 14 | b  (PULL: b =
//     aux offset).  la / lb mark the op that writes row a / b for the last time
//     in the window: its result is also stored to the matrix right away, so the
//     write-back runs during the levels instead of after them, and rows that
//     are only read are never written back.
constexpr uint32_t kStageBytes = 16384;
constexpr uint32_t kPackSegs = 64;
constexpr uint32_t kPackHead = 2 + kPackSegs / 4;          // units
constexpr uint32_t kPackOps = kStageBytes / 8 - kPackHead;  // 2,030
constexpr uint32_t kRecordWords = kStageBytes / 4 - 4;
constexpr uint32_t kPackLocal = 1u;   // a record
constexpr uint32_t kPackWindow = 2u;  // first pack of its window
constexpr uint32_t kPackEnd = 4u;     // no pack: the schedule ends here
constexpr uint32_t kPackTies = 8u;    // holds PULLs or COPYs
// One window of the schedule: `npacks` packs from unit `off` on; their sizes
// are pack[] while there are at most kDescPacks, else a uint32 table `tab`
// units behind `off`.
constexpr uint32_t kDescPacks = 4;
struct __align__(16) WinDesc {
    uint64_t off;
    uint32_t npacks, tab;
    uint32_t pack[kDescPacks];
};
static_assert(sizeof(WinDesc) == 32, "two 16-byte loads");
struct PlanHead;

constexpr uint32_t kLocalBits = 14;
constexpr uint32_t kLocalMask = 0x3FFFu;
constexpr uint32_t kLocalSlotLimit = 0x3FFFu;  // above the 10,240 slots a 160 KB row buffer can hold
// Widest column slab of one CTA: 128 words (1 KB row segments).
constexpr uint32_t kMaxSlabWords = 128;
constexpr uint32_t kLastA = 1u << 29;
constexpr uint32_t kLastB = 1u << 28;

__host__ __device__ inline uint32_t local_op(uint32_t kind, uint32_t a, uint32_t b)
{
    return (kind << kKindShift) | (a << kLocalBits) | b;
}

__device__ inline void record_status(int32_t *status, int32_t code)
{
    if (status) atomicCAS(status, 0, code);
}

// ---------------------------------------------------------------------------
// mbarrier and bulk-copy (TMA, non-tensor) PTX wrappers
// ---------------------------------------------------------------------------
__device__ inline uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ inline void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ inline void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ inline void mbar_arrive(uint64_t *bar)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
                 : "memory");
}

__device__ inline void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                     smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// One poll: true once the phase with the given parity has completed.
__device__ inline bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity), "r"(1000u)
        : "memory");
    return done != 0;
}

// Bounded wait; returns false on timeout.
__device__ inline bool mbar_wait_bounded(uint64_t *bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kWaitPolls; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// Bulk global -> shared copy of `bytes` (multiple of 16, both addresses
// 16-byte aligned), completion signalled on `bar` as transaction bytes.
__device__ inline void bulk_g2s(void *smem_dst, const void *gmem_src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(smem_dst)),
        "l"(gmem_src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// ---------------------------------------------------------------------------
// 128-bit row-segment access (L2-cached, not allocated in L1)
// ---------------------------------------------------------------------------
struct u64x2 {
    uint64_t x, y;
};

__device__ inline u64x2 ld_row16(const uint64_t *p)
{
    u64x2 r;
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(r.x), "=l"(r.y) : "l"(p) : "memory");
    return r;
}

__device__ inline void st_row16(uint64_t *p, u64x2 r)
{
    asm volatile("st.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(r.x), "l"(r.y) : "memory");
}

__device__ inline u64x2 or16(u64x2 a, u64x2 b) { return u64x2{a.x | b.x, a.y | b.y}; }

// Combine of two row chunks: OR of bitsets (component matrix), or byte-wise
// maximum (HyperLogLog registers, one byte each).
__device__ inline uint64_t max8x8(uint64_t a, uint64_t b)
{
    const uint32_t lo = __vmaxu4((uint32_t)a, (uint32_t)b);
    const uint32_t hi = __vmaxu4((uint32_t)(a >> 32), (uint32_t)(b >> 32));
    return ((uint64_t)hi << 32) | lo;
}

template <bool kMax>
__device__ inline u64x2 combine16(u64x2 a, u64x2 b)
{
    if (kMax) return u64x2{max8x8(a.x, b.x), max8x8(a.y, b.y)};
    return or16(a, b);
}

// Full adder of bit columns: (c, a, b) -> sum in c, carry returned.
__device__ inline uint32_t full_add(uint32_t &c, uint32_t a, uint32_t b)
{
    const uint32_t carry = (c & a) | (b & (c | a));
    c = c ^ a ^ b;
    return carry;
}

// ---------------------------------------------------------------------------
// Block-wide exclusive scan of an array (generic pointer: shared or global).
// All threads of the block must call it; returns the total.  `warp_sums` must
// hold 32 entries of shared memory.
// ---------------------------------------------------------------------------
__device__ inline uint32_t warp_incl_scan(uint32_t x)
{
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= (uint32_t)d) x += y;
    }
    return x;
}

__device__ inline uint32_t block_excl_scan_value(uint32_t x, uint32_t *warp_sums, uint32_t *total)
{
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t nwarps = (blockDim.x + 31u) >> 5;
    uint32_t incl = warp_incl_scan(x);
    if (lane == 31u) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t s = lane < nwarps ? warp_sums[lane] : 0u;
        uint32_t si = warp_incl_scan(s);
        if (lane < nwarps) warp_sums[lane] = si - s;
        if (lane == nwarps - 1u) *total = si;
    }
    __syncthreads();
    uint32_t r = warp_sums[warp] + incl - x;
    __syncthreads();
    return r;
}

template <typename I>
__device__ inline uint32_t block_excl_scan_array(I *a, uint32_t len, uint32_t *warp_sums, uint32_t *total)
{
    const uint32_t per = (len + blockDim.x - 1u) / blockDim.x;
    const uint32_t b = threadIdx.x * per;
    const uint32_t e = min(len, b + per);
    uint32_t sum = 0;
    for (uint32_t i = b; i < e; ++i) sum += a[i];
    uint32_t off = block_excl_scan_value(sum, warp_sums, total);
    for (uint32_t i = b; i < e; ++i) {
        uint32_t x = a[i];
        a[i] = (I)off;
        off += x;
    }
    __syncthreads();
    return *total;
}

}  // namespace tn

// Plan object (opaque in the ABI).
struct tn_plan {
    int device;
    uint64_t m;
    uint32_t n;
    uint64_t windows, levels, ops, aux, temps, big_windows, local_windows, items, blob8;
    int64_t t_first, t_last;
    uint32_t slab_words;  // 64-bit words of every row owned by one CTA (the widest, with wave_ctas)
    uint32_t auto_slab;   // slab_words was left open: chosen when the plan is applied, if it has no records
    uint32_t auto_form;   // the form (resident or column slabs) was left open: chosen when the plan is applied
    tn_plan *batch_plan;  // owned: the schedule as records, for launches where this plan is in column slabs (or NULL)
    uint32_t wave_ctas;   // 0, or the number of CTAs one matrix is spread over
    uint32_t dcap;        // row slots of the kernel's shared-memory row buffer
    uint32_t buffer_bytes;  // largest row buffer of a width chosen when the plan is applied (smem_rows was given: its bytes)
    uint32_t resident;    // 0, or 64-bit words of every row one CTA keeps in shared memory
    uint2 *d_blob;        // packs (8-byte units)
    tn::WinDesc *d_win;   // [windows]    their windows in time order
    uint32_t *d_aux;      // source lists outside the packs
    void *d_mem;          // owned: all of the below but the labels
    uint32_t *d_label;    // [n] component of every node, a node id (NULL: not computed)
    tn::PlanHead *d_head; // counters, time bounds, status word
    int64_t *d_tbounds;   // [2]          t_first, t_last (in d_head)
    int32_t *d_status;    // first asynchronous error (in d_head, or the owner's: tn::plan_use_status)
};

namespace tn {
// SMs of the current device (cached per device).
int multiprocessors();
// Resident-slab form (tn_plan_options.resident_words): whether a network of
// `rows` rows and `temps` saved-row slots fits one CTA's shared memory at
// `words` 64-bit words per row, beside the smallest schedule ring; and the
// largest row count that fits with no saved rows (0 for an unsupported width).
bool resident_fits(uint64_t rows, uint64_t temps, uint32_t words);
uint32_t resident_max_rows(uint32_t words);
// Words of a row per resident CTA that an open plan takes when it alone is applied to
// `ncols` columns; 0: column slabs.
uint32_t resident_form(const tn_plan *p, uint32_t ncols);
uint64_t resident_waves(const tn_plan *p, uint32_t ncols, uint32_t words);
// Whether the rows of a slab of `words` words can be tracked beside a row buffer of
// `bytes`: row groups that are whole parts of a warp, and copy rings that fit.
bool tracked_slab(uint32_t words, uint64_t bytes);
// Internal apply flag: combine rows by byte-wise maximum (HyperLogLog
// registers) instead of OR; no initialisation.
constexpr uint32_t kApplyMax = 1u << 16;
// Launch the column-slab streaming kernel for a list of (plan, matrix) jobs.
tn_status apply_jobs(const tn_plan *const *plans, uint64_t *const *S, const uint32_t *ncols,
                     const uint32_t *const *src, int64_t *const *t_last, uint32_t count, uint32_t flags,
                     cudaStream_t stream);
// Online state in two-stream mode (used by the serving engine): its matrix
// updates (and node growth) run on `apply_stream`, while the stream given to
// each tn_online_push carries the copies and the scheduling, so scheduling a
// batch never waits for the update of the one before.  Must be called right
// after tn_online_create, with the matrix's initialisation complete on both
// streams.  Up to kOnlineFlight applied batches stay in flight; a device error
// of one is returned once that batch has finished, and always by
// tn_online_status.
constexpr uint32_t kOnlineFlight = 8;
tn_status online_use_apply_stream(tn_online *online, cudaStream_t apply_stream);
// Two-stream mode: the device status word every batch's plan records errors
// in (0 = none), for a caller that copies it out behind the updates.
const int32_t *online_status_word(const tn_online *online);
// tn_plan_create for a plan whose use is known: applied alone, to `ncols` columns (0: not
// known), with the byte-wise maximum (kApplyMax).
struct PlanUse {
    uint32_t ncols;
    bool max;
};
tn_status plan_create_for(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                          const int64_t *t_after, const tn_plan_options *opt, const PlanUse &use, void *stream,
                          tn_plan **plan_out);
// tn_plan_create without its last host wait: the plan's device buffers are
// written by work enqueued on `stream`, so a use on another stream must first
// wait for an event recorded on `stream` after this call.
tn_status plan_create_ordered(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, uint32_t n,
                              const tn_plan_options *opt, cudaStream_t stream, tn_plan **plan_out);
// Points a plan's status word at `status` (owned by the caller, e.g. one word
// for every batch of an online state, so an error gates the later batches and
// is read once); the plan's own word is released on `stream`.
tn_status plan_use_status(tn_plan *plan, int32_t *status, cudaStream_t stream);
// Reversed copy of an event sequence (Section 3.4): event m-1-e becomes event e,
// t -> ~t; with `turn` the endpoints are swapped (directed events).  The three
// arrays come from the stream-ordered allocator; the caller frees them.
tn_status reversed_events(const uint32_t *u, const uint32_t *v, const int64_t *t, uint64_t m, bool turn,
                          uint32_t **ru, uint32_t **rv, int64_t **rt, cudaStream_t st);
}  // namespace tn
