// Error of hashed estimates against exact out-component sizes (Section 4.4:
// the estimated and exact size distributions are compared with the
// Earth-Mover distance; absolute and relative errors are reported beside it).
//
// One pass over the pairs accumulates the absolute and relative errors and two
// histograms of the values.  For integer samples of equal size the
// Wasserstein-1 distance is the area between the two empirical CDFs, i.e.
// sum over integers x of |#{est <= x} - #{exact <= x}| / count; a scan
// of the histogram difference gives that sum exactly, with no sort.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "tn_internal.cuh"

namespace tn {

struct ErrAccum {
    unsigned long long sum_abs, max_abs, w1_num, max_rel_bits;
    double rel_sum;
    int32_t bad;
    int32_t pad;
};

constexpr int kErrThreads = 256;

__global__ void __launch_bounds__(kErrThreads)
    error_pairs_kernel(const uint32_t *est, const uint32_t *exact, uint32_t count, uint32_t max_value,
                       uint32_t *hist_est, uint32_t *hist_exact, ErrAccum *acc)
{
    unsigned long long s = 0, mx = 0, mr = 0;
    double rs = 0.0;
    bool bad = false;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const uint32_t a = est[i], b = exact[i];
        if (a > max_value || b > max_value || b == 0) {
            bad = true;
            continue;
        }
        const unsigned long long d = a > b ? a - b : b - a;
        s += d;
        mx = d > mx ? d : mx;
        const double r = (double)d / (double)b;
        rs += r;
        // non-negative doubles order like their bit patterns
        const unsigned long long rb = (unsigned long long)__double_as_longlong(r);
        mr = rb > mr ? rb : mr;
        atomicAdd(hist_est + a, 1u);
        atomicAdd(hist_exact + b, 1u);
    }
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = x > mx ? x : mx;
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, mr, o);
        mr = y > mr ? y : mr;
        rs += __shfl_xor_sync(0xffffffffu, rs, o);
    }
    bad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31u) == 0) {
        if (s) atomicAdd(&acc->sum_abs, s);
        if (mx) atomicMax(&acc->max_abs, mx);
        if (mr) atomicMax(&acc->max_rel_bits, mr);
        if (rs != 0.0) atomicAdd(&acc->rel_sum, rs);
        if (bad) atomicExch(&acc->bad, 1);
    }
}

// w1_num = sum over x in [0, max_value] of |C(x)|, C(x) = prefix sum of
// hist_est - hist_exact up to x.  Every CTA takes `tiles` consecutive tiles of
// kW1Bins bins (four a thread), at most kW1Ctas CTAs: the first kernel sums the
// differences of a CTA's bins, the second adds the sums of the CTAs before it and
// scans its own.  max_value = 10^6: 9 us for both (863 us in one CTA).
constexpr int kW1Threads = 256;
constexpr uint32_t kW1Bins = 4 * kW1Threads;
constexpr uint64_t kW1Ctas = 2048;

// Differences of this thread's four bins of tile `tile`.
__device__ inline void w1_load(const uint32_t *hist_est, const uint32_t *hist_exact, uint64_t len, uint64_t tile,
                               long long d[4])
{
    const uint64_t x = tile * kW1Bins + 4 * threadIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        d[k] = x + k < len ? (long long)hist_est[x + k] - (long long)hist_exact[x + k] : 0;
}

__device__ inline long long w1_warp_sum(long long s)
{
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__global__ void __launch_bounds__(kW1Threads)
    error_w1_sums_kernel(const uint32_t *hist_est, const uint32_t *hist_exact, uint64_t len, uint64_t tiles,
                         long long *part)
{
    __shared__ long long warp_sum[kW1Threads / 32];
    long long s = 0, d[4];
    for (uint64_t i = 0; i < tiles; ++i) {
        w1_load(hist_est, hist_exact, len, blockIdx.x * tiles + i, d);
        s += d[0] + d[1] + d[2] + d[3];
    }
    s = w1_warp_sum(s);
    if ((threadIdx.x & 31u) == 0) warp_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < kW1Threads / 32; ++w) t += warp_sum[w];
        part[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kW1Threads)
    error_w1_kernel(const uint32_t *hist_est, const uint32_t *hist_exact, uint64_t len, uint64_t tiles,
                    const long long *part, ErrAccum *acc)
{
    __shared__ long long warp_sum[kW1Threads / 32], before[kW1Threads / 32];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    long long b = 0;  // the CTAs before this one
    for (uint32_t i = threadIdx.x; i < blockIdx.x; i += blockDim.x) b += part[i];
    b = w1_warp_sum(b);
    if (lane == 0) before[warp] = b;
    __syncthreads();
    long long carry = 0;
    for (int w = 0; w < kW1Threads / 32; ++w) carry += before[w];
    unsigned long long w1 = 0;
    for (uint64_t i = 0; i < tiles; ++i) {
        const uint64_t tile = blockIdx.x * tiles + i, x = tile * kW1Bins + 4 * threadIdx.x;
        long long d[4];
        w1_load(hist_est, hist_exact, len, tile, d);
        const long long mine = d[0] + d[1] + d[2] + d[3];
        long long incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        __syncthreads();  // the last tile's sums are read
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        long long c = carry + incl - mine;
        for (uint32_t w = 0; w < kW1Threads / 32; ++w) {
            if (w < warp) c += warp_sum[w];
            carry += warp_sum[w];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            c += d[k];
            if (x + k < len) w1 += (unsigned long long)(c < 0 ? -c : c);
        }
    }
    for (int o = 16; o > 0; o >>= 1) w1 += __shfl_xor_sync(0xffffffffu, w1, o);
    if (lane == 0 && w1) atomicAdd(&acc->w1_num, w1);
}

}  // namespace tn

using namespace tn;

extern "C" tn_status tn_error_stats_compute(const uint32_t *est, const uint32_t *exact, uint32_t count,
                                            uint32_t max_value, tn_error_stats *out, void *stream)
{
    if (!est || !exact || !out || count == 0 || max_value == 0 || max_value >= 0xFFFFFFFFu) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t len = (uint64_t)max_value + 1;
    uint32_t *hist = nullptr;
    ErrAccum *acc = nullptr;
    ErrAccum h;
    const uint64_t w1_tiles = (len + kW1Bins - 1) / kW1Bins, per_cta = (w1_tiles + kW1Ctas - 1) / kW1Ctas;
    const unsigned w1_blocks = (unsigned)((w1_tiles + per_cta - 1) / per_cta);
    long long *part = nullptr;
    TN_CUDA_TRY(cudaMallocAsync((void **)&hist, 2 * len * sizeof(uint32_t), st));
    TN_CUDA_TRY(cudaMallocAsync((void **)&part, w1_blocks * sizeof(long long), st));
    TN_CUDA_TRY(cudaMallocAsync((void **)&acc, sizeof(ErrAccum), st));
    TN_CUDA_TRY(cudaMemsetAsync(hist, 0, 2 * len * sizeof(uint32_t), st));
    TN_CUDA_TRY(cudaMemsetAsync(acc, 0, sizeof(ErrAccum), st));
    const unsigned blocks = (count + kErrThreads - 1) / kErrThreads < 2048 ? (count + kErrThreads - 1) / kErrThreads : 2048;
    tn_internal_count_launches(3);
    error_pairs_kernel<<<blocks, kErrThreads, 0, st>>>(est, exact, count, max_value, hist, hist + len, acc);
    error_w1_sums_kernel<<<w1_blocks, kW1Threads, 0, st>>>(hist, hist + len, len, per_cta, part);
    error_w1_kernel<<<w1_blocks, kW1Threads, 0, st>>>(hist, hist + len, len, per_cta, part, acc);
    TN_CUDA_TRY(cudaGetLastError());
    TN_CUDA_TRY(cudaMemcpyAsync(&h, acc, sizeof(h), cudaMemcpyDeviceToHost, st));
    TN_CUDA_TRY(cudaFreeAsync(hist, st));
    TN_CUDA_TRY(cudaFreeAsync(part, st));
    TN_CUDA_TRY(cudaFreeAsync(acc, st));
    TN_CUDA_TRY(cudaStreamSynchronize(st));
    if (h.bad) return TN_ERANGE;
    double max_rel;
    memcpy(&max_rel, &h.max_rel_bits, sizeof(max_rel));
    out->count = count;
    out->sum_abs = h.sum_abs;
    out->max_abs = h.max_abs;
    out->w1_num = h.w1_num;
    out->rel_sum = h.rel_sum;
    out->max_rel = max_rel;
    out->mean_abs = (double)h.sum_abs / count;
    out->mean_rel = h.rel_sum / count;
    out->w1 = (double)h.w1_num / count;
    return TN_OK;
}
