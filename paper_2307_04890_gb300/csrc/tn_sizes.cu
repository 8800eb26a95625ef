// Component sizes (Section 3.1: the out-component size of node j is the number
// of ones in column j; the in-component size of node i the number of ones in
// row i; Section 3.3: both sums have the same total n * mean size).
//
// One CTA covers 32 lanes x WPL 32-bit words of consecutive columns (4,096, or
// 1,024 for narrow matrices) and a block of rows; its 8 warps take eight rows at a
// time, all eight loads of a lane in flight.  Eight row words are added with full
// adders into 10-bit vertical counters (three operations a word and row, against
// sixteen for one row at a time); the counters are extracted once, at the end of
// the CTA's rows.  Row counts are popcounts of a lane's words and one warp
// reduction.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "tn_internal.cuh"

namespace tn {

constexpr int kSizeWarps = 8;
constexpr int kCounterBits = 10;               // vertical counters hold up to 1,023 rows
constexpr uint32_t kRowsMax = kSizeWarps * 1016;  // rows per CTA (127 batches of eight per warp)
constexpr uint32_t kRowsMin = kSizeWarps * 32;  // fewer would spend more on adding the CTAs' counts than on rows

// Bound by HBM: every word of S is read once.  n = 123,457 with row sizes 335 us
// (5.7 TB/s; 899 us with one word a lane and one row at a time into 8-bit counters),
// n = 10^5 208 us (424), n = 10^4 with row sizes 18 us (52), n = 1,000 7 us (27).
template <int WPL>
__global__ void __launch_bounds__(32 * kSizeWarps)
    column_counts_kernel(const uint32_t *S32, uint32_t n_rows, uint64_t ld32, uint32_t ncols, uint32_t rows_per_cta,
                         uint32_t *out, uint32_t *in)
{
    __shared__ uint32_t counts[32 * 32 * WPL];  // [bit][word][lane]
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint64_t word = ((uint64_t)blockIdx.x * 32 + lane) * WPL;
    const bool live = word < ld32;
    const uint32_t r0 = blockIdx.y * rows_per_cta;
    const uint32_t r1 = min(n_rows, r0 + rows_per_cta);
    for (uint32_t i = threadIdx.x; i < 32 * 32 * WPL; i += blockDim.x) counts[i] = 0;
    uint32_t c[kCounterBits][WPL];
#pragma unroll
    for (int i = 0; i < kCounterBits; ++i)
#pragma unroll
        for (int q = 0; q < WPL; ++q) c[i][q] = 0;
    for (uint32_t r = r0 + warp * 8; r < r1; r += kSizeWarps * 8) {
        uint32_t x[8][WPL];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t *p = S32 + (uint64_t)(r + k) * ld32 + word;
#pragma unroll
            for (int q = 0; q < WPL; ++q) x[k][q] = 0;
            if (live && r + k < r1) {
                if (WPL == 4) {
                    const uint4 v = __ldcs(reinterpret_cast<const uint4 *>(p));
                    x[k][0] = v.x;
                    x[k][1 % WPL] = v.y;
                    x[k][2 % WPL] = v.z;
                    x[k][3 % WPL] = v.w;
                } else {
                    x[k][0] = __ldcs(p);
                }
            }
        }
        if (in) {
            uint32_t mine = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                uint32_t pc = 0;
#pragma unroll
                for (int q = 0; q < WPL; ++q) pc += __popc(x[k][q]);
                pc = __reduce_add_sync(0xffffffffu, pc);
                if (lane == k) mine = pc;
            }
            if (lane < 8 && mine) atomicAdd(&in[r + lane], mine);
        }
#pragma unroll
        for (int q = 0; q < WPL; ++q) {
            const uint32_t t0 = full_add(c[0][q], x[0][q], x[1][q]), t1 = full_add(c[0][q], x[2][q], x[3][q]);
            const uint32_t t2 = full_add(c[0][q], x[4][q], x[5][q]), t3 = full_add(c[0][q], x[6][q], x[7][q]);
            const uint32_t f0 = full_add(c[1][q], t0, t1), f1 = full_add(c[1][q], t2, t3);
            uint32_t carry = full_add(c[2][q], f0, f1);
#pragma unroll
            for (int i = 3; i < kCounterBits; ++i) {
                const uint32_t next = c[i][q] & carry;
                c[i][q] ^= carry;
                carry = next;
            }
        }
    }
    __syncthreads();
    auto extract = [&](auto planes) {
#pragma unroll
        for (int q = 0; q < WPL; ++q)
#pragma unroll 4
            for (int b = 0; b < 32; ++b) {
                uint32_t v = 0;
#pragma unroll
                for (int i = 0; i < decltype(planes)::value; ++i) v |= ((c[i][q] >> b) & 1u) << i;
                if (v) atomicAdd(&counts[(b * WPL + q) * 32 + lane], v);
            }
    };
    if (rows_per_cta <= kSizeWarps * 56) extract(std::integral_constant<int, 6>());  // at most 63 rows a warp
    else extract(std::integral_constant<int, kCounterBits>());
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 32 * 32 * WPL; i += blockDim.x) {
        const uint32_t l = i % 32, q = (i / 32) % WPL, b = i / (32 * WPL);
        const uint64_t col = (((uint64_t)blockIdx.x * 32 + l) * WPL + q) * 32 + b;
        if (counts[i] && col < ncols) atomicAdd(&out[col], counts[i]);
    }
}

// Largest size, lowest column among equals; the last CTA to finish writes it.
struct Best {
    unsigned long long key;
    unsigned int done, pad;
};

__global__ void argmax_kernel(const uint32_t *out, uint32_t ncols, Best *best, uint32_t *argmax)
{
    unsigned long long key = 0;
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncols; c += gridDim.x * blockDim.x) {
        const unsigned long long k = ((unsigned long long)out[c] << 32) | (0xFFFFFFFFull - c);
        key = k > key ? k : key;
    }
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, key, d);
        key = o > key ? o : key;
    }
    if ((threadIdx.x & 31u) == 0) atomicMax(&best->key, key);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&best->done, 1u) == gridDim.x - 1) {
        __threadfence();
        *argmax = (uint32_t)(0xFFFFFFFFull - (atomicMax(&best->key, 0ull) & 0xFFFFFFFFull));
    }
}

}  // namespace tn

using namespace tn;

extern "C" tn_status tn_out_sizes(const uint64_t *S, uint32_t n_rows, uint32_t ncols, uint32_t *out_sizes,
                                  uint32_t *in_sizes, uint32_t *argmax, void *stream)
{
    if (!S || !out_sizes || n_rows == 0 || ncols == 0) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t ld32 = 2 * tn_row_words(ncols);
    TN_CUDA_TRY(cudaMemsetAsync(out_sizes, 0, (size_t)ncols * sizeof(uint32_t), st));
    if (in_sizes) TN_CUDA_TRY(cudaMemsetAsync(in_sizes, 0, (size_t)n_rows * sizeof(uint32_t), st));
    // four words a lane where they fill a warp; rows per CTA: as many as the
    // counters hold, in whole waves of two CTAs per SM, but a wave at least
    const int wpl = ld32 >= 96 && ((uintptr_t)S & 15u) == 0 ? 4 : 1;
    const uint64_t cols = (ld32 + 32 * wpl - 1) / (32 * wpl), slots = 2 * (uint64_t)multiprocessors();
    const uint64_t waves = (cols * ((n_rows + kRowsMax - 1) / kRowsMax) + slots - 1) / slots;
    uint64_t blocks = waves * slots / cols;
    if (blocks < 1) blocks = 1;
    uint64_t rows = ((n_rows + blocks - 1) / blocks + kRowsMin - 1) / kRowsMin * kRowsMin;
    if (rows > kRowsMax) rows = kRowsMax;
    const dim3 grid((unsigned)cols, (unsigned)((n_rows + rows - 1) / rows));
    const uint32_t *S32 = reinterpret_cast<const uint32_t *>(S);
    tn_internal_count_launches(1);
    if (wpl == 4)
        column_counts_kernel<4><<<grid, 32 * kSizeWarps, 0, st>>>(S32, n_rows, ld32, ncols, (uint32_t)rows, out_sizes,
                                                                  in_sizes);
    else
        column_counts_kernel<1><<<grid, 32 * kSizeWarps, 0, st>>>(S32, n_rows, ld32, ncols, (uint32_t)rows, out_sizes,
                                                                  in_sizes);
    TN_CUDA_TRY(cudaGetLastError());
    if (argmax) {
        Best *best = nullptr;
        TN_CUDA_TRY(cudaMallocAsync((void **)&best, sizeof(Best), st));
        TN_CUDA_TRY(cudaMemsetAsync(best, 0, sizeof(Best), st));
        const unsigned blocks = (unsigned)((ncols + 255) / 256 < 1024 ? (ncols + 255) / 256 : 1024);
        tn_internal_count_launches(1);
        argmax_kernel<<<blocks, 256, 0, st>>>(out_sizes, ncols, best, argmax);
        TN_CUDA_TRY(cudaGetLastError());
        TN_CUDA_TRY(cudaFreeAsync(best, st));
    }
    return TN_OK;
}
