// Network hashing (Section 4.1) and fusion of the hashed out-components
// (Section 4.2).
//
// Hash family (the paper's construction is garbled; this is its reading as
// Thorup-Zhang 2-character tabulation with a derived character, which the
// paper cites): for replica j the coefficients A(i, c), i < 3, c < 4, are
// ((r1 << 32) + r2) mod p with p = 2^61 - 1 and r = successive SplitMix64
// outputs reduced modulo 2^31 - 1, the stream starting at state
// splitmix64(seed XOR j).  T_i[x] is the cubic A(i,0) x^3 + ... + A(i,3) over
// GF(p) evaluated by the MultAddMod recursion acc <- x * acc + A(i, c), and
// h(u) = (T0[u & 0xFFFF] ^ T1[u >> 16] ^ T2[(u & 0xFFFF) + (u >> 16)]) mod k.
// The coefficients are derived on the host (12 per replica); the tables are
// evaluated on the fly on the device (three cubics per node).
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include "tn_internal.cuh"

namespace tn {

constexpr uint64_t kP61 = (1ull << 61) - 1;

// ---------------- host: coefficient derivation ----------------
static uint64_t sm64_step(uint64_t &state)
{
    state += 0x9E3779B97F4A7C15ull;
    uint64_t z = state;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

static void replica_coefficients(uint64_t seed, uint32_t j, uint64_t out[12])
{
    uint64_t st = seed ^ (uint64_t)j;
    uint64_t stream = sm64_step(st);
    for (int q = 0; q < 12; ++q) {
        const uint64_t hi = sm64_step(stream) % 2147483647ull;
        const uint64_t lo = sm64_step(stream) % 2147483647ull;
        out[q] = ((hi << 32) + lo) % kP61;
    }
}

// ---------------- device: arithmetic modulo 2^61 - 1 ----------------
// (a * x + c) mod p for a, c < p and x < 2^32: the 128-bit product is folded
// with 2^61 = 1 (mod p).
__device__ inline uint64_t mul_add_p61(uint64_t a, uint64_t x, uint64_t c)
{
    const uint64_t lo = a * x;
    const uint64_t hi = __umul64hi(a, x);
    uint64_t r = (lo & kP61) + ((lo >> 61) | (hi << 3));
    r = (r >= kP61) ? r - kP61 : r;
    r += c;
    r = (r >= kP61) ? r - kP61 : r;
    return r;
}

__device__ inline uint64_t cubic_p61(const uint64_t *A, uint64_t x)
{
    uint64_t acc = A[0];
    acc = mul_add_p61(acc, x, A[1]);
    acc = mul_add_p61(acc, x, A[2]);
    acc = mul_add_p61(acc, x, A[3]);
    return acc;
}

__device__ inline uint32_t bucket_of(const uint64_t *A, uint32_t u, uint32_t k)
{
    const uint64_t x0 = u & 0xFFFFu, x1 = u >> 16;
    const uint64_t h = cubic_p61(A, x0) ^ cubic_p61(A + 4, x1) ^ cubic_p61(A + 8, x0 + x1);
    return (uint32_t)(h % k);
}

__global__ void hash_nodes_kernel(const uint64_t *coef, uint32_t R, uint32_t k, uint32_t n, uint32_t *H)
{
    const uint64_t total = (uint64_t)R * n;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t j = (uint32_t)(i / n), x = (uint32_t)(i - (uint64_t)j * n);
        H[i] = bucket_of(coef + 12ull * j, x, k);
    }
}

// super-events (h_j(u), h_j(v), t) of every replica (Section 4.1)
__global__ void proxy_events_kernel(const uint32_t *u, const uint32_t *v, uint64_t m, uint32_t n, uint32_t R,
                                    const uint32_t *H, uint32_t *pu, uint32_t *pv)
{
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < m; e += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t a = u[e], b = v[e];
        for (uint32_t j = 0; j < R; ++j) {
            // an endpoint outside [0, n) becomes an invalid super-node, which a
            // later plan over the super-events rejects with TN_ERANGE
            pu[(uint64_t)j * m + e] = a < n ? __ldg(H + (uint64_t)j * n + a) : 0xFFFFFFFFu;
            pv[(uint64_t)j * m + e] = b < n ? __ldg(H + (uint64_t)j * n + b) : 0xFFFFFFFFu;
        }
    }
}

// ---------------- fusion ----------------
// CTA = 8 sources.  table[j * k + b] bit s = [super-node b reached from
// h_j(x_s) in proxy j] = bit h_j(x_s) of row b of P_j.  A node w belongs to
// the estimate of source s when bit s of AND_j table[j * k + h_j(w)] is set.
constexpr int kEstSources = 8;
constexpr uint32_t kBitsliceMinSources = 256;  // from here on the bit-sliced fusion is used
constexpr int kEstThreads = 256;

__global__ void check_sources_kernel(const uint32_t *src, uint32_t nsrc, uint32_t n, int32_t *bad)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nsrc; i += gridDim.x * blockDim.x)
        if (src[i] >= n) atomicExch(bad, 1);
}

__global__ void __launch_bounds__(kEstThreads)
    estimate_kernel(const uint64_t *P, uint32_t R, uint32_t k, uint64_t ldk, const uint32_t *H, uint32_t n,
                    const uint32_t *src, uint32_t nsrc, uint32_t *est, uint8_t *gtable)
{
    extern __shared__ uint8_t stable[];
    __shared__ uint32_t col[kEstSources * 64];  // h_j(x_s) for up to 64 replicas
    __shared__ uint32_t cnt[kEstSources];
    const uint32_t s0 = blockIdx.x * kEstSources;
    const uint32_t ns = min((uint32_t)kEstSources, nsrc - s0);
    uint8_t *table = gtable ? gtable + (uint64_t)blockIdx.x * R * k : stable;
    for (uint32_t q = threadIdx.x; q < kEstSources * R; q += blockDim.x) {
        const uint32_t s = q / R, j = q - s * R;
        const uint32_t x = s < ns ? (src ? src[s0 + s] : s0 + s) : 0u;
        col[s * R + j] = H[(uint64_t)j * n + x];
    }
    if (threadIdx.x < kEstSources) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (uint64_t q = threadIdx.x; q < (uint64_t)R * k; q += blockDim.x) {
        const uint32_t j = (uint32_t)(q / k), b = (uint32_t)(q - (uint64_t)j * k);
        const uint64_t *row = P + ((uint64_t)j * k + b) * ldk;
        uint32_t byte = 0;
        for (uint32_t s = 0; s < ns; ++s) {
            const uint32_t c = col[s * R + j];
            byte |= (uint32_t)((__ldg(row + (c >> 6)) >> (c & 63)) & 1ull) << s;
        }
        table[q] = (uint8_t)byte;
    }
    __syncthreads();
    uint32_t c[kEstSources];
#pragma unroll
    for (int s = 0; s < kEstSources; ++s) c[s] = 0;
    const uint32_t all = (1u << ns) - 1u;
    for (uint32_t w = blockIdx.y * blockDim.x + threadIdx.x; w < n; w += gridDim.y * blockDim.x) {
        uint32_t mask = all;
        for (uint32_t j = 0; j < R && mask; ++j) mask &= table[(uint64_t)j * k + __ldg(H + (uint64_t)j * n + w)];
#pragma unroll
        for (int s = 0; s < kEstSources; ++s) c[s] += (mask >> s) & 1u;
    }
#pragma unroll
    for (int s = 0; s < kEstSources; ++s) {
        uint32_t x = c[s];
        for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        if ((threadIdx.x & 31u) == 0 && x) atomicAdd(&cnt[s], x);
    }
    __syncthreads();
    if (threadIdx.x < ns && cnt[threadIdx.x]) atomicAdd(&est[s0 + threadIdx.x], cnt[threadIdx.x]);
}

// ---------------- fusion, bit-sliced over sources ----------------
// For many sources the fusion is reorganised around a transposed table, built for
// one chunk of sources at a time:
//   T[j][b] = bitset over the chunk's sources, bit s = bit h_j(x_s) of row b of P_j
// (Section 4.2: super-node b reaches h_j(x_s) in proxy j).  Then
//   est(x_s) = #{w : bit s of AND_j T[j][h_j(w)]},
// i.e. a column count of the n x chunk boolean matrix whose row w is the AND of R
// rows of T.  A chunk is 4,096 sources (512-byte rows of T, four words a lane) or,
// for few sources, 1,024: small enough that T stays in L2 (R = 8, k = 16,384: 64
// MB) while every node reads R of its rows.
constexpr int kTabThreads = 256;
constexpr int kTabRows = 32;            // proxy rows per CTA, in shared memory
constexpr uint32_t kTabSmem = 200 * 1024;  // largest such block of rows (k <= 51,200)

// Bits of 32 rows of P_j at 256 sources' columns per warp step: lane i holds
// source 32 s + i, reads the 32-bit word of its column in four rows at a time
// (rows are stored in groups of four, rotated by the 16-byte piece against bank
// conflicts), and a ballot per row gathers the 32 sources' bits; lane r keeps row
// r's words and stores a whole 32-byte sector.  Bound by the shared-memory reads
// of random columns.  R = 8, k = 16,384, 65,536 sources: about 4 ms in all (36 ms
// with one thread gathering 32 bits through L1 per word).
__global__ void __launch_bounds__(kTabThreads)
    bitslice_table_kernel(const uint64_t *P, uint32_t k, uint64_t ldk, const uint32_t *H, uint32_t n,
                          const uint32_t *src, uint32_t s0, uint32_t ns, uint32_t words, uint32_t *T)
{
    extern __shared__ uint4 rows4[];  // [ldk32][8]
    const uint32_t j = blockIdx.z, b0 = blockIdx.x * kTabRows;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t w4 = (k + 127) / 128;  // 16-byte pieces of a row that hold columns
    uint32_t *flat = reinterpret_cast<uint32_t *>(rows4);
    for (uint32_t i0 = threadIdx.x; i0 < w4 * kTabRows; i0 += 4 * blockDim.x) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {  // four loads in flight; consecutive threads read along a row
            const uint32_t i = i0 + u * blockDim.x, r = i / w4, c = i - r * w4;
            v[u] = make_uint4(0u, 0u, 0u, 0u);
            if (i < w4 * kTabRows && b0 + r < k)
                v[u] = __ldg(reinterpret_cast<const uint4 *>(P + ((uint64_t)j * k + b0 + r) * ldk) + c);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t i = i0 + u * blockDim.x, r = i / w4, c = i - r * w4;
            if (i >= w4 * kTabRows) continue;
            const uint32_t word[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (uint32_t h = 0; h < 4; ++h) {
                const uint32_t w = 4 * c + h;
                flat[w * kTabRows + (((r >> 2) + c) & 7u) * 4 + (r & 3u)] = word[h];
            }
        }
    }
    __syncthreads();
    const uint32_t groups = (ns + 255) / 256;
    for (uint32_t g = blockIdx.y * (kTabThreads / 32) + warp; g < groups; g += gridDim.y * (kTabThreads / 32)) {
        uint32_t col[8], mine[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const uint32_t q = g * 256 + s * 32 + lane;
            col[s] = 0xFFFFFFFFu;
            mine[s] = 0;
            if (q < ns) col[s] = __ldg(H + (uint64_t)j * n + (src ? __ldg(src + s0 + q) : s0 + q));
        }
#pragma unroll 1
        for (uint32_t q = 0; q < 8; ++q) {  // rows 4q .. 4q + 3
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const bool in = col[s] != 0xFFFFFFFFu;
                const uint32_t w = in ? col[s] >> 5 : 0u, bit = in ? 1u << (col[s] & 31u) : 0u;
                const uint4 v = rows4[w * 8 + ((q + (w >> 2)) & 7u)];
                const uint32_t x0 = __ballot_sync(0xffffffffu, v.x & bit), x1 = __ballot_sync(0xffffffffu, v.y & bit);
                const uint32_t x2 = __ballot_sync(0xffffffffu, v.z & bit), x3 = __ballot_sync(0xffffffffu, v.w & bit);
                if ((lane >> 2) == q) mine[s] = (lane & 2u) ? ((lane & 1u) ? x3 : x2) : ((lane & 1u) ? x1 : x0);
            }
        }
        if (b0 + lane < k) {
            uint4 *out = reinterpret_cast<uint4 *>(T + ((uint64_t)j * k + b0 + lane) * words + g * 8);
            out[0] = make_uint4(mine[0], mine[1], mine[2], mine[3]);
            out[1] = make_uint4(mine[4], mine[5], mine[6], mine[7]);
        }
    }
}

// The same table for proxies whose rows do not fit shared memory 32 at a time, and
// for a P that is not 16-byte aligned: one thread per 32-bit word of T, columns read
// through L1 in 8-byte loads.
__global__ void __launch_bounds__(kTabThreads)
    bitslice_table_wide_kernel(const uint64_t *P, uint32_t k, uint64_t ldk, const uint32_t *H, uint32_t n,
                               const uint32_t *src, uint32_t s0, uint32_t ns, uint32_t words, uint32_t *T)
{
    __shared__ uint32_t col[4096];
    const uint32_t j = blockIdx.z;
    for (uint32_t q = threadIdx.x; q < ns; q += blockDim.x)
        col[q] = H[(uint64_t)j * n + (src ? src[s0 + q] : s0 + q)];
    __syncthreads();
    const uint32_t b1 = min(k, (blockIdx.x + 1u) * 64u);
    for (uint32_t b = blockIdx.x * 64u; b < b1; ++b) {
        const uint64_t *row = P + ((uint64_t)j * k + b) * ldk;
        for (uint32_t wd = threadIdx.x; wd < words; wd += blockDim.x) {
            uint32_t bits = 0;
#pragma unroll 8
            for (uint32_t i = 0; i < 32; ++i) {
                const uint32_t q = wd * 32 + i;
                if (q < ns) bits |= (uint32_t)((__ldg(row + (col[q] >> 6)) >> (col[q] & 63)) & 1ull) << i;
            }
            T[((uint64_t)j * k + b) * words + wd] = bits;
        }
    }
}

constexpr int kCountWarps = 8;
constexpr int kCountBits = 10;                            // vertical counters hold up to 1,023 rows
constexpr uint32_t kCountMax = kCountWarps * 1016;        // nodes per CTA at most (1,016 = 127 x 8 per warp)

// Column counts of the chunk: a warp takes every eighth node of the CTA's range,
// lane l the WPL words at 32 WPL sources.  Eight nodes at a time are added with
// full adders into 10-bit vertical counters (three operations a word and node,
// against sixteen for one node at a time), two nodes' R rows in flight; buckets of
// the range are staged in shared memory.  Bound by the L2 reads of T (R rows a
// node): n = 10^6, R = 8, 65,536 sources 5.6 ms at 12.8 TB/s (56 ms with the whole
// table in DRAM, one word a lane and 4-bit counters); counts leave the registers
// once.
template <int WPL>
__global__ void __launch_bounds__(32 * kCountWarps)
    bitslice_count_kernel(const uint32_t *T, uint32_t words, uint32_t R, uint32_t k, const uint32_t *H, uint32_t n,
                          uint32_t per_cta, uint32_t ns, uint32_t *est)
{
    extern __shared__ uint32_t sh[];
    uint32_t *counts = sh;                       // [32 bits][32 WPL words]
    uint32_t *rows = sh + 32 * 32 * WPL;         // [R][256] T rows of a batch of nodes
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    for (uint32_t i = threadIdx.x; i < 32 * 32 * WPL; i += blockDim.x) counts[i] = 0;
    const uint32_t w0 = blockIdx.x * per_cta, w1 = min(n, w0 + per_cta);
    uint32_t c[kCountBits][WPL];
#pragma unroll
    for (int i = 0; i < kCountBits; ++i)
#pragma unroll
        for (int q = 0; q < WPL; ++q) c[i][q] = 0;
    for (uint32_t base = w0; base < w1; base += 256) {
        __syncthreads();
        const uint32_t cnt = min(256u, w1 - base);
        for (uint32_t j = warp; j < R; j += kCountWarps)
            for (uint32_t i = lane; i < 256; i += 32)
                rows[j * 256 + i] = i < cnt ? j * k + __ldg(H + (uint64_t)j * n + base + i) : 0xFFFFFFFFu;
        __syncthreads();
        // warp's nodes of the batch: 32 consecutive, eight at a time
#pragma unroll 1
        for (uint32_t e = 0; e < 4; ++e) {
            const uint32_t at = warp * 32 + e * 8;
            if (at >= cnt) break;
            uint32_t two[4][WPL], four[2][WPL];
#pragma unroll
            for (int p = 0; p < 4; ++p) {  // pairs of nodes
                uint32_t x[2][WPL];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < WPL; ++q) x[h][q] = at + 2 * p + h < cnt ? 0xFFFFFFFFu : 0u;
#pragma unroll 4
                for (uint32_t j = 0; j < R; ++j) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t r = rows[j * 256 + at + 2 * p + h];
                        const uint32_t *t = T + (uint64_t)(r == 0xFFFFFFFFu ? 0u : r) * words + lane * WPL;
                        if (WPL == 4) {
                            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(t));
                            x[h][0] &= v.x;
                            x[h][1 % WPL] &= v.y;
                            x[h][2 % WPL] &= v.z;
                            x[h][3 % WPL] &= v.w;
                        } else {
                            x[h][0] &= __ldg(t);
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < WPL; ++q) two[p][q] = full_add(c[0][q], x[0][q], x[1][q]);
            }
#pragma unroll
            for (int q = 0; q < WPL; ++q) {
                four[0][q] = full_add(c[1][q], two[0][q], two[1][q]);
                four[1][q] = full_add(c[1][q], two[2][q], two[3][q]);
                uint32_t carry = full_add(c[2][q], four[0][q], four[1][q]);
#pragma unroll
                for (int i = 3; i < kCountBits; ++i) {
                    const uint32_t next = c[i][q] & carry;
                    c[i][q] ^= carry;
                    carry = next;
                }
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < WPL; ++q)
#pragma unroll 1
        for (int b = 0; b < 32; ++b) {
            uint32_t v = 0;
#pragma unroll
            for (int i = 0; i < kCountBits; ++i) v |= ((c[i][q] >> b) & 1u) << i;
            if (v) atomicAdd(&counts[b * 32 * WPL + q * 32 + lane], v);
        }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 32 * 32 * WPL; i += blockDim.x) {
        const uint32_t b = i / (32 * WPL), q = (i / 32) % WPL, l = i % 32;
        const uint32_t s = (l * WPL + q) * 32 + b;
        if (s < ns && counts[i]) atomicAdd(&est[s], counts[i]);
    }
}

}  // namespace tn

using namespace tn;

extern "C" tn_status tn_hash_proxy(const uint32_t *u, const uint32_t *v, uint64_t m, uint32_t n, uint32_t k,
                                   uint32_t R, uint64_t seed, uint32_t *H, uint32_t *pu, uint32_t *pv,
                                   void *stream)
{
    if (!H || n == 0 || k == 0 || R == 0 || n >= (1u << 30) || k >= (1u << 30)) return TN_EINVAL;
    if (m > 0 && (pu || pv) && (!pu || !pv || !u || !v)) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    uint64_t *hcoef = (uint64_t *)malloc(12 * sizeof(uint64_t) * R);
    if (!hcoef) return TN_ENOMEM;
    for (uint32_t j = 0; j < R; ++j) replica_coefficients(seed, j, hcoef + 12ull * j);
    uint64_t *dcoef = nullptr;
    cudaError_t err = cudaMallocAsync((void **)&dcoef, 12 * sizeof(uint64_t) * R, st);
    if (err == cudaSuccess) err = cudaMemcpyAsync(dcoef, hcoef, 12 * sizeof(uint64_t) * R, cudaMemcpyHostToDevice, st);
    if (err == cudaSuccess) err = cudaStreamSynchronize(st);  // the host copy may be freed now
    free(hcoef);
    if (err != cudaSuccess) {
        tn_internal_set_cuda_error(err);
        return err == cudaErrorMemoryAllocation ? TN_ENOMEM : TN_ECUDA;
    }
    const uint64_t total = (uint64_t)R * n;
    tn_internal_count_launches(1);
    hash_nodes_kernel<<<(unsigned)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192), 256, 0, st>>>(dcoef, R,
                                                                                                          k, n, H);
    if (m > 0 && pu) {
        tn_internal_count_launches(1);
        proxy_events_kernel<<<(unsigned)((m + 255) / 256 < 8192 ? (m + 255) / 256 : 8192), 256, 0, st>>>(
            u, v, m, n, R, H, pu, pv);
    }
    TN_CUDA_TRY(cudaGetLastError());
    TN_CUDA_TRY(cudaFreeAsync(dcoef, st));
    return TN_OK;
}

static tn_status estimate_bitsliced(const uint64_t *P, uint32_t R, uint32_t k, uint64_t ldk, const uint32_t *H,
                                    uint32_t n, const uint32_t *src, uint32_t nsrc, uint32_t *est, cudaStream_t st)
{
    // four words a lane once that leaves no large part of a chunk empty
    const uint32_t chunk = nsrc > 3072 && (uint64_t)R * k * 512 <= (2ull << 30) ? 4096u : 1024u;
    const uint32_t words = chunk / 32;
    const size_t tab_smem = (size_t)((k + 127) / 128) * 4 * kTabRows * 4;
    const bool wide = tab_smem > kTabSmem || ((uintptr_t)P & 15u);  // (rows are whole 128-byte units)
    const size_t cnt_smem = (32ull * words + 256ull * R) * 4;
    uint32_t *T = nullptr;
    TN_CUDA_TRY(cudaMallocAsync((void **)&T, (uint64_t)R * k * words * 4, st));
    if (!wide) TN_CUDA_TRY(tn_internal_allow_max_dyn_smem((const void *)bitslice_table_kernel));
    const void *count = chunk == 4096 ? (const void *)bitslice_count_kernel<4> : (const void *)bitslice_count_kernel<1>;
    TN_CUDA_TRY(tn_internal_allow_max_dyn_smem(count));
    // nodes per CTA: a multiple of the 256-node batch, about four CTAs per SM
    uint32_t per_cta = (uint32_t)(((uint64_t)n / (4 * (uint64_t)multiprocessors()) + 255) / 256 * 256);
    if (per_cta < 256) per_cta = 256;
    if (per_cta > kCountMax / 256 * 256) per_cta = kCountMax / 256 * 256;
    const unsigned blocks = (n + per_cta - 1) / per_cta;
    for (uint32_t s0 = 0; s0 < nsrc; s0 += chunk) {
        const uint32_t ns = nsrc - s0 < chunk ? nsrc - s0 : chunk;
        tn_internal_count_launches(2);
        if (wide)
            bitslice_table_wide_kernel<<<dim3((k + 63) / 64, 1, R), kTabThreads, 0, st>>>(P, k, ldk, H, n, src, s0, ns,
                                                                                         words, T);
        else
            bitslice_table_kernel<<<dim3((k + kTabRows - 1) / kTabRows, 1, R), kTabThreads, tab_smem, st>>>(
                P, k, ldk, H, n, src, s0, ns, words, T);
        if (chunk == 4096)
            bitslice_count_kernel<4><<<blocks, 32 * kCountWarps, cnt_smem, st>>>(T, words, R, k, H, n, per_cta, ns, est + s0);
        else
            bitslice_count_kernel<1><<<blocks, 32 * kCountWarps, cnt_smem, st>>>(T, words, R, k, H, n, per_cta, ns, est + s0);
        TN_CUDA_TRY(cudaGetLastError());
    }
    TN_CUDA_TRY(cudaFreeAsync(T, st));
    return TN_OK;
}

extern "C" tn_status tn_hash_estimate(const uint64_t *P, uint32_t R, uint32_t k, const uint32_t *H, uint32_t n,
                                      const uint32_t *src, uint32_t nsrc, uint32_t *est, void *stream)
{
    if (!P || !H || !est || R == 0 || R > 64 || k == 0 || n == 0 || nsrc == 0) return TN_EINVAL;
    if (!src && nsrc != n) return TN_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (src) {  // validating: source ids must be node ids
        int32_t *dbad = nullptr, hbad = 0;
        TN_CUDA_TRY(cudaMallocAsync((void **)&dbad, sizeof(int32_t), st));
        TN_CUDA_TRY(cudaMemsetAsync(dbad, 0, sizeof(int32_t), st));
        tn_internal_count_launches(1);
        check_sources_kernel<<<(nsrc + 255) / 256 < 1024 ? (nsrc + 255) / 256 : 1024, 256, 0, st>>>(src, nsrc, n, dbad);
        TN_CUDA_TRY(cudaMemcpyAsync(&hbad, dbad, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        TN_CUDA_TRY(cudaFreeAsync(dbad, st));
        TN_CUDA_TRY(cudaStreamSynchronize(st));
        if (hbad) return TN_ERANGE;
    }
    const uint64_t ldk = tn_row_words(k);
    const uint64_t table_bytes = (uint64_t)R * k;
    const unsigned batches = (nsrc + kEstSources - 1) / kEstSources;
    TN_CUDA_TRY(cudaMemsetAsync(est, 0, (size_t)nsrc * sizeof(uint32_t), st));
    if (nsrc >= kBitsliceMinSources) return estimate_bitsliced(P, R, k, ldk, H, n, src, nsrc, est, st);
    uint8_t *gtable = nullptr;
    size_t smem = 0;
    if (table_bytes <= 200 * 1024) {
        smem = table_bytes;
        TN_CUDA_TRY(tn_internal_allow_max_dyn_smem((const void *)estimate_kernel));
    } else {
        TN_CUDA_TRY(cudaMallocAsync((void **)&gtable, table_bytes * batches, st));  // one table per CTA
    }
    tn_internal_count_launches(1);
    estimate_kernel<<<dim3(batches, 1), kEstThreads, smem, st>>>(P, R, k, ldk, H, n, src, nsrc, est, gtable);
    TN_CUDA_TRY(cudaGetLastError());
    if (gtable) TN_CUDA_TRY(cudaFreeAsync(gtable, st));
    return TN_OK;
}

// ---------------- fusion without allocation ----------------
// For callers that cannot allocate device memory during a call (code inside
// another framework's memory budget, latency-bound loops).  Same result as
// tn_hash_estimate, but only its byte-table fusion (one CTA per 8 sources):
// the bit-sliced path for many sources needs R * k * 128 or 512 bytes of transposed
// tables, more than a fixed array should hold, so every call here
// reads H once per 8 sources (about ceil(nsrc / 8) * R * n * 4 bytes).  The
// source-check flag and the per-CTA tables of the global-table path live in
// one fixed device array of this module instead of the stream-ordered
// allocator.  Host code never uses the array's name as an
// address: the address comes from cudaGetSymbolAddress, per device.  Bytes [0, 4) hold the
// flag, the tables start at byte 256.
#include <mutex>

namespace tn {
static __device__ __align__(256) uint8_t g_noalloc_scratch[TN_NOALLOC_SCRATCH_BYTES];
constexpr uint64_t kNoallocTableOffset = 256;
constexpr int kNoallocMaxDevices = 64;

// Address of the scratch on the current device, looked up once per device.
static tn_status noalloc_scratch(uint8_t **out)
{
    static std::mutex mu;
    static uint8_t *addr[kNoallocMaxDevices] = {nullptr};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) {
        tn_internal_set_cuda_error(err);
        return TN_ECUDA;
    }
    if (dev < 0 || dev >= kNoallocMaxDevices) return TN_EINVAL;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        err = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (err != cudaSuccess) {
            tn_internal_set_cuda_error(err);
            return TN_ECUDA;
        }
        addr[dev] = (uint8_t *)p;
    }
    *out = addr[dev];
    return TN_OK;
}
}  // namespace tn

extern "C" tn_status tn_hash_estimate_noalloc(const uint64_t *P, uint32_t R, uint32_t k, const uint32_t *H,
                                              uint32_t n, const uint32_t *src, uint32_t nsrc, uint32_t *est,
                                              void *stream)
{
    if (!P || !H || !est || R == 0 || R > 64 || k == 0 || n == 0 || nsrc == 0) return TN_EINVAL;
    if (!src && nsrc != n) return TN_EINVAL;
    const uint64_t ldk = tn_row_words(k);
    const uint64_t table_bytes = (uint64_t)R * k;
    const unsigned batches = (nsrc + kEstSources - 1) / kEstSources;
    const bool smem_table = table_bytes <= 200 * 1024;
    if (!smem_table && table_bytes * batches > TN_NOALLOC_TABLE_BYTES) return TN_ESCRATCH;
    uint8_t *scratch = nullptr;
    const tn_status s = noalloc_scratch(&scratch);
    if (s != TN_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    if (src) {  // validating: source ids must be node ids
        int32_t *dbad = reinterpret_cast<int32_t *>(scratch), hbad = 0;
        TN_CUDA_TRY(cudaMemsetAsync(dbad, 0, sizeof(int32_t), st));
        tn_internal_count_launches(1);
        check_sources_kernel<<<(nsrc + 255) / 256 < 1024 ? (nsrc + 255) / 256 : 1024, 256, 0, st>>>(src, nsrc, n, dbad);
        TN_CUDA_TRY(cudaMemcpyAsync(&hbad, dbad, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        TN_CUDA_TRY(cudaStreamSynchronize(st));
        if (hbad) return TN_ERANGE;
    }
    TN_CUDA_TRY(cudaMemsetAsync(est, 0, (size_t)nsrc * sizeof(uint32_t), st));
    size_t smem = 0;
    uint8_t *gtable = nullptr;
    if (smem_table) {
        smem = table_bytes;
        TN_CUDA_TRY(tn_internal_allow_max_dyn_smem((const void *)estimate_kernel));
    } else {
        gtable = scratch + kNoallocTableOffset;  // every byte is written by its CTA before it is read
    }
    tn_internal_count_launches(1);
    estimate_kernel<<<dim3(batches, 1), kEstThreads, smem, st>>>(P, R, k, ldk, H, n, src, nsrc, est, gtable);
    TN_CUDA_TRY(cudaGetLastError());
    return TN_OK;
}
