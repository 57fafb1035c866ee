// Time-randomised control (arXiv:1802.01685 Sect. 2.2 and Fig. 2): the series
// with its samples permuted, which keeps the sample histogram exactly and
// destroys all phase coherence.  The permutation is the argsort of the pairs
// (splitmix64(seed ^ i), i) -- a counter-based draw, so it does not depend on
// the device or thread count -- and out[rank of i] = in[i].
// splitmix64 is the published generator of Steele, Lea and Flood (2014).
//
// The keys are as good as uniform, so one pass of buckets on their leading
// bits leaves about 8-16 keys to a bucket (32-64 from 2^23 samples on), and a
// key's place inside its bucket is the number of smaller pairs there:
//   count    the bucket of every i; its slot in the bucket by arrival (atomic)
//   scan     where each bucket begins
//   scatter  i into its bucket, in arrival order
//   rank     the place of i among its bucket's pairs, and the sample moved
// Nothing is assumed of the keys but speed: any distribution gives the argsort
// (the pairs are compared in full), a crowded bucket only takes longer, and
// the arrival order does not reach the output.  Keys are computed again in
// every step (a dozen integer operations) rather than stored, so the scratch
// is 8 bytes a sample and 8 a bucket.  The work is latency, not bandwidth:
// 262,144 samples on the device took 241 us a call as a bitonic sort of (key,
// index) arrays in 37 launches, and take 38 us in these four.
#include <algorithm>

#include "bf_internal.h"

namespace bfi {

constexpr int SORT_T = 256;               // threads per block of the per-sample kernels
constexpr int SCAN_THREADS = 1024;        // of the scan; each takes four buckets
constexpr uint32_t SCAN_TILE = 4 * SCAN_THREADS;
constexpr uint32_t SMALL_N = 4096;        // sorted by one block, in shared memory
constexpr int SMALL_T = 1024;
constexpr uint32_t SMALL_BUCKETS = 1024;

__device__ __forceinline__ uint64_t splitmix64(uint64_t z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// (ka, ia) before (kb, ib) in the argsort's order
__device__ __forceinline__ bool pair_less(uint64_t ka, uint32_t ia, uint64_t kb, uint32_t ib)
{
    return ka < kb || (ka == kb && ia < ib);
}

// inclusive scan over the block's threads (all of them take part); sh: one word per warp
__device__ __forceinline__ uint32_t block_incl_scan(uint32_t v, uint32_t* sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = lane < nw ? sh[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        if (lane < nw) sh[lane] = s;
    }
    __syncthreads();
    return inc + (wid > 0 ? sh[wid - 1] : 0u);
}

// count[b] (zeroed before) and slot[i], bucket b = the key's bits above `shift`
__global__ void __launch_bounds__(SORT_T) k_perm_count(uint32_t n, uint64_t seed, int shift,
                                                       uint32_t* __restrict__ count, uint32_t* __restrict__ slot)
{
    const uint64_t i = blockIdx.x * (uint64_t)SORT_T + threadIdx.x;
    if (i >= n) return;
    slot[i] = atomicAdd(count + (splitmix64(seed ^ i) >> shift), 1u);
}

// begin[b] = the samples in buckets before b.  Every block scans its own
// SCAN_TILE buckets and sums all those before them itself, so that no block
// waits for another and one launch does (the last of 8 tiles at 2^19 samples
// reads 112 KB from L2).  n_buckets is a multiple of 4.
__global__ void __launch_bounds__(SCAN_THREADS) k_perm_scan(const uint32_t* __restrict__ count, uint32_t n_buckets,
                                                            uint32_t* __restrict__ begin)
{
    __shared__ uint32_t sh[SCAN_THREADS / 32];
    __shared__ uint32_t sh_base;
    const uint4* c4 = reinterpret_cast<const uint4*>(count);
    const uint32_t q = blockIdx.x * SCAN_THREADS + threadIdx.x;        // this thread's four buckets
    uint32_t before = 0;
    for (uint32_t p = threadIdx.x; p < blockIdx.x * SCAN_THREADS; p += SCAN_THREADS) {
        const uint4 v = c4[p];
        before += (v.x + v.y) + (v.z + v.w);
    }
    const uint32_t all = block_incl_scan(before, sh);
    if (threadIdx.x == SCAN_THREADS - 1) sh_base = all;
    __syncthreads();
    const uint32_t base = sh_base;
    const bool in = 4 * q < n_buckets;
    const uint4 v = in ? c4[q] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t mine = (v.x + v.y) + (v.z + v.w);
    const uint32_t e = base + block_incl_scan(mine, sh) - mine;
    if (in) reinterpret_cast<uint4*>(begin)[q] = make_uint4(e, e + v.x, e + v.x + v.y, e + v.x + v.y + v.z);
}

__global__ void __launch_bounds__(SORT_T) k_perm_scatter(uint32_t n, uint64_t seed, int shift,
                                                         const uint32_t* __restrict__ begin,
                                                         const uint32_t* __restrict__ slot,
                                                         uint32_t* __restrict__ idx)
{
    const uint64_t i = blockIdx.x * (uint64_t)SORT_T + threadIdx.x;
    if (i >= n) return;
    idx[begin[splitmix64(seed ^ i) >> shift] + slot[i]] = (uint32_t)i;
}

// One thread per place p of the bucket order: its sample's final place is its
// bucket's beginning plus the number of smaller pairs in the bucket.  The block
// first makes the keys of its own places and RANK_HALO on either side, once
// each, where every thread made those of its whole bucket again (6.7 us for
// 262,144 samples against 10.7).  A bucket that reaches further than that, far
// from the mean of at most 64, is ranked from its indices.
constexpr int RANK_HALO = 128;
__global__ void __launch_bounds__(SORT_T) k_perm_rank(const float* __restrict__ in, uint32_t n, uint64_t seed,
                                                      int shift, const uint32_t* __restrict__ begin,
                                                      const uint32_t* __restrict__ count,
                                                      const uint32_t* __restrict__ idx, float* __restrict__ out)
{
    constexpr int W = SORT_T + 2 * RANK_HALO;
    __shared__ uint64_t sk[W];
    __shared__ uint32_t si[W];
    const int64_t w0 = (int64_t)blockIdx.x * SORT_T - RANK_HALO;       // place of sk[0]
#pragma unroll
    for (int e = 0; e < W / SORT_T; ++e) {
        const int u = threadIdx.x + e * SORT_T;
        const int64_t q = w0 + u;
        if (q >= 0 && q < (int64_t)n) {
            const uint32_t i = idx[q];
            si[u] = i;
            sk[u] = splitmix64(seed ^ (uint64_t)i);
        }
    }
    __syncthreads();
    const uint64_t p = blockIdx.x * (uint64_t)SORT_T + threadIdx.x;
    if (p >= n) return;
    const uint32_t i = si[threadIdx.x + RANK_HALO];
    const uint64_t key = sk[threadIdx.x + RANK_HALO];
    const float v = in[i];
    const uint32_t b0 = begin[key >> shift], m = count[key >> shift];
    uint32_t rank = b0;
    if ((int64_t)b0 >= w0 && (int64_t)b0 + m <= w0 + W) {
        const int u0 = (int)((int64_t)b0 - w0);
#pragma unroll 4
        for (uint32_t q = 0; q < m; ++q) rank += pair_less(sk[u0 + q], si[u0 + q], key, i) ? 1u : 0u;
    } else {
        for (uint32_t q = 0; q < m; ++q) {
            const uint32_t k = idx[b0 + q];
            rank += pair_less(splitmix64(seed ^ (uint64_t)k), k, key, i) ? 1u : 0u;
        }
    }
    out[rank] = v;
}

// The four steps in one block for n <= SMALL_N.
__global__ void __launch_bounds__(SMALL_T) k_perm_small(const float* __restrict__ in, uint32_t n, uint64_t seed,
                                                        float* __restrict__ out)
{
    __shared__ uint32_t count[SMALL_BUCKETS], begin[SMALL_BUCKETS];
    __shared__ uint32_t sh[SMALL_T / 32];
    __shared__ uint64_t key[SMALL_N];
    __shared__ uint32_t idx[SMALL_N];
    constexpr int E = SMALL_N / SMALL_T;
    constexpr int SHIFT = 54;                                  // 2^10 buckets
    static_assert(SMALL_BUCKETS == 1024 && SMALL_T == 1024, "one thread per bucket");
    count[threadIdx.x] = 0u;
    __syncthreads();
    uint64_t k[E];
    uint32_t slot[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = threadIdx.x + e * SMALL_T;
        k[e] = splitmix64(seed ^ (uint64_t)i);
        if (i < n) slot[e] = atomicAdd(count + (k[e] >> SHIFT), 1u);
    }
    __syncthreads();
    const uint32_t c = count[threadIdx.x];
    begin[threadIdx.x] = block_incl_scan(c, sh) - c;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = threadIdx.x + e * SMALL_T;
        if (i < n) {
            const uint32_t p = begin[k[e] >> SHIFT] + slot[e];
            key[p] = k[e];
            idx[p] = i;
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = threadIdx.x + e * SMALL_T;
        if (i >= n) continue;
        const uint32_t b0 = begin[k[e] >> SHIFT], m = count[k[e] >> SHIFT];
        uint32_t rank = b0;
        for (uint32_t q = b0; q < b0 + m; ++q) rank += pair_less(key[q], idx[q], k[e], i) ? 1u : 0u;
        out[rank] = in[i];
    }
}

// log2 of the number of buckets for n > SMALL_N samples: 8-16 samples a bucket
// up to 2^23 samples (2^19 buckets), where the scan's re-reading of the tiles
// before each block is still microseconds; 32-64 beyond
static int bucket_bits(uint64_t n)
{
    int p = 0;
    while ((1ull << p) < n) ++p;           // 2^p >= n
    return n <= (1ull << 23) ? p - 4 : p - 6;
}

size_t permute_scratch_bytes(uint64_t n)
{
    if (n <= SMALL_N) return 256;
    const uint64_t B = 1ull << bucket_bits(n);
    return (size_t)((B + n) * 2 * sizeof(uint32_t)) + 256;
}

// Loads the code of the permutation kernels on the current device.  Under
// CUDA's lazy module loading a kernel's module (and the device memory it
// takes) is otherwise loaded at the kernel's first launch; asking for the
// kernels' attributes loads it now.
cudaError_t preload_permute()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, k_perm_count);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_perm_scan);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_perm_scatter);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_perm_rank);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_perm_small);
    return e;
}

// n < 2^32 - 1 (the callers check)
cudaError_t launch_permute(const float* in, uint64_t n, uint64_t seed, float* out, void* scratch,
                           cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    if (n > 0xFFFFFFFFull) return cudaErrorInvalidValue;
    if (n <= SMALL_N) {
        count_launches(1);
        k_perm_small<<<1, SMALL_T, 0, s>>>(in, (uint32_t)n, seed, out);
        return cudaGetLastError();
    }
    const int bits = bucket_bits(n), shift = 64 - bits;
    const uint32_t B = 1u << bits;
    uint32_t* count = reinterpret_cast<uint32_t*>(scratch);        // [B], 16-byte aligned
    uint32_t* begin = count + B;
    uint32_t* slot = begin + B;
    uint32_t* idx = slot + n;
    cudaError_t e = cudaMemsetAsync(count, 0, (size_t)B * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((n + SORT_T - 1) / SORT_T);
    count_launches(4);
    k_perm_count<<<grid, SORT_T, 0, s>>>((uint32_t)n, seed, shift, count, slot);
    k_perm_scan<<<(B + SCAN_TILE - 1) / SCAN_TILE, SCAN_THREADS, 0, s>>>(count, B, begin);
    k_perm_scatter<<<grid, SORT_T, 0, s>>>((uint32_t)n, seed, shift, begin, slot, idx);
    k_perm_rank<<<grid, SORT_T, 0, s>>>(in, (uint32_t)n, seed, shift, begin, count, idx, out);
    return cudaGetLastError();
}

}  // namespace bfi
