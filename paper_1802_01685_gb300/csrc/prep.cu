// Series preparation on the device.
//
// (1) Split rows for the tensor-core path.  Row w holds the eight samples
//     x[w .. w+7] rounded to bf16 (hi) and the bf16 rounding of the remainder
//     x - hi (lo; x - hi is exact in FP32).  Consecutive rows overlap by seven
//     samples, so the 8-row x 8-sample core matrix that starts at row w is the
//     Hankel block x[w + i + c] (i, c < 8) stored as 128 contiguous bytes: the
//     correlation kernel feeds it to tcgen05.mma as the lag operand with 16-byte
//     row pitch and no gather.  Rows past the series read zeros.
// (2) Inverse window norms.  S[n] = sum_{i<n} x[i]^2 in FP64 (every x^2 of an
//     FP32 sample is exact in FP64), nu(tau) = S[tau+M] - S[tau], and
//     inv(tau) = 1 / sqrt(nu) rounded to FP32.  A window without a nonzero
//     sample gets exactly 0 (rho := 0 there): an exact count prefix C[n] of
//     nonzero samples decides it, because the block-wise scan sums the energy
//     prefix in different orders on either side of a block edge, so S may
//     differ by rounding across an all-zero window.
//
// Four launches for up to 64 series: block sums, their scan, prefix, norms and
// rows.  What bounds them on the usual 10^4 to 10^5 samples is FP64
// issue on the few SMs that hold the blocks -- GB300 runs a warp's FP64
// instruction in 16 cycles -- and the launches themselves.  So a sample costs
// one conversion and one FMA per pass (x^2 is exact, so the FMA rounds as the
// addition would), counts are integers, the blocks are small (1024 samples),
// and 1/sqrt starts from the FP32 one.  With the clearing of the outputs in one
// launch a 4 s search of 256 templates went from 183 to 171 us, a served mix of
// six requests (prepared one by one) from 3.61 to 3.50 ms.
#include <algorithm>

#include "bf_internal.h"

namespace bfi {

// ---------------------------------------------------------------- FP64 scan
constexpr int SCAN_T = 256;              // threads per scan block
constexpr int SCAN_E = 4;                // elements per thread
constexpr int SCAN_B = SCAN_T * SCAN_E;  // elements per block

// block-sum scratch (doubles): energies and nonzero counts of every scan block
uint64_t inv_norm_scratch_blocks(uint64_t N) { return 2 * ((N + SCAN_B - 1) / SCAN_B + 1); }

// sum over the block's threads, in every thread (sh: one word per warp; ends
// with a barrier before which sh is read)
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    T tot = sh[0];
#pragma unroll
    for (int w = 1; w < SCAN_T / 32; ++w) tot += sh[w];
    __syncthreads();
    return tot;
}

// exclusive scan over the block's threads.  A thread's result holds only the
// threads before it: taking its own part off an inclusive total would leave that
// part's rounding in it, and S[t] must not depend on x[t ..] (quiet data before
// loud data).
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* sh, T* total = nullptr)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) sh[wid] = inc;
    T ex = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) ex = T(0);
    __syncthreads();
    T base = T(0), all = T(0);
#pragma unroll
    for (int w = 0; w < SCAN_T / 32; ++w) {
        if (w == wid) base = all;
        all += sh[w];
    }
    if (total) *total = all;
    __syncthreads();
    return base + ex;
}

__device__ __forceinline__ uint32_t* block_counts(double* bsum, uint64_t nb) { return reinterpret_cast<uint32_t*>(bsum + nb); }

// this thread's SCAN_E samples of scan block blockIdx.x (zero past N)
__device__ __forceinline__ void load_samples(const float* __restrict__ x, uint64_t N, float (&v)[SCAN_E])
{
    const uint64_t base = (uint64_t)blockIdx.x * SCAN_B + (uint64_t)threadIdx.x * SCAN_E;
    static_assert(SCAN_E == 4, "one 16-byte load");
    if (base + SCAN_E <= N) {
        const float4 f = *reinterpret_cast<const float4*>(x + base);
        v[0] = f.x;
        v[1] = f.y;
        v[2] = f.z;
        v[3] = f.w;
    } else {
#pragma unroll
        for (int e = 0; e < SCAN_E; ++e) v[e] = base + e < N ? x[base + e] : 0.f;
    }
}

// Per-block sums of x^2 (FP64) and counts of nonzero samples of series
// s = blockIdx.y.  The same launch zeroes the series' padding x[N, xcap) and its
// max |x| word.
__global__ void __launch_bounds__(SCAN_T) k_block_sq(const __grid_constant__ PrepBatch b)
{
    __shared__ double sh[SCAN_T / 32];
    __shared__ uint32_t shc[SCAN_T / 32];
    const int s = blockIdx.y;
    if (s >= b.n) return;
    const uint64_t N = b.N[s], nb = b.nb[s];
    for (uint64_t i = N + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < b.xcap[s];
         i += (uint64_t)gridDim.x * blockDim.x)
        b.x[s][i] = 0.f;
    if (b.mode == 2 && blockIdx.x == 0 && threadIdx.x == 0) *b.xmax[s] = 0u;
    if (blockIdx.x >= nb) return;
    float x[SCAN_E];
    load_samples(b.x[s], N, x);
    double v = 0.0;
    uint32_t c = 0;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e) {
        const double d = (double)x[e];
        v = fma(d, d, v);
        c += x[e] != 0.f ? 1u : 0u;
    }
    const double tot = block_sum(v, sh);
    const uint32_t ctot = block_sum(c, shc);
    if (threadIdx.x == 0) {
        b.bsum[s][blockIdx.x] = tot;
        block_counts(b.bsum[s], nb)[blockIdx.x] = ctot;
    }
}

// exclusive scan of n block sums, in place, E of them a thread and round
template <int E>
__device__ __forceinline__ void scan_sums(double* energy, uint32_t* count, uint64_t n, double* sh, uint32_t* shc)
{
    double carry = 0.0;
    uint32_t ccarry = 0;
    for (uint64_t c0 = 0; c0 < n; c0 += SCAN_T * E) {
        const uint64_t i0 = c0 + (uint64_t)threadIdx.x * E;
        double v[E], t = 0.0, tot;
        uint32_t c[E], ct = 0, ctot;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = i0 + e < n ? energy[i0 + e] : 0.0;
            c[e] = i0 + e < n ? count[i0 + e] : 0u;
            t += v[e];
            ct += c[e];
        }
        double ex = carry + block_excl_scan(t, sh, &tot);
        uint32_t cx = ccarry + block_excl_scan(ct, shc, &ctot);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (i0 + e < n) {
                energy[i0 + e] = ex;
                count[i0 + e] = cx;
            }
            ex += v[e];
            cx += c[e];
        }
        carry += tot;
        ccarry += ctot;
    }
}

// The block sums of series blockIdx.y, by one block: a round's time is its
// barriers', so past SCAN_T of them (262,144 samples) a thread takes 16 and the
// rounds are as many times fewer.  A search of 64 short templates over 10^7 samples
// takes 1.707 ms (1.772 with one a thread), over 4 x 10^8 64.7 (67.5).
__global__ void __launch_bounds__(SCAN_T) k_scan_sums(const __grid_constant__ PrepBatch b)
{
    __shared__ double sh[SCAN_T / 32];
    __shared__ uint32_t shc[SCAN_T / 32];
    const int s = blockIdx.y;
    if (s >= b.n) return;
    const uint64_t n = b.nb[s];
    double* energy = b.bsum[s];
    uint32_t* count = block_counts(energy, n);
    if (n <= (uint64_t)SCAN_T) scan_sums<1>(energy, count, n, sh, shc);
    else scan_sums<16>(energy, count, n, sh, shc);
}

// S[t] = sum_{i < t} x_i^2 and C[t] = #{i < t : x_i != 0}, t = 0..N, of
// series blockIdx.y; mode 2 also max |x| as float bits (non-negative floats
// order like unsigned integers) into *xmax (zeroed by k_block_sq)
__global__ void __launch_bounds__(SCAN_T) k_prefix(const __grid_constant__ PrepBatch b)
{
    __shared__ double sh[SCAN_T / 32];
    __shared__ uint32_t shc[SCAN_T / 32];
    const int s = blockIdx.y;
    if (s >= b.n || blockIdx.x >= b.nb[s]) return;
    const uint64_t N = b.N[s], nb = b.nb[s];
    double* S = b.S[s];
    uint32_t* C = reinterpret_cast<uint32_t*>(S + N + 1);
    float x[SCAN_E];
    load_samples(b.x[s], N, x);
    double t = 0.0;
    uint32_t c = 0;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e) {
        const double d = (double)x[e];
        t = fma(d, d, t);
        c += x[e] != 0.f ? 1u : 0u;
    }
    double ex = block_excl_scan(t, sh) + b.bsum[s][blockIdx.x];
    uint32_t cx = block_excl_scan(c, shc) + block_counts(b.bsum[s], nb)[blockIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S[0] = 0.0;
        C[0] = 0u;
    }
    const uint64_t at = (uint64_t)blockIdx.x * SCAN_B + (uint64_t)threadIdx.x * SCAN_E;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e) {
        const double d = (double)x[e];
        ex = fma(d, d, ex);
        cx += x[e] != 0.f ? 1u : 0u;
        if (at + e < N) {
            S[at + e + 1] = ex;
            C[at + e + 1] = cx;
        }
    }
    if (b.mode == 2) {
        uint32_t m = 0;
#pragma unroll
        for (int e = 0; e < SCAN_E; ++e) m = max(m, __float_as_uint(fabsf(x[e])));
        m = __reduce_max_sync(0xffffffffu, m);
        if ((threadIdx.x & 31) == 0) atomicMax(b.xmax[s], m);
    }
}

// 1/sqrt(m) for m in [1, 4) in FP64: from FP32's value y with h = 1 - m y^2, which
// is rounded once (y^2 is exact), y (1 - h)^(-1/2) = y (1 + h/2 + 3 h^2/8 + ...).
// |h| <= 2^-20, so the series ends below 2^-61 of the value: closer than the
// FP64 root and division that it stands for, in five instructions of the slow pipe.
__device__ __forceinline__ double inv_root(double m)
{
    const double y = (double)rsqrtf((float)m);
    const double h = fma(-m, y * y, 1.0);
    return fma(y, h * fma(0.375, h, 0.5), y);
}

// 1/sqrt(nu) for nu > 0, rounded to FP32 from FP64: of nu's mantissa with an even
// exponent, scaled back exactly.  Energies outside 2^+-240 (the result would leave
// the range of normal floats) take the FP64 root and division.
__device__ __forceinline__ float inv_sqrt(double nu)
{
    const int hi = __double2hiint(nu);
    const int e = ((hi >> 20) - 1023) & ~1;               // even exponent
    if (e < -240 || e > 240) return (float)(1.0 / sqrt(nu));
    const double m = __hiloint2double(hi - (e << 20), __double2loint(nu));
    return (float)inv_root(m) * __int_as_float((127 - e / 2) << 23);       // 2^(-e/2)
}

// Norms and split rows of series blockIdx.y, one index per thread.
// Norms: 1 / |window|, and exactly 0 for a window without a nonzero sample
// (rho := 0 there).  The count decides emptiness: a difference of FP64 prefix
// sums formed in different orders need not vanish over an all-zero window.
// The prefix difference S[t+M] - S[t] carries an absolute rounding error of a
// few ulps of S[t+M]; where the window holds less than 2^-30 of the energy
// before it (a quiet stretch after loud data) that would be a relative error
// above ~5e-6, so such windows are summed directly (x^2 is exact in FP64).
// The first thread of a series also reports a non-finite series: the FP64
// total of x^2 (at most 2^32 squares of floats, far below the FP64 range) is
// finite exactly when every sample is.
// Rows (mode 1 and 2): row w holds x[w .. w+7] (zero past N), in mode 2 as FP16
// of x 2^e: hi = fp16(x 2^e), lo = fp16(x 2^e - hi) (exact difference in FP32),
// e from the series' max |x|.
__global__ void k_norms_rows(const __grid_constant__ PrepBatch b)
{
    const int s = blockIdx.y;
    if (s >= b.n) return;
    const float* x = b.x[s];
    const uint32_t M = b.M;
    const uint64_t N = b.N[s], L = N - M + 1, rows = b.mode ? b.rows[s] : 0;
    const double* S = b.S[s];
    const uint32_t* C = reinterpret_cast<const uint32_t*>(S + N + 1);
    float* inv = b.inv[s];
    uint4* yhi = b.yhi[s];
    uint4* ylo = b.ylo[s];
    const float scale = b.mode == 2 ? ldexpf(1.f, f16_series_shift(*b.xmax[s])) : 1.f;
    if (b.status[s] && blockIdx.x == 0 && threadIdx.x == 0 && !isfinite(S[N])) atomicOr(b.status[s], 1u);
    const uint64_t n = rows > L ? rows : L;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < n;
         t += (uint64_t)gridDim.x * blockDim.x) {
        if (t < L) {
            const double end = S[t + M];
            double nu = end - S[t];
            const bool any = C[t + M] != C[t];
            if (any && nu < end * 0x1p-30) {
                double acc = 0.0;
                for (uint32_t m = 0; m < M; ++m) {
                    const double v = (double)x[t + m];
                    acc = fma(v, v, acc);
                }
                nu = acc;
            }
            inv[t] = (any && nu > 0.0) ? inv_sqrt(nu) : 0.f;
        }
        if (t >= rows) continue;
        uint32_t h[4], l[4];
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
            const float v0 = ((t + c < N) ? x[t + c] : 0.f) * scale;
            const float v1 = ((t + c + 1 < N) ? x[t + c + 1] : 0.f) * scale;
            if (b.mode == 1) {
                const __nv_bfloat16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
                const __nv_bfloat16 l0 = __float2bfloat16_rn(v0 - __bfloat162float(h0));
                const __nv_bfloat16 l1 = __float2bfloat16_rn(v1 - __bfloat162float(h1));
                h[c / 2] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                l[c / 2] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            } else {
                const __half h0 = __float2half_rn(v0), h1 = __float2half_rn(v1);
                const __half l0 = __float2half_rn(v0 - __half2float(h0));
                const __half l1 = __float2half_rn(v1 - __half2float(h1));
                h[c / 2] = (uint32_t)__half_as_ushort(h0) | ((uint32_t)__half_as_ushort(h1) << 16);
                l[c / 2] = (uint32_t)__half_as_ushort(l0) | ((uint32_t)__half_as_ushort(l1) << 16);
            }
        }
        yhi[t] = make_uint4(h[0], h[1], h[2], h[3]);
        ylo[t] = make_uint4(l[0], l[1], l[2], l[3]);
    }
}

size_t prefix_bytes(uint64_t N) { return (N + 1) * (sizeof(double) + sizeof(uint32_t)); }

uint64_t prep_scan_blocks(uint64_t N) { return (N + SCAN_B - 1) / SCAN_B; }

cudaError_t launch_prep(const PrepBatch& b, cudaStream_t st)
{
    if (b.n <= 0 || b.n > MAX_PREP) return cudaErrorInvalidValue;
    uint64_t nb = 0, work = 0;
    for (int i = 0; i < b.n; ++i) {
        if (b.N[i] < b.M || b.nb[i] != prep_scan_blocks(b.N[i]) || b.nb[i] == 0) return cudaErrorInvalidValue;
        nb = std::max(nb, b.nb[i]);
        work = std::max(work, std::max(b.N[i] - b.M + 1, b.mode ? b.rows[i] : 0));
    }
    const unsigned ny = (unsigned)b.n;
    const unsigned bx = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((work + 255) / 256, 65535ull * 16));
    count_launches(4);
    k_block_sq<<<dim3((unsigned)nb, ny), SCAN_T, 0, st>>>(b);
    k_scan_sums<<<dim3(1, ny), SCAN_T, 0, st>>>(b);
    k_prefix<<<dim3((unsigned)nb, ny), SCAN_T, 0, st>>>(b);
    k_norms_rows<<<dim3(bx, ny), 256, 0, st>>>(b);
    return cudaGetLastError();
}

}  // namespace bfi
