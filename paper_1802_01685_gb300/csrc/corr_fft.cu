// Correlation by FFT: the paper's own route to the filter output (Sect. 2.2
// and Fig. 5: the output of every template against data segments through
// single-precision FFTs on the GPU, with only the tails rho > kappa sigma
// leaving the device).  Overlap-save: with segments of F samples,
//
//   segment j of a series covers lags tau0 = j V .. tau0 + V - 1, V = F - M + 1,
//   X_j = DFT_F(x[tau0 .. tau0 + F))             (zero past the series end)
//   H_k = DFT_F(h_k zero-padded to F)
//   c_k[tau0 + t] = (1/F) sum_f X_j[f] conj(H_k[f]) e^{+2 pi i f t / F},  t < V,
//
// which is the circular correlation of the segment with the padded template;
// for t < V no product wraps around, so it equals the direct sum
// sum_m h_k[m] x[tau0 + t + m].  The result is normalised by the window norm
// and reduced exactly like the direct kernels (max |rho| with its first
// argmax, sum rho^2, tails).
//
// Every transform here is a complex FFT of N = 8192 points in one CTA.  Two
// ways of using it:
//  * the real route (plain banks): segments of F = 2N = 16384 samples.  The
//    real input of length F is packed as N complex values (even samples in
//    the real part, odd in the imaginary) and the half spectra of N + 1 bins
//    are separated from the complex transform by the usual even/odd split; the
//    inverse runs the same way backwards: the N complex outputs of one inverse
//    transform are the correlation at 2N consecutive lags of ONE template.
//    At M = 4096 that is 12289 useful lags per transform.
//  * the pair route (quadrature banks): segments of F = N = 8192 samples and
//    a template with its quadrature partner in one complex transform, output
//    |c_cos + i c_sin| at the V = 8193 - M lags of the segment.
//
// GB300 layout of the work:
//  * template spectra are kept by a stored bank in HBM (made once) and made
//    per call for a generated bank, chunk by chunk, in a two-slot ring on the
//    auxiliary stream;
//  * each segment spectrum is computed once per call; all of them stay in L2,
//    and so do the segments' window norms, and go straight into registers;
//  * the forward transforms (segments, templates, the predictor) are Stockham
//    autosort FFTs of one CTA with three radix-16 passes (each thread one
//    16-point DFT per pass, in registers) and a final radix-2 stage; the work
//    array holds index i at i + i/16, so that every pass moves a warp's 64-bit
//    values in the minimum two wavefronts.  Twiddles: the second pass reads a
//    [15][16] table, the third reads e^{2 pi i r k / 4096} for r = 1, 2, 3, 4, 8, 12
//    and forms the others as one product of two; the last stage and the real
//    route's even/odd split use per-thread constants (rounded from FP64 once
//    per thread) times exact-to-rounding roots of unity;
//  * the inverse transforms, nearly all of the work, are k_corr_fft's: the
//    product with a template's spectrum, the transform and the reduction of its
//    output in one kernel, so that the filter output never reaches HBM.
//  * The transform's rounding error scales with its whole segment, so lags
//    whose window holds almost none of the segment's energy are taken out of
//    the FFT route (k_fft_flags) and computed directly (k_fft_fixup).
#include "corr_common.cuh"
#include "device_once.h"
#include "synth.cuh"
#include "runtime.h"

namespace bfi {

namespace {

constexpr int FN = FFT_POINTS;            // 8192 complex points per transform
constexpr int FH = FN / 2;                // 4096
constexpr int FR = 2 * FN;                // 16384 samples per segment of the real route
constexpr int FT = 512;                   // threads per FFT block
constexpr int FBINS = FH / FT;            // 8 bins per thread (and their 8 mirrors)
constexpr int ZPAD = FN + FN / 16;        // padded complex values of the work array
constexpr int ROW = FT + FT / 16;         // padded distance of elements 512 apart (544)
constexpr int UPPER = FH + FH / 16;       // padded distance of elements 4096 apart (4352)
// twiddle tables e^{+2 pi i n / 8192}: pass 2 [15][16] (r (j mod 16) units of
// 32), pass 3 [6][256] (r (j mod 256) units of 2 for r = 1, 2, 3, 4, 8, 12)
constexpr int TW2 = 0, TW3 = 15 * 16, TW_N = TW3 + 6 * 256;     // 1776 entries
// shared memory of the forward transforms: work array, twiddles, then (template
// spectra of the real route only) a second work array, so that the passes
// alternate between the two, and the staged row
constexpr size_t FFT_SMEM = (ZPAD + TW_N) * sizeof(float2);
constexpr size_t BANK_SMEM = FFT_SMEM + ZPAD * sizeof(float2) + FH * sizeof(float2);
static_assert(FFT_SMEM % 16 == 0 && (FFT_SMEM + ZPAD * sizeof(float2)) % 16 == 0, "16-byte staging");
// the correlation kernel: two groups of GT threads, each with a work array of
// 16 blocks of 16 rows of 16 packed values at a pitch of 17 (so that the last
// pass, whose threads differ in the row, meets no bank conflict), a template's
// records, and twiddles: [6][256] of pass 1, e^{2 pi i q j / 4096} for q = 1, 2,
// 3, 4, 8, 12, [15][16] of pass 2, e^{2 pi i q n / 256}, and [256][2] of the
// product, e^{i pi j / 8192} and e^{i pi j / 4096}
constexpr int GT = FT / 2;
constexpr int ZROW = 17, ZBLK = 16 * ZROW, ZG = 16 * ZBLK;
constexpr int TWC_N = 6 * 256 + 15 * 16 + 2 * 256;          // float2 entries, after the TW_N of the forward transforms
// 2 x 9: column 0; the warps' max keys; two mbarriers; the threads' sums; the abort flag
constexpr int CORR_ACC = 2 * ZG + FH + TWC_N / 2 + 2 * 9;
constexpr size_t CORR_SMEM = (size_t)(CORR_ACC + FT / 64 + 1 + FT / 2 + 1) * sizeof(float4);
static_assert(CORR_SMEM <= 227 * 1024, "the correlation kernel fits one SM's shared memory");
static_assert(TW_N % 2 == 0 && TWC_N % 2 == 0, "16-byte tables");

__global__ void k_fft_tables(float2* __restrict__ tw)
{
    // the correlation kernel's tables
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < TWC_N; e += gridDim.x * blockDim.x) {
        double a;                                 // the angle over pi
        if (e < 6 * 256) {
            const int q = e / 256;
            a = (double)((q < 3 ? q + 1 : 4 * (q - 2)) * (e % 256)) / 2048.0;
        } else if (e < 6 * 256 + 15 * 16) {
            a = (double)(((e - 6 * 256) / 16 + 1) * (e % 16)) / 128.0;
        } else {
            const int i = e - 6 * 256 - 15 * 16;
            a = (double)(i / 2) / (i % 2 ? 4096.0 : 8192.0);
        }
        double sn, cs;
        sincospi(a, &sn, &cs);
        tw[TW_N + e] = make_float2((float)cs, (float)sn);
    }
    // the forward transforms' per-thread constants
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 2 * FT; e += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi((double)(e / 2) / (e % 2 ? 4096.0 : 8192.0), &sn, &cs);
        tw[TW_N + TWC_N + e] = make_float2((float)cs, (float)sn);
    }
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < TW_N; e += gridDim.x * blockDim.x) {
        int n;                                    // exponent in units of 2 pi / 8192
        if (e < TW3) {
            n = ((e - TW2) / 16 + 1) * ((e - TW2) % 16) * 32;
        } else {
            const int q = (e - TW3) / 256, k = (e - TW3) % 256;
            const int r = q < 4 ? q + 1 : 4 * (q - 2);           // 1, 2, 3, 4, 8, 12
            n = r * k * 2;
        }
        double sn, cs;
        sincospi((double)n / 4096.0, &sn, &cs);
        tw[e] = make_float2((float)cs, (float)sn);
    }
}

// Work array z (complex, index i stored at i + i/16), twiddle tables, and, for the
// template spectra of the real route (TWO), a second work array z2 and the staged
// row x.
struct Smem {
    float2* z;
    const float2* tw;
    float2* z2;
    float2* x;
};

template <bool TWO>
__device__ __forceinline__ Smem smem_setup(const float2* __restrict__ tw_global)
{
    extern __shared__ __align__(16) float2 fsm[];
    Smem m{fsm, fsm + ZPAD, TWO ? fsm + ZPAD + TW_N : nullptr, TWO ? fsm + 2 * ZPAD + TW_N : nullptr};
    float4* dst = reinterpret_cast<float4*>(fsm + ZPAD);
    const float4* src = reinterpret_cast<const float4*>(tw_global);
    for (int i = threadIdx.x; i < TW_N / 2; i += blockDim.x) dst[i] = __ldg(src + i);
    __syncthreads();
    return m;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

// waits until at most N of this thread's most recent groups are in flight
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

template <int SIGN>
__device__ __forceinline__ float2 tw_get(const float2* t, int e)
{
    const float2 w = t[e];
    return make_float2(w.x, SIGN > 0 ? w.y : -w.y);
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ void rotate(float& r, float& i, float2 w)
{
    const float a = r * w.x - i * w.y;
    i = r * w.y + i * w.x;
    r = a;
}

// e^{i pi a / 16} for a compile-time a in [0, 16): cos(pi a/16) for a <= 8 is
// C[a], past 8 it is -C[16 - a]; sin(pi a/16) is C[8 - a], past 8 C[a - 8]
__device__ __forceinline__ float2 root32(int a)
{
    const float C[9] = {1.0f, 0.9807852804032304491262f, 0.9238795325112867561282f,
                        0.8314696123025452370788f, 0.7071067811865475244008f,
                        0.5555702330196022247428f, 0.3826834323650897717285f,
                        0.1950903220161282678483f, 0.0f};
    return a <= 8 ? make_float2(C[a], C[8 - a]) : make_float2(-C[16 - a], C[a - 8]);
}

// this thread's constants e^{i pi tid / 8192} (.x, .y) and e^{i pi tid / 4096}
// (.z, .w), rounded from FP64 in the tables: computed here they were most of
// the 16 us that one transform took (GB300's FP64 rate)
__device__ __forceinline__ float4 thread_roots(const float2* __restrict__ tw)
{
    return __ldg(reinterpret_cast<const float4*>(tw + TW_N + TWC_N) + threadIdx.x);
}

// 4-point DFT with kernel e^{SIGN 2 pi i n k / 4}, in place
template <int SIGN>
__device__ __forceinline__ void dft4(float& ar, float& ai, float& br, float& bi, float& cr, float& ci,
                                     float& dr, float& di)
{
    const float t0r = ar + cr, t0i = ai + ci;
    const float t1r = ar - cr, t1i = ai - ci;
    const float t2r = br + dr, t2i = bi + di;
    const float t3r = br - dr, t3i = bi - di;
    const float ur = SIGN > 0 ? -t3i : t3i;       // SIGN * i * (b - d)
    const float ui = SIGN > 0 ? t3r : -t3r;
    ar = t0r + t2r;
    ai = t0i + t2i;
    cr = t0r - t2r;
    ci = t0i - t2i;
    br = t1r + ur;
    bi = t1i + ui;
    dr = t1r - ur;
    di = t1i - ui;
}

// 16-point DFT as 4 x 4 (Cooley-Tukey, n = 4 n1 + n2, k = k1 + 4 k2): DFTs
// over n1, twiddles e^{SIGN 2 pi i n2 k1 / 16}, DFTs over n2.  On return
// position 4 k1 + k2 holds output k1 + 4 k2.
template <int SIGN>
__device__ __forceinline__ void dft16(float (&r)[16], float (&i)[16])
{
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2)
        dft4<SIGN>(r[n2], i[n2], r[4 + n2], i[4 + n2], r[8 + n2], i[8 + n2], r[12 + n2], i[12 + n2]);
    constexpr float C1 = 0.923879532511286756f;   // cos(pi/8)
    constexpr float S1 = 0.382683432365089772f;   // sin(pi/8)
    constexpr float R2 = 0.707106781186547524f;   // cos(pi/4)
    constexpr float S = SIGN > 0 ? 1.f : -1.f;
    // position 4 k1 + n2 gets e^{SIGN 2 pi i (n2 k1) / 16}
    rotate(r[5], i[5], make_float2(C1, S * S1));      // n2 k1 = 1
    rotate(r[9], i[9], make_float2(R2, S * R2));      // 2
    rotate(r[13], i[13], make_float2(S1, S * C1));    // 3
    rotate(r[6], i[6], make_float2(R2, S * R2));      // 2
    rotate(r[10], i[10], make_float2(0.f, S));        // 4
    rotate(r[14], i[14], make_float2(-R2, S * R2));   // 6
    rotate(r[7], i[7], make_float2(S1, S * C1));      // 3
    rotate(r[11], i[11], make_float2(-R2, S * R2));   // 6
    rotate(r[15], i[15], make_float2(-C1, -S * S1));  // 9
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
        dft4<SIGN>(r[4 * k1], i[4 * k1], r[4 * k1 + 1], i[4 * k1 + 1], r[4 * k1 + 2], i[4 * k1 + 2],
                   r[4 * k1 + 3], i[4 * k1 + 3]);
}

// One radix-16 Stockham pass over 8192 points with stride NS (1, 16, 256):
// thread j reads in[j + 512 r], twiddles by e^{SIGN 2 pi i r (j mod NS) / (16 NS)},
// takes the 16-point DFT and writes out[(j / NS) 16 NS + j mod NS + q NS].
// Padded addresses (i + i/16) are a per-thread base plus constant offsets.
// The second half of a pass, from the 16 inputs already in registers, into
// the work array dst; it ends with a barrier.
template <int SIGN, int NS>
__device__ __forceinline__ void pass16_from(const Smem& m, float2* dst, float (&vr)[16], float (&vi)[16])
{
    const int j = threadIdx.x;
    if (NS == 16) {
        const float2* t = m.tw + TW2 + (j % 16);
#pragma unroll
        for (int r = 1; r < 16; ++r) rotate(vr[r], vi[r], tw_get<SIGN>(t, (r - 1) * 16));
    } else if (NS == 256) {
        // e^{2 pi i r k / 4096}, k = j mod 256, from r = 1, 2, 3, 4, 8, 12
        const float2* t = m.tw + TW3 + (j % 256);
        const float2 w1 = tw_get<SIGN>(t, 0), w2 = tw_get<SIGN>(t, 256), w3 = tw_get<SIGN>(t, 512);
        const float2 w4 = tw_get<SIGN>(t, 768), w8 = tw_get<SIGN>(t, 1024), w12 = tw_get<SIGN>(t, 1280);
        rotate(vr[1], vi[1], w1);
        rotate(vr[2], vi[2], w2);
        rotate(vr[3], vi[3], w3);
        rotate(vr[4], vi[4], w4);
        rotate(vr[5], vi[5], cmul(w4, w1));
        rotate(vr[6], vi[6], cmul(w4, w2));
        rotate(vr[7], vi[7], cmul(w4, w3));
        rotate(vr[8], vi[8], w8);
        rotate(vr[9], vi[9], cmul(w8, w1));
        rotate(vr[10], vi[10], cmul(w8, w2));
        rotate(vr[11], vi[11], cmul(w8, w3));
        rotate(vr[12], vi[12], w12);
        rotate(vr[13], vi[13], cmul(w12, w1));
        rotate(vr[14], vi[14], cmul(w12, w2));
        rotate(vr[15], vi[15], cmul(w12, w3));
    }
    dft16<SIGN>(vr, vi);
    int wb;                                       // padded address of output q = 0
    if (NS == 1) wb = 17 * j;
    else if (NS == 16) wb = (j / 16) * 272 + (j % 16);
    else wb = (j / 256) * 4352 + (j % 256) + ((j % 256) >> 4);
#pragma unroll
    for (int p = 0; p < 16; ++p) {
        const int q = 4 * (p % 4) + p / 4;
        const int off = NS == 1 ? q : NS == 16 ? 17 * q : 272 * q;
        dst[wb + off] = make_float2(vr[p], vi[p]);
    }
    __syncthreads();
}

// A pass from work array src to dst; in place (src == dst) every thread's
// reads complete at a barrier before the first write.
template <int SIGN, int NS, bool IN_PLACE = true>
__device__ __forceinline__ void pass16(const Smem& m, const float2* src, float2* dst)
{
    const int j = threadIdx.x;
    const int rd = j + (j >> 4);
    float vr[16], vi[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const float2 v = src[rd + ROW * r];
        vr[r] = v.x;
        vi[r] = v.y;
    }
    if (IN_PLACE) __syncthreads();
    pass16_from<SIGN, NS>(m, dst, vr, vi);
}

template <int SIGN>
__device__ __forceinline__ void fft_passes(const Smem& m)
{
    pass16<SIGN, 1>(m, m.z, m.z);
    pass16<SIGN, 16>(m, m.z, m.z);
    pass16<SIGN, 256>(m, m.z, m.z);
}

// twiddle e^{SIGN i pi k / 4096} of the final radix-2 stage for k = tid + 512 i
// (base_f = e^{i pi tid / 4096})
template <int SIGN>
__device__ __forceinline__ float2 final_tw(float2 base_f, int i)
{
    const float2 w = cmul(base_f, root32(2 * i));
    return make_float2(w.x, SIGN > 0 ? w.y : -w.y);
}

// The final radix-2 stage for output pair (k, k + 4096), k = tid + 512 i, with
// its twiddle w = final_tw<SIGN>(base_f, i), from the work array z.
__device__ __forceinline__ void fft_final(const float2* z, int i, float2 w, float2& lo, float2& hi)
{
    const int a = threadIdx.x + (threadIdx.x >> 4) + ROW * i;
    const float2 v = z[a + UPPER];
    float vr = v.x, vi = v.y;
    rotate(vr, vi, w);
    const float2 u = z[a];
    lo = make_float2(u.x + vr, u.y + vi);
    hi = make_float2(u.x - vr, u.y - vi);
}

// Z[8192 - k] = the upper output of the final stage at 4096 - k, 1 <= k < 4096,
// whose twiddle e^{SIGN i pi (4096 - k) / 4096} is -conj(w), w that of k
__device__ __forceinline__ float2 fft_final_mirror(const float2* z, int k, float2 w)
{
    const int kk = FH - k;
    const int a = kk + (kk >> 4);
    const float2 v = z[a + UPPER];
    float vr = v.x, vi = v.y;
    rotate(vr, vi, make_float2(-w.x, w.y));
    const float2 u = z[a];
    return make_float2(u.x - vr, u.y - vi);
}

// Half spectrum of a real signal s of F = 16384 samples from the complex
// transform U of u[n] = s[2n] + i s[2n+1] (in the work array after
// fft_passes<-1>): with E = (U[k] + conj U[N-k]) / 2 and
// O = (U[k] - conj U[N-k]) / 2i the transforms of the even and odd samples,
//   S[k] = E + e^{-i pi k / N} O,   S[N - k] = conj(E - e^{-i pi k / N} O),
//   S[N/2] = conj(U[N/2]),  S[0] = E_0 + O_0,  S[N] = E_0 - O_0 (real).
// Calls emit(i, slot, k, S[k]) for this thread's bins: slot 0 for
// k = tid + 512 i, slot 1 for N - k (i < 8); thread 0, i = 0 emits slot 0
// with k = 0 and (S[0], S[N]) packed, and slot 2 with k = N/2.  i is a
// compile-time constant in each call.
template <typename Emit>
__device__ __forceinline__ void real_spectrum(const Smem& m, float2 base_f, float2 base_r, Emit emit)
{
    const int tid = threadIdx.x;
#pragma unroll
    for (int i = 0; i < FBINS; ++i) {
        const int k = tid + FT * i;
        const float2 w = final_tw<-1>(base_f, i);
        float2 zk, zh;
        fft_final(m.z, i, w, zk, zh);                               // U[k], U[k + 4096]
        if (k == 0) {
            emit(i, 0, 0, make_float2(zk.x + zk.y, zk.x - zk.y));
            emit(i, 2, FH, make_float2(zh.x, -zh.y));
        } else {
            const float2 zm = fft_final_mirror(m.z, k, w);         // U[N - k]
            const float2 e = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
            const float2 o = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
            const float2 wr = cmul(base_r, root32(i));            // e^{i pi k / N}
            const float2 wo = cmul(make_float2(wr.x, -wr.y), o);
            emit(i, 0, k, make_float2(e.x + wo.x, e.y + wo.y));
            emit(i, 1, FN - k, make_float2(e.x - wo.x, wo.y - e.y));
        }
    }
}

// U[n], U[n + 4096], U[4096 - n], U[8192 - n] of the complex transform in the
// work array after fft_passes<-1>, n = tid + 512 i, i < 4; for n = 0 the last two
// are U[2048] and U[6144]
__device__ __forceinline__ void quad_bins(const float2* z, float2 base_f, int i, float2 (&u)[4])
{
    const int n = threadIdx.x + FT * i;
    const float2 w = final_tw<-1>(base_f, i);
    fft_final(z, i, w, u[0], u[1]);
    const int m = n ? FH - n : FH / 2;
    const int a = m + (m >> 4);
    const float2 v = z[a + UPPER], c = z[a];
    float vr = v.x, vi = v.y;
    rotate(vr, vi, n ? make_float2(-w.x, w.y) : make_float2(0.f, -1.f));    // e^{-i pi m / 4096}
    u[2] = make_float2(c.x + vr, c.y + vi);
    u[3] = make_float2(c.x - vr, c.y - vi);
}

// The place of column j among a row's 256 records: that of the thread which reads
// it in the correlation kernel, whose lanes 16-31 hold the mirrors of lanes
// 0-15's columns, so that a warp reads 512 bytes in a row.  In the order of j the
// mirrors' 256 bytes lay across three lines, one of them shared with the warp
// beside (3 % on the light curves, 0.5-1 % elsewhere).
__device__ __forceinline__ int record_place(int j)
{
    const int m = j < GT / 2 ? j : GT - j;            // a mirror's column: 1 .. 127; 128 is in the place of 0's
    return j == GT / 2 ? 16 : 32 * (m >> 4) + (j < GT / 2 ? 0 : 16) + (m & 15);
}

__device__ __forceinline__ float4 lanes(float2 a, float2 b) { return make_float4(a.x, b.x, a.y, b.y); }

// S[k] and S[N - k] from U[k] and U[N - k], w = e^{i pi k / N} (real_spectrum)
__device__ __forceinline__ void real_split(float2 uk, float2 um, float2 w, float2& sk, float2& sm)
{
    const float2 e = make_float2(0.5f * (uk.x + um.x), 0.5f * (uk.y - um.y));
    const float2 o = make_float2(0.5f * (uk.y + um.y), -0.5f * (uk.x - um.x));
    const float2 wo = cmul(make_float2(w.x, -w.y), o);
    sk = make_float2(e.x + wo.x, e.y + wo.y);
    sm = make_float2(e.x - wo.x, wo.y - e.y);
}

// The half spectrum of a real signal (as real_spectrum) as the records the
// correlation kernel reads: for n = j + 256 r < 2048, float4 number 2 r 256 +
// record_place(j) holds the bins n and 4096 - n as (re, re, im, im), number
// (2 r + 1) 256 + record_place(j) the bins 8192 - n and 4096 + n; the record of n = 0 holds bin 0 = (S[0], S[N]), bin
// 4096, bin 6144 and bin 2048.
__device__ __forceinline__ void real_spectrum_quads(const Smem& m, float2 base_f, float2 base_r,
                                                    float2* __restrict__ out)
{
    const int tid = threadIdx.x;
    float4* rec = reinterpret_cast<float4*>(out) + 2 * GT * (tid / GT) + record_place(tid % GT);
#pragma unroll
    for (int i = 0; i < FBINS / 2; ++i) {
        float2 u[4], s0, s1, s2, s3;                  // bins n, 4096 - n, 8192 - n, 4096 + n
        quad_bins(m.z, base_f, i, u);
        if (tid == 0 && i == 0) {
            s0 = make_float2(u[0].x + u[0].y, u[0].x - u[0].y);
            s1 = make_float2(u[1].x, -u[1].y);
            constexpr float R2 = 0.707106781186547524f;
            real_split(u[2], u[3], make_float2(R2, R2), s3, s2);
        } else {
            const float2 w = cmul(base_r, root32(i));                        // e^{i pi n / N}
            real_split(u[0], u[3], w, s0, s2);
            real_split(u[2], u[1], make_float2(w.y, w.x), s1, s3);           // e^{i pi (4096 - n) / N}
        }
        rec[4 * GT * i] = lanes(s0, s1);
        rec[4 * GT * i + GT] = lanes(s2, s3);
    }
}

// Spectra of segments of a batch of series, as the correlation kernel's
// records.  Pair route (F = 8192): the real segment through one complex
// transform, 4096 bins: for n = j + 256 r < 2048, float4 number r 256 +
// record_place(j) holds the bins n and 4096 - n (for n = 0: bin 0 = (DC, Nyquist) and bin 2048).  Real
// route (F = 16384): even/odd packed, 8192 bins (real_spectrum_quads).
template <bool REAL>
__global__ void __launch_bounds__(FT, 1) k_fft_series(const __grid_constant__ FftSeriesBatch p,
                                                      uint32_t total)
{
    const Smem m = smem_setup<false>(p.tw);
    const int tid = threadIdx.x;
    if (blockIdx.x == 0 && p.n_fix && tid < p.n) p.n_fix[tid] = 0u;       // k_fft_flags counts from 0
    const float4 roots = thread_roots(p.tw);
    const float2 base_f = make_float2(roots.z, roots.w), base_r = make_float2(roots.x, roots.y);
    for (uint32_t g = blockIdx.x; g < total; g += gridDim.x) {
        int s = 0;
        while (s + 1 < p.n && g >= p.seg_begin[s + 1]) ++s;
        const uint32_t j = g - p.seg_begin[s];
        const float* x = p.x[s];
        const uint64_t N = p.N[s], t0 = (uint64_t)j * p.V;
        if (REAL) {
            for (int n = tid; n < FN; n += FT) {
                const uint64_t a = t0 + 2 * (uint64_t)n;
                m.z[n + (n >> 4)] = make_float2(a < N ? x[a] : 0.f, a + 1 < N ? x[a + 1] : 0.f);
            }
        } else {
            for (int n = tid; n < FN; n += FT) m.z[n + (n >> 4)] = make_float2(t0 + n < N ? x[t0 + n] : 0.f, 0.f);
        }
        __syncthreads();
        fft_passes<-1>(m);
        if (REAL) {
            real_spectrum_quads(m, base_f, base_r, p.spec[s] + (size_t)j * FN);
        } else {
            float4* rec = reinterpret_cast<float4*>(p.spec[s] + (size_t)j * FH) + GT * (tid / GT) + record_place(tid % GT);
#pragma unroll
            for (int i = 0; i < FBINS / 2; ++i) {
                float2 u[4];
                quad_bins(m.z, base_f, i, u);
                rec[FT * i] = lanes(tid == 0 && i == 0 ? make_float2(u[0].x, u[1].x) : u[0], u[2]);
            }
        }
        __syncthreads();
    }
}

// Template spectra of a chunk of synthesised rows (rows of 8192 samples, zero
// past M), pair route: rows (2q, 2q + 1) through one complex transform of
// h_a + i h_b, separated by Hermitian symmetry into two half spectra of 4096
// bins (records as k_fft_series' pair route).
__global__ void __launch_bounds__(FT, 1) k_fft_bank_pair(const float* __restrict__ rows, uint32_t n_rows,
                                                         uint32_t n_items, const float2* __restrict__ tw,
                                                         float2* __restrict__ spec)
{
    const Smem m = smem_setup<false>(tw);
    const int tid = threadIdx.x;
    const float4 roots = thread_roots(tw);
    const float2 base_f = make_float2(roots.z, roots.w);
    for (uint32_t q = blockIdx.x; q < n_items; q += gridDim.x) {
        const uint32_t a = 2 * q, b = a + 1;
        const float* ra = rows + (size_t)a * FN;
        const float* rb = rows + (size_t)b * FN;
        for (int n = tid; n < FN; n += FT) m.z[n + (n >> 4)] = make_float2(ra[n], b < n_rows ? rb[n] : 0.f);
        __syncthreads();
        fft_passes<-1>(m);
        float4* sa = reinterpret_cast<float4*>(spec + (size_t)a * FH) + GT * (tid / GT) + record_place(tid % GT);
        float4* sb = reinterpret_cast<float4*>(spec + (size_t)b * FH) + GT * (tid / GT) + record_place(tid % GT);
#pragma unroll
        for (int i = 0; i < FBINS / 2; ++i) {
            float2 u[4];                           // Z[n], Z[n + 4096], Z[4096 - n], Z[8192 - n]
            quad_bins(m.z, base_f, i, u);
            // H_a = (Z[k] + conj Z[F-k]) / 2,  H_b = (Z[k] - conj Z[F-k]) / 2i
            auto ha = [](float2 k, float2 c) { return make_float2(0.5f * (k.x + c.x), 0.5f * (k.y - c.y)); };
            auto hb = [](float2 k, float2 c) { return make_float2(0.5f * (k.y + c.y), -0.5f * (k.x - c.x)); };
            if (tid == 0 && i == 0) {
                // DC and Nyquist of both real templates: real parts of Z[0], Z[4096]; bin 2048
                sa[0] = lanes(make_float2(u[0].x, u[1].x), ha(u[2], u[3]));
                if (b < n_rows) sb[0] = lanes(make_float2(u[0].y, u[1].y), hb(u[2], u[3]));
            } else {
                sa[FT * i] = lanes(ha(u[0], u[3]), ha(u[2], u[1]));
                if (b < n_rows) sb[FT * i] = lanes(hb(u[0], u[3]), hb(u[2], u[1]));
            }
        }
        __syncthreads();
    }
}

// Template spectra of the real route from synthesised rows (8192 samples each,
// zero past M): one row per transform, even/odd packed into 4096 complex
// values and zero past them (the 16384-sample segment), 8192 bins per row.
// While one row is transformed the next one's first M samples arrive by
// cp.async, and the passes alternate between the two work arrays: four
// barriers per row.  The route takes M <= 4096, so the inputs past the first
// quarter of the transform are zero, and the first pass knows it at compile
// time.
__global__ void __launch_bounds__(FT, 1) k_fft_bank_real(const float* __restrict__ rows, uint32_t n_rows,
                                                         uint32_t M, const float2* __restrict__ tw,
                                                         float2* __restrict__ spec)
{
    const Smem m = smem_setup<true>(tw);
    const int tid = threadIdx.x;
    const float4 roots = thread_roots(tw);
    const float2 base_f = make_float2(roots.z, roots.w), base_r = make_float2(roots.x, roots.y);
    const uint32_t n16 = (M + 3) / 4;             // 16-byte pieces holding a row's first M samples
    const uint32_t mh = 2 * n16;                  // complex values staged (M <= FH: mh <= FH / 2)
    uint32_t q = blockIdx.x;
    if (q >= n_rows) return;
    auto stage = [&](uint32_t r) {
        const float* src = rows + (size_t)r * FN;
        for (uint32_t c = tid; c < n16; c += FT) cp_async16(m.x + 2 * c, src + 4 * c);
    };
    stage(q);
    cp_async_commit();
    for (;;) {
        cp_async_wait<0>();
        __syncthreads();                          // the row staged; the previous spectrum read
        float vr[16], vi[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const uint32_t n = (uint32_t)(tid + FT * r);
            const float2 v = r < FBINS / 2 && n < mh ? m.x[n] : make_float2(0.f, 0.f);
            vr[r] = v.x;
            vi[r] = v.y;
        }
        pass16_from<-1, 1>(m, m.z, vr, vi);       // every thread has read its staged values
        const uint32_t qn = q + gridDim.x;
        if (qn < n_rows) stage(qn);
        cp_async_commit();
        pass16<-1, 16, false>(m, m.z, m.z2);
        pass16<-1, 256, false>(m, m.z2, m.z);
        real_spectrum_quads(m, base_f, base_r, spec + (size_t)q * FN);
        if (qn >= n_rows) break;
        q = qn;
    }
}

// ---- Parseval predictor of sigma (Sect. 2.2, Fig. 5 caption): periodograms
// and template power spectra on the real route's 16384-point transform.

// |S[k]|^2, k = 0 .. N, of this thread's bins into out (N + 1 floats)
__device__ __forceinline__ void real_power_out(const Smem& m, float2 base_f, float2 base_r,
                                               float* __restrict__ out)
{
    real_spectrum(m, base_f, base_r, [&](int, int, int k, float2 v) {
        if (k == 0) {
            out[0] = v.x * v.x;
            out[FN] = v.y * v.y;
        } else {
            out[k] = v.x * v.x + v.y * v.y;
        }
    });
}

// Periodograms of the Welch segments of a batch of series: segment g of
// series s covers samples [g F/2, g F/2 + F), zero past the end; row
// seg_begin[s] + g of pseg gets |S[k]|^2 for k = 0 .. N.
__global__ void __launch_bounds__(FT, 1) k_welch_segments(const __grid_constant__ WelchBatch p, uint32_t total)
{
    const Smem m = smem_setup<false>(p.tw);
    const int tid = threadIdx.x;
    const float4 roots = thread_roots(p.tw);
    const float2 base_f = make_float2(roots.z, roots.w), base_r = make_float2(roots.x, roots.y);
    for (uint32_t g = blockIdx.x; g < total; g += gridDim.x) {
        int s = 0;
        while (s + 1 < p.n && g >= p.seg_begin[s + 1]) ++s;
        const uint64_t N = p.N[s], a0 = (uint64_t)(g - p.seg_begin[s]) * FN;      // hop F/2 = N
        const float* x = p.x[s];
        for (int n = tid; n < FN; n += FT) {
            const uint64_t a = a0 + 2 * (uint64_t)n;
            m.z[n + (n >> 4)] = make_float2(a < N ? x[a] : 0.f, a + 1 < N ? x[a + 1] : 0.f);
        }
        __syncthreads();
        fft_passes<-1>(m);
        real_power_out(m, base_f, base_r, p.pseg + (size_t)g * PRED_BINS);
        __syncthreads();
    }
}

// P_s(k) = c_s / S_s sum_g pseg[g](k) over the S_s segments of series s, the
// sum in FP64 in segment order; c_s = 1, or F / N_s for a series shorter than
// F (one zero-padded segment).  Grid: (bins, series).
__global__ void k_welch_mean(const __grid_constant__ WelchBatch p)
{
    const int s = blockIdx.y;
    if (s >= p.n) return;
    const uint32_t g0 = p.seg_begin[s], S = p.seg_begin[s + 1] - g0;
    const double c = p.N[s] < (uint64_t)PRED_F ? (double)PRED_F / (double)p.N[s] : 1.0;
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < (uint32_t)PRED_BINS; k += gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (uint32_t g = 0; g < S; ++g) acc += (double)p.pseg[(size_t)(g0 + g) * PRED_BINS + k];
        p.P[(size_t)s * PRED_BINS + k] = (float)(acc * c / (double)S);
    }
}

// For template rows q < n_rows of a chunk (8192 samples each, zero past M):
// D[s][row0 + q] = sum over all F bins of P_s(f) |H_q(f)|^2, i.e. the bins
// 0 and N once and the others twice, for each series s < n_ser; the partial
// sums per thread in FP32 (16 terms), across the CTA in FP64.
__global__ void __launch_bounds__(FT, 1) k_template_power_dot(const float* __restrict__ rows, uint32_t n_rows,
                                                              const float2* __restrict__ tw,
                                                              const float* __restrict__ P, uint32_t n_ser,
                                                              float* __restrict__ D, uint32_t d_stride,
                                                              uint32_t row0)
{
    const Smem m = smem_setup<false>(tw);
    __shared__ double red[FT / 32];
    const int tid = threadIdx.x;
    const float4 roots = thread_roots(tw);
    const float2 base_f = make_float2(roots.z, roots.w), base_r = make_float2(roots.x, roots.y);
    for (uint32_t q = blockIdx.x; q < n_rows; q += gridDim.x) {
        const float2* r2 = reinterpret_cast<const float2*>(rows + (size_t)q * FN);
        for (int n = tid; n < FN; n += FT) m.z[n + (n >> 4)] = n < FH ? r2[n] : make_float2(0.f, 0.f);
        __syncthreads();
        fft_passes<-1>(m);
        // this thread's weighted powers: pw[i] at k = tid + 512 i, pm[i] at
        // N - k (thread 0, i = 0: S[0] and S[N], each once); thread 0 also
        // holds the middle bin N/2 in mid
        float pw[FBINS], pm[FBINS], mid = 0.f;
        real_spectrum(m, base_f, base_r, [&](int i, int slot, int k, float2 v) {
            const float a = 2.f * (v.x * v.x + v.y * v.y);
            if (slot == 0 && k == 0) {                      // S[0] and S[N], each once
                pw[i] = v.x * v.x;
                pm[i] = v.y * v.y;
            } else if (slot == 0) {
                pw[i] = a;
            } else if (slot == 1) {
                pm[i] = a;
            } else {
                mid = a;
            }
        });
        __syncthreads();                        // work array read: the next row may load
        for (uint32_t s = 0; s < n_ser; ++s) {
            const float* Ps = P + (size_t)s * PRED_BINS;
            float acc = tid == 0 ? mid * Ps[FH] : 0.f;
#pragma unroll
            for (int i = 0; i < FBINS; ++i) {
                const int k = tid + FT * i;
                acc = fmaf(pw[i], Ps[k], acc);
                acc = fmaf(pm[i], Ps[k == 0 ? FN : FN - k], acc);
            }
            double d = (double)acc;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if ((tid & 31) == 0) red[tid >> 5] = d;
            __syncthreads();
            if (tid == 0) {
                double tot = 0.0;
                for (int w = 0; w < FT / 32; ++w) tot += red[w];
                D[(size_t)s * d_stride + row0 + q] = (float)tot;
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ void push_tail(const FftParams& p, uint32_t series, uint32_t k, uint32_t tau,
                                          float rho)
{
    unsigned int i = atomicAdd(p.cand_count, 1u);
    if (i < p.cand_cap) p.cand[i] = Candidate{series, k, tau, rho};
}

// the warp's largest of the non-negative g (float bits order as values)
__device__ __forceinline__ float warp_max_abs(float g)
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(g)));
}

// a 128-byte line from DRAM into L2 (no register, no wait)
__device__ __forceinline__ void prefetch_l2(const void* g)
{
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(g));
}

// ---- The correlation kernel's transform: N = 8192 points by a group of 256
// threads, packed two to a register pair (Blackwell's FFMA2/FADD2/FMUL2 take
// two FP32 values per lane at half the issue rate and the full flop rate).
// The first radix-2 stage is taken while the product spectrum is formed:
//   a[n] = Z[n] + Z[n + 4096],  b[n] = (Z[n] - Z[n + 4096]) e^{2 pi i n / 8192},
// n < 4096, give the outputs 2k and 2k + 1 as two 4096-point transforms, which
// run side by side in the two halves of every register pair with the same
// twiddles.  Each is 16 x 16 x 16, decimated in frequency and in place: with
// n = 256 n2 + 16 n1 + n0, pass 1 turns n2 into k0, pass 2 n1 into k1, pass 3
// n0 into k2, k = k0 + 16 k1 + 256 k2, every thread writing back to the slots
// it read, so one array serves.  Passes 2 and 3 of a block of equal k0 belong to
// one half-warp: only pass 1 crosses warps, so a group meets at one barrier a
// transform, after pass 1 writes.  That all its warps have read the transform
// before is an mbarrier's: they arrive after pass 3's reads and wait before the
// next pass 1, long after, and so drift apart between the barriers, some in shared
// memory while others compute.  With a barrier in the mbarrier's place a
// transform took 3 % longer (16 s x 4096 templates in a plan: 541 us a run, 556
// before).

// two complex values, one per register half
struct cpk {
    float2 r, i;
};

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// v *= (wr + i wi), lane by lane
__device__ __forceinline__ void rotate2(cpk& v, float2 wr, float2 wi)
{
    const float2 r = fma2(v.r, wr, neg2(mul2(v.i, wi)));
    v.i = fma2(v.r, wi, mul2(v.i, wr));
    v.r = r;
}

// v *= w, one twiddle for both lanes: unpacked, as a packed FMA of three distinct
// register pairs takes the time of two and the pairs (w, w) would have to be made
__device__ __forceinline__ void rotate1(cpk& v, float2 w)
{
    const float ax = v.r.x * w.x - v.i.x * w.y, ay = v.r.y * w.x - v.i.y * w.y;
    const float bx = v.r.x * w.y + v.i.x * w.x, by = v.r.y * w.y + v.i.y * w.x;
    v.r = make_float2(ax, ay);
    v.i = make_float2(bx, by);
}

// dft4<+1> and dft16<+1> on packed values
__device__ __forceinline__ void dft4_pk(cpk& a, cpk& b, cpk& c, cpk& d)
{
    const cpk t0{add2(a.r, c.r), add2(a.i, c.i)}, t1{sub2(a.r, c.r), sub2(a.i, c.i)};
    const cpk t2{add2(b.r, d.r), add2(b.i, d.i)}, t3{sub2(b.r, d.r), sub2(b.i, d.i)};
    a = {add2(t0.r, t2.r), add2(t0.i, t2.i)};
    c = {sub2(t0.r, t2.r), sub2(t0.i, t2.i)};
    b = {sub2(t1.r, t3.i), add2(t1.i, t3.r)};
    d = {add2(t1.r, t3.i), sub2(t1.i, t3.r)};
}

__device__ __forceinline__ void dft16_pk(cpk (&v)[16])
{
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4_pk(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
    constexpr float C1 = 0.923879532511286756f;   // cos(pi/8)
    constexpr float S1 = 0.382683432365089772f;   // sin(pi/8)
    constexpr float R2 = 0.707106781186547524f;   // cos(pi/4)
    const float2 c1 = make_float2(C1, C1), s1 = make_float2(S1, S1), r2 = make_float2(R2, R2);
    // position 4 k1 + n2 gets e^{2 pi i n2 k1 / 16}
    auto eighth = [&](cpk& u) {                   // e^{i pi / 4}
        const float2 a = sub2(u.r, u.i), b = add2(u.r, u.i);
        u = {mul2(a, r2), mul2(b, r2)};
    };
    auto three_eighths = [&](cpk& u) {            // e^{3 i pi / 4}
        const float2 a = add2(u.r, u.i), b = sub2(u.r, u.i);
        u = {mul2(a, neg2(r2)), mul2(b, r2)};
    };
    rotate2(v[5], c1, s1);
    eighth(v[9]);
    rotate2(v[13], s1, c1);
    eighth(v[6]);
    v[10] = {neg2(v[10].i), v[10].r};
    three_eighths(v[14]);
    rotate2(v[7], s1, c1);
    three_eighths(v[11]);
    rotate2(v[15], neg2(c1), neg2(s1));
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4_pk(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
}

__device__ __forceinline__ float4 pack4(const cpk& v) { return make_float4(v.r.x, v.r.y, v.i.x, v.i.y); }
__device__ __forceinline__ cpk unpack4(float4 f) { return {make_float2(f.x, f.y), make_float2(f.z, f.w)}; }

// Hardware barriers: `id` over `count` threads of the CTA (bar.arrive does not
// wait).  A warp takes part as a whole, so its lanes meet first.
__device__ __forceinline__ void bar_sync(int id, int count)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int count)
{
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// A work array's mbarrier, of one phase a transform: the group's warps arrive
// when they have read their last of the transform from it, and wait for all
// before they write the next one's.  On expiry of the wait the status word is set
// and the kernel goes on without any further wait on these mbarriers, so that it
// ends (its outputs are not given out).
__device__ __forceinline__ void warp_arrive(uint32_t bar)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}
__device__ __forceinline__ void work_array_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err)
{
    if (mbar_try_wait(bar, parity) || *abort_flag || mbar_wait(bar, parity, abort_flag)) return;
    if (err && !*abort_flag) record_error(err, DEV_TIMEOUT_FFT);
    *abort_flag = 1;
}

// s.x + s.y += a, s.x rounded and s.y what the roundings left (Knuth's two-sum): the
// sum of rho^2 to 48 bits without FP64's pipe, whose conversions and additions made
// the GW step 115.6 ms instead of 113.0 (light curves 29.2, 28.5), and for the lanes'
// tree twelve series of one segment against 2048 templates 640 us instead of 600
__device__ __forceinline__ void add_exact(float2& s, float a)
{
    const float h = __fadd_rn(s.x, a), b = __fsub_rn(h, s.x);
    s.y = __fadd_rn(s.y, __fadd_rn(__fsub_rn(s.x, __fsub_rn(h, b)), __fsub_rn(a, b)));
    s.x = h;
}

// 16 bytes of global memory past L1: the norms, which would displace the segment
// spectra there (light curves 8.43 -> 8.27 ms, a 16 s plan 529 -> 526 us, the 64 s
// step 7.32 -> 7.38 ms; the spectra themselves past L1 cost 4 % there)
__device__ __forceinline__ float4 ldg_past_l1(const float4* p)
{
    float4 f;
    asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f.x), "=f"(f.y), "=f"(f.z), "=f"(f.w) : "l"(p));
    return f;
}

// e^{i pi a / 32} for a compile-time a in [0, 8)
__device__ __forceinline__ float2 root64(int a)
{
    const float C[8] = {1.0f, 0.9951847266721968862448f, 0.9807852804032304491262f, 0.9569403357322088649358f,
                        0.9238795325112867561282f, 0.8819212643483550297128f, 0.8314696123025452370788f,
                        0.7730104533627369608109f};
    const float S[8] = {0.0f, 0.0980171403295606019942f, 0.1950903220161282678483f, 0.2902846772544623676362f,
                        0.3826834323650897717285f, 0.4713967368259976485564f, 0.5555702330196022247428f,
                        0.6343932841636454982152f};
    return make_float2(C[a], S[a]);
}

// The correlation.  A CTA holds one template's spectra (real route: one row's;
// pair route: a template's and its partner's) in shared memory, and its two
// groups of 256 threads take the call's segments in turn, each with a work
// array of its own: while one group waits at a barrier or for shared memory,
// the other computes.  A CTA's items (template row, series, segment) are a
// contiguous share of all of them, so the load is even to one transform
// whatever the number of rows; a segment's spectrum is read from L2 straight
// into registers.
//
// Spectra are kept as records (see real_spectrum_quads): float4 number
// (2 r + side) 256 + t (real route) or r 256 + t (pair route) is thread t's; for
// its column j (record_place(j) = t) and n = j + 256 r it holds the bins n and
// 4096 - n (side 0), 8192 - n and 4096 + n (side 1), as (re, re, im, im).  One
// record gives Z[n], Z[n + 4096], and their mirrors Z[4096 - n], Z[8192 - n]:
// the packed inputs n and 4096 - n of the transform.  The second belongs to the
// thread of 256 - j, which sits 16 lanes away in the same warp: lanes 0-15 of
// warp w hold j = 16 w + lane, lanes 16-31 256 - j of them (and 128 in the place
// of 0's, both being their own mirrors).
//
// When both groups have formed their last product of a row (barrier EMPTY),
// the group with the row's last item fetches the next row's spectra during
// its first two passes and then opens them to the other group (barrier FULL,
// of two that alternate with the row: the fetching group may reach the next
// row's before the other has passed this one's).  All these
// are hardware barriers.
//
// What bounds it: the L1 data pipe, 4.6 K wavefronts a transform at five
// segments a template (work array 2.2 K, spectra 1.5 K, norms, mirrors, twiddles
// and sums 0.9 K), beside 4.2 K cycles of FP32 and 4.1 K of issue (63, 57 and
// 55 % busy).  A transform takes 7.3 K cycles (6.2 K at 84 segments a template):
// four warps a scheduler do not overlap the three any further, and the registers
// and the shared memory hold no third group.  16 s x 16,384 templates of 4096
// samples (81,920 transforms) run 1.90 ms; the form it replaced (one CTA-wide
// group with the template in registers, unpacked arithmetic, the radix-2 stage
// last through shared memory, 9 K warp instructions more per transform and four
// CTA-wide barriers) ran 2.60.  The 64 s x 4 series x 65,536 template step went
// from 163.7 to 112.0 ms.  Unpacked twiddle products (rotate1) are 1 % of that.
template <bool QUAD, bool DENSE>
__global__ void __launch_bounds__(FT, 1) k_corr_fft(const __grid_constant__ FftParams p, uint32_t total)
{
    extern __shared__ __align__(16) float4 csm[];
    const int g = threadIdx.x / GT, tg = threadIdx.x % GT, warp = tg >> 5, lane = tg & 31;
    // the transform's input column of this thread, and the lane that holds its mirror
    const int j = lane < 16 ? 16 * warp + lane : (tg == 16 ? GT / 2 : GT - (16 * warp + lane - 16));
    const int mate = tg == 0 || tg == 16 ? lane : lane ^ 16;
    float4* const z = csm + g * ZG;                       // this group's work array
    float4* const h = csm + 2 * ZG;                       // the template's records [4096]
    const float2* const twa = reinterpret_cast<const float2*>(h + FH);       // [6][256]
    const float2* const twb = twa + 6 * GT;               // [15][16]
    const float4* const twp = reinterpret_cast<const float4*>(twb + 15 * 16);   // [256] pairs
    float4* const col0 = h + FH + TWC_N / 2 + 9 * g;      // column 0's inputs 2048, 2304 .. 3840, and 0
    // the reductions over the (row, series) so far, kept out of the registers: the
    // warp's packed max key (0: none yet; a lag below its value and the tail threshold
    // changes nothing) and the thread's sum of rho^2, a pair of FP32 values
    unsigned long long& best = reinterpret_cast<unsigned long long*>(csm + CORR_ACC)[threadIdx.x >> 5];
    float2& ss = reinterpret_cast<float2*>(csm + CORR_ACC + FT / 64 + 1)[threadIdx.x];
    // the group's mbarrier: its work array is read
    const uint32_t zread = smem_u32(csm + CORR_ACC + FT / 64) + 8 * g;
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(csm + CORR_ACC + FT / 64 + 1 + FT / 2);
    const int BAR_G = 1 + g, BAR_EMPTY = 3, BAR_FULL = 4;          // FULL: two, by the parity of the row
    constexpr uint32_t BINS = QUAD ? FH : FN;             // complex bins per segment
    constexpr uint32_t KR = QUAD ? 2 : 1;                 // template rows per item

    const uint32_t n_rows = (p.k_hi - p.k_lo) / KR;
    // this CTA's items, and its first: segment seg0 of row row0
    const uint64_t T = (uint64_t)n_rows * total, i0 = T * blockIdx.x / gridDim.x;
    const uint32_t n_items = (uint32_t)(T * (blockIdx.x + 1) / gridDim.x - i0);
    if (n_items == 0) return;
    const uint32_t row0 = (uint32_t)(i0 / total), seg0 = (uint32_t)(i0 % total);
    const uint32_t row_last = row0 + (uint32_t)(((uint64_t)seg0 + n_items - 1) / total);
    auto spectra = [&](uint32_t row) {
        return reinterpret_cast<const float4*>(p.hspec + (size_t)(p.k_lo + row * KR - p.hrow0) * BINS);
    };
    if (tg == 0) mbar_init(zread, GT / 32);
    if (threadIdx.x == 0) *abort_flag = 0;
    {
        const float4* src = reinterpret_cast<const float4*>(p.tw + TW_N);
        for (int e = threadIdx.x; e < TWC_N / 2; e += FT) cp_async16(h + FH + e, src + e);
        src = spectra(row0);
        for (int e = threadIdx.x; e < FH; e += FT) cp_async16(h + e, src + e);
        cp_async_commit();
        if (row0 < row_last) prefetch_l2(reinterpret_cast<const char*>(spectra(row0 + 1)) + 128 * threadIdx.x);
        cp_async_wait<0>();
        __syncthreads();
    }
    if (g >= (int)n_items) return;                        // a single item: the first group's
    uint32_t item = g, row = row0, seg = seg0 + g;
    int s = 0;
    if (seg >= total) {                                   // the second group begins in the next row
        seg -= total;
        ++row;
        bar_arrive(BAR_EMPTY, FT);
        bar_sync(BAR_FULL + (row & 1), FT);
    }
    while (seg >= p.ser[s].nseg) seg -= p.ser[s++].nseg;
    bool fresh = true;
    float thr = 0.f;
    // the group's next item, two on
    auto advance = [&](uint32_t& row, int& s, uint32_t& seg) {
        seg += 2;
        while (seg >= p.ser[s].nseg) {
            seg -= p.ser[s].nseg;
            if (++s == p.n_ser) {
                s = 0;
                ++row;
            }
        }
    };

    for (;;) {
        const FftSeries& S = p.ser[s];
        const uint32_t k = p.k_lo + row * KR;
        const uint32_t o = (k - p.k_begin) / KR;          // output index
        (void)BF_BOUNDS(p.err, k + KR - 1 < p.k_end && k >= p.hrow0 && seg < S.nseg);
        if (fresh) {
            thr = S.sigma_pred ? S.kappa * S.sigma_pred[o] : p.thr;
            if (lane == 0) best = 0ull;
            ss = make_float2(0.f, 0.f);
        }
        const uint32_t t0 = seg * p.V;
        const uint32_t nv = min(p.V, S.L - t0);
        const float* nrm = S.inv + (size_t)seg * p.Vp;
        // Product spectrum and the first radix-2 stage.  Column 0 holds its own
        // mirrors one place further (256 r goes to 256 (16 - r)), and the record
        // of n = 0 other bins than the rest: its inputs go through `col0`.
        cpk v[16];
        const float4* X = reinterpret_cast<const float4*>(S.spec + (size_t)seg * BINS);
        if (j == 0) {
            float zr, zi, mr, mi, er, ei, fr, fi;         // Z[0], Z[4096], Z[2048], Z[6144]
            if (!QUAD) {
                // the real bins 0 and 8192 as (re, im) of bin 0, then bins 4096, 6144 and 2048
                const cpk xk = unpack4(__ldg(X)), xq = unpack4(__ldg(X + GT)), hk = unpack4(h[0]), hq = unpack4(h[GT]);
                const float y0 = xk.r.x * hk.r.x, yn = xk.i.x * hk.i.x;
                zr = y0 + yn;
                zi = y0 - yn;
                mr = 2.f * (xk.r.y * hk.r.y + xk.i.y * hk.i.y);                  // 2 conj(X) H
                mi = 2.f * (xk.r.y * hk.i.y - xk.i.y * hk.r.y);
                const float ykr = xq.r.y * hq.r.y + xq.i.y * hq.i.y, yki = xq.i.y * hq.r.y - xq.r.y * hq.i.y;
                const float yqr = xq.r.x * hq.r.x + xq.i.x * hq.i.x, yqi = xq.i.x * hq.r.x - xq.r.x * hq.i.x;
                const float ar = ykr + yqr, ai = yki - yqi, br = ykr - yqr, bi = yki + yqi;
                constexpr float R2 = 0.707106781186547524f;                     // w = e^{i pi / 4}
                const float wbr = R2 * (br - bi), wbi = R2 * (br + bi);
                er = ar - wbi;
                ei = ai + wbr;
                fr = ar + wbi;
                fi = wbr - ai;
            } else {
                // bin 0 holds the real bins 0 and 4096; the other lane bin 2048
                const cpk x = unpack4(__ldg(X)), ha = unpack4(h[0]), hb = unpack4(h[FH / 2]);
                zr = x.r.x * ha.r.x;
                zi = x.r.x * hb.r.x;
                mr = x.i.x * ha.i.x;
                mi = x.i.x * hb.i.x;
                const float yar = x.r.y * ha.r.y + x.i.y * ha.i.y, yai = x.i.y * ha.r.y - x.r.y * ha.i.y;
                const float ybr = x.r.y * hb.r.y + x.i.y * hb.i.y, ybi = x.i.y * hb.r.y - x.r.y * hb.i.y;
                er = yar - ybi;
                ei = yai + ybr;
                fr = yar + ybi;
                fi = ybr - yai;
            }
            col0[8] = make_float4(zr + mr, zr - mr, zi + mi, zi - mi);          // the input 0
            col0[0] = make_float4(er + fr, fi - ei, ei + fi, er - fr);          // the input 2048, twiddle i
        }
        const float4 roots = twp[j];
        const float2 base_w = make_float2(roots.x, roots.y), base_t = make_float2(roots.z, roots.w);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float2 w = r ? cmul(base_w, root64(r)) : base_w;          // e^{i pi n / 8192}
            const float2 t = r ? cmul(base_t, root32(r)) : base_t;          // e^{2 pi i n / 8192}
            float2 pr, pi, qr, qi;          // (Z[n], Z[4096 - n]) and (Z[8192 - n], Z[4096 + n])
            if (!QUAD) {
                const cpk xk = unpack4(__ldg(X + 2 * r * GT + tg)), xq = unpack4(__ldg(X + (2 * r + 1) * GT + tg));
                const cpk hk = unpack4(h[2 * r * GT + tg]), hq = unpack4(h[(2 * r + 1) * GT + tg]);
                const float2 wr = make_float2(w.x, w.y), wi = make_float2(w.y, w.x);     // lanes n, 4096 - n
                const float2 ykr = fma2(xk.r, hk.r, mul2(xk.i, hk.i)), yki = fma2(xk.i, hk.r, neg2(mul2(xk.r, hk.i)));
                const float2 yqr = fma2(xq.r, hq.r, mul2(xq.i, hq.i)), yqi = fma2(xq.i, hq.r, neg2(mul2(xq.r, hq.i)));
                // A = Y[k] + conj Y[N-k], B = Y[k] - conj Y[N-k], Z[k] = A + i w B, Z[N-k] = conj(A - i w B)
                const float2 ar = add2(ykr, yqr), ai = sub2(yki, yqi), br = sub2(ykr, yqr), bi = add2(yki, yqi);
                const float2 wbr = fma2(wr, br, neg2(mul2(wi, bi))), wbi = fma2(wr, bi, mul2(wi, br));
                pr = sub2(ar, wbi);
                pi = add2(ai, wbr);
                qr = add2(ar, wbi);
                qi = sub2(wbr, ai);
            } else {
                const cpk x = unpack4(__ldg(X + r * GT + tg));
                const cpk ha = unpack4(h[r * GT + tg]), hb = unpack4(h[FH / 2 + r * GT + tg]);
                const float2 yar = fma2(x.r, ha.r, mul2(x.i, ha.i)), yai = fma2(x.i, ha.r, neg2(mul2(x.r, ha.i)));
                const float2 ybr = fma2(x.r, hb.r, mul2(x.i, hb.i)), ybi = fma2(x.i, hb.r, neg2(mul2(x.r, hb.i)));
                // Z = Ya + i Yb, Z[N - k] = conj(Ya) + i conj(Yb)
                pr = sub2(yar, ybi);
                pi = add2(yai, ybr);
                qr = add2(yar, ybi);
                qi = sub2(ybr, yai);
            }
            // input n: from Z[n] and Z[n + 4096], twiddle t; input 4096 - n: from
            // Z[4096 - n] and Z[8192 - n], twiddle -conj(t)
            const float dr = pr.x - qr.y, di = pi.x - qi.y, er = pr.y - qr.x, ei = pi.y - qi.x;
            v[r] = {make_float2(pr.x + qr.y, dr * t.x - di * t.y), make_float2(pi.x + qi.y, dr * t.y + di * t.x)};
            const float4 f = make_float4(pr.y + qr.x, -er * t.x - ei * t.y, pi.y + qi.x, er * t.y - ei * t.x);
            if (r > 0 && j == 0) col0[8 - r] = f;
            v[15 - r] = {make_float2(__shfl_sync(0xffffffffu, f.x, mate), __shfl_sync(0xffffffffu, f.y, mate)),
                         make_float2(__shfl_sync(0xffffffffu, f.z, mate), __shfl_sync(0xffffffffu, f.w, mate))};
        }
        if (j == 0) {
            v[0] = unpack4(col0[8]);
#pragma unroll
            for (int r = 0; r < 8; ++r) v[8 + r] = unpack4(col0[r]);
        }
        // this group's last product of the row: the spectra may be replaced
        const bool more = item + 2 < n_items;
        bool loading = false, departed = false;
        if (row < row_last) {
            uint32_t nrow = row, nseg = seg;
            int ns = s;
            advance(nrow, ns, nseg);
            if (more && nrow == row) {
                // not the last
            } else if ((((row - row0 + 1) * total - seg0 - 1) & 1) == (uint32_t)g) {       // the row's last item is this group's
                bar_sync(BAR_EMPTY, FT);
                const float4* src = spectra(row + 1);
#pragma unroll
                for (int e = 0; e < FH / GT; ++e) cp_async16(h + e * GT + tg, src + e * GT + tg);
                cp_async_commit();
                if (row + 2 <= row_last) {                // the row after into L2 (64 KiB)
                    const char* nx = reinterpret_cast<const char*>(spectra(row + 2));
                    prefetch_l2(nx + 256 * tg);
                    prefetch_l2(nx + 256 * tg + 128);
                }
                loading = true;
            } else {
                bar_arrive(BAR_EMPTY, FT);
                departed = true;
            }
        }
        // every warp has read the transform before (item / 2 of them) from the work
        // array; asked for here, ahead of the arithmetic, and not at the writes (1 %)
        work_array_wait(zread, ((item >> 1) & 1) ^ 1, abort_flag, p.err);
        __syncwarp();
        // pass 1: out k0 = q at position 4 k1 + k2 of dft16, q = k1 + 4 k2; twiddle e^{2 pi i q j / 4096}
        dft16_pk(v);
        {
            float2 w[4], u[4];
#pragma unroll
            for (int e = 1; e < 4; ++e) {
                w[e] = twa[(e - 1) * GT + j];             // q = 1, 2, 3
                u[e] = twa[(e + 2) * GT + j];             // q = 4, 8, 12
            }
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2)
#pragma unroll
                for (int k1 = 0; k1 < 4; ++k1) {
                    if (k1 + k2 == 0) continue;
                    const float2 f = k1 == 0 ? u[k2] : k2 == 0 ? w[k1] : cmul(u[k2], w[k1]);
                    rotate1(v[4 * k1 + k2], f);
                }
            float4* const zz = z + (j >> 4) * ZROW + (j & 15);
#pragma unroll
            for (int c = 0; c < 16; ++c) zz[((c >> 2) + 4 * (c & 3)) * ZBLK] = pack4(v[c]);
        }
        bar_sync(BAR_G, GT);                              // pass 1 is written
        {
            // pass 2: thread (k0, n0) = (tg / 16, tg % 16); twiddle e^{2 pi i q n0 / 256}
            float4* const zz = z + (tg >> 4) * ZBLK + (tg & 15);
#pragma unroll
            for (int r = 0; r < 16; ++r) v[r] = unpack4(zz[ZROW * r]);
            dft16_pk(v);
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int q = (c >> 2) + 4 * (c & 3);
                if (q) {
                    const float2 f = twb[(q - 1) * 16 + (tg & 15)];
                    rotate1(v[c], f);
                }
                zz[ZROW * q] = pack4(v[c]);
            }
        }
        if (loading) {
            cp_async_wait<0>();                           // this thread's part of the next row's spectra
            bar_arrive(BAR_FULL + ((row + 1) & 1), FT);
        }
        __syncwarp();
        // pass 3: thread (k0, k1) = (tg / 16, tg % 16); output k = k0 + 16 k1 + 256 q
        {
            const float4* const zz = z + (tg >> 4) * ZBLK + (tg & 15) * ZROW;
#pragma unroll
            for (int r = 0; r < 16; ++r) v[r] = unpack4(zz[r]);
        }
        warp_arrive(zread);
        // norms of the lags of this thread's output q: lags 4 k .. 4 k + 3 in the order
        // 0, 2, 1, 3 (real route), lags 2 k, 2 k + 1 (pair route), stored by (q, tg);
        // zero past the segment's end
        auto norms = [&](int q) -> float4 {
            if ((QUAD ? 2u : 4u) * GT * q >= nv) return make_float4(0.f, 0.f, 0.f, 0.f);
            if (!QUAD) return ldg_past_l1(reinterpret_cast<const float4*>(nrm) + GT * q + tg);
            const float2 f = __ldg(reinterpret_cast<const float2*>(nrm) + GT * q + tg);
            return make_float4(f.x, f.y, 0.f, 0.f);
        };
        constexpr int AHEAD = 7;
        float4 iv[AHEAD];
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) iv[q] = norms(q);
        dft16_pk(v);
        // rho in place, the sum of its squares and this thread's largest |rho|
        float2 pa = make_float2(0.f, 0.f);
        float m = 0.f;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            // past the segment's lags (at M = 4096 half of the pair route's outputs;
            // the real route's, a fifth at most, cost less than the branches would)
            if (QUAD && q >= 4 && 2u * GT * q >= nv) continue;
            cpk& c = v[4 * (q & 3) + (q >> 2)];
            const float4 n = iv[q % AHEAD];
            if (q + AHEAD < 16) iv[q % AHEAD] = norms(q + AHEAD);
            if (!QUAD) {
                c.r = mul2(c.r, make_float2(n.x, n.y));           // lags t, t + 2
                c.i = mul2(c.i, make_float2(n.z, n.w));           // lags t + 1, t + 3
                pa = fma2(c.r, c.r, pa);
                pa = fma2(c.i, c.i, pa);
                m = fmaxf(m, fmaxf(fabsf(c.r.x), fabsf(c.r.y)));
                m = fmaxf(m, fmaxf(fabsf(c.i.x), fabsf(c.i.y)));
            } else {
                const float2 e = fma2(c.r, c.r, mul2(c.i, c.i));
                c.r = mul2(make_float2(sqrtf(e.x), sqrtf(e.y)), make_float2(n.x, n.y));
                pa = fma2(c.r, c.r, pa);
                m = fmaxf(m, fmaxf(c.r.x, c.r.y));
            }
        }
        // f(lag in the segment, rho) over this thread's lags in increasing order
        auto each = [&](auto f) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const cpk& c = v[4 * (q & 3) + (q >> 2)];
                const uint32_t t = (QUAD ? 2u : 4u) * (uint32_t)((tg >> 4) + 16 * (tg & 15) + GT * q);
                f(t, c.r.x);
                f(t + 1, QUAD ? c.r.y : c.i.x);
                if (!QUAD) {
                    f(t + 2, c.r.y);
                    f(t + 3, c.i.y);
                }
            }
        };
        if (DENSE && S.rho)
            each([&](uint32_t t, float r) {
                if (t < nv && BF_BOUNDS(p.err, t0 + t < S.L)) S.rho[(size_t)o * S.L + t0 + t] = r;
            });
        {
            float2 t = ss;                                // 32 terms each in FP32 (pair route 16)
            add_exact(t, pa.x);
            add_exact(t, pa.y);
            ss = t;
            // a NaN (finite samples that overflow the transform) counts as larger than any
            // |rho|, as its bits do; fmaxf drops it, the squares do not
            if (!(t.x == t.x)) m = __int_as_float(0x7fc00000);
        }
        // only a warp whose largest |rho| reaches its running max (ties
        // included: an earlier lag wins them) or the tail threshold looks at
        // single lags
        m = warp_max_abs(m);
        __syncwarp();
        const float best_v = __uint_as_float((uint32_t)(best >> 32));
        if (!(m < fminf(thr, best_v))) {
            if (!(m < best_v)) {
                // the earliest lag that has it (a padded lag has rho = 0 and is
                // later than the segment's), for a NaN the warp's earliest
                uint32_t first = 0xffffffffu;
                each([&](uint32_t t, float r) {
                    if (!(fabsf(r) < m)) first = min(first, t);
                });
                first = __reduce_min_sync(0xffffffffu, first);
                const unsigned long long key = pack_max(m, t0 + first);
                if (lane == 0 && first < nv && key > best) best = key;
            }
            if (!(m < thr))
                each([&](uint32_t t, float r) {
                    if (t < nv && fabsf(r) >= thr) push_tail(p, S.series_id, QUAD ? k >> 1 : k, t0 + t, r);
                });
        }
        uint32_t nrow = row;
        int ns = s;
        asm volatile("" : "+r"(seg));                     // recomputed here, not kept in registers
        advance(nrow, ns, seg);
        fresh = !more || ns != s || nrow != row;
        if (__any_sync(0xffffffffu, fresh)) {             // the whole warp's: as a vote it needs no convergence barrier
            float2 t = ss;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const float2 f = make_float2(__shfl_xor_sync(0xffffffffu, t.x, off), __shfl_xor_sync(0xffffffffu, t.y, off));
                add_exact(t, f.x);
                t.y += f.y;
            }
            const double sum = (double)t.x + (t.y == t.y ? (double)t.y : 0.0);     // an infinity leaves a NaN beside it
            if (lane == 0) {
                atomicMax(S.vmax + o, best);
                atomicAdd(S.sumsq + o, sum);
            }
        }
        if (!more) break;
        // the spectra of the next item's row: fetched by this group (all its
        // threads' parts) or by the other
        if (loading) {
            bar_sync(BAR_G, GT);
            ++row;
        }
        while (row < nrow) {
            if (!departed) bar_arrive(BAR_EMPTY, FT);
            ++row;
            bar_sync(BAR_FULL + (row & 1), FT);
            departed = false;
        }
        item += 2;
        s = ns;
    }
}

// Lags whose window holds less than 1/FFT_FIX_RATIO2 of the energy of its
// FFT segment (e.g. a quiet stretch or the tapered edge of a loud chirp next to
// silence): the transform's rounding error scales with the segment, so there it
// would swamp rho.  Their inverse norm is set to 0, so the correlation kernel
// gives them rho = 0 (no tail, nothing to the sum of squares, never above the
// true maximum), and they are listed, with the norm, for k_fft_fixup.  The
// energies come from the FP64 prefix of x^2.  One grid row per series.
// Every norm is also written, times the inverse transform's scale (a power of
// two, so exactly), to the per-segment copy the correlation kernel reads:
// segment j's lags at inv_seg[j Vp ..), Vp = V rounded up as said below,
// so every segment starts 16-byte aligned; past a segment's last lag its row
// holds zeros.  Inside a row the norms stand as the threads of the correlation
// kernel's last pass read them: outputs k = k0 + 16 k1 + 256 q in the order (q, k0,
// k1), each with its lags 4 k, 4 k + 2, 4 k + 1, 4 k + 3 (real route) or 2 k, 2 k + 1
// (pair route); Vp is V rounded up to whole q.
__global__ void __launch_bounds__(256) k_fft_flags(const __grid_constant__ FftSeriesBatch b)
{
    const int i = blockIdx.y;
    if (i >= b.n) return;
    const uint64_t L = b.L[i], N = b.N[i];
    const double* S = b.S[i];
    float* inv = b.inv[i];
    const uint32_t lane = threadIdx.x & 31;
    // the place of lag u of a segment in its row
    auto place = [&](uint64_t u) -> uint64_t {
        const uint64_t k = b.quad ? u >> 1 : u >> 2;
        const uint64_t at = (k & ~255ull) | ((k & 15) << 4) | ((k >> 4) & 15);
        return b.quad ? 2 * at + (u & 1) : 4 * at + ((u & 1) << 1 | ((u >> 1) & 1));
    };
    {
        // the zeros: Vp - V per full segment, Vp - (its lags) in the last one
        const uint64_t nseg = (L + b.V - 1) / b.V;
        const uint64_t last = L - (nseg - 1) * b.V;
        const uint64_t padv = b.Vp - b.V, n_full = (nseg - 1) * padv;
        const uint64_t n_pad = n_full + (b.Vp - last);
        for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < n_pad;
             q += (uint64_t)gridDim.x * blockDim.x) {
            const uint64_t pos = q < n_full ? (q / padv) * b.Vp + place(b.V + q % padv)
                                            : (nseg - 1) * b.Vp + place(last + (q - n_full));
            if (BF_BOUNDS(b.err, pos < nseg * b.Vp)) b.inv_seg[i][pos] = 0.f;
        }
    }
    // the loop bound is uniform over a warp, so each warp appends its lanes'
    // lags together, in lag order (the fixup reads them as coalesced runs)
    for (uint64_t base = blockIdx.x * (uint64_t)blockDim.x; base < L; base += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t t = base + threadIdx.x;
        bool flag = false;
        float iv = 0.f;
        if (t < L) {
            iv = inv[t];
            const uint64_t j = t / b.V;                 // the segment
            const uint64_t a = j * b.V;                 // its first sample
            if (iv > 0.f) {                             // empty window: rho = 0 exactly
                const uint64_t e = min(a + (uint64_t)b.F, N);
                const double E = S[e] - S[a];
                flag = E * (double)iv * (double)iv > FFT_FIX_RATIO2;
            }
            b.inv_seg[i][j * b.Vp + place(t - a)] = flag ? 0.f : iv * b.scale;
        }
        const uint32_t mask = __ballot_sync(0xffffffffu, flag);
        if (mask == 0u) continue;
        uint32_t slot0 = 0;
        if (lane == 0) slot0 = atomicAdd(b.n_fix + i, (uint32_t)__popc(mask));   // each lag once: < L entries
        slot0 = __shfl_sync(0xffffffffu, slot0, 0);
        const uint32_t slot = slot0 + __popc(mask & ((1u << lane) - 1u));
        if (flag && BF_BOUNDS(b.err, slot < L)) {
            inv[t] = 0.f;
            b.fix[i][2 * slot] = (uint32_t)t;
            b.fix[i][2 * slot + 1] = __float_as_uint(iv);
        }
    }
}

// The direct computation of the listed lags.  Each CTA takes FIX_ROWS template
// rows of the launch's range (FIX_ROWS / 2 quadrature pairs), synthesises them
// in shared memory as the bank does (FP32 rows at unit norm), and gives each
// lane one listed lag: the lane runs the FP32 dot products of its window with
// every row, four samples at a time (four window loads, one 16-byte broadcast
// per row), so one shared-memory wavefront feeds 32 FMAs of the warp rather
// than one.  The products then feed the same max keys, sums of rho^2, tails and
// dense output (written after the correlation kernel's 0 there) as the
// correlation kernel.  Returns at once when no series has a listed lag.
constexpr int FIX_T = 256;
constexpr int FIX_ROWS = 4;
constexpr size_t FIX_SMEM = (size_t)FIX_ROWS * FH * sizeof(float);      // rows of at most FH samples

template <bool QUAD>
__global__ void __launch_bounds__(FIX_T) k_fft_fixup(const __grid_constant__ FftParams p)
{
    constexpr int NOUT = QUAD ? FIX_ROWS / 2 : FIX_ROWS;
    extern __shared__ __align__(16) float fx_rows[];                     // [FIX_ROWS][M_s]
    __shared__ double red[8];
    __shared__ unsigned long long w_key[FIX_T / 32][NOUT];
    __shared__ double w_ss[FIX_T / 32][NOUT];
    uint32_t total = 0;
    for (int i = 0; i < p.n_ser; ++i) total += *p.ser[i].n_fix;
    if (total == 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t M = p.M, M_s = (M + 63u) & ~63u;
    const uint32_t n_groups = (p.k_hi - p.k_lo + FIX_ROWS - 1) / FIX_ROWS;   // a pair never splits
    for (uint32_t grp = blockIdx.x; grp < n_groups; grp += gridDim.x) {
        const uint32_t row0 = p.k_lo + grp * FIX_ROWS;
        const uint32_t nr = min((uint32_t)FIX_ROWS, p.k_hi - row0);
        for (uint32_t r = 0; r < (uint32_t)FIX_ROWS; ++r) {
            float* g = fx_rows + (size_t)r * M_s;
            const float nrm = synth_row(p.chirps, row0 + r, p.quad, r < nr, M, M_s, p.fs, g, red);
            for (uint32_t m = threadIdx.x; m < M_s; m += FIX_T) g[m] *= nrm;
        }
        __syncthreads();
        uint32_t o[NOUT], kt[NOUT];
        bool live[NOUT];
#pragma unroll
        for (int j = 0; j < NOUT; ++j) {
            const uint32_t row = row0 + (QUAD ? 2 * j : j);
            live[j] = row < p.k_hi;
            o[j] = QUAD ? (row - p.k_begin) >> 1 : row - p.k_begin;      // output index
            kt[j] = QUAD ? row >> 1 : row;                               // tail index
        }
        for (int i = 0; i < p.n_ser; ++i) {
            const FftSeries& S = p.ser[i];
            const uint32_t n = min(*S.n_fix, S.L);
            if (n == 0) continue;                                        // uniform over the CTA
            float thr[NOUT];
#pragma unroll
            for (int j = 0; j < NOUT; ++j)
                thr[j] = !live[j] ? INFINITY : (S.sigma_pred ? S.kappa * S.sigma_pred[o[j]] : p.thr);
            unsigned long long best[NOUT];
            double ss[NOUT];
#pragma unroll
            for (int j = 0; j < NOUT; ++j) {
                best[j] = 0ull;
                ss[j] = 0.0;
            }
            for (uint32_t f0 = warp * 32u; f0 < n; f0 += FIX_T) {
                const uint32_t f = f0 + lane;
                const bool act = f < n;
                const uint32_t tau = act ? S.fix[2 * f] : 0u;
                const float iv = act ? __uint_as_float(S.fix[2 * f + 1]) : 0.f;   // the window's norm
                const float* xw = S.x + tau;    // padded: reads up to tau + M + 2 stay inside
                float c[FIX_ROWS];
#pragma unroll
                for (int r = 0; r < FIX_ROWS; ++r) c[r] = 0.f;
                for (uint32_t m = 0; m < M; m += 4) {           // rows are zero past M
                    const float x0 = xw[m], x1 = xw[m + 1], x2 = xw[m + 2], x3 = xw[m + 3];
#pragma unroll
                    for (int r = 0; r < FIX_ROWS; ++r) {
                        const float4 gv = *reinterpret_cast<const float4*>(fx_rows + (size_t)r * M_s + m);
                        c[r] = fmaf(x0, gv.x, c[r]);
                        c[r] = fmaf(x1, gv.y, c[r]);
                        c[r] = fmaf(x2, gv.z, c[r]);
                        c[r] = fmaf(x3, gv.w, c[r]);
                    }
                }
                if (!act) continue;
#pragma unroll
                for (int j = 0; j < NOUT; ++j) {
                    if (!live[j]) continue;
                    const float rho = QUAD ? sqrtf(c[2 * j] * c[2 * j] + c[2 * j + 1] * c[2 * j + 1]) * iv
                                           : c[j] * iv;
                    const float a = fabsf(rho);
                    const unsigned long long key = pack_max(a, tau);
                    best[j] = key > best[j] ? key : best[j];
                    ss[j] += (double)rho * (double)rho;
                    if (a >= thr[j]) push_tail(p, S.series_id, kt[j], tau, rho);
                    if (S.rho) S.rho[(size_t)o[j] * S.L + tau] = rho;
                }
            }
#pragma unroll
            for (int j = 0; j < NOUT; ++j) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    const unsigned long long ok = __shfl_xor_sync(0xffffffffu, best[j], off);
                    best[j] = ok > best[j] ? ok : best[j];
                    ss[j] += __shfl_xor_sync(0xffffffffu, ss[j], off);
                }
                if (lane == 0) {
                    w_key[warp][j] = best[j];
                    w_ss[warp][j] = ss[j];
                }
            }
            __syncthreads();
            if (threadIdx.x < NOUT && live[threadIdx.x]) {
                const int j = threadIdx.x;
                unsigned long long kmax = 0ull;
                double tot = 0.0;
                for (int w = 0; w < FIX_T / 32; ++w) {
                    kmax = w_key[w][j] > kmax ? w_key[w][j] : kmax;
                    tot += w_ss[w][j];
                }
                if (kmax != 0ull) {
                    atomicMax(S.vmax + o[j], kmax);
                    atomicAdd(S.sumsq + o[j], tot);
                }
            }
            __syncthreads();
        }
    }
}

template <typename K>
cudaError_t smem_opt_in(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t fft_attributes()
{
    static DeviceOnce once;
    return once.run([] {
        cudaError_t e = smem_opt_in(k_corr_fft<false, false>, CORR_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_corr_fft<false, true>, CORR_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_corr_fft<true, false>, CORR_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_corr_fft<true, true>, CORR_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_fft_series<true>, FFT_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_fft_series<false>, FFT_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_fft_bank_real, BANK_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_fft_bank_pair, FFT_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_welch_segments, FFT_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_template_power_dot, FFT_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_fft_fixup<false>, FIX_SMEM);
        if (e == cudaSuccess) e = smem_opt_in(k_fft_fixup<true>, FIX_SMEM);
        return e;
    });
}

}  // namespace

// The context's twiddle tables, built on first use.
cudaError_t fft_tables(bf_ctx* ctx, cudaStream_t st, const float2** out)
{
    if (!ctx->fft_tw) {
        float2* t = nullptr;
        cudaError_t e = cudaMalloc(&t, (TW_N + TWC_N + 2 * FT) * sizeof(float2));
        if (e != cudaSuccess) return e;
        count_launches(1);
        k_fft_tables<<<(TW_N + 255) / 256, 256, 0, st>>>(t);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            cudaFree(t);
            return e;
        }
        ctx->fft_tw = t;
    }
    *out = ctx->fft_tw;
    return fft_attributes();
}

uint32_t fft_seg_len(bool quad) { return quad ? FN : FR; }
uint32_t fft_spec_bins(bool quad) { return quad ? FH : FN; }

// Spectra of template rows [row0, row0 + nrows) into out[0 ..] (fft_spec_bins
// complex values per row), through `scratch`, room for `scratch_rows`
// synthesised rows of 8192 samples.  The pair route rounds nrows up to even:
// an odd tail pairs with a zero row whose spectrum is not written.
// Asynchronous on st.
static cudaError_t template_spectra(const bf_bank* bank, size_t row0, size_t nrows, float* scratch,
                                    size_t scratch_rows, const float2* tw, float2* out, int n_sm,
                                    cudaStream_t st)
{
    const size_t bins = fft_spec_bins(bank->quad);
    if (bank->M > (uint32_t)FH) return cudaErrorInvalidValue;     // the route's limit (checked by the callers)
    cudaError_t e = cudaSuccess;
    for (size_t k = 0; k < nrows && e == cudaSuccess; k += scratch_rows) {
        const size_t kc = std::min(scratch_rows, nrows - k);     // rows of this sub-chunk
        const size_t nr = bank->quad ? kc + (kc & 1) : kc;        // scratch_rows is even
        e = launch_bank_synth(bank->d_params, (uint32_t)(row0 + k), bank->quad, (uint32_t)kc, (uint32_t)nr,
                              bank->M, FN, bank->fs, scratch, nullptr, nullptr, st);
        if (e != cudaSuccess) break;
        const uint32_t items = (uint32_t)(bank->quad ? nr / 2 : nr);
        const unsigned grid = std::min<uint32_t>(items, (uint32_t)n_sm);
        count_launches(1);
        if (bank->quad) k_fft_bank_pair<<<grid, FT, FFT_SMEM, st>>>(scratch, (uint32_t)kc, items, tw, out + k * bins);
        else k_fft_bank_real<<<grid, FT, BANK_SMEM, st>>>(scratch, (uint32_t)kc, bank->M, tw, out + k * bins);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t fft_template_spectra(const bf_bank* bank, size_t row0, size_t nrows, float* scratch,
                                 size_t scratch_rows, const float2* tw, float2* out, int n_sm, cudaStream_t st)
{
    return template_spectra(bank, row0, nrows, scratch, scratch_rows, tw, out, n_sm, st);
}

// Spectra of every template of the bank, [rows (rounded up to even for the
// pair route)][fft_spec_bins] complex, computed once and kept with the bank.
bf_status bank_fft_spectra(bf_ctx* ctx, bf_bank* bank, cudaStream_t st)
{
    if (bank->fspec) return BF_OK;
    if (bank->M > FFT_POINTS / 2) {
        set_error("the FFT route takes templates of at most %d samples (this bank: %u)", FFT_POINTS / 2,
                  bank->M);
        return BF_ENOTSUP;
    }
    const float2* tw = nullptr;
    cudaError_t e = fft_tables(ctx, st, &tw);
    if (e != cudaSuccess) return cuda_fail(e, "FFT tables");
    const size_t K2 = bank->quad ? bank->rows + (bank->rows & 1) : bank->rows;
    const size_t bins = fft_spec_bins(bank->quad);
    Allocator& mem = *ctx->mem;
    float2* spec = static_cast<float2*>(mem.alloc(K2 * bins * sizeof(float2)));
    const size_t chunk = std::min<size_t>(4096, K2 + (K2 & 1));
    float* rows = static_cast<float*>(mem.alloc(chunk * FN * sizeof(float)));
    if (!spec || !rows) {
        mem.release(spec);
        mem.release(rows);
        set_error("out of device memory for the template spectra (%zu MB)", (K2 * bins * 8) >> 20);
        return BF_ENOMEM;
    }
    e = template_spectra(bank, 0, bank->rows, rows, chunk, tw, spec, ctx->n_sm, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    mem.release(rows);
    if (e != cudaSuccess) {
        mem.release(spec);
        return cuda_fail(e, "template spectra");
    }
    bank->fspec = spec;
    return BF_OK;
}

uint32_t fft_lags_per_seg(uint32_t M, bool quad) { return fft_seg_len(quad) - M + 1; }
uint32_t fft_norm_stride(uint32_t M, bool quad)
{
    const uint32_t q = (quad ? 2 : 4) * GT;          // lags of one output of every thread
    return (fft_lags_per_seg(M, quad) + q - 1) / q * q;
}
// 1/F for the real route: the inverse transform is unnormalised and the
// even/odd split forms twice the packed spectrum; 1/N for the pair route
float fft_inverse_scale(bool quad) { return 1.f / (float)fft_seg_len(quad); }

size_t fft_series_bytes(uint32_t L, uint32_t M, bool quad)
{
    const size_t nseg = fft_segments(L, M, quad);
    return nseg * fft_spec_bins(quad) * sizeof(float2) + nseg * fft_norm_stride(M, quad) * sizeof(float);
}

uint32_t fft_segments(uint32_t L, uint32_t M, bool quad)
{
    const uint64_t V = fft_lags_per_seg(M, quad);
    return (uint32_t)(((uint64_t)L + V - 1) / V);          // L may be close to 2^32
}

uint32_t welch_segments(uint64_t N)
{
    return N >= (uint64_t)PRED_F ? (uint32_t)((N - PRED_F) / (PRED_F / 2) + 1) : 1u;
}

cudaError_t launch_welch(const WelchBatch& b, int n_sm, cudaStream_t st)
{
    const uint32_t total = b.seg_begin[b.n];
    if (b.n == 0 || total == 0) return cudaSuccess;
    count_launches(2);
    k_welch_segments<<<std::min<uint32_t>(total, (uint32_t)n_sm), FT, FFT_SMEM, st>>>(b, total);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_welch_mean<<<dim3((PRED_BINS + 255) / 256, (unsigned)b.n), 256, 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_template_power_dot(const float* rows, uint32_t n_rows, const float2* tw, const float* P,
                                      uint32_t n_ser, float* D, uint32_t d_stride, uint32_t row0, int n_sm,
                                      cudaStream_t st)
{
    if (n_rows == 0 || n_ser == 0) return cudaSuccess;
    count_launches(1);
    k_template_power_dot<<<std::min<uint32_t>(n_rows, (uint32_t)n_sm), FT, FFT_SMEM, st>>>(
        rows, n_rows, tw, P, n_ser, D, d_stride, row0);
    return cudaGetLastError();
}

cudaError_t launch_fft_series(const FftSeriesBatch& b, uint32_t total_segments, int n_sm, cudaStream_t st)
{
    if (total_segments == 0) return cudaSuccess;
    const unsigned grid = std::min<uint32_t>(total_segments, (uint32_t)n_sm);
    count_launches(1);
    if (b.quad) k_fft_series<false><<<grid, FT, FFT_SMEM, st>>>(b, total_segments);
    else k_fft_series<true><<<grid, FT, FFT_SMEM, st>>>(b, total_segments);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !b.n_fix) return e;
    // the lags for the direct fixup
    uint32_t L_max = 0;
    for (int i = 0; i < b.n; ++i) L_max = std::max(L_max, b.L[i]);
    const unsigned bx = (unsigned)std::max<uint32_t>(1, std::min<uint32_t>((L_max + 255) / 256, 1024));
    count_launches(1);
    k_fft_flags<<<dim3(bx, (unsigned)b.n), 256, 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_corr_fft(const FftParams& p, int n_sm, cudaStream_t st)
{
    const uint32_t rows = p.quad ? (p.k_hi - p.k_lo) / 2 : p.k_hi - p.k_lo;
    if (rows == 0 || p.n_ser == 0) return cudaSuccess;
    uint64_t total = 0;                       // segments of a row
    bool dense = false;
    for (int i = 0; i < p.n_ser; ++i) {
        total += p.ser[i].nseg;
        dense = dense || p.ser[i].rho != nullptr;
    }
    if (total == 0 || total > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    // contiguous shares of the rows x total transforms: a CTA needs one at least,
    // and counts its own in 32 bits
    const uint64_t T = rows * total;
    const unsigned grid = (unsigned)std::min<uint64_t>(T, std::max<uint64_t>((uint64_t)n_sm, T >> 30));
    count_launches(1);
    if (p.quad) {
        if (dense) k_corr_fft<true, true><<<grid, FT, CORR_SMEM, st>>>(p, (uint32_t)total);
        else k_corr_fft<true, false><<<grid, FT, CORR_SMEM, st>>>(p, (uint32_t)total);
    } else {
        if (dense) k_corr_fft<false, true><<<grid, FT, CORR_SMEM, st>>>(p, (uint32_t)total);
        else k_corr_fft<false, false><<<grid, FT, CORR_SMEM, st>>>(p, (uint32_t)total);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !p.chirps) return e;
    // the lags left to the direct computation (none: the CTAs return at once)
    const uint32_t n_groups = (p.k_hi - p.k_lo + FIX_ROWS - 1) / FIX_ROWS;
    if (n_groups == 0) return e;
    const unsigned fgrid = std::min<unsigned>(n_groups, (unsigned)n_sm * 3);
    const size_t smem = (size_t)FIX_ROWS * ((p.M + 63u) & ~63u) * sizeof(float);
    count_launches(1);
    if (p.quad) k_fft_fixup<true><<<fgrid, FIX_T, smem, st>>>(p);
    else k_fft_fixup<false><<<fgrid, FIX_T, smem, st>>>(p);
    return cudaGetLastError();
}

// A bank that keeps only its chirp parameters: the template spectra are made
// chunk by chunk (512 MiB of spectra: 8192 rows of the real route, 16384 of
// the pair route) into a two-slot ring on the auxiliary stream, and chunk c is
// correlated against every series batch on the main stream while chunk c+1 is
// made.  Events order the reuse of a slot after the launches that read it.
constexpr size_t FFT_CHUNK_BYTES = size_t(512) << 20;
constexpr size_t FFT_SYNTH_ROWS = 4096;

bf_status fft_ring_prepare(bf_ctx* ctx, const bf_bank* bank, uint32_t row_begin, uint32_t row_end,
                           std::vector<void*>& keep, FftRing* ring)
{
    const size_t bins = fft_spec_bins(bank->quad);
    const size_t n_rows = row_end - row_begin;
    ring->chunk = std::min(FFT_CHUNK_BYTES / (bins * sizeof(float2)), n_rows + (n_rows & 1));
    ring->n_chunks = (n_rows + ring->chunk - 1) / ring->chunk;
    ring->synth_rows = std::min(FFT_SYNTH_ROWS, ring->chunk + (ring->chunk & 1));    // even
    Allocator& mem = *ctx->mem;
    ring->scratch = static_cast<float*>(mem.alloc(ring->synth_rows * FN * sizeof(float)));
    if (ring->scratch) keep.push_back(ring->scratch);
    for (int i = 0; i < 2 && i < (int)ring->n_chunks; ++i) {
        ring->slot[i] = static_cast<float2*>(mem.alloc((ring->chunk + 2) * bins * sizeof(float2)));
        if (ring->slot[i]) keep.push_back(ring->slot[i]);
    }
    if (!ring->scratch || !ring->slot[0] || (ring->n_chunks > 1 && !ring->slot[1])) {
        set_error("out of device memory for the template-spectra ring");
        return BF_ENOMEM;
    }
    cudaError_t e = ring->ev.create();
    return e == cudaSuccess ? BF_OK : cuda_fail(e, "ring events");
}

cudaError_t fft_correlate_chunked(bf_ctx* ctx, const bf_bank* bank, std::vector<FftParams>& batches,
                                  uint32_t row_begin, uint32_t row_end, const FftRing& ring,
                                  cudaStream_t st)
{
    const bool quad = bank->quad;
    const float2* tw = batches.empty() ? nullptr : batches[0].tw;
    const RingEvents& ev = ring.ev;
    cudaError_t e = cudaEventRecord(ev.start, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->aux, ev.start, 0);
    for (size_t c = 0; c < ring.n_chunks && e == cudaSuccess; ++c) {
        const int sl = (int)(c & 1);
        const uint32_t c0 = row_begin + (uint32_t)(c * ring.chunk);
        const uint32_t c1 = (uint32_t)std::min<size_t>(c0 + ring.chunk, row_end);
        // the pair route makes the spectra of the even-aligned row pairs that a
        // stored bank uses, partner rows outside the slice included (each
        // spectrum carries its partner's rounding), so the outputs equal the
        // stored bank's; the real route makes one row per transform
        const uint32_t s0 = quad ? c0 & ~1u : c0;
        const uint32_t s1 = quad ? (uint32_t)std::min<size_t>((c1 + 1) & ~1u, bank->rows) : c1;
        if (c >= 2) e = cudaStreamWaitEvent(ctx->aux, ev.used[sl], 0);
        if (e == cudaSuccess)
            e = template_spectra(bank, s0, s1 - s0, ring.scratch, ring.synth_rows, tw, ring.slot[sl], ctx->n_sm,
                                 ctx->aux);
        if (e == cudaSuccess) e = cudaEventRecord(ev.made[sl], ctx->aux);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev.made[sl], 0);
        for (FftParams& p : batches) {
            if (e != cudaSuccess) break;
            p.hspec = ring.slot[sl];
            p.hrow0 = s0;
            p.k_lo = c0;
            p.k_hi = c1;
            e = launch_corr_fft(p, ctx->n_sm, st);
        }
        if (e == cudaSuccess) e = cudaEventRecord(ev.used[sl], st);
    }
    return e;
}

}  // namespace bfi
