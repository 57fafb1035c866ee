// Helpers shared by the correlation kernels: mbarriers whose waits are bounded in
// time, tile lookup over segments, and the reductions of the fused epilogue
// (arXiv:1802.01685 Sect. 2.1-2.2 and Fig. 2: per-template maxima of the filter
// output, sigma of the output, and the tails |rho| >= threshold that paint the
// chirp-based spectrogram).
#pragma once
#include "bf_internal.h"

namespace bfi {

// Locates the segment owning global tile t (segments are sorted by tile_begin).
__device__ __forceinline__ int find_seg(const CorrParams& p, uint64_t t)
{
    int lo = 0, hi = p.n_seg - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (p.seg[mid].tile_begin <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Max key of |rho| with ties resolved to the smallest lag: |rho| >= 0, so its
// float bits order like unsigned integers; the low word is ~tau.
__device__ __forceinline__ unsigned long long pack_max(float a, uint32_t tau)
{
    return ((unsigned long long)__float_as_uint(a) << 32) | (unsigned long long)(~tau);
}

__device__ __forceinline__ void push_candidate(const CorrParams& p, uint32_t series,
                                               uint32_t k, uint32_t tau, float rho)
{
    unsigned int i = atomicAdd(p.cand_count, 1u);
    if (i < p.cand_cap) p.cand[i] = Candidate{series, k, tau, rho};
}

// ---------------------------------------------------------------- mbarriers
// The longest that a wait lasts, against the microseconds that it takes: on expiry
// the kernel records a code and ends, so that no wait can hang the GPU.
constexpr uint64_t TIMEOUT_NS = 10ull * 1000 * 1000 * 1000;

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait.  Returns false on timeout or when another role aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity,
                                          volatile int* abort_flag, bool honour_abort = true,
                                          uint64_t limit_ns = TIMEOUT_NS)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63) == 0) {
            if (honour_abort && *abort_flag) return false;
            if (globaltimer() - t0 > limit_ns) return false;
        }
    }
}

// the first code recorded stays
__device__ __forceinline__ void record_error(int* err, int code)
{
    atomicCAS(err, 0, code);
}

}  // namespace bfi
