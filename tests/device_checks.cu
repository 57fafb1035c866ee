// Checks of device functions that no call of the library shows by itself.  The
// sources are included, so that the functions tested are the library's.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <numeric>

#include "prep.cu"
#include "permute.cu"
#include "corr_common.cuh"

namespace bfi {
std::atomic<uint64_t> g_launches{0};
}

using namespace bfi;

#define CK(x)                                                                     \
    do {                                                                          \
        const cudaError_t e_ = (x);                                               \
        if (e_ != cudaSuccess) {                                                  \
            fprintf(stderr, "%s: %s\n", #x, cudaGetErrorString(e_));              \
            return 2;                                                             \
        }                                                                         \
    } while (0)

// mantissas of window energies in [1, 4): the largest relative distance of the
// library's 1 / sqrt from FP64's, in units of 2^-53; and the norms of energies
// 2^e (1 + f), e in [-300, 300), that differ from FP64's rounded to FP32
__global__ void k_norm_check(uint64_t n, unsigned long long* worst, unsigned long long* wrong)
{
    double d = 0.0;
    unsigned long long w = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t z = splitmix64(i), f = z >> 12;
        const double m = __longlong_as_double((long long)((1023 + (z & 1)) << 52 | f)), r = 1.0 / sqrt(m);
        d = fmax(d, fabs(inv_root(m) - r) / r);
        const double nu = __longlong_as_double((long long)((1023 - 300 + splitmix64(~i) % 600) << 52 | f));
        w += inv_sqrt(nu) != (float)(1.0 / sqrt(nu)) ? 1ull : 0ull;
    }
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(wrong, w);
    atomicMax(worst, (unsigned long long)(d * 0x1p53 * 1000.0));
}

static int norms()
{
    unsigned long long* d = nullptr;
    unsigned long long h[2] = {0, 0};
    CK(cudaMalloc(&d, sizeof h));
    CK(cudaMemset(d, 0, sizeof h));
    k_norm_check<<<2048, 256>>>(1ull << 28, d, d + 1);
    CK(cudaGetLastError());
    CK(cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost));
    printf("norms %.3f %llu\n", (double)h[0] / 1000.0, h[1]);
    return 0;
}

// The control's four steps with 2^bits buckets for n samples, so few that every
// bucket reaches past a block's neighbourhood, against a stable sort by key.
static int crowded(uint32_t n, int bits, uint64_t seed)
{
    auto mix = [](uint64_t z) {
        z += 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    std::vector<float> x(n), got(n);
    std::iota(x.begin(), x.end(), 0.f);
    std::vector<uint32_t> want(n);
    std::iota(want.begin(), want.end(), 0u);
    std::stable_sort(want.begin(), want.end(),
                     [&](uint32_t a, uint32_t b) { return mix(seed ^ a) < mix(seed ^ b); });
    const uint32_t B = 1u << bits;
    const int shift = 64 - bits;
    float *in = nullptr, *out = nullptr;
    uint32_t* s = nullptr;
    CK(cudaMalloc(&in, n * 4));
    CK(cudaMalloc(&out, n * 4));
    CK(cudaMalloc(&s, (2 * (size_t)B + 2 * (size_t)n) * 4));
    uint32_t *count = s, *begin = s + B, *slot = begin + B, *idx = slot + n;
    CK(cudaMemcpy(in, x.data(), n * 4, cudaMemcpyHostToDevice));
    CK(cudaMemset(out, 0xff, n * 4));
    CK(cudaMemset(count, 0, B * 4));
    const unsigned grid = (n + SORT_T - 1) / SORT_T;
    k_perm_count<<<grid, SORT_T>>>(n, seed, shift, count, slot);
    k_perm_scan<<<(B + SCAN_TILE - 1) / SCAN_TILE, SCAN_THREADS>>>(count, B, begin);
    k_perm_scatter<<<grid, SORT_T>>>(n, seed, shift, begin, slot, idx);
    k_perm_rank<<<grid, SORT_T>>>(in, n, seed, shift, begin, count, idx, out);
    CK(cudaGetLastError());
    CK(cudaMemcpy(got.data(), out, n * 4, cudaMemcpyDeviceToHost));
    uint32_t wrong = 0;
    for (uint32_t j = 0; j < n; ++j) wrong += got[j] != (float)want[j] ? 1u : 0u;
    printf("crowded_wrong %u %d %u\n", n, bits, wrong);
    cudaFree(in);
    cudaFree(out);
    cudaFree(s);
    return 0;
}

// The wait that both correlation kernels use, on an mbarrier that nothing arrives
// at: with a limit of 20 ms, then with the abort flag set.
__global__ void k_wait_check(unsigned long long* ns, int* ok)
{
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_word;
    if (threadIdx.x != 0) return;
    mbar_init(smem_u32(&bar), 1);
    abort_word = 0;
    for (int i = 0; i < 2; ++i) {
        const uint64_t t0 = globaltimer();
        ok[i] = mbar_wait(smem_u32(&bar), 0, &abort_word, true, i ? 1000000000ull : 20000000ull) ? 1 : 0;
        ns[i] = globaltimer() - t0;
        abort_word = 1;
    }
}

static int waits()
{
    unsigned long long *d = nullptr, h[2];
    int *o = nullptr, ok[2];
    CK(cudaMalloc(&d, sizeof h));
    CK(cudaMalloc(&o, sizeof ok));
    k_wait_check<<<1, 32>>>(d, o);
    CK(cudaGetLastError());
    CK(cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(ok, o, sizeof ok, cudaMemcpyDeviceToHost));
    printf("wait %llu %d %llu %d\n", h[0], ok[0], h[1], ok[1]);
    return 0;
}

int main()
{
    int rc = norms();
    rc = rc ? rc : waits();
    for (uint32_t n : {257u, 5000u, 20001u})
        for (int bits : {2, 4, 6}) rc = rc ? rc : crowded(n, bits, 0x1234567ull + n);
    return rc;
}
