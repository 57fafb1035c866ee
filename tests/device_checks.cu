// Checks of device functions that no call of the library shows by itself.  The
// sources are included, so that the functions tested are the library's.
#include <cstdio>

#include "prep.cu"

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

// a counter-based draw (the splitmix64 finaliser)
__device__ uint64_t splitmix64(uint64_t z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

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

int main() { return norms(); }
