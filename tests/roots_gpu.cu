// The step's own roots and reciprocals on the GPU beside CUDA's.
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm_device.cuh"

using namespace lbm;

// n[0], n[1]: FP32 roots and reciprocals of both components that differ from sqrtf and division,
// for every significand at each of the exponents e0 .. e0 + ne - 1 (biased).
__global__ void check_f32(int e0, int ne, unsigned long long* n) {
    const unsigned long long total = (unsigned long long)ne << 23;
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < total;
         k += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t frac = (uint32_t)(k & 0x7FFFFFu), e = (uint32_t)(e0 + (int)(k >> 23));
        const float x = __uint_as_float(e << 23 | frac), z = __uint_as_float(e << 23 | (0x7FFFFFu - frac));
        const f2 p = f2(make_float2(x, z)), s = sqrt_pos<true>(p), r = rcp_pos<true>(p);
        if (__float_as_uint(s.v.x) != __float_as_uint(sqrtf(x)) || __float_as_uint(s.v.y) != __float_as_uint(sqrtf(z)))
            atomicAdd(n, 1ull);
        if (__float_as_uint(r.v.x) != __float_as_uint(1.0f / x) || __float_as_uint(r.v.y) != __float_as_uint(1.0f / z))
            atomicAdd(n + 1, 1ull);
    }
}

// The largest distance in units: n[2] FP64 root, n[3] reciprocal; n[4], n[5] the seeds' relative
// errors in 2^-30.  Exponents e0 .. e0 + ne - 1 (biased), significands from a linear generator.
__global__ void check_f64(int e0, int ne, int each, unsigned long long* n) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ne) return;
    unsigned long long state = 0x9E3779B97F4A7C15ull * (unsigned)(t + 1), far[4] = {0, 0, 0, 0};
    auto units = [](double a, double b) {
        const long long d = __double_as_longlong(a) - __double_as_longlong(b);
        return (unsigned long long)(d < 0 ? -d : d);
    };
    auto most = [](unsigned long long& a, unsigned long long b) { if (b > a) a = b; };
    for (int k = 0; k < each; ++k) {
        state = state * 6364136223846793005ull + 1442695040888963407ull;
        // both ends of the binade first, then anything
        const unsigned long long frac = k == 0 ? 0 : k == 1 ? (1ull << 52) - 1 : state >> 12;
        const double x = __longlong_as_double((long long)(((unsigned long long)(e0 + t) << 52) | frac));
        most(far[0], units(sqrt_pos<false>(x), sqrt(x)));
        most(far[1], units(rcp_pos<false>(x), 1.0 / x));
        const double y = rsqrt_seed(x), z = rcp_seed(x);
        most(far[2], (unsigned long long)(fabs(fma(y * x, y, -1.0)) * 0.5 * 1073741824.0));
        most(far[3], (unsigned long long)(fabs(fma(z, x, -1.0)) * 1073741824.0));
    }
    for (int k = 0; k < 4; ++k) atomicMax(n + 2 + k, far[k]);
}

extern "C" int check_roots(unsigned long long out[6]) {
    unsigned long long* n = nullptr;
    if (cudaMalloc(&n, 6 * sizeof *n) != cudaSuccess) return 1;
    cudaMemset(n, 0, 6 * sizeof *n);
    // |v|^2 + 1e-28 and Eq. 18's denominator: 2^-93 .. 2^120, in four ranges of two binades or more
    check_f32<<<608, 256>>>(127, 2, n);
    check_f32<<<608, 256>>>(127 - 93, 4, n);
    check_f32<<<608, 256>>>(127 - 30, 2, n);
    check_f32<<<608, 256>>>(127 + 119, 2, n);
    check_f64<<<(1990 + 127) / 128, 128>>>(1023 - 996, 1990, 4096, n);
    const cudaError_t e = cudaMemcpy(out, n, 6 * sizeof *n, cudaMemcpyDeviceToHost);
    cudaFree(n);
    return e == cudaSuccess ? 0 : 2;
}
