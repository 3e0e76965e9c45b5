// The sequences of lbm_roots.cuh on the CPU in FP32, from seeds that are off by up to `off`
// units of the rounded value, for every significand of two binades.
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
static inline uint32_t __float_as_uint(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }
static inline float __uint_as_float(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
namespace lbm {
static inline float mul_(float a, float b) { return a * b; }
static inline float fma_(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float fnma_(float a, float b, float c) { return std::fmaf(-a, b, c); }
}  // namespace lbm
#include "lbm_roots.cuh"

static float moved(float x, int units) { return __uint_as_float(__float_as_uint(x) + units); }

// wrong[0]: roots, wrong[1]: reciprocals that are not the rounded ones
extern "C" void check_roots(int off, long long wrong[2]) {
    wrong[0] = wrong[1] = 0;
    for (uint32_t b = 0x3F800000u; b < 0x40800000u; ++b) {
        const float x = __uint_as_float(b);
        const float root = (float)std::sqrt((double)x), rcp = 1.0f / x;
        const float seed_root = (float)(1.0 / std::sqrt((double)x));
        for (int k = -off; k <= off; ++k) {
            wrong[0] += lbm::sqrt_from(x, moved(seed_root, k)) != root;
            wrong[1] += lbm::rcp_from(x, moved(rcp, k)) != rcp;
        }
    }
}
