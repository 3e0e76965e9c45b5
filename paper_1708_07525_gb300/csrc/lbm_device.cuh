// Device-side building blocks of the fused three-lattice step.
//
// Storage holds deviations from the rest equilibria (u = 0, rho = rho0,
// T = T0, C = C0) of Eqs. 20 and 28:
//   f'_i = f_i - w_i rho0,  g'_i = g_i - g_i^eq(T0, 0),  h'_i = h_i - h_i^eq(C0, 0).
// Every equilibrium moment that is linear in rho, T or C (Eqs. 14, 24, 25)
// has its rest part cancelled exactly by the shift, so the collision below
// is the paper's collision rewritten in these variables (no approximation);
// it keeps small numbers small, which is what FP32 / FP16 / BF16 storage needs.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

namespace lbm {

// D2Q9 velocities (Eq. 8), same ordering as the paper; D2Q5 uses q = 0..4.
//   q : 0  1  2  3  4  5  6  7  8
//   ex: 0  1  0 -1  0  1 -1 -1  1
//   ey: 0  0  1  0 -1  1  1 -1 -1
__host__ __device__ constexpr int ex_of(int q) {
    return q == 1 || q == 5 || q == 8 ? 1 : (q == 3 || q == 6 || q == 7 ? -1 : 0);
}
__host__ __device__ constexpr int ey_of(int q) {
    return q == 2 || q == 5 || q == 6 ? 1 : (q == 4 || q == 7 || q == 8 ? -1 : 0);
}
__host__ __device__ constexpr int opp_of(int q) {
    return q == 0 ? 0 : (q <= 4 ? ((q + 1) & 3) + 1 : ((q - 3) & 3) + 5);
}
static_assert(opp_of(1) == 3 && opp_of(3) == 1 && opp_of(2) == 4 && opp_of(4) == 2, "opp");
static_assert(opp_of(5) == 7 && opp_of(7) == 5 && opp_of(6) == 8 && opp_of(8) == 6, "opp");

// D2Q9 weights (Eq. 20).
__host__ __device__ constexpr double w9_of(int q) {
    return q == 0 ? 4.0 / 9.0 : (q <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
}

// Plane index of each lattice inside the 19-plane state: f 0..8, g 9..13, h 14..18.
constexpr int QF = 0, QG = 9, QH = 14, NQ = 19;

// ---- storage conversions -------------------------------------------------------
// 32-bit mixing function (the MurmurHash3 finaliser): random bits for stochastic rounding.
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x85EBCA6Bu;
    x ^= x >> 13;
    x *= 0xC2B2AE35u;
    x ^= x >> 16;
    return x;
}

template <typename R> __device__ __forceinline__ R sqrt_(R x);
template <> __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
template <> __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
template <typename R> __device__ __forceinline__ bool finite_(R x);
template <> __device__ __forceinline__ bool finite_(float x) { return fabsf(x) <= 3.402823466e38f; }
template <> __device__ __forceinline__ bool finite_(double x) { return fabs(x) <= 1.7976931348623157e308; }

// st() rounds to nearest even; st_sr() rounds stochastically (up with probability
// equal to the distance to the lower neighbour in ulps), so that the expected stored
// value equals the computed one.  With 8-11 significand bits, rounding to nearest
// makes per-step changes smaller than half an ulp vanish (the state stagnates);
// stochastic rounding keeps them on average.
// ld_nc() reads through the non-coherent read-only path (__ldg).  gather_local() uses
// it: the in-place even step loads and stores the same array, and with coherent loads
// it was compiled to 98 registers (25 % occupancy) against 64 with ld_nc (GB300,
// 4096^2 FP32 in-place step 516 -> 483 us).  Valid there because each thread writes
// only the locations it has itself read before, and reads nothing another thread of
// the launch writes.  (For the pulls of the odd step the same change cost registers.)
template <typename S> struct Store;
template <> struct Store<double> {
    static constexpr bool kLow = false;
    __device__ static double ld(const double* p) { return *p; }
    __device__ static double ld_nc(const double* p) { return __ldg(p); }
    __device__ static void st(double* p, double v) { *p = v; }
    __device__ static void st_sr(double* p, double v, uint32_t) { *p = v; }
};
template <> struct Store<float> {
    static constexpr bool kLow = false;
    __device__ static float ld(const float* p) { return *p; }
    __device__ static float ld_nc(const float* p) { return __ldg(p); }
    __device__ static void st(float* p, float v) { *p = v; }
    __device__ static void st_sr(float* p, float v, uint32_t) { *p = v; }
};
template <> struct Store<__nv_bfloat16> {
    static constexpr bool kLow = true;
    __device__ static float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    __device__ static float ld_nc(const __nv_bfloat16* p) { return __bfloat162float(__ldg(p)); }
    __device__ static void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
    __device__ static void st_sr(__nv_bfloat16* p, float v, uint32_t r) {
        // bfloat16 is the top half of the float: add 16 random bits (r < 2^16) below it,
        // truncate (on the sign-magnitude encoding this rounds |v| away from zero with
        // the right odds).  v must be finite (put() routes non-finite nodes to st()).
        const uint32_t b = __float_as_uint(v) + r;
        *p = __ushort_as_bfloat16((unsigned short)(b >> 16));
    }
};
// FP16 holds the deviations scaled by 2^12 (exact in both directions), so that
// deviations down to ~1.5e-8 sit in FP16's normal range (11 significant bits)
// instead of its subnormals; |deviation| must stay below 16 (65504 / 2^12).
template <> struct Store<__half> {
    static constexpr bool kLow = true;
    static constexpr float kScale = 4096.0f, kInvScale = 1.0f / 4096.0f;
    __device__ static float ld(const __half* p) { return __half2float(*p) * kInvScale; }
    __device__ static float ld_nc(const __half* p) { return __half2float(__ldg(p)) * kInvScale; }
    __device__ static void st(__half* p, float v) { *p = __float2half_rn(v * kScale); }
    __device__ static void st_sr(__half* p, float v, uint32_t r) {
        // In FP16's normal range the 13 float mantissa bits below the 10 kept ones are
        // the fraction of an FP16 ulp: add 13 random bits there, then truncate.  v must
        // be finite (put() routes non-finite nodes to st()).
        const uint32_t b = __float_as_uint(v * kScale) + (r & 0x1FFFu);
        *p = __float2half_rz(__uint_as_float(b));
    }
};

// Store one of a node's populations: stochastic rounding for 16-bit storage when
// sr is set (see sr_node).  The random bits come from a per-node linear
// congruential stream (the 32-bit constants of Numerical Recipes) seeded by node_seed(); only its high
// 16 bits are used, which is enough for rounding decisions and costs one
// multiply-add per value.
template <typename S, typename R>
__device__ __forceinline__ void put(S* p, R v, int sr, uint32_t& state, int) {
    if (Store<S>::kLow && sr) {
        state = state * 1664525u + 1013904223u;
        Store<S>::st_sr(p, v, state >> 16);
    } else {
        Store<S>::st(p, v);
    }
}

// Whether a node's post-collision values are stored with stochastic rounding: 16-bit
// storage with rounding enabled and all 19 values finite (one check on their sum
// instead of one per value; a node holding a NaN or an infinity is rounded to
// nearest, which keeps it non-finite for the residual's divergence check).
template <typename S, typename R>
__device__ __forceinline__ int sr_node(int sr, const R f[9], const R g[5], const R h[5]) {
    if (!Store<S>::kLow || !sr) return 0;
    R s = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]));
    s += ((f[8] + g[0]) + (g[1] + g[2])) + ((g[3] + g[4]) + (h[0] + h[1]));
    s += (h[2] + h[3]) + h[4];
    return finite_(s) ? 1 : 0;
}

// Per-node seed of the random stream: a hash of the node's index and of the bits of
// two of its pre-collision populations.  The populations change from step to step,
// so the stream does too, with no step counter (graph replay stays valid) and the
// same result whenever the same state is stepped (runs are reproducible).
template <typename R>
__device__ __forceinline__ uint32_t node_seed(size_t node, R a, R b) {
    const uint32_t ia = __float_as_uint((float)a), ib = __float_as_uint((float)b);
    return mix32(ia ^ mix32(ib ^ mix32((uint32_t)node ^ (uint32_t)(node >> 32) * 0x27D4EB2Fu)));
}

// ---- arithmetic with every rounding written out ------------------------------------------
// One node's step is written with these operations only, so that its result does not hang
// on which products and sums a compiler fuses: the one-node kernels, the kernels with two
// nodes per thread and the batch kernels give the same bits, whatever surrounds the
// arithmetic.  fma_(a, b, c) = a b + c and fnma_(a, b, c) = c - a b round once.
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float fnma_(float a, float b, float c) { return __fmaf_rn(-a, b, c); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double fnma_(double a, double b, double c) { return __fma_rn(-a, b, c); }

// f2: the FP32 values of one quantity at two nodes, computed with the packed FP32x2
// instructions of sm_100 and later (one add, multiply or fused multiply-add for both
// nodes; each component rounds as the scalar operation does).  Constants stay scalar and
// are written R(c): an instruction takes one value for both components as it takes an
// immediate, where a pair of constants has to be brought into registers first.
struct f2 {
    float2 v;
    f2() = default;
    __host__ __device__ f2(float2 a) : v(a) {}
    template <typename T, typename std::enable_if<std::is_arithmetic<T>::value, int>::type = 0>
    __host__ __device__ explicit f2(T s) : v(make_float2((float)s, (float)s)) {}
};
#ifdef __CUDACC__
__device__ __forceinline__ f2 add_(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 sub_(f2 a, f2 b) {
    return f2(__ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v));   // round(a - b) exactly
}
__device__ __forceinline__ f2 mul_(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 fma_(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ f2 fnma_(f2 a, f2 b, f2 c) {
    return f2(__ffma2_rn(make_float2(-a.v.x, -a.v.y), b.v, c.v));
}
__device__ __forceinline__ float round_up_ones(float x, float y);
__device__ __forceinline__ f2 round_up_ones(f2 x, f2 y) {
    return f2(make_float2(round_up_ones(x.v.x, y.v.x), round_up_ones(x.v.y, y.v.y)));
}
#endif
}  // namespace lbm
#include "lbm_roots.cuh"
namespace lbm {

// sqrt(x) and 1 / x of a normal, finite x > 0.
//   FP32: CUDA's root and division in the one-node kernels, which have all loads issued by
//   the time these functions' branches come up (within one basic block the compiler
//   put loads between the sums that they feed: a 256^2 step took 4.5 instead of 3.4 us).
//   f2: per component, or (FLAT) without a branch for both at once from the special-function
//   unit's approximation (lbm_roots.cuh): the same bits, rounded to nearest.
//   FP64: the binomial series of (1 - e)^(-1/2) and (1 - e)^(-1) to second order in the
//   error e of the approximation (below 2^-19): within one unit of the rounded result, in 5
//   and 3 operations.
__device__ __forceinline__ float rsqrt_seed(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float rcp_seed(float x) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ double rsqrt_seed(double x) { double y; asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x)); return y; }
__device__ __forceinline__ double rcp_seed(double x) { double y; asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x)); return y; }

template <bool FLAT> __device__ __forceinline__ float sqrt_pos(float x) { return sqrtf(x); }
template <bool FLAT> __device__ __forceinline__ float rcp_pos(float x) { return 1.0f / x; }
template <bool FLAT> __device__ __forceinline__ double sqrt_pos(double x) {
    const double y = rsqrt_seed(x), g = mul_(x, y), e = fnma_(g, y, 1.0);
    return fma_(mul_(g, e), fma_(e, 0.375, 0.5), g);
}
template <bool FLAT> __device__ __forceinline__ double rcp_pos(double x) {
    const double y = rcp_seed(x), e = fnma_(x, y, 1.0);
    return fma_(y, fma_(e, e, e), y);
}
#ifdef __CUDACC__
template <bool FLAT> __device__ __forceinline__ f2 sqrt_pos(f2 x) {
    if (!FLAT) return f2(make_float2(sqrtf(x.v.x), sqrtf(x.v.y)));
    return sqrt_from(x, f2(make_float2(rsqrt_seed(x.v.x), rsqrt_seed(x.v.y))));
}
template <bool FLAT> __device__ __forceinline__ f2 rcp_pos(f2 x) {
    if (!FLAT) return f2(make_float2(1.0f / x.v.x, 1.0f / x.v.y));
    return rcp_from(x, f2(make_float2(rcp_seed(x.v.x), rcp_seed(x.v.y))));
}
#endif
// Added to |v|^2 under the root, which is then never zero, and whose residual in Markstein's
// sequence is never subnormal: far below half a unit of what the root is added to (Eq. 18's
// l0^2 >= 1/4 after a factor l1, Eq. 5's drag).
template <typename R> __device__ __forceinline__ R tiny_() { return R(1e-28); }
template <> __device__ __forceinline__ double tiny_<double>() { return 1e-300; }

// Compute type for a storage type: FP64 stays FP64, everything else is FP32.
template <typename S> struct Real { using type = float; };
template <> struct Real<double> { using type = double; };

// ---- per-instance constants (prepared on the host, passed by value) ------------
// The constants of the integer form of the FP64 collision (lbm_fixed.cuh).
// A positive constant c < 2^-B as the even integer c 2^(63 + B); fx_pair() and fx_one() shift their
// arguments by the other 3 - B bits.  `less` (of a pair or a lone constant) takes off what
// their offset-binary products hold too much, and adds the rounding.
template <int B> struct FxConst { unsigned long long c; };
struct FixedScalar {
    FxConst<0> b1, q1, b2, q2, p;   // r_1 / 2, (1 - r_1 / 2) / 2 and the same for r_2; the factor of
                                    // the scalar's sum in the third moment, |r_3 nc3 / (20 cap)|
    FxConst<3> b3;                  // r_3 / 20
    FxConst<1> b4;                  // r_4 / 4
    long long less1, less2, less3, less4;
    int p_neg;                      // the sign of p's factor
};
struct FixedCoef {
    int on;                         // 0: p's factor does not lie below 1 (extreme varpi / cap), FP64 instead
    FxConst<3> k1, k4F, k6F;
    FxConst<2> k1F, k2, k2F, k4, k6, k8F, sixth;
    FxConst<1> k7, k7F, k8;
    long long less1, less2, less4, less6, less7, less8, less_sixth;
    FixedScalar zs, es;
};

struct NoFixed {};
template <typename R> struct FixedOf { using type = NoFixed; };
template <> struct FixedOf<double> { using type = FixedCoef; };

template <typename R>
struct CoefScalar {
    R b1, q1, b2, q2, b3, b4;
};
template <typename R>
struct Coef {
    R T0, C0;
    R inv_sigma, inv_eps;      // Eq. 26
    R eps, half_eps;           // eps of Eqs. 5, 14, 15, 19
    R inv_eps_f;               // 1/eps for the flow equilibria (Eqs. 14, 15)
    R gbT, gbC, Gx;            // Eq. 6 (+ optional constant Gx)
    R l0, l0sq, l1;            // Eq. 19
    R ndrag_lin, ndrag_quad;   // -eps nu / K and -eps F_eps / sqrt(K) (Eq. 5)
    R half_epsGx, epsGx;       // eps Gx / 2, eps Gx
    // Relaxation and forcing of the moments with the factors of M^-1 (Eq. 10): Lambda_k
    // and 1 - Lambda_k / 2 times 1/36 (e, and 3/36 for eps), 1/12 (q), 1/4 (nu), see
    // collide_flow().  s_rho and s_j play no role: rho is conserved, and the momentum gains
    // exactly F whatever s_j (Eq. 17).
    R k1, k1F, k2, k2F, k4, k4F, k6, k6F, k7, k7F, k8, k8F;
    // Theta, Q and the source factors with those of N^-1 (Eqs. 21, 22, 27): r_1 / 2,
    // -(1 - r_1 / 2) / 2, the same for r_2, r_3 / 20, r_4 / 4.
    CoefScalar<R> zs, es;
    R nc3T, nc3C;              // 4 sigma - 5 varpi, 4 eps - 5 varpi (Eqs. 24, 25)
    // Per wall side (0 left, 1 right, 2 bottom, 3 top): 2 w~ (Phi_w - Phi0) with
    // w~ = varpi / 4, the anti-bounce-back constant in deviations.
    R wallT[4], wallC[4];
    int dirichlet_mask;        // bit s set: side s is Dirichlet for g and h, else adiabatic
    int sr;                    // 1: stochastic rounding when storing 16-bit populations
    // Moving walls: wmom[s] = 2 rho0 u_w / c_s^2 of side s; moving = 1 if any is nonzero.
    R wmom[4][2];
    int moving;
    // Spatially varying porous medium: NULL, or planes [2][ny][pitch] of (eps, K); then
    // the porous constants above are recomputed per node (porous_at).
    const R* poro;
    R nu, varpi5;              // fluid viscosity of Eq. 5, 5 varpi of Eq. 25
    // Walls with nodes on them (Sec. 3.3, nee = 1): wall values Phi_w - Phi0 by side,
    // Bi / L of convective sides (Eq. 39; 0 otherwise), wall velocities, and the D2Q5
    // equilibria as g_eq,0 = a0 Phi, g_eq,i = a1 Phi + (e_i . u) Phi / 2 (i = 1..4) with
    // a0 = (cap - c3) / 5, a1 = cap / 5 + c3 / 20 (N^-1 n_eq of Eqs. 24-25 / 30-31).
    int nee;
    // Added to a node's storage index to key its stochastic-rounding stream: 0 for a
    // cavity; for a slab of a cavity split along y, the offset that makes the key the
    // node's index in the undivided cavity (so a split run rounds as the whole one does).
    long long seed_off;
    R TwP[4], CwP[4];
    R bT[4], bC[4];
    R uwall[4][2];
    R aT0, aT1, aC0, aC1;
    typename FixedOf<R>::type fx;
};



// The constants of node `self` of a cavity with a porosity / permeability field:
// eps and K from the field, F_eps from Eq. 7, l0 and l1 from Eq. 19, the drag
// coefficients of Eq. 5 and the n_eq,3 factor of Eq. 25.
template <typename R>
__device__ __forceinline__ void porous_at(Coef<R>& c, size_t self, size_t plane) {
    const R e = c.poro[self], K = c.poro[plane + self];
    const R Fe = R(1.75) / sqrt_(R(150) * e * e * e);
    c.eps = e;
    c.half_eps = R(0.5) * e;
    c.inv_eps = R(1) / e;
    c.inv_eps_f = c.inv_eps;
    c.ndrag_lin = -(e * c.nu / K);
    c.ndrag_quad = -(e * Fe / sqrt_(K));
    c.half_epsGx = c.half_eps * c.Gx;
    c.epsGx = e * c.Gx;
    c.l0 = R(0.5) * (R(1) - R(0.5) * c.ndrag_lin);
    c.l0sq = c.l0 * c.l0;
    c.l1 = R(-0.5) * c.ndrag_quad;
    c.nc3C = R(4) * e - c.varpi5;
    c.aC0 = (e + c.nc3C) * R(0.2);
    c.aC1 = e * R(0.2) - c.nc3C * R(0.05);
    if constexpr (std::is_same<R, double>::value) c.fx.on = 0;   // its constants are the uniform medium's
}

// Macroscopic quantities of one node from pre-collision deviations.
template <typename R>
struct Macro {
    R rho, ux, uy, Tp, Cp, Fx, Fy;   // rho' (deviation), u, T - T0, C - C0, F
};

// Sums and differences of opposite populations of one lattice; collide_flow() and
// collide_d2q5() need the ones that macro() forms again (the compiler shares them).
template <typename R>
__device__ __forceinline__ R sum5(const R d[5]) {
    return add_(d[0], add_(add_(d[1], d[3]), add_(d[2], d[4])));
}

template <bool FLAT = false, typename K, typename R>
__device__ __forceinline__ Macro<R> macro(const Coef<K>& c, const R f[9], const R g[5],
                                          const R h[5]) {
    Macro<R> o;
    const R p = add_(add_(f[1], f[3]), add_(f[2], f[4])), d = add_(add_(f[5], f[7]), add_(f[6], f[8]));
    const R D57 = sub_(f[5], f[7]), D68 = sub_(f[6], f[8]);
    const R jx = add_(add_(sub_(f[1], f[3]), D57), sub_(f[8], f[6]));
    const R jy = add_(sub_(f[2], f[4]), add_(D57, D68));
    o.rho = add_(f[0], add_(p, d));                                  // Eq. 16
    o.Tp = mul_(sum5(g), R(c.inv_sigma));                               // Eq. 26
    o.Cp = mul_(sum5(h), R(c.inv_eps));
    const R Gy = fma_(R(c.gbT), o.Tp, mul_(R(c.gbC), o.Cp));               // Eq. 6
    const R vx = add_(jx, R(c.half_epsGx));                             // Eq. 19, rho0 = 1
    const R vy = fma_(R(c.half_eps), Gy, jy);
    const R vm = sqrt_pos<FLAT>(fma_(vx, vx, fma_(vy, vy, tiny_<R>())));
    const R inv_den = rcp_pos<FLAT>(add_(R(c.l0), sqrt_pos<FLAT>(fma_(R(c.l1), vm, R(c.l0sq)))));   // Eq. 18
    o.ux = mul_(vx, inv_den);
    o.uy = mul_(vy, inv_den);
    const R ndrag = fma_(R(c.ndrag_quad), mul_(vm, inv_den), R(c.ndrag_lin));        // Eq. 5, |u| = |v| / den
    o.Fx = fma_(ndrag, o.ux, R(c.epsGx));
    o.Fy = fma_(ndrag, o.uy, mul_(R(c.eps), Gy));
    return o;
}

// D2Q5 collision (Eq. 21 / 22 with Eq. 24 / 25 and the moment-space source
// (0, X_x, X_y, 0, 0) of Eq. 27), written as d* = d - N^-1 [Theta (n - n_eq)
// - (I - Theta/2) S] so that only the change is rounded; the zeroth moment
// (cap * Phi) is conserved exactly, its change is set to zero.  N^-1 uses the
// orthogonality of N: N^-1 = N^T D^-1, D = diag(5, 2, 2, 20, 4), whose factors r carries.
// Pp = Phi - Phi0, nc3 = 4 cap - 5 varpi, (Px, Py) = Phi u, (Xx, Xy) its change.
template <typename K, typename R>
__device__ __forceinline__ void collide_d2q5(R d[5], R Pp, R Px, R Py, R Xx, R Xy,
                                             const CoefScalar<K>& r, K nc3) {
    const R p13 = add_(d[1], d[3]), p24 = add_(d[2], d[4]);
    const R n3 = fma_(R(-4), d[0], add_(p13, p24));
    const R n4 = sub_(p13, p24);
    const R b1 = fma_(R(r.b1), sub_(sub_(d[1], d[3]), Px), mul_(R(r.q1), Xx));
    const R b2 = fma_(R(r.b2), sub_(sub_(d[2], d[4]), Py), mul_(R(r.q2), Xy));
    const R b3 = mul_(R(r.b3), fma_(R(nc3), Pp, n3));
    const R b4 = mul_(R(r.b4), n4);
    const R X = add_(b3, b4), Y = sub_(b3, b4);
    d[0] = fma_(R(4), b3, d[0]);
    d[1] = sub_(d[1], add_(X, b1));
    d[2] = sub_(d[2], add_(Y, b2));
    d[3] = sub_(d[3], sub_(X, b1));
    d[4] = sub_(d[4], sub_(Y, b2));
}

// The collision of one node, in place on the deviations f, g, h: collide_flow (the D2Q9
// part), then collide_scalars; collide() does both.  hist = (T u_x, T u_y, C u_x, C u_y)
// at the previous step; updated.  The D2Q9 part is Eq. 10 written as
// f* = f - M^-1 [Lambda (m - m_eq) - (I - Lambda/2) S] (only the change is rounded; the
// density moment is conserved exactly).  In that change (alpha1 = 1, alpha2 = -3, rho0 = 1)
//   e:   m_1 - m_eq,1 = 4 fd + fa - 2 f0 - 3 u^2/eps   (rho cancels; fa, fd: the sums over the
//   eps: m_2 - m_eq,2 = 3 (f0 - fa + u^2/eps)            axis and the diagonal populations)
//   j:   s_3 (j_x - u_x) - (1 - s_3/2) F_x = -F_x, since u = j + F/2 (Eq. 17) is what
//        macro() solves; the same in y
// and a_k below is the k-th component times the factor of M^-1 = M^T diag(1/9, 1/36, 1/36,
// 1/6, 1/12, 1/6, 1/12, 1/4, 1/4).  Opposite populations share their sums.  With the root
// of |u| and a division gone from macro(), a node takes 179 FP64 instructions instead of
// 250, and 170 FP32 operations.
template <typename K, typename R>
__device__ __forceinline__ void collide_flow(const Coef<K>& c, const Macro<R>& M, R f[9]) {
    const R ux = M.ux, uy = M.uy, Fx = M.Fx, Fy = M.Fy;
    const R p13 = add_(f[1], f[3]), d13 = sub_(f[1], f[3]), p24 = add_(f[2], f[4]), d24 = sub_(f[2], f[4]);
    const R p57 = add_(f[5], f[7]), D57 = sub_(f[5], f[7]), p68 = add_(f[6], f[8]), D68 = sub_(f[6], f[8]);
    const R fa = add_(p13, p24), fd = add_(p57, p68);
    const R uxe = mul_(ux, R(c.inv_eps_f)), uye = mul_(uy, R(c.inv_eps_f));
    const R A = mul_(ux, uxe), B = mul_(uy, uye);
    const R P = mul_(uxe, Fx), Q = mul_(uye, Fy);
    const R u2 = add_(A, B), uF = add_(P, Q);
    const R a1 = fma_(R(c.k1), fma_(R(4), fd, fma_(R(-2), f[0], fma_(R(-3), u2, fa))), mul_(R(c.k1F), uF));
    const R a2 = fma_(R(c.k2), sub_(add_(f[0], u2), fa), mul_(R(c.k2F), uF));
    const R a4 = fma_(R(c.k4), fma_(R(-2), d13, add_(sub_(D57, D68), ux)), mul_(R(c.k4F), Fx));
    const R a6 = fma_(R(c.k6), fma_(R(-2), d24, add_(add_(D57, D68), uy)), mul_(R(c.k6F), Fy));
    const R a7 = fma_(R(c.k7), sub_(sub_(p13, A), sub_(p24, B)), mul_(R(c.k7F), sub_(P, Q)));
    const R a8 = fma_(R(c.k8), sub_(sub_(p57, p68), mul_(ux, uye)), mul_(R(c.k8F), fma_(uxe, Fy, mul_(uye, Fx))));
    const R gx = mul_(Fx, R(1.0 / 6.0)), gy = mul_(Fy, R(1.0 / 6.0));
    const R ax = fma_(R(2), a2, a1), X = sub_(ax, a7), Y = add_(ax, a7);
    const R px = fma_(R(2), a4, gx), py = fma_(R(2), a6, gy);
    const R dg = fma_(R(2), a1, a2), U = add_(dg, a8), V = sub_(dg, a8);
    const R qx = sub_(gx, a4), qy = sub_(gy, a6), r = add_(qx, qy), t = sub_(qx, qy);
    f[0] = fma_(R(4), sub_(a1, a2), f[0]);
    f[1] = add_(f[1], add_(X, px));
    f[2] = add_(f[2], add_(Y, py));
    f[3] = add_(f[3], sub_(X, px));
    f[4] = add_(f[4], sub_(Y, py));
    f[5] = add_(f[5], sub_(r, U));
    f[6] = sub_(f[6], add_(V, t));
    f[7] = sub_(f[7], add_(U, r));
    f[8] = add_(f[8], sub_(t, V));
}

// The two D2Q5 collisions of a node (Eqs. 21-22) with the source of Eq. 27; hist is
// read and updated.
template <typename K, typename R>
__device__ __forceinline__ void collide_scalars(const Coef<K>& c, const Macro<R>& M, R g[5], R h[5],
                                                R hist[4]) {
    // Eq. 27 with d(Phi u)/dt = (Phi u)|t - (Phi u)|t-1 (Sec. 3.2)
    const R T = add_(R(c.T0), M.Tp), C = add_(R(c.C0), M.Cp);
    const R Tux = mul_(T, M.ux), Tuy = mul_(T, M.uy), Cux = mul_(C, M.ux), Cuy = mul_(C, M.uy);
    collide_d2q5(g, M.Tp, Tux, Tuy, sub_(Tux, hist[0]), sub_(Tuy, hist[1]), c.zs, c.nc3T);
    collide_d2q5(h, M.Cp, Cux, Cuy, sub_(Cux, hist[2]), sub_(Cuy, hist[3]), c.es, c.nc3C);
    hist[0] = Tux;
    hist[1] = Tuy;
    hist[2] = Cux;
    hist[3] = Cuy;
}

}  // namespace lbm
#include "lbm_fixed.cuh"
namespace lbm {

template <bool FLAT = false, typename K, typename R>
__device__ __forceinline__ void collide(const Coef<K>& c, R f[9], R g[5], R h[5], R hist[4]) {
    if constexpr (std::is_same<R, double>::value) {
        if (c.fx.on) {
            collide_fixed(c, f, g, h, hist);
            return;
        }
    }
    const Macro<R> M = macro<FLAT>(c, f, g, h);
    collide_flow(c, M, f);
    collide_scalars(c, M, g, h, hist);
}

// ---- SplitMix64 (Steele, Lea & Flood 2014): k-th output of a generator seeded with s
__host__ __device__ inline uint64_t splitmix64_at(uint64_t seed, uint64_t k) {
    uint64_t z = seed + (k + 1u) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__host__ __device__ inline double uniform01(uint64_t seed, uint64_t k) {
    return (double)(splitmix64_at(seed, k) >> 11) * (1.0 / 9007199254740992.0);
}

}  // namespace lbm
