// The FP64 collision with its linear part in 64-bit integers.
//
// GB300's FP64 pipe takes a warp's instruction every 64 clocks per SM sub-partition (measured;
// the number of active lanes makes no difference), its integer units one per clock or two.
// Most of a node's 179 FP64 operations are sums of its own populations.  Here a lattice's
// populations are brought to integers of one scale per node and lattice (block fixed point:
// the largest magnitude gets 57 bits), in which sums, differences and doublings are exact
// and cost two instructions; products with the relaxation constants are 64 x 64 -> 128 bit
// integer products; and what is not linear (Eqs. 5, 6, 18: two roots and a reciprocal; the
// products of Eqs. 14, 15 and T u, C u) stays in FP64: 53 instructions per node (ncu).
// Error: a population is rounded at 2^-58 of the node's largest (exact when within 2^4 of it;
// the FP64 sums rounded at 2^-53 of their operands at every step), sums are exact, and a
// result is rounded once, to nearest, when it goes back to FP64.  rho, T and C are
// conserved exactly by the update, up to that last rounding.
// A node that holds an infinity or a NaN becomes NaN as a whole.
#pragma once
namespace lbm {

// The smallest scale: a zero lies more than 2^57 below it (fx_in), and nothing of a cavity
// does (2^-959).
constexpr int FX_LOW = 64;

__device__ __forceinline__ int fx_exp(double x) {          // biased exponent
    return (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7FF;
}

// x as an integer, x 2^(1079 - E) for a biased exponent E: |result| < 2^57 times 2^(e - E) for
// an x of exponent e.  Bits that do not fit set the last one (von Neumann's rounding: within
// one unit and without bias; rounding halves up was not, since half of the values that lose
// one bit are halves: T drifted by 7e-18 a step).
__device__ __forceinline__ long long fx_in(double x, int E) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7FF;
    const unsigned long long m = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 10;
    // m 2^-6 at e = E; a zero (and all else below 2^-57 of the scale) ends as 0
    int s = E - e + 6;
    s = s > 63 ? 63 : s;
    unsigned long long v = m >> s;
    if (s < 63 && (v << s) != m) v |= 1;
    const long long n = (long long)b >> 63;
    return ((long long)v ^ n) - n;
}

// The FP64 value of v 2^(E - 1079), rounded to nearest even (0 below the normal numbers).
__device__ __forceinline__ double fx_out(long long v, int E) {
    const long long n = v >> 63;
    const unsigned long long a = (unsigned long long)((v ^ n) - n);
    const int z = __clzll((long long)a);
    const unsigned long long w = a << (z & 63);                     // top bit at 63
    unsigned long long r = w >> 11;                                 // 2^52 .. 2^53
    r += ((unsigned)w & 0x7FFu) + ((unsigned)r & 1u) > 0x400u;
    const int e = E + 6 - z;                                        // biased exponent less one
    if (a == 0 || e < 0) return 0.0;
    return __longlong_as_double((long long)((((unsigned long long)e << 52) + r) | ((unsigned long long)n << 63)));
}

// 4 v c + 2^62 (4 c), rounded down, |v| < 2^(60 + B): the high word of an unsigned product, v in
// offset binary (a signed high word takes 17 instructions, an unsigned one 9).
template <int B> __device__ __forceinline__ unsigned long long fx_mul(long long v, FxConst<B> k) {
    return __umul64hi(((unsigned long long)v << (3 - B)) ^ (1ull << 63), k.c);
}
// v c + w d or v c - w d, and v c, without bias: the products come as quarters; what the
// floors cost is in `less`, and the parity of the result evens out the last one.  (Rounding
// down gave every flux of Eq. 21 half a unit, which summed over a cavity's width to an
// error in T of 3e-15.)
__device__ __forceinline__ long long fx_near(unsigned long long t, long long less) {
    const long long q = (long long)t - less;
    return (q + ((q >> 2) & 1)) >> 2;
}
template <int B, int D>
__device__ __forceinline__ long long fx_plus(long long v, FxConst<B> c, long long w, FxConst<D> d, long long less) {
    return fx_near(fx_mul(v, c) + fx_mul(w, d), less);
}
template <int B, int D>
__device__ __forceinline__ long long fx_minus(long long v, FxConst<B> c, long long w, FxConst<D> d, long long less) {
    return fx_near(fx_mul(v, c) - fx_mul(w, d), less);
}
template <int B> __device__ __forceinline__ long long fx_one(long long v, FxConst<B> c, long long less) {
    return ((long long)fx_mul(v, c) - less) >> 2;
}

// v 2^-d rounded, d >= 0: to a coarser scale.
__device__ __forceinline__ long long fx_shift(long long v, int d) {
    d = d > 63 ? 63 : d;
    return d ? ((v >> (d - 1)) + 1) >> 1 : v;
}

__device__ __forceinline__ int fx_max(int a, int b) { return a > b ? a : b; }

// u, F of Eqs. 18, 5 (macro() from the moments).
struct FixedMacro {
    double ux, uy, Fx, Fy;
};
__device__ __forceinline__ FixedMacro fixed_macro(const Coef<double>& c, double jx, double jy, double Tp, double Cp) {
    const double Gy = fma_(c.gbT, Tp, mul_(c.gbC, Cp));
    const double vx = add_(jx, c.half_epsGx), vy = fma_(c.half_eps, Gy, jy);
    const double vm = sqrt_pos<false>(fma_(vx, vx, fma_(vy, vy, tiny_<double>())));
    const double inv_den = rcp_pos<false>(add_(c.l0, sqrt_pos<false>(fma_(c.l1, vm, c.l0sq))));
    FixedMacro M;
    M.ux = mul_(vx, inv_den);
    M.uy = mul_(vy, inv_den);
    const double ndrag = fma_(c.ndrag_quad, mul_(vm, inv_den), c.ndrag_lin);
    M.Fx = fma_(ndrag, M.ux, c.epsGx);
    M.Fy = fma_(ndrag, M.uy, mul_(c.eps, Gy));
    return M;
}

// The largest exponents of a lattice, at least FX_LOW, and its populations on that scale.
template <int N> __device__ __forceinline__ int fixed_in(const double* d, long long* v) {
    int E = FX_LOW;
#pragma unroll
    for (int q = 0; q < N; ++q) E = fx_max(E, fx_exp(d[q]));
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = fx_in(d[q], E);
    return E;
}
template <int N> __device__ __forceinline__ void fixed_nan(double* d) {
#pragma unroll
    for (int q = 0; q < N; ++q) d[q] = __longlong_as_double(0x7FF8000000000000ll);
}
constexpr int FX_TOP = 0x7FF - 8;        // exponents from here on count as not finite

// The D2Q9 update (collide_flow): f as integers v of scale E; `top` the largest exponent of the
// node so far.  The populations leave in f.
__device__ __forceinline__ void fixed_flow(const Coef<double>& c, const FixedMacro& M, double f[9], long long v[9],
                                           int E, int top) {
    const FixedCoef& k = c.fx;
    const double ux = M.ux, uy = M.uy, Fx = M.Fx, Fy = M.Fy;
    const double uxe = mul_(ux, c.inv_eps_f), uye = mul_(uy, c.inv_eps_f);
    const double dA = mul_(ux, uxe), dB = mul_(uy, uye), dXY = mul_(ux, uye);
    const double dP = mul_(uxe, Fx), dQ = mul_(uye, Fy), dW = fma_(uxe, Fy, mul_(uye, Fx));
    // a scale that holds u, F and their products too (a bit of headroom above it)
    const int most = fx_max(fx_max(fx_max(fx_exp(ux), fx_exp(uy)), fx_max(fx_exp(Fx), fx_exp(Fy))),
                            fx_max(fx_max(fx_exp(dA), fx_exp(dB)), fx_max(fx_exp(dW), fx_max(fx_exp(dP), fx_exp(dQ)))));
    if (fx_max(top, most) >= FX_TOP) {
        fixed_nan<9>(f);
        return;
    }
    if (most - 1 > E) {
        for (int q = 0; q < 9; ++q) v[q] = fx_shift(v[q], most - 1 - E);
        E = most - 1;
    }
    const long long d13 = v[1] - v[3], d24 = v[2] - v[4], D57 = v[5] - v[7], D68 = v[6] - v[8];
    const long long p13 = v[1] + v[3], p24 = v[2] + v[4], p57 = v[5] + v[7], p68 = v[6] + v[8];
    const long long fa = p13 + p24, fd = p57 + p68;
    const long long A = fx_in(dA, E), B = fx_in(dB, E), P = fx_in(dP, E), Q = fx_in(dQ, E);
    const long long iFx = fx_in(Fx, E), iFy = fx_in(Fy, E), u2 = A + B, uF = P + Q;
    const long long a1 = fx_minus(4 * fd + fa - 2 * v[0] - 3 * u2, k.k1, uF, k.k1F, k.less1);
    const long long a2 = fx_plus(v[0] - fa + u2, k.k2, uF, k.k2F, k.less2);
    const long long a4 = fx_plus(D57 - D68 - 2 * d13 + fx_in(ux, E), k.k4, iFx, k.k4F, k.less4);
    const long long a6 = fx_plus(D57 + D68 - 2 * d24 + fx_in(uy, E), k.k6, iFy, k.k6F, k.less6);
    const long long a7 = fx_minus(p13 - p24 - A + B, k.k7, P - Q, k.k7F, k.less7);
    const long long a8 = fx_minus(p57 - p68 - fx_in(dXY, E), k.k8, fx_in(dW, E), k.k8F, k.less8);
    const long long gx = fx_one(iFx, k.sixth, k.less_sixth), gy = fx_one(iFy, k.sixth, k.less_sixth);
    const long long ax = a1 + 2 * a2, X = ax - a7, Y = ax + a7;
    const long long px = 2 * a4 + gx, py = 2 * a6 + gy;
    const long long dg = 2 * a1 + a2, U = dg + a8, V = dg - a8;
    const long long qx = gx - a4, qy = gy - a6, r = qx + qy, t = qx - qy;
    f[0] = fx_out(v[0] + 4 * (a1 - a2), E);
    f[1] = fx_out(v[1] + X + px, E);
    f[2] = fx_out(v[2] + Y + py, E);
    f[3] = fx_out(v[3] + X - px, E);
    f[4] = fx_out(v[4] + Y - py, E);
    f[5] = fx_out(v[5] + r - U, E);
    f[6] = fx_out(v[6] - V - t, E);
    f[7] = fx_out(v[7] - U - r, E);
    f[8] = fx_out(v[8] + t - V, E);
}

// One D2Q5 lattice (collide_d2q5): d as integers v of scale E, their sum s; Phi the scalar's value;
// hist Phi u before, replaced by Phi u now.  The populations leave in d.
__device__ __forceinline__ void fixed_scalar(const FixedScalar& r, double Phi, const FixedMacro& M, double d[5],
                                             long long v[5], int E, long long s, double hist[2], int top) {
    const double Px = mul_(Phi, M.ux), Py = mul_(Phi, M.uy), Qx = hist[0], Qy = hist[1];
    hist[0] = Px;
    hist[1] = Py;
    // a scale that holds the fluxes as well (a bit of headroom above it)
    const int most = fx_max(fx_max(fx_exp(Px), fx_exp(Py)), fx_max(fx_exp(Qx), fx_exp(Qy)));
    if (fx_max(top, most) >= FX_TOP) {
        fixed_nan<5>(d);
        return;
    }
    if (most - 1 > E) {
        for (int q = 0; q < 5; ++q) v[q] = fx_shift(v[q], most - 1 - E);
        s = fx_shift(s, most - 1 - E);
        E = most - 1;
    }
    const long long px = fx_in(Px, E), py = fx_in(Py, E);
    const long long p13 = v[1] + v[3], p24 = v[2] + v[4];
    const long long b1 = fx_minus(v[1] - v[3] - px, r.b1, px - fx_in(Qx, E), r.q1, r.less1);
    const long long b2 = fx_minus(v[2] - v[4] - py, r.b2, py - fx_in(Qy, E), r.q2, r.less2);
    const long long b3 = fx_plus(p13 + p24 - 4 * v[0], r.b3, r.p_neg ? -s : s, r.p, r.less3);
    const long long b4 = fx_one(p13 - p24, r.b4, r.less4);
    const long long X = b3 + b4, Y = b3 - b4;
    d[0] = fx_out(v[0] + 4 * b3, E);
    d[1] = fx_out(v[1] - X - b1, E);
    d[2] = fx_out(v[2] - Y - b2, E);
    d[3] = fx_out(v[3] - X + b1, E);
    d[4] = fx_out(v[4] - Y + b2, E);
}

// The momentum and a scalar's sum from integers.
__device__ __forceinline__ double fixed_jx(const long long v[9], int E) {
    return fx_out(v[1] - v[3] + v[5] - v[7] - v[6] + v[8], E);
}
__device__ __forceinline__ double fixed_jy(const long long v[9], int E) {
    return fx_out(v[2] - v[4] + v[5] - v[7] + v[6] - v[8], E);
}
__device__ __forceinline__ long long fixed_sum(const long long v[5]) {
    return v[0] + (v[1] + v[3]) + (v[2] + v[4]);
}

// collide() of one FP64 node with uniform porous constants (the same update; see
// collide_flow for the algebra).
__device__ __forceinline__ void collide_fixed(const Coef<double>& c, double f[9], double g[5], double h[5],
                                              double hist[4]) {
    long long v[9], vg[5], vh[5];
    const int E = fixed_in<9>(f, v), Eg = fixed_in<5>(g, vg), Eh = fixed_in<5>(h, vh);
    const long long sg = fixed_sum(vg), sh = fixed_sum(vh);
    const double Tp = mul_(fx_out(sg, Eg), c.inv_sigma), Cp = mul_(fx_out(sh, Eh), c.inv_eps);     // Eq. 26
    const FixedMacro M = fixed_macro(c, fixed_jx(v, E), fixed_jy(v, E), Tp, Cp);
    const int top = fx_max(fx_max(E, Eg), Eh);
    fixed_flow(c, M, f, v, E, top);
    fixed_scalar(c.fx.zs, add_(c.T0, Tp), M, g, vg, Eg, sg, hist, top);
    fixed_scalar(c.fx.es, add_(c.C0, Cp), M, h, vh, Eh, sh, hist + 2, top);
}

}  // namespace lbm
