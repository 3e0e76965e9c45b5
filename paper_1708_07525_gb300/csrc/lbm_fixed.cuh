// The FP64 collision with its linear part in 64-bit integers.
//
// GB300's FP64 pipe takes a warp's instruction every 64 clocks per SM sub-partition (measured;
// the number of active lanes makes no difference), its integer units one per clock or two.
// Most of a node's 179 FP64 operations are sums of its own populations.  Here a lattice's
// populations are brought to integers of one scale per node and lattice (block fixed point:
// the largest magnitude gets 57 bits), in which sums, differences and doublings are exact
// and cost two instructions; products with the relaxation constants are 64 x 64 -> 128 bit
// integer products; and what is not linear (Eqs. 5, 6, 18: two roots and a reciprocal; the
// products of Eqs. 14, 15 and T u, C u) stays in FP64: 45 operations.
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

// One D2Q5 lattice (collide_d2q5): d as integers of scale E, their sum s; (Px, Py) = Phi u now
// and (Qx, Qy) before.  The populations leave in d.
__device__ __forceinline__ void fixed_d2q5(double d[5], long long v[5], int E, long long s, double Px,
                                                    double Py, double Qx, double Qy,
                                                    const FixedScalar& r) {
    // a scale that holds the fluxes as well (a bit of headroom above it)
    const int need = fx_max(fx_max(fx_exp(Px), fx_exp(Py)), fx_max(fx_exp(Qx), fx_exp(Qy))) - 1;
    if (need > E) {
        for (int q = 0; q < 5; ++q) v[q] = fx_shift(v[q], need - E);
        s = fx_shift(s, need - E);
        E = need;
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

// collide() of one FP64 node with uniform porous constants (the same update; see
// collide_flow for the algebra).
__device__ __forceinline__ void collide_fixed(const Coef<double>& c, double f[9], double g[5],
                                                       double h[5], double hist[4]) {
    const FixedCoef& k = c.fx;
    int E = FX_LOW, Eg = FX_LOW, Eh = FX_LOW;
#pragma unroll
    for (int q = 0; q < 9; ++q) E = fx_max(E, fx_exp(f[q]));
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        Eg = fx_max(Eg, fx_exp(g[q]));
        Eh = fx_max(Eh, fx_exp(h[q]));
    }
    long long v[9], vg[5], vh[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        vg[q] = fx_in(g[q], Eg);
        vh[q] = fx_in(h[q], Eh);
    }
    const long long sg = vg[0] + (vg[1] + vg[3]) + (vg[2] + vg[4]), sh = vh[0] + (vh[1] + vh[3]) + (vh[2] + vh[4]);
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q] = fx_in(f[q], E);
    long long d13 = v[1] - v[3], d24 = v[2] - v[4], D57 = v[5] - v[7], D68 = v[6] - v[8];
    const double jx = fx_out(d13 + D57 - D68, E), jy = fx_out(d24 + D57 + D68, E);
    // macro(): Eqs. 26, 6, 19, 18, 5
    const double Tp = mul_(fx_out(sg, Eg), c.inv_sigma), Cp = mul_(fx_out(sh, Eh), c.inv_eps);
    const double Gy = fma_(c.gbT, Tp, mul_(c.gbC, Cp));
    const double vx = add_(jx, c.half_epsGx), vy = fma_(c.half_eps, Gy, jy);
    const double vm = sqrt_pos<false>(fma_(vx, vx, fma_(vy, vy, tiny_<double>())));
    const double inv_den = rcp_pos<false>(add_(c.l0, sqrt_pos<false>(fma_(c.l1, vm, c.l0sq))));
    const double ux = mul_(vx, inv_den), uy = mul_(vy, inv_den);
    const double ndrag = fma_(c.ndrag_quad, mul_(vm, inv_den), c.ndrag_lin);
    const double Fx = fma_(ndrag, ux, c.epsGx), Fy = fma_(ndrag, uy, mul_(c.eps, Gy));
    const double uxe = mul_(ux, c.inv_eps_f), uye = mul_(uy, c.inv_eps_f);
    const double dA = mul_(ux, uxe), dB = mul_(uy, uye), dXY = mul_(ux, uye);
    const double dP = mul_(uxe, Fx), dQ = mul_(uye, Fy), dW = fma_(uxe, Fy, mul_(uye, Fx));
    const double T = add_(c.T0, Tp), C = add_(c.C0, Cp);
    const double Tux = mul_(T, ux), Tuy = mul_(T, uy), Cux = mul_(C, ux), Cuy = mul_(C, uy);
    // not finite somewhere: everything becomes NaN
    int top = fx_max(fx_max(E, Eg), Eh);
    const double all[] = {Tux, Tuy, Cux, Cuy, dA, dB, dP, dQ, dW, hist[0], hist[1], hist[2], hist[3]};
#pragma unroll
    for (int i = 0; i < 13; ++i) top = fx_max(top, fx_exp(all[i]));
    if (top >= 0x7FF - 8) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
#pragma unroll
        for (int q = 0; q < 9; ++q) f[q] = nan;
#pragma unroll
        for (int q = 0; q < 5; ++q) g[q] = h[q] = nan;
        return;
    }
    // the flow lattice: a scale that holds u, F and their products too
    const int need = fx_max(fx_max(fx_max(fx_exp(ux), fx_exp(uy)), fx_max(fx_exp(Fx), fx_exp(Fy))),
                            fx_max(fx_max(fx_exp(dA), fx_exp(dB)), fx_max(fx_exp(dW), fx_max(fx_exp(dP), fx_exp(dQ))))) - 1;
    if (need > E) {
        for (int q = 0; q < 9; ++q) v[q] = fx_shift(v[q], need - E);
        E = need;
        d13 = v[1] - v[3], d24 = v[2] - v[4], D57 = v[5] - v[7], D68 = v[6] - v[8];
    }
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
    fixed_d2q5(g, vg, Eg, sg, Tux, Tuy, hist[0], hist[1], k.zs);
    fixed_d2q5(h, vh, Eh, sh, Cux, Cuy, hist[2], hist[3], k.es);
    hist[0] = Tux;
    hist[1] = Tuy;
    hist[2] = Cux;
    hist[3] = Cuy;
}

}  // namespace lbm
