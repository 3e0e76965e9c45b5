// The FP64 two-buffer step of a small cavity: three warps for 32 nodes.
//
// A cavity of 64 x 64 nodes is 128 warps for 608 SM sub-partitions, and the step's time is one
// node's chain: gather, two roots and a reciprocal, 1200 integer instructions, with a warp
// alone on its sub-partition.  Here the node's three lattices go to three warps (f; g; h),
// which lie in different sub-partitions and share only the moments: jx, jy, T', C' go to the
// first warp through shared memory and u comes back (on wall nodes once more, whose rebuild
// needs the interior node's u first).  The arithmetic is collide_fixed()'s and nee_rebuild()'s,
// operation for operation, so the bits are those of one thread a node.
// GB300, us per step, one thread / one warp a lattice: 33^2 7.1 / 4.7, 64^2 7.1 / 5.3, 101^2 10.2 /
// 6.8, 128^2 12.5 / 8.6, 200^2 13.6 / 8.9, 249^2 13.8 / 13.2, 512^2 41 / 45; with wall nodes 33^2
// 14.2 / 7.9, 101^2 15.7 / 8.7, 200^2 19.6 / 11.1, 249^2 20.4 / 13.8, 300^2 20.6 / 18.3, 362^2
// 22.6 / 25.5.  Eq. 18 solved by each warp for itself, without the way back: 64^2 6.1, 101^2
// 9.8, 128^2 11.4 (the FP64 pipe is the scarce unit as soon as an SM has two blocks).
// With the next step let in late (late_start()), up to 532 blocks: 64^2 4.95, 101^2 5.5, 128^2 5.5;
// with wall nodes 101^2 8.2, 128^2 8.5.
// A block has a fourth warp, which leaves at once: a warp's sub-partition is its number
// modulo 4, so that each block's first warp, which has the FP64 chain, would lie elsewhere
// with three (101^2 7.9, 101^2 with wall nodes 10.9, elsewhere within 3 percent).
// Both scalars run one code, since a lone warp waits for instructions as long as for its own
// results (a code each: 64^2 5.7, 64^2 with wall nodes 8.2); seven blocks per SM (72 registers, 16
// bytes of spills; eight: 128^2 9.0, 200^2 9.4; left at 80 registers: 200^2 11.2).
#pragma once
#include "lbm_kernels.cuh"

namespace lbm {

constexpr int TRIO_NODES = 32, TRIO_THREADS = 4 * TRIO_NODES;

// f (N = 9) or a scalar (N = 5) of node (i, j), its slots from q0, as gather_pull() has them.
template <int N, bool MOVING>
__device__ __forceinline__ void trio_pull(const double* __restrict__ buf, const Geom& G, int i, int j,
                                          const Coef<double>& c, int q0, const double* wall, double* d) {
    const size_t self = (size_t)j * G.pitch + i;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const int si = i - ex_of(q), sj = j - ey_of(q);
        const bool in = (unsigned)si < (unsigned)G.nx && (unsigned)sj < (unsigned)G.ny;
        const size_t off = in ? (size_t)sj * G.pitch + si : self;
        d[q] = buf[(size_t)(q0 + (in ? q : opp_of(q))) * G.plane + off];
        if (N == 5 && q > 0 && !in) d[q] = wall_value(c, wall, pull_side(q), d[q]);
        if (N == 9 && MOVING && !in) d[q] = add_(d[q], wall_momentum(c, link_side(si, sj, G), q));
    }
}

// u of Eq. 18 (and F, for the first warp, which has the flow) from the moments m, by the first warp.
__device__ __forceinline__ FixedMacro trio_macro(const Coef<double>& c, int role, int lane,
                                                 const double (*m)[TRIO_NODES], double (*u)[TRIO_NODES]) {
    FixedMacro M;
    if (role == 0) {
        M = fixed_macro(c, m[0][lane], m[1][lane], m[2][lane], m[3][lane]);
        u[0][lane] = M.ux;
        u[1][lane] = M.uy;
    }
    __syncthreads();
    if (role > 0) {
        M.ux = u[0][lane];
        M.uy = u[1][lane];
    }
    return M;
}

// NEE: nodes on the walls (the first ring_blocks blocks take them); else MOVING: halfway walls
// that move.  Uniform porous constants, factors that fit (c.fx.on).
template <bool NEE, bool MOVING, int NEXT>
__global__ void __launch_bounds__(TRIO_THREADS, 7)
step_ab_trio_kernel(const double* __restrict__ src, double* __restrict__ dst, double* __restrict__ hist, Geom G,
                    const __grid_constant__ Coef<double> c, unsigned ring_blocks) {
    __shared__ double s_wall[4][TRIO_NODES], s_mom[4][TRIO_NODES];   // jx, jy, T', C'
    __shared__ double s_u[4][TRIO_NODES];
    __shared__ int s_top[3][TRIO_NODES];                             // the lattices' scales
    const int role = threadIdx.x / TRIO_NODES, lane = threadIdx.x % TRIO_NODES;
    const bool ring = NEE && blockIdx.x < ring_blocks;               // of the whole block
    if (NEXT == NEXT_AT_ONCE) pdl_trigger();
    if (role == 3) return;
    int i, j;
    bool on;                       // threads past the end repeat the last node and store nothing
    if (ring) {
        const long long n = ring_count(G), k = (long long)blockIdx.x * TRIO_NODES + lane;
        on = k < n;
        ring_node(G, on ? k : n - 1, i, j);
    } else {
        const unsigned w = (unsigned)G.nx - (NEE ? 2u : 0u), n = w * ((unsigned)G.ny - (NEE ? 2u : 0u));
        unsigned k = (blockIdx.x - ring_blocks) * TRIO_NODES + lane;
        on = k < n;
        k = on ? k : n - 1;
        j = (int)(k / w);
        i = (int)(k - (unsigned)j * w) + (NEE ? 1 : 0);
        j += NEE ? 1 : 0;
    }
    const size_t self = (size_t)j * G.pitch + i;
    const int q0 = role == 0 ? QF : role == 1 ? QG : QH;
    const double* wall = role == 1 ? c.wallT : c.wallC;
    pdl_wait();                                // launched by launch_step()
    if (NEXT == NEXT_LATE) pdl_trigger();
    double d[9], hv[2];
    const size_t hk = (size_t)(role == 2 ? 2 : 0) * G.plane + self;
    if (role > 0) {
        hv[0] = hist[hk];
        hv[1] = hist[hk + G.plane];
    }
    if (ring) {                    // nee_rebuild()
        const int di = i == 0 ? 1 : (i == G.nx - 1 ? -1 : 0), dj = j == 0 ? 1 : (j == G.ny - 1 ? -1 : 0);
        double Pf = 0.0, Pff = 0.0;
        if (role == 0) {
            trio_pull<9, false>(src, G, i + di, j + dj, c, q0, wall, d);
            const double D57 = sub_(d[5], d[7]), D68 = sub_(d[6], d[8]);
            s_wall[0][lane] = add_(add_(sub_(d[1], d[3]), D57), sub_(d[8], d[6]));
            s_wall[1][lane] = add_(sub_(d[2], d[4]), add_(D57, D68));
        } else {
            double d2[5];
            trio_pull<5, false>(src, G, i + di, j + dj, c, q0, wall, d);
            trio_pull<5, false>(src, G, i + 2 * di, j + 2 * dj, c, q0, wall, d2);
            const double inv = role == 1 ? c.inv_sigma : c.inv_eps;
            s_wall[role + 1][lane] = Pf = mul_(sum5(d), inv);
            Pff = mul_(sum5(d2), inv);
        }
        __syncthreads();
        const FixedMacro M = trio_macro(c, role, lane, s_wall, s_u);
        const int sv = dj ? (dj > 0 ? 2 : 3) : (di > 0 ? 0 : 1);
        const double ubx = c.uwall[sv][0], uby = c.uwall[sv][1];
        if (role == 0)
            nee_flow(M.ux, M.uy, ubx, uby, c.inv_eps_f, c.inv_eps_f, d);
        else if (role == 1)
            nee_heat(c, M.ux, M.uy, ubx, uby, Pf, nee_scalar(c, di, dj, c.TwP, c.bT, Pf, Pff), d);
        else
            nee_mass(c, c, c, M.ux, M.uy, ubx, uby, Pf, nee_scalar(c, di, dj, c.CwP, c.bC, Pf, Pff), d);
    } else if (role == 0) {
        trio_pull<9, MOVING>(src, G, i, j, c, q0, wall, d);
    } else {
        trio_pull<5, false>(src, G, i, j, c, q0, wall, d);
    }
    long long v[9], s = 0;         // collide_fixed()
    int E;
    if (role == 0) {
        E = fixed_in<9>(d, v);
        s_mom[0][lane] = fixed_jx(v, E);
        s_mom[1][lane] = fixed_jy(v, E);
    } else {
        E = fixed_in<5>(d, v);
        s = fixed_sum(v);
        s_mom[role + 1][lane] = mul_(fx_out(s, E), role == 1 ? c.inv_sigma : c.inv_eps);   // Eq. 26
    }
    s_top[role][lane] = E;
    __syncthreads();
    const FixedMacro M = trio_macro(c, role, lane, s_mom, s_u + 2);
    const int top = fx_max(fx_max(s_top[0][lane], s_top[1][lane]), s_top[2][lane]);
    double* p = dst + (size_t)q0 * G.plane + self;
    if (role == 0) {
        fixed_flow(c, M, d, v, E, top);
        if (!on) return;
#pragma unroll
        for (int q = 0; q < 9; ++q) p[(size_t)q * G.plane] = d[q];
        return;
    }
    const FixedScalar& r = role == 1 ? c.fx.zs : c.fx.es;
    fixed_scalar(r, add_(role == 1 ? c.T0 : c.C0, s_mom[role + 1][lane]), M, d, v, E, s, hv, top);
    if (!on) return;
#pragma unroll
    for (int q = 0; q < 5; ++q) p[(size_t)q * G.plane] = d[q];
    hist[hk] = hv[0];
    hist[hk + G.plane] = hv[1];
}

// Up to these sizes (the figures above); uniform constants whose factors fit.
inline bool trio_fits(const Geom& G, const Coef<double>& c) {
    return !c.poro && c.fx.on && (long long)G.nx * G.ny <= (c.nee ? 90000 : 62500);
}

}  // namespace lbm
