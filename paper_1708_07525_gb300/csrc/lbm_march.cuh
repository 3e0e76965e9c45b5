// Two time steps per launch for the FP32 two-buffer layout with halfway walls.
//
// A warp takes a strip of 32 columns and marches up a band of rows, two rows at a time.
// Stage A pulls the rows (r, r + 1) of level t from memory and collides them; stage B pulls
// the rows below them of level t + 1 out of the registers of stage A's last two row pairs
// (its own columns directly, the neighbouring columns by warp shuffles), collides, and
// stores level t + 2.  The outer columns of the strip and one row at either end of the band
// only feed their neighbours: 24 columns of 32 are stored, and a band of H rows takes
// H / 2 + 1 row pairs of stage A.
//   - HBM sees the state once per two steps (1.00 of the algorithmic bytes of one step), and a
//     run takes half the launches;
//   - both rows of a pair go through the collision as packed FP32x2 values (f2), whose
//     operations round as the scalar ones do, so that two steps here give the bits of two
//     steps of step_ab_kernel: 339 warp instructions per 32 nodes and step, repeated nodes
//     and staging included, against 545 there (ncu, 2048^2);
//   - a warp's rows come by asynchronous 16-byte copies into shared memory while it works on
//     the pair before (46 rows of 128 bytes in 12 instructions); a block is one warp, so
//     that there is no barrier, and row pointers are the same for all lanes.
// 24 columns and not 30: what a warp stores is then whole 32-byte sectors (30 columns, whose
// ends shared a sector with the next strip: 304 us per 4096^2 step, 24 columns: 277).  Four
// warps side by side that pass the edge columns through shared memory store 120 columns of
// 128, but a barrier per row pair costs more than that saves (295 us).
// Bound by issue and latency at 12 warps per SM (48 % issue; 5 TB/s of HBM traffic).
// The history of Eq. 27 has two buffers here: the neighbouring strips and bands read
// the old one while this warp writes the new one.
// GB300, us per step, one step per launch / two: 900^2 23.5 / 19.9, 1024^2 29.5 / 22.9, 2048^2
// 112 / 77, 4096^2 442 / 280; 768^2 13.6 / 14.2 and 512^2 6.2 / 7.5, where the two buffers stay in
// L2 and the shorter chain of one step wins.
#pragma once
#include "lbm_kernels.cuh"

namespace lbm {

constexpr int MARCH_COLS = 24;       // columns a warp stores

// Post-collision values of a node pair.
struct NodePair {
    f2 f[9], g[5], h[5], hv[4];
};

__device__ __forceinline__ f2 pair_of(float a, float b) { return f2(make_float2(a, b)); }
// Staging buffer of one row pair: 23 planes, two rows each.
constexpr int MARCH_ROWS = 2 * (NQ + 4);

struct MarchStage {
    float row[MARCH_ROWS][32];
    // element offsets of the staged rows from one row below the pair's first, inside the cavity
    unsigned off[MARCH_ROWS];
};

__device__ __forceinline__ void copy_async16(uint32_t dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// e_y of plane q of the state.
__device__ __forceinline__ int plane_ey(int q) {
    const unsigned up = 1u << 2 | 1u << 5 | 1u << 6 | 1u << 11 | 1u << 16;     // f2 f5 f6 g2 h2
    const unsigned down = 1u << 4 | 1u << 7 | 1u << 8 | 1u << 13 | 1u << 18;   // f4 f7 f8 g4 h4
    return (int)(up >> q & 1) - (int)(down >> q & 1);
}

// Starts the copies of the rows that the pair (r, r + 1) of level t pulls from: a row of
// eight 16-byte pieces by eight neighbouring lanes, four rows at a time.  x1: the first staged
// column.  Pieces and rows outside the storage or the cavity take the nearest ones inside;
// their values are not used.
__device__ __forceinline__ void march_issue(MarchStage& S, const float* __restrict__ src,
                                            const float* __restrict__ hist, const Geom& G, int x1, int r) {
    const int piece = (int)threadIdx.x % 8, sub = (int)threadIdx.x / 8;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&S.row[sub][4 * piece]);
    const unsigned dx = (unsigned)min(max(x1 + 4 * piece, 0), G.pitch - 4);
    const bool in = r >= 1 && r + 2 <= G.ny - 1;
    const float* ps = src + (size_t)(r - 1) * G.pitch + dx;
    const float* ph = hist + (size_t)(r - 1) * G.pitch + dx;
#pragma unroll
    for (int k = 0; k < (MARCH_ROWS + 3) / 4; ++k) {
        const int row = 4 * k + sub;
        if (4 * k + 4 > MARCH_ROWS && row >= MARCH_ROWS) break;
        const bool h = row >= 2 * NQ;
        if (in) {
            copy_async16(dst + k * 512, (h ? ph : ps) + S.off[row]);
        } else {
            const int q = row >> 1;
            const int j = min(max(r + (row & 1) - (h ? 0 : plane_ey(q)), 0), G.ny - 1);
            copy_async16(dst + k * 512, (h ? hist + (size_t)(q - NQ) * G.plane : src + (size_t)q * G.plane) +
                                            (size_t)j * G.pitch + dx);
        }
    }
    copy_commit();
}

// The staged values of the pair (x, r), (x, r + 1) of this thread's column.  Links
// through a wall take the node's own opposite population, straight from memory.
__device__ __forceinline__ void march_fetch(const MarchStage& S, const float* __restrict__ src, const Geom& G,
                                            int x, int r, bool inner, NodePair& n) {
    constexpr int P = 32;
    const float* s = &S.row[0][threadIdx.x];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int e = q < QG ? q : q < QH ? q - QG : q - QH;
        const f2 v = pair_of(s[2 * q * P - ex_of(e)], s[(2 * q + 1) * P - ex_of(e)]);
        if (q < QG) n.f[e] = v;
        else if (q < QH) n.g[e] = v;
        else n.h[e] = v;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        n.hv[k] = pair_of(s[2 * (NQ + k) * P], s[(2 * (NQ + k) + 1) * P]);
    if (!inner) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int j = r + k;
            if (x < 0 || x >= G.nx || j < 0 || j >= G.ny) continue;
            const float* own = src + (size_t)j * G.pitch + x;
            auto at = [&](f2& v) -> float& { return k ? v.v.y : v.v.x; };
#pragma unroll
            for (int q = 1; q < 9; ++q) {
                if ((ex_of(q) > 0 && x == 0) || (ex_of(q) < 0 && x == G.nx - 1) ||
                    (ey_of(q) > 0 && j == 0) || (ey_of(q) < 0 && j == G.ny - 1)) {
                    at(n.f[q]) = __ldg(own + (size_t)(QF + opp_of(q)) * G.plane);
                    if (q < 5) {
                        at(n.g[q]) = __ldg(own + (size_t)(QG + opp_of(q)) * G.plane);
                        at(n.h[q]) = __ldg(own + (size_t)(QH + opp_of(q)) * G.plane);
                    }
                }
            }
        }
    }
}

// The wall rules of the pair (x, y), (x, y + 1) whose links through a wall hold the node's
// own opposite population.
template <bool EXT>
__device__ __forceinline__ void march_walls(const Geom& G, const Coef<float>& c, int x, int y, NodePair& m) {
    const bool left = x == 0, right = x == G.nx - 1;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int j = y + k;
        auto at = [&](f2& v) -> float& { return k ? v.v.y : v.v.x; };
        if (left) {
            at(m.g[1]) = wall_value(c, c.wallT, 0, at(m.g[1]));
            at(m.h[1]) = wall_value(c, c.wallC, 0, at(m.h[1]));
        }
        if (right) {
            at(m.g[3]) = wall_value(c, c.wallT, 1, at(m.g[3]));
            at(m.h[3]) = wall_value(c, c.wallC, 1, at(m.h[3]));
        }
        if (j == 0) {
            at(m.g[2]) = wall_value(c, c.wallT, 2, at(m.g[2]));
            at(m.h[2]) = wall_value(c, c.wallC, 2, at(m.h[2]));
        }
        if (j == G.ny - 1) {
            at(m.g[4]) = wall_value(c, c.wallT, 3, at(m.g[4]));
            at(m.h[4]) = wall_value(c, c.wallC, 3, at(m.h[4]));
        }
        if (EXT && c.moving) {
#pragma unroll
            for (int q = 1; q < 9; ++q) {
                const bool outx = (ex_of(q) > 0 && left) || (ex_of(q) < 0 && right);
                const bool outy = (ey_of(q) > 0 && j == 0) || (ey_of(q) < 0 && j == G.ny - 1);
                if (outx || outy)
                    at(m.f[q]) = add_(at(m.f[q]), wall_momentum(c, link_side(x - ex_of(q), j - ey_of(q), G), q));
            }
        }
    }
}

// What stage B pulls along q: the rows y, y + 1 of level t + 1 from the post-collision row
// pairs p = (y - 1, y) and n = (y + 1, y + 2), in this column or the one beside it.
__device__ __forceinline__ f2 march_pull(int q, const f2* p, const f2* n) {
    f2 v = ey_of(q) > 0 ? p[q] : ey_of(q) < 0 ? n[q] : pair_of(p[q].v.y, n[q].v.x);
    if (ex_of(q) > 0) {
        v.v.x = __shfl_up_sync(0xffffffffu, v.v.x, 1);
        v.v.y = __shfl_up_sync(0xffffffffu, v.v.y, 1);
    } else if (ex_of(q) < 0) {
        v.v.x = __shfl_down_sync(0xffffffffu, v.v.x, 1);
        v.v.y = __shfl_down_sync(0xffffffffu, v.v.y, 1);
    }
    return v;
}

// Warps per SM the kernel is compiled for: at most 168 registers (it takes 152).  GB300,
// 4096^2, us per step: 12 warps 277, 14 and 16 (128 registers, 52 bytes of spills) 299 and 347.
constexpr int MARCH_WARPS = 12;

// Grid (strips, bands): block (s, b) is one warp; it stages the columns MARCH_COLS s - 4 .. + 31
// and stores rows b rows .. b rows + rows - 1 (rows even).
template <bool EXT>
__global__ void __launch_bounds__(32, MARCH_WARPS)
step2_ab_kernel(const float* __restrict__ src, float* __restrict__ dst, const float* __restrict__ hist,
                float* __restrict__ hist_out, Geom G, Coef<float> c, int rows) {
    __shared__ __align__(16) MarchStage S;
    const int x1 = (int)blockIdx.x * MARCH_COLS - 4;
    const int y0 = (int)blockIdx.y * rows, y1 = min(y0 + rows, G.ny);
    const int x = x1 + (int)threadIdx.x;
    const bool store = threadIdx.x >= 4 && threadIdx.x < 4 + MARCH_COLS && x < G.nx;
    const bool edge = x1 <= 0 || x1 + 32 >= G.nx;
    auto inner = [&](int r) { return r >= 1 && r + 1 <= G.ny - 2 && !edge; };
    for (int row = threadIdx.x; row < MARCH_ROWS; row += 32) {
        const int q = row >> 1, l = q < NQ ? q : q - NQ;
        S.off[row] = (unsigned)((size_t)l * G.plane + (size_t)((row & 1) + 1 - (q < NQ ? plane_ey(q) : 0)) * G.pitch);
    }
    __syncwarp();
    pdl_trigger();
    pdl_wait();                                // launched by launch_pdl()
    NodePair p, n;
    march_issue(S, src, hist, G, x1, y0 - 1);
    for (int r = y0 - 1; r <= y1; r += 2) {
        copy_wait();
        __syncwarp();                          // every lane's copies have landed
        march_fetch(S, src, G, x, r, inner(r), n);
        if (!inner(r)) march_walls<EXT>(G, c, x, r, n);
        collide<true>(c, n.f, n.g, n.h, n.hv);
        // the staged values are used up: the next pair's rows come while stage B works
        __syncwarp();
        if (r + 2 <= y1) march_issue(S, src, hist, G, x1, r + 2);
        if (r >= y0) {
            const int y = r - 1;                           // rows y, y + 1 of level t + 1
            NodePair m;
#pragma unroll
            for (int q = 0; q < 9; ++q) m.f[q] = march_pull(q, p.f, n.f);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                m.g[q] = march_pull(q, p.g, n.g);
                m.h[q] = march_pull(q, p.h, n.h);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) m.hv[k] = pair_of(p.hv[k].v.y, n.hv[k].v.x);
            if (edge || y == 0 || y + 1 >= G.ny - 1) {
                // links through the walls: the node's own opposite population of level t + 1
#pragma unroll
                for (int q = 1; q < 9; ++q) {
                    const int o = opp_of(q);
                    const bool outx = (ex_of(q) > 0 && x == 0) || (ex_of(q) < 0 && x == G.nx - 1);
                    const bool out0 = outx || (ey_of(q) > 0 && y == 0) || (ey_of(q) < 0 && y == G.ny - 1);
                    const bool out1 = outx || (ey_of(q) < 0 && y + 1 == G.ny - 1);
                    if (out0) m.f[q].v.x = p.f[o].v.y;
                    if (out1) m.f[q].v.y = n.f[o].v.x;
                    if (q < 5) {
                        if (out0) m.g[q].v.x = p.g[o].v.y;
                        if (out1) m.g[q].v.y = n.g[o].v.x;
                        if (out0) m.h[q].v.x = p.h[o].v.y;
                        if (out1) m.h[q].v.y = n.h[o].v.x;
                    }
                }
                march_walls<EXT>(G, c, x, y, m);
            }
            collide<true>(c, m.f, m.g, m.h, m.hv);
            if (store) {
                // 32-bit byte offsets from the buffers (see march_fits)
                const unsigned o = ((unsigned)y * (unsigned)G.pitch + (unsigned)x) * 4u;
                const unsigned row = (unsigned)G.pitch * 4u, plane = (unsigned)G.plane * 4u;
                char* d = reinterpret_cast<char*>(dst);
                char* e = reinterpret_cast<char*>(hist_out);
                auto put2 = [&](char* base, unsigned at, f2 v) {
                    *reinterpret_cast<float*>(base + at) = v.v.x;
                    if (y + 1 < y1) *reinterpret_cast<float*>(base + at + row) = v.v.y;
                };
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    put2(d, o + q * plane, q < QG ? m.f[q] : q < QH ? m.g[q - QG] : m.h[q - QH]);
#pragma unroll
                for (int k = 0; k < 4; ++k) put2(e, o + k * plane, m.hv[k]);
            }
        }
        p = n;
    }
}

}  // namespace lbm
