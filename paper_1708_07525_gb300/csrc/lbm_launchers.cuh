// Definitions of the launchers declared in lbm_launch.h (included by the
// per-precision translation units, which instantiate them).
#pragma once
#include <algorithm>
#include <type_traits>

#include "lbm_kernels.cuh"
#include "lbm_pair.cuh"
#include "lbm_trio.cuh"

namespace lbm {

inline dim3 grid_for(const Geom& G, int bx, int by) {
    return dim3((unsigned)((G.nx + bx - 1) / bx), (unsigned)((G.ny + by - 1) / by), 1);
}

// When a step lets the next launch in late (pdl_start()).  Let in at once, a launch that waits
// for its turn lets the next in at once as well, and launches pile up until every SM is full; of
// the last to fit, the blocks lie on the few SMs that had room left, and when its turn comes
// those SMs have all of it to do (an FP64 cavity of 128^2 in a porous field 34 us per step, of
// 64^2 11.7).  Let in late, one launch waits while one runs, at the price of a launch's latency.
// That is better where a grid covers most of the SMs and the GPU holds two of it, and for some
// kernels where one all but fills it.  Let in after its end, the next is placed on an empty
// GPU: FP64 steps in place or in a porous field, which take long, and 16-bit steps in place by
// one-node kernels.
// GB300, us per step, at once / late: FP32 two buffers 64^2 1.68 / 1.74, 128^2 2.19 / 1.74, 256^2 3.45 /
// 2.63, 257 x 200 (600 blocks) 2.92 / 3.40, with wall nodes 70 x 300 8.99 / 6.87; BF16 with wall nodes
// 140 x 285 (578 blocks) 7.8 / 7.9, 140 x 300 (608) 12.2 / 8.0; 16-bit pairs 129^2
// 5.34 / 5.51, 144^2 4.91 / 4.23, 70 x 300 6.12 / 4.07, 288^2 4.87 / 4.99, 366^2 13.4 / 5.07, 374^2 (763
// blocks) 4.97 / 5.05; FP64 (lbm_trio.cuh) 128^2 8.56 / 5.47, 70 x 300 (657 blocks) 7.08 / 7.84.  At
// once / after: FP64 in a porous field 128^2 34.0 / 11.6, 201 x 200 38.3 / 29.6, 1024^2 503 / 504;
// FP16 in place 103 x 301 3.97 / 2.38, 257 x 200 4.57 / 3.12, 383 x 260 4.61 / 4.07, 501 x 301 (1,204
// blocks) 12.3 / 5.9, lid 129 x 600 (1,200 blocks) 6.26 / 6.50.
struct LateRule {            // in twentieths of a block of 128 threads per SM
    int least, most;
    int full, filled;        // and from .. to here, where one grid (or two) fills the GPU
};
constexpr LateRule LATE_F32{13, 70, 0, 0};                                          // 8 blocks per SM
constexpr LateRule LATE_16BIT{13, 60, 78, 80}, LATE_16BIT_AA{13, 120, 0, 0};        // 8, 5 to 8
constexpr LateRule LATE_AA_SPLIT{157, 160, 0, 0};      // even steps beside step_aa_odd_fused_kernel
constexpr LateRule LATE_PAIR{19, 50, 95, 100}, LATE_TRIO{13, 70, 0, 0};             // 5, 7
inline bool late_start(const LateRule& r, long long blocks, int threads, int sms) {
    const long long n = 20 * blocks * threads, sm = 128LL * sms;
    return (n >= r.least * sm && n <= r.most * sm) || (n >= r.full * sm && n <= r.filled * sm);
}

// A step in one launch, a programmatic dependent one, by the kernel that lets the next one in
// at once or by the other.
template <typename... P, typename... A>
cudaError_t launch_step(void (*at_once)(P...), void (*late)(P...), const LateRule& r, dim3 grid, dim3 block,
                        const LaunchCfg& L, A... args) {
    const bool wait = late_start(r, (long long)grid.x * grid.y, (int)(block.x * block.y), L.sms);
    return launch_pdl(wait ? late : at_once, grid, block, L.stream, args...);
}

template <typename S>
cudaError_t launch_init(void* buf, void* hist, const Geom& G, const Coef<typename Real<S>::type>& c,
                        const InitSpec& I, bool pull, cudaStream_t st) {
    using R = typename Real<S>::type;
    dim3 b(128, 1), gr = grid_for(G, 128, 1);
    if (pull)
        init_kernel<S, true><<<gr, b, 0, st>>>((S*)buf, (R*)hist, G, c, I);
    else
        init_kernel<S, false><<<gr, b, 0, st>>>((S*)buf, (R*)hist, G, c, I);
    if (c.nee && pull) {   // wall nodes: the t = 0 state obeys the wall rules too
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        nee_hist_kernel<S><<<gr, b, 0, st>>>((const S*)buf, (R*)hist, G, c);
    }
    return cudaGetLastError();
}

// Grids of the two-nodes-per-thread kernels (lbm_pair.cuh); false if the cavity does
// not take them (too small, or too many rows for one launch).
// The pull grid: erows block rows of edge nodes, then the rows of inner pairs.
inline bool pair_grid_ab(const Geom& G, dim3& gr, int& erows) {
    const int np = inner_pairs(G.nx), rows = G.ny - 2;
    if (G.nx < 8 || rows < 1 || np < 1) return false;
    const long long gx = (np + PAIR_BX) / PAIR_BX;
    const long long eb = (edge_count(G) + PAIR_BX * PAIR_BY - 1) / (PAIR_BX * PAIR_BY);
    const long long er = (eb + gx - 1) / gx;
    const long long gy = (rows + PAIR_BY - 1) / PAIR_BY + er;
    if (gy > 65535) return false;
    erows = (int)er;
    gr = dim3((unsigned)gx, (unsigned)gy, 1);
    return true;
}
inline bool pair_grid_aa_even(const Geom& G, dim3& gr) {
    if (G.nx & 1) return false;
    gr = dim3((unsigned)((G.nx / 2 + PAIR_BX - 1) / PAIR_BX), (unsigned)((G.ny + PAIR_BY - 1) / PAIR_BY), 1);
    return gr.y <= 65535u;
}

// With FP32 arithmetic the in-place odd step splits the inner nodes (no wall logic) from
// the ring of outermost nodes from this many nodes on, below it runs as one kernel with
// the wall logic for every node.  GB300, FP32, us per step over alternating odd and even
// steps, one kernel / split with the ring on a second stream / split in one launch (the
// ring's block rows first): 128^2 2.5 / 4.6 / 3.9, 256^2 2.9 / 4.9 / 4.6, 512^2 6.9 / 7.8 /
// 6.3, 1024^2 28.2 / 27.5 / 25.5, 2048^2 121.3 / 117.0 / 114.6, 4096^2 - / 460.5 / 458.8.
#ifndef LBM_AA_SPLIT_MIN_NODES
#define LBM_AA_SPLIT_MIN_NODES (1LL << 17)
#endif
// With FP32 arithmetic the split odd step is one launch (step_aa_odd_fused_kernel: the
// ring's block rows, then the inner nodes), and so is the two-buffer step with wall nodes
// (Sec. 3.3; step_ab_nee_fused_kernel): no second stream, no fork / join, a programmatic
// dependent launch.  With wall nodes, FP32, us per step (second stream / one launch): 1024^2 33.3 / 30.5, 4096^2
// 459.2 / 456.7.
#ifndef LBM_AA_ODD_FUSED
#define LBM_AA_ODD_FUSED 1
#endif
#ifndef LBM_AB_NEE_FUSED
#define LBM_AB_NEE_FUSED 1
#endif

template <typename S>
cudaError_t launch_step_ab(const void* src, void* dst, void* hist, const Geom& G,
                           const Coef<typename Real<S>::type>& c, const LaunchCfg& L) {
    using R = typename Real<S>::type;
    dim3 b(L.bx, L.by), gr = grid_for(G, L.bx, L.by);
    constexpr LateRule rule = std::is_same<S, float>::value ? LATE_F32 : LATE_16BIT;
    if (G.jb != 0 || G.je != G.ny) {
        // a slab of a split cavity: the rows between its ghost rows, one launch with the
        // general pull (the ghost rows are ordinary neighbours, walls only where real)
        gr.y = (unsigned)((step_rows(G) + L.by - 1) / L.by);
        if (c.poro || c.moving)
            step_ab_kernel<S, true><<<gr, b, 0, L.stream>>>((const S*)src, (S*)dst, (R*)hist, G, c);
        else
            step_ab_kernel<S, false><<<gr, b, 0, L.stream>>>((const S*)src, (S*)dst, (R*)hist, G, c);
        return cudaGetLastError();
    }
    if constexpr (Store<S>::kLow) {
        dim3 gp;
        int erows = 0;
        if (L.pair && !c.nee && !c.poro && !c.moving && pair_grid_ab(G, gp, erows))
            // inner column pairs two nodes per thread, the edge set one node per thread,
            // in one programmatic dependent launch
            return launch_step(step_ab_pair_kernel<S>, step_ab_pair_kernel<S, NEXT_LATE>, LATE_PAIR, gp,
                               dim3(PAIR_BX, PAIR_BY), L, (const S*)src,
                              (S*)dst, (float*)hist, G, c, erows);
    }
    if constexpr (std::is_same<S, double>::value) {
        // one launch for all nodes, the wall nodes of Sec. 3.3 in its first blocks
        const bool ext = c.poro || c.moving;
        auto go = [&](auto* k, long long blocks, auto... more) {
            return launch_pdl(k, dim3((unsigned)blocks), dim3(128), L.stream, (const S*)src, (S*)dst, (R*)hist, G, c,
                              more...);
        };
        const long long nodes = (long long)G.nx * G.ny, ring = c.nee ? ring_count(G) : 0;
        if (trio_fits(G, c)) {   // three warps for 32 nodes
            const unsigned rb = (unsigned)((ring + TRIO_NODES - 1) / TRIO_NODES);
            const unsigned ib = (unsigned)((nodes - ring + TRIO_NODES - 1) / TRIO_NODES);
            auto go3 = [&](auto* at_once, auto* late) {
                return launch_step(at_once, late, LATE_TRIO, dim3(rb + ib), dim3(TRIO_THREADS), L,
                                   (const S*)src, (S*)dst, (R*)hist, G, c, rb);
            };
            if (c.nee)
                return go3(step_ab_trio_kernel<true, false, NEXT_AT_ONCE>, step_ab_trio_kernel<true, false, NEXT_LATE>);
            if (c.moving)
                return go3(step_ab_trio_kernel<false, true, NEXT_AT_ONCE>, step_ab_trio_kernel<false, true, NEXT_LATE>);
            return go3(step_ab_trio_kernel<false, false, NEXT_AT_ONCE>, step_ab_trio_kernel<false, false, NEXT_LATE>);
        }
        if (c.nee) {
            const long long rb = (ring_count(G) + 127) / 128;
            const long long ib = ((long long)(G.nx - 2) * (G.ny - 2) + 127) / 128;
            return c.poro ? go(step_ab_nee_flat_kernel<true>, rb + ib, (unsigned)rb)
                          : go(step_ab_nee_flat_kernel<false>, rb + ib, (unsigned)rb);
        }
        const long long nb = (nodes + 127) / 128;
        return ext ? go(step_ab_flat_kernel<true>, nb) : go(step_ab_flat_kernel<false>, nb);
    } else {
        if constexpr (LBM_AB_NEE_FUSED) {
            if (c.nee) {
                // the ring of wall nodes (the rebuild, Sec. 3.3) in the first block rows, the
                // inner nodes (the plain pull) after them: one programmatic dependent launch
                const long long threads = (long long)b.x * b.y;
                const long long rrows = ((2LL * G.nx + 2LL * (G.ny - 2) + threads - 1) / threads + gr.x - 1) / gr.x;
                if (gr.y + rrows <= 65535) {
                    const dim3 gf(gr.x, (unsigned)(gr.y + rrows), 1);
                    if (c.poro)
                        return launch_step(step_ab_nee_fused_kernel<S, true>,
                                           step_ab_nee_fused_kernel<S, true, NEXT_LATE>, rule, gf, b, L,
                                           (const S*)src, (S*)dst, (R*)hist, G, c, (int)rrows);
                    return launch_step(step_ab_nee_fused_kernel<S, false>,
                                       step_ab_nee_fused_kernel<S, false, NEXT_LATE>, rule, gf, b, L,
                                       (const S*)src, (S*)dst, (R*)hist, G, c, (int)rrows);
                }
            }
        }
        if (c.nee) {
            // the ring of wall nodes: the rebuild (Sec. 3.3); inner nodes: the plain pull
            cudaStream_t rs;
            cudaError_t e = ring_fork(L, &rs);
            if (e != cudaSuccess) return e;
            const long long nring = 2LL * G.nx + 2LL * (G.ny - 2);
            nee_ring_kernel<S><<<(unsigned)((nring + 127) / 128), 128, 0, rs>>>(
                (const S*)src, (S*)dst, (R*)hist, G, c);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if (c.poro)
                step_ab_kernel<S, true, true><<<gr, b, 0, L.stream>>>((const S*)src, (S*)dst, (R*)hist, G, c);
            else
                step_ab_kernel<S, false, true><<<gr, b, 0, L.stream>>>((const S*)src, (S*)dst, (R*)hist, G, c);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            return ring_join(L);
        } else if (!std::is_same<S, float>::value && G.nx >= 3 && G.ny >= 3) {
            // inner nodes with no wall logic, then the ring of outermost nodes.  GB300, 4096^2:
            // BF16 385 -> 377 us, FP16 442 -> 410 us; the DRAM-bound FP32 step measured slower
            // split (446 -> 460 us) and stays one kernel.
            const bool ext = c.poro || c.moving;
            cudaStream_t rs;
            cudaError_t e = ring_fork(L, &rs);
            if (e != cudaSuccess) return e;
            const long long nring = 2LL * G.nx + 2LL * (G.ny - 2);
            const unsigned nb = (unsigned)((nring + 127) / 128);
            if (ext)
                step_ab_ring_kernel<S, true><<<nb, 128, 0, rs>>>((const S*)src, (S*)dst, (R*)hist, G, c);
            else
                step_ab_ring_kernel<S, false><<<nb, 128, 0, rs>>>((const S*)src, (S*)dst, (R*)hist, G, c);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if (ext)
                step_ab_kernel<S, true, true><<<gr, b, 0, L.stream>>>((const S*)src, (S*)dst, (R*)hist, G, c);
            else
                step_ab_kernel<S, false, true><<<gr, b, 0, L.stream>>>((const S*)src, (S*)dst, (R*)hist, G, c);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            return ring_join(L);
        }
        // one kernel per step: a programmatic dependent launch, so that this step's CTAs are
        // placed while the step before drains
        if (c.poro || c.moving)
            return launch_step(step_ab_kernel<S, true>, step_ab_kernel<S, true, false, NEXT_LATE>, rule, gr, b, L,
                               (const S*)src, (S*)dst, (R*)hist, G, c);
        return launch_step(step_ab_kernel<S, false>, step_ab_kernel<S, false, false, NEXT_LATE>, rule, gr, b, L,
                               (const S*)src, (S*)dst, (R*)hist, G, c);
    }
}


template <typename S>
cudaError_t launch_step_aa(void* buf, void* hist, const Geom& G,
                           const Coef<typename Real<S>::type>& c, bool odd, const LaunchCfg& L) {
    using R = typename Real<S>::type;
    dim3 b(L.bx, L.by), gr = grid_for(G, L.bx, L.by);
    constexpr bool low = Store<S>::kLow;
    constexpr int later = low ? NEXT_AFTER : NEXT_LATE;
    const bool ext = c.poro || c.moving;
    if constexpr (Store<S>::kLow) {
        dim3 gp, ge;
        int erows = 0;
        if (L.pair && !ext && pair_grid_ab(G, gp, erows) && pair_grid_aa_even(G, ge)) {
            const dim3 pb(PAIR_BX, PAIR_BY);
            if (!odd)
                return launch_step(step_aa_even_pair_kernel<S>, step_aa_even_pair_kernel<S, NEXT_LATE>, LATE_PAIR,
                                   ge, pb, L, (S*)buf, (float*)hist, G,
                                  c);
            return launch_step(step_aa_odd_pair_kernel<S>, step_aa_odd_pair_kernel<S, NEXT_LATE>, LATE_PAIR, gp, pb,
                                   L, (S*)buf, (float*)hist, G,
                              c, erows);
        }
    }
    if constexpr (std::is_same<S, double>::value) {
        const long long nb = ((long long)G.nx * G.ny + 127) / 128;
        auto go = [&](auto* k) {
            return launch_pdl(k, dim3((unsigned)nb), dim3(128), L.stream, (S*)buf, (R*)hist, G, c);
        };
        if (odd) return ext ? go(step_aa_flat_kernel<true, true>) : go(step_aa_flat_kernel<true, false>);
        return ext ? go(step_aa_flat_kernel<false, true>) : go(step_aa_flat_kernel<false, false>);
    } else {
        const long long split_min = LBM_AA_SPLIT_MIN_NODES;
        const bool split = G.nx >= 3 && G.ny >= 3 && (long long)G.nx * G.ny >= split_min;
        if constexpr (LBM_AA_ODD_FUSED) {
            if (odd && split) {
                // ring and inner nodes in one programmatic dependent launch (the ring's block
                // rows first)
                const long long threads = (long long)b.x * b.y;
                const long long rrows = ((ring_count(G) + threads - 1) / threads + gr.x - 1) / gr.x;
                if (gr.y + rrows <= 65535) {
                    const dim3 gf(gr.x, (unsigned)(gr.y + rrows), 1);
                    if constexpr (low) {
                        if (!ext)
                            return launch_pdl(step_aa_odd_fused_kernel<S, false>, gf, b, L.stream, (S*)buf, (R*)hist,
                                              G, c, (int)rrows);
                    }
                    return launch_pdl(step_aa_odd_fused_kernel<S, true>, gf, b, L.stream, (S*)buf, (R*)hist, G, c,
                                      (int)rrows);
                }
            }
        }
        if (odd && split) {
            // the ring of outermost nodes beside the inner nodes (no wall logic); the two
            // launches touch disjoint locations
            cudaStream_t rs;
            cudaError_t e = ring_fork(L, &rs);
            if (e != cudaSuccess) return e;
            const long long nring = 2LL * G.nx + 2LL * (G.ny - 2);
            const unsigned nb = (unsigned)((nring + 127) / 128);
            if (ext)
                step_aa_odd_ring_kernel<S, true><<<nb, 128, 0, rs>>>((S*)buf, (R*)hist, G, c);
            else
                step_aa_odd_ring_kernel<S, false><<<nb, 128, 0, rs>>>((S*)buf, (R*)hist, G, c);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if (ext)
                step_aa_odd_inner_kernel<S, true><<<gr, b, 0, L.stream>>>((S*)buf, (R*)hist, G, c);
            else
                step_aa_odd_inner_kernel<S, false><<<gr, b, 0, L.stream>>>((S*)buf, (R*)hist, G, c);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            return ring_join(L);
        }
        // one kernel per step: a programmatic dependent launch, as in launch_step_ab
        constexpr LateRule alone = low ? LATE_16BIT_AA : LATE_F32;
        const LateRule& rule = split ? LATE_AA_SPLIT : alone;
        auto go = [&](auto* at_once, auto* late) {
            return launch_step(at_once, late, rule, gr, b, L, (S*)buf, (R*)hist, G, c);
        };
        if (split && ext) return go(step_aa_kernel<S, false, true>, step_aa_kernel<S, false, true, NEXT_AFTER>);
        if (split) return go(step_aa_kernel<S, false, false>, step_aa_kernel<S, false, false, NEXT_AFTER>);
        if (odd && ext) return go(step_aa_kernel<S, true, true>, step_aa_kernel<S, true, true, later>);
        if (odd) return go(step_aa_kernel<S, true, false>, step_aa_kernel<S, true, false, later>);
        if (ext) return go(step_aa_kernel<S, false, true>, step_aa_kernel<S, false, true, later>);
        return go(step_aa_kernel<S, false, false>, step_aa_kernel<S, false, false, later>);
    }
}

template <typename S>
cudaError_t launch_fields(const void* buf, const Geom& G, const Coef<typename Real<S>::type>& c,
                          int mode, int x0, int y0, int w, int h, double* out, cudaStream_t st) {
    if (w <= 0 || h <= 0) return cudaSuccess;
    dim3 b(128, 1), gr((unsigned)((w + 127) / 128), (unsigned)h, 1);
    fields_kernel<S><<<gr, b, 0, st>>>((const S*)buf, G, c, mode, x0, y0, w, h, out);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_nush(const void* buf, const Geom& G, const Coef<typename Real<S>::type>& c,
                        int mode, const WallSpec& W, double* scratch, double* out, cudaStream_t st) {
    const dim3 gr(nush_blocks(step_rows(G)), 2, 1);
    nush_kernel<S, true><<<gr, NUSH_THREADS, 0, st>>>((const S*)buf, G, c, mode, W, scratch,
                                                      (unsigned*)(scratch + NUSH_SCRATCH - 1), out);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_nush_tb(const void* buf, const Geom& G, const Coef<typename Real<S>::type>& c,
                           int mode, const WallSpec& W, double* scratch, double* out, cudaStream_t st) {
    const dim3 gr(nush_blocks(G.nx), 2, 1);
    nush_kernel<S, false><<<gr, NUSH_THREADS, 0, st>>>((const S*)buf, G, c, mode, W, scratch,
                                                       (unsigned*)(scratch + NUSH_SCRATCH - 1), out);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_residual(const void* buf, const Geom& G, const Coef<typename Real<S>::type>& c,
                            int mode, void* snap, double* slots, double* out,
                            cudaStream_t st) {
    using R = typename Real<S>::type;
    return launch_residual_pass<S, R>((const S*)buf, G, c, mode, (R*)snap, slots, out, st);
}

template <typename S>
cudaError_t launch_halo(void* buf, const Geom& G, int row, int up, void* face, int pack,
                        cudaStream_t st) {
    const dim3 gr((unsigned)((G.nx + 127) / 128), 5, 1);
    halo_kernel<S><<<gr, 128, 0, st>>>((S*)buf, G, row, up, (S*)face, pack);
    return cudaGetLastError();
}

#define LBM_INSTANTIATE(S)                                                                      \
    template cudaError_t launch_init<S>(void*, void*, const Geom&,                             \
                                        const Coef<Real<S>::type>&, const InitSpec&, bool,     \
                                        cudaStream_t);                                         \
    template cudaError_t launch_step_ab<S>(const void*, void*, void*, const Geom&,             \
                                           const Coef<Real<S>::type>&, const LaunchCfg&);      \
    template cudaError_t launch_step_aa<S>(void*, void*, const Geom&,                          \
                                           const Coef<Real<S>::type>&, bool,                   \
                                           const LaunchCfg&);                                  \
    template cudaError_t launch_fields<S>(const void*, const Geom&,                            \
                                          const Coef<Real<S>::type>&, int, int, int, int, int, \
                                          double*, cudaStream_t);                              \
    template cudaError_t launch_nush<S>(const void*, const Geom&, const Coef<Real<S>::type>&,  \
                                        int, const WallSpec&, double*, double*, cudaStream_t); \
    template cudaError_t launch_nush_tb<S>(const void*, const Geom&, const Coef<Real<S>::type>&,\
                                           int, const WallSpec&, double*, double*,             \
                                           cudaStream_t);                                      \
    template cudaError_t launch_residual<S>(const void*, const Geom&,                          \
                                            const Coef<Real<S>::type>&, int, void*, double*,   \
                                            double*, cudaStream_t);                            \
    template cudaError_t launch_halo<S>(void*, const Geom&, int, int, void*, int, cudaStream_t);

}  // namespace lbm
