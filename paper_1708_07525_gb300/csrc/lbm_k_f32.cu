// FP32 storage and arithmetic.
#include "lbm_launchers.cuh"
#include "lbm_march.cuh"

namespace lbm {

// Whether a cavity takes two steps per launch: its two buffers and history no longer stay in
// the 126 MB L2 between steps (168 bytes per node; the measurements stand in lbm_march.cuh),
// the state's byte offsets fit 32 bits, and strips and bands do not repeat too much of it.
// A band of n rows stages 2 (ceil(n / 2) + 1): with fewer than 6 rows, or 7, that is more than
// 1.4 n (us per step, two / one per launch, 760,000 nodes: 3 rows 30.6 / 19.8, 4 22.3 / 19.8,
// 5 24.0 / 19.9, 6 19.1 / 19.8, 7 21.5 / 19.7, 8 19.6 / 19.8, 9 19.0 / 19.9; 3 million: 4 rows
// 83 / 82, 5 86 / 81, 6 69 / 81, 7 75 / 82).  Rows of 32 columns are two strips, but one warp
// and whole lines to the one-step kernel (65,535 rows: 66.5 / 57.5; 31 columns 69.4 / 90.1,
// 33 columns 76.0 / 113).
bool march_fits(const Geom& G) {
    return (long long)G.nx * G.ny >= 750000 && (unsigned long long)(NQ + 1) * G.plane * 4 < (1ull << 32) &&
           10LL * ((G.ny + 1) / 2 + 1) <= 7LL * G.ny && G.nx != 32;
}

// Rows per band: the even number up to 32 for which the last wave of warps wastes least, a
// band of n rows costing n + 2.5 (one more row pair of stage A).  Longer bands measured slower
// although they repeat less (4096^2: 48 rows 279.5, 96 rows 287 us; 2048^2: 26 rows 77, 98
// rows 84 us): the warps of a wave drift apart over more rows of every plane.
static int march_rows_per_band(const Geom& G, int strips, int sms) {
    const long long resident = (long long)sms * MARCH_WARPS;
    int best = 4;
    double cost = 0;
    for (int rows = 4; rows <= 32; rows += 2) {
        const long long warps = (long long)strips * ((G.ny + rows - 1) / rows);
        const double w = (double)((warps + resident - 1) / resident) * (rows + 2.5);
        if (rows == 4 || w < cost) {
            cost = w;
            best = rows;
        }
    }
    return best;
}

cudaError_t launch_step2_ab(const void* src, void* dst, const void* hist, void* hist_out, const Geom& G,
                            const Coef<float>& c, const LaunchCfg& L) {
    const int strips = (G.nx + MARCH_COLS - 1) / MARCH_COLS;
    int rows = march_rows_per_band(G, strips, L.sms);
    while ((G.ny + rows - 1) / rows > 65535) rows *= 2;
    const dim3 gr((unsigned)strips, (unsigned)((G.ny + rows - 1) / rows), 1);
    if (c.moving)
        return launch_pdl(step2_ab_kernel<true>, gr, dim3(32), L.stream, (const float*)src, (float*)dst,
                          (const float*)hist, (float*)hist_out, G, c, rows);
    return launch_pdl(step2_ab_kernel<false>, gr, dim3(32), L.stream, (const float*)src, (float*)dst,
                      (const float*)hist, (float*)hist_out, G, c, rows);
}

LBM_INSTANTIATE(float)
}  // namespace lbm
