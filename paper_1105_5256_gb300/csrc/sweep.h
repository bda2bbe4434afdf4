// Index map of the true-residual sweep (k_residual_sweep in engine.cu), common to the kernel
// and to the host test that walks every lane of it.
#pragma once
#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

namespace ld {

constexpr int SWEEP_WARPS = 8;

// The lattice column of one lane: its warp's block of columns is 32 wide, 31 in the difference
// form, whose lane 0 only supplies its right neighbour's left difference.
template <bool D3, bool DIFF>
struct SweepLane {
    static constexpr int W = DIFF ? 31 : 32;
    int gx, gy;
    bool own;       // the lane forms and counts the residual of its column
    bool in;        // the lane loads x
    __host__ __device__ SweepLane(int nx, int ny, int bx, int yb, int wid, int lane) {
        gx = (D3 ? bx : bx * SWEEP_WARPS + wid) * W + lane - (DIFF ? 1 : 0);
        gy = D3 ? yb * SWEEP_WARPS + wid : 0;
        own = gx < nx && (!D3 || gy < ny) && (!DIFF || lane > 0);
        // lane 0 only where its right neighbour owns a column: the torus wrap below is by one period
        in = own || (DIFF && lane == 0 && gx + 1 < nx && (!D3 || gy < ny));
    }
};

// Launch of the sweep: xb x (yb * number of segments) blocks a tile; segments of the marching
// axis for about eight blocks an SM, at least 16 positions each.  ok: the grid's y and z
// extents hold it, and no lane's column or count leaves int (one block of columns is 256 wide).
struct SweepGrid {
    int xb, yb, seg;
    unsigned by;
    bool ok;
};
inline SweepGrid sweep_grid(bool d3, bool diff, int nx, int ny, int nz, int ntiles) {
    constexpr int64_t MAX = 65535;
    SweepGrid g{};
    constexpr int EDGE = 2147483647 - 512;
    if (nx > EDGE || ny > EDGE || nz > EDGE) return g;
    const int nm = d3 ? nz : ny, W = (d3 ? 1 : SWEEP_WARPS) * (diff ? 31 : 32);
    g.xb = (nx + W - 1) / W;
    g.yb = d3 ? (ny + SWEEP_WARPS - 1) / SWEEP_WARPS : 1;
    int64_t segs = (int64_t)152 * 8 / std::max<int64_t>(1, (int64_t)g.xb * g.yb * ntiles);
    segs = std::max<int64_t>(1, std::min<int64_t>(segs, (nm + 15) / 16));
    while (segs > 1 && segs * g.yb > MAX) segs = (segs + 1) / 2;
    g.seg = (int)((nm + segs - 1) / segs);
    g.by = (unsigned)(g.yb * (((int64_t)nm + g.seg - 1) / g.seg));
    g.ok = g.yb <= MAX && ntiles <= MAX;
    return g;
}

// The vertex at (x, y) of marching position m (nm of them): wrapped on a torus by one period,
// -1 outside a Dirichlet grid.
template <bool D3>
__host__ __device__ inline int64_t sweep_vertex(int nx, int ny, int nm, bool per, int x, int y, int m) {
    if (per) {
        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        if (D3) y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        m = m < 0 ? m + nm : (m >= nm ? m - nm : m);
    } else if (x < 0 || x >= nx || m < 0 || m >= nm || (D3 && (y < 0 || y >= ny))) {
        return -1;
    }
    return D3 ? ((int64_t)m * ny + y) * nx + x : (int64_t)m * nx + x;
}

}  // namespace ld
