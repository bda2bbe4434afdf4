// Index map of the true-residual sweep (k_residual_sweep in engine.cu), common to the kernel
// and to the host test that walks every lane of it.
#pragma once
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
