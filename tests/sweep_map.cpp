// Walks every block, warp, lane and marching position of the true-residual sweep on the host:
// each load must lie inside the lattice, and every vertex must be owned exactly once.
#include <cstdio>
#include <vector>

#include "sweep.h"

template <bool D3, bool DIFF>
static int walk(int nx, int ny, int nz, bool per) {
    const int nm = D3 ? nz : ny, yb = D3 ? (ny + 7) / 8 : 1;
    const int W = (D3 ? 1 : 8) * (DIFF ? 31 : 32), xb = (nx + W - 1) / W;
    const int64_t n = (int64_t)nx * ny * (D3 ? nz : 1);
    std::vector<int> owned(n, 0);
    int bad = 0;
    for (int bx = 0; bx < xb; ++bx)
        for (int by = 0; by < yb; ++by)
            for (int wid = 0; wid < ld::SWEEP_WARPS; ++wid)
                for (int lane = 0; lane < 32; ++lane) {
                    const ld::SweepLane<D3, DIFF> l(nx, ny, bx, by, wid, lane);
                    if (!l.in) continue;
                    for (int m = 0; m < nm; ++m) {
                        const int d[7][3] = {{0, 0, 0}, {0, 0, -1}, {0, 0, 1}, {1, 0, 0}, {-1, 0, 0}, {0, -1, 0}, {0, 1, 0}};
                        for (int q = 0; q < (D3 ? 7 : 5); ++q) {
                            // right neighbours are loaded by the last lane or column, left ones by the first
                            if (q == 3 && lane != 31 && l.gx != nx - 1) continue;
                            if (q == 4 && (DIFF || (lane != 0 && l.gx != 0))) continue;
                            const int64_t j = ld::sweep_vertex<D3>(nx, ny, nm, per, l.gx + d[q][0], l.gy + d[q][1], m + d[q][2]);
                            if (j >= n || (per && j < 0)) ++bad;
                            if (q == 0 && l.own && j >= 0 && j < n) ++owned[j];
                        }
                    }
                }
    for (int v : owned) bad += v != 1;
    if (bad) std::printf("%dx%dx%d %s %s: %d faults\n", nx, ny, nz, per ? "torus" : "grid", DIFF ? "difference" : "direct", bad);
    return bad;
}

// The launch: its extents hold, its segments cover the marching axis, and it is given up (for the
// gather kernel) exactly where its y blocks or tiles exceed a grid's extent.
static int launch(bool d3, bool diff, int nx, int ny, int nz, int ntiles) {
    const ld::SweepGrid g = ld::sweep_grid(d3, diff, nx, ny, nz, ntiles);
    const int nm = d3 ? nz : ny;
    const int64_t want = d3 ? ((int64_t)ny + 7) / 8 : 1;
    const int64_t edge = 2147483647 - 512;            // lane columns and block counts beyond it leave int
    int bad = g.ok != (want <= 65535 && ntiles <= 65535 && nx <= edge && ny <= edge && nz <= edge);
    if (g.ok) {
        const int segs = (int)g.by / g.yb;
        bad += g.by < 1 || g.by > 65535 || (int)g.by % g.yb != 0;
        bad += g.seg < 1 || (int64_t)segs * g.seg < nm || (int64_t)(segs - 1) * g.seg >= nm;
    }
    if (g.ok) {              // the last lane of the last warp still has a column number
        const int64_t last = ((int64_t)g.xb * (d3 ? 1 : ld::SWEEP_WARPS)) * (diff ? 31 : 32);
        bad += g.xb < 1 || last > 2147483647;
    }
    if (bad) std::printf("launch of %dx%dx%d, %d tiles: %d faults\n", nx, ny, nz, ntiles, bad);
    return bad;
}

int main() {
    int bad = 0;
    for (int diff = 0; diff < 2; ++diff)
        for (int ntiles : {1, 3, 9, 152, 5000, 65535, 65536})
            for (int nx : {1, 31, 32, 33, 500, 70000}) {
                for (int ny : {1, 15, 16, 17, 333, 100000, 2000000}) bad += launch(false, diff, nx, ny, 1, ntiles);
                for (int big : {2147483647, 2147483647 - 500, 2147483647 - 512}) {
                    bad += launch(false, diff, big, 1, 1, ntiles) + launch(false, diff, 1, big, 1, ntiles);
                    bad += launch(true, diff, big, 1, 1, ntiles) + launch(true, diff, 1, big, 1, ntiles) +
                           launch(true, diff, 1, 1, big, ntiles);
                }
                for (int ny : {1, 8, 9, 333, 30000, 262144, 524279, 524280, 524281, 600000})
                    for (int nz : {1, 2, 17, 400, 100000}) bad += launch(true, diff, nx, ny, nz, ntiles);
            }
    for (int per = 0; per < 2; ++per) {
        for (int nx : {1, 2, 3, 5, 30, 31, 32, 33, 48, 61, 62, 63, 92, 93, 94, 100, 108, 109, 124, 200, 217, 218, 247, 248, 249, 300, 500})
            for (int ny : {1, 2, 7}) bad += walk<false, true>(nx, ny, 1, per) + walk<false, false>(nx, ny, 1, per);
        for (int nx : {1, 2, 5, 30, 31, 32, 33, 62, 63, 64, 95})
            for (int ny : {1, 3, 8, 9, 17})
                for (int nz : {1, 2, 5}) bad += walk<true, true>(nx, ny, nz, per) + walk<true, false>(nx, ny, nz, per);
    }
    return bad != 0;
}
