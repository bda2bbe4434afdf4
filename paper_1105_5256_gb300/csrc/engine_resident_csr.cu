// Resident engine for CSR matrices, host side: row split, local column numbers, plan, launch.
#include "engine_resident_csr.cuh"

#include <algorithm>
#include <cmath>
#include <atomic>
#include <new>
#include <system_error>
#include <thread>

namespace ld {

// state of the columns the engine does not solve, and the counters (engine_resident.cu)
void resident_init(const Solve &s, int cb, int ce, cudaStream_t st);

namespace {

template <typename V, int NT>
const void *csr_fn(int ng) {
    if (ng == 1) return reinterpret_cast<const void *>(&k_resident_csr<V, 1, NT>);
    if (ng == 2) return reinterpret_cast<const void *>(&k_resident_csr<V, 2, NT>);
    return reinterpret_cast<const void *>(&k_resident_csr<V, 4, NT>);
}
// FP64: eight warps cover the gathers' latency (four: 49 against 40 us an iteration on a 13K-vertex
// second-order mesh, 31 vectors); more would only lengthen the warp sums
const void *csr_kernel(int precision, int ng) {
    return precision == 0 ? csr_fn<double, 256>(ng) : csr_fn<float, 512>(ng);
}

// external columns of rows [a, b), ascending
void external_columns(const int64_t *rowptr, const int32_t *colidx, int64_t a, int64_t b, std::vector<int32_t> &seen,
                      int stamp, std::vector<int32_t> &out) {
    out.clear();
    for (int64_t e = rowptr[a]; e < rowptr[b]; ++e) {
        const int32_t j = colidx[e];
        if ((j < a || j >= b) && seen[j] != stamp) {
            seen[j] = stamp;
            out.push_back(j);
        }
    }
    std::sort(out.begin(), out.end());
}

}  // namespace

// the parts of a plan that depend on T
static void csr_items(CsrPlan &p, int E) {
    const int rs = p.nt / (p.T / E);
    p.items_own = (p.own_max + rs - 1) / rs;
    p.items_ext = (p.ext_max + rs - 1) / rs;
    p.rec_team = (size_t)2 * p.T * p.M * 6 + (size_t)2 * p.T * 4;
}

int engine_csr_layout(int64_t n, const int64_t *rowptr, const int32_t *colidx, int precision, int ncolours, int nshift,
                      int sms, CsrPlan *out, std::vector<int32_t> &row0, std::vector<int32_t> &ext0,
                      std::vector<int32_t> &ext, std::vector<uint16_t> &lcol, int64_t *scanned) {
    const int word = precision == 0 ? 8 : 4, E = 16 / word, nt = precision == 0 ? 256 : 512;
    if (scanned) *scanned = 0;
    if (n < 2 || n >= (1ll << 30) || ncolours < 1) return 1;
    const double avg = (double)rowptr[n] / (double)n;
    // Cost of a plan in clocks, by the warps' rows and external columns.  FP64: 19 a warp
    // instruction (entries, r, p, dots); FP32: the shared-memory wavefronts of the product
    // (about nine an entry and warp) and the updates.  The exchange has two hops (partials to
    // the vector's owner, alpha and beta back); fewer teams of more vectors make it shorter
    // (13K-vertex second-order mesh, FP32, 31 vectors: T 4, 8 teams 11.5, T 8, 4 teams 10.2 us;
    // 3000-vertex graph, FP64, 15: T 2, 8 teams 10.3, T 4, 4 teams 9.2).
    double best = 1e300;
    CsrPlan bp{};
    std::vector<int32_t> seen(n, -1), tmp;
    int stamp = 0;
    for (int ng : {1, 2, 4}) {
        const int T = ng * E;
        if (T > RES_CSR_T) continue;
        for (int rounds = 1; rounds <= (ncolours + T - 1) / T; ++rounds) {
            const int J = (ncolours + rounds * T - 1) / (rounds * T);
            if (rounds > 1 && (ncolours + (rounds - 1) * T - 1) / ((rounds - 1) * T) == J) continue;
            int M = (int)std::min<int64_t>(sms / J, n);
            // at least a warp of rows a CTA
            M = (int)std::min<int64_t>(M, std::max<int64_t>(n / 32, T));
            if (M < T || M > n) continue;
            CsrPlan p{};
            p.M = M;
            p.J = J;
            p.T = T;
            p.nt = nt;
            // the largest CTA: every one of them for the rows and entries, a sample for the
            // external columns (the layout below takes the true maximum), which is only drawn
            // where the rows and entries alone would fit
            for (int m = 0; m < M; ++m) {
                const int64_t a = n * m / M, b = n * (m + 1) / M;
                p.own_max = std::max(p.own_max, (int)(b - a));
                p.nnz_max = (int)std::min<int64_t>(std::max<int64_t>(p.nnz_max, rowptr[b] - rowptr[a]), INT32_MAX);
            }
            const int room = 512 / (nt / 128) / 4;
            auto fits = [&]() {
                csr_items(p, E);
                return 3 * p.items_own + p.items_ext <= room && p.own_max + p.ext_max <= 65000 &&
                       csr_smem(p, word, nshift).bytes <= 227 * 1024;
            };
            if (!fits()) continue;
            for (int m : {0, M / 3, M / 2, M - 1}) {
                external_columns(rowptr, colidx, n * m / M, n * (m + 1) / M, seen, stamp++, tmp);
                if (scanned) *scanned += rowptr[n * (m + 1) / M] - rowptr[n * m / M];
                p.ext_max = std::max(p.ext_max, (int)tmp.size());
            }
            if (!fits()) continue;
            auto clocks = [&](const CsrPlan &q) {
                const double lanes = q.T / E / 32.0, own = std::ceil(q.own_max * lanes), ex = std::ceil(q.ext_max * lanes);
                const double fixed = (precision == 0 ? 14500 : 13000) + 20.0 * M + 400.0 * J;
                if (precision == 0) return fixed + own * (42 * avg + 310) + ex * 80.0 + nt / 32.0 * 250;
                return fixed + own * (9 * avg + 60) + ex * 22.0;
            };
            // whole rounds of J T vectors, then the remainder on the fewest vectors a team that hold it
            const int rest = ncolours % (J * T);
            p.split = ncolours - rest;
            p.T2 = 0;
            double t = (ncolours / (J * T)) * clocks(p);
            if (rest) {
                CsrPlan q = p;
                for (q.T = E; q.T * J < rest; q.T *= 2) {}
                csr_items(q, E);
                t += clocks(q);
                p.T2 = q.T;
                if (q.T == T) {
                    p.T2 = 0;
                    p.split = ncolours;
                }
            }
            if (t < best) {
                best = t;
                bp = p;
            }
        }
    }
    if (best >= 1e300) return 1;
    // Up to 32768 rows the alternative is one CTA a tile: slower than any plan by its serial
    // product.  Beyond, the streaming step and product (two launches; the gathers' latency and
    // the state from L2 or HBM).
    const double stream = n <= 32768 ? 1e300 : 45000 + (double)n * ncolours * (avg + 2) * (precision == 0 ? 0.006 : 0.0016);
    if (best >= stream) return 1;
    // ---- layout: external columns and local numbers, CTAs in parallel
    const int M = bp.M;
    row0.resize(M + 1);
    for (int m = 0; m <= M; ++m) row0[m] = (int32_t)(n * m / M);
    std::vector<std::vector<int32_t>> lists(M);
    lcol.resize(rowptr[n]);
    std::atomic<int> next{0};
    std::atomic<bool> failed{false};
    auto work = [&]() {
        try {
            std::vector<int32_t> mark(n, -1), loc(n);
            for (int m = next++; m < M; m = next++) {
                const int64_t a = row0[m], b = row0[m + 1];
                external_columns(rowptr, colidx, a, b, mark, m, lists[m]);
                for (size_t k = 0; k < lists[m].size(); ++k) loc[lists[m][k]] = (int32_t)(b - a + k);
                for (int64_t e = rowptr[a]; e < rowptr[b]; ++e) {
                    const int32_t j = colidx[e];
                    lcol[e] = (uint16_t)(j >= a && j < b ? j - a : loc[j]);
                }
            }
        } catch (const std::bad_alloc &) {
            failed = true;          // no plan: nothing leaves a thread or the C boundary
        }
    };
    const int nth = rowptr[n] > 200000 ? (int)std::min(8u, std::max(1u, std::thread::hardware_concurrency())) : 1;
    std::vector<std::thread> pool;
    pool.reserve(nth);
    try {
        for (int k = 1; k < nth; ++k) pool.emplace_back(work);
    } catch (const std::system_error &) {       // fewer helpers then
    }
    work();
    for (std::thread &t : pool) t.join();
    if (failed) return 1;
    ext0.assign(M + 1, 0);
    ext.clear();
    bp.ext_max = 1;
    for (int m = 0; m < M; ++m) {
        bp.ext_max = std::max(bp.ext_max, (int)lists[m].size());
        ext.insert(ext.end(), lists[m].begin(), lists[m].end());
        ext0[m + 1] = (int32_t)ext.size();
    }
    csr_items(bp, E);
    if (3 * bp.items_own + bp.items_ext > 512 / (nt / 128) / 4 || bp.own_max + bp.ext_max > 65000) return 1;
    bp.smem = csr_smem(bp, word, nshift).bytes;
    if (bp.smem > 227 * 1024) return 1;
    *out = bp;
    return 0;
}

int engine_csr_plan(int64_t n, const int64_t *rowptr, const int32_t *colidx, int precision, int ncolours, int nshift,
                    CsrPlan *out, std::vector<int32_t> &row0, std::vector<int32_t> &ext0, std::vector<int32_t> &ext,
                    std::vector<uint16_t> &lcol) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    CsrPlan bp{};
    if (engine_csr_layout(n, rowptr, colidx, precision, ncolours, nshift, sms, &bp, row0, ext0, ext, lcol, nullptr)) return 1;
    const int E = precision == 0 ? 2 : 4, nt = bp.nt;
    for (int T : {bp.T, bp.T2}) {
        if (T == 0) continue;
        const void *fn = csr_kernel(precision, T / E);
        int occ = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, nt + 64, bp.smem) != cudaSuccess ||
            (long)occ * sms < (long)bp.J * bp.M) {
            cudaGetLastError();
            return 1;
        }
    }
    *out = bp;
    return 0;
}

size_t engine_csr_rec_bytes(const CsrPlan &p) { return (size_t)p.J * p.rec_team * sizeof(ulonglong2); }

int engine_resident_csr(const Solve &s, const CsrPlan &p, const ResArgs &a, void *stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    resident_init(s, a.cb, a.ce, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    const int word = s.precision == 0 ? 8 : 4, E = 16 / word;
    for (int part = 0; part < 2; ++part) {
        // a colour's vectors-a-team follow from its index, so a partial range computes it alike
        CsrPlan pv = p;
        ResArgs av = a;
        if (part == 0) {
            av.ce = std::min(a.ce, p.split);
        } else {
            av.cb = std::max(a.cb, p.split);
            if (p.T2) {
                pv.T = p.T2;
                csr_items(pv, E);
                pv.smem = csr_smem(pv, word, s.nshift).bytes;
            }
        }
        if (av.cb >= av.ce) continue;
        if ((e = cudaMemsetAsync(a.rec, 0, (size_t)pv.J * pv.rec_team * sizeof(ulonglong2), st)) != cudaSuccess) return (int)e;
        const void *fn = csr_kernel(s.precision, pv.T / E);
        Solve sv = s;
        void *args[] = {&sv, &pv, &av};
        e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)(p.J * p.M - a.missing)), dim3((unsigned)(p.nt + 64)), args, pv.smem, st);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return (int)e;
        }
    }
    return 0;
}

}  // namespace ld
