// Resident engine, host side: plan (how many CTAs share a probing vector, and how they
// exchange) and launch.
#include "engine_resident.cuh"

#include <algorithm>
#include <cmath>

namespace ld {

namespace {

// items (16 bytes of a line) a thread owns at most: two private vectors in its 128 words of
// tensor memory, and a 64-bit mask of its own-colour vertices
constexpr int RES_ITEMS = 16;

template <typename V, int KIND>
const void *res_fn(int nt, bool kx) {
    if (kx)
        return nt == 256 ? reinterpret_cast<const void *>(&k_resident<V, KIND, 256, true, false>)
                         : reinterpret_cast<const void *>(&k_resident<V, KIND, 512, true, false>);
    return nt == 256 ? reinterpret_cast<const void *>(&k_resident<V, KIND, 256, false, false>)
                     : reinterpret_cast<const void *>(&k_resident<V, KIND, 512, false, false>);
}

template <typename V>
const void *res_fn_for(int kind, int nt, bool kx) {
    if (kind == KIND_2D5) return res_fn<V, KIND_2D5>(nt, kx);
    if (kind == KIND_3D7) return res_fn<V, KIND_3D7>(nt, kx);
    return res_fn<V, KIND_2D13_SQ>(nt, kx);
}

const void *res_kernel(const Solve &s, int nt, bool keep_x0) {
    return s.precision == 0 ? res_fn_for<double>(s.op.kind, nt, keep_x0) : res_fn_for<float>(s.op.kind, nt, keep_x0);
}

// geometry of a team of M CTAs; false when it does not fit
bool res_geometry(const Solve &s, bool keep_x0, int yw, int nt, int M, bool clustered, ResPlan &p) {
    const int word = s.precision == 0 ? 8 : 4, E = 16 / word;
    const bool mat = s.op.kind == KIND_2D13_SQ, d3 = s.op.kind == KIND_3D7;
    const int H = mat ? 2 : 1;
    p.M = M;
    p.nt = nt;
    p.clustered = clustered;
    p.yw = yw;
    p.G = (s.op.nx + E - 1) / E;
    if (p.G > nt) return false;
    p.pitch = (p.G + 2) * E;
    int best = -1;
    long best_cost = 0;
    for (int My = 1; My <= M; ++My) {       // y x z split of a 3D lattice with the fewest lines a CTA
        if (M % My || (!d3 && My != M)) continue;
        const int Mz = M / My;
        if (s.op.ny / My < H || (d3 && s.op.nz / Mz < 1)) continue;
        const long Ly = (s.op.ny + My - 1) / My, Lz = d3 ? (s.op.nz + Mz - 1) / Mz : 1;
        const long cost = 4 * Ly * Lz + (d3 ? 2 * (Ly + Lz) : 0);
        if (best < 0 || cost < best_cost) {
            best = My;
            best_cost = cost;
            p.My = My;
            p.Ly = (int)Ly;
            p.Lz = (int)Lz;
        }
    }
    if (best < 0) return false;
    const int L = p.Ly * p.Lz;
    p.nseg = std::min(nt / p.G, L);
    p.cmax = (L + p.nseg - 1) / p.nseg;
    if (p.cmax > RES_ITEMS || p.cmax * (4 * (mat && !keep_x0 ? 1 : 2) + yw) > 128) return false;
    p.slots = 2 * H * p.Lz + (d3 ? 2 * p.Ly : 0);
    const ResSmem lay = res_smem(p, word, s.op.kind, s.nshift, keep_x0, !mat && s.op.field_d != nullptr);
    p.smem = lay.bytes;
    return lay.bytes <= 227 * 1024;
}

// Clocks of one iteration of a team, from measured parts: a warp's 16-byte item in the
// vector phases (FP64: its FP64 instructions at 19 clocks each; FP32: issue), and the
// exchange with the scalar chain (grows with the warps whose partials are summed, and
// between cooperative CTAs with the records each reads).  Fits the measured iterations of
// 48 x 40 to 1024 x 1024 and 40^3 to 128^3 lattices within about 20 %.
double res_clocks(const Solve &s, const ResPlan &p, bool keep_x0) {
    const bool f64 = s.precision == 0;
    double item = s.op.kind == KIND_2D13_SQ ? (f64 ? 525 : 60) : s.op.kind == KIND_3D7 ? (f64 ? 470 : 96) : (f64 ? 390 : 42);
    if (keep_x0) item += f64 ? (s.op.kind == KIND_2D13_SQ ? 120 : 60) : (s.op.kind == KIND_3D7 ? 16 : 8);
    if (s.op.kind != KIND_2D13_SQ && s.op.field_d) item += f64 ? 10 : (s.op.kind == KIND_3D7 ? 13 : 2);
    if (!f64 && p.nt == 256) item *= 1.25;      // half the warps to cover the latencies
    const double warps = p.nt / 32.0, halo = (double)p.slots * p.G / p.nt;
    const double active = (p.G * p.nseg + 31) / 32;            // warps that own lines
    const double work = item * (active * p.cmax + 0.35 * warps * halo);
    const double fixed = p.clustered ? (f64 ? 4800 + 210 * warps + 50.0 * p.M : 1600 + 255 * warps + 300.0 * p.M)
                                     : (f64 ? 7400 + 500 * warps + 50.0 * p.M : 10800 + 150 * warps);
    return work + fixed;
}

// Clocks of one streamed pass over the same vectors (grid engine).  FP64: its launches and end
// of pass, or 13 or 18 FP64 instructions a vertex and column.  FP32: fitted to passes of 400^2
// to 1200^2 and 48^3 to 80^3 (18 to 45 columns) within 10 %, an intercept by kind and the state
// words at a rate.  Measured at the line, stream against resident, us: Matern 520^2 30.0 / 25.9,
// 640^2 36.6 / 39.3; 5-point 600^2 32.8 / 24.4, 900^2 48.7 / 51.7; 3D field 64^3 94 / 72, 80^3
// 135 / 200.
double stream_clocks(const Solve &s, int ncolours, bool keep_x0) {
    const double vc = (double)s.op.n * ncolours;
    const bool mat = s.op.kind == KIND_2D13_SQ, d3 = s.op.kind == KIND_3D7;
    if (s.precision == 0) {
        const double instr = mat ? 18 : d3 ? 15 : 13;
        return std::max(15.0 * 1950, vc * (instr + (keep_x0 ? 3 : 0)) / (152 * 1.5));
    }
    const int words = (mat && keep_x0 ? 8 : 4) + (keep_x0 && !mat ? 2 : 0);
    const double rate = d3 ? 2600 : mat ? (keep_x0 ? 2640 : 3000) : 4200;    // bytes a clock
    return (d3 ? 60000 : mat && keep_x0 ? 24000 : 32000) + vc * words * 4 / rate;
}

// Clocks of one streamed FP64 pass over `tiles` of the context's tiles: each block steps through
// its rows (planes in 3D) at the latency of a step or, with enough blocks an SM, at the FP64
// units' rate; a pass over few tiles has few blocks.  Fitted within 20 % to 400 passes over ranges
// of 1 to all of 7 to 111 colours, 190^2 to 640^2 and 33^3 to 64^3, with and without x.
double stream_range_clocks(const Solve &s, int tiles) {
    const bool mat = s.op.kind == KIND_2D13_SQ, d3 = s.op.kind == KIND_3D7, x = s.keep_x0 != 0;
    const double load = (double)tiles * s.bpt / 152.0;
    const double lat = d3 ? 1970 * (x ? 1.22 : 1) + 1740 * (s.T - 1)
                      : mat ? 2150 * (x ? 1.2 : 1) + 500 * (s.T - 1) : 1780 * (x ? 1.22 : 1) + 800 * (s.T - 1);
    const double rate = load * s.T * (d3 ? 1664 * (x ? 1.09 : 1) : mat ? 920 * (x ? 1.12 : 1) : 812 * (x ? 1.07 : 1));
    return (d3 ? 40700 : mat ? 24000 : 32000) + (s.seg + (mat ? 4 : 2)) * std::pow(std::pow(lat, 4) + std::pow(rate, 4), 0.25);
}

// Whether the grid engine's passes would take no longer than `clocks` on chip.  FP32: margins for
// what the two estimates miss at the line.  3D FP32 bodies spill, and a CTA that takes nearly all
// of the SM's shared memory leaves its spills no L1: measured 1.25 (1.6) times the estimate
// without x, 1.05 (1.35) with it.  Measured there, resident against streamed, us: 3D 60^3, 45
// columns 79 / 69, 130 x 20 x 50, 45, 61 / 59; 64^3, 45, 66 / 79; 3D FP64 60^3, 109, 806 / 748;
// Matern 450^2, 53 columns, 45 / 42, 400^2, 53, 36 / 40.
bool stream_faster(const Solve &s, const ResPlan &p, double clocks, int ncolours, bool keep_x0) {
    const double stream = stream_clocks(s, ncolours, keep_x0);
    const bool mat = s.op.kind == KIND_2D13_SQ, d3 = s.op.kind == KIND_3D7;
    if (s.precision == 0) {
        // the fit is to 3D passes whose blocks are partly padding; without any they are faster
        const double pad = !d3 ? 2.0 : (double)((s.op.nx + P3X - 3) / (P3X - 2) * (P3X - 2)) / s.op.nx *
                                           ((s.op.ny + P3Y - 3) / (P3Y - 2) * (P3Y - 2)) / s.op.ny;
        return clocks >= std::min(1.0, 0.95 * pad) * stream;
    }
    if (clocks >= (mat ? 0.85 : 0.9) * stream) return true;
    const bool full = p.smem > 196 * 1024;
    return d3 && clocks * (keep_x0 ? (full ? 1.35 : 1.05) : (full ? 1.6 : 1.25)) >= stream;
}

template <class F>
cudaError_t res_launch(const ResPlan &p, int missing, cudaStream_t st, F &&fn) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(p.J * p.M - missing));
    cfg.blockDim = dim3((unsigned)(p.nt + 64));
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    if (p.clustered) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)p.M;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return fn(cfg);
}

}  // namespace

static int resident_plan(const Solve &s, int ncolours, bool keep_x0, bool streams, int yw, ResPlan *out) {
    const int k = s.op.kind;
    if ((k != KIND_2D5 && k != KIND_2D13_SQ && k != KIND_3D7) || s.asig || ncolours < 1) return 1;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return (int)cudaGetLastError();
    double best = 1e300;
    for (int nt : {256, 512}) {
        const void *fn = res_kernel(s, nt, keep_x0);
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return (int)cudaGetLastError();
        // one cluster a vector
        for (int M : {1, 2, 3, 4, 6, 8, 10, 12, 16}) {
            ResPlan p{};
            if (!res_geometry(s, keep_x0, yw, nt, M, true, p)) continue;
            p.J = ncolours;
            int act = 0;
            cudaError_t e = res_launch(p, 0, nullptr, [&](cudaLaunchConfig_t &cfg) {
                return cudaOccupancyMaxActiveClusters(&act, fn, &cfg);
            });
            if (e != cudaSuccess || act < 1) {
                cudaGetLastError();
                continue;
            }
            const int rounds = (ncolours + act - 1) / act;
            p.clocks = res_clocks(s, p, keep_x0);
            p.wide = act;
            const double t = rounds * p.clocks;
            if (t < best) {
                best = t;
                *out = p;
            }
        }
        // teams over L2, all resident at once (one CTA an SM)
        for (int J = 1; J <= std::min(ncolours, sms); ++J) {
            const int rounds = (ncolours + J - 1) / J;
            if (J > 1 && (ncolours + J - 2) / (J - 1) == rounds) continue;   // fewer teams, as many rounds
            int M = sms / J;
            if (k != KIND_3D7) M = std::min(M, s.op.ny / (k == KIND_2D13_SQ ? 2 : 1));
            ResPlan p{}, q{};
            bool ok = false;
            for (int tries = 0; M >= 1 && tries < 24; --M, ++tries) {   // a 3D split wants a composite M
                if (!res_geometry(s, keep_x0, yw, nt, M, false, q)) {
                    if (k != KIND_3D7) break;
                    continue;
                }
                q.J = J;
                if (!ok || res_clocks(s, q, keep_x0) < res_clocks(s, p, keep_x0)) p = q;
                ok = true;
                if (k != KIND_3D7) break;
            }
            p.clocks = ok ? res_clocks(s, p, keep_x0) : 1e300;
            p.wide = J;
            const double t = rounds * p.clocks;
            int occ = 0;
            if (t < best &&
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, p.nt + 64, p.smem) == cudaSuccess &&
                (long)occ * sms >= (long)J * p.M) {
                best = t;
                *out = p;
            }
        }
    }
    cudaGetLastError();
    // contexts the grid engine would run: only where the passes would take longer
    if (streams && best < 1e300 && stream_faster(s, *out, best, ncolours, keep_x0)) return 1;
    return best < 1e300 ? 0 : 1;
}

int engine_resident_plan(const Solve &s, int ncolours, bool keep_x0, bool streams, ResPlan *out) {
    return resident_plan(s, ncolours, keep_x0, streams, 0, out);
}

int engine_resident_plan_vec(const Solve &s, int ncols, ResPlan *out) {
    return resident_plan(s, ncols, false, false, s.precision == 0 ? 4 : 8, out);
}

// FP32: a pass over few colours takes most of a pass over all (Matern 520^2, 19 colours: 30 us, 3
// of them 25, against 12 on chip for up to ten), so the plan holds for every range.  FP64: fewer
// blocks leave the streamed pass the FP64 units to itself (Matern 300^2, 19 colours: 77 us streamed, 59
// on chip; 3 of them 33 and still 59).
bool engine_resident_range(const Solve &s, const ResPlan &p, int cb, int ce) {
    if (s.precision != 0 || ce <= cb) return true;
    const int rounds = (ce - cb + p.wide - 1) / p.wide;
    return rounds * p.clocks < stream_range_clocks(s, (ce + s.T - 1) / s.T - cb / s.T);
}

size_t engine_resident_rec_bytes(const ResPlan &p) {
    return p.clustered ? 0 : (size_t)p.J * 2 * p.M * 8 * sizeof(ulonglong2);
}
size_t engine_resident_halo_bytes(const ResPlan &p) {
    return p.clustered ? 0 : (size_t)p.J * p.M * 2 * p.slots * p.G * 16;
}

bool engine_resident_cluster(const Solve &s, int M, ResPlan *out, double *clocks) {
    ResPlan p{};
    if (!res_geometry(s, false, 0, RES_BATCH_NT, M, true, p)) return false;
    if (p.smem > 225 * 1024) return false;          // beside the kernel's copies of Solve and plan
    p.J = 1;
    *out = p;
    *clocks = res_clocks(s, p, false);
    return true;
}

// state of the columns the engine does not solve, and the counters
__global__ void k_resident_init(Solve s, int cb, int ce) {
    __shared__ int cnt;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    for (int q = threadIdx.x; q < s.ncols * s.nshift; q += blockDim.x) s.pi[q] = make_double2(0.0, 0.0);
    for (int c = threadIdx.x; c < s.ncols; c += blockDim.x) {
        s.pi0[c] = 0.0;
        s.col_iters[c] = 0;
        s.rho[c] = s.class_size[c];
        s.col_active[c] = 0;
        if (c >= cb && c < ce && s.class_size[c] > 0.0) atomicAdd(&cnt, 1);
    }
    for (int t = threadIdx.x; t < s.ntiles; t += blockDim.x) {
        s.tile_done[t] = 1;
        s.tile_ctr[t] = 0;
        s.tile_par[t] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        *s.remaining = cnt;
        *s.status = 0;
    }
}

void resident_init(const Solve &s, int cb, int ce, cudaStream_t st) {
    k_resident_init<<<1, 1024, 0, st>>>(s, cb, ce);
}

int engine_resident(const Solve &s, const ResPlan &p, const ResArgs &a, void *stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    resident_init(s, a.cb, a.ce, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    if (a.rec && (e = cudaMemsetAsync(a.rec, 0, engine_resident_rec_bytes(p), st)) != cudaSuccess) return (int)e;
    const bool kx = s.keep_x0 != 0;
    const void *fn = res_kernel(s, p.nt, kx);
    Solve sv = s;
    ResPlan pv = p;
    ResArgs av = a;
    pv.smem = res_smem(p, s.precision == 0 ? 8 : 4, s.op.kind, s.nshift, kx, s.op.kind != KIND_2D13_SQ && s.op.field_d).bytes;
    void *args[] = {&sv, &pv, &av};
    e = res_launch(pv, a.missing, st, [&](cudaLaunchConfig_t &cfg) { return cudaLaunchKernelExC(&cfg, fn, args); });
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

// One CTA waits on a record that nobody writes (status bit 0: it gave up) and on a phase of its
// own barrier that nobody completes (bit 1).
__global__ void k_resident_wait_selftest(uint64_t limit_ns, const ulonglong2 *rec, int32_t *status) {
    __shared__ uint64_t bar;
    __shared__ volatile uint64_t limit;
    if (threadIdx.x == 0) {
        limit = limit_ns;
        mbar_init(&bar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    double v;
    const bool got = rec_wait(rec, 1, v, &limit);
    const bool done = res_bar_wait(smem_u32(&bar), 0u, &limit);
    __syncthreads();
    if (threadIdx.x == 0) *status = (got ? 0 : 1) | (done ? 0 : 2);
}

int engine_resident_wait_selftest(uint64_t limit_ns, void *rec_dev, int32_t *status_dev, void *stream) {
    k_resident_wait_selftest<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(
        limit_ns, static_cast<const ulonglong2 *>(rec_dev), status_dev);
    return (int)cudaGetLastError();
}

// one warp an item: {rr, pw, rw, ww} -> {alpha, beta, rho, code}
__global__ void k_resident_scalar_selftest(int64_t count, bool exact, const double *dots, double *out) {
    for (int64_t q = blockIdx.x; q < count; q += gridDim.x) {
        const double *d = dots + 4 * q;
        double na, nb, rho;
        const int code = exact ? res_scalars<true>(d[0], d[1], d[2], d[3], na, nb, rho)
                              : res_scalars<false>(d[0], d[1], d[2], d[3], na, nb, rho);
        if (threadIdx.x == 0) {
            out[4 * q] = na;
            out[4 * q + 1] = nb;
            out[4 * q + 2] = rho;
            out[4 * q + 3] = (double)code;
        }
    }
}

int engine_resident_scalar_selftest(int64_t count, bool exact, const double *dots_dev, double *out_dev, void *stream) {
    k_resident_scalar_selftest<<<(unsigned)std::min<int64_t>(count, 1 << 16), 32, 0, static_cast<cudaStream_t>(stream)>>>(
        count, exact, dots_dev, out_dev);
    return (int)cudaGetLastError();
}

// ------------------------------------------------------------------ vector form
// y = Re sum_l w_l x^{sigma_l}, every x^{sigma_l} a combination of the seed residuals r_k:
// with p_0 = r_0, p_{k+1} = zeta_{k+1} r_{k+1} + beta_k p_k, x += alpha_k p_k per shift, the
// weight of p_k in x is G_k = alpha_k + beta_k G_{k+1}, so y = sum_k coef_k r_k with
// coef_k = Re sum_l w_l zeta_k G_k.  The solve records the shift scalars of every iteration,
// the coefficients follow backwards, and the same CG runs again (its alpha and beta known: no
// dots) adding coef_k r_k: one FP64 update a vertex and iteration in place of one complex
// direction per shift.
__global__ void k_funmv_back(Solve s, ResArgs a) {
    const int c = blockIdx.x, l = threadIdx.x;
    const int J = s.col_iters[c];
    if (l >= s.nshift || !(s.class_size[c] > 0.0)) return;
    double2 *h = a.hist + (size_t)c * a.hcap * s.nshift * 3 + 3 * l;
    const size_t step = (size_t)s.nshift * 3;
    const double2 w = s.weight[l];
    double2 G = make_double2(0.0, 0.0);
    constexpr int U = 4;        // records in flight
    for (int k0 = J - 1; k0 >= 0; k0 -= U) {
        double2 as[U], bs[U], z[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const double2 *q = h + (size_t)max(k0 - u, 0) * step;
            as[u] = q[0];
            bs[u] = q[1];
            z[u] = q[2];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k0 - u < 0) break;
            G = cadd(as[u], cmul(bs[u], G));
            const double2 f = cmul(w, z[u]);
            h[(size_t)(k0 - u) * step].x = f.x * G.x - f.y * G.y;
        }
    }
}

// coef of every iteration: the shifts' parts in order
__global__ void k_funmv_coef(Solve s, ResArgs a) {
    const int c = blockIdx.y, J = s.col_iters[c];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < J; k += gridDim.x * blockDim.x) {
        const double2 *h = a.hist + ((size_t)c * a.hcap + k) * s.nshift * 3;
        double v = 0.0;
        for (int l = 0; l < s.nshift; ++l) v += h[3 * l].x;
        a.coef[(size_t)c * a.hcap + k] = v;
    }
}

template <typename V, int NT>
static const void *replay_fn(int kind) {
    if (kind == KIND_2D5) return reinterpret_cast<const void *>(&k_resident<V, KIND_2D5, NT, false, true>);
    if (kind == KIND_3D7) return reinterpret_cast<const void *>(&k_resident<V, KIND_3D7, NT, false, true>);
    return reinterpret_cast<const void *>(&k_resident<V, KIND_2D13_SQ, NT, false, true>);
}

int engine_resident_funmv(const Solve &s, const ResPlan &p, const ResArgs &a, int ncols, void *stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_funmv_back<<<ncols, (s.nshift + 31) / 32 * 32, 0, st>>>(s, a);
    k_funmv_coef<<<dim3(8, ncols), 128, 0, st>>>(s, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    if (a.rec && (e = cudaMemsetAsync(a.rec, 0, engine_resident_rec_bytes(p), st)) != cudaSuccess) return (int)e;
    const void *fn = s.precision == 0 ? (p.nt == 256 ? replay_fn<double, 256>(s.op.kind) : replay_fn<double, 512>(s.op.kind))
                                      : (p.nt == 256 ? replay_fn<float, 256>(s.op.kind) : replay_fn<float, 512>(s.op.kind));
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
        return (int)e;
    Solve sv = s;
    ResPlan pv = p;
    ResArgs av = a;
    void *args[] = {&sv, &pv, &av};
    e = res_launch(pv, 0, st, [&](cudaLaunchConfig_t &cfg) { return cudaLaunchKernelExC(&cfg, fn, args); });
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

}  // namespace ld
