// Resident engine for CSR matrices: CG-M solves of groups of probing vectors on chip.
//
// As engine_resident.cuh, for a general sparse matrix.  A team of M CTAs of a cooperative
// launch owns T = NG E probing vectors at once (E = 16 bytes of them: 4 FP32 or 2 FP64); CTA
// m owns the rows [row0[m], row0[m+1]) with their part of the matrix in shared memory
// (values, and 16-bit local column numbers).  Columns of the matrix outside the CTA's rows
// (its external columns) have local copies of r and p that it updates itself from w = Q p,
// which every CTA writes to a buffer in L2: the product then reads shared memory only, and an
// iteration gathers each external w once instead of p once per matrix entry.
//
// Per iteration: update r, p (x) of own rows and r, p of external columns; w = Q p; w to
// L2; dot partials of the T vectors.  CTA q < T of the team collects the partials of vector
// q (records as in engine_resident.cuh), forms its alpha and beta, and publishes them to the
// team; its shift warp runs the vector's shift recurrences.  A vector that has converged
// gets alpha = beta = 0 until the whole group has.
//
// r, w, x of own rows and r of external columns are private to a thread: tensor memory.
//
// Bound by the two hops of the exchange (about 7 us of an iteration) on small matrices, by
// shared-memory wavefronts of the gathers (FP32) or the FP64 units on larger ones.  Measured
// a CG iteration over all vectors (before: one CTA a tile, or the streaming step and product):
// 64^2 torus FP64, 25 vectors 38.7 -> 11 us; second-order FEM mesh of 13K vertices, 31
// vectors, FP32 220 -> 10.6, FP64 80 -> 39; of 90K vertices, 33 vectors, FP32 85 -> 46 (the
// last vector of 33 runs in a round of its own, on four vectors a team); FP64 of that size
// stays with the streaming passes (270 against 206).
#pragma once
#include "engine_resident.cuh"

namespace ld {

struct CsrCtl {
    int stop;                    // 1: every vector of the group is finished, 2: a wait ran out
    uint32_t tm;
    volatile int done, head, tail;
    int bad;                     // a vector warp's wait ran out
    volatile uint64_t wait_ns;   // limit of a wait
    ResCtl::Entry q[4];
    double alpha[RES_CSR_T], beta[RES_CSR_T];
    double tot[4];               // rr, pw, rw, ww of the vector this CTA owns
};
static_assert(sizeof(CsrCtl) <= RES_CSR_CTL_BYTES, "control block");

// ------------------------------------------------------------------ scalar warp
template <int NT, bool EXACT>
__device__ __noinline__ void csr_scalar_role(const Solve &s, const CsrPlan &pl, const ResArgs &ar, int team, int m,
                                             CsrCtl *ctl) {
    const int lane = threadIdx.x & 31, M = pl.M, T = pl.T;
    // records: partials [2][T][M][6], then scalars [2][T][4]
    ulonglong2 *const rec = ar.rec + (size_t)team * pl.rec_team;
    ulonglong2 *const rec2 = rec + (size_t)2 * T * M * 6;
    const bool owner = m < T;                    // of vector c0 + m
    unsigned long long tick = 0;
    int head = 0;
    auto timed = [&](uint64_t &t0) -> bool {     // the limit, from the first call
        const uint64_t t = global_ns();
        if (t0 == 0) t0 = t;
        return t - t0 > ctl->wait_ns;
    };
    for (int c0 = ar.cb + team * T; c0 < ar.ce; c0 += pl.J * T) {
        const int c = c0 + m;
        const bool live0 = owner && c < ar.ce && s.class_size[c] > 0.0;
        bool live = live0;
        double c_alpha = 0.0, c_beta = 0.0, c_rho = 0.0;
        int code = 0;
        const int base = head;
        for (int it = 0;; ++it, ++tick) {
            const int par = (int)(tick & 1);
            const unsigned long long tag = tick + 1;
            bool ok = true;
            double na = 0.0, nb = 0.0, rho = 0.0;
            int ncode = 0, fin = 1;
            const ulonglong2 *const rp = rec + ((size_t)par * T + m) * M * 6;      // (owner)
            if (owner) {
                bar_sync(3, 160);             // the sums of vector warps 0 to 3
                ok = !ctl->bad;
                if (live) {
                    // stop a fixed two iterations after the shift warp's verdict
                    while (ctl->tail < head - 1) {}
                    __threadfence_block();
                    const int d = ctl->done;
                    if (d > base && d <= head - 1) live = false;
                }
                fin = !live;
                const double rr = ctl->tot[0], pw = ctl->tot[1], rw = ctl->tot[2], ww = ctl->tot[3];
                rho = rr;
                if (live) ncode = res_scalars<EXACT>(rr, pw, rw, ww, na, nb, rho);
                if (lane < 3) rec_st(rec2 + ((size_t)par * T + m) * 4 + lane, lane == 0 ? na : lane == 1 ? nb : (double)fin, tag);
            }
            // every vector's alpha, beta and finished flag
            bool all_fin = true;
            for (int t = lane; t < T; t += 32) {
                double v[3];
                uint64_t t0 = 0;
                for (unsigned spin = 0;; ++spin) {
                    bool got = true;
#pragma unroll
                    for (int k = 0; k < 3; ++k) got &= rec_ld(rec2 + ((size_t)par * T + t) * 4 + k, tag, v[k]);
                    if (got) break;
                    if ((spin & 255) == 255 && timed(t0)) {
                        ok = false;
                        break;
                    }
                }
                ctl->alpha[t] = v[0];
                ctl->beta[t] = v[1];
                all_fin = all_fin && v[2] != 0.0;
            }
            __threadfence();
            int stop = __all_sync(0xffffffffu, all_fin) ? 1 : 0;
            if (!__all_sync(0xffffffffu, ok)) {
                set_status(s.status, DEV_TIMEOUT);
                stop = 2;
            }
            if (lane == 0) ctl->stop = stop;
            bar_sync(2, NT + 32);
            if (stop) break;
            if (live) {
                if (it > 0) {        // iteration it - 1 to the shift warp
                    double vr_sum = 0.0;
                    for (int q = lane; q < M; q += 32) {
                        double v = 0.0;
                        ok = rec_wait(rp + (size_t)q * 6 + 4, tag, v, &ctl->wait_ns) && ok;
                        vr_sum += v;
                    }
                    __syncwarp();
                    vr_sum = lane_sum(vr_sum);
                    if (!__all_sync(0xffffffffu, ok)) set_status(s.status, DEV_TIMEOUT);
                    while (head - ctl->tail >= 4) {}
                    if (lane == 0) {
                        ResCtl::Entry &e = ctl->q[head & 3];
                        e.alpha = c_alpha;
                        e.beta = c_beta;
                        e.rho = c_rho;
                        e.vr = vr_sum;
                        e.code = code;
                        __threadfence_block();
                        ctl->head = head + 1;
                    }
                    ++head;
                    __syncwarp();
                }
                c_alpha = na;
                c_beta = nb;
                c_rho = rho;
                code = ncode;
            }
        }
        // After a wait that ran out every owner posts the end, whether or not its vector of this group
        // is live: the shift warp passes over an empty colour class and may be waiting for a later
        // group's entries (or be gone, and the entry stays unread).
        if (live0 || (owner && ctl->stop == 2)) {
            while (head - ctl->tail >= 4) {}
            if (lane == 0) {
                ctl->q[head & 3].code = ctl->stop == 2 ? -2 : -1;
                __threadfence_block();
                ctl->head = head + 1;
            }
            ++head;
            __syncwarp();
        }
        ++tick;
        if (ctl->stop == 2) break;
    }
}

// ------------------------------------------------------------------ vector warps
template <typename V, int NG, int NT>
__device__ __forceinline__ void csr_vector_role(const Solve &s, const CsrPlan &pl, const ResArgs &ar, int team, int m,
                                                unsigned char *smem, const CsrSmem &lay, CsrCtl *ctl) {
    constexpr int E = res_epi<V>(), NW = NT / 32, RS = NT / NG;       // RS rows a sweep of the threads
    using It = ResItem<V>;
    using PM = PackMath<V, E>;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int T = pl.T, M = pl.M;
    const int r0 = pl.row0[m], own = pl.row0[m + 1] - r0, e0 = pl.ext0[m], ext = pl.ext0[m + 1] - e0;
    const int n = (int)s.op.n;
    double *const part = reinterpret_cast<double *>(smem + lay.part);
    V *const val = reinterpret_cast<V *>(smem + lay.val);
    uint16_t *const col = reinterpret_cast<uint16_t *>(smem + lay.col);
    int *const rowp = reinterpret_cast<int *>(smem + lay.row);
    int *const colour = reinterpret_cast<int *>(smem + lay.colour);
    V *const P = reinterpret_cast<V *>(smem + lay.p);                 // [own + ext][NG] items
    V *const coef = reinterpret_cast<V *>(smem + lay.coef);           // -alpha, beta, alpha: [3][T]
    V *const wbuf = static_cast<V *>(ar.halo) + (size_t)team * 2 * n * T;
    const int g = tid % NG, rs = tid / NG;
    const int io = pl.items_own, ie = pl.items_ext;
    // tensor memory: [w | r | x] of own items, r of external ones
    const uint32_t tmw = ctl->tm + ((uint32_t)(wid & 3) << 21) + (uint32_t)(wid >> 2) * (512u / (NT / 128));
    const uint32_t tmr = tmw + 4u * io, tmx = tmr + 4u * io, tme = tmx + (s.keep_x0 ? 4u * io : 0u);
    const bool keepx = s.keep_x0;
    // the matrix rows of this CTA
    const int64_t nz0 = s.op.rowptr[r0];
    const int nnz = (int)(s.op.rowptr[r0 + own] - nz0);
    for (int q = tid; q < nnz; q += NT) {
        if constexpr (sizeof(V) == 8) val[q] = s.op.val_d[nz0 + q];
        else val[q] = s.op.val_f[nz0 + q];
        col[q] = pl.lcol[nz0 + q];
    }
    for (int q = tid; q <= own; q += NT) rowp[q] = (int)(s.op.rowptr[r0 + q] - nz0);
    for (int q = tid; q < own; q += NT) colour[q] = s.colour[r0 + q];
    unsigned long long tick = 0;
    for (int c0 = ar.cb + team * T; c0 < ar.ce; c0 += pl.J * T) {
        const int hi = min(ar.ce - c0, T);           // vectors of this group
        bar_sync(1, NT);
        const It zz = zero_pack<V, E>();
        auto init = [&](int lc) {                    // the indicator of this thread's vectors
            It r = zz;
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (lc == g * E + e && lc < hi) r.v[e] = (V)1;
            return r;
        };
        for (int i = 0; i < io; ++i) {
            const int row = i * RS + rs;
            It r = zz;
            if (row < own) {
                r = init(colour[row] - c0);
                ri_st(P + ((size_t)row * NG + g) * E, zz);
            }
            __syncwarp();
            tm_st<V>(tmw + 4u * i, zz);
            tm_st<V>(tmr + 4u * i, r);
            if (keepx) tm_st<V>(tmx + 4u * i, zz);
        }
        for (int i = 0; i < ie; ++i) {
            const int q = i * RS + rs;
            It r = zz;
            if (q < ext) {
                r = init(s.colour[pl.ext[e0 + q]] - c0);
                ri_st(P + ((size_t)(own + q) * NG + g) * E, zz);
            }
            __syncwarp();
            tm_st<V>(tme + 4u * i, r);
        }
        tm_wait_st();
        for (int q = tid; q < 3 * T; q += NT) coef[q] = (V)0;
        bar_sync(1, NT);
        int stop = 0;
        for (int it = 0;; ++it, ++tick) {
            const int par = (int)(tick & 1);
            const It na = ri_ld(coef + g * E), be = ri_ld(coef + T + g * E), aa = ri_ld(coef + 2 * T + g * E);
            // ---- r, p (x) of own rows, r and p of external columns
            const V *wprev = wbuf + (size_t)(par ^ 1) * n * T;
            // four items at a time: their gathers from L2 are in flight together
            constexpr int U = 4;
            for (int i0 = 0; i0 < ie; i0 += U) {
                It wv[U];
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const int q = (i0 + k) * RS + rs;
                    wv[k] = zz;
                    if (q < ext && it > 0) wv[k] = ri_ldcg(wprev + ((size_t)pl.ext[e0 + q] * NG + g) * E);
                }
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const int i = i0 + k, q = i * RS + rs;
                    if (i >= ie) break;
                    __syncwarp();
                    TmItem tr;
                    tm_ld(tr, tme + 4u * i);
                    V *pp = P + ((size_t)(own + min(q, ext - 1)) * NG + g) * E;
                    const It old = ri_ld(pp);
                    tm_wait(tr);
                    const It r = PM::fma(na, wv[k], tm_get<V>(tr));
                    tm_st<V>(tme + 4u * i, r);
                    if (q < ext) ri_st(pp, PM::fma(be, old, r));
                }
            }
#pragma unroll 2
            for (int i = 0; i < io; ++i) {
                const int row = i * RS + rs;
                __syncwarp();
                TmItem tw, tr;
                tm_ld(tw, tmw + 4u * i);
                tm_ld(tr, tmr + 4u * i);
                V *pp = P + ((size_t)min(row, own - 1) * NG + g) * E;
                const It old = ri_ld(pp);
                tm_wait(tw, tr);
                const It r = PM::fma(na, tm_get<V>(tw), tm_get<V>(tr));
                tm_st<V>(tmr + 4u * i, r);
                if (keepx) {
                    TmItem tx;
                    tm_ld(tx, tmx + 4u * i);
                    tm_wait(tx);
                    tm_st<V>(tmx + 4u * i, PM::fma(aa, old, tm_get<V>(tx)));
                }
                if (row < own) ri_st(pp, PM::fma(be, old, r));
            }
            __syncwarp();
            tm_wait_st();
            bar_sync(1, NT);
            // ---- w = Q p, dots
            It d[5] = {zz, zz, zz, zz, zz};
            V *wout = wbuf + (size_t)par * n * T;
            for (int i = 0; i < io; ++i) {
                const int row = i * RS + rs;
                TmItem tr;
                tm_ld(tr, tmr + 4u * i);
                It w = zz;
                const V *pg = P + g * E;
                if (row < own) {
                    int e = rowp[row];
                    const int e1 = rowp[row + 1];
                    It w2 = zz;
                    for (; e + 4 <= e1; e += 4) {        // four gathers in flight, two sums
                        It q[4];
                        V c[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            q[k] = ri_ld(pg + (size_t)col[e + k] * (NG * E));
                            c[k] = val[e + k];
                        }
                        w = PM::fma(PM::splat(c[0]), q[0], w);
                        w2 = PM::fma(PM::splat(c[1]), q[1], w2);
                        w = PM::fma(PM::splat(c[2]), q[2], w);
                        w2 = PM::fma(PM::splat(c[3]), q[3], w2);
                    }
                    for (; e < e1; ++e) w = PM::fma(PM::splat(val[e]), ri_ld(pg + (size_t)col[e] * (NG * E)), w);
                    w = PM::add(w, w2);
                }
                __syncwarp();
                tm_wait(tr);
                tm_st<V>(tmw + 4u * i, w);
                if (row < own) {
                    ri_st(wout + ((size_t)(r0 + row) * NG + g) * E, w);
                    const It r = tm_get<V>(tr), p = ri_ld(pg + (size_t)row * (NG * E));
                    d[0] = PM::fma(r, r, d[0]);
                    d[1] = PM::fma(p, w, d[1]);
                    d[2] = PM::fma(r, w, d[2]);
                    d[3] = PM::fma(w, w, d[3]);
                    const int lc = colour[row] - c0 - g * E;
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (lc == e) d[4].v[e] += r.v[e];
                }
                __syncwarp();
            }
            tm_wait_st();
            // partials [par][warp][vector][dot]
            double *pp = part + ((size_t)par * NW + wid) * 5 * T;
            constexpr int NS = group_sum_left(5 * E, NG);
            // beyond a thread's rows the sums of FP32 vectors keep their rounding errors, as the
            // streaming product's do in FP64
            V v[5 * E];
            std::conditional_t<sizeof(V) == 8, double, Sum2> sum[NS];
#pragma unroll
            for (int k = 0; k < 5 * E; ++k) v[k] = d[k % 5].v[k / 5];
            int at = 0, end = 5 * E;
            group_sum<NG>(v, sum, at, end);
#pragma unroll
            for (int k = 0; k < NS; ++k)
                if (at + k < end) pp[g * 5 * E + at + k] = (double)sum[k];
            bar_sync(1, NT);           // every warp's w and partials, before the fence of who publishes
            const unsigned long long tag = tick + 1;
            ulonglong2 *const rec = ar.rec + (size_t)team * pl.rec_team;
            // one thread a sum, to the vector's owner; then the owner's vector's dots over the
            // team, one a warp (see engine_resident.cuh: FP64 sums want warps of all SM quarters)
            if (tid < 5 * T) {
                const double *q = part + (size_t)par * NW * 5 * T + tid;
                double a = q[0];
#pragma unroll
                for (int w = 1; w < NW; ++w) a += q[(size_t)w * 5 * T];
                __threadfence();
                const int t = tid / 5, k = tid - 5 * t;
                rec_st(rec + (((size_t)par * T + t) * M + m) * 6 + k, a, tag);
            }
            if (m < T && wid < 4) {
                __syncwarp();
                const ulonglong2 *rp = rec + ((size_t)par * T + m) * M * 6 + wid;
                bool ok = true;
                double a = 0.0;
                for (int q0 = lane; q0 < M; q0 += 160) {         // five records a lane in flight
                    double v[5];
                    uint64_t t0 = 0;
                    for (unsigned spin = 0;; ++spin) {
                        bool got = true;
#pragma unroll
                        for (int b = 0; b < 5; ++b) {
                            v[b] = 0.0;
                            if (q0 + 32 * b < M) got &= rec_ld(rp + (size_t)(q0 + 32 * b) * 6, tag, v[b]);
                        }
                        if (got) break;
                        if ((spin & 255) == 255) {
                            const uint64_t t = global_ns();
                            if (t0 == 0) t0 = t;
                            else if (t - t0 > ctl->wait_ns) {
                                ok = false;
                                break;
                            }
                        }
                    }
                    a = q0 == lane ? v[0] : a + v[0];
#pragma unroll
                    for (int b = 1; b < 5; ++b)
                        if (q0 - lane + 32 * b < M) a += v[b];
                }
                __syncwarp();
                if (!ok) ctl->bad = 1;
                a = lane_sum(a);
                if (lane == 0) ctl->tot[wid] = a;
                __threadfence();         // every CTA's w before the owner's alpha and beta
                bar_arrive(3, 160);
            }
            bar_sync(2, NT + 32);
            stop = ctl->stop;
            if (stop) break;
            if (tid < T) {
                const V a = (V)ctl->alpha[tid];
                coef[tid] = -a;
                coef[T + tid] = (V)ctl->beta[tid];
                coef[2 * T + tid] = a;
            }
            bar_sync(1, NT);
        }
        ++tick;
        if (keepx) {
            for (int i = 0; i < io; ++i) {
                const int row = i * RS + rs;
                TmItem tx;
                tm_ld(tx, tmx + 4u * i);
                tm_wait(tx);
                const It xv = tm_get<V>(tx);
                if (row < own) {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int c = c0 + g * E + e, tile = c / s.T;
                        if (g * E + e < hi)
                            static_cast<V *>(s.x)[((int64_t)tile * n + r0 + row) * s.T + (c - tile * s.T)] = xv.v[e];
                    }
                }
                __syncwarp();
            }
        }
        if (stop == 2) break;
    }
}

template <typename V, int NG, int NT>
__global__ void __launch_bounds__(NT + 64, 1) k_resident_csr(const __grid_constant__ Solve s, const __grid_constant__ CsrPlan pl,
                                                             const __grid_constant__ ResArgs ar) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int wid = threadIdx.x >> 5;
    const int team = blockIdx.x / pl.M, m = blockIdx.x - team * pl.M;
    const CsrSmem lay = csr_smem(pl, (int)sizeof(V), s.nshift);
    CsrCtl *const ctl = reinterpret_cast<CsrCtl *>(smem + lay.ctl);
    if (wid == NW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&ctl->tm)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
        if ((threadIdx.x & 31) == 0) {
            ctl->done = 0;
            ctl->head = ctl->tail = 0;
            ctl->bad = 0;
            ctl->wait_ns = ar.wait_ns;
        }
        __syncwarp();
    }
    __syncthreads();
    if (wid < NW) {
        csr_vector_role<V, NG, NT>(s, pl, ar, team, m, smem, lay, ctl);
    } else if (wid == NW) {
        csr_scalar_role<NT, sizeof(V) == 8>(s, pl, ar, team, m, ctl);
    } else if (m < pl.T) {
        res_shift_role(s, pl.J * pl.T, ar.cb + team * pl.T + m, ar, ctl->q, &ctl->head, &ctl->tail, &ctl->done,
                       reinterpret_cast<double2 *>(smem + lay.shift));
    }
    __syncwarp();
    __syncthreads();
    if (wid == NW) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(ctl->tm));
}

}  // namespace ld
