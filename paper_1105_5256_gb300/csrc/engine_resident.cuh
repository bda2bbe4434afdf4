// Resident engine: a probing vector's whole CG-M solve on chip (sm_103a).
//
// The streaming engines read and write the CG state (r, p, and w or x) through L2 or HBM
// once per iteration and end every pass with a kernel boundary.  Here the state never
// leaves the SMs: a team of M CTAs owns one probing vector, each CTA a block of lattice
// lines (rows of nx vertices), and one launch runs every iteration of the solve.
//
//   5- and 7-point kinds   p in shared memory (with one halo line on each side); r,
//                          w = Q p, x (when kept) and a kappa^2 field's diagonal private
//   Matern kind s Q1^2     r (two halo lines) and u = Q1 p (one) in shared memory:
//                          u_k = Q1 r_k + beta u_{k-1}, w = s Q1 u, p.w = s |u|^2;
//                          w private.  With x kept, p (two halo lines) and u = Q1 p formed
//                          from it, r, w and x private: with u by its own recurrence w
//                          drifts from Q p, and FP32 x was two to nine times less exact
//
// Private vectors (read and written only by the thread that owns the vertex) live in tensor
// memory: 128 words a thread, addressed by a loop index (registers would need the loop
// unrolled, and hold half as many), with a bandwidth of its own beside shared memory's.
// x and the diagonal move to shared memory when tensor memory is full.
//
// The recurrences are those of the streaming passes (one reduction per iteration; r.r,
// p.w, r.w, w.w and v.r).  A halo costs no synchronisation of its own: a CTA keeps copies
// of r and p on its halo lines and updates them itself from the neighbours' boundary rows
// of w, which travel with the partial sums of the same iteration.  So an iteration has one
// exchange: boundary w and dots out, then alpha and beta (computed by every CTA from the
// same partials in the same order, so all agree to the bit).
//
// Team forms: one thread-block cluster (M <= 16; exchange through distributed shared
// memory and the cluster barrier), or, where a vector needs more CTAs, a cooperative
// launch whose teams exchange through L2 (16-byte {value, tag} records read until their
// tag is the iteration's, with a bounded wait).
//
// FP64 is slow here (an add takes 65 clocks, a quotient 600, two lanes a clock), so the
// scalar chains have warps of their own: in every CTA one warp sums the partials and forms
// alpha and beta; in the team's first CTA another runs the shift recurrences from a small
// queue while the vector warps are in later iterations.  v^T r_{k+1} is the next
// iteration's measured v.r; a converged vector is found an iteration or two late, and the
// iterations past its last are discarded (counts and projections are unaffected).
//
// Bound by what the SMs issue (FP32: about 45 to 65 instructions a 16-byte item and level, 16
// warps an SM) or by their FP64 units (19 clocks a warp instruction), plus one exchange of 2
// to 4.5 us an iteration, most of it dependent FP64 instructions; the state costs no DRAM or
// L2 traffic at all.  Measured a CG iteration over all vectors (before: the streaming or the
// one-CTA engine): 48 x 40 Matern FP64, 52 vectors, with x 63 -> 8.5 us; 128^2 5-point FP64,
// 18, with x 143 -> 13.5; 300 x 200 Matern FP32, 19, with x 22.6 -> 7.2; 500 x 333 torus
// field FP32, 26, with x 29.6 -> 17.5; 512 x 384 Matern FP64, 18 (FP64 units busy in both) 137
// -> 114.  Large FP32 problems stay with the lean passes: 1024^2 Matern, 18 vectors: 77 us
// here, 60 streamed.
//
// Where x, r or w live was tried three ways: registers with unrolled loops (12 items a
// thread spilled, half the capacity), shared memory only (two thirds of the capacity), and
// tensor memory (kept).  The runtime's occupancy query gives one CTA an SM to any kernel that
// allocates tensor memory (a 288-thread, 12-register kernel with 1 KB of shared memory: 7 without
// the tcgen05.alloc of 256 columns, 1 with it), and the registers here allow no second one
// either, so a team's iterations are not overlapped with another team's.
#pragma once
#include "engine_device.cuh"
#include "resident.h"

namespace ld {

constexpr int RES_NDOT = 5;     // rr, pw, rw, ww, vr

// elements of one item: 16 bytes of a lattice line
template <typename V>
__host__ __device__ constexpr int res_epi() { return 16 / (int)sizeof(V); }

template <typename V>
using ResItem = Pack<V, 16 / (int)sizeof(V)>;

template <typename V>
__device__ __forceinline__ ResItem<V> ri_ld(const V *p) {
    return *reinterpret_cast<const ResItem<V> *>(p);
}
template <typename V>
__device__ __forceinline__ void ri_st(V *p, const ResItem<V> &v) {
    *reinterpret_cast<ResItem<V> *>(p) = v;
}
template <typename V>
__device__ __forceinline__ ResItem<V> ri_ldcg(const V *p) {
    const float4 a = __ldcg(reinterpret_cast<const float4 *>(p));
    ResItem<V> o;
    *reinterpret_cast<float4 *>(&o) = a;
    return o;
}

// one level of the lattice operator: FP32 in difference form (see diff5p), FP64 in the
// direct form with c already holding the stencil's centre count; nz: the z neighbours' part
template <typename V, int NB>
__device__ __forceinline__ ResItem<V> res_level(const ResItem<V> &c, const ResItem<V> &m, V l, V r,
                                                const ResItem<V> &dn, const ResItem<V> &up,
                                                const ResItem<V> &fr, const ResItem<V> &bk) {
    constexpr int E = res_epi<V>();
    using M = PackMath<V, E>;
    ResItem<V> ml, mr;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        ml.v[e] = e == 0 ? l : m.v[e - 1];
        mr.v[e] = e == E - 1 ? r : m.v[e + 1];
    }
    if constexpr (sizeof(V) == 8) {
        ResItem<V> o;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            V sum = (ml.v[e] + mr.v[e]) + (dn.v[e] + up.v[e]);
            if constexpr (NB == 6) sum += fr.v[e] + bk.v[e];
            o.v[e] = fma(c.v[e], m.v[e], -sum);
        }
        return o;
    } else {
        ResItem<V> s = M::add(M::add(M::sub(m, ml), M::sub(m, mr)), M::add(M::sub(m, dn), M::sub(m, up)));
        if constexpr (NB == 6) s = M::add(s, M::add(M::sub(m, fr), M::sub(m, bk)));
        return M::fma(c, m, s);
    }
}

// The FP32 level of a 2D lattice with each difference formed once: e between neighbours of
// the line (scalar adds, which need no re-paired operands and leave the paired pipe free),
// d = m - (next line) kept for the next line's level as its dp.  Bits as in res_level.
__device__ __forceinline__ ResItem<float> res_level_sh(const ResItem<float> &c, const ResItem<float> &m, float l,
                                                       float r, const ResItem<float> &d, const ResItem<float> &dp) {
    using M = PackMath<float, 4>;
    const float el = l - m.v[0], e0 = m.v[0] - m.v[1], e1 = m.v[1] - m.v[2], e2 = m.v[2] - m.v[3], er = m.v[3] - r;
    ResItem<float> h;
    h.v[0] = e0 - el;
    h.v[1] = e1 - e0;
    h.v[2] = e2 - e1;
    h.v[3] = er - e2;
    return M::fma(c, m, M::add(h, M::sub(d, dp)));
}

// An FP32 sum that carries its rounding errors: hi + lo (Knuth's two-sum), within 2^-46 of the
// terms' magnitudes over a warp, for sums that must not lose bits to FP32.  An FP64 add would do
// it at 16 issue slots.  Lane sums of the CSR engine, us an iteration in FP32 / this / FP64 (the
// last two agree to all digits of the results): second-order mesh of 90K vertices 36.1 / 37.0 /
// 42.7, of 13K 10.7 / 11.0 / 14.6.
struct Sum2 {
    float hi, lo;
    __device__ __forceinline__ Sum2() {}
    __device__ __forceinline__ Sum2(float v) : hi(v), lo(0.f) {}
    __device__ __forceinline__ Sum2(float h, float l) : hi(h), lo(l) {}
    // an overflowed sum is infinite, whatever its errors
    __device__ __forceinline__ explicit operator double() const { return isfinite(hi) ? (double)hi + (double)lo : (double)hi; }
};
__device__ __forceinline__ Sum2 operator+(const Sum2 &a, const Sum2 &b) {
    const float s = a.hi + b.hi, t = s - a.hi;
    return Sum2(s, ((a.hi - (s - t)) + (b.hi - t)) + (a.lo + b.lo));
}
template <typename A>
__device__ __forceinline__ A lane_xor(const A &v, int o) {
    return __shfl_xor_sync(0xffffffffu, v, o);
}
template <>
__device__ __forceinline__ Sum2 lane_xor(const Sum2 &v, int o) {
    return Sum2(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}

// Sums of K values over the lanes with equal lane % NG by halving exchange: each step a lane
// sends one half of its values and adds to the other, (K + 1) / 2 left.  A lane ends with the
// totals of values [at, at + N) (those below K) in v[0 .. N), N = group_sum_left(K, NG).
// The sums are formed in type A, the lanes' values come in type I.
__host__ __device__ constexpr int group_sum_left(int K, int NG) {
    for (int o = 16; o >= NG; o /= 2) K = (K + 1) / 2;
    return K;
}
template <int NG, int O = 16, typename I, int K, typename A, int R>
__device__ __forceinline__ void group_sum(const I (&v)[K], A (&out)[R], int &at, int &end) {
    constexpr int N = (K + 1) / 2;
    const bool up = threadIdx.x & O;
    A w[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const I hi = N + k < K ? v[N + k < K ? N + k : 0] : (I)0.f;
        w[k] = A(up ? hi : v[k]) + A(lane_xor<I>(up ? v[k] : hi, O));
    }
    if (up) at += N;
    else end = min(end, at + N);
    if constexpr (O == NG) {
        static_assert(N == R, "values left");
#pragma unroll
        for (int k = 0; k < N; ++k) out[k] = w[k];
    } else {
        group_sum<NG, O / 2>(w, out, at, end);
    }
}

// sum over the warp's lanes below W, the same in all of them
template <int W = 32>
__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- the scalar chain of an iteration, every step of which the vector warps wait for.
// FP64 compares and quotients cost as much as several adds here (one warp's FP64 instruction takes
// 64 clocks whatever it waits for), so signs are read from the bits and the quotients are formed
// from the hardware's 20-bit reciprocal estimate by one third-order Householder step,
// y += y (e + e^2) with e = 1 - a y (2^-60 before its last rounding).  b y is then off by up to 1.5
// units in the last place.  For FP64 vectors (EXACT) one correction by its exact residual,
// q += y (b - a q) (Markstein 1990), leaves 2^-51 of a unit before the last rounding: the correctly
// rounded quotient but for ties that close; 0.13 us an iteration (48 x 40 Matern 8.26 -> 8.39).  FP32
// vectors round alpha and beta to FP32, and their dots are FP32 sums: there the 1.5 units stay.
__device__ __forceinline__ bool res_positive(double v) {           // v > 0
    const long long b = __double_as_longlong(v);
    return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool res_plain(double v) {              // 2^-400 < v < 2^400: quotients are normal numbers
    return (unsigned)((__double2hiint(v) >> 20) - 623) < 800u;
}
__device__ __forceinline__ double res_recip(double a) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-a, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// b / a, y = res_recip(a)
template <bool EXACT>
__device__ __forceinline__ double res_quotient(double b, double a, double y) {
    const double q = b * y;
    return EXACT ? fma(y, fma(-a, q, b), q) : q;
}
// outside the plain range; a function of its own to keep its code out of the loop's
static __device__ __noinline__ double res_divide(double b, double a) { return b / a; }
// alpha, beta and the predicted |r_{k+1}|^2 of one iteration from its dots; all lanes alike.
// Returns a DEV_ code or 0.
template <bool EXACT>
__device__ __forceinline__ int res_scalars(double rr, double pw, double rw, double ww, double &na, double &nb, double &rho) {
    const int lane = threadIdx.x & 31;
    na = nb = 0.0;
    rho = rr;
    if (!res_positive(pw)) return isfinite(pw) ? DEV_NOTSPD : DEV_NUMERIC;
    const double m2 = -2.0 * rw;
    const bool plain = res_plain(rr) && res_plain(pw);
    double irr = 0.0;
    if (plain) {
        // lane 1 takes 1 / rr while lane 0 takes 1 / pw
        const double y = res_recip(lane & 1 ? rr : pw);
        na = res_quotient<EXACT>(rr, pw, __shfl_sync(0xffffffffu, y, 0));
        irr = __shfl_sync(0xffffffffu, y, 1);
    } else {
        na = res_divide(rr, pw);
    }
    const double x = fma(na, fma(na, ww, m2), rr);
    rho = res_positive(x) ? x : 0.0;
    if (res_positive(rr)) nb = plain ? res_quotient<EXACT>(rho, rr, irr) : res_divide(rho, rr);
    return 0;
}

// 16-byte record {value, tag}: one 128-bit access each way, so that a reader that sees the
// iteration's tag sees its value
__device__ __forceinline__ void rec_st(ulonglong2 *p, double v, unsigned long long tag) {
    asm volatile(
        "{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}\n" ::"l"(p),
        "l"(__double_as_longlong(v)), "l"(tag)
        : "memory");
}
__device__ __forceinline__ bool rec_ld(const ulonglong2 *p, unsigned long long tag, double &v) {
    long long a;
    unsigned long long b;
    asm volatile(
        "{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
        : "=l"(a), "=l"(b)
        : "l"(p)
        : "memory");
    v = __longlong_as_double(a);
    return b == tag;
}
__device__ __forceinline__ uint64_t res_limit(const volatile uint64_t *limit_ns) { return limit_ns ? *limit_ns : RES_WAIT_NS; }
// Wait for a record's tag; false after *limit_ns (in shared memory: a limit in a register of the
// vector warps cost 1 %; null: RES_WAIT_NS).  The wait proper is a function of its own, out of the
// scalar warp's loop: with x kept 300 x 200 Matern 7.12 -> 7.04 us an iteration.
static __device__ __noinline__ bool rec_poll(const ulonglong2 *p, unsigned long long tag, double *out,
                                             const volatile uint64_t *limit_ns) {
    uint64_t t0 = 0;
    double v;
    for (unsigned it = 0;; ++it) {
        if (rec_ld(p, tag, v)) {
            *out = v;
            return true;
        }
        if ((it & 255) == 0) {
            const uint64_t t = global_ns();
            if (it == 0) t0 = t;
            else if (t - t0 > res_limit(limit_ns)) return false;
        }
    }
}
__device__ __forceinline__ bool rec_wait(const ulonglong2 *p, unsigned long long tag, double &v, const volatile uint64_t *limit_ns) {
    return rec_ld(p, tag, v) || rec_poll(p, tag, &v, limit_ns);
}

// ---- private vectors in tensor memory: 16 bytes a lane, the warp's own 32 lanes.  These are
// .sync.aligned: a __syncwarp() stands between them and a branch on a thread's own lines or rows
struct TmItem {
    uint32_t r[4];
};
__device__ __forceinline__ void tm_ld(TmItem &o, uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(o.r[0]), "=r"(o.r[1]), "=r"(o.r[2]), "=r"(o.r[3])
                 : "r"(addr));
}
// completes the loads into a (and b): their registers are named so that no use moves above
__device__ __forceinline__ void tm_wait(TmItem &a) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+r"(a.r[0]), "+r"(a.r[1]), "+r"(a.r[2]), "+r"(a.r[3]));
}
__device__ __forceinline__ void tm_wait(TmItem &a, TmItem &b) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(a.r[0]), "+r"(a.r[1]), "+r"(a.r[2]), "+r"(a.r[3]), "+r"(b.r[0]), "+r"(b.r[1]), "+r"(b.r[2]),
                   "+r"(b.r[3]));
}
template <int N>
__device__ __forceinline__ void tm_wait(TmItem (&a)[N]) {
    tm_wait(a[0]);
#pragma unroll
    for (int k = 1; k < N; ++k)      // the wait above covered them: no instruction, only the dependence
        asm volatile("" : "+r"(a[k].r[0]), "+r"(a[k].r[1]), "+r"(a[k].r[2]), "+r"(a[k].r[3]));
}
template <typename V>
__device__ __forceinline__ ResItem<V> tm_get(const TmItem &a) {
    ResItem<V> o;
    if constexpr (sizeof(V) == 8) {
        o.v[0] = __hiloint2double((int)a.r[1], (int)a.r[0]);
        o.v[1] = __hiloint2double((int)a.r[3], (int)a.r[2]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) o.v[k] = __uint_as_float(a.r[k]);
    }
    return o;
}
template <typename V>
__device__ __forceinline__ void item_words(const ResItem<V> v, uint32_t (&r)[4]) {
    if constexpr (sizeof(V) == 8) {
        r[0] = (uint32_t)__double2loint(v.v[0]);
        r[1] = (uint32_t)__double2hiint(v.v[0]);
        r[2] = (uint32_t)__double2loint(v.v[1]);
        r[3] = (uint32_t)__double2hiint(v.v[1]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) r[k] = __float_as_uint(v.v[k]);
    }
}
template <typename V>
__device__ __forceinline__ void tm_st(uint32_t addr, const ResItem<V> v) {
    uint32_t r[4];
    item_words<V>(v, r);
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3]));
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n"); }

// Scalar state of one column, in the registers of the scalar warp (all lanes alike), and
// its shift state in shared memory.
struct ResShift {
    double2 *z, *zp, *pi, *phi;
    uint8_t *act;
};

// Shift recurrences of one finished iteration (alpha, beta, predicted rho = |r_{k+1}|^2,
// measured vrn = v^T r_{k+1}); one warp.  Returns whether the column is still active.
__device__ __forceinline__ bool res_tail(const Solve &s, const ResShift &h, double alpha, double beta, double rho,
                                         double vrn, double ap, double bp, double lim2, double2 *hist, bool &bad) {
    const int lane = threadIdx.x & 31;
    bool any = rho > lim2;
    bad = !isfinite(vrn) || !isfinite(alpha) || !isfinite(beta);
    for (int l = lane; l < s.nshift; l += 32) {
        if (!h.act[l]) {
            if (hist) hist[3 * l] = hist[3 * l + 1] = hist[3 * l + 2] = make_double2(0.0, 0.0);
            continue;
        }
        const double2 sl = s.shift[l];
        const double2 z = h.z[l], zp = h.zp[l], phi = h.phi[l];
        // zeta_{k+1} / zeta_k as one complex quotient (see fused_tail)
        const double2 one_sa = make_double2(fma(sl.x, alpha, 1.0), sl.y * alpha);
        const double2 den = cadd(cscale(ap, cmul(zp, one_sa)), cscale(alpha * bp, csub(zp, z)));
        const double inv = ap / (den.x * den.x + den.y * den.y);
        const double2 ratio = cscale(inv, cmul(zp, make_double2(den.x, -den.y)));
        const double2 zn = cmul(ratio, z);
        const double2 as = cscale(alpha, ratio);
        const double2 bs = cscale(beta, cmul(ratio, ratio));
        h.pi[l] = cadd(h.pi[l], cmul(as, phi));
        if (hist) {
            hist[3 * l] = as;
            hist[3 * l + 1] = bs;
            hist[3 * l + 2] = z;
        }
        h.phi[l] = cadd(cscale(vrn, zn), cmul(bs, phi));
        h.zp[l] = z;
        h.z[l] = zn;
        // |zeta_{k+1}| ||r_{k+1}|| > tol ||v||, squared
        const double res2 = (zn.x * zn.x + zn.y * zn.y) * rho;
        if (!isfinite(res2)) bad = true;
        if (res2 > lim2) any = true;
        else h.act[l] = 0;
    }
    bad = __any_sync(0xffffffffu, bad);
    return __any_sync(0xffffffffu, any);
}

// ------------------------------------------------------------------ exchange primitives
__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// remote stores that count their bytes on the destination CTA's mbarrier
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, double v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n" ::"r"(addr),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
template <typename V>
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, const ResItem<V> v) {
    uint32_t r[4];
    item_words<V>(v, r);
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(
                     addr),
                 "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(bar)
                 : "memory");
}
// wait for a phase of this CTA's mbarrier, with the remote stores it counted; false after *limit_ns
__device__ __forceinline__ bool res_bar_wait(uint32_t bar, unsigned parity, const volatile uint64_t *limit_ns) {
    uint64_t t0 = 0;
    for (unsigned it = 0;; ++it) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 63) == 0) {
            const uint64_t t = global_ns();
            if (it == 0) t0 = t;
            else if (t - t0 > res_limit(limit_ns)) return false;
        }
    }
}
__device__ __forceinline__ void bar_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Control block of a CTA in shared memory.
struct ResCtl {
    double alpha, beta;          // of the next vector update
    int stop;                    // 1: the column is finished, 2: a wait ran out
    uint32_t tm;                 // tensor memory base
    volatile int done;           // queue entries processed when the last column's shifts converged
    volatile int head, tail;     // queue entries posted, processed
    int bad;                     // a vector warp's wait ran out
    volatile uint64_t wait_ns;   // limit of a wait
    uint64_t bar[2];             // exchange barriers by iteration parity
    double dflag[2];             // done flag of the team's first CTA, by parity
    double tot[4];               // the team's rr, pw, rw, ww
    struct Entry {
        double alpha, beta, rho, vr;
        int code, pad;
    } q[4];
};
static_assert(sizeof(ResCtl) <= RES_CTL_BYTES, "control block");

// This CTA's block of lattice lines and its neighbours in the team.
template <int KIND>
struct ResBlock {
    static constexpr bool D3 = KIND == KIND_3D7;
    static constexpr int H = KIND == KIND_2D13_SQ ? 2 : 1;
    int nx, ny, nz, my, mz, My, Mz, ya, Ly, za, Lz, L, slots;
    bool per;
    struct Has {
        unsigned bits;
        __device__ bool operator[](int d) const { return bits >> d & 1u; }
    } has;
    __device__ ResBlock(const Solve &s, const ResPlan &pl, int m) {
        nx = s.op.nx;
        ny = s.op.ny;
        nz = s.op.nz;
        per = s.op.periodic;
        My = pl.My;
        Mz = pl.M / My;
        my = m % My;
        mz = m / My;
        ya = (int)((int64_t)my * ny / My);
        Ly = (int)((int64_t)(my + 1) * ny / My) - ya;
        za = D3 ? z_begin(mz) : 0;
        Lz = D3 ? z_begin(mz + 1) - za : 1;
        L = Ly * Lz;
        slots = 2 * H * Lz + (D3 ? 2 * Ly : 0);
        has.bits = (per || my > 0 ? 1u : 0u) | (per || my < My - 1 ? 2u : 0u) |
                   (D3 && (per || mz > 0) ? 4u : 0u) | (D3 && (per || mz < Mz - 1) ? 8u : 0u);
    }
    __device__ int z_begin(int k) const { return (int)((int64_t)k * nz / Mz); }
    // halo slots: [y- : H Lz][y+ : H Lz][z- : Ly][z+ : Ly]
    __device__ int halo_lines(int dir) const { return !has[dir] ? 0 : dir < 2 ? H * Lz : Ly; }
    __device__ int nb(int dir) const {
        int a = my, b = mz;
        if (dir == 0) a = my == 0 ? My - 1 : my - 1;
        if (dir == 1) a = my == My - 1 ? 0 : my + 1;
        if (dir == 2) b = mz == 0 ? Mz - 1 : mz - 1;
        if (dir == 3) b = mz == Mz - 1 ? 0 : mz + 1;
        return b * My + a;
    }
    // shared line of a halo slot; its lattice line (y, z, unwrapped) and direction
    __device__ int hline(int q, int &y, int &z, int &dir) const {
        if constexpr (D3) {
            const int PY = Ly + 2;
            if (q < Lz) { dir = 0; y = ya - 1; z = za + q; return (q + 1) * PY; }
            if (q < 2 * Lz) { dir = 1; y = ya + Ly; z = za + q - Lz; return (q - Lz + 1) * PY + Ly + 1; }
            if (q < 2 * Lz + Ly) { dir = 2; y = ya + q - 2 * Lz; z = za - 1; return q - 2 * Lz + 1; }
            dir = 3;
            y = ya + q - 2 * Lz - Ly;
            z = za + Lz;
            return (Lz + 1) * PY + (q - 2 * Lz - Ly) + 1;
        } else {
            z = 0;
            if (q < H) { dir = 0; y = ya - H + q; return q; }
            dir = 1;
            y = ya + Ly + q - H;
            return Ly + q;
        }
    }
};

// ------------------------------------------------------------------ shift warp
// columns first, first + stride, ...
static __device__ __noinline__ void res_shift_role(const Solve &s, int stride, int first, const ResArgs &ar,
                                                   ResCtl::Entry *queue, volatile int *head, volatile int *tail_out,
                                                   volatile int *done_out, double2 *shm) {
    const int lane = threadIdx.x & 31;
    ResShift sh;
    sh.z = shm;
    sh.zp = sh.z + s.nshift;
    sh.pi = sh.zp + s.nshift;
    sh.phi = sh.pi + s.nshift;
    sh.act = reinterpret_cast<uint8_t *>(sh.phi + s.nshift);
    int tail = 0;
    for (int c = first; c < ar.ce; c += stride) {
        const double vv = s.class_size[c];
        if (!(vv > 0.0)) continue;
        for (int l = lane; l < s.nshift; l += 32) {
            sh.z[l] = sh.zp[l] = make_double2(1.0, 0.0);
            sh.pi[l] = make_double2(0.0, 0.0);
            sh.phi[l] = make_double2(vv, 0.0);
            sh.act[l] = 1;
        }
        __syncwarp();
        const double lim2 = s.tol * s.tol * vv;
        double alpha_p = 1.0, beta_p = 0.0, pi0 = 0.0, phi0 = vv;
        int iters = 0;
        bool done = false;
        for (;;) {
            while (*head == tail) __nanosleep(20);     // the scalar warp always posts an end
            __threadfence_block();
            const ResCtl::Entry e = queue[tail & 3];
            if (e.code < 0) {
                __syncwarp();
                ++tail;
                if (lane == 0) *tail_out = tail;
                if (e.code == -2) return;                // a wait ran out
                break;
            }
            if (!done) {
                if (e.code || (ar.hist && iters >= ar.hcap)) {
                    if (lane == 0) set_status(s.status, e.code ? e.code : DEV_OVERFLOW);
                    done = true;
                } else {
                    bool bad;
                    double2 *const hist = ar.hist ? ar.hist + ((size_t)c * ar.hcap + iters) * s.nshift * 3 : nullptr;
                    if (hist && lane == 0) ar.ab[(size_t)c * ar.hcap + iters] = make_double2(e.alpha, e.beta);
                    const bool still = res_tail(s, sh, e.alpha, e.beta, e.rho, e.vr, alpha_p, beta_p, lim2, hist, bad);
                    pi0 += e.alpha * phi0;
                    phi0 = e.vr + e.beta * phi0;
                    ++iters;
                    alpha_p = e.alpha;
                    beta_p = e.beta;
                    if (bad && lane == 0) set_status(s.status, DEV_NUMERIC);
                    if (!still || bad) {
                        done = true;
                        if (lane == 0 && !bad) atomicSub(s.remaining, 1);
                    } else if (iters >= ar.cap) {
                        done = true;                      // not converged: `remaining` keeps the column
                    }
                    if (done && lane == 0) s.rho[c] = e.rho;
                }
                if (done && lane == 0) *done_out = tail + 1;
            }
            __threadfence_block();
            __syncwarp();
            ++tail;
            if (lane == 0) *tail_out = tail;
        }
        for (int l = lane; l < s.nshift; l += 32) s.pi[(size_t)c * s.nshift + l] = sh.pi[l];
        if (lane == 0) {
            if (ar.terms) {
                double t = 0.0;
                for (int l = 0; l < s.nshift; ++l) t += s.weight[l].x * sh.pi[l].x - s.weight[l].y * sh.pi[l].y;
                s.terms[c] = t;
            }
            s.pi0[c] = pi0;
            s.col_iters[c] = iters;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ scalar warp
// BATCH: every team is a cluster and the limits are literals, so the cooperative code goes (eight
// lattices of 40^2 to 400^2: 13.3 -> 12.6 ms)
template <int NT, bool EXACT, bool BATCH>
__device__ __noinline__ void res_scalar_role(const Solve &s, const ResPlan &pl, const ResArgs &ar, int team, int m,
                                             ResCtl *ctl, const double *part, int NP, unsigned in_bytes) {
    const int lane = threadIdx.x & 31, M = pl.M;
    const bool clustered = BATCH || pl.clustered;
    const double ds = s.precision == 0 ? s.op.scale : (double)s.op.scale_f;
    const double ds2 = ds * ds;
    const bool scaled = ds != 1.0;
    ulonglong2 *const rec = clustered ? nullptr : ar.rec + (size_t)team * 2 * M * 8;
    unsigned long long tick = 0;
    int head = 0;
    // The team stops a fixed two iterations after the shift warp's verdict (the verdict on the
    // last but one posted iteration is waited for, a later one is not looked at), so that the
    // iterations a kept seed solution receives do not depend on timing.
    auto finished = [&](int base) -> int {
        while (ctl->tail < head - 1) {}
        __threadfence_block();
        const int d = ctl->done;
        return d > base && d <= head - 1;
    };
    for (int c = ar.cb + team; c < ar.ce; c += pl.J) {
        if (!(s.class_size[c] > 0.0)) continue;
        double c_alpha = 0.0, c_beta = 0.0, c_rho = 0.0;
        int code = 0;
        const int base = head;
        for (int it = 0;; ++it, ++tick) {
            const int par = (int)(tick & 1);
            const double *pp = part + (size_t)par * RES_NDOT * NP;
            const unsigned long long tag = tick + 1;
            ulonglong2 *const rp = rec + (size_t)par * M * 8;
            double fl = 0.0;
            bool ok = true;
            if (m == 0) fl = finished(base) ? 1.0 : 0.0;
            if (clustered) {
                if (m == 0 && lane < M)
                    st_async(mapa(smem_u32(&ctl->dflag[par]), lane), mapa(smem_u32(&ctl->bar[par]), lane), fl);
            } else {
                if (m == 0 && lane == 0) rec_st(rp + 5, fl, tag);
                ok = rec_wait(rp + 5, tag, fl, BATCH ? nullptr : &ctl->wait_ns);
            }
            bar_sync(3, 160);                 // the sums of vector warps 0 to 3
            if (clustered) {
                if (lane == 0) mbar_arrive_tx(&ctl->bar[par], in_bytes);      // armed for tick + 2
                fl = ctl->dflag[par];
            }
            int stop = __double2hiint(fl) != 0;
            if (!__all_sync(0xffffffffu, ok) || ctl->bad) {
                set_status(s.status, DEV_TIMEOUT);
                stop = 2;
            }
            // the levels ran unscaled: p.w and r.w carry one factor s, w.w two
            const double rr = ctl->tot[0];
            double pw = ctl->tot[1], rw = ctl->tot[2], ww = ctl->tot[3];
            if (scaled) {
                pw *= ds;
                rw *= ds;
                ww *= ds2;
            }
            double na, nb, rho;
            const int ncode = res_scalars<EXACT>(rr, pw, rw, ww, na, nb, rho);
            if (lane == 0) {
                ctl->alpha = na;
                ctl->beta = nb;
                ctl->stop = stop;
            }
            bar_sync(2, NT + 32);
            if (stop) break;
            if (m == 0) {
                // iteration it - 1 to the shift warp: its v^T r_{it} is this iteration's v.r
                if (it > 0) {
                    double vr_sum = 0.0;
                    for (int q = lane; q < (clustered ? NP : M); q += 32) {
                        double v = 0.0;
                        if (clustered) v = pp[(size_t)4 * NP + q];
                        else ok = rec_wait(rp + (size_t)q * 8 + 4, tag, v, BATCH ? nullptr : &ctl->wait_ns) && ok;
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
        if (m == 0) {
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

// The scalar warp of a replay: waits for the boundary rows, hands out the recorded alpha and
// beta.  A CTA waits for its neighbours only.
template <int NT, int KIND>
__device__ __noinline__ void res_replay_role(const Solve &s, const ResPlan &pl, const ResArgs &ar, int team, int m,
                                             ResCtl *ctl, unsigned in_bytes) {
    const int lane = threadIdx.x & 31, M = pl.M;
    const bool clustered = pl.clustered;
    const ResBlock<KIND> bk(s, pl, m);
    ulonglong2 *const rec = clustered ? nullptr : ar.rec + (size_t)team * 2 * M * 8;
    unsigned long long tick = 0;
    for (int c = ar.cb + team; c < ar.ce; c += pl.J) {
        if (!(s.class_size[c] > 0.0)) continue;
        const int last = s.col_iters[c] - 1;
        int stop = 0;
        for (int it = 0; it < last; ++it, ++tick) {
            const int par = (int)(tick & 1);
            const double2 ab = ar.ab[(size_t)c * ar.hcap + it];
            bool ok = true;
            // every vector warp has read the last alpha and beta (and, cooperative, sent its rows):
            // a neighbour's rows may be here before this CTA's own warps have come that far
            bar_sync(3, NT + 32);
            if (clustered) {
                ok = res_bar_wait(smem_u32(&ctl->bar[par]), (unsigned)(tick >> 1) & 1u, &ctl->wait_ns);
                __syncwarp();
                if (lane == 0) mbar_arrive_tx(&ctl->bar[par], in_bytes);      // armed for tick + 2
            } else {
                __threadfence();
                ulonglong2 *rp = rec + (size_t)par * M * 8;
                if (lane == 0) rec_st(rp + (size_t)m * 8, 0.0, tick + 1);
                double v;
                if (lane < 4 && bk.has[lane]) ok = rec_wait(rp + (size_t)bk.nb(lane) * 8, tick + 1, v, &ctl->wait_ns);
                __threadfence();
            }
            if (!__all_sync(0xffffffffu, ok)) {
                set_status(s.status, DEV_TIMEOUT);
                stop = 2;
            }
            if (lane == 0) {
                ctl->alpha = ab.x;
                ctl->beta = ab.y;
                ctl->stop = stop;
            }
            bar_sync(2, NT + 32);
            if (stop) return;
        }
        tick += 2;      // the last iteration exchanges nothing: its parity's buffers are free, see below
    }
}

// ------------------------------------------------------------------ vector warps
// RP: replay of a finished solve (vector form): alpha, beta from its records, no dots,
// y += coef_k r_k
template <typename V, int KIND, int NT, bool KX, bool RP, bool BATCH>
__device__ __forceinline__ void res_vector_role(const Solve &s, const ResPlan &pl, const ResArgs &ar, int team, int m,
                                                unsigned char *smem, const ResSmem &lay, ResCtl *ctl,
                                                const volatile uint64_t *limit_ns) {
    constexpr int E = res_epi<V>(), NW = NT / 32;
    constexpr bool MAT = KIND == KIND_2D13_SQ, D3 = KIND == KIND_3D7;
    constexpr int H = MAT ? 2 : 1, NB = D3 ? 6 : 4;
    constexpr bool SH = sizeof(V) == 4 && !D3;   // differences shared between lines
    constexpr bool RS = MAT && !KX;            // r in shared memory and u by its recurrence (else p shared, r private)
    constexpr bool PRIV = !RS;
    using It = ResItem<V>;
    using PM = PackMath<V, E>;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool clustered = BATCH || pl.clustered;
    const int M = pl.M, G = pl.G, GE = G * E, pitch = pl.pitch, cmax = pl.cmax;
    const ResBlock<KIND> bk(s, pl, m);
    const int nx = bk.nx, L = bk.L, Ly = bk.Ly;
    const bool per = bk.per;
    const int PY = Ly + 2 * H;                 // shared lines per z-plane
    double *const part = reinterpret_cast<double *>(smem + lay.part);     // [2][5][NP]
    const int NP = clustered ? NW * M : NW;
    V *const A = reinterpret_cast<V *>(smem + lay.a);       // p, or r (Matern without x), with halo lines
    V *const B = reinterpret_cast<V *>(smem + lay.b);       // u (Matern), one halo line a side
    V *const RH = reinterpret_cast<V *>(smem + lay.rh);     // r on the halo lines (where A is p)
    const V *const HB = reinterpret_cast<const V *>(smem + lay.hb);   // incoming boundary w (clustered), [2][slots][GE]
    V *const XS = reinterpret_cast<V *>(smem + lay.x) + (size_t)tid * E;   // + i * NT * E
    V *const XLS = reinterpret_cast<V *>(smem + lay.xl) + (size_t)tid * E;
    V *const DS = reinterpret_cast<V *>(smem + lay.d) + (size_t)tid * E;
    // tensor memory: [w | r | x | its low words | diagonal], cmax items of 4 words each, in the 128
    // columns of this warp (two warps of a CTA of 256 share a lane quarter, four of 512)
    const uint32_t tmw = ctl->tm + ((uint32_t)(wid & 3) << 21) + (uint32_t)(wid >> 2) * 128u;    // w
    const uint32_t tma = tmw + 4u * cmax;                                                        // r
    constexpr uint32_t YW = sizeof(V) == 8 ? 4 : 8;            // words of an item's y (FP64)
    const uint32_t tmy = tma + (PRIV ? 4u * cmax : 0u);
    const uint32_t tmx = tmy + (uint32_t)pl.yw * cmax, tmxl = tmx + (lay.x_tm ? 4u * cmax : 0u);
    const uint32_t tmd = tmxl + (lay.xl_tm ? 4u * cmax : 0u);
    const bool x_tm = lay.x_tm, xl_tm = lay.xl_tm, d_tm = lay.d_tm;
    constexpr bool keepx = KX;
    const size_t hstride = (size_t)pl.slots * GE;   // one parity of one CTA's halo buffer
    V *const hglob = clustered ? nullptr : static_cast<V *>(ar.halo) + (size_t)team * M * 2 * hstride;
    // ---- this thread's run: group g of lines [l0, l0 + cnt)
    const int g = tid % G, seg = tid / G;
    const int l0 = seg < pl.nseg ? (int)((int64_t)seg * L / pl.nseg) : 0;
    const int cnt = seg < pl.nseg ? (int)((int64_t)(seg + 1) * L / pl.nseg) - l0 : 0;   // cmax or cmax - 1, or 0
    const int items = __any_sync(0xffffffffu, cnt > 0) ? cmax : 0;      // a warp without lines skips the loops
    const int ev = min(E, nx - g * E);              // valid elements of the group
    const bool ragged = nx % E != 0;                // the last group is partial
    const bool lfix = lane == 0 || g == 0, rfix = lane == 31 || g == G - 1;
    const int go = E + g * E;                       // offset of the group in a shared line
    const int jz0 = D3 ? l0 / Ly : 0, jy0 = l0 - jz0 * Ly;     // its first line
    auto clip = [&](It &v) {
        if (ragged) {
#pragma unroll
            for (int e = 1; e < E; ++e) v.v[e] = e < ev ? v.v[e] : (V)0;
        }
    };
    // store an item of a shared line with its torus ghosts
    auto put = [&](V *line, int gg, const It &v) {
        if (!per) {
            ri_st(line + E + gg * E, v);
            return;
        }
        const int nv = min(E, nx - gg * E);
        V *q = line + E + gg * E;
        if (nv < E) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (e < nv) q[e] = v.v[e];
        } else {
            ri_st(q, v);
        }
        if (gg == 0) line[E + nx] = v.v[0];
        if (gg == G - 1) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (e == nv - 1) line[E - 1] = v.v[e];
        }
    };
    const V sc = op_scale<V>(s.op);
    const V centre = sizeof(V) == 8 ? (V)(D3 ? 6 : 4) : (V)0;    // the direct form's neighbour count
    const V k2 = op_kappa2<V>(s.op) + centre;
    const V k2m = op_kappa2<V>(s.op) + op_tau<V>(s.op) + centre;
    const bool use_d = !MAT && s.op.field_d != nullptr, use_m = !MAT && s.op.mask && !use_d;
    const int64_t plane = (int64_t)nx * bk.ny;
    auto own_vertex = [&](int jy, int jz) { return (int64_t)(bk.za + jz) * plane + (int64_t)(bk.ya + jy) * nx + g * E; };
    // own lines in order: y fastest
    auto next_line = [&](int &jy, int &jz) {
        ++jy;
        if constexpr (D3) {
            if (jy == Ly) {
                jy = 0;
                ++jz;
            }
        }
    };
    auto sline = [&](int jy, int jz) { return D3 ? (jz + 1) * PY + jy + 1 : jy + H; };
    // x += alpha p.  FP32 Matern solves run hundreds of iterations, and the roundings of these
    // additions are most of the gradient's error: there x carries a low word (compensated
    // summation: t = x + y, low = y - (t - x)), dropped when x is written.  300 x 200, eight
    // kappa^2: median relative error of the gradient 4.8e-7 -> 7e-8, 4.9 -> 5.5 ms; sums of 32
    // terms added to x at a time: 4.1e-7
    constexpr bool XL = MAT && KX && sizeof(V) == 4;
    auto x_get = [&](bool tmem, uint32_t col, const V *sh, int i) -> It {
        if (!tmem) return ri_ld(sh + (size_t)i * NT * E);
        TmItem t;
        tm_ld(t, col + 4u * i);
        tm_wait(t);
        return tm_get<V>(t);
    };
    auto x_put = [&](bool tmem, uint32_t col, V *sh, int i, const It &v) {
        if (tmem) tm_st<V>(col + 4u * i, v);
        else ri_st(sh + (size_t)i * NT * E, v);
    };
    auto x_add = [&](int i, const It &aa, const It &p) {
        if constexpr (XL) {
            const It x = x_get(x_tm, tmx, XS, i), y = PM::fma(aa, p, x_get(xl_tm, tmxl, XLS, i)), t = PM::add(x, y);
            x_put(x_tm, tmx, XS, i, t);
            x_put(xl_tm, tmxl, XLS, i, PM::sub(y, PM::sub(t, x)));
        } else {
            x_put(x_tm, tmx, XS, i, PM::fma(aa, p, x_get(x_tm, tmx, XS, i)));
        }
    };
    unsigned long long tick = 0;                    // iterations of this launch: parity and record tags

    // diagonal terms (kappa^2 field) and mask bits do not depend on the column
    uint64_t mbits = 0;
    for (int i = 0, jy = jy0, jz = jz0; i < items; ++i, next_line(jy, jz)) {
        It d = zero_pack<V, E>();
        if (i < cnt) {
            const int64_t v0 = own_vertex(jy, jz);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e < ev && use_d) d.v[e] = diag_ptr<V>(s.op)[v0 + e] + centre;
                if (e < ev && use_m && s.op.mask[v0 + e]) mbits |= 1ull << (i * E + e);
            }
        }
        __syncwarp();
        if (use_d && d_tm) tm_st<V>(tmd + 4u * i, d);
        else if (use_d) ri_st(DS + (size_t)i * NT * E, d);
    }

    for (int c = ar.cb + team; c < ar.ce; c += pl.J) {
        if (!(s.class_size[c] > 0.0)) continue;
        // ---- initial state: r = v, everything else zero
        for (int q = tid; q < (int)(lay.zero_bytes / 16); q += NT)
            reinterpret_cast<float4 *>(smem + lay.a)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        bar_sync(1, NT);
        // the column's starting vector: its colour's indicator, or (vector form) a right-hand side
        auto start = [&](int64_t v) -> V {
            return ar.rhs ? (V)ar.rhs[v * ar.ld + c] : (s.colour[v] == c ? (V)1 : (V)0);
        };
        uint64_t vbits = 0;                         // own-colour bits of the thread's vertices
        for (int i = 0, jy = jy0, jz = jz0; i < items; ++i, next_line(jy, jz)) {
            It r = zero_pack<V, E>();
            if (i < cnt) {
                const int64_t v0 = own_vertex(jy, jz);
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (e < ev) {
                        r.v[e] = start(v0 + e);
                        if (!ar.rhs && r.v[e] != (V)0) vbits |= 1ull << (i * E + e);
                    }
                if constexpr (RS) put(A + (size_t)sline(jy, jz) * pitch, g, r);
            }
            __syncwarp();
            const It zz = zero_pack<V, E>();
            tm_st<V>(tmw + 4u * i, zz);
            if constexpr (PRIV) tm_st<V>(tma + 4u * i, r);
            if (keepx && x_tm) tm_st<V>(tmx + 4u * i, zz);
            if (XL && xl_tm) tm_st<V>(tmxl + 4u * i, zz);
            if constexpr (RP) {
#pragma unroll
                for (uint32_t k = 0; k < YW; k += 4) tm_st<V>(tmy + YW * i + k, zz);
            }
        }
        tm_wait_st();
        for (int q = tid; q < bk.slots * G; q += NT) {
            const int sl = q / G, gg = q - sl * G;
            int y, z, dir;
            const int line = bk.hline(sl, y, z, dir);
            if (!bk.has[dir]) continue;
            if (per) {
                y = y < 0 ? y + bk.ny : (y >= bk.ny ? y - bk.ny : y);
                if constexpr (D3) z = z < 0 ? z + bk.nz : (z >= bk.nz ? z - bk.nz : z);
            }
            const int64_t v0 = (int64_t)z * plane + (int64_t)y * nx + gg * E;
            It r = zero_pack<V, E>();
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (gg * E + e < nx) r.v[e] = start(v0 + e);
            if constexpr (RS) put(A + (size_t)line * pitch, gg, r);
            else ri_st(RH + (size_t)sl * GE + gg * E, r);
        }
        V al = (V)0, be = (V)0;
        int stop = 0;
        double al64 = 0.0, ck = 0.0;
        int last = -1;
        if constexpr (RP) {
            last = s.col_iters[c] - 1;
            ck = ar.coef[(size_t)c * ar.hcap];
        }
        // y += coef (r - alpha w) with r, w of the last iteration, in FP64 before rounding
        auto y_add = [&](int i, const It &rold, const It &wv) {
            if constexpr (sizeof(V) == 8) {
                TmItem t;
                tm_ld(t, tmy + YW * i);
                const It r = PM::fma(PM::splat(-al * sc), wv, rold);
                tm_wait(t);
                tm_st<V>(tmy + YW * i, PM::fma(PM::splat((V)ck), r, tm_get<V>(t)));
            } else {
                TmItem t[2];
                tm_ld(t[0], tmy + YW * i);
                tm_ld(t[1], tmy + YW * i + 4);
                const double a64 = -al64 * (double)sc;
                tm_wait(t);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    ResItem<double> yv = tm_get<double>(t[h]);
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        yv.v[e] = ::fma(ck, ::fma(a64, (double)wv.v[2 * h + e], (double)rold.v[2 * h + e]), yv.v[e]);
                    tm_st<double>(tmy + YW * i + 4 * h, yv);
                }
            }
        };
        for (int it = 0;; ++it, ++tick) {
            const int par = (int)(tick & 1);
            const It bb = PM::splat(be);
            double ckn = 0.0;
            if constexpr (RP) ckn = it < last ? ar.coef[(size_t)c * ar.hcap + it + 1] : 0.0;
            {
                // ---- update r (and p, x) on own and halo lines
                const It nas = PM::splat(-al * sc), aa = PM::splat(al);
                // four items at a time, their loads in flight together
                int jy = jy0, jz = jz0;
                constexpr int U = MAT && KX ? 2 : 4;
                for (int i0 = 0; i0 < items; i0 += U) {
                    TmItem tw[U], ta[PRIV ? U : 1];
                    V *line[U];
                    It old[U];
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const int i = min(i0 + k, cmax - 1);
                        tm_ld(tw[k], tmw + 4u * i);
                        if constexpr (PRIV) tm_ld(ta[k], tma + 4u * i);
                        line[k] = A + (i0 + k < cnt ? sline(jy, jz) : 0) * pitch;
                        next_line(jy, jz);
                        old[k] = ri_ld(line[k] + go);
                    }
                    tm_wait(tw);
                    if constexpr (PRIV) tm_wait(ta);
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const int i = i0 + k;
                        if (i >= items) break;
                        const bool act = i < cnt;
                        const It wv = tm_get<V>(tw[k]);
                        if constexpr (!RS || RP) __syncwarp();
                        if constexpr (RP) y_add(i, RS ? old[k] : tm_get<V>(ta[PRIV ? k : 0]), wv);
                        It next;                    // r, or p
                        if constexpr (RS) {
                            next = PM::fma(nas, wv, old[k]);
                        } else {
                            if constexpr (keepx) x_add(i, aa, old[k]);
                            const It r = PM::fma(nas, wv, tm_get<V>(ta[k]));
                            tm_st<V>(tma + 4u * i, r);
                            next = PM::fma(bb, old[k], r);
                        }
                        if (act) put(line[k], g, next);
                    }
                }
                __syncwarp();
                tm_wait_st();
                if (RP && it == last) break;          // y has its last term
                const V *in = clustered ? HB + (size_t)(par ^ 1) * hstride : hglob + (size_t)(2 * m + (par ^ 1)) * hstride;
                for (int q = tid; q < bk.slots * G; q += NT) {
                    const int sl = q / G, gg = q - sl * G;
                    int y, z, dir;
                    const int li = bk.hline(sl, y, z, dir);
                    if (!bk.has[dir]) continue;
                    It wn = zero_pack<V, E>();
                    if (it > 0) {
                        const V *src = in + (size_t)sl * GE + gg * E;
                        wn = clustered ? ri_ld(src) : ri_ldcg(src);
                    }
                    V *line = A + (size_t)li * pitch;
                    if constexpr (RS) {
                        put(line, gg, PM::fma(nas, wn, ri_ld(line + E + gg * E)));
                    } else {
                        V *rp = RH + (size_t)sl * GE + gg * E;
                        const It r = PM::fma(nas, wn, ri_ld(rp));
                        ri_st(rp, r);
                        put(line, gg, PM::fma(bb, ri_ld(line + E + gg * E), r));
                    }
                }
            }
            bar_sync(1, NT);
            const It zz = zero_pack<V, E>();
            It d_rr = zz, d_pw = zz, d_rw = zz, d_ww = zz;
            V d_vr = (V)0;
            if constexpr (MAT) {
                // ---- u = Q1 r + beta u, or Q1 p, on own lines and one line beyond on each side
                const It cc = PM::splat(k2);
                // a row ahead: the line below, the old u and the side neighbours of the next row
                // load while this row is formed.  Loads past the run's end are clamped to the
                // block's lines and not used.
                int om = (H + l0) * pitch + go, od = om + pitch, ou = (1 + l0) * pitch + go;
                const int odmax = (L + 2 * H - 1) * pitch + go, oumax = (L + 1) * pitch + go;
                V *ul = B + (size_t)(1 + l0) * pitch;
                It up = ri_ld(A + om - pitch), mid = ri_ld(A + om), dn = ri_ld(A + od), uo = ri_ld(B + ou);
                if constexpr (SH) up = PM::sub(up, mid);
                V l = A[om - 1], r = A[om + E];
#pragma unroll 2
                for (int i = 0; i < items; ++i) {
                    om = od;
                    od = min(od + pitch, odmax);
                    ou = min(ou + pitch, oumax);
                    const It dn2 = ri_ld(A + od), uo2 = RS ? ri_ld(B + ou) : zz;
                    // side neighbours: across the lanes, and from the line at the warp's ends
                    const V ls = __shfl_up_sync(0xffffffffu, dn.v[E - 1], 1), rs = __shfl_down_sync(0xffffffffu, dn.v[0], 1);
                    V le = (V)0, re = (V)0;
                    if (lfix) le = A[om - 1];
                    if (rfix) re = A[om + E];
                    It u;
                    if constexpr (SH) {
                        const It d = PM::sub(mid, dn);
                        u = res_level_sh(cc, mid, l, r, d, up);
                        up = d;
                    } else {
                        u = res_level<V, 4>(cc, mid, l, r, dn, up, zz, zz);
                        up = mid;
                    }
                    if constexpr (RS) u = PM::fma(bb, uo, u);
                    clip(u);
                    if (i < cnt) {
                        if constexpr (!RP) d_pw = PM::fma(u, u, d_pw);
                        put(ul, g, u);
                    }
                    mid = dn;
                    dn = dn2;
                    uo = uo2;
                    l = lfix ? le : ls;
                    r = rfix ? re : rs;
                    ul += pitch;
                }
                for (int q = tid; q < 2 * G; q += NT) {
                    const int side = q / G, gg = q - side * G;
                    if (!bk.has[side]) continue;
                    const V *rw = A + (size_t)(side ? H + L : H - 1) * pitch + E + gg * E;
                    V *uo = B + (size_t)(side ? L + 1 : 0) * pitch;
                    It u = res_level<V, 4>(cc, ri_ld(rw), rw[-1], rw[E], ri_ld(rw + pitch), ri_ld(rw - pitch), zz, zz);
                    if constexpr (RS) u = PM::fma(bb, ri_ld(uo + E + gg * E), u);
                    const int nv = min(E, nx - gg * E);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e >= nv) u.v[e] = (V)0;
                    put(uo, gg, u);
                }
                bar_sync(1, NT);
            }
            {
                // ---- w = Q p (unscaled): 5/7-point from p, Matern from u; dots; boundary rows out
                const uint32_t hb_addr = smem_u32(HB) + (uint32_t)((par * hstride + g * E) * sizeof(V));
                const uint32_t bar_addr = smem_u32(&ctl->bar[par]);
                auto send = [&](int dir, int slot, const It v) {
                    const int to = bk.nb(dir);
                    if (clustered)
                        st_async<V>(mapa(hb_addr + (uint32_t)(slot * GE * sizeof(V)), to), mapa(bar_addr, to), v);
                    else
                        ri_st(hglob + (size_t)(2 * to + par) * hstride + (size_t)slot * GE + g * E, v);
                };
                constexpr int SO = MAT ? 1 : H;
                // as above, a row ahead: lines, lane exchange, and the private vectors
                int jy = jy0, jz = jz0;
                auto row_of = [&](int i) -> const V * {       // 3D: lines of the block, clamped to it
                    return A + (size_t)(i < cnt ? sline(jy, jz) : PY + 1) * pitch + go;
                };
                V *const S = MAT ? B : A;
                int om = (SO + l0) * pitch + go, od = om + pitch;        // 2D: this line, the next
                const int odmax = (L + 2 * SO - 1) * pitch + go;
                const V *row = D3 ? row_of(0) : S + om;
                const V *rrow = A + (size_t)(H + l0) * pitch + go;       // r (Matern)
                It up = ri_ld(row - pitch), mid = ri_ld(row), dn = ri_ld(row + pitch), fr = zz, bck = zz, rv = zz;
                if constexpr (SH) up = PM::sub(up, mid);
                if constexpr (D3) {
                    fr = ri_ld(row - PY * pitch);
                    bck = ri_ld(row + PY * pitch);
                }
                if constexpr (RS) rv = ri_ld(rrow);
                V l, r;
                if constexpr (D3) {
                    l = __shfl_up_sync(0xffffffffu, mid.v[E - 1], 1);
                    r = __shfl_down_sync(0xffffffffu, mid.v[0], 1);
                    if (lfix) l = row[-1];
                    if (rfix) r = row[E];
                } else {
                    l = row[-1];
                    r = row[E];
                }
                __syncwarp();
                TmItem ta, td;
                if constexpr (PRIV) tm_ld(ta, tma);
                if (!MAT && d_tm) tm_ld(td, tmd);
                uint64_t vb = vbits, mb = mbits;
#pragma unroll 2
                for (int i = 0; i < items; ++i) {
                    const bool act = i < cnt;
                    It cc;
                    const int in = min(i + 1, cmax - 1);
                    __syncwarp();
                    if constexpr (PRIV) {
                        if (!MAT && d_tm) tm_wait(ta, td);
                        else tm_wait(ta);
                        rv = tm_get<V>(ta);
                        tm_ld(ta, tma + 4u * in);
                    }
                    if constexpr (!MAT) {
                        if (use_d) {
                            if (d_tm) {
                                cc = tm_get<V>(td);
                                tm_ld(td, tmd + 4u * in);
                            } else {
                                cc = ri_ld(DS + (size_t)i * NT * E);
                            }
                        } else if (use_m) {
#pragma unroll
                            for (int e = 0; e < E; ++e) cc.v[e] = (unsigned)mb & (1u << e) ? k2m : k2;
                            mb >>= E;
                        } else {
                            cc = PM::splat(k2);
                        }
                    } else {
                        cc = PM::splat(k2);
                    }
                    const int jyc = jy, jzc = jz;
                    It up2, mid2, dn2, fr2 = zz, bck2 = zz, rv2 = rv;
                    V l2, r2, le = (V)0, re = (V)0;
                    const V *nrow = nullptr;
                    if constexpr (D3) {
                        next_line(jy, jz);
                        nrow = row_of(i + 1);
                        mid2 = ri_ld(nrow);
                        dn2 = ri_ld(nrow + pitch);
                        up2 = ri_ld(nrow - pitch);
                        fr2 = ri_ld(nrow - PY * pitch);
                        bck2 = ri_ld(nrow + PY * pitch);
                        const bool more = i + 1 < cnt;
                        l2 = __shfl_up_sync(0xffffffffu, mid2.v[E - 1], 1);
                        r2 = __shfl_down_sync(0xffffffffu, mid2.v[0], 1);
                        if (lfix && more) l2 = nrow[-1];
                        if (rfix && more) r2 = nrow[E];
                    } else {
                        ++jy;
                        om = od;
                        od = min(od + pitch, odmax);      // past the run's end: not used
                        mid2 = dn;
                        dn2 = ri_ld(S + od);
                        l2 = __shfl_up_sync(0xffffffffu, mid2.v[E - 1], 1);
                        r2 = __shfl_down_sync(0xffffffffu, mid2.v[0], 1);
                        if (lfix) le = S[om - 1];
                        if (rfix) re = S[om + E];
                        if constexpr (RS) {
                            rrow += pitch;
                            rv2 = ri_ld(rrow);
                        }
                    }
                    It wv;
                    if constexpr (SH) {
                        up2 = PM::sub(mid, dn);
                        wv = res_level_sh(cc, mid, l, r, up2, up);
                    } else {
                        if constexpr (!D3) up2 = mid;
                        wv = res_level<V, NB>(cc, mid, l, r, dn, up, fr, bck);
                    }
                    clip(wv);
                    if constexpr (RS) clip(rv);    // a torus ghost inside a partial item is not r
                    __syncwarp();
                    tm_st<V>(tmw + 4u * i, wv);
                    if (act) {
                        if constexpr (!RP) {
                            d_rr = PM::fma(rv, rv, d_rr);
                            if constexpr (!MAT) d_pw = PM::fma(mid, wv, d_pw);
                            d_rw = PM::fma(rv, wv, d_rw);
                            d_ww = PM::fma(wv, wv, d_ww);
#pragma unroll
                            for (int e = 0; e < E; ++e)
                                if ((unsigned)vb & (1u << e)) d_vr += rv.v[e];
                        }
                        // boundary rows to the neighbours' halo slots
                        if constexpr (D3) {
                            if (jyc == 0 && bk.has[0]) send(0, bk.Lz + jzc, wv);
                            if (jyc == Ly - 1 && bk.has[1]) send(1, jzc, wv);
                            // z neighbours share this CTA's y range; their Lz may differ
                            if (jzc == 0 && bk.has[2]) {
                                const int zn = bk.mz == 0 ? bk.Mz - 1 : bk.mz - 1;
                                send(2, 2 * (bk.z_begin(zn + 1) - bk.z_begin(zn)) + Ly + jyc, wv);
                            }
                            if (jzc == bk.Lz - 1 && bk.has[3]) {
                                const int zn = bk.mz == bk.Mz - 1 ? 0 : bk.mz + 1;
                                send(3, 2 * (bk.z_begin(zn + 1) - bk.z_begin(zn)) + jyc, wv);
                            }
                        } else {
                            if (jyc < H || jyc >= L - H) {
                                if (jyc < H && bk.has[0]) send(0, H + jyc, wv);
                                if (jyc >= L - H && bk.has[1]) send(1, jyc - (L - H), wv);
                            }
                        }
                    }
                    vb >>= E;
                    up = up2;
                    mid = mid2;
                    dn = dn2;
                    fr = fr2;
                    bck = bck2;
                    rv = rv2;
                    l = !D3 && lfix ? le : l2;
                    r = !D3 && rfix ? re : r2;
                    row = nrow;
                }
                __syncwarp();
                if constexpr (PRIV) {
                    if (!MAT && d_tm) tm_wait(ta, td);     // the load past the last item
                    else tm_wait(ta);
                }
                tm_wait_st();
                if constexpr (RP) {
                    if (!clustered) __threadfence();
                    bar_arrive(3, NT + 32);
                } else {
                V flat[RES_NDOT] = {d_rr.v[0], d_pw.v[0], d_rw.v[0], d_ww.v[0], d_vr}, sum[1];
#pragma unroll
                for (int e = 1; e < E; ++e) {
                    flat[0] += d_rr.v[e];
                    flat[1] += d_pw.v[e];
                    flat[2] += d_rw.v[e];
                    flat[3] += d_ww.v[e];
                }
                int k = 0, end = RES_NDOT;                // four lanes hold dot k, where k < end
                group_sum<4>(flat, sum, k, end);
#pragma unroll
                for (int o = 2; o > 0; o >>= 1) sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
                const double tot = (double)sum[0];
                // One warp adds FP64 numbers at a quarter of the SM's rate (64 clocks an
                // instruction whatever its lanes), so the team's sums are formed by four or five
                // vector warps, one a dot, and the scalar warp starts from the totals.
                if (clustered) {
                    if (k < end) {
                        const uint32_t slot = smem_u32(part + (size_t)(par * RES_NDOT + k) * NP + m * NW + wid);
                        for (int q = lane & 3; q < M; q += 4) st_async(mapa(slot, q), mapa(bar_addr, q), tot);
                    }
                    if (wid < 4) {
                        if (!res_bar_wait(bar_addr, (unsigned)(tick >> 1) & 1u, limit_ns)) ctl->bad = 1;
                        const double *pp = part + (size_t)(par * RES_NDOT + wid) * NP;
                        double a = lane < NP ? pp[lane] : 0.0;
                        for (int q = lane + 32; q < NP; q += 32) a += pp[q];
                        __syncwarp();
                        a = lane_sum(a);
                        if (lane == 0) ctl->tot[wid] = a;
                        bar_arrive(3, 160);
                    }
                } else {
                    if (k < end && (lane & 3) == 0) part[(size_t)(par * RES_NDOT + k) * NP + wid] = tot;
                    // every thread's boundary rows on their way: a fence by the publishers alone
                    // orders them too, but waits for all of them at the end (FP64 Matern 200 x
                    // 150, four vectors: 19.9 against 18.8 ms)
                    __threadfence();
                    bar_sync(1, NT);
                    const unsigned long long tag = tick + 1;
                    ulonglong2 *const rp = ar.rec + ((size_t)team * 2 + par) * M * 8;
                    if (wid < RES_NDOT) {
                        const double a = lane_sum<NW>(lane < NW ? part[(size_t)(par * RES_NDOT + wid) * NP + lane] : 0.0);
                        __threadfence();
                        if (lane == 0) rec_st(rp + (size_t)m * 8 + wid, a, tag);
                    }
                    if (wid < 4) {
                        bool ok = true;
                        double a = 0.0;
                        for (int q0 = lane; q0 < M; q0 += 128) {      // four records a lane in flight
                            double v[4];
                            uint64_t t0 = 0;
                            for (unsigned spin = 0;; ++spin) {
                                bool got = true;
#pragma unroll
                                for (int b = 0; b < 4; ++b) {
                                    v[b] = 0.0;
                                    if (q0 + 32 * b < M) got &= rec_ld(rp + (size_t)(q0 + 32 * b) * 8 + wid, tag, v[b]);
                                }
                                if (got) break;
                                if ((spin & 255) == 255) {
                                    const uint64_t t = global_ns();
                                    if (t0 == 0) t0 = t;
                                    else if (t - t0 > res_limit(limit_ns)) {
                                        ok = false;
                                        break;
                                    }
                                }
                            }
                            a = q0 == lane ? v[0] : a + v[0];
#pragma unroll
                            for (int b = 1; b < 4; ++b)
                                if (q0 - lane + 32 * b < M) a += v[b];
                        }
                        __syncwarp();
                        if (!ok) ctl->bad = 1;
                        a = lane_sum(a);
                        if (lane == 0) ctl->tot[wid] = a;
                        __threadfence();     // the neighbours' boundary rows after their records
                        bar_arrive(3, 160);
                    }
                }
                }
            }
            bar_sync(2, NT + 32);
            al = (V)ctl->alpha;
            be = (V)ctl->beta;
            stop = ctl->stop;
            if constexpr (RP) {
                al64 = ctl->alpha;
                ck = ckn;
            }
            if (stop) break;
        }
        ++tick;
        if constexpr (RP) {
            // The next column starts on the parity the last iteration did not send: a neighbour
            // may still read the other one.
            ++tick;
            for (int i = 0, jy = jy0, jz = jz0; i < items; ++i, next_line(jy, jz)) {
                double yv[E];
                if constexpr (sizeof(V) == 8) {
                    TmItem t;
                    tm_ld(t, tmy + YW * i);
                    tm_wait(t);
                    const It q = tm_get<V>(t);
#pragma unroll
                    for (int e = 0; e < E; ++e) yv[e] = q.v[e];
                } else {
                    TmItem t[2];
                    tm_ld(t[0], tmy + YW * i);
                    tm_ld(t[1], tmy + YW * i + 4);
                    tm_wait(t);
#pragma unroll
                    for (int e = 0; e < E; ++e) yv[e] = tm_get<double>(t[e >> 1]).v[e & 1];
                }
                if (i < cnt) {
                    const int64_t v0 = own_vertex(jy, jz);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e < ev) ar.y[(v0 + e) * ar.ld + c] = yv[e];
                }
                __syncwarp();
            }
        }
        if constexpr (keepx) {
            const int tile = c / s.T, t = c - tile * s.T;
            V *x = static_cast<V *>(s.x) + (int64_t)tile * s.op.n * s.T + t;
            for (int i = 0, jy = jy0, jz = jz0; i < items; ++i, next_line(jy, jz)) {
                const It xv = x_get(x_tm, tmx, XS, i);
                if (i < cnt) {
                    const int64_t v0 = own_vertex(jy, jz);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e < ev) x[(v0 + e) * s.T] = xv.v[e];
                }
                __syncwarp();
            }
        }
        bar_sync(1, NT);
        if (stop == 2) break;
    }
}

// ------------------------------------------------------------------ kernel
// NT vector threads, then the scalar warp and the shift warp
template <typename V, int KIND, int NT, bool KX, bool RP, bool BATCH>
__device__ __forceinline__ void resident_body(const Solve &s, const ResPlan &pl, const ResArgs &ar, int team, int m,
                                              unsigned char *smem) {
    constexpr int NW = NT / 32;
    const int wid = threadIdx.x >> 5;
    const ResSmem lay = res_smem(pl, (int)sizeof(V), KIND, s.nshift, KX, KIND != KIND_2D13_SQ && s.op.field_d != nullptr);
    ResCtl *const ctl = reinterpret_cast<ResCtl *>(smem + lay.bc);
    constexpr uint32_t TM_COLS = NT == 256 ? 256 : 512;
    const int NP = pl.clustered ? NW * pl.M : NW;
    unsigned in_bytes = 0;
    if (pl.clustered) {
        const ResBlock<KIND> bk(s, pl, m);
        for (int d = 0; d < 4; ++d) in_bytes += (unsigned)(bk.halo_lines(d) * pl.G * 16);
        if (!RP) in_bytes += (unsigned)(NP * RES_NDOT * 8) + 8u;
    }
    if (wid == NW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&ctl->tm)),
                     "n"(TM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
        if ((threadIdx.x & 31) == 0) {
            ctl->done = 0;
            ctl->head = ctl->tail = 0;
            ctl->bad = 0;
            ctl->wait_ns = ar.wait_ns;
            if (pl.clustered) {
                mbar_init(&ctl->bar[0], 1);
                mbar_init(&ctl->bar[1], 1);
                mbar_init_fence();
                mbar_arrive_tx(&ctl->bar[0], in_bytes);
                mbar_arrive_tx(&ctl->bar[1], in_bytes);
            }
        }
        __syncwarp();
    }
    __syncthreads();
    if (pl.clustered) cluster_sync_all();          // barriers armed before any remote store
    if (wid < NW)
        res_vector_role<V, KIND, NT, KX, RP, BATCH>(s, pl, ar, team, m, smem, lay, ctl, BATCH ? nullptr : &ctl->wait_ns);
    else if (RP && wid == NW)
        res_replay_role<NT, KIND>(s, pl, ar, team, m, ctl, in_bytes);
    else if (wid == NW)
        res_scalar_role<NT, sizeof(V) == 8, BATCH>(s, pl, ar, team, m, ctl, reinterpret_cast<const double *>(smem + lay.part), NP, in_bytes);
    else if (m == 0 && !RP)
        res_shift_role(s, pl.J, ar.cb + team, ar, ctl->q, &ctl->head, &ctl->tail, &ctl->done,
                       reinterpret_cast<double2 *>(smem + lay.shift));
    __syncwarp();
    __syncthreads();
    if (pl.clustered) cluster_sync_all();          // no CTA leaves while another may still store to it
    if (wid == NW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(ctl->tm), "n"(TM_COLS));
}

template <typename V, int KIND, int NT, bool KX, bool RP>
__global__ void __launch_bounds__(NT + 64, 1) k_resident(const __grid_constant__ Solve s, const __grid_constant__ ResPlan pl,
                                                         const __grid_constant__ ResArgs ar) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int team = blockIdx.x / pl.M;
    resident_body<V, KIND, NT, KX, RP, false>(s, pl, ar, team, blockIdx.x - team * pl.M, smem);
}

// A batch's items (instance, column) of one kind and cluster size: a cluster solves one item.
template <typename V, int KIND, int NT>
__global__ void __launch_bounds__(NT + 64, 1) k_resident_batch(const Solve *solves, const ResPlan *plans, const int2 *items,
                                                               int M, int cap) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Solve s;
    __shared__ ResPlan pl;
    const int2 it = items[blockIdx.x / M];
    for (int q = threadIdx.x; q < (int)(sizeof(Solve) / 4); q += blockDim.x)
        reinterpret_cast<uint32_t *>(&s)[q] = reinterpret_cast<const uint32_t *>(solves + it.x)[q];
    for (int q = threadIdx.x; q < (int)(sizeof(ResPlan) / 4); q += blockDim.x)
        reinterpret_cast<uint32_t *>(&pl)[q] = reinterpret_cast<const uint32_t *>(plans + it.x)[q];
    __syncthreads();
    ResArgs ar{};
    ar.wait_ns = RES_WAIT_NS;
    ar.cb = it.y;
    ar.ce = it.y + 1;
    ar.cap = cap;
    ar.terms = 1;
    resident_body<V, KIND, NT, false, false, true>(s, pl, ar, 0, blockIdx.x % M, smem);
}

}  // namespace ld
