// Plan and shared-memory layout of the resident engine, common to its kernel
// (engine_resident.cuh) and its host side (engine_resident.cu).
#pragma once
#include <cstddef>
#include <cstdint>

#include "internal.h"

namespace ld {

constexpr int RES_CTL_BYTES = 288;

// bytes of one CTA's shared memory by purpose (offsets from the dynamic base)
struct ResSmem {
    size_t part, bc, shift, a, b, rh, hb, x, xl, d, bytes;
    size_t zero_bytes;      // from `a`: what a new column starts from zero
    bool xl_on;             // x carries its low words (FP32 Matern, see x_add)
    bool x_tm, xl_tm, d_tm; // x, its low words, diagonal in tensor memory (else in shared memory)
};

__host__ __device__ inline ResSmem res_smem(const ResPlan &p, int word, int kind, int nshift, int keepx, bool field) {
    const bool mat = kind == KIND_2D13_SQ, d3 = kind == KIND_3D7;
    const int E = 16 / word, H = mat ? 2 : 1, NW = p.nt / 32;
    const size_t ge = (size_t)p.G * E * word, pitch = (size_t)p.pitch * word;
    const size_t np = p.clustered ? (size_t)NW * p.M : NW;
    const size_t priv = (size_t)p.cmax * p.nt * 16;
    ResSmem s;
    // private vectors in tensor memory, 128 words a thread: w; r (but Matern without x); then
    // x and the diagonal while they fit
    int room = 32 - p.cmax * ((mat && !keepx ? 1 : 2) + p.yw / 4);
    s.x_tm = keepx && room >= p.cmax;
    if (s.x_tm) room -= p.cmax;
    s.xl_on = mat && keepx && word == 4;
    s.xl_tm = s.xl_on && room >= p.cmax;
    if (s.xl_tm) room -= p.cmax;
    s.d_tm = field && room >= p.cmax;
    size_t o = 0;
    s.part = o;
    o += (2 * 5 * np * 8 + 15) / 16 * 16;
    s.bc = o;
    o += RES_CTL_BYTES;
    s.shift = o;
    o += ((size_t)nshift * 65 + 15) / 16 * 16;
    s.a = o;
    o += (size_t)(d3 ? (p.Ly + 2) * (p.Lz + 2) : p.Ly + 2 * H) * pitch;
    s.b = o;
    if (mat) o += (size_t)(p.Ly + 2) * pitch;
    s.rh = o;
    if (!mat || keepx) o += (size_t)p.slots * ge;
    s.x = o;
    if (keepx && !s.x_tm) o += priv;
    s.xl = o;
    if (s.xl_on && !s.xl_tm) o += priv;
    s.zero_bytes = o - s.a;
    s.hb = o;
    if (p.clustered) o += 2 * (size_t)p.slots * ge;
    s.d = o;
    if (field && !s.d_tm) o += priv;
    s.bytes = o;
    return s;
}

// ---- CSR (engine_resident_csr.cuh)
constexpr int RES_CSR_T = 16;            // vectors of a team at most
constexpr int RES_CSR_CTL_BYTES = 24 + 4 * 40 + 16 * RES_CSR_T + 32 + 8;

struct CsrSmem {
    size_t part, ctl, shift, val, col, row, colour, coef, p, bytes;
};

__host__ __device__ inline CsrSmem csr_smem(const CsrPlan &p, int word, int nshift) {
    const size_t a16 = 15;
    CsrSmem s;
    size_t o = 0;
    s.p = o;
    o += (size_t)(p.own_max + p.ext_max) * p.T * word;
    s.part = o;
    o += (size_t)2 * 5 * p.T * (p.nt / 32) * 8;
    s.ctl = o;
    o += (RES_CSR_CTL_BYTES + a16) / 16 * 16;
    s.shift = o;
    o += ((size_t)nshift * 65 + a16) / 16 * 16;
    s.coef = o;
    o += (size_t)3 * p.T * word;
    s.val = o;
    o += ((size_t)p.nnz_max * word + a16) / 16 * 16;
    s.col = o;
    o += ((size_t)p.nnz_max * 2 + a16) / 16 * 16;
    s.row = o;
    o += ((size_t)(p.own_max + 1) * 4 + a16) / 16 * 16;
    s.colour = o;
    o += ((size_t)p.own_max * 4 + a16) / 16 * 16;
    s.bytes = o;
    return s;
}

}  // namespace ld
