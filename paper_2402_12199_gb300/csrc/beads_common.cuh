// Bead-sum device code shared by the pair kernel (beads.cu) and the
// training-pair sampler (train.cu).
//
// Paper mapping: the traditional interaction of two composite bodies is the
// double sum U = sum_i sum_j u_bead(r_ij) over their beads (Methods), with
// every inter-body bead distance evaluated (abstract).  Everything here runs
// in the frame of body i: its beads are the template d_k, body j's beads are
// b_l = s + R_rel d_l with s = R(q_i)^T R_ij and R_rel = R(q_i^* q_j).
#pragma once

#include "rb_internal.cuh"

namespace rb {

constexpr int kPadBeads = 3;  // far-away template entries after the last bead

// Bead potential.  Lennard-Jones (kind 0): rc2, sig2, eps4, eps24, u_shift.
// Half-power half-cosine of Eq. 1 (kind 1: the continuous reading, kind 2:
// as printed): A, b, c, p; eps4 = 1 and u_shift = 0 so that the accumulated
// sum is the energy itself.  rc2 is the squared cutoff in every kind.
struct BeadPot {
    float rc2, sig2, eps4, eps24, u_shift;
    float rc2_test;  // rc2 + a bound on the rounding of the expanded and the box distance tests
    int kind;
    float hA, hb, hc, hp;
    // (r_c + r_circ)^2 with a rounding margin: a column of body i farther
    // than this from body j's centre has no bead within r_c of any bead of j
    float cull2 = 3.0e38f;
};

BeadPot bead_pot(const rb_system* s);

// Per-CTA shared template: sT[k] = (x, y, z, 0); sN[2k], sN[2k+1] =
// (-2x, -2x, -2y, -2y), (-2z, -2z, thr - |d|^2, thr - |d|^2): duplicated for
// packed FP32x2 arithmetic (0.5 * (-2x) = -x exactly); thr is the distance
// test's threshold: |b|^2 - 2 b.d < thr - |d|^2 flags a possible hit.
// The template is padded with kPadBeads entries far away (never within any
// cutoff), so the distance loop can take up to kPadBeads + 1 template beads
// per iteration.
__device__ inline void load_template(const float4* __restrict__ tmpl, int n_beads, float thr,
                                     float4* sT, float4* sN) {
    for (int t = threadIdx.x; t < n_beads + kPadBeads; t += blockDim.x) {
        if (t < n_beads) {
            const float4 d = tmpl[t];
            sT[t] = d;
            const float dd = thr - (d.x * d.x + d.y * d.y + d.z * d.z);
            sN[2 * t] = make_float4(-2.f * d.x, -2.f * d.x, -2.f * d.y, -2.f * d.y);
            sN[2 * t + 1] = make_float4(-2.f * d.z, -2.f * d.z, dd, dd);
        } else {  // padding bead at 1e18 sigma
            sN[2 * t] = make_float4(-2e18f, -2e18f, 0.f, 0.f);
            sN[2 * t + 1] = make_float4(0.f, 0.f, -1e36f, -1e36f);
        }
    }
}

// Three-input minimum (one instruction on sm_100 and later).
__device__ inline float fmin3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Body j's beads owned by this lane, b_l = s + R_rel d_l for l = lane + 32 m
// (m < 2 NP), as scalars and as packed pairs, with |b_l|^2; unused slots sit
// far away (never within any cutoff).
template <int NP>
__device__ inline void slots_setup(const float3 s, const Mat3& Rr, const float4* sT, int n_beads,
                                   int lane, float (&bx)[2 * NP], float (&by)[2 * NP],
                                   float (&bz)[2 * NP], float2 (&Bx)[NP], float2 (&By)[NP],
                                   float2 (&Bz)[NP], float2 (&BB)[NP]) {
#pragma unroll
    for (int m = 0; m < 2 * NP; ++m) {
        const int l = lane + 32 * m;
        if (l < n_beads) {
            const float4 d = sT[l];
            const float3 b = mul(Rr, make_float3(d.x, d.y, d.z));
            bx[m] = s.x + b.x;
            by[m] = s.y + b.y;
            bz[m] = s.z + b.z;
        } else {
            bx[m] = by[m] = bz[m] = 1e18f;
        }
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        Bx[q] = make_float2(bx[2 * q], bx[2 * q + 1]);
        By[q] = make_float2(by[2 * q], by[2 * q + 1]);
        Bz[q] = make_float2(bz[2 * q], bz[2 * q + 1]);
        BB[q] = __ffma2_rn(Bz[q], Bz[q], __ffma2_rn(By[q], By[q], __fmul2_rn(Bx[q], Bx[q])));
    }
}

// Lennard-Jones accumulators of one lane: force on each owned bead (packed),
// sum of (s^12 - s^6) and number of pairs inside r_c.
template <int NP>
struct LJAcc {
    float2 Fx[NP], Fy[NP], Fz[NP];
    float2 acc, cnt;
    __device__ void zero() {
#pragma unroll
        for (int q = 0; q < NP; ++q) Fx[q] = Fy[q] = Fz[q] = make_float2(0.f, 0.f);
        acc = cnt = make_float2(0.f, 0.f);
    }
};

// One template bead d (given as md = -2 d, duplicated) against every owned
// slot: exact separations r = b - d, the strict cutoff r^2 < r_c^2 and the
// masked Lennard-Jones body.
template <int NP>
__device__ inline void lj_bead(const float2 md0, const float2 md1, const float2 md2,
                               const float2 (&Bx)[NP], const float2 (&By)[NP],
                               const float2 (&Bz)[NP], const BeadPot& pot, LJAcc<NP>& a) {
    const float2 half2 = make_float2(0.5f, 0.5f);
    const float2 sig2v = make_float2(pot.sig2, pot.sig2);
    const float2 e48 = make_float2(2.f * pot.eps24, 2.f * pot.eps24);
    const float2 me24 = make_float2(-pot.eps24, -pot.eps24);
    const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const float2 rx = __ffma2_rn(half2, md0, Bx[q]);
        const float2 ry = __ffma2_rn(half2, md1, By[q]);
        const float2 rz = __ffma2_rn(half2, md2, Bz[q]);
        float2 r2 = __fmul2_rn(rx, rx);
        r2 = __ffma2_rn(ry, ry, r2);
        r2 = __ffma2_rn(rz, rz, r2);
        const bool inx = r2.x < pot.rc2, iny = r2.y < pot.rc2;
        const float2 inv2 = make_float2(inx ? __fdividef(1.f, r2.x) : 0.f,
                                        iny ? __fdividef(1.f, r2.y) : 0.f);
        const float2 s2 = __fmul2_rn(sig2v, inv2);
        const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
        const float2 s12 = __fmul2_rn(s6, s6);
        a.acc = __fadd2_rn(a.acc, __ffma2_rn(s6, m1, s12));
        a.cnt = __fadd2_rn(a.cnt, make_float2(inx ? 1.f : 0.f, iny ? 1.f : 0.f));
        const float2 fr = __fmul2_rn(inv2, __ffma2_rn(s12, e48, __fmul2_rn(s6, me24)));
        a.Fx[q] = __ffma2_rn(fr, rx, a.Fx[q]);
        a.Fy[q] = __ffma2_rn(fr, ry, a.Fy[q]);
        a.Fz[q] = __ffma2_rn(fr, rz, a.Fz[q]);
    }
}

// The half-power half-cosine (paper, Eq. 1) counterpart of lj_bead, per
// slot: x = b - r; r <= b: u = x^p - 2A, -u'/r = p x^(p-1) / r; b < r < r_c:
// u = -A (1 + cos t) (kind 1) or -A cos t (kind 2) with t = c (r - b),
// -u'/r = -A c sin t / r; nothing from r_c on.  Both branches are evaluated
// and one selected (no divergence inside the warp).
template <int NP>
__device__ inline void hphc_bead(const float2 md0, const float2 md1, const float2 md2,
                                 const float2 (&Bx)[NP], const float2 (&By)[NP],
                                 const float2 (&Bz)[NP], const BeadPot& pot, LJAcc<NP>& a) {
    const float2 half2 = make_float2(0.5f, 0.5f);
    const float u_base = pot.kind == 2 ? 0.f : -pot.hA;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const float2 rx = __ffma2_rn(half2, md0, Bx[q]);
        const float2 ry = __ffma2_rn(half2, md1, By[q]);
        const float2 rz = __ffma2_rn(half2, md2, Bz[q]);
        float2 r2 = __fmul2_rn(rx, rx);
        r2 = __ffma2_rn(ry, ry, r2);
        r2 = __ffma2_rn(rz, rz, r2);
        const float r2s[2] = {r2.x, r2.y};
        float us[2], fs[2], ns[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool in = r2s[h] < pot.rc2;
            const float ir = rsqrtf(r2s[h]);
            const float r = r2s[h] * ir;
            const float x = pot.hb - r;
            const float xp = fmaxf(x, 0.f);
            const float xp1 = __powf(xp, pot.hp - 1.f);  // 0 at x = 0 (p > 1)
            float sn, cs;
            __sincosf(pot.hc * (r - pot.hb), &sn, &cs);
            const bool rep = x >= 0.f;
            const float u = rep ? fmaf(xp1, xp, -2.f * pot.hA) : fmaf(-pot.hA, cs, u_base);
            const float f = rep ? pot.hp * xp1 * ir : -pot.hA * pot.hc * sn * ir;
            us[h] = in ? u : 0.f;
            fs[h] = in ? f : 0.f;
            ns[h] = in ? 1.f : 0.f;
        }
        a.acc = __fadd2_rn(a.acc, make_float2(us[0], us[1]));
        a.cnt = __fadd2_rn(a.cnt, make_float2(ns[0], ns[1]));
        const float2 fr = make_float2(fs[0], fs[1]);
        a.Fx[q] = __ffma2_rn(fr, rx, a.Fx[q]);
        a.Fy[q] = __ffma2_rn(fr, ry, a.Fy[q]);
        a.Fz[q] = __ffma2_rn(fr, rz, a.Fz[q]);
    }
}

// One template bead against every owned slot with the potential POT
// (0: Lennard-Jones, 1: half-power half-cosine, either reading).
template <int NP, int POT>
__device__ inline void bead_terms(const float2 md0, const float2 md1, const float2 md2,
                                  const float2 (&Bx)[NP], const float2 (&By)[NP],
                                  const float2 (&Bz)[NP], const BeadPot& pot, LJAcc<NP>& a) {
    if constexpr (POT == 0)
        lj_bead<NP>(md0, md1, md2, Bx, By, Bz, pot, a);
    else
        hphc_bead<NP>(md0, md1, md2, Bx, By, Bz, pot, a);
}

// Reduce-scatter of seven sums over the warp: lanes with bit 16 set keep sums
// 4..6 (and a zero) and hand 0..3 to their partner, then bits 8 and 4 halve
// the kept set again and xor 2 and 1 complete it: lane 4 k returns sum k.
__device__ inline float warp_scatter7(const float (&v)[7]) {
    const int lane = threadIdx.x & 31;
    float w[4];
    {
        const bool b = lane & 16;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float keep = b ? (j + 4 < 7 ? v[j + 4] : 0.f) : v[j];
            const float give = b ? v[j] : (j + 4 < 7 ? v[j + 4] : 0.f);
            w[j] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
        }
    }
    float u[2];
    {
        const bool b = lane & 8;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float keep = b ? w[j + 2] : w[j];
            const float give = b ? w[j] : w[j + 2];
            u[j] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
        }
    }
    const bool b = lane & 4;
    float t = (b ? u[1] : u[0]) + __shfl_xor_sync(0xffffffffu, b ? u[0] : u[1], 4);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    return t;
}

// v[0..2] = F_j, v[3..5] = T = sum_l b_l x f_l, v[6] = E, reduced over the
// warp with xor shuffles (every lane gets the sums).
template <int NP>
__device__ inline void warp_finish(const float (&bx)[2 * NP], const float (&by)[2 * NP],
                                   const float (&bz)[2 * NP], const LJAcc<NP>& a,
                                   const BeadPot& pot, float (&v)[7]) {
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = 0.f;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const float fx[2] = {a.Fx[q].x, a.Fx[q].y}, fy[2] = {a.Fy[q].x, a.Fy[q].y},
                    fz[2] = {a.Fz[q].x, a.Fz[q].y};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int m = 2 * q + h;
            v[0] += fx[h];
            v[1] += fy[h];
            v[2] += fz[h];
            v[3] += by[m] * fz[h] - bz[m] * fy[h];
            v[4] += bz[m] * fx[h] - bx[m] * fz[h];
            v[5] += bx[m] * fy[h] - by[m] * fx[h];
        }
    }
    v[6] = pot.eps4 * (a.acc.x + a.acc.y) - pot.u_shift * (a.cnt.x + a.cnt.y);
    const float t = warp_scatter7(v);
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = __shfl_sync(0xffffffffu, t, 4 * k);
}

// Whole-warp bead double sum of one body pair in the frame of body i, any
// template.  NP = packed slot pairs per lane: the lane owns beads
// l = lane + 32 m, m = 0 .. 2 NP - 1, of body j.  Every bead-pair distance is
// tested (expanded form, with a rounding margin); one warp vote per U
// template beads decides whether any slot may be inside r_c, and then the
// exact separations, the strict cutoff and the masked Lennard-Jones body run
// for those U beads.  Result as in warp_finish.
template <int NP, int POT = 0, int U = 2>
__device__ inline void bead_pair_warp(const float3 s, const Mat3& Rr, const float4* sT,
                                      const float4* sN, int n_beads, const BeadPot& pot,
                                      int lane, float (&v)[7]) {
    float bx[2 * NP], by[2 * NP], bz[2 * NP];
    float2 Bx[NP], By[NP], Bz[NP], BB[NP];
    slots_setup<NP>(s, Rr, sT, n_beads, lane, bx, by, bz, Bx, By, Bz, BB);
    LJAcc<NP> a;
    a.zero();
    static_assert(U >= 1 && U <= kPadBeads + 1, "template padding");
    for (int k = 0; k < n_beads; k += U) {
        float2 md[U][3];
        float th[U], mn[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float4 n0 = sN[2 * (k + u)], n1 = sN[2 * (k + u) + 1];
            md[u][0] = make_float2(n0.x, n0.y);
            md[u][1] = make_float2(n0.z, n0.w);
            md[u][2] = make_float2(n1.x, n1.y);
            th[u] = n1.z;
            mn[u] = 3.0e38f;
        }
        // test: |b|^2 - 2 b.d < thr - |d|^2, i.e. r^2 < thr in expanded form
        // (3 packed FMAs per 2 slots, one three-input min per 2 slots, one
        // compare per template bead); the rounding bound is folded into thr,
        // so no pair inside r_c is missed
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                float2 t = __ffma2_rn(Bx[q], md[u][0], BB[q]);
                t = __ffma2_rn(By[q], md[u][1], t);
                t = __ffma2_rn(Bz[q], md[u][2], t);
                mn[u] = fmin3(mn[u], t.x, t.y);
            }
        bool hit = false;
#pragma unroll
        for (int u = 0; u < U; ++u) hit |= mn[u] < th[u];
        if (__any_sync(0xffffffffu, hit)) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                bead_terms<NP, POT>(md[u][0], md[u][1], md[u][2], Bx, By, Bz, pot, a);
        }
    }
    warp_finish<NP>(bx, by, bz, a, pot, v);
}

// Shared-memory form of a column-structured template (see BeadCols): the
// columns' (x, y) and the z values that all of them hold.
constexpr int kMaxCols = kMaxBeads / 5;
constexpr int kColWords = (kMaxCols + 31) / 32;  // column masks of 32 bits
struct ColShared {
    float2 xy[kMaxCols + 1];
    float z[kMaxColLen];
};
__device__ inline void load_columns(const float4* __restrict__ tmpl, const BeadCols& cols, ColShared& sc) {
    for (int c = threadIdx.x; c < cols.n_cols; c += blockDim.x) {
        const float4 d = tmpl[c * cols.len];
        sc.xy[c] = make_float2(d.x, d.y);
    }
    for (int m = threadIdx.x; m < cols.len; m += blockDim.x) sc.z[m] = cols.z[m];
}

// Lane's share of a column test: column c (< n_cols) within sqrt(r2) of the point s.
template <int C>
__device__ inline bool column_near(const float3 s, const ColShared& sc, const BeadCols& cols, int c, float r2) {
    if (c >= cols.n_cols) return false;
    const float dx = s.x - sc.xy[c].x, dy = s.y - sc.xy[c].y;
    const float dz = fmaxf(fmaxf(cols.z[0] - s.z, s.z - cols.z[C - 1]), 0.f);
    return dx * dx + dy * dy + dz * dz <= r2;
}

// Squared distance of (x, y, z) from the box [xl, xh] x [yl, yh] x [zl, zh].
__device__ inline float box_dist2(float x, float y, float z, float xl, float xh, float yl, float yh,
                                  float zl, float zh) {
    const float dx = fmaxf(fmaxf(xl - x, x - xh), 0.f);
    const float dy = fmaxf(fmaxf(yl - y, y - yh), 0.f);
    const float dz = fmaxf(fmaxf(zl - z, z - zh), 0.f);
    return dx * dx + dy * dy + dz * dz;
}

__device__ inline float warp_fmin(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ inline float warp_fmax(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// One bead pair at (dx, dy, dz), squared distance r2 (on: inside the cutoff,
// else it adds nothing): force on j's bead, energy sum and count, as lj_bead
// and hphc_bead form them.
template <int POT>
__device__ inline void bead_term(float dx, float dy, float dz, float r2, bool on, const BeadPot& pot,
                                 float& Fx, float& Fy, float& Fz, float& acc, float& cnt) {
    float fr;
    if constexpr (POT == 0) {
        const float inv2 = on ? __fdividef(1.f, r2) : 0.f;
        const float s2 = pot.sig2 * inv2, s6 = s2 * s2 * s2, s12 = s6 * s6;
        acc += s12 - s6;
        fr = inv2 * (2.f * pot.eps24 * s12 - pot.eps24 * s6);
    } else {
        const float ir = rsqrtf(r2), r = r2 * ir, x = pot.hb - r;
        float u;
        if (x >= 0.f) {
            const float xp1 = __powf(x, pot.hp - 1.f);  // 0 at x = 0 (p > 1)
            u = fmaf(xp1, x, -2.f * pot.hA);
            fr = pot.hp * xp1 * ir;
        } else {
            float sn, cs;
            __sincosf(pot.hc * (r - pot.hb), &sn, &cs);
            u = fmaf(-pot.hA, cs, pot.kind == 2 ? 0.f : -pot.hA);
            fr = -pot.hA * pot.hc * sn * ir;
        }
        acc += on ? u : 0.f;
        fr = on ? fr : 0.f;
    }
    cnt += on ? 1.f : 0.f;
    Fx = fmaf(fr, dx, Fx);
    Fy = fmaf(fr, dy, Fy);
    Fz = fmaf(fr, dz, Fz);
}

// Whole-warp bead double sum of one body pair for a column-structured template
// of columns of C beads, in the frame of body i: b[m] is body j's bead
// l = lane + 32 m (unused slots far away).
//   1. j's beads within the cutoff of the box around body i's beads are packed
//      into `buf` (room for 32 NS); the others cannot interact.  Of a touching
//      pair's 125 beads 10 to 40 are left, so a lane holds one bead from here
//      on instead of four.
//   2. Per 32 packed beads: the columns of i that come within the cutoff of
//      those beads' box (a lane per column), then column by column the squared
//      distances of every lane's bead to its C beads, (dx^2 + dy^2) + dz^2 with
//      dz^2 kept per lane, and one vote.
//   3. A lane with beads inside the cutoff evaluates its own ones, the warp
//      until no lane has any left.
// What is skipped would have added exact zeros.  Returns false (v untouched)
// if no bead pair is inside the cutoff; else the lane's partial sums of F_j
// (v[0..2]), T = sum_l b_l x f_l (v[3..5]) and E (v[6]).
template <int NS, int C, int POT>
__device__ inline bool bead_pair_cols(const float (&bx)[NS], const float (&by)[NS], const float (&bz)[NS],
                                      const ColShared& sc, const BeadCols& cols, const BeadPot& pot,
                                      float4* buf, int lane, float (&v)[7]) {
    const unsigned lt = (1u << lane) - 1u;
    int nb = 0;
#pragma unroll
    for (int m = 0; m < NS; ++m) {
        const bool near = box_dist2(bx[m], by[m], bz[m], cols.x_lo, cols.x_hi, cols.y_lo, cols.y_hi,
                                    cols.z[0], cols.z[C - 1]) <= pot.rc2_test;
        const unsigned w = __ballot_sync(0xffffffffu, near);
        if (near) buf[nb + __popc(w & lt)] = make_float4(bx[m], by[m], bz[m], 0.f);
        nb += __popc(w);
    }
    if (nb == 0) return false;
    __syncwarp();
    bool any = false;
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = 0.f;
    float acc = 0.f, cnt = 0.f;
    for (int k0 = 0; k0 < nb; k0 += 32) {
        const bool own = k0 + lane < nb;
        const float4 b = buf[min(k0 + lane, nb - 1)];  // surplus lanes repeat the last bead, masked below
        const float xl = warp_fmin(b.x), xh = warp_fmax(b.x), yl = warp_fmin(b.y), yh = warp_fmax(b.y);
        const float zl = warp_fmin(b.z), zh = warp_fmax(b.z);
        float zz[C];
#pragma unroll
        for (int m = 0; m < C; ++m) {
            const float dz = b.z - cols.z[m];
            zz[m] = own ? __fmul_rn(dz, dz) : 3.0e38f;
        }
        float Fx = 0.f, Fy = 0.f, Fz = 0.f;
#pragma unroll
        for (int wd = 0; wd < kColWords; ++wd) {
            if (32 * wd >= cols.n_cols) break;
            const int cl = min(32 * wd + lane, cols.n_cols - 1);
            const float2 cxy = sc.xy[cl];
            // the column as the point nearest to the beads' box
            const bool near = 32 * wd + lane < cols.n_cols &&
                              box_dist2(cxy.x, cxy.y, fminf(fmaxf(cols.z[0], zl), cols.z[C - 1]), xl, xh, yl,
                                        yh, zl, zh) <= pot.rc2_test;
            unsigned todo = __ballot_sync(0xffffffffu, near);
            while (todo) {
                const int c = 32 * wd + __ffs(todo) - 1;
                todo &= todo - 1u;
                const float2 xy = sc.xy[c];
                const float dx = b.x - xy.x, dy = b.y - xy.y;
                const float p = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
                float r2[C], mn = 3.0e38f;
#pragma unroll
                for (int m = 0; m < C; ++m) r2[m] = __fadd_rn(p, zz[m]);
#pragma unroll
                for (int m = 0; m + 1 < C; m += 2) mn = fmin3(mn, r2[m], r2[m + 1]);
                if (C & 1) mn = fminf(mn, r2[C - 1]);
                if (!__any_sync(0xffffffffu, mn < pot.rc2)) continue;
                any = true;
                unsigned mine = 0;
#pragma unroll
                for (int m = 0; m < C; ++m) mine |= r2[m] < pot.rc2 ? 1u << m : 0u;
                do {
                    const bool on = mine != 0u;
                    const int m = on ? __ffs(mine) - 1 : 0;
                    mine &= mine - 1u;
                    const float dz = b.z - sc.z[m];
                    bead_term<POT>(dx, dy, dz, __fadd_rn(p, __fmul_rn(dz, dz)), on, pot, Fx, Fy, Fz, acc, cnt);
                } while (__any_sync(0xffffffffu, mine != 0u));
            }
        }
        v[0] += Fx;
        v[1] += Fy;
        v[2] += Fz;
        v[3] += b.y * Fz - b.z * Fy;
        v[4] += b.z * Fx - b.x * Fz;
        v[5] += b.x * Fy - b.y * Fx;
    }
    __syncwarp();  // buf is read before the next pair's beads are packed
    v[6] = pot.eps4 * acc - pot.u_shift * cnt;
    return any;
}

}  // namespace rb
