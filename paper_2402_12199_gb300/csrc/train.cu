// Training of the pair energy network: on-device sampling of pair
// configurations labelled by the bead sum, the force-matching loss and its
// weight gradient, and Adam.
//
// Paper mapping: the paper trains a fully connected energy network on pair
// configurations sampled from bead-level simulations and expressed in the
// frame of body 1 (Methods; SI Sec. 1), then takes forces and torques as the
// energy's gradients (SI Sec. 6).  Here configurations are drawn directly
// (uniform direction, uniform orientation, separation uniform between contact
// and the body-pair cutoff) and labelled with E, F_j, tau_i, tau_j by the bead
// double sum; the network is fitted to forces and torques (and optionally the
// energy) with a loss whose weight gradient needs the derivative of the
// network's input gradient:
//
//   l_b  = w_b [ |F_j - F*|^2 + lam_tau (|tau_i - tau_i*|^2 + |tau_j - tau_j*|^2)
//          + lam_E (E - E*)^2 ],         L = mean_b l_b,
//   w_b  = min(1, exp(-E* / kT_w)) / (1 + (|F*|^2 + lam_tau (|tau_i*|^2 +
//          |tau_j*|^2)) / f_scale^2)
//   (each factor 1 when its parameter is 0).  The paper's training pairs come
//   from simulations at T = 0.2 - 2.0, i.e. Boltzmann-weighted, and it caps
//   large force/torque targets (SI Sec. 6); pairs drawn uniformly here get the
//   Boltzmann factor and a smooth force cap as importance weights instead.
//   With G = dE/d(s, q) the outputs are linear in G, so dl/dG = v (7 numbers)
//   and dL/dW = d/dW sum_b [u_b . grad_(s,q) E_hat_b + c_b E_hat_b]
//   (u = e_scale v / B, c = e_scale dl/dE / B): a forward pass carrying the
//   tangent along u (z, z_dot, h, h_dot) followed by its reverse pass,
//     a_zdot = a_hdot phi'(z),  a_z = a_h phi'(z) + a_hdot phi''(z) z_dot,
//     dW_l += a_z h_{l-1}^T + a_zdot h_dot_{l-1}^T,  db_l += a_z,
//     a_h_{l-1} = W_l^T a_z,  a_hdot_{l-1} = W_l^T a_zdot,
//   with phi(z) = z sigma(z).  The seed a_hdot_D = w_o is that of the plain
//   reverse pass, so a_zdot_l is its signal g_l and is formed once, with the
//   predicted forces.  All arithmetic FP32; every sum in a fixed order.
#include <algorithm>
#include <cmath>
#include <new>

#include "beads_common.cuh"
#include "nn_f32_common.cuh"

struct rb_trainer {
    rb_mlp* mlp = nullptr;
    int64_t max_batch = 0;
    float lr = 1e-3f, beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    int64_t t = 0;
    float* m = nullptr;        // Adam first moment (n_params)
    float* v = nullptr;        // Adam second moment
    float* grad = nullptr;     // gradient of the last rb_train_grad / vjp
    float* pred = nullptr;     // predicted pair outputs of a batch (12 floats per pair)
    float* part = nullptr;     // per CTA: its share of the gradient (n_params)
    float* scratch = nullptr;  // per CTA: phi', phi'' terms of its tile (kTrSlots)
    double* loss_part = nullptr;
    double* loss_out = nullptr;
    int sms = 1;
};

namespace rb {

// ------------------------------------------------------------- sampler
// One warp per sample.  The contact separation is a bisection on "some bead
// distance is below `contact`", 40 halvings of [0, Rc].  Testing all n_beads^2
// distances in each of them was 140 thousand instructions a sample (8.9 ms for
// 65536 cube pairs, 1.6% of the time being the label); here
//   * the first halvings (kCoarse, to a bracket of about 0.3 sigma) scan the
//     beads exactly, but for a column template only the columns of body i
//     within contact + r_circ of body j's centre (no bead of another column can
//     be closer than contact to a bead of j), leaving at the first hit;
//   * one scan at the bracket's middle then lists the bead pairs closer than
//     contact + half the bracket: a centre that moves by d changes a distance
//     by at most d, so only these can decide the halvings that are left;
//   * those test the listed pairs alone, two per lane, and stop when the middle
//     no longer differs from an end of the bracket in FP32.
// A list longer than kCand (parallel faces; contacts far beyond the bead spacing,
// where many pairs are nearly equally far) is given up and tried again after two
// more halvings.
// A grazing contact amplifies the last bit of a distance and the label's
// repulsion that of the separation (by up to 3e-3 of the labels' rms in one
// element), so every quantity that a halving or a label depends on is rounded as
// the scan of all pairs rounds it, operation by operation (rotation, place,
// bead_dist2, bead_terms): separations and labels are those of the full scan, bit
// for bit.  The label takes the columns near body j only, and of those the beads
// inside the cutoff; the others would add exact zeros.  Measured: 8885 -> 370 us
// for 65536 cube pairs at contact 0.85; bound by instruction issue.
constexpr int kCoarse = 5;
constexpr int kCand = 64;

// Squared distance from its components, in the full scan's rounding: the x-y
// part first, so that it is shared along a column.
__device__ __forceinline__ float bead_dist2_xy(float rx, float ry) {
    return __fmaf_rn(rx, rx, __fmul_rn(ry, ry));
}
__device__ __forceinline__ float bead_dist2(float rx, float ry, float rz) {
    return __fmaf_rn(rz, rz, bead_dist2_xy(rx, ry));
}
// R(q) (as qmat) with the roundings spelled out: the compiler's choice of which
// product of a sum is fused differs between instantiations.
__device__ __forceinline__ Mat3 rotation(const float4& q) {
    const float w = q.x, x = q.y, y = q.z, z = q.w;
    const float xx = __fmul_rn(x, x), zz = __fmul_rn(z, z), xz = __fmul_rn(x, z), wz = __fmul_rn(w, z),
                wx = __fmul_rn(w, x);
    Mat3 R;
    R.m[0] = __fmaf_rn(-2.f, __fmaf_rn(y, y, zz), 1.f);
    R.m[1] = 2.f * __fmaf_rn(x, y, -wz);
    R.m[2] = 2.f * __fmaf_rn(w, y, xz);
    R.m[3] = 2.f * __fmaf_rn(x, y, wz);
    R.m[4] = __fmaf_rn(-2.f, __fmaf_rn(z, z, xx), 1.f);
    R.m[5] = 2.f * __fmaf_rn(y, z, -wx);
    R.m[6] = 2.f * __fmaf_rn(-w, y, xz);
    R.m[7] = 2.f * __fmaf_rn(y, z, wx);
    R.m[8] = __fmaf_rn(-2.f, __fmaf_rn(y, y, xx), 1.f);
    return R;
}
// R d, the products of each component fused except the second.
__device__ __forceinline__ float3 rotate_bead(const Mat3& R, const float4& d) {
    return make_float3(__fmaf_rn(R.m[2], d.z, __fmaf_rn(R.m[0], d.x, __fmul_rn(R.m[1], d.y))),
                       __fmaf_rn(R.m[5], d.z, __fmaf_rn(R.m[3], d.x, __fmul_rn(R.m[4], d.y))),
                       __fmaf_rn(R.m[8], d.z, __fmaf_rn(R.m[6], d.x, __fmul_rn(R.m[7], d.y))));
}

// Smallest squared distance between the beads of one column of body i (at x, y)
// and the lane's beads of j.
template <int NP, int C>
__device__ inline float column_min(float x, float y, const BeadCols& cols, const float (&bx)[2 * NP],
                                   const float (&by)[2 * NP], const float (&bz)[2 * NP]) {
    float mn = 3.0e38f;
#pragma unroll
    for (int m = 0; m < 2 * NP; ++m) {
        const float p = bead_dist2_xy(bx[m] - x, by[m] - y);
#pragma unroll
        for (int z = 0; z < C; ++z) {
            const float rz = bz[m] - cols.z[z];
            mn = fminf(mn, __fmaf_rn(rz, rz, p));
        }
    }
    return mn;
}
// The column's beads (bit z) with one of the lane's beads within sqrt(r2).
template <int NP, int C>
__device__ inline unsigned column_hits(float x, float y, const BeadCols& cols, const float (&bx)[2 * NP],
                                       const float (&by)[2 * NP], const float (&bz)[2 * NP], float r2) {
    float mn[C];
#pragma unroll
    for (int z = 0; z < C; ++z) mn[z] = 3.0e38f;
#pragma unroll
    for (int m = 0; m < 2 * NP; ++m) {
        const float p = bead_dist2_xy(bx[m] - x, by[m] - y);
#pragma unroll
        for (int z = 0; z < C; ++z) {
            const float rz = bz[m] - cols.z[z];
            mn[z] = fminf(mn[z], __fmaf_rn(rz, rz, p));
        }
    }
    unsigned hits = 0u;
#pragma unroll
    for (int z = 0; z < C; ++z) hits |= mn[z] < r2 ? 1u << z : 0u;
    return hits;
}

template <int NP, int C, int POT>
__global__ void __launch_bounds__(256, NP <= 3 || C == 0 ? 2 : 1)
    k_sample_pairs(int64_t n, const float* __restrict__ u, const float4* __restrict__ tmpl,
                   int n_beads, BeadCols cols, float r_circ, float Rc, float contact, BeadPot pot,
                   float4* __restrict__ cfg, float4* __restrict__ lab, float* __restrict__ rho_c) {
    constexpr int MB = 2 * NP;
    __shared__ float4 sT[kMaxBeads + 1];
    __shared__ float4 sN[C == 0 ? 2 * (kMaxBeads + kPadBeads) : 1];  // any template: its distance-test form
    __shared__ ColShared sc;
    __shared__ unsigned short s_cand[8][kCand];  // bead of i << 8 | bead of j
    if (C == 0) {
        load_template(tmpl, n_beads, pot.rc2_test, sT, sN);
    } else {
        for (int t = threadIdx.x; t < n_beads; t += blockDim.x) sT[t] = tmpl[t];
        load_columns(tmpl, cols, sc);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    const float sig2 = contact * contact;
    // what rounding can take from a listed pair's distance
    const float slack = 1e-3f + 4e-6f * (Rc + contact);
    unsigned short* cand = s_cand[warp];
    for (int64_t b = gw; b < n; b += nw) {
        const float* ub = u + 6 * b;
        const float z = 2.f * ub[0] - 1.f;
        float sp, cp;
        sincospif(2.f * ub[1], &sp, &cp);
        const float rxy = sqrtf(fmaxf(0.f, 1.f - z * z));
        const float3 dir = make_float3(rxy * cp, rxy * sp, z);
        float s3, c3, s4, c4;
        sincospif(2.f * ub[3], &s3, &c3);
        sincospif(2.f * ub[4], &s4, &c4);
        const float a = sqrtf(1.f - ub[2]), bq = sqrtf(ub[2]);
        const float4 q = make_float4(a * s3, a * c3, bq * s4, bq * c4);
        const Mat3 Rr = rotation(q);
        float px[MB], py[MB], pz[MB];  // R d_l of the lane's beads l = lane + 32 m
#pragma unroll
        for (int m = 0; m < MB; ++m) {
            const int l = lane + 32 * m;
            const float3 r = rotate_bead(Rr, sT[min(l, n_beads - 1)]);
            px[m] = l < n_beads ? r.x : 1e18f;
            py[m] = l < n_beads ? r.y : 1e18f;
            pz[m] = l < n_beads ? r.z : 1e18f;
        }
        float bx[MB], by[MB], bz[MB];
        auto centre = [&](float rho) {
            return make_float3(__fmul_rn(rho, dir.x), __fmul_rn(rho, dir.y), __fmul_rn(rho, dir.z));
        };
        auto place = [&](float rho) {  // the lane's beads with j's centre at rho dir
            const float3 s = centre(rho);
#pragma unroll
            for (int m = 0; m < MB; ++m) {
                bx[m] = __fadd_rn(s.x, px[m]);
                by[m] = __fadd_rn(s.y, py[m]);
                bz[m] = __fadd_rn(s.z, pz[m]);
            }
            return s;
        };
        // columns of body i within r_circ + reach of j's centre s, 32 per word
        auto columns_near = [&](const float3 s, float reach, unsigned (&near)[kColWords]) {
            const float t = (reach + r_circ) * 1.0001f + 1e-3f;
#pragma unroll
            for (int wd = 0; wd < kColWords; ++wd) {
                near[wd] = 0u;
                if constexpr (C > 0) {
                    if (32 * wd < cols.n_cols)
                        near[wd] = __ballot_sync(0xffffffffu, column_near<C>(s, sc, cols, 32 * wd + lane, t * t));
                }
            }
        };
        auto close = [&](float rho) {  // some bead distance below contact (all beads)
            const float3 s = place(rho);
            if constexpr (C > 0) {
                unsigned near[kColWords];
                columns_near(s, contact, near);
                for (int wd = 0; wd < kColWords; ++wd)
                    while (near[wd]) {
                        const int c = 32 * wd + __ffs(near[wd]) - 1;
                        near[wd] &= near[wd] - 1u;
                        const float mn = column_min<NP, C>(sc.xy[c].x, sc.xy[c].y, cols, bx, by, bz);
                        if (__any_sync(0xffffffffu, mn < sig2)) return true;
                    }
                return false;
            } else {
                for (int k0 = 0; k0 < n_beads; k0 += 32) {
                    float mn = 3.0e38f;
                    for (int k = k0; k < min(k0 + 32, n_beads); ++k) {
                        const float4 d = sT[k];
#pragma unroll
                        for (int m = 0; m < MB; ++m)
                            mn = fminf(mn, bead_dist2(bx[m] - d.x, by[m] - d.y, bz[m] - d.z));
                    }
                    if (__any_sync(0xffffffffu, mn < sig2)) return true;
                }
                return false;
            }
        };
        // bead pairs closer than `reach` with j's centre at rho: their number
        // (some number above kCand if there are more), the first kCand of them in cand
        auto list_pairs = [&](float rho, float reach) {
            const float3 s = place(rho);
            const float r2 = reach * reach;
            int nc = 0;
            auto test = [&](int k, float x, float y, float zz) {
#pragma unroll
                for (int m = 0; m < MB; ++m) {
                    const bool hit = bead_dist2(bx[m] - x, by[m] - y, bz[m] - zz) < r2;
                    const unsigned w = __ballot_sync(0xffffffffu, hit);
                    if (w) {
                        const int at = nc + __popc(w & ((1u << lane) - 1u));
                        if (hit && at < kCand) cand[at] = (unsigned short)(k << 8 | (lane + 32 * m));
                        nc += __popc(w);
                    }
                }
            };
            if constexpr (C > 0) {
                unsigned near[kColWords];
                columns_near(s, reach, near);
                for (int wd = 0; wd < kColWords; ++wd)
                    while (near[wd]) {
                        const int c = 32 * wd + __ffs(near[wd]) - 1;
                        near[wd] &= near[wd] - 1u;
                        const float x = sc.xy[c].x, y = sc.xy[c].y;
                        const float mn = column_min<NP, C>(x, y, cols, bx, by, bz);
                        if (!__any_sync(0xffffffffu, mn < r2)) continue;
                        for (int k = 0; k < C; ++k) test(C * c + k, x, y, cols.z[k]);
                        if (nc > kCand) return nc;
                    }
            } else {
                for (int k = 0; k < n_beads; ++k) {
                    const float4 d = sT[k];
                    float mn = 3.0e38f;
#pragma unroll
                    for (int m = 0; m < MB; ++m) mn = fminf(mn, bead_dist2(bx[m] - d.x, by[m] - d.y, bz[m] - d.z));
                    if (!__any_sync(0xffffffffu, mn < r2)) continue;
                    test(k, d.x, d.y, d.z);
                    if (nc > kCand) return nc;
                }
            }
            __syncwarp();
            return nc;
        };
        float lo = 0.f, hi = Rc;
        int nc = kCand + 1;            // listed pairs (> kCand: none listed yet)
        float3 o0, o1, d0, d1;         // the lane's two listed pairs: R d_l and d_k
        o0 = o1 = make_float3(1e18f, 0.f, 0.f);
        d0 = d1 = make_float3(0.f, 0.f, 0.f);
        for (int it = 0; it < 40; ++it) {
            const float mid = 0.5f * (lo + hi);
            if ((lo > 0.f && mid <= lo) || (hi < Rc && mid >= hi)) break;  // an end tested before: settled
            if (nc > kCand && it >= kCoarse && ((it - kCoarse) & 1) == 0) {
                nc = list_pairs(mid, contact + 0.5f * (hi - lo) + slack);
                if (nc <= kCand) {
                    auto entry = [&](int e, float3& o, float3& d) {
                        if (e >= nc) return;
                        const int k = cand[e] >> 8, l = cand[e] & 0xFF;
                        o = rotate_bead(Rr, sT[l]);
                        d = xyz(sT[k]);
                    };
                    entry(lane, o0, d0);
                    entry(lane + 32, o1, d1);
                }
                __syncwarp();  // the list is read before it is written again
            }
            bool hit;
            if (nc <= kCand) {
                const float3 s = centre(mid);
                auto dist2 = [&](const float3& o, const float3& d) {
                    return bead_dist2(__fadd_rn(s.x, o.x) - d.x, __fadd_rn(s.y, o.y) - d.y, __fadd_rn(s.z, o.z) - d.z);
                };
                hit = __any_sync(0xffffffffu, fminf(dist2(o0, d0), dist2(o1, d1)) < sig2);
            } else {
                hit = close(mid);
            }
            if (hit)
                lo = mid;
            else
                hi = mid;
        }
        const float rc = 0.5f * (lo + hi);
        const float rho = rc + ub[5] * (Rc - rc);
        const float3 s = centre(rho);
        float v[7];
        if constexpr (C > 0) {
            place(rho);
            float2 Bx[NP], By[NP], Bz[NP];
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                Bx[p] = make_float2(bx[2 * p], bx[2 * p + 1]);
                By[p] = make_float2(by[2 * p], by[2 * p + 1]);
                Bz[p] = make_float2(bz[2 * p], bz[2 * p + 1]);
            }
            LJAcc<NP> acc;
            acc.zero();
#pragma unroll
            for (int wd = 0; wd < kColWords; ++wd) {
                if (32 * wd >= cols.n_cols) break;
                unsigned near = __ballot_sync(0xffffffffu, column_near<C>(s, sc, cols, 32 * wd + lane, pot.cull2));
                while (near) {
                    const int c = 32 * wd + __ffs(near) - 1;
                    near &= near - 1u;
                    const float x = sc.xy[c].x, y = sc.xy[c].y;
                    unsigned hits = __reduce_or_sync(0xffffffffu,
                                                     column_hits<NP, C>(x, y, cols, bx, by, bz, pot.rc2_test));
                    while (hits) {
                        const float mz = -2.f * sc.z[__ffs(hits) - 1];
                        hits &= hits - 1u;
                        bead_terms<NP, POT>(make_float2(-2.f * x, -2.f * x), make_float2(-2.f * y, -2.f * y),
                                            make_float2(mz, mz), Bx, By, Bz, pot, acc);
                    }
                }
            }
            warp_finish<NP>(bx, by, bz, acc, pot, v);
        } else {
            bead_pair_warp<NP, POT>(s, Rr, sT, sN, n_beads, pot, lane, v);
        }
        if (lane == 0) {
            cfg[2 * b] = make_float4(s.x, s.y, s.z, 0.f);
            cfg[2 * b + 1] = q;
            const float3 F = make_float3(v[0], v[1], v[2]);
            const float3 T = make_float3(v[3], v[4], v[5]);
            const float3 sxF = cross3(s, F);
            lab[3 * b] = make_float4(F.x, F.y, F.z, v[6]);
            lab[3 * b + 1] = make_float4(-T.x, -T.y, -T.z, 0.f);
            lab[3 * b + 2] = make_float4(T.x - sxF.x, T.y - sxF.y, T.z - sxF.z, 0.f);
            if (rho_c) rho_c[b] = rc;
        }
    }
}

// ------------------------------------------------------------- weight gradient
// One CTA computes a tile of S = 1024 CPT / W samples from the configurations
// to its share of every parameter's gradient; k_train_update sums the shares
// and applies Adam.  A thread owns CPT samples x 4 units of every layer;
// activations and signals live in shared memory as [unit][sample] (row stride
// S + 4: the weight-gradient loop reads rows of consecutive units, which then
// fall on different banks), weights stream through the cp.async ring of
// nn.cu.  phi'(z), phi''(z) terms and h_D are only needed by the thread that
// formed them: they go to a global scratch (coalesced per thread, L2-resident).
// Per tile: forward and plain reverse (energy, dE/dx, g_l), the residual and
// its tangent u per sample, tangent forward, one reverse stream (a_h), and for
// every layer dW += a_z h^T + g h_dot^T.  Samples past the batch have u = c = 0
// and so add zeros.
// What bounds it: FP32 FMA issue at about half rate (8 warps per SM).  A step
// of this pass was 45 launches (split-TF32 GEMMs of 4096 x 128 x 128, each bound
// by its load latency, and elementwise kernels between them); the GEMMs of one
// tile are too small to pay for splitting operands and moving tiles to tensor
// memory, and without the kernels between them there is no traffic to save.
// Measured, batch 4096 at width 128: step 375 -> 79 us (this kernel 65 us, the
// update 10 us), error of the gradient against FP64 2.5e-6 -> 1.8e-7; width 256:
// 606 -> 362 us, where the shares of the 256 x 256 gradients (0.5 MB a tile)
// weigh as much as the arithmetic.
constexpr int kTrSlotFloats = 4 * 256;  // x CPT: one quantity of one layer, all threads
__host__ __device__ inline int tr_slots(int D) { return 2 * D + 1; }  // phi', phi'' term per layer, h_D

// DG: h_dot_1 .. h_dot_{D-1} in the CTA's global scratch instead of shared memory
// (width 256 at depth 4, whose arrays for four samples a thread would not fit).
template <int W, int CPT, int KC, bool DG = false>
struct TrShape {
    static constexpr int S = 1024 * CPT / W;  // samples per tile
    static constexpr int LD = S + 4;
    static constexpr int NTP = S / CPT;       // thread groups along samples
    static constexpr int NG = 256 / NTP;      // along units
    static_assert(NG * 4 == W && NTP <= 32, "4 units per thread; a unit's samples within a warp");
    // floats of a CTA's scratch
    __host__ __device__ static size_t scratch(int D) {
        return (size_t)tr_slots(D) * kTrSlotFloats * CPT + (DG ? (size_t)(D - 1) * W * LD : 0);
    }
    static size_t smem(int D) {
        return sizeof(float) * ((size_t)(DG ? 2 * D : 3 * D - 1) * W * LD + 2 * (size_t)KC * W + 2 * (size_t)kInPad * LD +
                                (size_t)NG * S + 32 + (size_t)D * W + W + S);
    }
};

// What a sample's tangent comes from: labels (force matching) or a given (u, c).
struct TrArgs {
    int64_t n;
    const float4 *cfg, *lab, *ucfg;
    const float* c;
    float4* pred;
    float lam_tau, lam_E, inv_f2, inv_kTw, inv_n, sw_on, sw_inv;
};

// u (tangent in (s, q) space), c and the loss of one sample from its residuals.
__device__ inline double tr_residual(const TrArgs& A, int64_t b, float e_scale, float4& u0, float4& u1, float& c) {
    const float scale = e_scale * A.inv_n;  // dE/dE_hat over the batch mean
    const float4 c0 = A.cfg[2 * b], q = A.cfg[2 * b + 1];
    const float3 s = make_float3(c0.x, c0.y, c0.z);
    const float4 p0 = A.pred[3 * b], p1 = A.pred[3 * b + 1], p2 = A.pred[3 * b + 2];
    const float4 l0 = A.lab[3 * b], l1 = A.lab[3 * b + 1], l2 = A.lab[3 * b + 2];
    const float3 dF = make_float3(p0.x - l0.x, p0.y - l0.y, p0.z - l0.z);
    const float3 di = make_float3(p1.x - l1.x, p1.y - l1.y, p1.z - l1.z);
    const float3 dj = make_float3(p2.x - l2.x, p2.y - l2.y, p2.z - l2.z);
    const float dE = p0.w - l0.w;
    // per-sample weight 1 / (1 + |label|^2 / f_scale^2): relative error for
    // large forces, absolute for small ones (1 when inv_f2 = 0)
    const float mag2 = l0.x * l0.x + l0.y * l0.y + l0.z * l0.z +
                       A.lam_tau * (l1.x * l1.x + l1.y * l1.y + l1.z * l1.z + l2.x * l2.x + l2.y * l2.y +
                                    l2.z * l2.z);
    // Boltzmann importance weight min(1, exp(-E* / kT_w)) (1 when inv_kTw = 0)
    const float wgt = __expf(-fmaxf(l0.w, 0.f) * A.inv_kTw) / (1.f + mag2 * A.inv_f2);
    const double l = wgt * ((double)(dF.x * dF.x + dF.y * dF.y + dF.z * dF.z) +
                            A.lam_tau * (double)(di.x * di.x + di.y * di.y + di.z * di.z + dj.x * dj.x +
                                                 dj.y * dj.y + dj.z * dj.z) +
                            A.lam_E * (double)dE * dE);
    // dl/dF = 2 w dF, dl/dtau_i = 2 w lam di, dl/dtau_j = 2 w lam dj
    const float a2 = 2.f * wgt, b2 = 2.f * wgt * A.lam_tau;
    const float3 rF = make_float3(a2 * dF.x, a2 * dF.y, a2 * dF.z);
    const float3 ri = make_float3(b2 * di.x, b2 * di.y, b2 * di.z);
    const float3 rj = make_float3(b2 * dj.x, b2 * dj.y, b2 * dj.z);
    // F_j = -G_s, tau_i = s x G_s - tau_j, tau_j = -1/2 (-G_w v + w G_v + v x G_v)
    const float3 rixs = cross3(ri, s);
    const float3 us = make_float3(-rF.x + rixs.x, -rF.y + rixs.y, -rF.z + rixs.z);
    const float3 rv = make_float3(rj.x - ri.x, rj.y - ri.y, rj.z - ri.z);
    const float w = q.x;
    const float3 v = make_float3(q.y, q.z, q.w);
    const float uw = 0.5f * (rv.x * v.x + rv.y * v.y + rv.z * v.z);
    const float3 rvxv = cross3(rv, v);
    const float3 uv = make_float3(-0.5f * (w * rv.x + rvxv.x), -0.5f * (w * rv.y + rvxv.y),
                                  -0.5f * (w * rv.z + rvxv.z));
    u0 = make_float4(scale * us.x, scale * us.y, scale * us.z, 0.f);
    u1 = make_float4(scale * uw, scale * uv.x, scale * uv.y, scale * uv.z);
    c = scale * 2.f * wgt * A.lam_E * dE;
    return l;
}

// Tangent of the 10 (or the paper's six) features along (u0, u1), which are
// given for the configuration as passed.  With the smooth cutoff the output is
// S(rho) E_hat: d/dW [u . grad(S E_hat) + c S E_hat] = d/dW [u' . grad E_hat +
// c' E_hat] with u' = S u and c' = S c + S' (u_s . s / rho).  With a point group
// the tangent is mapped with the configuration: u_s' = sg R(Q_k) u_s,
// u_q' = Q_k u_q Q_j.  desc = 1: the tangent follows from the rotation
// delta theta = 2 vec(delta q (x) q^*) of cube 2 (paper6_geometry).
__device__ inline void tr_tangent(const TrArgs& A, const PairGeom& g, const float4& c0, float4 u0, float4 u1,
                                  float& c, float (&xd)[kIn]) {
    if (A.sw_inv > 0.f) {
        const float rho = sqrtf(c0.x * c0.x + c0.y * c0.y + c0.z * c0.z);
        float S, dS;
        cutoff_switch(rho, A.sw_on, A.sw_inv, S, dS);
        c = S * c + dS * (u0.x * c0.x + u0.y * c0.y + u0.z * c0.z) / rho;
        u0 = make_float4(S * u0.x, S * u0.y, S * u0.z, 0.f);
        u1 = make_float4(S * u1.x, S * u1.y, S * u1.z, S * u1.w);
    }
    if (g.sym) {
        const float3 r = mul(qmat(g.sym_qk), make_float3(u0.x, u0.y, u0.z));
        u0 = make_float4(g.sym_sg * r.x, g.sym_sg * r.y, g.sym_sg * r.z, 0.f);
        u1 = qmul(qmul(g.sym_qk, u1), g.sym_qj);
    }
    const float rd = (g.s.x * u0.x + g.s.y * u0.y + g.s.z * u0.z) / g.rho;
    xd[0] = u0.x;
    xd[1] = u0.y;
    xd[2] = u0.z;
    xd[3] = g.sgn * u1.x;
    xd[4] = g.sgn * u1.y;
    xd[5] = g.sgn * u1.z;
    xd[6] = g.sgn * u1.w;
    xd[7] = rd;
    xd[8] = -rd / (g.rho * g.rho);
    xd[9] = 2.f * g.rho * rd;
    if (g.paper6) {
        const Paper6 P = paper6_geometry(g.s, g.qc);
        const float4 t = qmul(make_float4(xd[3], xd[4], xd[5], xd[6]), qconj(g.qc));
        const float3 th = make_float3(2.f * t.y, 2.f * t.z, 2.f * t.w);
        const float e1t = P.e1.x * th.x + P.e1.y * th.y + P.e1.z * th.z;
        xd[3] = P.e2.y * th.y + P.e2.z * th.z;
        xd[4] = -e1t * P.inv_sin;
        xd[5] = P.w.x * th.x + P.w.y * th.y + P.w.z * th.z + P.cot * e1t;
        xd[6] = xd[7] = xd[8] = xd[9] = 0.f;
    }
}

// acc[i][j / 2].(x, y) = sum_k A[k][p0 + i] B[k][o0 + j]: A in shared memory
// [K][LD], B the next K / KC weight chunks.
template <int W, int CPT, int KC>
__device__ __forceinline__ void tr_gemm(const float* __restrict__ As, int K, ChunkFeed<W, KC>& feed, int p0,
                                        int o0, float2 (&acc)[CPT][2]) {
    constexpr int LD = TrShape<W, CPT, KC>::LD;
#pragma unroll
    for (int i = 0; i < CPT; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
    for (int kc = 0; kc < K; kc += KC) {
        const float* Bs = feed.acquire();
        const int kn = min(KC, K - kc);
#pragma unroll 16
        for (int k = 0; k < kn; ++k) {
            const TrVec<CPT> a = tr_ld<CPT>(As + (size_t)(kc + k) * LD + p0);
            const float4 b = *reinterpret_cast<const float4*>(Bs + (size_t)k * W + o0);
            const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
#pragma unroll
            for (int i = 0; i < CPT; ++i) {
                const float2 aa = make_float2(a.v[i], a.v[i]);
                acc[i][0] = __ffma2_rn(aa, b0, acc[i][0]);
                acc[i][1] = __ffma2_rn(aa, b1, acc[i][1]);
            }
        }
        feed.release();
    }
}
// out[o * W + i] (+)= sum_c A1[o][c] B1[i][c] + A2[o][c] B2[i][c] over the
// tile's samples: a warp per 8 units o, lanes on consecutive i; FP32x2 over
// pairs of samples.
template <int W, int S, int LD>
__device__ __forceinline__ void tr_weight_grad(const float* __restrict__ A1, const float* __restrict__ B1,
                                               const float* __restrict__ A2, const float* __restrict__ B2,
                                               float* __restrict__ out, bool first) {
    constexpr int JN = W / 32 < 4 ? W / 32 : 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o0 = 8 * warp; o0 < W; o0 += 64)
        for (int i0 = 0; i0 < W; i0 += 32 * JN) {
            float2 acc[8][JN];
#pragma unroll
            for (int o = 0; o < 8; ++o)
#pragma unroll
                for (int j = 0; j < JN; ++j) acc[o][j] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int t = 0; t < 2; ++t) {
                const float* A = t == 0 ? A1 : A2;
                const float* B = t == 0 ? B1 : B2;
#pragma unroll 2
                for (int c = 0; c < S; c += 4) {
                    float4 b[JN];
#pragma unroll
                    for (int j = 0; j < JN; ++j)
                        b[j] = *reinterpret_cast<const float4*>(B + (size_t)(i0 + lane + 32 * j) * LD + c);
#pragma unroll
                    for (int o = 0; o < 8; ++o) {
                        const float4 a = *reinterpret_cast<const float4*>(A + (size_t)(o0 + o) * LD + c);
#pragma unroll
                        for (int j = 0; j < JN; ++j) {
                            acc[o][j] = __ffma2_rn(make_float2(a.x, a.y), make_float2(b[j].x, b[j].y), acc[o][j]);
                            acc[o][j] = __ffma2_rn(make_float2(a.z, a.w), make_float2(b[j].z, b[j].w), acc[o][j]);
                        }
                    }
                }
            }
#pragma unroll
            for (int o = 0; o < 8; ++o)
#pragma unroll
                for (int j = 0; j < JN; ++j) {
                    float* p = out + (size_t)(o0 + o) * W + i0 + lane + 32 * j;
                    const float v = acc[o][j].x + acc[o][j].y;
                    *p = first ? v : *p + v;
                }
        }
}

template <int W, int CPT, int KC, bool DG>
__global__ void __launch_bounds__(256, 1)
    k_train_tile(const float* __restrict__ flat, const float* __restrict__ prep, FlatLayout fl, F32Layout pl,
                 int D, PairSrc src, TrArgs A, float* __restrict__ part, int64_t np,
                 float* __restrict__ scratch, double* __restrict__ loss_part) {
    using Sh = TrShape<W, CPT, KC, DG>;
    constexpr int S = Sh::S, LD = Sh::LD, NTP = Sh::NTP, NG = Sh::NG;
    constexpr int NS = 256 / S < W / 16 ? 256 / S : W / 16;  // unit slices of the dE/dx reduction
    static_assert(NS * kIn * S <= W * LD, "dE/dx partial sums fit in one array");
    pdl_wait();
    extern __shared__ float4 smem4[];
    float* Hs = reinterpret_cast<float*>(smem4);   // h_1 .. h_{D-1}
    float* own = scratch + (size_t)blockIdx.x * Sh::scratch(D);
    float* Ds = DG ? own + (size_t)tr_slots(D) * kTrSlotFloats * CPT  // h_dot_1 .. h_dot_{D-1}
                   : Hs + (size_t)(D - 1) * W * LD;
    float* Gs = Hs + (size_t)(DG ? 1 : 2) * (D - 1) * W * LD;  // g_1 .. g_D, then a_z_{l-1} in the place of g_l
    float* Zs = Gs + (size_t)D * W * LD;           // dE/dx partial sums, then a_z_D
    float* Bs = Zs + (size_t)W * LD;               // 2 x [KC][W] weight chunks
    float* Xs = Bs + (size_t)2 * KC * W;           // [16][LD] normalised features
    float* Us = Xs + (size_t)kInPad * LD;          // [16][LD] their tangent
    float* Red = Us + (size_t)kInPad * LD;         // [NG][S] energy partial sums
    float* mu = Red + (size_t)NG * S;              // 16
    float* isd = mu + 16;                          // 16
    float* bias = isd + 16;                        // D x W
    float* wo = bias + (size_t)D * W;              // W
    float* cs = wo + W;                            // S
    const int tid = threadIdx.x, tp = tid % NTP, to = tid / NTP;
    const int p0 = tp * CPT, o0 = to * 4;
    float* mine = own + (size_t)tid * CPT;
    auto slot = [&](int k, int j) { return mine + ((size_t)k * 4 + j) * 256 * CPT; };  // unit j of the thread
    float* gp = part + (size_t)blockIdx.x * np;

    for (int t = tid; t < 16; t += 256) {
        mu[t] = t < kIn ? flat[fl.mu + t] : 0.f;
        isd[t] = t < kIn ? flat[fl.inv_sd + t] : 0.f;
    }
    for (int t = tid; t < D * W; t += 256) bias[t] = flat[fl.b_(1 + t / W, W) + t % W];
    for (int t = tid; t < W; t += 256) wo[t] = flat[fl.wo + t];
    const float b_o = flat[fl.bo], e_scale = flat[fl.escale], e_shift = flat[fl.eshift];
    const int64_t n_tiles = (A.n + S - 1) / S;
    ChunkFeed<W, KC> feed;
    feed.prep = prep;
    feed.pl = pl;
    feed.D = D;
    feed.n_chunks = 1 + 2 * (D - 1) * ChunkFeed<W, KC>::NK;
    feed.c = 0;
    feed.total = ((n_tiles - 1 - blockIdx.x) / gridDim.x + 1) * 2 * feed.n_chunks;  // two passes per tile
    feed.buf = Bs;
    feed.issue(0);
    __syncthreads();

    double loss = 0.0;
    float bo_sum = 0.f;  // this sample thread's c
    bool first = true;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, first = false) {
        const int64_t b = tile * S + tid;
        const bool sample = tid < S, valid = sample && b < A.n;
        PairGeom geo;
        if (sample) {
            geo = load_pair<false>(src, b, valid);
            float x[kIn];
            raw_features(geo, x);
#pragma unroll
            for (int k = 0; k < kInPad; ++k) Xs[k * LD + tid] = k < kIn ? (x[k] - mu[k]) * isd[k] : 0.f;
        }
        float2 acc[CPT][2];
        // ---- forward: h_l, phi'(z_l), phi''(z_l); at the top g_D = w_o phi', w_o phi''
        for (int l = 1; l <= D; ++l) {
            tr_gemm<W, CPT, KC>(l == 1 ? Xs : Hs + (size_t)(l - 2) * W * LD, l == 1 ? kInPad : W, feed, p0, o0, acc);
            TrVec<CPT> e;
#pragma unroll
            for (int i = 0; i < CPT; ++i) e.v[i] = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float bj = bias[(l - 1) * W + o0 + j], w = wo[o0 + j];
                TrVec<CPT> h, d1, d2;
#pragma unroll
                for (int i = 0; i < CPT; ++i) {
                    const float z = tr_at<CPT>(acc, i, j) + bj;
                    const float sg = 1.f / (1.f + __expf(-z));
                    h.v[i] = z * sg;
                    d1.v[i] = sg * (1.f + z * (1.f - sg));
                    d2.v[i] = sg * (1.f - sg) * (2.f + z * (1.f - 2.f * sg));
                    e.v[i] = fmaf(w, h.v[i], e.v[i]);
                }
                tr_st<CPT>(slot(l - 1, j), d1);
                if (l < D) {
                    tr_st<CPT>(slot(D + l - 1, j), d2);
                    tr_st<CPT>(Hs + (size_t)(l - 1) * W * LD + (size_t)(o0 + j) * LD + p0, h);
                } else {
                    tr_st<CPT>(slot(2 * D, j), h);
#pragma unroll
                    for (int i = 0; i < CPT; ++i) {
                        d1.v[i] *= w;
                        d2.v[i] *= w;
                    }
                    tr_st<CPT>(slot(2 * D - 1, j), d2);
                    tr_st<CPT>(Gs + (size_t)(D - 1) * W * LD + (size_t)(o0 + j) * LD + p0, d1);
                }
            }
            if (l == D) tr_st<CPT>(Red + (size_t)to * S + p0, e);
        }
        // ---- plain reverse: g_{l-1} = (W_l^T g_l) phi', and (W_l^T g_l) phi''
        for (int l = D; l >= 2; --l) {
            tr_gemm<W, CPT, KC>(Gs + (size_t)(l - 1) * W * LD, W, feed, p0, o0, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                TrVec<CPT> d1 = tr_ld<CPT>(slot(l - 2, j)), d2 = tr_ld<CPT>(slot(D + l - 2, j));
#pragma unroll
                for (int i = 0; i < CPT; ++i) {
                    const float a = tr_at<CPT>(acc, i, j);
                    d1.v[i] *= a;
                    d2.v[i] *= a;
                }
                tr_st<CPT>(slot(D + l - 2, j), d2);
                tr_st<CPT>(Gs + (size_t)(l - 2) * W * LD + (size_t)(o0 + j) * LD + p0, d1);
            }
        }
        __syncthreads();
        // ---- dE/dx_hat = W_1^T g_1 in unit slices; outputs, residual, tangent
        if (A.lab) {
            const int pp = tid % S, ks = tid / S;
            constexpr int SL = W / NS;
            const float4* W1p = reinterpret_cast<const float4*>(prep + pl.w1p);
            float g[kIn];
#pragma unroll
            for (int k = 0; k < kIn; ++k) g[k] = 0.f;
#pragma unroll 4
            for (int o = ks * SL; o < (ks < NS ? ks + 1 : ks) * SL; ++o) {
                const float gv = Gs[(size_t)o * LD + pp];
                const float4 w0 = W1p[4 * o], w1 = W1p[4 * o + 1], w2 = W1p[4 * o + 2];
                g[0] = fmaf(gv, w0.x, g[0]);
                g[1] = fmaf(gv, w0.y, g[1]);
                g[2] = fmaf(gv, w0.z, g[2]);
                g[3] = fmaf(gv, w0.w, g[3]);
                g[4] = fmaf(gv, w1.x, g[4]);
                g[5] = fmaf(gv, w1.y, g[5]);
                g[6] = fmaf(gv, w1.z, g[6]);
                g[7] = fmaf(gv, w1.w, g[7]);
                g[8] = fmaf(gv, w2.x, g[8]);
                g[9] = fmaf(gv, w2.y, g[9]);
            }
#pragma unroll
            for (int k = 0; k < kIn; ++k)
                if (ks < NS) Zs[(size_t)(ks * kIn + k) * S + pp] = g[k];
            __syncthreads();
        }
        if (sample) {
            float xd[kIn], c = 0.f;
#pragma unroll
            for (int k = 0; k < kIn; ++k) xd[k] = 0.f;
            if (valid) {
                float4 u0, u1;
                if (A.lab) {
                    float e = 0.f;
                    for (int g = 0; g < NG; ++g) e += Red[(size_t)g * S + tid];
                    float gx[kIn];
#pragma unroll
                    for (int k = 0; k < kIn; ++k) {
                        float a = 0.f;
                        for (int q = 0; q < NS; ++q) a += Zs[(size_t)(q * kIn + k) * S + tid];
                        gx[k] = e_scale * a * isd[k];
                    }
                    PairDst dst{};
                    dst.sw_on = A.sw_on;
                    dst.sw_inv = A.sw_inv;
                    dst.out = A.pred;
                    write_pair_outputs<false>(dst, b, geo, gx, e_scale * (e + b_o) + e_shift);
                    loss += tr_residual(A, b, e_scale, u0, u1, c);
                } else {
                    u0 = A.ucfg[2 * b];
                    u1 = A.ucfg[2 * b + 1];
                    c = A.c[b];
                }
                tr_tangent(A, geo, A.cfg[2 * b], u0, u1, c, xd);
            }
#pragma unroll
            for (int k = 0; k < kInPad; ++k) Us[k * LD + tid] = k < kIn ? xd[k] * isd[k] : 0.f;
            cs[tid] = c;
            bo_sum += c;
        }
        // ---- tangent forward: h_dot_l = phi' z_dot, (phi'' terms) z_dot; at the
        // top the gradient of w_o and a_z_D = c g_D + (phi'' terms) z_dot
        for (int l = 1; l <= D; ++l) {
            tr_gemm<W, CPT, KC>(l == 1 ? Us : Ds + (size_t)(l - 2) * W * LD, l == 1 ? kInPad : W, feed, p0, o0, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                TrVec<CPT> d1 = tr_ld<CPT>(slot(l - 1, j)), d2 = tr_ld<CPT>(slot(D + l - 1, j));
#pragma unroll
                for (int i = 0; i < CPT; ++i) {
                    const float zd = tr_at<CPT>(acc, i, j);
                    d1.v[i] *= zd;
                    d2.v[i] *= zd;
                }
                const size_t at = (size_t)(o0 + j) * LD + p0;
                if (l < D) {
                    tr_st<CPT>(slot(D + l - 1, j), d2);
                    tr_st<CPT>(Ds + (size_t)(l - 1) * W * LD + at, d1);
                } else {
                    const TrVec<CPT> h = tr_ld<CPT>(slot(2 * D, j)), g = tr_ld<CPT>(Gs + (size_t)(D - 1) * W * LD + at);
                    float sum = 0.f;
#pragma unroll
                    for (int i = 0; i < CPT; ++i) {
                        const float c = cs[p0 + i];
                        sum += fmaf(c, h.v[i], d1.v[i]);
                        d2.v[i] = fmaf(c, g.v[i], d2.v[i]);
                    }
                    tr_st<CPT>(Zs + at, d2);
#pragma unroll
                    for (int o = 1; o < NTP; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                    if (tp == 0) {
                        float* q = gp + fl.wo + o0 + j;
                        *q = first ? sum : *q + sum;
                    }
                }
            }
        }
        // ---- reverse: dW_l, db_l, then a_z_{l-1} = (W_l^T a_z_l) phi' + (phi'' terms) z_dot
        float* az = Zs;
        for (int l = D; l >= 1; --l) {
            __syncthreads();
            const float* g = Gs + (size_t)(l - 1) * W * LD;
            for (int o = tid; o < W; o += 256) {
                float a = 0.f;
                for (int c = 0; c < S; ++c) a += az[(size_t)o * LD + c];
                float* q = gp + fl.b_(l, W) + o;
                *q = first ? a : *q + a;
            }
            if (l == 1) {
                for (int t = tid; t < W * 16; t += 256) {
                    const int o = t >> 4, k = t & 15;
                    if (k >= kIn) continue;
                    float a = 0.f;
                    for (int c = 0; c < S; ++c)
                        a += az[(size_t)o * LD + c] * Xs[k * LD + c] + g[(size_t)o * LD + c] * Us[k * LD + c];
                    float* q = gp + fl.W1 + o * kIn + k;
                    *q = first ? a : *q + a;
                }
                break;
            }
            tr_weight_grad<W, S, LD>(az, Hs + (size_t)(l - 2) * W * LD, g, Ds + (size_t)(l - 2) * W * LD,
                                     gp + fl.W_(l, W), first);
            tr_gemm<W, CPT, KC>(az, W, feed, p0, o0, acc);
            float* nz = Gs + (size_t)(l - 1) * W * LD;  // g_l has been used
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                TrVec<CPT> d1 = tr_ld<CPT>(slot(l - 2, j));
                const TrVec<CPT> d2 = tr_ld<CPT>(slot(D + l - 2, j));
#pragma unroll
                for (int i = 0; i < CPT; ++i) d1.v[i] = fmaf(tr_at<CPT>(acc, i, j), d1.v[i], d2.v[i]);
                tr_st<CPT>(nz + (size_t)(o0 + j) * LD + p0, d1);
            }
            az = nz;
        }
        __syncthreads();  // the next tile overwrites what this one read
    }
    // the sample threads' sums, in order (Red and the arrays are free)
    double* sl = reinterpret_cast<double*>(smem4);
    float* sb = reinterpret_cast<float*>(sl + 256);
    if (tid < S) {
        sl[tid] = loss;
        sb[tid] = bo_sum;
    }
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        float f = 0.f;
        for (int k = 0; k < S; ++k) {
            a += sl[k];
            f += sb[k];
        }
        loss_part[blockIdx.x] = a;
        gp[fl.bo] = f;
    }
}

// Sum of the CTAs' gradient shares (in order), Adam on the trainable parameters
// when `step`, and the updated weights' prepared FP32 copies.  Block 0 also
// sums the loss.
struct AdamArgs {
    float *p, *m, *v, *prep;
    float lr, b1, b2, eps, c1, c2;
};
__global__ void __launch_bounds__(256)
    k_train_update(int64_t np, int W, int D, int n_part, const float* __restrict__ part,
                   float* __restrict__ grad, bool step, AdamArgs a, const double* __restrict__ loss_part,
                   double inv_n, double* __restrict__ loss_out) {
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double x = 0.0;
        for (int k = threadIdx.x; k < n_part; k += 32) x += loss_part[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (threadIdx.x == 0) *loss_out = x * inv_n;
    }
    // 64 parameters per block, four threads each: a quarter of the shares, in
    // order, then the quarters in order
    __shared__ float s_q[4][64];
    const int lane = threadIdx.x & 63, q = threadIdx.x >> 6;
    const int64_t t = blockIdx.x * (int64_t)64 + lane;
    const FlatLayout f = flat_layout(W, D);
    const bool train = t >= f.W1 && t < f.escale;
    float g = 0.f;
    if (train) {
        const int per = (n_part + 3) / 4, e = min(n_part, (q + 1) * per);
        int k = q * per;
        for (; k + 16 <= e; k += 16) {
            float v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = part[(size_t)(k + u) * np + t];
#pragma unroll
            for (int u = 0; u < 16; ++u) g += v[u];
        }
        for (; k < e; ++k) g += part[(size_t)k * np + t];
    }
    s_q[q][lane] = g;
    __syncthreads();
    if (q > 0 || t >= np) return;
    g = ((s_q[0][lane] + s_q[1][lane]) + s_q[2][lane]) + s_q[3][lane];
    grad[t] = g;
    if (!step || !train) return;
    const float p = adam_update(a.p[t], g, a.m[t], a.v[t], a.lr, a.b1, a.b2, a.eps, a.c1, a.c2);
    a.p[t] = p;
    const F32Layout L = f32_layout(W, D);
    if (t < f.b1) {
        const int e = (int)(t - f.W1), o = e / kIn, k = e % kIn;
        a.prep[L.wt1 + (int64_t)k * W + o] = p;
        a.prep[L.w1p + (int64_t)o * kInPad + k] = p;
    } else if (t >= f.Wl && t < f.wo) {
        const int64_t r = t - f.Wl, wl = (int64_t)W * W + W;
        const int l = (int)(r / wl);  // layer l + 2
        const int64_t e = r % wl;
        if (e < (int64_t)W * W) {
            const int64_t o = e / W, k = e % W;
            a.prep[L.wt + (int64_t)l * W * W + k * W + o] = p;
            a.prep[L.wr + (int64_t)l * W * W + e] = p;
        }
    }
}

static inline unsigned nblk(int64_t n, int t) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

// Tiles of 4 samples per thread; 2 where a batch would leave half of the SMs
// without a tile (a step of width 128: 59.6 against 73.9 us for 1000 samples,
// 63.7 against 75.9 us for 2048; from 3000 on both forms fill the GPU), and at
// depth 4 below width 256, whose arrays would not fit.  At width 256 the gradient
// shares of a tile (0.8 MB at depth 4) are most of its traffic, so there h_dot
// leaves shared memory instead: a gradient of 4096 samples 1020 -> 668 us, of 65536
// 14.1 -> 8.9 ms (as separate GEMMs 858 us and 8.3 ms).
static int tr_cols(const rb_trainer* t, int64_t B) {
    const int W = t->mlp->width;
    return (t->mlp->depth > 3 && W < 256) || B * W <= (int64_t)4096 * (t->sms / 2) ? 2 : 4;
}
static int tr_grid(const rb_trainer* t, int64_t B, int cols) {
    const int64_t S = 1024 * cols / t->mlp->width;
    return (int)std::min<int64_t>((B + S - 1) / S, t->sms);
}

template <int W, int CPT, int KC, bool DG = false>
static rb_status launch_tile(rb_trainer* t, int grid, const PairSrc& src, const TrArgs& A) {
    rb_mlp* m = t->mlp;
    const size_t smem = TrShape<W, CPT, KC, DG>::smem(m->depth);
    static std::atomic<size_t> allowed{0};
    if (smem > allowed.load()) {
        RB_CUDA(cudaFuncSetAttribute(k_train_tile<W, CPT, KC, DG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     227 * 1024));
        allowed.store(227 * 1024);
    }
    RB_CUDA(launch_pdl(k_train_tile<W, CPT, KC, DG>, grid, 256, smem, m->stream, m->params, m->f32_prep,
                       flat_layout(W, m->depth), f32_layout(W, m->depth), m->depth, src, A, t->part,
                       m->n_params, t->scratch, t->loss_part));
    return RB_OK;
}

// The gradient of a batch into `grad` (and the parameters' Adam step).
static rb_status train_pass(rb_trainer* t, TrArgs A, float* grad, bool step) {
    rb_mlp* m = t->mlp;
    PairSrc src{};
    set_symmetry(src, m);
    src.cfg = A.cfg;
    src.n_explicit = A.n;
    A.pred = reinterpret_cast<float4*>(t->pred);
    A.sw_on = m->sw_on;
    A.sw_inv = m->sw_off > m->sw_on ? 1.f / (m->sw_off - m->sw_on) : 0.f;
    A.inv_n = 1.f / (float)A.n;
    const int cols = tr_cols(t, A.n), grid = tr_grid(t, A.n, cols);
    switch (m->width * 8 + cols) {
        case 64 * 8 + 4: RB_TRY((launch_tile<64, 4, 64>(t, grid, src, A))); break;
        case 64 * 8 + 2: RB_TRY((launch_tile<64, 2, 64>(t, grid, src, A))); break;
        case 128 * 8 + 4: RB_TRY((launch_tile<128, 4, 64>(t, grid, src, A))); break;
        case 128 * 8 + 2: RB_TRY((launch_tile<128, 2, 32>(t, grid, src, A))); break;
        case 256 * 8 + 4:
            if (m->depth > 3)
                RB_TRY((launch_tile<256, 4, 16, true>(t, grid, src, A)));
            else
                RB_TRY((launch_tile<256, 4, 16>(t, grid, src, A)));
            break;
        case 256 * 8 + 2: RB_TRY((launch_tile<256, 2, 16>(t, grid, src, A))); break;
        default: return fail(RB_ENOTSUP, "training supports widths 64, 128, 256");
    }
    AdamArgs a{m->params, t->m, t->v, m->f32_prep, t->lr, t->beta1, t->beta2, t->eps, 1.f, 1.f};
    if (step) {
        t->t += 1;
        // Bias corrections 1 - beta^t in FP64: in FP32, 1 - beta2^t loses about
        // five digits to cancellation (beta2^t is within 1e-3 of 1 early on).
        a.c1 = (float)(1.0 - std::pow((double)t->beta1, (double)t->t));
        a.c2 = (float)(1.0 - std::pow((double)t->beta2, (double)t->t));
    }
    RB_CUDA(launch_pdl(k_train_update, nblk(m->n_params, 64), 256, 0, m->stream, m->n_params, m->width, m->depth,
                       grid, t->part, grad, step, a, t->loss_part, 1.0 / (double)A.n, t->loss_out));
    if (step) m->version++;  // the BF16 / F16X3 images follow on their next use (ensure_images)
    return RB_OK;
}

static rb_status train_batch(rb_trainer* t, int64_t B, const float* cfg, const float* labels, float lam_tau,
                             float lam_E, float f_scale, float kT_w, bool step, double* loss_host) {
    RB_TRY(check_mlp(t->mlp));
    TrArgs A{};
    A.n = B;
    A.cfg = reinterpret_cast<const float4*>(cfg);
    A.lab = reinterpret_cast<const float4*>(labels);
    A.lam_tau = lam_tau;
    A.lam_E = lam_E;
    A.inv_f2 = f_scale > 0.f ? 1.f / (f_scale * f_scale) : 0.f;
    A.inv_kTw = kT_w > 0.f ? 1.f / kT_w : 0.f;
    RB_TRY(train_pass(t, A, t->grad, step));
    if (loss_host) {
        RB_CUDA(cudaMemcpyAsync(loss_host, t->loss_out, sizeof(double), cudaMemcpyDeviceToHost, t->mlp->stream));
        RB_CUDA(cudaStreamSynchronize(t->mlp->stream));
    }
    return RB_OK;
}

// The same pairs with the other body as the reference, in place: cfg
// (s, 0 | q) -> (R(q)^T (-s), 0 | q^*), labels (F, E | tau_i | tau_j) ->
// (R(q)^T (-F), E | R(q)^T tau_j | R(q)^T tau_i).
__global__ void k_swap_reference(int64_t n, float4* __restrict__ cfg, float4* __restrict__ lab) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const float4 s = cfg[2 * p], q = cfg[2 * p + 1];
        const Mat3 R = qmat(q);
        const float3 s2 = mulT(R, make_float3(-s.x, -s.y, -s.z));
        cfg[2 * p] = make_float4(s2.x, s2.y, s2.z, 0.f);
        cfg[2 * p + 1] = make_float4(q.x, -q.y, -q.z, -q.w);
        if (lab) {
            const float4 F = lab[3 * p], ti = lab[3 * p + 1], tj = lab[3 * p + 2];
            const float3 F2 = mulT(R, make_float3(-F.x, -F.y, -F.z));
            const float3 a = mulT(R, make_float3(tj.x, tj.y, tj.z));
            const float3 b = mulT(R, make_float3(ti.x, ti.y, ti.z));
            lab[3 * p] = make_float4(F2.x, F2.y, F2.z, F.w);
            lab[3 * p + 1] = make_float4(a.x, a.y, a.z, 0.f);
            lab[3 * p + 2] = make_float4(b.x, b.y, b.z, 0.f);
        }
    }
}

}  // namespace rb

using namespace rb;

extern "C" {

rb_status rb_pairs_swap_reference(int64_t n, float* cfg, float* labels, void* stream) {
    if (n < 0 || (n > 0 && !cfg)) return fail(RB_EINVAL, "bad pair arrays");
    if (n == 0) return RB_OK;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8);
    k_swap_reference<<<grid, 256, 0, (cudaStream_t)stream>>>(n, reinterpret_cast<float4*>(cfg),
                                                            reinterpret_cast<float4*>(labels));
    RB_CUDA(cudaGetLastError());
    return RB_OK;
}

rb_status rb_sample_pairs(const rb_system* s, int64_t n, const float* uniforms, float* cfg,
                          float* labels, float* rho_contact) {
    if (!s) return fail(RB_EINVAL, "null system");
    return rb_sample_pairs_at(s, n, uniforms, s->sigma, cfg, labels, rho_contact);
}

rb_status rb_sample_pairs_at(const rb_system* s, int64_t n, const float* uniforms, float contact,
                             float* cfg, float* labels, float* rho_contact) {
    if (!s) return fail(RB_EINVAL, "null system");
    if (!(contact > 0.f)) return fail(RB_EINVAL, "contact distance must be positive");
    if (n < 0 || (n > 0 && (!uniforms || !cfg || !labels))) return fail(RB_EINVAL, "bad arrays");
    if (n == 0) return RB_OK;
    const int np = (s->n_beads + 63) / 64;
    BeadPot pot = bead_pot(s);
    const int grid = (int)std::min<int64_t>((n + 7) / 8, (int64_t)s->num_sms * 4);  // a warp per sample
#define RB_SAMPLE(NP, C, POT)                                                                \
    k_sample_pairs<NP, C, POT><<<grid, 256, 0, s->stream>>>(                                 \
        n, uniforms, s->tmpl_dev, s->n_beads, s->cols, s->r_circ, s->Rc, contact, pot,       \
        reinterpret_cast<float4*>(cfg), reinterpret_cast<float4*>(labels), rho_contact)
#define RB_SAMPLE_C(NP, POT)                                                                 \
    do {                                                                                     \
        if (s->cols.len == 5) RB_SAMPLE(NP, 5, POT);                                         \
        else if (s->cols.len == 8) RB_SAMPLE(NP, 8, POT);                                    \
        else RB_SAMPLE(NP, 0, POT);                                                          \
    } while (0)
    const bool lj = s->pot_kind == RB_POT_LJ;
    if (np <= 2) {
        if (lj) RB_SAMPLE_C(2, 0); else RB_SAMPLE_C(2, 1);
    } else if (np <= 3) {
        if (lj) RB_SAMPLE_C(3, 0); else RB_SAMPLE_C(3, 1);
    } else {
        if (lj) RB_SAMPLE_C(4, 0); else RB_SAMPLE_C(4, 1);
    }
#undef RB_SAMPLE_C
#undef RB_SAMPLE
    RB_CUDA(cudaGetLastError());
    return RB_OK;
}

rb_status rb_trainer_create(rb_mlp* mlp, int64_t max_batch, float lr, float beta1, float beta2,
                            float eps, rb_trainer** out) {
    if (!mlp || !out) return fail(RB_EINVAL, "null argument");
    *out = nullptr;
    if (max_batch < 1 || max_batch > (1 << 22)) return fail(RB_EINVAL, "max_batch out of range");
    rb_trainer* t = new (std::nothrow) rb_trainer();
    if (!t) return fail(RB_ENOMEM, "host allocation");
    t->mlp = mlp;
    t->max_batch = max_batch;
    t->lr = lr;
    t->beta1 = beta1;
    t->beta2 = beta2;
    t->eps = eps;
    const int64_t np = mlp->n_params;
    cudaDeviceGetAttribute(&t->sms, cudaDevAttrMultiProcessorCount, mlp->device);
    // the most CTAs a batch of up to max_batch takes, in either tile form
    const size_t ctas = std::max(tr_grid(t, max_batch, 2), tr_grid(t, max_batch, 4));
    cudaError_t e = cudaMalloc(&t->m, sizeof(float) * np);
    if (e == cudaSuccess) e = cudaMalloc(&t->v, sizeof(float) * np);
    if (e == cudaSuccess) e = cudaMalloc(&t->grad, sizeof(float) * np);
    if (e == cudaSuccess) e = cudaMalloc(&t->pred, sizeof(float4) * 3 * max_batch);
    if (e == cudaSuccess) e = cudaMalloc(&t->part, sizeof(float) * np * ctas);
    if (e == cudaSuccess)
        e = cudaMalloc(&t->scratch, sizeof(float) * ctas *
                                        (mlp->width == 256 && mlp->depth > 3
                                             ? TrShape<256, 4, 16, true>::scratch(mlp->depth)
                                             : (size_t)tr_slots(mlp->depth) * kTrSlotFloats * 4));
    if (e == cudaSuccess) e = cudaMalloc(&t->loss_part, sizeof(double) * ctas);
    if (e == cudaSuccess) e = cudaMalloc(&t->loss_out, sizeof(double));
    if (e == cudaSuccess) e = cudaMemsetAsync(t->m, 0, sizeof(float) * np, mlp->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(t->v, 0, sizeof(float) * np, mlp->stream);
    if (e != cudaSuccess) {
        rb_trainer_destroy(t);
        return cuda_fail(e, "cudaMalloc (trainer)");
    }
    *out = t;
    return RB_OK;
}

rb_status rb_trainer_set_lr(rb_trainer* t, float lr) {
    if (!t || !(lr > 0.f)) return fail(RB_EINVAL, "need a trainer and lr > 0");
    t->lr = lr;
    return RB_OK;
}

rb_status rb_trainer_destroy(rb_trainer* t) {
    if (!t) return RB_OK;
    // the network may be gone already (destroyed in any order at a process's end):
    // cudaFree waits for the work in flight
    void* ptrs[] = {t->m, t->v, t->grad, t->pred, t->part, t->scratch, t->loss_part, t->loss_out};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete t;
    return RB_OK;
}

rb_status rb_train_grad(rb_trainer* t, int64_t batch, const float* cfg, const float* labels,
                        float lam_tau, float lam_E, float f_scale, float kT_w, float* grad_out,
                        double* loss_host) {
    if (!t || !cfg || !labels) return fail(RB_EINVAL, "null argument");
    if (batch < 1 || batch > t->max_batch) return fail(RB_EINVAL, "batch out of range");
    RB_TRY(train_batch(t, batch, cfg, labels, lam_tau, lam_E, f_scale, kT_w, false, loss_host));
    if (grad_out)
        RB_CUDA(cudaMemcpyAsync(grad_out, t->grad, sizeof(float) * t->mlp->n_params,
                                cudaMemcpyDeviceToDevice, t->mlp->stream));
    return RB_OK;
}

rb_status rb_train_step(rb_trainer* t, int64_t batch, const float* cfg, const float* labels,
                        float lam_tau, float lam_E, float f_scale, float kT_w,
                        double* loss_host) {
    if (!t || !cfg || !labels) return fail(RB_EINVAL, "null argument");
    if (batch < 1 || batch > t->max_batch) return fail(RB_EINVAL, "batch out of range");
    return train_batch(t, batch, cfg, labels, lam_tau, lam_E, f_scale, kT_w, true, loss_host);
}

rb_status rb_nn_weight_vjp(rb_trainer* t, int64_t n, const float* cfg, const float* u_cfg,
                           const float* c, float* grad_out) {
    if (!t || !cfg || !u_cfg || !c || !grad_out) return fail(RB_EINVAL, "null argument");
    if (n < 1 || n > t->max_batch) return fail(RB_EINVAL, "n out of range");
    RB_TRY(check_mlp(t->mlp));
    TrArgs A{};
    A.n = n;
    A.cfg = reinterpret_cast<const float4*>(cfg);
    A.ucfg = reinterpret_cast<const float4*>(u_cfg);
    A.c = c;
    return train_pass(t, A, grad_out, false);
}

}  // extern "C"
