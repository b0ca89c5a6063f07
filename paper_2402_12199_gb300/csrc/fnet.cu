// Per-component force/torque networks for cylinders (paper, Methods: five
// separate networks for f_1, f_2, f_3, tau_1, tau_2, used directly in the
// simulation, tau_3 about the cylinder's axis not needed; SI Sec. 2: the
// four-number description of a cylinder pair).
//
// Description of a pair (i = cylinder 1, j = cylinder 2), in the frame of
// body i (s = R(q_i)^T R_ij, q_rel = q_i^* q_j; a cylinder's axis is its body
// z axis):
//   z_hat = sign(s_z) e_z (+e_z for s_z = 0), p_z = |s_z|;
//   x_hat = (s_x, s_y, 0) / p_r, p_r = |(s_x, s_y)| (e_x for p_r = 0);
//   y_hat = z_hat x x_hat;
//   u = cylinder 2's axis R(q_rel) e_z in (x_hat, y_hat, z_hat), turned end
//       over end when u_z < 0 (for u_z = 0 the first non-zero of u_x, u_y is
//       made positive); theta = atan2(|(u_x, u_y)|, u_z) (= arccos u_z
//       without the rounding blow-up of arccos near u_z = 1),
//       phi = atan2(u_y, u_x).
// Five networks (4 -> W x D SiLU -> 1) give the force on cylinder 2 and the
// torque on cylinder 1 in that frame; F_i = -F_j and tau_j = -tau_i - s x F_j
// (angular-momentum balance).  The pair energy is not modelled (0).
//
// Inference: a thread evaluates two pairs (one at width 64); the five networks
// sit in shared memory (weight matrices transposed, so one 16-byte load gives
// four outputs' weights of one input); activations stay in registers; layers
// accumulate pairs of outputs with packed FP32x2 FMAs.
// Training: regression of the five components on bead-sum labels,
// L = mean_b w_b sum_c (y_c - t_c)^2, the targets optionally capped to
// [-cap, cap] (the paper caps the wide force and torque range of its training
// data, SI Sec. 6) and optionally weighted, w_b = 1 / (1 + |t_b|^2 / f^2)
// (else 1); one kernel for the gradient (a CTA per network and tile of
// samples), one for the fixed-order sum of its shares and Adam.
#include <algorithm>
#include <cmath>
#include <new>

#include "nn_f32_common.cuh"

struct rb_fnet {
    int device = 0;
    cudaStream_t stream = nullptr;
    int width = 0, depth = 0;
    int64_t net_floats = 0;   // one network, flat layout
    int64_t img_floats = 0;   // one network, kernel image (multiple of 4)
    float* params = nullptr;  // 5 networks, flat FP32 (device), the ABI layout
    float* img = nullptr;     // 5 networks, kernel image (device)
    float* wr = nullptr;      // 5 x (D-1) hidden matrices as stored, [out][in] (training's reverse pass)
    uint64_t version = 1;
    std::atomic<uint64_t> ready_version{0};  // the version other streams have waited for
};

struct rb_fnet_trainer {
    rb_fnet* f = nullptr;
    int64_t max_batch = 0;
    float lr = 1e-3f, beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    int64_t t = 0;
    float *m = nullptr, *v = nullptr, *grad = nullptr;
    float* part = nullptr;        // per CTA: its share of one network's gradient (net_floats)
    float* scratch = nullptr;     // per CTA: silu' of its tile and the top activations
    double* loss_part = nullptr;  // per CTA
    double* loss_out = nullptr;
    int sms = 1;
    float cap = 0.f;      // targets clamped to [-cap, cap] (0: no cap)
    float f_scale = 0.f;  // sample weight 1 / (1 + |t|^2 / f_scale^2) (0: none)
};

namespace rb {

constexpr int kFnIn = 4;
constexpr int kFnNets = 5;
constexpr int kFnThreads = 128;

__host__ __device__ inline int64_t fn_net_size(int W, int D) {
    return 8 + (int64_t)W * kFnIn + W + (int64_t)(D - 1) * ((int64_t)W * W + W) + W + 3;
}
__host__ __device__ inline int64_t fn_img_size(int W, int D) { return (fn_net_size(W, D) + 3) & ~3LL; }

// Offsets of one network's flat layout: weights and bias of layer l
// (0-based), then w_o, b_o, y_scale, y_shift.
struct FnLayout {
    int W;
    int64_t wo, bo, ys, yt;
    __host__ __device__ int64_t w(int l) const {
        return l == 0 ? 8 : 8 + 5LL * W + (int64_t)(l - 1) * ((int64_t)W * W + W);
    }
    __host__ __device__ int64_t b(int l) const { return w(l) + (l == 0 ? 4LL * W : (int64_t)W * W); }
};
__host__ __device__ inline FnLayout fn_layout(int W, int D) {
    FnLayout L{};
    L.W = W;
    L.wo = 8 + 5LL * W + (int64_t)(D - 1) * ((int64_t)W * W + W);
    L.bo = L.wo + W;
    L.ys = L.wo + W + 1;
    L.yt = L.wo + W + 2;
    return L;
}

// Kernel image: the flat layout with every weight matrix transposed
// ([out][in] -> [in][out]), padded to a multiple of 4 floats.
// wr: the hidden matrices as stored, 16-byte aligned.
__global__ void k_fn_prepare(const float* __restrict__ flat, int W, int D, float* __restrict__ img,
                             float* __restrict__ wr) {
    const int64_t n = fn_net_size(W, D), m = fn_img_size(W, D);
    const FnLayout L = fn_layout(W, D);
    const int64_t ww = (int64_t)W * W, nw = (int64_t)kFnNets * (D - 1) * ww;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nw;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / ww;  // network and layer
        wr[t] = flat[k / (D - 1) * n + L.w(1 + (int)(k % (D - 1))) + t % ww];
    }
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < kFnNets * m;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(t / m);
        const int64_t e = t % m;
        const float* f = flat + c * n;
        float v = 0.f;
        if (e < n) {
            v = f[e];
            for (int l = 0; l < D; ++l) {
                const int in = l == 0 ? kFnIn : W;
                if (e >= L.w(l) && e < L.w(l) + (int64_t)W * in) {
                    const int64_t r = e - L.w(l);  // image index [k][o]
                    const int k = (int)(r / W), o = (int)(r % W);
                    v = f[L.w(l) + (int64_t)o * in + k];
                }
            }
        }
        img[t] = v;
    }
}

struct FnFrame {
    float3 xh, yh, zh;
    float d[kFnIn];
};

__device__ inline FnFrame fn_frame(const float3 s, const float4 q) {
    FnFrame f;
    const float sz = s.z < 0.f ? -1.f : 1.f;
    f.zh = make_float3(0.f, 0.f, sz);
    const float pr = sqrtf(s.x * s.x + s.y * s.y);
    f.xh = pr > 0.f ? make_float3(s.x / pr, s.y / pr, 0.f) : make_float3(1.f, 0.f, 0.f);
    f.yh = make_float3(-sz * f.xh.y, sz * f.xh.x, 0.f);
    // cylinder 2's axis: third column of R(q), q = (w, x, y, z) stored as (x, y, z, w) lanes
    const float qw = q.x, qx = q.y, qy = q.z, qz = q.w;
    const float3 a = make_float3(2.f * (qx * qz + qw * qy), 2.f * (qy * qz - qw * qx),
                                 1.f - 2.f * (qx * qx + qy * qy));
    float ux = a.x * f.xh.x + a.y * f.xh.y, uy = a.x * f.yh.x + a.y * f.yh.y, uz = a.z * sz;
    const bool flip = uz < 0.f || (uz == 0.f && (ux < 0.f || (ux == 0.f && uy < 0.f)));
    if (flip) {
        ux = -ux;
        uy = -uy;
        uz = -uz;
    }
    f.d[0] = pr;
    f.d[1] = fabsf(s.z);
    f.d[2] = atan2f(sqrtf(ux * ux + uy * uy), uz);
    f.d[3] = atan2f(uy, ux);
    return f;
}

// SiLU of two pre-activations, z sigma(z) with sigma(z) = 1 / (1 + 2^(-z log2 e))
// (e^-z written with base 2), by the hardware base-2 exponential and reciprocal,
// which flush what is below 2^-126: for z < -88 the exponential or the
// reciprocal saturates and the result is -0 instead of some -1e-36, for z > 88
// it is z.  An IEEE division in the place of the reciprocal was a third of the
// kernel's instructions and gained no accuracy (error against FP64 of the forces
// of 30000 cylinders 1.5e-6 both ways); __expf and __fdividef, which treat
// subnormals, give the same accuracy at 68 us a step instead of 61.
__device__ __forceinline__ float2 fn_silu2(float2 z) {
    constexpr float kLog2e = 1.4426950408889634f;
    const float2 t = __fmul2_rn(z, make_float2(-kLog2e, -kLog2e));
    float ex, ey, rx, ry;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(t.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ey) : "f"(t.y));
    const float2 den = __fadd2_rn(make_float2(ex, ey), make_float2(1.f, 1.f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rx) : "f"(den.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ry) : "f"(den.y));
    return __fmul2_rn(z, make_float2(rx, ry));
}

// One network (image layout in shared memory) on PP descriptions.  Outputs
// (o, o + 1) share a packed accumulator; a 16-byte load of four outputs'
// weights serves all PP pairs.
template <int W, int PP>
__device__ inline void fn_forward(const float* __restrict__ w, const FnLayout& L, int D,
                                  const float (&d)[PP][kFnIn], float (&y)[PP]) {
    float2 h[PP][W / 2];
    {
        const float* p = w + L.w(0);
        const float* b = w + L.b(0);
#pragma unroll
        for (int o = 0; o < W; o += 2)
#pragma unroll
            for (int q = 0; q < PP; ++q) h[q][o / 2] = make_float2(b[o], b[o + 1]);
#pragma unroll
        for (int k = 0; k < kFnIn; ++k) {
            float2 x[PP];
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                const float v = (d[q][k] - w[k]) * w[4 + k];
                x[q] = make_float2(v, v);
            }
#pragma unroll
            for (int o = 0; o < W; o += 4) {
                const float4 w4 = *reinterpret_cast<const float4*>(p + k * W + o);
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    h[q][o / 2] = __ffma2_rn(make_float2(w4.x, w4.y), x[q], h[q][o / 2]);
                    h[q][o / 2 + 1] = __ffma2_rn(make_float2(w4.z, w4.w), x[q], h[q][o / 2 + 1]);
                }
            }
        }
#pragma unroll
        for (int o = 0; o < W / 2; ++o)
#pragma unroll
            for (int q = 0; q < PP; ++q) h[q][o] = fn_silu2(h[q][o]);
    }
    for (int l = 1; l < D; ++l) {
        const float* p = w + L.w(l);
        const float* b = w + L.b(l);
        float2 z[PP][W / 2];
#pragma unroll
        for (int o = 0; o < W; o += 2)
#pragma unroll
            for (int q = 0; q < PP; ++q) z[q][o / 2] = make_float2(b[o], b[o + 1]);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            float2 hk[PP];
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                const float v = (k & 1) ? h[q][k / 2].y : h[q][k / 2].x;
                hk[q] = make_float2(v, v);
            }
#pragma unroll
            for (int o = 0; o < W; o += 4) {
                const float4 w4 = *reinterpret_cast<const float4*>(p + k * W + o);
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    z[q][o / 2] = __ffma2_rn(make_float2(w4.x, w4.y), hk[q], z[q][o / 2]);
                    z[q][o / 2 + 1] = __ffma2_rn(make_float2(w4.z, w4.w), hk[q], z[q][o / 2 + 1]);
                }
            }
        }
#pragma unroll
        for (int o = 0; o < W / 2; ++o)
#pragma unroll
            for (int q = 0; q < PP; ++q) h[q][o] = fn_silu2(z[q][o]);
    }
#pragma unroll
    for (int q = 0; q < PP; ++q) {
        float a = w[L.bo];
#pragma unroll
        for (int o = 0; o < W; o += 2) {
            a = fmaf(w[L.wo + o], h[q][o / 2].x, a);
            a = fmaf(w[L.wo + o + 1], h[q][o / 2].y, a);
        }
        y[q] = fmaf(w[L.ys], a, w[L.yt]);
    }
}

// Pair source: the system's pair list (SYSTEM) or explicit configurations
// (s, 0), (q_rel) per pair.
struct FnSrc {
    const int2* pairs;
    const int* n_pairs;
    const float4 *pos, *quat;
    float3 L, invL;
    float Rc2;
    const float4* cfg;
    int64_t n;
};
struct FnDst {
    float4 *F, *ti, *tj;   // SYSTEM: per-pair results (space frame)
    float4* out;           // explicit: 3 float4 per pair (frame of body i)
};

// A warp evaluates 32 PP pairs at a time, PP per lane (two where the
// activations of both fit the registers), so that a weight load feeds 2 PP
// packed FMAs.  RESIDENT: all five networks stay in shared memory and the warps
// run on their own; else the CTA stages one network after the other.  A thread
// per pair with one network staged at a time took 116 us for the 88 thousand
// listed pairs of 30000 cylinders at width 32 (a 16-byte weight load for every
// two packed FMAs, and an IEEE division per SiLU); this form takes 48 us, bound
// by issue at two CTAs of 244 registers per SM.
template <int W, int PP, bool SYSTEM, bool RESIDENT>
__global__ void __launch_bounds__(kFnThreads)
    k_fnet_pairs(const float* __restrict__ img, int D, int img_sz, FnSrc src, FnDst dst) {
    extern __shared__ float4 sm4[];
    const float* sw = reinterpret_cast<const float*>(sm4);
    if (RESIDENT) {
        // the parameters were written before this stream's work (fnet_ready)
        for (int k = threadIdx.x; k < kFnNets * img_sz / 4; k += kFnThreads)
            sm4[k] = __ldg(reinterpret_cast<const float4*>(img) + k);
    }
    if (SYSTEM) pdl_wait();
    if (RESIDENT) __syncthreads();
    const FnLayout L = fn_layout(W, D);
    const int64_t n = SYSTEM ? (int64_t)(*src.n_pairs) : src.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // RESIDENT: tasks of 32 PP pairs per warp; else of a CTA's warps together
    constexpr int kTask = 32 * PP, kWarps = kFnThreads / 32;
    const int64_t stride = (int64_t)gridDim.x * kWarps * kTask;
    for (int64_t cbase = (int64_t)blockIdx.x * kWarps * kTask; cbase < n; cbase += stride) {
        const int64_t base = cbase + warp * kTask + lane;
        if (RESIDENT && cbase + warp * kTask >= n) break;
        float3 s[PP];
        float4 qi[PP];
        bool inside[PP];
        FnFrame f[PP];
#pragma unroll
        for (int e = 0; e < PP; ++e) {
            const int64_t t = base + 32 * e;
            s[e] = make_float3(1.f, 0.f, 0.f);
            float4 q = make_float4(1.f, 0.f, 0.f, 0.f);
            qi[e] = q;
            inside[e] = t < n;
            if (t < n) {
                if (SYSTEM) {
                    const int2 ij = src.pairs[t];
                    const float4 pi = src.pos[ij.x], pj = src.pos[ij.y];
                    qi[e] = src.quat[ij.x];
                    const float4 qj = src.quat[ij.y];
                    const float3 R = min_image(make_float3(pj.x - pi.x, pj.y - pi.y, pj.z - pi.z), src.L,
                                               src.invL);
                    inside[e] = R.x * R.x + R.y * R.y + R.z * R.z < src.Rc2;
                    s[e] = mulT(qmat(qi[e]), R);
                    q = qmul(qconj(qi[e]), qj);
                } else {
                    const float4 c0 = src.cfg[2 * t], c1 = src.cfg[2 * t + 1];
                    s[e] = make_float3(c0.x, c0.y, c0.z);
                    q = c1;
                }
            }
            f[e] = fn_frame(s[e], q);
        }
        float d[PP][kFnIn], out[kFnNets][PP];
#pragma unroll
        for (int e = 0; e < PP; ++e)
#pragma unroll
            for (int k = 0; k < kFnIn; ++k) d[e][k] = f[e].d[k];
#pragma unroll 1
        for (int c = 0; c < kFnNets; ++c) {
            const float* w = sw + (RESIDENT ? c * img_sz : 0);
            if (!RESIDENT) {
                __syncthreads();  // the previous network's readers are done
                const float4* g = reinterpret_cast<const float4*>(img + (int64_t)c * img_sz);
                for (int k = threadIdx.x; k < img_sz / 4; k += kFnThreads) sm4[k] = __ldg(g + k);
                __syncthreads();
            }
            float y[PP];
            fn_forward<W, PP>(w, L, D, d, y);
#pragma unroll
            for (int k = 0; k < kFnNets; ++k)
#pragma unroll
                for (int e = 0; e < PP; ++e) out[k][e] = k == c ? y[e] : out[k][e];
        }
#pragma unroll
        for (int e = 0; e < PP; ++e) {
            const int64_t t = base + 32 * e;
            if (t >= n) continue;
            const float3 Fj = make_float3(out[0][e] * f[e].xh.x + out[1][e] * f[e].yh.x,
                                          out[0][e] * f[e].xh.y + out[1][e] * f[e].yh.y, out[2][e] * f[e].zh.z);
            const float3 ti = make_float3(out[3][e] * f[e].xh.x + out[4][e] * f[e].yh.x,
                                          out[3][e] * f[e].xh.y + out[4][e] * f[e].yh.y, 0.f);
            const float3 sxF = cross3(s[e], Fj);
            const float3 tj = make_float3(-ti.x - sxF.x, -ti.y - sxF.y, -ti.z - sxF.z);
            if (SYSTEM) {
                if (inside[e]) {
                    const Mat3 Ri = qmat(qi[e]);
                    const float3 a = mul(Ri, Fj), b = mul(Ri, ti), c2 = mul(Ri, tj);
                    dst.F[t] = make_float4(a.x, a.y, a.z, 0.f);
                    dst.ti[t] = make_float4(b.x, b.y, b.z, 0.f);
                    dst.tj[t] = make_float4(c2.x, c2.y, c2.z, 0.f);
                } else {  // listed within the skin only: exactly nothing
                    dst.F[t] = dst.ti[t] = dst.tj[t] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            } else {
                dst.out[3 * t] = make_float4(Fj.x, Fj.y, Fj.z, 0.f);
                dst.out[3 * t + 1] = make_float4(ti.x, ti.y, ti.z, 0.f);
                dst.out[3 * t + 2] = make_float4(tj.x, tj.y, tj.z, 0.f);
            }
        }
    }
}

// All five networks in shared memory where two CTAs per SM still fit.
static bool fn_resident(const rb_fnet* f) {
    return sizeof(float) * kFnNets * (size_t)f->img_floats <= 100 * 1024;
}

template <int W, int PP, bool SYSTEM, bool RESIDENT>
static rb_status launch_fnet_form(const rb_fnet* f, cudaStream_t st, int64_t ctas, int sms, const FnSrc& src,
                                  const FnDst& dst) {
    const size_t smem = sizeof(float) * (size_t)f->img_floats * (RESIDENT ? kFnNets : 1);
    static std::atomic<bool> allowed{false};
    if (!allowed.load()) {
        RB_CUDA(cudaFuncSetAttribute(k_fnet_pairs<W, PP, SYSTEM, RESIDENT>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        allowed.store(true);
    }
    int per_sm = 1;  // one wave of CTAs, each with its own copy of the weights
    RB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fnet_pairs<W, PP, SYSTEM, RESIDENT>,
                                                          kFnThreads, smem));
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ctas, (int64_t)sms * std::max(1, per_sm)));
    if (SYSTEM)
        RB_CUDA(launch_pdl(k_fnet_pairs<W, PP, SYSTEM, RESIDENT>, grid, kFnThreads, smem, st,
                           (const float*)f->img, f->depth, (int)f->img_floats, src, dst));
    else
        k_fnet_pairs<W, PP, SYSTEM, RESIDENT><<<grid, kFnThreads, smem, st>>>(f->img, f->depth,
                                                                            (int)f->img_floats, src, dst);
    RB_CUDA(cudaGetLastError());
    return RB_OK;
}

template <int W, int PP, bool SYSTEM>
static rb_status launch_fnet_w(const rb_fnet* f, cudaStream_t st, int64_t ctas, int sms, const FnSrc& src,
                               const FnDst& dst) {
    ctas = (ctas + PP - 1) / PP;
    return fn_resident(f) ? launch_fnet_form<W, PP, SYSTEM, true>(f, st, ctas, sms, src, dst)
                          : launch_fnet_form<W, PP, SYSTEM, false>(f, st, ctas, sms, src, dst);
}

// ctas: CTAs of kFnThreads pairs
template <bool SYSTEM>
static rb_status launch_fnet(const rb_fnet* f, cudaStream_t st, int64_t ctas, const FnSrc& src, const FnDst& dst) {
    int sms = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, f->device);
    switch (f->width) {
        case 16: return launch_fnet_w<16, 2, SYSTEM>(f, st, ctas, sms, src, dst);
        case 32: return launch_fnet_w<32, 2, SYSTEM>(f, st, ctas, sms, src, dst);
        case 64: return launch_fnet_w<64, 1, SYSTEM>(f, st, ctas, sms, src, dst);
        default: return fail(RB_ENOTSUP, "per-component networks support widths 16, 32, 64");
    }
}

rb_status check_fnet(const rb_fnet* f) {
    if (!f) return fail(RB_EINVAL, "null per-component network");
    return RB_OK;
}

uint64_t fnet_version(const rb_fnet* f) { return f->version; }

rb_status fnet_ready(const rb_fnet* cf) {
    // the parameters and the kernel image are written on the network's stream;
    // the system's stream reads them, so it waits for that stream once per change
    rb_fnet* f = const_cast<rb_fnet*>(cf);
    if (f->ready_version.load() == f->version) return RB_OK;
    RB_CUDA(cudaStreamSynchronize(f->stream));
    f->ready_version.store(f->version);
    return RB_OK;
}

rb_status fnet_pairs_system_async(rb_system* s, const rb_fnet* f) {
    RB_TRY(check_fnet(f));
    FnSrc src{};
    src.pairs = s->pl.pairs;
    src.n_pairs = s->pl.n_pairs;
    src.pos = s->pos;
    src.quat = s->quat;
    src.L = make_float3(s->box[0], s->box[1], s->box[2]);
    src.invL = make_float3(1.f / s->box[0], 1.f / s->box[1], 1.f / s->box[2]);
    src.Rc2 = s->Rc * s->Rc;
    FnDst dst{};
    dst.F = s->pair_F;
    dst.ti = s->pair_ti;
    dst.tj = s->pair_tj;
    return launch_fnet<true>(f, s->stream, pair_grid(s, kFnThreads, s->num_sms * 8), src, dst);
}

// ------------------------------------------------------------- training
// The gradient of L for one network and a tile of S = 4096 / W samples per CTA
// and pass (blockIdx: network x share of the tiles): description, target and
// weight of every sample, forward, residual, backward, and the layer gradients
// added to the CTA's own share.  A thread owns 4 samples x 4 units of every
// layer; activations and signals live in shared memory as [unit][sample] (row
// stride S + 4, so that rows of consecutive units fall on different banks),
// silu' and the top activations, which only their own thread reads again, in a
// global scratch; the network's weights (17 KB at width 32, depth 3) are staged in shared
// memory or come through L1 (FnTile::staged).
// A step was about 130 launches (GEMMs, column sums and elementwise kernels of
// the five networks one after the other, 880 us at batch 4096 and width 32, for
// 0.27 GFLOP); it is two, 36 us (this kernel 30 us), and the gradient's error
// against FP64 went from 8.6e-7 to 1.1e-7.  Bound by latency: a dozen dependent
// short stages.
struct FnTrainArgs {
    int64_t n;
    const float4 *cfg, *lab;
    float cap, f_scale;
};

constexpr int kFnCpt = 4;
template <int W>
struct FnTile {
    static constexpr int S = 1024 * kFnCpt / W, LD = S + 4;
    static constexpr int NTP = S / kFnCpt, NG = W / 4;
    static constexpr int kWarpsPerUnit = NTP > 32 ? NTP / 32 : 1;
    static size_t smem(int D) {
        return sizeof(float) * ((size_t)(D + 1) * W * LD + kFnIn * LD + NG * S + 2 * S + kWarpsPerUnit * W + 16) +
               sizeof(double) * 256;
    }
    // a network's image and stored matrices beside them, where two CTAs per SM
    // still fit (width 32: 39.5 -> 35.7 us a step of 4096; width 64, where only
    // one would: 74 -> 82 us)
    static size_t weights(int D) { return sizeof(float) * ((size_t)fn_img_size(W, D) + (size_t)(D - 1) * W * W); }
    static bool staged(int D) { return smem(D) + weights(D) <= 112 * 1024; }
};
__host__ __device__ inline size_t fn_scratch_floats(int D) { return (size_t)(D + 1) * 4 * 256 * kFnCpt; }

// out[o * W + i] (+)= sum_c A[o][c] B[i][c], every thread W * W / 256 outputs.
template <int W>
__device__ inline void fn_weight_grad(const float* __restrict__ A, const float* __restrict__ B,
                                      float* __restrict__ out, bool first) {
    constexpr int S = FnTile<W>::S, LD = FnTile<W>::LD;
    constexpr int LI = W < 32 ? W : 32;               // lanes along i
    constexpr int IN = W / LI, RO = 8 * (32 / LI), ON = W / RO;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = lane % LI, r0 = warp * (32 / LI) + lane / LI;
    float2 acc[ON][IN];
#pragma unroll
    for (int o = 0; o < ON; ++o)
#pragma unroll
        for (int j = 0; j < IN; ++j) acc[o][j] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int c = 0; c < S; c += 4) {
        float4 b[IN];
#pragma unroll
        for (int j = 0; j < IN; ++j) b[j] = *reinterpret_cast<const float4*>(B + (i0 + LI * j) * LD + c);
#pragma unroll
        for (int o = 0; o < ON; ++o) {
            const float4 a = *reinterpret_cast<const float4*>(A + (r0 + RO * o) * LD + c);
#pragma unroll
            for (int j = 0; j < IN; ++j) {
                acc[o][j] = __ffma2_rn(make_float2(a.x, a.y), make_float2(b[j].x, b[j].y), acc[o][j]);
                acc[o][j] = __ffma2_rn(make_float2(a.z, a.w), make_float2(b[j].z, b[j].w), acc[o][j]);
            }
        }
    }
#pragma unroll
    for (int o = 0; o < ON; ++o)
#pragma unroll
        for (int j = 0; j < IN; ++j) {
            float* p = out + (r0 + RO * o) * W + i0 + LI * j;
            const float v = acc[o][j].x + acc[o][j].y;
            *p = first ? v : *p + v;
        }
}

// acc[i][.] = sum_k A[k][p0 + i] B[k][o0 + .], A in shared memory, B global.
template <int W>
__device__ inline void fn_gemm(const float* __restrict__ As, const float* __restrict__ B, int K, int p0, int o0,
                               float2 (&acc)[kFnCpt][2]) {
#pragma unroll
    for (int i = 0; i < kFnCpt; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const TrVec<kFnCpt> a = tr_ld<kFnCpt>(As + k * FnTile<W>::LD + p0);
        const float4 b = *reinterpret_cast<const float4*>(B + k * W + o0);
        const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
#pragma unroll
        for (int i = 0; i < kFnCpt; ++i) {
            const float2 aa = make_float2(a.v[i], a.v[i]);
            acc[i][0] = __ffma2_rn(aa, b0, acc[i][0]);
            acc[i][1] = __ffma2_rn(aa, b1, acc[i][1]);
        }
    }
}

template <int W>
__global__ void __launch_bounds__(256)
    k_fn_tile(const float* __restrict__ img, int64_t img_sz, const float* __restrict__ wr, int D, FnTrainArgs A,
              float* __restrict__ part, int64_t nn, float* __restrict__ scratch, double* __restrict__ loss_part,
              int staged) {
    using T = FnTile<W>;
    constexpr int S = T::S, LD = T::LD, NTP = T::NTP, NG = T::NG;
    pdl_wait();
    extern __shared__ double smem_d[];
    double* s_loss = smem_d;                                 // 256
    float* Hs = reinterpret_cast<float*>(smem_d + 256);      // h_1 .. h_{D-1}
    float* G0 = Hs + (size_t)(D - 1) * W * LD;               // signals of a layer, two in turn
    float* G1 = G0 + W * LD;
    float* Xs = G1 + W * LD;                                 // [4][LD] normalised inputs
    float* Red = Xs + kFnIn * LD;                            // [NG][S] partial sums of w_o . h
    float* ts = Red + NG * S;                                // S residuals
    float* Wp = ts + 2 * S;                                  // [warps per unit][W] partial sums of w_o's gradient
    const int tid = threadIdx.x, tp = tid % NTP, to = tid / NTP;
    const int p0 = tp * kFnCpt, o0 = to * 4;
    const int c = blockIdx.x, share = blockIdx.y, n_share = gridDim.y;
    const int cta = c * n_share + share;
    const FnLayout L = fn_layout(W, D);
    const float* net = img + c * img_sz;  // matrices [in][out], everything else as in the flat layout
    const float* wrc = wr + (int64_t)c * (D - 1) * W * W;
    if (staged) {
        float4* w4 = reinterpret_cast<float4*>(Wp + T::kWarpsPerUnit * W);
        const int ni = (int)img_sz / 4, nr = (D - 1) * W * W / 4;
        for (int k = tid; k < ni; k += 256) w4[k] = reinterpret_cast<const float4*>(net)[k];
        for (int k = tid; k < nr; k += 256) w4[ni + k] = reinterpret_cast<const float4*>(wrc)[k];
        net = reinterpret_cast<const float*>(w4);
        wrc = reinterpret_cast<const float*>(w4 + ni);
        __syncthreads();
    }
    float* gp = part + (size_t)cta * nn;
    float* mine = scratch + (size_t)cta * fn_scratch_floats(D) + (size_t)tid * kFnCpt;
    auto slot = [&](int k, int j) { return mine + ((size_t)k * 4 + j) * 256 * kFnCpt; };
    const float bo = net[L.bo], ys = net[L.ys], yt = net[L.yt];
    const int64_t n_tiles = (A.n + S - 1) / S;
    double loss = 0.0;
    float r_sum = 0.f;
    bool first = true;
    for (int64_t tile = share; tile < n_tiles; tile += n_share, first = false) {
        const int64_t b = tile * S + tid;
        const bool valid = tid < S && b < A.n;
        float target = 0.f, weight = 0.f;
        if (tid < S) {
            float d[kFnIn] = {0.f, 0.f, 0.f, 0.f};
            if (valid) {
                const float4 c0 = A.cfg[2 * b], c1 = A.cfg[2 * b + 1];
                const FnFrame f = fn_frame(make_float3(c0.x, c0.y, c0.z), c1);
                const float4 F = A.lab[3 * b], ti = A.lab[3 * b + 1];
                float t[5] = {F.x * f.xh.x + F.y * f.xh.y, F.x * f.yh.x + F.y * f.yh.y, F.z * f.zh.z,
                              ti.x * f.xh.x + ti.y * f.xh.y, ti.x * f.yh.x + ti.y * f.yh.y};
                float t2 = 0.f;
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    t[k] = A.cap > 0.f ? fminf(fmaxf(t[k], -A.cap), A.cap) : t[k];
                    t2 = fmaf(t[k], t[k], t2);
                    target = k == c ? t[k] : target;
                }
                weight = A.f_scale > 0.f ? 1.f / (1.f + t2 / (A.f_scale * A.f_scale)) : 1.f;
#pragma unroll
                for (int k = 0; k < kFnIn; ++k) d[k] = f.d[k];
            }
#pragma unroll
            for (int k = 0; k < kFnIn; ++k) Xs[k * LD + tid] = (d[k] - net[k]) * net[4 + k];
        }
        __syncthreads();
        // ---- forward
        float2 acc[kFnCpt][2];
        for (int l = 0; l < D; ++l) {
            fn_gemm<W>(l == 0 ? Xs : Hs + (size_t)(l - 1) * W * LD, net + L.w(l), l == 0 ? kFnIn : W, p0, o0, acc);
            TrVec<kFnCpt> e;
#pragma unroll
            for (int i = 0; i < kFnCpt; ++i) e.v[i] = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float bj = net[L.b(l) + o0 + j], w = net[L.wo + o0 + j];
                TrVec<kFnCpt> h, d1;
#pragma unroll
                for (int i = 0; i < kFnCpt; ++i) {
                    const float z = tr_at<kFnCpt>(acc, i, j) + bj;
                    const float sg = 1.f / (1.f + __expf(-z));
                    h.v[i] = z * sg;
                    d1.v[i] = sg * (1.f + z * (1.f - sg));
                    e.v[i] = fmaf(w, h.v[i], e.v[i]);
                }
                tr_st<kFnCpt>(slot(l, j), d1);
                if (l < D - 1)
                    tr_st<kFnCpt>(Hs + (size_t)l * W * LD + (size_t)(o0 + j) * LD + p0, h);
                else
                    tr_st<kFnCpt>(slot(D, j), h);
            }
            if (l == D - 1) tr_st<kFnCpt>(Red + (size_t)to * S + p0, e);
            __syncthreads();
        }
        // ---- residual r = 2 w (y - t) / n, scaled by y_scale
        if (tid < S) {
            float y = bo;
            for (int g = 0; g < NG; ++g) y += Red[(size_t)g * S + tid];
            const float dv = fmaf(ys, y, yt) - target;
            const float r = valid ? 2.f * weight * dv / (float)A.n * ys : 0.f;
            ts[tid] = r;
            r_sum += r;
            if (valid) loss += (double)weight * dv * dv;
        }
        __syncthreads();
        // ---- top: the gradient of w_o and the signal r w_o silu'
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const TrVec<kFnCpt> h = tr_ld<kFnCpt>(slot(D, j));
            TrVec<kFnCpt> d1 = tr_ld<kFnCpt>(slot(D - 1, j));
            const float w = net[L.wo + o0 + j];
            float sum = 0.f;
#pragma unroll
            for (int i = 0; i < kFnCpt; ++i) {
                const float r = ts[p0 + i];
                sum = fmaf(r, h.v[i], sum);
                d1.v[i] *= r * w;
            }
            tr_st<kFnCpt>(G0 + (size_t)(o0 + j) * LD + p0, d1);
            constexpr int kGroup = NTP < 32 ? NTP : 32;
#pragma unroll
            for (int o = 1; o < kGroup; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (tp % kGroup == 0) Wp[(tp / kGroup) * W + o0 + j] = sum;
        }
        __syncthreads();
        if (tid < W) {
            float a = Wp[tid];
            if (T::kWarpsPerUnit > 1) a += Wp[W + tid];
            float* q = gp + L.wo + tid;
            *q = first ? a : *q + a;
        }
        // ---- backward
        float* g = G0;
        float* gn = G1;
        for (int l = D - 1; l >= 0; --l) {
            for (int o = tid; o < W; o += 256) {
                float a = 0.f;
                for (int k = 0; k < S; k += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(g + (size_t)o * LD + k);
                    a += (v.x + v.y) + (v.z + v.w);
                }
                float* q = gp + L.b(l) + o;
                *q = first ? a : *q + a;
            }
            if (l == 0) {
                for (int t = tid; t < W * kFnIn; t += 256) {
                    const int o = t / kFnIn, k = t % kFnIn;
                    float a = 0.f;
                    for (int s = 0; s < S; ++s) a = fmaf(g[(size_t)o * LD + s], Xs[k * LD + s], a);
                    float* q = gp + L.w(0) + t;
                    *q = first ? a : *q + a;
                }
                break;
            }
            fn_weight_grad<W>(g, Hs + (size_t)(l - 1) * W * LD, gp + L.w(l), first);
            fn_gemm<W>(g, wrc + (size_t)(l - 1) * W * W, W, p0, o0, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                TrVec<kFnCpt> d1 = tr_ld<kFnCpt>(slot(l - 1, j));
#pragma unroll
                for (int i = 0; i < kFnCpt; ++i) d1.v[i] *= tr_at<kFnCpt>(acc, i, j);
                tr_st<kFnCpt>(gn + (size_t)(o0 + j) * LD + p0, d1);
            }
            __syncthreads();
            float* tmp = g;
            g = gn;
            gn = tmp;
        }
        __syncthreads();  // the next tile overwrites what this one read
    }
    s_loss[tid] = loss;
    if (tid < S) ts[tid] = r_sum;
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        float r = 0.f;
        for (int k = 0; k < S; ++k) {
            a += s_loss[k];
            r += ts[k];
        }
        loss_part[cta] = a;
        gp[L.bo] = r;
    }
}

// Sum of each network's shares (in order), the loss, Adam when `step`, and the
// kernel images of the updated parameters.
struct FnAdam {
    float *p, *m, *v, *img, *wr;
    float lr, b1, b2, eps, c1, c2;
};
__global__ void __launch_bounds__(256)
    k_fn_update(int W, int D, int64_t nn, int64_t img_sz, int n_share, const float* __restrict__ part,
                float* __restrict__ grad, bool step, FnAdam a, const double* __restrict__ loss_part,
                double inv_n, double* __restrict__ loss_out) {
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double x = 0.0;
        for (int k = threadIdx.x; k < kFnNets * n_share; k += 32) x += loss_part[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (threadIdx.x == 0) *loss_out = x * inv_n;
    }
    const int64_t t = blockIdx.x * (int64_t)256 + threadIdx.x;
    if (t >= kFnNets * nn) return;
    const int64_t c = t / nn, e = t % nn;
    const FnLayout L = fn_layout(W, D);
    const bool train = e >= 8 && e <= L.bo;
    float g = 0.f;
    if (train) {
        const float* q = part + (size_t)c * n_share * nn + e;
        int k = 0;
        for (; k + 8 <= n_share; k += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = q[(size_t)(k + u) * nn];
#pragma unroll
            for (int u = 0; u < 8; ++u) g += v[u];
        }
        for (; k < n_share; ++k) g += q[(size_t)k * nn];
    }
    grad[t] = g;
    if (!step || !train) return;
    const float p = adam_update(a.p[t], g, a.m[t], a.v[t], a.lr, a.b1, a.b2, a.eps, a.c1, a.c2);
    a.p[t] = p;
    // the image's place of entry e: matrices transposed, the rest as it is
    float* im = a.img + c * img_sz;
    int64_t at = e;
    if (e < L.b(0)) {
        const int64_t r = e - 8;
        at = 8 + r % kFnIn * W + r / kFnIn;
    } else if (e >= L.w(1) && e < L.wo) {
        const int64_t per = (int64_t)W * W + W, r = (e - L.w(1)) % per, l = (e - L.w(1)) / per;
        if (r < (int64_t)W * W) {
            at = e - r + r % W * W + r / W;
            a.wr[(c * (D - 1) + l) * W * W + r] = p;
        }
    }
    im[at] = p;
}

static inline int nblk(int64_t n, int t = 256) { return (int)std::max<int64_t>(1, (n + t - 1) / t); }

// Shares per network: a CTA per tile, at most two per SM over the five networks.
static int fn_shares(const rb_fnet_trainer* t, int64_t B) {
    const int64_t S = 1024 * kFnCpt / t->f->width;
    return (int)std::max<int64_t>(1, std::min<int64_t>((B + S - 1) / S, 2 * t->sms / kFnNets));
}

template <int W>
static rb_status launch_fn_tile(rb_fnet_trainer* t, int shares, const FnTrainArgs& A) {
    rb_fnet* f = t->f;
    static std::atomic<bool> allowed{false};
    if (!allowed.load()) {
        RB_CUDA(cudaFuncSetAttribute(k_fn_tile<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        allowed.store(true);
    }
    const bool staged = FnTile<W>::staged(f->depth);
    RB_CUDA(launch_pdl(k_fn_tile<W>, dim3(kFnNets, shares), 256,
                       FnTile<W>::smem(f->depth) + (staged ? FnTile<W>::weights(f->depth) : 0), f->stream, f->img,
                       f->img_floats, f->wr, f->depth, A, t->part, f->net_floats, t->scratch, t->loss_part,
                       staged ? 1 : 0));
    return RB_OK;
}

// Gradient of L for a batch of B sampled pairs (cfg: 2 float4, labels: 3
// float4 per pair, as rb_sample_pairs writes them) into t->grad (the flat
// layout; zero for mu, inv_sd, y_scale, y_shift), and the Adam step.
static rb_status fn_train(rb_fnet_trainer* t, int64_t B, const float4* cfg, const float4* lab, bool step,
                          double* loss_host) {
    rb_fnet* f = t->f;
    const FnTrainArgs A{B, cfg, lab, t->cap, t->f_scale};
    const int shares = fn_shares(t, B);
    switch (f->width) {
        case 16: RB_TRY(launch_fn_tile<16>(t, shares, A)); break;
        case 32: RB_TRY(launch_fn_tile<32>(t, shares, A)); break;
        default: RB_TRY(launch_fn_tile<64>(t, shares, A)); break;
    }
    FnAdam a{f->params, t->m, t->v, f->img, f->wr, t->lr, t->beta1, t->beta2, t->eps, 1.f, 1.f};
    if (step) {
        ++t->t;
        // bias corrections in FP64 (1 - beta2^t cancels badly in FP32)
        a.c1 = (float)(1.0 - std::pow((double)t->beta1, (double)t->t));
        a.c2 = (float)(1.0 - std::pow((double)t->beta2, (double)t->t));
    }
    RB_CUDA(launch_pdl(k_fn_update, nblk(kFnNets * f->net_floats), 256, 0, f->stream, f->width, f->depth,
                       f->net_floats, f->img_floats, shares, t->part, t->grad, step, a, t->loss_part,
                       1.0 / (double)B, t->loss_out));
    if (step) ++f->version;
    if (loss_host) {
        RB_CUDA(cudaMemcpyAsync(loss_host, t->loss_out, sizeof(double), cudaMemcpyDeviceToHost, f->stream));
        RB_CUDA(cudaStreamSynchronize(f->stream));
    }
    return RB_OK;
}

static rb_status fn_prepare(rb_fnet* f) {
    k_fn_prepare<<<nblk(kFnNets * f->img_floats), 256, 0, f->stream>>>(f->params, f->width, f->depth,
                                                                      f->img, f->wr);
    RB_CUDA(cudaGetLastError());
    ++f->version;
    return RB_OK;
}

}  // namespace rb

using namespace rb;

extern "C" {

int64_t rb_fnet_n_params(int32_t width, int32_t depth) {
    if (width < 1 || depth < 1 || depth > 8) return -1;
    return kFnNets * fn_net_size(width, depth);
}

rb_status rb_fnet_create(int32_t width, int32_t depth, void* stream, rb_fnet** out) {
    if (!out) return fail(RB_EINVAL, "null argument");
    *out = nullptr;
    if (width != 16 && width != 32 && width != 64)
        return fail(RB_ENOTSUP, "per-component networks support widths 16, 32, 64");
    if (depth < 1 || depth > 8) return fail(RB_EINVAL, "depth must be in [1, 8]");
    rb_fnet* f = new (std::nothrow) rb_fnet();
    if (!f) return fail(RB_ENOMEM, "host allocation");
    f->stream = (cudaStream_t)stream;
    cudaGetDevice(&f->device);
    f->width = width;
    f->depth = depth;
    f->net_floats = fn_net_size(width, depth);
    f->img_floats = fn_img_size(width, depth);
    cudaError_t e = cudaMalloc((void**)&f->params, sizeof(float) * kFnNets * f->net_floats);
    if (e == cudaSuccess) e = cudaMalloc((void**)&f->img, sizeof(float) * kFnNets * f->img_floats);
    if (e == cudaSuccess)
        e = cudaMalloc((void**)&f->wr, sizeof(float) * std::max<int64_t>(16, (int64_t)kFnNets * (depth - 1) * width * width));
    if (e == cudaSuccess) e = cudaMemsetAsync(f->params, 0, sizeof(float) * kFnNets * f->net_floats, f->stream);
    if (e != cudaSuccess) {
        cudaFree(f->params);
        cudaFree(f->img);
        cudaFree(f->wr);
        delete f;
        return cuda_fail(e, "per-component network allocation");
    }
    if (sizeof(float) * f->img_floats > 227 * 1024) {
        cudaFree(f->params);
        cudaFree(f->img);
        cudaFree(f->wr);
        delete f;
        return fail(RB_ENOTSUP, "one network's weights must fit in shared memory (227 KB)");
    }
    *out = f;
    return fn_prepare(f);
}

rb_status rb_fnet_destroy(rb_fnet* f) {
    if (!f) return RB_OK;
    if (f->stream) cudaStreamSynchronize(f->stream);
    cudaFree(f->params);
    cudaFree(f->img);
    cudaFree(f->wr);
    delete f;
    return RB_OK;
}

rb_status rb_fnet_set_params(rb_fnet* f, const float* flat, int64_t n, int32_t from_host) {
    if (!f || !flat) return fail(RB_EINVAL, "null argument");
    if (n != kFnNets * f->net_floats) return fail(RB_EINVAL, "wrong parameter count");
    RB_CUDA(cudaMemcpyAsync(f->params, flat, sizeof(float) * n,
                            from_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, f->stream));
    if (from_host) RB_CUDA(cudaStreamSynchronize(f->stream));
    return fn_prepare(f);
}

rb_status rb_fnet_get_params(const rb_fnet* f, float* flat, int64_t n, int32_t to_host) {
    if (!f || !flat) return fail(RB_EINVAL, "null argument");
    if (n != kFnNets * f->net_floats) return fail(RB_EINVAL, "wrong parameter count");
    RB_CUDA(cudaMemcpyAsync(flat, f->params, sizeof(float) * n,
                            to_host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, f->stream));
    if (to_host) RB_CUDA(cudaStreamSynchronize(f->stream));
    return RB_OK;
}

rb_status rb_fnet_pairs(const rb_fnet* f, int64_t n, const float* cfg, float* out) {
    RB_TRY(check_fnet(f));
    if (n < 0 || (n > 0 && (!cfg || !out))) return fail(RB_EINVAL, "bad arrays");
    if (n == 0) return RB_OK;
    FnSrc src{};
    src.cfg = reinterpret_cast<const float4*>(cfg);
    src.n = n;
    FnDst dst{};
    dst.out = reinterpret_cast<float4*>(out);
    return launch_fnet<false>(f, f->stream, (n + kFnThreads - 1) / kFnThreads, src, dst);
}

rb_status rb_fnet_trainer_create(rb_fnet* f, int64_t max_batch, float lr, float beta1, float beta2,
                                 float eps, rb_fnet_trainer** out) {
    if (!f || !out) return fail(RB_EINVAL, "null argument");
    *out = nullptr;
    if (max_batch < 1) return fail(RB_EINVAL, "max_batch must be positive");
    rb_fnet_trainer* t = new (std::nothrow) rb_fnet_trainer();
    if (!t) return fail(RB_ENOMEM, "host allocation");
    t->f = f;
    t->max_batch = max_batch;
    t->lr = lr;
    t->beta1 = beta1;
    t->beta2 = beta2;
    t->eps = eps;
    const int64_t np = kFnNets * f->net_floats;
    cudaDeviceGetAttribute(&t->sms, cudaDevAttrMultiProcessorCount, f->device);
    const size_t ctas = (size_t)kFnNets * fn_shares(t, max_batch);
    cudaError_t e = cudaMalloc((void**)&t->m, sizeof(float) * np);
    if (e == cudaSuccess) e = cudaMalloc((void**)&t->v, sizeof(float) * np);
    if (e == cudaSuccess) e = cudaMalloc((void**)&t->grad, sizeof(float) * np);
    if (e == cudaSuccess) e = cudaMalloc((void**)&t->part, sizeof(float) * f->net_floats * ctas);
    if (e == cudaSuccess) e = cudaMalloc((void**)&t->scratch, sizeof(float) * fn_scratch_floats(f->depth) * ctas);
    if (e == cudaSuccess) e = cudaMalloc((void**)&t->loss_part, sizeof(double) * ctas);
    if (e == cudaSuccess) e = cudaMalloc((void**)&t->loss_out, sizeof(double));
    if (e == cudaSuccess) e = cudaMemsetAsync(t->m, 0, sizeof(float) * np, f->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(t->v, 0, sizeof(float) * np, f->stream);
    if (e != cudaSuccess) {
        cudaFree(t->m);
        cudaFree(t->v);
        cudaFree(t->grad);
        cudaFree(t->part);
        cudaFree(t->scratch);
        cudaFree(t->loss_part);
        cudaFree(t->loss_out);
        delete t;
        return cuda_fail(e, "trainer allocation");
    }
    *out = t;
    return RB_OK;
}

rb_status rb_fnet_trainer_destroy(rb_fnet_trainer* t) {
    if (!t) return RB_OK;
    // the network may be gone already (destroyed in any order at a process's end):
    // cudaFree waits for the work in flight
    cudaFree(t->m);
    cudaFree(t->v);
    cudaFree(t->grad);
    cudaFree(t->part);
    cudaFree(t->scratch);
    cudaFree(t->loss_part);
    cudaFree(t->loss_out);
    delete t;
    return RB_OK;
}

rb_status rb_fnet_train_grad(rb_fnet_trainer* t, int64_t batch, const float* cfg, const float* labels,
                             float* grad_out, double* loss_host) {
    if (!t) return fail(RB_EINVAL, "null trainer");
    if (batch < 1 || batch > t->max_batch || !cfg || !labels)
        return fail(RB_EINVAL, "batch must be in [1, max_batch] with cfg and labels");
    RB_TRY(fn_train(t, batch, reinterpret_cast<const float4*>(cfg), reinterpret_cast<const float4*>(labels), false,
                    loss_host));
    if (grad_out)
        RB_CUDA(cudaMemcpyAsync(grad_out, t->grad, sizeof(float) * kFnNets * t->f->net_floats,
                                cudaMemcpyDeviceToDevice, t->f->stream));
    return RB_OK;
}

rb_status rb_fnet_train_step(rb_fnet_trainer* t, int64_t batch, const float* cfg, const float* labels,
                             double* loss_host) {
    if (!t) return fail(RB_EINVAL, "null trainer");
    if (batch < 1 || batch > t->max_batch || !cfg || !labels)
        return fail(RB_EINVAL, "batch must be in [1, max_batch] with cfg and labels");
    return fn_train(t, batch, reinterpret_cast<const float4*>(cfg), reinterpret_cast<const float4*>(labels), true,
                    loss_host);
}

rb_status rb_fnet_trainer_set_lr(rb_fnet_trainer* t, float lr) {
    if (!t) return fail(RB_EINVAL, "null trainer");
    t->lr = lr;
    return RB_OK;
}

rb_status rb_fnet_trainer_set_cap(rb_fnet_trainer* t, float cap, float f_scale) {
    if (!t) return fail(RB_EINVAL, "null trainer");
    if (!(cap >= 0.f) || !(f_scale >= 0.f)) return fail(RB_EINVAL, "cap and f_scale must be >= 0");
    t->cap = cap;
    t->f_scale = f_scale;
    return RB_OK;
}

}  // extern "C"
