// FP32 network pieces shared by the SIMT inference kernel (nn.cu) and the
// training kernels (train.cu, fnet.cu): the prepared weight copies, the cp.async
// ring that streams them through shared memory, register tiles and Adam.
#pragma once

#include "nn_common.cuh"

namespace rb {

constexpr int kF32Threads = 256;

// Prepared FP32 weights (device), built from the flat parameters:
//   WT1p [16][W]      W1 transposed, rows 10..15 zero          (forward, layer 1)
//   WT_l [W][W]       W_l transposed, l = 2..D                 (forward)
//   W1p  [W][16]      W1 with columns 10..15 zero              (dE/dx)
//   WR_l [W][W]       W_l as stored ([out][in]), l = 2..D      (reverse)
// Every block starts on a 64-byte boundary (W is a multiple of 64).
struct F32Layout {
    int64_t wt1 = 0, wt = 0, w1p = 0, wr = 0, total = 0;
};
__host__ __device__ inline F32Layout f32_layout(int W, int D) {
    F32Layout L;
    L.wt1 = 0;
    L.wt = L.wt1 + (int64_t)kInPad * W;
    L.w1p = L.wt + (int64_t)(D - 1) * W * W;
    L.wr = L.w1p + (int64_t)W * kInPad;
    L.total = L.wr + (int64_t)(D - 1) * W * W;
    return L;
}

__device__ inline void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ inline void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// The weight chunks one tile consumes, in order: layer-1 (16 rows), the
// forward chunks of W_2..W_D, the reverse chunks of W_D..W_2.  A CTA consumes
// this sequence once per tile; chunk c lives in buffer c % 2.
template <int W, int KC, int T = kF32Threads>
struct ChunkFeed {
    static_assert(KC >= kInPad && W % KC == 0, "chunk rows must divide the width");
    static constexpr int NK = W / KC;  // chunks per hidden matrix
    const float* prep;
    F32Layout pl;
    int D;
    int n_chunks;
    int64_t c, total;
    float* buf;

    __device__ void source(int ci, const float*& p, int& rows) const {
        if (ci == 0) {
            p = prep + pl.wt1;
            rows = kInPad;
            return;
        }
        int r = ci - 1;
        rows = KC;
        const int nf = (D - 1) * NK;
        if (r < nf) {
            p = prep + pl.wt + (int64_t)(r / NK) * W * W + (int64_t)(r % NK) * KC * W;
            return;
        }
        r -= nf;
        const int l = D - r / NK;
        p = prep + pl.wr + (int64_t)(l - 2) * W * W + (int64_t)(r % NK) * KC * W;
    }
    // All threads: start the copy of chunk cc into its buffer.
    __device__ void issue(int64_t cc) {
        if (cc >= total) return;
        const float* p;
        int rows;
        source((int)(cc % n_chunks), p, rows);
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(buf + (cc & 1) * KC * W));
        const int pieces = rows * W / 4;
        for (int t = threadIdx.x; t < pieces; t += T) cp_async16(dst + 16u * t, p + 4 * t);
        cp_async_commit();
    }
    // Wait for chunk c (this thread's copies, then everyone's via the
    // barrier, which also retires every read of chunk c-1's buffer), start
    // chunk c+1 into that buffer and return chunk c.
    __device__ const float* acquire() {
        cp_async_wait_all();
        __syncthreads();
        issue(c + 1);
        return buf + (c & 1) * KC * W;
    }
    __device__ void release() { ++c; }
};

// ---- pieces of the training kernels (train.cu, fnet.cu)
// CPT consecutive samples of one unit.
template <int CPT>
struct TrVec {
    float v[CPT];
};
template <int CPT>
__device__ __forceinline__ TrVec<CPT> tr_ld(const float* p) {
    TrVec<CPT> r;
    if constexpr (CPT == 4) {
        const float4 a = *reinterpret_cast<const float4*>(p);
        r.v[0] = a.x, r.v[1] = a.y, r.v[2] = a.z, r.v[3] = a.w;
    } else {
        const float2 a = *reinterpret_cast<const float2*>(p);
        r.v[0] = a.x, r.v[1] = a.y;
    }
    return r;
}
template <int CPT>
__device__ __forceinline__ void tr_st(float* p, const TrVec<CPT>& r) {
    if constexpr (CPT == 4)
        *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
    else
        *reinterpret_cast<float2*>(p) = make_float2(r.v[0], r.v[1]);
}

template <int CPT>
__device__ __forceinline__ float tr_at(const float2 (&acc)[CPT][2], int i, int j) {
    const float2 v = acc[i][j >> 1];
    return (j & 1) ? v.y : v.x;
}

// One Adam step of a parameter; m and v in place.
__device__ __forceinline__ float adam_update(float p, float g, float& m, float& v, float lr, float b1, float b2,
                                             float eps, float c1, float c2) {
    m = b1 * m + (1.f - b1) * g;
    v = b2 * v + (1.f - b2) * g * g;
    return p - lr * (m / c1) / (sqrtf(v / c2) + eps);
}

}  // namespace rb
