// Bead-sum kernel: the traditional composite-body interaction (paper, Methods:
// U = sum_i sum_j u_bead(r_ij) over the beads of two bodies; the abstract
// names the evaluation of every bead-bead distance between two bodies as the
// cost of this form).
//
// One warp per body pair, in the frame of body i: its beads are the template
// d_k itself, body j's beads are b_l = s + R_rel d_l with s = R(q_i)^T R_ij and
// R_rel = R(q_i^* q_j).  For templates made of columns of beads with equal
// (x, y) (the cube and the cylinder) only the beads of j within the cutoff of
// the box of i's beads and the columns of i near those are tested
// (k_bead_cols); for other templates every distance is (k_bead_pairs_any).  Per
// lane the force f_l on each owned bead is accumulated; then
//   F_j = sum_l f_l,   T = sum_l b_l x f_l,
//   tau_i = -T (central bead forces: sum_kl d_k x f_kl = sum_kl b_l x f_kl),
//   tau_j = T - s x F_j,
// reduced over the warp with xor shuffles (fixed order, deterministic) and
// rotated back to the space frame with R(q_i).
#include <algorithm>
#include <utility>

#include "beads_common.cuh"

namespace rb {

// Both kernels: pairs with |R|^2 >= cut2 are skipped: with zero_beyond they get
// zero results (the bead path, cut2 = Rc^2, pairs listed only because of the
// skin); without it they keep what is there.  With sel (the network path's bead
// fallback, cut2 = rho_min^2) only the pairs sel[0 .. *sel_count) are visited:
// the network kernel listed those closer than rho_min.  POT = 0: Lennard-Jones
// beads; POT = 1: the half-power half-cosine beads of Eq. 1 (either reading).

// Any template: one warp per listed body pair, grid-stride.  Lanes 0..2 store
// the pair's results in the space frame: F_j (with E), tau_i, tau_j = T - s x F
// (T: the bead torques about body i's centre, in i's frame).
template <int NP, int POT>
__global__ void __launch_bounds__(256)
    k_bead_pairs_any(const int2* __restrict__ pairs, const int* __restrict__ n_pairs_ptr,
                     const float4* __restrict__ pos, const float4* __restrict__ quat,
                     const float4* __restrict__ tmpl, int n_beads, float3 L, float3 invL, BeadPot pot,
                     float cut2, int zero_beyond, float4* __restrict__ out_F,
                     float4* __restrict__ out_ti, float4* __restrict__ out_tj,
                     const int* __restrict__ sel, const int* __restrict__ sel_count) {
    __shared__ float4 sT[kMaxBeads + 1];
    __shared__ float4 sN[2 * (kMaxBeads + kPadBeads)];  // 2 float4 per template bead
    pdl_wait();
    const int n_pairs = sel ? *sel_count : *n_pairs_ptr;
    // a CTA with no pair (most of them when only the few fallback pairs are
    // listed) leaves before staging the template
    if ((int64_t)blockIdx.x * (blockDim.x >> 5) >= n_pairs) return;
    load_template(tmpl, n_beads, pot.rc2_test, sT, sN);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warps_per_block = blockDim.x >> 5;
    const int gw = blockIdx.x * warps_per_block + (threadIdx.x >> 5);
    const int nw = gridDim.x * warps_per_block;
    for (int t = gw; t < n_pairs; t += nw) {
        const int p = sel ? sel[t] : t;
        const int2 ij = pairs[p];
        const float4 pi = pos[ij.x], pj = pos[ij.y];
        const float4 qi = quat[ij.x], qj = quat[ij.y];
        const float3 R = min_image(make_float3(pj.x - pi.x, pj.y - pi.y, pj.z - pi.z), L, invL);
        if (R.x * R.x + R.y * R.y + R.z * R.z >= cut2) {
            if (zero_beyond && lane == 0)
                out_F[p] = out_ti[p] = out_tj[p] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        const Mat3 Rr = qmat(qmul(qconj(qi), qj));
        const float3 s = mulT(qmat(qi), R);
        float v[7];
        bead_pair_warp<NP, POT>(s, Rr, sT, sN, n_beads, pot, lane, v);
        if (lane >= 3) continue;
        const Mat3 Ri = qmat(qi);
        const float3 F = make_float3(v[0], v[1], v[2]);
        const float3 T = make_float3(v[3], v[4], v[5]);
        if (lane == 0) {
            const float3 Fs = mul(Ri, F);
            out_F[p] = make_float4(Fs.x, Fs.y, Fs.z, v[6]);
        } else if (lane == 1) {
            const float3 ti = mul(Ri, make_float3(-T.x, -T.y, -T.z));
            out_ti[p] = make_float4(ti.x, ti.y, ti.z, 0.f);
        } else {
            const float3 sxF = cross3(s, F);
            const float3 tj = mul(Ri, make_float3(T.x - sxF.x, T.y - sxF.y, T.z - sxF.z));
            out_tj[p] = make_float4(tj.x, tj.y, tj.z, 0.f);
        }
    }
}

// Column-structured templates (the cube and the cylinder), up to 32 NS beads in
// columns of C.  Every CTA takes an equal contiguous share of the list, 256
// pairs at a time: a thread per pair loads its bodies, forms its frame and
// tests it against the box of body i's columns grown by r_c + r_circ; the pairs
// that can interact go into a queue that the eight warps empty one pair at a
// time (bead_pair_cols), and the threads then rotate their pairs' sums into the
// space frame and store them.  Equal shares and the queue level the work, which
// varies by more than ten between a pair at the cutoff and two touching faces;
// the per-pair geometry costs a 32nd of a warp instead of a fourth.  Measured,
// 32768 cubes at phi = 0.20 in contact (92 thousand pairs): 100 -> 48 us (MD step
// 114 -> 62 us); the kernel before tested a lane's four beads against every column
// near j's bounding sphere and gave every warp its pairs up front.  Bound by
// instruction issue.
// BATCH (no sel): the concatenated pair lists of n_seg systems with this
// template and potential (segs: their lists, bodies, boxes and outputs).
template <int NS, int C, int POT, bool BATCH = false>
__global__ void __launch_bounds__(256, NS <= 5 ? 4 : 3)
    k_bead_cols(const int2* __restrict__ pairs, const int* __restrict__ n_pairs_ptr,
                const float4* __restrict__ pos, const float4* __restrict__ quat,
                const float4* __restrict__ tmpl, int n_beads, BeadCols cols, float3 L, float3 invL,
                BeadPot pot, float cut2, int zero_beyond, float4* __restrict__ out_F,
                float4* __restrict__ out_ti, float4* __restrict__ out_tj,
                const int* __restrict__ sel, const int* __restrict__ sel_count,
                const PairSeg* __restrict__ segs, int n_seg) {
    __shared__ ColShared sc;
    __shared__ float4 s_q[256][3];        // per pair: s, R_rel; then its seven sums
    __shared__ float4 s_buf[8][32 * NS];  // per warp: the packed beads of j
    __shared__ int s_todo[256];
    __shared__ int s_n, s_next;
    // BATCH: each system's first pair (inclusive scan over n_seg <= 32 lanes)
    __shared__ int s_b0[BATCH ? kMaxSeg + 1 : 1];
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int n_pairs;
    if constexpr (BATCH) {
        if (tid < 32) {
            int t = lane < n_seg ? *segs[lane].n_pairs : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += v;
            }
            s_b0[lane + 1] = t;
            if (lane == 0) s_b0[0] = 0;
        }
        __syncthreads();
        n_pairs = s_b0[n_seg];
    } else {
        n_pairs = sel ? *sel_count : *n_pairs_ptr;
    }
    const int share = (n_pairs + (int)gridDim.x - 1) / (int)gridDim.x;
    const int64_t first = (int64_t)blockIdx.x * share;
    if (first >= n_pairs) return;  // nothing left for this CTA
    const int beg = (int)first, end = min(beg + share, n_pairs);
    load_columns(tmpl, cols, sc);
    float tx[NS], ty[NS], tz[NS];  // the lane's template beads lane + 32 m
#pragma unroll
    for (int m = 0; m < NS; ++m) {
        const float4 d = tmpl[min(lane + 32 * m, n_beads - 1)];
        tx[m] = d.x;
        ty[m] = d.y;
        tz[m] = d.z;
    }
    for (int base = beg; base < end; base += 256) {
        if (tid == 0) s_n = s_next = 0;
        __syncthreads();
        // this thread's pair, its system (BATCH: the last k with s_b0[k] <= t)
        const int t = base + tid;
        const bool live = t < end;
        int sg = 0, p = 0;
        if (live) {
            if constexpr (BATCH) {
                int lo = 0, hi = n_seg - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_b0[mid] <= t) lo = mid; else hi = mid - 1;
                }
                sg = lo;
                p = t - s_b0[lo];
            } else {
                p = sel ? sel[t] : t;
            }
        }
        float4 qi = make_float4(1.f, 0.f, 0.f, 0.f);
        float3 sv = make_float3(0.f, 0.f, 0.f);
        bool work = false, store = false;
        if (live) {
            const int2* __restrict__ prs = BATCH ? segs[sg].pairs : pairs;
            const float4* __restrict__ ps = BATCH ? segs[sg].pos : pos;
            const float4* __restrict__ qs = BATCH ? segs[sg].quat : quat;
            const int2 ij = prs[p];
            const float4 pi = ps[ij.x], pj = ps[ij.y], qj = qs[ij.y];
            qi = qs[ij.x];
            const float3 R = min_image(make_float3(pj.x - pi.x, pj.y - pi.y, pj.z - pi.z),
                                       BATCH ? segs[sg].L : L, BATCH ? segs[sg].invL : invL);
            const bool in = R.x * R.x + R.y * R.y + R.z * R.z < cut2;
            store = in || zero_beyond;
            sv = mulT(qmat(qi), R);
            work = in && box_dist2(sv.x, sv.y, sv.z, cols.x_lo, cols.x_hi, cols.y_lo, cols.y_hi, cols.z[0],
                                   cols.z[C - 1]) <= pot.cull2;
            if (work) {
                const Mat3 Rr = qmat(qmul(qconj(qi), qj));
                s_q[tid][0] = make_float4(sv.x, sv.y, sv.z, Rr.m[0]);
                s_q[tid][1] = make_float4(Rr.m[1], Rr.m[2], Rr.m[3], Rr.m[4]);
                s_q[tid][2] = make_float4(Rr.m[5], Rr.m[6], Rr.m[7], Rr.m[8]);
            }
        }
        {
            const unsigned w = __ballot_sync(0xffffffffu, work);
            int at = 0;
            if (lane == 0 && w) at = atomicAdd(&s_n, __popc(w));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (work) s_todo[at + __popc(w & ((1u << lane) - 1u))] = tid;
        }
        __syncthreads();
        const int n_todo = s_n;
        for (;;) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&s_next, 1);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= n_todo) break;
            const int o = s_todo[k];
            const float4 a0 = s_q[o][0], a1 = s_q[o][1], a2 = s_q[o][2];
            float bx[NS], by[NS], bz[NS];
#pragma unroll
            for (int m = 0; m < NS; ++m) {
                const bool bead = lane + 32 * m < n_beads;
                bx[m] = bead ? fmaf(a0.w, tx[m], fmaf(a1.x, ty[m], fmaf(a1.y, tz[m], a0.x))) : 1e18f;
                by[m] = bead ? fmaf(a1.z, tx[m], fmaf(a1.w, ty[m], fmaf(a2.x, tz[m], a0.y))) : 1e18f;
                bz[m] = bead ? fmaf(a2.y, tx[m], fmaf(a2.z, ty[m], fmaf(a2.w, tz[m], a0.z))) : 1e18f;
            }
            float v[7];
            float sum = 0.f;
            if (bead_pair_cols<NS, C, POT>(bx, by, bz, sc, cols, pot, s_buf[warp], lane, v))
                sum = warp_scatter7(v);
            __syncwarp();  // the pair's geometry has been read
            if ((lane & 3) == 0 && lane < 28) reinterpret_cast<float*>(s_q[o])[lane >> 2] = sum;
        }
        __syncthreads();
        if (store) {
            float4 oF = make_float4(0.f, 0.f, 0.f, 0.f), oti = oF, otj = oF;
            if (work) {
                const float4 v0 = s_q[tid][0], v1 = s_q[tid][1];
                const Mat3 Ri = qmat(qi);
                const float3 F = make_float3(v0.x, v0.y, v0.z), T = make_float3(v0.w, v1.x, v1.y);
                const float3 a = mul(Ri, F), b = mul(Ri, make_float3(-T.x, -T.y, -T.z));
                const float3 sxF = cross3(sv, F);
                const float3 c = mul(Ri, make_float3(T.x - sxF.x, T.y - sxF.y, T.z - sxF.z));
                oF = make_float4(a.x, a.y, a.z, v1.z);
                oti = make_float4(b.x, b.y, b.z, 0.f);
                otj = make_float4(c.x, c.y, c.z, 0.f);
            }
            (BATCH ? segs[sg].F : out_F)[p] = oF;
            (BATCH ? segs[sg].ti : out_ti)[p] = oti;
            (BATCH ? segs[sg].tj : out_tj)[p] = otj;
        }
    }
}

BeadPot bead_pot(const rb_system* s) {
    BeadPot p;
    p.rc2 = s->rcut * s->rcut;
    p.sig2 = s->sigma * s->sigma;
    p.eps4 = 4.f * s->eps;
    p.eps24 = 24.f * s->eps;
    p.u_shift = s->u_shift;
    p.kind = s->pot_kind;
    p.hA = s->hphc[0];
    p.hb = s->hphc[1];
    p.hc = s->hphc[2];
    p.hp = s->hphc[3];
    if (s->pot_kind != RB_POT_LJ) {  // the sum of u itself is the energy
        p.eps4 = 1.f;
        p.u_shift = 0.f;
    }
    // |r^2_expanded - r^2| <= a few roundings of values up to (Rc + r_circ)^2
    // + r_circ^2 (b within Rc + r_circ of body i's centre, d within r_circ)
    const float big = (s->Rc + s->r_circ) * (s->Rc + s->r_circ) + s->r_circ * s->r_circ;
    p.rc2_test = p.rc2 + 4e-6f * big;
    // column cull radius r_c + r_circ, widened well past the FP32 rounding of
    // the test's squared distance (a few ulps of values below (Rc + r_circ)^2)
    const float rct = (sqrtf(p.rc2_test) + s->r_circ) * 1.0001f + 1e-3f;
    p.cull2 = rct * rct;
    return p;
}

template <int NP, int POT>
static rb_status launch_beads_any(rb_system* s, float cut2, int zero_beyond, const int* sel) {
    static int occ = 0;
    if (occ == 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bead_pairs_any<NP, POT>, 256, 0);
        if (occ <= 0) occ = 1;
    }
    const float3 L = make_float3(s->box[0], s->box[1], s->box[2]);
    const float3 invL = make_float3(1.f / s->box[0], 1.f / s->box[1], 1.f / s->box[2]);
    const int grid = pair_grid(s, 8, s->num_sms * occ);  // a warp per pair, 8 per CTA
    RB_CUDA(launch_pdl(k_bead_pairs_any<NP, POT>, grid, 256, 0, s->stream, s->pl.pairs, s->pl.n_pairs,
                       s->pos, s->quat, s->tmpl_dev, s->n_beads, L, invL, bead_pot(s), cut2, zero_beyond,
                       s->pair_F, s->pair_ti, s->pair_tj, sel, s->fallback_count));
    return RB_OK;
}

// grid: one wave of CTAs (their shares are equal), fewer for a small system:
// eight pairs per CTA, one per warp
template <int NS, int C, int POT>
static rb_status launch_beads_cols(rb_system* s, float cut2, int zero_beyond, const int* sel) {
    static int occ = 0;
    if (occ == 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bead_cols<NS, C, POT>, 256, 0);
        if (occ <= 0) occ = 1;
    }
    const float3 L = make_float3(s->box[0], s->box[1], s->box[2]);
    const float3 invL = make_float3(1.f / s->box[0], 1.f / s->box[1], 1.f / s->box[2]);
    const int grid = pair_grid(s, 8, s->num_sms * occ);
    RB_CUDA(launch_pdl(k_bead_cols<NS, C, POT>, grid, 256, 0, s->stream, s->pl.pairs, s->pl.n_pairs,
                       s->pos, s->quat, s->tmpl_dev, s->n_beads, s->cols, L, invL, bead_pot(s), cut2,
                       zero_beyond, s->pair_F, s->pair_ti, s->pair_tj, sel, s->fallback_count,
                       (const PairSeg*)nullptr, 0));
    return RB_OK;
}

template <int NS, int C, int POT>
static rb_status launch_beads_batch(const rb_system* s, const PairSeg* segs, int n_seg, int grid_hint,
                                    cudaStream_t st) {
    static int occ = 0;
    if (occ == 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bead_cols<NS, C, POT, true>, 256, 0);
        if (occ <= 0) occ = 1;
    }
    const int grid = std::max(1, std::min(grid_hint, s->num_sms * occ));
    RB_CUDA(launch_pdl(k_bead_cols<NS, C, POT, true>, grid, 256, 0, st, (const int2*)nullptr,
                       (const int*)nullptr, (const float4*)nullptr, (const float4*)nullptr,
                       s->tmpl_dev, s->n_beads, s->cols, make_float3(0.f, 0.f, 0.f),
                       make_float3(0.f, 0.f, 0.f), bead_pot(s), s->Rc * s->Rc, 1,
                       (float4*)nullptr, (float4*)nullptr, (float4*)nullptr, (const int*)nullptr,
                       (const int*)nullptr, segs, n_seg));
    return RB_OK;
}

// The bead sum over the pair lists of several systems whose template and
// potential are those of `like` (the caller groups them).  Batched kernels
// exist for the column templates of the built-in cube (125 beads in columns
// of 5) and cylinder (152 beads in columns of 8); for other templates *done
// is false and nothing is launched.
rb_status bead_pairs_batch_async(const rb_system* like, const PairSeg* segs_dev, int n_seg,
                                 int grid_hint, cudaStream_t st, bool* done) {
    *done = false;
    if (n_seg < 1 || n_seg > kMaxSeg) return fail(RB_EINVAL, "batch of 1 to 32 systems");
    const bool lj = like->pot_kind == RB_POT_LJ;
    if (like->cols.len == 5 && like->n_beads <= 128) {
        *done = true;
        return lj ? launch_beads_batch<4, 5, 0>(like, segs_dev, n_seg, grid_hint, st)
                  : launch_beads_batch<4, 5, 1>(like, segs_dev, n_seg, grid_hint, st);
    }
    if (like->cols.len == 8 && like->n_beads > 128 && like->n_beads <= 160) {
        *done = true;
        return lj ? launch_beads_batch<5, 8, 0>(like, segs_dev, n_seg, grid_hint, st)
                  : launch_beads_batch<5, 8, 1>(like, segs_dev, n_seg, grid_hint, st);
    }
    return RB_OK;
}

template <int C, int POT>
static rb_status launch_beads_len(rb_system* s, float cut2, int zero_beyond, const int* sel) {
    if (s->n_beads <= 128) return launch_beads_cols<4, C, POT>(s, cut2, zero_beyond, sel);
    if (s->n_beads <= 160) return launch_beads_cols<5, C, POT>(s, cut2, zero_beyond, sel);
    return launch_beads_cols<8, C, POT>(s, cut2, zero_beyond, sel);
}

template <int POT>
static rb_status launch_beads_pot(rb_system* s, float cut2, int zero_beyond, const int* sel) {
    if (s->cols.len == 5) return launch_beads_len<5, POT>(s, cut2, zero_beyond, sel);
    if (s->cols.len == 8) return launch_beads_len<8, POT>(s, cut2, zero_beyond, sel);
    if (s->n_beads <= 128) return launch_beads_any<2, POT>(s, cut2, zero_beyond, sel);
    if (s->n_beads <= 192) return launch_beads_any<3, POT>(s, cut2, zero_beyond, sel);
    return launch_beads_any<4, POT>(s, cut2, zero_beyond, sel);
}

static rb_status launch_beads(rb_system* s, float cut2, int zero_beyond, const int* sel) {
    if (s->pot_kind == RB_POT_LJ) return launch_beads_pot<0>(s, cut2, zero_beyond, sel);
    return launch_beads_pot<1>(s, cut2, zero_beyond, sel);
}

// The pairs the network kernel listed (closer than rho_min) by the bead sum.
rb_status bead_fallback_async(rb_system* s) {
    if (!(s->nn_fallback_rho > 0.f)) {
        RB_CUDA(cudaMemsetAsync(s->fallback_count, 0, sizeof(int), s->stream));
        return RB_OK;
    }
    const float r = std::min(s->nn_fallback_rho, s->Rc);
    return launch_beads(s, r * r, 0, s->fb_list);
}

rb_status bead_pairs_async(rb_system* s) { return launch_beads(s, s->Rc * s->Rc, 1, nullptr); }

void bead_columns(float4* t, int n, BeadCols* c) {
    *c = BeadCols();
    if (n < 1 || n > kMaxBeads) return;
    // group by exact (x, y), in order of first appearance (fixed-size arrays:
    // no allocation, so the allocation-free entry point can call this)
    float gx[kMaxBeads], gy[kMaxBeads];
    int gid[kMaxBeads], gsize[kMaxBeads];
    int ng = 0;
    for (int k = 0; k < n; ++k) {
        int g = 0;
        while (g < ng && !(gx[g] == t[k].x && gy[g] == t[k].y)) ++g;
        if (g == ng) {
            gx[ng] = t[k].x;
            gy[ng] = t[k].y;
            gsize[ng++] = 0;
        }
        gid[k] = g;
        ++gsize[g];
    }
    const int len = gsize[0];
    if ((len != 5 && len != 8) || ng * len != n || ng > kMaxBeads / 5) return;
    float4 out[kMaxBeads];
    for (int g = 0; g < ng; ++g) {
        if (gsize[g] != len) return;
        float4* col = out + g * len;
        int m = 0;
        for (int k = 0; k < n; ++k)
            if (gid[k] == g) col[m++] = t[k];
        for (int i = 1; i < len; ++i)  // z ascending
            for (int j = i; j > 0 && col[j].z < col[j - 1].z; --j) std::swap(col[j], col[j - 1]);
        for (int i = 0; i < len; ++i) {
            if (col[i].z != out[i].z) return;            // same z values in every column
            if (i > 0 && col[i].z == col[i - 1].z) return;
        }
    }
    c->n_cols = ng;
    c->len = len;
    for (int m = 0; m < len; ++m) c->z[m] = out[m].z;
    c->x_lo = c->x_hi = gx[0];
    c->y_lo = c->y_hi = gy[0];
    for (int g = 1; g < ng; ++g) {
        c->x_lo = std::min(c->x_lo, gx[g]);
        c->x_hi = std::max(c->x_hi, gx[g]);
        c->y_lo = std::min(c->y_lo, gy[g]);
        c->y_hi = std::max(c->y_hi, gy[g]);
    }
    for (int k = 0; k < n; ++k) t[k] = out[k];
}

}  // namespace rb
