// Kernels of the reverse-time (adjoint) march: the transposed pieces of one step, each a thin
// launch around a body of adjoint.cuh (the derivation is at the top of that file).  The type-1
// and type-2 transforms of the reverse step run through a standalone NUFFT plan on the springs.
//
// Adjoint state (internal spring order):
//   sb   ring of m_max + 1 slots x M: sigmabar^q in slot q mod (m_max + 1)
//   Sb   ring of W slots x (K + 1) complex: Sbar^q in slot q mod W
//   ab, apb  alphabar, alpha'bar (K + 1 complex)
// Every launch has one writer per output element and sums in a fixed order: no atomics, and the
// gradient is the same bit for bit from run to run.
#include <cuda_runtime.h>

#include <cstdint>

#include "adjoint.cuh"
#include "internal.h"
#include "range.cuh"

namespace wave1d {

// receivers' transposed readout over the receiver weights regrouped by source (m >= 0: the m = 0 terms
// of sources closer than dt included): one thread per source and eighth of the m (blockIdx.y: m = y,
// y + 8, ..), so each ring entry has one writer, which meets the receivers in order
__global__ void k_adj_receivers(int64_t M, int ring, int64_t n, const int64_t* __restrict__ ptr,
                                const int32_t* __restrict__ rcv, const int32_t* __restrict__ mrange,
                                const int64_t* __restrict__ woff, const double* __restrict__ w,
                                const double* __restrict__ ubar, double* sb) {
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < M; l += (int64_t)gridDim.x * blockDim.x)
        adj::receivers_T_part(l, (int)blockIdx.y, ptr, rcv, mrange, woff, w, ubar, n + 1, ring,
                              [&](int s, double v) { sb[(int64_t)s * M + l] += v; });
}

// transposed block solve, one thread per member position e of blk_members (blk_of[e] = its
// block), then the step's gradient terms and the adjoints of the local sum and of u_H:
//   grad_j += rhsbar_j (sigma_j^{n+1} + g_j^{n+1}) / beta_j   (g: a forcing that does not scale
//             with beta; for the incident wave g = beta f is part of rhs and the term is
//             rhsbar_j sigma_j^{n+1} / beta_j),
//   gbar_j^{n+1} = -rhsbar_j,  cbar_j = -beta_j rhsbar_j / 2,  u_Hbar_j = -beta_j rhsbar_j.
// sigma_next, g_next and gbar_next are rows in caller order; g_next, grad and gbar_next may be null.
// sigbar: the ring slot of sigmabar^{n+1} itself (k_adj_gather clears it afterwards).
__global__ void k_adj_solve(DevPlan P, const int32_t* __restrict__ blk_of, const double* __restrict__ sigbar,
                            const double* __restrict__ sigma_next, const double* __restrict__ g_next, double* grad,
                            double* __restrict__ gbar_next, double* cbar, double* uHbar) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < P.M; e += (int64_t)gridDim.x * blockDim.x) {
        const int b = blk_of[e];
        const int64_t m0 = P.blk_ptr[b];
        const int s = (int)(P.blk_ptr[b + 1] - m0);
        const double rb = adj::solve_T(P.inv + P.blk_inv_off[b], P.blk_members, m0, s, (int)(e - m0), sigbar);
        const int j = P.blk_members[e];
        const int jc = P.perm[j];
        const double bj = P.beta[j];
        if (grad) grad[j] += rb * (g_next ? sigma_next[jc] + g_next[jc] : sigma_next[jc]) / bj;
        if (gbar_next) gbar_next[jc] = -rb;
        cbar[j] = -0.5 * bj * rb;
        uHbar[j] = -bj * rb;
    }
}

// transposed local sum of the springs, one warp per row l (the row's items read in the transposed
// direction, Q_m being symmetric in the pair), in the compensated FP32 arithmetic of the forward
// local sum: each lane accumulates its slices into the warp's shared pairs acc[m][lane] (row
// stride kAdjAccStride), eight slices' weights in flight, then lane i adds m = i, i + 32, ... over the
// 32 lanes in lane order, in three floats (acc3_add, more than FP64's bits), and adds the result to
// sigmabar^{n+1-m}[l].  Dynamic shared memory: warps per block x (m_max + 1) x kAdjAccStride float pairs.
// With the lanes' sums in FP64 (4 x 32 instructions a row and m of the FP64 pipe) and one slice in flight
// it took 137 us for 1.1e7 weights; now 48 (45 with the sums as one pair, which holds less).
constexpr int kAdjAccStride = 33;

__global__ void k_adj_local(DevPlan P, int64_t n, const double* __restrict__ cbar, double* sb) {
    extern __shared__ float2 adj_acc[];
    const int lane = threadIdx.x & 31;
    const int nm = P.m_max + 1;
    float2* acc = adj_acc + (int64_t)(threadIdx.x >> 5) * nm * kAdjAccStride;
    const int64_t l = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (l >= P.M) return;                                  // the whole warp: l is the warp's row
    for (int m = 0; m < nm; m++) acc[m * kAdjAccStride + lane] = make_float2(0.f, 0.f);
    for (int64_t it = P.l_item_ptr[l]; it < P.l_item_ptr[l + 1]; it++) {
        float ch, cl;
        adj::split_pair(cbar[P.l_src[it * 32 + lane]], ch, cl);
        const float4* w = (const float4*)(P.l_w + 2 * P.l_wbase[it]) + lane;     // slices 2i, 2i + 1
        float2* a = acc + (P.l_mfirst + P.l_s0[it]) * kAdjAccStride + lane;
        const int len = P.l_len[it];
        auto mac = [&](int t, float wh, float wl) {
            if (wh != 0.0f) {                              // zero: padding, maybe past the last m
                float2 v = a[t * kAdjAccStride];
                adj::pair_mac(v.x, v.y, wh, wl, ch, cl);
                a[t * kAdjAccStride] = v;
            }
        };
        int t = 0;
        for (; t + 8 <= len; t += 8) {
            float4 q[4];
#pragma unroll
            for (int u = 0; u < 4; u++) q[u] = __ldcs(w + 32 * ((t >> 1) + u));
#pragma unroll
            for (int u = 0; u < 4; u++) {
                mac(t + 2 * u, q[u].x, q[u].y);
                mac(t + 2 * u + 1, q[u].z, q[u].w);
            }
        }
        for (; t < len; t += 2) {
            const float4 q = __ldcs(w + 32 * (t >> 1));
            mac(t, q.x, q.y);
            mac(t + 1, q.z, q.w);
        }
    }
    __syncwarp();
    for (int m = lane; m < nm; m += 32) {
        float sh = 0.f, sm = 0.f, sl = 0.f;
        for (int i = 0; i < 32; i++) {
            const float2 a = acc[m * kAdjAccStride + i];
            rs::acc3_add(sh, sm, sl, a.x, a.y);
        }
        const double s = rs::acc3_value(sh, sm, sl);
        if (s != 0.0) sb[(int64_t)adj::slot(n + 1 - m, P.ring) * P.M + l] += s;
    }
}

size_t adj_local_smem(int m_max, int warps) { return (size_t)warps * (m_max + 1) * kAdjAccStride * sizeof(float2); }

// out[i] = in[perm[i]] (spring order -> NUFFT point order); clear: the ring slot of sigmabar^{n+1}, read by
// the solve, becomes sigma^{n-m_max}'s
__global__ void k_adj_gather(int64_t M, const int64_t* __restrict__ perm, const double* __restrict__ in,
                             double* __restrict__ out, double* __restrict__ clear) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        out[i] = in[perm[i]];
        if (clear) clear[i] = 0.0;
    }
}

// acc[perm[i]] += in[i] (NUFFT point order -> spring order; perm is a permutation)
__global__ void k_adj_scatter_add(int64_t M, const int64_t* __restrict__ perm, const double* __restrict__ in,
                                  double* __restrict__ acc) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
        acc[perm[i]] += in[i];
}

// e^{i k x_r} of the receivers, [r][k], once per call (a sine and cosine of FP64 are some 200 instructions of
// the FP64 pipe: 26 us a step for eight receivers)
__global__ void k_adj_receiver_waves(int K, const double* __restrict__ xr, int64_t R, double2* __restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > K) return;
    for (int64_t r = blockIdx.y; r < R; r += gridDim.y) {
        const double a = (double)k * xr[r];
        out[r * (K + 1) + k] = make_double2(cos(a), sin(a));
    }
}

// alphabar_k += w_k (2 pi S1_k + sum_r ubar_r e^{i k x_r}) (adj::modes_in); waves may be null (too many
// receivers for the table): the waves are then formed here
__global__ void k_adj_modes_in(int K, const double* __restrict__ S1, const double* __restrict__ xr,
                               const double2* __restrict__ waves, const double* __restrict__ ubar, int64_t R,
                               double* ab) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > K) return;
    if (!waves) {
        adj::modes_in(k, S1, xr, ubar, R, ab);
        return;
    }
    const double two_pi = 6.283185307179586476925286766559, wk = k == 0 ? 1.0 : 2.0;
    double re = two_pi * S1[2 * k], im = two_pi * S1[2 * k + 1];
#pragma unroll 4
    for (int64_t r = 0; r < R; r++) {
        const double2 e = __ldg(waves + r * (K + 1) + k);
        const double u = __ldg(ubar + r);
        re = fma(u, e.x, re);
        im = fma(u, e.y, im);
    }
    ab[2 * k] = fma(wk, re, ab[2 * k]);
    ab[2 * k + 1] = fma(wk, im, ab[2 * k + 1]);
}

// transposed projection, grid part: a block per rolled-off point (cf. adj::rbc_grid_T; the block's sum
// in a fixed order)
__global__ void __launch_bounds__(256) k_adj_rbc_grid(int K, int npts, const int32_t* __restrict__ idx,
                                                      const double* __restrict__ tw2K, const double* __restrict__ phi,
                                                      const double* __restrict__ dphi, const double* __restrict__ ab,
                                                      const double* __restrict__ apb, double* __restrict__ uvbar) {
    __shared__ double red[2][8];
    const int pt = blockIdx.x;
    double su = 0.0, sv = 0.0;
    adj::rbc_grid_sum(idx[pt], K, 1 + threadIdx.x, blockDim.x, tw2K, ab, apb, su, sv);
    for (int o = 16; o > 0; o >>= 1) {
        su += __shfl_xor_sync(0xffffffffu, su, o);
        sv += __shfl_xor_sync(0xffffffffu, sv, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = su;
        red[1][threadIdx.x >> 5] = sv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        su = ab[0];
        sv = apb[0];
        for (int w = 0; w < 8; w++) {
            su += red[0][w];
            sv += red[1][w];
        }
        adj::rbc_grid_values(K, su, sv, phi[pt], dphi[pt], uvbar + 2 * pt);
    }
}

// mode part (cf. adj::rbc_update_T): eight lanes per mode, each every eighth point, a fixed tree
__global__ void __launch_bounds__(256) k_adj_rbc_update(int K, int npts, const int32_t* __restrict__ idx,
                                                        const double* __restrict__ tw2K,
                                                        const double* __restrict__ uvbar, double* ab, double* apb) {
    const int k = blockIdx.x * 32 + (threadIdx.x >> 3), q = threadIdx.x & 7;
    adj::Complex u = {0.0, 0.0}, v = {0.0, 0.0};
    if (k < K) adj::rbc_update_sum(k, K, q, 8, npts, idx, tw2K, uvbar, u, v);
    for (int o = 4; o > 0; o >>= 1) {
        u.x += __shfl_xor_sync(0xffffffffu, u.x, o);
        u.y += __shfl_xor_sync(0xffffffffu, u.y, o);
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    if (q == 0 && k <= K) adj::rbc_update_values(k, K, u, v, ab, apb);
}

// rotation and FIR transposed, one thread per mode and kModeTaps of the W taps (blockIdx.y; adj::modes_T_taps).
// One thread per mode took 33 us for 36 taps, a chain of ring reads and writes.
__global__ void k_adj_modes(int K, int W, int64_t n, const double* __restrict__ rot, const double* __restrict__ pq,
                            const double* __restrict__ ab, const double* __restrict__ apb, double* __restrict__ ab_out,
                            double* __restrict__ apb_out, double* Sb, double* __restrict__ a2) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k <= K) adj::modes_T_taps(k, K + 1, W, n, blockIdx.y * adj::kModeTaps, rot, pq, ab, apb, ab_out, apb_out, Sb, a2);
}

// Checkpoint restore (wave1d_adjoint_checkpointed): the float-pair copy of the density ring
// (both halves of its doubled ring) from the FP64 ring, the same split store_sigma makes, so a
// march resumed from a checkpoint of the FP64 ring alone repeats the original bit for bit
__global__ void k_ck_sig2(int64_t n, const double* __restrict__ sig, float2* __restrict__ sig2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = sig[i];
        const float hi = (float)v;
        const float2 pr = make_float2(hi, (float)(v - (double)hi));
        sig2[i] = pr;
        sig2[i + n] = pr;
    }
}

// the device step counter of a restored march
__global__ void k_ck_step(int64_t* step, int64_t n) {
    step[0] = n;
    step[1] = 0;
}

}  // namespace wave1d
