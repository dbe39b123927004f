// Local sum of plans without pair lists with FP32 spreading and interpolation (opts.precision = 1): the
// fold and the pairs chunk by chunk in shared memory.  The FP64 form (range.cu) makes the same e-vectors
// bit for bit but sums the pairs in another order, and here the order counts: the FP32 passes round every
// grid value and u_H to 2^-24, so a density that differs by 1e-12 flips roundings and moves results by 1e-7
// of the field.  A mixed march keeps this order of sums, and its results stay the same bit for bit.
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"
#include "phases.cuh"
#include "range.cuh"
#include "range_dev.cuh"

namespace wave1d {

namespace {
constexpr int kRsChunk = 32;      // sources per chunk (one per lane of warp 0 in the set-up)
constexpr int kRsIvCap = 32;      // intervals whose e-vectors are held at once (3 blocks of 256 threads per SM)
// one interval's row of e-vector records: 32 records of 12 floats and 4 floats of padding, so the
// rows of consecutive intervals start 4 banks apart (threads of a warp read the records of the 2-3
// intervals their distances fall in)
constexpr int kRsRow = kRsChunk * rs::kERecord + 4;
}  // namespace

// shared memory of k_rs_local (bytes): e-vector rows, the chunk's densities, the interval table
size_t rs_local_smem(int nint, int nm) {
    return (size_t)kRsIvCap * kRsRow * sizeof(float) + (size_t)nm * kRsChunk * sizeof(float2) +
           (size_t)4 * nint * sizeof(float);
}

// ---------------------------------------------------------------------------------------------
// Local explicit sum, one block per kRsTargets consecutive targets (thread t: target j0 + t).
// The block's sources (window [wlo, whi) of extended indices) are visited twice over as
// "left" sources (strictly left of the target: d = x_j - x_e) and "right" sources (at or right
// of it: d = x_e - x_j), in chunks of 32.  Per chunk:
//   1. once per 8 chunks, one thread per source: its position on the block grid (range.cuh) and
//      the interval range its distances to the block's targets fall in;
//   2. the chunk's densities sigma^{n+1-m}, m = 1 .. m_max, into shared memory;
//   3. for each interval of the chunk's range (at most kRsIvCap at a time), one warp folds the
//      densities of all 32 sources into their e-vectors (coefficients are warp-uniform loads);
//   4. each thread walks the 32 sources: z on the tracked interval of the side (it moves by about
//      one interval from one source to the next), and the polynomial of the source's e-vector at z
//      into the thread's compensated accumulator.
// Which side counts a source is decided by index: e < lb_j (the first spring at x_j's position) is
// strictly left.  Q_m is continuous across the breakpoints other than dt, so a pair within
// rounding of one takes either neighbouring interval's polynomial; at dt the spring's FP64 window
// of near sources decides (near_side in range.cuh).
// ---------------------------------------------------------------------------------------------
template <int S>
__device__ __forceinline__ void rs_pairs(const float* sE, const float4* sMeta, const float* ivt, const int* cell,
                                         float cscale, int nint, int iv_dt, int k0, int k1, int W0, int W1, int lbj,
                                         int nbl, int nbc, float bh, float bl, rs::Track& tr, float& a0h, float& a0l,
                                         float& a1h, float& a1l) {
    for (int k = k0; k < k1; k += 2) {
        // the record and z of sources k and k + 1 (null where the pair does not count in this
        // window), then both polynomials as independent chains.  z is computed for every slot
        // (the group's meta holds 256 defined entries, so slot k + 1 >= k1 reads one); only a
        // pair that counts moves the tracked interval.
        const float* rec[2];
        float zh[2], zl[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int kk = k + u;
            const float4 mt = sMeta[kk];
            const int e = __float_as_int(mt.z), lohi = __float_as_int(mt.w);
            const int lo = max(lohi & 0x7fff, W0), hi = min(lohi >> 16, W1);
            const bool valid = kk < k1 && lo <= hi && (S < 0 ? e < lbj : e >= lbj);
            float h0, l0;
            rs::z_of<S>(tr, mt.x, mt.y, h0, l0);
            if (valid && fabsf(h0) > rs::kZTol) rs::walk<S>(ivt, cell, cscale, nint, bh, bl, mt.x, mt.y, tr, h0, l0);
            if (valid && (lohi & 0x8000))
                rs::near_side<S>(ivt, iv_dt, (unsigned)(e - nbl) < (unsigned)nbc, bh, bl, mt.x, mt.y, tr, h0, l0);
            const bool ok = valid && fabsf(h0) <= rs::kZTol && tr.iv >= lo && tr.iv <= hi;
            rec[u] = ok ? sE + (tr.iv - W0) * kRsRow + kk * rs::kERecord : nullptr;
            zh[u] = h0;
            zl[u] = l0;
        }
        if (rec[0]) rs::evec_eval(rec[0], zh[0], zl[0], a0h, a0l);
        if (rec[1]) rs::evec_eval(rec[1], zh[1], zl[1], a1h, a1l);
    }
}

// The pairs of one side for one target in a chunk whose interval range takes several windows of
// e-vectors: the sources in walk order (right: k ascending; left: k descending, so the distance
// grows along both) from the thread's cursor cur, evaluated in the window that holds their
// interval.  A source whose interval lies beyond the window stops the walk there (the tracked
// interval kept, the cursor on it) until the next window; so each source is walked once per
// thread and chunk, not once per window.  Sources beyond delta end the side.  k0 .. k1 - 1: the
// side's sources in the chunk; par alternates the two accumulators.
template <int S>
__device__ __forceinline__ void rs_pairs_cursor(const float* sE, const float4* sMeta, const float* ivt, const int* cell,
                                                float cscale, int nint, int iv_dt, int k0, int k1, int& cur, int W0,
                                                int W1, int lbj, int nbl, int nbc, float bh, float bl, rs::Track& tr,
                                                int& par, float& a0h, float& a0l, float& a1h, float& a1l) {
    while (S > 0 ? cur < k1 : cur >= k0) {
        const int k = cur;
        const float4 mt = sMeta[k];
        const int e = __float_as_int(mt.z), lohi = __float_as_int(mt.w);
        const int lo = lohi & 0x7fff, hi = lohi >> 16;
        if (lo > hi || (S < 0 ? e >= lbj : e < lbj)) {
            cur += S;
            continue;
        }
        if (lo > W1) break;                                   // its interval lies in a later window
        float zh, zl;
        rs::z_of<S>(tr, mt.x, mt.y, zh, zl);
        if (fabsf(zh) > rs::kZTol) rs::walk<S>(ivt, cell, cscale, nint, bh, bl, mt.x, mt.y, tr, zh, zl);
        if (lohi & 0x8000)
            rs::near_side<S>(ivt, iv_dt, (unsigned)(e - nbl) < (unsigned)nbc, bh, bl, mt.x, mt.y, tr, zh, zl);
        if (tr.iv > W1 && fabsf(zh) <= rs::kZTol) break;     // a later window
        if (fabsf(zh) <= rs::kZTol && tr.iv >= lo && tr.iv <= hi && tr.iv >= W0) {
            const float* rec = sE + (tr.iv - W0) * kRsRow + k * rs::kERecord;
            if (par) rs::evec_eval(rec, zh, zl, a1h, a1l);
            else rs::evec_eval(rec, zh, zl, a0h, a0l);
            par ^= 1;
        } else if (zh > rs::kZTol && tr.iv == nint - 1) {
            cur = S > 0 ? k1 : k0 - 1;                         // beyond delta, and the rest farther
            break;
        }
        cur += S;
    }
}

// The pairs of one side for one target in a chunk where e-vectors would hardly be shared (the
// chunk's interval range holds more than twice as many (source, interval) e-vectors as it has
// pairs, as where springs lie farther apart than the intervals are wide): each pair folds its own
// source's densities on its interval (the same e-vector, bit for bit, as the shared fold) and
// evaluates it, with no interval windows.  Sources k0 .. k1 - 1 of the chunk.
template <int S>
__device__ __forceinline__ void rs_direct(const float4* sMeta, const float2* sSig, const float* ivt, const int* cell,
                                          float cscale, int nint, int iv_dt, const float4* __restrict__ coef,
                                          const int32_t* __restrict__ mr, int nm, int k0, int k1, int lbj, int nbl,
                                          int nbc, float bh, float bl, rs::Track& tr, float& a0h, float& a0l,
                                          float& a1h, float& a1l) {
    for (int k = k0; k < k1; k++) {
        const float4 mt = sMeta[k];
        const int e = __float_as_int(mt.z), lohi = __float_as_int(mt.w);
        const int lo = lohi & 0x7fff, hi = lohi >> 16;
        if (lo > hi || (S < 0 ? e >= lbj : e < lbj)) continue;
        float zh, zl;
        rs::z_of<S>(tr, mt.x, mt.y, zh, zl);
        if (fabsf(zh) > rs::kZTol) rs::walk<S>(ivt, cell, cscale, nint, bh, bl, mt.x, mt.y, tr, zh, zl);
        if (lohi & 0x8000)
            rs::near_side<S>(ivt, iv_dt, (unsigned)(e - nbl) < (unsigned)nbc, bh, bl, mt.x, mt.y, tr, zh, zl);
        if (!(fabsf(zh) <= rs::kZTol && tr.iv >= lo && tr.iv <= hi)) continue;
        rs::EVec ev;
        rs::evec_zero(ev);
        const int m0 = __ldg(mr + 2 * tr.iv), m1 = __ldg(mr + 2 * tr.iv + 1);
        const float4* c = coef + (size_t)tr.iv * nm * 3;
        const int kk = k & (kRsChunk - 1);
#pragma unroll 1
        for (int m = m0; m <= m1; m++) {
            const float2 sg = sSig[m * kRsChunk + kk];
            const float4 c01 = __ldg(c + 3 * m), c23 = __ldg(c + 3 * m + 1), c47 = __ldg(c + 3 * m + 2);
            rs::acc_mac(ev.e0h, ev.e0l, c01.x, c01.y, sg.x, sg.y);
            rs::acc_mac(ev.e1h, ev.e1l, c01.z, c01.w, sg.x, sg.y);
            ev.e2 = rs::fma_(c23.y, sg.x, rs::fma_(c23.x, sg.x, ev.e2));
            ev.e3 = rs::fma_(c23.w, sg.x, rs::fma_(c23.z, sg.x, ev.e3));
            ev.e4 = rs::fma_(c47.x, sg.x, ev.e4);
            ev.e5 = rs::fma_(c47.y, sg.x, ev.e5);
            ev.e6 = rs::fma_(c47.z, sg.x, ev.e6);
            ev.e7 = rs::fma_(c47.w, sg.x, ev.e7);
        }
        if (k & 1) rs::evec_eval_v(ev, zh, zl, a1h, a1l);
        else rs::evec_eval_v(ev, zh, zl, a0h, a0l);
    }
}

// One side of one target in a block whose targets lie farther apart than two window widths (each
// target meets few of the block's sources): the thread walks its own sources nearest first (left:
// e = lb_j - 1, lb_j - 2, ..; right: e = lb_j, lb_j + 1, ..) until they lie beyond delta, with the
// shared path's per-source data (position on the block grid, interval range over the block, the
// walk and the near/far rule) and one e-vector per pair folded from the density ring itself; no
// shared staging, no barriers.
template <int S>
__device__ __forceinline__ void rs_sparse_side(const DevPlan& P, const RangeDev& R, const float* ivt, float cscale,
                                               rs::Grid G, double xa, double span, double xj, int64_t n, int wlo,
                                               int whi, int lbj, int nbl, int nbc, float bh, float bl, rs::Track& tr,
                                               float& a0h, float& a0l, float& a1h, float& a1l) {
    const double reach = R.delta * (1.0 + 8.0 * rs::kRangeMargin);
    const float4* coef = (const float4*)R.coef;
    for (int q = 0;; q++) {
        const int e = S > 0 ? lbj + q : lbj - 1 - q;
        if (S > 0 ? e >= whi : e < wlo) break;
        const double xe = rs_xext(P, e);
        if (!((S > 0 ? xe - xj : xj - xe) < reach)) break;     // the farther ones lie farther still
        const double xr = xe - xa;
        const int lohi = rs::source_range(xr, S < 0, span, R.delta, P.dt, R.bp2, R.cell, cscale, R.nint);
        const int lo = lohi & 0x7fff, hi = lohi >> 16;
        if (lo > hi) continue;
        float h, l;
        rs::grid_split(xr, G, h, l);
        float zh, zl;
        rs::z_of<S>(tr, h, l, zh, zl);
        if (fabsf(zh) > rs::kZTol) rs::walk<S>(ivt, R.cell, cscale, R.nint, bh, bl, h, l, tr, zh, zl);
        if (lohi & 0x8000) rs::near_side<S>(ivt, R.iv_dt, (unsigned)(e - nbl) < (unsigned)nbc, bh, bl, h, l, tr, zh, zl);
        if (!(fabsf(zh) <= rs::kZTol && tr.iv >= lo && tr.iv <= hi)) continue;
        const int64_t sp = rs_spring(e, P.M);
        rs::EVec ev;
        rs::evec_zero(ev);
        const int m0 = __ldg(R.mr + 2 * tr.iv), m1 = __ldg(R.mr + 2 * tr.iv + 1);
        const float4* c = coef + (size_t)tr.iv * R.nm * 3;
#pragma unroll 1
        for (int m = m0; m <= m1; m++) {
            const float2 sg = __ldg((const float2*)P.sig2 + (int64_t)ring_slot(n + 1 - m, P.ring) * P.M + sp);
            const float4 c01 = __ldg(c + 3 * m), c23 = __ldg(c + 3 * m + 1), c47 = __ldg(c + 3 * m + 2);
            rs::acc_mac(ev.e0h, ev.e0l, c01.x, c01.y, sg.x, sg.y);
            rs::acc_mac(ev.e1h, ev.e1l, c01.z, c01.w, sg.x, sg.y);
            ev.e2 = rs::fma_(c23.y, sg.x, rs::fma_(c23.x, sg.x, ev.e2));
            ev.e3 = rs::fma_(c23.w, sg.x, rs::fma_(c23.z, sg.x, ev.e3));
            ev.e4 = rs::fma_(c47.x, sg.x, ev.e4);
            ev.e5 = rs::fma_(c47.y, sg.x, ev.e5);
            ev.e6 = rs::fma_(c47.z, sg.x, ev.e6);
            ev.e7 = rs::fma_(c47.w, sg.x, ev.e7);
        }
        if (q & 1) rs::evec_eval_v(ev, zh, zl, a1h, a1l);
        else rs::evec_eval_v(ev, zh, zl, a0h, a0l);
    }
}

__global__ void __launch_bounds__(kRsTargets, 3) k_rs_local(DevPlan P, RangeDev R) {
    extern __shared__ __align__(16) float rs_sm[];
    float* sE = rs_sm;
    float2* sSig = (float2*)(sE + kRsIvCap * kRsRow);
    float* sIv = (float*)(sSig + (size_t)R.nm * kRsChunk);
    // per source of a group of kRsTargets sources (8 chunks): (h, l, extended index, packed
    // interval range), and the interval union of each chunk
    __shared__ float4 sMeta[kRsTargets];
    __shared__ int sU[2][kRsTargets / kRsChunk];
    // targets' positions relative to the first (float, sorted), and per chunk an estimate of its
    // pairs (sources' targets within delta) for the choice between shared and per-pair e-vectors
    __shared__ float sT[kRsTargets];
    __shared__ int sP[kRsTargets / kRsChunk];

    const int64_t M = P.M;
    const int64_t n = load_step(P);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarps = blockDim.x >> 5;
    const int b = blockIdx.x;
    const int64_t j0 = (int64_t)b * kRsTargets;
    const int nT = (int)min((int64_t)kRsTargets, M - j0);
    const double xa = P.x[j0], span = P.x[j0 + nT - 1] - xa;
    const rs::Grid G = rs::grid_of(span, R.delta);
    for (int iv = t; iv < R.nint; iv += blockDim.x) rs::interval_on_grid(__ldg(R.mid + iv), __ldg(R.ih + iv), G, sIv + 4 * iv);
    const float cscale = R.cell_scale;

    const bool valid = t < nT;
    const int64_t j = j0 + (valid ? t : 0);
    const double xj = P.x[j];
    float hj, lj;
    rs::grid_split(xj - xa, G, hj, lj);
    // lb_j: the first spring at x_j's position (sources below it are strictly left of x_j)
    int64_t lbj = j;
    if (j > 0 && P.x[j - 1] == xj) {
        int64_t lo = 0;
        while (lo < lbj) {
            const int64_t mid = (lo + lbj) >> 1;
            if (P.x[mid] < xj) lo = mid + 1;
            else lbj = mid;
        }
    }
    sT[t] = valid ? (float)(xj - xa) : 3.0e38f;
    const int nbl = __ldg(R.nb_lo + j), nbc = __ldg(R.nb_cnt + j);
    const int wlo = __ldg(R.blk_win + 4 * b), inlo = __ldg(R.blk_win + 4 * b + 1);
    const int inhi = __ldg(R.blk_win + 4 * b + 2), whi = __ldg(R.blk_win + 4 * b + 3);
    const int nL = max(0, inhi - wlo), total = nL + max(0, whi - inlo);
    __syncthreads();

    // two accumulators (even and odd sources), so consecutive pairs are independent chains
    float a0h = 0.f, a0l = 0.f, a1h = 0.f, a1l = 0.f;
    rs::Track trL, trR;
    rs::track_to(sIv, 0, hj, lj, trL);
    rs::track_to(sIv, 0, -hj, -lj, trR);

    if (span > 2.0 * R.delta) {
        // targets farther apart than two window widths: no shared e-vectors to speak of
        if (valid) {
            rs_sparse_side<-1>(P, R, sIv, cscale, G, xa, span, xj, n, wlo, whi, (int)lbj, nbl, nbc, hj, lj, trL, a0h, a0l,
                               a1h, a1l);
            rs_sparse_side<1>(P, R, sIv, cscale, G, xa, span, xj, n, wlo, whi, (int)lbj, nbl, nbc, -hj, -lj, trR, a0h,
                              a0l, a1h, a1l);
            P.clocal[j] = ((double)a0h + (double)a0l) + ((double)a1h + (double)a1l);
        }
        return;
    }
    for (int base = 0; base < total; base += kRsChunk) {
        const int grp = base & (kRsTargets - 1);       // the chunk's place in its group of 8
        if (grp == 0) {
            // set-up of the group's 256 sources, one per thread: position on the block grid and
            // interval range; warp w reduces the union of chunk w
            if (base > 0) __syncthreads();             // the previous group's last chunk is done
            const int v = base + t;
            int lohi = 1, e = 0, cnt = 0;
            float h = 0.f, l = 0.f;
            if (v < total) {
                const bool left = v < nL;
                e = left ? wlo + v : inlo + (v - nL);
                const double xr = rs_xext(P, e) - xa;
                rs::grid_split(xr, G, h, l);
                lohi = rs::source_range(xr, left, span, R.delta, P.dt, R.bp2, R.cell, cscale, R.nint);
                if ((lohi & 0x7fff) <= (lohi >> 16)) {
                    // targets within delta of the source (an estimate: float positions)
                    const float xf = (float)xr, df = (float)R.delta;
                    int a = 0, bnd = nT;
                    while (a < bnd) {
                        const int mid = (a + bnd) >> 1;
                        if (sT[mid] > xf - df) bnd = mid;
                        else a = mid + 1;
                    }
                    int c = a;
                    bnd = nT;
                    while (c < bnd) {
                        const int mid = (c + bnd) >> 1;
                        if (sT[mid] >= xf + df) bnd = mid;
                        else c = mid + 1;
                    }
                    cnt = c - a;
                }
            }
            sMeta[t] = make_float4(h, l, __int_as_float(e), __int_as_float(lohi));
            const int lo = lohi & 0x7fff, hi = lohi >> 16;
            int u0 = lo <= hi ? lo : 0x7fffffff, u1 = lo <= hi ? hi : -1;
            for (int o = 16; o > 0; o >>= 1) {
                u0 = min(u0, __shfl_xor_sync(0xffffffffu, u0, o));
                u1 = max(u1, __shfl_xor_sync(0xffffffffu, u1, o));
                cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            }
            if (lane == 0) {
                sU[0][warp] = u0;
                sU[1][warp] = u1;
                sP[warp] = cnt;
            }
        }
        // the chunk's densities, sigma^{n+1-m} of source k at sSig[m][k] (pairs)
        for (int i = t; i < (R.nm - 1) * kRsChunk; i += blockDim.x) {
            const int k = i & (kRsChunk - 1), m = 1 + i / kRsChunk, v = base + k;
            float2 s = make_float2(0.f, 0.f);
            if (v < total) {
                const int64_t l = rs_spring(v < nL ? wlo + v : inlo + (v - nL), M);
                s = __ldg((const float2*)P.sig2 + (int64_t)ring_slot(n + 1 - m, P.ring) * M + l);
            }
            sSig[m * kRsChunk + k] = s;
        }
        __syncthreads();
        const float4* meta = sMeta + grp;
        const int U0 = sU[0][grp / kRsChunk], U1 = sU[1][grp / kRsChunk];
        if (U1 >= U0 && 2 * sP[grp / kRsChunk] < kRsChunk * (U1 - U0 + 1)) {
            // few pairs per e-vector: each pair folds its own (no windows, no shared records)
            if (valid) {
                const int kend = min(kRsChunk, total - base), kL = min(kend, max(0, nL - base));
                const float4* cf = (const float4*)R.coef;
                rs_direct<-1>(meta, sSig, sIv, R.cell, cscale, R.nint, R.iv_dt, cf, R.mr, R.nm, 0, kL, (int)lbj, nbl, nbc,
                              hj, lj, trL, a0h, a0l, a1h, a1l);
                rs_direct<1>(meta, sSig, sIv, R.cell, cscale, R.nint, R.iv_dt, cf, R.mr, R.nm, kL, kend, (int)lbj, nbl,
                             nbc, -hj, -lj, trR, a0h, a0l, a1h, a1l);
            }
            __syncthreads();
            continue;
        }
        const int lohi_lane = __float_as_int(meta[lane].w);
        const int lo_lane = lohi_lane & 0x7fff, hi_lane = lohi_lane >> 16;
        const bool multi = U1 - U0 + 1 > kRsIvCap;
        const int kend_c = min(kRsChunk, total - base), kL_c = min(kend_c, max(0, nL - base));
        int curL = kL_c - 1, curR = kL_c, par = 0;
        for (int W0 = U0; W0 <= U1; W0 += kRsIvCap) {
            const int W1 = min(U1, W0 + kRsIvCap - 1);
            // e-vectors of the intervals [W0, W1]: warp per interval, lane per source
            for (int iv = W0 + warp; iv <= W1; iv += nwarps) {
                const bool act = lo_lane <= iv && iv <= hi_lane;
                if (!__any_sync(0xffffffffu, act)) continue;
                rs::EVec ev;
                rs::evec_zero(ev);
                const int m0 = __ldg(R.mr + 2 * iv), m1 = __ldg(R.mr + 2 * iv + 1);
                const float4* c = (const float4*)R.coef + (size_t)iv * R.nm * 3;
                // two m per iteration: six coefficient loads in flight (they come from L2)
                int m = m0;
                for (; m < m1; m += 2) {
                    const float4 c01 = __ldg(c + 3 * m), c23 = __ldg(c + 3 * m + 1), c47 = __ldg(c + 3 * m + 2);
                    const float4 d01 = __ldg(c + 3 * m + 3), d23 = __ldg(c + 3 * m + 4), d47 = __ldg(c + 3 * m + 5);
                    const float2 s = sSig[m * kRsChunk + lane], s2 = sSig[(m + 1) * kRsChunk + lane];
                    const float a01[4] = {c01.x, c01.y, c01.z, c01.w}, a23[4] = {c23.x, c23.y, c23.z, c23.w},
                                a47[4] = {c47.x, c47.y, c47.z, c47.w};
                    rs::evec_mac(ev, a01, a23, a47, s.x, s.y);
                    const float b01[4] = {d01.x, d01.y, d01.z, d01.w}, b23[4] = {d23.x, d23.y, d23.z, d23.w},
                                b47[4] = {d47.x, d47.y, d47.z, d47.w};
                    rs::evec_mac(ev, b01, b23, b47, s2.x, s2.y);
                }
                if (m == m1) {
                    const float4 c01 = __ldg(c + 3 * m), c23 = __ldg(c + 3 * m + 1), c47 = __ldg(c + 3 * m + 2);
                    const float2 s = sSig[m * kRsChunk + lane];
                    const float a01[4] = {c01.x, c01.y, c01.z, c01.w}, a23[4] = {c23.x, c23.y, c23.z, c23.w},
                                a47[4] = {c47.x, c47.y, c47.z, c47.w};
                    rs::evec_mac(ev, a01, a23, a47, s.x, s.y);
                }
                float4* rec = (float4*)(sE + (iv - W0) * kRsRow + lane * rs::kERecord);
                rec[0] = make_float4(ev.e0h, ev.e0l, ev.e1h, ev.e1l);
                rec[1] = make_float4(ev.e2, ev.e3, ev.e4, ev.e5);
                rec[2] = make_float4(ev.e6, ev.e7, 0.f, 0.f);
            }
            __syncthreads();
            if (valid && multi) {
                rs_pairs_cursor<-1>(sE, meta, sIv, R.cell, cscale, R.nint, R.iv_dt, 0, kL_c, curL, W0, W1, (int)lbj, nbl,
                                    nbc, hj, lj, trL, par, a0h, a0l, a1h, a1l);
                rs_pairs_cursor<1>(sE, meta, sIv, R.cell, cscale, R.nint, R.iv_dt, kL_c, kend_c, curR, W0, W1, (int)lbj,
                                   nbl, nbc, -hj, -lj, trR, par, a0h, a0l, a1h, a1l);
            } else if (valid) {
                rs_pairs<-1>(sE, meta, sIv, R.cell, cscale, R.nint, R.iv_dt, 0, kL_c, W0, W1, (int)lbj, nbl, nbc, hj, lj,
                             trL, a0h, a0l, a1h, a1l);
                rs_pairs<1>(sE, meta, sIv, R.cell, cscale, R.nint, R.iv_dt, kL_c, kend_c, W0, W1, (int)lbj, nbl, nbc, -hj,
                            -lj, trR, a0h, a0l, a1h, a1l);
            }
            __syncthreads();
        }
    }
    if (valid) P.clocal[j] = ((double)a0h + (double)a0l) + ((double)a1h + (double)a1l);
}

}  // namespace wave1d
