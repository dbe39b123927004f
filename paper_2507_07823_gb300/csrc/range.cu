// Time step of plans opened with opts.local_weights = 1: no per-pair data on the device.  The
// springs are sorted, so the sources within delta of a target are an index window, and the local
// weights Q_m(d) (Sec. 4.1) come from their polynomials in the distance (range.cuh).  One step:
//
//   local explicit sum c_j over m >= 1 (Sec. 4.1), compensated FP32 pairs:
//     per slab of intervals of the distance:
//     k_rs_fold     e-vectors of every spring and interval (k_rs_fold_used: those that some pair reads)
//     k_rs_pairs    the polynomials of all pairs whose distance lies in the slab
//   (k_rs_local, range_fp32.cu, with FP32 spreading and interpolation)
//   history pipeline (type-1 NUFFT, mode update, [projection], type-2 NUFFT): the per-stage
//                   kernels of every plan; the interpolation leaves rhs_j = -g_j - beta_j u_H(x_j)
//   k_rs_solve_init rhs_j -= (beta_j / 2) c_j; first iterate extrapolated from sigma^{n-7..n}
//   k_rs_jacobi     Jacobi sweeps of (I + S) sigma^{n+1} = rhs (eq. linearSystem), S_jl =
//                   (beta_j / 2) Q_0(d_jl) over the sources closer than dt, until the largest
//                   change is below kRsTol of the largest density (launches after that return at
//                   once, so the step is a fixed sequence of launches and can be captured);
//                   k_rs_sweeps: all of them in one launch, for small plans
//   k_rs_store      sigma^{n+1} into the rings (status WAVE1D_ENOTCONV if no sweep converged)
//   k_rs_receivers  u_L at the receivers (eq. localSol2, all m including m = 0), FP64
//   k_rs_finish     u = u_L + u_H at the receivers, step counter
//
// Every kernel reads the step index from the device counter (graphs of steps are replayed).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "internal.h"
#include "phases.cuh"
#include "range.cuh"
#include "range_dev.cuh"
#include "../../include/wave1d.h"

namespace wave1d {

namespace {
constexpr int kRsPosChunk = 1024; // source positions staged at once by a block of k_rs_pairs
}  // namespace

// interval of an FP64 distance
__device__ __forceinline__ int rs_locate64(const RangeDev& R, double d) {
    int lo = 0, hi = R.nint;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (d < __ldg(R.bp + mid)) hi = mid;
        else lo = mid;
    }
    return lo;
}

// Chebyshev series of degree 7 (Clenshaw), FP64
__device__ __forceinline__ double rs_cheb(const double* c, double z) {
    double b0 = 0.0, b1 = 0.0;
    for (int r = 7; r >= 1; r--) {
        const double b2 = b1;
        b1 = b0;
        b0 = fma(2.0 * z, b1, __ldg(c + r) - b2);
    }
    return fma(z, b0, __ldg(c) - b1);
}

// Q_0(d) from its series (zero at d >= dt, where m_min = 1)
__device__ __forceinline__ double rs_q0(const RangeDev& R, double d) {
    const int iv = rs_locate64(R, d);
    if (iv >= R.iv_dt) return 0.0;
    const double z = (d - __ldg(R.mid + iv)) * (double)__ldg(R.ih + iv);
    return rs_cheb(R.cheb + (size_t)iv * R.nm * 8, z);
}

// ---------------------------------------------------------------------------------------------
// The fold: e-vectors e_{l,iv,r} = sum_m a_{iv,m,r} sigma_l^{n+1-m} for the intervals [s0, s0 + slab), in the
// compensated FP32 pairs of range.cuh, m ascending; records (e0h e0l e1h e1l | e2 e3 e4 e5 | e6 e7 - -).
// Bound by FP32 issue: 32 instructions per record and m (evec_mac).
// Every product is one of float pairs.  A contraction of 11-bit slices on the tensor cores took 1.2 ms for
// 1e5 springs (2.7 here), but a slice's unit is that of the largest density of the window and the largest
// coefficient of the interval: where an interval is reached by small coefficients or old densities alone
// (a march from rest, a growing history) e_0 kept 1e-8 of sum_m |a_m sigma_m| or nothing, against 1e-13.
//
// k_rs_fold makes every record, where springs are dense.  A block takes 32 springs, one to a lane, whose
// densities of the window it holds in shared memory, and tiles of 8 intervals, one to a warp, whose
// coefficient rows (read by all lanes alike) each warp copies ahead of the tile that needs them.  Records
// are staged and written as whole rows, two buffers, one barrier a tile.  1e5 springs, 676 intervals, 26 m on
// average: 2.7 ms, of which the FP32 pipe needs 1.5; two springs to a lane the same; coefficients by loads
// from L2 3.5; a lane to an interval 2.7 to 3.3.
// ---------------------------------------------------------------------------------------------
constexpr int kRsFoldSprings = 32;
constexpr int kRsFoldTile = 8;
constexpr int kRsFoldRow = kRsFoldTile * kRsRecord + 4;      // floats of a spring's staged records
size_t rs_fold_smem(int nm, bool copied) {
    return (size_t)2 * kRsFoldSprings * kRsFoldRow * sizeof(float) + (size_t)(nm - 1) * kRsFoldSprings * sizeof(float2) +
           (copied ? (size_t)2 * kRsFoldTile * nm * 3 * sizeof(float4) : 0);
}

// COPIED: the tile's coefficients come through shared memory; windows too long for that read them in place
template <bool COPIED>
__device__ __forceinline__ void rs_fold_block(const DevPlan& P, const RangeDev& R, int s0) {
    extern __shared__ __align__(16) float fold_sm[];         // staged records, densities [m - 1][spring], coefficients
    float2* sSig = (float2*)(fold_sm + 2 * kRsFoldSprings * kRsFoldRow);
    float4* sCoef = (float4*)(sSig + (R.nm - 1) * kRsFoldSprings);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t n = load_step(P), l0 = (int64_t)blockIdx.x * kRsFoldSprings;
    // this block's tiles of the slab
    const int s1 = min(R.nint, s0 + R.slab), ntile = (s1 - s0 + kRsFoldTile - 1) / kRsFoldTile;
    const int t0 = (int)((int64_t)ntile * blockIdx.y / gridDim.y), t1 = (int)((int64_t)ntile * (blockIdx.y + 1) / gridDim.y);
    auto fetch = [&](int tile) {
        const int iv = s0 + kRsFoldTile * tile + warp;
        if (iv < s1) {
            const int m0 = __ldg(R.mr + 2 * iv), rows = 3 * (__ldg(R.mr + 2 * iv + 1) - m0 + 1);
            const float4* src = (const float4*)R.coef + ((size_t)iv * R.nm + m0) * 3;
            float4* dst = sCoef + ((tile & 1) * kRsFoldTile + warp) * R.nm * 3;
            for (int i = lane; i < rows; i += 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst + i)),
                             "l"(src + i));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (COPIED && t0 < t1) fetch(t0);
    for (int i = t; i < (R.nm - 1) * kRsFoldSprings; i += blockDim.x) {
        const int k = i & (kRsFoldSprings - 1), m = 1 + i / kRsFoldSprings;
        float2 v = make_float2(0.f, 0.f);
        if (l0 + k < P.M) v = __ldg((const float2*)P.sig2 + (int64_t)ring_slot(n + 1 - m, P.ring) * P.M + l0 + k);
        sSig[i] = v;
    }
    __syncthreads();
    for (int tile = t0; tile < t1; tile++) {
        float* stage = fold_sm + (tile & 1) * kRsFoldSprings * kRsFoldRow;
        const int iv0 = s0 + kRsFoldTile * tile, iv = iv0 + warp;
        if (COPIED) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();                                     // the warp's rows have arrived, its other buffer is free
            if (tile + 1 < t1) fetch(tile + 1);
        }
        if (iv < s1) {
            rs::EVec ev;
            rs::evec_zero(ev);
            const int m0 = __ldg(R.mr + 2 * iv), m1 = __ldg(R.mr + 2 * iv + 1);
            const float2* sg = sSig + (m0 - 1) * kRsFoldSprings + lane;
            const float4* c = COPIED ? sCoef + ((tile & 1) * kRsFoldTile + warp) * R.nm * 3
                                     : (const float4*)R.coef + ((size_t)iv * R.nm + m0) * 3;
#pragma unroll 2
            for (int m = m0; m <= m1; m++, sg += kRsFoldSprings, c += 3) {
                const float4 a = c[0], b = c[1], d = c[2];
                const float2 s = *sg;
                const float c01[4] = {a.x, a.y, a.z, a.w}, c23[4] = {b.x, b.y, b.z, b.w}, c47[4] = {d.x, d.y, d.z, d.w};
                rs::evec_mac(ev, c01, c23, c47, s.x, s.y);
            }
            float4* rec = (float4*)(stage + lane * kRsFoldRow + warp * kRsRecord);
            rec[0] = make_float4(ev.e0h, ev.e0l, ev.e1h, ev.e1l);
            rec[1] = make_float4(ev.e2, ev.e3, ev.e4, ev.e5);
            rec[2] = make_float4(ev.e6, ev.e7, 0.f, 0.f);
        }
        __syncthreads();                                      // the tile is staged; the other buffer has been written out
        constexpr int rowq = kRsFoldTile * kRsRecord / 4;
        const int per = min(kRsFoldTile, s1 - iv0) * (kRsRecord / 4);
        float* dst = R.evec + ((size_t)l0 * R.slab + (iv0 - s0)) * kRsRecord;
#pragma unroll
        for (int i = t; i < kRsFoldSprings * rowq; i += 32 * kRsFoldTile) {
            const int r = i / rowq, o = i - r * rowq;
            if (o < per && l0 + r < P.M)
                *(float4*)(dst + (size_t)r * R.slab * kRsRecord + 4 * o) = *(const float4*)(stage + r * kRsFoldRow + 4 * o);
        }
    }
}
__global__ void __launch_bounds__(32 * kRsFoldTile, 3) k_rs_fold(DevPlan P, RangeDev R, int s0) {
    rs_fold_block<true>(P, R, s0);
}
__global__ void __launch_bounds__(32 * kRsFoldTile, 3) k_rs_fold_long(DevPlan P, RangeDev R, int s0) {
    rs_fold_block<false>(P, R, s0);
}

// k_rs_fold_used makes the records that some pair reads (R.used), where there is less than a pair to a
// record: a block lists the used records of 32 springs and kRsUsedIntervals intervals, interval by
// interval, and its threads take one each, so a warp reads the coefficients of one or two intervals.  A step
// of uniform springs in free space, every record against the used ones, by pairs per record: 0.11 (6,000
// springs) 0.55 and 0.42 ms, 0.27 0.97 and 0.73, 0.54 1.33 and 1.12, 0.9 2.43 and 2.35, 1.1 2.81 and 2.84,
// 1.8 (100,000) 4.62 and 5.17.
constexpr int kRsUsedIntervals = 64;
size_t rs_used_smem(int nm) { return (size_t)(nm - 1) * kRsFoldSprings * sizeof(float2); }
int rs_used_blocks(int intervals) { return (intervals + kRsUsedIntervals - 1) / kRsUsedIntervals; }
__global__ void __launch_bounds__(256, 3) k_rs_fold_used(DevPlan P, RangeDev R, int s0) {
    extern __shared__ __align__(16) float2 used_sm[];        // densities [m - 1][spring]
    __shared__ unsigned sWord[kRsUsedIntervals];             // per interval: the springs that use it
    __shared__ int sFirst[kRsUsedIntervals + 1];
    __shared__ uint16_t sItem[kRsUsedIntervals * kRsFoldSprings];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarps = blockDim.x >> 5;
    const int64_t n = load_step(P), l0 = (int64_t)blockIdx.x * kRsFoldSprings;
    const int b0 = s0 + kRsUsedIntervals * blockIdx.y, nb = min(kRsUsedIntervals, min(R.nint, s0 + R.slab) - b0);
    for (int k = warp; k < nb; k += nwarps) {
        const int iv = b0 + k;
        const bool u = l0 + lane < P.M && (__ldg(R.used + (size_t)(l0 + lane) * R.used_words + (iv >> 5)) >> (iv & 31) & 1u);
        const unsigned w = __ballot_sync(0xffffffffu, u);
        if (lane == 0) sWord[k] = w;
    }
    __syncthreads();
    if (warp == 0) {
        static_assert(kRsUsedIntervals == 64, "two intervals a lane");
        const int a = 2 * lane < nb ? __popc(sWord[2 * lane]) : 0, b = 2 * lane + 1 < nb ? __popc(sWord[2 * lane + 1]) : 0;
        int sum = a + b;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += v;
        }
        sFirst[2 * lane + 1] = sum - b;
        sFirst[2 * lane + 2] = sum;
        if (lane == 0) sFirst[0] = 0;
    }
    __syncthreads();
    const int total = sFirst[kRsUsedIntervals];
    if (total == 0) return;
    for (int k = warp; k < nb; k += nwarps) {
        const unsigned w = sWord[k];
        if (w >> lane & 1u) sItem[sFirst[k] + __popc(w & ((1u << lane) - 1u))] = (uint16_t)(k * kRsFoldSprings + lane);
    }
    for (int i = t; i < (R.nm - 1) * kRsFoldSprings; i += blockDim.x) {
        const int k = i & (kRsFoldSprings - 1), m = 1 + i / kRsFoldSprings;
        float2 v = make_float2(0.f, 0.f);
        if (l0 + k < P.M) v = __ldg((const float2*)P.sig2 + (int64_t)ring_slot(n + 1 - m, P.ring) * P.M + l0 + k);
        used_sm[i] = v;
    }
    __syncthreads();
    for (int i = t; i < total; i += blockDim.x) {
        const int item = sItem[i], iv = b0 + item / kRsFoldSprings, sp = item & (kRsFoldSprings - 1);
        rs::EVec ev;
        rs::evec_zero(ev);
        const int m0 = __ldg(R.mr + 2 * iv), m1 = __ldg(R.mr + 2 * iv + 1);
        const float4* c = (const float4*)R.coef + ((size_t)iv * R.nm + m0) * 3;
        const float2* sg = used_sm + (m0 - 1) * kRsFoldSprings + sp;
#pragma unroll 2
        for (int m = m0; m <= m1; m++, sg += kRsFoldSprings, c += 3) {
            const float4 a = __ldg(c), b = __ldg(c + 1), d = __ldg(c + 2);
            const float2 s = *sg;
            const float c01[4] = {a.x, a.y, a.z, a.w}, c23[4] = {b.x, b.y, b.z, b.w}, c47[4] = {d.x, d.y, d.z, d.w};
            rs::evec_mac(ev, c01, c23, c47, s.x, s.y);
        }
        float4* rec = (float4*)(R.evec + ((size_t)(l0 + sp) * R.slab + (iv - s0)) * kRsRecord);
        rec[0] = make_float4(ev.e0h, ev.e0l, ev.e1h, ev.e1l);
        rec[1] = make_float4(ev.e2, ev.e3, ev.e4, ev.e5);
        rec[2] = make_float4(ev.e6, ev.e7, 0.f, 0.f);
    }
}

// ---------------------------------------------------------------------------------------------
// Pairs whose distances lie in the intervals [p0, p1) of a slab: one block per kRsPairTargets
// consecutive targets and side (0: sources strictly left of the target, d = x_j - x_e; 1: at or right
// of it, d = x_e - x_j).  The block stages the positions of the sources that some target meets at such
// a distance on the block grid (range.cuh), kRsPosChunk at a time; a warp takes its own run of them one
// by one for its 32 targets together, whose records lie next to one another (same source,
// neighbouring intervals).  The interval of a pair comes from a table of fine cells of the distance and
// the next breakpoints, in FP32, and is checked by z, so it depends on the pair alone and each pair falls
// in one part whatever the parts are.  Two sources are in flight at a time: the chain position - cell -
// interval - record of a pair is four dependent loads.
// Which side counts a source is decided by index: e < lb_j (the first spring at x_j's position) is
// strictly left.  Q_m is continuous across the breakpoints other than dt, so a pair within
// rounding of one takes either neighbouring interval's polynomial; at dt the spring's FP64 window
// of near sources decides.
// ---------------------------------------------------------------------------------------------
// acc += the polynomial of a record at z
__device__ __forceinline__ void rs_eval(const float4& a, const float4& b, const float2& c, float zh, float zl, float& ah,
                                        float& al) {
    rs::evec_eval4(rs::F4{a.x, a.y, a.z, a.w}, rs::F4{b.x, b.y, b.z, b.w}, rs::F4{c.x, c.y, 0.f, 0.f}, zh, zl, ah, al);
}

// the first k in [0, n) with pred(k), or n (pred monotone), by a warp: 32 probes a round
template <typename F>
__device__ __forceinline__ int rs_warp_first(int n, F&& pred) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;                      // the answer lies in [lo, hi]
    while (hi > lo) {
        const int step = (hi - lo + 31) / 32, k = lo + lane * step;
        const unsigned yes = __ballot_sync(0xffffffffu, k >= hi || pred(k));
        if (yes == 0u) {
            lo = lo + 31 * step + 1;         // none of the probes
            continue;
        }
        const int f = __ffs(yes) - 1;
        hi = min(hi, lo + f * step);
        if (f > 0) lo = lo + (f - 1) * step + 1;
    }
    return hi;
}

// One side of one block's pairs of the intervals [p0, p1): v.stage(k, e) is called for each of the
// block's sources as their positions are staged (k: place in the chunk), v.pair(u, k, e, iv, zh, zl)
// for each pair of this thread's target in the order of its sources (u: the source's parity).
template <int S, typename Visitor>
__device__ __forceinline__ void rs_pair_block(const DevPlan& P, const RangeDev& R, int p0, int p1, float4* sIv, float2* sPos,
                                              int* sRed, Visitor& v) {
    const int64_t M = P.M;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * kRsPairTargets;
    const int nT = (int)min((int64_t)kRsPairTargets, M - j0);
    const double xa = P.x[j0], xb = P.x[j0 + nT - 1];
    const rs::Grid G = rs::grid_of(xb - xa, R.delta);
    const float gf = (float)G.g, igf = (float)G.ig;
    // the part's intervals and those a pair of it may be looked up as first
    const int v0 = max(0, p0 - R.fine_span - 2), v1 = min(R.nint, p1 + 2);
    for (int iv = v0 + t; iv < v1; iv += blockDim.x) {
        const rs::F4 q = rs::interval_entry(__ldg(R.mid + iv), __ldg(R.ih + iv),
                                            iv + 1 < R.nint ? __ldg(R.bp2 + 2 * (iv + 1)) : __uint_as_float(0x7f800000u), gf, igf);
        sIv[iv - v0] = make_float4(q.x, q.y, q.z, q.w);
    }
    const bool valid = t < nT;
    const int64_t j = j0 + (valid ? t : nT - 1);
    const double xj = P.x[j];
    float bh, bl;
    rs::grid_split(xj - xa, G, bh, bl);
    if (S > 0) {
        bh = -bh;
        bl = -bl;
    }
    const int nbl = __ldg(R.nb_lo + j), nbc = __ldg(R.nb_cnt + j);
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
    const int lb = (int)lbj;
    // the block's sources in the order of their distance: from the first one that may lie at the
    // part's near end from some target to the first one beyond its far end from all of them, inside
    // the window of its 256-target block
    const int* win = R.blk_win + 4 * (j0 / kRsTargets);
    const int top = S > 0 ? __ldg(win) : (int)(j0 + nT - 1), all = max(0, S > 0 ? __ldg(win + 3) - top : top - __ldg(win) + 1);
    const double marg = rs::part_margin(R.delta, G.g), d0 = __ldg(R.bp + p0) - marg, d1 = __ldg(R.bp + p1) + marg;
    if (warp < 2) {
        const int c = rs_warp_first(all, [&](int k) {
            const double x = rs_xext(P, top + S * k);
            return warp == 0 ? (S > 0 ? x - xa : xb - x) >= d0 : !((S > 0 ? x - xb : xa - x) < d1);
        });
        if (lane == 0) sRed[warp] = c;
    }
    __syncthreads();
    const int start = top + S * sRed[0], count = sRed[1] - sRed[0];
    const bool at_dt = p0 <= R.iv_dt && R.iv_dt <= p1;    // the part touches the breakpoint dt
    const float bfar = __shfl_sync(0xffffffffu, bh, S > 0 ? 0 : 31), bnear = __shfl_sync(0xffffffffu, bh, S > 0 ? 31 : 0);
    const float df0 = (float)d0, df1 = (float)d1;
    const int ns = v1 - v0, ivd = R.iv_dt - v0;
    for (int base = 0; base < count; base += kRsPosChunk) {
        const int lim = min(count - base, kRsPosChunk), e0 = start + S * base;
        if (base > 0) __syncthreads();
        for (int k = t; k < lim; k += blockDim.x) {
            float h, l;
            rs::grid_split(rs_xext(P, e0 + S * k) - xa, G, h, l);
            sPos[k] = make_float2(h, l);
            v.stage(k, e0 + S * k);
        }
        __syncthreads();
        // the warp's run of the chunk
        const int klo = rs_warp_first(lim, [&](int k) { return (S < 0 ? bfar - sPos[k].x : bfar + sPos[k].x) >= df0; });
        const int khi = rs_warp_first(lim, [&](int k) { return (S < 0 ? bnear - sPos[k].x : bnear + sPos[k].x) >= df1; });
        for (int k0 = klo; k0 < khi; k0 += 2) {
            float zh[2], zl[2];
            int iv[2];
            bool in[2];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int k = k0 + u, e = e0 + S * k;
                const float2 ps = sPos[min(k, lim - 1)];
                const int i = rs::place_pair<S>([&](int k2) { return rs::load4((const float*)(sIv + k2)); },
                                                [&](int c) { return (int)__ldg(R.fine + c); }, R.fine_scale, v0, ns, at_dt, ivd,
                                                (unsigned)(e - nbl) < (unsigned)nbc, valid && k < khi && (S > 0 ? e >= lb : e < lb), bh,
                                                bl, ps.x, ps.y, zh[u], zl[u]);
                iv[u] = i + v0;
                in[u] = i >= 0 && iv[u] >= p0 && iv[u] < p1;
            }
            v.pairs(in, k0, e0 + S * k0, S, iv, zh, zl);
        }
    }
    __syncthreads();                                      // the staged positions are free again
}

// the local sum of one side and part: each target's polynomials, two sources at a time into two pairs
struct RsSum {
    const DevPlan& P;
    const RangeDev& R;
    int s0;                   // the slab's first interval
    float ah[2], al[2];
    __device__ __forceinline__ void stage(int, int) {}
    __device__ __forceinline__ void pairs(const bool (&in)[2], int, int e, int step, const int (&iv)[2], const float (&zh)[2],
                                          const float (&zl)[2]) {
        float4 r[2][2];
        float2 q[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const float4* rec = (const float4*)(R.evec + ((size_t)rs_spring(e + u * step, P.M) * R.slab + (iv[u] - s0)) * kRsRecord);
            if (in[u]) {
                r[u][0] = __ldg(rec);
                r[u][1] = __ldg(rec + 1);
                q[u] = __ldg((const float2*)(rec + 2));
            }
        }
#pragma unroll
        for (int u = 0; u < 2; u++)
            if (in[u]) rs_eval(r[u][0], r[u][1], q[u], zh[u], zl[u], ah[u], al[u]);
    }
};

// ten blocks to an SM (48 registers, five words spilled): the loads' latency is what a warp waits for, and
// more warps gain more than the spills cost.  A million clustered springs, the whole step: 72.2 ms with six
// blocks (66 registers, no spills), 69.8 with eight, 66.2 with ten (measured with a fold 12 ms faster)
constexpr int kRsPairBlocks = 10;
__global__ void __launch_bounds__(kRsPairTargets, kRsPairBlocks) k_rs_pairs(DevPlan P, RangeDev R, int s0) {
    extern __shared__ __align__(16) float4 pair_sm[];
    __shared__ float2 sPos[kRsPosChunk];
    __shared__ int sRed[2];
    const int p0 = s0 + blockIdx.z * R.part, p1 = min(R.nint, p0 + R.part);
    RsSum v{P, R, s0, {0.f, 0.f}, {0.f, 0.f}};
    if (blockIdx.y == 0) rs_pair_block<-1>(P, R, p0, p1, pair_sm, sPos, sRed, v);
    else rs_pair_block<1>(P, R, p0, p1, pair_sm, sPos, sRed, v);
    rs::acc_add(v.ah[0], v.al[0], v.ah[1], v.al[1]);
    const int64_t j = (int64_t)blockIdx.x * kRsPairTargets + threadIdx.x;
    if (j < P.M) ((float2*)R.csum)[((size_t)(p0 / R.part) * 2 + blockIdx.y) * P.M + j] = make_float2(v.ah[0], v.al[0]);
}

// plan time: the records that k_rs_pairs reads, by its own walk (R.used zero on entry)
struct RsUse {
    const DevPlan& P;
    const RangeDev& R;
    __device__ __forceinline__ void stage(int, int) {}
    __device__ __forceinline__ void pairs(const bool (&in)[2], int, int e, int step, const int (&iv)[2], const float (&)[2],
                                          const float (&)[2]) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            if (!in[u]) continue;
            unsigned* w = R.used + (size_t)rs_spring(e + u * step, P.M) * R.used_words + (iv[u] >> 5);
            const unsigned bit = 1u << (iv[u] & 31);
            if (!(__ldcg(w) & bit)) atomicOr(w, bit);
        }
    }
};
__global__ void __launch_bounds__(kRsPairTargets) k_rs_mark_used(DevPlan P, RangeDev R) {
    extern __shared__ __align__(16) float4 pair_sm[];
    __shared__ float2 sPos[kRsPosChunk];
    __shared__ int sRed[2];
    const int p0 = blockIdx.z * R.part, p1 = min(R.nint, p0 + R.part);
    RsUse v{P, R};
    if (blockIdx.y == 0) rs_pair_block<-1>(P, R, p0, p1, pair_sm, sPos, sRed, v);
    else rs_pair_block<1>(P, R, p0, p1, pair_sm, sPos, sRed, v);
}

// shared memory of a pair block's interval table
size_t rs_pair_smem(int part, int fine_span) { return (size_t)(part + fine_span + 4) * sizeof(float4); }

// plan time: the terms of the local sum, sum over pairs (j, l) closer than delta of the number of
// m >= 1 with a non-zero weight on the pair's interval (the multiply-adds sum_m Q_m sigma_l^{n+1-m}
// the method performs per step), by a walk over each target's sources on both sides
__global__ void k_rs_count_terms(DevPlan P, RangeDev R, unsigned long long* total) {
    unsigned long long acc = 0;
    const bool per = P.bc == WAVE1D_PERIODIC;
    const int64_t elo = per ? -P.M : 0, ehi = per ? 2 * P.M : P.M;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P.M; j += (int64_t)gridDim.x * blockDim.x) {
        const double xj = P.x[j];
        for (int side = 0; side < 2; side++) {
            int64_t e = side ? j : j - 1;                  // right: the spring itself first (d = 0)
            int iv = 0;
            for (;;) {
                if (side ? e >= min(ehi, j + P.M) : e < max(elo, j - P.M)) break;
                const double d = side ? rs_xext(P, e) - xj : xj - rs_xext(P, e);
                if (!(d < R.delta)) break;
                while (iv + 1 < R.nint && !(d < __ldg(R.bp + iv + 1))) iv++;
                const int m0 = __ldg(R.mr + 2 * iv), m1 = __ldg(R.mr + 2 * iv + 1);
                acc += (unsigned long long)max(0, m1 - m0 + 1);
                e += side ? 1 : -1;
            }
        }
    }
    atomicAdd(total, acc);
}

// ---------------------------------------------------------------------------------------------
// Implicit solve of eq. linearSystem: (I + S) sigma^{n+1} = rhs by Jacobi sweeps
// ---------------------------------------------------------------------------------------------

// plan time: S_jl = (beta_j / 2) Q_0(d_jl) for the sources of spring j's window (warp per spring)
__global__ void k_rs_nearby_weights(DevPlan P, RangeDev R) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < P.M; j += nw) {
        const double xj = P.x[j], hb = 0.5 * P.beta[j];
        const int lo = R.nb_lo[j], cnt = R.nb_cnt[j];
        const int64_t off = R.nb_off[j];
        for (int k = lane; k < cnt; k += 32) {
            const int64_t e = (int64_t)lo + k;
            const double w = e == j ? 0.0 : hb * rs_q0(R, fabs(rs_xext(P, e) - xj));
            const rs::Pair pw = rs::split(w);
            R.nb_w[2 * (off + k)] = pw.hi;
            R.nb_w[2 * (off + k) + 1] = pw.lo;
        }
        if (lane == 0) {
            const double diag = 1.0 + hb * rs_q0(R, 0.0);
            R.diag[j] = diag;
            R.idiag[j] = 1.0 / diag;
        }
    }
}

__device__ __forceinline__ double rs_from_bits(unsigned long long v) { return __longlong_as_double((long long)v); }

// right-hand side and first iterate: sigma^{n+1} extrapolated from sigma^{n-7..n} (the
// degree-7 polynomial through them), or rhs / (1 + S_jj) in the first steps
__global__ void k_rs_solve_init(DevPlan P, RangeDev R) {
    const int64_t n = load_step(P);
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < 2 * (kRsMaxIter + 1); i += blockDim.x) R.stats[i] = 0ull;
    const double ex[8] = {8.0, -28.0, 56.0, -70.0, 56.0, -28.0, 8.0, -1.0};
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P.M; j += (int64_t)gridDim.x * blockDim.x) {
        // the two sides of the local sum
        double c;
        if (R.folded) {
            // the parts and sides of the local sum, in order
            float h = 0.f, l = 0.f;
            for (int q = 0; q < 2 * R.nparts; q++) {
                const float2 a = ((const float2*)R.csum)[(size_t)q * P.M + j];
                rs::acc_add(h, l, a.x, a.y);
            }
            c = (double)h + (double)l;
            P.clocal[j] = c;
        } else {
            c = P.clocal[j];                            // the mixed form's k_rs_local
        }
        const double rhs = fma(-0.5 * P.beta[j], c, __ldcg(P.rhs + j));
        P.rhs[j] = rhs;
        double x0;
        if (n >= 8) {
            x0 = 0.0;
            for (int q = 0; q < 8; q++) x0 = fma(ex[q], P.sig[(int64_t)ring_slot(n - q, P.ring) * P.M + j], x0);
        } else {
            x0 = rhs / R.diag[j];
        }
        R.it64[0][j] = x0;
        const rs::Pair p2 = rs::split(x0);
        R.it2[0][2 * j] = p2.hi;
        R.it2[0][2 * j + 1] = p2.lo;
    }
}

// sweep `it` (1 .. kRsMaxIter): iterate it from iterate it - 1, unless sweep it - 1 converged.  A warp
// takes kRsRows consecutive springs: each row's sum sum_{l != j} S_jl sigma_l in compensated pairs over
// the lanes, then one lane per row does the row's FP64 work (the division above all: some 20
// instructions of 16 cycles of an SM each, whether one lane or 32 take part; with one row at a time it
// bound the sweep, 120 us at 1e5 springs and 0.9 ms at a million).
constexpr int kRsRows = 8;
__global__ void __launch_bounds__(256) k_rs_jacobi(DevPlan P, RangeDev R, int it) {
    if (it >= 2) {
        const double dmax = rs_from_bits(__ldcg(R.stats + 2 * (it - 1)));
        const double smax = rs_from_bits(__ldcg(R.stats + 2 * (it - 1) + 1));
        if (dmax <= kRsTol * smax) return;
    }
    __shared__ double red[2][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float* src2 = R.it2[(it - 1) & 1];
    const double* src = R.it64[(it - 1) & 1];
    double* dst = R.it64[it & 1];
    float* dst2 = R.it2[it & 1];
    double dmax = 0.0, smax = 0.0;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5, groups = (P.M + kRsRows - 1) / kRsRows;
    for (int64_t gr = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; gr < groups; gr += nw) {
        const int64_t j0 = gr * kRsRows, mine = j0 + lane;
        const bool own = lane < kRsRows && mine < P.M;
        // the rows' windows, one per lane, and what their FP64 work reads
        const int lo_r = own ? __ldg(R.nb_lo + mine) : 0, cnt_r = own ? __ldg(R.nb_cnt + mine) : 0;
        const int64_t off_r = own ? __ldg(R.nb_off + mine) : 0;
        const double rhs = own ? __ldcg(P.rhs + mine) : 0.0, diag = own ? R.diag[mine] : 1.0, prev = own ? __ldcg(src + mine) : 0.0;
        float sh = 0.f, sl = 0.f;
#pragma unroll 2
        for (int r = 0; r < kRsRows; r++) {
            const int lo = __shfl_sync(0xffffffffu, lo_r, r), cnt = __shfl_sync(0xffffffffu, cnt_r, r);
            const int64_t off = __shfl_sync(0xffffffffu, off_r, r);
            // four entries per lane in flight (their weight and iterate loads issued together), two
            // accumulators; the row's entries are streamed once per sweep
            float ah = 0.f, al = 0.f, bh = 0.f, bl = 0.f;
            int k = lane;
            for (; k + 96 < cnt; k += 128) {
                float2 w[4], sv[4];
#pragma unroll
                for (int u = 0; u < 4; u++) w[u] = __ldcs((const float2*)R.nb_w + off + k + 32 * u);
#pragma unroll
                for (int u = 0; u < 4; u++) sv[u] = __ldcg((const float2*)src2 + rs_spring((int64_t)lo + k + 32 * u, P.M));
                rs::acc_mac(ah, al, w[0].x, w[0].y, sv[0].x, sv[0].y);
                rs::acc_mac(bh, bl, w[1].x, w[1].y, sv[1].x, sv[1].y);
                rs::acc_mac(ah, al, w[2].x, w[2].y, sv[2].x, sv[2].y);
                rs::acc_mac(bh, bl, w[3].x, w[3].y, sv[3].x, sv[3].y);
            }
            for (; k < cnt; k += 32) {
                const float2 w = __ldcs((const float2*)R.nb_w + off + k);
                const float2 s = __ldcg((const float2*)src2 + rs_spring((int64_t)lo + k, P.M));
                rs::acc_mac(ah, al, w.x, w.y, s.x, s.y);
            }
            rs::acc_add(ah, al, bh, bl);
            for (int o = 16; o > 0; o >>= 1) {
                const float oh = __shfl_xor_sync(0xffffffffu, ah, o), ol = __shfl_xor_sync(0xffffffffu, al, o);
                rs::acc_add(ah, al, oh, ol);
            }
            // lane 0's sum (the tree's order differs from lane to lane) goes to the row's lane
            const float th = __shfl_sync(0xffffffffu, ah, 0), tl = __shfl_sync(0xffffffffu, al, 0);
            if (lane == r) {
                sh = th;
                sl = tl;
            }
        }
        if (own) {
            const double x = (rhs - ((double)sh + (double)sl)) / diag;
            dmax = fmax(dmax, fabs(x - prev));
            smax = fmax(smax, fabs(x));
            dst[mine] = x;
            const rs::Pair p2 = rs::split(x);
            ((float2*)dst2)[mine] = make_float2(p2.hi, p2.lo);
        }
    }
    for (int o = kRsRows / 2; o > 0; o >>= 1) {
        dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    }
    if (lane == 0) {
        red[0][wid] = dmax;
        red[1][wid] = smax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); w++) {
            dmax = fmax(dmax, red[0][w]);
            smax = fmax(smax, red[1][w]);
        }
        // non-negative doubles order as their bit patterns (a NaN sorts above every number)
        atomicMax(R.stats + 2 * it, (unsigned long long)__double_as_longlong(dmax));
        atomicMax(R.stats + 2 * it + 1, (unsigned long long)__double_as_longlong(smax));
    }
}

// All sweeps of a small plan in one launch: one cluster (8 or 16 blocks, api.cu), four lanes to a
// row (rows of these plans hold a few tens of sources), the cluster's barrier between sweeps, until the stopping rule
// is met.  Forty launches, of which 7 to 10 do work, cost a plan of 3e4 springs more than its sweeps, and
// a batch runs many such plans side by side.  Four lanes to a row: the weights of a row lie together, and a
// lane per row fetched 32 lines an instruction.  The FP64 epilogue (16 cycles of the SM an instruction)
// takes 32 rows at once: the quotient by the stored reciprocal with one residual correction, the two
// largest moduli as bit patterns on the integer pipe.  A reverse march of 3e4 springs (30 solves) 46.1 ms
// with eight blocks, a lane per row, the division and FP64 maxima; 40.8 with sixteen blocks and the new
// epilogue; 39.5 with four lanes to a row.
__device__ __forceinline__ unsigned long long rs_modulus_bits(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b;       // a NaN does not count, as with fmax
}
__global__ void __launch_bounds__(1024) k_rs_sweeps(DevPlan P, RangeDev R) {
    __shared__ unsigned long long red[2][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int it = 1; it <= kRsMaxIter; it++) {
        const float2* src2 = (const float2*)R.it2[(it - 1) & 1];
        const double* src = R.it64[(it - 1) & 1];
        double* dst = R.it64[it & 1];
        float2* dst2 = (float2*)R.it2[it & 1];
        unsigned long long dmax = 0, smax = 0;
        for (int64_t j0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; j0 < P.M; j0 += (int64_t)gridDim.x * blockDim.x) {
            const bool own = j0 + lane < P.M;
            const int64_t j = own ? j0 + lane : P.M - 1;
            const int lo = __ldg(R.nb_lo + j), cnt = own ? __ldg(R.nb_cnt + j) : 0;
            const long long off = __ldg(R.nb_off + j);
            const double rhs = __ldcg(P.rhs + j), prev = __ldcg(src + j), diag = __ldg(R.diag + j), inv = __ldg(R.idiag + j);
            float sh = 0.f, sl = 0.f;
            // four lanes a row, eight rows at a time; each row's sum goes to the row's lane
#pragma unroll 1
            for (int g = 0; g < 4; g++) {
                const int r = 8 * g + (lane >> 2);
                const int rlo = __shfl_sync(0xffffffffu, lo, r), rcnt = __shfl_sync(0xffffffffu, cnt, r);
                const float2* w = (const float2*)R.nb_w + __shfl_sync(0xffffffffu, off, r);
                float ah = 0.f, al = 0.f, bh = 0.f, bl = 0.f;
                for (int k = lane & 3; k < rcnt; k += 16) {
                    float2 wv[4], sv[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const bool in = k + 4 * u < rcnt;
                        wv[u] = in ? __ldg(w + k + 4 * u) : make_float2(0.f, 0.f);
                        sv[u] = in ? __ldcg(src2 + rs_spring((int64_t)rlo + k + 4 * u, P.M)) : make_float2(0.f, 0.f);
                    }
                    rs::acc_mac(ah, al, wv[0].x, wv[0].y, sv[0].x, sv[0].y);
                    rs::acc_mac(bh, bl, wv[1].x, wv[1].y, sv[1].x, sv[1].y);
                    rs::acc_mac(ah, al, wv[2].x, wv[2].y, sv[2].x, sv[2].y);
                    rs::acc_mac(bh, bl, wv[3].x, wv[3].y, sv[3].x, sv[3].y);
                }
                __syncwarp();
                rs::acc_add(ah, al, bh, bl);
#pragma unroll
                for (int o = 2; o > 0; o >>= 1) {
                    const float oh = __shfl_xor_sync(0xffffffffu, ah, o), ol = __shfl_xor_sync(0xffffffffu, al, o);
                    rs::acc_add(ah, al, oh, ol);
                }
                const float th = __shfl_sync(0xffffffffu, ah, 4 * (lane & 7)), tl = __shfl_sync(0xffffffffu, al, 4 * (lane & 7));
                if (lane >> 3 == g) {
                    sh = th;
                    sl = tl;
                }
            }
            if (!own) continue;
            const double t = rhs - ((double)sh + (double)sl);
            const double q = t * inv, x = fma(fma(-diag, q, t), inv, q);
            dmax = max(dmax, rs_modulus_bits(x - prev));
            smax = max(smax, rs_modulus_bits(x));
            dst[j] = x;
            const rs::Pair p2 = rs::split(x);
            dst2[j] = make_float2(p2.hi, p2.lo);
        }
        __syncwarp();
        for (int o = 16; o > 0; o >>= 1) {
            dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
            smax = max(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        }
        if (lane == 0) {
            red[0][wid] = dmax;
            red[1][wid] = smax;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < (int)(blockDim.x >> 5); w++) {
                dmax = max(dmax, red[0][w]);
                smax = max(smax, red[1][w]);
            }
            atomicMax(R.stats + 2 * it, dmax);
            atomicMax(R.stats + 2 * it + 1, smax);
            __threadfence();
        }
        __syncthreads();
        // every block's rows and its part of the record are in place for the whole cluster
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rs_from_bits(__ldcg(R.stats + 2 * it)) <= kRsTol * rs_from_bits(__ldcg(R.stats + 2 * it + 1))) break;
    }
}

// the converged iterate into the rings: the first sweep whose record meets the stopping rule
// (sweeps after it did not run and left zero records)
__global__ void k_rs_store(DevPlan P, RangeDev R) {
    const int64_t n = load_step(P);
    int fin = kRsMaxIter;
    bool ok = false;
    for (int it = 1; it <= kRsMaxIter; it++) {
        const double dmax = rs_from_bits(__ldcg(R.stats + 2 * it)), smax = rs_from_bits(__ldcg(R.stats + 2 * it + 1));
        if (dmax <= kRsTol * smax) {
            fin = it;
            ok = true;
            break;
        }
    }
    const double* x = R.it64[fin & 1];
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P.M; j += (int64_t)gridDim.x * blockDim.x)
        store_sigma(P, n, (int)j, __ldcg(x + j));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *R.iters = fin;
        if (!ok) atomicCAS(P.status, 0, (int)WAVE1D_ENOTCONV);
    }
}

// T_0(z) .. T_7(z); a series is then 7 FMAs (a Clenshaw sum per m would be 15)
__device__ __forceinline__ void rs_cheb_basis(double z, double (&T)[8]) {
    T[0] = 1.0;
    T[1] = z;
#pragma unroll
    for (int r = 2; r < 8; r++) T[r] = fma(2.0 * z, T[r - 1], -T[r - 2]);
}
__device__ __forceinline__ double rs_cheb_sum(const double* c, const double (&T)[8]) {
    double v = __ldg(c);
#pragma unroll
    for (int r = 1; r < 8; r++) v = fma(__ldg(c + r), T[r], v);
    return v;
}

// receivers' local part (eq. localSol2), block (chunk c of kRsRecvChunk sources, receiver r): every m of
// the pair's interval, m = 0 with sigma^{n+1} (already stored), FP64; block sums in a fixed order.  Four
// threads share a source, each every fourth m: with one thread each the 25 to 40 series in a row took
// 73 us whatever the number of receivers.
constexpr int kRsRecvChunk = 64;
int rs_receiver_chunks(int64_t window) { return (int)((window + kRsRecvChunk - 1) / kRsRecvChunk); }
__global__ void __launch_bounds__(4 * kRsRecvChunk) k_rs_receivers(DevPlan P, RangeDev R) {
    __shared__ double red[kRsRecvChunk / 8];
    const int64_t n = load_step(P);
    const int r = blockIdx.y, c = blockIdx.x;
    const int lo = R.r_win[2 * r], hi = R.r_win[2 * r + 1];
    const int64_t e = (int64_t)lo + (int64_t)c * kRsRecvChunk + (threadIdx.x & (kRsRecvChunk - 1));
    const int q = threadIdx.x / kRsRecvChunk;
    double v = 0.0;
    if (e < hi) {
        const int64_t l = rs_spring(e, P.M);
        const double d = fabs(rs_xext(P, e) - P.xr[r]);
        if (d < R.delta) {
            const int iv = rs_locate64(R, d);
            double T[8];
            rs_cheb_basis((d - __ldg(R.mid + iv)) * (double)__ldg(R.ih + iv), T);
            const int m0 = __ldg(R.mr0 + 2 * iv), m1 = __ldg(R.mr0 + 2 * iv + 1);
            for (int m = m0 + q; m <= m1; m += 4)
                v = fma(rs_cheb_sum(R.cheb + ((size_t)iv * R.nm + m) * 8, T),
                        __ldcg(P.sig + (int64_t)ring_slot(n + 1 - m, P.ring) * P.M + l), v);
        }
    }
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += red[w];
        R.r_part[(size_t)r * R.rchunks + c] = s;
    }
}

// u = u_L + u_H at the receivers (a warp per receiver over its chunks' partials), then the step counter
__global__ void k_rs_finish(DevPlan P, RangeDev R) {
    const int64_t n = load_step(P);
    const int lane = threadIdx.x & 31;
    for (int64_t r = threadIdx.x >> 5; r < P.R; r += blockDim.x >> 5) {
        double s = 0.0;
        for (int c = lane; c < R.rchunks; c += 32) s += __ldcg(R.r_part + r * R.rchunks + c);
        s = warp_sum(s);
        if (lane == 0) P.rec_hist[(n % P.chunk) * P.R + r] = 0.5 * s + __ldcg(P.uHr + r);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        *P.item_ctr = 0ull;
        P.step[1] = 0;
        __threadfence();
        P.step[0] = n + 1;
    }
}

// ---------------------------------------------------------------------------------------------
// Reverse march (wave1d_adjoint on a plan without pair lists): the transposed local sum,
//   sigmabar_l^{n+1-m} += sum_j Q_m(d_jl) cbar_j,   m >= 1,
// over the same pairs as k_rs_pairs (every j within delta of l, each once).  On interval iv,
// Q_m(d) = sum_r a_{iv,m,r} z^r, so the pairs of output l that fall in iv enter only through the
// moments F_{l,iv,r} = sum_{j in iv} z_jl^r cbar_j (k_rs_moments: F_0, F_1 as pairs, F_2 .. F_7 single),
// and the rest is a sum over intervals and powers with the same coefficients for every output,
// sum_{iv,r} a_{iv,m,r} F_{l,iv,r} (k_rs_unfold).  No atomics: every output has one writer, in a fixed order.
// ---------------------------------------------------------------------------------------------
struct RsMoments {
    const DevPlan& P;
    const RangeDev& R;
    const double* cbar;
    float2* sC;               // cbar of the staged sources as pairs
    float* rec;               // this output's records of the slab
    int s0;                   // the slab's first interval
    int cur;                  // the interval whose moments are held, -1: none
    float f0h, f0l, f1h, f1l, f2, f3, f4, f5, f6, f7;
    __device__ __forceinline__ void clear() { f0h = f0l = f1h = f1l = f2 = f3 = f4 = f5 = f6 = f7 = 0.f; }
    __device__ __forceinline__ void flush() {
        if (cur < 0) return;
        float4* o = (float4*)(rec + (size_t)cur * kRsRecord);
        const float4 a = o[0], b = o[1], c = o[2];        // (the records start as zeros)
        rs::acc_add(f0h, f0l, a.x, a.y);
        rs::acc_add(f1h, f1l, a.z, a.w);
        f2 = __fadd_rn(f2, b.x);
        f3 = __fadd_rn(f3, b.y);
        f4 = __fadd_rn(f4, b.z);
        f5 = __fadd_rn(f5, b.w);
        f6 = __fadd_rn(f6, c.x);
        f7 = __fadd_rn(f7, c.y);
        o[0] = make_float4(f0h, f0l, f1h, f1l);
        o[1] = make_float4(f2, f3, f4, f5);
        o[2] = make_float4(f6, f7, 0.f, 0.f);
    }
    __device__ __forceinline__ void stage(int k, int e) {
        const double c = cbar[rs_spring(e, P.M)];
        const float hi = (float)c;
        sC[k] = make_float2(hi, (float)(c - (double)hi));
    }
    __device__ __forceinline__ void pairs(const bool (&in)[2], int k, int, int, const int (&iv)[2], const float (&zh)[2],
                                          const float (&zl)[2]) {
#pragma unroll
        for (int u = 0; u < 2; u++)
            if (in[u]) pair(k + u, iv[u] - s0, zh[u], zl[u]);
    }
    __device__ __forceinline__ void pair(int k, int iv, float zh, float zl) {
        if (iv != cur) {
            flush();
            cur = iv;
            clear();
        }
        const float2 c = sC[k];
        rs::acc_add(f0h, f0l, c.x, c.y);
        rs::acc_mac(f1h, f1l, zh, zl, c.x, c.y);
        float p = __fmul_rn(__fmul_rn(zh, zh), c.x);
        f2 = __fadd_rn(f2, p);
        p = __fmul_rn(p, zh);
        f3 = __fadd_rn(f3, p);
        p = __fmul_rn(p, zh);
        f4 = __fadd_rn(f4, p);
        p = __fmul_rn(p, zh);
        f5 = __fadd_rn(f5, p);
        p = __fmul_rn(p, zh);
        f6 = __fadd_rn(f6, p);
        p = __fmul_rn(p, zh);
        f7 = __fadd_rn(f7, p);
    }
};

// the moments of a slab, both sides (the records are zero on entry), parts in blocks of their own
__global__ void __launch_bounds__(kRsPairTargets) k_rs_moments(DevPlan P, RangeDev R, int s0,
                                                              const double* __restrict__ cbar) {
    extern __shared__ __align__(16) float4 pair_sm[];
    __shared__ float2 sPos[kRsPosChunk], sC[kRsPosChunk];
    __shared__ int sRed[2];
    const int64_t j = min((int64_t)blockIdx.x * kRsPairTargets + threadIdx.x, P.M - 1);
    RsMoments v{P, R, cbar, sC, R.evec + (size_t)j * R.slab * kRsRecord, s0, -1};
    v.clear();
    const int p0 = s0 + blockIdx.z * R.part, p1 = min(R.nint, p0 + R.part);
    rs_pair_block<-1>(P, R, p0, p1, pair_sm, sPos, sRed, v);
    rs_pair_block<1>(P, R, p0, p1, pair_sm, sPos, sRed, v);
    v.flush();
}

// The sums over a slab's intervals: out_{l,m} = sum_{iv} sum_r a_{iv,m,r} F_{l,iv,r}, in float pairs per interval
// (r = 0, 1 as pairs, the rest single, as the fold's e-vectors), added up over the intervals in three floats (acc3_add), which
// hold more than FP64's bits.  A block takes 64 outputs, two to a lane, a run of the slab's intervals
// (blockIdx.z) and a group of steps (blockIdx.y); it stages records and coefficients of 8 intervals at a time (two
// buffers, asynchronous copies).  Warp w takes the group's steps w, w + nwarps, .., four at most, so that the warps'
// work is even.  sums: [blockIdx.z][m][M], carried from slab to slab; k_rs_unfold_add puts them into the ring.
// Bound by FP32 issue, 52 instructions per output, interval and m: 30,000 outputs and 676 intervals 1.5 ms,
// of which the FP32 pipe needs 0.7 (one run of intervals with four warps' steps of eight: 3.3 ms, 469 blocks in two
// uneven rounds).  11-bit slices on the tensor cores took 0.84 ms, held moments and coefficients in common
// units and the sums as pairs, and gave NaN at p = 16.
constexpr int kRsOutputs = 64;
constexpr int kRsOutPer = 4;
constexpr int kRsOutWarps = 10;                       // 40 steps to a group at most: one group for windows of 36 steps
constexpr int kRsOutTile = 8;
constexpr int kRsOutRow = kRsOutTile * kRsRecord + 4;
constexpr int kRsOutRows = kRsOutputs * kRsOutRow;    // floats of a tile's records
int rs_unfold_groups(int m_max) { return (m_max + kRsOutPer * kRsOutWarps - 1) / (kRsOutPer * kRsOutWarps); }
int rs_unfold_warps(int m_max) {
    const int g = rs_unfold_groups(m_max) * kRsOutPer;
    return (m_max + g - 1) / g;
}
size_t rs_unfold_smem() {
    return (size_t)2 * (kRsOutRows * sizeof(float) + kRsOutTile * kRsOutPer * kRsOutWarps * 3 * sizeof(float4));
}
// runs of a slab's intervals: enough blocks for the chip (six resident rounds) where there are few outputs
int rs_unfold_runs(int64_t M, int slab, int sms) {
    const int64_t gx = (M + kRsOutputs - 1) / kRsOutputs;
    return (int)std::max<int64_t>(1, std::min<int64_t>(slab / (2 * kRsOutTile), (12 * (int64_t)sms + gx - 1) / gx));
}
__global__ void __launch_bounds__(32 * kRsOutWarps, 2) k_rs_unfold(DevPlan P, RangeDev R, int s0, int s1,
                                                                  double* __restrict__ sums) {
    extern __shared__ __align__(16) float unfold_sm[];       // 2 x records, 2 x coefficients [interval][step][3]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarps = blockDim.x >> 5, steps = nwarps * kRsOutPer;
    const int64_t l0 = (int64_t)blockIdx.x * kRsOutputs;
    const int mg = 1 + blockIdx.y * steps, mfirst = mg + warp;               // the group's and the warp's first step
    float4* const sCoef = (float4*)(unfold_sm + 2 * kRsOutRows);
    sums += (int64_t)blockIdx.z * (R.nm - 1) * P.M;
    // this block's tiles of the slab
    const int ntile = (s1 - s0 + kRsOutTile - 1) / kRsOutTile;
    const int t0 = (int)((int64_t)ntile * blockIdx.z / gridDim.z), t1 = (int)((int64_t)ntile * (blockIdx.z + 1) / gridDim.z);
    float acc[kRsOutPer][2][3];
#pragma unroll
    for (int i = 0; i < kRsOutPer; i++)
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int m = mfirst + i * nwarps;
            const int64_t l = l0 + lane + 32 * u;
            rs::acc3_set(s0 > 0 && m < R.nm && l < P.M ? sums[(int64_t)(m - 1) * P.M + l] : 0.0, acc[i][u][0], acc[i][u][1],
                         acc[i][u][2]);
        }
    auto copy = [&](void* dst, const void* src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
    };
    auto fetch = [&](int tile) {
        const int i0 = s0 + kRsOutTile * tile, n = min(kRsOutTile, s1 - i0), buf = tile & 1;
        constexpr int rowq = kRsOutTile * kRsRecord / 4;
        const float* src = R.evec + ((size_t)l0 * R.slab + (i0 - s0)) * kRsRecord;
        for (int i = t; i < kRsOutputs * rowq; i += blockDim.x) {
            const int r = i / rowq, o = i - r * rowq;
            if (o < n * (kRsRecord / 4) && l0 + r < P.M)
                copy(unfold_sm + buf * kRsOutRows + r * kRsOutRow + 4 * o, src + (size_t)r * R.slab * kRsRecord + 4 * o);
        }
        const int rows = 3 * min(steps, R.nm - mg);          // (the steps of an interval lie together)
        for (int k = warp; k < n; k += nwarps) {
            const float4* c = (const float4*)R.coef + ((size_t)(i0 + k) * R.nm + mg) * 3;
            for (int i = lane; i < rows; i += 32) copy(sCoef + (buf * kRsOutTile + k) * steps * 3 + i, c + i);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (t0 < t1) fetch(t0);
    for (int tile = t0; tile < t1; tile++) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                              // this tile has arrived, the other buffers are free
        if (tile + 1 < t1) fetch(tile + 1);
        const int i0 = s0 + kRsOutTile * tile, buf = tile & 1;
        const float* rec0 = unfold_sm + buf * kRsOutRows + lane * kRsOutRow;
        for (int k = 0; k < min(kRsOutTile, s1 - i0); k++) {
            const int m0 = __ldg(R.mr + 2 * (i0 + k)), m1 = __ldg(R.mr + 2 * (i0 + k) + 1);
            if (mfirst + (kRsOutPer - 1) * nwarps < m0) continue;
            float4 a[2], b[2];
            float2 c[2];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const float* rec = rec0 + 32 * u * kRsOutRow + k * kRsRecord;
                a[u] = *(const float4*)rec;
                b[u] = *(const float4*)(rec + 4);
                c[u] = *(const float2*)(rec + 8);
            }
            const float4* cf = sCoef + ((buf * kRsOutTile + k) * steps + warp) * 3;
#pragma unroll
            for (int i = 0; i < kRsOutPer; i++) {
                const int m = mfirst + i * nwarps;
                if (m < m0 || m > m1) continue;
                const float4 c01 = cf[3 * i * nwarps], c23 = cf[3 * i * nwarps + 1], c47 = cf[3 * i * nwarps + 2];
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    float h, l;
                    rs::moments_sum(h, l, rs::F4{c01.x, c01.y, c01.z, c01.w}, rs::F4{c23.x, c23.y, c23.z, c23.w},
                                    rs::F4{c47.x, c47.y, c47.z, c47.w}, rs::F4{a[u].x, a[u].y, a[u].z, a[u].w},
                                    rs::F4{b[u].x, b[u].y, b[u].z, b[u].w}, c[u].x, c[u].y);
                    rs::acc3_add(acc[i][u][0], acc[i][u][1], acc[i][u][2], h, l);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kRsOutPer; i++)
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int m = mfirst + i * nwarps;
            const int64_t l = l0 + lane + 32 * u;
            if (m < R.nm && l < P.M) sums[(int64_t)(m - 1) * P.M + l] = rs::acc3_value(acc[i][u][0], acc[i][u][1], acc[i][u][2]);
        }
}

// the runs' sums in order into the ring: sigmabar_l^{n+1-m} += sum_z sums[z][m][l] (blockIdx.y: m - 1)
__global__ void k_rs_unfold_add(DevPlan P, RangeDev R, int runs, int64_t n, const double* __restrict__ sums, double* __restrict__ sb) {
    const int m = 1 + blockIdx.y;
    double* out = sb + (int64_t)ring_slot(n + 1 - m, P.ring) * P.M;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < P.M; l += (int64_t)gridDim.x * blockDim.x) {
        double v = 0.0;
        for (int z = 0; z < runs; z++) v += __ldg(sums + ((int64_t)z * (R.nm - 1) + m - 1) * P.M + l);
        if (v != 0.0) out[l] += v;
    }
}

// Transposed implicit solve.  With S_jl = (beta_j / 2) Q_0(d_jl), (I + S)^T rb = b is
// rb = y / beta with (I + S) y = beta b (beta > 0), so the forward Jacobi sweeps solve it on the
// right-hand side beta b.  Set-up: that right-hand side (k_rs_jacobi reads it as P.rhs) and the
// first iterate rhs / (1 + S_jj); b = sigmabar^{n+1}, taken out of its ring slot.
__global__ void k_rs_adj_init(DevPlan P, RangeDev R, double* __restrict__ slot_vals, double* __restrict__ rhs) {
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < 2 * (kRsMaxIter + 1); i += blockDim.x) R.stats[i] = 0ull;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P.M; j += (int64_t)gridDim.x * blockDim.x) {
        const double r = P.beta[j] * slot_vals[j];
        slot_vals[j] = 0.0;
        rhs[j] = r;
        const double x0 = r / R.diag[j];
        R.it64[0][j] = x0;
        const rs::Pair p2 = rs::split(x0);
        R.it2[0][2 * j] = p2.hi;
        R.it2[0][2 * j + 1] = p2.lo;
    }
}

// the converged sweep's y (as k_rs_store chooses it), then rb_j = y_j / beta_j and the step's
// gradient terms and adjoints as the block-solve form gives them (k_adj_solve):
//   grad_j += rb_j (sigma_j^{n+1} [+ g_j^{n+1}]) / beta_j,  gbar_j^{n+1} = -rb_j,  cbar_j = -beta_j rb_j / 2,
//   u_Hbar_j = -beta_j rb_j  (sigma_next, gbar_next in caller order; grad, gbar_next may be null)
__global__ void k_rs_adj_post(DevPlan P, RangeDev R, const double* __restrict__ sigma_next,
                              const double* __restrict__ g_next, double* grad, double* __restrict__ gbar_next,
                              double* cbar, double* uHbar) {
    int fin = kRsMaxIter;
    bool ok = false;
    for (int it = 1; it <= kRsMaxIter; it++) {
        const double dmax = rs_from_bits(__ldcg(R.stats + 2 * it)), smax = rs_from_bits(__ldcg(R.stats + 2 * it + 1));
        if (dmax <= kRsTol * smax) {
            fin = it;
            ok = true;
            break;
        }
    }
    const double* y = R.it64[fin & 1];
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P.M; j += (int64_t)gridDim.x * blockDim.x) {
        const double bj = P.beta[j];
        const double rb = __ldcg(y + j) / bj;
        const int jc = P.perm[j];
        if (grad) grad[j] += rb * (g_next ? sigma_next[jc] + g_next[jc] : sigma_next[jc]) / bj;
        if (gbar_next) gbar_next[jc] = -rb;
        cbar[j] = -0.5 * bj * rb;
        uHbar[j] = -bj * rb;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && !ok) atomicCAS(P.status, 0, (int)WAVE1D_ENOTCONV);
}

// Transposed receiver read-out (eq. localSol2, every m including m = 0, FP64): for spring l and
// each receiver r in order, the extended indices of l inside r's window (those of the forward
// read-out), sigmabar_l^{n+1-m} += (1/2) Q_m(d) ubar_r.  One thread per spring and eighth of the m
// (blockIdx.y: m = y, y + 8, ..), so each output has one writer; no atomics.
__global__ void k_rs_adj_receivers(DevPlan P, RangeDev R, int64_t n, const double* __restrict__ ubar, double* sb) {
    const int64_t M = P.M;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < M; l += (int64_t)gridDim.x * blockDim.x) {
        for (int64_t r = 0; r < P.R; r++) {
            const int lo = R.r_win[2 * r], hi = R.r_win[2 * r + 1];
            for (int k = -1; k <= 1; k++) {
                const int64_t e = l + k * M;
                if (e < lo || e >= hi) continue;
                const double d = fabs(rs_xext(P, e) - P.xr[r]);
                if (!(d < R.delta)) continue;
                const int iv = rs_locate64(R, d);
                double T[8];
                rs_cheb_basis((d - __ldg(R.mid + iv)) * (double)__ldg(R.ih + iv), T);
                const int m0 = __ldg(R.mr0 + 2 * iv), m1 = __ldg(R.mr0 + 2 * iv + 1);
                for (int m = m0 + ((blockIdx.y - m0) & 7); m <= m1; m += 8) {
                    int64_t s = (n + 1 - m) % P.ring;
                    if (s < 0) s += P.ring;
                    sb[s * M + l] += 0.5 * rs_cheb_sum(R.cheb + ((size_t)iv * R.nm + m) * 8, T) * ubar[r];
                }
            }
        }
    }
}

}  // namespace wave1d
