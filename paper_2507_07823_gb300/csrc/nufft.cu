// Standalone NUFFTs of the history part (Sec. 3.1) on fixed points: the type-1 transform
// S_k = (1/2 pi) sum_j c_j e^{+i k x_j}, k = 0..K (eq. densco), and the type-2 transform
// u_j = sum_{|k| <= K} alpha_k e^{-i k x_j} with alpha_{-k} = conj(alpha_k) (eq. historySol1), each
// split into its spreading (A1) or interpolation (A6) pass and the FFT, with the same Kaiser-Bessel
// kernel, fine grid and deconvolution as the time-step plan.  A plan may hold many point sets
// (instances) with the same K; one launch per pass covers all of them.
//
// Two precisions:
//   FP64   kernel weights precomputed (w per point) and streamed from HBM.  Relative accuracy set
//          by tol, like the time-step plan.
//   mixed  each tap's kernel a Chebyshev series in the point's offset within its first cell
//          (fitted on the host to about 2e-7 of the kernel's peak); spreading by per-cell
//          Chebyshev moments and interpolation by per-cell Chebyshev sums of the grid, in FP32
//          with the dominant terms compensated; the FFT and the deconvolution stay FP64.  GB300
//          runs FP32 about 60 times faster than FP64, so these passes read little more than the
//          points' cells, offsets and values.
// Points are kept in an internal order sorted by first grid cell, instance by instance
// (wave1d_nufft_perm gives it).  Spreading: each instance's grid is cut into cell ranges, one
// block per range writes its grid reals complete (recomputing the sums of the w - 1 cells before
// the range), so clustered points, with hundreds per cell, spread over many blocks and lanes.
// Interpolation: blocks of consecutive points.  Neither uses atomics: the results do not depend
// on scheduling.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <string>
#include <type_traits>
#include <utility>
#include <vector>

#include "internal.h"
#include "nufft_host.h"
#include "nufft_units.cuh"
#include "device_common.cuh"
#include "../../include/wave1d.h"

using namespace wave1d;

namespace {

constexpr double kPiN = 3.14159265358979323846264338327950288;
constexpr int kMaxDegree = 16;      // polynomial degree limit of the mixed-precision kernel

thread_local std::string g_nu_error;

int nfail(int code, const std::string& msg) {
    g_nu_error = msg;
    return code;
}

// ---------------------------------------------------------------------------------------------
// Moving between FP64 and FP32 with integer operations on the IEEE-754 bit patterns.  On this GPU
// the FP64 pipe, conversions included, issues about 60 times slower than FP32, so the mixed passes
// convert each value with a few integer operations instead.
// ---------------------------------------------------------------------------------------------
// double -> float, rounded to nearest (ties away from zero); magnitudes below 2^-126 give a signed
// zero, magnitudes above the float range a signed infinity
__device__ __forceinline__ float nu_f64_to_f32(double d) {
    unsigned hw = (unsigned)__double2hiint(d);
    const unsigned lw = (unsigned)__double2loint(d);
    const unsigned lr = lw + 0x10000000u;                 // half a unit of the 29 dropped bits
    hw += lr < lw ? 1u : 0u;                              // a carry may step the exponent: still exact
    const unsigned s = hw & 0x80000000u;
    const int e = (int)((hw >> 20) & 0x7ffu) - 896;       // biased float exponent
    const unsigned b = s | ((unsigned)e << 23) | ((hw & 0xfffffu) << 3) | (lr >> 29);
    return __uint_as_float(e <= 0 ? s : (e >= 255 ? (s | 0x7f800000u) : b));
}
// float -> double, exact for zero and normal floats (subnormals give a signed zero)
__device__ __forceinline__ double nu_f32_to_f64(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xffu, s = b & 0x80000000u;
    const unsigned hw = e == 0u ? s : (e == 255u ? (s | 0x7ff00000u) : (s | ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3)));
    const unsigned lw = (e == 0u || e == 255u) ? 0u : (b << 29);
    return __hiloint2double((int)hw, (int)lw);
}

// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ void nu_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (sh, sl) += (ph, pl)
__device__ __forceinline__ void nu_pair_add(float& sh, float& sl, float ph, float pl) {
    float s, t;
    nu_two_sum(sh, ph, s, t);
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(t, pl));
}

// Mixed-precision kernel: tap t (0 <= t < w) of a point with offset variable y in [-1, 1] has the
// value psi_t(y) = sum_d a[t][d] T_d(y), a Chebyshev series of degree D fitted on the host (well
// conditioned: sum_d |a[t][d]| stays near max psi_t, so FP32 evaluation loses little).  The
// kernel is even, so psi_{w-1-t}(y) = psi_t(-y) and a[w-1-t][d] = (-1)^d a[t][d]: the host fits
// the first half of the taps and mirrors them.  The table is a kernel parameter, so the unrolled
// FMAs take their coefficients straight from the constant bank.
struct NuPoly {
    float c[16][kMaxDegree + 1];
};
template <int D>
struct NuCheb {                    // T_0(y) .. T_D(y) by the three-term recurrence
    float T[D + 1];
    __device__ __forceinline__ explicit NuCheb(float y) {
        const float y2 = __fadd_rn(y, y);
        T[0] = 1.f;
        T[1] = y;
#pragma unroll
        for (int d = 2; d <= D; d++) T[d] = __fmaf_rn(y2, T[d - 1], -T[d - 2]);
    }
};
// all w kernel values of a point: even and odd parts of the first half, mirrored
template <int W, int D>
__device__ __forceinline__ void nu_taps(const NuPoly& P, const NuCheb<D>& ch, float (&psi)[W]) {
#pragma unroll
    for (int t = 0; t < (W + 1) / 2; t++) {
        float e = P.c[t][0], o = __fmul_rn(P.c[t][1], ch.T[1]);
#pragma unroll
        for (int d = 2; d <= D; d += 2) e = __fmaf_rn(P.c[t][d], ch.T[d], e);
#pragma unroll
        for (int d = 3; d <= D; d += 2) o = __fmaf_rn(P.c[t][d], ch.T[d], o);
        psi[t] = __fadd_rn(e, o);
        if (W - 1 - t != t) psi[W - 1 - t] = __fsub_rn(e, o);
    }
}

// ---------------------------------------------------------------------------------------------
// Spreading (A1).  The points are sorted by first cell; the grid is cut into cell ranges, each
// range handled by one block that writes its grid reals complete (below).  No atomics: the result
// does not depend on scheduling, and a dense cluster (hundreds of points per cell) spreads over
// many ranges and lanes.
// ---------------------------------------------------------------------------------------------

// Mixed precision by Chebyshev moments.  With psi_t(y) = sum_d a[t][d] T_d(y),
//   G[g] = sum_t sum_{q: i0_q = g - t} c_q psi_t(y_q) = sum_t sum_d a[t][d] M_d(g - t),
//   M_d(f) = sum_{q: i0_q = f} c_q T_d(y_q),
// so a point costs D + 1 FMAs (its moments) and each grid real w (D + 1) multiply-adds.
//
// Work split: the grid is tiled by cell ranges [c0, c0 + nc) (at most kRangeCells cells, and at
// most kRangePoints points counting the w - 1 cells before the range, the halo).  A block takes a
// range: it stages the (c, y) of the points whose first cell lies in [c0 - w + 1, c0 + nc) in
// shared memory (one or two slices of the sorted points: the halo of the first range wraps round
// the periodic box), gives each of those nc + w - 1 cells a group of G lanes that accumulate the
// cell's moments (a fixed shuffle tree closes each group), and then writes every grid real of its
// range complete.  The halo cells' moments are computed twice, by this block and by the
// previous one; in exchange no block depends on another (no partials, atomics or second pass),
// each grid real is written once, and the result does not depend on scheduling.  A range whose
// points exceed kStage (a cell holding thousands of points) reads them from global memory.
// M_0 and the d = 0 terms are compensated FP32 pairs (they carry the magnitude); the higher
// moments cancel over a cell and carry small coefficients, so they are plain FP32.
constexpr int kStage = 2048;        // staging capacity (points) of a range
constexpr int kRangePoints = 2048;  // points a range is cut at, halo included (one cell may exceed it)
constexpr int kRangeCells = 240;    // cells of a mixed range (w - 1 halo cells more fit one thread each)
constexpr int kRangePoints64 = 4096;  // FP64: its halo costs FP64 FMAs, so fewer, larger ranges
constexpr int kEmptyCells = 8192;   // cells of a range no point reaches (zeros only)
template <int W, int D>
__global__ void __launch_bounds__(kUnitThreads) k_nu_spread_mixed(const NuRange* __restrict__ ranges,
                                                                  const int32_t* __restrict__ runs,
                                                                  const double* __restrict__ c,
                                                                  const float* __restrict__ soff, const NuPoly P,
                                                                  double* __restrict__ grid) {
    constexpr int R = (D + 2 + 3) / 4 * 4;            // moment row: M_0 (hi, lo), M_1 .. M_D, padded to float4
    constexpr int kPer = kStage / kUnitThreads;
    __shared__ int rp[kRangeCells + 16 + 1];
    __shared__ float2 cy[kStage];
    __shared__ __align__(16) float mo[kRangeCells + 16][R];
    const NuRange u = ranges[blockIdx.x];
    const int nr = u.nc + W - 1, np = u.na + u.nb;
    if (np == 0) {                                    // no point reaches the range: zeros
        for (int l = threadIdx.x; l < u.nc; l += kUnitThreads) grid[u.c0 + l] = 0.0;
        return;
    }
    const bool staged = np <= kStage;
    if ((int)threadIdx.x <= nr) rp[threadIdx.x] = __ldg(runs + u.roff + threadIdx.x);
    if (staged) {
        double cd[kPer];
        float sv[kPer];
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const int q = (int)threadIdx.x + i * kUnitThreads;
            if (q < np) {
                const int j = q < u.na ? u.a0 + q : u.b0 + (q - u.na);
                cd[i] = __ldcs(c + j);
                sv[i] = __ldcs(soff + j);
            }
        }
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const int q = (int)threadIdx.x + i * kUnitThreads;
            if (q < np) cy[q] = make_float2(nu_f64_to_f32(cd[i]), __fmaf_rn(2.f, sv[i], -1.f));
        }
    }
    __syncthreads();
    const int G = 1 << u.lg, f = (int)threadIdx.x >> u.lg, gl = (int)threadIdx.x & (G - 1);
    float m[D + 1];
#pragma unroll
    for (int d = 0; d <= D; d++) m[d] = 0.f;
    if (f < nr) {
        const int q1 = rp[f + 1];
        for (int q = rp[f] + gl; q < q1; q += G) {
            float2 v;
            if (staged) {
                v = cy[q];
            } else {
                const int j = q < u.na ? u.a0 + q : u.b0 + (q - u.na);
                v = make_float2(nu_f64_to_f32(__ldcs(c + j)), __fmaf_rn(2.f, __ldcs(soff + j), -1.f));
            }
            const NuCheb<D> ch(v.y);
            m[0] = __fadd_rn(m[0], v.x);
#pragma unroll
            for (int d = 1; d <= D; d++) m[d] = __fmaf_rn(ch.T[d], v.x, m[d]);
        }
    }
    float m0l = 0.f;
    for (int o = G >> 1; o > 0; o >>= 1) {
        nu_pair_add(m[0], m0l, __shfl_xor_sync(0xffffffffu, m[0], o), __shfl_xor_sync(0xffffffffu, m0l, o));
#pragma unroll
        for (int d = 1; d <= D; d++) m[d] = __fadd_rn(m[d], __shfl_xor_sync(0xffffffffu, m[d], o));
    }
    if (gl == 0 && f < nr) {
        mo[f][0] = m[0];
        mo[f][1] = m0l;
#pragma unroll
        for (int d = 1; d <= D; d++) mo[f][d + 1] = m[d];
    }
    __syncthreads();
    if ((int)threadIdx.x < u.nc && rp[threadIdx.x + W] == rp[threadIdx.x]) {
        grid[u.c0 + threadIdx.x] = 0.0;               // none of the w cells feeding it holds a point
    } else if ((int)threadIdx.x < u.nc) {
        // grid real c0 + l takes tap t of cell c0 + l - t, i.e. run (l + w - 1) - t
        const int l = threadIdx.x;
        float h = 0.f, lo = 0.f, r = 0.f;
#pragma unroll
        for (int t = 0; t < W; t++) {
            float mf[R];
#pragma unroll
            for (int k = 0; k < R; k += 4)
                *reinterpret_cast<float4*>(mf + k) = *reinterpret_cast<const float4*>(&mo[l + W - 1 - t][k]);
            const float p = __fmul_rn(P.c[t][0], mf[0]);
            const float e = __fmaf_rn(P.c[t][0], mf[1], __fmaf_rn(P.c[t][0], mf[0], -p));
            nu_pair_add(h, lo, p, e);
#pragma unroll
            for (int d = 1; d <= D; d++) r = __fmaf_rn(P.c[t][d], mf[d + 1], r);
        }
        nu_pair_add(h, lo, r, 0.f);
        grid[u.c0 + l] = nu_f32_to_f64(h) + nu_f32_to_f64(lo);
    }
}

// FP64 spreading on the same cell ranges, one block per range (spread64_unit, nufft_units.cuh).
// Like the mixed pass, no block depends on another.
template <int W>
__global__ void __launch_bounds__(kUnitThreads) k_nu_spread64(const NuRange* __restrict__ ranges,
                                                              const int32_t* __restrict__ runs,
                                                              const double* __restrict__ c,
                                                              const double* __restrict__ ker,
                                                              double* __restrict__ grid) {
    __shared__ int rp[kSpread64Runs];
    __shared__ double seg[kRangeCells64 + 16][W];
    spread64_unit<W>(ranges[blockIdx.x], runs, c, ker, grid, seg, rp);
}

// ---------------------------------------------------------------------------------------------
// FP64 spreading of a standalone plan, in two launches over all instances.  k_nu_tap_sums: each cell's points
// are cut into segments of at most kSegPoints, a half-warp per segment with a lane per tap, so the
// weights (w doubles a point, the pass's stream) are read in order; the partial sums S_t of every
// segment go to memory.  k_nu_assemble: grid real g = sum_t S_t(g - t) over the segments of w cells.
// Bound by the FP64 pipe (90 % busy): 44 us and 9 us at 1e6 clustered points and w = 11.  The form by
// cell ranges (spread64_unit) recomputes its halos, rounds cells up to whole groups of lanes and reads the
// weights lane by lane, 88 bytes apart: 67 us there.  (Compensated FP32 pairs in place of FP64 here: 43 us
// with unequal segments, as splitting each weight costs what they save.)
// ---------------------------------------------------------------------------------------------
constexpr int kSegPoints = 64;      // points of a segment at most, unless the autotuner finds better

template <int W>
__global__ void __launch_bounds__(256) k_nu_tap_sums(const int32_t* __restrict__ seg, int64_t nseg,
                                                     const double* __restrict__ c, const double* __restrict__ ker,
                                                     double* __restrict__ S) {
    const int64_t sg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
    const int t = threadIdx.x & 15;
    if (sg >= nseg || t >= W) return;
    const int j0 = __ldg(seg + sg), np = __ldg(seg + sg + 1) - j0;
    const double* kr = ker + (int64_t)j0 * W + t;
    const double* cr = c + j0;
    double out = 0.0;
    int i = 0;
    for (; i + 8 <= np; i += 8) {
        double k[8], v[8];
#pragma unroll
        for (int p = 0; p < 8; p++) {
            k[p] = __ldcs(kr + (i + p) * W);
            v[p] = __ldg(cr + i + p);
        }
#pragma unroll
        for (int p = 0; p < 8; p++) out = fma(k[p], v[p], out);
    }
    {
        double k[7], v[7];
#pragma unroll
        for (int p = 0; p < 7; p++) {
            k[p] = i + p < np ? __ldcs(kr + (i + p) * W) : 0.0;
            v[p] = i + p < np ? __ldg(cr + i + p) : 0.0;
        }
#pragma unroll
        for (int p = 0; p < 7; p++)
            if (i + p < np) out = fma(k[p], v[p], out);
    }
    S[sg * W + t] = out;
}

// cseg: first segment of each cell (instance x nf + cell), one more at the end
template <int W>
__global__ void __launch_bounds__(256) k_nu_assemble(const int32_t* __restrict__ cseg, const double* __restrict__ S,
                                                     double* __restrict__ grid, int64_t cells, int nf) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= cells) return;
    const int64_t gb = g & ~(int64_t)(nf - 1);
    int s0[W], s1[W];
#pragma unroll
    for (int t = 0; t < W; t++) {
        const int64_t f = gb | ((g - t) & (nf - 1));
        s0[t] = __ldg(cseg + f);
        s1[t] = __ldg(cseg + f + 1);
    }
    double a = 0.0;
#pragma unroll
    for (int t = 0; t < W; t++)
        for (int s = s0[t]; s < s1[t]; s++) a += __ldg(S + (int64_t)s * W + t);
    grid[g] = a;
}

// ---------------------------------------------------------------------------------------------
// The FFTs of the transforms (L = L1 L2 complex points per instance, z[i2 + L2 i1] -> X[k1 + L1 k2]),
// blockIdx.y = instance: one launch per pass covers all instances.  A block takes two lines at a time
// (two adjacent columns or rows: 32-byte pieces, and two threads per butterfly of both lines,
// fft_lines), type-1's row pass forms S_k from its pair of rows and type-2's column pass forms the
// spectrum as it loads, so neither takes a pass over memory of its own.  Bound by the FP64 pipe: 2
// instructions per point, component and stage; 64 instances of L = 8192 both ways about 90 us of it.
// One instance at a time, six launches each, the 64 took 2.5 ms.
// ---------------------------------------------------------------------------------------------
constexpr int kFftThreads = 256;
size_t nu_fft_smem(int N) { return (size_t)(2 * N + N / 2) * sizeof(double2); }

__device__ __forceinline__ void nu_line_twiddles(double2* twN, const double2* __restrict__ tw, int L, int N, int sign) {
    for (int j = threadIdx.x; j < N / 2; j += blockDim.x) {
        double2 w = __ldg(tw + (int64_t)j * (L / N));
        if (sign < 0) w.y = -w.y;
        twN[j] = w;
    }
}

// columns 2c, 2c + 1 (c = blockIdx.x) of z, from load(i2, i1): FFT over i1, twiddle -> Y[k1 L2 + i2]
template <int SIGN, typename Load>
__device__ __forceinline__ void nu_columns(Load load, double2* __restrict__ Y, const double2* __restrict__ tw, int L,
                                           int L1, int L2, double2* sm) {
    double2 *a = sm, *b = sm + L1, *twN = sm + 2 * L1;
    const int logL1 = 31 - __clz(L1), c = 2 * blockIdx.x;
    nu_line_twiddles(twN, tw, L, L1, SIGN);
    for (int t = threadIdx.x; t < 2 * L1; t += blockDim.x)
        (t & 1 ? b : a)[__brev(t >> 1) >> (32 - logL1)] = load(c + (t & 1), t >> 1);
    __syncthreads();
    fft_lines(a, b, twN, L1, logL1);
    for (int t = threadIdx.x; t < 2 * L1; t += blockDim.x) {
        const int i2 = c + (t & 1), k1 = t >> 1;
        double2 w = __ldg(tw + (((int64_t)i2 * k1) & (L - 1)));
        if (SIGN < 0) w.y = -w.y;
        Y[(int64_t)k1 * L2 + i2] = cmul((t & 1 ? b : a)[k1], w);
    }
}

__global__ void __launch_bounds__(kFftThreads) k_nu_cols1(const double2* __restrict__ grids, double2* __restrict__ works,
                                                          const double2* __restrict__ tw, int L, int L1, int L2) {
    extern __shared__ __align__(16) double2 nu_sm[];
    const double2* z = grids + (int64_t)blockIdx.y * L;
    nu_columns<1>([&](int i2, int i1) { return __ldg(z + i2 + (int64_t)L2 * i1); }, works + (int64_t)blockIdx.y * L, tw, L,
                  L1, L2, nu_sm);
}

// type-2 spectrum for the inverse real FFT: Zs[k] = alpha_k (f3 + i f4), Zs[L - k] = conj(alpha_k)
// (f5 + i f6), zero where no mode lands
__global__ void __launch_bounds__(kFftThreads) k_nu_cols2(const double* __restrict__ alphas, double2* __restrict__ works,
                                                          const double* __restrict__ modefac,
                                                          const double2* __restrict__ tw, int K, int L, int L1, int L2) {
    extern __shared__ __align__(16) double2 nu_sm[];
    const double* alpha = alphas + (int64_t)blockIdx.y * 2 * (K + 1);
    nu_columns<-1>(
        [&](int i2, int i1) {
            const int idx = i2 + L2 * i1;
            if (idx <= K) {
                const double* f = modefac + 8 * (int64_t)idx;
                return cmul(make_double2(alpha[2 * idx], alpha[2 * idx + 1]), make_double2(__ldg(f + 3), __ldg(f + 4)));
            }
            if (idx >= L - K) {
                const int k = L - idx;
                const double* f = modefac + 8 * (int64_t)k;
                return cmul(make_double2(alpha[2 * k], -alpha[2 * k + 1]), make_double2(__ldg(f + 5), __ldg(f + 6)));
            }
            return make_double2(0.0, 0.0);
        },
        works + (int64_t)blockIdx.y * L, tw, L, L1, L2, nu_sm);
}

// rows k1 and L1 - k1 (k1 = blockIdx.x <= L1 / 2): FFT over i2, then S_k of the rows' modes from the
// half-length FFT (E, O split) with the deconvolution factors, S_k = f0 E_k + (f1 + i f2) O_k; the
// partner Z_{L-k} lies in the other row (in the same one for k1 = 0 and L1 / 2)
__global__ void __launch_bounds__(kFftThreads) k_nu_rows1(const double2* __restrict__ works, double* __restrict__ Ss,
                                                          const double* __restrict__ modefac,
                                                          const double2* __restrict__ tw, int K, int L, int L1, int L2,
                                                          bool wide) {
    extern __shared__ __align__(16) double2 nu_sm[];
    double2 *a = nu_sm, *b = nu_sm + L2, *twN = nu_sm + 2 * L2;
    const double2* Y = works + (int64_t)blockIdx.y * L;
    double* S = Ss + (int64_t)blockIdx.y * 2 * (K + 1);
    const int logL2 = 31 - __clz(L2), k1 = blockIdx.x, k1p = (L1 - k1) % L1;
    const bool pair = k1p != k1;
    nu_line_twiddles(twN, tw, L, L2, 1);
    for (int i2 = threadIdx.x; i2 < L2; i2 += blockDim.x) {
        const int rv = __brev(i2) >> (32 - logL2);
        a[rv] = __ldg(Y + (int64_t)k1 * L2 + i2);
        if (pair) b[rv] = __ldg(Y + (int64_t)k1p * L2 + i2);
    }
    __syncthreads();
    fft_lines(a, pair ? b : nullptr, twN, L2, logL2);
    for (int t = threadIdx.x; t < (pair ? 2 : 1) * L2; t += blockDim.x) {
        const bool second = t >= L2;
        const int k2 = second ? t - L2 : t, k = (second ? k1p : k1) + L1 * k2;
        if (k > K) continue;
        const double2 zk = (second ? b : a)[k2];
        const double2 zm = (pair ? (second ? a : b) : a)[k1 == 0 ? (L2 - k2) & (L2 - 1) : L2 - 1 - k2];
        const double* f = modefac + 8 * (int64_t)k;
        const double f0 = __ldg(f);
        const double2 E = make_double2(0.5 * (zk.x + zm.x), 0.5 * (zk.y - zm.y));
        const double2 D = make_double2(0.5 * (zk.x - zm.x), 0.5 * (zk.y + zm.y));
        const double2 O = make_double2(D.y, -D.x);
        const double2 s = cadd(make_double2(f0 * E.x, f0 * E.y), cmul(make_double2(__ldg(f + 1), __ldg(f + 2)), O));
        if (wide) {
            ((double2*)S)[k] = s;
        } else {
            S[2 * k] = s.x;
            S[2 * k + 1] = s.y;
        }
    }
}

// rows 2c, 2c + 1: FFT over i2 (sign -) -> grid points k1 + L1 k2
__global__ void __launch_bounds__(kFftThreads) k_nu_rows2(const double2* __restrict__ works, double2* __restrict__ grids,
                                                          const double2* __restrict__ tw, int L, int L1, int L2) {
    extern __shared__ __align__(16) double2 nu_sm[];
    double2 *a = nu_sm, *b = nu_sm + L2, *twN = nu_sm + 2 * L2;
    const double2* Y = works + (int64_t)blockIdx.y * L;
    double2* X = grids + (int64_t)blockIdx.y * L;
    const int logL2 = 31 - __clz(L2), c = 2 * blockIdx.x;
    nu_line_twiddles(twN, tw, L, L2, -1);
    for (int t = threadIdx.x; t < 2 * L2; t += blockDim.x) {
        const int r = t >= L2, i2 = r ? t - L2 : t;
        (r ? b : a)[__brev(i2) >> (32 - logL2)] = __ldg(Y + (int64_t)(c + r) * L2 + i2);
    }
    __syncthreads();
    fft_lines(a, b, twN, L2, logL2);
    for (int t = threadIdx.x; t < 2 * L2; t += blockDim.x) X[c + (t & 1) + (int64_t)L1 * (t >> 1)] = (t & 1 ? b : a)[t >> 1];
}

// FP64 interpolation, tiles of kInterpTile consecutive points (interp64_unit, nufft_units.cuh).
template <int W>
__global__ void __launch_bounds__(kInterpTile) k_nu_interp64(const double* __restrict__ grid, double* __restrict__ u,
                                                             const int32_t* __restrict__ i0,
                                                             const double* __restrict__ ker, int64_t M, int nf) {
    __shared__ __align__(16) double ks[kInterpTile * W];
    interp64_unit<W>(blockIdx.x, grid, u, i0, ker, M, nf, ks);
}

// mixed interpolation (A6).  With psi_t(y) = sum_d a[t][d] T_d(y),
//   u_j = sum_t psi_t(y_j) G[i0_j + t] = sum_d T_d(y_j) H_d(i0_j),  H_d(i) = sum_t a[t][d] G[i + t],
// and H depends only on the first cell.  A block takes 1024 consecutive points (sorted by first
// cell, four per thread), converts the grid cells they reach to FP32 in shared memory, forms H
// for each of their first cells (W (D + 1) FMAs per cell), and then each point costs D + 1 FMAs.
// FP32 throughout (rounding of the order of the kernel's fit, below the requested tolerance).  A
// block whose points start in more than kHCells cells evaluates the taps per point instead.
constexpr int kHCells = 512;
constexpr int kInterpPer = 4;
template <int W, int D>
__global__ void __launch_bounds__(256) k_nu_interp_mixed(const double* __restrict__ grid, double* __restrict__ u,
                                                         const int32_t* __restrict__ first,
                                                         const float* __restrict__ soff, const NuPoly P, int64_t M,
                                                         int nf) {
    constexpr int R = (D + 1 + 3) / 4 * 4;            // H row, padded to float4
    __shared__ float gs[kHCells + 16];
    __shared__ __align__(16) float H[kHCells * R];
    __shared__ int fr[2];
    const int64_t base = (int64_t)blockIdx.x * (256 * kInterpPer);
    const int64_t last = M - 1 < base + 256 * kInterpPer - 1 ? M - 1 : base + 256 * kInterpPer - 1;
    int a[kInterpPer];
    float y[kInterpPer];
#pragma unroll
    for (int i = 0; i < kInterpPer; i++) {
        const int64_t j = base + threadIdx.x + i * 256;
        a[i] = j <= last ? __ldg(first + j) : 0;
        y[i] = j <= last ? __fmaf_rn(2.f, __ldcs(soff + j), -1.f) : 0.f;
        if (j == base) fr[0] = a[i];
        if (j == last) fr[1] = a[i];
    }
    __syncthreads();
    // cells are instance x nf + cell (nf a power of two): a block within one instance wraps inside
    // it; a block that straddles two instances takes the per-point path
    const int c0 = fr[0], ncell = fr[1] - c0 + 1, gbase = c0 & ~(nf - 1);
    const bool fits = ncell <= kHCells && (fr[1] & ~(nf - 1)) == gbase;   // the same in every thread
    if (fits) {
        for (int l = threadIdx.x; l < ncell + W - 1; l += 256)
            gs[l] = nu_f64_to_f32(__ldg(grid + (gbase | ((c0 + l) & (nf - 1)))));
        __syncthreads();
        for (int l = threadIdx.x; l < ncell; l += 256) {
            float g[W];
#pragma unroll
            for (int t = 0; t < W; t++) g[t] = gs[l + t];
#pragma unroll
            for (int d = 0; d <= D; d++) {
                float h = __fmul_rn(P.c[0][d], g[0]);
#pragma unroll
                for (int t = 1; t < W; t++) h = __fmaf_rn(P.c[t][d], g[t], h);
                H[l * R + d] = h;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kInterpPer; i++) {
        const int64_t j = base + threadIdx.x + i * 256;
        if (j > last) break;
        const NuCheb<D> ch(y[i]);
        float acc;
        if (fits) {
            float h[R];
#pragma unroll
            for (int k = 0; k < R; k += 4) *reinterpret_cast<float4*>(h + k) = *reinterpret_cast<const float4*>(H + (a[i] - c0) * R + k);
            acc = h[0];
#pragma unroll
            for (int d = 1; d <= D; d++) acc = __fmaf_rn(ch.T[d], h[d], acc);
        } else {
            float psi[W];
            nu_taps<W, D>(P, ch, psi);
            acc = 0.f;
            const int pb = a[i] & ~(nf - 1);
#pragma unroll
            for (int t = 0; t < W; t++)
                acc = __fmaf_rn(psi[t], nu_f64_to_f32(__ldg(grid + (pb | ((a[i] + t) & (nf - 1))))), acc);
        }
        __stcs(u + j, nu_f32_to_f64(acc));
    }
}

// compile-time kernel widths and polynomial degrees: FP64 takes w = 4..16; mixed precision
// (tol >= 1e-6) takes w = 4..7 with degrees 6, 8 or 10
constexpr int kMixedMaxW = 7;
template <int W, typename F>
bool nu_try_w(int w, F& f) {
    if (w != W) return false;
    f(std::integral_constant<int, W>{});
    return true;
}
template <typename F>
bool nu_with_w(int w, F&& f) {
    return nu_try_w<4>(w, f) || nu_try_w<5>(w, f) || nu_try_w<6>(w, f) || nu_try_w<7>(w, f) ||
           nu_try_w<8>(w, f) || nu_try_w<9>(w, f) || nu_try_w<10>(w, f) || nu_try_w<11>(w, f) ||
           nu_try_w<12>(w, f) || nu_try_w<13>(w, f) || nu_try_w<14>(w, f) || nu_try_w<15>(w, f) ||
           nu_try_w<16>(w, f);
}
template <typename F>
bool nu_with_mixed(int w, int D, F&& f) {
    auto wd = [&](auto wc, auto dc) {
        if (wc.value != w || dc.value != D) return false;
        f(wc, dc);
        return true;
    };
    using I4 = std::integral_constant<int, 4>;
    using I5 = std::integral_constant<int, 5>;
    using I6 = std::integral_constant<int, 6>;
    using I7 = std::integral_constant<int, 7>;
    using I8 = std::integral_constant<int, 8>;
    using I10 = std::integral_constant<int, 10>;
    return wd(I4{}, I6{}) || wd(I4{}, I8{}) || wd(I4{}, I10{}) || wd(I5{}, I6{}) || wd(I5{}, I8{}) ||
           wd(I5{}, I10{}) || wd(I6{}, I6{}) || wd(I6{}, I8{}) || wd(I6{}, I10{}) || wd(I7{}, I6{}) ||
           wd(I7{}, I8{}) || wd(I7{}, I10{});
}

}  // namespace

// How a plan's spreading is cut.  Ranges (mixed plans; FP64 plans of a batch, whose one-launch step spreads by
// them): cell ranges tiling every instance's grid, with their run tables.  Segments (FP64): `points` points of one
// cell at most, the first segment of every cell, tap sums.
struct NuSplit {
    int cells = 0, points = 0;       // the caps it was cut with (segments: one cell)
    NuRange* ranges = nullptr;
    int64_t nunits = 0;
    int32_t* runs = nullptr;
    int32_t *seg = nullptr, *cseg = nullptr;
    int64_t nseg = 0;
    double* tap_sums = nullptr;
};

struct wave1d_nufft_s {
    int device = 0;
    int precision = 0;
    int64_t M = 0;                   // points over all instances
    int B = 1;                       // instances (each with its own grid of nf reals)
    Params P{};
    int D = 0;                       // polynomial degree (mixed)
    double kernel_err = 0.0;         // max |Chebyshev series (FP32) - kernel| over the taps (mixed)
    cudaStream_t stream = nullptr;
    std::vector<int64_t> perm;       // internal point i -> caller index
    std::vector<void*> allocs;
    // points (internal order): first cell, offset in it (mixed), kernel weights (FP64)
    int32_t* first = nullptr;
    float* soff = nullptr;
    NuPoly poly{};                   // tap polynomials (mixed), passed to the kernels by value
    double* ker = nullptr;
    NuSplit split;                   // the work split of the spreading
    std::vector<int32_t> i0_host;    // points' first cells (sorted within each instance), for re-cutting
    std::vector<int64_t> off_host;   // instance offsets
    // FFT and deconvolution
    double *grid = nullptr, *work = nullptr, *twiddle = nullptr, *modefac = nullptr;
    int group = 1;                   // instances whose FFTs share a launch (their work arrays fit 256 MB)
};

namespace {

template <typename T>
int nu_upload(wave1d_nufft_t h, const std::vector<T>& v, T** out) {
    void* p = nullptr;
    size_t bytes = std::max<size_t>(1, v.size()) * sizeof(T);
    if (cudaMalloc(&p, bytes) != cudaSuccess) return nfail(WAVE1D_ENOMEM, "cudaMalloc failed");
    h->allocs.push_back(p);
    if (!v.empty() && cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
        return nfail(WAVE1D_ECUDA, "cudaMemcpy failed");
    *out = (T*)p;
    return WAVE1D_OK;
}

template <typename T>
int nu_alloc(wave1d_nufft_t h, size_t count, T** out) {
    void* p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(1, count) * sizeof(T)) != cudaSuccess)
        return nfail(WAVE1D_ENOMEM, "cudaMalloc failed");
    h->allocs.push_back(p);
    *out = (T*)p;
    return WAVE1D_OK;
}

void nu_free(wave1d_nufft_t h, void* p) {
    if (!p) return;
    h->allocs.erase(std::find(h->allocs.begin(), h->allocs.end(), p));
    cudaFree(p);
}

void nu_drop(wave1d_nufft_t h, NuSplit& s) {
    for (void* p : {(void*)s.ranges, (void*)s.runs, (void*)s.seg, (void*)s.cseg, (void*)s.tap_sums}) nu_free(h, p);
    s = NuSplit();
}

// ranges of at most `cells` cells and `points` points
int nu_cut_ranges(wave1d_nufft_t h, int cells, int points, NuSplit& s) {
    std::vector<NuRange> ranges;
    std::vector<int32_t> runs;
    nufft_ranges(h->i0_host, h->off_host.data(), h->B, h->P.nf, h->P.nufft_w, cells, points, kEmptyCells, kUnitThreads, ranges,
                 runs);
    s.cells = cells;
    s.points = points;
    s.nunits = (int64_t)ranges.size();
    int rc = nu_upload(h, ranges, &s.ranges);
    return rc ? rc : nu_upload(h, runs, &s.runs);
}

// segments of at most `points` points of one cell
int nu_cut_segments(wave1d_nufft_t h, int points, NuSplit& s) {
    const int64_t cells = (int64_t)h->B * h->P.nf;
    std::vector<int32_t> seg, cseg((size_t)cells + 1, 0);
    int64_t cell = 0;                                // cells below it know their first segment
    for (int b = 0; b < h->B; b++)
        for (int64_t i = h->off_host[b]; i < h->off_host[b + 1];) {
            int64_t e = i;
            while (e < h->off_host[b + 1] && h->i0_host[e] == h->i0_host[i]) e++;
            for (const int64_t at = (int64_t)b * h->P.nf + h->i0_host[i]; cell <= at; cell++) cseg[cell] = (int32_t)seg.size();
            const int64_t parts = (e - i + points - 1) / points;              // equal, as a warp takes two
            for (int64_t q = 0; q < parts; q++) seg.push_back((int32_t)(i + (e - i) * q / parts));
            i = e;
        }
    for (; cell <= cells; cell++) cseg[cell] = (int32_t)seg.size();
    s.cells = 1;
    s.points = points;
    s.nseg = (int64_t)seg.size();
    seg.push_back((int32_t)h->M);
    int rc;
    if ((rc = nu_upload(h, seg, &s.seg)) || (rc = nu_upload(h, cseg, &s.cseg))) return rc;
    return nu_alloc(h, (size_t)s.nseg * h->P.nufft_w, &s.tap_sums);
}

}  // namespace

namespace wave1d {
int nufft_build_ranges(wave1d_nufft_t h) {
    if (!h || h->precision != 0) return WAVE1D_EINVAL;
    if (h->split.ranges) return WAVE1D_OK;
    NuSplit s;
    const int rc = nu_cut_ranges(h, kRangeCells64, kRangePoints64, s);
    if (rc) {
        nu_drop(h, s);
        return rc;
    }
    h->split.ranges = s.ranges;
    h->split.runs = s.runs;
    h->split.nunits = s.nunits;
    return WAVE1D_OK;
}
int nufft_dev64(wave1d_nufft_t h, NuDev64& out) {
    if (!h || h->precision != 0) return WAVE1D_EINVAL;
    out.ranges = h->split.ranges;
    out.runs = h->split.runs;
    out.nunits = h->split.nunits;
    out.ker = h->ker;
    out.i0 = h->first;
    out.M = h->M;
    out.w = h->P.nufft_w;
    out.nf = h->P.nf;
    return WAVE1D_OK;
}
int nufft_spread_ranges(wave1d_nufft_t h, const double* c, double* grid) {
    if (!h || h->precision != 0 || !h->split.ranges) return WAVE1D_EINVAL;
    if (!nu_with_w(h->P.nufft_w, [&](auto wc) {
            k_nu_spread64<decltype(wc)::value><<<(unsigned)h->split.nunits, kUnitThreads, 0, h->stream>>>(h->split.ranges, h->split.runs,
                                                                                                   c, h->ker, grid);
        }))
        return nfail(WAVE1D_EUNSUPPORTED, "kernel width not built");
    return cudaGetLastError() == cudaSuccess ? WAVE1D_OK : nfail(WAVE1D_ECUDA, "spread launch failed");
}
}  // namespace wave1d

extern "C" {

int wave1d_nufft_plan(const double* x, int64_t M, int K, double tol, int precision, void* stream,
                      wave1d_nufft_t* out) {
    if (!out) return nfail(WAVE1D_EINVAL, "out is NULL");
    *out = nullptr;
    const int64_t off[2] = {0, M};
    return wave1d_nufft_plan_many(x, off, 1, K, tol, precision, stream, out);
}

int wave1d_nufft_plan_many(const double* x, const int64_t* offsets, int n_inst, int K, double tol, int precision,
                           void* stream, wave1d_nufft_t* out) {
    if (!out) return nfail(WAVE1D_EINVAL, "out is NULL");
    *out = nullptr;
    if (!x || !offsets || n_inst < 1 || K < 1 || !(tol > 0.0 && tol < 0.1) || (precision != 0 && precision != 1))
        return nfail(WAVE1D_EINVAL, "need x, offsets, n_instances >= 1, K >= 1, 0 < tol < 0.1, precision 0 or 1");
    if (offsets[0] != 0) return nfail(WAVE1D_EINVAL, "offsets[0] must be 0");
    for (int b = 0; b < n_inst; b++)
        if (offsets[b + 1] <= offsets[b]) return nfail(WAVE1D_EINVAL, "every instance needs at least one point");
    const int64_t M = offsets[n_inst];
    if (M > INT32_MAX / 32) return nfail(WAVE1D_EINVAL, "at most 2^26 points in all");
    if (precision == 1 && tol < 1e-6) return nfail(WAVE1D_EINVAL, "mixed precision needs tol >= 1e-6");
    wave1d_nufft_t h = new (std::nothrow) wave1d_nufft_s();
    if (!h) return nfail(WAVE1D_ENOMEM, "host allocation");
    auto cleanup = [&](int code) {
        wave1d_nufft_destroy(h);
        return code;
    };
    h->precision = precision;
    h->M = M;
    h->B = n_inst;
    h->stream = (cudaStream_t)stream;
    if (cudaGetDevice(&h->device) != cudaSuccess) return cleanup(nfail(WAVE1D_ECUDA, "no CUDA device"));
    Params& P = h->P;
    nufft_grid(P, K, tol, 0);
    if (P.L2 > 1024) return cleanup(nfail(WAVE1D_EUNSUPPORTED, "fine grid too large for this build (nf > 2^21)"));
    if ((int64_t)n_inst * P.nf > INT32_MAX / 2) return cleanup(nfail(WAVE1D_EINVAL, "instances x fine grid above 2^30"));
    const int w = P.nufft_w, nf = P.nf;
    // positions wrapped into [-pi, pi), kernel weights, internal order: instance by instance, each
    // sorted by first cell
    std::vector<double> xw(M);
    for (int64_t j = 0; j < M; j++) {
        double v = x[j];
        if (!std::isfinite(v)) return cleanup(nfail(WAVE1D_EINVAL, "non-finite position"));
        v = std::fmod(v + kPiN, 2.0 * kPiN);
        if (v < 0) v += 2.0 * kPiN;
        v -= kPiN;
        if (v >= kPiN) v -= 2.0 * kPiN;
        xw[j] = v;
    }
    std::vector<int32_t> i0c;
    std::vector<double> kerc;
    spread_weights(P, xw, i0c, kerc);
    h->perm.resize(M);
    std::iota(h->perm.begin(), h->perm.end(), 0);
    for (int b = 0; b < n_inst; b++)
        std::stable_sort(h->perm.begin() + offsets[b], h->perm.begin() + offsets[b + 1], [&](int64_t p, int64_t q) {
            return i0c[p] != i0c[q] ? i0c[p] < i0c[q] : xw[p] < xw[q];
        });
    std::vector<int32_t> i0(M), gfirst(M);           // cell in the instance; instance x nf + cell
    std::vector<double> xs(M);
    for (int b = 0; b < n_inst; b++)
        for (int64_t i = offsets[b]; i < offsets[b + 1]; i++) {
            i0[i] = i0c[h->perm[i]];
            gfirst[i] = b * nf + i0[i];
            xs[i] = xw[h->perm[i]];
        }
    int rc;
    if (precision == 0) {
        std::vector<double> ker((size_t)M * w);
        for (int64_t i = 0; i < M; i++)
            std::memcpy(&ker[(size_t)i * w], &kerc[(size_t)h->perm[i] * w], sizeof(double) * w);
        if ((rc = nu_upload(h, ker, &h->ker))) return cleanup(rc);
    } else {
        // offsets s = first - u + w/2 in [0, 1), y = 2 s - 1; tap t's kernel as a polynomial in y
        std::vector<float> soff(M);
        for (int64_t i = 0; i < M; i++) {
            const double u = (xs[i] + kPiN) / P.h_f;
            const double fst = std::ceil(u - 0.5 * w);
            soff[i] = (float)(fst - u + 0.5 * w);
        }
        const int ns = 96;
        std::vector<double> ys(ns);
        for (int i = 0; i < ns; i++) ys[i] = std::cos(kPiN * (i + 0.5) / ns);
        const double inv_i0b = 1.0 / std::cyl_bessel_i(0.0, P.kb_beta);
        auto kernel = [&](double y, int t) {
            double s = 0.5 * (y + 1.0);
            double z = (s + t - 0.5 * w) * 2.0 / w;
            double r = 1.0 - z * z;
            return r > 0.0 ? std::cyl_bessel_i(0.0, P.kb_beta * std::sqrt(r)) * inv_i0b : 0.0;
        };
        // Chebyshev series of degree 6, 8 or 10 (the ones the kernels are built for): the first
        // within max(3e-7, tol / 5) of the kernel (FP32 evaluation alone errs by about 1.7e-7), checked
        // in FP32 in the device's order.  Taps
        // t < w/2 are fitted (coefficients from the discrete Chebyshev transform at ns nodes, a
        // near-minimax truncation); tap w-1-t mirrors t, and the middle tap of an odd w keeps only
        // its even terms.
        if (w > kMixedMaxW) return cleanup(nfail(WAVE1D_EINVAL, "mixed precision: kernel width above 7"));
        const double fit_tol = std::max(3e-7, tol / 5);
        int D = 6;
        double err = 1.0;
        for (;; D += 2) {
            std::memset(&h->poly, 0, sizeof(h->poly));
            for (int t = 0; t < (w + 1) / 2; t++) {
                for (int d = 0; d <= D; d++) {
                    double acc = 0.0;
                    for (int i = 0; i < ns; i++) acc += kernel(ys[i], t) * std::cos(d * kPiN * (i + 0.5) / ns);
                    double ad = (d == 0 ? 1.0 : 2.0) * acc / ns;
                    if (2 * t + 1 == w && d % 2 == 1) ad = 0.0;
                    h->poly.c[t][d] = (float)ad;
                    h->poly.c[w - 1 - t][d] = (float)(d % 2 ? -ad : ad);
                }
            }
            // interior points: at y = -1 and +1 an end tap touches the support edge, where the
            // kernel drops from 1/I0(beta) to 0 (a jump of the kernel itself, not of the fit)
            err = 0.0;
            for (int i = 1; i < 400; i++) {
                const float y = (float)(-1.0 + 2.0 * i / 400.0);
                float T[kMaxDegree + 1];
                T[0] = 1.f;
                T[1] = y;
                for (int d = 2; d <= D; d++) T[d] = std::fma(y + y, T[d - 1], -T[d - 2]);
                for (int t = 0; t < (w + 1) / 2; t++) {
                    float e = h->poly.c[t][0], o = h->poly.c[t][1] * T[1];
                    for (int d = 2; d <= D; d += 2) e = std::fma(h->poly.c[t][d], T[d], e);
                    for (int d = 3; d <= D; d += 2) o = std::fma(h->poly.c[t][d], T[d], o);
                    err = std::max(err, std::fabs((double)(e + o) - kernel((double)y, t)));
                    err = std::max(err, std::fabs((double)(e - o) - kernel((double)y, w - 1 - t)));
                }
            }
            if (err < fit_tol || D == 10) break;
        }
        h->D = D;
        h->kernel_err = err;
        if ((rc = nu_upload(h, soff, &h->soff))) return cleanup(rc);
    }
    h->i0_host = i0;
    h->off_host.assign(offsets, offsets + n_inst + 1);
    rc = precision == 1 ? nu_cut_ranges(h, kRangeCells, kRangePoints, h->split) : nu_cut_segments(h, kSegPoints, h->split);
    if (rc || (rc = nu_upload(h, gfirst, &h->first))) return cleanup(rc);
    std::vector<double> d1, d2, mf, tw((size_t)P.L * 2);
    nufft_factors(P, d1, d2, mf);
    for (int j = 0; j < P.L; j++) {
        double ang = 2.0 * kPiN * (double)j / (double)P.L;
        tw[2 * j] = std::cos(ang);
        tw[2 * j + 1] = std::sin(ang);
    }
    h->group = std::max(1, std::min({n_inst, (1 << 25) / nf, 65535}));
    if ((rc = nu_upload(h, mf, &h->modefac)) || (rc = nu_upload(h, tw, &h->twiddle)) ||
        (rc = nu_alloc(h, (size_t)n_inst * nf, &h->grid)) || (rc = nu_alloc(h, (size_t)h->group * nf, &h->work)))
        return cleanup(rc);
    for (const void* k : {(const void*)k_nu_cols1, (const void*)k_nu_cols2, (const void*)k_nu_rows1, (const void*)k_nu_rows2})
        if (!allow_smem(k, nu_fft_smem(std::max(P.L1, P.L2))))
            return cleanup(nfail(WAVE1D_ECUDA, "cannot size the shared memory of the FFT passes"));
    if (cudaDeviceSynchronize() != cudaSuccess) return cleanup(nfail(WAVE1D_ECUDA, "upload failed"));
    *out = h;
    return WAVE1D_OK;
}

int wave1d_nufft_info(wave1d_nufft_t h, int* nf, int* w, int* degree, double* kernel_err) {
    if (!h) return nfail(WAVE1D_EINVAL, "plan is NULL");
    if (nf) *nf = h->P.nf;
    if (w) *w = h->P.nufft_w;
    if (degree) *degree = h->D;
    if (kernel_err) *kernel_err = h->kernel_err;
    return WAVE1D_OK;
}

int wave1d_nufft_perm(wave1d_nufft_t h, int64_t* perm) {
    if (!h || !perm) return nfail(WAVE1D_EINVAL, "bad arguments");
    std::memcpy(perm, h->perm.data(), sizeof(int64_t) * h->M);
    return WAVE1D_OK;
}

int wave1d_nufft_spread(wave1d_nufft_t h, const double* c, double* grid) {
    if (!h || !c || !grid) return nfail(WAVE1D_EINVAL, "bad arguments");
    if (cudaSetDevice(h->device) != cudaSuccess) return nfail(WAVE1D_ECUDA, "cudaSetDevice");
    const int w = h->P.nufft_w;
    const NuSplit& sp = h->split;
    bool ok;
    if (h->precision == 0) {
        const int64_t cells = (int64_t)h->B * h->P.nf;
        ok = nu_with_w(w, [&](auto wc) {
            constexpr int W = decltype(wc)::value;
            k_nu_tap_sums<W><<<(unsigned)((sp.nseg * 16 + 255) / 256), 256, 0, h->stream>>>(sp.seg, sp.nseg, c, h->ker, sp.tap_sums);
            k_nu_assemble<W><<<(unsigned)((cells + 255) / 256), 256, 0, h->stream>>>(sp.cseg, sp.tap_sums, grid, cells, h->P.nf);
        });
    } else {
        ok = nu_with_mixed(w, h->D, [&](auto wc, auto dc) {
            k_nu_spread_mixed<decltype(wc)::value, decltype(dc)::value><<<(unsigned)sp.nunits, kUnitThreads, 0, h->stream>>>(
                sp.ranges, sp.runs, c, h->soff, h->poly, grid);
        });
    }
    if (!ok) return nfail(WAVE1D_EUNSUPPORTED, "kernel width / degree not built");
    return cudaGetLastError() == cudaSuccess ? WAVE1D_OK : nfail(WAVE1D_ECUDA, "spread launch failed");
}

int wave1d_nufft_interp(wave1d_nufft_t h, const double* grid, double* u) {
    if (!h || !grid || !u) return nfail(WAVE1D_EINVAL, "bad arguments");
    if (cudaSetDevice(h->device) != cudaSuccess) return nfail(WAVE1D_ECUDA, "cudaSetDevice");
    if (h->precision == 0) {
        if (!nu_with_w(h->P.nufft_w, [&](auto wc) {
                k_nu_interp64<decltype(wc)::value><<<(unsigned)((h->M + kInterpTile - 1) / kInterpTile), kInterpTile, 0,
                                                     h->stream>>>(grid, u, h->first, h->ker, h->M, h->P.nf);
            }))
            return nfail(WAVE1D_EUNSUPPORTED, "kernel width not built");
    } else if (!nu_with_mixed(h->P.nufft_w, h->D, [&](auto wc, auto dc) {
                   const unsigned nb = (unsigned)((h->M + 256 * kInterpPer - 1) / (256 * kInterpPer));
                   k_nu_interp_mixed<decltype(wc)::value, decltype(dc)::value><<<nb, 256, 0, h->stream>>>(
                       grid, u, h->first, h->soff, h->poly, h->M, h->P.nf);
               })) {
        return nfail(WAVE1D_EUNSUPPORTED, "kernel width / degree not built");
    }
    return cudaGetLastError() == cudaSuccess ? WAVE1D_OK : nfail(WAVE1D_ECUDA, "interp launch failed");
}

int wave1d_nufft_type1(wave1d_nufft_t h, const double* c, double* S) {
    if (!h || !c || !S) return nfail(WAVE1D_EINVAL, "bad arguments");
    int rc = wave1d_nufft_spread(h, c, h->grid);
    if (rc) return rc;
    const Params& P = h->P;
    const double2* tw = (const double2*)h->twiddle;
    double2* work = (double2*)h->work;
    // S_k in one store where the caller's array allows it (two take 1 % longer over 64 instances)
    const bool wide = ((uintptr_t)S & 15) == 0;
    for (int b = 0; b < h->B; b += h->group) {
        const unsigned nb = (unsigned)std::min(h->group, h->B - b);
        k_nu_cols1<<<dim3(P.L2 / 2, nb), kFftThreads, nu_fft_smem(P.L1), h->stream>>>(
            (const double2*)(h->grid + (size_t)b * P.nf), work, tw, P.L, P.L1, P.L2);
        k_nu_rows1<<<dim3(P.L1 / 2 + 1, nb), kFftThreads, nu_fft_smem(P.L2), h->stream>>>(
            work, S + (size_t)b * 2 * (P.K + 1), h->modefac, tw, P.K, P.L, P.L1, P.L2, wide);
    }
    return cudaGetLastError() == cudaSuccess ? WAVE1D_OK : nfail(WAVE1D_ECUDA, "type-1 launch failed");
}

int wave1d_nufft_type2(wave1d_nufft_t h, const double* alpha, double* u) {
    if (!h || !alpha || !u) return nfail(WAVE1D_EINVAL, "bad arguments");
    if (cudaSetDevice(h->device) != cudaSuccess) return nfail(WAVE1D_ECUDA, "cudaSetDevice");
    const Params& P = h->P;
    const double2* tw = (const double2*)h->twiddle;
    double2* work = (double2*)h->work;
    for (int b = 0; b < h->B; b += h->group) {
        const unsigned nb = (unsigned)std::min(h->group, h->B - b);
        k_nu_cols2<<<dim3(P.L2 / 2, nb), kFftThreads, nu_fft_smem(P.L1), h->stream>>>(
            alpha + (size_t)b * 2 * (P.K + 1), work, h->modefac, tw, P.K, P.L, P.L1, P.L2);
        k_nu_rows2<<<dim3(P.L1 / 2, nb), kFftThreads, nu_fft_smem(P.L2), h->stream>>>(
            work, (double2*)(h->grid + (size_t)b * P.nf), tw, P.L, P.L1, P.L2);
    }
    if (cudaGetLastError() != cudaSuccess) return nfail(WAVE1D_ECUDA, "type-2 launch failed");
    return wave1d_nufft_interp(h, h->grid, u);
}

int wave1d_nufft_destroy(wave1d_nufft_t h) {
    if (!h) return WAVE1D_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    else cudaDeviceSynchronize();
    for (void* a : h->allocs) cudaFree(a);
    delete h;
    return WAVE1D_OK;
}

// Picks the work split of the spreading for this plan's points by timing: each candidate is cut from the
// points' first cells and timed over `reps` spreads of c (after one untimed spread) with CUDA events on the
// plan's stream; the fastest stays, the others' tables go.  Mixed: cells and points a range is cut at, at or below the
// kernel's shared-memory capacities.  FP64: points of one cell to a segment.  The grid is overwritten.  Every
// candidate takes every point once, so results change only in rounding.
int wave1d_nufft_autotune(wave1d_nufft_t h, const double* c, double* grid, int reps, int* cells, int* points) {
    if (!h || !c || !grid || reps < 1) return nfail(WAVE1D_EINVAL, "bad arguments");
    if (cudaSetDevice(h->device) != cudaSuccess) return nfail(WAVE1D_ECUDA, "cudaSetDevice");
    std::vector<std::pair<int, int>> candidates;
    if (h->precision == 1)
        for (int cc : {kRangeCells / 4, kRangeCells / 2, kRangeCells})
            for (int pp : {kRangePoints / 4, kRangePoints / 2, kRangePoints}) candidates.push_back({cc, pp});
    else
        for (int pp : {kSegPoints / 4, kSegPoints / 2, kSegPoints, 2 * kSegPoints, 4 * kSegPoints}) candidates.push_back({1, pp});
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return nfail(WAVE1D_ECUDA, "cudaEventCreate");
    }
    NuSplit before = h->split, best;
    float best_ms = 0.f;
    int rc = WAVE1D_OK;
    for (const auto& cand : candidates) {
        NuSplit s;
        rc = h->precision == 1 ? nu_cut_ranges(h, cand.first, cand.second, s) : nu_cut_segments(h, cand.second, s);
        h->split = s;
        if (!rc) rc = wave1d_nufft_spread(h, c, grid);
        cudaEventRecord(e0, h->stream);
        for (int r = 0; r < reps && rc == WAVE1D_OK; r++) rc = wave1d_nufft_spread(h, c, grid);
        cudaEventRecord(e1, h->stream);
        if (cudaEventSynchronize(e1) != cudaSuccess && !rc) rc = nfail(WAVE1D_ECUDA, "timing the spreading failed");
        float ms = 0.f;
        if (!rc) cudaEventElapsedTime(&ms, e0, e1);
        if (!rc && (best.points == 0 || ms < best_ms)) {
            nu_drop(h, best);
            best = s;
            best_ms = ms;
        } else {
            nu_drop(h, s);
        }
        if (rc) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    h->split = before;
    if (rc) {
        nu_drop(h, best);
        return rc;
    }
    if (h->precision == 0) {                         // a batch's ranges stay
        std::swap(best.ranges, before.ranges);
        std::swap(best.runs, before.runs);
        best.nunits = before.nunits;
    }
    nu_drop(h, before);
    h->split = best;
    if (cells) *cells = best.cells;
    if (points) *points = best.points;
    return WAVE1D_OK;
}

const char* wave1d_nufft_strerror(void) { return g_nu_error.c_str(); }

}  // extern "C"
