// The tensor-core fold's operands on the CPU: the coefficient slices of the plan builder and the
// density slices of range.cuh, contracted as the kernel contracts them (whole-number products, one
// accumulator per i + j), against the FP64 polynomials times the densities.
// input: dt tol p spread; output: ok <error of e_r summed at |z| = 1, relative to the largest
// |Q| max |sigma|> <largest |partial sum| of any accumulator>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "internal.h"
#include "range.cuh"

using namespace wave1d;

static double half_value(uint16_t h) {
    if ((h & 0x7fff) == 0) return 0.0;
    const double m = 1.0 + (h & 0x3ff) / 1024.0;
    return (h & 0x8000 ? -1.0 : 1.0) * std::ldexp(m, ((h >> 10) & 31) - 15);
}

int main() {
    double dt, tol, spread;
    int p;
    if (std::scanf("%lf %lf %d %lf", &dt, &tol, &p, &spread) != 4) return 1;
    HostPlan hp;
    std::string err;
    const double x[2] = {0.0, 1.0}, b[2] = {1.0, 1.0};
    if (build_host_plan(x, b, 2, 0, dt, 10, tol, p, 0.5, 0, 0, 32, 0, 0, 4096, 1ll << 30, hp, err, true)) return 2;
    const RangeTables& rt = hp.rt;
    const int nm = rt.nm;
    // the transposed sum's table holds the same slices
    for (int sl = 0; sl < kRsAllSlices; sl++)
        for (int iv = 0; iv < rt.nint; iv++)
            for (int m = 1; m < nm; m++)
                if (rt.fold[fold_index(sl, m, iv, rt.nk, rt.nivp)] != rt.unfold[unfold_index(sl, m, iv, rt.nis, rt.nmp)]) return 3;
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    double maxq = 0.0, worst = 0.0, most = 0.0;
    for (double v : rt.cheb) maxq = std::max(maxq, std::fabs(v));
    for (int iv = 0; iv < rt.nint; iv++) {
        // a history whose samples span `spread` decades
        std::vector<double> sig(nm);
        double smax = 0.0;
        for (int m = 1; m < nm; m++) {
            sig[m] = U(rng) * std::pow(10.0, -spread * std::fabs(U(rng)));
            smax = std::max(smax, std::fabs(sig[m]));
        }
        float hi[512], lo[512];
        unsigned mx = 0;
        for (int m = 1; m < nm; m++) {
            const rs::Pair q = rs::split(sig[m]);
            hi[m] = q.hi;
            lo[m] = q.lo;
            const float a = std::fabs(q.hi);
            unsigned bits;
            std::memcpy(&bits, &a, 4);
            mx = std::max(mx, bits);
        }
        const int E = rs::slice_exponent(mx);
        const float inv = std::ldexp(1.0f, 10 - E);
        double err_iv = 0.0;
        for (int r = 0; r < kRsPowers; r++) {
            double acc[kRsSlices + 1] = {}, exact = 0.0;
            for (int m = 1; m < nm; m++) {
                float s[kRsSlices];
                rs::density_slices(hi[m], lo[m], inv, s);
                for (int g = 0; g < kRsDiagonals[r]; g++)
                    for (int i = 0; i <= g; i++) {
                        if (i >= kRsSlices || g - i >= kRsSlicesOf[r]) continue;
                        acc[g] += s[i] * half_value(rt.fold[fold_index(kRsFirstSlice[r] + g - i, m, iv, rt.nk, rt.nivp)]);
                        most = std::max(most, std::fabs(acc[g]));
                    }
                // the monomial coefficient from the FP64 Chebyshev series
                const double* c = &rt.cheb[((size_t)iv * nm + m) * 8];
                static const double T[8][8] = {{1}, {0, 1}, {-1, 0, 2}, {0, -3, 0, 4}, {1, 0, -8, 0, 8},
                                               {0, 5, 0, -20, 0, 16}, {-1, 0, 18, 0, -48, 0, 32},
                                               {0, -7, 0, 56, 0, -112, 0, 64}};
                double a = 0.0;
                for (int q = r; q < 8; q++) a += c[q] * T[q][r];
                exact += a * ((double)hi[m] + (double)lo[m]);
            }
            double v = 0.0;
            for (int g = kRsDiagonals[r] - 1; g >= 0; g--) v = v / 2048.0 + acc[g];
            v *= (double)rt.fold_scale[(size_t)iv * kRsPowers + r] * std::ldexp(1.0, E - 10);
            err_iv += std::fabs(v - exact);
        }
        worst = std::max(worst, err_iv / (maxq * smax));
    }
    std::printf("ok %.3e %.0f\n", worst, most);
    return 0;
}
