// Sums of float pairs in three floats (acc3_add, range.cuh) against long double.
// output: ok <largest error / (2^-53 sum |v|) over the cases> <the same of a sum kept as one pair>
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "range.cuh"

using namespace wave1d;

int main() {
    std::mt19937_64 rng(11);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    double worst = 0.0, pair = 0.0;
    for (int kind = 0; kind < 6; kind++)
        for (int n : {1, 2, 16, 676, 20000}) {
            float h = 0.f, m = 0.f, l = 0.f, ah = 0.f, al = 0.f;
            long double sum = 0.0L, mag = 0.0L;
            for (int i = 0; i < n; i++) {
                double v = U(rng);
                if (kind == 1) v = 1.0 / 3.0 + 1e-3 * v;                       // aligned
                if (kind == 2) v *= std::pow(10.0, 8.0 * U(rng));              // many sizes
                if (kind == 3) v = (i & 1 ? -1.0 : 1.0) * (1.0 + 1e-9 * i);    // cancelling
                if (kind == 4) v *= 1e-30;                                     // small, its low parts still normal
                if (kind == 5) v = std::pow(1.03, i % 2000) * (1.0 + 0.1 * v); // growing
                const rs::Pair q = rs::split(v);
                rs::acc3_add(h, m, l, q.hi, q.lo);
                rs::acc_add(ah, al, q.hi, q.lo);
                sum += (long double)q.hi + (long double)q.lo;
                mag += std::fabs((long double)q.hi);
                if (i == n / 2) {                                              // carried through a double
                    const double d = rs::acc3_value(h, m, l);
                    rs::acc3_set(d, h, m, l);
                    if (rs::acc3_value(h, m, l) != d) return 1;
                }
            }
            worst = std::max(worst, (double)(std::fabs(rs::acc3_value(h, m, l) - sum) / (0x1p-53L * mag)));
            pair = std::max(pair, (double)(std::fabs((long double)ah + (long double)al - sum) / (0x1p-53L * mag)));
        }
    std::printf("ok %.3f %.3f\n", worst, pair);
    return 0;
}
