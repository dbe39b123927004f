// The parts that the reverse march's kernels split their work into (adjoint.cuh: receivers_T_part, rbc_grid_sum,
// rbc_update_sum, modes_T_taps), run for every thread and added up as the kernels do, against the plain forms.
// output: ok <largest difference / largest value>; receivers and taps bit for bit (exit 3, 4 otherwise)
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "adjoint.cuh"

using namespace wave1d;

int main() {
    std::mt19937_64 rng(5);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    auto fill = [&](size_t n) {
        std::vector<double> v(n);
        for (auto& x : v) x = U(rng);
        return v;
    };
    double worst = 0.0;
    auto compare = [&](const std::vector<double>& a, const std::vector<double>& b) {
        double d = 0.0, s = 0.0;
        for (size_t i = 0; i < a.size(); i++) {
            d = std::max(d, std::fabs(a[i] - b[i]));
            s = std::max(s, std::fabs(a[i]));
        }
        worst = std::max(worst, d / s);
    };
    // receivers: rows of every first m and length a window can have
    for (int ring : {3, 9, 41, 48}) {
        std::vector<int64_t> ptr = {0}, woff;
        std::vector<int32_t> rcv, mrange;
        std::vector<double> w;
        for (int lo = 0; lo < ring; lo++)
            for (int cnt = 0; lo + cnt <= ring; cnt++) {
                rcv.push_back((lo + cnt) % 4);
                mrange.push_back(lo | cnt << 16);
                woff.push_back((int64_t)w.size());
                for (int c = 0; c < cnt; c++) w.push_back(U(rng));
            }
        ptr.push_back((int64_t)rcv.size());
        const std::vector<double> ubar = {0.5, 0.0, -1.25, 3.0};
        for (int64_t q : {(int64_t)0, (int64_t)7, (int64_t)123456789}) {
            std::vector<double> a(ring, 0.0), b(ring, 0.0);
            adj::receivers_T_source(0, ptr.data(), rcv.data(), mrange.data(), woff.data(), w.data(), ubar.data(), q, ring,
                                    [&](int s, double v) { a[s] += v; });
            for (int part = adj::kReceiverParts - 1; part >= 0; part--)
                adj::receivers_T_part(0, part, ptr.data(), rcv.data(), mrange.data(), woff.data(), w.data(), ubar.data(), q, ring,
                                      [&](int s, double v) { b[s] += v; });
            if (a != b) return 3;
        }
    }
    for (int K : {3, 50, 315, 849}) {
        const int K1 = K + 1, npts = std::min(37, K);
        std::vector<double> tw(4 * (size_t)K);
        for (int a = 0; a < 2 * K; a++) {
            tw[2 * a] = std::cos(3.141592653589793 * a / K);
            tw[2 * a + 1] = std::sin(3.141592653589793 * a / K);
        }
        const std::vector<double> ab = fill(2 * K1), apb = fill(2 * K1), phi = fill(npts), dphi = fill(npts), uvbar = fill(2 * npts);
        std::vector<int32_t> idx;
        for (int i = 0; i < npts; i++) idx.push_back((K - npts / 2 + i) % (2 * K));
        // grid part: 256 threads to a point
        std::vector<double> plain(2 * npts), parts(2 * npts);
        for (int pt = 0; pt < npts; pt++) {
            adj::rbc_grid_T(idx[pt], K, tw.data(), ab.data(), apb.data(), phi[pt], dphi[pt], &plain[2 * pt], &plain[2 * pt + 1]);
            double su = ab[0], sv = apb[0];
            for (int t = 0; t < 256; t++) adj::rbc_grid_sum(idx[pt], K, 1 + t, 256, tw.data(), ab.data(), apb.data(), su, sv);
            adj::rbc_grid_values(K, su, sv, phi[pt], dphi[pt], &parts[2 * pt]);
        }
        compare(plain, parts);
        // mode part: eight lanes to a mode
        std::vector<double> a0 = ab, p0 = apb, a1 = ab, p1 = apb;
        for (int k = 0; k <= K; k++) {
            adj::rbc_update_T(k, K, npts, idx.data(), tw.data(), uvbar.data(), a0.data(), p0.data());
            adj::Complex u = {0.0, 0.0}, v = {0.0, 0.0};
            for (int q = 0; q < 8; q++)
                if (k < K) adj::rbc_update_sum(k, K, q, 8, npts, idx.data(), tw.data(), uvbar.data(), u, v);
            adj::rbc_update_values(k, K, u, v, a1.data(), p1.data());
        }
        compare(a0, a1);
        compare(p0, p1);
        // modes: kModeTaps taps to a thread, any order of the threads
        for (int W : {1, 2, 4, 9, 36}) {
            const std::vector<double> rot = fill(3 * K1), pq = fill(2 * (size_t)W * K1), S0 = fill(2 * (size_t)W * K1);
            for (int64_t n : {(int64_t)0, (int64_t)5, (int64_t)1000}) {
                std::vector<double> xa = ab, xp = apb, xS = S0, x2(2 * K1), ya(2 * K1), yp(2 * K1), yS = S0, y2(2 * K1);
                for (int k = 0; k <= K; k++) {
                    adj::modes_T(k, K1, W, n, rot.data(), pq.data(), xa.data(), xp.data(), xS.data(), x2.data());
                    for (int ma = (W - 1) / adj::kModeTaps * adj::kModeTaps; ma >= 0; ma -= adj::kModeTaps)
                        adj::modes_T_taps(k, K1, W, n, ma, rot.data(), pq.data(), ab.data(), apb.data(), ya.data(), yp.data(), yS.data(),
                                          y2.data());
                }
                if (xa != ya || xp != yp || xS != yS || x2 != y2) return 4;
            }
        }
    }
    std::printf("ok %.3e\n", worst);
    return 0;
}
