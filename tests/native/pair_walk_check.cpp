// Host-side check (no GPU) of the pair kernels' walk of plans without pair lists (rs_pair_block, range.cu): blocks of
// 128 targets, both sides, parts of the distance intervals, each warp's run of the block's sources in chunks, every
// pair placed by place_pair (range.cuh).
//   * every pair closer than delta is met once, in one part and on one side, none that lies farther;
//   * the local sums through the e-vectors (in the kernel's order) equal the stored FP64 weights';
//   * so do the transposed sums through the moments per interval (moments_sum, acc3_add).
// Input: M dt tol bc part (0: range_split's), then M positions.  Output: ok <pairs met wrongly> <max |difference| of the
// local sums / max |row sum|> <the same of the transposed sums> <pairs>.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"
#include "range.cuh"
#include "wave1d.h"

using namespace wave1d;

namespace {

constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr int kChunk = 1024;        // kRsPosChunk of range.cu

double hist(int m, int64_t l) { return std::cos(0.41 * m + 0.9 * (double)l) + 0.02 * m; }
double cbar_of(int64_t l) { return std::sin(1.3 * (double)l) + 0.1; }

double xext(const HostPlan& hp, int64_t e) {
    const int64_t M = hp.P.M;
    if (e < 0) return hp.x[e + M] - 2.0 * kPi;
    if (e >= M) return hp.x[e - M] + 2.0 * kPi;
    return hp.x[e];
}
int64_t spring(const HostPlan& hp, int64_t e) { return e < 0 ? e + hp.P.M : (e >= hp.P.M ? e - hp.P.M : e); }

void evec_of(const RangeTables& rt, int iv, int64_t l, float* rec) {
    rs::EVec ev;
    rs::evec_zero(ev);
    for (int m = rt.mr[2 * iv]; m <= rt.mr[2 * iv + 1]; m++) {
        const float* c = &rt.coef[((size_t)iv * rt.nm + m) * 12];
        const rs::Pair s = rs::split(hist(m, l));
        rs::evec_mac(ev, c, c + 4, c + 8, s.hi, s.lo);
    }
    const float r[12] = {ev.e0h, ev.e0l, ev.e1h, ev.e1l, ev.e2, ev.e3, ev.e4, ev.e5, ev.e6, ev.e7, 0.f, 0.f};
    std::memcpy(rec, r, sizeof(r));
}

struct Moments {                     // RsMoments of range.cu
    float f[10] = {};
    void add(float zh, float zl, float ch, float cl) {
        rs::acc_add(f[0], f[1], ch, cl);
        rs::acc_mac(f[2], f[3], zh, zl, ch, cl);
        float p = rs::mul(rs::mul(zh, zh), ch);
        for (int r = 4; r < 10; r++) {
            f[r] = rs::add(f[r], p);
            p = rs::mul(p, zh);
        }
    }
    void flush(float* rec) {
        rs::acc_add(f[0], f[1], rec[0], rec[1]);
        rs::acc_add(f[2], f[3], rec[2], rec[3]);
        for (int r = 4; r < 10; r++) f[r] = rs::add(f[r], rec[r]);
        std::memcpy(rec, f, sizeof(f));
        std::memset(f, 0, sizeof(f));
    }
};

struct Target {
    Moments mo;
    int cur = -1;
    float ah[2], al[2];
};

struct Walk {
    const HostPlan& hp;
    int part;
    std::vector<std::vector<int>> met;          // [target][e - wlo]
    std::vector<double> sums;
    std::vector<float> records;                 // [target of the block][interval][12]
    std::vector<float> accs;                    // [target of the block][2]

    template <int S>
    void side(int64_t j0, int p0, int p1, std::vector<Target>& st) {
        const RangeTables& rt = hp.rt;
        const int64_t M = hp.P.M;
        const int nT = (int)std::min<int64_t>(kRsPairTargets, M - j0);
        const double xa = hp.x[j0], xb = hp.x[j0 + nT - 1];
        const rs::Grid G = rs::grid_of(xb - xa, hp.P.delta);
        const int v0 = std::max(0, p0 - rt.fine_span - 2), v1 = std::min(rt.nint, p1 + 2), ns = v1 - v0;
        std::vector<rs::F4> tab;
        for (int iv = v0; iv < v1; iv++)
            tab.push_back(rs::interval_entry(rt.mid[iv], rt.ih[iv], iv + 1 < rt.nint ? rt.bp2[2 * (iv + 1)] : INFINITY, (float)G.g,
                                             (float)G.ig));
        const int* win = &hp.blk_win[4 * (j0 / kRsTargets)];
        const int top = S > 0 ? win[0] : (int)(j0 + nT - 1), all = std::max(0, S > 0 ? win[3] - top : top - win[0] + 1);
        const double marg = rs::part_margin(hp.P.delta, G.g), d0 = rt.bp[p0] - marg, d1 = rt.bp[p1] + marg;
        int lo = 0, hi = 0;
        while (lo < all && !((S > 0 ? xext(hp, top + lo) - xa : xb - xext(hp, top - lo)) >= d0)) lo++;
        while (hi < all && ((S > 0 ? xext(hp, top + hi) - xb : xa - xext(hp, top - hi)) < d1)) hi++;
        const int start = top + S * lo, count = hi - lo;
        const bool at_dt = p0 <= rt.iv_dt && rt.iv_dt <= p1;
        const float scale = (float)(kRsFineCells / hp.P.delta), df0 = (float)d0, df1 = (float)d1;
        for (int w = 0; w < kRsPairTargets / 32; w++) {
            float bh[32], bl[32];
            for (int i = 0; i < 32; i++) {
                rs::grid_split(hp.x[j0 + std::min(32 * w + i, nT - 1)] - xa, G, bh[i], bl[i]);
                if (S > 0) bh[i] = -bh[i], bl[i] = -bl[i];
            }
            const float bfar = bh[S > 0 ? 0 : 31], bnear = bh[S > 0 ? 31 : 0];
            for (int base = 0; base < count; base += kChunk) {
                const int lim = std::min(count - base, kChunk), e0 = start + S * base;
                std::vector<float> ph(lim), pl(lim);
                for (int k = 0; k < lim; k++) rs::grid_split(xext(hp, e0 + S * k) - xa, G, ph[k], pl[k]);
                int klo = 0, khi = 0;
                while (klo < lim && !((S < 0 ? bfar - ph[klo] : bfar + ph[klo]) >= df0)) klo++;
                while (khi < lim && !((S < 0 ? bnear - ph[khi] : bnear + ph[khi]) >= df1)) khi++;
                for (int i = 0; i < 32 && 32 * w + i < nT; i++) {
                    const int64_t j = j0 + 32 * w + i;
                    int64_t lb = j;
                    while (lb > 0 && hp.x[lb - 1] == hp.x[j]) lb--;
                    for (int k = klo; k < khi; k++) {
                        const int64_t e = e0 + S * k;
                        float zh, zl;
                        const int at = rs::place_pair<S>([&](int q) { return tab[q]; }, [&](int c) { return (int)rt.fine[c]; }, scale, v0,
                                                         ns, at_dt, rt.iv_dt - v0, (unsigned)((int)e - hp.nb_lo[j]) < (unsigned)hp.nb_cnt[j],
                                                         S > 0 ? e >= lb : e < lb, bh[i], bl[i], ph[k], pl[k], zh, zl);
                        const int iv = at + v0;
                        if (at < 0 || iv < p0 || iv >= p1) continue;
                        met[j][e - win[0]]++;
                        Target& t = st[32 * w + i];
                        float rec[12];
                        evec_of(rt, iv, spring(hp, e), rec);
                        const int u = (k - klo) & 1;
                        rs::evec_eval(rec, zh, zl, t.ah[u], t.al[u]);
                        if (iv != t.cur) {
                            if (t.cur >= 0) t.mo.flush(&records[((size_t)(32 * w + i) * rt.nint + t.cur) * 12]);
                            t.cur = iv;
                        }
                        const double c = cbar_of(spring(hp, e));
                        t.mo.add(zh, zl, (float)c, (float)(c - (double)(float)c));
                    }
                }
            }
        }
    }
};

}  // namespace

int main() {
    long M;
    double dt, tol;
    int bc, part;
    if (std::scanf("%ld %lf %lf %d %d", &M, &dt, &tol, &bc, &part) != 5) return 2;
    std::vector<double> x(M), beta(M, 3.0);
    for (auto& v : x)
        if (std::scanf("%lf", &v) != 1) return 2;
    std::string err;
    HostPlan hr, hs;
    if (build_host_plan(x.data(), beta.data(), M, bc, dt, 100, tol, 8, 0.5, 0, 0, 32, 0, 0, 4096, (int64_t)1 << 34, hr, err, true) ||
        build_host_plan(x.data(), beta.data(), M, bc, dt, 100, tol, 8, 0.5, 0, 0, 32, 0, 0, 4096, (int64_t)1 << 34, hs, err)) {
        std::printf("error %s\n", err.c_str());
        return 1;
    }
    const RangeTables& rt = hr.rt;
    if (part == 0) part = range_split(rt.nint, M, hr.range_pairs, (size_t)1 << 40).part;
    Walk w{hr, part, {}, std::vector<double>(M, 0.0), {}, {}};
    std::vector<double> tgot((size_t)M * rt.nm, 0.0);
    w.met.resize(M);
    for (int64_t j = 0; j < M; j++) {
        const int* win = &hr.blk_win[4 * (j / kRsTargets)];
        w.met[j].assign(std::max(0, win[3] - win[0]), 0);
    }
    for (int64_t j0 = 0; j0 < M; j0 += kRsPairTargets) {
        const int nT = (int)std::min<int64_t>(kRsPairTargets, M - j0);
        w.records.assign((size_t)nT * rt.nint * 12, 0.f);
        w.accs.assign(2 * (size_t)nT, 0.f);
        for (int p0 = 0; p0 < rt.nint; p0 += part) {
            const int p1 = std::min(rt.nint, p0 + part);
            std::vector<Target> st(kRsPairTargets);
            for (int side = 0; side < 2; side++) {
                for (auto& t : st) t.ah[0] = t.ah[1] = t.al[0] = t.al[1] = 0.f;
                if (side == 0) w.side<-1>(j0, p0, p1, st);
                else w.side<1>(j0, p0, p1, st);
                for (int t = 0; t < nT; t++) {
                    rs::acc_add(st[t].ah[0], st[t].al[0], st[t].ah[1], st[t].al[1]);
                    rs::acc_add(w.accs[2 * t], w.accs[2 * t + 1], st[t].ah[0], st[t].al[0]);
                }
            }
            for (int t = 0; t < nT; t++)
                if (st[t].cur >= 0) st[t].mo.flush(&w.records[((size_t)t * rt.nint + st[t].cur) * 12]);
        }
        for (int t = 0; t < nT; t++) {
            w.sums[j0 + t] = (double)w.accs[2 * t] + (double)w.accs[2 * t + 1];
            for (int m = 1; m < rt.nm; m++) {
                float a = 0.f, b = 0.f, c = 0.f;
                for (int iv = 0; iv < rt.nint; iv++) {
                    if (m < rt.mr[2 * iv] || m > rt.mr[2 * iv + 1]) continue;
                    const float* q = &rt.coef[((size_t)iv * rt.nm + m) * 12];
                    const float* f = &w.records[((size_t)t * rt.nint + iv) * 12];
                    float h, l;
                    rs::moments_sum(h, l, rs::load4(q), rs::load4(q + 4), rs::load4(q + 8), rs::load4(f), rs::load4(f + 4), f[8], f[9]);
                    rs::acc3_add(a, b, c, h, l);
                }
                tgot[(size_t)(j0 + t) * rt.nm + m] = rs::acc3_value(a, b, c);
            }
        }
    }
    // every pair once (e is a right source from lb_j on), none beyond delta; at delta itself either is right
    long wrong = 0, pairs = 0;
    for (int64_t j = 0; j < M; j++) {
        const int* win = &hr.blk_win[4 * (j / kRsTargets)];
        for (size_t k = 0; k < w.met[j].size(); k++) {
            const double d = std::fabs(xext(hr, win[0] + (int64_t)k) - hr.x[j]), rel = d / hr.P.delta - 1.0;
            pairs += w.met[j][k];
            if (rel < -1e-6 ? w.met[j][k] != 1 : (rel > 1e-5 ? w.met[j][k] != 0 : w.met[j][k] > 1)) wrong++;
        }
    }
    std::vector<double> ref(M, 0.0), tref((size_t)M * rt.nm, 0.0);
    const LocalCSR& C = hs.loc;
    for (int64_t j = 0; j < M; j++)
        for (int64_t e = C.row_ptr[j]; e < C.row_ptr[j + 1]; e++) {
            const int lo = C.mrange[e] & 0xffff, cnt = C.mrange[e] >> 16;
            for (int c = 0; c < cnt; c++) {
                ref[j] += lo + c >= 1 ? C.w[C.woff[e] + c] * hist(lo + c, C.src[e]) : 0.0;
                if (lo + c >= 1) tref[(size_t)j * rt.nm + lo + c] += C.w[C.woff[e] + c] * cbar_of(C.src[e]);
            }
        }
    double worst = 0.0, scale = 0.0, tworst = 0.0, tscale = 0.0;
    for (int64_t j = 0; j < M; j++) {
        worst = std::max(worst, std::fabs(w.sums[j] - ref[j]));
        scale = std::max(scale, std::fabs(ref[j]));
    }
    for (size_t i = 0; i < tref.size(); i++) {
        tworst = std::max(tworst, std::fabs(tgot[i] - tref[i]));
        tscale = std::max(tscale, std::fabs(tref[i]));
    }
    std::printf("ok %ld %.3e %.3e %ld\n", wrong, worst / scale, tworst / tscale, pairs);
    return 0;
}
