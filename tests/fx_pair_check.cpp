// Host check of the FP64 operators' fixed-point pair arithmetic (csrc/fx.h,
// csrc/fx_pair.h): sums of every operator over one tile of points against long
// double, for near, touching, coincident and far tiles, several smoothing radii
// and density scales.  Prints the largest error of a row in units of the sum of
// its absolute terms, one line per operator and case.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "../paper_2110_10749_gb300/csrc/fx_table.cu"
namespace ssd {
enum Op { OP_LSL, OP_LDL, OP_SSL, OP_SDL, OP_SSLDL, OP_LSLDL, OP_LDLT, OP_SDLT };
}
#include "../paper_2110_10749_gb300/csrc/fx_pair.h"
using namespace ssd;

namespace {
struct Pt { double x[3], m[3], u[3], f[3], p, g; };
Sigma sig;

int top(double m) { return m > 0 ? std::ilogb(m) + 1 : 0; }

template <int OP> double check(const std::vector<Pt> &src, const std::vector<Pt> &tgt, double delta) {
    typedef FxOp<OP> T;
    constexpr int NC = T::vec ? 3 : 1;
    double lo[3] = {1e9, 1e9, 1e9}, hi[3] = {-1e9, -1e9, -1e9}, um = 0, fm = 0, mm = 0, ext = 0;
    for (const auto *v : {&src, &tgt})
        for (const Pt &a : *v) {
            for (int c = 0; c < 3; ++c) {
                lo[c] = std::min(lo[c], a.x[c]);
                hi[c] = std::max(hi[c], a.x[c]);
                mm = std::max(mm, std::fabs(a.m[c]));
                if (T::vec) { um = std::max(um, std::fabs(a.u[c])); fm = std::max(fm, std::fabs(a.f[c])); }
            }
            if (!T::vec) { um = std::max(um, std::fabs(a.p)); fm = std::max(fm, std::fabs(a.g)); }
        }
    for (int c = 0; c < 3; ++c) ext = std::max(ext, (hi[c] - lo[c]) / delta);
    if (ext < kFxMinExt) return 0;   // left to the generic kernel
    int ps = ext > 0 ? 62 - top(ext) : 58;
    if (ps > 58) ps = 58;
    auto grid = [&](double v, int c) {
        return (int64_t)llrintl(((ld)v - 0.5 * (lo[c] + hi[c])) / (ld)delta * ldexpl(1, ps));
    };
    const bool only_f = OP == OP_LSL || OP == OP_SSL;
    int ed;
    std::frexp(1.0 / delta, &ed);
    const FxScale sc = fx_scale<OP>(top(only_f ? fm : um), top(fm), top(mm), llrintl(ldexpl(1 / (ld)delta, 62 - ed)), ed);
    int64_t dmax = 0, gap = 0;
    for (int c = 0; c < 3; ++c) {
        int64_t b[4] = {INT64_MAX, INT64_MIN, INT64_MAX, INT64_MIN};
        for (int k = 0; k < 2; ++k)
            for (const Pt &a : k ? tgt : src) {
                const int64_t h = grid(a.x[c], c) >> 32;
                b[2 * k] = std::min(b[2 * k], h);
                b[2 * k + 1] = std::max(b[2 * k + 1], h);
            }
        dmax = std::max(dmax, std::max(b[3] - b[0], b[1] - b[2]) + 1);
        gap = std::max(gap, std::max(b[2] - b[1], b[0] - b[3]) - 1);
    }
    int L = 32 - ps, r = 0;
    while (std::ldexp((double)dmax, 32) > std::ldexp(1.0, L + ps)) ++L;
    if (L < 0) L = 0;
    while (gap > 0 && std::ldexp((double)gap, 32) >= std::ldexp(1.0, r + 1 + ps)) ++r;
    const FxTile tl = fx_tile<OP>(sc, L, r);
    const int ks = 61 - L - ps;
    auto conv = [&](const Pt &a) {
        FxPoint<OP> q{};
        for (int c = 0; c < 3; ++c) {
            const int64_t X = grid(a.x[c], c);
            fx_split(ks >= 0 ? (int64_t)((uint64_t)X << ks) : X >> -ks, q.x.h[c], q.x.l[c]);
            fx_split(fx_fix(a.m[c], sc.em, 59), q.m.h[c], q.m.l[c]);
            if (T::vec) {
                fx_split(fx_fix(a.u[c], sc.eu, 58), q.u.h[c], q.u.l[c]);
                fx_split(fx_fix(a.f[c], sc.ef, 58), q.f.h[c], q.f.l[c]);
            }
        }
        if (!T::vec) { q.p = fx_fix(a.p, sc.eu, 60); q.g = fx_fix(a.g, sc.ef, 60); }
        return q;
    };
    const FxI4 *tab = fx_table_host();
    auto entry = [&](int k, uint32_t i, int w) { return tab[((size_t)T::tab(k) * kFxMaxOct * kFxSeg + i) * kFxEntry + w]; };
    const double fac = T::dl && !T::fused ? 1 / (delta * delta) : 1 / delta;
    double worst = 0;
    for (const Pt &y : tgt) {
        const FxPoint<OP> Y = conv(y);
        FxSum<OP> acc;
        std::memset(&acc, 0, sizeof(acc));
        ld ref[3] = {0, 0, 0}, mag[3] = {0, 0, 0};
        for (const Pt &x : src) {
            fx_pair<OP, kFxFull>(Y, conv(x), tl, sc, kFxMaxOct * kFxSeg - 1, entry, acc);
            ld d[3], r2 = 0, s[4], v[3] = {0, 0, 0}, av[3] = {0, 0, 0};
            for (int c = 0; c < 3; ++c) { d[c] = (ld)y.x[c] - x.x[c]; r2 += d[c] * d[c]; }
            const ld de = delta;
            sig.at(r2 / (de * de), s);
            const ld k1 = s[0] / de, k2 = s[1] / (de * de * de), k3 = s[2] / (de * de * de),
                     k4 = s[3] / (de * de * de * de * de);
            auto dot = [&](const double *a) { return d[0] * a[0] + d[1] * a[1] + d[2] * a[2]; };
            auto add = [&](int c, ld t) { v[c] += t; av[c] += fabsl(t); };
            if (OP == OP_LSL || OP == OP_LSLDL) add(0, k1 * x.g);
            if (OP == OP_LDL || OP == OP_LSLDL) add(0, ((ld)x.p - y.p) * dot(x.m) * k2);
            if (OP == OP_LDLT) { add(0, k2 * dot(y.m) * x.p); add(0, k2 * dot(x.m) * y.p); }
            for (int c = 0; c < NC && T::vec; ++c) {
                if (T::sl) { add(c, x.f[c] * k1); add(c, d[c] * dot(x.f) * k3); }
                if (OP == OP_SDL || OP == OP_SSLDL) add(c, k4 * (dot(x.u) - dot(y.u)) * dot(x.m) * d[c]);
                if (OP == OP_SDLT) { add(c, k4 * dot(y.m) * dot(x.u) * d[c]); add(c, k4 * dot(x.m) * dot(y.u) * d[c]); }
            }
            for (int c = 0; c < NC; ++c) { ref[c] += v[c]; mag[c] += av[c]; }
        }
        ld err = 0, all = 0;
        for (int c = 0; c < NC; ++c) {
            const double got = (T::vec ? std::ldexp(fx_value(acc.v[c]), tl.ex)
                                       : std::ldexp((double)acc.f.h + std::ldexp((double)acc.f.l, -32), tl.ex)) * fac;
            err = fmaxl(err, fabsl(got - ref[c]));
            all = fmaxl(all, mag[c]);
        }
        if (all > 0) worst = std::max(worst, (double)(err / all));
        else if (err > 0) worst = 1;
    }
    return worst;
}
}  // namespace

int main() {
    std::mt19937_64 gen(3);
    std::normal_distribution<double> N;
    std::uniform_real_distribution<double> U(-1, 1);
    // (smoothing radius, tile radius, centre distance) on the unit sphere, density scales
    const double cases[][5] = {{0.375, 0.5, 0, 1, 1},      {0.375, 0.5, 2.0, 1e-9, 1e7}, {0.09, 0.3, 0, 1, 1},
                               {0.09, 0.3, 1.5, 1, 1e-30}, {0.03, 0.1, 0, 1e40, 1},      {0.03, 0.1, 1.9, 1, 1},
                               {0.03, 1.0, 0, 1, 1},       {0.008, 0.02, 1.99, 1, 1},    {0.01, 0.0, 0, 1, 1}};
    for (const auto &k : cases) {
        const double delta = k[0], rad = k[1];
        auto points = [&](double th, int n) {
            std::vector<Pt> v;
            for (int i = 0; i < n; ++i) {
                Pt a;
                const double t = th + rad * U(gen), f = 0.7 + rad * U(gen);
                const double nx[3] = {std::sin(t) * std::cos(f), std::sin(t) * std::sin(f), std::cos(t)};
                for (int c = 0; c < 3; ++c) {
                    a.x[c] = nx[c] + 0.05;
                    a.m[c] = 1e-3 * (1.2 + U(gen)) * nx[c];
                    a.u[c] = k[3] * N(gen);
                    a.f[c] = k[4] * N(gen);
                }
                a.p = k[3] * N(gen);
                a.g = k[4] * N(gen);
                v.push_back(a);
            }
            return v;
        };
        std::vector<Pt> tgt = points(0.9, 40), src = points(0.9 + 1.5 * k[2], 128);
        for (int i = 0; k[2] == 0 && i < 40; ++i) {   // self and coincident pairs, pairs a rounding apart
            src[i] = tgt[i];
            for (int c = 0; i >= 20 && c < 3; ++c) src[i].x[c] = std::nextafter(src[i].x[c], (i + c) % 2 ? 9.0 : -9.0);
        }
        std::printf("LSL %.3e\n", check<OP_LSL>(src, tgt, delta));
        std::printf("LDL %.3e\n", check<OP_LDL>(src, tgt, delta));
        std::printf("SSL %.3e\n", check<OP_SSL>(src, tgt, delta));
        std::printf("SDL %.3e\n", check<OP_SDL>(src, tgt, delta));
        std::printf("SSLDL %.3e\n", check<OP_SSLDL>(src, tgt, delta));
        std::printf("LSLDL %.3e\n", check<OP_LSLDL>(src, tgt, delta));
        std::printf("LDLT %.3e\n", check<OP_LDLT>(src, tgt, delta));
        std::printf("SDLT %.3e\n", check<OP_SDLT>(src, tgt, delta));
    }
    return 0;
}
