// Tables of the kernel factors sigma_i(t) = s_i(rho) / rho^p, t = rho^2
// (s_i of Section 5.3; p = 1, 3, 3, 5), for the fixed-point pair sums.
//
// The variable is v = 1 + t: 64 segments of equal width per octave of v, so
// the segments are narrow where the smoothing acts (t < 64) and scale with t
// where the kernels are bare powers.  On each segment sigma_i is a polynomial
// of degree 7 in s in [-1, 1]: the Chebyshev interpolant on 12 nodes,
// truncated to degree 7 (largest neglected term below 2^-56 of the value) and
// rewritten in powers of s.  From c4 on the coefficients have 32 bits, which sets the
// error: over all octaves at most 2^-53.7 of sigma_1 to sigma_3 and t^(-1/2) (rms
// 2^-57.1) and 2^-51.9 of sigma_4 (2^-55.1).  Node values come from the closed forms in long
// double, below t = 2 from the Maclaurin series (the closed forms cancel).
// Where long double is 128 bits in software the entries take 47 ms on one thread;
// they go to up to 16, and creating a process's first context takes 8 ms (50 on one).
#include <math.h>

#include <algorithm>
#include <exception>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "fx.h"

namespace ssd {
namespace {

typedef long double ld;
constexpr int kNodes = 12, kDeg = 7, kTerms = 48;
const ld kPiL = 3.141592653589793238462643383279502884L;

struct Sigma {
    ld ser[4][kTerms];
    Sigma() {
        const ld q[4][4] = {{5.0L / 3, -2.0L / 3, 0, 0}, {-1, 2.0L / 3, 0, 0}, {-1, 14.0L / 3, -4.0L / 3, 0},
                            {-1, -6.0L / 9, 4, -8.0L / 9}};
        const int skip[4] = {0, 1, 1, 2};
        const ld c = 2 / sqrtl(kPiL);
        for (int i = 0; i < 4; ++i)
            for (int k = 0; k < kTerms; ++k) {
                const int n = k + skip[i];
                ld f[4] = {0, 0, 0, 0}, fact = 1;   // (-1)^(n-m) / (n-m)!
                std::vector<ld> inv(n + 1, 1.0L);
                for (int j = 1; j <= n; ++j) { fact *= j; inv[j] = 1 / fact; }
                ld a = ((n & 1) ? -1 : 1) * inv[n] / (2 * n + 1);
                for (int m = 0; m < 4 && m <= n; ++m) {
                    f[m] = (((n - m) & 1) ? -1 : 1) * inv[n - m];
                    a += q[i][m] * f[m];
                }
                ser[i][k] = c * a;
            }
    }
    // sigma_1 .. sigma_4 at t
    void at(ld t, ld out[4]) const {
        if (t < 2) {
            for (int i = 0; i < 4; ++i) {
                ld s = 0;
                for (int k = kTerms - 1; k >= 0; --k) s = s * t + ser[i][k];
                out[i] = s;
            }
            return;
        }
        const ld rho = sqrtl(t);
        ld er = 1, g = 0;
        if (t < 80) {   // beyond, erf = 1 and e^{-t} = 0 to the table's precision
            er = erfl(rho);
            g = 2 / sqrtl(kPiL) * rho * expl(-t);
        }
        const ld s1 = er + g * (5 - 2 * t) / 3, s2 = er + g * (2 * t - 3) / 3,
                 s3 = er + g * (t * (14 - 4 * t) - 3) / 3,
                 s4 = er - g * (t * (t * (8 * t - 36) + 6) + 9) / 9;
        out[0] = s1 / rho;
        out[1] = s2 / (rho * t);
        out[2] = s3 / (rho * t);
        out[3] = s4 / (rho * t * t);
    }
};

int64_t round_ll(ld x) { return (int64_t)llrintl(x); }

std::vector<FxI4> build() {
    static const Sigma sig;
    std::vector<FxI4> tab((size_t)kFxTabEntries * kFxEntry);
    ld node[kNodes], cheb[kNodes][kNodes];   // nodes, T_k(node_j)
    for (int j = 0; j < kNodes; ++j) {
        node[j] = cosl(kPiL * (j + 0.5L) / kNodes);
        for (int k = 0; k < kNodes; ++k) cheb[k][j] = cosl(kPiL * k * (j + 0.5L) / kNodes);
    }
    ld mono[kDeg + 1][kDeg + 1] = {};        // T_k in powers of s
    mono[0][0] = 1;
    mono[1][1] = 1;
    for (int k = 2; k <= kDeg; ++k)
        for (int p = 0; p <= k; ++p) mono[k][p] = (p ? 2 * mono[k - 1][p - 1] : 0) - mono[k - 2][p];
    // entry of the polynomial through val (at the nodes), coefficient units 2^unit ..
    auto entry = [&](const ld *val, int unit, FxI4 *t) {
        ld c[kDeg + 1] = {}, top = 0;
        for (int j = 0; j < kNodes; ++j) top = fmaxl(top, fabsl(val[j]));
        for (int k = 0; k <= kDeg; ++k) {
            ld a = 0;
            for (int j = 0; j < kNodes; ++j) a += val[j] * cheb[k][j];
            a *= (k ? 2.0L : 1.0L) / kNodes;
            for (int p = 0; p <= k; ++p) c[p] += a * mono[k][p];
        }
        int ex;
        frexpl(top * 1.002L, &ex);          // top < 2^ex: mantissa below 2^62 over the whole segment
        const int e = 1 - ex;
        const ld u = ldexpl(1, 61 + e);
        int64_t q[kDeg + 1];
        for (int p = 0; p <= 3; ++p) q[p] = round_ll(c[p] * u);
        for (int p = 4; p <= kDeg; ++p) q[p] = round_ll(ldexpl(c[p] * u, p - 4 - unit));
        auto lo = [](int64_t x) { return (int)(uint32_t)x; };
        auto hi = [](int64_t x) { return (int)(x >> 32); };
        t[0] = FxI4{lo(q[0]), hi(q[0]), lo(q[1]), hi(q[1])};
        t[1] = FxI4{lo(q[2]), hi(q[2]), lo(q[3]), hi(q[3])};
        t[2] = FxI4{(int)q[4], (int)q[5], (int)q[6], (int)((uint32_t)(int)q[7] << 8 | (uint32_t)(e + kFxEBias))};
    };
    auto segments = [&](int first, int step) {
        for (int n = first; n < kFxMaxOct * kFxSeg; n += step) {
            const int o = n / kFxSeg, g = n % kFxSeg;
            const ld base = ldexpl(1, o), hw = base / (2 * kFxSeg);
            const ld vc = base + (2 * g + 1) * hw;
            ld val[4][kNodes], bare[kNodes];
            for (int j = 0; j < kNodes; ++j) {
                ld v4[4];
                sig.at(vc - 1 + hw * node[j], v4);
                for (int i = 0; i < 4; ++i) val[i][j] = v4[i];
                bare[j] = 1 / sqrtl(vc + hw * node[j]);
            }
            for (int i = 0; i < 4; ++i)
                entry(val[i], fx_unit(i), &tab[((size_t)i * kFxMaxOct * kFxSeg + (size_t)o * kFxSeg + g) * kFxEntry]);
            if (o < 2)
                entry(bare, fx_unit(0), &tab[((size_t)4 * kFxMaxOct * kFxSeg + (size_t)o * kFxSeg + g) * kFxEntry]);
        }
    };
    const int step = std::min(16, std::max(1, (int)std::thread::hardware_concurrency()));
    std::vector<std::thread> helpers;
    helpers.reserve(step);
    int first = 1;
    try {
        for (; first < step; ++first) helpers.emplace_back(segments, first, step);
    } catch (const std::exception &) {   // no more threads: the rest here
    }
    segments(0, step);
    for (; first < step; ++first) segments(first, step);
    for (auto &t : helpers) t.join();
    return tab;
}

}  // namespace

const FxI4 *fx_table_host() {
    static std::once_flag once;
    static std::vector<FxI4> tab;
    try {
        std::call_once(once, [] { tab = build(); });
    } catch (const std::bad_alloc &) {   // the next call tries again
        return nullptr;
    }
    return tab.data();
}

}  // namespace ssd
