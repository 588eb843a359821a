// Fixed-point grid of a point set at a length scale delta (fx.h): constants and
// the conversion of positions.
#pragma once

#include <math.h>

#include "fx.h"
#include "internal.h"

namespace ssd {

constexpr int kFxExpMax = 400;

struct FxGeo {
    double c[3];          // grid origin
    double inv, inv_lo;   // 1 / delta to twice double precision
    double grid;          // 2^ps
    int ps;               // positions: (x - c) / delta in units of 2^-ps
    int em;               // |w n| < 2^em
    int ed, pad;
    int64_t dq;           // 1 / delta = dq 2^(ed - 62)
    double f_sl, f_dl;    // 1 / delta, 1 / delta^2
};

__device__ __forceinline__ int64_t fx_grid(double x, double c, const FxGeo &g) {
    const double hi = x - c, bb = hi - x, lo = (x - (hi - bb)) - (c + bb);   // x - c = hi + lo exactly
    const double q = hi * g.inv;
    const double e = fma(hi, g.inv, -q) + (hi * g.inv_lo + lo * g.inv);
    const double r = q * g.grid;
    const long long a = __double2ll_rn(r);
    return a + __double2ll_rn((r - (double)a) + e * g.grid);
}

// Constants of a point set and smoothing radius; false when the fixed-point
// kernel does not serve it (extent outside kFxMinExt .. kFxMaxExt delta, values
// that are not finite or far from unit scale).  noct: octaves of 1 + rho^2 that
// occur.  head: the grid reaches 2^head times further than the points.
inline bool fx_geo(const Extent &e, double delta, FxGeo *g, int *noct, double max_ext = kFxMaxExt, int head = 0) {
    if (!(e.fin > 0.0)) return false;
    double ext = 0.0, r2 = 0.0;
    for (int c = 0; c < 3; ++c) {
        const double d = e.hi[c] - e.lo[c];
        g->c[c] = 0.5 * (e.lo[c] + e.hi[c]);
        ext = fmax(ext, d / delta);
        r2 += d / delta * (d / delta);
    }
    g->em = 0;
    if (e.mmax > 0.0) frexp(e.mmax, &g->em);
    int xd;
    frexp(delta, &xd);
    double cm = 0.0;
    for (int c = 0; c < 3; ++c) cm = fmax(cm, fabs(g->c[c]));
    if (!(ext >= kFxMinExt && ext <= max_ext) || g->em > kFxExpMax || g->em < -kFxExpMax || xd > 60 || xd < -60 || !(cm < 1e100))
        return false;
    int xe;
    frexp(ext, &xe);
    g->ps = 62 - xe - head < 58 ? 62 - xe - head : 58;   // |x - c| / delta <= 2^(xe - 1): grid values below 2^(62 - head)
    g->grid = ldexp(1.0, g->ps);
    g->inv = 1.0 / delta;
    g->inv_lo = fma(-g->inv, delta, 1.0) / delta;
    const double m = frexp(g->inv, &g->ed);    // 1 / delta = (m + lo) 2^ed, 62 bits
    g->dq = (int64_t)ldexp(m, 53) * 512 + llrint(ldexp(g->inv_lo, 62 - g->ed));
    g->f_sl = 1.0 / delta;
    g->f_dl = 1.0 / (delta * delta);
    g->pad = 0;
    const int k = (int)floor(log2(1.0 + r2 * (1.0 + 1e-12))) + 1;
    *noct = k < kFxMaxOct ? k : kFxMaxOct;
    return true;
}

}  // namespace ssd
