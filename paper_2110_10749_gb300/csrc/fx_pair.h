// One (target, source) pair of an FP64 layer operator in fixed point (fx.h).
// Host and device code; OpInfo and the operator numbers come from the
// including file.
//
// Formats: positions in units of delta, |d| < 2^61 in units of 2^(L-61), L the
// exponent of the tile's largest distance; vector densities |U| <= 2^58 in
// units of 2^(eu-58); weighted normals |M| <= 2^59 in units of 2^(em-59);
// scalar densities |P| <= 2^60 in units of 2^(eu-60).  Each term is shifted to
// fixed point in units of 2^U.  With rho >= 2^r for every pair of the tile,
// |sigma_4 rho^2| < 1.5 2^-3r, |sigma_2 rho| < 0.75 2^-2r,
// |sigma_3 rho| < 2.5 2^-2r and sigma_1 < 3.01 2^-r keep it within 2^57
// whatever the points, so the sums cannot overflow.
#pragma once

#include "fx.h"

namespace ssd {

// operator traits: tables used (sigma_{i+1}), record fields, density kinds
template <int OP> struct FxOp {
    static constexpr bool vec = OP == OP_SSL || OP == OP_SDL || OP == OP_SSLDL || OP == OP_SDLT;
    static constexpr bool dl = OP != OP_LSL && OP != OP_SSL;
    static constexpr bool sl = OP == OP_LSL || OP == OP_SSL || OP == OP_SSLDL || OP == OP_LSLDL;
    static constexpr bool tr = OP == OP_LDLT || OP == OP_SDLT;
    static constexpr bool fused = OP == OP_SSLDL || OP == OP_LSLDL;
    static constexpr bool rest = fused || OP == OP_SDL;   // densities less the first one where those are smaller
    static constexpr int k1 = sl ? 0 : -1;                                   // index among the staged tables
    static constexpr int k3 = vec && sl ? 1 : -1;
    static constexpr int kd = dl ? (fused ? (vec ? 2 : 1) : 0) : -1;
    static constexpr int ntab = (sl ? (vec ? 2 : 1) : 0) + (dl ? 1 : 0);
    static constexpr int tab(int k) { return k == kd ? (vec ? 3 : 1) : (k == 0 ? 0 : 2); }   // sigma index
};

template <int OP> struct FxPoint {       // target or source in a tile's format
    FxV x, m, u, f;                      // unused members are dead code
    int64_t p, g;
};

// per-tile constants
struct FxTile {
    int64_t one;                         // 1 in units of the squared distance's 2^62
    int oct0;                            // segment origin
    int c_dl, c_sl, c_k;                 // shift constants of the double layer, the single
                                         // layer's second part and its first part
    int ex;                              // the tile sum is fx_value 2^ex (vector) or (h + l 2^-32) 2^ex
};

// exponents of a launch: densities eu (double layer, or the only one) and ef
// (single layer of a fused operator), normals em, 1/delta = dq 2^(ed-62)
struct FxScale {
    int eu, ef, em, ed;
    int64_t dq;
};

template <int OP> FX_HD FxScale fx_scale(int eu, int ef, int em, int64_t dq, int ed) {
    typedef FxOp<OP> T;
    FxScale s;
    s.eu = eu; s.ef = T::fused ? ef : eu; s.em = em; s.dq = dq; s.ed = T::fused ? ed : 0;
    return s;
}

// L: exponent of the tile's largest distance; 2^r: a lower bound of its distances (0 <= r <= L)
template <int OP> FX_HD FxTile fx_tile(const FxScale &s, int L, int r) {
    typedef FxOp<OP> T;
    FxTile t;
    t.one = (int64_t)1 << (60 - 2 * L);
    t.oct0 = (2 + 2 * L) * kFxSeg;
    const int ud = s.eu + s.em + s.ed - (T::vec ? 53 + 3 * r : 48 + 2 * r),
              us = s.ef - (T::vec ? 52 + 2 * r : 48 + r);
    const int U = !T::dl ? us : (!T::sl ? ud : (ud > us ? ud : us));
    t.c_dl = T::vec ? U + 52 - 2 * L - s.eu - s.em - s.ed : U + 55 - L - s.eu - s.em - s.ed;
    t.c_sl = U + 56 - L - s.ef;
    t.c_k = T::vec ? 58 + U - s.ef + L : U + 59 - s.ef;
    t.ex = T::vec ? U + L - 22 : U;
    return t;
}

template <int OP> struct FxSum { FxMac v[FxOp<OP>::vec ? 3 : 1]; FxF f; };

// Modes.  kFxFar: every pair of the tile has rho >= 8, where sigma_3 = sigma_1^3
// (bare kernels): the Stokes single layer then needs one table instead of two.
// kFxBare: bare kernels at any rho >= 1, all from one table of t^(-1/2) over
// 1 <= t < 4 (kFxBareEntries segments; t scales by powers of 4), with t.one = 0.
enum FxMode { kFxFull = 0, kFxFar = 1, kFxBare = 2 };

FX_HD FxQ fx_cube(const FxQ &a, int64_t sq) {   // (m 2^-(61+e))^3, sq = m^2 2^-62
    FxQ r;
    r.m = fx_mul(sq, a.m);
    r.e = 3 * a.e - 2;
    return r;
}

// tab(k, idx, w): word w of entry idx of staged table k
template <int OP, FxMode MODE, typename Tab>
FX_HD void fx_pair(const FxPoint<OP> &y, const FxPoint<OP> &x, const FxTile &t, const FxScale &s, uint32_t idx_max,
                   const Tab &tab, FxSum<OP> &acc) {
    typedef FxOp<OP> T;
    FxV d;
    for (int c = 0; c < 3; ++c) { d.h[c] = y.x.h[c] - x.x.h[c]; d.l[c] = y.x.l[c] - x.x.l[c]; }
    const FxArgSeg a = fx_index(d, t.one, t.oct0);
    const uint32_t idx = a.idx < idx_max ? a.idx : idx_max;
    FxQ K1, K3, KD;
    if constexpr (MODE == kFxBare) {
        const uint32_t i = a.idx & (kFxBareEntries - 1);
        K1 = fx_poly<fx_unit(0)>(tab(0, i, 0), tab(0, i, 1), tab(0, i, 2), a.sh, a.sl);
        K1.e += (int)(a.idx / kFxBareEntries);
        const int64_t sq = fx_mul(K1.m, K1.m);
        K3 = fx_cube(K1, sq);
        KD = K3;
        if constexpr (T::vec) { KD.m = fx_mul(K3.m, sq); KD.e = K3.e + 2 * K1.e - 2; }
    } else {
        if constexpr (T::k1 >= 0)
            K1 = fx_poly<fx_unit(0)>(tab(T::k1, idx, 0), tab(T::k1, idx, 1), tab(T::k1, idx, 2), a.sh, a.sl);
        if constexpr (T::k3 >= 0 && MODE == kFxFar)
            K3 = fx_cube(K1, fx_mul(K1.m, K1.m));
        else if constexpr (T::k3 >= 0)
            K3 = fx_poly<fx_unit(2)>(tab(T::k3, idx, 0), tab(T::k3, idx, 1), tab(T::k3, idx, 2), a.sh, a.sl);
        if constexpr (T::kd >= 0)
            KD = fx_poly<fx_unit(T::vec ? 3 : 1)>(tab(T::kd, idx, 0), tab(T::kd, idx, 1), tab(T::kd, idx, 2), a.sh, a.sl);
    }
    if constexpr (!T::vec) {
        if constexpr (OP == OP_LDL || OP == OP_LSLDL) {
            const FxQ B = fx_dot(d, x.m);
            int64_t b = fx_mul(fx_mul(x.p - y.p, KD.m), B.m);
            if constexpr (T::fused) b = fx_mul(b, s.dq);
            acc.f = fx_add(acc.f, fx_shift(b, t.c_dl + KD.e + B.e));
        }
        if constexpr (OP == OP_LDLT) {
            const FxQ Bt = fx_dot(d, y.m), Bs = fx_dot(d, x.m);
            acc.f = fx_add(acc.f, fx_shift(fx_mul(fx_mul(x.p, KD.m), Bt.m), t.c_dl + KD.e + Bt.e));
            acc.f = fx_add(acc.f, fx_shift(fx_mul(fx_mul(y.p, KD.m), Bs.m), t.c_dl + KD.e + Bs.e));
        }
        if constexpr (T::sl) acc.f = fx_add(acc.f, fx_shift(fx_mul(x.g, K1.m), t.c_k + K1.e));
    } else {
        FxF b;
        b.h = 0; b.l = 0;
        if constexpr (OP == OP_SDL || OP == OP_SSLDL) {
            FxV du;
            for (int c = 0; c < 3; ++c) { du.h[c] = x.u.h[c] - y.u.h[c]; du.l[c] = x.u.l[c] - y.u.l[c]; }
            const FxQ A = fx_dot(d, du), B = fx_dot(d, x.m);
            int64_t q = fx_mul(fx_mul(A.m, KD.m), B.m);
            if constexpr (T::fused) q = fx_mul(q, s.dq);
            b = fx_shift(q, t.c_dl + KD.e + A.e + B.e);
        }
        if constexpr (OP == OP_SDLT) {
            const FxQ Bt = fx_dot(d, y.m), Bs = fx_dot(d, x.m), As = fx_dot(d, x.u), At = fx_dot(d, y.u);
            b = fx_shift(fx_mul(fx_mul(As.m, KD.m), Bt.m), t.c_dl + KD.e + As.e + Bt.e);
            b = fx_add(b, fx_shift(fx_mul(fx_mul(At.m, KD.m), Bs.m), t.c_dl + KD.e + At.e + Bs.e));
        }
        if constexpr (T::sl) {
            const FxQ A = fx_dot(d, x.f);
            const FxF q = fx_shift(fx_mul(A.m, K3.m), t.c_sl + K3.e + A.e);
            b = T::dl ? fx_add(b, q) : q;
            const FxB k = fx_limbs(fx_shift(K1.m, t.c_k + K1.e));
            for (int c = 0; c < 3; ++c) fx_mac(acc.v[c], k, x.f.h[c], x.f.l[c]);
        }
        const FxB l = fx_limbs(b);
        for (int c = 0; c < 3; ++c) fx_mac(acc.v[c], l, d.h[c], d.l[c]);
    }
}

}  // namespace ssd
