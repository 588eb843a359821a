// Off-surface evaluation (FP64): the Darcy pressure inside the body from
// Green's representation (eq. Greens), the Stokes velocity outside from the
// Stokes representation (eq. Stokes) and the Stokes pressure outside from the
// pressures that go with its two kernels, given the boundary data of a D-N
// solve.  Bare kernels: the surface quadrature is accurate for field points a
// few grid spacings away from the surface.
//
// Prepared point sets: the velocity and the Darcy pressure run in fixed point
// on the integer pipes (fx.h), one field point per thread, bare kernels from
// one table of t^(-1/2) (csrc/fx_pair.h).  Everything else, and there the field
// points closer than a point spacing or far outside, in double precision.
#include <math.h>

#include "fx_geo.h"
#include "fx_pair.h"
#include "internal.h"

namespace ssd {
namespace {

constexpr int kFieldTPB = 256;
constexpr int kFieldT = 32;          // field points per CTA of the double-precision kernels
constexpr int kFieldG = kFieldTPB / kFieldT;   // source groups (warps)
constexpr int kFieldTile = 128;      // sources staged at a time
constexpr double kPiF = 3.14159265358979323846;

struct FieldArgs {
    int64_t n, nt;
    const double *xyz, *nrm, *w;   // surface [3][n], [3][n], [n]
    const double *a, *b;           // Darcy: q [n], p [n]; Stokes: f [3][n], u [3][n]
    const double *y;               // field points [3][nt]
    double ca, cb;                 // coefficients of the single and double layer sums
    double u0[3];                  // far field (Stokes)
    double *out;                   // pressures [nt]; velocity [3][nt]
};

enum FieldKind { kDarcy, kVelocity, kPressure };

// One warp per source group: lane = field point, sources by broadcast from
// shared memory, the groups' sums added in order.  FP64 issues 1.6 operations a
// clock and SM, so what counts is their number (reciprocal square roots instead
// of square roots and divisions) and an even load: 32 field points per CTA
// (20001 points: 626 CTAs; one thread per point left 157 CTAs of 128 on 152
// SMs, two on five of them).
//   Darcy:    ca w q / r + cb w p (yh . n) / r^3
//   velocity: ca w [f / r + yh (yh . f) / r^3] + cb w (u . yh)(yh . n) yh / r^5
//   pressure: ca w (yh . f) / r^3 + cb w [(u . n) / r^3 - 3 (yh . u)(yh . n) / r^5]
// with yh = y - x_j, high powers of 1 / r multiplied in parts (r^-5 leaves the
// range first).
template <FieldKind KIND>
__global__ void __launch_bounds__(kFieldTPB) field_kernel(const FieldArgs A) {
    constexpr int NC = KIND == kVelocity ? 3 : 1, NB = KIND == kDarcy ? 1 : 3;
    __shared__ double sx[3][kFieldTile], sn[3][kFieldTile], sa[NB][kFieldTile], sb[NB][kFieldTile];
    __shared__ double red[NC][kFieldG][kFieldT];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t t = (int64_t)blockIdx.x * kFieldT + lane;
    const bool act = t < A.nt;
    double y[3] = {0.0, 0.0, 0.0}, s[NC] = {};
    if (act)
        for (int e = 0; e < 3; ++e) y[e] = A.y[e * A.nt + t];
    for (int64_t base = 0; base < A.n; base += kFieldTile) {
        __syncthreads();
        const int64_t m = base + threadIdx.x;
        if (threadIdx.x < kFieldTile && m < A.n) {
            const double w = A.w[m], wa = A.ca * w, wb = A.cb * w;
            for (int e = 0; e < 3; ++e) {
                sx[e][threadIdx.x] = A.xyz[e * A.n + m];
                sn[e][threadIdx.x] = (KIND == kDarcy ? 1.0 : wb) * A.nrm[e * A.n + m];
            }
            for (int e = 0; e < NB; ++e) {
                sa[e][threadIdx.x] = wa * A.a[e * A.n + m];
                sb[e][threadIdx.x] = (KIND == kDarcy ? wb : 1.0) * A.b[e * A.n + m];
            }
        }
        __syncthreads();
        const int cnt = (int)((A.n - base) < kFieldTile ? (A.n - base) : kFieldTile);
        for (int j = g; j < cnt; j += kFieldG) {
            const double d[3] = {y[0] - sx[0][j], y[1] - sx[1][j], y[2] - sx[2][j]};
            const double ri = rsqrt(fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])));
            const double ri2 = ri * ri, ri3 = ri2 * ri;
            const double dn = fma(d[2], sn[2][j], fma(d[1], sn[1][j], d[0] * sn[0][j]));
            if constexpr (KIND == kDarcy) {
                s[0] = fma(fma(sb[0][j], dn * ri2, sa[0][j]), ri, s[0]);
            } else {
                const double df = fma(d[2], sa[2][j], fma(d[1], sa[1][j], d[0] * sa[0][j]));
                const double du = fma(d[2], sb[2][j], fma(d[1], sb[1][j], d[0] * sb[0][j]));
                if constexpr (KIND == kVelocity) {
                    const double b = fma(df, ri3, (du * ri2) * (dn * ri3));
                    for (int e = 0; e < 3; ++e) s[e] = fma(sa[e][j], ri, fma(d[e], b, s[e]));
                } else {
                    const double un = fma(sb[2][j], sn[2][j], fma(sb[1][j], sn[1][j], sb[0][j] * sn[0][j]));
                    s[0] = fma(ri3, df + (un - 3.0 * du * (dn * ri2)), s[0]);   // n_S = -n flips both terms
                }
            }
        }
    }
    for (int e = 0; e < NC; ++e) red[e][g][lane] = s[e];
    __syncthreads();
    if (g == 0 && act)
        for (int e = 0; e < NC; ++e) {
            double v = red[e][0][lane];
            for (int k = 1; k < kFieldG; ++k) v += red[e][k][lane];
            A.out[e * A.nt + t] = v + A.u0[e];
        }
}

// ------------------------------------------------------------- fixed point
// Bounds of the fixed-point units need a lower bound of the distances.  Field
// points come in any order, so each thread takes its own per tile, from a pass
// over the tile in single precision (8 of about 350 instructions a pair).
// Lengths are in units of the point spacing sqrt(sum w / n): a thread whose
// nearest source of a tile is closer than that, whose point lies more than 8
// extents out or is not finite, or all threads when the densities have no
// common scale, run the tile in double precision.
constexpr double kFieldMaxExt = 512.0;
constexpr int kFieldHead = 4;

struct FieldFx {
    int64_t n, n_pad, nt;
    const int32_t *perm;
    const d4 *pos, *wn;           // layout order
    const double *a, *b, *y;      // caller order
    double ca, cb;
    double u0[3];
    FxGeo geo;
    l4 *X;                        // packed, layout order
    int4 *cbox;
    d4 *d0, *d1;                  // velocity: cb u, ca w f; Darcy: d0 = (cb p, ca w q)
    unsigned long long *bmax;     // [block][2]
    int nblk;
    const FxI4 *tab;
    int64_t chunk;
    int nsplit;
    double *part;                 // [split][NC][nt]; one split: not used
    double *out;
};

constexpr int kFieldPack = 64;

template <bool VEL>
__global__ void __launch_bounds__(kFieldPack) field_pack_kernel(const FieldFx A) {
    __shared__ unsigned long long smax[2][kFieldPack / 32];
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * kFieldPack + threadIdx.x;   // n_pad is a multiple of 512
    pdl_wait();
    pdl_release();
    const int32_t o = A.perm[i];
    d4 r0 = {0.0, 0.0, 0.0, 0.0}, r1 = r0;
    if (o >= 0) {
        const double wa = A.ca * A.pos[i].w;
        if (VEL) {
            r0 = d4{A.cb * A.b[o], A.cb * A.b[A.n + o], A.cb * A.b[2 * A.n + o], 0.0};
            r1 = d4{wa * A.a[o], wa * A.a[A.n + o], wa * A.a[2 * A.n + o], 0.0};
        } else {
            r0 = d4{A.cb * A.b[o], wa * A.a[o], 0.0, 0.0};
        }
    }
    A.d0[i] = r0;
    if (VEL) A.d1[i] = r1;
    const unsigned long long am = 0x7fffffffffffffffull;
    auto bits = [&](double v) { return (unsigned long long)__double_as_longlong(v) & am; };
    unsigned long long m0 = bits(r0.x), m1;
    if (VEL) { m0 = max(m0, max(bits(r0.y), bits(r0.z))); m1 = max(bits(r1.x), max(bits(r1.y), bits(r1.z))); }
    else m1 = bits(r0.y);
    for (int off = 16; off > 0; off >>= 1) {
        m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, off));
        m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, off));
    }
    if (lane == 0) { smax[0][threadIdx.x >> 5] = m0; smax[1][threadIdx.x >> 5] = m1; }
    __syncthreads();
    if (threadIdx.x < 2) A.bmax[2 * blockIdx.x + threadIdx.x] = max(smax[threadIdx.x][0], smax[threadIdx.x][1]);
    const d4 p = A.pos[i < A.n ? i : A.n - 1];   // padding: a copy of the last point, with zero densities
    const int64_t x = fx_grid(p.x, A.geo.c[0], A.geo), y = fx_grid(p.y, A.geo.c[1], A.geo), z = fx_grid(p.z, A.geo.c[2], A.geo);
    A.X[i] = l4{x, y, z, 0};
    const int xh = (int)(x >> 32), yh = (int)(y >> 32), zh = (int)(z >> 32);
    const int4 lo = make_int4(__reduce_min_sync(0xffffffffu, xh), __reduce_min_sync(0xffffffffu, yh),
                              __reduce_min_sync(0xffffffffu, zh), 0);
    const int4 hi = make_int4(__reduce_max_sync(0xffffffffu, xh), __reduce_max_sync(0xffffffffu, yh),
                              __reduce_max_sync(0xffffffffu, zh), 0);
    if (lane == 0) { A.cbox[2 * (i / kChunk)] = lo; A.cbox[2 * (i / kChunk) + 1] = hi; }
}

// GROUPS as in the pair kernel: threads that share a field point and split the sources.
template <bool VEL, int GROUPS>
__global__ void __launch_bounds__(kFieldTPB, 2) field_fx_kernel(const FieldFx A) {
    constexpr int OP = VEL ? OP_SSLDL : OP_LSLDL;
    constexpr int NC = VEL ? 3 : 1, NT = kFieldTPB / GROUPS, NW = kFieldTPB / 32;
    __shared__ int4 s_tab[kFxBareEntries * kFxEntry];
    __shared__ int4 s_xh[kFieldTile], s_xl[kFieldTile], s_mh[kFieldTile], s_ml[kFieldTile];
    __shared__ int4 s_uh[VEL ? kFieldTile : 1], s_ul[VEL ? kFieldTile : 1], s_fh[VEL ? kFieldTile : 1],
        s_fl[VEL ? kFieldTile : 1];
    __shared__ float4 s_pos[kFieldTile];
    __shared__ unsigned long long s_max[2][NW];
    __shared__ int s_box[6][NW];
    __shared__ double s_sum[GROUPS > 1 ? NC : 1][GROUPS > 1 ? kFieldTPB : 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = threadIdx.x / NT;
    const int64_t t = (int64_t)blockIdx.x * NT + threadIdx.x % NT;
    const bool act = t < A.nt;
    for (int k = threadIdx.x; k < kFxBareEntries * kFxEntry; k += kFieldTPB)
        s_tab[k] = reinterpret_cast<const int4 *>(A.tab)[(int64_t)4 * kFxMaxOct * kFxSeg * kFxEntry + k];
    pdl_wait();
    pdl_release();
    double yt[3] = {0.0, 0.0, 0.0};
    if (act)
        for (int e = 0; e < 3; ++e) yt[e] = A.y[e * A.nt + t];
    // the point on the grid, where it fits
    const double lim = 1152921504606846976.0 / A.geo.grid;   // 2^60 grid steps
    bool ok = act;
    int64_t Y[3] = {0, 0, 0};
    for (int e = 0; e < 3; ++e) ok = ok && fabs((yt[e] - A.geo.c[e]) * A.geo.inv) < lim;
    if (ok)
        for (int e = 0; e < 3; ++e) Y[e] = fx_grid(yt[e], A.geo.c[e], A.geo);
    unsigned long long m0 = 0, m1 = 0;
    for (int b = threadIdx.x; b < A.nblk; b += kFieldTPB) { m0 = max(m0, A.bmax[2 * b]); m1 = max(m1, A.bmax[2 * b + 1]); }
    for (int off = 16; off > 0; off >>= 1) {
        m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, off));
        m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, off));
    }
    if (lane == 0) { s_max[0][warp] = m0; s_max[1][warp] = m1; }
    for (int e = 0; e < 3; ++e) {
        const int lo = __reduce_min_sync(0xffffffffu, ok ? (int)(Y[e] >> 32) : 0x7fffffff);
        const int hi = __reduce_max_sync(0xffffffffu, ok ? (int)(Y[e] >> 32) : -0x7fffffff);
        if (lane == 0) { s_box[e][warp] = lo; s_box[3 + e][warp] = hi; }
    }
    __syncthreads();
    int ee[2];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        unsigned long long m = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) m = max(m, s_max[k][w]);
        const int ex = (int)(m >> 52);
        ee[k] = m == 0 ? -kFxExpMax : ex - 1022;
        bad |= m != 0 && (ee[k] > kFxExpMax || ee[k] < -kFxExpMax);
    }
    int tlo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, thi[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
#pragma unroll
    for (int w = 0; w < NW; ++w)
#pragma unroll
        for (int e = 0; e < 3; ++e) { tlo[e] = min(tlo[e], s_box[e][w]); thi[e] = max(thi[e], s_box[3 + e][w]); }
    const FxGeo &g = A.geo;
    const FxScale sc = fx_scale<OP>(ee[0], ee[1], g.em, g.dq, g.ed);
    const float tf[3] = {(float)(int)(Y[0] >> 32), (float)(int)(Y[1] >> 32), (float)(int)(Y[2] >> 32)};
    const float unit = ldexpf(1.f, 32 - g.ps);
    FxPoint<OP> y;
    for (int c = 0; c < 3; ++c) y.u.h[c] = y.u.l[c] = 0;
    y.p = 0;
    auto tab = [&](int, uint32_t idx, int w) {
        const int4 v = s_tab[idx * kFxEntry + w];
        return FxI4{v.x, v.y, v.z, v.w};
    };
    double sum[NC] = {}, low[NC] = {};
    const int64_t top = (A.n + kChunk - 1) / kChunk * kChunk;
    const int64_t s_beg = blockIdx.y * A.chunk, s_end = s_beg + A.chunk < top ? s_beg + A.chunk : top;
    for (int64_t tile = s_beg; tile < s_end; tile += kFieldTile) {
        const int cnt = (int)(s_end - tile < kFieldTile ? s_end - tile : kFieldTile);
        // exponent of the largest distance of the tile (of the points on the grid)
        int dmax = 1;
        for (int k = 0; k < cnt / kChunk; ++k) {
            const int4 l = A.cbox[2 * (tile / kChunk + k)], h = A.cbox[2 * (tile / kChunk + k) + 1];
            if (tlo[0] <= thi[0]) {
                dmax = max(dmax, max(thi[0] - l.x, h.x - tlo[0]) + 1);
                dmax = max(dmax, max(thi[1] - l.y, h.y - tlo[1]) + 1);
                dmax = max(dmax, max(thi[2] - l.z, h.z - tlo[2]) + 1);
            }
        }
        const int L = max(0, 32 - g.ps + (32 - __clz(dmax - 1)));
        const int ks = 61 - L - g.ps;
        auto grid = [&](int64_t v) { return ks >= 0 ? (int64_t)((uint64_t)v << ks) : v >> -ks; };
        __syncthreads();
        if (threadIdx.x < cnt) {
            const int64_t j = tile + threadIdx.x;
            const l4 p = A.X[j];
            const d4 e0 = A.d0[j], m = A.wn[j];
            s_pos[threadIdx.x] = make_float4((float)(int)(p.x >> 32), (float)(int)(p.y >> 32), (float)(int)(p.z >> 32), 0.f);
            if (!bad) {
                int4 h, l;
                fx_split(grid(p.x), h.x, l.x);
                fx_split(grid(p.y), h.y, l.y);
                fx_split(grid(p.z), h.z, l.z);
                if constexpr (!VEL) {
                    const int64_t q = fx_fix(e0.x, sc.eu, 60);
                    h.w = (int)(q >> 32);
                    l.w = (int)q;
                }
                s_xh[threadIdx.x] = h;
                s_xl[threadIdx.x] = l;
                fx_split(fx_fix(m.x, sc.em, 59), h.x, l.x);
                fx_split(fx_fix(m.y, sc.em, 59), h.y, l.y);
                fx_split(fx_fix(m.z, sc.em, 59), h.z, l.z);
                if constexpr (!VEL) {
                    const int64_t q = fx_fix(e0.y, sc.ef, 60);
                    h.w = (int)(q >> 32);
                    l.w = (int)q;
                }
                s_mh[threadIdx.x] = h;
                s_ml[threadIdx.x] = l;
                if constexpr (VEL) {
                    fx_split(fx_fix(e0.x, sc.eu, 58), h.x, l.x);
                    fx_split(fx_fix(e0.y, sc.eu, 58), h.y, l.y);
                    fx_split(fx_fix(e0.z, sc.eu, 58), h.z, l.z);
                    s_uh[threadIdx.x] = h;
                    s_ul[threadIdx.x] = l;
                    const d4 e1 = A.d1[j];
                    fx_split(fx_fix(e1.x, sc.ef, 58), h.x, l.x);
                    fx_split(fx_fix(e1.y, sc.ef, 58), h.y, l.y);
                    fx_split(fx_fix(e1.z, sc.ef, 58), h.z, l.z);
                    s_fh[threadIdx.x] = h;
                    s_fl[threadIdx.x] = l;
                }
            }
        }
        __syncthreads();
        // lower bound of this thread's distances (grid positions to 2^-24: 2% are plenty)
        float r2 = 3e38f;
        for (int j = grp; j < cnt; j += GROUPS) {
            const float4 p = s_pos[j];
            const float dx = tf[0] - p.x, dy = tf[1] - p.y, dz = tf[2] - p.z;
            r2 = fminf(r2, fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
        }
        r2 *= 0.98f * unit * unit;
        double v[NC] = {};
        if (!bad && ok && r2 >= 1.f) {
            const int r = min(L, ((__float_as_int(r2) >> 23) - 127) >> 1);
            FxTile tl = fx_tile<OP>(sc, L, r);
            tl.one = 0;
            for (int c = 0; c < 3; ++c) fx_split(grid(Y[c]), y.x.h[c], y.x.l[c]);
            FxSum<OP> acc{};
#pragma unroll 2
            for (int j = grp; j < cnt; j += GROUPS) {
                FxPoint<OP> x;
                auto vec = [](FxV &q, const int4 &h, const int4 &l) {
                    q.h[0] = h.x; q.h[1] = h.y; q.h[2] = h.z;
                    q.l[0] = l.x; q.l[1] = l.y; q.l[2] = l.z;
                };
                const int4 xh = s_xh[j], xl = s_xl[j], mh = s_mh[j], ml = s_ml[j];
                vec(x.x, xh, xl);
                vec(x.m, mh, ml);
                if constexpr (VEL) {
                    vec(x.u, s_uh[j], s_ul[j]);
                    vec(x.f, s_fh[j], s_fl[j]);
                } else {
                    x.p = ((int64_t)xh.w << 32) | (uint32_t)xl.w;
                    x.g = ((int64_t)mh.w << 32) | (uint32_t)ml.w;
                }
                fx_pair<OP, kFxBare>(y, x, tl, sc, 0u, tab, acc);
            }
            const double f = __longlong_as_double((long long)(1023 + tl.ex) << 52) * g.f_sl;
            if constexpr (VEL) {
                for (int c = 0; c < 3; ++c) v[c] = fx_value(acc.v[c]) * f;
            } else {
                v[0] = ((double)acc.f.h + (double)acc.f.l * 2.3283064365386963e-10) * f;
            }
        } else if (act) {
            for (int j = grp; j < cnt; j += GROUPS) {
                if (tile + j >= A.n) break;
                const d4 p = A.pos[tile + j], m = A.wn[tile + j], e0 = A.d0[tile + j];
                const double d[3] = {yt[0] - p.x, yt[1] - p.y, yt[2] - p.z};
                const double ri = rsqrt(fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0])));
                const double ri2 = ri * ri, ri3 = ri2 * ri;
                const double dn = fma(d[2], m.z, fma(d[1], m.y, d[0] * m.x));
                if constexpr (VEL) {
                    const d4 e1 = A.d1[tile + j];
                    const double df = fma(d[2], e1.z, fma(d[1], e1.y, d[0] * e1.x));
                    const double du = fma(d[2], e0.z, fma(d[1], e0.y, d[0] * e0.x));
                    const double b = fma(df, ri3, (du * ri2) * (dn * ri3));
                    v[0] = fma(e1.x, ri, fma(d[0], b, v[0]));
                    v[1] = fma(e1.y, ri, fma(d[1], b, v[1]));
                    v[2] = fma(e1.z, ri, fma(d[2], b, v[2]));
                } else {
                    v[0] = fma(fma(e0.x, dn * ri2, e0.y), ri, v[0]);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {   // TwoSum over the tiles
            const double q = sum[c] + v[c], b = q - sum[c];
            low[c] += (sum[c] - (q - b)) + (v[c] - b);
            sum[c] = q;
        }
    }
    // (a sum that is not finite has no low part)
#pragma unroll
    for (int c = 0; c < NC; ++c)
        if (isfinite(sum[c])) sum[c] += low[c];
    if constexpr (GROUPS > 1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) s_sum[c][threadIdx.x] = sum[c];
        __syncthreads();
        if (grp) return;
        for (int k = 1; k < GROUPS; ++k)
#pragma unroll
            for (int c = 0; c < NC; ++c) sum[c] += s_sum[c][threadIdx.x + k * NT];
    }
    if (!act) return;
    if (A.nsplit == 1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) A.out[c * A.nt + t] = sum[c] + A.u0[c];
        return;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) A.part[((int64_t)blockIdx.y * NC + c) * A.nt + t] = sum[c];
}

template <bool VEL>
__global__ void __launch_bounds__(64) field_sum_kernel(const FieldFx A) {
    constexpr int NC = VEL ? 3 : 1;
    pdl_wait();
    pdl_release();
    const int64_t g = (int64_t)blockIdx.x * 64 + threadIdx.x;
    if (g >= NC * A.nt) return;
    double s0 = 0.0, s1 = 0.0;
    int k = 0;
    for (; k + 1 < A.nsplit; k += 2) {
        s0 += A.part[(int64_t)k * NC * A.nt + g];
        s1 += A.part[(int64_t)(k + 1) * NC * A.nt + g];
    }
    if (k < A.nsplit) s0 += A.part[(int64_t)k * NC * A.nt + g];
    A.out[g] = (s0 + s1) + A.u0[g / A.nt];
}

// Fixed-point evaluation on a prepared layout; *done is false where it does not serve
// the point set, or has no workspace: a captured call whose pool has no block of the
// size, a device without the memory.  The kernel in double needs none.
template <bool VEL> int field_fx(ssd_ctx *ctx, const ssd_points *pts, const FieldArgs &F, cudaStream_t s, bool *done) {
    *done = false;
    if (!pts->layout) return SSD_OK;
    const Layout &L = pts->layout->L;
    FieldFx A{};
    int noct = 0;
    if (!fx_geo(L.ext, sqrt(L.wsum / (double)L.n), &A.geo, &noct, kFieldMaxExt, kFieldHead)) return SSD_OK;
    constexpr int NC = VEL ? 3 : 1;
    const int groups = F.nt < 4096 ? 4 : 1;
    const int64_t span = kFieldTPB / groups, ntt = (F.nt + span - 1) / span, units = (L.n + kChunk - 1) / kChunk;
    if (ntt > 0x7fffffff) return SSD_OK;
    int64_t ns = ((int64_t)ctx->num_sms * 2 * (groups > 1 ? 2 : 8) + ntt - 1) / ntt;
    ns = ns < 1 ? 1 : (ns > units ? units : ns);
    int64_t cu = (units + ns - 1) / ns;
    if (cu > 4) cu = (cu + 3) / 4 * 4;
    A.n = L.n; A.n_pad = L.n_pad; A.nt = F.nt; A.perm = L.perm; A.pos = L.pos64; A.wn = L.wn64;
    A.a = F.a; A.b = F.b; A.y = F.y; A.ca = F.ca; A.cb = F.cb; A.out = F.out;
    for (int e = 0; e < 3; ++e) A.u0[e] = F.u0[e];
    A.chunk = cu * kChunk;
    A.nsplit = (int)((units + cu - 1) / cu);
    A.nblk = (int)(L.n_pad / kFieldPack);
    A.tab = static_cast<const FxI4 *>(ctx->fx_tab);
    size_t off = 0;
    auto carve = [&](size_t b) { size_t o = off; off += (b + 255) & ~size_t(255); return o; };
    const size_t o_x = carve(sizeof(l4) * L.n_pad), o_b = carve(sizeof(int4) * 2 * (L.n_pad / kChunk)),
                 o_0 = carve(sizeof(d4) * L.n_pad), o_1 = VEL ? carve(sizeof(d4) * L.n_pad) : 0,
                 o_m = carve(sizeof(unsigned long long) * 2 * A.nblk),
                 o_p = A.nsplit > 1 ? carve(sizeof(double) * NC * F.nt * A.nsplit) : 0;
    void *ws = nullptr;
    if (!dev_cached(ctx, off)) {
        if (capturing(s)) return SSD_OK;
        const int st = dev_alloc(ctx, off, &ws);
        if (st == SSD_ENOMEM) {
            ctx->err.clear();
            cudaGetLastError();
            return SSD_OK;
        }
        SSD_TRY(st);
    } else {
        SSD_TRY(dev_alloc(ctx, off, &ws));
    }
    struct Release { ssd_ctx *c; void *p; ~Release() { dev_free(c, p); } } release{ctx, ws};
    char *b = static_cast<char *>(ws);
    A.X = reinterpret_cast<l4 *>(b + o_x);
    A.cbox = reinterpret_cast<int4 *>(b + o_b);
    A.d0 = reinterpret_cast<d4 *>(b + o_0);
    A.d1 = reinterpret_cast<d4 *>(b + o_1);
    A.bmax = reinterpret_cast<unsigned long long *>(b + o_m);
    A.part = reinterpret_cast<double *>(b + o_p);
    SSD_TRY(cuda_check(ctx, launch_pdl(field_pack_kernel<VEL>, dim3(A.nblk), dim3(kFieldPack), 0, s, A), "field packing"));
    const dim3 grid((unsigned)ntt, (unsigned)A.nsplit);
    SSD_TRY(cuda_check(ctx, groups == 1 ? launch_pdl(field_fx_kernel<VEL, 1>, grid, dim3(kFieldTPB), 0, s, A)
                                        : launch_pdl(field_fx_kernel<VEL, 4>, grid, dim3(kFieldTPB), 0, s, A),
                       "field kernel"));
    ctx->launches += 2;
    if (A.nsplit > 1) {
        SSD_TRY(cuda_check(ctx, launch_pdl(field_sum_kernel<VEL>, dim3((unsigned)((NC * F.nt + 63) / 64)), dim3(64), 0, s,
                                           A), "field sums"));
        ctx->launches++;
    }
    *done = true;
    return SSD_OK;
}

template <FieldKind KIND> int field_launch(ssd_ctx *ctx, const FieldArgs &A, cudaStream_t s) {
    field_kernel<KIND><<<(unsigned)((A.nt + kFieldT - 1) / kFieldT), kFieldTPB, 0, s>>>(A);
    ctx->launches++;
    return launch_check(ctx, "field kernel");
}

int field_common(ssd_ctx *ctx, const ssd_points *pts, int64_t nt, const double *targets, double *out) {
    SSD_TRY(check_points(ctx, pts));
    if (nt < 0) return set_error(ctx, SSD_EINVAL, "negative field-point count");
    if (nt > 0 && (!targets || !out)) return set_error(ctx, SSD_EINVAL, "NULL field points or output");
    return SSD_OK;
}

}  // namespace
}  // namespace ssd

using namespace ssd;

extern "C" {

int ssd_darcy_pressure_field(ssd_ctx *ctx, const ssd_points *pts, double mu, double kappa, const double *q,
                             const double *p, int64_t nt, const double *targets, double *out, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    ctx->err.clear();
    SSD_TRY(field_common(ctx, pts, nt, targets, out));
    if (!(mu > 0.0) || !(kappa > 0.0) || !isfinite(mu) || !isfinite(kappa))
        return set_error(ctx, SSD_EINVAL, "mu and kappa must be positive");
    if (!q || !p) return set_error(ctx, SSD_EINVAL, "NULL boundary data");
    if (nt == 0) return SSD_OK;
    FieldArgs A;
    A.n = pts->n; A.nt = nt; A.xyz = pts->xyz; A.nrm = pts->nrm; A.w = pts->w;
    A.a = q; A.b = p; A.y = targets; A.out = out;
    A.ca = -(mu / kappa) / (4.0 * kPiF);
    A.cb = -1.0 / (4.0 * kPiF);
    A.u0[0] = A.u0[1] = A.u0[2] = 0.0;
    bool done = false;
    SSD_TRY(field_fx<false>(ctx, pts, A, (cudaStream_t)stream, &done));
    return done ? SSD_OK : field_launch<kDarcy>(ctx, A, (cudaStream_t)stream);
}

int ssd_stokes_velocity_field(ssd_ctx *ctx, const ssd_points *pts, double mu, const double uinf[3], const double *f,
                              const double *u, int64_t nt, const double *targets, double *out, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    ctx->err.clear();
    SSD_TRY(field_common(ctx, pts, nt, targets, out));
    if (!(mu > 0.0) || !isfinite(mu)) return set_error(ctx, SSD_EINVAL, "mu must be positive");
    if (!f || !u || !uinf) return set_error(ctx, SSD_EINVAL, "NULL boundary data or far field");
    if (nt == 0) return SSD_OK;
    FieldArgs A;
    A.n = pts->n; A.nt = nt; A.xyz = pts->xyz; A.nrm = pts->nrm; A.w = pts->w;
    A.a = f; A.b = u; A.y = targets; A.out = out;
    A.ca = -1.0 / (8.0 * kPiF * mu);
    A.cb = 6.0 / (8.0 * kPiF);
    for (int e = 0; e < 3; ++e) A.u0[e] = uinf[e];
    bool done = false;
    SSD_TRY(field_fx<true>(ctx, pts, A, (cudaStream_t)stream, &done));
    return done ? SSD_OK : field_launch<kVelocity>(ctx, A, (cudaStream_t)stream);
}

int ssd_stokes_pressure_field(ssd_ctx *ctx, const ssd_points *pts, double mu, const double *f, const double *u,
                              int64_t nt, const double *targets, double *out, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    ctx->err.clear();
    SSD_TRY(field_common(ctx, pts, nt, targets, out));
    if (!(mu > 0.0) || !isfinite(mu)) return set_error(ctx, SSD_EINVAL, "mu must be positive");
    if (!f || !u) return set_error(ctx, SSD_EINVAL, "NULL boundary data");
    if (nt == 0) return SSD_OK;
    FieldArgs A;
    A.n = pts->n; A.nt = nt; A.xyz = pts->xyz; A.nrm = pts->nrm; A.w = pts->w;
    A.a = f; A.b = u; A.y = targets; A.out = out;
    A.ca = -2.0 / (8.0 * kPiF);
    A.cb = -4.0 * mu / (8.0 * kPiF);
    A.u0[0] = A.u0[1] = A.u0[2] = 0.0;
    return field_launch<kPressure>(ctx, A, (cudaStream_t)stream);
}

}  // extern "C"
