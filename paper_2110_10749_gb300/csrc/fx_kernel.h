// FP64 pair sums in fixed point: kernel, packing and host set-up (included by
// pair.cu inside its namespace, after the generic pair kernel).
//
// What bounds it: the integer pipes.  One Stokes double-layer pair is about
// 70 wide multiply-adds and 90 shifts, adds and logic operations, two thirds
// of them replacing 31 double-precision operations that issue at 1.6 per
// clock and SM; a smoothed pair costs the same as a bare one, where the
// double-precision kernel also evaluates erf and exp (33 clocks per pair and
// SM).  So there is no near/far split within a launch, every tile costs the same,
// and the grid needs no launch order.  (On a plan the far block pairs are a launch of
// their own, the FAR form below.)
//
// A CTA holds 256 targets, one per thread, and walks its sources 128 at a time
// in shared memory next to the kernel tables (3 KB per octave of 1 + rho^2 and
// table).  Positions keep one global grid; each tile shifts it so that its
// largest distance fills 61 bits.  The tile's sums are integers (exact, so
// their order does not matter); they enter a double accumulator once per tile.
// Tables are read by lane-dependent index, sources by broadcast.
// Measured on the h = 1/32 sphere (N = 17070), against the double-precision
// kernel: Laplace double layer 2.21 ms (18.9), and on small sets, where every
// pair is smoothed, with packing and epilogue: Stokes double layer 0.028 ms
// (0.62) at N = 1062, fused Stokes layers 0.095 ms (1.44) at N = 1742, transposed
// Stokes double layer 0.334 ms (3.7) at N = 4302; errors against long double at
// or below the double kernel's, on densities whose values are within a few orders
// of magnitude (below).  The wide multiplier is 71% busy (32 a clock and
// SM) on large sets, the ALU that shifts and adds 64%; clocks per pair and SM: LSL 1.6, LDL 2.2, SDL 3.3, SSL 4.0,
// SDLT 4.4, SSLDL 6.
//
// Densities are scaled by their largest magnitude, which the packing kernel
// leaves per block; the kernel reduces those at its start.  The double layers see
// differences of densities only.  Where a constant can cost digits (more than one
// component, or a single layer beside it) the packing also leaves the densities less the
// surface's first one, and where these are smaller by 2^5 or more the kernel takes them:
// the scale is then that of the variation, and what a component keeps of its constant
// subtracts exactly (Sterbenz).  (Errors with a constant 1 and a variation of 1e-8 in
// another component: 1.4e-10 without, 1e-16 with it; of a single layer of 1e-8 beside a
// constant double-layer density 3e-12 and 1e-16.)  What remains is relative to the
// largest value: a source 1e12 times the others costs the targets that its kernel
// vanishes on, as those of one plane do for a double layer, 6e-6 of their sums.  When the scale
// does not exist (a NaN, an infinity, or a magnitude outside 2^+-400) the CTA
// evaluates its pairs in double precision instead, as the generic kernel
// does, so non-finite densities give the same results as there.  Point sets
// whose extent is over 256 or under 1/16 delta, or that are not finite, keep the
// generic kernel (fx_geo).

constexpr int kFxGroups = 4;   // source groups of a CTA on small sets
constexpr int kFxUnit = 8;     // and the granularity of their chunks of sources

struct FxArgs {
    const l4 *X;
    const int4 *cbox;            // per 32-point chunk: (lo, hi) of X >> 32
    const unsigned long long *bmax;   // [rhs][pack block][2], see fx_pack
    int64_t nblk;                // pack blocks per right-hand side
    const FxI4 *tab;
    int noct;
    FxGeo geo;
    const FxGeo *geos;           // batched: per surface
    KArgs<double> k;             // the rest, as for the generic kernel
    int64_t n;
};

// what the packing kernels leave for it: the densities' block maxima
struct FxPack {
    unsigned long long *bmax = nullptr;   // NULL: not wanted
    int two = 0;                 // LSLDL: .y of the first record is the second density
    d4 *rest = nullptr;          // double layers: first records less the surface's first one
    const int32_t *elem_surf = nullptr;   // batched: surface of a caller index, and the surfaces
    const BSurf *surfs = nullptr;
};

// magnitude of a double for comparisons and its exponent: the high word without the
// sign, 0 for zero only
__device__ __forceinline__ uint32_t fx_mag(double v) {
    return ((uint32_t)__double2hiint(v) & 0x7fffffffu) | (__double2loint(v) != 0 ? 1u : 0u);
}
__device__ __forceinline__ uint32_t fx_mag(double x, double y, double z) { return max(fx_mag(x), max(fx_mag(y), fx_mag(z))); }

// a record less the first point's, s v; both are rounded records (no contraction)
__device__ __forceinline__ double fx_rest(double r, double s, double v) { return __dsub_rn(r, __dmul_rn(s, v)); }

// Block maxima (every thread of a 256-thread block calls this), 16 bytes per block: the
// bits of the largest |d0| and |d1|, or, with P.rest, a uint4 of fx_mag of the first
// density, of the second one and of the first one's rest.  rest: record r0 less the
// surface's first one (zero for padding); it goes to P.rest[i].
__device__ __forceinline__ void fx_pack(const FxPack &P, const d4 &r0, const d4 &r1, const d4 &rest, int64_t i, int rhs,
                                        int64_t nblk) {
    __shared__ unsigned long long smax[2][8];
    __shared__ uint32_t smag[3][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (P.rest) {
        P.rest[i] = rest;
        const uint32_t m[3] = {P.two ? fx_mag(r0.x) : fx_mag(r0.x, r0.y, r0.z), P.two ? fx_mag(r0.y) : fx_mag(r1.x, r1.y, r1.z),
                               P.two ? fx_mag(rest.x) : fx_mag(rest.x, rest.y, rest.z)};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t v = __reduce_max_sync(0xffffffffu, m[k]);
            if (lane == 0) smag[k][warp] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t[3] = {0u, 0u, 0u};
            for (int w = 0; w < 8; ++w)
                for (int k = 0; k < 3; ++k) t[k] = max(t[k], smag[k][w]);
            reinterpret_cast<uint4 *>(P.bmax)[(int64_t)rhs * nblk + blockIdx.x] = make_uint4(t[0], t[1], t[2], 0u);
        }
        return;
    }
    const unsigned long long am = 0x7fffffffffffffffull;
    auto bits = [&](double v) { return (unsigned long long)__double_as_longlong(v) & am; };
    unsigned long long m0 = max(bits(r0.x), max(bits(r0.y), bits(r0.z))), m1 = max(bits(r1.x), max(bits(r1.y), bits(r1.z)));
    for (int off = 16; off > 0; off >>= 1) {
        m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, off));
        m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, off));
    }
    if (lane == 0) { smax[0][warp] = m0; smax[1][warp] = m1; }
    __syncthreads();
    if (threadIdx.x < 2) {
        unsigned long long m = smax[threadIdx.x][0];
        for (int w = 1; w < 8; ++w) m = max(m, smax[threadIdx.x][w]);
        P.bmax[((int64_t)rhs * nblk + blockIdx.x) * 2 + threadIdx.x] = m;
    }
}

// Positions on the fixed-point grid and their chunk boxes, once per point set
// and smoothing radius (32-thread blocks: about 50 double-precision operations
// a point, so few points per SM).
struct FxGrid {
    const d4 *pos;
    int64_t n_pad, n_last;       // one surface: last real point
    FxGeo geo;
    const FxGeo *geos;           // batched: per surface
    const BSurf *surfs;
    int nsurf;
    l4 *X;
    int4 *cbox;
};

__global__ void __launch_bounds__(kChunk) fx_grid_kernel(const __grid_constant__ FxGrid P) {
    const int64_t i = (int64_t)blockIdx.x * kChunk + threadIdx.x;
    int64_t last = P.n_last;
    const FxGeo *g = &P.geo;
    if (P.geos) {
        int lo = 0, hi = P.nsurf - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (P.surfs[mid].poff <= i) lo = mid; else hi = mid - 1;
        }
        g = P.geos + lo;
        last = P.surfs[lo].poff + P.surfs[lo].n_real - 1;
    }
    const d4 p = P.pos[i <= last ? i : last];   // padding: a copy of the last point, with zero weight and density
    const int64_t x = fx_grid(p.x, g->c[0], *g), y = fx_grid(p.y, g->c[1], *g), z = fx_grid(p.z, g->c[2], *g);
    P.X[i] = l4{x, y, z, 0};
    const int xh = (int)(x >> 32), yh = (int)(y >> 32), zh = (int)(z >> 32);
    const int4 lo = make_int4(__reduce_min_sync(0xffffffffu, xh), __reduce_min_sync(0xffffffffu, yh),
                              __reduce_min_sync(0xffffffffu, zh), 0);
    const int4 hi = make_int4(__reduce_max_sync(0xffffffffu, xh), __reduce_max_sync(0xffffffffu, yh),
                              __reduce_max_sync(0xffffffffu, zh), 0);
    if (threadIdx.x == 0) { P.cbox[2 * blockIdx.x] = lo; P.cbox[2 * blockIdx.x + 1] = hi; }
}

// The generic kernel's pair terms for one target in double precision, all
// pairs of [s_beg, s_end) in order (densities without a common scale).
template <int OP>
__device__ __noinline__ void fx_fallback(const KArgs<double> *ap, const Consts<double> *cp, const d4 *d0, const d4 *d1,
                                         int64_t i, int64_t s_beg, int64_t s_end, double out[3]) {
    const KArgs<double> &a = *ap;
    const Consts<double> c = *cp;
    const d4 yp = a.pos[i], yd = d0[i], yw = a.wn[i];
    const double dt[3] = {yd.x, yd.y, yd.z}, twn[3] = {yw.x, yw.y, yw.z};
    double acc[3] = {0.0, 0.0, 0.0};
    for (int64_t j = s_beg; j < s_end; ++j) {
        const d4 sp = a.pos[j], sw = a.wn[j], s0 = d0[j], s1 = d1[j];
        const double d[3] = {yp.x - sp.x, yp.y - sp.y, yp.z - sp.z};
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        if (r2 < c.rfar2) pair_term<double, OP, true>(d, r2, dt, sw, s0, s1, c, true, false, acc, twn);
        else pair_term<double, OP, false>(d, r2, dt, sw, s0, s1, c, false, false, acc, twn);
    }
    out[0] = acc[0]; out[1] = acc[1]; out[2] = acc[2];
}

// FAR: all items are block pairs at least 8 delta apart (the second launch of a
// plan).  Only the octaves from there on are staged, and the Stokes single
// layer takes sigma_3 from sigma_1: one table of noct - 6 octaves instead of two
// of noct.  Stokes single layer at N = 68166: 58.9 ms with the plan against 64.9
// with every tile on the general kernel; the other layers gain 1-2%.
constexpr int kFxFarOct = 6;                     // 1 + 8^2 > 2^6
template <int OP, bool FAR> constexpr int fx_ntab() { return FAR && OP == OP_SSL ? 1 : FxOp<OP>::ntab; }

// GROUPS > 1: the threads form groups that share the CTA's 256 / GROUPS targets
// and take sources grp, grp + GROUPS, .. of each staged tile; their integer
// sums are added before they become a double.
template <int OP, bool FAR, int GROUPS>
__global__ void __launch_bounds__(kFxTPB, 2) fx_kernel(const FxArgs a) {
    typedef FxOp<OP> T;
    constexpr int kOct0 = FAR ? kFxFarOct : 0;
    const int tstride = (a.noct - kOct0) * kFxSeg * kFxEntry;
    constexpr int NC = OpInfo<OP>::NC;
    constexpr bool M = T::dl, VU = T::dl && T::vec, VF = T::sl && T::vec;
    extern __shared__ __align__(16) FxI4 s_tab[];           // [ntab][noct * kFxSeg][kFxEntry]
    // staged sources: limbs of the vectors, scalars in the spare words
    __shared__ int4 s_xh[kTile], s_xl[kTile];
    __shared__ int4 s_mh[M ? kTile : 1], s_ml[M ? kTile : 1];
    __shared__ int4 s_uh[VU ? kTile : 1], s_ul[VU ? kTile : 1];
    __shared__ int4 s_fh[VF ? kTile : 1], s_fl[VF ? kTile : 1];
    __shared__ __align__(16) unsigned long long s_max[2][kFxTPB / 32];   // or a uint4 per warp
    __shared__ int64_t s_acc[GROUPS > 1 ? 2 * NC : 1][GROUPS > 1 ? kFxTPB : 1];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t tbase, s_beg, s_end, part_base, pstride, b0 = 0, b1 = a.nblk;
    const d4 *d0 = a.k.d0, *d1 = a.k.d1;
    const FxGeo *gp = &a.geo;
    const Consts<double> *cp = &a.k.c;
    if (a.k.items) {
        const BItem it = a.k.items[blockIdx.x];
        const BSurf sf = a.k.surfs[it.surf];
        tbase = it.tbase; s_beg = it.s_beg; s_end = it.s_end;
        if (a.geos) {
            gp = a.geos + it.surf;
            b0 = sf.poff / 256; b1 = (sf.poff + sf.n_pad) / 256;
        }
        cp = a.k.consts + it.surf;
        d0 += blockIdx.y * a.k.rec_stride;
        d1 += blockIdx.y * a.k.rec_stride;
        part_base = blockIdx.y * a.k.part_stride + NC * sf.pbase + (int64_t)it.split * NC * sf.n_pad - sf.poff;
        pstride = sf.n_pad;
    } else {
        tbase = (blockIdx.x + a.k.tile0) * (kFxTPB / GROUPS);
        s_beg = blockIdx.y * a.k.chunk;
        s_end = s_beg + a.k.chunk;
        const int64_t top = (a.n + kChunk - 1) / kChunk * kChunk;
        if (s_end > top) s_end = top;
        part_base = blockIdx.y * NC * a.k.n_pad;
        pstride = a.k.n_pad;
    }
    constexpr int nt = kFxTPB / GROUPS;
    const int grp = threadIdx.x / nt;
    const int64_t i = tbase + threadIdx.x % nt;
    // the tables arrive while the densities' scale is found
    for (int k = 0; k < fx_ntab<OP, FAR>(); ++k) {
        const int4 *src = reinterpret_cast<const int4 *>(a.tab) +
                          ((int64_t)T::tab(k) * kFxMaxOct + kOct0) * kFxSeg * kFxEntry;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_tab) + (uint32_t)(k * tstride) * 16u;
        for (int q = threadIdx.x; q < tstride; q += kFxTPB)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + q * 16u), "l"(src + q));
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    // and, where it pays, the target's grid position and its block's box, which are
    // kept with the layout: Stokes double layer at N = 17070 3.37 ms, 3.48 with these
    // loads after the scale and the tile's boxes one by one; transposed at N = 4302
    // 339 and 350 us; the Laplace layers and the Stokes single layer of large sets
    // lose 0.5%.
    constexpr bool kEarly = GROUPS > 1 || (T::vec && T::dl);
    l4 Y;
    d4 Yd;
    int tlo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, thi[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
    auto grow = [&](int (&lo)[3], int (&hi)[3], int64_t box) {
        const int4 l = a.cbox[2 * box], h = a.cbox[2 * box + 1];
        lo[0] = min(lo[0], l.x); lo[1] = min(lo[1], l.y); lo[2] = min(lo[2], l.z);
        hi[0] = max(hi[0], h.x); hi[1] = max(hi[1], h.y); hi[2] = max(hi[2], h.z);
    };
    auto load_target = [&] {
        Y = a.X[i];
#pragma unroll
        for (int k = 0; k < nt / kChunk; ++k) grow(tlo, thi, tbase / kChunk + k);
    };
    if constexpr (kEarly) load_target();
    pdl_wait();
    pdl_release();
    if constexpr (kEarly) Yd = d0[i];
    // largest densities of this surface and right-hand side
    int ee[2];
    bool bad = false;
    if constexpr (T::rest) {
        uint4 *s_mag = reinterpret_cast<uint4 *>(s_max);
        uint4 m = make_uint4(0u, 0u, 0u, 0u);
        const uint4 *bm = reinterpret_cast<const uint4 *>(a.bmax) + (a.geos ? blockIdx.y : 0) * a.nblk;
        for (int64_t b = b0 + threadIdx.x; b < b1; b += kFxTPB) {
            const uint4 v = bm[b];
            m.x = max(m.x, v.x);
            m.y = max(m.y, v.y);
            m.z = max(m.z, v.z);
        }
        m.x = __reduce_max_sync(0xffffffffu, m.x);
        m.y = __reduce_max_sync(0xffffffffu, m.y);
        m.z = __reduce_max_sync(0xffffffffu, m.z);
        if (lane == 0) s_mag[warp] = m;
        __syncthreads();
        m = s_mag[0];
#pragma unroll
        for (int w = 1; w < kFxTPB / 32; ++w) {
            const uint4 v = s_mag[w];
            m.x = max(m.x, v.x);
            m.y = max(m.y, v.y);
            m.z = max(m.z, v.z);
        }
        // the rest where it is smaller by 2^5 (not below the range)
        if (m.x < 0x7ff00000u && m.z + (5u << 20) <= m.x && (m.z == 0u || m.z >= (uint32_t)(1022 - kFxExpMax) << 20)) {
            m.x = m.z;
            d0 += (a.geos ? (int64_t)gridDim.y : 1) * a.k.n_pad;
            if constexpr (kEarly) Yd = d0[i];
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t t = k ? m.y : m.x;
            ee[k] = t == 0u ? -kFxExpMax : (int)(t >> 20) - 1022;   // all zero: any scale
            bad |= t != 0u && (ee[k] > kFxExpMax || ee[k] < -kFxExpMax);
        }
    } else {
        unsigned long long m0 = 0, m1 = 0;
        const unsigned long long *bm = a.bmax + (a.geos ? blockIdx.y : 0) * a.nblk * 2;
        for (int64_t b = b0 + threadIdx.x; b < b1; b += kFxTPB) { m0 = max(m0, bm[2 * b]); m1 = max(m1, bm[2 * b + 1]); }
        for (int off = 16; off > 0; off >>= 1) {
            m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, off));
            m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, off));
        }
        if (lane == 0) { s_max[0][warp] = m0; s_max[1][warp] = m1; }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            unsigned long long m = 0;
#pragma unroll
            for (int w = 0; w < kFxTPB / 32; ++w) m = max(m, s_max[k][w]);
            const int ex = (int)(m >> 52);
            ee[k] = m == 0 ? -kFxExpMax : ex - 1022;            // all zero: any scale
            bad |= m != 0 && (ee[k] > kFxExpMax || ee[k] < -kFxExpMax);
        }
    }
    double sum[3] = {0.0, 0.0, 0.0}, low[3] = {0.0, 0.0, 0.0};
    if (bad) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (grp == 0) fx_fallback<OP>(&a.k, cp, d0, d1, i, s_beg, s_end, sum);
    } else {
        const FxGeo &g = *gp;
        const FxScale sc = fx_scale<OP>(ee[0], ee[1], g.em, g.dq, g.ed);
        FxPoint<OP> y;
        if constexpr (!kEarly) {
            load_target();
            Yd = d0[i];
        }
        if constexpr (VU) {
            fx_split(fx_fix(Yd.x, sc.eu, 58), y.u.h[0], y.u.l[0]);
            fx_split(fx_fix(Yd.y, sc.eu, 58), y.u.h[1], y.u.l[1]);
            fx_split(fx_fix(Yd.z, sc.eu, 58), y.u.h[2], y.u.l[2]);
        }
        if constexpr (!T::vec && T::dl) y.p = fx_fix(Yd.x, sc.eu, 60);
        if constexpr (T::tr) {
            const d4 m = a.k.wn[i];
            fx_split(fx_fix(m.x, sc.em, 59), y.m.h[0], y.m.l[0]);
            fx_split(fx_fix(m.y, sc.em, 59), y.m.h[1], y.m.l[1]);
            fx_split(fx_fix(m.z, sc.em, 59), y.m.h[2], y.m.l[2]);
        }
        const uint32_t idx_max = (uint32_t)((a.noct - kOct0) * kFxSeg - 1);
        const int4 *tab4 = reinterpret_cast<const int4 *>(s_tab);
        auto tab = [&](int k, uint32_t idx, int w) {
            const int4 v = tab4[k * tstride + idx * kFxEntry + w];
            return FxI4{v.x, v.y, v.z, v.w};
        };
        for (int64_t tile = s_beg; tile < s_end; tile += kTile) {
            const int cnt = (int)(s_end - tile < kTile ? s_end - tile : kTile);   // a multiple of kChunk, or of kFxUnit
            // the tile's largest distance exponent L and a lower bound 2^r of its distances
            int dmax = 0, gap = 0;
            {
                int slo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, shi[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
                if constexpr (kEarly) {   // overlapping loads (a short tile's last box again)
                    // (tiles of small sets start and end at multiples of kFxUnit)
                    constexpr int kBoxes = kTile / kChunk + (GROUPS > 1 ? 1 : 0);
                    const int64_t b = tile / kChunk;
                    const int top = (int)((tile + cnt - 1) / kChunk - b);
#pragma unroll
                    for (int k = 0; k < kBoxes; ++k) grow(slo, shi, b + (k < top ? k : top));
                    if (GROUPS == 1 && top >= kBoxes) grow(slo, shi, b + top);
                } else {
                    const int64_t b = tile / kChunk;
                    for (int k = 0; k < cnt / kChunk; ++k) grow(slo, shi, b + k);
                    if ((tile | cnt) % kChunk) {   // (a loop over all boxes costs large sets 0.3%)
                        const int64_t e = (tile + cnt - 1) / kChunk;
                        grow(slo, shi, min(b + cnt / kChunk, e));
                        grow(slo, shi, e);
                    }
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    dmax = max(dmax, max(thi[c] - slo[c], shi[c] - tlo[c]) + 1);
                    gap = max(gap, max(tlo[c] - shi[c], slo[c] - thi[c]) - 1);
                }
            }
            // distances < dmax 2^(32 - ps) <= 2^L, >= gap 2^(32 - ps) >= 2^r
            const int L = max(0, 32 - g.ps + (32 - __clz(dmax - 1)));
            const int r = gap > 0 ? max(0, 31 - __clz(gap) + 32 - g.ps) : 0;
            FxTile tl = fx_tile<OP>(sc, L, r);
            tl.oct0 -= kOct0 * kFxSeg;
            const int ks = 61 - L - g.ps;
            auto grid = [&](int64_t v) { return ks >= 0 ? (int64_t)((uint64_t)v << ks) : v >> -ks; };
            if constexpr (GROUPS == 1) __syncthreads();   // (with groups the one before their sums)
            if (threadIdx.x < cnt) {
                const int64_t j = tile + threadIdx.x;
                const l4 p = a.X[j];
                const d4 e0 = d0[j];
                int4 h, l;
                fx_split(grid(p.x), h.x, l.x);
                fx_split(grid(p.y), h.y, l.y);
                fx_split(grid(p.z), h.z, l.z);
                if constexpr (!T::vec) {
                    const int64_t q = fx_fix(e0.x, sc.eu, 60);
                    h.w = (int)(q >> 32);
                    l.w = (int)q;
                }
                s_xh[threadIdx.x] = h;
                s_xl[threadIdx.x] = l;
                if constexpr (M) {
                    const d4 m = a.k.wn[j];
                    fx_split(fx_fix(m.x, sc.em, 59), h.x, l.x);
                    fx_split(fx_fix(m.y, sc.em, 59), h.y, l.y);
                    fx_split(fx_fix(m.z, sc.em, 59), h.z, l.z);
                    if constexpr (OP == OP_LSLDL) {
                        const int64_t q = fx_fix(e0.y, sc.ef, 60);
                        h.w = (int)(q >> 32);
                        l.w = (int)q;
                    }
                    s_mh[threadIdx.x] = h;
                    s_ml[threadIdx.x] = l;
                }
                if constexpr (VU) {
                    fx_split(fx_fix(e0.x, sc.eu, 58), h.x, l.x);
                    fx_split(fx_fix(e0.y, sc.eu, 58), h.y, l.y);
                    fx_split(fx_fix(e0.z, sc.eu, 58), h.z, l.z);
                    s_uh[threadIdx.x] = h;
                    s_ul[threadIdx.x] = l;
                }
                if constexpr (VF) {
                    const d4 e1 = T::dl ? d1[j] : e0;
                    fx_split(fx_fix(e1.x, sc.ef, 58), h.x, l.x);
                    fx_split(fx_fix(e1.y, sc.ef, 58), h.y, l.y);
                    fx_split(fx_fix(e1.z, sc.ef, 58), h.z, l.z);
                    s_fh[threadIdx.x] = h;
                    s_fl[threadIdx.x] = l;
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");   // the tables, before the first tile
            __syncthreads();
            fx_split(grid(Y.x), y.x.h[0], y.x.l[0]);
            fx_split(grid(Y.y), y.x.h[1], y.x.l[1]);
            fx_split(grid(Y.z), y.x.h[2], y.x.l[2]);
            FxSum<OP> acc{};
            // 4 pairs in flight fill the wide multiplier's latency (Stokes double layer
            // 3.10 clocks per pair and SM against 3.50 unrolled once; the transposed
            // Stokes layer has no registers left beyond 2).  3 resident CTAs of the Laplace
            // layers with 2 pairs in flight are slower: 2.29 ms against 2.20 at N = 17070.  The
            // fused Laplace layers keep their values in registers with 2: 3.52 ms, 3.54 with 4.
            constexpr int kUnroll = OP == OP_SDLT || OP == OP_LSLDL ? 2 : 4;
#pragma unroll kUnroll
            for (int j = grp; j < cnt; j += GROUPS) {
                FxPoint<OP> x;
                auto vec = [](FxV &v, const int4 &h, const int4 &l) {
                    v.h[0] = h.x; v.h[1] = h.y; v.h[2] = h.z;
                    v.l[0] = l.x; v.l[1] = l.y; v.l[2] = l.z;
                };
                auto word = [](const int4 &h, const int4 &l) { return ((int64_t)h.w << 32) | (uint32_t)l.w; };
                const int4 xh = s_xh[j], xl = s_xl[j];
                vec(x.x, xh, xl);
                if constexpr (T::dl && !T::vec) x.p = word(xh, xl);
                if constexpr (OP == OP_LSL) x.g = word(xh, xl);
                if constexpr (M) {
                    const int4 mh = s_mh[j], ml = s_ml[j];
                    vec(x.m, mh, ml);
                    if constexpr (OP == OP_LSLDL) x.g = word(mh, ml);
                }
                if constexpr (VU) vec(x.u, s_uh[j], s_ul[j]);
                if constexpr (VF) vec(x.f, s_fh[j], s_fl[j]);
                fx_pair<OP, FAR ? kFxFar : kFxFull>(y, x, tl, sc, idx_max, tab, acc);
            }
            const double f = __longlong_as_double((long long)(1023 + tl.ex) << 52) *
                             (T::fused || !T::dl ? g.f_sl : g.f_dl);
            auto value = [&](int64_t h, int64_t l) {   // of a component's two integers
                return T::vec ? ((double)h * 16777216.0 + (double)l) * f
                              : ((double)h + (double)l * 2.3283064365386963e-10) * f;
            };
            auto add = [&](int c, double v) {   // TwoSum: the tiles add no rounding of their own
                const double t = sum[c] + v, b = t - sum[c];
                low[c] += (sum[c] - (t - b)) + (v - b);
                sum[c] = t;
            };
            if constexpr (GROUPS == 1) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if constexpr (T::vec) add(c, value(acc.v[c].h, fx_low(acc.v[c])));
                    else add(c, value(acc.f.h, acc.f.l));
                }
            } else {
                // The groups' integers are added first, exactly: together they hold the
                // tile's 128 terms.  A thread then takes one component of one target.
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if constexpr (T::vec) {
                        s_acc[c][threadIdx.x] = acc.v[c].h;
                        s_acc[NC + c][threadIdx.x] = fx_low(acc.v[c]);
                    } else {
                        s_acc[0][threadIdx.x] = acc.f.h;
                        s_acc[1][threadIdx.x] = acc.f.l;
                    }
                }
                __syncthreads();
                if (grp < NC) {
                    int64_t h = 0, l = 0;
#pragma unroll
                    for (int q = 0; q < GROUPS; ++q) {
                        h += s_acc[grp][q * nt + threadIdx.x % nt];
                        l += s_acc[NC + grp][q * nt + threadIdx.x % nt];
                    }
                    add(0, value(h, l));
                }
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) sum[c] += low[c];
    }
    if constexpr (GROUPS > 1) {
        if (grp >= (bad ? 1 : NC)) return;
        if (!bad) {   // component grp of target i
            const int64_t q = grp;
            if (a.k.acc) atomicAdd(a.k.acc + q * a.k.n_pad + i, sum[0]);
            else a.k.part[part_base + q * pstride + i] = sum[0];
            return;
        }
    }
    if (a.k.acc) {
#pragma unroll
        for (int q = 0; q < NC; ++q) atomicAdd(a.k.acc + q * a.k.n_pad + i, sum[q]);
        return;
    }
#pragma unroll
    for (int q = 0; q < NC; ++q) a.k.part[part_base + (int64_t)q * pstride + i] = sum[q];
}

template <int OP, bool FAR> size_t fx_smem(int noct) {
    return (size_t)fx_ntab<OP, FAR>() * (noct - (FAR ? kFxFarOct : 0)) * kFxSeg * kFxEntry * sizeof(FxI4);
}

template <int OP, bool FAR = false, int GROUPS = 1>
cudaError_t launch_fx1(dim3 grid, const FxArgs &a, cudaStream_t s) {
    return launch_pdl(fx_kernel<OP, FAR, GROUPS>, grid, dim3(kFxTPB), fx_smem<OP, FAR>(a.noct), s, a);
}
template <int OP> cudaError_t launch_fx1(dim3 grid, const FxArgs &a, int groups, cudaStream_t s) {
    return groups == 1 ? launch_fx1<OP, false, 1>(grid, a, s) : launch_fx1<OP, false, kFxGroups>(grid, a, s);
}

cudaError_t launch_fx(int op, dim3 grid, const FxArgs &a, int groups, cudaStream_t s) {
    switch (op) {
        case OP_LSL: return launch_fx1<OP_LSL>(grid, a, groups, s);
        case OP_LDL: return launch_fx1<OP_LDL>(grid, a, groups, s);
        case OP_SSL: return launch_fx1<OP_SSL>(grid, a, groups, s);
        case OP_SDL: return launch_fx1<OP_SDL>(grid, a, groups, s);
        case OP_SSLDL: return launch_fx1<OP_SSLDL>(grid, a, groups, s);
        case OP_LSLDL: return launch_fx1<OP_LSLDL>(grid, a, groups, s);
        case OP_LDLT: return launch_fx1<OP_LDLT>(grid, a, groups, s);
        default: return launch_fx1<OP_SDLT>(grid, a, groups, s);
    }
}

template <int OP, bool FAR = false> cudaError_t fx_attr1() {
    const int bytes = (int)fx_smem<OP, FAR>(kFxMaxOct);
    cudaError_t e = cudaFuncSetAttribute(fx_kernel<OP, FAR, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if constexpr (!FAR)
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fx_kernel<OP, false, kFxGroups>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}

// Uploads the kernel tables of a context and lets the kernels use them.
int fx_init(ssd_ctx *ctx) {
    const size_t bytes = (size_t)kFxTabEntries * kFxEntry * sizeof(FxI4);
    const FxI4 *host = fx_table_host();
    if (!host) return set_error(ctx, SSD_ENOMEM, "kernel tables: no host memory");
    SSD_TRY(dev_alloc(ctx, bytes, &ctx->fx_tab));
    SSD_TRY(cuda_check(ctx, cudaMemcpy(ctx->fx_tab, host, bytes, cudaMemcpyHostToDevice), "kernel tables"));
    cudaError_t e = fx_attr1<OP_LSL>();
    if (e == cudaSuccess) e = fx_attr1<OP_LDL>();
    if (e == cudaSuccess) e = fx_attr1<OP_SSL>();
    if (e == cudaSuccess) e = fx_attr1<OP_SDL>();
    if (e == cudaSuccess) e = fx_attr1<OP_SSLDL>();
    if (e == cudaSuccess) e = fx_attr1<OP_LSLDL>();
    if (e == cudaSuccess) e = fx_attr1<OP_LDLT>();
    if (e == cudaSuccess) e = fx_attr1<OP_SDLT>();
    if (e == cudaSuccess) e = fx_attr1<OP_LSL, true>();
    if (e == cudaSuccess) e = fx_attr1<OP_LDL, true>();
    if (e == cudaSuccess) e = fx_attr1<OP_SSL, true>();
    if (e == cudaSuccess) e = fx_attr1<OP_SDL, true>();
    return cuda_check(ctx, e, "kernel attributes");
}
