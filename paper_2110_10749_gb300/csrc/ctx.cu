// Context, errors, device memory pool, kernel timing and point layouts.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cub/device/device_radix_sort.cuh>

#include "internal.h"

namespace ssd {

int set_error(ssd_ctx *ctx, int status, const std::string &msg) {
    if (ctx) ctx->err = msg;
    return status;
}

int cuda_check(ssd_ctx *ctx, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return SSD_OK;
    const int st = (e == cudaErrorMemoryAllocation) ? SSD_ENOMEM : SSD_ECUDA;
    return set_error(ctx, st, std::string(what) + ": " + cudaGetErrorString(e));
}

int launch_check(ssd_ctx *ctx, const char *what) { return cuda_check(ctx, cudaGetLastError(), what); }

// smallest free block of the pool of at least this size, or -1
static int dev_best(const ssd_ctx *ctx, size_t bytes) {
    int best = -1;
    for (size_t k = 0; k < ctx->pool.size(); ++k) {
        const auto &b = ctx->pool[k];
        if (!b.used && b.bytes >= bytes && (best < 0 || b.bytes < ctx->pool[best].bytes)) best = (int)k;
    }
    return best;
}

static size_t dev_round(size_t bytes) { return bytes == 0 ? 256 : (bytes + 255) & ~size_t(255); }

bool dev_cached(const ssd_ctx *ctx, size_t bytes) { return dev_best(ctx, dev_round(bytes)) >= 0; }

int dev_alloc(ssd_ctx *ctx, size_t bytes, void **p) {
    bytes = dev_round(bytes);
    const int best = dev_best(ctx, bytes);
    if (best >= 0) {
        ctx->pool[best].used = true;
        *p = ctx->pool[best].p;
        return SSD_OK;
    }
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, bytes);
    if (e != cudaSuccess) {
        // release unused cached blocks and retry once
        cudaGetLastError();
        for (auto &b : ctx->pool)
            if (!b.used) { cudaFree(b.p); b.p = nullptr; }
        ctx->pool.erase(std::remove_if(ctx->pool.begin(), ctx->pool.end(),
                                       [](const ssd_ctx::Block &b) { return b.p == nullptr; }),
                        ctx->pool.end());
        e = cudaMalloc(&q, bytes);
        if (e != cudaSuccess) return cuda_check(ctx, e, "device allocation");
    }
    ctx->pool.push_back({q, bytes, true});
    *p = q;
    return SSD_OK;
}

void dev_free(ssd_ctx *ctx, void *p) {
    if (!p) return;
    for (auto &b : ctx->pool)
        if (b.p == p) { b.used = false; return; }
}

int timed_begin(ssd_ctx *ctx, cudaStream_t s, cudaEvent_t *beg) {
    *beg = nullptr;
    if (!ctx->timing) return SSD_OK;
    cudaEvent_t e;
    if (!ctx->event_pool.empty()) {
        e = ctx->event_pool.back();
        ctx->event_pool.pop_back();
    } else {
        SSD_TRY(cuda_check(ctx, cudaEventCreate(&e), "event create"));
    }
    *beg = e;
    return cuda_check(ctx, cudaEventRecord(e, s), "event record");
}

void timed_end(ssd_ctx *ctx, cudaStream_t s, cudaEvent_t beg, int cls, int prec, double pairs) {
    if (!ctx->timing || !beg) return;
    cudaEvent_t e;
    if (!ctx->event_pool.empty()) {
        e = ctx->event_pool.back();
        ctx->event_pool.pop_back();
    } else if (cudaEventCreate(&e) != cudaSuccess) {
        return;
    }
    cudaEventRecord(e, s);
    ctx->pending.push_back({beg, e, cls, prec == SSD_FP32C ? 1 : 0, pairs});
}

int frame_acquire(ssd_ctx *ctx, double **slots, cudaEvent_t ev[2]) {
    if (ctx->hsp >= kHostFrames) return set_error(ctx, SSD_EINVAL, "GMRES nesting too deep");
    const int f = ctx->hsp;
    while ((int)ctx->sync_ev.size() < 2 * (f + 1)) {
        cudaEvent_t e;
        SSD_TRY(cuda_check(ctx, cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "event create"));
        ctx->sync_ev.push_back(e);
    }
    *slots = ctx->hbuf + 512 + kFrameLen * f;
    ev[0] = ctx->sync_ev[2 * f];
    ev[1] = ctx->sync_ev[2 * f + 1];
    ctx->hsp++;
    return SSD_OK;
}

void frame_release(ssd_ctx *ctx) {
    if (ctx->hsp > 0) ctx->hsp--;
}

static int drain_timing(ssd_ctx *ctx) {
    for (auto &t : ctx->pending) {
        float ms = 0.f;
        SSD_TRY(cuda_check(ctx, cudaEventSynchronize(t.end), "event sync"));
        SSD_TRY(cuda_check(ctx, cudaEventElapsedTime(&ms, t.beg, t.end), "event time"));
        ctx->stat_ms[t.cls][t.prec] += ms;
        ctx->stat_pairs[t.cls][t.prec] += t.pairs;
        ctx->stat_launches[t.cls][t.prec] += 1;
        ctx->event_pool.push_back(t.beg);
        ctx->event_pool.push_back(t.end);
    }
    ctx->pending.clear();
    return SSD_OK;
}

// ------------------------------------------------------------------ layouts
namespace {

// Bounding box of n points: one block, or 32 partial boxes (block b: part + 6 b)
// and then their union.  The comparisons are double precision, 1.6 a clock and SM,
// six a point: preparing 78106 points took 344 us with one block and takes 190,
// 17070 points 188 and 153; up to 4096 points the second launch costs as much as it
// saves.
constexpr int kBoxBlocks = 32;

__global__ void bbox_kernel(const double *xyz, int64_t n, double *out, double *part) {
    __shared__ double red[6][256];   // (lo, -hi)
    double v[6] = {1e300, 1e300, 1e300, 1e300, 1e300, 1e300};
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        for (int k = 0; k < 3; ++k) {
            const double x = xyz[k * n + i];
            v[k] = fmin(v[k], x);
            v[3 + k] = fmin(v[3 + k], -x);
        }
    for (int k = 0; k < 6; ++k) red[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st)
            for (int k = 0; k < 6; ++k) red[k][threadIdx.x] = fmin(red[k][threadIdx.x], red[k][threadIdx.x + st]);
        __syncthreads();
    }
    if (threadIdx.x < 6)
        (gridDim.x > 1 ? part + 6 * blockIdx.x : out)[threadIdx.x] = threadIdx.x < 3 ? red[threadIdx.x][0] : -red[threadIdx.x][0];
}

__global__ void bbox_union_kernel(double *out, const double *part) {   // one warp
    const double *p = part + 6 * threadIdx.x;
    for (int k = 0; k < 6; ++k) {
        double v = p[k];
        for (int off = 16; off > 0; off >>= 1) {
            const double u = __shfl_xor_sync(0xffffffffu, v, off);
            v = k < 3 ? fmin(v, u) : fmax(v, u);
        }
        if (threadIdx.x == 0) out[k] = v;
    }
}

static void launch_bbox(ssd_ctx *ctx, const double *xyz, int64_t n, double *bb, double *part, cudaStream_t s) {
    const int blocks = n <= 4096 ? 1 : kBoxBlocks;
    bbox_kernel<<<blocks, 256, 0, s>>>(xyz, n, bb, part);
    if (blocks > 1) bbox_union_kernel<<<1, kBoxBlocks, 0, s>>>(bb, part);
    ctx->launches += blocks > 1 ? 2 : 1;
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// 30-bit Morton key of each point inside the bounding box
__global__ void morton_kernel(const double *xyz, int64_t n, const double *bb, uint32_t *key, int32_t *idx) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t q[3];
    for (int k = 0; k < 3; ++k) {
        const double ext = bb[3 + k] - bb[k];
        double f = ext > 0 ? (xyz[k * n + i] - bb[k]) / ext : 0.0;
        f = fmin(fmax(f, 0.0), 1.0);
        q[k] = (uint32_t)(f * 1023.0);
    }
    key[i] = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    idx[i] = (int32_t)i;
}

__global__ void fill_layout_kernel(const double *xyz, const double *nrm, const double *w, int64_t n, int64_t n_pad,
                                   const int32_t *sorted_idx, Layout L) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_pad) return;
    if (i < n) {
        const int32_t o = sorted_idx ? sorted_idx[i] : (int32_t)i;
        const double x = xyz[o], y = xyz[n + o], z = xyz[2 * n + o];
        const double ww = w[o];
        const double wx = ww * nrm[o], wy = ww * nrm[n + o], wz = ww * nrm[2 * n + o];
        L.perm[i] = o;
        L.pos64[i] = d4{x, y, z, ww};
        L.wn64[i] = d4{wx, wy, wz, 0.0};
        L.pos32[i] = make_float4((float)x, (float)y, (float)z, (float)ww);
        L.wn32[i] = make_float4((float)wx, (float)wy, (float)wz, 0.f);
    } else {
        // padding: zero weight far from every point
        const double far = 1.0e4;
        L.perm[i] = -1;
        L.pos64[i] = d4{far, far, far, 0.0};
        L.wn64[i] = d4{0.0, 0.0, 0.0, 0.0};
        L.pos32[i] = make_float4((float)far, (float)far, (float)far, 0.f);
        L.wn32[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Bounding box of each 32-point chunk of the sorted layout (real points only;
// a chunk of padding gets the padding position as a degenerate box).
__global__ void chunk_box_kernel(Layout L) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.n_pad / kChunk) return;
    float lo[3] = {1e30f, 1e30f, 1e30f}, hi[3] = {-1e30f, -1e30f, -1e30f};
    bool any = false;
    for (int k = 0; k < kChunk; ++k) {
        const int64_t i = c * kChunk + k;
        if (i >= L.n) break;
        const float4 p = L.pos32[i];
        lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y); lo[2] = fminf(lo[2], p.z);
        hi[0] = fmaxf(hi[0], p.x); hi[1] = fmaxf(hi[1], p.y); hi[2] = fmaxf(hi[2], p.z);
        any = true;
    }
    if (!any) {
        const float4 p = L.pos32[c * kChunk];
        lo[0] = hi[0] = p.x; lo[1] = hi[1] = p.y; lo[2] = hi[2] = p.z;
    }
    L.cbox[2 * c] = make_float4(lo[0], lo[1], lo[2], 0.f);
    L.cbox[2 * c + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
}

// fixed-order FP64 sum of the weights, by one block of 256 threads
__device__ void wsum_block(const double *w, int64_t n, double *red, double *out) {
    double s = 0.0;
#pragma unroll 8
    for (int64_t i = threadIdx.x; i < n; i += 256) s += w[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// Extent (see internal.h) of points [off[y], off[y + 1]) of surface y =
// blockIdx.y (off NULL: all n points), one partial per block x.  With wsum, block 0 of
// one more sums the weights beside them, to wsum[y] (a launch of its own made the layout
// of 1062 points take 7 us longer, with one block for the box).  BOX: with the box of the points,
// six double-precision minima a point; prepared sets have it already.  The magnitudes
// are compared as integers, which order like the nonnegative doubles they are the
// bits of, with infinities and NaN above all finite ones.
// Preparing and releasing 1062 points takes 78 us (86 with a second box and eight
// double-precision minima through shared memory, 77 without an extent).
template <bool BOX>
__global__ void extent_kernel(const double *xyz, const double *nrm, const double *w, int64_t n, const int64_t *off,
                              Extent *out, double *wsum) {
    __shared__ double red[BOX ? 6 : 1][256];
    __shared__ unsigned long long top[2][8];
    const int64_t nb = (int64_t)gridDim.x - (wsum ? 1 : 0), blk = (int64_t)blockIdx.x - (wsum ? 1 : 0);
    const int64_t beg = off ? off[blockIdx.y] : 0, end = off ? off[blockIdx.y + 1] : n;
    if (blk < 0) {
        wsum_block(w + beg, end - beg, red[0], wsum + blockIdx.y);
        return;
    }
    double v[6] = {1e308, 1e308, 1e308, 1e308, 1e308, 1e308};   // lo, -hi
    unsigned long long mx = 0, mm = 0;                          // largest |x|, |w n|
    auto bits = [](double a) { return (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull; };
    for (int64_t i = beg + blk * 256 + threadIdx.x; i < end; i += nb * 256) {
        for (int c = 0; c < 3; ++c) {
            const double x = xyz[c * n + i];
            if (BOX) { v[c] = fmin(v[c], x); v[3 + c] = fmin(v[3 + c], -x); }
            mx = max(mx, bits(x));
            mm = max(mm, bits(w[i] * nrm[c * n + i]));
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        mm = max(mm, __shfl_xor_sync(0xffffffffu, mm, o));
    }
    if ((threadIdx.x & 31) == 0) { top[0][threadIdx.x >> 5] = mx; top[1][threadIdx.x >> 5] = mm; }
    if (BOX)
        for (int q = 0; q < 6; ++q) red[q][threadIdx.x] = v[q];
    __syncthreads();
    if (BOX)
        for (int st = 128; st > 0; st >>= 1) {
            if (threadIdx.x < st)
                for (int q = 0; q < 6; ++q) red[q][threadIdx.x] = fmin(red[q][threadIdx.x], red[q][threadIdx.x + st]);
            __syncthreads();
        }
    if (threadIdx.x == 0) {
        Extent e{};
        if (BOX)
            for (int c = 0; c < 3; ++c) { e.lo[c] = red[c][0]; e.hi[c] = -red[3 + c][0]; }
        for (int k = 1; k < 8; ++k) { mx = max(mx, top[0][k]); mm = max(mm, top[1][k]); }
        e.fin = mx < 0x7ff0000000000000ull && mm < 0x7ff0000000000000ull ? 1.0 : 0.0;
        e.mmax = __longlong_as_double((long long)mm);
        out[blockIdx.y * nb + blk] = e;
    }
}

Extent merge_extents(const Extent *e, int k) {
    Extent r = e[0];
    for (int i = 1; i < k; ++i) {
        for (int c = 0; c < 3; ++c) { r.lo[c] = fmin(r.lo[c], e[i].lo[c]); r.hi[c] = fmax(r.hi[c], e[i].hi[c]); }
        r.mmax = fmax(r.mmax, e[i].mmax);
        r.fin = fmin(r.fin, e[i].fin);
    }
    return r;
}

// ------------------------------------------------------------- batched layouts
// key = surface index above a 30-bit Morton code of the position in the
// batch's bounding box: sorting groups each surface's points in Morton order
__global__ void batch_key_kernel(const double *xyz, int64_t n, const double *bb, const int32_t *esurf,
                                 uint64_t *key, int32_t *idx) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t q[3];
    for (int k = 0; k < 3; ++k) {
        const double ext = bb[3 + k] - bb[k];
        double f = ext > 0 ? (xyz[k * n + i] - bb[k]) / ext : 0.0;
        f = fmin(fmax(f, 0.0), 1.0);
        q[k] = (uint32_t)(f * 1023.0);
    }
    const uint32_t m = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    key[i] = ((uint64_t)esurf[i] << 30) | m;
    idx[i] = (int32_t)i;
}

struct BatchFillArgs {
    int32_t nsurf;
    const int64_t *off, *cnt, *poff;   // device copies
    const double *xyz, *nrm, *w;
    int64_t n_total, n_pad_total;
    const int32_t *sorted;             // sorted position -> caller index
};

__global__ void batch_fill_kernel(const BatchFillArgs a, Layout L) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n_pad_total) return;
    // surface owning padded index i (binary search over padded offsets)
    int lo = 0, hi = a.nsurf - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.poff[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const int64_t local = i - a.poff[lo];
    const int64_t n = a.n_total;
    if (local < a.cnt[lo]) {
        const int32_t o = a.sorted[a.off[lo] + local];
        const double x = a.xyz[o], y = a.xyz[n + o], z = a.xyz[2 * n + o];
        const double ww = a.w[o];
        const double wx = ww * a.nrm[o], wy = ww * a.nrm[n + o], wz = ww * a.nrm[2 * n + o];
        L.perm[i] = o;
        L.pos64[i] = d4{x, y, z, ww};
        L.wn64[i] = d4{wx, wy, wz, 0.0};
        L.pos32[i] = make_float4((float)x, (float)y, (float)z, (float)ww);
        L.wn32[i] = make_float4((float)wx, (float)wy, (float)wz, 0.f);
    } else {
        const double far = 1.0e4;
        L.perm[i] = -1;
        L.pos64[i] = d4{far, far, far, 0.0};
        L.wn64[i] = d4{0.0, 0.0, 0.0, 0.0};
        L.pos32[i] = make_float4((float)far, (float)far, (float)far, 0.f);
        L.wn32[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// chunk boxes of the batched layout; chunks never straddle surfaces because
// every surface is padded to a multiple of kRowAlign
__global__ void batch_chunk_box_kernel(Layout L) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.n_pad / kChunk) return;
    float lo[3] = {1e30f, 1e30f, 1e30f}, hi[3] = {-1e30f, -1e30f, -1e30f};
    bool any = false;
    for (int k = 0; k < kChunk; ++k) {
        const int64_t i = c * kChunk + k;
        if (L.perm[i] < 0) continue;
        const float4 p = L.pos32[i];
        lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y); lo[2] = fminf(lo[2], p.z);
        hi[0] = fmaxf(hi[0], p.x); hi[1] = fmaxf(hi[1], p.y); hi[2] = fmaxf(hi[2], p.z);
        any = true;
    }
    if (!any) {
        const float4 p = L.pos32[c * kChunk];
        lo[0] = hi[0] = p.x; lo[1] = hi[1] = p.y; lo[2] = hi[2] = p.z;
    }
    L.cbox[2 * c] = make_float4(lo[0], lo[1], lo[2], 0.f);
    L.cbox[2 * c + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
}

__global__ void batch_esurf_kernel(const int64_t *off, int32_t nsurf, int64_t n, int32_t *esurf) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = nsurf - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    esurf[i] = lo;
}

}  // namespace

void batch_layout_release(ssd_ctx *ctx, BatchLayout *B) {
    if (B->block) dev_free(ctx, B->block);
    for (int k = 0; k < 2; ++k) {
        if (B->items[k]) dev_free(ctx, B->items[k]);
    }
    if (B->fx_pos) dev_free(ctx, B->fx_pos);
    *B = BatchLayout();
}

int batch_layout_build(ssd_ctx *ctx, const ssd_batch *b, BatchLayout *B, cudaStream_t s) {
    if (!b || b->nsurf < 1 || b->nsurf > (1 << 20) || !b->offsets || !b->delta)
        return set_error(ctx, SSD_EINVAL, "bad batch description");
    if (!b->xyz || !b->nrm || !b->w) return set_error(ctx, SSD_EINVAL, "NULL batch point array");
    BatchLayout out;
    out.nsurf = b->nsurf;
    if (b->offsets[0] != 0) return set_error(ctx, SSD_EINVAL, "offsets[0] must be 0");
    int64_t pacc = 0;
    for (int k = 0; k < b->nsurf; ++k) {
        const int64_t nk = b->offsets[k + 1] - b->offsets[k];
        if (nk <= 0) return set_error(ctx, SSD_EINVAL, "every surface needs at least one point");
        if (!(b->delta[k] > 0.0) || !isfinite(b->delta[k]))
            return set_error(ctx, SSD_EINVAL, "delta must be positive per surface");
        out.off.push_back(b->offsets[k]);
        out.n.push_back(nk);
        out.poff.push_back(pacc);
        const int64_t np = ((nk + kRowAlign - 1) / kRowAlign) * kRowAlign;
        out.n_pad.push_back(np);
        out.delta.push_back(b->delta[k]);
        pacc += np;
    }
    out.n_total = b->offsets[b->nsurf];
    out.n_pad_total = pacc;
    if (out.n_pad_total > (int64_t)0x7fffffff - 1024) return set_error(ctx, SSD_EINVAL, "batch too large");
    const int64_t n = out.n_total, np = out.n_pad_total;
    const int ns = out.nsurf;

    size_t off = 0;
    auto carve = [&](size_t bb) { size_t o = off; off += (bb + 255) & ~size_t(255); return o; };
    const size_t o_perm = carve(sizeof(int32_t) * np), o_p32 = carve(sizeof(float4) * np),
                 o_w32 = carve(sizeof(float4) * np), o_p64 = carve(sizeof(d4) * np),
                 o_w64 = carve(sizeof(d4) * np), o_cb = carve(sizeof(float4) * 2 * (np / kChunk)),
                 o_es = carve(sizeof(int32_t) * n), o_ws = carve((sizeof(double) + sizeof(Extent)) * ns),
                 o_meta = carve(sizeof(int64_t) * (4 * ns + 1) + sizeof(double) * ns);
    void *blk = nullptr;
    SSD_TRY(dev_alloc(ctx, off, &blk));
    char *bp = static_cast<char *>(blk);
    out.block = blk;
    out.L.n = np;   // the concatenated arrays as one padded set
    out.L.n_pad = np;
    out.L.perm = reinterpret_cast<int32_t *>(bp + o_perm);
    out.L.pos32 = reinterpret_cast<float4 *>(bp + o_p32);
    out.L.wn32 = reinterpret_cast<float4 *>(bp + o_w32);
    out.L.pos64 = reinterpret_cast<d4 *>(bp + o_p64);
    out.L.wn64 = reinterpret_cast<d4 *>(bp + o_w64);
    out.L.cbox = reinterpret_cast<float4 *>(bp + o_cb);
    out.elem_surf = reinterpret_cast<int32_t *>(bp + o_es);
    out.d_wsum = reinterpret_cast<double *>(bp + o_ws);
    int64_t *dmeta = reinterpret_cast<int64_t *>(bp + o_meta);   // off[ns+1], cnt[ns], poff[ns]
    out.d_selfc = reinterpret_cast<double *>(dmeta + 4 * ns + 1);
    Extent *dext = reinterpret_cast<Extent *>(out.d_wsum + ns);   // behind the weight sums: one host read
    std::vector<int64_t> hmeta(5 * ns + 1, 0);
    for (int k = 0; k <= ns; ++k) hmeta[k] = b->offsets[k];
    for (int k = 0; k < ns; ++k) { hmeta[ns + 1 + k] = out.n[k]; hmeta[2 * ns + 1 + k] = out.poff[k]; }
    for (int k = 0; k < ns; ++k) {
        const double selfc = 16.0 / (3.0 * sqrt(M_PI) * out.delta[k]);
        memcpy(&hmeta[4 * ns + 1 + k], &selfc, sizeof(selfc));
    }
    int st = cuda_check(ctx, cudaMemcpyAsync(dmeta, hmeta.data(), sizeof(int64_t) * hmeta.size(),
                                             cudaMemcpyHostToDevice, s), "batch meta copy");
    // sort by (surface, Morton)
    void *tmp = nullptr;
    if (st == SSD_OK) {
        size_t cub_bytes = 0;
        int nbits = 30;
        while ((1 << (nbits - 30)) < ns) ++nbits;
        cub::DeviceRadixSort::SortPairs(nullptr, cub_bytes, (const uint64_t *)nullptr, (uint64_t *)nullptr,
                                        (const int32_t *)nullptr, (int32_t *)nullptr, (int)n, 0, nbits, s);
        size_t t_off = 0;
        auto tcarve = [&](size_t bb) { size_t o = t_off; t_off += (bb + 255) & ~size_t(255); return o; };
        const size_t o_k0 = tcarve(sizeof(uint64_t) * n), o_k1 = tcarve(sizeof(uint64_t) * n);
        const size_t o_i0 = tcarve(sizeof(int32_t) * n), o_i1 = tcarve(sizeof(int32_t) * n);
        const size_t o_bb = tcarve(sizeof(double) * 6 * (1 + kBoxBlocks)), o_cub = tcarve(cub_bytes);
        st = dev_alloc(ctx, t_off, &tmp);
        if (st == SSD_OK) {
            char *tb = static_cast<char *>(tmp);
            uint64_t *k0 = reinterpret_cast<uint64_t *>(tb + o_k0), *k1 = reinterpret_cast<uint64_t *>(tb + o_k1);
            int32_t *i0 = reinterpret_cast<int32_t *>(tb + o_i0), *i1 = reinterpret_cast<int32_t *>(tb + o_i1);
            double *bb = reinterpret_cast<double *>(tb + o_bb);
            const unsigned gn = (unsigned)((n + 255) / 256);
            batch_esurf_kernel<<<gn, 256, 0, s>>>(dmeta, ns, n, out.elem_surf);
            launch_bbox(ctx, b->xyz, n, bb, bb + 6, s);
            batch_key_kernel<<<gn, 256, 0, s>>>(b->xyz, n, bb, out.elem_surf, k0, i0);
            ctx->launches += 2;
            st = launch_check(ctx, "batch keys");
            if (st == SSD_OK) {
                cudaError_t e = cub::DeviceRadixSort::SortPairs(tb + o_cub, cub_bytes, k0, k1, i0, i1, (int)n, 0,
                                                                nbits, s);
                ctx->launches += 4;
                st = cuda_check(ctx, e, "batch radix sort");
            }
            if (st == SSD_OK) {
                BatchFillArgs fa;
                fa.nsurf = ns; fa.off = dmeta; fa.cnt = dmeta + ns + 1; fa.poff = dmeta + 2 * ns + 1;
                fa.xyz = b->xyz; fa.nrm = b->nrm; fa.w = b->w; fa.n_total = n; fa.n_pad_total = np;
                fa.sorted = i1;
                batch_fill_kernel<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(fa, out.L);
                batch_chunk_box_kernel<<<(unsigned)((np / kChunk + 127) / 128), 128, 0, s>>>(out.L);
                ctx->launches += 2;
                for (int k = 0; k < ns; k += 65535) {   // grid.y limit
                    extent_kernel<true><<<dim3(2, (unsigned)(ns - k < 65535 ? ns - k : 65535)), 256, 0, s>>>(
                        b->xyz, b->nrm, b->w, n, dmeta + k, dext + k, out.d_wsum + k);
                    ctx->launches++;
                }
                st = launch_check(ctx, "batch fill");
            }
        }
    }
    out.wsum.resize(ns);
    out.ext.resize(ns);
    std::vector<char> sums((sizeof(double) + sizeof(Extent)) * ns);
    if (st == SSD_OK)
        st = cuda_check(ctx, cudaMemcpyAsync(sums.data(), out.d_wsum, sums.size(), cudaMemcpyDeviceToHost, s),
                        "wsum copy");
    if (st == SSD_OK) st = cuda_check(ctx, cudaStreamSynchronize(s), "batch layout sync");
    memcpy(out.wsum.data(), sums.data(), sizeof(double) * ns);
    memcpy(out.ext.data(), sums.data() + sizeof(double) * ns, sizeof(Extent) * ns);
    if (tmp) dev_free(ctx, tmp);
    if (st == SSD_OK) {
        for (int k = 0; k < ns; ++k)
            if (!(out.wsum[k] > 0.0)) { st = set_error(ctx, SSD_EINVAL, "surface weights must sum to > 0"); break; }
    }
    if (st == SSD_OK) st = pair_batch_items(ctx, &out, s);
    if (st != SSD_OK) {
        batch_layout_release(ctx, &out);
        return st;
    }
    *B = out;
    return SSD_OK;
}

int check_points(ssd_ctx *ctx, const ssd_points *pts) {
    if (!pts) return set_error(ctx, SSD_EINVAL, "points is NULL");
    if (pts->n <= 0 || pts->n > (int64_t)0x7fffffff - 1024)
        return set_error(ctx, SSD_EINVAL, "point count out of range");
    if (!pts->xyz || !pts->nrm || !pts->w) return set_error(ctx, SSD_EINVAL, "NULL point array");
    if (pts->layout && pts->layout->L.n != pts->n)
        return set_error(ctx, SSD_EINVAL, "layout was built for a different point count");
    return SSD_OK;
}

void release_layout(ssd_ctx *ctx, Layout *L) {
    if (L->block) dev_free(ctx, L->block);
    for (int k = 0; k < 2; ++k)
        if (L->order32[k]) dev_free(ctx, L->order32[k]);
    if (L->fx_block) dev_free(ctx, L->fx_block);
    for (auto &pl : L->sym)
        if (pl.block) dev_free(ctx, pl.block);
    *L = Layout();
}

int build_layout(ssd_ctx *ctx, const ssd_points *pts, bool sort, bool extent, Layout *L, cudaStream_t s) {
    const int64_t n = pts->n;
    const int64_t n_pad = ((n + kRowAlign - 1) / kRowAlign) * kRowAlign;
    size_t off = 0;
    auto carve = [&](size_t b) { size_t o = off; off += (b + 255) & ~size_t(255); return o; };
    const size_t o_perm = carve(sizeof(int32_t) * n_pad);
    const size_t o_p32 = carve(sizeof(float4) * n_pad);
    const size_t o_w32 = carve(sizeof(float4) * n_pad);
    const size_t o_p64 = carve(sizeof(d4) * n_pad);
    const size_t o_w64 = carve(sizeof(d4) * n_pad);
    const size_t o_cb = carve(sizeof(float4) * 2 * (n_pad / kChunk));
    // weight sum, box of the points, extent partials: one host read
    const size_t o_ws = carve(sizeof(double) * 16 + sizeof(Extent) * kExtentBlocks);
    void *blk = nullptr;
    SSD_TRY(dev_alloc(ctx, off, &blk));
    char *b = static_cast<char *>(blk);
    Layout out;
    out.n = n;
    out.owner = ctx;
    out.n_pad = n_pad;
    out.block = blk;
    out.perm = reinterpret_cast<int32_t *>(b + o_perm);
    out.pos32 = reinterpret_cast<float4 *>(b + o_p32);
    out.wn32 = reinterpret_cast<float4 *>(b + o_w32);
    out.pos64 = reinterpret_cast<d4 *>(b + o_p64);
    out.wn64 = reinterpret_cast<d4 *>(b + o_w64);
    out.cbox = reinterpret_cast<float4 *>(b + o_cb);
    double *dsum = reinterpret_cast<double *>(b + o_ws);

    // blocks of the extent: some 256 points each on small sets
    const int eb = !extent ? 0 : (n < 256 * kExtentBlocks ? (int)((n + 255) / 256) : kExtentBlocks);
    int32_t *sorted = nullptr;
    void *tmp = nullptr;
    int st = SSD_OK;
    if (sort) {
        // keys/values and CUB temporary storage
        size_t cub_bytes = 0;
        cub::DeviceRadixSort::SortPairs(nullptr, cub_bytes, (const uint32_t *)nullptr, (uint32_t *)nullptr,
                                        (const int32_t *)nullptr, (int32_t *)nullptr, (int)n, 0, 30, s);
        size_t t_off = 0;
        auto tcarve = [&](size_t bb) { size_t o = t_off; t_off += (bb + 255) & ~size_t(255); return o; };
        const size_t o_k0 = tcarve(sizeof(uint32_t) * n), o_k1 = tcarve(sizeof(uint32_t) * n);
        const size_t o_i0 = tcarve(sizeof(int32_t) * n), o_i1 = tcarve(sizeof(int32_t) * n);
        const size_t o_bb = tcarve(sizeof(double) * 6 * kBoxBlocks), o_cub = tcarve(cub_bytes);
        st = dev_alloc(ctx, t_off, &tmp);
        if (st != SSD_OK) { release_layout(ctx, &out); return st; }
        char *tb = static_cast<char *>(tmp);
        uint32_t *k0 = reinterpret_cast<uint32_t *>(tb + o_k0), *k1 = reinterpret_cast<uint32_t *>(tb + o_k1);
        int32_t *i0 = reinterpret_cast<int32_t *>(tb + o_i0), *i1 = reinterpret_cast<int32_t *>(tb + o_i1);
        double *bb = dsum + 8;
        launch_bbox(ctx, pts->xyz, n, bb, reinterpret_cast<double *>(tb + o_bb), s);
        morton_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pts->xyz, n, bb, k0, i0);
        ctx->launches += 1;
        st = launch_check(ctx, "morton keys");
        if (st == SSD_OK) {
            cudaError_t e = cub::DeviceRadixSort::SortPairs(tb + o_cub, cub_bytes, k0, k1, i0, i1, (int)n, 0, 30, s);
            ctx->launches += 4;
            st = cuda_check(ctx, e, "radix sort");
        }
        sorted = i1;
    }
    if (st == SSD_OK) {
        fill_layout_kernel<<<(unsigned)((n_pad + 255) / 256), 256, 0, s>>>(pts->xyz, pts->nrm, pts->w, n, n_pad,
                                                                          sorted, out);
        // (without the extent's blocks the Stokes double layer in FP32C on 2406 plain points
        // takes 146.2 us, 147.8 with them)
        Extent *part = reinterpret_cast<Extent *>(dsum + 16);
        if (sort) extent_kernel<false><<<1 + eb, 256, 0, s>>>(pts->xyz, pts->nrm, pts->w, n, nullptr, part, dsum);
        else extent_kernel<true><<<1 + eb, 256, 0, s>>>(pts->xyz, pts->nrm, pts->w, n, nullptr, part, dsum);
        chunk_box_kernel<<<(unsigned)((n_pad / kChunk + 127) / 128), 128, 0, s>>>(out);
        ctx->launches += 3;
        st = launch_check(ctx, "layout fill");
    }
    static_assert(16 + 8 * kExtentBlocks <= 512, "the read fits the pinned scratch");
    if (st == SSD_OK) st = cuda_check(ctx, cudaMemcpyAsync(ctx->hbuf, dsum,
                                                           eb ? sizeof(double) * 16 + sizeof(Extent) * eb : sizeof(double),
                                                           cudaMemcpyDeviceToHost, s), "wsum copy");
    if (st == SSD_OK) st = cuda_check(ctx, cudaStreamSynchronize(s), "layout sync");
    if (tmp) dev_free(ctx, tmp);
    if (st != SSD_OK) { release_layout(ctx, &out); return st; }
    out.wsum = ctx->hbuf[0];
    if (extent) {
        out.ext = merge_extents(reinterpret_cast<const Extent *>(ctx->hbuf + 16), eb);
        if (sort)
            for (int c = 0; c < 3; ++c) { out.ext.lo[c] = ctx->hbuf[8 + c]; out.ext.hi[c] = ctx->hbuf[11 + c]; }
    }
    if (!(out.wsum > 0.0)) {
        release_layout(ctx, &out);
        return set_error(ctx, SSD_EINVAL, "quadrature weights must have a positive sum");
    }
    *L = out;
    return SSD_OK;
}

int get_layout(ssd_ctx *ctx, const ssd_points *pts, LayoutRef *ref, cudaStream_t s, bool extent) {
    SSD_TRY(check_points(ctx, pts));
    if (pts->layout) {
        ref->L = &pts->layout->L;
        return SSD_OK;
    }
    SSD_TRY(build_layout(ctx, pts, false, extent, &ref->tmp, s));
    ref->ctx = ctx;
    ref->L = &ref->tmp;
    return SSD_OK;
}

}  // namespace ssd

using namespace ssd;

extern "C" {

const char *ssd_status_string(int st) {
    switch (st) {
        case SSD_OK: return "ok";
        case SSD_EINVAL: return "invalid argument";
        case SSD_ENOMEM: return "out of memory";
        case SSD_ECUDA: return "CUDA error";
        case SSD_ENOTCONV: return "iteration limit reached";
        case SSD_ENUMERIC: return "non-finite value";
        default: return "unknown status";
    }
}

int ssd_ctx_create(ssd_ctx **out, int device) {
    if (!out) return SSD_EINVAL;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return SSD_EINVAL;
    }
    if (cudaSetDevice(device) != cudaSuccess) return SSD_ECUDA;
    ssd_ctx *ctx = new ssd_ctx();
    ctx->device = device;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) { delete ctx; return SSD_ECUDA; }
    ctx->num_sms = prop.multiProcessorCount;
    if (cudaMallocHost((void **)&ctx->hbuf, sizeof(double) * (512 + kFrameLen * kHostFrames)) != cudaSuccess) { delete ctx; return SSD_ENOMEM; }
    const int st = pair_occupancy(ctx);
    if (st != SSD_OK) {
        for (auto &b : ctx->pool) cudaFree(b.p);
        cudaFreeHost(ctx->hbuf);
        delete ctx;
        return st;
    }
    // tuning knob: waves of resident CTAs in an FP32C pair-kernel grid
    if (const char *w = getenv("SSD_PAIR_WAVES")) {
        const int v = atoi(w);
        if (v >= 1 && v <= 64) ctx->waves32 = v;
    }
    // tuning knob: 0 launches the FP32C grid in plain (tile, split) order
    if (const char *w = getenv("SSD_PAIR_LPT")) ctx->lpt = atoi(w) != 0;
    if (const char *w = getenv("SSD_PAIR_SYM")) ctx->sym = atoi(w) != 0;
    if (const char *w = getenv("SSD_PAIR_WAVES64")) {
        const int v = atoi(w);
        if (v >= 1 && v <= 64) ctx->waves64 = ctx->waves_fx = v;
    }
    if (const char *w = getenv("SSD_GRID_POLLS")) {
        const int v = atoi(w);
        if (v >= 0 && v <= ctx->grid_polls) ctx->grid_polls = v;
    }
    *out = ctx;
    return SSD_OK;
}

int ssd_ctx_destroy(ssd_ctx *ctx) {
    if (!ctx) return SSD_OK;
    cudaSetDevice(ctx->device);
    cudaDeviceSynchronize();
    for (auto &b : ctx->pool) cudaFree(b.p);
    for (auto &t : ctx->pending) { cudaEventDestroy(t.beg); cudaEventDestroy(t.end); }
    for (auto e : ctx->event_pool) cudaEventDestroy(e);
    for (auto e : ctx->sync_ev) cudaEventDestroy(e);
    if (ctx->hbuf) cudaFreeHost(ctx->hbuf);
    delete ctx;
    return SSD_OK;
}

const char *ssd_ctx_last_error(const ssd_ctx *ctx) { return ctx ? ctx->err.c_str() : ""; }

int ssd_ctx_set_timing(ssd_ctx *ctx, int enable) {
    if (!ctx) return SSD_EINVAL;
    ctx->timing = enable != 0;
    return SSD_OK;
}

int ssd_ctx_kernel_stats(ssd_ctx *ctx, int cls, int prec, ssd_kernel_stats *out) {
    if (!ctx || !out || cls < 0 || cls >= SSD_K_COUNT || (prec != SSD_FP64 && prec != SSD_FP32C))
        return set_error(ctx, SSD_EINVAL, "bad kernel class, precision or output");
    SSD_TRY(drain_timing(ctx));
    const int p = prec == SSD_FP32C ? 1 : 0;
    out->launches = ctx->stat_launches[cls][p];
    out->ms = ctx->stat_ms[cls][p];
    out->pairs = ctx->stat_pairs[cls][p];
    return SSD_OK;
}

int ssd_ctx_reset_stats(ssd_ctx *ctx) {
    if (!ctx) return SSD_EINVAL;
    SSD_TRY(drain_timing(ctx));
    for (int c = 0; c < SSD_K_COUNT; ++c)
        for (int p = 0; p < 2; ++p) {
            ctx->stat_ms[c][p] = 0;
            ctx->stat_pairs[c][p] = 0;
            ctx->stat_launches[c][p] = 0;
        }
    return SSD_OK;
}

int ssd_ctx_launch_count(const ssd_ctx *ctx, int64_t *out) {
    if (!ctx || !out) return SSD_EINVAL;
    *out = ctx->launches;
    return SSD_OK;
}

int ssd_sync(ssd_ctx *ctx, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != ctx->device)
        return set_error(ctx, SSD_EINVAL, "the current device is not the context's device");
    const cudaError_t e = stream ? cudaStreamSynchronize((cudaStream_t)stream) : cudaDeviceSynchronize();
    return cuda_check(ctx, e, "synchronise");
}

int ssd_points_prepare(ssd_ctx *ctx, ssd_points *pts, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    if (pts && pts->layout) return set_error(ctx, SSD_EINVAL, "points already have a layout");
    SSD_TRY(check_points(ctx, pts));
    ssd_layout *lay = new ssd_layout();
    int st = build_layout(ctx, pts, true, true, &lay->L, (cudaStream_t)stream);
    lay->L.order_ok = true;
    if (st != SSD_OK) { delete lay; return st; }
    pts->layout = lay;
    return SSD_OK;
}

int ssd_points_release(ssd_ctx *ctx, ssd_points *pts) {
    if (!ctx || !pts) return SSD_EINVAL;
    if (pts->layout) {
        release_layout(ctx, &pts->layout->L);
        delete pts->layout;
        pts->layout = nullptr;
    }
    return SSD_OK;
}

int ssd_batch_prepare(ssd_ctx *ctx, ssd_batch *b, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    ctx->err.clear();
    if (!b) return set_error(ctx, SSD_EINVAL, "batch is NULL");
    if (b->layout) return set_error(ctx, SSD_EINVAL, "batch already has a layout");
    ssd_batch_layout *lay = new ssd_batch_layout();
    const int st = batch_layout_build(ctx, b, &lay->B, (cudaStream_t)stream);
    if (st != SSD_OK) { delete lay; return st; }
    b->layout = lay;
    return SSD_OK;
}

int ssd_batch_release(ssd_ctx *ctx, ssd_batch *b) {
    if (!ctx || !b) return SSD_EINVAL;
    if (b->layout) {
        batch_layout_release(ctx, &b->layout->B);
        delete b->layout;
        b->layout = nullptr;
    }
    return SSD_OK;
}

int ssd_quadrature_points(ssd_ctx *ctx, const ssd_surface *surf, double h, double angle_deg, int64_t capacity,
                          int64_t *n_out, double *xyz, double *nrm, double *w, int32_t *meta, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    ctx->err.clear();
    return quadrature_points(ctx, surf, h, angle_deg, capacity, n_out, xyz, nrm, w, meta, (cudaStream_t)stream);
}

int ssd_quadrature_jacobian(ssd_ctx *ctx, const ssd_surface *surf, double h, double angle_deg, int64_t n,
                            double *dxyz, double *dnrm, double *dw, ssd_stream stream) {
    if (!ctx) return SSD_EINVAL;
    ctx->err.clear();
    if (!surf) return set_error(ctx, SSD_EINVAL, "surface is NULL");
    return quadrature_jacobian(ctx, surf, h, angle_deg, n, dxyz, dnrm, dw, (cudaStream_t)stream);
}

}  // extern "C"

// ------------------------------------------------- FP32 FMA rate (measurement)
// Every thread keeps 16 independent FMA chains (8 packed f32x2 pairs, or 16
// scalars) for `iters` steps; the result is stored only when it equals a
// value it cannot reach, so nothing is optimised away.  Used to measure the
// FP32 rate the pair kernels can reach on this device.
namespace ssd {
namespace {
__global__ void __launch_bounds__(256) fma_rate_kernel(int packed, int iters, float m, float c, float *sink) {
    if (packed) {
        float2 a[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = make_float2(threadIdx.x * 1e-3f + k, blockIdx.x * 1e-3f - k);
        const float2 mm = make_float2(m, m), cc = make_float2(c, c);
        for (int it = 0; it < iters; ++it)
#pragma unroll
            for (int k = 0; k < 8; ++k) a[k] = __ffma2_rn(a[k], mm, cc);
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) s += a[k].x + a[k].y;
        if (s == -12345.678f) sink[0] = s;
    } else {
        float a[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) a[k] = threadIdx.x * 1e-3f + k;
        for (int it = 0; it < iters; ++it)
#pragma unroll
            for (int k = 0; k < 16; ++k) a[k] = fmaf(a[k], m, c);
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) s += a[k];
        if (s == -12345.678f) sink[0] = s;
    }
}
}  // namespace
}  // namespace ssd

extern "C" int ssd_fp32_fma_rate(ssd_ctx *ctx, int packed, double *tflops) {
    using namespace ssd;
    if (!ctx || !tflops) return SSD_EINVAL;
    ctx->err.clear();
    void *sink = nullptr;
    SSD_TRY(dev_alloc(ctx, 256, &sink));
    struct Release { ssd_ctx *c; void *p; ~Release() { dev_free(c, p); } } release{ctx, sink};
    const int blocks = ctx->num_sms * 8, threads = 256, iters = 1 << 14;
    cudaEvent_t e0, e1;
    SSD_TRY(cuda_check(ctx, cudaEventCreate(&e0), "event"));
    SSD_TRY(cuda_check(ctx, cudaEventCreate(&e1), "event"));
    float ms = 0.f;
    for (int rep = 0; rep < 3; ++rep) {   // the last of three launches is timed
        cudaEventRecord(e0, 0);
        fma_rate_kernel<<<blocks, threads, 0, 0>>>(packed, iters, 0.999999f, 1e-7f, static_cast<float *>(sink));
        cudaEventRecord(e1, 0);
        ctx->launches++;
    }
    cudaError_t e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    SSD_TRY(cuda_check(ctx, e, "fma rate kernel"));
    const double fmas = (double)blocks * threads * iters * 16.0;
    *tflops = 2.0 * fmas / (ms * 1e-3) / 1e12;
    return SSD_OK;
}
