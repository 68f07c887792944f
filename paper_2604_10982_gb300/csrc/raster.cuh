// Per-pixel surfel evaluation shared by the forward (a4) and adjoint (a5)
// compositing kernels, and the staging of tile-list batches.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace psi {
namespace raster {

constexpr int kTile = 16;    // tile width in pixels (16x16 or 16x8 tiles), one thread per pixel
constexpr int kRecF4 = 5;    // render record: 80 bytes = 5 float4
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kAlphaMax = 0.99f;
constexpr float kNegHalfLog2e = -0.72134752044448170f; // -log2(e)/2: exp(-d2/2) = 2^(d2 * k)

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Thread -> pixel inside the 16x16 tile: warp w owns the 8x4 block at
// ((w & 1) * 8, (w >> 1) * 4). Its four groups of eight consecutive lanes
// own the block's 4x2 quarters: group g = l >> 3 is the quarter at
// ((g >> 1) * 4, (g & 1) * 2), lane l pixel (l & 3, (l >> 2) & 1) of it.
__device__ __forceinline__ void pixel_of_thread(int tid, int &lx, int &ly)
{
    const int w = tid >> 5, l = tid & 31;
    lx = (w & 1) * 8 + ((l >> 4) & 1) * 4 + (l & 3);
    ly = (w >> 1) * 4 + ((l >> 2) & 3);
}

// Staged render record after the per-tile transform: q = A (lx, ly, 1) with
// (lx, ly) the pixel's integer offset inside the tile; (ox, oy) = centre of the
// tile's first pixel minus the projected centre (the low-pass term's offset).
struct Rec {
    float a00, a01, c0, a10, a11, c1, a20, a21, c2;
    float o, r2;
    float ox, oy;
};

__device__ __forceinline__ Rec load_rec(const float4 *r)
{
    const float4 x = r[0], y = r[1], z = r[2], w = r[3];
    Rec q;
    q.a00 = x.x; q.a01 = x.y; q.c0 = x.z; q.a10 = x.w;
    q.a11 = y.x; q.c1 = y.y; q.a20 = y.z; q.a21 = y.w;
    q.c2 = z.x; q.o = z.w; q.r2 = w.x;
    q.ox = z.y; q.oy = z.z;
    return q;
}

struct Eval {
    float q0, q1, q2, d2, G, alpha;
    bool clamped;
    bool filt;    // low-pass filter only: its screen-space term won
    float dx, dy; // low-pass filter only: pixel centre minus projected centre
};

// alpha = min(0.99, o exp(-(u^2+v^2)/2)) of one surfel at one pixel (Sec. 3.1),
// (u, v) = (q0/q2, q1/q2). Returns false if the pixel lies outside the support
// disc (u^2+v^2 > r^2) or alpha < 1/255. Every operation is an explicitly
// rounded intrinsic, so forward and adjoint kernels reproduce the same alpha
// (and hence the same Top-K sets) bit for bit.
// LP: the 2DGS object-space low-pass filter. The Gaussian's argument is
// min(u^2+v^2, 2 (dx^2+dy^2)), (dx, dy) the pixel centre minus the projected
// centre (a screen-space Gaussian of standard deviation sqrt(2)/2 pixel), and
// the support is that argument <= r^2. The surfel's own term wins ties.
template <bool LP = false>
__device__ __forceinline__ bool eval_alpha(const Rec &r, float lx, float ly, Eval &e)
{
    e.q0 = __fmaf_rn(r.a00, lx, __fmaf_rn(r.a01, ly, r.c0));
    e.q1 = __fmaf_rn(r.a10, lx, __fmaf_rn(r.a11, ly, r.c1));
    e.q2 = __fmaf_rn(r.a20, lx, __fmaf_rn(r.a21, ly, r.c2));
    const float nn = __fmaf_rn(e.q0, e.q0, __fmul_rn(e.q1, e.q1));
    const float dd = __fmul_rn(e.q2, e.q2);
    if constexpr (LP) {
        const bool ell = (nn <= __fmul_rn(r.r2, dd)) && (dd > 0.0f);
        const float rho3 = ell ? __fmul_rn(nn, rcp_approx(dd)) : __int_as_float(0x7f800000);
        e.dx = __fadd_rn(lx, r.ox);
        e.dy = __fadd_rn(ly, r.oy);
        const float rho2 = __fmul_rn(2.0f, __fmaf_rn(e.dx, e.dx, __fmul_rn(e.dy, e.dy)));
        e.filt = rho2 < rho3;
        if (e.filt ? !(rho2 <= r.r2) : !ell) return false;
        e.d2 = e.filt ? rho2 : rho3;
    } else {
        if (!(nn <= __fmul_rn(r.r2, dd)) || !(dd > 0.0f)) return false;
        e.d2 = __fmul_rn(nn, rcp_approx(dd));
    }
    e.G = ex2_approx(__fmul_rn(e.d2, kNegHalfLog2e));
    const float a = __fmul_rn(r.o, e.G);
    e.clamped = a > kAlphaMax;
    e.alpha = e.clamped ? kAlphaMax : a;
    return e.alpha >= kAlphaMin;
}

// ------------------------------------------------------------ Top-K
// The K largest weights of one pixel with their list positions (Sec. 5, Top-K
// Hard Selection), kept sorted by weight (descending; among equal weights the
// earlier list position first), so the worst kept weight is always the last
// slot. A new weight enters only if it is strictly larger than that worst one
// -- it comes later in the list than everything kept, so ties favour the
// earlier surfel -- by one compare-and-shift pass. With a runtime K below
// KMAX the first KMAX-K slots hold +inf and never move. The insertion runs
// under a warp vote, so lanes pay one compare per surfel unless some lane of
// the warp improves its set.
template <int KMAX>
struct TopK {
    float w[KMAX];
    int p[KMAX];

    __device__ __forceinline__ void init(int K)
    {
#pragma unroll
        for (int s = 0; s < KMAX; ++s) {
            w[s] = (s < KMAX - K) ? __int_as_float(0x7f800000) : -1.0f;
            p[s] = 0x7fffffff;
        }
    }

    __device__ __forceinline__ void offer(bool hit, float wt, int pos)
    {
        const bool better = hit && wt > w[KMAX - 1];
        if (__any_sync(0xffffffffu, better)) {
            if (better) {
                bool gt[KMAX];
#pragma unroll
                for (int s = 0; s < KMAX; ++s) gt[s] = wt > w[s];
#pragma unroll
                for (int s = KMAX - 1; s > 0; --s) {
                    w[s] = gt[s - 1] ? w[s - 1] : (gt[s] ? wt : w[s]);
                    p[s] = gt[s - 1] ? p[s - 1] : (gt[s] ? pos : p[s]);
                }
                w[0] = gt[0] ? wt : w[0];
                p[0] = gt[0] ? pos : p[0];
            }
        }
    }

    // order the slots by list position (empty slots last)
    __device__ __forceinline__ void sort_by_pos()
    {
#pragma unroll
        for (int round = 0; round < KMAX; ++round) {
#pragma unroll
            for (int s = (round & 1); s + 1 < KMAX; s += 2) {
                if (p[s] > p[s + 1]) {
                    const int tp = p[s];
                    p[s] = p[s + 1];
                    p[s + 1] = tp;
                    const float tw = w[s];
                    w[s] = w[s + 1];
                    w[s + 1] = tw;
                }
            }
        }
    }

    __device__ __forceinline__ bool valid(int s, int K) const { return s < K && p[s] != 0x7fffffff; }
};

// ------------------------------------------------------------ decoupled pipeline
// A tile's list is streamed through shared-memory stages of kPB records,
// each transformed for the tile on its way in. The first 32 records per pixel
// warp are brought in by the pixel warps themselves (pipe_prefill: one record
// per thread, so a tile starts after one round of loads instead of after a
// single warp has moved a whole batch); the rest by a dedicated producer warp
// (the last warp), one record per lane, the next chunk's records prefetched
// while one is transformed. Records go through registers: a bulk copy per
// 80-byte record is issued lane by lane, and its producer then read and
// rewrote the stage for the transform (first batch ready after 21k cycles on
// the 3M-surfel 1080p frame). The producer refills a stage after every pixel
// warp (8 for a 16x16 tile, 4 for 16x8) has released it. Pixel warps only wait for
// ready stages, so a warp with little work in a batch runs ahead instead of
// waiting at a CTA barrier; released[w] counts the batches pixel warp w is
// done with, so that a warp whose pixels are all saturated can leave the walk
// (kLeft) and finish its pixels while the others composite, instead of
// following the stream to its end (the producer stops when all have). Every wait is bounded; a waiting warp is
// suspended in hardware.
constexpr int kPB = 128;          // records per stage (four 32-bit hit words per warp)
// pixel warps of a 16 x TH tile (8x4-pixel blocks, two per block row) and the
// CTA size with the producer warp
__host__ __device__ constexpr int pixel_warps(int TH) { return TH / 2; }
__host__ __device__ constexpr int pipe_threads(int TH) { return 32 * (pixel_warps(TH) + 1); }
constexpr int kPixelWarps = pixel_warps(16);
constexpr int kPipeThreads = pipe_threads(16);

constexpr int kLeft = 0x7fffffff;  // released[w] of a warp that left the walk
constexpr uint32_t kSuspendNs = 20000; // longest hardware suspension per poll of a wait

// NS stages: 4, or 3 where a fourth costs a resident CTA or the L1 (with two of them
// prefilled, each further one lets a fast warp run ahead of a slow one: 4
// against 3 is 0.90 against 1.00 ms for the adjoint of the depth/normal maps)
template <int NS>
struct PipeT {
    static constexpr int kPS = NS;
    float4 rec[kPS][kPB][kRecF4];
    uint32_t val[kPS][kPB];
    uint64_t ready[kPS]; // one arrival per pixel warp (the producer arrives for all of them)
    int released[kPixelWarps]; // batches each pixel warp is done with (unused ones: kLeft)
    int abort;
    unsigned long long limit; // the context's wait limit (ns)
};

using Pipe = PipeT<4>;

// Index lists of a warp's groups (build_hits), and whether `occ` CTAs of a
// compositing kernel -- stages, lists, `dyn` bytes of dynamic shared memory,
// 16 bytes of its own and the 1 KB the system takes -- fit an SM's shared memory. The
// launches assert it for the CTAs per SM that their build is for: one CTA fewer
// than that runs with the registers of more, and a persistent grid would hold
// CTAs that start only when the others have finished.
constexpr int kGroups = 4;
using HitLists = uint8_t[kGroups][kPB];
template <class PP>
constexpr bool smem_fits(int occ, int TH, size_t dyn)
{
    return occ * (sizeof(PP) + sizeof(HitLists) * pixel_warps(TH) + 16 + dyn + 1024) <= 228 * 1024;
}

__device__ __forceinline__ int vload(const int &x) { return *reinterpret_cast<const volatile int *>(&x); }

// thread 0; the caller synchronises the CTA afterwards. warps = the number of
// pixel warps (each releases every stage once per batch), limit = wait_limit()
template <class PP>
__device__ __forceinline__ void pipe_init(PP &P, int warps, unsigned long long limit)
{
    P.limit = limit;
    for (int s = 0; s < PP::kPS; ++s) {
        mbar_init(&P.ready[s], warps);
    }
    for (int w = 0; w < kPixelWarps; ++w) P.released[w] = w < warps ? 0 : kLeft;
    P.abort = 0;
    fence_mbar_init();
}

// thread 0, between two tiles of a persistent CTA (after a CTA barrier):
// retire the barriers so that pipe_init may initialise them again
template <class PP>
__device__ __forceinline__ void pipe_inval(PP &P)
{
    for (int s = 0; s < PP::kPS; ++s) {
        asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(&P.ready[s])) : "memory");
    }
}

// Grid of a persistent compositing launch: occ CTAs per SM, at most one per tile.
inline unsigned persistent_grid(uint32_t n_tiles, int occ)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return static_cast<unsigned>(std::min<int64_t>(n_tiles, static_cast<int64_t>(occ) * sms));
}

// Batch b of a walk over n list entries (forward: from the front; reverse:
// from the back); returns the first list position and sets the count.
__device__ __forceinline__ int batch_range(int b, int n, bool reverse, int &cnt)
{
    const int nb = (n + kPB - 1) / kPB;
    const int bi = reverse ? nb - 1 - b : b;
    cnt = min(kPB, n - bi * kPB);
    return bi * kPB;
}

// Per-tile transform of one staged record: fold the tile origin into the
// third column so that q = A (lx, ly, 1) with small, exact pixel offsets, and
// replace the covered-pixel rectangle by the mask of the 8x4 warp blocks it
// meets (bit w = warp w), so a warp skips a record with one shared load.
//
// Without the low-pass filter the record also gets the chord form of its
// support, from which build_hits takes each pixel row's covered columns: on
// row y, u^2 + v^2 <= r^2 asks |c(y) + a x| <= r |q2| with c(y) = (q0, q1) at
// x = 0 and a = d(q0, q1)/dx, that is (x - X)^2 <= M - S^2 with
//     X(y) = -(a . c) / |a|^2,  S(y) = (a x c) / |a|^2,  both linear in y,
//     M = r^2 max|q2|^2 / |a|^2 (the maximum over the tile's pixels).
// The cross product keeps thin ellipses exact where the conic's determinant
// would cancel. r is cut to the radius where o exp(-r^2/2) reaches 1/255. The
// form only has to hold everything eval_alpha accepts, so M carries a margin
// far above both sides' rounding: the half-width grows by 2^-8 of itself, 0.02
// pixel and 2^-18 of the distance |c| / |a| (eight times the rounding of the
// folded coefficients); a record it cannot be formed for covers every pixel.
// Layout afterwards: r[4] = (X0, X1, mask, S0), r[2].y = S1, r[2].z = M (with
// the filter r[4] = (rectangle, rectangle, mask, 0), r[2].yz = offset from p0).
template <bool LP>
__device__ __forceinline__ void transform_record(float4 (&r)[kRecF4], int tile_x0, int tile_y0)
{
    float4 q = r[4];
    const uint32_t bx = __float_as_uint(q.x), by = __float_as_uint(q.y);
    const int x0 = static_cast<int>(bx & 0xFFFFu) - tile_x0, x1 = static_cast<int>(bx >> 16) - tile_x0;
    const int y0 = static_cast<int>(by & 0xFFFFu) - tile_y0, y1 = static_cast<int>(by >> 16) - tile_y0;
    uint32_t mask = 0;
    if (y0 <= 15 && y1 >= 0) {
        // block rows first .. last of the columns met: two bits per block row
        const int lo = 2 * (max(y0, 0) >> 2), hi = 2 * (min(y1, 15) >> 2) + 2;
        const uint32_t cols = ((x0 <= 7 && x1 >= 0) ? 0x55u : 0u) | ((x0 <= 15 && x1 >= 8) ? 0xAAu : 0u);
        mask = cols & ((1u << hi) - (1u << lo));
    }
    float4 x = r[0], y = r[1], z = r[2];
    const float ox = (static_cast<float>(tile_x0) + 0.5f) - z.y;
    const float oy = (static_cast<float>(tile_y0) + 0.5f) - z.z;
    x.z = __fmaf_rn(x.x, ox, __fmaf_rn(x.y, oy, x.z));
    y.y = __fmaf_rn(x.w, ox, __fmaf_rn(y.x, oy, y.y));
    z.x = __fmaf_rn(y.z, ox, __fmaf_rn(y.w, oy, z.x));
    q.z = __uint_as_float(mask);
    if constexpr (LP) {
        z.y = ox; // the projected centre becomes the tile-relative offset (low-pass term)
        z.z = oy;
        q.w = 0.0f;
    } else {
        const float r2 = fminf(r[3].x, 2.0f * __logf(255.0f * z.w) + 0.01f);
        const float inv = 1.0f / (x.x * x.x + x.w * x.w);
        const float X0 = -(x.x * x.z + x.w * y.y) * inv, X1 = -(x.x * x.y + x.w * y.x) * inv;
        const float S0 = (x.x * y.y - x.w * x.z) * inv, S1 = (x.x * y.x - x.w * x.y) * inv;
        const float q2 = fabsf(z.x + 7.5f * (y.z + y.w)) + 7.5f * (fabsf(y.z) + fabsf(y.w));
        const float dist = fabsf(X0) + fabsf(S0) + 15.0f * (fabsf(X1) + fabsf(S1));
        const float h = sqrt_approx(r2 * inv) * q2 * (1.0f + 0x1p-8f) + 0.02f + dist * 0x1p-18f;
        const bool ok = h < 1e8f && dist < 1e8f;
        q.x = ok ? X0 : 0.0f;
        q.y = ok ? X1 : 0.0f;
        q.w = ok ? S0 : 0.0f;
        z.y = ok ? S1 : 0.0f;
        z.z = ok ? h * h : 1e30f;
    }
    r[4] = q;
    r[0] = x;
    r[1] = y;
    r[2] = z;
}

__device__ __forceinline__ void load_record(float4 (&r)[kRecF4], const float4 *__restrict__ records, uint32_t i)
{
    const float4 *src = records + kRecF4 * static_cast<size_t>(i);
#pragma unroll
    for (int k = 0; k < kRecF4; ++k) r[k] = __ldg(src + k);
}

__device__ __forceinline__ void prefetch_record(const float4 *__restrict__ records, uint32_t i)
{
    const float4 *p = records + kRecF4 * static_cast<size_t>(i);
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p + kRecF4 - 1));
}

// What else is staged with a record: nothing, or (StageFeat, further down) its
// feature channels.
struct NoExtra {
    __device__ __forceinline__ void operator()(int, int, uint32_t) const {}
};

// One record, transformed, into its place of a stage.
template <bool LP, class PP, class Extra>
__device__ __forceinline__ void stage_record(PP &P, int s, int j, float4 (&r)[kRecF4], uint32_t i, int tile_x0,
                                             int tile_y0, const Extra &extra)
{
    transform_record<LP>(r, tile_x0, tile_y0);
#pragma unroll
    for (int k = 0; k < kRecF4; ++k) P.rec[s][j][k] = r[k];
    P.val[s][j] = i;
    extra(s, j, i);
}

// Record index of list entry `pos` of the tile; debug builds check that it is
// a record of the tile's view.
__device__ __forceinline__ uint32_t list_entry(const uint32_t *__restrict__ vals, int64_t pos, uint32_t rec_lo,
                                               uint32_t rec_hi, DevStatus *st)
{
    uint32_t r = __ldg(vals + pos);
    (void)rec_lo;
    (void)rec_hi;
    if (!PSI_CHECK(r >= rec_lo && r < rec_hi, kChkRecord, st)) r = rec_lo;
    return r;
}

// The batches the PW pixel warps stage themselves (32 records per warp).
template <int PW>
__device__ __forceinline__ constexpr int prefill_batches() { return PW * 32 / kPB; }

// Pixel warp w of PW: its 32 records of the first batches (the same walk as
// pipe_produce, after pipe_init is visible to the CTA).
template <bool LP, int PW, class PP, class Extra = NoExtra>
__device__ __forceinline__ void pipe_prefill(PP &P, int w, const uint32_t *__restrict__ vals, int64_t list0, int n,
                                             bool reverse, const float4 *__restrict__ records, int tile_x0,
                                             int tile_y0, DevStatus *st, uint32_t rec_lo, uint32_t rec_hi,
                                             const Extra &extra = Extra())
{
    if constexpr (prefill_batches<PW>() == 0) return; // fewer threads than a batch: the producer stages all
    constexpr int kShare = PW / (kPB / 32); // arrivals per warp: kPB / 32 warps stage one batch
    const int b = w * 32 / kPB, lane = threadIdx.x & 31;
    const int j = (w * 32) % kPB + lane;
    if (b >= (n + kPB - 1) / kPB) return;
    int cnt;
    const int lo = batch_range(b, n, reverse, cnt);
    if (j < cnt) {
        const uint32_t i = list_entry(vals, list0 + lo + j, rec_lo, rec_hi, st);
        float4 r[kRecF4];
        load_record(r, records, i);
        stage_record<LP>(P, b, j, r, i, tile_x0, tile_y0, extra);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive_n(&P.ready[b], kShare);
}

// Batches that every pixel warp in the walk is done with: kLeft when all have
// left it, -1 after an abort. One answer for the whole (producer) warp, as the
// warp-wide operations of its loop need; lane w has acquired warp w's release.
template <class PP>
__device__ __forceinline__ int pipe_progress(const PP &P)
{
    const int lane = threadIdx.x & 31;
    int done = kLeft;
    if (lane < kPixelWarps)
        done = ld_acquire_cta_shared(&P.released[lane]);
    else if (lane == kPixelWarps && vload(P.abort))
        done = -1;
    return __reduce_min_sync(0xffffffffu, done);
}

// Producer warp: waits until the stage of batch b is free (every pixel warp is
// done with the batch before it there). False if there is nothing more to
// stage for: every warp has left, or an abort -- its own, when the wait runs
// out. One exit, for all lanes together.
template <class PP>
__device__ __forceinline__ bool pipe_wait_free(PP &P, int b, DevStatus *st, int site)
{
    unsigned long long t0 = 0;
    int done = pipe_progress(P);
    while (done >= 0 && done <= b - PP::kPS) {
        if (wait_expired(t0, P.limit)) {
            if (st) {
                atomicCAS(&st->wait_site, 0, site);
                raise_status(st, PSI_ERR_TIMEOUT);
            }
            atomicExch(&P.abort, 1);
        }
        __nanosleep(64);
        done = pipe_progress(P);
    }
    __syncwarp(); // what one lane acquired orders every lane's refill of the stage
    return done >= 0 && done != kLeft;
}

// Producer warp: stages the batches after the prefilled ones of the list
// (entries [list0, list0+n)), forward or reverse, until all are staged, every
// pixel warp has left the walk, or a wait runs out (status raised, abort set).
template <bool LP, int PW, class PP, class Extra = NoExtra>
__device__ __forceinline__ void pipe_produce(PP &P, const uint32_t *__restrict__ vals, int64_t list0, int n,
                                             bool reverse, const float4 *__restrict__ records, int tile_x0,
                                             int tile_y0, DevStatus *st, int site, uint32_t rec_lo, uint32_t rec_hi,
                                             const Extra &extra = Extra())
{
    constexpr int kChunks = kPB / 32;
    const int lane = threadIdx.x & 31;
    const int nb = (n + kPB - 1) / kPB;
    // chunk c: entries [32 (c % kChunks), + 32) of batch c / kChunks
    auto entry = [&](int c, uint32_t &i) {
        if (c >= nb * kChunks) return false;
        int cnt;
        const int lo = batch_range(c / kChunks, n, reverse, cnt);
        const int j = (c % kChunks) * 32 + lane;
        if (j >= cnt) return false;
        i = list_entry(vals, list0 + lo + j, rec_lo, rec_hi, st);
        return true;
    };
    int c = prefill_batches<PW>() * kChunks;
    uint32_t i0 = 0, i1 = 0; // this chunk's and the next chunk's record index
    bool v0 = entry(c, i0), v1 = entry(c + 1, i1);
#pragma unroll 1
    for (; c < nb * kChunks; ++c) {
        const int b = c / kChunks, s = b % PP::kPS;
        if (c % kChunks == 0 && !pipe_wait_free(P, b, st, site)) return;
        const int j = (c % kChunks) * 32 + lane;
        if (v1) prefetch_record(records, i1);
        if (v0) {
            float4 r[kRecF4];
            load_record(r, records, i0);
            stage_record<LP>(P, s, j, r, i0, tile_x0, tile_y0, extra);
        }
        v0 = v1;
        i0 = i1;
        v1 = entry(c + 2, i1);
        if (c % kChunks == kChunks - 1) {
            __syncwarp();
            if (lane == 0) mbar_arrive_n(&P.ready[s], PW);
        }
    }
}

// Pixel warp (all 32 lanes): wait until batch b is ready. Returns false
// after an abort. The answer is the same in every lane of the warp: once one
// lane has seen the batch ready it stays ready (the stage cannot be refilled
// before this warp releases it), so the others wait for it too.
template <class PP>
__device__ __forceinline__ bool pipe_wait_ready(PP &P, int b, DevStatus *st, int site)
{
    const int s = b % PP::kPS;
    const uint32_t par = (b / PP::kPS) & 1;
    bool ready = mbar_test_wait(&P.ready[s], par);
    if (!ready) {
        const unsigned long long limit = P.limit;
        const unsigned long long t0 = global_ns();
        while (true) {
            if (limit >= kTimerTickNs && mbar_try_wait_for(&P.ready[s], par, limit < kSuspendNs ? static_cast<uint32_t>(limit) : kSuspendNs)) {
                ready = true;
                break;
            }
            if (vload(P.abort)) break;
            // a limit below the timer's resolution has run out at the first poll that fails
            if (global_ns() - t0 > limit || limit < kTimerTickNs) {
                if (st) {
                    atomicCAS(&st->wait_site, 0, site);
                    raise_status(st, PSI_ERR_TIMEOUT);
                }
                atomicExch(&P.abort, 1);
                break;
            }
        }
    }
    if (!__any_sync(0xffffffffu, ready)) return false;
    if (!ready) mbar_wait(&P.ready[s], par, st, site); // complete already: returns at once
    return true;
}

// Pixel warp w: done with batch b and all before it.
template <class PP>
__device__ __forceinline__ void pipe_release(PP &P, int w, int b)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) st_release_cta_shared(&P.released[w], b + 1);
}

// Pixel warp w: no pixel of it composites any further.
template <class PP>
__device__ __forceinline__ void pipe_leave(PP &P, int w)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) st_release_cta_shared(&P.released[w], kLeft);
}

// The records of one staged batch that can reach a pixel of each group of
// lanes, as index lists in shared memory (ascending). A group walks its own
// list: the lanes of a warp then work on up to four records at a time, and the
// warp's trip count is the longest of its lists rather than the number of
// records that meet its 8x4 block. On a 1080p street of 3M surfels (median
// splat 8 pixels wide) that is 8.3M against 16.4M trips before the first
// pixel saturates.
//
// Builds the lists of pixel warp vw (its block's place in the 16x16 tile) for
// the first `cnt` records of stage s, taking record j into group g's list
// only if j < lim[g]; n[g] = length. NG = 4: one list per group; NG = 1: one
// list (0) for the whole warp. One record per lane; every lane gets n.
template <bool LP, int NG, class PP>
__device__ __forceinline__ void build_hits(const PP &P, int s, int cnt, int vw, int tile_x0, int tile_y0,
                                           const int lim[NG], HitLists &list, int n[NG])
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const int bx = (vw & 1) * 8, by = (vw >> 1) * 4;
#pragma unroll
    for (int g = 0; g < NG; ++g) n[g] = 0;
    __syncwarp(); // every lane is done with the previous batch's lists
#pragma unroll 1
    for (int q = 0; q < cnt; q += 32) {
        const int j = q + lane;
        bool hit[kGroups] = {false, false, false, false};
        if (j < cnt) {
            const float4 t = P.rec[s][j][4];
            if ((__float_as_uint(t.z) >> vw) & 1u) {
                if constexpr (LP) {
                    const uint32_t rx = __float_as_uint(t.x), ry = __float_as_uint(t.y);
                    const int x0 = static_cast<int>(rx & 0xFFFFu) - tile_x0 - bx, x1 = static_cast<int>(rx >> 16) - tile_x0 - bx;
                    const int y0 = static_cast<int>(ry & 0xFFFFu) - tile_y0 - by, y1 = static_cast<int>(ry >> 16) - tile_y0 - by;
                    hit[0] = x0 <= 3 && x1 >= 0 && y0 <= 1 && y1 >= 0;
                    hit[1] = x0 <= 3 && x1 >= 0 && y0 <= 3 && y1 >= 2;
                    hit[2] = x0 <= 7 && x1 >= 4 && y0 <= 1 && y1 >= 0;
                    hit[3] = x0 <= 7 && x1 >= 4 && y0 <= 3 && y1 >= 2;
                } else {
                    const float4 u = P.rec[s][j][2];
                    const float fx = static_cast<float>(bx);
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float y = static_cast<float>(by + r);
                        const float S = fmaf(u.y, y, t.w), X = fmaf(t.y, y, t.x) - fx;
                        const float h = sqrt_approx(fmaf(-S, S, u.z)); // NaN where the row is missed
                        const float lo = X - h, hi = X + h;
                        hit[r >> 1] |= hi >= 0.0f && lo <= 3.0f;
                        hit[2 + (r >> 1)] |= hi >= 4.0f && lo <= 7.0f;
                    }
                }
            }
        }
        if constexpr (NG == 1) {
            const bool h = (hit[0] || hit[1] || hit[2] || hit[3]) && j < lim[0];
            const uint32_t w = __ballot_sync(0xffffffffu, h);
            if (h) list[0][n[0] + __popc(w & lt)] = static_cast<uint8_t>(j);
            n[0] += __popc(w);
        } else {
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const bool h = hit[g] && j < lim[g];
                const uint32_t w = __ballot_sync(0xffffffffu, h);
                if (h) list[g][n[g] + __popc(w & lt)] = static_cast<uint8_t>(j);
                n[g] += __popc(w);
            }
        }
    }
    __syncwarp();
}

// ------------------------------------------------------------ features
// 32 bytes of read-only global memory (address 32-byte aligned).
__device__ __forceinline__ void ldg32(const void *p, uint32_t w[8])
{
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
        : "l"(p));
}

// Whether feature rows can be read 32 bytes at a time: the table starts on a
// 32-byte boundary and every row is a whole number of 32-byte units.
inline bool feat_rows_wide(const void *base, int D, int dtype)
{
    const int esize = dtype == PSI_F32 ? 4 : (dtype == PSI_BF16 ? 2 : 1);
    return (reinterpret_cast<uintptr_t>(base) % 32 == 0) && ((D * esize) % 32 == 0);
}

// CH (16 or 32) channels [c0, c0+CH) of feature row i as float32, before the
// per-channel scale. Rows are read with 16-byte vector loads, or 32-byte ones
// when `wide` (see feat_rows_wide; c0 is a multiple of 16): a lane then
// touches one whole 32-byte sector per load when the rows of a warp differ.
template <int DT, int CH>
__device__ __forceinline__ void load_feat(const void *__restrict__ base, int64_t i, int D, int c0, float *f,
                                          bool wide = false)
{
    if (wide && DT != PSI_FP8_E4M3) {
        const unsigned char *row = static_cast<const unsigned char *>(base) + (i * D + c0) * (DT == PSI_F32 ? 4 : 2);
        if constexpr (DT == PSI_F32) {
#pragma unroll
            for (int k = 0; k < CH / 8; ++k) {
                uint32_t w[8];
                ldg32(row + 32 * k, w);
#pragma unroll
                for (int h = 0; h < 8; ++h) f[8 * k + h] = __uint_as_float(w[h]);
            }
        } else {
#pragma unroll
            for (int k = 0; k < CH / 16; ++k) {
                uint32_t w[8];
                ldg32(row + 32 * k, w);
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    f[16 * k + 2 * h] = __uint_as_float(w[h] << 16);
                    f[16 * k + 2 * h + 1] = __uint_as_float(w[h] & 0xFFFF0000u);
                }
            }
        }
        return;
    }
    if constexpr (DT == PSI_F32) {
        const float4 *p = reinterpret_cast<const float4 *>(static_cast<const float *>(base) + i * D + c0);
#pragma unroll
        for (int k = 0; k < CH / 4; ++k) {
            const float4 v = __ldg(p + k);
            f[4 * k] = v.x; f[4 * k + 1] = v.y; f[4 * k + 2] = v.z; f[4 * k + 3] = v.w;
        }
    } else if constexpr (DT == PSI_BF16) {
        const uint4 *p = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(base) + i * D + c0);
#pragma unroll
        for (int k = 0; k < CH / 8; ++k) {
            const uint4 v = __ldg(p + k);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                f[8 * k + 2 * h] = __uint_as_float(w[h] << 16);
                f[8 * k + 2 * h + 1] = __uint_as_float(w[h] & 0xFFFF0000u);
            }
        }
    } else {
        // FP8 E4M3 (sign, 4 exponent bits with bias 7, 3 mantissa bits): placing
        // the 7 magnitude bits at float bits [20, 27) gives 2^(e-127)(1+m/8)
        // (or the denormal m 2^-129 when e = 0); times 2^120 that is exactly
        // 2^(e-7)(1+m/8) (or m 2^-9).
        const uint4 *p = reinterpret_cast<const uint4 *>(static_cast<const uint8_t *>(base) + i * D + c0);
#pragma unroll
        for (int k = 0; k < CH / 16; ++k) {
            const uint4 v = __ldg(p + k);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const uint32_t byte = (w[h] >> (8 * b)) & 0xFFu;
                    const uint32_t bits = ((byte & 0x80u) << 24) | ((byte & 0x7Fu) << 20);
                    f[16 * k + 4 * h + b] = __uint_as_float(bits) * 0x1p120f;
                }
            }
        }
    }
}

// Dense features: CH channels of each staged record's row, as float32 before
// the scale, beside the record. The walk then reads a hit's channels from
// shared memory instead of waiting for a global row per trip (depth/normal
// maps of 700k surfels at 1237x701, D = 16: forward 545 -> 266 us, adjoint 870
// -> 658 us). Rows of 16 channels are padded to 20 floats, which keeps lanes storing neighbouring
// records, and groups reading different ones, in different banks.
__host__ __device__ constexpr int feat_stride(int CH) { return CH == 16 ? 20 : CH; }
__host__ __device__ constexpr size_t feat_stage_bytes(int CH) { return sizeof(float) * Pipe::kPS * kPB * feat_stride(CH); }
template <int DT, int CH>
struct StageFeat {
    const void *feat; // NULL: no features
    int D, c0;
    bool wide;
    uint32_t rec0; // the view's first record
    float4 *dst;
    __device__ __forceinline__ void operator()(int s, int j, uint32_t rec) const
    {
        if (!feat) return;
        float f[CH];
        load_feat<DT, CH>(feat, static_cast<int64_t>(rec - rec0), D, c0, f, wide);
        float4 *d = dst + (s * kPB + j) * (feat_stride(CH) / 4);
#pragma unroll
        for (int k = 0; k < CH / 4; ++k) d[k] = make_float4(f[4 * k], f[4 * k + 1], f[4 * k + 2], f[4 * k + 3]);
    }
};
template <int CH>
__device__ __forceinline__ void staged_feat(const float4 *stage, int s, int j, float (&f)[CH])
{
    const float4 *d = stage + (s * kPB + j) * (feat_stride(CH) / 4);
#pragma unroll
    for (int k = 0; k < CH / 4; ++k) {
        const float4 v = d[k];
        f[4 * k] = v.x;
        f[4 * k + 1] = v.y;
        f[4 * k + 2] = v.z;
        f[4 * k + 3] = v.w;
    }
}

// Four channels [c, c + 4) of feature row i as float32 (before the scale).
template <int DT>
__device__ __forceinline__ float4 load_feat4(const void *__restrict__ base, int64_t i, int D, int c)
{
    if constexpr (DT == PSI_F32) {
        return __ldg(reinterpret_cast<const float4 *>(static_cast<const float *>(base) + i * D + c));
    } else if constexpr (DT == PSI_BF16) {
        const uint2 u = __ldg(reinterpret_cast<const uint2 *>(static_cast<const __nv_bfloat16 *>(base) + i * D + c));
        return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                           __uint_as_float(u.y & 0xFFFF0000u));
    } else {
        // FP8 E4M3: the 7 magnitude bits at float bits [20, 27), times 2^120
        // (as in load_feat)
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(static_cast<const uint8_t *>(base) + i * D + c));
        float f[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const uint32_t byte = (w >> (8 * b)) & 0xFFu;
            f[b] = __uint_as_float(((byte & 0x80u) << 24) | ((byte & 0x7Fu) << 20)) * 0x1p120f;
        }
        return make_float4(f[0], f[1], f[2], f[3]);
    }
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

// Store CH channels (times scale) of one pixel's feature row as FP32 or BF16.
template <int CH>
__device__ __forceinline__ void store_feat(void *F, bool bf16, int64_t pix, int D, int c0, const float *acc,
                                           const float *__restrict__ scale)
{
    float v[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) v[c] = scale ? acc[c] * __ldg(scale + c0 + c) : acc[c];
    if (bf16) {
        uint4 *dst = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(F) + pix * D + c0);
#pragma unroll
        for (int k = 0; k < CH / 8; ++k) {
            uint32_t w4[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const __nv_bfloat162 p2 = __floats2bfloat162_rn(v[8 * k + 2 * h], v[8 * k + 2 * h + 1]);
                w4[h] = *reinterpret_cast<const uint32_t *>(&p2);
            }
            dst[k] = make_uint4(w4[0], w4[1], w4[2], w4[3]);
        }
    } else {
        float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(F) + pix * D + c0);
#pragma unroll
        for (int k = 0; k < CH / 4; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    }
}

// ------------------------------------------------------------ warp sums
// Sum 16 per-lane values over the warp (transposing butterfly, 16 shuffles):
// afterwards lane l (and l ^ 1) holds the total of value index
// 8 b4 + 4 b3 + 2 b2 + b1 (b_k = bit k of l).
__device__ __forceinline__ float warp_transpose_sum16(float v[16], int lane)
{
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const bool hi = lane & 16;
        const float send = hi ? v[k] : v[k + 8];
        const float keep = hi ? v[k + 8] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool hi = lane & 8;
        const float send = hi ? v[k] : v[k + 4];
        const float keep = hi ? v[k + 4] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool hi = lane & 4;
        const float send = hi ? v[k] : v[k + 2];
        const float keep = hi ? v[k + 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    {
        const bool hi = lane & 2;
        const float send = hi ? v[0] : v[1];
        const float keep = hi ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

} // namespace raster
} // namespace psi
