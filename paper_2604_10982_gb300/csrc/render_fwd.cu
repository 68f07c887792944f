// a4: per-tile compositing with Top-K Hard Selection.
//
// One CTA per 16x16 tile, one thread per pixel. The tile's sorted list is
// streamed through shared-memory stages of 128 records (raster.cuh); each
// warp lists, per group of eight pixels, the records that can reach the group
// and every group walks its own list. Per pixel (Sec. 3.1, Eq. 1): alpha =
// min(0.99, o exp(-(u^2+v^2)/2)), RGB blended densely front to back with FP32
// transmittance T, and the K largest weights omega_j = alpha_j T_j kept
// (Sec. 5, Top-K Hard Selection; TopK, TopKShared). After the walk
// the K selected features are gathered row by row and summed in list order in
// FP32: F = scale * sum_{j in K} omega_j q_j (gather_rows).
// Dense features (K = 0) accumulate 32 channels per pass over the list.
#include "raster.cuh"

namespace psi {
namespace {

using namespace raster;

struct FwdArgs {
    const float4 *records;
    const uint32_t *vals;
    const uint32_t *ranges;
    const void *feat;
    const float *fscale;
    int D;
    bool wide; // feature rows read 32 bytes at a time
    int c0;          // dense mode: first channel of this pass
    int write_rgb;   // dense mode: only the first pass writes rgb / T / ids
    float *rgb;
    float *T;
    int32_t *n_last;
    void *F;
    int F_bf16;
    int32_t *topk_ids;
    float *topk_w;
    int32_t *argmax;
    DevStatus *status;
    unsigned int *work; // persistent launch: the context's tile counter pair; NULL: one tile per CTA
};

// 16 bytes of a feature row as CPL float32 values' products with a weight:
// acc[c] = fma(w, f_c, acc[c]), channel pairs by packed FMAs (each lane
// rounded as the scalar one).
template <int DT>
__device__ __forceinline__ void fma_row(const uint4 v, float w, float2 *acc)
{
    const uint32_t x[4] = {v.x, v.y, v.z, v.w};
    if constexpr (DT == PSI_F32) {
        const float2 ww = make_float2(w, w);
#pragma unroll
        for (int k = 0; k < 2; ++k)
            acc[k] = __ffma2_rn(ww, make_float2(__uint_as_float(x[2 * k]), __uint_as_float(x[2 * k + 1])), acc[k]);
    } else if constexpr (DT == PSI_BF16) {
        const float2 ww = make_float2(w, w);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            acc[k] = __ffma2_rn(ww, make_float2(__uint_as_float(x[k] << 16), __uint_as_float(x[k] & 0xFFFF0000u)), acc[k]);
    } else {
        // FP8 E4M3: the byte's sign at bit 31 and its 7 magnitude bits at bits
        // [20, 27) are the value times 2^-120 (a shift that copies the sign
        // down, the copies masked off); the weight carries the 2^120, so the
        // product is the exact one of the decoded value
        const float ws = w * 0x1p120f;
        const float2 ww = make_float2(ws, ws);
        auto val = [](uint32_t top) { return __uint_as_float(static_cast<uint32_t>(static_cast<int32_t>(top) >> 4) & 0x87F00000u); };
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[2 * k] = __ffma2_rn(ww, make_float2(val(x[k] << 24), val(x[k] << 16)), acc[2 * k]);
            acc[2 * k + 1] = __ffma2_rn(ww, make_float2(val(x[k] << 8), val(x[k])), acc[2 * k + 1]);
        }
    }
}

// The K largest weights of one pixel with their list positions (Sec. 5, Top-K
// Hard Selection), in shared memory: slot c of a lane is the float2 (weight,
// position bits) c & 1 of the float4 at [c >> 1][lane]. The first K weights
// are appended, which is most of what a pixel ever keeps, so a new surfel costs one
// store; after that a weight larger than the smallest kept one takes its
// slot and the new smallest is looked up. Ties favour the earlier position:
// among equal smallest weights the latest is replaced, and only by a strictly
// larger one. In registers (TopK: sorted, shifted on every insertion) the set
// costs 5 instructions per slot whenever any lane of the warp improves its own
// -- nearly always while sets fill -- and K = 16 leaves room for two CTAs per
// SM instead of three. For K <= 8 the registers are the better place (1.52
// against 1.60 ms for the 3M-surfel 1080p frame).
struct TopKShared {
    int cnt, cmin; // entries; slot of the smallest
    float wmin;    // the smallest weight
    bool replaced; // some entry is out of list order

    __device__ __forceinline__ void init()
    {
        cnt = cmin = 0;
        wmin = __int_as_float(0x7f800000);
        replaced = false;
    }

    __device__ __forceinline__ void offer(float4 *ent, int lane, int K, float w, int pos)
    {
        float2 *e2 = reinterpret_cast<float2 *>(ent) + 2 * lane;
        if (cnt < K) {
            e2[64 * (cnt >> 1) + (cnt & 1)] = make_float2(w, __int_as_float(pos));
            if (w <= wmin) {
                wmin = w;
                cmin = cnt;
            }
            ++cnt;
        } else if (w > wmin) {
            e2[64 * (cmin >> 1) + (cmin & 1)] = make_float2(w, __int_as_float(pos));
            replaced = true;
            wmin = __int_as_float(0x7f800000);
            int pmin = -1;
#pragma unroll 4
            for (int c = 0; c < K; ++c) {
                const float2 e = e2[64 * (c >> 1) + (c & 1)];
                const int pc = __float_as_int(e.y);
                if (e.x < wmin || (e.x == wmin && pc > pmin)) {
                    wmin = e.x;
                    pmin = pc;
                    cmin = c;
                }
            }
        }
    }
};

// float4 of shared memory per warp for the sets: K rounded up to four slots
__host__ __device__ constexpr int topk_entries(int K) { return (K + 3) / 4 * 64; }

// The Top-K feature sum of the warp's 32 pixels, F = scale * sum_{j in K}
// omega_j q_j, and / or its channel argmax. ent holds each pixel's selection
// in list order as (surfel, weight) pairs, two slots to a float4 at [slot / 2]
// [lane], weight -1 past its end. Rows are read by whole lanes' worths of 16
// bytes: D * esize / 16 lanes share one pixel, so the warp works on 32 / lanes
// pixels at a time, every load covers whole rows and every store a whole row
// of F; the kernel is bound by instruction issue, and this costs one address,
// one load and the packed FMAs per 16 bytes of a row. (One pixel per lane,
// 32 bytes of 32 different rows per load, was bound by the L1's tag lookups
// and, in FP8, by five instructions per value to decode.) The order of the
// additions is that of one lane summing alone in list order.
template <int KMAX, int DT>
__device__ __forceinline__ void gather_rows(const ViewParams &cam, const FwdArgs &a, int vw, int tile_x0, int tile_y0,
                                            int K, const float4 *ent, float T)
{
    constexpr int CPL = DT == PSI_F32 ? 4 : (DT == PSI_BF16 ? 8 : 16); // channels per lane: 16 bytes
    const int lane = threadIdx.x & 31;
    const int row_lanes = a.D / CPL; // 1 .. 64
    int lp = 1;                      // lanes per pixel: row_lanes rounded up to a power of two, at most 32
    while (lp < row_lanes && lp < 32) lp <<= 1;
    const int sub = lane & (lp - 1);
    const int row_bytes = row_lanes * 16;
#pragma unroll 1
    for (int t = 0; t < lp; ++t) {
        const int src = t * (32 / lp) + lane / lp; // the lane whose pixel this lane works on
        int lxi, lyi;
        pixel_of_thread(vw * 32 + src, lxi, lyi);
        const int px = tile_x0 + lxi, py = tile_y0 + lyi;
        const bool in = px < cam.W && py < cam.H;
        const int64_t pix = cam.pix_base + static_cast<int64_t>(py) * cam.W + px;
        float best = -__int_as_float(0x7f800000);
        int arg = 0;
#pragma unroll 1
        for (int cb = 0; cb < row_lanes; cb += 32) {
            const bool on = cb + sub < row_lanes;
            // lanes past the row read its last 16 bytes and drop them
            const unsigned char *base = static_cast<const unsigned char *>(a.feat) + 16 * min(cb + sub, row_lanes - 1);
            float2 acc[CPL / 2];
#pragma unroll
            for (int c = 0; c < CPL / 2; ++c) acc[c] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int s0 = 0; s0 < KMAX; s0 += 4) {
                if (s0 >= K) break;
                float4 e[2];
                e[0] = ent[(s0 / 2) * 32 + src];
                e[1] = ent[(s0 / 2 + 1) * 32 + src];
                // selections are packed: nothing further if no pixel has this slot
                if (!__any_sync(0xffffffffu, e[0].y >= 0.0f)) break;
                uint4 v[4];
                v[0] = __ldg(reinterpret_cast<const uint4 *>(base + static_cast<int64_t>(__float_as_int(e[0].x)) * row_bytes));
                v[1] = __ldg(reinterpret_cast<const uint4 *>(base + static_cast<int64_t>(__float_as_int(e[0].z)) * row_bytes));
                v[2] = __ldg(reinterpret_cast<const uint4 *>(base + static_cast<int64_t>(__float_as_int(e[1].x)) * row_bytes));
                v[3] = __ldg(reinterpret_cast<const uint4 *>(base + static_cast<int64_t>(__float_as_int(e[1].z)) * row_bytes));
                if (e[0].y >= 0.0f) fma_row<DT>(v[0], e[0].y, acc);
                if (e[0].w >= 0.0f) fma_row<DT>(v[1], e[0].w, acc);
                if (e[1].y >= 0.0f) fma_row<DT>(v[2], e[1].y, acc);
                if (e[1].w >= 0.0f) fma_row<DT>(v[3], e[1].w, acc);
            }
            const int c0 = (cb + sub) * CPL;
            if (on && in) {
                float f[CPL];
#pragma unroll
                for (int c = 0; c < CPL / 2; ++c) {
                    f[2 * c] = acc[c].x;
                    f[2 * c + 1] = acc[c].y;
                }
                if (a.fscale) {
#pragma unroll
                    for (int c = 0; c < CPL; ++c) f[c] *= __ldg(a.fscale + c0 + c);
                }
                if (a.F) {
                    if (a.F_bf16) {
                        uint32_t h[CPL / 2];
#pragma unroll
                        for (int c = 0; c < CPL / 2; ++c) {
                            const __nv_bfloat162 p2 = __floats2bfloat162_rn(f[2 * c], f[2 * c + 1]);
                            h[c] = *reinterpret_cast<const uint32_t *>(&p2);
                        }
                        __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(a.F) + pix * a.D + c0;
                        if constexpr (CPL == 4) {
                            *reinterpret_cast<uint2 *>(dst) = make_uint2(h[0], h[1]);
                        } else {
#pragma unroll
                            for (int k = 0; k < CPL / 8; ++k)
                                reinterpret_cast<uint4 *>(dst)[k] = make_uint4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
                        }
                    } else {
                        float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(a.F) + pix * a.D + c0);
#pragma unroll
                        for (int k = 0; k < CPL / 4; ++k)
                            dst[k] = make_float4(f[4 * k], f[4 * k + 1], f[4 * k + 2], f[4 * k + 3]);
                    }
                }
                if (a.argmax) {
#pragma unroll
                    for (int c = 0; c < CPL; ++c)
                        if (f[c] > best) {
                            best = f[c];
                            arg = c0 + c;
                        }
                }
            }
        }
        if (a.argmax) {
            // largest value of the pixel's lanes, lowest channel on ties
            for (int o = lp >> 1; o > 0; o >>= 1) {
                const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
                if (ob > best || (ob == best && oa < arg)) {
                    best = ob;
                    arg = oa;
                }
            }
            const float Tp = __shfl_sync(0xffffffffu, T, src);
            if (in && sub == 0) a.argmax[pix] = (1.0f - Tp < 1e-4f) ? -1 : arg;
        }
    }
}

// One tile of the frame (the whole CTA; P freshly initialised by thread 0
// below). TH: tile height (16x16 or 16x8 tiles).
template <int KMAX, int DT, int CH, bool LP, int TH, class PP>
__device__ __forceinline__ void fwd_tile(const FrameParams &fp, const FwdArgs &a, PP &P, HitLists *hits,
                                         float4 *entries, uint32_t tile)
{
    constexpr int PW = pixel_warps(TH);
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const unsigned long long wlimit = wait_limit(a.status); // in flight with the tile's own loads
    const int v = view_of_tile(fp, tile);
    const ViewParams &cam = fp.v[v];
    const int local = static_cast<int>(tile - cam.tile_base);
    const int tx = local % cam.tiles_x, ty = local / cam.tiles_x;
    const int64_t list0 = a.ranges[2 * tile];
    int n = static_cast<int>(a.ranges[2 * tile + 1] - a.ranges[2 * tile]);
    if (!PSI_CHECK(a.ranges[2 * tile + 1] >= a.ranges[2 * tile], kChkRange, a.status)) n = 0;
    const int nb = (n + kPB - 1) / kPB;
    const uint32_t rec_lo = static_cast<uint32_t>(static_cast<int64_t>(v) * fp.n);
    const uint32_t rec_hi = static_cast<uint32_t>(static_cast<int64_t>(v + 1) * fp.n);

    // A 16x8 tile is the upper or lower half of the 16x16 tile it lies in:
    // records are folded at that 16x16 tile's origin and its pixel warps play
    // warps 0-3 or 4-7 of it, so every pixel evaluates exactly the float32
    // sequence of the 16x16 launch (same results bit for bit).
    const int oy = (ty * TH) & 15;
    const int vw = wid + (oy ? pixel_warps(16) / 2 : 0); // warp of the 16x16 tile this warp plays
    if (tid == 0) pipe_init(P, PW, wlimit);
    __syncthreads();
    auto stage = [&](const auto &extra) {
        if (wid == PW)
            pipe_produce<LP, PW>(P, a.vals, list0, n, false, a.records, tx * kTile, ty * TH - oy, a.status,
                                 kSiteRenderFwd, rec_lo, rec_hi, extra);
        else
            pipe_prefill<LP, PW>(P, wid, a.vals, list0, n, false, a.records, tx * kTile, ty * TH - oy, a.status, rec_lo,
                                 rec_hi, extra);
    };
    // dense features: this pass's channels are staged with the records
    if constexpr (KMAX == 0)
        stage(StageFeat<DT, CH>{a.feat, a.D, a.c0, a.wide, rec_lo, entries});
    else
        stage(NoExtra());
    if (wid == PW) return;

    int lxi, lyi;
    pixel_of_thread(vw * 32 + lane, lxi, lyi);
    const int px = tx * kTile + lxi, py = ty * TH - oy + lyi;
    const bool inside = px < cam.W && py < cam.H;
    const float lx = static_cast<float>(lxi), ly = static_cast<float>(lyi);
    const int64_t surf0 = static_cast<int64_t>(v) * fp.n;
    const int K = KMAX > 0 ? fp.top_k : 0;
    const int grp = lane >> 3;

    float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
    int last = 0;
    bool done = !inside;
    // K <= 8: sorted in registers (top); larger K: in shared memory (set)
    constexpr bool kShared = KMAX > 8;
    TopK<(KMAX > 0 && !kShared ? KMAX : 1)> top;
    top.init(K);
    TopKShared set;
    set.init();
    float4 *ent = entries + wid * topk_entries(K);
    float facc[KMAX == 0 ? CH : 1];
#pragma unroll
    for (int c = 0; c < (KMAX == 0 ? CH : 1); ++c) facc[c] = 0.0f;

    bool in_walk = !__all_sync(0xffffffffu, done);
    if (!in_walk) pipe_leave(P, wid);
    for (int b = 0; b < nb && in_walk; ++b) {
        if (!pipe_wait_ready(P, b, a.status, kSiteRenderFwd)) break;
        const int st = b % PP::kPS;
        int cnt;
        const int lo = batch_range(b, n, false, cnt);
        // only the records that can reach a pixel of this lane's group, in list order
        int ng[kGroups];
        const int lim[kGroups] = {kPB, kPB, kPB, kPB};
        build_hits<LP, kGroups>(P, st, cnt, vw, tx * kTile, ty * TH - oy, lim, hits[wid], ng);
        const int mine = grp == 0 ? ng[0] : grp == 1 ? ng[1] : grp == 2 ? ng[2] : ng[3];
        const int most = max(max(ng[0], ng[1]), max(ng[2], ng[3]));
        const uint8_t *list = hits[wid][grp];
#pragma unroll 1
        for (int i = 0; i < most; ++i) {
            if (__all_sync(0xffffffffu, done)) break;
            const int j = list[i] & (kPB - 1); // past the group's list: any staged record, not used
            const Rec r = load_rec(P.rec[st][j]);
            Eval e;
            const bool hit = i < mine && !done && eval_alpha<LP>(r, lx, ly, e);
            const float w = hit ? __fmul_rn(e.alpha, T) : 0.0f;
            const int pos = lo + j;
            if (hit) {
                const float4 col = P.rec[st][j][3];
                cr = __fmaf_rn(w, col.y, cr);
                cg = __fmaf_rn(w, col.z, cg);
                cb = __fmaf_rn(w, col.w, cb);
                if constexpr (KMAX == 0) {
                    if (a.feat) {
                        float f[CH];
                        staged_feat<CH>(entries, st, j, f);
#pragma unroll
                        for (int c = 0; c < CH; ++c) facc[c] = __fmaf_rn(w, f[c], facc[c]);
                    }
                }
            }
            if constexpr (KMAX > 0 && !kShared) top.offer(hit, w, pos);
            if (hit) {
                if constexpr (kShared) set.offer(ent, lane, K, w, pos);
                T = __fmul_rn(T, __fsub_rn(1.0f, e.alpha));
                last = pos + 1;
                if (T < fp.t_eps) done = true;
            }
        }
        if (__all_sync(0xffffffffu, done)) {
            in_walk = false;
            pipe_leave(P, wid);
        } else {
            pipe_release(P, wid, b);
        }
    }
    // one answer for the warp, whose gather is warp-wide (as a vote, which the
    // compiler knows to be uniform, 1.3 % slower at K = 8)
    if (__shfl_sync(0xffffffffu, vload(P.abort), 0)) return;

    const int64_t pix = cam.pix_base + static_cast<int64_t>(py) * cam.W + px;
    if (inside && a.write_rgb) {
        a.rgb[pix] = cr;
        a.rgb[fp.n_pix_total + pix] = cg;
        a.rgb[2 * fp.n_pix_total + pix] = cb;
        a.T[pix] = T;
        if (a.n_last) a.n_last[pix] = last;
    }

    if constexpr (KMAX == 0) {
        if (inside && a.F && a.feat) store_feat<CH>(a.F, a.F_bf16 != 0, pix, a.D, a.c0, facc, a.fscale);
    } else {
        TopK<KMAX> sel; // the set in list order (empty slots last)
        if constexpr (kShared) {
#pragma unroll
            for (int s = 0; s < KMAX; ++s) {
                const bool ok = s < K && s < set.cnt;
                const float2 e = ok ? reinterpret_cast<const float2 *>(ent)[64 * (s >> 1) + 2 * lane + (s & 1)]
                                    : make_float2(-1.0f, __int_as_float(0x7fffffff));
                sel.w[s] = e.x;
                sel.p[s] = __float_as_int(e.y);
            }
            if (__any_sync(0xffffffffu, set.replaced)) sel.sort_by_pos();
        } else {
            sel = top;
            sel.sort_by_pos();
        }
#pragma unroll
        for (int s = 0; s < KMAX; ++s) {
            int32_t id = sel.valid(s, K) ? static_cast<int32_t>(static_cast<int64_t>(a.vals[list0 + sel.p[s]]) - surf0) : -1;
            if (!PSI_CHECK(id >= -1 && id < fp.n, kChkFeatRow, a.status)) id = -1;
            sel.p[s] = id;
        }
        if (inside && a.topk_ids) {
            int32_t *dst = a.topk_ids + pix * K;
#pragma unroll
            for (int s = 0; s < KMAX; ++s)
                if (s < K) dst[s] = sel.p[s];
        }
        if (inside && a.topk_w) {
            float *dst = a.topk_w + pix * K;
#pragma unroll
            for (int s = 0; s < KMAX; ++s)
                if (s < K) dst[s] = sel.p[s] >= 0 ? sel.w[s] : 0.0f;
        }
        if ((a.F || a.argmax) && a.feat) {
            auto pair = [&](int s) {
                return make_float2(__int_as_float(max(sel.p[s], 0)), sel.p[s] >= 0 ? sel.w[s] : -1.0f);
            };
#pragma unroll
            for (int s = 0; s < KMAX; s += 2)
                if (s < (K + 3) / 4 * 4) {
                    const float2 e0 = pair(s), e1 = pair(s + 1);
                    ent[(s >> 1) * 32 + lane] = make_float4(e0.x, e0.y, e1.x, e1.y);
                }
            __syncwarp();
            gather_rows<KMAX, DT>(cam, a, vw, tx * kTile, ty * TH - oy, K, ent, T);
        }
    }
}

// Record stages: four where the CTAs per SM that the build is for fit with them
// (K <= 8 at three, dense features). With the sets (2 KB per slot and 16x16 tile,
// half for 16x8) four stages let only three of four and four of five CTAs be
// resident: 1.58 against 1.51 ms at four CTAs, 1.63 against 1.44 ms for 16x8
// tiles at five (3M-surfel 1080p frame, K = 8; three CTAs and four stages: 1.46).
__host__ __device__ constexpr int fwd_stages(int KMAX, int OCC, int TH)
{
    return KMAX > 8 || (KMAX > 0 && (OCC > 3 || TH == 8)) ? 3 : 4;
}

// OCC: CTAs per SM the kernel is built for (the launch shape the autotuner
// picks). Tiles are taken longest list first: CTA b starts with entry b of the
// launch order; in the persistent launch (a.work set, grid of a few CTAs per
// SM) each CTA then fetches the next entry from the context's counter until
// the order is exhausted, and the last CTA to finish resets the counter pair
// for the next launch (launches through one context must not overlap).
template <int KMAX, int DT, int CH, bool LP, int OCC, int TH = 16>
__global__ void __launch_bounds__(pipe_threads(TH), OCC)
    render_fwd_kernel(const __grid_constant__ FrameParams fp, FwdArgs a)
{
    __shared__ __align__(128) PipeT<fwd_stages(KMAX, OCC, TH)> P;
    __shared__ HitLists hits[pixel_warps(TH)];
    __shared__ uint32_t s_next;
    extern __shared__ __align__(16) float4 entries[]; // K > 0: topk_entries(K) per pixel warp; dense: feature stages
    uint32_t i = blockIdx.x;
    while (true) {
        const uint32_t tile = a.ranges[2 * fp.n_tiles_total + i];
        // debug builds: the launch order must name a tile of the frame (uniform for the CTA)
        if (PSI_CHECK(tile < fp.n_tiles_total, kChkTile, a.status)) fwd_tile<KMAX, DT, CH, LP, TH>(fp, a, P, hits, entries, tile);
        if (!a.work) break;
        __syncthreads(); // every warp is done with this tile's pipeline
        if (threadIdx.x == 0) {
            s_next = vload(P.abort) ? 0xffffffffu : gridDim.x + atomicAdd(&a.work[0], 1u);
            pipe_inval(P);
        }
        __syncthreads();
        i = s_next;
        if (i >= fp.n_tiles_total) break;
    }
    if (a.work && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&a.work[1], 1u) == gridDim.x - 1) {
            a.work[0] = 0u;
            a.work[1] = 0u;
        }
    }
}

template <int KMAX, int DT, int CH, bool LP, int OCC, int TH>
cudaError_t launch_one(const FrameParams &fp, const FwdArgs &a, cudaStream_t st)
{
    const auto kernel = render_fwd_kernel<KMAX, DT, CH, LP, OCC, TH>;
    const unsigned grid = a.work ? persistent_grid(fp.n_tiles_total, OCC) : fp.n_tiles_total;
    constexpr auto set_bytes = [](int K) constexpr { return static_cast<size_t>(pixel_warps(TH)) * topk_entries(K) * sizeof(float4); };
    const size_t dyn = KMAX > 0 ? set_bytes(fp.top_k) : (a.feat ? feat_stage_bytes(CH) : 0);
    constexpr size_t most = KMAX > 0 ? set_bytes(KMAX) : feat_stage_bytes(CH);
    static_assert(smem_fits<PipeT<fwd_stages(KMAX, OCC, TH)>>(OCC, TH, most), "fewer CTAs fit than the build is for");
    // the sets or features and the record stages together pass 48 KB
    const cudaError_t e = allow_dynamic_smem(kernel, most);
    if (e != cudaSuccess) return e;
    kernel<<<grid, pipe_threads(TH), dyn, st>>>(fp, a);
    return cudaGetLastError();
}

template <int KMAX, int CH, bool LP, int OCC, int TH = 16>
cudaError_t launch_kclo(const FrameParams &fp, const FeatView &f, const FwdArgs &a, cudaStream_t st)
{
    switch (f.data ? f.dtype : PSI_F32) {
    case PSI_BF16: return launch_one<KMAX, PSI_BF16, CH, LP, OCC, TH>(fp, a, st);
    case PSI_FP8_E4M3: return launch_one<KMAX, PSI_FP8_E4M3, CH, LP, OCC, TH>(fp, a, st);
    default: return launch_one<KMAX, PSI_F32, CH, LP, OCC, TH>(fp, a, st);
    }
}

// 16x8 tiles (Top-K with K <= 8, no low-pass filter): 4 pixel warps, 5 CTAs per SM
constexpr int kOccTile8 = 5;

template <int KMAX, int CH, bool LP>
cudaError_t launch_kcl(const FrameParams &fp, const FeatView &f, const FwdArgs &a, bool alt, cudaStream_t st)
{
    // CTAs per SM: K <= 8: 3 (4 as the alternative); K <= 16: 3 (2), 37 KB of
    // stages and lists and 2 KB per slot of the sets; larger K and dense: 2 (1)
    constexpr int occ = (KMAX > 0 && KMAX <= 16) ? 3 : 2;
    constexpr int occ_alt = (KMAX > 0 && KMAX <= 8) ? 4 : occ - 1;
    return alt ? launch_kclo<KMAX, CH, LP, occ_alt>(fp, f, a, st) : launch_kclo<KMAX, CH, LP, occ>(fp, f, a, st);
}

template <int KMAX, int CH>
cudaError_t launch_kc(const FrameParams &fp, const FeatView &f, const FwdArgs &a, bool alt, cudaStream_t st)
{
    return fp.lowpass ? launch_kcl<KMAX, CH, true>(fp, f, a, alt, st) : launch_kcl<KMAX, CH, false>(fp, f, a, alt, st);
}

template <int KMAX>
cudaError_t launch_k(const FrameParams &fp, const FeatView &f, const FwdArgs &a, int ch, bool alt, cudaStream_t st)
{
    if (fp.n_tiles_total == 0) return cudaSuccess;
    // the channel chunk only shapes the dense (K = 0) accumulation
    if constexpr (KMAX > 0)
        return launch_kc<KMAX, 16>(fp, f, a, alt, st);
    else
        return ch == 32 ? launch_kc<KMAX, 32>(fp, f, a, alt, st) : launch_kc<KMAX, 16>(fp, f, a, alt, st);
}

} // namespace

cudaError_t launch_render_fwd(const FrameParams &fp, const FeatView &f, const float4 *records, const uint32_t *vals,
                              const uint32_t *ranges, const psi_fwd_out &out, DevStatus *status, cudaStream_t st,
                              int shape)
{
    FwdArgs a{};
    a.records = records;
    a.vals = vals;
    a.ranges = ranges;
    a.feat = f.data;
    a.wide = f.data && feat_rows_wide(f.data, f.dim, f.dtype);
    a.fscale = f.scale;
    a.D = f.dim;
    a.c0 = 0;
    a.write_rgb = 1;
    a.rgb = out.rgb;
    a.T = out.T;
    a.n_last = out.n_last;
    a.F = out.F;
    a.F_bf16 = out.F_dtype == PSI_BF16;
    a.topk_ids = out.topk_ids;
    a.topk_w = out.topk_w;
    a.argmax = out.argmax;
    a.status = status;
    const int K = fp.top_k;
    const int ch = render_channel_chunk(f.dim, K, shape);
    const bool alt = shape & kShapeAltOcc;
    a.work = (shape & kShapePersistent) ? status->work : nullptr;
    if (K == 0) {
        // dense: one pass per chunk of channels (the first also writes rgb/T)
        cudaError_t e = launch_k<0>(fp, f, a, ch, alt, st);
        for (int c0 = ch; e == cudaSuccess && f.data && out.F && c0 < f.dim; c0 += ch) {
            a.c0 = c0;
            a.write_rgb = 0;
            e = launch_k<0>(fp, f, a, ch, alt, st);
        }
        return e;
    }
    if (fp.tile_h == 8) return launch_kclo<8, 16, false, kOccTile8, 8>(fp, f, a, st);
    if (K <= 8) return launch_k<8>(fp, f, a, ch, alt, st);
    if (K <= 16) return launch_k<16>(fp, f, a, ch, alt, st);
    return launch_k<32>(fp, f, a, ch, alt, st);
}

} // namespace psi
