// a2: tile intersection and (tile|depth, record) key emission.
//
// Every visible record writes one pair per touched tile, in record order,
// tiles row-major: key = (global tile << 32) | float bits of the camera depth
// (positive, so the bit pattern orders like the value), value = record index.
// Which tiles a record touches is decided by the same float32 sequence that
// counted them (Sec. 5, Precise Tile Intersection; EXACT refines each tile row
// to the ellipse).
//
// One kernel: a block takes the next 1024 records (a ticket, so that every
// predecessor is already running), sums their tile counts, learns where its
// pairs start from its predecessors' published sums (decoupled look-back, a
// bounded wait per word; if one runs out the frame has no pairs), gathers its visible records -- half of a street's
// are culled -- and emits them one per thread. The counts are read once and no
// offsets are stored; up to 3072 pairs of a block are assembled in shared
// memory, so that its stores are contiguous (a thread writing its record's pairs
// to global memory directly touches a different sector per lane); a block with
// more writes them directly. Against a three-kernel scan, a count kernel and a
// direct emission from every record: four launches fewer, and 137 -> 124 us
// for 4.8M pairs of 3M records, 465 -> 352 us for 11.2M of 16M.
#include "discrete.cuh"

namespace psi {
namespace {

using namespace disc;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 4;                    // consecutive records per thread
constexpr int kRecords = kThreads * kItems;  // records per block
constexpr int kStage = 3072;                 // pairs assembled in shared memory
constexpr unsigned long long kOneRecord = 1ull << 48; // a visible record in the sums of pairs

// look-back word of a block: flag in bits 62-63, bit 61 set if the sum is not
// known because a wait gave up, the pair count below
constexpr unsigned long long kFlagAgg = 1ull << 62;  // the block's own count
constexpr unsigned long long kFlagIncl = 2ull << 62; // the count of all blocks up to this one
constexpr unsigned long long kFlags = 3ull << 62;
constexpr unsigned long long kPoison = 1ull << 61;
constexpr unsigned long long kValueMask = kPoison - 1ull;

// Pairs of all blocks before `part` (one warp; every lane gets the sum): the
// predecessors' words, 32 at a time, back to the first inclusive one. `ok` is
// false, and the sum meaningless, if a wait ran out here or at a predecessor.
__device__ __forceinline__ unsigned long long look_back(const unsigned long long *words, int64_t part,
                                                        DevStatus *status, bool &ok)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long limit = wait_limit(status);
    unsigned long long excl = 0;
    ok = true;
    for (int64_t q = part - 1; q >= 0; q -= 32) {
        const int64_t idx = q - lane;
        unsigned long long w = kFlagIncl; // before the first block: nothing
        unsigned long long t0 = 0;
        while (true) {
            if (idx >= 0) w = *reinterpret_cast<const volatile unsigned long long *>(words + idx);
            if (__all_sync(0xffffffffu, (w & kFlags) != 0)) break;
            if (__any_sync(0xffffffffu, wait_expired(t0, limit))) {
                if (lane == 0 && status) {
                    atomicCAS(&status->wait_site, 0, kSiteIntersect);
                    raise_status(status, PSI_ERR_TIMEOUT);
                }
                ok = false;
                return 0;
            }
        }
        const uint32_t incl = __ballot_sync(0xffffffffu, (w & kFlagIncl) != 0);
        const int first = incl ? __ffs(incl) - 1 : 31;
        if (__any_sync(0xffffffffu, lane <= first && (w & kPoison))) {
            ok = false;
            return 0;
        }
        unsigned long long v = lane <= first ? (w & kValueMask) : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        excl += v;
        if (incl) break;
    }
    return excl;
}

__global__ void __launch_bounds__(kThreads) intersect_kernel(const __grid_constant__ FrameParams fp,
                                                             const float4 *__restrict__ bins,
                                                             const uint32_t *__restrict__ counts,
                                                             uint64_t *__restrict__ keys, uint32_t *__restrict__ vals,
                                                             int64_t capacity, int64_t *__restrict__ d_num_pairs,
                                                             unsigned long long *words, unsigned int *ticket,
                                                             unsigned long long *finished, DevStatus *status)
{
    __shared__ uint64_t s_keys[kStage];
    __shared__ uint32_t s_vals[kStage];
    __shared__ uint32_t s_off[kRecords];
    __shared__ uint16_t s_rec[kRecords];
    __shared__ unsigned long long warp_sum[kWarps];
    __shared__ unsigned long long s_base;
    __shared__ bool s_ok;
    __shared__ unsigned int s_part;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) s_part = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t part = s_part;
    const int64_t total = fp.n * fp.n_views;
    const int64_t rec0 = part * kRecords;
    // the thread's records: pairs in the low 48 bits of each sum, visible
    // records (at most 1024 of a block) above
    uint32_t cnt[kItems];
    unsigned long long mine = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const int64_t r = rec0 + tid * kItems + k;
        cnt[k] = r < total ? counts[r] : 0u;
        mine += cnt[k] ? kOneRecord + cnt[k] : 0ull;
    }
    unsigned long long inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) warp_sum[wid] = inc;
    __syncthreads();
    unsigned long long before = inc - mine, both = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        if (w < wid) before += warp_sum[w];
        both += warp_sum[w];
    }
    const unsigned long long all = both & (kOneRecord - 1ull);
    const int visible = static_cast<int>(both / kOneRecord);
    // the visible records and where each one's pairs start in the block
#pragma unroll
    for (int k = 0; k < kItems; ++k)
        if (cnt[k]) {
            const int v = static_cast<int>(before / kOneRecord);
            const unsigned long long off = before & (kOneRecord - 1ull);
            s_rec[v] = static_cast<uint16_t>(tid * kItems + k);
            s_off[v] = off < 0xffffffffull ? static_cast<uint32_t>(off) : 0xffffffffu; // past any capacity
            before += kOneRecord + cnt[k];
        }
    if (wid == 0) {
        volatile unsigned long long *my = words + part;
        unsigned long long excl = 0;
        bool ok = true;
        if (part > 0) {
            if (lane == 0) *my = kFlagAgg | all;
            excl = look_back(words, part, status, ok);
        }
        if (lane == 0) {
            *my = kFlagIncl | (ok ? excl + all : kPoison);
            s_base = excl;
            s_ok = ok;
        }
    }
    __syncthreads();
    const unsigned long long base = s_base;
    const unsigned long long cap = static_cast<unsigned long long>(capacity);
    if (tid == kThreads - 1) {
        // The block that finishes last (not the frame's last block: one before
        // it may still give up) knows whether every block has its place, and
        // the frame's count: without it the list would have holes, so there is none.
        __threadfence();
        const unsigned long long old = atomicAdd(finished, s_ok ? 1ull : (1ull << 32) + 1ull);
        if (static_cast<uint32_t>(old) == gridDim.x - 1) {
            __threadfence();
            const bool whole = s_ok && (old >> 32) == 0;
            const unsigned long long w = *reinterpret_cast<const volatile unsigned long long *>(words + gridDim.x - 1);
            const unsigned long long pairs = whole ? w & kValueMask : 0ull;
            if (pairs > cap) {
                raise_status(status, PSI_ERR_CAPACITY);
                atomicMax(&status->required_pairs, pairs);
            }
            *d_num_pairs = static_cast<int64_t>(pairs < cap ? pairs : cap);
        }
    }
    if (!s_ok || base >= cap) return;

    // one visible record per thread
    const bool staged = all <= kStage;
    const bool lp = fp.lowpass != 0;
    const int tw = fp.tile_w, th = fp.tile_h;
    for (int v = tid; v < visible; v += kThreads) {
        const int64_t r = rec0 + s_rec[v];
        unsigned long long off = s_off[v];
        if (base + off >= cap) continue;
        float depth;
        const Bin b = load_bin(bins + bin_stride(lp) * r, depth, lp);
        const ViewParams &cam = fp.v[fp.n_views > 1 ? static_cast<uint32_t>(r) / static_cast<uint32_t>(fp.n) : 0u];
        const uint64_t dbits = __float_as_uint(depth);
        const uint32_t val = static_cast<uint32_t>(r);
        for (int ty = b.py0 / th; ty <= b.py1 / th; ++ty) {
            int c0, c1;
            if (!row_tiles(b, fp.mode, ty, tw, th, c0, c1)) continue;
            const uint32_t rowbase = cam.tile_base + static_cast<uint32_t>(ty * cam.tiles_x);
            for (int tx = c0; tx <= c1; ++tx, ++off) {
                const uint64_t key = (static_cast<uint64_t>(rowbase + static_cast<uint32_t>(tx)) << 32) | dbits;
                if (staged) {
                    if (off < kStage) {
                        s_keys[off] = key;
                        s_vals[off] = val;
                    }
                } else if (base + off < cap) { // pairs past the capacity are dropped
                    keys[base + off] = key;
                    vals[base + off] = val;
                }
            }
        }
    }
    if (!staged) return;
    __syncthreads();
    const int m = static_cast<int>(all < cap - base ? all : cap - base);
    for (int j = tid; j < m; j += kThreads) {
        keys[base + j] = s_keys[j];
        vals[base + j] = s_vals[j];
    }
}

int64_t blocks_of(int64_t n_records) { return (n_records + kRecords - 1) / kRecords; }

} // namespace

// the look-back words, the ticket and the finished blocks' count
size_t intersect_workspace_bytes(int64_t n_records)
{
    return align_up(static_cast<size_t>(blocks_of(std::max<int64_t>(n_records, 1))) * 8 + 16, 256);
}

cudaError_t launch_intersect(const FrameParams &fp, const float4 *bin_records, const uint32_t *tiles_touched,
                             uint64_t *keys, uint32_t *vals, int64_t capacity, int64_t *d_num_pairs, void *ws,
                             DevStatus *status, cudaStream_t st)
{
    const int64_t R = fp.n * fp.n_views;
    if (R == 0) return cudaMemsetAsync(d_num_pairs, 0, sizeof(int64_t), st);
    const int64_t nb = blocks_of(R);
    auto *words = static_cast<unsigned long long *>(ws);
    auto *ticket = reinterpret_cast<unsigned int *>(words + nb);
    cudaError_t e = cudaMemsetAsync(ws, 0, static_cast<size_t>(nb) * 8 + 16, st);
    if (e != cudaSuccess) return e;
    intersect_kernel<<<static_cast<unsigned>(nb), kThreads, 0, st>>>(fp, bin_records, tiles_touched, keys, vals, capacity,
                                                                    d_num_pairs, words, ticket, words + nb + 1, status);
    return cudaGetLastError();
}

} // namespace psi
