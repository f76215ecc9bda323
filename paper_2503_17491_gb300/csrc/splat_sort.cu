// K2-K4: tile binning, from the projection's pixel rectangles to the per-tile lists in
// (range, primitive id) order (Sec. 3.2.1).
//
//   count    list lengths: a CTA counts the tiles of a band of one view over a chunk of its
//            touching pairs in shared memory and adds its counts to the global ones;
//   layout   one CTA: [start, end) of every tile's list by an exclusive scan of the counts, the
//            work order (longest lists first) and the total;
//   emission (range key << 32 | pair id) into each touched tile's slice: a CTA reserves as many
//            places of each tile as it counted with one atomic and hands them out in shared
//            memory;
//   split    only lists of kListCap entries and more: one CTA, or a cluster, cuts a list by its
//            leading key bits into segments of at most kListCap entries;
//   lists    every list or segment is sorted in shared memory by the 64-bit key, by one warp up
//            to 255 entries, by one CTA above, and written back with each entry's pixel
//            rectangle inside its tile and the 4 x 8 blocks it meets.
// The keys are unique (the pair id is part of them), so the order in which places are handed out
// does not matter: the sorted lists are the same bits in every run.
//
// Why not a global radix sort: sorting all pairs by range and the entries by tile takes four plus
// two passes of three launches each, whose per-tile ranking is one serial chain of shared memory
// per warp; here an entry is written once and read by the list sort, in five launches.  From
// pairs to lists, 12 views x 500 k primitives (5.3 M entries): 0.51 ms in 24 launches -> 0.23 ms
// (count 0.032, layout 0.010, emission 0.067, split 0.030, lists 0.095); 64 tiles of 1,500
// entries: 0.13 -> 0.022 ms.  Counting is bound by instruction issue (68 % of the slots), emission
// by its scattered 8-byte stores (41 %), the list sort by the latency of its gathers (46 %; waits
// for global memory lead its stalls).
// Everything runs on counts that stay on the device, with fixed launch shapes, so the pipeline
// can be captured in a CUDA graph.

#include <cooperative_groups.h>

#include "splat_internal.cuh"

namespace splat {
namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kListThreads = 256, kListCtas = 3;   // CTAs per SM
constexpr int kListWarps = kListThreads / 32;
constexpr int kWarpCap = 256;             // lists below this are sorted by one warp
constexpr int kMaxItems = kListCap / kListThreads;   // 16 keys a thread

// ---------------------------------------------------------------------------------------------
// layout (one CTA)
// ---------------------------------------------------------------------------------------------
constexpr int kLayoutThreads = 1024;

// Four buckets an octave of list length: bucket b holds [bucket_len(b), bucket_len(b + 1)).
constexpr int kBuckets = 128;
__host__ __device__ constexpr int log2_floor(uint32_t x)
{
    int l = 0;
    while (x >>= 1) ++l;
    return l;
}
__device__ __forceinline__ int len_bucket(uint32_t len)
{
    if (len < 4u) return static_cast<int>(len);
    const int l = 31 - __clz(len);
    return 4 * (l - 1) + static_cast<int>(len >> (l - 2) & 3u);
}
constexpr int kMidBucket = 4 * (log2_floor(kWarpCap) - 1);    // lists of kWarpCap and more
constexpr int kLongBucket = 4 * (log2_floor(kListCap) - 1);   // lists of kListCap and more
constexpr int kHugeBucket = 4 * (log2_floor(kHugeList) - 1);
static_assert(kWarpCap == 1 << log2_floor(kWarpCap) && kListCap == 1 << log2_floor(kListCap) &&
                  kHugeList == 1 << log2_floor(kHugeList),
              "bucket bounds");

// exclusive sum over the CTA's threads; *total gets the sum of all
template <int kThreads, typename T>
__device__ __forceinline__ T block_excl_scan(T v, T *s_warp, T *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const T w = lane < kThreads / 32 ? s_warp[lane] : T(0);
        T z = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(kFull, z, o);
            if (lane >= o) z += y;
        }
        if (lane < kThreads / 32) s_warp[lane] = z - w;
        if (lane == 31) s_warp[32] = z;
    }
    __syncthreads();
    if (total) *total = s_warp[32];
    return x - v + s_warp[warp];
}

// Which tiles' blocks the compositing kernels split: with L = 8 entries / warps a warp's even share
// of the frame (in entries of one block's list), lists of at least kSplit2Share L go to two warps a
// block and lists of at least kSplit4Share L to four, both rounded up to a bucket of the work
// order, which the split tiles lead.  Measured, forward / backward in ms, whole | split at 0.4 and
// 0.8 of a share | at 0.7 and 1.2:
//   64x1024, 100 k primitives, longest list 15 shares   .125 .112 | .066 .047 | .066 .048
//   three ragged scans, 83 k, 7 shares                  .102 .100 | .064 .057 | .068 .060
//   four 64x1024, 200 k, 4 shares                       .245 .217 | .154 .150 | .154 .157
//   eight 128x1024 along a street, 3 shares             .446      | .315      | .318
//   128x2048, 1 M, urban block, 2.1 shares              .249 .225 |           | .274 .250
//   12 keyframes, 500 k, 1.8 shares                     .729 .816 |           | .768 .842
// Where even the longest list is below kSplitFrom shares the queue evens the warps out by itself
// and splitting mostly costs, so such a frame is left whole.  The line is taken over random frames
// (rooms, streets, blocks and a city, 1 to 12 views of 32 x 512 to 128 x 2048, 5,000 to 2 M
// primitives, all tile shapes, longest lists of 1 to 12 shares), forward and backward.  Splitting
// against whole blocks, geometric mean of 600 frames by the shares of their longest list: 0.93 at 1
// to 1.5, 0.97 up to 2, 1.02 up to 2.5, 1.11 up to 3, 1.17 up to 4, 1.33 up to 6, 1.63 above.
// Single frames scatter widely about that, so the mean hardly depends on the line (660, against
// the better of both in each: 1.024 splitting all, 1.016 with the line at 2.0, 1.020 at 2.4, 1.024
// at 2.65, 1.031 at 3.0, 1.228 splitting none), but the frames that splitting makes slower do: of
// 600, 149 by more than 3 % without a line, 72 with the line at 2.0, 48 at 2.4, 28 at 2.65, the
// worst by 30, 27, 25 and 16 %.  Each part also adds its own rounded gradient sums.  Hence the
// highest line that costs less than 1 % of the mean.  The longest list is taken exactly: rounded
// up to a bucket the line lay anywhere up to 3.1 shares.
// A split block keeps one contributor record per part and primitive, so nothing is split when the
// record pool might not hold one record for every row of 8 pixels that every pair meets (n_rows
// counts those): the pool then overflows for no frame that it held unsplit.
constexpr float kSplit2Share = 0.4f, kSplit4Share = 0.8f, kSplitFrom = 2.65f;
constexpr uint32_t kSplitLeast = 64;

__global__ void __launch_bounds__(kLayoutThreads) k_layout(
    const uint32_t *__restrict__ tile_count, int64_t n_tiles, int64_t max_pairs,
    uint2 *__restrict__ ranges, uint32_t *__restrict__ order, uint32_t *__restrict__ d_count,
    uint32_t *status, uint32_t *__restrict__ bin, uint32_t warps, uint32_t rec_cap,
    const unsigned long long *n_rows, const RefineStart start)
{
    chain_wait();
    __shared__ unsigned long long s_warp[33];
    __shared__ uint32_t s_cnt[kBuckets], s_off[kBuckets], s_longest;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < kBuckets) s_cnt[tid] = 0;
    if (tid == 0) s_longest = 0;
    __syncthreads();
    // each thread takes a run of consecutive tiles; the loop bounds are uniform so that the
    // whole warp takes part in the matches
    const int64_t per = (n_tiles + kLayoutThreads - 1) / kLayoutThreads;
    const int64_t t0 = per * tid;
    unsigned long long sum = 0;
    uint32_t longest = 0;
    for (int64_t k = 0; k < per; ++k) {
        const bool in = t0 + k < n_tiles;
        const uint32_t len = in ? tile_count[t0 + k] : 0u;
        sum += len;
        longest = max(longest, len);
        const int b = in ? len_bucket(len) : kBuckets;
        const uint32_t peers = __match_any_sync(kFull, b);
        if (in && lane == __ffs(peers) - 1) atomicAdd(&s_cnt[b], __popc(peers));
    }
    longest = __reduce_max_sync(kFull, longest);
    if (lane == 0 && longest) atomicMax(&s_longest, longest);
    unsigned long long total;
    const unsigned long long run0 = block_excl_scan<kLayoutThreads>(sum, s_warp, &total);
    __syncthreads();
    // s_off[b]: tiles in the buckets above b
    const unsigned long long above = block_excl_scan<kLayoutThreads, unsigned long long>(
        tid < kBuckets ? s_cnt[kBuckets - 1 - tid] : 0u, s_warp, nullptr);
    if (tid < kBuckets) s_off[kBuckets - 1 - tid] = static_cast<uint32_t>(above);
    __syncthreads();
    unsigned long long run = run0;
    if (tid == 0) {
        bin[kBinLong] = s_off[kLongBucket - 1];
        bin[kBinHuge] = s_off[kHugeBucket - 1];
        bin[kBinSegments] = 0u;
        bin[kBinQueueSeg] = 0u;
        bin[kBinMid] = s_off[kMidBucket - 1];
        const float share = static_cast<float>(total) * 8.0f / static_cast<float>(warps);
        // tiles of clearly more than x shares
        auto tiles_above = [&](float x) {
            return s_off[len_bucket(max(kSplitLeast, static_cast<uint32_t>(
                                                         fminf(share * x, 2147483647.0f))))];
        };
        uint32_t n4 = tiles_above(kSplit4Share), n2 = tiles_above(kSplit2Share) - n4;
        if (static_cast<float>(s_longest) < share * kSplitFrom) n4 = n2 = 0u;
        const unsigned long long items =
            8ull * (static_cast<unsigned long long>(n_tiles) + n2 + 3ull * n4);
        if (rec_cap && *n_rows / 32 + items > rec_cap) n4 = n2 = 0u;
        bin[kBinSplit4] = n4;
        bin[kBinSplit2] = n2;
        if (start.queue) *start.queue = 0u;
        if (start.evals) *start.evals = 0ull;
        if (start.loss) *start.loss = 0.0;
        if (start.step) *start.step += 1;
        const bool over = total > static_cast<unsigned long long>(max_pairs);
        bin[kBinOver] = over ? 1u : 0u;
        if (over) atomicOr(status, SPLAT_STATUS_CAPACITY);
        *d_count = static_cast<uint32_t>(over ? max_pairs : static_cast<int64_t>(total));
    }
    for (int k = tid; k < start.n_pose; k += kLayoutThreads) start.pose[k] = 0.0f;
    __syncthreads();
    // past the capacity a list keeps the places below it (the status bit marks the result)
    const unsigned long long cap = static_cast<unsigned long long>(max_pairs);
    for (int64_t k = 0; k < per; ++k) {
        const bool in = t0 + k < n_tiles;
        const uint32_t len = in ? tile_count[t0 + k] : 0u;
        const int b = in ? len_bucket(len) : kBuckets;
        const uint32_t peers = __match_any_sync(kFull, b);
        const int lead = __ffs(peers) - 1;
        uint32_t at = 0;
        if (in && lane == lead) at = atomicAdd(&s_off[b], __popc(peers));
        at = __shfl_sync(kFull, at, lead) + __popc(peers & ((1u << lane) - 1u));
        if (in) {
            order[at] = static_cast<uint32_t>(t0 + k);
            const unsigned long long e = run + len;
            ranges[t0 + k] = len == 0 ? make_uint2(0u, 0u)
                                      : make_uint2(static_cast<uint32_t>(run < cap ? run : cap),
                                                   static_cast<uint32_t>(e < cap ? e : cap));
            run = e;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// count and emission: a CTA takes a chunk of one view's touching pairs and a band of its tiles
// ---------------------------------------------------------------------------------------------
constexpr int kChunkThreads = 512;

struct Chunk {
    int view;
    const uint2 *touch;
    const float *kappa;
    const uint32_t *touch_count;
    int begin, end;        // units of 32 places: unit u is places 32 u .. of the view
    int unit_shift;        // log2 of the units a block
    int tiles_c;
    int row0, rows;        // the band's tile rows
    int n_tiles;           // and tiles, which the three arrays below begin with
    uint32_t *tile_count;
    uint32_t *cta_count;   // this CTA's count of every tile of the band
    const uint2 *ranges;
};

// The chunk of this CTA; false when its view is not drawn.  kBanded: at least one view has more
// than one band.
template <bool kBanded>
__device__ __forceinline__ bool chunk_of(const BinArgs &A, Chunk &c)
{
    int v = 0, band = 0, row = 0;   // row: rank of the band among those of the drawn views
    if (kBanded) {
        band = blockIdx.y;
        for (;; ++v) {
            const int nb = view_bands(A.views[v].tiles_r, A.views[v].tiles_c);
            if (band < nb) break;
            band -= nb;
            if (!A.active || A.active[v]) row += nb;
        }
        row += band;
    } else {
        v = row = blockIdx.y;
        if (A.active) {
            row = 0;
            for (int k = 0; k < v; ++k) row += A.active[k] ? 1 : 0;
        }
    }
    if (A.active && !A.active[v]) return false;
    const ViewDesc &vd = A.views[v];
    const int64_t p0 = static_cast<int64_t>(v) * A.n;
    const int first = A.chunk * static_cast<int>(blockIdx.x);
    c.view = v;
    c.touch = A.touch + p0;
    c.kappa = A.kappa + p0;
    c.touch_count = A.touch_count + static_cast<int64_t>(v) * A.blocks;
    c.unit_shift = __ffs(A.block_prims) - 1 - 5;   // block_prims is a power of two
    c.begin = first << c.unit_shift;
    c.end = min(first + A.chunk, A.blocks) << c.unit_shift;
    c.tiles_c = vd.tiles_c;
    c.row0 = kBanded ? band * band_rows(vd.tiles_c) : 0;
    c.rows = kBanded ? min(vd.tiles_r - c.row0, band_rows(vd.tiles_c)) : vd.tiles_r;
    c.n_tiles = c.rows * vd.tiles_c;
    const int64_t t0 = vd.tile_offset + static_cast<int64_t>(c.row0) * vd.tiles_c;
    c.tile_count = A.tile_count + t0;
    c.cta_count = A.cta_count +
                  (static_cast<int64_t>(row) * gridDim.x + blockIdx.x) * A.max_band_tiles;
    c.ranges = A.ranges + t0;
    return true;
}

// f(tile of the band, range key bits, primitive in the view) for every tile of the band of every
// touching pair of the chunk, 32 pairs a warp at a time, kUnitLoads of them read ahead (the range
// keys only with kKeys).  While no pair of a warp touches more than kLaneTiles tiles, every lane
// walks its own; otherwise the warp numbers the tiles of its 32 pairs by a prefix sum and gives one
// to every lane, so that one wide pair costs its warp no more than as many narrow ones.
constexpr int kLaneTiles = 8, kUnitLoads = 4;

template <bool kBanded, bool kKeys, typename F>
__device__ __forceinline__ void for_each_entry(const Chunk &c, F f)
{
    const int lane = threadIdx.x & 31;
    const uint32_t tiles_c = static_cast<uint32_t>(c.tiles_c);
    constexpr int kWarps = kChunkThreads / 32;
    for (int u0 = c.begin + static_cast<int>(threadIdx.x >> 5); u0 < c.end;
         u0 += kWarps * kUnitLoads) {
        uint32_t live[kUnitLoads];   // the unit's pairs
        uint2 word[kUnitLoads];
        uint32_t keys[kUnitLoads];
#pragma unroll
        for (int i = 0; i < kUnitLoads; ++i) {
            const int u = u0 + i * kWarps;
            const uint32_t n = u < c.end ? c.touch_count[u >> c.unit_shift] : 0u;
            const uint32_t b = static_cast<uint32_t>(u - (u >> c.unit_shift << c.unit_shift)) * 32u;
            live[i] = n > b ? n - b : 0u;
        }
#pragma unroll
        for (int i = 0; i < kUnitLoads; ++i) {
            const int64_t at = 32 * static_cast<int64_t>(u0 + i * kWarps) + lane;
            const bool in = static_cast<uint32_t>(lane) < live[i];
            word[i] = in ? c.touch[at] : make_uint2(0u, 0u);
            keys[i] = kKeys && in ? __float_as_uint(c.kappa[at]) : 0u;
        }
#pragma unroll 1
        for (int i = 0; i < kUnitLoads; ++i) {
            if (live[i] == 0u) continue;
            const int u = u0 + i * kWarps;
            const uint32_t first = 32u * static_cast<uint32_t>(u >> c.unit_shift << c.unit_shift);
            TileRect t{};
            uint32_t local = 0, cnt = 0;
            if (static_cast<uint32_t>(lane) < live[i]) {
                t = unpack_touch(word[i], local);
                if (kBanded) {   // the part inside the band
                    const int r0 = max(t.r0 - c.row0, 0);
                    t.nr = max(min(t.r0 - c.row0 + t.nr, c.rows) - r0, 0);
                    t.r0 = r0;
                }
                cnt = static_cast<uint32_t>(t.nr) * static_cast<uint32_t>(t.nc);
            }
            if (!__any_sync(kFull, cnt > kLaneTiles)) {
                uint32_t row = static_cast<uint32_t>(t.r0) * tiles_c;
                uint32_t col = static_cast<uint32_t>(t.c0);
                int left = t.nc;
                for (uint32_t k = 0; k < cnt; ++k) {
                    f(row + col, keys[i], first + local);
                    col = col + 1 == tiles_c ? 0u : col + 1;
                    if (--left == 0) {   // the next tile row
                        left = t.nc;
                        col = static_cast<uint32_t>(t.c0);
                        row += tiles_c;
                    }
                }
                continue;
            }
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(kFull, incl, 31);
            const uint32_t rc = static_cast<uint32_t>(t.r0) | static_cast<uint32_t>(t.c0) << 16;
            const uint32_t cl = static_cast<uint32_t>(t.nc) | local << 16;
            for (uint32_t q0 = 0; q0 < total; q0 += 32) {
                const uint32_t q = q0 + lane;
                int src = 0;   // the first lane whose run ends after q
#pragma unroll
                for (int s = 16; s > 0; s >>= 1)
                    if (__shfl_sync(kFull, incl, src + s - 1) <= q) src += s;
                const uint32_t k = q - __shfl_sync(kFull, incl - cnt, src);
                const uint32_t r = __shfl_sync(kFull, rc, src), m = __shfl_sync(kFull, cl, src);
                const uint32_t key = kKeys ? __shfl_sync(kFull, keys[i], src) : 0u;
                if (q < total) {
                    const uint32_t nc = m & 0xFFFFu, row = k / nc;
                    uint32_t col = (r >> 16) + (k - row * nc);
                    col = col >= tiles_c ? col - tiles_c : col;
                    f(((r & 0xFFFFu) + row) * tiles_c + col, key, first + (m >> 16));
                }
            }
        }
    }
}

// Counted in shared memory, a tile sees one global atomic per CTA instead of one per entry:
// neighbouring threads' pairs fall on a few hundred tiles of one view, and same-address atomics
// in L2 serialise (emission of 5.3 M entries: 0.95 ms with an atomic per entry).  A view of more
// tiles than the counters hold is taken in bands, each by its own CTAs, which pass over the pairs
// that miss their band: eleven 64 x 1024 views and one of 128 x 32,000 over 500 k primitives (11.6
// M entries), counted and emitted with global atomics 0.63 ms, in bands 0.29; the wide view alone
// (16,000 tiles, 6.2 M entries) 0.13 either way.
template <bool kBanded>
__global__ void __launch_bounds__(kChunkThreads) k_count(const BinArgs A)
{
    chain_wait();
    extern __shared__ uint32_t s_cnt[];
    Chunk c;
    if (!chunk_of<kBanded>(A, c)) return;
    for (int t = threadIdx.x; t < c.n_tiles; t += kChunkThreads) s_cnt[t] = 0u;
    __syncthreads();
    for_each_entry<kBanded, false>(
        c, [&](uint32_t t, uint32_t, uint32_t) { atomicAdd(s_cnt + t, 1u); });
    __syncthreads();
    for (int t = threadIdx.x; t < c.n_tiles; t += kChunkThreads) {
        const uint32_t n = s_cnt[t];
        if (n) atomicAdd(c.tile_count + t, n);
        c.cta_count[t] = n;
    }
}

template <bool kBanded>
__global__ void __launch_bounds__(kChunkThreads) k_emit(const BinArgs A)
{
    chain_wait();
    extern __shared__ uint32_t s_cnt[];
    Chunk c;
    if (!chunk_of<kBanded>(A, c)) return;
    // (a frame past its capacity checks every place against its list's end)
    const bool over = A.bin[kBinOver] != 0u;
    for (int t = threadIdx.x; t < c.n_tiles; t += kChunkThreads) {
        const uint32_t n = c.cta_count[t];   // the tile's count counts down: this CTA takes n
        if (n) s_cnt[t] = atomicSub(c.tile_count + t, n) - n + (over ? 0u : c.ranges[t].x);
    }
    __syncthreads();
    const uint32_t p0 = static_cast<uint32_t>(static_cast<int64_t>(c.view) * A.n);
    if (!over) {
        for_each_entry<kBanded, true>(c, [&](uint32_t t, uint32_t key, uint32_t i) {
            A.entries[atomicAdd(s_cnt + t, 1u)] = static_cast<uint64_t>(key) << 32 | (p0 + i);
        });
        return;
    }
    for_each_entry<kBanded, true>(c, [&](uint32_t t, uint32_t key, uint32_t i) {
        const uint32_t k = atomicAdd(s_cnt + t, 1u);
        const uint2 rg = c.ranges[t];
        if (k < rg.y - rg.x) A.entries[rg.x + k] = static_cast<uint64_t>(key) << 32 | (p0 + i);
    });
}

// ---------------------------------------------------------------------------------------------
// long lists: cut into segments by the leading key bits
// ---------------------------------------------------------------------------------------------
constexpr int kSplitThreads = 1024;
constexpr int kSplitBits = 12, kSplitBins = 1 << kSplitBits;
constexpr int kBinsPer = kSplitBins / kSplitThreads;

// f(key) for the keys src[0 .. n), kSplitLoads loads in flight a thread
constexpr int kSplitLoads = 8;
template <typename F>
__device__ __forceinline__ void for_each_key(const uint64_t *src, uint32_t n, F f)
{
    for (uint32_t b = 0; b < n; b += kSplitThreads * kSplitLoads) {
        uint64_t k[kSplitLoads];
#pragma unroll
        for (int u = 0; u < kSplitLoads; ++u) {
            const uint32_t j = b + u * kSplitThreads + threadIdx.x;
            k[u] = j < n ? src[j] : ~0ull;
        }
#pragma unroll
        for (int u = 0; u < kSplitLoads; ++u)
            if (b + u * kSplitThreads + threadIdx.x < n) f(k[u]);
    }
}

struct SplitShared {
    uint32_t bin[kSplitBins];         // this CTA's count of every bin, then its cursor
    uint32_t start[kSplitBins + 1];   // the bins' first places, then the segments'
    uint32_t warp[33];
    uint32_t base, next;
    unsigned long long lo[32], hi[32];   // smallest and largest key by warp
};

// The CTAs that cut one list, each with a slice of the keys: this one, or all of its cluster.
struct OneCta {
    static constexpr uint32_t ranks = 1, rank = 0;
    __device__ void sync() const { __syncthreads(); }
    template <typename T>
    __device__ T *of(T *shared, uint32_t) const { return shared; }
};
struct WholeCluster {
    uint32_t ranks, rank;
    __device__ void sync() const { cooperative_groups::this_cluster().sync(); }
    template <typename T>
    __device__ T *of(T *shared, uint32_t r) const
    {
        return cooperative_groups::this_cluster().map_shared_rank(shared, r);
    }
};

struct SegmentRun {
    uint32_t begin, end;   // places in A.segments
    bool oversized;        // at least one of them holds more than kListCap entries
};

// smallest lo and largest hi of the warp
__device__ __forceinline__ void warp_range(unsigned long long &lo, unsigned long long &hi)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(kFull, lo, o);
        const unsigned long long y = __shfl_xor_sync(kFull, hi, o);
        lo = x < lo ? x : lo;
        hi = y > hi ? y : hi;
    }
}

// Cuts the keys [start, start + len) of the buffer that `level` reads: a histogram over bins, bins
// gathered into segments of at most kListCap entries by the kSegTarget-entry stretch of the keys
// their first entry falls into, and the keys scattered by bin into the other buffer.  A segment
// above kListCap is a single bin.  The bins are linear in the keys' bits, which for floats spaces
// them like the logarithm: with kExact between the smallest and the largest key, which takes one
// more pass over them, else 128 an octave of range from 2^-12 on (the ends take what lies beyond).
// Bound by the latency of those passes and of the barriers between them, one CTA an SM.
template <bool kExact, typename Group>
__device__ __forceinline__ SegmentRun cut(const BinArgs &A, uint32_t start, uint32_t len,
                                          uint32_t tile, int level, SplitShared &sh, const Group &g)
{
    const int tid = threadIdx.x;
    const uint32_t s0 = static_cast<uint32_t>(uint64_t{len} * g.rank / g.ranks);
    const uint32_t n = static_cast<uint32_t>(uint64_t{len} * (g.rank + 1) / g.ranks) - s0;
    const uint64_t *src = (level & 1 ? A.entries2 : A.entries) + start + s0;
    uint64_t *dst = (level & 1 ? A.entries : A.entries2) + start;
    for (int k = tid; k < kSplitBins; k += kSplitThreads) sh.bin[k] = 0u;
    unsigned long long lo = 0ull;
    int down = 0;
    if constexpr (kExact) {
        unsigned long long hi = 0ull;
        lo = ~0ull;
        for_each_key(src, n, [&](uint64_t e) {
            lo = e < lo ? e : lo;
            hi = e > hi ? e : hi;
        });
        warp_range(lo, hi);
        if ((tid & 31) == 0) {
            sh.lo[tid >> 5] = lo;
            sh.hi[tid >> 5] = hi;
        }
        g.sync();
        for (uint32_t r = 0; r < g.ranks; ++r) {
            const unsigned long long x = g.of(sh.lo, r)[tid & 31], y = g.of(sh.hi, r)[tid & 31];
            lo = x < lo ? x : lo;
            hi = y > hi ? y : hi;
        }
        warp_range(lo, hi);
        down = max(0, 64 - __clzll(hi - lo) - kSplitBits);
    } else {
        __syncthreads();
    }
    auto bin = [=](uint64_t e) -> uint32_t {
        if constexpr (kExact) return static_cast<uint32_t>((e - lo) >> down);
        const int b = static_cast<int>(e >> 48) - ((127 - 12) << 7);
        return static_cast<uint32_t>(min(max(b, 0), kSplitBins - 1));
    };
    for_each_key(src, n, [&](uint64_t e) { atomicAdd(&sh.bin[bin(e)], 1u); });
    g.sync();
    uint32_t c[kBinsPer] = {}, below[kBinsPer] = {}, sum = 0;   // of all ranks, of lower ranks
    for (uint32_t r = 0; r < g.ranks; ++r) {
        const uint32_t *counts = g.of(sh.bin, r);
#pragma unroll
        for (int i = 0; i < kBinsPer; ++i) {
            const uint32_t m = counts[tid * kBinsPer + i];
            c[i] += m;
            below[i] += r < g.rank ? m : 0u;
        }
    }
    uint32_t longest = 0;
#pragma unroll
    for (int i = 0; i < kBinsPer; ++i) {
        sum += c[i];
        longest = max(longest, c[i]);
    }
    uint32_t at = block_excl_scan<kSplitThreads>(sum, sh.warp, static_cast<uint32_t *>(nullptr));
    uint32_t pre[kBinsPer];
#pragma unroll
    for (int i = 0; i < kBinsPer; ++i) {
        pre[i] = at;
        sh.start[tid * kBinsPer + i] = at;
        at += c[i];
    }
    const bool oversized = __syncthreads_or(longest > kListCap);
    // a segment starts at every bin whose first entry lies in another kSegTarget stretch than the
    // previous bin's (so also after every bin above kSegTarget), and at a bin that would take the
    // segment of its stretch above kListCap
    uint32_t first[kBinsPer], ns = 0;
#pragma unroll
    for (int i = 0; i < kBinsPer; ++i) {
        const int b = tid * kBinsPer + i;
        const uint32_t before = b == 0 ? 0u : (i > 0 ? pre[i - 1] : sh.start[b - 1]);
        first[i] = pre[i] < len && (b == 0 || pre[i] / kSegTarget != before / kSegTarget ||
                                    pre[i] % kSegTarget + c[i] > kListCap)
                       ? 1u : 0u;
        ns += first[i];
    }
    uint32_t n_seg;
    uint32_t q = block_excl_scan<kSplitThreads>(ns, sh.warp, &n_seg);
    g.sync();   // the counts and the bins' places have been read by all
#pragma unroll
    for (int i = 0; i < kBinsPer; ++i) {
        sh.bin[tid * kBinsPer + i] = pre[i] + below[i];
        if (first[i]) sh.start[q++] = pre[i];
    }
    if (tid == 0) {
        sh.start[n_seg] = len;
        if (g.rank == 0) sh.base = atomicAdd(A.bin + kBinSegments, n_seg);
    }
    __syncthreads();
    for_each_key(src, n, [&](uint64_t e) { dst[atomicAdd(&sh.bin[bin(e)], 1u)] = e; });
    g.sync();   // sh.base
    const uint32_t base = *g.of(&sh.base, 0);
    if (g.rank == 0)
        for (uint32_t k = tid; k < n_seg; k += kSplitThreads)
            A.segments[base + k] = ListSegment{start + sh.start[k], sh.start[k + 1] - sh.start[k],
                                               tile, static_cast<uint32_t>(level & 1)};
    g.sync();   // keys and segments are written, and no rank reads another's memory any more
    return SegmentRun{base, base + n_seg, oversized};
}

// Cuts the segments of `run`, left by a cut at `level`, again until none holds more than kListCap
// entries, depth first, by this CTA alone; it takes every ranks-th of the run.
template <typename Group>
__device__ __noinline__ void recut(const BinArgs &A, SegmentRun run, uint32_t tile, int level,
                                   SplitShared &sh, const Group &g)
{
    uint32_t next[kSplitLevels], end[kSplitLevels];   // by level: segments not yet looked at
    const int first = level;
    next[level] = run.begin;
    end[level] = run.oversized ? run.end : run.begin;
    while (level >= first) {
        // the level's next oversized segment
        if (threadIdx.x == 0) sh.next = kFull;
        __syncthreads();
        uint32_t at = kFull;
        for (uint32_t k0 = next[level]; k0 < end[level] && at == kFull; k0 += kSplitThreads) {
            const uint32_t k = k0 + threadIdx.x;
            if (k < end[level] && (level > first || k % g.ranks == g.rank) &&
                __ldcg(&A.segments[k].len) > kListCap)
                atomicMin(&sh.next, k);
            __syncthreads();
            at = sh.next;
            __syncthreads();   // read by all before the next writes
        }
        if (at == kFull || level + 1 == kSplitLevels) {
            --level;
            continue;
        }
        next[level] = at + 1;
        const uint32_t start = __ldcg(&A.segments[at].start), len = __ldcg(&A.segments[at].len);
        ++level;
        run = cut<true>(A, start, len, tile, level, sh, OneCta{});
        if (threadIdx.x == 0) A.segments[at].len = 0u;   // read by all before the cut
        next[level] = run.begin;
        end[level] = run.oversized ? run.end : run.begin;
    }
}

// Cuts one list until no segment is above kListCap.  The first cut of a list that one CTA cuts
// takes the fixed bins, where few lists of that length have more than kListCap entries in a bin;
// what is oversized after it (a wall at one distance, a dense map) is cut again, exactly.  An
// oversized segment is one bin, and a bin of an exact cut spans at most 2^-11 of the keys' range:
// keys have 63 bits at most and are unique, so that the bins of the fifth exact cut span no more
// than 8 keys.
// A cluster cuts exactly from the start, goes on as one while more than half of the list stays in
// one segment, and shares the rest out to its CTAs.
// What the exact pass costs a list of 5,000 or 20,000 entries on one CTA: 4 us on 4.5 and 18.  What
// it saves: 150,000 primitives of one tile within 0.1 mm of range, cut and sorted, 0.105 ms; left
// in one segment and merged by one CTA 2.99.
__device__ void split_list(const BinArgs &A, uint32_t tile, SplitShared &sh)
{
    const uint2 rg = A.ranges[tile];
    const SegmentRun run = cut<false>(A, rg.x, rg.y - rg.x, tile, 0, sh, OneCta{});
    if (run.oversized) recut(A, run, tile, 0, sh, OneCta{});
}

__device__ void split_list(const BinArgs &A, uint32_t tile, SplitShared &sh, const WholeCluster &g)
{
    const uint2 rg = A.ranges[tile];
    uint32_t start = rg.x, len = rg.y - rg.x;
    for (int level = 0;; ++level) {
        const SegmentRun run = cut<true>(A, start, len, tile, level, sh, g);
        if (!run.oversized) return;
        // a huge segment that the cluster goes on with
        uint32_t at = kFull;
        if (level + 1 < kSplitLevels) {
            if (threadIdx.x == 0) sh.next = kFull;
            __syncthreads();
            for (uint32_t k = run.begin + threadIdx.x; k < run.end; k += kSplitThreads) {
                const uint32_t m = __ldcg(&A.segments[k].len);
                if (m > len / 2 && m >= kHugeList) sh.next = k;   // there is one at most
            }
            __syncthreads();
            at = sh.next;
            if (at != kFull) {
                start = __ldcg(&A.segments[at].start);
                len = __ldcg(&A.segments[at].len);
            }
            g.sync();   // read by all ranks
            if (at != kFull && g.rank == 0 && threadIdx.x == 0) A.segments[at].len = 0u;
            g.sync();
        }
        recut(A, run, tile, level, sh, g);
        if (at == kFull) return;
        __syncthreads();
    }
}

// Launched in clusters when lists of kHugeList entries can occur: those are cut by a whole cluster
// each, the others by one CTA each.
__global__ void __launch_bounds__(kSplitThreads) k_split(const BinArgs A)
{
    chain_wait();
    __shared__ SplitShared sh;
    const auto cluster = cooperative_groups::this_cluster();
    const WholeCluster all{cluster.num_blocks(), cluster.block_rank()};
    const uint32_t n_long = A.bin[kBinLong], n_huge = all.ranks > 1 ? A.bin[kBinHuge] : 0u;
    for (uint32_t l = blockIdx.x / all.ranks; l < n_huge; l += gridDim.x / all.ranks)
        split_list(A, A.order[l], sh, all);
    // the longest of the others first to the CTAs that had no part in a huge one
    const uint32_t busy = min(n_huge * all.ranks, gridDim.x);
    const uint32_t place = blockIdx.x < busy ? blockIdx.x + gridDim.x - busy : blockIdx.x - busy;
    for (uint32_t l = n_huge + place; l < n_long; l += gridDim.x) {
        split_list(A, A.order[l], sh);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// list sort
// ---------------------------------------------------------------------------------------------

// one spare word per 16 keys: threads that walk runs a power of two apart spread over the banks
__device__ __forceinline__ int pad(int i) { return i + (i >> 4); }

template <int G>
__device__ __forceinline__ void group_sync()
{
    if (G == 32) __syncwarp();
    else __syncthreads();
}

__device__ __forceinline__ void order_pair(uint64_t &a, uint64_t &b)
{
    const uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort (Sorting networks and their applications, 1968) of E keys in
// registers: phase p merges sorted runs of p keys, in steps of comparison distance q = p, p / 2,
// ..., 1
template <int E, int P, int Q>
__device__ __forceinline__ void network(uint64_t (&k)[E])
{
    if constexpr (P < E) {
#pragma unroll
        for (int i = 0; i + Q < E; ++i)
            if (i >= Q % P && (i - Q % P) / Q % 2 == 0 && i / (2 * P) == (i + Q) / (2 * P))
                order_pair(k[i], k[i + Q]);
        if constexpr (Q > 1) network<E, P, Q / 2>(k);
        else network<E, 2 * P, 2 * P>(k);
    }
}

// Sorts the n <= G * E keys src[0 .. n) into s (padded places), with G threads (a warp or the
// CTA) of E keys each: every thread sorts its keys in registers (network), then
// runs of E, 2E, ... keys are merged pairwise, each thread finding its E outputs by a binary
// search along its diagonal (merge path: Odeh, Green, Mwassi, Shmueli, Birk 2012).
template <int E, int G>
__device__ __forceinline__ void sort_keys(const uint64_t *src, int n, uint64_t *s, int g)
{
    uint64_t k[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {   // coalesced read, then each thread's own run
        const int j = g + i * G;
        if (j < n) s[pad(j)] = src[j];
    }
    group_sync<G>();
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int j = g * E + i;
        k[i] = j < n ? s[pad(j)] : ~0ull;
    }
    network<E, 1, 1>(k);
    group_sync<G>();
#pragma unroll
    for (int i = 0; i < E; ++i) s[pad(g * E + i)] = k[i];
    group_sync<G>();
    for (int w = E; w < n; w <<= 1) {
        const int base = (g * E) & ~(2 * w - 1), diag = g * E - base;
        if (base + w < n) {   // otherwise the run has no partner and stays
            const int a0 = base, b0 = base + w;
            int lo = diag > w ? diag - w : 0, hi = diag < w ? diag : w;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s[pad(a0 + mid)] < s[pad(b0 + diag - 1 - mid)]) lo = mid + 1;
                else hi = mid;
            }
            int i = lo, j = diag - lo;
            uint64_t a = i < w ? s[pad(a0 + i)] : ~0ull, b = j < w ? s[pad(b0 + j)] : ~0ull;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const bool left = a < b || j >= w;
                k[e] = left ? a : b;
                if (left) {
                    ++i;
                    a = i < w ? s[pad(a0 + i)] : ~0ull;
                } else {
                    ++j;
                    b = j < w ? s[pad(b0 + j)] : ~0ull;
                }
            }
        }
        group_sync<G>();
        if (base + w < n) {
#pragma unroll
            for (int e = 0; e < E; ++e) s[pad(g * E + e)] = k[e];
        }
        group_sync<G>();
    }
}

// an entry of the list: pair id, pixel rectangle inside the tile, blocks met
struct ListTile {
    int rb, cb, cols;   // the tile's first row and column, the image's width
};

__device__ __forceinline__ uint32_t entry_rect(const BinArgs &A, uint64_t word, const ListTile &t)
{
    return tile_local_rect(unpack_pixel_rect(word), t.rb, t.cb, t.cols, A.tile_h, A.tile_w);
}

__device__ __forceinline__ void write_entry(const BinArgs &A, uint32_t at, uint32_t p, uint32_t r)
{
    reinterpret_cast<uint2 *>(A.entries)[at] = make_uint2(p, r);
    A.entry_blocks[at] =
        static_cast<uint8_t>(rect_blocks(r & ~kRectFlip, A.tile_h, A.tile_w));
}

__device__ __forceinline__ ListTile list_tile(const BinArgs &A, uint32_t tile)
{
    const TileInfo &ti = A.tiles[tile];
    return ListTile{ti.tr * A.tile_h, ti.tc * A.tile_w, ti.cols};
}

// bins of a list: two to four a key, 16-bit counters in pairs
constexpr int kMaxBins = 2 * kListCap;
// lists with a bin above this are merge sorted: an entry is compared with its whole bin
constexpr int kMaxInBin = 32;

struct ListShared {
    uint64_t key[kListCap + kListCap / 16];
    uint32_t bins[kMaxBins / 2 + kMaxBins / 64];
    uint32_t item, lo, hi, worst;
    uint32_t warp[33];
};

static_assert(kListWarps * (kWarpCap + kWarpCap / 16) <= kListCap + kListCap / 16 &&
                  kListWarps * (kWarpCap + kWarpCap / 32) <= kMaxBins / 2 + kMaxBins / 64,
              "the warps' slices lie inside the CTA's arrays");

// place of a counter word: one spare per 32, so that threads scanning runs of words spread over
// the banks
__device__ __forceinline__ uint32_t bin_word(uint32_t w) { return w + (w >> 5); }

// exclusive scan of the 16-bit counters packed two to a word, in place, by a group of G threads
template <int G>
__device__ __forceinline__ uint32_t scan_bins(uint32_t *bins, int words, uint32_t *s_warp, int g)
{
    // each thread takes a run of consecutive words; returns the largest counter it saw
    const int per = (words + G - 1) / G;
    uint32_t sum = 0, worst = 0;
    for (int i = 0; i < per; ++i) {
        const int w = g * per + i;
        if (w < words) {
            const uint32_t c = bins[bin_word(w)], a = c & 0xFFFFu, b = c >> 16;
            sum += a + b;
            worst = max(worst, max(a, b));
        }
    }
    uint32_t at;
    if (G == 32) {
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, x, o);
            if (g >= o) x += y;
        }
        at = x - sum;
    } else {
        at = block_excl_scan<G>(sum, s_warp, static_cast<uint32_t *>(nullptr));
    }
    for (int i = 0; i < per; ++i) {
        const int w = g * per + i;
        if (w < words) {
            const uint32_t c = bins[bin_word(w)], a = c & 0xFFFFu, b = c >> 16;
            bins[bin_word(w)] = at | (at + a) << 16;
            at += a + b;
        }
    }
    return worst;
}

__device__ __forceinline__ uint32_t add_bin(uint32_t *bins, uint32_t b)
{
    const int sh = (b & 1u) << 4;
    return (atomicAdd(bins + bin_word(b >> 1), 1u << sh) >> sh) & 0xFFFFu;
}

__device__ __forceinline__ uint32_t get_bin(const uint32_t *bins, uint32_t b)
{
    return (bins[bin_word(b >> 1)] >> ((b & 1u) << 4)) & 0xFFFFu;
}

// Sorts one list of n keys and writes its entries, with a group of G threads (a warp or the CTA).
// The keys go into two to four bins a key, linear in the range key's bits between the list's
// smallest and largest (floats of one sign order as integers), are laid out by bin, and each is
// then ranked against the other keys of its bin -- one or two on lists whose ranges spread.  A
// list with a bin above kMaxInBin (a wall behind a near object) is merge sorted.  The keys are
// read three times rather than held: they stay in L1, and short loops keep the code in the
// instruction cache.  24 warps with 52 KB a CTA leave a third of an SM's memory to L1, which bounds
// the misses in flight: with the rectangles gathered into shared memory as well (68 KB a CTA) the
// stage took 0.178 ms instead of 0.121 on 5.3 M entries, with four CTAs per SM 0.157.
template <int G>
__device__ __forceinline__ void sort_list(const BinArgs &A, const uint64_t *src, uint32_t start,
                                          int n, uint32_t tile, uint64_t *key,
                                          uint32_t *bins, ListShared &sh, int g)
{
    src += start;
    const int log_bins = min(32 - __clz(n) + 1, G == 32 ? 9 : 13);
    const int words = 1 << (log_bins - 1);
    for (int w = g; w < words; w += G) bins[bin_word(w)] = 0u;
    const uint32_t *hi_word = reinterpret_cast<const uint32_t *>(src) + 1;   // the range keys
    uint32_t lo = kFull, hi = 0u;
#pragma unroll 4
    for (int j = g; j < n; j += G) {
        const uint32_t k = hi_word[2 * j];
        lo = min(lo, k);
        hi = max(hi, k);
    }
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    if (G > 32) {
        if (g == 0) {
            sh.lo = kFull;
            sh.hi = 0u;
            sh.worst = 0u;
        }
        __syncthreads();
        if ((g & 31) == 0) {
            atomicMin(&sh.lo, lo);
            atomicMax(&sh.hi, hi);
        }
        __syncthreads();
        lo = sh.lo;
        hi = sh.hi;
    } else {
        __syncwarp();
    }
    const int down = max(0, 32 - __clz(hi - lo) - log_bins);
#pragma unroll 4
    for (int j = g; j < n; j += G) add_bin(bins, (hi_word[2 * j] - lo) >> down);
    group_sync<G>();
    uint32_t worst = __reduce_max_sync(kFull, scan_bins<G>(bins, words, sh.warp, g));
    if (G > 32) {
        if ((g & 31) == 0) atomicMax(&sh.worst, worst);
        __syncthreads();
        worst = sh.worst;
    } else {
        __syncwarp();
    }
    const ListTile t = list_tile(A, tile);
    if (worst <= kMaxInBin) {
#pragma unroll 4
        for (int j = g; j < n; j += G) {
            const uint64_t k = src[j];
            key[add_bin(bins, (static_cast<uint32_t>(k >> 32) - lo) >> down)] = k;
        }
        group_sync<G>();   // every counter now stands at its bin's end
        for (int j = g; j < n; j += G) {
            const uint64_t k = key[j];
            const uint64_t word = A.prect[static_cast<uint32_t>(k)];
            const uint32_t b = (static_cast<uint32_t>(k >> 32) - lo) >> down;
            const int b0 = b == 0 ? 0 : static_cast<int>(get_bin(bins, b - 1));
            const int b1 = static_cast<int>(get_bin(bins, b));
            int at = b0;
            if (b1 - b0 > 1)
                for (int q = b0; q < b1; ++q) at += key[q] < k ? 1 : 0;
            write_entry(A, start + at, static_cast<uint32_t>(k), entry_rect(A, word, t));
        }
    } else {
        constexpr int E = G == 32 ? kWarpCap / 32 : kMaxItems;
        sort_keys<E, G>(src, n, key, g);
        for (int j = g; j < n; j += G) {
            const uint32_t p = static_cast<uint32_t>(key[pad(j)]);
            write_entry(A, start + j, p, entry_rect(A, A.prect[p], t));
        }
    }
    group_sync<G>();
}

// Persistent: the CTAs take segments and lists of 256 entries and more, longest first; then their
// warps take the shorter lists.
__global__ void __launch_bounds__(kListThreads, kListCtas) k_lists(const BinArgs A)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char s_raw[];
    ListShared &sh = *reinterpret_cast<ListShared *>(s_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n_long = A.bin[kBinLong], n_seg = A.bin[kBinSegments];
    const uint32_t n_mid = A.bin[kBinMid];
    const uint32_t n_cta = n_seg + (n_mid - n_long);
    for (uint32_t item = blockIdx.x; item < n_cta;) {
        ListSegment sg;
        const uint64_t *src = A.entries;
        if (item < n_seg) {
            sg = A.segments[item];
            if (!sg.in_entries) src = A.entries2;
        } else {
            sg.tile = A.order[n_long + item - n_seg];
            const uint2 rg = A.ranges[sg.tile];
            sg.start = rg.x;
            sg.len = rg.y - rg.x;
        }
        if (sg.len > 0 && sg.len <= kListCap)
            sort_list<kListThreads>(A, src, sg.start, static_cast<int>(sg.len), sg.tile, sh.key,
                                    sh.bins, sh, tid);
        if (tid == 0) sh.item = atomicAdd(A.bin + kBinQueueSeg, 1u) + gridDim.x;
        __syncthreads();
        item = sh.item;
        __syncthreads();
    }
    uint64_t *key = sh.key + warp * (kWarpCap + kWarpCap / 16);
    uint32_t *bins = sh.bins + warp * (kWarpCap + kWarpCap / 32);
    for (uint32_t item = n_mid + blockIdx.x * kListWarps + warp; item < A.n_tiles;
         item += gridDim.x * kListWarps) {
        const uint32_t tile = A.order[item];
        const uint2 rg = A.ranges[tile];
        if (rg.y > rg.x)
            sort_list<32>(A, A.entries, rg.x, static_cast<int>(rg.y - rg.x), tile, key, bins, sh,
                          lane);
    }
}

// blocks a CTA counts or emits: at most kBinCtas CTAs per SM over the drawn views' bands, at least
// kMinChunk primitives (below that the CTA's counters cost more than its pairs)
dim3 chunk_grid(BinArgs &a)
{
    a.block_prims = block_prims(a.n);
    a.blocks = static_cast<int>(project_blocks(a.n));
    const int64_t c = int64_t{a.blocks} * a.max_active_bands / (int64_t{kBinCtas} * a.sms) + 1;
    const int64_t least = kMinChunk / a.block_prims;
    a.chunk = static_cast<int>(c < least ? least : c);
    return dim3(static_cast<unsigned>((a.blocks + a.chunk - 1) / a.chunk),
                static_cast<unsigned>(a.bands));
}

bool chained(const BinArgs &a) { return chained_size(a.n * a.n_views); }

}  // namespace

// k_lists' shared memory is above the 48 KB static limit.  Its three CTAs need 159 of an SM's 228
// KB; what is left is L1, which the list sort lives on.  Left to the driver, a build whose
// registers allow a fourth CTA gets the shared memory for one at the cost of the L1: 12 x 500 k
// primitives 0.096 -> 0.130 ms.
cudaError_t prepare_lists()
{
    constexpr int kShared = kListCtas * (sizeof(ListShared) + 1024);   // 1 KB a CTA is the system's
    constexpr int kPerSm = 228 << 10;
    static SharedLimit limit;
    return limit.raise(k_lists, sizeof(ListShared), (100 * kShared + kPerSm - 1) / kPerSm);
}

int bin_launches(int64_t n) { return n >= kListCap ? 5 : 4; }

cudaError_t launch_bin_counts(const BinArgs &args, cudaStream_t st)
{
    BinArgs a = args;
    if (a.n > 0) {
        const dim3 grid = chunk_grid(a);
        const cudaError_t e =
            launch_chained(chained(a), a.bands > a.n_views ? k_count<true> : k_count<false>, grid,
                           kChunkThreads, 4 * a.max_band_tiles, st, a);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(chained(a), k_layout, dim3(1), kLayoutThreads, 0, st, a.tile_count,
                          a.n_tiles, a.max_pairs, a.ranges, a.order, a.d_count, a.status, a.bin,
                          a.warps, a.rec_cap, a.n_rows, a.refine);
}

cudaError_t launch_emit(const BinArgs &args, cudaStream_t st)
{
    BinArgs a = args;
    if (a.n <= 0) return cudaSuccess;
    const dim3 grid = chunk_grid(a);
    return launch_chained(chained(a), a.bands > a.n_views ? k_emit<true> : k_emit<false>, grid,
                          kChunkThreads, 4 * a.max_band_tiles, st, a);
}

cudaError_t launch_lists(const BinArgs &a, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    // a list holds each primitive once: below kListCap primitives none is long
    if (a.n >= kListCap) {
        const int ranks = a.n >= kHugeList ? kSplitCluster : 1;
        const int grid = a.sms >= ranks ? a.sms / ranks * ranks : ranks;
        const cudaError_t e =
            launch_cluster(chained(a), ranks, k_split, dim3(grid), kSplitThreads, 0, st, a);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(chained(a), k_lists, dim3(kListCtas * a.sms), kListThreads,
                          sizeof(ListShared), st, a);
}

}  // namespace splat
