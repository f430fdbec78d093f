// a2 - a4 for maps of up to 2,048 records a tile on average: the tile lists by
// counting, scattering and sorting each tile on its own.
//
//   1. tile_count_kernel adds up each tile's pairs and tile_scan_kernel turns
//      the counts into every tile's [start, end) and lists the long tiles;
//   2. tile_scatter_kernel writes each pair's (depth bits, Gaussian index) as
//      one 64-bit word at its tile's next free slot (an atomic again, so the
//      order within a tile is arbitrary here);
//   3. tile_sort_kernel sorts each tile's words: depth first, equal depths by
//      index.  The words of a tile are distinct, so the sorted list does not
//      depend on the order they arrived in: it is the list a stable sort of
//      the 64-bit keys (tile << 32) | depth bits gives;
//   4. tile_merge_kernel puts together the chunks of the tiles of more than
//      kTileChunk words, spread over the GPU however few such tiles there are;
//      it has nothing to do on most calls.
//
// Against sorting all records by depth, emitting their pairs in that order and
// sorting the pairs by tile id (binning.cu: 13 to 16 dependent launches, of
// which a small map fills few blocks) this is five launches, reads each drawn
// record twice and each pair twice, and has no pass over all pairs that waits
// on its predecessors.  Bound: with many pairs the instruction issue of the
// sort (about log^2 of the list length a word); on small maps the five
// launches.  Kernel times, this against binning.cu:
//   100k Gaussians, 640x480, 49k pairs            36 against 125 us
//   300k Gaussians, 1200x680, 174k pairs          42 against 111 us
//   1M, 8 views of 1200x680 (32x16 tiles), 4.0M   235 against 305 us
//   4M, 16 views (lists up to 59,000), 28.2M      1.51 against 2.36 ms
// and whole calls on a map crowded into a few tiles:
//   100k in one tile of 640x480                   150 against 144 us
//   300k in 16 tiles of 1200x680                  124 against 152 us
//   1M in one tile of 1200x680, in four           215, 207 against 217, 220 us
//   4M in four tiles of 1200x680, in one          527, 848 against 558, 560 us
#include "binning.cuh"
#include "chain.cuh"
#include "common.cuh"

namespace gs {

constexpr int kListThreads = 256;
constexpr int kSortGroup = 128;                    // threads that sort a tile
constexpr int kSortBlock = 4 * kSortGroup;         // threads of a block: four tiles, or a long tile's chunk
constexpr int kMergeThreads = 256;
constexpr int kMergePer = 8;                       // words a thread of the merge sorts
constexpr uint32_t kMergeWords = kMergeThreads * kMergePer;
constexpr uint32_t kMergeParts = 5;                // blocks that share a chunk's part of the sorted tile
constexpr uint32_t kMergeSlack = 128;              // how far a cut may lie from its rank
// Chunks of a tile up to which the merge searches for each word's rank in the
// other chunks (beyond, it sorts parts of the tile again).  8M words in lists of
// two to six chunks took 583, 630, 700, 749 and 804 us of binning by search against
// 872 to 885; 100k in two lists of seven 142 against 150.
constexpr uint32_t kSearchChunks = 6;
constexpr int kSearchAhead = 4;                    // searches a thread makes side by side
constexpr int kCutThreads = kMergeThreads / 2;     // threads that look for a cut
constexpr int kCutKept = 4;                        // chunks a thread follows
constexpr int kScanThreads = 1024;
// Records up to which the pairs beyond the capacity are cut in the scan kernel, by
// a cluster of kCutCluster blocks: a call that cuts nothing pays 0.3 to 1.5 us for
// the cluster's launch (300k-Gaussian render, 100k-Gaussian tracking step; as much with
// four blocks).  A launch a step, over the whole GPU, cuts faster but costs every
// call 4 to 7 us: 300k records, 333k pairs at a capacity of 3/4, 192 against 106 us,
// 1M 403 against 155.
constexpr int kCutCluster = 8;
constexpr uint32_t kCutInScan = 1u << 20;
constexpr int kBlocksPerSm = 6;                    // counting and scattering blocks, resident
constexpr size_t kMaxTileSmem = 64 * 1024;         // a view's tiles in shared memory (16,384)
constexpr uint32_t kGroupWords = 16 * kSortGroup;  // words a group sorts (16 KB of shared memory)
constexpr uint32_t kTileChunk = 16 * kSortBlock;   // words a block sorts (64 KB)
static_assert(kTileChunk / kMergeParts + 1 + 2 * kMergeSlack <= kMergeWords, "a part of a chunk and both slacks fit");

// Words of the small region this path uses.
struct ListState {
    uint64_t room;       // pairs that still fit, while the cut is looked for
    uint32_t n_long;     // chunks listed in long_chunks
    uint32_t cut;        // 1: the pairs exceed the capacity and only the nearest are kept
    uint32_t cut_z, cut_r;  // (depth bits, record id) of the last record kept
    uint32_t cut_pairs;  // how many of its pairs
    uint32_t arrived;    // blocks that are done with a step of the cut
};

struct ListArgs {
    const float *rec;
    const uint2 *rect;
    const unsigned long long *mask;
    const uint32_t *tt;
    uint32_t total, n;  // records (views x Gaussians), Gaussians
    uint32_t cap;
    uint2 *ranges;
    uint32_t *n_pairs, *status;
    ListState *state;
    uint2 *long_chunks;         // (tile, chunk of kTileChunk) of the tiles longer than kGroupWords
    unsigned long long *words;  // [cap] unsorted (depth bits, index)
    uint32_t *table;  // [blocks][table_pitch] a block's first slot in each tile of its view
    unsigned long long *cut_hist;  // [kCutBins] of a cut by several launches (then there is no table)
    uint32_t table_pitch;
    uint64_t *keys;
    uint32_t *vals;
};

// A drawn record's tiles.
struct Splat {
    uint32_t tile0;        // tile of the rectangle's corner, within the view
    uint32_t wh;           // width | height << 16
    uint32_t z, idx;       // depth bits, Gaussian
    uint32_t rbase;        // record 0 of the view
    unsigned long long mask;
};

// The ordinal of a record's tile i (row-major in its rectangle) among its pairs.
__device__ __forceinline__ uint32_t pair_ordinal(const Splat &s, uint32_t i)
{
    if ((s.wh & 0xffffu) * (s.wh >> 16) > 64) return i;
    return (uint32_t)__popcll(s.mask & ((1ull << i) - 1ull));
}

// Whether a pair is among the nearest that fit (state.cut).
__device__ __forceinline__ bool pair_kept(const ListState &st, const Splat &s, uint32_t i)
{
    if (s.z != st.cut_z) return s.z < st.cut_z;
    if (s.rbase + s.idx != st.cut_r) return s.rbase + s.idx < st.cut_r;
    return pair_ordinal(s, i) < st.cut_pairs;
}

// What a walk does with tile i of splat s, tile `tile` of the view; alone: the
// lanes of a warp are at tiles of different splats, which may be the same.
struct CountPut {
    uint32_t *count;  // the view's tiles
    __device__ __forceinline__ void operator()(uint32_t tile, const Splat &, uint32_t, bool) const
    {
        atomicAdd(count + tile, 1u);
    }
};

struct ScatterPut {
    uint32_t *slot;
    unsigned long long *words;
    __device__ __forceinline__ void operator()(uint32_t tile, const Splat &s, uint32_t, bool) const
    {
        words[atomicAdd(slot + tile, 1u)] = ((unsigned long long)s.z << 32) | s.idx;
    }
};

// The same in the ranges' ends, where the additions of a crowded tile wait for
// one another: lanes alone at the same tile add together.
__device__ __forceinline__ uint32_t add_to_end(uint2 *ranges, uint32_t tile, bool alone)
{
    if (!alone) return atomicAdd(&ranges[tile].y, 1u);
    const uint32_t same = __match_any_sync(__activemask(), tile);
    const int lane = threadIdx.x & 31, leader = __ffs(same) - 1;
    uint32_t at = 0;
    if (lane == leader) at = atomicAdd(&ranges[tile].y, (uint32_t)__popc(same));
    return __shfl_sync(same, at, leader) + __popc(same & ((1u << lane) - 1u));
}

struct GlobalCountPut {
    uint2 *ranges;
    __device__ __forceinline__ void operator()(uint32_t tile, const Splat &, uint32_t, bool alone) const
    {
        add_to_end(ranges, tile, alone);
    }
};

struct GlobalScatterPut {
    uint2 *ranges;
    unsigned long long *words;
    __device__ __forceinline__ void operator()(uint32_t tile, const Splat &s, uint32_t, bool alone) const
    {
        words[add_to_end(ranges, tile, alone)] = ((unsigned long long)s.z << 32) | s.idx;
    }
};

// The same for the pairs that fit the capacity only, in the ranges' ends;
// without words they are only counted.
struct CutPut {
    ListState cut;
    uint2 *ranges;
    unsigned long long *words;
    __device__ __forceinline__ void operator()(uint32_t tile, const Splat &s, uint32_t i, bool alone) const
    {
        if (!pair_kept(cut, s, i)) return;
        const uint32_t pos = add_to_end(ranges, tile, alone);
        if (words) words[pos] = ((unsigned long long)s.z << 32) | s.idx;
    }
};

// The walk over all pairs of view v: put for each kept tile of a record's
// rectangle.  Warps take granules of 32 records, warp
// `first` of `stride`: drawn records come in runs (the map is in spatial order),
// so granules far apart go to one warp and every warp gets a share of a run.
// A lane walks its record's mask alone up to four tiles; larger records are
// walked by half a warp, a tile a lane.
template <bool DEPTH, typename PUT>
__device__ __forceinline__ void walk_view(const ListArgs &a, const ViewInfo &V, uint32_t v, uint32_t first,
                                          uint32_t stride, PUT put)
{
    constexpr int kAhead = 4;  // granules whose counts are loaded together
    const int lane = threadIdx.x & 31;
    const uint32_t granules = (a.n + 31) / 32;
    const size_t rbase = (size_t)v * a.n;
    const uint32_t tiles_x = (uint32_t)V.tiles_x;
    for (uint64_t g0 = first; g0 < granules; g0 += (uint64_t)kAhead * stride) {
        uint32_t cnt[kAhead];
        #pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint64_t i = (g0 + (uint64_t)k * stride) * 32 + lane;
            cnt[k] = i < a.n ? a.tt[rbase + i] : 0u;
        }
        #pragma unroll 1
        for (int k = 0; k < kAhead; k++) {
            const uint32_t c = k == 0 ? cnt[0] : k == 1 ? cnt[1] : k == 2 ? cnt[2] : cnt[3];
            if (!__any_sync(kFullMask, c > 0)) continue;
            Splat s = {};
            s.idx = (uint32_t)((g0 + (uint64_t)k * stride) * 32) + lane;
            s.rbase = (uint32_t)rbase;
            if (c) {
                const size_t r = rbase + s.idx;
                const uint2 rr = a.rect[r];
                s.mask = a.mask[r];
                s.z = DEPTH ? __float_as_uint(a.rec[12 * r + 2]) : 0u;
                s.tile0 = (rr.x >> 16) * tiles_x + (rr.x & 0xffffu);
                s.wh = ((rr.y & 0xffffu) - (rr.x & 0xffffu) + 1) | (((rr.y >> 16) - (rr.x >> 16) + 1) << 16);
            }
            const uint32_t w = s.wh & 0xffffu;
            const uint32_t recip = c ? (65536u + w - 1) / w : 0u;  // i / w = i * recip >> 16 for i < 64
            const bool alone = c > 0 && c <= 4 && w * (s.wh >> 16) <= 64;
            if (alone) {
                unsigned long long m = s.mask;
                while (m) {
                    const uint32_t i = (uint32_t)__ffsll((long long)m) - 1u;
                    m &= m - 1ull;
                    const uint32_t ky = (i * recip) >> 16;
                    put(s.tile0 + ky * tiles_x + (i - ky * w), s, i, true);
                }
            }
            // two of the larger records at a time, half a warp each
            uint32_t todo = __ballot_sync(kFullMask, c > 0 && !alone);
            while (todo) {
                const int s0 = __ffs(todo) - 1;
                todo &= todo - 1;
                const int s1 = __ffs(todo) - 1;  // -1: none
                todo &= todo - 1;
                const int src = lane < 16 ? s0 : s1;
                const bool have = src >= 0;
                Splat q;
                q.rbase = s.rbase;
                q.tile0 = __shfl_sync(kFullMask, s.tile0, src & 31);
                q.wh = __shfl_sync(kFullMask, s.wh, src & 31);
                q.mask = __shfl_sync(kFullMask, s.mask, src & 31);
                const uint32_t inv = __shfl_sync(kFullMask, recip, src & 31);
                q.z = DEPTH ? __shfl_sync(kFullMask, s.z, src & 31) : 0u;
                q.idx = DEPTH ? __shfl_sync(kFullMask, s.idx, src & 31) : 0u;
                const uint32_t qw = q.wh & 0xffffu, tiles = have ? qw * (q.wh >> 16) : 0u;
                for (uint32_t i = lane & 15; i < tiles; i += 16) {
                    const uint32_t ky = tiles <= 64 ? (i * inv) >> 16 : i / qw;
                    if (tiles > 64 || ((q.mask >> i) & 1ull)) put(q.tile0 + ky * tiles_x + (i - ky * qw), q, i, false);
                }
                __syncwarp();
            }
        }
    }
}

// One block of kScanThreads: the tile counts (ranges[t].y) to each tile's
// [start, end) ([0, 0) when empty), the long tiles' chunks to the list.  With
// `advance` the end is left at the start, for a scatter that moves it on.
// Returns the total; the ranges are complete only when it fits.
__device__ __forceinline__ uint64_t scan_tiles(const ListArgs &a, uint32_t n_tiles, bool advance)
{
    constexpr int kPer = 4;
    __shared__ uint64_t tmp[32];
    __shared__ uint32_t s_long;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_long = 0;
    uint64_t carry = 0;
    uint32_t c[kPer], next[kPer];
    auto load = [&](uint32_t t0, uint32_t (&x)[kPer]) {
        #pragma unroll
        for (int k = 0; k < kPer; k++) {
            const uint32_t t = t0 + threadIdx.x * kPer + k;
            x[k] = t < n_tiles ? __ldcg(&a.ranges[t].y) : 0u;  // (counted by blocks on other SMs)
        }
    };
    load(0, c);
    for (uint32_t t0 = 0; t0 < n_tiles; t0 += kScanThreads * kPer) {
        load(t0 + kScanThreads * kPer, next);
        uint64_t x = 0;
        #pragma unroll
        for (int k = 0; k < kPer; k++) x += c[k];
        uint64_t inc = x;
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(kFullMask, inc, o);
            if (lane >= o) inc += y;
        }
        __syncthreads();  // the last round's sums have been read
        if (lane == 31) tmp[warp] = inc;
        __syncthreads();
        const uint64_t w = tmp[lane];  // every warp scans the warps' sums
        uint64_t wi = w;
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(kFullMask, wi, o);
            if (lane >= o) wi += y;
        }
        uint64_t at = carry + __shfl_sync(kFullMask, wi - w, warp) + inc - x;
        carry += __shfl_sync(kFullMask, wi, 31);
        #pragma unroll
        for (int k = 0; k < kPer; k++) {
            const uint32_t t = t0 + threadIdx.x * kPer + k;
            if (t < n_tiles && c[k] && at + c[k] <= a.cap) {
                a.ranges[t] = make_uint2((uint32_t)at, (uint32_t)(advance ? at : at + c[k]));
                if (c[k] > kGroupWords) {
                    const uint32_t chunks = (c[k] + kTileChunk - 1) / kTileChunk;
                    const uint32_t slot = atomicAdd(&s_long, chunks);
                    for (uint32_t j = 0; j < chunks; j++) a.long_chunks[slot + j] = make_uint2(t, j);
                }
            }
            at += c[k];
            c[k] = next[k];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) a.state->n_long = s_long;
    return carry;
}

// When the pairs exceed the capacity, the nearest records' pairs stay: the (depth,
// record id) up to which they fit is found by a radix selection over all drawn
// records, weighted by their pairs.  Steps 0 to 2 add up the pairs by 11, 11 and
// 10 bits of the depth, step 3 those of the last depth by record id; after each,
// one block picks the bin in which the room ends.  Step 4 counts the tiles' pairs
// that stay.  Maps of few records do it in the scan kernel, a cluster of
// kCutCluster blocks; more take a launch a step, which return at once when nothing
// is cut (see kCutInScan).  Bound by the latency of the records' loads, with few
// warps in flight in the cluster and by the reads of all depths beyond.  Whole calls
// that cut a quarter of their pairs, this against one block that did it all and
// against the radix path:
//   100k records, 113k pairs            110, 855, 144 us
//   300k, 333k                          192, 2,306, 152 us
//   1M, 1.2M                            403, 7,553, 185 us
//   8M (1M in 8 views), 9.2M            641, 72,108, 531 us
constexpr int kCutBins = 2048;
constexpr int kCutSteps = 5;

__device__ __forceinline__ int cut_shift(int step) { return step == 0 ? 21 : step == 1 ? 10 : 0; }

// Bits of a record id below its bin in step 3.
__device__ __forceinline__ int cut_id_shift(uint32_t total)
{
    const int bits = 32 - __clz((int)(total - 1));
    return bits > 11 ? bits - 11 : 0;
}

// This thread's share (records first, first + stride, ...) of a step's sums, into
// hist in shared memory.  z: the bits of the depth that are known.
__device__ __forceinline__ void cut_sums(const ListArgs &a, int step, uint32_t z, unsigned long long *hist,
                                         uint64_t first, uint64_t stride)
{
    constexpr int kAhead = 8;
    const int known = step == 0 ? 32 : step == 1 ? 21 : step == 2 ? 10 : 0;  // the bits above are known
    const int shift = cut_shift(step), id_shift = cut_id_shift(a.total);
    for (uint64_t r0 = first; r0 < a.total; r0 += kAhead * stride) {
        uint32_t c[kAhead], d[kAhead];
        #pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const uint64_t r = r0 + k * stride;
            c[k] = r < a.total ? a.tt[r] : 0u;
        }
        #pragma unroll
        for (int k = 0; k < kAhead; k++) d[k] = c[k] ? __float_as_uint(a.rec[12 * (r0 + k * stride) + 2]) : 0u;
        #pragma unroll
        for (int k = 0; k < kAhead; k++) {
            if (!c[k] || (known < 32 && ((d[k] ^ z) >> known) != 0)) continue;
            const uint32_t bin = step == 3 ? (uint32_t)(r0 + k * stride) >> id_shift : (d[k] >> shift) & (kCutBins - 1);
            // lanes with the same bin (nearly all of them in step 0) add once
            const uint32_t same = __match_any_sync(__activemask(), bin);
            const uint32_t sum = __reduce_add_sync(same, c[k]);
            if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(hist + bin, (unsigned long long)sum);
        }
    }
}

// Sum of the block's kScanThreads values in front of this thread's, and of all.
__device__ __forceinline__ uint64_t scan_before(uint64_t x, uint64_t *tmp, uint64_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t inc = x;
    #pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(kFullMask, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();  // tmp is free
    if (lane == 31) tmp[warp] = inc;
    __syncthreads();
    const uint64_t w = tmp[lane];
    uint64_t wi = w;
    #pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(kFullMask, wi, o);
        if (lane >= o) wi += y;
    }
    *total = __shfl_sync(kFullMask, wi, 31);
    return __shfl_sync(kFullMask, wi - w, warp) + inc - x;
}

// One block: the bin in which the room ends, from the sums of bins 2 tid and
// 2 tid + 1, into the state; after step 3 the record, among those of the bin.
__device__ __forceinline__ void cut_pick(const ListArgs &a, int step, unsigned long long h0, unsigned long long h1)
{
    __shared__ uint64_t tmp[32];
    __shared__ uint32_t s_bin, s_found;
    const uint64_t room = __ldcg(&a.state->room);
    const uint32_t z = __ldcg(&a.state->cut_z);
    uint64_t all;
    const uint64_t before = scan_before(h0 + h1, tmp, &all);
    if (threadIdx.x == 0) s_bin = 0;
    __syncthreads();  // every thread has read the state
    if (before <= room && room < before + h0 + h1) {  // one thread's: the sums exceed the room
        const bool second = room >= before + h0;
        const uint32_t bin = 2 * threadIdx.x + second;
        s_bin = bin;
        if (step < 3) a.state->cut_z = z | (bin << cut_shift(step));
        a.state->room = room - before - (second ? h0 : 0);
    }
    if (threadIdx.x == 0) s_found = 0;
    __threadfence();
    __syncthreads();
    if (step < 3) return;
    const int id_shift = cut_id_shift(a.total);
    uint64_t left = __ldcg(&a.state->room);
    const uint64_t r0 = (uint64_t)s_bin << id_shift, r1 = r0 + (1ull << id_shift);
    for (uint64_t b = r0; b < r1; b += kScanThreads) {
        const uint64_t r = b + threadIdx.x;
        uint32_t c = r < r1 && r < a.total ? a.tt[r] : 0u;
        if (c && __float_as_uint(a.rec[12 * r + 2]) != z) c = 0;
        const uint64_t at = scan_before(c, tmp, &all);
        if (at <= left && left < at + c) {
            a.state->cut_r = (uint32_t)r;
            a.state->cut_pairs = (uint32_t)(left - at);
            s_found = 1;
        }
        __threadfence();
        __syncthreads();
        if (s_found) break;
        left -= all;
    }
}

// Step 4, the warps from `first` on of `stride`: the pairs that stay, in the
// ranges' ends (cleared before).
__device__ __forceinline__ void cut_count(const ListArgs &a, const ViewTable &vt, uint32_t first, uint32_t stride)
{
    ListState cut = {};
    cut.cut_z = __ldcg(&a.state->cut_z);
    cut.cut_r = __ldcg(&a.state->cut_r);
    cut.cut_pairs = __ldcg(&a.state->cut_pairs);
    for (int v = 0; v < vt.n_views; v++)
        walk_view<true>(a, vt.v[v], v, first, stride, CutPut{cut, a.ranges + vt.v[v].tile_base, nullptr});
}

// CLUSTER: a cluster of kCutCluster blocks, of which the first scans and all cut
// when the pairs do not fit.  Otherwise one block, which leaves a cut to the
// launches behind it.
template <bool CLUSTER>
__global__ void __launch_bounds__(kScanThreads) tile_scan_kernel(ListArgs a, ViewTable vt, bool advance)
{
    chain_go();
    chain_wait();
    const uint32_t n_tiles = (uint32_t)vt.n_tiles_total, rank = CLUSTER ? cluster_rank() : 0u;
    if (rank == 0) {
        if (threadIdx.x == 0) *a.state = ListState{};
        const uint64_t pairs = scan_tiles(a, n_tiles, advance);
        if (threadIdx.x == 0) {
            *a.n_pairs = pairs > 0xffffffffull ? 0xffffffffu : (uint32_t)pairs;
            if (pairs > a.cap) {
                raise_status(a.status, GS_ERR_CAPACITY);
                a.state->cut = 1;
                a.state->room = a.cap;
            }
        }
        if (!CLUSTER && pairs > a.cap)
            for (int k = threadIdx.x; k < kCutBins; k += kScanThreads) a.cut_hist[k] = 0;
    }
    if constexpr (CLUSTER) {
        __shared__ unsigned long long hist[kCutBins];
        cluster_sync();
        if (!__ldcg(&a.state->cut)) return;
        const uint32_t first = rank * kScanThreads + threadIdx.x, stride = kCutCluster * kScanThreads;
        for (uint32_t t = first; t < n_tiles; t += stride) a.ranges[t] = make_uint2(0u, 0u);
        for (int step = 0; step < kCutSteps - 1; step++) {
            for (int k = threadIdx.x; k < kCutBins; k += kScanThreads) hist[k] = 0;
            __syncthreads();
            cut_sums(a, step, __ldcg(&a.state->cut_z), hist, first, stride);
            cluster_sync();  // every block's sums are complete
            if (rank == 0) {
                unsigned long long h[2] = {};
                for (int b = 0; b < kCutCluster; b++)
                    for (int k = 0; k < 2; k++) h[k] += ld_cluster(hist + 2 * threadIdx.x + k, b);
                cut_pick(a, step, h[0], h[1]);
            }
            cluster_sync();  // the state is written, the sums are read
        }
        cut_count(a, vt, first / 32, stride / 32);
        cluster_sync();
        if (rank == 0) scan_tiles(a, n_tiles, true);
    }
}

// A step of the cut over the whole GPU; the last block to end picks the bin or
// scans the tiles.
__global__ void __launch_bounds__(kScanThreads) tile_cut_kernel(ListArgs a, ViewTable vt, int step)
{
    chain_go();
    chain_wait();
    if (!a.state->cut) return;
    __shared__ unsigned long long hist[kCutBins];
    __shared__ bool s_last;
    const uint32_t n_tiles = (uint32_t)vt.n_tiles_total;
    const uint32_t first = blockIdx.x * kScanThreads + threadIdx.x, stride = gridDim.x * kScanThreads;
    if (step < kCutSteps - 1) {
        if (step == 0)
            for (uint32_t t = first; t < n_tiles; t += stride) a.ranges[t] = make_uint2(0u, 0u);
        for (int k = threadIdx.x; k < kCutBins; k += kScanThreads) hist[k] = 0;
        __syncthreads();
        cut_sums(a, step, a.state->cut_z, hist, first, stride);
        __syncthreads();
        for (int k = threadIdx.x; k < kCutBins; k += kScanThreads)
            if (hist[k]) atomicAdd(a.cut_hist + k, hist[k]);
    } else {
        cut_count(a, vt, first / 32, stride / 32);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&a.state->arrived, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) a.state->arrived = 0;
    if (step < kCutSteps - 1) {
        const unsigned long long h0 = __ldcg(a.cut_hist + 2 * threadIdx.x), h1 = __ldcg(a.cut_hist + 2 * threadIdx.x + 1);
        a.cut_hist[2 * threadIdx.x] = a.cut_hist[2 * threadIdx.x + 1] = 0;
        cut_pick(a, step, h0, h1);
    } else {
        scan_tiles(a, n_tiles, true);
    }
}

// Grid: blocks of view 0, of view 1, ...  PRIVATE: a block counts its view's
// tiles in shared memory and adds them up at the end; the sum that an addition
// finds is the block's first slot in that tile's list, kept in its row of the
// table for the scatter.  (On the tiles' global words directly, the additions of
// a 60,000-word tile wait for one another: 1.2 ms on a 4M-Gaussian floor.)
// Without, the additions are global ones: for small maps, where a table row a
// block would not fit the workspace.
template <bool PRIVATE>
__global__ void __launch_bounds__(kListThreads, kBlocksPerSm) tile_count_kernel(ListArgs a, ViewTable vt, uint32_t blocks_per_view)
{
    chain_go();
    extern __shared__ __align__(16) unsigned char s_raw[];
    uint32_t *s_tile = reinterpret_cast<uint32_t *>(s_raw);  // the view's tiles
    const uint32_t v = blockIdx.x / blocks_per_view, b = blockIdx.x - v * blocks_per_view;
    const ViewInfo &V = vt.v[v];
    const uint32_t tiles = (uint32_t)(V.tiles_x * V.tiles_y);
    uint2 *ranges = a.ranges + V.tile_base;
    if (PRIVATE) {
        for (uint32_t t = threadIdx.x; t < tiles; t += kListThreads) s_tile[t] = 0;
        __syncthreads();
    }
    chain_wait();
    const uint32_t first = b * (kListThreads / 32) + threadIdx.x / 32, stride = blocks_per_view * (kListThreads / 32);
    if (!PRIVATE) {
        walk_view<false>(a, V, v, first, stride, GlobalCountPut{ranges});
    } else {
        walk_view<false>(a, V, v, first, stride, CountPut{s_tile});
        __syncthreads();
        uint32_t *row = a.table + (size_t)blockIdx.x * a.table_pitch;
        // four additions in flight a thread; the blocks start at different
        // tiles, so that they do not queue for the same words
        const uint32_t start = (uint32_t)(((uint64_t)tiles * b) / blocks_per_view);
        for (uint32_t t0 = threadIdx.x; t0 < tiles; t0 += 4 * kListThreads) {
            uint32_t t[4], c[4];
            #pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t u = t0 + k * kListThreads;
                t[k] = u + start < tiles ? u + start : u + start - tiles;
                c[k] = u < tiles ? s_tile[t[k]] : 0u;
            }
            #pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t n = c[k];
                if (n) c[k] = atomicAdd(&ranges[t[k]].y, n);
                t[k] = n ? t[k] : ~0u;
            }
            #pragma unroll
            for (int k = 0; k < 4; k++)
                if (t[k] != ~0u) row[t[k]] = c[k];
        }
    }
}

// The same grid and walk: each pair to its tile's next slot, from the block's
// first slot in shared memory (PRIVATE) or the tile's end in the ranges (which
// then advances to the list's end).
template <bool PRIVATE>
__global__ void __launch_bounds__(kListThreads, kBlocksPerSm) tile_scatter_kernel(ListArgs a, ViewTable vt, uint32_t blocks_per_view)
{
    chain_go();
    chain_wait();
    extern __shared__ __align__(16) unsigned char s_raw[];
    uint32_t *s_tile = reinterpret_cast<uint32_t *>(s_raw);
    const uint32_t v = blockIdx.x / blocks_per_view, b = blockIdx.x - v * blocks_per_view;
    const ViewInfo &V = vt.v[v];
    const uint32_t tiles = (uint32_t)(V.tiles_x * V.tiles_y);
    uint2 *ranges = a.ranges + V.tile_base;
    const ListState st = *a.state;
    const uint32_t first = b * (kListThreads / 32) + threadIdx.x / 32, stride = blocks_per_view * (kListThreads / 32);
    if (PRIVATE && !st.cut) {
        // (rows are written only where the block has pairs: other slots are not used)
        const uint32_t *row = a.table + (size_t)blockIdx.x * a.table_pitch;
        #pragma unroll 4
        for (uint32_t t = threadIdx.x; t < tiles; t += kListThreads) s_tile[t] = ranges[t].x + row[t];
        __syncthreads();
        walk_view<true>(a, V, v, first, stride, ScatterPut{s_tile, a.words});
    } else if (!st.cut) {
        walk_view<true>(a, V, v, first, stride, GlobalScatterPut{ranges, a.words});
    } else {
        walk_view<true>(a, V, v, first, stride, CutPut{st, ranges, a.words});
    }
}

// Ascending bitonic sort of a warp's 32 PER words, word lane * PER + r in
// register r of a lane: strides below PER stay in the lane.
template <int PER>
__device__ __forceinline__ void warp_sort(unsigned long long (&k)[PER], int lane)
{
    #pragma unroll
    for (int size = 2; size <= 32 * PER; size <<= 1) {
        #pragma unroll
        for (int stride = size / 2; stride > 0; stride >>= 1) {
            if (stride >= PER) {
                const int ls = stride / PER;
                const bool low = (lane & ls) == 0;
                const bool up = size >= 32 * PER || ((lane * PER) & size) == 0;
                #pragma unroll
                for (int r = 0; r < PER; r++) {
                    const unsigned long long o = __shfl_xor_sync(kFullMask, k[r], ls);
                    k[r] = (k[r] < o) == (low == up) ? k[r] : o;
                }
            } else {
                #pragma unroll
                for (int r = 0; r < PER; r++) {
                    if (r & stride) continue;
                    const bool up = size >= 32 * PER || ((size < PER ? r : lane * PER) & size) == 0;
                    const unsigned long long x = k[r], y = k[r | stride];
                    const bool swap = (x > y) == up;
                    k[r] = swap ? y : x;
                    k[r | stride] = swap ? x : y;
                }
            }
        }
    }
}

// Sorts words [0, m) of src, m <= THREADS PER, by THREADS threads: each warp a
// run of 32 PER in registers, then rounds of merging by rank in shared memory.
// s[0, m) holds the result; sync() is a barrier of the THREADS threads.
template <int PER, int THREADS, typename SYNC>
__device__ __forceinline__ void group_sort(const unsigned long long *src, uint32_t m, unsigned long long *s, int tid,
                                           SYNC sync)
{
    constexpr uint32_t kRun = 32 * PER;
    const int lane = tid & 31, warp = tid >> 5;
    unsigned long long k[PER];
    const uint32_t first = warp * kRun;
    if (first < m) {
        // coalesced loads; the order within the run does not matter
        #pragma unroll
        for (int r = 0; r < PER; r++) {
            const uint32_t i = first + r * 32 + lane;
            k[r] = i < m ? src[i] : ~0ull;
        }
        warp_sort<PER>(k, lane);
    } else {
        #pragma unroll
        for (int r = 0; r < PER; r++) k[r] = ~0ull;
    }
    #pragma unroll
    for (int r = 0; r < PER; r++) s[first + lane * PER + r] = k[r];
    sync();
    #pragma unroll 1
    for (uint32_t run = kRun; run < m; run *= 2) {  // until one run holds every word (the rest is padding)
        uint32_t to[PER];
        #pragma unroll
        for (int r = 0; r < PER; r++) {
            const uint32_t p = r * THREADS + tid;
            to[r] = ~0u;
            k[r] = ~0ull;
            if (p >= m) continue;  // padding: already behind every word
            k[r] = s[p];
            // words of the sibling run below this one
            const uint32_t sib = (p & ~(run - 1)) ^ run;
            uint32_t lo = 0;
            for (uint32_t half = run >> 1; half > 0; half >>= 1) lo += s[sib + lo + half - 1] < k[r] ? half : 0u;
            lo += s[sib + lo] < k[r] ? 1u : 0u;
            to[r] = (p & ~(2 * run - 1)) + (p & (run - 1)) + lo;
        }
        sync();
        #pragma unroll
        for (int r = 0; r < PER; r++)
            if (to[r] != ~0u) s[to[r]] = k[r];
        sync();
    }
}

// A block per listed chunk of a long tile (the first `extra` blocks), then four
// tiles a block, 128 threads each with a barrier of their own.  A long tile of
// one chunk is finished here; the chunks of longer ones go back sorted.
__global__ void __launch_bounds__(kSortBlock, 2) tile_sort_kernel(ListArgs a, uint32_t n_tiles, uint32_t extra)
{
    chain_go();
    chain_wait();
    extern __shared__ __align__(16) unsigned char s_raw[];
    unsigned long long *s = reinterpret_cast<unsigned long long *>(s_raw);
    if (blockIdx.x < extra) {
        const uint32_t n_long = a.state->n_long;
        for (uint32_t j = blockIdx.x; j < n_long; j += extra) {
            const uint2 tc = a.long_chunks[j];
            const uint2 r = a.ranges[tc.x];
            const uint32_t b = r.x + tc.y * kTileChunk, m = min(kTileChunk, r.y - b);
            auto sync = []() { __syncthreads(); };
            if (m <= 8 * kSortBlock) group_sort<8, kSortBlock>(a.words + b, m, s, threadIdx.x, sync);
            else group_sort<16, kSortBlock>(a.words + b, m, s, threadIdx.x, sync);
            const bool whole = r.y - r.x <= kTileChunk;
            for (uint32_t i = threadIdx.x; i < m; i += kSortBlock) {
                const unsigned long long w = s[i];
                if (whole) {
                    a.keys[b + i] = ((uint64_t)tc.x << 32) | (w >> 32);
                    a.vals[b + i] = (uint32_t)w;
                } else {
                    a.words[b + i] = w;
                }
            }
            __syncthreads();
        }
        return;
    }
    const int group = threadIdx.x / kSortGroup, tid = threadIdx.x % kSortGroup;
    const uint32_t tile = (blockIdx.x - extra) * (kSortBlock / kSortGroup) + group;
    if (tile >= n_tiles) return;
    const uint2 r = a.ranges[tile];
    const uint32_t m = r.y - r.x;
    if (m == 0 || m > kGroupWords) return;
    s += group * kGroupWords;
    const unsigned long long *src = a.words + r.x;
    auto sync = [group]() { asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kSortGroup) : "memory"); };
    if (m <= kSortGroup) group_sort<1, kSortGroup>(src, m, s, tid, sync);
    else if (m <= 2 * kSortGroup) group_sort<2, kSortGroup>(src, m, s, tid, sync);
    else if (m <= 4 * kSortGroup) group_sort<4, kSortGroup>(src, m, s, tid, sync);
    else if (m <= 8 * kSortGroup) group_sort<8, kSortGroup>(src, m, s, tid, sync);
    else group_sort<16, kSortGroup>(src, m, s, tid, sync);
    for (uint32_t i = tid; i < m; i += kSortGroup) {
        const unsigned long long w = s[i];
        a.keys[r.x + i] = ((uint64_t)tile << 32) | (w >> 32);
        a.vals[r.x + i] = (uint32_t)w;
    }
}

// Words of the sorted run below x; lo and hi bound the answer.
__device__ __forceinline__ uint32_t words_below(const unsigned long long *run, uint32_t lo, uint32_t hi,
                                                unsigned long long x)
{
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (run[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// A value with rank words of the tile below it, give or take kMergeSlack: by a
// search over values, interpolated and halved in turn, with kCutThreads threads
// that follow the answer in the tile's sorted chunks (kCutKept each; the chunks
// beyond, of a list of over 4.2M words, start afresh every time: 6M words in one
// tile 1.80 ms against 0.76 by the radix path).  A thread's searches side by side
// instead of one after another: 896 against 848 us for 4M words in one tile.  The words are distinct, so halving alone
// ends with the exact rank in 64 steps; with depths spread over the list it takes
// four to eight.  It is a function of the chunks and the rank only: the blocks on both
// sides of a cut find the same one.  bar: a barrier of the threads' own.
__device__ __noinline__ unsigned long long cut_value(const unsigned long long *w, uint32_t m, uint32_t chunks,
                                                     uint32_t rank, int tid, int bar, unsigned long long (*red)[4])
{
    if (rank == 0) return 0ull;
    if (rank >= m) return ~0ull;
    auto sync = [bar]() { asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(kCutThreads) : "memory"); };
    const int lane = tid & 31, warp = tid >> 5;
    uint32_t lo[kCutKept], hi[kCutKept];
    unsigned long long a = ~0ull, b = 0ull;  // the smallest word, and one above the largest
    #pragma unroll
    for (int k = 0; k < kCutKept; k++) {
        const uint32_t c = tid + k * kCutThreads;
        lo[k] = 0;
        hi[k] = c < chunks ? min(kTileChunk, m - c * kTileChunk) : 0u;
    }
    for (uint32_t c = tid; c < chunks; c += kCutThreads) {
        a = min(a, w[c * kTileChunk]);
        b = max(b, w[min(m, (c + 1) * kTileChunk) - 1] + 1);
    }
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = min(a, __shfl_xor_sync(kFullMask, a, o));
        b = max(b, __shfl_xor_sync(kFullMask, b, o));
    }
    if (lane == 0) {
        red[0][warp] = a;
        red[1][warp] = b;
    }
    sync();
    a = min(min(red[0][0], red[0][1]), min(red[0][2], red[0][3]));
    b = max(max(red[1][0], red[1][1]), max(red[1][2], red[1][3]));
    uint32_t ra = 0, rb = m;  // words below a (at most rank) and below b (more than rank)
    #pragma unroll 1
    for (int step = 0; step < 132 && b - a > 1; step++) {
        unsigned long long x = a + ((b - a) >> 1);
        if (!(step & 1)) {
            x = a + (unsigned long long)((float)(b - a) * ((float)(rank - ra) / (float)(rb - ra)));
            x = min(max(x, a + 1), b - 1);
        }
        uint32_t at[kCutKept], r = 0;
        #pragma unroll
        for (int k = 0; k < kCutKept; k++) {
            at[k] = words_below(w + (size_t)(tid + k * kCutThreads) * kTileChunk, lo[k], hi[k], x);
            r += at[k];
        }
        for (uint32_t c = tid + kCutKept * kCutThreads; c < chunks; c += kCutThreads)
            r += words_below(w + (size_t)c * kTileChunk, 0u, min(kTileChunk, m - c * kTileChunk), x);
        r = __reduce_add_sync(kFullMask, r);
        unsigned long long *part = red[2 + (step & 1)];  // (written again two barriers later)
        if (lane == 0) part[warp] = r;
        sync();
        r = (uint32_t)(part[0] + part[1] + part[2] + part[3]);
        if (r <= rank) {
            if (rank - r <= kMergeSlack) return x;
            a = x;
            ra = r;
        } else {
            if (r - rank <= kMergeSlack) return x;
            b = x;
            rb = r;
        }
        #pragma unroll
        for (int k = 0; k < kCutKept; k++) {
            if (r <= rank) lo[k] = at[k];
            else hi[k] = at[k];
        }
    }
    return a;
}

// Words [first, end) of a tile's chunk tc.y to their ranks in the tile: the place
// in the chunk plus the words below in the other chunks, kSearchAhead words at a time.
__device__ __forceinline__ void rank_words(const ListArgs &a, uint2 tc, uint2 r, uint32_t m, uint32_t chunks,
                                           uint32_t first, uint32_t end, int tid)
{
    const unsigned long long *w = a.words + r.x;
    for (uint32_t i0 = first + tid; i0 < end; i0 += kSearchAhead * kMergeThreads) {
        unsigned long long x[kSearchAhead];
        uint32_t rank[kSearchAhead];
        #pragma unroll
        for (int u = 0; u < kSearchAhead; u++) {
            const uint32_t i = i0 + u * kMergeThreads;
            x[u] = i < end ? w[i] : 0ull;
            rank[u] = i - tc.y * kTileChunk;
        }
        for (uint32_t c = 0; c < chunks; c++) {
            if (c == tc.y) continue;
            const unsigned long long *run = w + c * kTileChunk;
            uint32_t lo[kSearchAhead] = {};
            uint32_t n = min(kTileChunk, m - c * kTileChunk);
            while (n > 1) {
                const uint32_t half = n >> 1;
                #pragma unroll
                for (int u = 0; u < kSearchAhead; u++) lo[u] += run[lo[u] + half - 1] < x[u] ? half : 0u;
                n -= half;
            }
            #pragma unroll
            for (int u = 0; u < kSearchAhead; u++) rank[u] += lo[u] + (run[lo[u]] < x[u] ? 1u : 0u);
        }
        #pragma unroll
        for (int u = 0; u < kSearchAhead; u++) {
            if (i0 + u * kMergeThreads >= end) continue;
            a.keys[r.x + rank[u]] = ((uint64_t)tc.x << 32) | (x[u] >> 32);
            a.vals[r.x + rank[u]] = (uint32_t)x[u];
        }
    }
}

// The tiles of several sorted chunks.  A block takes a fifth of a chunk: of up to
// kSearchChunks chunks, the words at those places, each to its rank; of more, the
// words of those ranks: it finds the values that cut the tile in front of and
// behind them, gathers what lies in between from all chunks and sorts it again, so
// that a word's work does not grow with the list but for the cuts (a few searches
// in every chunk for 1,638 words).  Bound by the latency of the searches' loads.
// One list of 1M words: 80 us (8.3 ms when a block searched for a whole chunk's
// words, one by one, in all other chunks), of 100k 55 (450); the 28.2M pairs of a
// 4M-Gaussian floor 154 (334).
__global__ void __launch_bounds__(kMergeThreads, 4) tile_merge_kernel(ListArgs a)
{
    chain_go();
    chain_wait();
    __shared__ unsigned long long s[kMergeWords];
    __shared__ unsigned long long s_red[2][4][4], s_cut[2];
    __shared__ uint32_t s_end[kMergeThreads], s_src[kMergeThreads], s_sum[2][kMergeThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t items = a.state->n_long * kMergeParts;
    for (uint32_t q = blockIdx.x; q < items; q += gridDim.x) {
        const uint2 tc = a.long_chunks[q / kMergeParts];
        const uint2 r = a.ranges[tc.x];
        const uint32_t m = r.y - r.x, chunks = (m + kTileChunk - 1) / kTileChunk, part = q % kMergeParts;
        const uint32_t first = tc.y * kTileChunk + part * kTileChunk / kMergeParts;
        if (chunks == 1 || first >= m) continue;  // finished by the sort, or behind the last word
        const uint32_t end = tc.y * kTileChunk + (part + 1) * kTileChunk / kMergeParts;
        const unsigned long long *w = a.words + r.x;
        if (chunks <= kSearchChunks) {
            rank_words(a, tc, r, m, chunks, first, min(end, m), tid);
            continue;
        }
        {
            const int g = tid / kCutThreads;
            const unsigned long long x = cut_value(w, m, chunks, g ? end : first, tid % kCutThreads, 1 + g, s_red[g]);
            if (tid % kCutThreads == 0) s_cut[g] = x;
        }
        __syncthreads();
        const unsigned long long from = s_cut[0], to = s_cut[1];
        uint32_t have = 0, before = 0;  // words gathered; words below `from` in this thread's chunks
        for (uint32_t c0 = 0; c0 < chunks; c0 += kMergeThreads) {
            const uint32_t c = c0 + tid;
            uint32_t lo = 0, n = 0;
            if (c < chunks) {
                const unsigned long long *run = w + (size_t)c * kTileChunk;
                const uint32_t len = min(kTileChunk, m - c * kTileChunk);
                lo = words_below(run, 0u, len, from);
                n = words_below(run, lo, len, to) - lo;
            }
            before += lo;
            uint32_t inc = n;
            #pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFullMask, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) s_sum[0][warp] = inc;
            __syncthreads();
            for (int k = 0; k < warp; k++) inc += s_sum[0][k];
            s_end[tid] = inc;
            s_src[tid] = c * kTileChunk + lo - (inc - n);  // word i of the gathered ones: w[s_src + i]
            __syncthreads();
            const uint32_t here = s_end[kMergeThreads - 1];
            for (uint32_t i = tid; i < here; i += kMergeThreads) {
                uint32_t k = 0;  // the first chunk that ends behind word i
                #pragma unroll
                for (uint32_t half = kMergeThreads / 2; half > 0; half >>= 1) k += s_end[k + half - 1] <= i ? half : 0u;
                if (have + i < kMergeWords) s[have + i] = w[s_src[k] + i];  // (always: see kMergeWords)
            }
            have += here;
            __syncthreads();
        }
        have = min(have, kMergeWords);
        before = __reduce_add_sync(kFullMask, before);
        if (lane == 0) s_sum[1][warp] = before;
        group_sort<kMergePer, kMergeThreads>(s, have, s, tid, []() { __syncthreads(); });
        uint32_t out = r.x;
        for (int k = 0; k < kMergeThreads / 32; k++) out += s_sum[1][k];
        for (uint32_t i = tid; i < have; i += kMergeThreads) {
            const unsigned long long x = s[i];
            a.keys[out + i] = ((uint64_t)tc.x << 32) | (x >> 32);
            a.vals[out + i] = (uint32_t)x;
        }
        __syncthreads();
    }
}

// Allows the kernels `bytes` of dynamic shared memory, once a device.
template <typename... K>
static bool told_smem(PerDevice &allowed, size_t bytes, K... kernels)
{
    return allowed([&](int) {
        const cudaFuncAttribute most = cudaFuncAttributeMaxDynamicSharedMemorySize;
        return (... && (cudaFuncSetAttribute(kernels, most, (int)bytes) == cudaSuccess)) ? 1 : 0;
    }) == 1;
}

template <bool PRIVATE>
static gs_status_t launch_walks(const ListArgs &a, const ViewTable &vt, uint32_t blocks_per_view, size_t smem,
                                cudaStream_t s)
{
    const unsigned grid = blocks_per_view * (unsigned)vt.n_views;
    // the limit belongs to the kernel, not to the launch: one constant, told once
    // a device, so that no call lowers it between another thread's two launches
    static PerDevice allowed;
    if (smem > 48 * 1024 && !told_smem(allowed, kMaxTileSmem, tile_count_kernel<PRIVATE>, tile_scatter_kernel<PRIVATE>))
        return GS_ERR_CUDA;
    gs_status_t st = launch_chained(tile_count_kernel<PRIVATE>, grid, kListThreads, smem, s, a, vt, blocks_per_view);
    if (st != GS_OK) return st;
    if (a.total <= kCutInScan) {
        st = launch_with(true, kCutCluster, tile_scan_kernel<true>, kCutCluster, kScanThreads, 0, s, a, vt, !PRIVATE);
    } else {
        st = launch_chained(tile_scan_kernel<false>, 1, kScanThreads, 0, s, a, vt, !PRIVATE);
        for (int step = 0; step < kCutSteps && st == GS_OK; step++)
            st = launch_chained(tile_cut_kernel, (unsigned)num_sms(), kScanThreads, 0, s, a, vt, step);
    }
    if (st != GS_OK) return st;
    return launch_chained(tile_scatter_kernel<PRIVATE>, grid, kListThreads, smem, s, a, vt, blocks_per_view);
}

// Where a tile's list could grow very long, its chunks' merge (a search in
// every other chunk) would cost more than the radix passes: the records per
// tile decide, since the host knows no pair counts.  At 2,000 records a tile
// (950k Gaussians, four views of 400x304) whole mapping steps took 1,385
// against 1,522 us with the radix path (a room), 1,677 against 1,776 (a long
// floor, the lists most uneven); 200k Gaussians on 176x144: renders of 126
// against 193 us and 222 against 272.  The scan of the tiles is one block's,
// hence the limit on their number.
bool tile_lists_fit(int64_t n_records, int64_t n_tiles)
{
    return n_records <= 2048 * n_tiles && n_tiles <= (int64_t(1) << 18);
}

gs_status_t tile_lists(const gs_projected_t *proj, int64_t total, int64_t n, const ViewTable &vt, gs_bins_t *bins,
                       const TileListBuffers &buf, cudaStream_t s)
{
    ListArgs a;
    a.rec = proj->rec;
    a.rect = reinterpret_cast<const uint2 *>(proj->rect);
    a.mask = reinterpret_cast<const unsigned long long *>(proj->tile_mask);
    a.tt = proj->tiles_touched;
    a.total = (uint32_t)total;
    a.n = (uint32_t)n;
    a.cap = (uint32_t)bins->capacity;
    a.ranges = reinterpret_cast<uint2 *>(bins->ranges);
    a.n_pairs = bins->n_pairs;
    a.status = bins->status;
    a.state = reinterpret_cast<ListState *>(buf.small);
    a.long_chunks = static_cast<uint2 *>(buf.chunks);
    a.words = static_cast<unsigned long long *>(buf.words);
    a.keys = bins->keys;
    a.vals = bins->vals;
    a.cut_hist = static_cast<unsigned long long *>(buf.table);
    static_assert((size_t)kCutInScan * 4 >= kCutBins * sizeof(unsigned long long), "the table has room for the sums");
    const uint32_t n_tiles = (uint32_t)vt.n_tiles_total;
    gs_status_t st = launch_clear(reinterpret_cast<uint32_t *>(a.ranges), 2 * n_tiles, s);
    if (st != GS_OK) return st;
    uint32_t most_tiles = 0;
    for (int v = 0; v < vt.n_views; v++) {
        const uint32_t t = (uint32_t)(vt.v[v].tiles_x * vt.v[v].tiles_y);
        most_tiles = t > most_tiles ? t : most_tiles;
    }
    // blocks a view: a granule of 32 records a warp at least, a few waves at
    // most (views differ in what they see: with one wave the fullest view's
    // blocks finish last, 420 against 300 us on a 4M-Gaussian floor)
    const int64_t wanted = (n + kListThreads - 1) / kListThreads;
    const int64_t slots = (int64_t)num_sms() * 4 * kBlocksPerSm / vt.n_views;
    int64_t per_view = wanted < slots ? wanted : slots;
    const size_t smem = sizeof(uint32_t) * most_tiles;
    const int64_t rows = (int64_t)(buf.table_bytes / smem) / vt.n_views;  // table rows a view
    const bool priv = smem <= kMaxTileSmem && (rows >= per_view || rows * vt.n_views >= num_sms());
    if (priv) {
        per_view = per_view < rows ? per_view : rows;
        a.table = static_cast<uint32_t *>(buf.table);
        a.table_pitch = most_tiles;
        st = launch_walks<true>(a, vt, (uint32_t)per_view, smem, s);
    } else {
        a.table = nullptr;
        a.table_pitch = 0;
        st = launch_walks<false>(a, vt, (uint32_t)per_view, 0, s);
    }
    if (st != GS_OK) return st;
    const uint32_t extra = (uint32_t)num_sms() * 2;
    const size_t sort_smem = sizeof(unsigned long long) * kTileChunk;
    static PerDevice allowed;
    if (!told_smem(allowed, sort_smem, tile_sort_kernel)) return GS_ERR_CUDA;
    const unsigned groups = kSortBlock / kSortGroup;
    st = launch_chained(tile_sort_kernel, (n_tiles + groups - 1) / groups + extra, kSortBlock, sort_smem, s, a, n_tiles,
                        extra);
    // (no list is longer than a view has Gaussians)
    if (st != GS_OK || n <= kTileChunk) return st;
    return launch_chained(tile_merge_kernel, (unsigned)num_sms() * 4, kMergeThreads, 0, s, a);
}

}  // namespace gs
