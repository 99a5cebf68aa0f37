// (c) tile binning with a hand-written stable LSD radix sort.
//
// The per-tile lists are ordered by the composite key (tile, depth, primitive).
// Every pair of one primitive carries the same depth, so the primitives are sorted
// by depth once (32-bit depth bits, 4 stable passes of 8 bits, values = primitive
// index, ties kept in index order; small scenes in one block), and their (tile,
// primitive) pairs, in that order, are dealt to the tiles' lists: by counting, for
// most grids of up to kDirectTiles tiles (listed_by_counting), else by writing the pairs
// out and sorting them stably by tile id (ceil(log2 tiles / 8) passes).  The result equals a stable sort
// of (tile << 32 | depth bits) keys emitted in primitive order, with depth ties
// broken by primitive index.
//
// One radix pass = histogram kernel (per-block digit counts) + column scan (one
// block per digit: its counts over the blocks, and the digit's total) + scatter
// kernel (the lower digits' totals added per block; stable in-block ranking
// with warp match/ballot, block-local reorder in shared memory, coalesced
// write-out).  Item counts may live on the device so the whole pipeline runs
// without a host round trip.
#include <algorithm>

#include "gs_internal.h"

namespace gs {

namespace {

constexpr int kRT = 256;              // radix threads per block
constexpr int kScanT = 1024;

// Items per thread of a radix pass over up to cap items (kRI below; kRT * kRI per
// block).  More items make longer runs in the write-out, fewer make more blocks: 4
// up to 2^19 items (134,826 keys: 22 us a pass of three kernels at 16 items, 17 at
// 4), 8 up to 2^22 (2M keys: 31 against 28 us; 4 items: 32), 16 beyond (6.6M pairs of
// 600,000 primitives: depth sort and lists 271 us at 16 items, 287 at 8; 9.4M: 327, 353).
constexpr uint64_t kItems4 = 1ull << 19, kItems8 = 1ull << 22;
int radix_items(uint64_t cap) { return cap <= kItems4 ? 4 : (cap <= kItems8 ? 8 : 16); }

__device__ __forceinline__ uint64_t item_count(const unsigned long long* dcount, uint64_t scount) {
    if (!dcount) return scount;
    uint64_t c = dcount[0];
    return c < scount ? c : scount;   // scount is the capacity
}

// zero_tail: blocks past the item count write zero counts (the whole-table
// scan reads them; the column scan stops at the last block that holds items)
template <int kRI>
__global__ __launch_bounds__(kRT) void k_radix_hist(const uint32_t* __restrict__ keys,
                                                   const unsigned long long* dcount, uint64_t scount, int shift,
                                                   uint32_t* __restrict__ hist, int nblocks, int zero_tail) {
    constexpr int kRTile = kRT * kRI;
    __shared__ uint32_t h[256];
    uint64_t count = item_count(dcount, scount);
    uint64_t base = (uint64_t)blockIdx.x * kRTile;
    if (!zero_tail && base >= count) return;   // uniform over the block
    h[threadIdx.x] = 0;
    __syncthreads();
    // all loads first (kRI in flight per thread), then the shared counts
    uint32_t kk[kRI];
#pragma unroll
    for (int r = 0; r < kRI; r++) {
        const uint64_t i = base + (uint64_t)r * kRT + threadIdx.x;
        kk[r] = i < count ? keys[i] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kRI; r++) {
        const uint64_t i = base + (uint64_t)r * kRT + threadIdx.x;
        if (i < count) atomicAdd(&h[(kk[r] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(uint64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// block d: exclusive scan of digit d's counts over the blocks that hold items
// (in place; the others hold zeros and their scatter blocks return at once) and
// the digit's total; the scatter adds the totals of the lower digits itself
__global__ __launch_bounds__(kRT) void k_radix_colscan(uint32_t* __restrict__ hist, int nblocks, int tile,
                                                     const unsigned long long* dcount, uint64_t scount,
                                                     uint32_t* __restrict__ dtot) {
    __shared__ uint32_t wsum[kRT / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t* col = hist + (uint64_t)blockIdx.x * nblocks;
    const int nb = (int)min((uint64_t)nblocks, (item_count(dcount, scount) + tile - 1) / tile);
    const int chunk = (nb + kRT - 1) / kRT;
    const int b = min(tid * chunk, nb), e = min(b + chunk, nb);
    uint32_t s = 0;
    for (int i = b; i < e; i++) s += col[i];
    uint32_t x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    uint32_t run = x - s;
    for (int w = 0; w < wid; w++) run += wsum[w];
    for (int i = b; i < e; i++) {
        const uint32_t v = col[i];
        col[i] = run;
        run += v;
    }
    if (tid == kRT - 1) dtot[blockIdx.x] = run;
}

template <int kRI>
__global__ __launch_bounds__(kRT) void k_radix_scatter(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                      uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                      const unsigned long long* dcount, uint64_t scount, int shift,
                                                      const uint32_t* __restrict__ hist, int nblocks,
                                                      const uint32_t* __restrict__ dtot) {
    // Stable block-local ranking with warp-private digit counters: warp w owns
    // the contiguous items [w * 32 kRI, (w + 1) * 32 kRI) of the block's tile, so
    // ordering by (digit, warp, rank inside the warp) keeps input order.
    constexpr int kRTile = kRT * kRI;
    __shared__ uint32_t sk[kRTile];
    __shared__ uint32_t sv[kRTile];
    __shared__ uint16_t wh[kRT / 32][256];   // per-warp digit counts, then per-warp digit offsets
    __shared__ uint32_t bexcl[256];
    __shared__ uint32_t gbase[256];
    __shared__ uint32_t wsum[kRT / 32];
    __shared__ uint32_t dsum[kRT / 32];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t count = item_count(dcount, scount);
    const uint64_t base = (uint64_t)blockIdx.x * kRTile;
    if (base >= count) return;
    const uint32_t nitems = (uint32_t)(count - base < (uint64_t)kRTile ? count - base : (uint64_t)kRTile);

#pragma unroll
    for (int w = 0; w < kRT / 32; w++) wh[w][tid] = 0;
    // all loads first (kRI in flight per thread)
    uint32_t kr[kRI], vr[kRI];
    const uint32_t wbase = (uint32_t)warp * 32u * kRI;
#pragma unroll
    for (int r = 0; r < kRI; r++) {
        const uint32_t i = wbase + (uint32_t)r * 32u + (uint32_t)lane;
        kr[r] = i < nitems ? kin[base + i] : 0u;
        vr[r] = i < nitems ? vin[base + i] : 0u;
    }
    __syncthreads();
    // rank inside the warp, round by round (the rounds are in item order)
    const unsigned lt_mask = (1u << lane) - 1u;
    uint32_t lrank[kRI];
#pragma unroll
    for (int r = 0; r < kRI; r++) {
        const bool valid = wbase + (uint32_t)r * 32u + (uint32_t)lane < nitems;
        const uint32_t d = valid ? ((kr[r] >> shift) & 255u) : 256u;
        // lanes holding the same digit (9 bits, so the invalid sentinel 256 stands apart)
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int bit = 0; bit < 9; bit++) {
            const unsigned m = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
            peers &= ((d >> bit) & 1u) ? m : ~m;
        }
        const uint32_t before = valid ? wh[warp][d] : 0u;
        __syncwarp();
        if (valid && (peers & lt_mask) == 0u) wh[warp][d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
        lrank[r] = before + __popc(peers & lt_mask);
    }
    __syncthreads();
    // thread tid = digit: offsets of each warp inside the digit, digit totals,
    // block-exclusive scan of the totals
    {
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < kRT / 32; w++) {
            const uint32_t c = wh[w][tid];
            wh[w][tid] = (uint16_t)tot;
            tot += c;
        }
        uint32_t x = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        // start of digit tid in the output: the lower digits' totals (none when the
        // histogram was scanned as one table over (digit, block))
        const uint32_t dt = dtot ? dtot[tid] : 0u;
        uint32_t dx = dt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, dx, o);
            if (lane >= o) dx += y;
        }
        if (lane == 31) {
            wsum[warp] = x;
            dsum[warp] = dx;
        }
        __syncthreads();
        uint32_t add = 0, dadd = 0;
        for (int w = 0; w < warp; w++) {
            add += wsum[w];
            dadd += dsum[w];
        }
        bexcl[tid] = x - tot + add;
        gbase[tid] = hist[(uint64_t)tid * nblocks + blockIdx.x] + dx - dt + dadd;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRI; r++) {
        if (wbase + (uint32_t)r * 32u + (uint32_t)lane < nitems) {
            const uint32_t d = (kr[r] >> shift) & 255u;
            const uint32_t pos = bexcl[d] + wh[warp][d] + lrank[r];
            sk[pos] = kr[r];
            sv[pos] = vr[r];
        }
    }
    __syncthreads();
    for (uint32_t i = tid; i < nitems; i += kRT) {
        uint32_t key = sk[i];
        uint32_t d = (key >> shift) & 255u;
        uint64_t dst = (uint64_t)gbase[d] + (i - bexcl[d]);
        kout[dst] = key;
        vout[dst] = sv[i];
    }
}

// ---------------------------------------------------------------------------
// tiles per primitive (depth order), scan, pair emission, ranges
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t rect_tiles(uint2 r) {
    uint32_t x0 = r.x & 0xffff, y0 = r.x >> 16, x1 = r.y & 0xffff, y1 = r.y >> 16;
    return (x1 > x0 && y1 > y0) ? (x1 - x0) * (y1 - y0) : 0u;
}

// srect: the rects in depth order (the list kernels read them in that order)
__global__ void k_count_tiles(const uint32_t* __restrict__ sorted_ids, const uint2* __restrict__ rects, uint64_t n,
                              uint32_t* __restrict__ cnt, uint2* __restrict__ srect) {
    uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const uint2 r = rects[sorted_ids[j]];
    cnt[j] = rect_tiles(r);
    srect[j] = r;
}

constexpr int kScanItems = 16;
constexpr int kScanBlockT = 256;
constexpr int kScanTile = kScanItems * kScanBlockT;

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += sh[w];
    __syncthreads();
    return s;
}

__global__ __launch_bounds__(kScanBlockT) void k_scan_partials(const uint32_t* __restrict__ in, uint64_t n,
                                                              unsigned long long* __restrict__ part) {
    __shared__ unsigned long long sh[kScanBlockT / 32];
    uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    unsigned long long s = 0;
    for (int r = 0; r < kScanItems; r++) {
        uint64_t i = base + (uint64_t)r * kScanBlockT + threadIdx.x;
        if (i < n) s += in[i];
    }
    s = block_sum_u64(s, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// exclusive scan of the block partials (single block) and the grand total
__global__ __launch_bounds__(kScanT) void k_scan_partials_top(unsigned long long* part, int nparts,
                                                             unsigned long long* total, uint64_t cap) {
    __shared__ unsigned long long wsum[kScanT / 32];
    int chunk = (nparts + kScanT - 1) / kScanT;
    int b = threadIdx.x * chunk, e = min(b + chunk, nparts);
    unsigned long long s = 0;
    for (int i = b; i < e; i++) s += part[i];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x = s;
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long t = wsum[lane];
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        wsum[lane] = t;
    }
    __syncthreads();
    unsigned long long run = x - s + (wid > 0 ? wsum[wid - 1] : 0ull);
    for (int i = b; i < e; i++) {
        unsigned long long v = part[i];
        part[i] = run;
        run += v;
    }
    if (threadIdx.x == kScanT - 1) {
        total[0] = run < cap ? run : cap;     // usable pair count
        total[1] = run > cap ? 1ull : 0ull;   // overflow flag
        total[2] = run;                       // true pair count
    }
}

// in and out may be the same array: every element is read and then written by
// the same thread, and by no other
__global__ __launch_bounds__(kScanBlockT) void k_scan_apply(const uint32_t* in, uint64_t n,
                                                           const unsigned long long* __restrict__ part,
                                                           uint32_t* out) {
    __shared__ uint32_t wsum[kScanBlockT / 32];
    __shared__ uint32_t carry;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    if (threadIdx.x == 0) carry = (uint32_t)part[blockIdx.x];
    // all loads first (kScanItems in flight per thread): the barriers of the
    // rounds below would otherwise expose one load latency per round
    uint32_t vv[kScanItems];
#pragma unroll
    for (int r = 0; r < kScanItems; r++) {
        const uint64_t i = base + (uint64_t)r * kScanBlockT + threadIdx.x;
        vv[r] = i < n ? in[i] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kScanItems; r++) {
        uint64_t i = base + (uint64_t)r * kScanBlockT + threadIdx.x;
        uint32_t v = vv[r];
        uint32_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        uint32_t add = carry;
        for (int w = 0; w < wid; w++) add += wsum[w];
        if (i < n) out[i] = add + x - v;
        __syncthreads();
        if (threadIdx.x == kScanBlockT - 1) carry = add + x;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Tile lists by counting: the pairs of the primitives in depth order, dealt to the
// lists without sorting them.  The pairs (never stored) are cut into segments of
// equal length, one per block, and each segment into one run per warp.
//   k_tile_hist: each warp counts its run's pairs per tile in shared memory; out go
//     the warps' exclusive counts inside the segment and the segment's totals.
//   k_tile_colscan, k_tile_starts: exclusive counts over the segments, the tiles'
//     totals, their starts and ranges.
//   k_tile_place: each warp walks its run again and writes every pair's primitive
//     at its place: tile start + earlier segments + earlier warps + rank in the run.
// A list is then in (segment, warp, pair) order, the depth order.  The counters of
// a warp take 2 bytes a tile, so this runs for grids of up to kDirectTiles tiles; larger
// ones, and large scenes on large ones, keep the radix sort of (tile, primitive) pairs
// below.  Per pair it
// moves 4 B (the primitive, written once) where the sort of 12-bit to 16-bit tile
// ids moved 60 (emission, two passes, ranges).  Bound by the placing walk's chain per
// 64 pairs and its stores, a sector per pair: 12.25M pairs of a 2M-primitive,
// 1600x1040 view take 203 us (count 54, scans 18, place 131), the sort 290 us; the
// same with 6 or 16 warps per SM.
// ---------------------------------------------------------------------------
constexpr int kDirectTiles = 13900;
constexpr int kWalkGroups = 4;   // see walk_pairs

// Is a grid of nt tiles listed by counting for a scene of n primitives?  Up to about 7,000
// tiles two blocks fit an SM; with one, the walks of long pair streams fall behind the
// sort: 2M primitives on 7,684 tiles (12.4M pairs) 440 us against 478, on 10,000 tiles
// (12.2M) 498 against 474, on 13,000 (17.4M) 620 against 554; 600,000 primitives on 13,000
// tiles (5.7M) 241 against 271.
bool listed_by_counting(uint64_t n, int nt) { return nt <= 9000 || (nt <= kDirectTiles && n <= (1ull << 20)); }

// Blocks, warps and shared memory of the two walks for a grid of nt tiles.
struct DirectShape {
    int warps, per_sm, segs;
    size_t hist_smem, place_smem;
};

DirectShape direct_shape(int nt, uint64_t cap) {
    DirectShape d;
    // the placing walk needs 2 bytes a tile and warp and 4 a tile; a block's segment
    // must stay below 2^16 pairs (the warps' exclusive counts are 16-bit)
    const size_t t = ((size_t)nt + 7) & ~(size_t)7;
    d.warps = t * 20 <= 54 * 1024 ? 8 : 6;
    d.hist_smem = t * 2 * (size_t)d.warps;
    d.place_smem = t * (2 * (size_t)d.warps + 4);
    d.per_sm = (int)std::max<size_t>(1, std::min<size_t>(2, (220 * 1024) / (d.place_smem + 1024)));
    const uint64_t fill = (uint64_t)num_sms() * d.per_sm;
    // no segment shorter than 8 steps of its warps, none of 2^16 pairs or more
    d.segs = (int)std::max<uint64_t>({(uint64_t)1, std::min<uint64_t>(fill, div_up(cap, (uint64_t)d.warps * 256)), div_up(cap, 60000)});
    return d;
}

// Words of the counting tables of such a shape: the segments' totals, the tiles'
// totals, the warps' 16-bit counts.
size_t direct_words(const DirectShape& d, int nt) {
    const size_t t = ((size_t)nt + 7) & ~(size_t)7;
    return t * d.segs + t + t * d.warps / 2 * d.segs;
}

// Words that serve every grid of up to nt tiles at a pair capacity of cap.  A block's
// shared memory bounds tiles x warps per SM, so one wave of blocks takes the same at
// any grid (34 MB); beyond it the segments go with the capacity.  Small scenes have few
// segments: 1 MB serves them, and a render of another size mostly finds its tables there
// (a first render of 6,741 primitives at 800x800: 350 us with 1 or 34 MB, 460 with 3).
size_t direct_tab_words(int nt, uint64_t cap) {
    const auto tables = [nt](uint64_t segs) { return (size_t)segs * (size_t)(nt + 8) * (4 + 1) + (size_t)nt + 64; };
    constexpr size_t kSmall = 1ull << 18;
    const size_t wave = (size_t)num_sms() * (220 * 1024 / 4) + kDirectTiles + 64;   // tiles x (warps + 2) x blocks, two bytes each
    const size_t few = tables(div_up(std::max<uint64_t>(cap, 1), 6 * 256));
    return std::max(few <= kSmall ? kSmall : wave, tables(div_up(cap, 60000)));
}

// The pairs [p0, p1) in order, 2 x 32 at a time: f(tile, primitive, active of the
// first 32, the same of the second); called by whole warps.
template <class F>
__device__ __forceinline__ void walk_pairs(const uint32_t* __restrict__ sid, const uint2* __restrict__ srect,
                                           const uint32_t* __restrict__ off, uint32_t n, uint32_t p0, uint32_t p1,
                                           int tiles_x, const F& f) {
    const int lane = threadIdx.x & 31;
    if (p0 >= p1) return;
    // the primitive of pair p0: the last one whose offset is <= p0 (32-ary search)
    uint32_t lo = 0, hi = n;   // the answer is in [lo, hi)
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31u) / 32u, at = lo + (uint32_t)lane * step;
        const unsigned m = __ballot_sync(0xffffffffu, at < hi && off[at] <= p0);
        const uint32_t k = 31u - (uint32_t)__clz(m);   // lane 0 always holds (off[lo] <= p0)
        lo += k * step;
        hi = min(hi, lo + step);
    }
    auto load = [&](uint32_t j, uint32_t& o, uint2& r, uint32_t& id) {
        const bool in = j < n;
        o = in ? off[j] : 0xffffffffu;
        r = in ? srect[j] : make_uint2(0u, 0u);
        id = in ? sid[j] : 0u;
    };
    // kWalkGroups groups of 32 primitives at a time, the next ones in flight over them:
    // far primitives have one or two pairs each, and a group's loads take longer than
    // its pairs
    uint32_t o[kWalkGroups], id[kWalkGroups], no[kWalkGroups], nid[kWalkGroups];
    uint2 r[kWalkGroups], nr[kWalkGroups];
#pragma unroll
    for (int k = 0; k < kWalkGroups; k++) load(lo + 32u * k + (uint32_t)lane, o[k], r[k], id[k]);
    for (uint32_t j0 = lo; j0 < n; j0 += 32u * kWalkGroups) {
#pragma unroll
        for (int k = 0; k < kWalkGroups; k++)
            load(j0 + 32u * (kWalkGroups + k) + (uint32_t)lane, no[k], nr[k], nid[k]);
        uint32_t gend = 0;
#pragma unroll
        for (int k = 0; k < kWalkGroups; k++) {
            const uint32_t first = max(p0, __shfl_sync(0xffffffffu, o[k], 0));
            if (first >= p1) return;   // past the run, or past the last primitive
            const uint32_t c = rect_tiles(r[k]), w = (r[k].y & 0xffffu) - (r[k].x & 0xffffu);
            const float inv = 1.0f / (float)max(w, 1u);
            gend = __reduce_max_sync(0xffffffffu, o[k] == 0xffffffffu ? 0u : o[k] + c);
            const uint32_t end = min(p1, gend);
            // the source lane, tile and primitive of pair b + lane.  Primitives without tiles
            // come last in depth order, so the lanes with pairs are the first ones and the
            // source of a pair is the number of primitives that start at or before it, less
            // one: those at or before b, plus the starts marked inside the 32 pairs.
            auto pair_of = [&](uint32_t b, uint32_t& tile, uint32_t& prim) {
                const uint32_t d = o[k] - b;   // start inside (b, b + 32): 1 ... 31
                const unsigned begun = __ballot_sync(0xffffffffu, o[k] <= b);
                const unsigned marks = __reduce_or_sync(0xffffffffu, d - 1u < 31u ? 1u << d : 0u);
                const int s = __popc(begun) - 1 + __popc(marks & (0xffffffffu >> (31 - lane)));
                const uint32_t t = b + (uint32_t)lane - __shfl_sync(0xffffffffu, o[k], s);
                const uint32_t xy = __shfl_sync(0xffffffffu, r[k].x, s), sw = __shfl_sync(0xffffffffu, w, s);
                prim = __shfl_sync(0xffffffffu, id[k], s);
                // t / sw: exact for t < 2^20 (the half keeps it off the integers by more than the
                // rounding of the reciprocal and the product)
                const uint32_t ty = (uint32_t)(((float)t + 0.5f) * __shfl_sync(0xffffffffu, inv, s));
                tile = ((xy >> 16) + ty) * (uint32_t)tiles_x + (xy & 0xffffu) + (t - ty * sw);
            };
            // two groups of 32 pairs at a time: their chains overlap
            if (first < end) {
                uint32_t b = first;
                do {
                    const uint32_t left = end - b;
                    uint32_t t0, i0, t1, i1;
                    pair_of(b, t0, i0);
                    pair_of(b + 32u, t1, i1);
                    f(t0, i0, (uint32_t)lane < left, t1, i1, 32u + (uint32_t)lane < left);
                } while (pair_next(b, end));
            }
        }
        if (gend >= p1) return;
#pragma unroll
        for (int k = 0; k < kWalkGroups; k++) {
            o[k] = no[k];
            r[k] = nr[k];
            id[k] = nid[k];
        }
    }
}

// run of this warp
__device__ __forceinline__ void warp_run(uint32_t total, uint32_t& p0, uint32_t& p1) {
    pair_run(total, gridDim.x * (blockDim.x >> 5), blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), p0, p1);
}

__global__ void k_tile_hist(const uint32_t* __restrict__ sid, const uint2* __restrict__ srect,
                            const uint32_t* __restrict__ off, uint32_t n, int tiles_x, int nt,
                            const unsigned long long* __restrict__ total, uint16_t* __restrict__ wtab,
                            uint32_t* __restrict__ tab) {
    extern __shared__ __align__(16) uint32_t hsm[];   // two 16-bit counters a word, a row per warp
    if (total[1]) return;   // the pairs overflow the capacity: nothing is listed (uniform)
    const int tpad = (nt + 7) & ~7, row = tpad / 2, warps = blockDim.x >> 5;
    for (int i = threadIdx.x; i < row * warps / 4; i += blockDim.x) reinterpret_cast<uint4*>(hsm)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    uint32_t p0, p1;
    warp_run((uint32_t)total[0], p0, p1);
    uint32_t* h = hsm + (threadIdx.x >> 5) * row;
    walk_pairs(sid, srect, off, n, p0, p1, tiles_x,
               [&](uint32_t t0, uint32_t, bool a0, uint32_t t1, uint32_t, bool a1) {
                   if (a0) atomicAdd(&h[t0 >> 1], 1u << ((t0 & 1u) * 16u));
                   if (a1) atomicAdd(&h[t1 >> 1], 1u << ((t1 & 1u) * 16u));
               });
    __syncthreads();
    // two tiles at a time (16-bit halves: a segment has fewer than 2^16 pairs)
    uint32_t* wout = reinterpret_cast<uint32_t*>(wtab) + (size_t)blockIdx.x * warps * row;
    for (int i = threadIdx.x; i < row; i += blockDim.x) {
        uint32_t run = 0;
        for (int w = 0; w < warps; w++) {
            wout[(size_t)w * row + i] = run;
            run += hsm[w * row + i];
        }
        reinterpret_cast<uint2*>(tab + (size_t)blockIdx.x * tpad)[i] = make_uint2(run & 0xffffu, run >> 16);
    }
}

// Column t of tab: exclusive counts over the segments (in place) and the tile's total.
__global__ __launch_bounds__(1024) void k_tile_colscan(uint32_t* __restrict__ tab, int nt, int tpad, int segs,
                                                     const unsigned long long* __restrict__ total,
                                                     uint32_t* __restrict__ tot) {
    __shared__ uint32_t part[32][33];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, t = blockIdx.x * 32 + lane;
    const int per = (segs + 31) / 32, b = min(g * per, segs), e = min(b + per, segs);
    if (total[1]) return;   // uniform
    uint32_t s = 0;
    if (t < nt) {
#pragma unroll 8
        for (int i = b; i < e; i++) s += tab[(size_t)i * tpad + t];
    }
    part[g][lane] = s;
    __syncthreads();
    uint32_t run = 0, all = 0;
#pragma unroll
    for (int k = 0; k < 32; k++) {
        run += k < g ? part[k][lane] : 0u;
        all += part[k][lane];
    }
    if (t >= nt) return;
    if (g == 0) tot[t] = all;
#pragma unroll 8
    for (int i = b; i < e; i++) {
        const uint32_t c = tab[(size_t)i * tpad + t];
        tab[(size_t)i * tpad + t] = run;
        run += c;
    }
}

// The tiles' starts (in place of their totals) and ranges (empty tiles: 0, 0).
__global__ __launch_bounds__(kScanT) void k_tile_starts(uint32_t* __restrict__ tot, int nt,
                                                       const unsigned long long* __restrict__ total,
                                                       uint2* __restrict__ ranges) {
    __shared__ uint32_t wsum[kScanT / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (total[1]) {   // uniform: no lists
        for (int t = threadIdx.x; t < nt; t += kScanT) ranges[t] = make_uint2(0u, 0u);
        return;
    }
    uint32_t carry = 0;
    for (int base = 0; base < nt; base += kScanT) {
        const int t = base + threadIdx.x;
        const uint32_t c = t < nt ? tot[t] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        const uint32_t ws = wsum[lane];
        uint32_t add = __reduce_add_sync(0xffffffffu, lane < wid ? ws : 0u);
        const uint32_t all = __reduce_add_sync(0xffffffffu, ws);
        const uint32_t at = carry + add + x - c;
        if (t < nt) {
            tot[t] = at;
            ranges[t] = c ? make_uint2(at, at + c) : make_uint2(0u, 0u);
        }
        carry += all;
        __syncthreads();
    }
}

__global__ void k_tile_place(const uint32_t* __restrict__ sid, const uint2* __restrict__ srect,
                             const uint32_t* __restrict__ off, uint32_t n, int tiles_x, int nt,
                             const unsigned long long* __restrict__ total, const uint16_t* __restrict__ wtab,
                             const uint32_t* __restrict__ tab, const uint32_t* __restrict__ start,
                             uint32_t* __restrict__ ids) {
    extern __shared__ __align__(16) uint32_t psm[];   // place of each tile's next pair, then the warps' counters
    if (total[1]) return;   // uniform
    const int tpad = (nt + 7) & ~7, warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* cnt = psm + tpad + (size_t)warp * (tpad / 2);   // two 16-bit counters a word
    for (int i = threadIdx.x; i < tpad / 4; i += blockDim.x) {
        const uint4 a = reinterpret_cast<const uint4*>(start)[i];
        const uint4 c = reinterpret_cast<const uint4*>(tab + (size_t)blockIdx.x * tpad)[i];
        reinterpret_cast<uint4*>(psm)[i] = make_uint4(a.x + c.x, a.y + c.y, a.z + c.z, a.w + c.w);
    }
    for (int i = threadIdx.x; i < warps * tpad / 8; i += blockDim.x)
        reinterpret_cast<uint4*>(psm + tpad)[i] =
            reinterpret_cast<const uint4*>(wtab + (size_t)blockIdx.x * warps * tpad)[i];
    __syncthreads();
    uint32_t p0, p1;
    warp_run((uint32_t)total[0], p0, p1);
    const unsigned lt = (1u << lane) - 1u;
    walk_pairs(sid, srect, off, n, p0, p1, tiles_x,
               [&](uint32_t t0, uint32_t i0, bool a0, uint32_t t1, uint32_t i1, bool a1) {
                   // the first pair of each tile draws the places of all of them
                   const unsigned m0 = __match_any_sync(0xffffffffu, a0 ? t0 : 0xffffffffu);
                   const unsigned m1 = __match_any_sync(0xffffffffu, a1 ? t1 : 0xffffffffu);
                   const uint32_t b0 = a0 ? psm[t0] : 0u, b1 = a1 ? psm[t1] : 0u;
                   const unsigned s0 = (t0 & 1u) * 16u, s1 = (t1 & 1u) * 16u;
                   uint32_t c0 = 0, c1 = 0;
                   if (a0 && (m0 & lt) == 0u) c0 = atomicAdd(&cnt[t0 >> 1], (uint32_t)__popc(m0) << s0);
                   __syncwarp();   // the second 32 pairs come behind the first
                   if (a1 && (m1 & lt) == 0u) c1 = atomicAdd(&cnt[t1 >> 1], (uint32_t)__popc(m1) << s1);
                   c0 = (__shfl_sync(0xffffffffu, c0, __ffs(m0) - 1) >> s0) & 0xffffu;
                   c1 = (__shfl_sync(0xffffffffu, c1, __ffs(m1) - 1) >> s1) & 0xffffu;
                   if (a0) ids[b0 + c0 + (uint32_t)__popc(m0 & lt)] = i0;
                   if (a1) ids[b1 + c1 + (uint32_t)__popc(m1 & lt)] = i1;
                   __syncwarp();
               });
}

constexpr uint32_t kBigPrim = 256;   // primitives with more tiles are emitted by a whole block

// thread per primitive (depth order): write its (tile, primitive) pairs, row-major over its rect
__global__ void k_emit(const uint32_t* __restrict__ sorted_ids, const uint2* __restrict__ rects,
                       const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ off, uint64_t n, int tiles_x,
                       const unsigned long long* __restrict__ total, uint32_t* __restrict__ pkey,
                       uint32_t* __restrict__ pval, uint32_t* big_list, unsigned int* big_count) {
    // one warp per 32 consecutive primitives (depth order); their pairs are
    // written by consecutive lanes, so the stores coalesce
    const int lane = threadIdx.x & 31;
    const uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (total[1]) return;   // nothing is emitted when the pairs overflow the capacity (uniform)
    uint32_t c = j < n ? cnt[j] : 0u;
    if (c > kBigPrim) {   // emitted by k_emit_big
        big_list[atomicAdd(big_count, 1u)] = (uint32_t)j;
        c = 0u;
    }
    uint32_t p = 0, o = 0, x0 = 0, y0 = 0, w = 1;
    if (c) {
        p = sorted_ids[j];
        const uint2 r = rects[p];
        x0 = r.x & 0xffff;
        y0 = r.x >> 16;
        w = (r.y & 0xffff) - x0;
        o = off[j];
    }
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    const uint32_t excl = incl - c;
    const uint32_t wtotal = __shfl_sync(0xffffffffu, incl, 31);
    for (uint32_t b = 0; b < wtotal; b += 32) {
        const uint32_t q = b + (uint32_t)lane;
        // source lane: the last lane whose exclusive offset is <= q (lanes without
        // pairs share their neighbour's offset and are skipped by taking the last)
        int s = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const int m = s + step;
            if (__shfl_sync(0xffffffffu, excl, m) <= q) s = m;
        }
        const uint32_t t = q - __shfl_sync(0xffffffffu, excl, s);
        const uint32_t so = __shfl_sync(0xffffffffu, o, s), sp = __shfl_sync(0xffffffffu, p, s);
        const uint32_t sx = __shfl_sync(0xffffffffu, x0, s), sy = __shfl_sync(0xffffffffu, y0, s);
        const uint32_t sw = __shfl_sync(0xffffffffu, w, s);
        if (q < wtotal) {
            pkey[so + t] = (sy + t / sw) * (uint32_t)tiles_x + sx + t % sw;
            pval[so + t] = sp;
        }
    }
}

__global__ void k_emit_big(const uint32_t* __restrict__ sorted_ids, const uint2* __restrict__ rects,
                           const uint32_t* __restrict__ off, int tiles_x, const unsigned long long* __restrict__ total,
                           uint32_t* __restrict__ pkey, uint32_t* __restrict__ pval, const uint32_t* big_list,
                           const unsigned int* big_count) {
    if (total[1]) return;
    unsigned int nb = *big_count;
    for (unsigned int b = blockIdx.x; b < nb; b += gridDim.x) {
        uint32_t j = big_list[b];
        uint32_t p = sorted_ids[j];
        uint2 r = rects[p];
        uint32_t x0 = r.x & 0xffff, y0 = r.x >> 16, x1 = r.y & 0xffff;
        uint32_t w = x1 - x0;
        uint32_t c = rect_tiles(r);
        uint32_t o = off[j];
        for (uint32_t m = threadIdx.x; m < c; m += blockDim.x) {
            uint32_t y = y0 + m / w, x = x0 + m % w;
            pkey[o + m] = y * (uint32_t)tiles_x + x;
            pval[o + m] = p;
        }
    }
}

__global__ void k_ranges(const uint32_t* __restrict__ keys, const unsigned long long* __restrict__ total,
                         uint64_t cap, uint2* __restrict__ ranges) {
    uint64_t cnt = total[0];
    if (total[1]) return;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t k = keys[i];
        if (i == 0 || keys[i - 1] != k) ranges[k].x = (uint32_t)i;
        if (i == cnt - 1 || keys[i + 1] != k) ranges[k].y = (uint32_t)(i + 1);
    }
}

__global__ void k_ranges_to_offsets(const uint2* ranges, int ntiles, uint32_t* offsets) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    // lists are contiguous in tile order: offset[t] = start of tile t's list or the running end
    if (t < ntiles) {
        uint2 r = ranges[t];
        offsets[t] = r.x;
        if (r.y == 0) offsets[t] = 0xffffffffu;   // empty: filled by the fix-up pass
    }
}

__global__ void k_offsets_fixup(uint32_t* offsets, int ntiles, const unsigned long long* total) {
    // single thread: empty tiles take the start of the next non-empty tile
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    uint32_t next = (uint32_t)total[0];
    offsets[ntiles] = next;
    for (int t = ntiles - 1; t >= 0; t--) {
        if (offsets[t] == 0xffffffffu)
            offsets[t] = next;
        else
            next = offsets[t];
    }
}

// rects clipped to the grid [0, tiles_x) x [0, tiles_y) here, so no list index
// can leave it whatever the caller passes
__global__ void k_rects_to_keys(const float* depth, const int32_t* rects, uint64_t n, int tiles_x, int tiles_y,
                                uint32_t* keys, uint32_t* vals, uint2* prect) {
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int x0 = min(max(rects[4 * i + 0], 0), tiles_x), y0 = min(max(rects[4 * i + 1], 0), tiles_y);
    const int x1 = min(max(rects[4 * i + 2], 0), tiles_x), y1 = min(max(rects[4 * i + 3], 0), tiles_y);
    bool vis = x1 > x0 && y1 > y0;
    // primitives without tiles come last (walk_pairs counts on it), whatever the depth bits
    keys[i] = vis ? min(__float_as_uint(depth[i]), 0xfffffffeu) : 0xffffffffu;
    vals[i] = (uint32_t)i;
    prect[i] = vis ? make_uint2((uint32_t)x0 | ((uint32_t)y0 << 16), (uint32_t)x1 | ((uint32_t)y1 << 16))
                   : make_uint2(0, 0);
}

// ---------------------------------------------------------------------------
// Depth order of a small scene in one block: the four 8-bit passes on registers and
// shared memory, ranked like a scatter block's (stable), then the tile counts and
// their scan in the same kernel.  Up to kSmallN primitives this replaces 16 launches
// whose time is latency (6,741 primitives: 60 us against 15).
// ---------------------------------------------------------------------------
constexpr int kSmallT = 1024, kSmallI = 8, kSmallN = kSmallT * kSmallI;
struct SmallSort {
    uint32_t k[kSmallN], v[kSmallN];
    uint16_t wh[kSmallT / 32][256];   // per-warp digit counts, then offsets
    uint32_t bexcl[256];
    uint32_t wsum[kSmallT / 32];
};

__global__ __launch_bounds__(kSmallT) void k_order_small(uint32_t* __restrict__ key, uint32_t* __restrict__ val,
                                                        const uint2* __restrict__ rects, uint32_t n,
                                                        uint32_t* __restrict__ cnt, uint32_t* __restrict__ off,
                                                        uint2* __restrict__ srect, unsigned long long* total,
                                                        uint64_t cap) {
    extern __shared__ __align__(16) unsigned char small_mem[];
    SmallSort& s = *reinterpret_cast<SmallSort*>(small_mem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t i0 = (uint32_t)warp * 32u * kSmallI + (uint32_t)lane;   // this lane's items: i0 + 32 r
    uint32_t kr[kSmallI], vr[kSmallI], rank[kSmallI];
#pragma unroll
    for (int r = 0; r < kSmallI; r++) {
        const uint32_t i = i0 + 32u * r;
        kr[r] = i < n ? key[i] : 0u;
        vr[r] = i < n ? val[i] : 0u;
    }
    for (int shift = 0; shift < 32; shift += 8) {
        for (int i = lane; i < 256; i += 32) s.wh[warp][i] = 0;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < kSmallI; r++) {
            const bool valid = i0 + 32u * r < n;
            const uint32_t d = valid ? ((kr[r] >> shift) & 255u) : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = valid ? s.wh[warp][d] : 0u;
            __syncwarp();
            if (valid && (peers & lt) == 0u) s.wh[warp][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            rank[r] = before + (uint32_t)__popc(peers & lt);
        }
        __syncthreads();
        uint32_t tot = 0, x = 0;
        if (tid < 256) {   // thread = digit: offsets of the warps inside it, then of the digits
#pragma unroll 8
            for (int w = 0; w < kSmallT / 32; w++) {
                const uint32_t c = s.wh[w][tid];
                s.wh[w][tid] = (uint16_t)tot;
                tot += c;
            }
            x = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) s.wsum[warp] = x;
        }
        __syncthreads();
        if (tid < 256) {
            uint32_t add = 0;
            for (int w = 0; w < warp; w++) add += s.wsum[w];
            s.bexcl[tid] = x - tot + add;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSmallI; r++) {
            if (i0 + 32u * r < n) {
                const uint32_t d = (kr[r] >> shift) & 255u, p = s.bexcl[d] + s.wh[warp][d] + rank[r];
                s.k[p] = kr[r];
                s.v[p] = vr[r];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSmallI; r++) {
            const uint32_t i = i0 + 32u * r;
            kr[r] = i < n ? s.k[i] : 0u;
            vr[r] = i < n ? s.v[i] : 0u;
        }
    }
    // keys and primitives in order; tiles of each primitive and their exclusive scan
    // (thread t: items 8 t ... 8 t + 7)
#pragma unroll
    for (int r = 0; r < kSmallI; r++) {
        const uint32_t i = i0 + 32u * r;
        if (i < n) {
            key[i] = kr[r];
            val[i] = vr[r];
        }
    }
    uint2 rc[kSmallI];
    uint32_t c[kSmallI];
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < kSmallI; k++) {
        const uint32_t j = (uint32_t)tid * kSmallI + (uint32_t)k;
        rc[k] = j < n ? rects[s.v[j]] : make_uint2(0u, 0u);
        c[k] = rect_tiles(rc[k]);
        sum += c[k];
    }
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __shared__ unsigned long long wtot[kSmallT / 32];
    if (lane == 31) wtot[warp] = x;
    __syncthreads();
    unsigned long long run = x - sum, all = 0;
    for (int w = 0; w < kSmallT / 32; w++) {
        run += w < warp ? wtot[w] : 0ull;
        all += wtot[w];
    }
#pragma unroll
    for (int k = 0; k < kSmallI; k++) {
        const uint32_t j = (uint32_t)tid * kSmallI + (uint32_t)k;
        if (j < n) {
            cnt[j] = c[k];
            off[j] = (uint32_t)run;
            srect[j] = rc[k];
        }
        run += c[k];
    }
    if (tid == 0) {
        total[0] = all < cap ? all : cap;     // usable pair count
        total[1] = all > cap ? 1ull : 0ull;   // overflow flag
        total[2] = all;                       // true pair count
    }
}

int radix_blocks(uint64_t cap) { return (int)std::max<uint64_t>(1, div_up(cap, (uint64_t)kRT * radix_items(cap))); }
// the most blocks of any pass over up to cap items
int radix_blocks_upto(uint64_t cap) {
    return std::max({radix_blocks(cap), radix_blocks(std::min(cap, kItems4)), radix_blocks(std::min(cap, kItems8))});
}

int hist_parts(int nblocks) { return (int)div_up((uint64_t)256 * nblocks, kScanTile); }

// one stable LSD radix sort over `bits` key bits; `cur` returns the index
// (0/1) of the buffer holding the result.  The (digit, block) histogram is
// scanned by block partials -> single-block scan of the partials -> apply.
gs_status radix_sort(uint32_t* k[2], uint32_t* v[2], const unsigned long long* dcount, uint64_t cap, int bits,
                     uint32_t* hist, unsigned long long* hpart, int& cur, cudaStream_t st) {
    const int nblocks = radix_blocks(cap);
    // up to 16,384 blocks a column per digit is short enough for one block to scan
    // (only the blocks that hold items are scanned); beyond, the table is scanned
    // by all blocks (partials, their scan, apply)
    const bool by_column = nblocks <= 16384;
    uint32_t* dtot = by_column ? reinterpret_cast<uint32_t*>(hpart) : nullptr;   // 256 digit totals
    const uint64_t hlen = (uint64_t)256 * nblocks;
    const int nparts = hist_parts(nblocks), items = radix_items(cap);
    unsigned long long* htot = hpart + nparts + 1;   // scratch for the partial scan's totals
    auto khist = items == 4 ? k_radix_hist<4> : (items == 8 ? k_radix_hist<8> : k_radix_hist<16>);
    auto kscatter = items == 4 ? k_radix_scatter<4> : (items == 8 ? k_radix_scatter<8> : k_radix_scatter<16>);
    for (int shift = 0; shift < bits; shift += 8) {
        khist<<<nblocks, kRT, 0, st>>>(k[cur], dcount, cap, shift, hist, nblocks, by_column ? 0 : 1);
        if (by_column) {
            k_radix_colscan<<<256, kRT, 0, st>>>(hist, nblocks, kRT * items, dcount, cap, dtot);
        } else {
            k_scan_partials<<<nparts, kScanBlockT, 0, st>>>(hist, hlen, hpart);
            k_scan_partials_top<<<1, kScanT, 0, st>>>(hpart, nparts, htot, ~0ull);
            k_scan_apply<<<nparts, kScanBlockT, 0, st>>>(hist, hlen, hpart, hist);
        }
        kscatter<<<nblocks, kRT, 0, st>>>(k[cur], v[cur], k[cur ^ 1], v[cur ^ 1], dcount, cap, shift, hist, nblocks,
                                          dtot);
        cur ^= 1;
    }
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

}  // namespace

// Grows w to n primitives, cap_pairs pairs and a grid of ntiles tiles.  What a growth
// frees is NULL, and its size 0, until all of it is there again: a failure part way
// leaves nothing that a later, smaller call could take for usable.
gs_status alloc_render_work(RenderWork& w, uint64_t n, uint64_t cap_pairs, int ntiles) {
    auto A = [](auto*& p, uint64_t items) -> gs_status {   // p: room for `items`, its old content gone
        cudaFree(p);
        p = nullptr;
        const cudaError_t e = cudaMalloc((void**)&p, std::max<uint64_t>(items, 1) * sizeof(*p));
        if (e == cudaSuccess) return GS_OK;
        cudaGetLastError();
        p = nullptr;
        return set_error(GS_ERR_OOM, std::string("cudaMalloc failed for render scratch: ") + cudaGetErrorString(e));
    };
    if (n > w.n || !w.recs) {
        w.n = 0;
        GS_TRY(A(w.srect, n));
        GS_TRY(A(w.rects, n));
        for (int i = 0; i < 2; i++) {
            GS_TRY(A(w.dkey[i], n));
            GS_TRY(A(w.dval[i], n));
        }
        GS_TRY(A(w.cnt, n));
        GS_TRY(A(w.off, n));
        // block sums of the scans (8 B each), then the large primitives' list and its length
        GS_TRY(A(w.scan_tmp, 2 * (div_up(std::max<uint64_t>(n, 1), kScanTile) + 1) + n + 16));
        GS_TRY(A(w.recs, n));   // last: it says that they are all there
        w.n = n;
    }
    if (cap_pairs > w.cap_pairs || !w.pval[0]) {
        w.cap_pairs = 0;
        GS_TRY(A(w.pval[0], cap_pairs));
        w.cap_pairs = cap_pairs;
    }
    // the pair sort's other buffers: only for grids that are not listed by counting
    const bool radix = !listed_by_counting(n, ntiles);
    if (radix && w.cap_pairs > w.radix_pairs) {
        w.radix_pairs = 0;
        GS_TRY(A(w.pkey[0], w.cap_pairs));
        GS_TRY(A(w.pkey[1], w.cap_pairs));
        GS_TRY(A(w.pval[1], w.cap_pairs));
        w.radix_pairs = w.cap_pairs;
    }
    const uint64_t big = std::max<uint64_t>({w.radix_pairs, w.n, (uint64_t)1});
    if (big > w.hist_items) {
        w.hist_items = 0;
        const int hb = radix_blocks_upto(big);
        GS_TRY(A(w.hist, 256ull * hb));
        GS_TRY(A(w.hpart, std::max(hist_parts(hb) + 8, 136)));
        w.hist_items = big;
    }
    if (!radix) {
        const size_t need = direct_tab_words(std::max(ntiles, 1), w.cap_pairs);
        if (need > w.tab_words) {
            w.tab_words = 0;
            GS_TRY(A(w.tab, need));
            w.tab_words = need;
        }
    }
    if (ntiles > w.ntiles_cap || !w.ranges) {
        w.ntiles_cap = 0;
        GS_TRY(A(w.ranges, std::max(ntiles, 1)));
        w.ntiles_cap = ntiles;
    }
    if (!w.total) GS_TRY(A(w.total, 8));
    if (!w.host_total && cudaMallocHost((void**)&w.host_total, sizeof(unsigned long long) * 8) != cudaSuccess) {
        cudaGetLastError();
        w.host_total = nullptr;
        return set_error(GS_ERR_OOM, "cudaMallocHost failed");
    }
    return GS_OK;
}

// Device bytes of a scratch of these sizes (see alloc_render_work).
static size_t work_bytes(uint64_t n, uint64_t pairs, uint64_t radix_pairs, uint64_t hist_items, size_t tab_words,
                         int ntiles) {
    const int hb = radix_blocks_upto(std::max<uint64_t>(hist_items, 1));
    const size_t prims = n * (sizeof(BlendRec) + 2 * sizeof(uint2) + 7 * 4) + 8 * (div_up(n, kScanTile) + 1) + 64;
    const size_t radix = 12 * radix_pairs + 1024ull * hb + 8ull * std::max(hist_parts(hb) + 8, 136);
    return prims + 4 * pairs + radix + 4 * tab_words + sizeof(uint2) * (size_t)ntiles + 64;
}
size_t render_work_bytes(uint64_t n, uint64_t pairs, int ntiles) {
    const bool radix = !listed_by_counting(n, ntiles);
    return work_bytes(n, pairs, radix ? pairs : 0, std::max<uint64_t>(radix ? pairs : 0, n),
                      radix ? 0 : direct_tab_words(std::max(ntiles, 1), pairs), ntiles);
}
size_t render_work_bytes(const RenderWork& w) {
    return w.recs ? work_bytes(w.n, w.cap_pairs, w.radix_pairs, w.hist_items, w.tab_words, w.ntiles_cap) : 0;
}

void free_render_work(RenderWork& w) {
    cudaFree(w.recs);
    cudaFree(w.rects);
    for (int i = 0; i < 2; i++) {
        cudaFree(w.dkey[i]);
        cudaFree(w.dval[i]);
        cudaFree(w.pkey[i]);
        cudaFree(w.pval[i]);
    }
    cudaFree(w.cnt);
    cudaFree(w.off);
    cudaFree(w.srect);
    cudaFree(w.tab);
    cudaFree(w.hist);
    cudaFree(w.hpart);
    cudaFree(w.scan_tmp);
    cudaFree(w.ranges);
    cudaFree(w.total);
    if (w.host_total) cudaFreeHost(w.host_total);
    w = RenderWork();
}

// Sorts the preprocess output in w (dkey[0] = depth keys, dval[0] = primitive
// ids, rects) into per-tile lists: w.ranges[tile] and the id array returned in
// *ids_out.  total[0] = usable pair count, total[1] = overflow flag.
gs_status build_tile_lists(RenderWork& w, uint64_t n, int tiles_x, int tiles_y, uint32_t** ids_out, cudaStream_t st) {
    int ntiles = tiles_x * tiles_y;
    // every segment's rows are written, so the tables have to hold them all
    const bool counting = listed_by_counting(n, ntiles);
    if (counting && direct_words(direct_shape(ntiles, w.cap_pairs), ntiles) > w.tab_words)
        return set_error(GS_ERR_CAPACITY, "the counting tables were not sized for this tile grid");
    int cur = 0;
    unsigned blocks = (unsigned)div_up(std::max<uint64_t>(n, 1), 256);
    int nparts = (int)std::max<uint64_t>(div_up(n, kScanTile), 1);
    unsigned long long* part = (unsigned long long*)w.scan_tmp;
    uint32_t* big_list = (uint32_t*)(part + nparts + 1);
    unsigned int* big_count = big_list + std::max<uint64_t>(n, 1);
    if (n <= kSmallN) {   // one block does all of it
        const int smem = (int)sizeof(SmallSort);
        GS_CUDA(cudaFuncSetAttribute(k_order_small, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        k_order_small<<<1, kSmallT, smem, st>>>(w.dkey[0], w.dval[0], w.rects, (uint32_t)n, w.cnt, w.off, w.srect,
                                               w.total, w.cap_pairs);
    } else {
        // depth order of the primitives, then tiles per primitive in that order, their
        // exclusive scan and the pair count
        GS_TRY(radix_sort(w.dkey, w.dval, nullptr, n, 32, w.hist, w.hpart, cur, st));
        k_count_tiles<<<blocks, 256, 0, st>>>(w.dval[cur], w.rects, n, w.cnt, w.srect);
        k_scan_partials<<<nparts, kScanBlockT, 0, st>>>(w.cnt, n, part);
        k_scan_partials_top<<<1, kScanT, 0, st>>>(part, nparts, w.total, w.cap_pairs);
        k_scan_apply<<<nparts, kScanBlockT, 0, st>>>(w.cnt, n, part, w.off);
    }
    const uint32_t* sorted_ids = w.dval[cur];
    w.cur = cur;
    w.passes[0] = 4;   // 32-bit depth keys, 8 bits a digit
    int tbits = 1;
    while ((1 << tbits) < ntiles) tbits++;
    w.passes[1] = (tbits + 7) / 8;
    if (counting) {
        const DirectShape d = direct_shape(ntiles, w.cap_pairs);
        const int thr = d.warps * 32;
        const int tpad = (ntiles + 7) & ~7;   // table rows: whole 16-byte pieces
        uint32_t *tab = w.tab, *tot = tab + (size_t)d.segs * tpad;
        uint16_t* wtab = reinterpret_cast<uint16_t*>(tot + tpad);
        // the largest any grid needs, not this one's: the attribute is the process's, and
        // another thread may list another grid between these lines and the launches
        const DirectShape most = direct_shape(kDirectTiles, 1);
        GS_CUDA(cudaFuncSetAttribute(k_tile_hist, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most.hist_smem));
        GS_CUDA(cudaFuncSetAttribute(k_tile_place, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most.place_smem));
        k_tile_hist<<<d.segs, thr, d.hist_smem, st>>>(sorted_ids, w.srect, w.off, (uint32_t)n, tiles_x, ntiles, w.total,
                                                      wtab, tab);
        GS_CUDA(cudaGetLastError());   // the placing walk writes where these counts say
        k_tile_colscan<<<(ntiles + 31) / 32, 1024, 0, st>>>(tab, ntiles, tpad, d.segs, w.total, tot);
        k_tile_starts<<<1, kScanT, 0, st>>>(tot, ntiles, w.total, w.ranges);
        k_tile_place<<<d.segs, thr, d.place_smem, st>>>(sorted_ids, w.srect, w.off, (uint32_t)n, tiles_x, ntiles,
                                                        w.total, wtab, tab, tot, w.pval[0]);
        GS_CUDA(cudaGetLastError());
        *ids_out = w.pval[0];
        return GS_OK;
    }
    GS_CUDA(cudaMemsetAsync(big_count, 0, sizeof(unsigned int), st));
    k_emit<<<blocks, 256, 0, st>>>(sorted_ids, w.rects, w.cnt, w.off, n, tiles_x, w.total, w.pkey[0], w.pval[0],
                                   big_list, big_count);
    k_emit_big<<<num_sms() * 2, 256, 0, st>>>(sorted_ids, w.rects, w.off, tiles_x, w.total, w.pkey[0], w.pval[0],
                                              big_list, big_count);
    // stable sort of the pairs by tile id
    int pcur = 0;
    GS_TRY(radix_sort(w.pkey, w.pval, w.total, w.cap_pairs, tbits, w.hist, w.hpart, pcur, st));
    GS_CUDA(cudaMemsetAsync(w.ranges, 0, sizeof(uint2) * ntiles, st));
    k_ranges<<<num_sms() * 8, 256, 0, st>>>(w.pkey[pcur], w.total, w.cap_pairs, w.ranges);
    GS_CUDA(cudaGetLastError());
    *ids_out = w.pval[pcur];
    return GS_OK;
}

// exclusive scan of n u32 values into out (n entries); total[0..2] (device) gets
// the sum; scratch: div_up(n, kScanTile) + 1 u64
gs_status launch_exclusive_scan(const uint32_t* in, uint64_t n, uint32_t* out, unsigned long long* scratch,
                                unsigned long long* total, cudaStream_t st) {
    const int nparts = (int)std::max<uint64_t>(div_up(n, kScanTile), 1);
    k_scan_partials<<<nparts, kScanBlockT, 0, st>>>(in, n, scratch);
    k_scan_partials_top<<<1, kScanT, 0, st>>>(scratch, nparts, total, ~0ull);
    k_scan_apply<<<nparts, kScanBlockT, 0, st>>>(in, n, scratch, out);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}
uint64_t scan_scratch_len(uint64_t n) { return std::max<uint64_t>(div_up(n, kScanTile), 1) + 1; }

gs_status launch_ranges_to_offsets(const uint2* ranges, int ntiles, uint32_t* offsets,
                                   const unsigned long long* total, cudaStream_t st) {
    k_ranges_to_offsets<<<(ntiles + 255) / 256, 256, 0, st>>>(ranges, ntiles, offsets);
    k_offsets_fixup<<<1, 32, 0, st>>>(offsets, ntiles, total);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_rects_to_keys(const float* depth, const int32_t* rects, uint64_t n, int tiles_x, int tiles_y,
                               uint32_t* keys, uint32_t* vals, uint2* prects, cudaStream_t st) {
    if (n == 0) return GS_OK;
    k_rects_to_keys<<<(unsigned)div_up(n, 256), 256, 0, st>>>(depth, rects, n, tiles_x, tiles_y, keys, vals, prects);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

}  // namespace gs
