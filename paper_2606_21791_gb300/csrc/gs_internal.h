// Internal declarations shared by the libgs translation units (GPU path only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/gs.h"

namespace gs {

// Render tiles are tw x th pixels, tw and th in {8, 16, 32} with 64 <= tw * th
// <= 256 (a scene's shape is set by gs_set_tile; 16 x 16 by default).  A tile's
// pixels are numbered in 8x4 blocks ("natural order"): pixel u = 32 w + lane of
// block w sits at (8 (w % nbx) + lane % 8, 4 (w / nbx) + lane / 8), nbx = tw / 8.
// The dirty-tile blend works on 8x8 blocks (one warp, two pixels per lane):
// block b is the 8x4 blocks wA = b % nbx + 2 nbx (b / nbx) and wA + nbx.
constexpr int kTile = 16;                   // default tile edge; the full-frame SSIM's own tile edge
constexpr int kTilePix = 256;               // most pixels in a tile
constexpr int kDirtyBlocks = kTilePix / 64; // most 8x8 blocks in a tile
__host__ __device__ inline bool tile_shape_ok(int tw, int th) {
    const bool ew = tw == 8 || tw == 16 || tw == 32, eh = th == 8 || th == 16 || th == 32;
    return ew && eh && tw * th >= 64 && tw * th <= kTilePix;
}
// log2 of the 8x4 blocks per tile row (tw / 8 = 1, 2, 4)
__host__ __device__ inline int tile_lgx(int tw) { return tw == 8 ? 0 : (tw == 16 ? 1 : 2); }
constexpr int kMaxWords = 59;
constexpr int kMaxPairs = 65536;      // (variant, view) pairs per dirty-tile batch
constexpr uint64_t kMaxCands = 1ull << 28;   // candidate tiles a batch has room for, unless it is small (20 B each)
constexpr int kSmallPairs = 8192, kSmallBatch = 2048;   // such a batch; also the largest with SSIM on
constexpr int kRowStride = 64;        // list entries from one row to the next (see ViewPtrs)
constexpr int kRowsPerTile = 64;      // rows of a tile after row 0
constexpr int kWalk = 4;              // blend-list entries taken at a time: 64 bytes
// first bit of the sign and exponent bits a sign+exponent code protects
__host__ __device__ inline int ecc_first_bit(int fmt) { return fmt == GS_FP32 ? 23 : (fmt == GS_FP16 ? 10 : 7); }
constexpr int kSseFracBits = 39;      // fixed-point scale of per-pixel squared errors (3 * 2^39 * 5.1e6 px < 2^64)

// ----------------------------------------------------------------------------
// error reporting
// ----------------------------------------------------------------------------
gs_status set_error(gs_status st, const std::string& msg);
gs_status cuda_error(cudaError_t e, const char* what);
#define GS_CUDA(call)                                          \
    do {                                                       \
        cudaError_t _e = (call);                               \
        if (_e != cudaSuccess) return gs::cuda_error(_e, #call); \
    } while (0)
#define GS_TRY(call)                          \
    do {                                      \
        gs_status _s = (call);                \
        if (_s != GS_OK) return _s;           \
    } while (0)

inline int words_for_degree(int d) { return 14 + ((d + 1) * (d + 1) - 1) * 3; }
inline int word_bytes(int fmt) { return fmt == GS_FP32 ? 4 : 2; }
inline uint64_t div_up(uint64_t a, uint64_t b) { return (a + b - 1) / b; }

// ----------------------------------------------------------------------------
// device-side records
// ----------------------------------------------------------------------------
// Blend record of one primitive in one view (48 B, 16-B aligned).  ex, ey are
// the half extents (pixels) of a box that contains every pixel centre where the
// primitive's alpha can reach 1/255 (NaN if the opacity is NaN: never culled;
// negative if it can never reach 1/255).
struct __align__(16) BlendRec {
    float mx, my, ca, cb;
    float cc, opac, ex, ey;
    float r, g, b, depth;
};

// Camera with the per-view constants the preprocess needs.
struct DevCamera {
    float R[9];
    float t[3];
    float fx, fy, cx, cy;
    int W, H;
    float znear, zfar;
    int tiles_x, tiles_y;
    int tile_w, tile_h;   // render tile shape
};

// Per (variant, view) comparison accumulator (integer/ordered atomics only, so
// the result does not depend on the order in which tiles finish).
struct CmpAcc {
    unsigned long long sse_fx;  // sum of per-pixel squared errors, each rounded to fixed point 2^-kSseFracBits
    unsigned int maxabs_bits;   // float bits of the max |diff| (non-negative floats order as uints)
    unsigned int footprint;
    unsigned int nonfinite;
    unsigned int clamps;
    unsigned int clean_nonfinite_replaced;   // dirty engine: re-blended pixels whose clean value was non-finite
    unsigned int pad;
    unsigned long long reg_actual;   // dirty engine: 8x8 screen cells holding a footprint pixel
    unsigned long long reg_pred;     // dirty engine: cells met by the changed primitive's tile rects
    unsigned long long ssim_fx;      // sum over pixels and channels of (1 - SSIM), fixed point 2^-32 (signed)
};

// Screen cells of the contamination masks: an 8x8 grid, cell of pixel (x, y) =
// (8x / W, 8y / H), bit 8 cy + cx.
__host__ __device__ inline unsigned long long cell_bit(int x, int y, int W, int H) {
    // x < W <= 65535 * 16, so 8 x fits 32 bits
    const int cx = (int)((unsigned)x * 8u / (unsigned)W), cy = (int)((unsigned)y * 8u / (unsigned)H);
    return 1ull << (cy * 8 + cx);
}
// cells met by the pixels of a tile rect (packed x0 | y0 << 16, x1 | y1 << 16, half
// open in tiles of tw x th pixels)
__host__ __device__ inline unsigned long long rect_cells(uint2 rect, int W, int H, int tw, int th) {
    const int x0 = rect.x & 0xffff, y0 = rect.x >> 16, x1 = rect.y & 0xffff, y1 = rect.y >> 16;
    if (x1 <= x0 || y1 <= y0) return 0ull;
    const int px1 = min(x1 * tw, W) - 1, py1 = min(y1 * th, H) - 1;
    const int cx0 = (int)(((long long)x0 * tw * 8) / W), cx1 = (int)(((long long)px1 * 8) / W);
    const int cy0 = (int)(((long long)y0 * th * 8) / H), cy1 = (int)(((long long)py1 * 8) / H);
    unsigned long long m = 0ull;
    for (int cy = cy0; cy <= cy1; cy++)
        for (int cx = cx0; cx <= cx1; cx++) m |= 1ull << (cy * 8 + cx);
    return m;
}

struct ViewPtrs {
    const BlendRec* recs;
    const uint32_t* ids;
    const uint32_t* rank;    // place of each primitive in the view's (depth, index) order
    const uint32_t* sdk;     // that order: depth keys
    const uint32_t* sid;     // and primitives
    const uint2* rects;
    const uint2* ranges;
    const float* clean;
    const uint32_t* stop;        // rank of the entry that stopped each clean pixel (tile, natural order)
    const uint32_t* tile_stop;   // the largest of them in each tile
    const uint32_t* row_idx;     // rows of every pixel of a tile, tile order: where its blend list continues (into ent / rk)
    const uint32_t* row_off;     // first row of each tile (row 0: the lists' starts)
    const uint32_t* row_key;     // [tile][kRowsPerTile] rank of the last entry before row 1, 2, ... (0xffffffff: no row)
    const float4* ent;           // pixel blend lists: (alpha, colour) of the entries a pixel blends, front to back
    const uint32_t* rk;          // their ranks
    const float4* state;         // clean blend (T, C) in front of every kWalk-th entry of the lists
    int W, H, tiles_x, tile_w, tile_h;
    uint32_t bin0;               // tiles of the views before this one
    // a dense view (no blend lists): per 8x8 block the entries of its tile's list that
    // its cull leaves, as (primitive, rank), and the clean blend (T, C) of its pixels in
    // front of every kRowStride-th of them
    const uint2* sub;
    const uint32_t* sub_off;
    const uint32_t* sub_cnt;
    const float4* row_state;
};

constexpr uint32_t kNoRank = 0xfffffffeu;   // above every primitive's rank, below a list's end (0xffffffff)

// Candidate tile of a batch: x = (variant, view) | 8x8 blocks to look at << 20 |
// view << 24, y = tile x | tile y << 16.
constexpr int kUnitVars = 16;   // candidates a block of the dirty blend takes at a time
constexpr uint32_t kCandPair = (1u << 20) - 1u;
static_assert(kMaxPairs <= (1 << 20), "a candidate packs its pair into 20 bits");

// One dirty tile that is re-blended, kept for the dirty-tile SSIM (48 B): mask
// marks the tile's active pixels (natural order, 8 x 32 bits).
struct __align__(16) PlanItem {
    uint32_t mask[kTilePix / 32];
    uint32_t bk;      // (variant, view) = variant * K + view
    uint32_t tile;
    uint32_t pad[2];
};
static_assert(sizeof(PlanItem) == 48, "k_plan writes PlanItem as 3 16-byte parts");

// Buffers of the dirty-tile SSIM (all NULL when it is off): per plan slot the
// delta index of each of its 8x4 blocks (0xffffffff: none), per delta index the
// new values of the block's 32 pixels, per (variant, view) and tile the plan
// slot (generation << 32 | slot) and the SSIM claim (generation << 32).
struct SsimBufs {
    PlanItem* plan;                    // [slot_cap] the re-blended tiles
    uint32_t* slot_group;              // [slot_cap * 8]
    uint32_t* slot_flags;              // [slot_cap] changed pixels: bit 4 any, 0-3 within 5 of the left/right/top/bottom edge
    float4* deltas;                    // [delta_cap * 32]
    unsigned long long* tile_map;      // [B*K * max_tiles]
    unsigned long long* ssim_map;      // [B*K * max_tiles]
    unsigned int* overflow;            // set when a capacity is exceeded
    uint32_t* claims;                  // [slot_cap * 9] claimed tiles: plan slot * 9 + neighbour
    uint32_t slot_cap, delta_cap, max_tiles, pad;
};

// Dirty-tile work descriptor of one (variant, view).  An empty rect: the record
// is not there (not binned, or alpha < 1/255 everywhere).
struct __align__(16) DirtyDesc {
    BlendRec rec;          // corrupted primitive's record
    BlendRec old;          // clean primitive's record
    uint16_t nx0, ny0, nx1, ny1;   // corrupted rect
    uint16_t ox0, oy0, ox1, oy1;   // clean rect
    uint32_t new_rank;     // clean entries of lower rank lie in front of the corrupted one (kNoRank: not there)
    uint32_t old_rank;     // the clean entry's rank (kNoRank: not there)
    uint32_t pad[2];
};

// The union of the half-open intervals [n0, n1) and [o0, o1) as a list: first
// [n0, n1), then what [o0, o1) has outside it.
struct Union1 {
    int n0, nlen, o0, left, right0, len;
    __host__ __device__ Union1(int a0, int a1, int b0, int b1) {
        const bool none = a1 <= a0;
        n0 = none ? b0 : a0;
        nlen = none ? 0 : a1 - a0;
        o0 = b0;
        const int n1 = n0 + nlen;
        left = max(0, min(b1, n0) - b0);
        right0 = max(b0, n1);
        len = nlen + left + max(0, b1 - right0);
    }
    __host__ __device__ int at(int j) const {
        if (j < nlen) return n0 + j;
        const int r = j - nlen;
        return r < left ? o0 + r : right0 + (r - left);
    }
};

// The tile lists' pair stream: run w of `runs` equal ones over pairs [0, total), and the
// step from 64 pairs to the next of [.., end).  Totals go up to 2^32 - 2: no sum here
// passes 32 bits.
__host__ __device__ inline void pair_run(uint32_t total, uint32_t runs, uint32_t w, uint32_t& p0, uint32_t& p1) {
    const uint32_t len = total / runs + (total % runs != 0u ? 1u : 0u);
    const uint64_t at = (uint64_t)w * len;
    p0 = at < total ? (uint32_t)at : total;
    p1 = total - p0 > len ? p0 + len : total;
}
__host__ __device__ inline bool pair_next(uint32_t& b, uint32_t end) {
    if (end - b <= 64u) return false;
    b += 64u;
    return true;
}

// ----------------------------------------------------------------------------
// per-view clean state and scratch
// ----------------------------------------------------------------------------
// A device allocation that its owner keeps and reuses (reserve / release in
// gs_api.cu).
struct Buf {
    void* p = nullptr;
    size_t cap = 0;
};

struct ViewState {
    DevCamera cam{};
    BlendRec* recs = nullptr;        // [n]
    uint2* rects = nullptr;          // [n] (x0 | y0 << 16, x1 | y1 << 16)
    uint32_t* rank = nullptr;        // [n] place in the view's (depth, index) order
    uint32_t* sdk = nullptr;         // [n] depth keys in that order
    uint32_t* sid = nullptr;         // [n] primitives in that order
    uint32_t* ids = nullptr;         // [npairs] sorted tile lists
    uint2* ranges = nullptr;         // [ntiles] (start, end)
    float* clean = nullptr;          // [H*W*3]
    uint32_t* stop = nullptr;        // [ntiles][pixels of a tile] rank of the entry that stopped the clean pixel
    uint32_t* tile_stop = nullptr;   // [ntiles] the largest of them
    uint32_t* tile_last = nullptr;   // [ntiles] largest list position that stopped a pixel (build only)
    uint32_t* row_idx = nullptr;     // [rows][pixels of a tile] where each pixel's blend list continues
    uint32_t* row_off = nullptr;     // [ntiles] first row
    uint32_t* row_cnt = nullptr;     // [ntiles] rows after row 0 (build only)
    uint32_t* row_key = nullptr;     // [ntiles][kRowsPerTile] rank of the last entry before each row after row 0
    float4* ent = nullptr;           // pixel blend lists (alpha, r, g, b)
    uint32_t* rk = nullptr;          // their ranks
    float4* state = nullptr;         // clean blend in front of every kWalk-th entry of the lists
    uint2* sub = nullptr;            // dense views, in place of the five above: block lists (see ViewPtrs)
    uint32_t* sub_off = nullptr;
    uint32_t* sub_cnt = nullptr;     // [8x8 blocks] entries that a block's cull leaves
    float4* row_state = nullptr;
    uint64_t npairs = 0;
    uint64_t cap_pairs = 0;
};

// Scratch of the full render pipeline for one view.
struct RenderWork {
    uint64_t n = 0;
    uint64_t cap_pairs = 0;
    int ntiles_cap = 0;
    BlendRec* recs = nullptr;
    uint2* rects = nullptr;
    uint32_t* dkey[2] = {nullptr, nullptr};    // depth keys (ping-pong)
    uint32_t* dval[2] = {nullptr, nullptr};    // primitive ids (ping-pong)
    uint32_t* cnt = nullptr;                    // tiles per primitive, in depth order
    uint32_t* off = nullptr;                    // exclusive scan of cnt
    uint2* srect = nullptr;                     // tile rects, in depth order
    uint32_t* tab = nullptr;                    // counting tables of the tile lists [tab_words]
    size_t tab_words = 0;
    uint32_t* pkey[2] = {nullptr, nullptr};    // pair tile keys
    uint32_t* pval[2] = {nullptr, nullptr};    // pair primitive ids ([0]: the lists when made by counting)
    uint64_t radix_pairs = 0;                   // pairs that pkey and pval[1] hold (large grids only)
    uint64_t hist_items = 0;                    // items that hist and hpart serve
    uint32_t* hist = nullptr;                   // radix histograms
    unsigned long long* hpart = nullptr;        // block partials of the histogram scan
    uint32_t* scan_tmp = nullptr;               // block sums for scans
    uint2* ranges = nullptr;
    unsigned long long* total = nullptr;        // [0] pair count, [1] overflow flag
    unsigned long long* host_total = nullptr;   // pinned mirror
    int passes[2] = {0, 0};                     // 8-bit digits of the last build's keys: depths, tile ids
    int cur = 0;                                // dkey / dval buffer that holds the last build's depth order
};

struct GraphEntry {
    int B = 0;
    int guard = -2;
    uint64_t mask = 0;
    bool ssim = false;
    bool regions = false;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

}  // namespace gs

struct gs_scene {
    uint64_t n = 0;
    int sh_degree = 0;
    int fmt = 0;
    int nwords = 0;
    void* planes = nullptr;                 // [nwords][n]
    uint32_t box_lo[gs::kMaxWords] = {};    // FIELD box (storage words)
    uint32_t box_hi[gs::kMaxWords] = {};
    void* pbox_lo = nullptr;                // PRIM box planes [nbox][n]
    void* pbox_hi = nullptr;
    int nbox_words = 0;
    uint32_t* dev_box = nullptr;            // FIELD box on device: lo[59], hi[59]
    unsigned int* dev_err = nullptr;        // sticky device error flags (bit 0: bad flip site)
    unsigned long long* dev_clamps = nullptr;

    // clean per-view state of the campaign
    int K = 0;
    std::vector<gs::ViewState> views;
    std::vector<gs::Buf> view_bufs;         // two per view: they hold all of its state; kept from one gs_set_views to the next
    gs::Buf list_tmp;                       // scratch of a view's build
    gs::DevCamera* dev_cams = nullptr;
    void* dev_views = nullptr;              // ViewPtrs[K]
    uint64_t full_cap_pairs = 0;
    int max_tiles = 0;
    int max_tiles_y = 0;
    uint32_t all_tiles = 0;                 // tiles of all views
    gs::RenderWork work;                    // scratch of the full render pipeline
    int tile_w = gs::kTile, tile_h = gs::kTile;   // render tile shape (gs_set_tile)
    std::vector<gs_camera> host_cams;       // the cameras of gs_set_views (rebuilt on a tile change)

    // batch buffers (dirty engine and plain loop)
    size_t batch_room = ~(size_t)0;         // most bytes the batch buffers may take (see allow_batch_growth)
    bool batch_short = false;               // the last campaign ran in smaller batches for lack of memory
    int cap_B = 0;
    int cap_flips = 0;
    uint64_t cap_flip_mem = 0, cap_pairs = 0, cap_cands = 0, cap_rows = 0, cap_bins = 0;   // elements the buffers below hold
    gs_flip* flip_stage = nullptr;
    gs_flip* host_io_flips = nullptr;       // device copies of gs_inject_and_render_host's inputs / outputs
    gs_result* host_io_out = nullptr;
    size_t host_io_flips_cap = 0, host_io_out_cap = 0;
    gs::DirtyDesc* desc = nullptr;
    gs::CmpAcc* acc = nullptr;
    gs_result* res_stage = nullptr;
    unsigned int* queue = nullptr;          // batch counters (see k_plan)
    uint2* rows = nullptr;                  // tile rows to look at: (pair, tile y | view << 16) [pairs * max_tiles_y]
    uint2* cand = nullptr;                  // candidate tiles [pairs * max_tiles]
    uint32_t* cand_at = nullptr;            // their places inside their tile's bin (large batches)
    uint2* cand_sorted = nullptr;           // the same by tile (large batches)
    uint32_t* bins = nullptr;               // candidates per tile, then bin starts [all_tiles] (zero between batches)
    gs::SsimBufs ssim{};                    // dirty-tile SSIM buffers (allocated on first use, else NULL)
    unsigned int* clean_nonfin = nullptr;   // [K] non-finite pixels of each clean view
    uint32_t* saved = nullptr;
    bool use_graphs = true;
    int batch = 0;                          // variants per dirty-tile launch (0: default)
    unsigned long long* work_ctr = nullptr; // work counters, non-NULL while counting is on (no graphs then)
    cudaEvent_t ev_k0 = nullptr;            // timing on: before the plan kernel of the last batch,
    cudaEvent_t ev_kp = nullptr;            // between the plan and the blend kernel,
    cudaEvent_t ev_k1 = nullptr;            // after the blend kernel
    cudaEvent_t ev_r[4] = {};               // timing on, gs_render: before preprocess, after it, after the tile
                                            // lists, after the blend (last view of the last call)
    bool render_timed = false;              // ev_r holds a complete record
    uint64_t render_pairs = 0;              // tile pairs of that view
    std::vector<gs::GraphEntry> graphs;
};

namespace gs {

// k_guard.cu
int num_sms();
gs_status launch_field_box(const void* planes, int fmt, uint64_t n, int nwords, uint32_t* dev_keys, cudaStream_t st);
gs_status launch_guard(gs_scene* s, int mode, uint64_t mask, unsigned long long* dev_clamps, cudaStream_t st);
gs_status launch_guard_mark(gs_scene* s, int mode, uint64_t mask, uint32_t* bitmap, cudaStream_t st);
gs_status launch_save_sites(const void* planes, int fmt, uint64_t n, int nwords, const gs_flip* flips, int count,
                            uint32_t* saved, cudaStream_t st);
gs_status launch_restore_sites(void* planes, int fmt, uint64_t n, int nwords, const gs_flip* flips, int count,
                               const uint32_t* saved, cudaStream_t st);

// k_preprocess.cu
DevCamera make_dev_camera(const gs_camera& c, int tile_w, int tile_h);

// gs_api.cu: the camera sizes and focal lengths the kernels accept
bool valid_camera(const gs_camera& c);
// Device bytes a scene holds: parameters, boxes, views, scratch, batch buffers.
size_t scene_bytes(const gs_scene* s);
// Lets a campaign of B single upsets grow the scene's batch buffers by up to `room` bytes
// (it runs in smaller batches otherwise); returns by how much it will.
size_t allow_batch_growth(gs_scene* s, int B, size_t room);
void trim_batch_buffers(gs_scene* s);   // back to what gs_set_views allocates

// k_sort.cu
gs_status alloc_render_work(RenderWork& w, uint64_t n, uint64_t cap_pairs, int ntiles);
void free_render_work(RenderWork& w);
size_t render_work_bytes(const RenderWork& w);                                // device bytes it holds
size_t render_work_bytes(uint64_t n, uint64_t pairs, int ntiles);             // ... and would hold for one view
gs_status launch_rects_to_keys(const float* depth, const int32_t* rects, uint64_t n, int tiles_x, int tiles_y,
                               uint32_t* keys, uint32_t* vals, uint2* prects, cudaStream_t st);

// k_blend.cu (full-frame kernels take the view's camera for its size and tile shape)
gs_status launch_blend_image(const BlendRec* recs, const uint32_t* ids, const uint2* ranges, const DevCamera& cam,
                             float* img, cudaStream_t st);
gs_status launch_blend_compare(const BlendRec* recs, const uint32_t* ids, const uint2* ranges, const DevCamera& cam,
                               const float* clean, CmpAcc* acc, unsigned long long* work, cudaStream_t st);
gs_status launch_compare(const float* a, const float* b, int H, int W, int K, CmpAcc* acc, cudaStream_t st);
gs_status launch_finalize(const CmpAcc* acc, int count, gs_result* out, cudaStream_t st);
gs_status launch_records_to_blend(const gs_record* in, uint64_t n, BlendRec* out, cudaStream_t st);

}  // namespace gs
