// C ABI of libgs: scene lifetime, the full render pipeline, the batched
// dirty-tile injection campaign (captured in CUDA graphs), the plain
// one-variant-at-a-time loop, and stage entry points.  All device work is done
// by the kernels in k_*.cu; this file only orchestrates.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <mutex>
#include <string>

#include "gs_internal.h"

namespace gs {

// implemented in the kernel translation units
gs_status launch_apply_flips(void* planes, int fmt, uint64_t n, int nwords, const gs_flip* flips, int64_t count,
                             unsigned int* err, uint64_t ecc_mask, cudaStream_t st);
gs_status launch_preprocess(const gs_scene* s, const DevCamera& cam, BlendRec* recs, uint2* rects, uint32_t* keys,
                            uint32_t* vals, gs_record* dbg, cudaStream_t st);
gs_status launch_inject_prep(const gs_scene* s, const DevCamera* dev_cams, int K, const gs_flip* flips, int B,
                             int guard_mode, uint64_t mask, const void* dev_views, DirtyDesc* desc, uint2* rows,
                             CmpAcc* acc, unsigned int* queue, cudaStream_t st);
gs_status build_tile_lists(RenderWork& w, uint64_t n, int tiles_x, int tiles_y, uint32_t** ids_out, cudaStream_t st);
gs_status launch_ranges_to_offsets(const uint2* ranges, int ntiles, uint32_t* offsets, const unsigned long long* total,
                                   cudaStream_t st);
gs_status launch_zero_acc(CmpAcc* acc, int count, cudaStream_t st);
gs_status launch_dirty_blend(gs_scene* s, int BK, bool regions, const SsimBufs& sb, cudaStream_t st);
gs_status launch_ssim_out(const CmpAcc* acc, int count, const void* dev_views, int K, double* out, cudaStream_t st);
gs_status launch_regions_out(const CmpAcc* acc, int count, unsigned long long* out, cudaStream_t st);
gs_status launch_finalize_dirty(const CmpAcc* acc, int count, gs_result* out, const unsigned int* clean_nonfin, int K,
                                unsigned int* queue, cudaStream_t st);
size_t view_ptrs_size();
void fill_view_ptrs(void* host_dst, const ViewState& vs, uint32_t bin0);
gs_status launch_exclusive_scan(const uint32_t* in, uint64_t n, uint32_t* out, unsigned long long* scratch,
                                unsigned long long* total, cudaStream_t st);
uint64_t scan_scratch_len(uint64_t n);
gs_status launch_blend_clean(const ViewState& v, uint32_t* counts, uint32_t* blk_cnt, unsigned int* clean_nonfin,
                             cudaStream_t st);
gs_status launch_ranks(const uint32_t* key, const uint32_t* id, uint64_t n, const ViewState& v, cudaStream_t st);
gs_status launch_row_counts(const ViewState& v, uint32_t* rows, cudaStream_t st);
gs_status launch_list_lens(const uint32_t* counts, uint64_t n, uint32_t* lens, cudaStream_t st);
gs_status launch_fill_lists(const ViewState& v, const uint32_t* off, cudaStream_t st);
gs_status launch_offsets_to_ranges(const uint32_t* offsets, int ntiles, uint2* ranges, cudaStream_t st);
uint32_t key_to_bits(uint32_t key, int fmt);
void dirty_grids();

static thread_local std::string g_last_error;

gs_status set_error(gs_status st, const std::string& msg) {
    g_last_error = msg;
    return st;
}

gs_status cuda_error(cudaError_t e, const char* what) {
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    if (e == cudaErrorMemoryAllocation) return set_error(GS_ERR_OOM, m);
    return set_error(GS_ERR_CUDA, m);
}

// the camera sizes and focal lengths the kernels accept (tile coordinates fit 16
// bits for the smallest tile edge, 8)
bool valid_camera(const gs_camera& c) {
    return c.width > 0 && c.height > 0 && c.width <= 65535 * 8 && c.height <= 65535 * 8 && c.fx > 0 &&
           c.fy > 0 && std::isfinite(c.fx) && std::isfinite(c.fy);
}

namespace {

__global__ void k_move_clamps(unsigned long long* ctr, CmpAcc* acc) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        acc->clamps = (unsigned int)(*ctr < 0xffffffffull ? *ctr : 0xffffffffull);
        *ctr = 0ull;
    }
}

gs_status dmalloc(void** p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return set_error(GS_ERR_OOM, std::string("cudaMalloc(") + std::to_string(bytes) + "): " + cudaGetErrorString(e));
    }
    return GS_OK;
}

void release(Buf& b) {
    cudaFree(b.p);
    b = Buf{};
}

// At least `bytes` in b; what it holds stays unless it is too small, or far too
// large (twice the size and 64 MB).
gs_status reserve(Buf& b, size_t bytes) {
    if (b.p && b.cap >= bytes && b.cap <= 2 * bytes + (64ull << 20)) return GS_OK;
    release(b);
    GS_TRY(dmalloc(&b.p, bytes));
    b.cap = bytes;
    return GS_OK;
}

// Full render pipeline of one view on scratch `w`: preprocess, depth sort,
// pair emission, tile sort, ranges.  Leaves records in w.recs, lists in *ids.
// ev (optional, 3 events): recorded before the preprocess, after it and after the tile lists.
gs_status render_lists(gs_scene* s, RenderWork& w, const DevCamera& cam, uint32_t** ids, cudaStream_t st,
                       cudaEvent_t* ev = nullptr) {
    if (ev) GS_CUDA(cudaEventRecord(ev[0], st));
    GS_TRY(launch_preprocess(s, cam, w.recs, w.rects, w.dkey[0], w.dval[0], nullptr, st));
    if (ev) GS_CUDA(cudaEventRecord(ev[1], st));
    GS_TRY(build_tile_lists(w, s->n, cam.tiles_x, cam.tiles_y, ids, st));
    if (ev) GS_CUDA(cudaEventRecord(ev[2], st));
    return GS_OK;
}

// Like render_lists but grows the pair capacity until the lists fit (host sync).
gs_status render_lists_sized(gs_scene* s, RenderWork& w, const DevCamera& cam, uint32_t** ids, uint64_t* npairs,
                             cudaStream_t st, cudaEvent_t* ev = nullptr) {
    int ntiles = cam.tiles_x * cam.tiles_y;
    uint64_t cap = std::max<uint64_t>(w.cap_pairs, std::max<uint64_t>(s->n * 2, 1024));
    for (int attempt = 0; attempt < 4; attempt++) {
        GS_TRY(alloc_render_work(w, s->n, cap, ntiles));
        GS_TRY(render_lists(s, w, cam, ids, st, ev));
        GS_CUDA(cudaMemcpyAsync(w.host_total, w.total, 3 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
        w.host_total[3] = 0ull;
        GS_CUDA(cudaMemcpyAsync(&w.host_total[3], s->dev_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, st));
        GS_CUDA(cudaStreamSynchronize(st));
        if (w.host_total[3] & 2ull)
            return set_error(GS_ERR_TIMEOUT, "a bounded wait of the preprocess gave up (device error word bit 1)");
        if (!w.host_total[1]) {
            *npairs = w.host_total[0];
            return GS_OK;
        }
        uint64_t need = w.host_total[2];
        if (need >= 0xffffffffull) return set_error(GS_ERR_CAPACITY, "tile pair count exceeds 2^32");
        cap = need + need / 4 + 1024;
    }
    return set_error(GS_ERR_CAPACITY, "could not size the tile pair buffers");
}

void destroy_graphs(gs_scene* s) {
    for (auto& g : s->graphs) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        if (g.graph) cudaGraphDestroy(g.graph);
    }
    s->graphs.clear();
}

void free_ssim_buffers(gs_scene* s);

void free_views(gs_scene* s) {
    destroy_graphs(s);
    free_ssim_buffers(s);
    s->views.clear();
    s->K = 0;
    cudaFree(s->dev_cams);
    cudaFree(s->dev_views);
    cudaFree(s->clean_nonfin);
    s->clean_nonfin = nullptr;
    s->dev_cams = nullptr;
    s->dev_views = nullptr;
}

// the views' memory as well
void free_view_memory(gs_scene* s) {
    free_views(s);
    for (auto& b : s->view_bufs) release(b);
    s->view_bufs.clear();
    release(s->list_tmp);
}

void free_ssim_buffers(gs_scene* s) {
    cudaFree(s->ssim.plan);
    cudaFree(s->ssim.slot_group);
    cudaFree(s->ssim.slot_flags);
    cudaFree(s->ssim.deltas);
    cudaFree(s->ssim.tile_map);
    cudaFree(s->ssim.ssim_map);
    cudaFree(s->ssim.overflow);
    cudaFree(s->ssim.claims);
    s->ssim = SsimBufs{};
}

// Variants per batch with SSIM on: its buffers are sized for them.
int ssim_batch(int K) { return std::max(1, std::min(kSmallBatch, kSmallPairs / K)); }

// SSIM buffers (zeroed: generation 0 is never current)
static gs_status alloc_ssim_buffers(gs_scene* s) {
    const int K = std::max(s->K, 1), B = std::min(s->cap_B, ssim_batch(K));
    SsimBufs b{};
    b.max_tiles = (uint32_t)std::max(s->max_tiles, 1);
    const size_t maps = (size_t)B * K * b.max_tiles;
    b.slot_cap = (uint32_t)std::min<uint64_t>(maps, 3ull << 17);
    b.delta_cap = (uint32_t)std::min<uint64_t>((kTilePix / 32) * maps, 1ull << 19);
    s->ssim = b;   // caps now; pointers below
    GS_TRY(dmalloc((void**)&s->ssim.plan, sizeof(PlanItem) * b.slot_cap));
    GS_TRY(dmalloc((void**)&s->ssim.slot_group, sizeof(uint32_t) * 8 * b.slot_cap));
    GS_TRY(dmalloc((void**)&s->ssim.slot_flags, sizeof(uint32_t) * b.slot_cap));
    GS_TRY(dmalloc((void**)&s->ssim.deltas, sizeof(float4) * 32 * (size_t)b.delta_cap));
    GS_TRY(dmalloc((void**)&s->ssim.tile_map, sizeof(unsigned long long) * maps));
    GS_TRY(dmalloc((void**)&s->ssim.ssim_map, sizeof(unsigned long long) * maps));
    GS_TRY(dmalloc((void**)&s->ssim.overflow, sizeof(unsigned int)));
    GS_TRY(dmalloc((void**)&s->ssim.claims, sizeof(uint32_t) * 9 * (size_t)b.slot_cap));
    GS_CUDA(cudaMemset(s->ssim.tile_map, 0, sizeof(unsigned long long) * maps));
    GS_CUDA(cudaMemset(s->ssim.ssim_map, 0, sizeof(unsigned long long) * maps));
    GS_CUDA(cudaMemset(s->ssim.overflow, 0, sizeof(unsigned int)));
    return GS_OK;
}

// All or nothing: a set tile_map means every SSIM buffer is allocated and zeroed.
gs_status ensure_ssim_buffers(gs_scene* s) {
    if (s->ssim.tile_map) return GS_OK;
    const gs_status rs = alloc_ssim_buffers(s);
    if (rs != GS_OK) free_ssim_buffers(s);
    return rs;
}

void free_batch_buffers(gs_scene* s) {
    cudaFree(s->flip_stage);
    cudaFree(s->desc);
    cudaFree(s->acc);
    cudaFree(s->res_stage);
    cudaFree(s->queue);
    cudaFree(s->saved);
    cudaFree(s->rows);
    cudaFree(s->cand);
    cudaFree(s->cand_at);
    cudaFree(s->cand_sorted);
    cudaFree(s->bins);
    s->flip_stage = nullptr;
    s->desc = nullptr;
    s->acc = nullptr;
    s->res_stage = nullptr;
    s->queue = nullptr;
    s->saved = nullptr;
    s->rows = s->cand = s->cand_sorted = nullptr;
    s->cand_at = s->bins = nullptr;
    s->cap_B = 0;
    s->cap_flips = 0;
    s->cap_flip_mem = s->cap_pairs = s->cap_cands = s->cap_rows = s->cap_bins = 0;
}

// Elements of the batch buffers for cb variants and cf upsets: every (variant, view) can
// dirty at most every tile of its view.
struct BatchSize {
    uint64_t flips = 0, pairs = 0, cands = 0, rows = 0, bins = 0;
    size_t bytes() const {
        return flips * (sizeof(gs_flip) + 4) + pairs * (sizeof(DirtyDesc) + sizeof(CmpAcc) + sizeof(gs_result)) +
               cands * (2 * sizeof(uint2) + 4) + rows * sizeof(uint2) + bins * 4;
    }
};
BatchSize batch_size(const gs_scene* s, int cb, int cf) {
    BatchSize b;
    b.flips = (uint64_t)cf;
    b.pairs = (uint64_t)cb * std::max(s->K, 1);
    b.cands = b.pairs * (uint64_t)std::max(s->max_tiles, 1);
    b.rows = b.pairs * (uint64_t)std::max(s->max_tiles_y, 1);
    b.bins = std::max(s->all_tiles, 1u);
    return b;
}
BatchSize batch_held(const gs_scene* s) {
    return BatchSize{s->cap_flip_mem, s->cap_pairs, s->cap_cands, s->cap_rows, s->cap_bins};
}
bool batch_fits(const BatchSize& b, const BatchSize& held) {
    return b.flips <= held.flips && b.pairs <= held.pairs && b.cands <= held.cands && b.rows <= held.rows &&
           b.bins <= held.bins;
}

gs_status ensure_batch_buffers(gs_scene* s, int B, int fpv) {
    if (B <= s->cap_B && fpv * B <= s->cap_flips) return GS_OK;
    const int cb = std::max(B, s->cap_B);
    const int cf = std::max(fpv * B, s->cap_flips);
    const BatchSize need = batch_size(s, cb, cf);
    const uint64_t pairs = need.pairs, cands = need.cands, rows = need.rows, bins = need.bins;
    if (cands >= (1ull << 29)) return set_error(GS_ERR_CAPACITY, "too many dirty tiles per batch for this view size");
    destroy_graphs(s);
    free_ssim_buffers(s);
    // new views (which reset cap_B) fit the memory of the last ones as often as not
    if (!batch_fits(need, batch_held(s))) {
        // no capacity until every buffer below is allocated: a failure part way (out
        // of memory) leaves nothing that a later call could take for usable
        free_batch_buffers(s);
        GS_TRY(dmalloc((void**)&s->flip_stage, sizeof(gs_flip) * cf));
        GS_TRY(dmalloc((void**)&s->desc, sizeof(DirtyDesc) * pairs));
        GS_TRY(dmalloc((void**)&s->acc, sizeof(CmpAcc) * pairs));
        GS_TRY(dmalloc((void**)&s->res_stage, sizeof(gs_result) * pairs));
        GS_TRY(dmalloc((void**)&s->queue, sizeof(unsigned int) * 16));
        const unsigned int q0[16] = {0u, 0u, 0u, 0u, 0u, 0u, 1u};   // [6]: batch generation
        GS_CUDA(cudaMemcpy(s->queue, q0, sizeof(q0), cudaMemcpyHostToDevice));
        GS_TRY(dmalloc((void**)&s->saved, sizeof(uint32_t) * cf));
        GS_TRY(dmalloc((void**)&s->rows, sizeof(uint2) * rows));
        GS_TRY(dmalloc((void**)&s->cand, sizeof(uint2) * cands));
        GS_TRY(dmalloc((void**)&s->cand_at, sizeof(uint32_t) * cands));
        GS_TRY(dmalloc((void**)&s->cand_sorted, sizeof(uint2) * cands));
        GS_TRY(dmalloc((void**)&s->bins, sizeof(uint32_t) * bins));
        GS_CUDA(cudaMemset(s->bins, 0, sizeof(uint32_t) * bins));
        s->cap_flip_mem = (uint64_t)cf;
        s->cap_pairs = pairs;
        s->cap_cands = cands;
        s->cap_rows = rows;
        s->cap_bins = bins;
    }
    s->cap_B = cb;
    s->cap_flips = cf;
    return GS_OK;
}

// Most variants per dirty-tile batch: kMaxPairs (variant, view) pairs and
// kMaxCands candidate tiles, or a small batch whatever its tiles.  A large batch
// amortises the launches and the tail of the longest walks, and lets the variants
// that re-blend a tile share its blend lists in the L2: 50,000 upsets of a 134,826-
// primitive scene took 2.07 ms in 25 batches, 0.55 ms in one.
int max_batch(const gs_scene* s) {
    const uint64_t K = (uint64_t)std::max(s->K, 1), tiles = (uint64_t)std::max(s->max_tiles, 1);
    const uint64_t small = std::min<uint64_t>(kSmallBatch, kSmallPairs / K);
    return (int)std::max<uint64_t>(1, std::max(small, std::min<uint64_t>(kMaxPairs / K, kMaxCands / (K * tiles))));
}

// Allocations from this size on look at the free memory first (cudaMemGetInfo: 100 us).
constexpr size_t kLookBytes = 256ull << 20;

// Variants per batch of a campaign: the caller's choice, or the most.
int campaign_batch(const gs_scene* s) { return s->batch > 0 ? std::min(s->batch, max_batch(s)) : max_batch(s); }

// Variants the buffers of a call of B variants, at most `chunk` a batch, are sized for:
// powers of two, so that small calls hold little.
int batch_cap(int B, int chunk) {
    int cap = 64;
    while (cap < B && cap < chunk) cap *= 2;
    return std::min(cap, chunk);
}

// Buffers for a call of B variants (at most `chunk` a batch): a smaller batch where they
// would take more than batch_room, or than there is memory.  Free memory is looked at
// before large buffers are given up for larger ones, and before any once memory has run
// out: the next call of this size then settles for the same batch and keeps its buffers.
// Returns the variants a batch can have in *chunk.
gs_status size_batch(gs_scene* s, int B, int* chunk) {
    constexpr size_t kSlack = 16ull << 20;   // the allocator's granules
    while (true) {
        const int cap = batch_cap(B, *chunk);
        const BatchSize need = batch_size(s, std::max(cap, s->cap_B), std::max(cap, s->cap_flips)), held = batch_held(s);
        const size_t bytes = need.bytes();
        bool room = true;
        if (cap > 64 && !batch_fits(need, held)) {
            room = bytes <= s->batch_room;
            if (room && (bytes >= kLookBytes || s->batch_short)) {
                size_t avail = 0, all = 0;
                GS_CUDA(cudaMemGetInfo(&avail, &all));
                room = bytes + kSlack <= avail + held.bytes();
            }
        }
        const gs_status rs = room ? ensure_batch_buffers(s, cap, 1) : GS_ERR_OOM;
        if (rs == GS_OK) s->batch_short = s->batch_short && cap < batch_cap(B, campaign_batch(s));
        if (rs != GS_ERR_OOM || cap <= 64) return rs;
        s->batch_short = true;
        *chunk = cap / 2;
    }
}

gs_status check_flip_args(gs_scene* s, const gs_flip* flips, int B, int fpv, int guard_mode, uint64_t mask) {
    if (!s || (!flips && B > 0) || B < 0 || fpv < 1) return set_error(GS_ERR_ARG, "bad campaign arguments");
    if (s->K == 0 || s->views.empty()) return set_error(GS_ERR_STATE, "gs_set_views was not called");
    if (guard_mode < -1 || guard_mode > 2) return set_error(GS_ERR_ARG, "guard_mode must be -1, 0, 1 or 2");
    if (guard_mode == GS_GUARD_PRIM) {
        if (!s->pbox_lo) return set_error(GS_ERR_STATE, "no per-primitive box set");
        uint64_t allowed = s->nbox_words >= 64 ? ~0ull : ((1ull << s->nbox_words) - 1ull);
        if (mask & ~allowed) return set_error(GS_ERR_ARG, "PRIM guard mask covers words without boxes");
    }
    return GS_OK;
}

// enqueue one dirty-tile batch (B <= cap_B, flips already in flip_stage)
gs_status enqueue_dirty(gs_scene* s, int B, int guard_mode, uint64_t mask, bool ssim, bool regions, cudaStream_t st) {
    int K = s->K;
    GS_TRY(launch_inject_prep(s, s->dev_cams, K, s->flip_stage, B, guard_mode, mask, s->dev_views, s->desc, s->rows,
                              s->acc, s->queue, st));
    // external records: inside a stream capture they become event-record nodes of the graph
    if (s->ev_k0) GS_CUDA(cudaEventRecordWithFlags(s->ev_k0, st, cudaEventRecordExternal));
    GS_TRY(launch_dirty_blend(s, B * K, regions, ssim ? s->ssim : SsimBufs{}, st));
    if (s->ev_k1) GS_CUDA(cudaEventRecordWithFlags(s->ev_k1, st, cudaEventRecordExternal));
    GS_TRY(launch_finalize_dirty(s->acc, B * K, s->res_stage, s->clean_nonfin, K, s->queue, st));
    return GS_OK;
}

gs_status run_dirty_batch(gs_scene* s, int B, int guard_mode, uint64_t mask, bool ssim, bool regions,
                          cudaStream_t st) {
    if (!s->use_graphs || s->work_ctr) return enqueue_dirty(s, B, guard_mode, mask, ssim, regions, st);
    GraphEntry* ge = nullptr;
    for (auto& g : s->graphs)
        if (g.B == B && g.guard == guard_mode && g.mask == mask && g.ssim == ssim && g.regions == regions) ge = &g;
    if (!ge) {
        dirty_grids();
        cudaStream_t cs;
        GS_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        GraphEntry g;
        g.B = B;
        g.guard = guard_mode;
        g.mask = mask;
        g.ssim = ssim;
        g.regions = regions;
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) {
            cudaStreamDestroy(cs);
            return cuda_error(e, "cudaStreamBeginCapture");
        }
        gs_status qs = enqueue_dirty(s, B, guard_mode, mask, ssim, regions, cs);
        e = cudaStreamEndCapture(cs, &g.graph);
        cudaStreamDestroy(cs);
        if (qs != GS_OK) {
            if (g.graph) cudaGraphDestroy(g.graph);
            return qs;
        }
        if (e != cudaSuccess) return cuda_error(e, "cudaStreamEndCapture");
        e = cudaGraphInstantiate(&g.exec, g.graph, 0);
        if (e != cudaSuccess) {
            cudaGraphDestroy(g.graph);
            return cuda_error(e, "cudaGraphInstantiate");
        }
        s->graphs.push_back(g);
        ge = &s->graphs.back();
    }
    GS_CUDA(cudaGraphLaunch(ge->exec, st));
    return GS_OK;
}

void free_prim_box(gs_scene* s) {
    cudaFree(s->pbox_lo);
    cudaFree(s->pbox_hi);
    s->pbox_lo = s->pbox_hi = nullptr;
    s->nbox_words = 0;
}

gs_status load_prim_box(gs_scene* s, const void* lo, const void* hi, int src_on_device, int nbox_words) {
    const size_t bytes = (size_t)s->n * nbox_words * word_bytes(s->fmt);
    GS_TRY(dmalloc(&s->pbox_lo, (bytes + 15) & ~(size_t)15));
    GS_TRY(dmalloc(&s->pbox_hi, (bytes + 15) & ~(size_t)15));
    const cudaMemcpyKind kind = src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    GS_CUDA(cudaMemcpy(s->pbox_lo, lo, bytes, kind));
    GS_CUDA(cudaMemcpy(s->pbox_hi, hi, bytes, kind));
    s->nbox_words = nbox_words;
    return GS_OK;
}

}  // namespace

size_t scene_bytes(const gs_scene* s) {
    size_t b = (size_t)s->n * (s->nwords + (s->pbox_lo ? 2 * s->nbox_words : 0)) * word_bytes(s->fmt);
    for (const Buf& v : s->view_bufs) b += v.cap;
    b += s->list_tmp.cap + render_work_bytes(s->work) + batch_held(s).bytes();
    b += sizeof(gs_flip) * s->host_io_flips_cap + sizeof(gs_result) * s->host_io_out_cap;
    if (s->ssim.tile_map) {
        const SsimBufs& q = s->ssim;
        const size_t pairs = (size_t)std::min(s->cap_B, ssim_batch(std::max(s->K, 1))) * std::max(s->K, 1);
        b += (size_t)q.slot_cap * (sizeof(PlanItem) + 4 * (8 + 1 + 9)) + (size_t)q.delta_cap * 32 * sizeof(float4) +
             2 * sizeof(unsigned long long) * pairs * q.max_tiles;
    }
    return b;
}

size_t allow_batch_growth(gs_scene* s, int B, size_t room) {
    const BatchSize held = batch_held(s);
    s->batch_room = room > ~held.bytes() ? ~(size_t)0 : held.bytes() + room;
    if (s->K == 0 || B < 1) return 0;
    for (int chunk = campaign_batch(s);; chunk /= 2) {   // as size_batch will settle
        const int cap = batch_cap(B, chunk);
        const BatchSize need = batch_size(s, std::max(cap, s->cap_B), std::max(cap, s->cap_flips));
        if (batch_fits(need, held)) return 0;
        if (cap <= 64 || need.bytes() <= s->batch_room) return need.bytes() - std::min(need.bytes(), held.bytes());
        chunk = cap;
    }
}

void trim_batch_buffers(gs_scene* s) {
    destroy_graphs(s);
    free_ssim_buffers(s);
    free_batch_buffers(s);
    if (s->K > 0) ensure_batch_buffers(s, 64, 1);   // (out of memory: the next campaign tries again)
}

gs_status render_lists_sized_ext(gs_scene* s, RenderWork& w, const DevCamera& cam, uint32_t** ids, uint64_t* npairs,
                                 cudaStream_t st) {
    return render_lists_sized(s, w, cam, ids, npairs, st);
}

}  // namespace gs

using namespace gs;

extern "C" {

const char* gs_last_error(void) { return g_last_error.c_str(); }

const char* gs_version(void) { return "libgs 0.1 (sm_103a)"; }

gs_status gs_load_scene(const void* planes, int src_on_device, uint64_t n, int sh_degree, gs_format fmt,
                        gs_scene** out) {
    if (!out) return set_error(GS_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (sh_degree < 0 || sh_degree > 3) return set_error(GS_ERR_ARG, "sh_degree must be 0..3");
    if (fmt != GS_FP32 && fmt != GS_FP16 && fmt != GS_BF16) return set_error(GS_ERR_ARG, "unknown storage format");
    if (n > 0xffffffffull) return set_error(GS_ERR_ARG, "at most 2^32 - 1 primitives");
    if (n > 0 && !planes) return set_error(GS_ERR_ARG, "planes is NULL");
    gs_scene* s = new gs_scene();
    s->n = n;
    s->sh_degree = sh_degree;
    s->fmt = fmt;
    s->nwords = words_for_degree(sh_degree);
    size_t bytes = (size_t)n * s->nwords * word_bytes(fmt);
    // rounded up to 16 bytes: 16-bit words are flipped with 32-bit atomics on
    // the aligned word that contains them
    gs_status st = dmalloc(&s->planes, (bytes + 15) & ~(size_t)15);
    if (st == GS_OK) st = dmalloc((void**)&s->dev_box, sizeof(uint32_t) * 2 * kMaxWords);
    if (st == GS_OK) st = dmalloc((void**)&s->dev_err, sizeof(unsigned int) * 4);
    if (st == GS_OK) st = dmalloc((void**)&s->dev_clamps, sizeof(unsigned long long) * 2);
    if (st != GS_OK) {
        gs_free_scene(s);
        return st;
    }
    cudaError_t e = cudaMemcpy(s->planes, planes, bytes, src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(s->dev_err, 0, sizeof(unsigned int) * 4);
    if (e == cudaSuccess) e = cudaMemset(s->dev_clamps, 0, sizeof(unsigned long long) * 2);
    if (e != cudaSuccess) {
        gs_free_scene(s);
        return cuda_error(e, "gs_load_scene copy");
    }
    // Algorithm 1 precompute: per-word min/max box
    st = launch_field_box(s->planes, fmt, n, s->nwords, s->dev_box, 0);
    uint32_t keys[2 * kMaxWords];
    if (st == GS_OK) {
        e = cudaMemcpy(keys, s->dev_box, sizeof(keys), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) st = cuda_error(e, "field box readback");
    }
    if (st != GS_OK) {
        gs_free_scene(s);
        return st;
    }
    for (int w = 0; w < s->nwords; w++) {
        if (keys[w] == 0xffffffffu && keys[kMaxWords + w] == 0u) {   // no finite... no non-NaN value
            s->box_lo[w] = s->box_hi[w] = 0u;
        } else {
            s->box_lo[w] = key_to_bits(keys[w], fmt);
            s->box_hi[w] = key_to_bits(keys[kMaxWords + w], fmt);
        }
        keys[w] = s->box_lo[w];
        keys[kMaxWords + w] = s->box_hi[w];
    }
    e = cudaMemcpy(s->dev_box, keys, sizeof(keys), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        gs_free_scene(s);
        return cuda_error(e, "field box upload");
    }
    *out = s;
    return GS_OK;
}

gs_status gs_free_scene(gs_scene* s) {
    if (!s) return GS_OK;
    free_view_memory(s);
    free_render_work(s->work);
    cudaFree(s->planes);
    free_prim_box(s);
    cudaFree(s->dev_box);
    cudaFree(s->dev_err);
    cudaFree(s->dev_clamps);
    cudaFree(s->host_io_flips);
    cudaFree(s->host_io_out);
    free_batch_buffers(s);
    free_ssim_buffers(s);
    cudaFree(s->clean_nonfin);
    cudaFree(s->work_ctr);
    if (s->ev_k0) cudaEventDestroy(s->ev_k0);
    if (s->ev_kp) cudaEventDestroy(s->ev_kp);
    if (s->ev_k1) cudaEventDestroy(s->ev_k1);
    for (auto& e : s->ev_r)
        if (e) cudaEventDestroy(e);
    delete s;
    return GS_OK;
}

gs_status gs_scene_info(const gs_scene* s, uint64_t* n, int* sh_degree, int* fmt, int* nwords) {
    if (!s) return set_error(GS_ERR_ARG, "scene is NULL");
    if (n) *n = s->n;
    if (sh_degree) *sh_degree = s->sh_degree;
    if (fmt) *fmt = s->fmt;
    if (nwords) *nwords = s->nwords;
    return GS_OK;
}

gs_status gs_scene_planes(gs_scene* s, void** dev_planes) {
    if (!s || !dev_planes) return set_error(GS_ERR_ARG, "NULL argument");
    *dev_planes = s->planes;
    return GS_OK;
}

gs_status gs_read_planes(gs_scene* s, void* dst, int dst_on_device, void* stream) {
    if (!s || !dst) return set_error(GS_ERR_ARG, "NULL argument");
    size_t bytes = (size_t)s->n * s->nwords * word_bytes(s->fmt);
    GS_CUDA(cudaMemcpyAsync(dst, s->planes, bytes, dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                            (cudaStream_t)stream));
    if (!dst_on_device) GS_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    return GS_OK;
}

gs_status gs_write_planes(gs_scene* s, const void* src, int src_on_device, void* stream) {
    if (!s || !src) return set_error(GS_ERR_ARG, "NULL argument");
    size_t bytes = (size_t)s->n * s->nwords * word_bytes(s->fmt);
    GS_CUDA(cudaMemcpyAsync(s->planes, src, bytes, src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                            (cudaStream_t)stream));
    if (!src_on_device) GS_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    return GS_OK;
}

gs_status gs_scene_errors(gs_scene* s, uint32_t* host_flags) {
    if (!s || !host_flags) return set_error(GS_ERR_ARG, "NULL argument");
    GS_CUDA(cudaMemcpy(host_flags, s->dev_err, sizeof(uint32_t), cudaMemcpyDeviceToHost));
    GS_CUDA(cudaMemset(s->dev_err, 0, sizeof(uint32_t)));
    return GS_OK;
}

gs_status gs_apply_flips(gs_scene* s, const gs_flip* dev_flips, int64_t count, void* stream) {
    if (!s || (count > 0 && !dev_flips) || count < 0) return set_error(GS_ERR_ARG, "bad gs_apply_flips arguments");
    return launch_apply_flips(s->planes, s->fmt, s->n, s->nwords, dev_flips, count, s->dev_err, 0ull,
                              (cudaStream_t)stream);
}

gs_status gs_field_box(gs_scene* s, uint32_t* host_lo, uint32_t* host_hi) {
    if (!s || !host_lo || !host_hi) return set_error(GS_ERR_ARG, "NULL argument");
    memcpy(host_lo, s->box_lo, sizeof(uint32_t) * s->nwords);
    memcpy(host_hi, s->box_hi, sizeof(uint32_t) * s->nwords);
    return GS_OK;
}

gs_status gs_set_prim_box(gs_scene* s, const void* lo, const void* hi, int src_on_device, int nbox_words) {
    if (!s || !lo || !hi || nbox_words < 1 || nbox_words > s->nwords)
        return set_error(GS_ERR_ARG, "bad gs_set_prim_box arguments");
    destroy_graphs(s);
    free_prim_box(s);
    const gs_status rs = load_prim_box(s, lo, hi, src_on_device, nbox_words);
    if (rs != GS_OK) free_prim_box(s);   // both halves or none: half a box is no box
    return rs;
}

gs_status gs_guard(gs_scene* s, int mode, uint64_t word_mask, uint64_t* dev_clamps, void* stream) {
    if (!s) return set_error(GS_ERR_ARG, "scene is NULL");
    if (mode != GS_GUARD_FIELD && mode != GS_GUARD_PRIM) return set_error(GS_ERR_ARG, "mode must be FIELD or PRIM");
    return launch_guard(s, mode, word_mask, (unsigned long long*)dev_clamps, (cudaStream_t)stream);
}

gs_status gs_guard_bitmap(gs_scene* s, int mode, uint64_t word_mask, uint64_t* dev_clamps, uint32_t* dev_bitmap,
                          void* stream) {
    if (!s) return set_error(GS_ERR_ARG, "scene is NULL");
    if (mode != GS_GUARD_FIELD && mode != GS_GUARD_PRIM) return set_error(GS_ERR_ARG, "mode must be FIELD or PRIM");
    if (!dev_bitmap && s->n > 0) return set_error(GS_ERR_ARG, "dev_bitmap is NULL");
    const cudaStream_t st = (cudaStream_t)stream;
    GS_TRY(launch_guard_mark(s, mode, word_mask, dev_bitmap, st));   // the decisions, on the words before the clamp
    return launch_guard(s, mode, word_mask, (unsigned long long*)dev_clamps, st);
}

gs_status gs_render(gs_scene* s, const gs_camera* host_cams, int K, float* dev_rgb, void* stream) {
    if (!s || !host_cams || !dev_rgb || K < 1) return set_error(GS_ERR_ARG, "bad gs_render arguments");
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t* ev = s->ev_r[0] ? s->ev_r : nullptr;
    s->render_timed = false;
    size_t off = 0;
    for (int k = 0; k < K; k++) {
        if (!valid_camera(host_cams[k])) return set_error(GS_ERR_ARG, "invalid camera");
        DevCamera cam = make_dev_camera(host_cams[k], s->tile_w, s->tile_h);
        uint32_t* ids = nullptr;
        uint64_t np = 0;
        GS_TRY(render_lists_sized(s, s->work, cam, &ids, &np, st, ev));
        GS_TRY(launch_blend_image(s->work.recs, ids, s->work.ranges, cam, dev_rgb + off, st));
        if (ev) GS_CUDA(cudaEventRecord(ev[3], st));
        s->render_pairs = np;
        off += (size_t)cam.W * cam.H * 3;
    }
    s->render_timed = ev != nullptr;
    return GS_OK;
}

gs_status gs_compare(const float* dev_a, const float* dev_b, int H, int W, int K, gs_result* dev_out, void* stream) {
    if (!dev_a || !dev_b || !dev_out || H < 1 || W < 1 || K < 1) return set_error(GS_ERR_ARG, "bad gs_compare arguments");
    cudaStream_t st = (cudaStream_t)stream;
    CmpAcc* acc = nullptr;
    GS_CUDA(cudaMallocAsync((void**)&acc, sizeof(CmpAcc) * K, st));
    gs_status rs = launch_zero_acc(acc, K, st);
    if (rs == GS_OK) rs = launch_compare(dev_a, dev_b, H, W, K, acc, st);
    if (rs == GS_OK) rs = launch_finalize(acc, K, dev_out, st);
    cudaFreeAsync(acc, st);
    return rs;
}

// Several arrays in one device allocation, each on a 256-byte boundary.
struct Part {
    void** p;
    size_t bytes;
};
static gs_status place(Buf& buf, std::initializer_list<Part> parts) {
    size_t total = 0;
    for (const Part& q : parts) total += (q.bytes + 255) & ~(size_t)255;
    GS_TRY(reserve(buf, total));
    char* at = (char*)buf.p;
    for (const Part& q : parts) {
        *q.p = at;
        at += (q.bytes + 255) & ~(size_t)255;
    }
    return GS_OK;
}

// Is a view with E blend-list entries, whose 8x8 blocks keep S entries for 64 pixels
// each, dense: better re-blended from its block lists?  The walk of a pixel's
// own list costs 20 B an entry, an evaluation of a block's entry serves 64 pixels.  Lists
// win where a pixel takes few of its block's entries or has few to walk.  Campaigns of
// 4,000 upsets at 1600x1040, lists against blocks: 0.88 of the entries taken, 89 a pixel:
// 1.85 and 1.28 ms; 0.78, 58: 0.79 and 0.68; 0.66, 55: 0.48 and 0.43; 0.62, 60: 0.82 and
// 0.90; 0.45, 50: 0.42 and 0.60; 1.0, 32 a pixel: 356 and 911.
constexpr uint64_t kDenseLength = 48;   // entries of a pixel's list (on average) from which a view may be dense
static bool dense_view(uint64_t E, uint64_t S) { return (double)E >= 0.65 * 64.0 * (double)S; }

// The lists of view v (its first pass is done): sizes on the device, a read-back of the
// totals, then the second pass.  Blend lists (24 B an entry) take at most this view's
// share of the memory that is free -- one for each view still to come, one for what
// comes behind them -- else, as in a dense view, the block lists take their place.
static gs_status build_lists(gs_scene* s, ViewState& v, Buf& buf, uint32_t* counts, int views_left, cudaStream_t st) {
    const uint64_t ntiles = (uint64_t)v.cam.tiles_x * v.cam.tiles_y;
    const uint64_t P = (uint64_t)v.cam.tile_w * v.cam.tile_h, npix = ntiles * P, nblk = npix / 64;
    uint32_t *rows = nullptr, *lens = nullptr, *off = nullptr, *boff = nullptr;
    unsigned long long *scratch = nullptr, *total = nullptr;
    GS_TRY(place(s->list_tmp, {{(void**)&rows, 4 * ntiles},
                               {(void**)&lens, 4 * npix},
                               {(void**)&off, 4 * npix},
                               {(void**)&boff, 4 * nblk},
                               {(void**)&scratch, 8 * scan_scratch_len(npix)},
                               {(void**)&total, 8 * 6}}));
    unsigned long long tot[6];
    auto read_totals = [&]() -> gs_status {
        GS_CUDA(cudaMemcpyAsync(tot, total, sizeof(tot), cudaMemcpyDeviceToHost, st));
        GS_CUDA(cudaStreamSynchronize(st));
        return GS_OK;
    };
    GS_TRY(launch_row_counts(v, rows, st));
    GS_TRY(launch_exclusive_scan(rows, ntiles, v.row_off, scratch, total, st));
    GS_TRY(launch_list_lens(counts, npix, lens, st));
    GS_TRY(launch_exclusive_scan(lens, npix, off, scratch, total + 3, st));
    GS_TRY(read_totals());
    const uint64_t nrows = tot[2], E = tot[5];
    const uint64_t bytes = 4 * P * nrows + (16 + 4) * E + 16 * (E / kWalk);   // and at most 1 KB to align the parts
    bool lists = nrows < 0xffffffffull && E < 0xffffffffull;
    if (lists && bytes >= kLookBytes && (!buf.p || bytes > buf.cap)) {
        size_t avail = 0, all = 0;
        GS_CUDA(cudaMemGetInfo(&avail, &all));
        lists = bytes <= (avail + buf.cap) / (uint64_t)(views_left + 1);
    }
    bool counted = false;   // tot[2]: entries of the block lists
    auto count_blocks = [&]() -> gs_status {
        if (counted) return GS_OK;
        counted = true;
        GS_TRY(launch_exclusive_scan(v.sub_cnt, nblk, boff, scratch, total, st));
        return read_totals();
    };
    if (lists && E >= kDenseLength * npix) {
        GS_TRY(count_blocks());
        lists = !dense_view(E, tot[2]);
    }
    if (lists) {
        const gs_status rs = place(buf, {{(void**)&v.row_idx, 4 * P * nrows},
                                         {(void**)&v.ent, sizeof(float4) * E},
                                         {(void**)&v.rk, 4 * E},
                                         {(void**)&v.state, sizeof(float4) * (E / kWalk)}});
        if (rs != GS_OK && rs != GS_ERR_OOM) return rs;
        lists = rs == GS_OK;
    }
    if (!lists) {
        v.row_idx = v.rk = nullptr;
        v.ent = v.state = nullptr;
        GS_TRY(count_blocks());
        if (tot[2] >= 0xffffffffull) return set_error(GS_ERR_CAPACITY, "too many block-list entries");
        GS_TRY(place(buf, {{(void**)&v.sub, sizeof(uint2) * tot[2]},
                           {(void**)&v.sub_off, 4 * nblk},
                           {(void**)&v.row_state, sizeof(float4) * 64 * (tot[2] / kRowStride + nblk)}}));
        GS_CUDA(cudaMemcpyAsync(v.sub_off, boff, 4 * nblk, cudaMemcpyDeviceToDevice, st));
    }
    return launch_fill_lists(v, off, st);
}

// The clean per-view state of gs_set_views, for validated arguments.
static gs_status build_views(gs_scene* s, const gs_camera* host_cams, int K, cudaStream_t st) {
    free_views(s);
    for (size_t i = 2 * (size_t)K; i < s->view_bufs.size(); i++) release(s->view_bufs[i]);
    s->view_bufs.resize(2 * (size_t)K);
    s->views.resize(K);
    s->K = K;
    std::vector<DevCamera> dcams(K);
    std::vector<char> vptrs(view_ptrs_size() * K);
    GS_TRY(dmalloc((void**)&s->clean_nonfin, sizeof(unsigned int) * K));
    GS_CUDA(cudaMemsetAsync(s->clean_nonfin, 0, sizeof(unsigned int) * K, st));
    uint64_t max_pairs = 0;
    int max_tiles = 0, max_tiles_y = 0;
    uint32_t all_tiles = 0;
    for (int k = 0; k < K; k++) {
        ViewState& v = s->views[k];
        v.cam = make_dev_camera(host_cams[k], s->tile_w, s->tile_h);
        dcams[k] = v.cam;
        int ntiles = v.cam.tiles_x * v.cam.tiles_y;
        const size_t pix = (size_t)v.cam.W * v.cam.H, tpix = (size_t)ntiles * v.cam.tile_w * v.cam.tile_h;
        uint32_t* ids = nullptr;
        uint64_t np = 0;
        GS_TRY(render_lists_sized(s, s->work, v.cam, &ids, &np, st));
        uint32_t* counts = nullptr;   // scratch of this build
        GS_TRY(place(s->view_bufs[2 * k], {{(void**)&v.recs, sizeof(BlendRec) * s->n},
                                           {(void**)&v.rects, sizeof(uint2) * s->n},
                                           {(void**)&v.rank, 4 * s->n},
                                           {(void**)&v.sdk, 4 * s->n},
                                           {(void**)&v.sid, 4 * s->n},
                                           {(void**)&v.ids, 4 * np},
                                           {(void**)&v.ranges, sizeof(uint2) * ntiles},
                                           {(void**)&v.clean, 12 * pix},
                                           {(void**)&v.stop, 4 * tpix},
                                           {(void**)&v.tile_stop, (size_t)4 * ntiles},
                                           {(void**)&v.tile_last, (size_t)4 * ntiles},
                                           {(void**)&v.row_key, (size_t)4 * ntiles * kRowsPerTile},
                                           {(void**)&v.row_off, (size_t)4 * ntiles},
                                           {(void**)&v.row_cnt, (size_t)4 * ntiles},
                                           {(void**)&v.sub_cnt, 4 * tpix / 64},
                                           {(void**)&counts, 4 * tpix}}));
        GS_CUDA(cudaMemcpyAsync(v.recs, s->work.recs, sizeof(BlendRec) * s->n, cudaMemcpyDeviceToDevice, st));
        GS_CUDA(cudaMemcpyAsync(v.rects, s->work.rects, sizeof(uint2) * s->n, cudaMemcpyDeviceToDevice, st));
        GS_CUDA(cudaMemcpyAsync(v.ids, ids, sizeof(uint32_t) * np, cudaMemcpyDeviceToDevice, st));
        GS_CUDA(cudaMemcpyAsync(v.ranges, s->work.ranges, sizeof(uint2) * ntiles, cudaMemcpyDeviceToDevice, st));
        GS_TRY(launch_ranks(s->work.dkey[s->work.cur], s->work.dval[s->work.cur], s->n, v, st));
        GS_TRY(launch_blend_clean(v, counts, v.sub_cnt, s->clean_nonfin + k, st));
        v.npairs = np;
        GS_TRY(build_lists(s, v, s->view_bufs[2 * k + 1], counts, K - k, st));
        fill_view_ptrs(vptrs.data() + view_ptrs_size() * k, v, all_tiles);
        all_tiles += (uint32_t)ntiles;
        max_pairs = std::max(max_pairs, np);
        max_tiles = std::max(max_tiles, ntiles);
        max_tiles_y = std::max(max_tiles_y, v.cam.tiles_y);
    }
    GS_TRY(dmalloc((void**)&s->dev_cams, sizeof(DevCamera) * K));
    GS_TRY(dmalloc(&s->dev_views, vptrs.size()));
    GS_CUDA(cudaMemcpyAsync(s->dev_cams, dcams.data(), sizeof(DevCamera) * K, cudaMemcpyHostToDevice, st));
    GS_CUDA(cudaMemcpyAsync(s->dev_views, vptrs.data(), vptrs.size(), cudaMemcpyHostToDevice, st));
    // the plain loop re-renders a single-flip variant: at most one primitive
    // changes, adding at most one grid's worth of pairs
    s->full_cap_pairs = max_pairs + (uint64_t)max_tiles + 1024;
    s->max_tiles = max_tiles;
    s->max_tiles_y = max_tiles_y;
    s->all_tiles = all_tiles;
    // buffers for the dirty engine
    s->cap_B = 0;
    s->cap_flips = 0;
    GS_TRY(ensure_batch_buffers(s, 64, 1));
    GS_CUDA(cudaStreamSynchronize(st));
    return GS_OK;
}

gs_status gs_set_views(gs_scene* s, const gs_camera* host_cams, int K, void* stream) {
    if (!s || !host_cams || K < 1 || K > 16) return set_error(GS_ERR_ARG, "bad gs_set_views arguments (1 <= K <= 16)");
    for (int k = 0; k < K; k++)
        if (!valid_camera(host_cams[k])) return set_error(GS_ERR_ARG, "invalid camera");
    const gs_status rs = build_views(s, host_cams, K, (cudaStream_t)stream);
    // a failure part way (out of memory, a capacity limit) leaves no half-built
    // views behind: campaign calls then report GS_ERR_STATE instead of reading them
    if (rs != GS_OK) {
        free_view_memory(s);
        s->host_cams.clear();
        return rs;
    }
    s->host_cams.assign(host_cams, host_cams + K);
    return GS_OK;
}

gs_status gs_set_tile(gs_scene* s, int tile_w, int tile_h, void* stream) {
    if (!s || !tile_shape_ok(tile_w, tile_h))
        return set_error(GS_ERR_ARG, "tile shape must be tw x th with tw, th in {8, 16, 32} and 64 <= tw * th <= 256");
    if (tile_w == s->tile_w && tile_h == s->tile_h) return GS_OK;
    s->tile_w = tile_w;
    s->tile_h = tile_h;
    if (s->host_cams.empty()) return GS_OK;
    // rebuild the clean per-view state for the new tiles
    const std::vector<gs_camera> cams = s->host_cams;
    return gs_set_views(s, cams.data(), (int)cams.size(), stream);
}

gs_status gs_get_tile(gs_scene* s, int* tile_w, int* tile_h) {
    if (!s || !tile_w || !tile_h) return set_error(GS_ERR_ARG, "bad gs_get_tile arguments");
    *tile_w = s->tile_w;
    *tile_h = s->tile_h;
    return GS_OK;
}

gs_status gs_clean_image(gs_scene* s, int k, float* dev_rgb, void* stream) {
    if (!s || !dev_rgb || k < 0 || k >= s->K) return set_error(GS_ERR_ARG, "bad gs_clean_image arguments");
    const ViewState& v = s->views[k];
    GS_CUDA(cudaMemcpyAsync(dev_rgb, v.clean, sizeof(float) * (size_t)v.cam.W * v.cam.H * 3, cudaMemcpyDeviceToDevice,
                            (cudaStream_t)stream));
    return GS_OK;
}

namespace {
gs_status inject_and_render(gs_scene* s, const gs_flip* dev_flips, int B, int guard_mode, uint64_t word_mask,
                            gs_result* dev_out, uint64_t* dev_regions, double* dev_ssim, void* stream);
}

gs_status gs_inject_and_render(gs_scene* s, const gs_flip* dev_flips, int B, int flips_per_variant, int guard_mode,
                               uint64_t word_mask, gs_result* dev_out, void* stream) {
    GS_TRY(check_flip_args(s, dev_flips, B, flips_per_variant, guard_mode, word_mask));
    if (!dev_out && B > 0) return set_error(GS_ERR_ARG, "dev_out is NULL");
    if (flips_per_variant != 1)
        return gs_inject_and_render_full(s, dev_flips, B, flips_per_variant, guard_mode, word_mask, dev_out, stream);
    return inject_and_render(s, dev_flips, B, guard_mode, word_mask, dev_out, nullptr, nullptr, stream);
}

gs_status gs_inject_and_render_regions(gs_scene* s, const gs_flip* dev_flips, int B, int guard_mode,
                                       uint64_t word_mask, gs_result* dev_out, uint64_t* dev_regions, void* stream) {
    GS_TRY(check_flip_args(s, dev_flips, B, 1, guard_mode, word_mask));
    if ((!dev_out || !dev_regions) && B > 0) return set_error(GS_ERR_ARG, "dev_out or dev_regions is NULL");
    return inject_and_render(s, dev_flips, B, guard_mode, word_mask, dev_out, dev_regions, nullptr, stream);
}

gs_status gs_inject_and_render_ex(gs_scene* s, const gs_flip* dev_flips, int B, int guard_mode, uint64_t word_mask,
                                  gs_result* dev_out, uint64_t* dev_regions, double* dev_ssim, void* stream) {
    GS_TRY(check_flip_args(s, dev_flips, B, 1, guard_mode, word_mask));
    if (!dev_out && B > 0) return set_error(GS_ERR_ARG, "dev_out is NULL");
    return inject_and_render(s, dev_flips, B, guard_mode, word_mask, dev_out, dev_regions, dev_ssim, stream);
}

namespace {
gs_status inject_and_render(gs_scene* s, const gs_flip* dev_flips, int B, int guard_mode, uint64_t word_mask,
                            gs_result* dev_out, uint64_t* dev_regions, double* dev_ssim, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int K = s->K;
    int chunk = campaign_batch(s);
    const bool ssim = dev_ssim != nullptr;
    if (ssim) chunk = std::min(chunk, ssim_batch(K));
    if (ssim && (s->tile_w != kTile || s->tile_h != kTile))
        return set_error(GS_ERR_STATE, "the dirty-tile SSIM needs 16 x 16 render tiles (gs_set_tile)");
    GS_TRY(size_batch(s, B, &chunk));
    if (ssim) GS_TRY(ensure_ssim_buffers(s));
    for (int b0 = 0; b0 < B; b0 += chunk) {
        int nb = std::min(chunk, B - b0);
        GS_CUDA(cudaMemcpyAsync(s->flip_stage, dev_flips + b0, sizeof(gs_flip) * nb, cudaMemcpyDeviceToDevice, st));
        GS_TRY(run_dirty_batch(s, nb, guard_mode, word_mask, ssim, dev_regions != nullptr, st));
        GS_CUDA(cudaMemcpyAsync(dev_out + (size_t)b0 * K, s->res_stage, sizeof(gs_result) * nb * K,
                                cudaMemcpyDeviceToDevice, st));
        if (dev_regions)
            GS_TRY(launch_regions_out(s->acc, nb * K, (unsigned long long*)dev_regions + (size_t)2 * b0 * K, st));
        if (ssim) GS_TRY(launch_ssim_out(s->acc, nb * K, s->dev_views, K, dev_ssim + (size_t)b0 * K, st));
    }
    if (ssim) {   // a capacity overflow leaves some SSIM values incomplete: report it
        unsigned int over = 0;
        GS_CUDA(cudaMemcpyAsync(&over, s->ssim.overflow, sizeof(over), cudaMemcpyDeviceToHost, st));
        GS_CUDA(cudaStreamSynchronize(st));
        if (over) {
            GS_CUDA(cudaMemset(s->ssim.overflow, 0, sizeof(unsigned int)));
            return set_error(GS_ERR_CAPACITY, "SSIM buffers too small for this batch: use a smaller batch");
        }
    }
    return GS_OK;
}
}  // namespace

gs_status gs_inject_and_render_host(gs_scene* s, const gs_flip* host_flips, int B, int flips_per_variant,
                                    int guard_mode, uint64_t word_mask, gs_result* host_out, void* stream) {
    GS_TRY(check_flip_args(s, host_flips, B, flips_per_variant, guard_mode, word_mask));
    if (!host_out && B > 0) return set_error(GS_ERR_ARG, "host_out is NULL");
    if (B == 0) return GS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nf = (size_t)B * flips_per_variant, nr = (size_t)B * s->K;
    if (nf > s->host_io_flips_cap) {
        cudaFree(s->host_io_flips);
        s->host_io_flips = nullptr;
        s->host_io_flips_cap = 0;
        GS_TRY(dmalloc((void**)&s->host_io_flips, sizeof(gs_flip) * nf));
        s->host_io_flips_cap = nf;
    }
    if (nr > s->host_io_out_cap) {
        cudaFree(s->host_io_out);
        s->host_io_out = nullptr;
        s->host_io_out_cap = 0;
        GS_TRY(dmalloc((void**)&s->host_io_out, sizeof(gs_result) * nr));
        s->host_io_out_cap = nr;
    }
    GS_CUDA(cudaMemcpyAsync(s->host_io_flips, host_flips, sizeof(gs_flip) * nf, cudaMemcpyHostToDevice, st));
    GS_TRY(gs_inject_and_render(s, s->host_io_flips, B, flips_per_variant, guard_mode, word_mask, s->host_io_out,
                                stream));
    GS_CUDA(cudaMemcpyAsync(host_out, s->host_io_out, sizeof(gs_result) * nr, cudaMemcpyDeviceToHost, st));
    GS_CUDA(cudaStreamSynchronize(st));
    return GS_OK;
}

gs_status gs_inject_and_render_full(gs_scene* s, const gs_flip* dev_flips, int B, int flips_per_variant,
                                    int guard_mode, uint64_t word_mask, gs_result* dev_out, void* stream) {
    GS_TRY(check_flip_args(s, dev_flips, B, flips_per_variant, guard_mode, word_mask));
    if (!dev_out && B > 0) return set_error(GS_ERR_ARG, "dev_out is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    const int K = s->K;
    const int fpv = flips_per_variant;
    GS_TRY(ensure_batch_buffers(s, 1, fpv));
    uint64_t cap = s->full_cap_pairs + (uint64_t)(fpv - 1) * s->max_tiles;
    // for every view's own grid: a smaller one may be listed by counting where the largest is not
    for (const ViewState& v : s->views) GS_TRY(alloc_render_work(s->work, s->n, cap, v.cam.tiles_x * v.cam.tiles_y));
    for (int b = 0; b < B; b++) {
        const gs_flip* f = dev_flips + (size_t)b * fpv;
        GS_TRY(launch_zero_acc(s->acc, K, st));
        GS_TRY(launch_save_sites(s->planes, s->fmt, s->n, s->nwords, f, fpv, s->saved, st));
        GS_TRY(launch_apply_flips(s->planes, s->fmt, s->n, s->nwords, f, fpv, s->dev_err,
                                  guard_mode == GS_GUARD_ECC ? word_mask : 0ull, st));
        if (guard_mode == GS_GUARD_FIELD || guard_mode == GS_GUARD_PRIM) {
            GS_TRY(launch_guard(s, guard_mode, word_mask, s->dev_clamps, st));
            k_move_clamps<<<1, 32, 0, st>>>(s->dev_clamps, s->acc);
            GS_CUDA(cudaGetLastError());
        }
        for (int k = 0; k < K; k++) {
            const ViewState& v = s->views[k];
            uint32_t* ids = nullptr;
            GS_TRY(render_lists(s, s->work, v.cam, &ids, st));
            GS_TRY(launch_blend_compare(s->work.recs, ids, s->work.ranges, v.cam, v.clean, s->acc + k,
                                        s->work_ctr, st));
        }
        GS_TRY(launch_restore_sites(s->planes, s->fmt, s->n, s->nwords, f, fpv, s->saved, st));
        GS_TRY(launch_finalize(s->acc, K, dev_out + (size_t)b * K, st));
    }
    return GS_OK;
}

gs_status gs_preprocess(gs_scene* s, const gs_camera* host_cam, gs_record* dev_out, void* stream) {
    if (!s || !host_cam || !dev_out) return set_error(GS_ERR_ARG, "bad gs_preprocess arguments");
    if (!valid_camera(*host_cam)) return set_error(GS_ERR_ARG, "invalid camera");
    DevCamera cam = make_dev_camera(*host_cam, s->tile_w, s->tile_h);
    return launch_preprocess(s, cam, nullptr, nullptr, nullptr, nullptr, dev_out, (cudaStream_t)stream);
}

gs_status gs_bin_tiles(const float* dev_depth, const int32_t* dev_rects, uint64_t n, int tiles_x, int tiles_y,
                       uint32_t* dev_offsets, uint32_t* dev_ids, uint64_t ids_cap, uint64_t* host_total,
                       void* stream) {
    if ((!dev_depth || !dev_rects) && n > 0) return set_error(GS_ERR_ARG, "NULL input");
    if (!dev_offsets || !host_total || tiles_x < 1 || tiles_y < 1 || tiles_x > 65535 || tiles_y > 65535)
        return set_error(GS_ERR_ARG, "bad gs_bin_tiles arguments");
    cudaStream_t st = (cudaStream_t)stream;
    int ntiles = tiles_x * tiles_y;
    RenderWork w;
    gs_status rs = alloc_render_work(w, n, std::max<uint64_t>(ids_cap, 1), ntiles);
    if (rs == GS_OK) rs = launch_rects_to_keys(dev_depth, dev_rects, n, tiles_x, tiles_y, w.dkey[0], w.dval[0], w.rects, st);
    uint32_t* ids = nullptr;
    if (rs == GS_OK) rs = build_tile_lists(w, n, tiles_x, tiles_y, &ids, st);
    if (rs == GS_OK) rs = launch_ranges_to_offsets(w.ranges, ntiles, dev_offsets, w.total, st);
    if (rs == GS_OK) {
        cudaError_t e = cudaMemcpyAsync(w.host_total, w.total, 3 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rs = cuda_error(e, "gs_bin_tiles readback");
    }
    if (rs == GS_OK) {
        *host_total = w.host_total[2];
        if (w.host_total[1]) {
            rs = set_error(GS_ERR_CAPACITY, "ids_cap too small");
        } else if (*host_total > 0) {
            if (!dev_ids) {
                rs = set_error(GS_ERR_ARG, "dev_ids is NULL");
            } else {
                cudaError_t e = cudaMemcpyAsync(dev_ids, ids, sizeof(uint32_t) * (*host_total), cudaMemcpyDeviceToDevice, st);
                if (e == cudaSuccess) e = cudaStreamSynchronize(st);
                if (e != cudaSuccess) rs = cuda_error(e, "gs_bin_tiles copy");
            }
        }
    }
    cudaStreamSynchronize(st);
    free_render_work(w);
    return rs;
}

gs_status gs_blend_lists(const gs_record* dev_recs, uint64_t n, const uint32_t* dev_offsets, const uint32_t* dev_ids,
                         int W, int H, float* dev_rgb, void* stream) {
    if (!dev_offsets || !dev_rgb || W < 1 || H < 1 || (n > 0 && !dev_recs)) return set_error(GS_ERR_ARG, "bad gs_blend_lists arguments");
    cudaStream_t st = (cudaStream_t)stream;
    gs_camera hc{};   // lists of 16 x 16 tiles
    hc.width = W;
    hc.height = H;
    const DevCamera cam = make_dev_camera(hc, kTile, kTile);
    const int ntiles = cam.tiles_x * cam.tiles_y;
    BlendRec* recs = nullptr;
    uint2* ranges = nullptr;
    GS_CUDA(cudaMallocAsync((void**)&recs, sizeof(BlendRec) * std::max<uint64_t>(n, 1), st));
    GS_CUDA(cudaMallocAsync((void**)&ranges, sizeof(uint2) * ntiles, st));
    gs_status rs = launch_records_to_blend(dev_recs, n, recs, st);
    if (rs == GS_OK) rs = launch_offsets_to_ranges(dev_offsets, ntiles, ranges, st);
    if (rs == GS_OK) rs = launch_blend_image(recs, dev_ids, ranges, cam, dev_rgb, st);
    cudaFreeAsync(recs, st);
    cudaFreeAsync(ranges, st);
    return rs;
}

gs_status gs_set_batch(gs_scene* s, int batch) {
    if (!s || batch < 0) return set_error(GS_ERR_ARG, "bad gs_set_batch arguments");
    s->batch = batch;
    return GS_OK;
}

gs_status gs_autotune(gs_scene* s, const gs_flip* dev_flips, int count, int guard_mode, uint64_t word_mask,
                      int* best_batch, float* best_us_per_variant, void* stream) {
    GS_TRY(check_flip_args(s, dev_flips, count, 1, guard_mode, word_mask));
    if (count < 1 || !best_batch) return set_error(GS_ERR_ARG, "bad gs_autotune arguments");
    cudaStream_t st = (cudaStream_t)stream;
    const int K = s->K;
    const int max_chunk = max_batch(s);
    gs_result* out = nullptr;
    GS_CUDA(cudaMallocAsync((void**)&out, sizeof(gs_result) * (size_t)count * K, st));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        cudaGetLastError();
        if (e0) cudaEventDestroy(e0);
        cudaFreeAsync(out, st);
        return set_error(GS_ERR_CUDA, "gs_autotune: event creation failed");
    }
    const int prev_batch = s->batch;
    int best = std::min(8, max_chunk);
    float best_t = 1e30f;
    gs_status rs = GS_OK;
    // powers of two up to the largest allowed, and up to the first that takes the list whole
    for (int c = 8; c <= max_chunk && (c == 8 || c / 2 < count); c *= 2) {
        s->batch = c;
        // warm (graph capture), then time the whole list at this batch size
        int warm = std::min(count, c);
        rs = gs_inject_and_render(s, dev_flips, warm, 1, guard_mode, word_mask, out, stream);
        if (rs != GS_OK) break;
        cudaEventRecord(e0, st);
        rs = gs_inject_and_render(s, dev_flips, count, 1, guard_mode, word_mask, out, stream);
        cudaEventRecord(e1, st);
        if (rs != GS_OK) break;
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        float per = ms * 1000.0f / count;
        if (per < best_t) {
            best_t = per;
            best = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFreeAsync(out, st);
    if (rs != GS_OK) {
        s->batch = prev_batch;   // a failed tuning run leaves the setting as it was
        return rs;
    }
    s->batch = best;
    *best_batch = best;
    if (best_us_per_variant) *best_us_per_variant = best_t;
    return GS_OK;
}

gs_status gs_autotune_tile(gs_scene* s, const gs_flip* dev_flips, int count, int guard_mode, uint64_t word_mask,
                           int* best_tile_w, int* best_tile_h, int* best_batch, float* best_us_per_variant,
                           void* stream) {
    GS_TRY(check_flip_args(s, dev_flips, count, 1, guard_mode, word_mask));
    if (count < 1 || !best_tile_w || !best_tile_h || !best_batch)
        return set_error(GS_ERR_ARG, "bad gs_autotune_tile arguments");
    const int shapes[3][2] = {{16, 16}, {8, 8}, {32, 8}};
    const int prev_w = s->tile_w, prev_h = s->tile_h, prev_batch = s->batch;
    int bw = prev_w, bh = prev_h, bb = 0;
    float bt = 1e30f;
    gs_status rs = GS_OK;
    for (const auto& sh : shapes) {
        rs = gs_set_tile(s, sh[0], sh[1], stream);
        if (rs != GS_OK) break;
        int b = 0;
        float us = 0.0f;
        rs = gs_autotune(s, dev_flips, count, guard_mode, word_mask, &b, &us, stream);
        if (rs != GS_OK) break;
        if (us < bt) {
            bt = us;
            bw = sh[0];
            bh = sh[1];
            bb = b;
        }
    }
    if (rs != GS_OK) {   // leave the scene as it was (views rebuilt for the previous tiles)
        const std::string msg = gs_last_error();
        gs_set_tile(s, prev_w, prev_h, stream);
        s->batch = prev_batch;
        return set_error(rs, msg);
    }
    GS_TRY(gs_set_tile(s, bw, bh, stream));
    s->batch = bb;
    *best_tile_w = bw;
    *best_tile_h = bh;
    *best_batch = bb;
    if (best_us_per_variant) *best_us_per_variant = bt;
    return GS_OK;
}

gs_status gs_count_work(gs_scene* s, int enable) {
    if (!s) return set_error(GS_ERR_ARG, "scene is NULL");
    if (enable && !s->work_ctr) {
        GS_TRY(dmalloc((void**)&s->work_ctr, sizeof(unsigned long long) * 16));
        GS_CUDA(cudaMemset(s->work_ctr, 0, sizeof(unsigned long long) * 16));
    }
    if (!enable && s->work_ctr) {
        cudaFree(s->work_ctr);
        s->work_ctr = nullptr;
    }
    return GS_OK;
}

gs_status gs_read_work(gs_scene* s, uint64_t* host_counts) {
    if (!s || !host_counts) return set_error(GS_ERR_ARG, "NULL argument");
    if (!s->work_ctr) return set_error(GS_ERR_STATE, "work counting is off");
    GS_CUDA(cudaMemcpy(host_counts, s->work_ctr, sizeof(unsigned long long) * 16, cudaMemcpyDeviceToHost));
    GS_CUDA(cudaMemset(s->work_ctr, 0, sizeof(unsigned long long) * 16));
    return GS_OK;
}

gs_status gs_time_kernels(gs_scene* s, int enable) {
    if (!s) return set_error(GS_ERR_ARG, "scene is NULL");
    destroy_graphs(s);   // the event records are part of the captured graph
    if (enable && !s->ev_k0) {
        GS_CUDA(cudaEventCreate(&s->ev_k0));
        GS_CUDA(cudaEventCreate(&s->ev_kp));
        GS_CUDA(cudaEventCreate(&s->ev_k1));
        for (auto& e : s->ev_r) GS_CUDA(cudaEventCreate(&e));
    }
    if (!enable && s->ev_k0) {
        cudaEventDestroy(s->ev_k0);
        cudaEventDestroy(s->ev_kp);
        cudaEventDestroy(s->ev_k1);
        s->ev_k0 = s->ev_kp = s->ev_k1 = nullptr;
        for (auto& e : s->ev_r) {
            cudaEventDestroy(e);
            e = nullptr;
        }
    }
    s->render_timed = false;
    return GS_OK;
}

gs_status gs_read_kernel_ms(gs_scene* s, float* ms) {
    if (!s || !ms) return set_error(GS_ERR_ARG, "NULL argument");
    if (!s->ev_k0) return set_error(GS_ERR_STATE, "kernel timing is off");
    GS_CUDA(cudaEventSynchronize(s->ev_k1));
    GS_CUDA(cudaEventElapsedTime(&ms[0], s->ev_k0, s->ev_kp));
    GS_CUDA(cudaEventElapsedTime(&ms[1], s->ev_kp, s->ev_k1));
    return GS_OK;
}

gs_status gs_read_render_ms(gs_scene* s, float* ms, uint64_t* counts) {
    if (!s || !ms || !counts) return set_error(GS_ERR_ARG, "NULL argument");
    if (!s->ev_r[0]) return set_error(GS_ERR_STATE, "kernel timing is off");
    if (!s->render_timed) return set_error(GS_ERR_STATE, "no gs_render since kernel timing was switched on");
    GS_CUDA(cudaEventSynchronize(s->ev_r[3]));
    for (int i = 0; i < 3; i++) GS_CUDA(cudaEventElapsedTime(&ms[i], s->ev_r[i], s->ev_r[i + 1]));
    counts[0] = s->n;
    counts[1] = s->render_pairs;
    counts[2] = (uint64_t)s->work.passes[0];
    counts[3] = (uint64_t)s->work.passes[1];
    return GS_OK;
}

gs_status gs_set_graphs(gs_scene* s, int enable) {
    if (!s) return set_error(GS_ERR_ARG, "scene is NULL");
    s->use_graphs = enable != 0;
    if (!enable) destroy_graphs(s);
    return GS_OK;
}

}  // extern "C"
