// SSIM of a corrupted frame against the clean one (Sec. 3 "Metrics and
// severity", Wang et al. 2004): per channel, Gaussian-weighted local means,
// variances and covariance over an 11x11 window (sigma 1.5, weights normalised
// to sum 1), SSIM = (2 mx my + C1)(2 sxy + C2) / ((mx^2 + my^2 + C1)(sx^2 + sy^2
// + C2)), C1 = 0.01^2, C2 = 0.03^2, on [0,1]-clamped values; the frame's SSIM is
// the mean over the windows inside the frame (pixels at least 5 from every
// edge) and over the channels.
//
// One 16x16 tile per block: the tile and a 5-pixel halo (26x26) of both images
// are staged in shared memory, a horizontal pass of the 11-tap filter, then a
// vertical one.  Every operation is explicitly rounded, so the full-frame and
// the dirty-tile kernels compute the same bits per pixel.  The sum of
// (1 - SSIM) over the pixels is accumulated in fixed point (2^-32), so totals do
// not depend on the order tiles finish.  Where both images agree on a whole
// window the numerator and denominator are computed identically and SSIM is
// exactly 1 (a zero term), so the dirty-tile engine only visits tiles within
// one tile of a re-blended tile.
//
// Both passes are bound by the FP32 pipe and shared memory (about 111,000 fused
// multiply-adds a tile).  Each thread computes a run of outputs and takes every
// staged value once into all the sums that use it -- 8 columns of one row
// horizontally (18 values of each image instead of 88), 4 rows of one column
// vertically (14 values of each sum instead of 44) -- with each sum's taps in the
// same order as one output at a time.  One output per thread and tap read took
// 86 us for a 1600x1040 pair, this form 49 us (0.37 of the FP32 pipe).
#include "gs_internal.h"

namespace gs {
namespace {

constexpr int kSR = 5;               // window radius
constexpr int kSS = kTile + 2 * kSR; // staged edge (26)
constexpr float kSsimFx = 4294967296.0f;   // 2^32

struct SsimW {
    float w[2 * kSR + 1];
};

// The two images' values, and their means and squares, lie in pairs: the sums of a
// pair share their weights, so one packed fp32x2 multiply-add takes both (each
// component rounded like the scalar operation).  Row pitches: 27 pairs keep the
// staged rows of neighbouring threads in different banks, 18 pairs and 20 floats do
// so for 16-byte stores of neighbouring rows.
constexpr int kPitchIn = 27, kPitchH2 = 18, kPitchH = 20;
constexpr int kSsimThreads = 192;   // the vertical pass has 192 runs, the horizontal one 156
struct __align__(16) SsimStage {
    float2 m[3][kSS][kPitchH2];   // horizontal sums of x, y
    float2 q[3][kSS][kPitchH2];   // of xx, yy
    float p[3][kSS][kPitchH];     // of xy
    float2 in[3][kSS][kPitchIn];  // image under test (corrupted), clean image; clamped
};

__device__ __forceinline__ float clamp01(float v) { return v > 0.0f ? (v < 1.0f ? v : 1.0f) : 0.0f; }

// Horizontal then vertical filtering of the staged tile, then the SSIM of
// this thread's pixels and channels; returns the sum over them of (1 - SSIM) in
// fixed point (0 outside the valid region or the frame).
__device__ __forceinline__ long long ssim_tile_sum(SsimStage& s, const SsimW& W11, int tx, int ty, int W, int H) {
    constexpr int kRunH = 8, kRunV = 4, kTaps = 2 * kSR + 1;
    if (threadIdx.x < 3 * kSS * (kTile / kRunH)) {
        const int r = threadIdx.x % kSS, t = threadIdx.x / kSS, ch = t % 3, c0 = (t / 3) * kRunH;
        float2 am[kRunH], aq[kRunH];
        float ap[kRunH];
#pragma unroll
        for (int o = 0; o < kRunH; o++) {
            am[o] = aq[o] = make_float2(0.0f, 0.0f);
            ap[o] = 0.0f;
        }
#pragma unroll
        for (int i = 0; i < kRunH + kTaps - 1; i++) {
            const float2 v = s.in[ch][r][c0 + i], vv = __fmul2_rn(v, v);
            const float xy = __fmul_rn(v.x, v.y);
#pragma unroll
            for (int o = 0; o < kRunH; o++) {
                if (i < o || i > o + kTaps - 1) continue;
                const float w = W11.w[i - o];
                const float2 w2 = make_float2(w, w);
                am[o] = __ffma2_rn(w2, v, am[o]);
                aq[o] = __ffma2_rn(w2, vv, aq[o]);
                ap[o] = __fmaf_rn(w, xy, ap[o]);
            }
        }
        float4* dm = reinterpret_cast<float4*>(&s.m[ch][r][c0]);
        float4* dq = reinterpret_cast<float4*>(&s.q[ch][r][c0]);
        float4* dp = reinterpret_cast<float4*>(&s.p[ch][r][c0]);
#pragma unroll
        for (int o = 0; o < kRunH; o += 2) {
            dm[o / 2] = make_float4(am[o].x, am[o].y, am[o + 1].x, am[o + 1].y);
            dq[o / 2] = make_float4(aq[o].x, aq[o].y, aq[o + 1].x, aq[o + 1].y);
        }
        dp[0] = make_float4(ap[0], ap[1], ap[2], ap[3]);
        dp[1] = make_float4(ap[4], ap[5], ap[6], ap[7]);
    }
    __syncthreads();
    long long fx = 0;
    {
        static_assert(kSsimThreads == 3 * kTile * (kTile / kRunV), "a thread per vertical run");
        const int lj = threadIdx.x % kTile, r0 = (threadIdx.x / kTile) % (kTile / kRunV) * kRunV;
        const int ch = threadIdx.x / (kTile * (kTile / kRunV));
        float2 am[kRunV], aq[kRunV];
        float ap[kRunV];
#pragma unroll
        for (int o = 0; o < kRunV; o++) {
            am[o] = aq[o] = make_float2(0.0f, 0.0f);
            ap[o] = 0.0f;
        }
#pragma unroll
        for (int i = 0; i < kRunV + kTaps - 1; i++) {
            const float2 vm = s.m[ch][r0 + i][lj], vq = s.q[ch][r0 + i][lj];
            const float vp = s.p[ch][r0 + i][lj];
#pragma unroll
            for (int o = 0; o < kRunV; o++) {
                if (i < o || i > o + kTaps - 1) continue;
                const float w = W11.w[i - o];
                const float2 w2 = make_float2(w, w);
                am[o] = __ffma2_rn(w2, vm, am[o]);
                aq[o] = __ffma2_rn(w2, vq, aq[o]);
                ap[o] = __fmaf_rn(w, vp, ap[o]);
            }
        }
        const float C1 = 1e-4f, C2 = 9e-4f;
        const int px = tx * kTile + lj;
#pragma unroll
        for (int o = 0; o < kRunV; o++) {
            const int py = ty * kTile + r0 + o;
            if (px < kSR || px >= W - kSR || py < kSR || py >= H - kSR) continue;
            const float mx = am[o].x, my = am[o].y, exx = aq[o].x, eyy = aq[o].y, exy = ap[o];
            const float mxy = __fmul_rn(mx, my), mxx = __fmul_rn(mx, mx), myy = __fmul_rn(my, my);
            const float num = __fmul_rn(__fadd_rn(__fmul_rn(2.0f, mxy), C1),
                                        __fadd_rn(__fmul_rn(2.0f, __fsub_rn(exy, mxy)), C2));
            const float den = __fmul_rn(__fadd_rn(__fadd_rn(mxx, myy), C1),
                                        __fadd_rn(__fadd_rn(__fsub_rn(exx, mxx), __fsub_rn(eyy, myy)), C2));
            const float one_minus = __fsub_rn(1.0f, __fdiv_rn(num, den));
            fx += __float2ll_rn(__fmul_rn(one_minus, kSsimFx));
        }
    }
    return fx;
}

// block-wide sum of a 64-bit value, added to *dst by thread 0
__device__ __forceinline__ void block_add_ll(long long v, unsigned long long* dst) {
    __shared__ long long red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[w];
        if (t) atomicAdd(dst, (unsigned long long)t);
    }
    __syncthreads();
}

// stage the 26x26 neighbourhood of tile (tx, ty): x from `test` (or the clean
// image with dirty-tile deltas, see below), y from `clean`; outside the frame 0
__device__ __forceinline__ void stage_pair(SsimStage& s, const float* __restrict__ test,
                                           const float* __restrict__ clean, int tx, int ty, int W, int H) {
    constexpr int kRounds = (kSS * kSS + kSsimThreads - 1) / kSsimThreads;
    float u[kRounds][3], v[kRounds][3];   // all loads first: the block has nothing else to do meanwhile
#pragma unroll
    for (int k = 0; k < kRounds; k++) {
        const int q = (int)threadIdx.x + k * kSsimThreads, r = q / kSS, c = q % kSS;
        const int gx = tx * kTile - kSR + c, gy = ty * kTile - kSR + r;
        const bool in = q < kSS * kSS && gx >= 0 && gx < W && gy >= 0 && gy < H;
        const size_t o = in ? ((size_t)gy * W + gx) * 3 : 0;
#pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            u[k][ch] = in ? __ldg(test + o + ch) : 0.0f;
            v[k][ch] = in ? __ldg(clean + o + ch) : 0.0f;
        }
    }
#pragma unroll
    for (int k = 0; k < kRounds; k++) {
        const int q = (int)threadIdx.x + k * kSsimThreads, r = q / kSS, c = q % kSS;
        if (q >= kSS * kSS) continue;
#pragma unroll
        for (int ch = 0; ch < 3; ch++) s.in[ch][r][c] = make_float2(clamp01(u[k][ch]), clamp01(v[k][ch]));
    }
    __syncthreads();
}

// full frames: one block per tile of an image pair (blockIdx.y)
__global__ __launch_bounds__(kSsimThreads) void k_ssim_full(const float* __restrict__ test, const float* __restrict__ clean,
                                                       int W, int H, int tiles_x, SsimW w11,
                                                       unsigned long long* __restrict__ acc) {
    __shared__ SsimStage s;
    const int tx = blockIdx.x % tiles_x, ty = blockIdx.x / tiles_x;
    const size_t img = (size_t)blockIdx.y * W * H * 3;
    stage_pair(s, test + img, clean + img, tx, ty, W, H);
    block_add_ll(ssim_tile_sum(s, w11, tx, ty, W, H), acc + blockIdx.y);
}

__global__ void k_ssim_finalize(const unsigned long long* acc, int count, int W, int H, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const double nvalid = 3.0 * (double)max(W - 2 * kSR, 0) * (double)max(H - 2 * kSR, 0);
    out[i] = nvalid > 0 ? 1.0 - (double)(long long)acc[i] * (1.0 / 4294967296.0) / nvalid : 1.0;
}

}  // namespace

SsimW ssim_weights() {
    SsimW w;
    double v[2 * kSR + 1], t = 0.0;
    for (int i = -kSR; i <= kSR; i++) t += (v[i + kSR] = std::exp(-(double)(i * i) / (2.0 * 1.5 * 1.5)));
    for (int i = 0; i < 2 * kSR + 1; i++) w.w[i] = (float)(v[i] / t);
    return w;
}

// ---------------------------------------------------------------------------
// dirty-tile engine: the SSIM of every (variant, view) from the re-blended
// pixels.  Corrupted values: the clean image with each active pixel's new
// value (deltas written by the blend kernel, found through the per-(variant,
// view) tile -> plan slot map and the slot's block -> delta index table).
// Each tile within one tile of a planned tile is claimed once (atomicMax of a
// per-batch generation tag) by the claim kernel, which lists it (queue[7] counts);
// the tiles listed are then processed by one block each.
// ---------------------------------------------------------------------------

// Thread per (plan slot, one of the 3x3 tiles around it): claims the tile if a
// changed pixel's window reaches it -- the tile itself if any pixel changed, a
// neighbour if one changed within 5 pixels of the shared edge.  (Claimed by the
// processing blocks, one pair after another, the 9 tests of each slot cost more
// than the tiles.)
__global__ __launch_bounds__(256) void k_ssim_claim(const ViewPtrs* __restrict__ views, int K,
                                                    unsigned int* __restrict__ queue, SsimBufs sb) {
    const uint32_t n_items = min(queue[9], sb.slot_cap);   // beyond it the batch reports an overflow
    const unsigned long long gen = (unsigned long long)queue[6] << 32;
    const int lane = threadIdx.x & 31;
    for (uint32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < n_items * 9u;
         base += gridDim.x * blockDim.x) {
        const uint32_t pair = base + (uint32_t)lane;
        bool claim = false;
        if (pair < n_items * 9u) {
            const uint32_t slot = pair / 9u, nb = pair % 9u;
            const unsigned f = sb.slot_flags[slot];
            const int dx = (int)(nb % 3u) - 1, dy = (int)(nb / 3u) - 1;
            if ((f & 16u) && (dx == 0 || (f & (dx < 0 ? 1u : 2u))) && (dy == 0 || (f & (dy < 0 ? 4u : 8u)))) {
                const uint32_t bk = sb.plan[slot].bk, tile = sb.plan[slot].tile;
                const ViewPtrs& v = views[bk % (uint32_t)K];
                const int tiles_y = (v.H + kTile - 1) / kTile;
                const int tx = (int)(tile % (uint32_t)v.tiles_x) + dx, ty = (int)(tile / (uint32_t)v.tiles_x) + dy;
                if (tx >= 0 && ty >= 0 && tx < v.tiles_x && ty < tiles_y)
                    claim = atomicMax(&sb.ssim_map[(size_t)bk * sb.max_tiles + (size_t)(ty * v.tiles_x + tx)], gen) < gen;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, claim);
        uint32_t at = 0;
        if (lane == 0 && m) at = atomicAdd(&queue[7], (unsigned)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + (uint32_t)__popc(m & ((1u << lane) - 1u));
        if (claim) sb.claims[at] = pair;
    }
}

__global__ __launch_bounds__(kSsimThreads) void k_dirty_ssim(const ViewPtrs* __restrict__ views, int K,
                                                        const unsigned int* __restrict__ queue, SsimBufs sb,
                                                        SsimW w11, CmpAcc* __restrict__ acc) {
    __shared__ SsimStage s;
    const PlanItem* __restrict__ plan = sb.plan;
    const unsigned long long gen = (unsigned long long)queue[6] << 32;
    const uint32_t n_tiles = queue[7];
    for (uint32_t k = blockIdx.x; k < n_tiles; k += gridDim.x) {
        const uint32_t pair = sb.claims[k], nb = pair % 9u;
        const PlanItem& it = plan[pair / 9u];
        const ViewPtrs& v = views[it.bk % (uint32_t)K];
        const int tiles_y = (v.H + kTile - 1) / kTile;
        const int tx = (int)(it.tile % (uint32_t)v.tiles_x) + (int)(nb % 3u) - 1;
        const int ty = (int)(it.tile / (uint32_t)v.tiles_x) + (int)(nb / 3u) - 1;
        // the 3x3 tiles around (tx, ty): delta index and active mask of each 8x4 block
        // (0xffffffff / 0: no delta), resolved once for the staging below
        __shared__ uint32_t nb_gi[9][8], nb_mask[9][8];
        if (threadIdx.x < 72) {
            const int t = threadIdx.x / 8, w = threadIdx.x % 8;
            const int ntx = tx + t % 3 - 1, nty = ty + t / 3 - 1;
            uint32_t gi = 0xffffffffu, m = 0u;
            if (ntx >= 0 && nty >= 0 && ntx < v.tiles_x && nty < tiles_y) {
                const unsigned long long e = sb.tile_map[(size_t)it.bk * sb.max_tiles + (size_t)(nty * v.tiles_x + ntx)];
                if ((e & 0xffffffff00000000ull) == gen) {
                    const uint32_t slot2 = (uint32_t)e;
                    gi = sb.slot_group[(size_t)slot2 * 8 + w];
                    m = gi != 0xffffffffu ? plan[slot2].mask[w] : 0u;
                }
            }
            nb_gi[t][w] = gi;
            nb_mask[t][w] = m;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < kSS * kSS; q += blockDim.x) {
            const int r = q / kSS, c = q % kSS;
            const int gx = tx * kTile - kSR + c, gy = ty * kTile - kSR + r;
            const bool in = gx >= 0 && gx < v.W && gy >= 0 && gy < v.H;
            float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f;
            if (in) {
                const float* cl = v.clean + ((size_t)gy * v.W + gx) * 3;
                c0 = cl[0];
                c1 = cl[1];
                c2 = cl[2];
            }
            float t0 = c0, t1 = c1, t2 = c2;
            if (in) {
                const int t = (gy / kTile - ty + 1) * 3 + (gx / kTile - tx + 1);   // 0..8 (the halo is < 1 tile)
                const int lx = gx % kTile, ly = gy % kTile;
                const int w = (ly / 4) * 2 + lx / 8, lane = (ly % 4) * 8 + lx % 8;
                if ((nb_mask[t][w] >> lane) & 1u) {
                    const float4 d = sb.deltas[(size_t)nb_gi[t][w] * 32 + lane];
                    t0 = d.x;
                    t1 = d.y;
                    t2 = d.z;
                }
            }
            s.in[0][r][c] = make_float2(clamp01(t0), clamp01(c0));
            s.in[1][r][c] = make_float2(clamp01(t1), clamp01(c1));
            s.in[2][r][c] = make_float2(clamp01(t2), clamp01(c2));
        }
        __syncthreads();
        block_add_ll(ssim_tile_sum(s, w11, tx, ty, v.W, v.H), &acc[it.bk].ssim_fx);
    }
}


gs_status launch_ssim_full(const float* test, const float* clean, int W, int H, int K, unsigned long long* acc,
                           cudaStream_t st) {
    const int tx = (W + kTile - 1) / kTile, ty = (H + kTile - 1) / kTile;
    const size_t img = (size_t)W * H * 3;
    for (int k = 0; k < K && tx * ty > 0; k += 65535) {
        const dim3 grid(tx * ty, std::min(K - k, 65535));
        k_ssim_full<<<grid, kSsimThreads, 0, st>>>(test + k * img, clean + k * img, W, H, tx, ssim_weights(), acc + k);
    }
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_ssim_finalize(const unsigned long long* acc, int count, int W, int H, double* out, cudaStream_t st) {
    if (count > 0) k_ssim_finalize<<<(count + 255) / 256, 256, 0, st>>>(acc, count, W, H, out);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_dirty_ssim(const void* dev_views, int K, unsigned int* queue, const SsimBufs& sb, CmpAcc* acc,
                            cudaStream_t st) {
    k_ssim_claim<<<num_sms() * 4, 256, 0, st>>>((const ViewPtrs*)dev_views, K, queue, sb);
    k_dirty_ssim<<<num_sms() * 4, kSsimThreads, 0, st>>>((const ViewPtrs*)dev_views, K, queue, sb, ssim_weights(), acc);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

// per (variant, view): SSIM = 1 - sum (1 - SSIM) / (3 x valid pixels)
__global__ void k_ssim_out(const CmpAcc* acc, int count, const ViewPtrs* views, int K, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const ViewPtrs& v = views[i % K];
    const double nvalid = 3.0 * (double)max(v.W - 2 * kSR, 0) * (double)max(v.H - 2 * kSR, 0);
    out[i] = nvalid > 0 ? 1.0 - (double)(long long)acc[i].ssim_fx * (1.0 / 4294967296.0) / nvalid : 1.0;
}

gs_status launch_ssim_out(const CmpAcc* acc, int count, const void* dev_views, int K, double* out, cudaStream_t st) {
    if (count > 0) k_ssim_out<<<(count + 255) / 256, 256, 0, st>>>(acc, count, (const ViewPtrs*)dev_views, K, out);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

}  // namespace gs

// SSIM of K image pairs (see gs.h)
extern "C" gs_status gs_ssim(const float* dev_test, const float* dev_clean, int H, int W, int K, double* dev_out,
                             void* stream) {
    using namespace gs;
    if (!dev_test || !dev_clean || !dev_out || H < 1 || W < 1 || K < 1)
        return set_error(GS_ERR_ARG, "bad gs_ssim arguments");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned long long* acc = nullptr;
    GS_CUDA(cudaMallocAsync((void**)&acc, sizeof(unsigned long long) * K, st));
    gs_status rs = GS_OK;
    if (cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * K, st) != cudaSuccess) rs = set_error(GS_ERR_CUDA, "memset");
    if (rs == GS_OK) rs = launch_ssim_full(dev_test, dev_clean, W, H, K, acc, st);
    if (rs == GS_OK) rs = launch_ssim_finalize(acc, K, W, H, dev_out, st);
    cudaFreeAsync(acc, st);
    return rs;
}
