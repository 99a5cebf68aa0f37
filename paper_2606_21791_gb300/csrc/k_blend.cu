// (d) front-to-back alpha blending and (e) comparison against the clean frame.
//
// Blend (3DGS forward pass, composited over white as in Sec. 3 "Metrics and
// severity"): one block of tw th / 2 threads per tw x th tile, a warp per 8x8 block of
// pixels, two pixels per lane.  The tile's sorted list is staged through shared memory a
// tile's pixels' worth of records at a time.  Each warp skips every staged primitive
// whose alpha >= 1/255 box (BlendRec::ex/ey, conservative) misses its block, 32 at a
// time.  Per pixel: power = -(a dx^2 + c dy^2)/2 - b dx dy; skip power > 0;
// alpha = opacity exp(power); skip alpha < 1/255; alpha capped at 0.99; stop
// before the primitive that would take T below 1e-4; C += colour alpha T.
// The block leaves as soon as all of its pixels have stopped.
//
// Compare (Definitions 1-2): squared differences of [0,1]-clamped images (NaN counts
// as 0), each pixel's rounded to a fixed-point integer, are summed and added
// atomically, so a (variant, view) record does not depend on which tiles ran or in
// what order: a dirty-tile re-blend and a full re-render give identical records.
//
// Dirty-tile engine: the plan lists the (variant, view, tile) candidates that the
// flipped primitive's clean or corrupted record can reach; the dirty blend decides
// per pixel, re-blends the pixels that can change from their own blend lists (in dense
// views from their block's list; both kept with the clean view), with the clean entry
// left out and the corrupted record at its (depth, index) place, and compares them on
// the fly.
#include <algorithm>
#include <mutex>

#include "gs_internal.h"

namespace gs {

namespace {

constexpr int kBT = 256;

// Shared staging of one batch of list entries.  box = conservative alpha box
// (x0, x1, y0, y1); q0 = (mean x, mean y, ca, cb), q1 = (cc, opacity, r, g), qb = b.
struct Stage {
    float4 box[kBT];
    float4 q0[kBT];
    float4 q1[kBT];
    float qb[kBT];
};

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ void stage_put(Stage& s, int j, const BlendRec& q) {
    s.box[j] = make_float4(q.mx - q.ex, q.mx + q.ex, q.my - q.ey, q.my + q.ey);
    s.q0[j] = make_float4(q.mx, q.my, q.ca, q.cb);
    s.q1[j] = make_float4(q.cc, q.opac, q.r, q.g);
    s.qb[j] = q.b;
}

__device__ __forceinline__ BlendRec load_rec(const BlendRec* recs, uint32_t id) {
    const float4* p = reinterpret_cast<const float4*>(recs + id);
    float4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    BlendRec q;
    q.mx = a.x;
    q.my = a.y;
    q.ca = a.z;
    q.cb = a.w;
    q.cc = b.x;
    q.opac = b.y;
    q.ex = b.z;
    q.ey = b.w;
    q.r = c.x;
    q.g = c.y;
    q.b = c.z;
    q.depth = c.w;
    return q;
}

struct Pix {
    float T, c0, c1, c2;
    bool done;
};

// 8x8 block b of a tile with 8x4 blocks per row nbx = 1 << lg: its upper 8x4
// block in the natural order (the lower one is that + nbx) and its offset in the tile.
__host__ __device__ inline int block_upper(int b, int lg) { return (b & ((1 << lg) - 1)) + ((b >> lg) << (lg + 1)); }
__host__ __device__ inline int block_x0(int b, int lg) { return (b & ((1 << lg) - 1)) * 8; }
__host__ __device__ inline int block_y0(int b, int lg) { return (b >> lg) * 8; }

// 2^x (hardware approximation, flushes subnormal results to zero)
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Each warp tests 32 staged entries at a time against its pixel block (one box
// load per lane, a ballot), then walks only the survivors in list order.  An
// entry culled here cannot reach alpha >= 1/255 at any of the warp's pixels, so
// skipping it changes no pixel; a NaN box never culls.
// Survivors a warp takes at a time: their alphas do not depend on the pixel
// state, so they are computed as independent chains, then applied in list order.
// The front-to-back step of one entry at one pixel (alpha capped at 0.99, NaN
// kept; stop when T would drop below 1e-4; C += colour * alpha * T) has explicit
// rounding in every operation, so the full-frame, clean and dirty-tile kernels
// compute the same bits wherever it is inlined.
constexpr int kAlphaGroup = 4;

// A staged entry as the walk needs it.
struct EntryQ {
    float4 q0;          // mx, my, ca, cb
    float cc, opac, r, g, b;
};

// One front-to-back step of an entry at one pixel, alpha already computed (ok:
// the blend takes the entry there; live: the pixel has not stopped): alpha
// capped at 0.99 (NaN kept), stop when T would drop below 1e-4, else
// C += colour * alpha * T.  Every operation is rounded on its own, so each
// kernel that inlines it computes the same bits.  Returns whether the pixel
// stopped at this entry.  (Packing the two pixels' steps into fp32x2
// operations computes the same bits but costs more than it saves: the state
// has to be packed and the updates selected per pixel.)
__device__ __forceinline__ bool apply_entry(Pix& p, bool live, bool ok, float a, float cr, float cg, float cb) {
    const bool act = live && ok;
    const float al = a > 0.99f ? 0.99f : a;   // keeps NaN
    const float Tn = __fmul_rn(p.T, __fsub_rn(1.0f, al));
    const bool stop_here = act && Tn < 1e-4f;
    const bool upd = act && !(Tn < 1e-4f);
    const float w = __fmul_rn(al, p.T);
    p.c0 = upd ? __fmaf_rn(cr, w, p.c0) : p.c0;
    p.c1 = upd ? __fmaf_rn(cg, w, p.c1) : p.c1;
    p.c2 = upd ? __fmaf_rn(cb, w, p.c2) : p.c2;
    p.T = upd ? Tn : p.T;
    p.done = p.done || stop_here;
    return stop_here;
}

// alpha of an entry at this lane's two pixels, which share a column (centres
// (pxc, pyA) and (pxc, pyB), npy = (-pyA, -pyB)); ok: the blend takes the entry there
// (power <= 0 or NaN, alpha not below 1/255).  The exponent of the Gaussian at offset
// (dx, dy), power = -(ca dx^2 + cc dy^2)/2 - cb dx dy, is evaluated as s = fma(cc dy, dy,
// ca dx dx), power = fma(-cb dx, dy, -s/2): each product rounded on its own, each sum
// fused with its product (one rounding).  Every evaluation here (and the oracle's) takes
// this order, so it is reproducible bit for bit -- which matters for near-degenerate
// conics, where cancellation makes the rounding error large compared with the value.
// The x offset and the terms that depend on it alone are computed once for both pixels,
// the rest as packed fp32x2 operations: no product feeds a separate addition, so they
// compute the bits of the scalar order.
__device__ __forceinline__ float2 alpha_pair(const EntryQ& q, float pxc, float2 npy, bool& okA, bool& okB) {
    const float dx = __fsub_rn(q.q0.x, pxc);
    const float t1 = __fmul_rn(__fmul_rn(q.q0.z, dx), dx);
    const float bdxn = __fmul_rn(-q.q0.w, dx);
    const float2 dy = __fadd2_rn(make_float2(q.q0.y, q.q0.y), npy);   // my - py, one rounding each
    const float2 sq = __ffma2_rn(__fmul2_rn(make_float2(q.cc, q.cc), dy), dy, make_float2(t1, t1));
    const float2 pw = __ffma2_rn(make_float2(bdxn, bdxn), dy, __fmul2_rn(make_float2(-0.5f, -0.5f), sq));
    const float2 pl = __fmul2_rn(pw, make_float2(kLog2e, kLog2e));
    const float2 a = __fmul2_rn(make_float2(q.opac, q.opac), make_float2(ex2_approx(pl.x), ex2_approx(pl.y)));
    okA = !(pw.x > 0.0f) && !(a.x < 1.0f / 255.0f);
    okB = !(pw.y > 0.0f) && !(a.y < 1.0f / 255.0f);
    return a;
}

// Walk the survivors m (bit i: entry c + i) in list order for this lane's two
// pixels: apply(entry index, live, ok flags, alphas, colour) takes them one by
// one, kAlphaGroup at a time; after() follows each such group.
template <class Fetch, class Apply, class After>
__device__ __forceinline__ void walk_survivors2(unsigned m, int c, const Fetch& fetch, float pxc, float pyA,
                                                float pyB, const Apply& apply, const After& after) {
    const float2 npy = make_float2(-pyA, -pyB);
    while (m) {
        int e[kAlphaGroup];
        bool v[kAlphaGroup], okA[kAlphaGroup], okB[kAlphaGroup];
        float2 a[kAlphaGroup];
        float cr[kAlphaGroup], cg[kAlphaGroup], cb[kAlphaGroup];
#pragma unroll
        for (int k = 0; k < kAlphaGroup; k++) {
            v[k] = m != 0u;
            e[k] = v[k] ? c + __ffs(m) - 1 : c;
            m &= m - 1u;
        }
#pragma unroll
        for (int k = 0; k < kAlphaGroup; k++) {
            const EntryQ q = fetch(e[k]);
            a[k] = alpha_pair(q, pxc, npy, okA[k], okB[k]);
            cr[k] = q.r;
            cg[k] = q.g;
            cb[k] = q.b;
        }
        // apply in list order with selects (no divergent branch per entry)
#pragma unroll
        for (int k = 0; k < kAlphaGroup; k++) apply(e[k], v[k], okA[k], okB[k], a[k], cr[k], cg[k], cb[k]);
        after();
    }
}

// The two pixels of a lane in 8x8 block b of a tile (the full-frame kernels: b =
// warp): pixel A at (lane % 8, lane / 8) of the block, B four rows below; u0 and
// u1 are their indices in the tile's natural (8x4 block) order.
struct Pix2Geo {
    int px, pyA, pyB, u0, u1;
    float pxc, pycA, pycB;
    float wx0, wx1, wy0, wy1;   // pixel-centre box of the 8x8 block
    bool inA, inB;
};

__device__ __forceinline__ Pix2Geo pix2_geo(int tile_x, int tile_y, int tw, int th, int W, int H, int b) {
    const int lane = threadIdx.x & 31, lg = tile_lgx(tw);
    Pix2Geo g;
    const int bx = tile_x * tw + block_x0(b, lg), by = tile_y * th + block_y0(b, lg);
    g.px = bx + (lane & 7);
    g.pyA = by + (lane >> 3);
    g.pyB = g.pyA + 4;
    g.u0 = block_upper(b, lg) * 32 + lane;
    g.u1 = g.u0 + (32 << lg);
    g.pxc = (float)g.px + 0.5f;
    g.pycA = (float)g.pyA + 0.5f;
    g.pycB = (float)g.pyB + 0.5f;
    g.wx0 = (float)bx + 0.5f;
    g.wx1 = (float)bx + 7.5f;
    g.wy0 = (float)by + 0.5f;
    g.wy1 = (float)by + 7.5f;
    g.inA = g.px < W && g.pyA < H;
    g.inB = g.px < W && g.pyB < H;
    return g;
}

// Conservative test of a rectangle, all in fp32: false only if the blend cannot reach
// alpha >= 1/255 for record q at any pixel centre of the rectangle
// [x0, x1] x [y0, y1].  The blend's offsets d = mean - pixel are fp32
// differences, and rounding is monotone, so every pixel's d lies in the box
// spanned by the rounded corner offsets.  Its power is -q(d)/2 for
// q(d) = ca dx^2 + 2 cb dx dy + cc dy^2 up to a few ulps of
// M = ((|ca| + |cb|) max dx^2 + (|cc| + |cb|) max dy^2)/2 >= the sum of |terms|;
// g = 1e-5 covers that and the rounding of this test's own q (both about
// 1e-6 M).  alpha >= 1/255 needs -q/2 + g M >= -L with L = ln(255 opacity)
// + 1e-3 (the margin covers the fast log and exp2), so the rectangle is
// unreachable when the minimum of q over it exceeds 2 L + 2 g M.  With ca, cc > 0
// the minimum over each edge is that of a convex 1-D quadratic; it is 0 if the
// mean lies inside (then: reachable).  NaN opacity, or terms near overflow
// (where the blend's own power can be NaN, which it blends): reachable.
__device__ __forceinline__ bool rect_reachable(float mx, float my, float ca, float cb, float cc, float opac, float x0,
                                               float x1, float y0, float y1) {
    const float L = __logf(255.0f * opac) + 1e-3f;
    if (!(ca > 1e-30f) || !(cc > 1e-30f) || !(L < 3.0e38f)) return true;
    const float dx0 = mx - x1, dx1 = mx - x0;
    const float dy0 = my - y1, dy1 = my - y0;
    const float mdx = fmaxf(dx0 * dx0, dx1 * dx1), mdy = fmaxf(dy0 * dy0, dy1 * dy1);
    const float M = 0.5f * ((ca + fabsf(cb)) * mdx + (cc + fabsf(cb)) * mdy);
    if (!(M < 1.0e37f)) return true;   // terms near overflow: the blend's power may be NaN
    if (L < 0.0f) return false;        // alpha <= opacity < 1/255 everywhere (with margin)
    if (dx0 <= 0.0f && dx1 >= 0.0f && dy0 <= 0.0f && dy1 >= 0.0f) return true;
    auto qf = [&](float dx, float dy) { return ca * dx * dx + 2.0f * cb * dx * dy + cc * dy * dy; };
    // approximate reciprocals: they only place the nearest point of an edge, and
    // a relative error e there raises q by about e^2 M, far inside the margin
    const float rca = __fdividef(1.0f, ca), rcc = __fdividef(1.0f, cc);
    // the nearest point of each edge (dx fixed: dy = -cb dx / cc; dy fixed: dx = -cb dy / ca), clamped to it
    const float e0 = qf(dx0, fminf(fmaxf(-cb * dx0 * rcc, dy0), dy1));
    const float e1 = qf(dx1, fminf(fmaxf(-cb * dx1 * rcc, dy0), dy1));
    const float e2 = qf(fminf(fmaxf(-cb * dy0 * rca, dx0), dx1), dy0);
    const float e3 = qf(fminf(fmaxf(-cb * dy1 * rca, dx0), dx1), dy1);
    const float qmin = fminf(fminf(e0, e1), fminf(e2, e3));
    return !(qmin > 2.0f * L + 2.0e-5f * M);
}

// The clean views' stages: records as they are, one entry per thread and batch.
constexpr int kStageMax = kBT / 2;
template <int N>
struct RawStageN {
    float4 q0[N];   // mx, my, ca, cb
    float4 q1[N];   // cc, opacity, ex, ey
    float4 q2[N];   // r, g, b, depth
};
using RawStage = RawStageN<kStageMax>;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned saddr = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(saddr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    const unsigned saddr = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(saddr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Streams a tile's list [rg.x, rg.y) through two stages, one entry per thread and
// batch: while a batch is blended, the records of the next one are copied into the
// other stage and the indices of the one after are loaded, so a batch costs one
// barrier and no memory latency.  copy(stage, id) may bring more of this thread's
// entry; blend(stage, its number, entries, list index of entry 0); done: this
// thread's pixels need no more entries (the block leaves when all do).  For the
// clean views' two passes, which have few warps per SM to hide a batch's loads
// behind (registers, list rings): with the ellipse test, 0.44 + 0.90 ms for two
// 1600x1040 views of 300k primitives against 0.44 + 0.97 staged in turn, and 0.48 +
// 1.01 staged without the test.  The plain renders have warps enough: 208 us
// streamed, 207 staged.
template <class Copy, class Blend, class Done>
__device__ __forceinline__ void stream_list(RawStage (&st)[2], const BlendRec* __restrict__ recs,
                                            const uint32_t* __restrict__ ids, uint2 rg, const Copy& copy,
                                            const Blend& blend, const Done& done) {
    const uint32_t nb = blockDim.x, t = threadIdx.x;
    auto fetch = [&](int k, uint32_t id) {
        const float4* src = reinterpret_cast<const float4*>(recs + id);
        cp_async16(&st[k].q0[t], src);
        cp_async16(&st[k].q1[t], src + 1);
        cp_async16(&st[k].q2[t], src + 2);
        copy(k, id);
    };
    if (rg.x + t < rg.y) fetch(0, ids[rg.x + t]);
    uint32_t next = rg.x + nb + t < rg.y ? ids[rg.x + nb + t] : 0u;
    int k = 0;
    for (uint32_t base = rg.x; base < rg.y; base += nb, k ^= 1) {
        cp_async_wait_all();
        // the batch has landed for every thread, and every thread is done with the other stage
        if (__syncthreads_count(done()) == (int)nb) break;
        if (base + nb + t < rg.y) fetch(k ^ 1, next);
        next = base + 2 * nb + t < rg.y ? ids[base + 2 * nb + t] : 0u;
        blend(st[k], k, (int)min(nb, rg.y - base), base - rg.x);
    }
    cp_async_wait_all();   // leave no copy in flight
}

// Entries [c, c + 32) of a staged batch for one warp: cull 32 boxes against the
// warp's 8x8 pixel block with one ballot, then walk the survivors in list order.
// CONIC: survivors whose ellipse misses the block (rect_reachable: no pixel of it
// would take them) are dropped as well, 32 tests side by side, when at least
// kConicMin are left to gain from it: a box keeps the blocks at the corners of a
// slanted ellipse.  One 1600x1040 view of 2M primitives: 206 us without, 195 at 5,
// 197 at 8, 201 at 2 (189 to 195 over boxes of the same kind).  Not for the compared
// renders of corrupted scenes: there most of a deep list is exploded primitives whose
// ellipse does cover the block (four renders with 1000 upsets each: 558 us without,
// 630 with).
constexpr int kConicMin = 5;

template <bool CONIC, class Apply, class After>
__device__ __forceinline__ void blend_chunk2(const Stage& s, int c, int cnt, const Pix2Geo& g, const Apply& apply,
                                             const After& after) {
    const int lane = threadIdx.x & 31;
    const int j = c + lane;
    bool pass = false;
    if (j < cnt) {
        const float4 bx = s.box[j];
        pass = !(bx.y < g.wx0 || bx.x > g.wx1 || bx.w < g.wy0 || bx.z > g.wy1);
    }
    unsigned m = __ballot_sync(0xffffffffu, pass);
    if (CONIC && __popc(m) >= kConicMin) {
        if (pass) {
            const float4 q0 = s.q0[j], q1 = s.q1[j];
            pass = rect_reachable(q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, g.wx0, g.wx1, g.wy0, g.wy1);
        }
        m = __ballot_sync(0xffffffffu, pass);
    }
    auto fetch = [&](int e) {
        const float4 q1 = s.q1[e];
        return EntryQ{s.q0[e], q1.x, q1.y, q1.z, q1.w, s.qb[e]};
    };
    walk_survivors2(m, c, fetch, g.pxc, g.pycA, g.pycB, apply, after);
}

// survivors of entries [c, c + 32) of a raw stage
template <bool CONIC, int N>
__device__ __forceinline__ unsigned chunk_survivors(const RawStageN<N>& s, int c, int cnt, const Pix2Geo& g) {
    const int j = c + (threadIdx.x & 31);
    bool pass = false;
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
    if (j < cnt) {
        a = s.q0[j];
        b = s.q1[j];
        pass = !(a.x + b.z < g.wx0 || a.x - b.z > g.wx1 || a.y + b.w < g.wy0 || a.y - b.w > g.wy1);
    }
    unsigned m = __ballot_sync(0xffffffffu, pass);
    if (CONIC && __popc(m) >= kConicMin) {
        pass = pass && rect_reachable(a.x, a.y, a.z, a.w, b.x, b.y, g.wx0, g.wx1, g.wy0, g.wy1);
        m = __ballot_sync(0xffffffffu, pass);
    }
    return m;
}

template <int N, class Apply, class After>
__device__ __forceinline__ void walk_raw2(unsigned m, const RawStageN<N>& s, int c, const Pix2Geo& g,
                                          const Apply& apply, const After& after) {
    auto fetch = [&](int e) {
        const float4 q1 = s.q1[e], q2 = s.q2[e];
        return EntryQ{s.q0[e], q1.x, q1.y, q2.x, q2.y, q2.z};
    };
    walk_survivors2(m, c, fetch, g.pxc, g.pycA, g.pycB, apply, after);
}

__device__ __forceinline__ float clamp01(float v) { return v > 0.0f ? (v < 1.0f ? v : 1.0f) : 0.0f; }

// One pixel's comparison terms: squared error of the [0,1]-clamped values in
// fixed point (integer sums do not depend on the order of accumulation), peak
// |difference|, footprint flag (> 1/255), non-finite flag of the new value.
struct PixCmp {
    unsigned long long fx;
    float m;
    bool foot, nonfin;
};

__device__ __forceinline__ PixCmp pixel_compare(float v0, float v1, float v2, const float* c) {
    PixCmp r;
    const float d0 = clamp01(v0) - clamp01(c[0]);
    const float d1 = clamp01(v1) - clamp01(c[1]);
    const float d2 = clamp01(v2) - clamp01(c[2]);
    const float sq = d0 * d0 + d1 * d1 + d2 * d2;
    r.fx = __float2ull_rn(sq * 549755813888.0f);   // 2^kSseFracBits
    r.m = fmaxf(fmaxf(fabsf(d0), fabsf(d1)), fabsf(d2));   // differences are finite
    r.foot = r.m > 1.0f / 255.0f;
    r.nonfin = !(isfinite(v0) && isfinite(v1) && isfinite(v2));
    return r;
}

__device__ __forceinline__ void add_work(unsigned long long* work, unsigned int nev, unsigned int staged) {
    unsigned int w = __reduce_add_sync(0xffffffffu, nev);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(&work[0], (unsigned long long)w);
    if (threadIdx.x == 0) {
        atomicAdd(&work[1], 1ull);
        atomicAdd(&work[2], (unsigned long long)staged);
    }
}

// Both pixels of a lane against the clean image, added to *acc for the block
// (fixed-point squared errors: the sum does not depend on the order).
__device__ __forceinline__ void compare_tile2(const Pix2Geo& g, float a0, float a1, float a2, float b0, float b1,
                                              float b2, const float* clean, int W, CmpAcc* acc) {
    __shared__ unsigned long long wsse[kBT / 32];
    __shared__ float wmax[kBT / 32];
    __shared__ unsigned wfoot[kBT / 32], wbad[kBT / 32];
    PixCmp rA{0ull, 0.0f, false, false}, rB{0ull, 0.0f, false, false};
    if (g.inA) rA = pixel_compare(a0, a1, a2, clean + ((size_t)g.pyA * W + g.px) * 3);
    if (g.inB) rB = pixel_compare(b0, b1, b2, clean + ((size_t)g.pyB * W + g.px) * 3);
    unsigned long long fx = rA.fx + rB.fx;
    float m = fmaxf(rA.m, rB.m);
    for (int o = 16; o > 0; o >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    const unsigned nf = __reduce_add_sync(0xffffffffu, (rA.foot ? 1u : 0u) + (rB.foot ? 1u : 0u));
    const unsigned nb = __reduce_add_sync(0xffffffffu, (rA.nonfin ? 1u : 0u) + (rB.nonfin ? 1u : 0u));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        wsse[warp] = fx;
        wmax[warp] = m;
        wfoot[warp] = nf;
        wbad[warp] = nb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        float mm = 0.0f;
        unsigned nfoot = 0, nbad = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            t += wsse[w];
            mm = fmaxf(mm, wmax[w]);
            nfoot += wfoot[w];
            nbad += wbad[w];
        }
        if (t) atomicAdd(&acc->sse_fx, t);
        if (mm > 0.0f) atomicMax(&acc->maxabs_bits, __float_as_uint(mm));
        if (nfoot) atomicAdd(&acc->footprint, nfoot);
        if (nbad) atomicAdd(&acc->nonfinite, nbad);
    }
}

// MODE 0: write the image; 1: compare with the clean image.
// One block of tw * th / 2 threads per tw x th tile: warp b blends the tile's
// 8x8 block b, two pixels per lane.
template <int MODE, bool COUNT>
__global__ __launch_bounds__(kBT / 2) void k_blend_full(const BlendRec* __restrict__ recs,
                                                       const uint32_t* __restrict__ ids,
                                                       const uint2* __restrict__ ranges, int W, int H, int tiles_x,
                                                       int tw, int th, float* __restrict__ img,
                                                       const float* __restrict__ clean, CmpAcc* acc,
                                                       unsigned long long* work) {
    __shared__ Stage s;
    const int tile = blockIdx.x;
    const uint32_t P = (uint32_t)(tw * th);   // pixels of a tile = records staged per batch
    const Pix2Geo g = pix2_geo(tile % tiles_x, tile / tiles_x, tw, th, W, H, threadIdx.x >> 5);
    Pix pA{1.0f, 0.0f, 0.0f, 0.0f, !g.inA}, pB{1.0f, 0.0f, 0.0f, 0.0f, !g.inB};
    const uint2 rg = ranges[tile];
    unsigned int nev = 0, staged = 0;
    auto apply = [&](int, bool v, bool okA, bool okB, float2 a, float cr, float cg, float cb) {
        const bool liveA = v && !pA.done, liveB = v && !pB.done;
        if (COUNT) nev += (liveA ? 1u : 0u) + (liveB ? 1u : 0u);
        apply_entry(pA, liveA, okA, a.x, cr, cg, cb);
        apply_entry(pB, liveB, okB, a.y, cr, cg, cb);
    };
    for (uint32_t base = rg.x; base < rg.y; base += P) {
        const int cnt = (int)min(P, rg.y - base);
        for (int j = threadIdx.x; j < cnt; j += blockDim.x) stage_put(s, j, load_rec(recs, ids[base + j]));
        __syncthreads();
        staged += cnt;
        for (int c = 0; c < cnt && !__all_sync(0xffffffffu, pA.done && pB.done); c += 32)
            blend_chunk2<MODE == 0>(s, c, cnt, g, apply, [] {});
        // also the barrier that lets the next batch overwrite the stage
        if (__syncthreads_count(pA.done && pB.done) == (int)blockDim.x) break;
    }
    if (COUNT) add_work(work, nev, staged);
    const float a0 = __fadd_rn(pA.c0, pA.T), a1 = __fadd_rn(pA.c1, pA.T), a2 = __fadd_rn(pA.c2, pA.T);   // over white
    const float b0 = __fadd_rn(pB.c0, pB.T), b1 = __fadd_rn(pB.c1, pB.T), b2 = __fadd_rn(pB.c2, pB.T);
    if (MODE == 0) {
        if (g.inA) {
            const size_t px = (size_t)g.pyA * W + g.px;
            img[px * 3] = a0;
            img[px * 3 + 1] = a1;
            img[px * 3 + 2] = a2;
        }
        if (g.inB) {
            const size_t px = (size_t)g.pyB * W + g.px;
            img[px * 3] = b0;
            img[px * 3 + 1] = b1;
            img[px * 3 + 2] = b2;
        }
    } else {
        compare_tile2(g, a0, a1, a2, b0, b1, b2, clean, W, acc);
    }
}

// ---------------------------------------------------------------------------
// Clean views: the blend of k_blend_full, and what the dirty-tile engine keeps
// of it.  Two passes of the same blend, the second in one of two forms:
//   kImage: the image, the rank of the entry that stopped each pixel (0xffffffff if
//     none), each tile's largest stop and the length of each pixel's blend list;
//   kLists: the pixels' blend lists, the blend's state in front of every kWalk-th of
//     their entries, and the rows that say where each list stands at every
//     kRowStride-th entry of the tile's list;
//   kBlocks: of a view without blend lists (a dense one, see dense_view in gs_api.cu),
//     each 8x8 block's list -- the entries of the tile's list that its cull leaves --
//     and the pixels' states in front of every kRowStride-th of its entries.
//
// A pixel's blend list holds the entries its blend takes (power <= 0 and alpha >=
// 1/255), front to back, as (capped alpha, colour) and rank in the view's order.
// Only the flipped primitive's entry differs between a variant and the clean
// scene, so a dirty pixel is re-blended from its list: no exponent, and no entry
// that the pixel skips (2M primitives at 1600x1040 leave 20-35 entries a pixel of
// tile lists of 1,885).  The list goes on past the clean stop, because a variant
// that lacks an entry stops later: it ends where the product of (1 - alpha) over
// its entries has fallen below kListEndT.  A variant lacks at most one entry,
// whose alpha is at most 0.99, so its own T there is below 100 kListEndT (1 +
// rounding) < 1e-4: it has stopped.  (A NaN alpha makes the product NaN, which
// ends no list; a NaN corrupted alpha makes every channel NaN for good, wherever
// the walk ends.)  The end is marked by an alpha so large that T (1 - alpha) <
// 1e-4 for any T, kListEnd at rank 0xffffffff.
// ---------------------------------------------------------------------------
constexpr float kListEndT = 0.9e-6f;
constexpr float kListEnd = 1e30f;
enum CleanPass { kImage, kLists, kBlocks };

struct CleanPix {
    float T, c0, c1, c2;   // the clean blend (frozen where it stopped)
    float Tv;              // product of (1 - alpha) over every entry taken, stopped or not
    bool stopped, done;    // done: the list ends here
    uint32_t stop, last;   // rank and list position of the entry that stopped it
    uint32_t n;            // entries taken
    uint32_t off, flushed; // kLists: start of the list, entries written out
};

struct ListOut {
    float4* ent;
    uint32_t* rk;
    const uint32_t* off;   // [tiles * pixels of a tile] start of each pixel's list
    float4* state;
    uint32_t* row_idx;
    const uint32_t* row_off;
    const uint32_t* row_cnt;
    uint2* sub;            // kBlocks: (primitive, rank) of the blocks' entries
    const uint32_t* sub_off;
    float4* row_state;
};

// First row of the states of a block whose list starts at `off` (tb: the block's number
// in its view): a block of n entries has n / kRowStride + 1.
__device__ __forceinline__ size_t block_rows(uint32_t off, uint32_t tb) {
    return (size_t)(off / (uint32_t)kRowStride) + tb;
}

// Entries of a pixel on their way to its list: a lane takes an entry here and
// there, so writing each by itself would cost two partial stores per entry (0.72
// ms per pass of a 1600x1040 view of 300k primitives, 0.44 ms this way); four at a
// time they leave as whole 64-byte pieces.  Ring of 8 per pixel: a walk group adds at most
// kAlphaGroup.
struct ListRing {
    float4 e[8][64];    // [entry % 8][pixel of the 8x8 block]
    uint32_t r[8][64];
};

// two entries to a 32-byte aligned place, one 256-bit store
__device__ __forceinline__ void store_pair(float4* p, const float4& a, const float4& b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// four entries [p.flushed, p.flushed + 4) of ring column `col` to the list
static_assert(kWalk == 4, "lists start and end on the pieces written here and read by the dirty walk");
__device__ __forceinline__ void flush4(CleanPix& p, const ListRing& ring, int col, const ListOut& lo) {
    const int k = (int)(p.flushed & 4u);
    const size_t at = (size_t)p.off + p.flushed;
    store_pair(lo.ent + at, ring.e[k][col], ring.e[k + 1][col]);
    store_pair(lo.ent + at + 2, ring.e[k + 2][col], ring.e[k + 3][col]);
    *reinterpret_cast<uint4*>(lo.rk + at) =
        make_uint4(ring.r[k][col], ring.r[k + 1][col], ring.r[k + 2][col], ring.r[k + 3][col]);
    p.flushed += 4u;
}

template <CleanPass PASS>
__device__ __forceinline__ void clean_entry(CleanPix& p, bool live, bool ok, float a, float cr, float cg, float cb,
                                            uint32_t rank, uint32_t li, const ListOut& lo, ListRing* ring, int col) {
    const bool act = live && ok;
    const float al = a > 0.99f ? 0.99f : a;   // keeps NaN
    const float Tn = __fmul_rn(p.Tv, __fsub_rn(1.0f, al));
    const bool run = act && !p.stopped;       // then Tv is the blend's T
    const bool upd = run && !(Tn < 1e-4f);
    const float w = __fmul_rn(al, p.Tv);
    const float4 before = make_float4(p.T, p.c0, p.c1, p.c2);
    p.c0 = upd ? __fmaf_rn(cr, w, p.c0) : p.c0;
    p.c1 = upd ? __fmaf_rn(cg, w, p.c1) : p.c1;
    p.c2 = upd ? __fmaf_rn(cb, w, p.c2) : p.c2;
    p.T = upd ? Tn : p.T;
    if (PASS == kImage) {
        p.stop = (run && !upd) ? rank : p.stop;
        p.last = (run && !upd) ? li : p.last;
    }
    p.stopped = p.stopped || (run && !upd);
    p.Tv = act ? Tn : p.Tv;
    if (PASS == kLists && act) {
        ring->e[p.n & 7u][col] = make_float4(al, cr, cg, cb);
        ring->r[p.n & 7u][col] = rank;
        if ((p.n & (kWalk - 1u)) == 0u) lo.state[(p.off + p.n) / kWalk] = before;   // the state in front of this entry
    }
    p.n += act ? 1u : 0u;
    p.done = p.done || (act && Tn < kListEndT);
}

template <CleanPass PASS>
__global__ __launch_bounds__(kBT / 2) void k_blend_clean(const BlendRec* __restrict__ recs,
                                                        const uint32_t* __restrict__ ids,
                                                        const uint32_t* __restrict__ rank,
                                                        const uint2* __restrict__ ranges, int W, int H, int tiles_x,
                                                        int tw, int th, float* __restrict__ img,
                                                        uint32_t* __restrict__ stop, uint32_t* __restrict__ tile_stop,
                                                        uint32_t* __restrict__ tile_last, uint32_t* __restrict__ counts,
                                                        uint32_t* __restrict__ blk_cnt,
                                                        unsigned int* __restrict__ clean_nonfin, ListOut lo) {
    extern __shared__ __align__(16) unsigned char ring_mem[];   // kLists: one ListRing per warp
    __shared__ RawStage st[2];
    __shared__ uint32_t rks[2][kStageMax];   // ranks of the staged entries
    const int tile = blockIdx.x, lane = threadIdx.x & 31;
    ListRing* ring = PASS == kLists ? reinterpret_cast<ListRing*>(ring_mem) + (threadIdx.x >> 5) : nullptr;
    const uint32_t P = (uint32_t)(tw * th);
    const Pix2Geo g = pix2_geo(tile % tiles_x, tile / tiles_x, tw, th, W, H, threadIdx.x >> 5);
    CleanPix pA{1.0f, 0.0f, 0.0f, 0.0f, 1.0f, !g.inA, !g.inA, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u};
    CleanPix pB{1.0f, 0.0f, 0.0f, 0.0f, 1.0f, !g.inB, !g.inB, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u};
    const uint2 rg = ranges[tile];
    const uint32_t row0 = PASS == kLists ? lo.row_off[tile] : 0u, rows = PASS == kLists ? lo.row_cnt[tile] : 0u;
    const uint32_t tb = (uint32_t)tile * (blockDim.x >> 5) + (threadIdx.x >> 5);   // this warp's block
    const uint32_t sub0 = PASS == kBlocks ? lo.sub_off[tb] : 0u;
    uint32_t nsub = 0;   // entries that the cull has left
    if (PASS == kLists) {
        pA.off = lo.off[(size_t)tile * P + g.u0];
        pB.off = lo.off[(size_t)tile * P + g.u1];
    }
    auto put_row = [&](uint32_t j) {
        if (PASS == kLists) {   // after the first j kRowStride entries of the tile's list
            const size_t r = (size_t)(row0 + j) * P;
            lo.row_idx[r + g.u0] = pA.off + pA.n;
            lo.row_idx[r + g.u1] = pB.off + pB.n;
        } else {                // ... of the block's list
            float4* r = lo.row_state + (block_rows(sub0, tb) + j) * 64 + lane;
            r[0] = make_float4(pA.T, pA.c0, pA.c1, pA.c2);
            r[32] = make_float4(pB.T, pB.c0, pB.c1, pB.c2);
        }
    };
    if (PASS != kImage) put_row(0u);
    uint32_t at = 0;   // list index of entry 0 of the staged batch
    const uint32_t* rk = rks[0];
    auto apply = [&](int e, bool v, bool okA, bool okB, float2 a, float cr, float cg, float cb) {
        clean_entry<PASS>(pA, v && !pA.done, okA, a.x, cr, cg, cb, rk[e], at + (uint32_t)e, lo, ring, lane);
        clean_entry<PASS>(pB, v && !pB.done, okB, a.y, cr, cg, cb, rk[e], at + (uint32_t)e, lo, ring, lane + 32);
    };
    auto pending = [&](const CleanPix& p) { return (int)(p.n - p.flushed); };   // entries of the ring not yet written out
    auto drain = [&]() {   // after each walk group: make room for the next
        if (PASS != kLists) return;
        if (!__any_sync(0xffffffffu, max(pending(pA), pending(pB)) > 8 - kAlphaGroup)) return;
        if (pending(pA) >= 4) flush4(pA, *ring, lane, lo);
        if (pending(pB) >= 4) flush4(pB, *ring, lane + 32, lo);
    };
    stream_list(
        st, recs, ids, rg, [&](int k, uint32_t id) { cp_async4(&rks[k][threadIdx.x], rank + id); },
        [&](const RawStage& s, int k, int cnt, uint32_t li0) {
            at = li0;
            rk = rks[k];
            for (int c = 0; c < cnt && !__all_sync(0xffffffffu, pA.done && pB.done); c += 32) {
                const uint32_t li = at + (uint32_t)c;
                if (PASS == kLists && li > 0 && li % kRowStride == 0 && li / kRowStride <= rows) put_row(li / kRowStride);
                unsigned m = chunk_survivors<true>(s, c, cnt, g);
                if (PASS != kBlocks) {
                    nsub += (unsigned)__popc(m);
                    walk_raw2(m, s, c, g, apply, drain);
                    continue;
                }
                if ((m >> lane) & 1u)
                    lo.sub[(size_t)sub0 + nsub + (uint32_t)__popc(m & ((1u << lane) - 1u))] =
                        make_uint2(ids[rg.x + li + (uint32_t)lane], rk[c + lane]);
                while (m) {   // up to the next row, then the rest
                    const unsigned room = (unsigned)kRowStride - nsub % (unsigned)kRowStride;
                    const unsigned part = (unsigned)__popc(m) <= room ? m : m & (0xffffffffu >> (31u - __fns(m, 0, (int)room)));
                    walk_raw2(part, s, c, g, apply, drain);
                    nsub += (unsigned)__popc(part);
                    m &= ~part;
                    if (nsub % (unsigned)kRowStride == 0u) put_row(nsub / (unsigned)kRowStride);
                }
            }
        },
        [&] { return pA.done && pB.done; });
    if (PASS == kBlocks) return;
    if (PASS == kImage && lane == 0) blk_cnt[tb] = nsub;
    if (PASS == kLists) {
        auto finish = [&](CleanPix& p, int col) {
            ring->e[p.n & 7u][col] = make_float4(kListEnd, 0.0f, 0.0f, 0.0f);
            ring->r[p.n & 7u][col] = 0xffffffffu;
            if ((p.n & (kWalk - 1u)) == 0u)   // a walk may resume at the mark itself
                lo.state[(p.off + p.n) / kWalk] = make_float4(p.T, p.c0, p.c1, p.c2);
            // the list's space is a multiple of kWalk entries: whole pieces, up to the mark
            while (p.flushed <= p.n) flush4(p, *ring, col, lo);
        };
        finish(pA, lane);
        finish(pB, lane + 32);
        return;
    }
    const size_t t0 = (size_t)tile * P;
    counts[t0 + g.u0] = pA.n;
    counts[t0 + g.u1] = pB.n;
    stop[t0 + g.u0] = pA.stop;
    stop[t0 + g.u1] = pB.stop;
    const float a0 = __fadd_rn(pA.c0, pA.T), a1 = __fadd_rn(pA.c1, pA.T), a2 = __fadd_rn(pA.c2, pA.T);   // over white
    const float b0 = __fadd_rn(pB.c0, pB.T), b1 = __fadd_rn(pB.c1, pB.T), b2 = __fadd_rn(pB.c2, pB.T);
    if (g.inA) {
        const size_t px = (size_t)g.pyA * W + g.px;
        img[px * 3] = a0;
        img[px * 3 + 1] = a1;
        img[px * 3 + 2] = a2;
    }
    if (g.inB) {
        const size_t px = (size_t)g.pyB * W + g.px;
        img[px * 3] = b0;
        img[px * 3 + 1] = b1;
        img[px * 3 + 2] = b2;
    }
    const unsigned bad = (g.inA && !(isfinite(a0) && isfinite(a1) && isfinite(a2)) ? 1u : 0u) +
                         (g.inB && !(isfinite(b0) && isfinite(b1) && isfinite(b2)) ? 1u : 0u);
    const unsigned wb = __reduce_add_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && wb) atomicAdd(clean_nonfin, wb);
    // the tile's largest stop: a change at or after it leaves every pixel as it is
    __shared__ uint32_t wmax[2][kBT / 32];
    const uint32_t m = __reduce_max_sync(0xffffffffu, max(g.inA ? pA.stop : 0u, g.inB ? pB.stop : 0u));
    const uint32_t ml = __reduce_max_sync(0xffffffffu, max(g.inA ? pA.last : 0u, g.inB ? pB.last : 0u));
    if (lane == 0) {
        wmax[0][threadIdx.x >> 5] = m;
        wmax[1][threadIdx.x >> 5] = ml;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0, l = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            t = max(t, wmax[0][w]);
            l = max(l, wmax[1][w]);
        }
        tile_stop[tile] = t;
        tile_last[tile] = l;
    }
}

// The view's order: rank of every primitive, and the order's own keys (kept for
// the corrupted entries' places).
__global__ void k_ranks(const uint32_t* __restrict__ key, const uint32_t* __restrict__ id, uint64_t n,
                        uint32_t* __restrict__ rank, uint32_t* __restrict__ sdk, uint32_t* __restrict__ sid) {
    const uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const uint32_t p = id[j];
    rank[p] = (uint32_t)j;
    sdk[j] = key[j];
    sid[j] = p;
}

// Rows of each tile: row 0 and one every kRowStride list entries up to the tile's
// last stop, at most kRowsPerTile.
__global__ void k_row_counts(const uint2* __restrict__ ranges, const uint32_t* __restrict__ tile_last, int ntiles,
                             uint32_t* __restrict__ row_cnt, uint32_t* __restrict__ rows) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntiles) return;
    const uint32_t L = ranges[t].y - ranges[t].x;
    const uint32_t last = L > 0 ? min(tile_last[t], L - 1u) : 0u;
    const uint32_t c = min(last / (uint32_t)kRowStride, (uint32_t)kRowsPerTile);
    row_cnt[t] = c;
    rows[t] = c + 1u;
}

// Rank of the last entry before each row after row 0 (0xffffffff: no such row).
__global__ void k_row_keys(const uint2* __restrict__ ranges, const uint32_t* __restrict__ ids,
                           const uint32_t* __restrict__ rank, const uint32_t* __restrict__ row_cnt, int ntiles,
                           uint32_t* __restrict__ row_key) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = i / kRowsPerTile, r = i % kRowsPerTile + 1;
    if (t >= ntiles) return;
    row_key[i] = (uint32_t)r <= row_cnt[t] ? rank[ids[ranges[t].x + (uint32_t)(r * kRowStride) - 1u]] : 0xffffffffu;
}

// Space of each pixel's blend list: its entries and the end mark, in whole groups of
// kWalk.
__global__ void k_list_lens(const uint32_t* __restrict__ counts, uint64_t n, uint32_t* __restrict__ lens) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) lens[i] = (counts[i] + (uint32_t)kWalk) & ~(uint32_t)(kWalk - 1);
}

// Image pairs (blockIdx.y): a stream over both images, four pixels (three 16-byte
// loads of each image) per thread and step when both images of the pair start on
// 16-byte boundaries, one pixel otherwise.  HBM-bound: 24 B per pixel.  The terms
// of a pixel do not depend on which thread takes it and their sums are exact, so
// the result does not depend on the split.  (One block per 16x16 tile read 96-byte
// pieces of rows: 14 us for a 1600x1040 pair against 7.4 us, 0.8 of the copy peak.)
__global__ __launch_bounds__(kBT) void k_compare(const float* __restrict__ a, const float* __restrict__ b, uint64_t pix,
                                                CmpAcc* acc) {
    a += blockIdx.y * pix * 3;
    b += blockIdx.y * pix * 3;
    unsigned long long fx = 0ull;
    float m = 0.0f;
    unsigned nfoot = 0u, nbad = 0u;
    auto add = [&](float v0, float v1, float v2, float c0, float c1, float c2) {
        const float c[3] = {c0, c1, c2};
        const PixCmp r = pixel_compare(v0, v1, v2, c);
        fx += r.fx;
        m = fmaxf(m, r.m);
        nfoot += r.foot ? 1u : 0u;
        nbad += r.nonfin ? 1u : 0u;
    };
    const uint64_t tid = (uint64_t)blockIdx.x * kBT + threadIdx.x, nthr = (uint64_t)gridDim.x * kBT;
    const bool wide = (((uintptr_t)a | (uintptr_t)b) & 15u) == 0u;
    const uint64_t quads = wide ? pix / 4 : 0;
    for (uint64_t q = tid; q < quads; q += nthr) {
        const float4* va = reinterpret_cast<const float4*>(a) + 3 * q;
        const float4* vb = reinterpret_cast<const float4*>(b) + 3 * q;
        const float4 a0 = __ldcs(va), a1 = __ldcs(va + 1), a2 = __ldcs(va + 2);
        const float4 b0 = __ldcs(vb), b1 = __ldcs(vb + 1), b2 = __ldcs(vb + 2);
        add(a0.x, a0.y, a0.z, b0.x, b0.y, b0.z);
        add(a0.w, a1.x, a1.y, b0.w, b1.x, b1.y);
        add(a1.z, a1.w, a2.x, b1.z, b1.w, b2.x);
        add(a2.y, a2.z, a2.w, b2.y, b2.z, b2.w);
    }
    for (uint64_t i = 4 * quads + tid; i < pix; i += nthr)
        add(a[3 * i], a[3 * i + 1], a[3 * i + 2], b[3 * i], b[3 * i + 1], b[3 * i + 2]);
    __shared__ unsigned long long wsse[kBT / 32];
    __shared__ unsigned wmax[kBT / 32], wfoot[kBT / 32], wbad[kBT / 32];
    for (int o = 16; o > 0; o >>= 1) fx += __shfl_xor_sync(0xffffffffu, fx, o);
    const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));   // m >= 0
    const unsigned wf = __reduce_add_sync(0xffffffffu, nfoot), wb = __reduce_add_sync(0xffffffffu, nbad);
    if ((threadIdx.x & 31) == 0) {
        wsse[threadIdx.x >> 5] = fx;
        wmax[threadIdx.x >> 5] = wm;
        wfoot[threadIdx.x >> 5] = wf;
        wbad[threadIdx.x >> 5] = wb;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    CmpAcc* A = acc + blockIdx.y;
    unsigned long long t = 0;
    unsigned mm = 0, f = 0, n = 0;
    for (int w = 0; w < kBT / 32; w++) {
        t += wsse[w];
        mm = max(mm, wmax[w]);
        f += wfoot[w];
        n += wbad[w];
    }
    if (t) atomicAdd(&A->sse_fx, t);
    if (mm) atomicMax(&A->maxabs_bits, mm);
    if (f) atomicAdd(&A->footprint, f);
    if (n) atomicAdd(&A->nonfinite, n);
}

// clean_nonfin (dirty engine only): per view, the clean image's non-finite
// pixels, which count for every variant except where a pixel was re-blended.
// queue (dirty engine only): the batch's counters, cleared for the next one.
__global__ void k_finalize(const CmpAcc* acc, int count, gs_result* out, const unsigned int* clean_nonfin, int K,
                           unsigned int* queue) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (queue && i < 16) queue[i] = i == 6 ? queue[6] + 1u : 0u;   // [6]: batch generation (tags of the SSIM maps)
    if (i >= count) return;
    CmpAcc a = acc[i];
    gs_result r;
    r.sse = (double)a.sse_fx * (1.0 / 549755813888.0);
    r.maxabs = __uint_as_float(a.maxabs_bits);
    r.footprint = a.footprint;
    r.nonfinite = a.nonfinite + (clean_nonfin ? clean_nonfin[i % K] - a.clean_nonfinite_replaced : 0u);
    r.clamps = a.clamps;
    out[i] = r;
}

__global__ void k_zero_acc(CmpAcc* acc, int count) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) acc[i] = CmpAcc{0ull, 0u, 0u, 0u, 0u, 0u, 0u, 0ull, 0ull, 0ull};
}

// ---------------------------------------------------------------------------
// dirty-tile persistent kernel
// ---------------------------------------------------------------------------


// Tiles [t0, t1) of tile columns [c0, c1) whose pixel centres record q can reach
// with alpha >= 1/255 somewhere in the rows of pixel centres [y0, y1]:
// conservative, by the extent of the record's conic over the band.  The blend's
// power is within g M of -q(d)/2, M = ((|ca| + |cb|) dx^2 + (|cc| + |cb|) dy^2)/2
// and g = 1e-6 (several ulps), so with margins of 4e-5 on the diagonal the
// candidates satisfy d^T Q'' d <= R, Q'' = [[ca - 4e-5 (|ca| + |cb|), cb], [cb, cc
// - 4e-5 (|cc| + |cb|)]], R = 2 ln(255 opacity) + 2e-3 (the margin covers the
// fast log and exp2).  At a fixed dy they lie between -cb dy / q_xx +- sqrt(q_xx R -
// det dy^2) / q_xx, whatever the sign of the determinant: of an ellipse (det > 0)
// the right end is concave in dy, with its maximum at dy* = -(cb / q_yy) sqrt(R
// q_yy / det), and the left end mirrors it; with det <= 0 (needles, whose
// determinant is lost in the margins) the right end is convex and the left one
// concave, so the band's ends bound both.  The determinant is lowered by its own
// rounding error (the region only grows); the rounding of the ends is covered by a
// slack of one pixel, 2e-3 of the half width at dy = 0 (the root of a cancelling
// difference) and 1e-4 of the largest half width.  No bound (all columns): opacity
// NaN, a first diagonal term that the margin makes negative, or terms near overflow.
__device__ __forceinline__ void band_tiles(const BlendRec& q, float y0, float y1, int c0, int c1, int tw, int& t0,
                                           int& t1) {
    t0 = c0;
    t1 = c1;
    const float L = __logf(255.0f * q.opac) + 1e-3f;
    if (L < 0.0f) {   // alpha <= opacity < 1/255 everywhere (with margin); NaN falls through
        t1 = c0;
        return;
    }
    const float acb = fabsf(q.cb);
    const float qxx = q.ca - 4e-5f * (fabsf(q.ca) + acb), qyy = q.cc - 4e-5f * (fabsf(q.cc) + acb);
    const float pxy = qxx * qyy, pcb = q.cb * q.cb;
    const float det = (pxy - pcb) - 4.8e-7f * (fabsf(pxy) + pcb);
    if (!(qxx > 1e-30f) || !(fabsf(det) < 1e20f) || !(pcb < 1e20f) || !(L < 3.0e38f) || !(fabsf(q.mx) < 4e6f) ||
        !(fabsf(q.my) < 4e6f))
        return;
    const float R = 2.0f * L + 2e-3f, rq = 1.0f / qxx, h0 = sqrtf(R * rq);
    float da = q.my - y1, db = q.my - y0, dp0, dp1, dm0, dm1, hx;   // where the right / left end is furthest out
    if (det > 0.0f && qyy > 1e-30f) {
        const float rdet = R / det;
        const float hy = sqrtf(rdet * qxx) * (1.0f + 1e-4f) + 1.0f;
        hx = sqrtf(rdet * qyy);
        if (!(hy < 1e12f) || !(hx < 1e12f)) return;
        da = fmaxf(da, -hy);
        db = fminf(db, hy);
        if (da > db) {   // the band misses the ellipse
            t1 = c0;
            return;
        }
        const float dys = -q.cb / qyy * hx;
        dp0 = dp1 = fminf(fmaxf(dys, da), db);
        dm0 = dm1 = fminf(fmaxf(-dys, da), db);
    } else {
        dp0 = dm0 = da;
        dp1 = dm1 = db;
        const float far = fmaxf(fabsf(da), fabsf(db));
        hx = sqrtf(fmaxf(qxx * R - det * far * far, 0.0f)) * rq;
    }
    auto half = [&](float dy) { return sqrtf(fmaxf(qxx * R - det * dy * dy, 0.0f)); };
    const float xp = fmaxf(-q.cb * dp0 + half(dp0), -q.cb * dp1 + half(dp1)) * rq;
    const float xm = fminf(-q.cb * dm0 - half(dm0), -q.cb * dm1 - half(dm1)) * rq;
    const float slack = 1.0f + 2e-3f * h0 + 1e-4f * hx + 1e-5f * (fabsf(xp) + fabsf(xm));
    const float inv = 1.0f / (float)tw;   // tile edges are powers of two: exact
    const float f0 = floorf((q.mx - xp - slack) * inv), f1 = floorf((q.mx - xm + slack) * inv) + 1.0f;
    if (!isfinite(f0) || !isfinite(f1)) return;
    t0 = (int)fminf(fmaxf(f0, (float)c0), (float)c1);
    t1 = (int)fminf(fmaxf(f1, (float)t0), (float)c1);
}

// A pixel of a dirty tile keeps its clean value, bit for bit, when its clean
// blend stopped before the first changed list position, or when its blend skips
// both the removed (clean) and the inserted (corrupted) record (power > 0 or
// alpha < 1/255, decided by the blend's own arithmetic): the state changes of
// its blend are then those of the clean blend.  Every other pixel is "active"
// and must be re-blended.

// Plan: the candidate tiles of a batch.  Lane = tile row of a pair (the
// injector's list): the columns that either record reaches in that row
// (band_tiles), then the warp's 32 rows' tiles are taken 32 at a time.  A tile is
// dropped when every pixel's clean blend stopped in front of both changed entries
// (tile_stop, exact) or when neither record can reach any of its 8x8 blocks
// (rect_reachable, conservative); the others become candidates with the blocks to
// look at.
// Issue-bound; the row step is what keeps it small: an exploded primitive's rect
// spans the frame, but its ellipse crosses a few columns of each row (20,000 upsets
// of a 2M-primitive scene, 4 views: 28.5M tiles by rects, 1.4M by rows; 0.16 ms,
// and 0.82 ms where needles kept their whole rows).
// counts[1] rows, [2] candidates, [3] their blocks to look at, [9] SSIM plan slots.
// BIN: also count the candidates of each tile (bins) and keep each one's place.
template <bool COUNT, bool BIN>
__global__ __launch_bounds__(256) void k_plan(const ViewPtrs* __restrict__ views, const DirtyDesc* __restrict__ desc,
                                              const uint2* __restrict__ rows, uint2* __restrict__ cand,
                                              uint32_t* __restrict__ cand_at, uint32_t* __restrict__ bins,
                                              unsigned int* __restrict__ counts, unsigned long long* work,
                                              SsimBufs sb) {
    // tiles that some pixel's clean blend reached behind the change, waiting for the
    // block tests: x = pair | 1 << 20 (corrupted record there) | 1 << 21 (clean record
    // there) | view << 24, y = tile x | tile y << 16
    __shared__ uint2 wait[256 / 32][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nrows = counts[1], nwarps = (gridDim.x * blockDim.x) >> 5;
    // rows a warp takes at a time: all lanes when there is enough work for every warp
    const uint32_t per = min(32u, (nrows + nwarps - 1u) / nwarps);
    unsigned int drop_key = 0, drop_box = 0;
    int nwait = 0;
    // the block tests of the first (at most 32) waiting tiles, one per lane
    auto test_blocks = [&](int n) {
        uint32_t blocks = 0u, bin = 0u, tile = 0u;
        const uint2 w = lane < n ? wait[warp][lane] : make_uint2(0u, 0u);
        if (lane < n) {
            const DirtyDesc& d = desc[w.x & kCandPair];
            const ViewPtrs& v = views[w.x >> 24];
            const bool has_new = (w.x >> 20) & 1u, has_old = (w.x >> 21) & 1u;
            const int tx = (int)(w.y & 0xffffu), ty = (int)(w.y >> 16);
            tile = (uint32_t)ty * (uint32_t)v.tiles_x + (uint32_t)tx;
            bin = v.bin0 + tile;
            const int lg = tile_lgx(v.tile_w), nb = (v.tile_w * v.tile_h) >> 6;
            for (int b = 0; b < nb; b++) {
                const int bx = tx * v.tile_w + block_x0(b, lg), by = ty * v.tile_h + block_y0(b, lg);
                const float x0 = (float)bx + 0.5f, x1 = fminf((float)(bx + 7), (float)(v.W - 1)) + 0.5f;
                const float y0 = (float)by + 0.5f, y1 = fminf((float)(by + 7), (float)(v.H - 1)) + 0.5f;
                if (bx >= v.W || by >= v.H) continue;
                const bool r = (has_new && rect_reachable(d.rec.mx, d.rec.my, d.rec.ca, d.rec.cb, d.rec.cc,
                                                          d.rec.opac, x0, x1, y0, y1)) ||
                               (has_old && rect_reachable(d.old.mx, d.old.my, d.old.ca, d.old.cb, d.old.cc,
                                                          d.old.opac, x0, x1, y0, y1));
                blocks |= r ? 1u << b : 0u;
            }
            if (COUNT && !blocks) drop_box++;
            if (COUNT && blocks) atomicAdd(&work[1], 1ull);
        }
        const unsigned m = __ballot_sync(0xffffffffu, blocks != 0u);
        if (!m) return;
        const unsigned nblk = __reduce_add_sync(0xffffffffu, (unsigned)__popc(blocks));
        uint32_t c0 = 0, s0 = 0;
        if (lane == 0) {   // both counts in one addition
            c0 = (uint32_t)atomicAdd(reinterpret_cast<unsigned long long*>(&counts[2]),
                                     (unsigned long long)__popc(m) | ((unsigned long long)nblk << 32));
            if (sb.plan) s0 = atomicAdd(&counts[9], (unsigned)__popc(m));
        }
        c0 = __shfl_sync(0xffffffffu, c0, 0) + __popc(m & ((1u << lane) - 1u));
        s0 = __shfl_sync(0xffffffffu, s0, 0) + __popc(m & ((1u << lane) - 1u));
        if (!blocks) return;
        const uint32_t bk = w.x & kCandPair;
        cand[c0] = make_uint2(bk | (blocks << 20) | (w.x & 0xff000000u), w.y);
        if (BIN) cand_at[c0] = atomicAdd(&bins[bin], 1u);
        if (sb.plan) {   // dirty-tile SSIM: tile -> slot of this batch, nothing re-blended yet
            if (s0 < sb.slot_cap) {
                const uint4 none = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
                uint4* sg = reinterpret_cast<uint4*>(sb.slot_group + (size_t)s0 * 8);
                sg[0] = none;
                sg[1] = none;
                uint4* item = reinterpret_cast<uint4*>(&sb.plan[s0]);
                item[0] = make_uint4(0u, 0u, 0u, 0u);
                item[1] = make_uint4(0u, 0u, 0u, 0u);
                item[2] = make_uint4(bk, tile, 0u, 0u);
                sb.slot_flags[s0] = 0u;
                sb.tile_map[(size_t)bk * sb.max_tiles + tile] = ((unsigned long long)counts[6] << 32) | s0;
            } else {
                atomicOr(sb.overflow, 1u);
            }
        }
    };
    for (uint32_t base = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per; base < nrows; base += nwarps * per) {
        const bool have = (uint32_t)lane < per && base + (uint32_t)lane < nrows;
        uint2 row = make_uint2(0u, 0u);
        int n0 = 0, n1 = 0, o0 = 0, o1 = 0;   // columns either record reaches
        if (have) {
            row = rows[base + (uint32_t)lane];
            const DirtyDesc& d = desc[row.x];
            const ViewPtrs& v = views[row.y >> 16];
            const int ty = (int)(row.y & 0xffffu), th = v.tile_h, tw = v.tile_w;
            const float y0 = (float)(ty * th) + 0.5f, y1 = fminf((float)(ty * th + th - 1), (float)(v.H - 1)) + 0.5f;
            const bool rn = ty >= d.ny0 && ty < d.ny1, ro = ty >= d.oy0 && ty < d.oy1;
            if (rn) band_tiles(d.rec, y0, y1, d.nx0, d.nx1, tw, n0, n1);
            if (ro) band_tiles(d.old, y0, y1, d.ox0, d.ox1, tw, o0, o1);
            if (COUNT)
                drop_box += (unsigned)(Union1(rn ? d.nx0 : 0, rn ? d.nx1 : 0, ro ? d.ox0 : 0, ro ? d.ox1 : 0).len -
                                       Union1(n0, n1, o0, o1).len);
        }
        const uint32_t cnt = (uint32_t)Union1(n0, n1, o0, o1).len;
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t excl = incl - cnt, total = __shfl_sync(0xffffffffu, incl, 31);
        for (uint32_t q0 = 0; q0 < total; q0 += 32) {
            const uint32_t q = q0 + (uint32_t)lane;
            int s = 0;   // the row this tile belongs to: the last lane whose offset is <= q
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int m = s + step;
                if (__shfl_sync(0xffffffffu, excl, m) <= q) s = m;
            }
            const int j = (int)(q - __shfl_sync(0xffffffffu, excl, s));
            const uint32_t bk = __shfl_sync(0xffffffffu, row.x, s), yv = __shfl_sync(0xffffffffu, row.y, s);
            const int a0 = __shfl_sync(0xffffffffu, n0, s), a1 = __shfl_sync(0xffffffffu, n1, s);
            const int b0 = __shfl_sync(0xffffffffu, o0, s), b1 = __shfl_sync(0xffffffffu, o1, s);
            bool keep = false;
            uint2 w = make_uint2(0u, 0u);
            if (q < total) {
                const int tx = Union1(a0, a1, b0, b1).at(j), ty = (int)(yv & 0xffffu);
                const DirtyDesc& d = desc[bk];
                const ViewPtrs& v = views[yv >> 16];
                const bool has_new = tx >= a0 && tx < a1, has_old = tx >= b0 && tx < b1;
                const uint32_t cut = min(has_new ? d.new_rank : kNoRank, has_old ? d.old_rank : kNoRank);
                keep = v.tile_stop[(uint32_t)ty * (uint32_t)v.tiles_x + (uint32_t)tx] >= cut;
                w = make_uint2(bk | (has_new ? 1u << 20 : 0u) | (has_old ? 1u << 21 : 0u) | ((yv >> 16) << 24),
                               (uint32_t)tx | ((uint32_t)ty << 16));
                if (COUNT && !keep) drop_key++;
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (keep) wait[warp][nwait + __popc(m & ((1u << lane) - 1u))] = w;
            nwait += __popc(m);
            __syncwarp();
            if (nwait >= 32) {
                test_blocks(32);
                __syncwarp();
                const uint2 rest = wait[warp][32 + lane];
                __syncwarp();
                wait[warp][lane] = rest;
                nwait -= 32;
                __syncwarp();
            }
        }
    }
    if (nwait) test_blocks(nwait);
    if (COUNT) {
        const unsigned k = __reduce_add_sync(0xffffffffu, drop_key), x = __reduce_add_sync(0xffffffffu, drop_box);
        if (lane == 0 && (k + x)) {
            atomicAdd(&work[3], (unsigned long long)(k + x));
            atomicAdd(&work[4], (unsigned long long)k);
            atomicAdd(&work[5], (unsigned long long)x);
        }
    }
}

// Candidates by tile, so that the warps that run side by side re-blend the same
// pixels for different variants and find their blend lists in the L2: the bins'
// starts (each block scans 1024 bins and draws its place from counts[4]; the
// order of the blocks does not matter) and the candidates' copy into them.
__global__ __launch_bounds__(1024) void k_bin_starts(uint32_t* __restrict__ bins, uint32_t nbins,
                                                    unsigned int* __restrict__ counts) {
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t start;
    const uint32_t i = blockIdx.x * 1024u + threadIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t c = i < nbins ? bins[i] : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t t = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        wsum[lane] = t;
        if (lane == 31) start = t ? atomicAdd(&counts[4], t) : 0u;
    }
    __syncthreads();
    if (i < nbins) bins[i] = start + x - c + (wid > 0 ? wsum[wid - 1] : 0u);
}

__global__ __launch_bounds__(256) void k_bin_cands(const ViewPtrs* __restrict__ views,
                                                   const uint2* __restrict__ cand, const uint32_t* __restrict__ cand_at,
                                                   const uint32_t* __restrict__ bins,
                                                   const unsigned int* __restrict__ counts, uint2* __restrict__ out) {
    const uint32_t n = counts[2];
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint2 c = cand[i];
        const ViewPtrs& v = views[c.x >> 24];
        const uint32_t tile = (c.y >> 16) * (uint32_t)v.tiles_x + (c.y & 0xffffu);
        out[bins[v.bin0 + tile] + cand_at[i]] = c;
    }
}

// One pixel's part of a unit's comparison, in words that add up without overflow
// over the 256 pixels of a tile: the fixed-point squared error (< 2^41) in a low
// part of 20 bits and a high one, the peak difference, and the footprint /
// non-finite / clean-non-finite counts 10 bits apart.
struct DirtySum {
    uint32_t fx_lo, fx_hi, maxbits, counts;
    bool foot;
};

__device__ __forceinline__ DirtySum dirty_sum(float v0, float v1, float v2, float k0, float k1, float k2) {
    const float c[3] = {k0, k1, k2};
    const PixCmp r = pixel_compare(v0, v1, v2, c);
    DirtySum s;
    s.fx_lo = (uint32_t)r.fx & 0xfffffu;
    s.fx_hi = (uint32_t)(r.fx >> 20);
    s.maxbits = __float_as_uint(r.m);   // r.m >= 0
    s.foot = r.foot;
    s.counts = (r.foot ? 1u : 0u) | (r.nonfin ? 1u << 10 : 0u) |
               (!(isfinite(k0) && isfinite(k1) && isfinite(k2)) ? 1u << 20 : 0u);
    return s;
}

// Two neighbouring entries of a blend list (32-byte aligned), one 256-bit load.
__device__ __forceinline__ void load_pair(const float4* p, float4& a, float4& b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

// The state of one dirty pixel's walk.
struct DirtyPix {
    float T, c0, c1, c2;
    // Takes an entry of capped alpha al; true when the walk ends there: the pixel
    // stops before it (T would drop below 1e-4), an end mark, or T became NaN, after
    // which every channel is NaN whatever follows (poison()).
    __device__ __forceinline__ bool take(float al, float r, float g, float b) {
        const float Tn = __fmul_rn(T, __fsub_rn(1.0f, al));
        if (!(Tn >= 1e-4f)) return true;
        const float w = __fmul_rn(al, T);
        c0 = __fmaf_rn(r, w, c0);
        c1 = __fmaf_rn(g, w, c1);
        c2 = __fmaf_rn(b, w, c2);
        T = Tn;
        return false;
    }
    __device__ __forceinline__ void poison(float al) {   // al: the alpha that ended the walk
        if (isnan(al)) T = c0 = c1 = c2 = NAN;
    }
};

// Dirty-tile blend.  A block of kDirtyWarps warps takes up to kUnitVars consecutive
// candidate tiles (in a large batch, mostly variants of a few tiles) in two steps.
//
// (1) Per candidate and 8x8 pixel block, by a warp: which pixels are active.  A
// pixel keeps its clean value, bit for bit, when its clean blend stopped in front of
// both changed entries, or when its blend skips the removed (clean) and the inserted
// (corrupted) record (power > 0 or alpha < 1/255, by the blend's own arithmetic):
// its state changes are then those of the clean blend.
//
// (2) The active (pixel, candidate) pairs, ordered by pixel, 32 at a time, one per
// lane: the pair resumes from the clean blend's state kept at or in front of the
// first change and walks the pixel's blend list from there -- without the removed
// entry and with the corrupted one at its place -- by the same operations in the
// same order as the full-frame blend, and compares the result with the clean pixel.
//
// Why by pixel: a lane's gather of its list costs one L1 lookup per load and list,
// and pairs of one pixel of one tile read the same lines.  With one variant's
// pixels over the lanes (32 lists per warp) the walk took 150 SM cycles per group of
// 8 entries whatever the occupancy.  Why 16 candidates: a tile of a 2M-primitive
// view holds three of a batch's, which would leave most of a block's warps idle.
// Bound by the gathers' latency and the longest walk of a unit: 42% of issue slots, 49%
// of the DRAM rate, 17 of a walk step's 32 lanes blending (1,024 upsets of 500,000
// primitives, four views).  20,000 upsets of a 2M-primitive scene in four 1600x1040 views:
// 40 warps of 48 registers per SM and 4 entries at a time 4.6 to 3.6 ms (the walk over
// block lists with every alpha evaluated took 6.0); drawn units took 8,192 of them from
// 1.56 to 1.38 ms.
constexpr int kDirtyWarps = 8;   // warps per block
constexpr int kDirtyThreads = kDirtyWarps * 32;
static_assert(kDirtyThreads >= kTilePix, "a thread per pixel of the tile");
struct __align__(16) DirtyVar {   // one candidate
    const uint32_t* row_idx;      // the tile's row to resume from
    const float* clean;           // the clean image's pixel at the tile's corner
    const float4* ent;            // blend lists, their ranks and states
    const uint32_t* rk;
    const float4* state;
    int W3;                       // floats per image row
    uint32_t bk, ins, pp;         // pair; ranks of the changed entries
    float r, g, b;                // the corrupted record's colour
    uint32_t cx, cy, tile;        // the candidate
    uint32_t fx_lo, fx_hi, maxbits, counts;   // sums over its pixels (see DirtySum)
    uint32_t cells_lo, cells_hi, edge, pad;
    uint32_t unit[kDirtyBlocks];              // SSIM: delta units of the blocks (0xffffffff: none)
    unsigned long long mask[kDirtyBlocks];    // active pixels of each 8x8 block
};

// DENSE: the candidates of dense views, which keep block lists: step (2) takes a
// candidate's 8x8 block per warp, two pixels per lane, and evaluates the block's list
// from the last row in front of the change, as the full-frame blend does, records
// streamed through two stages per warp.  Where nearly every entry of a block is taken
// at every pixel, 64 pixels then share a record of 48 B instead of reading 20 B of list
// each.  mixed: the views are of both kinds, each kernel skips the other's candidates.
template <bool COUNT, bool DENSE>
__global__ __launch_bounds__(kDirtyThreads, DENSE ? 4 : 5) void k_dirty(
    const ViewPtrs* __restrict__ views, const DirtyDesc* __restrict__ desc, const uint2* __restrict__ cand, int tw,
    int th, unsigned int* __restrict__ counts, uint32_t* __restrict__ bins, uint32_t nbins, CmpAcc* __restrict__ acc,
    bool regions, bool mixed, unsigned long long* work, SsimBufs sb) {
    __shared__ DirtyVar var[kUnitVars];
    __shared__ float alpha[kUnitVars][kTilePix];   // the corrupted entry's capped alpha at each pixel, -1: not taken
    __shared__ uint16_t pairs[DENSE ? 1 : kUnitVars * kTilePix];   // candidate << 8 | 8x8 block << 6 | pixel of the block
    __shared__ RawStageN<DENSE ? 32 : 1> stage[DENSE ? kDirtyWarps : 1][2];
    __shared__ uint32_t wsum[kDirtyWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lg = tile_lgx(tw), nb = (tw * th) >> 6;
    const uint32_t P = (uint32_t)(tw * th), ncand = counts[2];
    // Candidates of a unit, which blocks draw one after another.  A second unit costs its
    // set-up (6 us) again, so a block's share is one unit where the candidates are light.
    // Where most are reached in most of their blocks (the corrupted record covers them), a
    // unit may hold many times another's pixels: an eighth of a share, of at least one
    // candidate from 0.6 of the blocks on, two from 0.55.  300 upsets of 2M primitives, four
    // views (0.70, share 12): 202 us in shares, 124 in eighths; 3,000 of 134,826 (0.44,
    // share 10): 48 us in shares, 70 in eighths.
    const uint32_t share = (ncand + gridDim.x - 1u) / gridDim.x;
    const float covered = (float)counts[3] / ((float)max(ncand, 1u) * (float)nb);
    const uint32_t least = nb < 4 || covered < 0.55f ? (uint32_t)kUnitVars : (covered < 0.6f ? 2u : 1u);
    const uint32_t per = min((uint32_t)kUnitVars, share <= least + 1u ? share : max(least, (share + 7u) / 8u));
    __shared__ uint32_t next_unit;
    // the bins are free again: clear them for the next batch
    for (uint32_t i = blockIdx.x * kDirtyThreads + (uint32_t)tid; i < nbins; i += gridDim.x * kDirtyThreads) bins[i] = 0u;
    // measurement builds: SM cycles each warp spends per phase (the activity of the
    // candidates' pixels, the walk, the comparison and reductions)
    long long t_pro = 0, t_walk = 0, t_epi = 0;
    // units are drawn: the first by place, the next ones while this one is at work (none
    // where every unit has its block: the blocks' additions to one word take 2 us)
    const bool more = ncand > gridDim.x * per;
    for (uint32_t unit = blockIdx.x, drawn = ncand;; unit = next_unit) {
        const uint32_t c0 = unit * per;
        if (unit >= ncand || c0 >= ncand) break;   // the same for the whole block
        if (tid == 0 && more) drawn = gridDim.x + atomicAdd(&counts[DENSE ? 8 : 0], 1u);
        const long long t0 = COUNT ? clock64() : 0;
        const int nv = (int)min(per, ncand - c0);
        __syncthreads();   // the previous candidates are done with the shared arrays
        for (int task = warp; task < nv * nb; task += kDirtyWarps) {
            const int vi = task / nb, b = task % nb;
            const uint2 c = cand[c0 + (uint32_t)vi];
            const uint32_t bk = c.x & kCandPair;
            const int tx = (int)(c.y & 0xffffu), ty = (int)(c.y >> 16);
            const ViewPtrs& v = views[c.x >> 24];
            const uint32_t tile = (uint32_t)ty * (uint32_t)v.tiles_x + (uint32_t)tx;
            const DirtyDesc& d = desc[bk];
            const uint4 rects = *reinterpret_cast<const uint4*>(&d.nx0);   // corrupted x0 | y0 << 16, x1 | y1 << 16, clean
            auto in_rect = [&](uint32_t q0, uint32_t q1) {
                return tx >= (int)(q0 & 0xffffu) && tx < (int)(q1 & 0xffffu) && ty >= (int)(q0 >> 16) &&
                       ty < (int)(q1 >> 16);
            };
            const bool has_new = in_rect(rects.x, rects.y), has_old = in_rect(rects.z, rects.w);
            const uint32_t ins = has_new ? d.new_rank : kNoRank, pp = has_old ? d.old_rank : kNoRank;
            const uint32_t cut = min(ins, pp);
            unsigned mA = 0u, mB = 0u;
            if (((c.x >> (20 + b)) & 1u) && (!mixed || (v.sub != nullptr) == DENSE)) {
                const int wA = block_upper(b, lg), wB = wA + (1 << lg);
                // this lane's two pixels of the block: (lane % 8, lane / 8) and four rows below
                const uint32_t* stop = v.stop + (size_t)tile * P + lane;
                const uint32_t stA = stop[wA * 32], stB = stop[wB * 32];
                const int px = tx * tw + block_x0(b, lg) + (lane & 7), pyA = ty * th + block_y0(b, lg) + (lane >> 3);
                const float pxc = (float)px + 0.5f, pycA = (float)pyA + 0.5f;
                const float2 npy = make_float2(-pycA, -(pycA + 4.0f));
                bool okA = false, okB = false;
                if (has_old) {
                    const BlendRec& q = d.old;
                    alpha_pair(EntryQ{make_float4(q.mx, q.my, q.ca, q.cb), q.cc, q.opac, 0.0f, 0.0f, 0.0f}, pxc, npy,
                               okA, okB);
                }
                float aA = -1.0f, aB = -1.0f;
                if (has_new) {
                    const BlendRec& q = d.rec;
                    bool nA, nB;
                    const float2 a = alpha_pair(
                        EntryQ{make_float4(q.mx, q.my, q.ca, q.cb), q.cc, q.opac, 0.0f, 0.0f, 0.0f}, pxc, npy, nA, nB);
                    aA = nA ? (a.x > 0.99f ? 0.99f : a.x) : -1.0f;   // keeps NaN
                    aB = nB ? (a.y > 0.99f ? 0.99f : a.y) : -1.0f;
                    okA |= nA;
                    okB |= nB;
                }
                alpha[vi][b * 64 + lane] = aA;
                alpha[vi][b * 64 + 32 + lane] = aB;
                okA = okA && px < v.W && pyA < v.H;
                okB = okB && px < v.W && pyA + 4 < v.H;
                mA = __ballot_sync(0xffffffffu, okA && stA >= cut);
                mB = __ballot_sync(0xffffffffu, okB && stB >= cut);
                if (COUNT) {
                    const bool any = __any_sync(0xffffffffu, okA || okB);
                    if (lane == 0 && (mA | mB)) atomicAdd(&work[10], 1ull);
                    if (lane == 0 && !(mA | mB)) {
                        atomicAdd(&work[3], 1ull);
                        atomicAdd(&work[any ? 7 : 6], 1ull);
                    }
                }
            }
            if (lane == 0) var[vi].mask[b] = (unsigned long long)mA | ((unsigned long long)mB << 32);
            if (b == 0) {
                uint32_t row = 0u;
                if (!DENSE && (!mixed || v.sub == nullptr)) {   // the rows in front of the first change (the keys ascend)
                    const uint32_t* key = v.row_key + (size_t)tile * kRowsPerTile + lane;
                    const uint32_t key0 = key[0], key1 = key[32];
                    row = v.row_off[tile] + (uint32_t)(__popc(__ballot_sync(0xffffffffu, key0 < cut)) +
                                                       __popc(__ballot_sync(0xffffffffu, key1 < cut)));
                }
                if (lane == 0) {
                    DirtyVar& q = var[vi];
                    q.row_idx = v.row_idx + (size_t)row * P;
                    q.W3 = 3 * v.W;
                    q.clean = v.clean + ((size_t)(ty * th) * v.W + tx * tw) * 3;
                    q.ent = v.ent;
                    q.rk = v.rk;
                    q.state = v.state;
                    q.bk = bk;
                    q.ins = ins;
                    q.pp = pp;
                    q.r = d.rec.r;
                    q.g = d.rec.g;
                    q.b = d.rec.b;
                    q.cx = c.x;
                    q.cy = c.y;
                    q.tile = tile;
                    q.fx_lo = q.fx_hi = q.maxbits = q.counts = 0u;
                    q.cells_lo = q.cells_hi = q.edge = 0u;
                }
            }
        }
        __syncthreads();
        if (sb.plan && warp < (kUnitVars * kDirtyBlocks) / 32) {   // dirty-tile SSIM: two 32-pixel delta units per block
            const int vi = tid / nb, b = tid % nb;
            const unsigned long long mask = vi < nv ? var[vi].mask[b] : 0ull;
            const unsigned am = __ballot_sync(0xffffffffu, mask != 0ull);
            uint32_t unit = 0;
            if (lane == 0 && am) unit = atomicAdd(&counts[5], (unsigned)__popc(am));
            unit = __shfl_sync(0xffffffffu, unit, 0) + (uint32_t)__popc(am & ((1u << lane) - 1u));
            if (mask) {
                const unsigned long long e = sb.tile_map[(size_t)var[vi].bk * sb.max_tiles + var[vi].tile];
                const uint32_t slot = (uint32_t)e;
                const int wA = block_upper(b, lg), wB = wA + (1 << lg);
                if ((uint32_t)(e >> 32) == counts[6] && 2u * unit + 1u < sb.delta_cap) {
                    sb.plan[slot].mask[wA] = (uint32_t)mask;
                    sb.plan[slot].mask[wB] = (uint32_t)(mask >> 32);
                    sb.slot_group[(size_t)slot * 8 + wA] = 2u * unit;
                    sb.slot_group[(size_t)slot * 8 + wB] = 2u * unit + 1u;
                    var[vi].unit[b] = unit;
                } else {
                    var[vi].unit[b] = 0xffffffffu;
                    atomicOr(sb.overflow, 1u);
                }
            }
        }
        unsigned int nev = 0, nst = 0;
        if (DENSE) {
            __syncthreads();   // the delta units, where there are any
            if (COUNT) t_pro += clock64() - t0;
            for (int task = warp; task < nv * nb; task += kDirtyWarps) {
                const int vi = task / nb, b = task % nb;
                DirtyVar& q = var[vi];
                const unsigned long long mask = q.mask[b];
                if (!mask) continue;
                const long long t1 = COUNT ? clock64() : 0;
                const ViewPtrs& v = views[q.cx >> 24];
                const Pix2Geo g = pix2_geo((int)(q.cy & 0xffffu), (int)(q.cy >> 16), tw, th, v.W, v.H, b);
                const bool actA = (mask >> lane) & 1ull, actB = (mask >> (32 + lane)) & 1ull;
                const uint32_t ins = q.ins, pp = q.pp, cut = min(ins, pp);
                // the block's list, and how many of its entries lie in front of the first change
                const uint32_t tb = q.tile * (uint32_t)nb + (uint32_t)b, n = v.sub_cnt[tb], off = v.sub_off[tb];
                const uint2* __restrict__ sub = v.sub + off;
                uint32_t lo = 0, hi = n;
                while (lo < hi) {
                    const uint32_t step = (hi - lo + 31u) / 32u, i = lo + (uint32_t)lane * step;
                    const int k = __popc(__ballot_sync(0xffffffffu, i < hi && sub[i].y < cut));   // they come first
                    hi = k == 0 ? lo : min(hi, lo + (uint32_t)k * step);
                    lo = k == 0 ? lo : lo + (uint32_t)(k - 1) * step + 1u;
                }
                const uint32_t row = lo / (uint32_t)kRowStride;   // resume from this row
                const float4* rs = v.row_state + (block_rows(off, tb) + row) * 64 + lane;
                const float4 sA = rs[0], sB = rs[32];
                Pix pA{sA.x, sA.y, sA.z, sA.w, !actA}, pB{sB.x, sB.y, sB.z, sB.w, !actB};
                const float naA = alpha[vi][b * 64 + lane], naB = alpha[vi][b * 64 + 32 + lane];
                bool pend = ins != kNoRank;   // the corrupted entry is still to be inserted
                auto insert = [&] {
                    pend = false;
                    apply_entry(pA, !pA.done, !(naA < 0.0f), naA, q.r, q.g, q.b);
                    apply_entry(pB, !pB.done, !(naB < 0.0f), naB, q.r, q.g, q.b);
                };
                auto apply = [&](int, bool has, bool okA, bool okB, float2 a, float cr, float cg, float cb) {
                    const bool liveA = has && !pA.done, liveB = has && !pB.done;
                    if (COUNT) nev += (liveA && okA ? 1u : 0u) + (liveB && okB ? 1u : 0u);
                    apply_entry(pA, liveA, okA, a.x, cr, cg, cb);
                    apply_entry(pB, liveB, okB, a.y, cr, cg, cb);
                };
                auto fetch = [&](int k, uint32_t id) {
                    const float4* src = reinterpret_cast<const float4*>(v.recs + id);
                    cp_async16(&stage[warp][k].q0[lane], src);
                    cp_async16(&stage[warp][k].q1[lane], src + 1);
                    cp_async16(&stage[warp][k].q2[lane], src + 2);
                };
                const uint2 none = make_uint2(0u, 0xffffffffu);   // behind the list's end: of the last rank
                uint32_t i = row * (uint32_t)kRowStride + (uint32_t)lane;   // this lane's entries: i, i + 32, ...
                uint2 cur = i < n ? sub[i] : none;
                if (i < n) fetch(0, cur.x);
                uint2 next = i + 32u < n ? sub[i + 32u] : none;
                for (uint32_t base = row * (uint32_t)kRowStride, k = 0; base < n; base += 32u, k ^= 1u) {
                    cp_async_wait_all();
                    __syncwarp();   // the entries are there for every lane, and every lane is done with the other stage
                    const uint32_t rank = cur.y;
                    if (i + 32u < n) fetch((int)k ^ 1, next.x);
                    cur = next;
                    next = i + 64u < n ? sub[i + 64u] : none;
                    i += 32u;
                    if (COUNT) nst++;
                    const uint32_t left = n - base;
                    unsigned m = (left >= 32u ? 0xffffffffu : (1u << left) - 1u) & ~__ballot_sync(0xffffffffu, rank == pp);
                    if (pend) {
                        const unsigned behind = __ballot_sync(0xffffffffu, rank >= ins);   // (past the list's end too)
                        if (behind) {
                            walk_raw2(m & ~behind, stage[warp][k], 0, g, apply, [] {});
                            insert();
                            m &= behind;
                        }
                    }
                    walk_raw2(m, stage[warp][k], 0, g, apply, [] {});
                    if (__all_sync(0xffffffffu, pA.done && pB.done)) break;
                }
                cp_async_wait_all();   // leave no copy in flight
                __syncwarp();
                if (pend) insert();   // (pixels that have stopped take no more)
                const long long t2 = COUNT ? clock64() : 0;
                DirtySum s{};
                uint32_t maxb = 0u;
                auto finish = [&](const Pix& p, bool act, int py, int half) {
                    if (!act) return;
                    const int lx = g.px - (int)(q.cy & 0xffffu) * tw, ly = py - (int)(q.cy >> 16) * th;   // in the tile
                    const float* kp = q.clean + (ly * q.W3 + lx * 3);
                    const float k0 = kp[0], k1 = kp[1], k2 = kp[2];
                    const float a0 = __fadd_rn(p.c0, p.T), a1 = __fadd_rn(p.c1, p.T), a2 = __fadd_rn(p.c2, p.T);
                    const DirtySum d = dirty_sum(a0, a1, a2, k0, k1, k2);
                    s.fx_lo += d.fx_lo;
                    s.fx_hi += d.fx_hi;
                    s.counts += d.counts;
                    maxb = max(maxb, d.maxbits);
                    if (regions && d.foot) {
                        const unsigned long long cell = cell_bit(g.px, py, v.W, v.H);
                        if ((unsigned)cell) atomicOr(&q.cells_lo, (unsigned)cell);
                        if ((unsigned)(cell >> 32)) atomicOr(&q.cells_hi, (unsigned)(cell >> 32));
                    }
                    if (sb.plan && q.unit[b] != 0xffffffffu) {
                        sb.deltas[(size_t)(2u * q.unit[b] + (uint32_t)half) * 32 + lane] = make_float4(a0, a1, a2, 0.0f);
                        const bool ch = __float_as_uint(a0) != __float_as_uint(k0) ||
                                        __float_as_uint(a1) != __float_as_uint(k1) || __float_as_uint(a2) != __float_as_uint(k2);
                        if (ch)
                            atomicOr(&q.edge, 16u | (lx < 5 ? 1u : 0u) | (lx > tw - 6 ? 2u : 0u) | (ly < 5 ? 4u : 0u) |
                                                  (ly > th - 6 ? 8u : 0u));
                    }
                };
                finish(pA, actA, g.pyA, 0);
                finish(pB, actB, g.pyB, 1);
                s.fx_lo = __reduce_add_sync(0xffffffffu, s.fx_lo);   // 64 pixels: below 2^26 and 2^27, counts below 2^7 a field
                s.fx_hi = __reduce_add_sync(0xffffffffu, s.fx_hi);
                s.counts = __reduce_add_sync(0xffffffffu, s.counts);
                maxb = __reduce_max_sync(0xffffffffu, maxb);
                if (lane == 0) {
                    if (s.fx_lo) atomicAdd(&q.fx_lo, s.fx_lo);
                    if (s.fx_hi) atomicAdd(&q.fx_hi, s.fx_hi);
                    if (s.counts) atomicAdd(&q.counts, s.counts);
                    if (maxb) atomicMax(&q.maxbits, maxb);
                }
                if (COUNT) {
                    t_walk += t2 - t1;
                    t_epi += clock64() - t2;
                    if (lane == 0) {
                        const unsigned npix = (unsigned)__popcll(mask);
                        atomicAdd(&work[8], (unsigned long long)nst * 32ull);
                        atomicAdd(&work[9], (unsigned long long)nst * 32ull);
                        atomicAdd(&work[14], (unsigned long long)npix);
                        atomicAdd(&work[15], (unsigned long long)nst * 32ull * npix);
                    }
                    nst = 0;
                }
            }
        }
        if (!DENSE) {
            // the pairs by pixel: thread t lists the candidates of pixel t
            uint32_t m = 0u;
            if (tid < nb * 64)
                for (int vi = 0; vi < nv; vi++) m |= ((unsigned)(var[vi].mask[tid >> 6] >> (tid & 63)) & 1u) << vi;
            const uint32_t cnt = (uint32_t)__popc(m);
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            uint32_t at = incl - cnt, npairs = 0;
#pragma unroll
            for (int w = 0; w < kDirtyWarps; w++) {
                at += w < warp ? wsum[w] : 0u;
                npairs += wsum[w];
            }
            for (; m; m &= m - 1u) pairs[at++] = (uint16_t)((__ffs(m) - 1) << 8 | tid);
            __syncthreads();
            if (COUNT) t_pro += clock64() - t0;
            for (uint32_t r0 = (uint32_t)warp * 32u; r0 < npairs; r0 += kDirtyThreads) {
                const long long t1 = COUNT ? clock64() : 0;
                const bool act = r0 + (uint32_t)lane < npairs;
                const int code = pairs[act ? r0 + (uint32_t)lane : r0];
                const int vi = code >> 8, u8 = code & 255, b = u8 >> 6, u6 = u8 & 63;
                DirtyVar& q = var[vi];
                const int lx = block_x0(b, lg) + (u6 & 7), ly = block_y0(b, lg) + (u6 >> 3);   // in the tile
                const int u = (block_upper(b, lg) + ((u6 >> 5) << lg)) * 32 + (u6 & 31);
                DirtyPix p{1.0f, 0.0f, 0.0f, 0.0f};
                float k0 = 0.0f, k1 = 0.0f, k2 = 0.0f;   // the clean pixel
                if (act) {
                    const float4* ent = q.ent;
                    uint32_t i = q.row_idx[u] & ~(uint32_t)(kWalk - 1);
                    const float* kp = q.clean + (ly * q.W3 + lx * 3);
                    k0 = kp[0];
                    k1 = kp[1];
                    k2 = kp[2];
                    const float4 st = q.state[i / kWalk];
                    p.T = st.x;
                    p.c0 = st.y;
                    p.c1 = st.z;
                    p.c2 = st.w;
                    const uint32_t ins = q.ins, pp = q.pp;
                    const float na = alpha[vi][u8];   // the corrupted entry at this pixel, when its blend takes it
                    bool pend = !(na < 0.0f);         // still to be inserted (a NaN alpha too)
                    bool old = pp != kNoRank;         // the removed entry may still lie ahead
                    float4 e[kWalk];
                    float last = 0.0f;                // the alpha that ended the walk
                    bool end = false;
                    do {
#pragma unroll
                        for (int k = 0; k < kWalk; k += 2) load_pair(ent + i + k, e[k], e[k + 1]);
                        if (COUNT) nst++;
                        if (pend || old) {   // ranks matter until both changes are behind
                            // the first entry of this group behind the corrupted one (the end's rank is
                            // above every other) and the removed entry
                            const uint4 x = __ldg(reinterpret_cast<const uint4*>(q.rk + i));
                            const int first = x.x >= ins ? 0 : (x.y >= ins ? 1 : (x.z >= ins ? 2 : (x.w >= ins ? 3 : 4)));
                            const int at_new = pend ? first : kWalk;
                            const int at_old = x.x == pp ? 0 : (x.y == pp ? 1 : (x.z == pp ? 2 : (x.w == pp ? 3 : kWalk)));
#pragma unroll
                            for (int k = 0; k < kWalk; k++) {
                                if (k == at_new && !end) {
                                    pend = false;
                                    if (COUNT) nev++;
                                    last = na;
                                    end = p.take(na, q.r, q.g, q.b);
                                }
                                if (!end && k != at_old) {
                                    if (COUNT) nev++;
                                    last = e[k].x;
                                    end = p.take(e[k].x, e[k].y, e[k].z, e[k].w);
                                }
                            }
                            old = old && x.w < pp;
                        } else {
#pragma unroll
                            for (int k = 0; k < kWalk; k++) {
                                if (end) continue;
                                if (COUNT) nev++;
                                last = e[k].x;
                                end = p.take(e[k].x, e[k].y, e[k].z, e[k].w);
                            }
                        }
                        i += kWalk;
                    } while (!end);
                    p.poison(last);
                }
                __syncwarp();
                const long long t2 = COUNT ? clock64() : 0;
                // compare with the clean image; every inactive pixel keeps its clean value
                // (Delta = 0), and the clean image's non-finite pixels are counted once per
                // view at finalize
                const float a0 = __fadd_rn(p.c0, p.T), a1 = __fadd_rn(p.c1, p.T), a2 = __fadd_rn(p.c2, p.T);
                DirtySum s{};
                if (act) s = dirty_sum(a0, a1, a2, k0, k1, k2);
                const bool one = nv == 1;   // block-uniform
                if (one) {
                    s.fx_lo = __reduce_add_sync(0xffffffffu, s.fx_lo);
                    s.fx_hi = __reduce_add_sync(0xffffffffu, s.fx_hi);
                    s.counts = __reduce_add_sync(0xffffffffu, s.counts);
                    s.maxbits = __reduce_max_sync(0xffffffffu, s.maxbits);
                }
                if (one ? lane == 0 : act) {
                    if (s.fx_lo) atomicAdd(&q.fx_lo, s.fx_lo);
                    if (s.fx_hi) atomicAdd(&q.fx_hi, s.fx_hi);
                    if (s.counts) atomicAdd(&q.counts, s.counts);
                    if (s.maxbits) atomicMax(&q.maxbits, s.maxbits);
                }
                if (regions && act && s.foot) {   // screen cells holding a footprint pixel
                    const ViewPtrs& v = views[q.cx >> 24];
                    const unsigned long long cell = cell_bit((int)(q.cy & 0xffffu) * tw + lx, (int)(q.cy >> 16) * th + ly, v.W, v.H);
                    if ((unsigned)cell) atomicOr(&q.cells_lo, (unsigned)cell);
                    if ((unsigned)(cell >> 32)) atomicOr(&q.cells_hi, (unsigned)(cell >> 32));
                }
                if (sb.plan && act && q.unit[b] != 0xffffffffu) {   // dirty-tile SSIM: the new values
                    sb.deltas[(size_t)(2u * q.unit[b] + (uint32_t)(u6 >> 5)) * 32 + (u6 & 31)] = make_float4(a0, a1, a2, 0.0f);
                    // where the changed pixels are: which neighbouring tiles their SSIM windows reach
                    const bool ch = __float_as_uint(a0) != __float_as_uint(k0) || __float_as_uint(a1) != __float_as_uint(k1) ||
                                    __float_as_uint(a2) != __float_as_uint(k2);
                    if (ch)
                        atomicOr(&q.edge, 16u | (lx < 5 ? 1u : 0u) | (lx > tw - 6 ? 2u : 0u) | (ly < 5 ? 4u : 0u) |
                                              (ly > th - 6 ? 8u : 0u));
                }
                if (COUNT) {
                    const unsigned steps = __reduce_max_sync(0xffffffffu, nst);
                    nst = 0;
                    t_walk += t2 - t1;
                    t_epi += clock64() - t2;
                    if (lane == 0) {
                        const unsigned npix = min(32u, npairs - r0);
                        atomicAdd(&work[8], (unsigned long long)(steps * kWalk));
                        atomicAdd(&work[9], (unsigned long long)(steps * kWalk));
                        atomicAdd(&work[14], (unsigned long long)npix);
                        atomicAdd(&work[15], (unsigned long long)steps * kWalk * npix);
                    }
                }
            }
        }
        if (tid == 0) next_unit = drawn;
        __syncthreads();
        if (tid < nv) {
            const DirtyVar& q = var[tid];
            CmpAcc* A = &acc[q.bk];
            const unsigned long long fx = (unsigned long long)q.fx_lo + ((unsigned long long)q.fx_hi << 20);
            const unsigned long long cells = (unsigned long long)q.cells_lo | ((unsigned long long)q.cells_hi << 32);
            const unsigned foot = q.counts & 1023u, bad = (q.counts >> 10) & 1023u, clean_bad = q.counts >> 20;
            if (cells) atomicOr(&A->reg_actual, cells);
            if (fx) atomicAdd(&A->sse_fx, fx);
            if (q.maxbits) atomicMax(&A->maxabs_bits, q.maxbits);
            if (foot) atomicAdd(&A->footprint, foot);
            if (bad) atomicAdd(&A->nonfinite, bad);
            if (clean_bad) atomicAdd(&A->clean_nonfinite_replaced, clean_bad);
            if (q.edge)   // set only where the tile has a slot
                atomicOr(&sb.slot_flags[(uint32_t)sb.tile_map[(size_t)q.bk * sb.max_tiles + q.tile]], q.edge);
        }
        if (COUNT) {
            const unsigned wn = __reduce_add_sync(0xffffffffu, nev);
            if (lane == 0 && wn) {
                atomicAdd(&work[0], (unsigned long long)wn);
                atomicAdd(&work[2], (unsigned long long)wn);
            }
        }
    }
    if (COUNT && lane == 0) {
        atomicAdd(&work[11], (unsigned long long)t_pro);
        atomicAdd(&work[12], (unsigned long long)t_walk);
        atomicAdd(&work[13], (unsigned long long)t_epi);
    }
}

__global__ void k_records_to_blend(const gs_record* in, uint64_t n, BlendRec* out) {
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    gs_record r = in[i];
    BlendRec q;
    q.mx = r.mx;
    q.my = r.my;
    q.ca = r.ca;
    q.cb = r.cb;
    q.cc = r.cc;
    q.opac = r.opac;
    q.r = r.r;
    q.g = r.g;
    q.b = r.b;
    q.depth = r.depth;
    // records from outside carry no alpha box: never cull
    q.ex = NAN;
    q.ey = NAN;
    out[i] = q;
}

__global__ void k_offsets_to_ranges(const uint32_t* offsets, int ntiles, uint2* ranges) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ntiles) ranges[t] = make_uint2(offsets[t], offsets[t + 1]);
}

}  // namespace

gs_status launch_blend_image(const BlendRec* recs, const uint32_t* ids, const uint2* ranges, const DevCamera& cam,
                             float* img, cudaStream_t st) {
    const int tx = cam.tiles_x, ty = cam.tiles_y, P = cam.tile_w * cam.tile_h / 2;   // threads: two pixels each
    if (tx * ty == 0) return GS_OK;
    k_blend_full<0, false><<<tx * ty, P, 0, st>>>(recs, ids, ranges, cam.W, cam.H, tx, cam.tile_w, cam.tile_h, img,
                                                   nullptr, nullptr, nullptr);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_blend_compare(const BlendRec* recs, const uint32_t* ids, const uint2* ranges, const DevCamera& cam,
                               const float* clean, CmpAcc* acc, unsigned long long* work, cudaStream_t st) {
    const int tx = cam.tiles_x, ty = cam.tiles_y, P = cam.tile_w * cam.tile_h / 2;   // threads: two pixels each
    if (tx * ty == 0) return GS_OK;
    if (work)
        k_blend_full<1, true><<<tx * ty, P, 0, st>>>(recs, ids, ranges, cam.W, cam.H, tx, cam.tile_w, cam.tile_h,
                                                     nullptr, clean, acc, work);
    else
        k_blend_full<1, false><<<tx * ty, P, 0, st>>>(recs, ids, ranges, cam.W, cam.H, tx, cam.tile_w, cam.tile_h,
                                                      nullptr, clean, acc, nullptr);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

// First pass over a clean view: image, stops, list lengths.
gs_status launch_blend_clean(const ViewState& v, uint32_t* counts, uint32_t* blk_cnt, unsigned int* clean_nonfin,
                             cudaStream_t st) {
    const DevCamera& cam = v.cam;
    const int tx = cam.tiles_x, ty = cam.tiles_y, P = cam.tile_w * cam.tile_h / 2;
    if (tx * ty == 0) return GS_OK;
    k_blend_clean<kImage><<<tx * ty, P, 0, st>>>(v.recs, v.ids, v.rank, v.ranges, cam.W, cam.H, tx, cam.tile_w,
                                                 cam.tile_h, v.clean, v.stop, v.tile_stop, v.tile_last, counts,
                                                 blk_cnt, clean_nonfin, ListOut{});
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

// Second pass: blend lists (off: their starts), or, of a dense view, block lists.
gs_status launch_fill_lists(const ViewState& v, const uint32_t* off, cudaStream_t st) {
    const DevCamera& cam = v.cam;
    const int tx = cam.tiles_x, ty = cam.tiles_y, P = cam.tile_w * cam.tile_h / 2;
    if (tx * ty == 0) return GS_OK;
    const bool dense = v.sub != nullptr;
    const int smem = dense ? 0 : (int)sizeof(ListRing) * (P / 32);
    // the largest tile's, not this one's: the attribute is the process's, and another
    // thread may fill lists of another tile shape between these lines
    constexpr int most = (int)sizeof(ListRing) * (kBT / 2 / 32);
    GS_CUDA(cudaFuncSetAttribute(k_blend_clean<kLists>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    auto fill = dense ? k_blend_clean<kBlocks> : k_blend_clean<kLists>;
    fill<<<tx * ty, P, smem, st>>>(v.recs, v.ids, v.rank, v.ranges, cam.W, cam.H, tx, cam.tile_w, cam.tile_h, nullptr,
                                   nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                                   ListOut{v.ent, v.rk, off, v.state, v.row_idx, v.row_off, v.row_cnt, v.sub, v.sub_off,
                                           v.row_state});
    if (!dense)
        k_row_keys<<<(tx * ty * kRowsPerTile + 255) / 256, 256, 0, st>>>(v.ranges, v.ids, v.rank, v.row_cnt, tx * ty,
                                                                           v.row_key);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_ranks(const uint32_t* key, const uint32_t* id, uint64_t n, const ViewState& v, cudaStream_t st) {
    if (n > 0) k_ranks<<<(unsigned)div_up(n, 256), 256, 0, st>>>(key, id, n, v.rank, v.sdk, v.sid);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_row_counts(const ViewState& v, uint32_t* rows, cudaStream_t st) {
    const int ntiles = v.cam.tiles_x * v.cam.tiles_y;
    if (ntiles > 0) k_row_counts<<<(ntiles + 255) / 256, 256, 0, st>>>(v.ranges, v.tile_last, ntiles, v.row_cnt, rows);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_list_lens(const uint32_t* counts, uint64_t n, uint32_t* lens, cudaStream_t st) {
    if (n > 0) k_list_lens<<<(unsigned)div_up(n, 256), 256, 0, st>>>(counts, n, lens);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_compare(const float* a, const float* b, int H, int W, int K, CmpAcc* acc, cudaStream_t st) {
    const uint64_t pix = (uint64_t)W * H;
    // enough blocks for one resident wave, at least four pixels a thread
    const uint64_t want = std::max<uint64_t>(1, (uint64_t)num_sms() * 8 / (uint64_t)std::min(K, 65535));
    const unsigned bx = (unsigned)std::min<uint64_t>(div_up(pix, 4 * kBT), want);
    for (int k = 0; k < K; k += 65535)
        k_compare<<<dim3(bx, std::min(K - k, 65535)), kBT, 0, st>>>(a + k * pix * 3, b + k * pix * 3, pix, acc + k);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_zero_acc(CmpAcc* acc, int count, cudaStream_t st) {
    if (count <= 0) return GS_OK;
    k_zero_acc<<<(count + 255) / 256, 256, 0, st>>>(acc, count);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_finalize(const CmpAcc* acc, int count, gs_result* out, cudaStream_t st) {
    if (count <= 0) return GS_OK;
    k_finalize<<<(count + 255) / 256, 256, 0, st>>>(acc, count, out, nullptr, 1, nullptr);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

__global__ void k_regions_out(const CmpAcc* acc, int count, unsigned long long* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    out[2 * i] = acc[i].reg_actual;
    out[2 * i + 1] = acc[i].reg_pred;
}

gs_status launch_regions_out(const CmpAcc* acc, int count, unsigned long long* out, cudaStream_t st) {
    if (count > 0) k_regions_out<<<(count + 255) / 256, 256, 0, st>>>(acc, count, out);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_finalize_dirty(const CmpAcc* acc, int count, gs_result* out, const unsigned int* clean_nonfin, int K,
                                unsigned int* queue, cudaStream_t st) {
    if (count <= 0) return GS_OK;
    k_finalize<<<(count + 255) / 256, 256, 0, st>>>(acc, count, out, clean_nonfin, K, queue);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

template <bool DENSE>
static int resident_blocks() {
    static const int blocks = [] {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dirty<false, DENSE>, kDirtyThreads, 0);
        return std::max(per_sm, 1) * num_sms();
    }();
    return blocks;
}
// the occupancy queries, outside any stream capture
void dirty_grids() {
    resident_blocks<false>();
    resident_blocks<true>();
}

gs_status launch_dirty_ssim(const void* dev_views, int K, unsigned int* queue, const SsimBufs& sb, CmpAcc* acc,
                            cudaStream_t st);

// Candidates are put in tile order from this many (variant, view) pairs on: with
// fewer, hardly two variants meet in a tile, and the two launches cost 10 us (1,024
// pairs of a 300k-primitive scene: 1.14 ms in order, 1.18 ms as planned; 200 pairs
// of a 5k-primitive one: no difference).
constexpr int kSortPairs = 512;

// One batch after the injector.  ev_mid (optional): recorded between the plan and
// the blend kernel.  s->queue, cleared by the finaliser but for [6]: [0] units drawn (of
// dense views: [8]), [1] tile rows, [2] candidates and [3] their blocks to look at, [4]
// bin places, [5] SSIM delta units, [6] batch generation, [7] tiles the SSIM visits, [9]
// SSIM plan slots.
gs_status launch_dirty_blend(gs_scene* s, int BK, bool regions, const SsimBufs& sb, cudaStream_t st) {
    const ViewPtrs* views = (const ViewPtrs*)s->dev_views;
    const int plan_blocks = num_sms() * 8;
    const uint32_t nbins = s->all_tiles;
    const bool bin = BK >= kSortPairs;
    unsigned long long* work = s->work_ctr;
    auto plan = work ? (bin ? k_plan<true, true> : k_plan<true, false>) : (bin ? k_plan<false, true> : k_plan<false, false>);
    plan<<<plan_blocks, 256, 0, st>>>(views, s->desc, s->rows, s->cand, s->cand_at, s->bins, s->queue, work, sb);
    if (bin) {
        k_bin_starts<<<(nbins + 1023) / 1024, 1024, 0, st>>>(s->bins, nbins, s->queue);
        k_bin_cands<<<plan_blocks, 256, 0, st>>>(views, s->cand, s->cand_at, s->bins, s->queue, s->cand_sorted);
    }
    if (s->ev_kp) {
        cudaError_t e = cudaEventRecordWithFlags(s->ev_kp, st, cudaEventRecordExternal);
        if (e != cudaSuccess) return set_error(GS_ERR_CUDA, cudaGetErrorString(e));
    }
    const int dense_views = (int)std::count_if(s->views.begin(), s->views.end(), [](const ViewState& v) { return v.sub != nullptr; });
    const bool mixed = dense_views > 0 && dense_views < s->K;
    auto dirty = [&](auto kernel, int blocks) {
        kernel<<<blocks, kDirtyThreads, 0, st>>>(views, s->desc, bin ? s->cand_sorted : s->cand, s->tile_w, s->tile_h,
                                                 s->queue, s->bins, bin ? nbins : 0u, s->acc, regions, mixed, work, sb);
    };
    if (dense_views < s->K) dirty(work ? k_dirty<true, false> : k_dirty<false, false>, resident_blocks<false>());
    if (dense_views > 0) dirty(work ? k_dirty<true, true> : k_dirty<false, true>, resident_blocks<true>());
    if (sb.plan) GS_TRY(launch_dirty_ssim(s->dev_views, s->K, s->queue, sb, s->acc, st));
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

size_t view_ptrs_size() { return sizeof(ViewPtrs); }

void fill_view_ptrs(void* host_dst, const ViewState& vs, uint32_t bin0) {
    ViewPtrs v{};
    v.recs = vs.recs;
    v.ids = vs.ids;
    v.rank = vs.rank;
    v.sdk = vs.sdk;
    v.sid = vs.sid;
    v.rects = vs.rects;
    v.ranges = vs.ranges;
    v.clean = vs.clean;
    v.stop = vs.stop;
    v.tile_stop = vs.tile_stop;
    v.row_idx = vs.row_idx;
    v.row_off = vs.row_off;
    v.row_key = vs.row_key;
    v.ent = vs.ent;
    v.rk = vs.rk;
    v.state = vs.state;
    v.sub = vs.sub;
    v.sub_off = vs.sub_off;
    v.sub_cnt = vs.sub_cnt;
    v.row_state = vs.row_state;
    v.W = vs.cam.W;
    v.H = vs.cam.H;
    v.tiles_x = vs.cam.tiles_x;
    v.tile_w = vs.cam.tile_w;
    v.tile_h = vs.cam.tile_h;
    v.bin0 = bin0;
    memcpy(host_dst, &v, sizeof(v));
}

gs_status launch_records_to_blend(const gs_record* in, uint64_t n, BlendRec* out, cudaStream_t st) {
    if (n == 0) return GS_OK;
    k_records_to_blend<<<(unsigned)div_up(n, 256), 256, 0, st>>>(in, n, out);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

gs_status launch_offsets_to_ranges(const uint32_t* offsets, int ntiles, uint2* ranges, cudaStream_t st) {
    if (ntiles <= 0) return GS_OK;
    k_offsets_to_ranges<<<(ntiles + 255) / 256, 256, 0, st>>>(offsets, ntiles, ranges);
    GS_CUDA(cudaGetLastError());
    return GS_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free comparison.  The per-image accumulators live in one fixed
// device array instead of memory obtained at call time, for callers that may
// not allocate (see gs_compare_noalloc in gs.h).  Every GPU that loads this
// library holds the array until the process exits.
// ---------------------------------------------------------------------------
constexpr int kNoAllocMaxImages = 64;
constexpr int kNoAllocMaxDevices = 64;
static __device__ __align__(256) CmpAcc g_noalloc_acc[kNoAllocMaxImages];

namespace {
std::mutex g_noalloc_mu;
CmpAcc* g_noalloc_ptr[kNoAllocMaxDevices] = {};   // device address of the array, per device
}  // namespace

// Once per device, with that device current: the array's device address.  In
// host code the array's name is only a host-side stand-in, so kernels are given
// this address, never the name.
static gs_status noalloc_scratch(CmpAcc** out) {
    int dev = 0;
    GS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kNoAllocMaxDevices) return set_error(GS_ERR_ARG, "device index out of range");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_acc);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(no-alloc comparison scratch)");
        g_noalloc_ptr[dev] = (CmpAcc*)p;
    }
    *out = g_noalloc_ptr[dev];
    return GS_OK;
}

}  // namespace gs

extern "C" gs_status gs_compare_noalloc(const float* dev_a, const float* dev_b, int H, int W, int K,
                                        gs_result* dev_out, void* stream) {
    using namespace gs;
    if (!dev_a || !dev_b || !dev_out || H < 1 || W < 1 || K < 1)
        return set_error(GS_ERR_ARG, "bad gs_compare_noalloc arguments");
    if (K > kNoAllocMaxImages)
        return set_error(GS_ERR_ARG, "gs_compare_noalloc: at most 64 image pairs per call (fixed scratch size)");
    CmpAcc* acc = nullptr;
    GS_TRY(noalloc_scratch(&acc));
    cudaStream_t st = (cudaStream_t)stream;
    // the array keeps the previous call's sums: clear the K accumulators first
    GS_TRY(launch_zero_acc(acc, K, st));
    GS_TRY(launch_compare(dev_a, dev_b, H, W, K, acc, st));
    return launch_finalize(acc, K, dev_out, st);
}
