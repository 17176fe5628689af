// A-5 forward compositing (Sec. 2.1, Step 3: Eq. 2, Eq. 3), A-6 loss
// (Sec. 4.1, Eq. 6) and A-7 backward compositing (Sec. 2.2, Step 4: Eq. 4,
// Eq. 5) on sm_103a.
//
// Two forms of the compositing, chosen per frame (fwd_entry_parallel,
// bwd_entry_parallel):
//
// Pixel-parallel: one pixel per thread; a full 16x16 tile takes a CTA of 256
// threads, the smaller tiles of a downsampled frame share one.  Tiles are
// issued in the heavy-first order produced by the binning, so the longest
// lists start first (the GPU counterpart of the paper's subtile streaming,
// Sec. 5.2).  Warps cover 8x4 pixel blocks.  The forward stages a tile's
// sorted list in batches, an entry a thread, with a mask per warp of the
// pixels that can blend the entry; each warp compacts the entries it may
// blend and composites them in pairs (their geometry in packed f32x2
// operations), four a step.  The alpha of a fragment is one FMA and one ex2:
// op e^(-q/2) = 2^(log2 op - q log2(e)/2), with q = d.(Q d) and log2 op staged
// per entry.  The forward also records, per pixel and run of 32 list entries,
// the entries it blended (the blend masks).
//
// Entry-parallel (tiles of at most 64 sampled pixels): see the section of
// that name below.
//
// The backward, given the blend masks, runs every 8x4 warp block as its own
// one-warp CTA: it visits the entries one of its pixels blended, takes each
// lane's decision from the lane's own mask bit, walks the fragments in
// reverse recovering T_k by division (Eq. 5), and sums the per-pixel terms
// of each Gaussian over the warp through shared memory, four entries at a
// time, before one global atomic per (Gaussian, warp, field).  Without masks
// a CTA per tile stages the list, visits the entries whose pixel box meets
// each warp's block, merges the per-pixel gradients with a reduce-scatter
// butterfly (each level halves the fields a lane carries) and sums the warps
// in shared memory first.  This replaces the paper's Gradient
// Merging Unit (Sec. 5.3).
#include <algorithm>
#include <type_traits>

#include "gs_internal.cuh"

namespace gs {

#define R_THREADS 256            // largest CTA (16x16 tile)
#define R_BATCH 1024             // largest batch of entries a tile stages at a time (32 mask words: lane q holds word q)
#define R_BWD_SMEM (70 * 1024)          // backward staging budget per CTA (512 entries: 51 KB, 4 CTAs per SM)

#define EP_B 256     // entries an entry-parallel tile stages per batch (64-pixel
                     // tiles 512: fewer CTA barriers per list)

struct StagedSplat {
    float4 a;   // x, y, conic_a, conic_b
    float4 b;   // conic_c, opacity, depth, log2(opacity)
    float4 c;   // r, g, b, unused
    int4 box;   // full-resolution integer box x0, x1, y0, y1
};

struct PixelMap {
    int i, j;        // sampled pixel
    bool inside;
    int px, py;      // full-resolution pixel
    int wx0, wx1, wy0, wy1;  // full-resolution extent of this warp's 8x4 block
};

// Threads serving one tile: tw * th, at least one warp.  Warps cover BW x BH
// pixel blocks (8x4, or 4x8 for 4-wide tiles).
__host__ __device__ inline int tile_threads(const Grid& g) {
    const int t = g.tw * g.th;
    return t < 32 ? 32 : t;
}

// Every CTA has R_THREADS threads and serves R_THREADS / TT tiles (TT =
// tile_threads): a full-resolution 16x16 tile takes the whole CTA, the
// smaller sampled tiles of a downsampled frame take groups of 2 or 1 warps,
// each group with its own slice of the staging buffer and its own named
// barrier, so a CTA always holds 8 warps.
struct Group {
    int TT;     // threads of the group
    int gi;     // group index in the CTA
    int lt;     // thread index in the group
    int B;      // entries staged per batch
    int tile;   // tile served, -1 if none
};

// `blk` numbers the CTA among those serving tiles this way; its groups take
// tile slots blk * gpc + gi of the tile order.
__device__ __forceinline__ Group make_group(const Grid& g, const uint32_t* order, int B, int blk) {
    Group G;
    G.TT = tile_threads(g);
    const int gpc = R_THREADS / G.TT;
    G.gi = threadIdx.x / G.TT;
    G.lt = threadIdx.x % G.TT;
    G.B = B;
    const int t = blk * gpc + G.gi;
    G.tile = t < g.TX * g.TY ? (order ? (int)__ldg(order + t) : t) : -1;
    return G;
}

__device__ __forceinline__ void group_sync(const Group& G) {
    if (G.TT == R_THREADS) __syncthreads();
    else if (G.TT == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + G.gi), "r"(G.TT) : "memory");
}

__device__ __forceinline__ PixelMap map_pixel(const Grid& g, int tile, int lt) {
    PixelMap m;
    const int tx = tile % g.TX, ty = tile / g.TX;
    const int lane = lt & 31, w = lt >> 5;
    const int BW = g.tw < 8 ? g.tw : 8, BH = 32 / BW, WX = g.tw / BW;
    const int bx = (w % WX) * BW, by = (w / WX) * BH;
    const int lx = lane % BW, ly = lane / BW;
    m.i = tx * g.tw + bx + lx;
    m.j = ty * g.th + by + ly;
    m.inside = by + ly < g.th && m.i < g.Ws && m.j < g.Hs;
    m.px = m.i * g.sx;
    m.py = m.j * g.sy;
    m.wx0 = (tx * g.tw + bx) * g.sx;
    m.wx1 = (tx * g.tw + bx + BW - 1) * g.sx;
    m.wy0 = (ty * g.th + by) * g.sy;
    m.wy1 = (ty * g.th + by + BH - 1) * g.sy;
    return m;
}

// Sampled pixel q of the tile: full-resolution coordinates, and whether it
// lies in the image.
__device__ __forceinline__ bool ep_pixel(const Grid& g, int tile, int q, int& i, int& j) {
    const int tx = tile % g.TX, ty = tile / g.TX;
    i = tx * g.tw + q % g.tw;
    j = ty * g.th + q / g.tw;
    return q < g.tw * g.th && i < g.Ws && j < g.Hs;
}

// The 2D Gaussian at offset d = (dx, dy) from its mean (Eq. 2): with the
// conic Q = [[ca, cb], [cb, cc]], (a, b) = Q d and q = d^T Q d = dx a + dy b,
// the exponent is -q/2 and the backward's mean gradient is (a, b) times
// dL/dexponent.  The operations are spelled out (no contraction left to the
// compiler) so that every compositing kernel, forward and backward, computes
// the same value and so takes the same blending decisions; q < 0 (a positive
// exponent, from rounding) skips the fragment.
struct Quad {
    float a, b, q;
};

__device__ __forceinline__ Quad quad_form(float ca, float cb, float cc, float dx, float dy) {
    Quad r;
    r.a = __fmaf_rn(cb, dy, __fmul_rn(ca, dx));
    r.b = __fmaf_rn(cc, dy, __fmul_rn(cb, dx));
    r.q = __fmaf_rn(dx, r.a, __fmul_rn(dy, r.b));
    return r;
}

// 2^x with the SFU's ex2 instruction.
__device__ __forceinline__ float exp2_sfu(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 1 / x with the SFU's rcp instruction (x well inside the normal range).
__device__ __forceinline__ float rcp_sfu(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// log2 of a staged opacity (the same instruction for every kernel that
// stages an entry, so all of them see the same value).
__device__ __forceinline__ float log2_opacity(float op) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(op));
    return y;
}

// -log2(e) / 2: op e^(-q/2) = 2^(log2(op) - q log2(e) / 2).
#define R_NEG_HALF_LOG2E (-0.721347520444481703680f)

// Unclamped alpha op e^(-q/2) of a fragment, one FMA and one ex2.
__device__ __forceinline__ float raw_alpha(float q, float log2_op) {
    return exp2_sfu(__fmaf_rn(q, R_NEG_HALF_LOG2E, log2_op));
}

// Two float32 values in one 64-bit register for the packed f32x2
// instructions (add, sub, mul, fma with round-to-nearest: one instruction for
// both halves, each half rounded exactly as the scalar operation).
typedef unsigned long long x2f;

__device__ __forceinline__ x2f x2_pack(float lo, float hi) {
    x2f r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void x2_unpack(x2f v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ x2f x2_add(x2f a, x2f b) {
    x2f r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ x2f x2_sub(x2f a, x2f b) {
    x2f r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ x2f x2_mul(x2f a, x2f b) {
    x2f r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ x2f x2_fma(x2f a, x2f b, x2f c) {  // a b + c
    x2f r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ x2f x2_dup(float v) { return x2_pack(v, v); }

__device__ __forceinline__ void x2_ld2(const float4* p, x2f& lo, x2f& hi) {  // one 16-byte load: two packed pairs
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    lo = v.x;
    hi = v.y;
}

// Pixel box of a staged Gaussian: its integer 3-sigma box (the definition of
// which pixels see it), shrunk to the pixels whose centre lies in the
// axis-aligned bounding box of the ellipse where alpha can reach alpha_min,
//     d^T Q d <= 2 ln(opacity / alpha_min),  half extents
//     sqrt(2 ln(opacity / alpha_min) (Q^-1)_xx), ... (Q = conic),
// widened against rounding (1e-4 added to the log threshold, a relative
// 1e-3 and 1e-3 px on the extent).  Every pixel it drops would fail the alpha
// test, so the image and gradients are unchanged; the compositing loops just
// visit fewer entries.  A Gaussian whose opacity is clearly below alpha_min
// gets an empty box.  Forward and backward use the same box.
// t2 receives the widened threshold 2 (ln(opacity / alpha_min) + 1e-4), or
// -1 when the box is the 3-sigma box alone (no usable ellipse).
__device__ __forceinline__ int4 pixel_box(const Splat& v, float alpha_min, float& t2) {
    const int xi = pix_floor(v.x), yi = pix_floor(v.y), r = v.radius;
    int4 box = make_int4(xi - r, xi + r, yi - r, yi + r);
    t2 = -1.f;
    const float det = v.ca * v.cc - v.cb * v.cb;
    if (!(det > 0.f) || !(v.op > 0.f) || !(alpha_min > 0.f)) return box;
    const float thr = logf(v.op / alpha_min);
    if (thr < -1e-4f) return make_int4(1, 0, 1, 0);  // empty: opacity < alpha_min
    const float t = 2.f * (fmaxf(thr, 0.f) + 1e-4f);
    const float ex = sqrtf(t * v.cc / det) * 1.001f + 1e-3f;
    const float ey = sqrtf(t * v.ca / det) * 1.001f + 1e-3f;
    if (!(ex < 1e8f) || !(ey < 1e8f)) return box;
    t2 = t;
    // pixel p qualifies when |p + 0.5 - x| <= ex
    box.x = max(box.x, (int)ceilf(v.x - ex - 0.5f));
    box.y = min(box.y, (int)floorf(v.x + ex - 0.5f));
    box.z = max(box.z, (int)ceilf(v.y - ey - 0.5f));
    box.w = min(box.w, (int)floorf(v.y + ey - 0.5f));
    return box;
}

// Stages a Gaussian for the unmasked backward.
__device__ __forceinline__ void fill_staged(const Splat& v, float alpha_min, StagedSplat& s) {
    s.a = make_float4(v.x, v.y, v.ca, v.cb);
    s.b = make_float4(v.cc, v.op, v.depth, log2_opacity(v.op));
    // the box as (x0, x1 - x0, y0, y1 - y0), clamped far outside any image;
    // an empty box never matches
    float t2;
    const int4 bx = pixel_box(v, alpha_min, t2);
    const int lo = -(1 << 28), hi = 1 << 28;
    const int x0 = max(bx.x, lo), x1 = min(bx.y, hi), y0 = max(bx.z, lo), y1 = min(bx.w, hi);
    s.box = x1 < x0 || y1 < y0 ? make_int4(hi, 0, hi, 0) : make_int4(x0, x1 - x0, y0, y1 - y0);
    s.c = make_float4(v.r, v.g, v.b, 0.f);
}

// Stages list entries [0, n_in) of `ids` into sp[] (and their ids into sid[]
// when given) with the group's TT threads.  Each thread gathers KST records
// before it converts any, so KST dependent id -> record loads are in flight
// per thread (KST = 4 for the small groups of downsampled frames, which
// stage several entries per thread; 1 for full-resolution tiles).
template <int DT, int KST>
__device__ __forceinline__ void stage_batch(const void* __restrict__ splats, const uint32_t* __restrict__ ids,
                                            int n_in, int lt, int TT, float alpha_min, StagedSplat* sp,
                                            uint32_t* sid) {
    for (int e0 = lt; e0 < n_in; e0 += KST * TT) {
        uint32_t id[KST];
#pragma unroll
        for (int k = 0; k < KST; ++k) id[k] = e0 + k * TT < n_in ? __ldg(ids + e0 + k * TT) : 0u;
        Splat v[KST];
#pragma unroll
        for (int k = 0; k < KST; ++k)
            if (e0 + k * TT < n_in) v[k] = load_splat<DT>(splats, id[k]);
#pragma unroll
        for (int k = 0; k < KST; ++k)
            if (e0 + k * TT < n_in) {
                fill_staged(v[k], alpha_min, sp[e0 + k * TT]);
                sid[e0 + k * TT] = id[k];
            }
    }
}

// Overlap masks of the staged entries with the warp's block: bit e of word q
// is set when entry 32q + e (below `limit`) meets the block.  Lane q returns
// word q (words at or beyond `words` are zero), so a word is one shuffle away
// and the masks stay in registers.  Only the words that hold entries are
// built (a loop to the batch's last word rather than over all 32:
// tracking step 236.6 -> 231.5 us).
__device__ __forceinline__ unsigned warp_masks(const StagedSplat* sp, int limit, int words, const PixelMap& m) {
    const int lane = threadIdx.x & 31;
    unsigned mine = 0u;
    const int nq = min(words, (limit + 31) >> 5);  // the words holding entries
#pragma unroll 4
    for (int q = 0; q < nq; ++q) {
        const int e = q * 32 + lane;
        bool hit = false;
        if (e < limit) {
            const int4 box = sp[e].box;
            hit = !(box.x + box.y < m.wx0 || box.x > m.wx1 || box.z + box.w < m.wy0 || box.z > m.wy1);
        }
        const unsigned w = __ballot_sync(0xffffffffu, hit);
        if (lane == q) mine = w;
    }
    return mine;
}

// Forward outputs (gs_render_fwd) and, when trgb is given, the fused loss
// (gs_render_fwd_loss).
struct FwdOut {
    float* rgb;
    float* depth;
    float* t;
    uint32_t* last;
    uint32_t* nb;
    const float* trgb;  // NULL: no loss
    const float* tdepth;
    float* d_rgb;
    float* d_depth;
    double* loss;
    uint32_t* bmask;    // NULL: no blend masks
};

// Blend masks: for each pixel of a tile and each run of 32 list entries,
// the entries the forward blended into that pixel (bit e of run r: entry
// 32 r + e of the tile's list).  A pixel-parallel tile (TT <= 256 threads,
// pixel = thread lt of the group) with list [s, s + len) keeps run r of
// pixel lt at word 256 (floor(s / 32) + t) + r TT + lt: run-major, so a
// warp's 32 pixels read one 128-byte line; the TT ceil(len / 32) words of a
// tile end before the next tile's first word.
__host__ __device__ inline size_t blend_mask_base(int tile, uint32_t start) {
    return (size_t)256 * ((size_t)(start >> 5) + (size_t)tile);
}

// Tiles of at most 64 sampled pixels keep run r of pixel q (in row order) at
// word 64 (floor(s / 32) + t) + 64 r + q.
__host__ __device__ inline size_t blend_mask_base_ep(int tile, uint32_t start) {
    return (size_t)64 * ((size_t)(start >> 5) + (size_t)tile);
}

// Writes sampled pixel (i, j)'s results; with the fused loss also its image
// gradient (the formulas of k_loss_l1 on the same float values) and returns
// its share of the loss.
__device__ __forceinline__ float write_pixel(const gs_config& cfg, const Grid& g, const FwdOut& O, int i, int j,
                                             float C0, float C1, float C2, float D, float T, uint32_t last,
                                             uint32_t nb) {
    const size_t P = (size_t)g.Ws * g.Hs;
    const size_t pix = (size_t)j * g.Ws + i;
    const float c[3] = {C0 + T * cfg.bg[0], C1 + T * cfg.bg[1], C2 + T * cfg.bg[2]};
    O.rgb[pix] = c[0];
    O.rgb[P + pix] = c[1];
    O.rgb[2 * P + pix] = c[2];
    O.depth[pix] = D;
    O.t[pix] = T;
    O.last[pix] = last;
    if (O.nb) O.nb[pix] = nb;
    if (!O.trgb) return 0.f;
    const float inv3 = 1.f / (3.f * (float)P), inv1 = 1.f / (float)P;
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float r = c[k] - O.trgb[k * P + pix];
        acc += cfg.w_rgb * fabsf(r) * inv3;
        O.d_rgb[k * P + pix] = cfg.w_rgb * (r > 0.f ? inv3 : (r < 0.f ? -inv3 : 0.f));
    }
    const float td = O.tdepth[pix];
    float gd = 0.f;
    if (td != 0.f) {
        const float r = D - td;
        acc += cfg.w_depth * fabsf(r) * inv1;
        gd = cfg.w_depth * (r > 0.f ? inv1 : (r < 0.f ? -inv1 : 0.f));
    }
    O.d_depth[pix] = gd;
    return acc;
}

// Warp sum of the pixels' loss shares, one float64 atomic per warp (all 32
// lanes call it).
__device__ __forceinline__ void add_loss(const FwdOut& O, float part) {
    if (!O.trgb) return;
    part = warp_sum(part);
    if ((threadIdx.x & 31) == 0 && part != 0.f) atomicAdd(O.loss, (double)part);
}

// ---------------------------------------------------------------------------
// Forward compositing, pixel-parallel
// ---------------------------------------------------------------------------
// A tile of NW warps (32 NW threads, one pixel each; a CTA of 256 threads
// serves 8 / NW tiles) stages its list in batches.  The thread that stages an
// entry also forms, for each warp's block of 32 pixels, the mask of the
// pixels that can blend it: the entry's pixel box, which the definition makes
// exact, intersected with its alpha >= alpha_min ellipse, which only saves
// work.  Each warp then compacts the entries whose mask is not empty, 32 list
// entries at a time, into pairs of slots of its own, and composites two
// entries a step: their geometry in packed f32x2 operations (each half the
// scalar operation), the alpha test, transmittance and blending entry by entry, each
// lane's box test one bit of the slot's mask.
//
// Issue-bound (64 % issue-active, then barriers and fixed latencies): box tests
// of four words in every lane, scalar geometry and steps of three entries
// padded with dummies took 74 instructions a (warp, entry) visit, 65.9 M for
// the tracking frame, against 41.4 M now.  Forward + loss 640x480 / 200k 84 ->
// 61.4 us, forward 1200x680 / 1M 180 -> 100, 1296x968 / 750k bf16 232 -> 144.
// Measured and not kept: records by cp.async a batch ahead (raw records
// in shared memory cost each warp their unpacking: 61.4 / 105.8 / 152.7), the
// next batch staged beside the compositing (60.9 / 112 / 157), two entries a
// step (68.9 / 102 / 146).
// Staged entries of a tile, an entry a thread.
template <int NW>
struct __align__(16) FwdStage {
    float4 a[32 * NW];           // x, y, conic_a, conic_b
    float4 col[32 * NW];         // r, g, b, depth
    float2 cl[32 * NW];          // conic_c, log2(opacity)
    uint32_t pm[NW][32 * NW];    // per warp: the pixels that can blend the entry
};

// A warp's compacted entries of one run: slots 2 p and 2 p + 1 as pair p.
struct __align__(16) FwdSlots {
    float4 xy[16];   // x0 x1 y0 y1
    float4 ab[16];   // conic a, b
    float4 cl[16];   // conic c, log2(opacity)
    uint4 pb[16];    // pixel masks, run bits
    float4 col[32];  // r, g, b, depth
};

__device__ __forceinline__ float sqrt_sfu(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Pixel masks of a Gaussian over the tile's warp blocks: bit p of pm[w] is
// set when pixel p of warp w's block lies in the Gaussian's box and may lie
// in the region d^T Q d <= t (t = t2 widened by 1 %; t2 < 0: the box alone).
// Blocks are 8 x 4 pixels, WX of them across the tile.  Per strip of blocks
// (a band of rows) the ellipse's x extent over the band follows from its
// chord [(-cb dy -+ sqrt(t ca - det dy^2)) / ca] at the band's rows closest
// to the rightmost point (dy = -cb ex / cc) and the leftmost point (dy = cb
// ex / cc): the chord's right end is concave in dy and its left end convex.
// The extent is widened by 1e-2 ex + 0.05 px, well beyond the float32
// rounding of the fragment test, so no pixel the alpha test accepts is
// dropped.
template <int NW>
__device__ __forceinline__ void pixel_masks(const Splat& v, float alpha_min, const Grid& g, int tile,
                                            uint32_t (&pm)[NW]) {
#pragma unroll
    for (int w = 0; w < NW; ++w) pm[w] = 0u;
    float t2;
    int4 bx = pixel_box(v, alpha_min, t2);  // x0, x1, y0, y1
    const int lo = -(1 << 28), hi = 1 << 28;
    bx = make_int4(max(bx.x, lo), min(bx.y, hi), max(bx.z, lo), min(bx.w, hi));
    // (NW == 8: 16x16 pixels at stride 1; else 16x8 or 8x16)
    constexpr int BW = 8;
    const int sx = NW == 8 ? 1 : g.sx, sy = NW == 8 ? 1 : g.sy, tw = NW == 8 ? 16 : g.tw, th = NW == 8 ? 16 : g.th;
    const int WX = tw / BW;
    constexpr int BH = 4;
    const int tx = tile % g.TX, ty = tile / g.TX;
    const int X0 = tx * tw * sx, Y0 = ty * th * sy;
    const bool ell = t2 > 0.f;
    float det = 0.f, tA = 0.f, ey = 0.f, yr = 0.f, ia = 0.f, sl = 0.f;
    if (ell) {
        const float t = t2 * 1.01f;
        det = v.ca * v.cc - v.cb * v.cb;
        const float ex = sqrt_sfu(__fdividef(t * v.cc, det));
        tA = t * v.ca;
        ey = sqrt_sfu(__fdividef(tA, det));
        yr = __fdividef(-v.cb * ex, v.cc);
        ia = rcp_sfu(v.ca);
        sl = 1e-2f * ex + 0.05f;
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        if (NW != 8 && s * WX >= NW) break;
        // the strip's rows inside the box: sampled rows jlo .. jhi
        const int ry = Y0 + s * BH * sy;
        const int jlo = max(0, ceil_div_i(bx.z - ry, sy)), jhi = min(BH - 1, floor_div(bx.w - ry, sy));
        if (jlo > jhi) continue;
        int c0 = bx.x, c1 = bx.y;
        if (ell) {
            const float ylo = fminf(fmaxf((float)(ry + jlo * sy) + 0.5f - v.y, -ey), ey);
            const float yhi = fminf(fmaxf((float)(ry + jhi * sy) + 0.5f - v.y, -ey), ey);
            const float dr = fminf(fmaxf(yr, ylo), yhi), dl = fminf(fmaxf(-yr, ylo), yhi);
            const float xr = (sqrt_sfu(fmaxf(tA - det * dr * dr, 0.f)) - v.cb * dr) * ia;
            const float xl = (-sqrt_sfu(fmaxf(tA - det * dl * dl, 0.f)) - v.cb * dl) * ia;
            c0 = max(c0, (int)ceilf(v.x + xl - sl - 0.5f));
            c1 = min(c1, (int)floorf(v.x + xr + sl - 0.5f));
        }
        const int ilo = max(0, ceil_div_i(max(c0, lo) - X0, sx)), ihi = min(tw - 1, floor_div(min(c1, hi) - X0, sx));
        if (ilo > ihi) continue;
        const uint32_t cols = (2u << ihi) - (1u << ilo);
        const int rows = jhi - jlo;
        const uint32_t rsel = (0x01010101u >> (8 * (3 - rows))) << (8 * jlo);
        // (constant indices, so that pm stays in registers)
#pragma unroll
        for (int w = 0; w < NW; ++w)
            if (w >= s * WX && w < (s + 1) * WX) pm[w] = ((cols >> ((w - s * WX) * BW)) & ((1u << BW) - 1u)) * rsel;
    }
}

template <int DT, int NW>
__device__ __forceinline__ void fwd_pp(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                       const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                       const FwdOut& O, int tile, FwdStage<NW>& S, FwdSlots& R) {
    constexpr int TT = 32 * NW;  // a batch: an entry a thread
    const int lane = threadIdx.x & 31, lt = threadIdx.x % TT, w = lt >> 5, gi = threadIdx.x / TT;
    const PixelMap m = map_pixel(g, tile, lt);
    const uint32_t start = ranges[2 * tile], end = ranges[2 * tile + 1];
    const x2f PXC = x2_dup((float)m.px + 0.5f), PYC = x2_dup((float)m.py + 0.5f);
    const uint32_t bit = 1u << lane;
    const float never = __int_as_float(0x7f800000);
    float T = 1.f;
    x2f C01 = x2_dup(0.f), C2D = x2_dup(0.f);
    uint32_t last = 0, nb = 0;
    float amin = m.inside ? cfg.alpha_min : never;  // `never`: the pixel has stopped
    // this pixel's blend-mask words (run r at bm_pix[r TT])
    uint32_t* const bm_pix = O.bmask ? O.bmask + blend_mask_base(tile, start) + lt : nullptr;
    auto barrier = [&] {
        if (NW == 8) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + gi), "r"(TT) : "memory");
    };
    // this thread's entry of a batch; its id is loaded a batch ahead
    uint32_t id = start + lt < end ? __ldg(vals + start + lt) : 0u;
    for (uint32_t b = start; b < end; b += TT) {
        if (b != start) {
            // the previous batch is no longer read; every pixel stopped: the tile ends
            const bool done = amin == never;
            int stopped;
            if (NW == 8) stopped = __syncthreads_count(done);
            else
                asm volatile("{ .reg .pred p; setp.ne.u32 p, %3, 0; bar.red.popc.u32 %0, %1, %2, p; }"
                             : "=r"(stopped) : "r"(1 + gi), "r"(TT), "r"((unsigned)done) : "memory");
            if (stopped == TT) break;
        }
        const int n_in = (int)min((uint32_t)TT, end - b);
        if (lt < n_in) {
            const Splat v = load_splat<DT>(splats, id);
            S.a[lt] = make_float4(v.x, v.y, v.ca, v.cb);
            S.col[lt] = make_float4(v.r, v.g, v.b, v.depth);
            S.cl[lt] = make_float2(v.cc, log2_opacity(v.op));
            uint32_t pm[NW];
            pixel_masks<NW>(v, cfg.alpha_min, g, tile, pm);
#pragma unroll
            for (int q = 0; q < NW; ++q) S.pm[q][lt] = pm[q];
        }
        if (b + TT + lt < end) id = __ldg(vals + b + TT + lt);
        barrier();
        if (__all_sync(0xffffffffu, amin == never)) continue;
        const uint32_t base = b - start;
#pragma unroll 1
        for (int q = 0; q < n_in; q += 32) {
            const int e = q + lane;
            const uint32_t pix = e < n_in ? S.pm[w][e] : 0u;
            const unsigned hit = __ballot_sync(0xffffffffu, pix != 0u);
            const int cnt = __popc(hit);
            uint32_t bq = 0u;  // entries of the run this pixel blended
            if (pix != 0u) {
                const int slot = __popc(hit & (bit - 1u));
                const float4 A = S.a[e];
                const float2 L = S.cl[e];
                float* const xy = reinterpret_cast<float*>(R.xy + (slot >> 1)) + (slot & 1);
                float* const ab = reinterpret_cast<float*>(R.ab + (slot >> 1)) + (slot & 1);
                float* const cl = reinterpret_cast<float*>(R.cl + (slot >> 1)) + (slot & 1);
                uint32_t* const pb = reinterpret_cast<uint32_t*>(R.pb + (slot >> 1)) + (slot & 1);
                xy[0] = A.x;
                xy[2] = A.y;
                ab[0] = A.z;
                ab[2] = A.w;
                cl[0] = L.x;
                cl[2] = L.y;
                pb[0] = pix;
                pb[2] = bit;
                R.col[slot] = S.col[e];
            }
            if ((cnt & 1) && lane == cnt) {  // the last pair's empty half
                reinterpret_cast<uint32_t*>(R.pb + (cnt >> 1))[1] = 0u;
                R.col[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            __syncwarp();
            // NP pairs of entries from pair p
            auto step = [&](auto NP_, int p) {
                constexpr int NP = decltype(NP_)::value;
                float al[2 * NP];  // the alphas do not depend on T
                bool in[2 * NP];
                uint32_t rb[2 * NP];
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    x2f X, Y, CA, CB, CC, LOP;
                    x2_ld2(R.xy + p + h, X, Y);
                    x2_ld2(R.ab + p + h, CA, CB);
                    x2_ld2(R.cl + p + h, CC, LOP);
                    const uint4 pb = R.pb[p + h];
                    const x2f DX = x2_sub(PXC, X), DY = x2_sub(PYC, Y);
                    const x2f QA = x2_fma(CB, DY, x2_mul(CA, DX));  // Q d, as quad_form
                    const x2f QB = x2_fma(CC, DY, x2_mul(CB, DX));
                    const x2f Q = x2_fma(DX, QA, x2_mul(DY, QB));
                    float q0, q1, e0, e1;
                    x2_unpack(Q, q0, q1);
                    x2_unpack(x2_fma(Q, x2_dup(R_NEG_HALF_LOG2E), LOP), e0, e1);
                    al[2 * h] = fminf(cfg.alpha_max, exp2_sfu(e0));
                    al[2 * h + 1] = fminf(cfg.alpha_max, exp2_sfu(e1));
                    in[2 * h] = (pb.x & bit) != 0u && !(q0 < 0.f);
                    in[2 * h + 1] = (pb.y & bit) != 0u && !(q1 < 0.f);
                    rb[2 * h] = pb.z;
                    rb[2 * h + 1] = pb.w;
                }
                // Front to back: a fragment in the box with alpha >= alpha_min
                // is blended unless it would take T below t_eps, where the
                // pixel stops (Eq. 3); a skipped one has factor 1 and adds
                // zero weight.
#pragma unroll
                for (int u = 0; u < 2 * NP; ++u) {
                    const bool valid = in[u] && al[u] >= amin;
                    const float Tn = T * (1.f - al[u]);
                    const bool stop = valid && Tn < cfg.t_eps;
                    const bool ok = valid && !stop;
                    const x2f W = x2_dup(ok ? al[u] * T : 0.f);
                    const float4 c = R.col[2 * p + u];
                    C01 = x2_fma(W, x2_pack(c.x, c.y), C01);
                    C2D = x2_fma(W, x2_pack(c.z, c.w), C2D);
                    T = ok ? Tn : T;
                    amin = stop ? never : amin;
                    bq |= ok ? rb[u] : 0u;
                }
            };
            int p = 0;
#pragma unroll 1
            for (; 2 * p + 2 < cnt; p += 2) step(std::integral_constant<int, 2>(), p);
            if (2 * p < cnt) step(std::integral_constant<int, 1>(), p);
            // the count and the last position follow from the run's blended bits
            nb += __popc(bq);
            if (bq != 0u) last = base + (uint32_t)(q + 32 - __clz(bq));
            // every run up to the one where the warp stops is written (a
            // run past every pixel's last position is never read)
            if (bm_pix) bm_pix[(size_t)((base + q) >> 5) * TT] = bq;
            if (__all_sync(0xffffffffu, amin == never)) break;
            __syncwarp();  // the next run reuses the slots
        }
    }
    float C0, C1, C2, D;
    x2_unpack(C01, C0, C1);
    x2_unpack(C2D, C2, D);
    float lpart = 0.f;
    if (m.inside) lpart = write_pixel(cfg, g, O, m.i, m.j, C0, C1, C2, D, T, last, nb);
    add_loss(O, lpart);
}

// The CTA's tiles: 8 / NW consecutive ones of the order.
template <int NW>
struct FwdSmem {
    FwdStage<NW> S[8 / NW];
    FwdSlots R[8];
};

template <int DT, int NW>
__device__ __forceinline__ void fwd_cta(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                        const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                        const uint32_t* __restrict__ order, const FwdOut& O, int blk) {
    extern __shared__ __align__(16) unsigned char r_smem[];
    FwdSmem<NW>& M = *reinterpret_cast<FwdSmem<NW>*>(r_smem);
    const int gi = (int)threadIdx.x / (32 * NW), t = blk * (8 / NW) + gi;
    if (t >= g.TX * g.TY) return;
    const int tile = order ? (int)__ldg(order + t) : t;
    fwd_pp<DT, NW>(cfg, g, splats, vals, ranges, O, tile, M.S[gi], M.R[threadIdx.x >> 5]);
}

// CT: CTAs per SM.  Three (80 registers) finish a tile sooner, four (64) keep
// more warps in flight: 1200 tiles 61.4 against 64.7 us (640x480 / 200k), but
// 3225 tiles 105.6 against 100.2 (1200x680 / 1M) and 4941 tiles 154 against 144
// (1296x968 / 750k): three up to 8 CTAs per SM.
static bool fwd_three(int64_t ctas) { return ctas <= 8 * (int64_t)num_sms(); }

template <int DT, int NW, int CT>
__global__ void __launch_bounds__(R_THREADS, CT)
    k_render_fwd(gs_config cfg, Grid g, const void* __restrict__ splats, const uint32_t* __restrict__ vals,
                 const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order, FwdOut O) {
    fwd_cta<DT, NW>(cfg, g, splats, vals, ranges, order, O, (int)blockIdx.x);
}

// ---------------------------------------------------------------------------
// Loss (Eq. 6) with L1 residuals
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_loss_l1(gs_config cfg, int64_t P, const float* __restrict__ rgb,
                                                 const float* __restrict__ depth, const float* __restrict__ trgb,
                                                 const float* __restrict__ tdepth, float* __restrict__ d_rgb,
                                                 float* __restrict__ d_depth, double* __restrict__ loss) {
    __shared__ float s_w[8];
    const float inv3 = 1.f / (3.f * (float)P), inv1 = 1.f / (float)P;
    float acc = 0.f;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < P; q += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float r = rgb[c * P + q] - trgb[c * P + q];
            acc += cfg.w_rgb * fabsf(r) * inv3;
            d_rgb[c * P + q] = cfg.w_rgb * (r > 0.f ? inv3 : (r < 0.f ? -inv3 : 0.f));
        }
        const float td = tdepth[q];
        float gd = 0.f;
        if (td != 0.f) {
            const float r = depth[q] - td;
            acc += cfg.w_depth * fabsf(r) * inv1;
            gd = cfg.w_depth * (r > 0.f ? inv1 : (r < 0.f ? -inv1 : 0.f));
        }
        d_depth[q] = gd;
    }
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += (double)s_w[w];
        atomicAdd(loss, s);
    }
}

// ---------------------------------------------------------------------------
// Backward compositing
// ---------------------------------------------------------------------------
// Fields merged per fragment, in the order the backward forms them:
//   GS_TRACK  a h, b h, u dx, u dy, v dy, w gD                      (6)
//   GS_MAP    a h, b h, u dx, u dy, v dy, G T (dL/dalpha T^-1), w gD,
//             w gR, w gG, w gB                                      (10)
// with h = -dL/d(exponent) / 2 = -alpha dL/dalpha / 2, (u, v) = h (dx, dy),
// (a, b) = Q d and w = T alpha.  The gradients follow by exact power-of-two
// scalings applied once per entry when a batch is written out:
// dL/dmean = -2 (a h, b h) (since dL/dmean = Q d dL/d(exponent)),
// dL/dconic = (u dx, 2 u dy, v dy) (the exponent is -(A dx^2 + 2 B dx dy +
// C dy^2) / 2).
template <int MODE>
struct Fields {
    static constexpr int N = MODE == GS_MAP ? 10 : 6;
};

// grad2d column of a merged field, and its scale.
template <int MODE>
__device__ __forceinline__ int field_col(int f) {
    if (MODE == GS_MAP) return f < 7 ? f : f + 1;  // du dv dA dB dC dop dd | dr dg db
    return f < 5 ? f : 6;                          // du dv dA dB dC | dd
}
__device__ __forceinline__ float field_scale(int f) { return f < 2 ? -2.f : (f == 3 ? 2.f : 1.f); }

// Per-fragment quantities of the backward that do not depend on the
// running state: offsets, Gaussian falloff G, unclamped and clamped alpha,
// and whether the fragment was blended.
struct FragGeo {
    float dx, dy, a, b, q, raw, alpha, dep;  // offset, Q d, d^T Q d, alphas, depth
    bool contrib;
};

// The geometry of a staged entry at the pixel, with the forward's arithmetic
// (so the same alpha).  Without blend masks the decision is re-derived: inside
// the box, exponent <= 0, alpha >= alpha_min, before the pixel's last blended
// position.
__device__ __forceinline__ FragGeo frag_geo(const StagedSplat& s, const PixelMap& m, float pxc, float pyc,
                                            const gs_config& cfg, bool before_last) {
    FragGeo f;
    const float4 A = s.a;
    const float4 Bv = s.b;
    const int4 box = s.box;
    f.dep = Bv.z;
    f.dx = pxc - A.x;
    f.dy = pyc - A.y;
    const Quad Qd = quad_form(A.z, A.w, Bv.x, f.dx, f.dy);
    f.a = Qd.a;
    f.b = Qd.b;
    f.q = Qd.q;
    f.raw = raw_alpha(Qd.q, Bv.w);
    f.alpha = fminf(cfg.alpha_max, f.raw);
    f.contrib = before_last && (unsigned)(m.px - box.x) <= (unsigned)box.y &&
                (unsigned)(m.py - box.z) <= (unsigned)box.w && !(f.q < 0.f) && !(f.alpha < cfg.alpha_min);
    return f;
}

// A pixel's running state in the backward walk: the transmittance in front
// of the current entry, s = A . g (the normalised suffix sum A of colour and
// depth behind it -- the background entering with weight T_final -- dotted
// with the image gradient g) and g itself.
struct BackState {
    float T, sg, gC0, gC1, gC2, gD;
};

// Loads a pixel's backward inputs (t_final, image gradients); pixels outside
// the image keep T = 1 and zero gradients.  Returns its last_idx (0 outside).
__device__ __forceinline__ uint32_t back_start(const gs_config& cfg, const Grid& g, const PixelMap& m,
                                               const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                                               const float* __restrict__ d_rgb, const float* __restrict__ d_depth,
                                               BackState& S) {
    S.T = 1.f;
    S.gC0 = S.gC1 = S.gC2 = S.gD = 0.f;
    uint32_t last = 0;
    if (m.inside) {
        const size_t P = (size_t)g.Ws * g.Hs;
        const size_t pix = (size_t)m.j * g.Ws + m.i;
        S.T = t_final[pix];
        last = last_idx[pix];
        S.gC0 = d_rgb[pix];
        S.gC1 = d_rgb[P + pix];
        S.gC2 = d_rgb[2 * P + pix];
        S.gD = d_depth[pix];
    }
    S.sg = cfg.bg[0] * S.gC0 + cfg.bg[1] * S.gC1 + cfg.bg[2] * S.gC2;
    return last;
}

// One fragment, back to front: T_k recovered by division (Eq. 5).  With
// w = T_k alpha_k and c_k . g (colour and depth dotted with the image
// gradient),
//   dL/dalpha_k = T_k (c_k . g - s_k),  s_k = A_k . g,
//   s_{k-1} = s_k + alpha_k (c_k . g - s_k),
// and alpha dL/dalpha = w (c . g - s) is the exponent's gradient.  Writes the
// fragment's merged fields f[0, Fields<MODE>::N).  Branch-free: every lane
// evaluates the recursion (all values are finite: 1 - alpha >= 1 -
// alpha_max); a lane whose pixel did not blend the entry keeps its state and
// contributes zeros.
template <int MODE>
__device__ __forceinline__ void back_frag(BackState& S, const FragGeo& fg, const float4& Cc, const gs_config& cfg,
                                          float* f) {
    const float alpha = fg.alpha;
    // fast division (at most 2 ulp for these operands: 1 - alpha in
    // [0.01, 1], T in [t_eps, 1]); over the few hundred entries a pixel
    // recovers the relative drift stays near 1e-5
    S.T = fg.contrib ? __fdividef(S.T, 1.f - alpha) : S.T;
    const float w = fg.contrib ? alpha * S.T : 0.f;
    const float cg = __fmaf_rn(fg.dep, S.gD, __fmaf_rn(Cc.z, S.gC2, __fmaf_rn(Cc.y, S.gC1, Cc.x * S.gC0)));
    const float dif = cg - S.sg;
    S.sg = fg.contrib ? __fmaf_rn(alpha, dif, S.sg) : S.sg;
    // the clamp passes no gradient to opacity or shape
    const bool clamped = fg.raw > cfg.alpha_max;
    const float h = clamped ? 0.f : (-0.5f * w) * dif;  // -dL/d(exponent) / 2
    const float u = h * fg.dx, v = h * fg.dy;
    f[0] = fg.a * h;
    f[1] = fg.b * h;
    f[2] = u * fg.dx;
    f[3] = u * fg.dy;
    f[4] = v * fg.dy;
    if (MODE == GS_MAP) {
        // dalpha/dopacity = e^(-q/2)
        f[5] = (fg.contrib && !clamped) ? exp2_sfu(__fmul_rn(fg.q, R_NEG_HALF_LOG2E)) * (S.T * dif) : 0.f;
        f[6] = w * S.gD;
        f[7] = w * S.gC0;
        f[8] = w * S.gC1;
        f[9] = w * S.gC2;
    } else {
        f[5] = w * S.gD;
    }
}

// Backward compositing of group G's tile, pixel-parallel, without blend
// masks (smem: the CTA's staging, id and accumulator buffers for gpc groups
// of G.B entries; s_max_all: one word per warp).  Each warp visits the
// staged entries whose pixel box meets its block, up to the furthest last
// position of its pixels.
template <int DT, int MODE, int KST>
__device__ __forceinline__ void bwd_pp(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                       const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                       const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                                       const float* __restrict__ d_rgb, const float* __restrict__ d_depth,
                                       float* __restrict__ grad2d, const Group& G, unsigned char* smem,
                                       uint32_t* s_max_all) {
    constexpr int NF = Fields<MODE>::N;
    constexpr int BSTEP = 2;  // entries per backward step, merged together
    static_assert(BSTEP * NF <= 32, "one lane per merged value");
    const int gpc = R_THREADS / G.TT;
    StagedSplat* sp_all = reinterpret_cast<StagedSplat*>(smem);
    uint32_t* sid_all = reinterpret_cast<uint32_t*>(sp_all + gpc * G.B);
    float(*acc_all)[NF] = reinterpret_cast<float(*)[NF]>(sid_all + gpc * G.B);
    StagedSplat* sp = sp_all + G.gi * G.B;
    uint32_t* sid = sid_all + G.gi * G.B;
    float(*acc)[NF] = acc_all + G.gi * G.B;
    uint32_t* s_wl = s_max_all + G.gi * (G.TT >> 5);  // the group's per-warp maxima
    const int tile = G.tile;
    const PixelMap m = map_pixel(g, tile, G.lt);
    const uint32_t start = ranges[2 * tile], end = ranges[2 * tile + 1];
    const float pxc = (float)m.px + 0.5f, pyc = (float)m.py + 0.5f;
    const int lane = threadIdx.x & 31;
    // the merged field this lane adds (entry owner / NF of a step, field
    // owner % NF), or -1
    const int owner = merge_owner<BSTEP * NF>();
    BackState S;
    uint32_t last = back_start(cfg, g, m, t_final, last_idx, d_rgb, d_depth, S);
    // a last_idx beyond the tile's list (inconsistent inputs) is clamped
    last = min(last, end - start);
    uint32_t wlast = last;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wlast = max(wlast, __shfl_xor_sync(0xffffffffu, wlast, o));
    if (lane == 0) s_wl[G.lt >> 5] = wlast;
    group_sync(G);
    uint32_t s_max = 0;
    for (int w = 0; w < (G.TT >> 5); ++w) s_max = max(s_max, s_wl[w]);
    const int words = G.B / 32;
    // batches [start + k B, start + (k + 1) B) from the last one holding a
    // blended entry back to the first (whole mask words for every batch)
    for (int k = (int)((s_max + G.B - 1) / G.B) - 1; k >= 0; --k) {
        const uint32_t base_pos = (uint32_t)k * G.B;
        const uint32_t lo = start + base_pos, hi = start + min(s_max, base_pos + G.B);
        const int n_in = (int)(hi - lo);
        stage_batch<DT, KST>(splats, vals + lo, n_in, G.lt, G.TT, cfg.alpha_min, sp, sid);
        for (int q = G.lt; q < G.B * NF; q += G.TT) (&acc[0][0])[q] = 0.f;
        group_sync(G);
        // entries at or beyond the warp's furthest blended position are skipped
        const int wlimit = (int)min((uint32_t)n_in, wlast > base_pos ? wlast - base_pos : 0u);
        const unsigned mword = warp_masks(sp, wlimit, words, m);
#pragma unroll 1
        for (int q = words - 1; q >= 0; --q) {
            unsigned mq = __shfl_sync(0xffffffffu, mword, q);
            while (mq) {
                // BSTEP entries per step, last first: their geometry does
                // not depend on the running state
                int eu[BSTEP];
#pragma unroll
                for (int u = 0; u < BSTEP; ++u) {
                    const int bit = mq ? 31 - __clz(mq) : -1;
                    eu[u] = bit >= 0 ? q * 32 + bit : -1;
                    if (bit >= 0) mq &= ~(1u << bit);
                }
                FragGeo gu[BSTEP];
#pragma unroll
                for (int u = 0; u < BSTEP; ++u) {
                    const int e = eu[u] >= 0 ? eu[u] : 0;
                    gu[u] = frag_geo(sp[e], m, pxc, pyc, cfg, eu[u] >= 0 && base_pos + (uint32_t)e < last);
                }
                float f[BSTEP * NF];
#pragma unroll
                for (int u = 0; u < BSTEP; ++u) back_frag<MODE>(S, gu[u], sp[eu[u] >= 0 ? eu[u] : 0].c, cfg, f + u * NF);
                // the step's fields merged at once
                bool any = false;
#pragma unroll
                for (int u = 0; u < BSTEP; ++u) any = any || gu[u].contrib;
                if (__any_sync(0xffffffffu, any)) {
                    const float v = warp_merge<BSTEP * NF>(f);
                    if (owner >= 0) {
                        const int u = owner / NF;
                        int e = eu[0];
#pragma unroll
                        for (int x = 1; x < BSTEP; ++x) e = u == x ? eu[x] : e;
                        if (e >= 0) atomicAdd(&acc[e][owner - u * NF], v);
                    }
                }
            }
        }
        group_sync(G);
        for (int q = G.lt; q < n_in * NF; q += G.TT) {
            const float v = (&acc[0][0])[q];
            const int f = q % NF;
            if (v != 0.f) atomicAdd(grad2d + (size_t)sid[q / NF] * GS_GRAD2D_STRIDE + field_col<MODE>(f),
                                    v * field_scale(f));
        }
        if (k > 0) group_sync(G);  // the next batch reuses the buffers
    }
}

// 4 CTAs per SM for the pose-only backward (64 registers); 3 when mapping,
// whose 16-slot merge would spill at 64 (measured 363 vs 342 us at 1200x680).
template <int DT, int MODE, int KST>
__global__ void __launch_bounds__(R_THREADS, KST == 1 ? (MODE == GS_TRACK ? 4 : 3) : 2)
    k_render_bwd(gs_config cfg, Grid g, const void* __restrict__ splats, const uint32_t* __restrict__ vals,
                 const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order,
                 const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                 const float* __restrict__ d_rgb, const float* __restrict__ d_depth, float* __restrict__ grad2d,
                 int B) {
    extern __shared__ __align__(16) unsigned char r_smem[];
    __shared__ uint32_t s_max_all[R_THREADS / 32];
    const Group G = make_group(g, order, B, blockIdx.x);
    if (G.tile < 0) return;
    bwd_pp<DT, MODE, KST>(cfg, g, splats, vals, ranges, t_final, last_idx, d_rgb, d_depth, grad2d, G, r_smem,
                          s_max_all);
}

// The masked backward's working set of one warp: a ring of 64 staged entries
// (slot s: pair s / 2, half s & 1, so that two consecutive slots load as
// packed pairs, two fields per 16-byte load) and what the lanes hand over to
// be summed in a step of two pairs.
#define PW_TERMS 6  // per pair: a h, b h, u dx, u dy, v dy, and w gD (pose only) or the opacity's (mapping)
struct __align__(16) PwRing {
    float4 xy[32];     // x0 x1 y0 y1
    float4 ab[32];     // conic a, b
    float4 cl[32];     // conic c, log2(opacity)
    float4 dr[32];     // depth, red
    float4 gb[32];     // green, blue
    uint32_t id[64];
    uint32_t pm[64];   // pixels that blended the entry
    // [half of the block's pixels][pair, term][pixel]: the terms of the pair's
    // two entries (18: eight rows' 16-byte words lie in different banks)
    x2f term[2][2 * PW_TERMS][18];
};
struct __align__(16) PwRingMap : PwRing {
    float w[4][36];    // w = T alpha of the step's entries over the pixels (36: as above)
};
template <int MODE>
using PwShared = typename std::conditional<MODE == GS_MAP, PwRingMap, PwRing>::type;

// 32 x 32 bit transpose over the warp: bit p of lane e's result is bit e of
// lane p's word (five butterfly exchanges; at distance s the partners swap
// the half words of s-bit groups that belong to the other).
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const uint32_t keep_lo = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu
                                 : s == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
        const bool up = (lane & s) != 0;
        const uint32_t keep = up ? ~keep_lo : keep_lo;
        const uint32_t z = __funnelshift_l(y, y, up ? 32 - s : s);  // the partner's half into place
        x = (x & keep) | (z & ~keep);
    }
    return x;
}

// Two consecutive fragments of a warp's ring, back to front (slot s first):
// the geometry and the gradient products of both in packed pairs with the
// forward's arithmetic in every half (the same alpha), the transmittance and
// suffix recursions (Eq. 5) fragment by fragment as in back_frag.  c0, c1:
// whether the forward blended them into this pixel; a fragment that was not
// keeps the state (alpha 0: T / 1, s + 0) and adds zeros.  Writes the pair's
// terms, term k to term[18 k], and when mapping w to wcol[0] and wcol[36].
template <int MODE>
__device__ __forceinline__ void back_pair(BackState& S, const PwRing& R, int pair, bool c0, bool c1, x2f PXC,
                                          x2f PYC, float alpha_max, x2f* term, float* wcol) {
    x2f X, Y, CA, CB, CC, LOP, DEP, CR, CG, CL;
    x2_ld2(R.xy + pair, X, Y);
    x2_ld2(R.ab + pair, CA, CB);
    x2_ld2(R.cl + pair, CC, LOP);
    x2_ld2(R.dr + pair, DEP, CR);
    x2_ld2(R.gb + pair, CG, CL);
    const x2f DX = x2_sub(PXC, X), DY = x2_sub(PYC, Y);
    const x2f A = x2_fma(CB, DY, x2_mul(CA, DX));  // Q d, as quad_form
    const x2f B = x2_fma(CC, DY, x2_mul(CB, DX));
    const x2f Q = x2_fma(DX, A, x2_mul(DY, B));
    float e0, e1, cg0, cg1;
    x2_unpack(x2_fma(Q, x2_dup(R_NEG_HALF_LOG2E), LOP), e0, e1);
    const float raw0 = exp2_sfu(e0), raw1 = exp2_sfu(e1);
    x2_unpack(x2_fma(DEP, x2_dup(S.gD),
                     x2_fma(CL, x2_dup(S.gC2), x2_fma(CG, x2_dup(S.gC1), x2_mul(CR, x2_dup(S.gC0))))),
              cg0, cg1);
    const float al0 = c0 ? fminf(alpha_max, raw0) : 0.f, al1 = c1 ? fminf(alpha_max, raw1) : 0.f;
    // T / (1 - alpha) by the reciprocal instruction (at most 1 ulp) and a
    // product, as the fast division of back_frag
    const float T0 = S.T *= rcp_sfu(1.f - al0);
    const float w0 = al0 * T0;
    const float dif0 = c0 ? cg0 - S.sg : 0.f;
    S.sg = __fmaf_rn(al0, dif0, S.sg);
    const float T1 = S.T *= rcp_sfu(1.f - al1);
    const float w1 = al1 * T1;
    const float dif1 = c1 ? cg1 - S.sg : 0.f;
    S.sg = __fmaf_rn(al1, dif1, S.sg);
    // the clamp passes no gradient to opacity or shape
    const bool cl0 = raw0 > alpha_max, cl1 = raw1 > alpha_max;
    const x2f H = x2_mul(x2_pack(cl0 ? 0.f : -0.5f * w0, cl1 ? 0.f : -0.5f * w1), x2_pack(dif0, dif1));
    const x2f U = x2_mul(H, DX), V = x2_mul(H, DY);
    term[0] = x2_mul(A, H);
    term[18] = x2_mul(B, H);
    term[36] = x2_mul(U, DX);
    term[54] = x2_mul(U, DY);
    term[72] = x2_mul(V, DY);
    if (MODE == GS_MAP) {
        // dalpha/dopacity = e^(-q/2): not alpha / opacity, which an opacity
        // that rounds to 0 (blended where alpha_min is 0) does not have
        x2_unpack(x2_mul(Q, x2_dup(R_NEG_HALF_LOG2E)), e0, e1);
        term[90] = x2_pack(c0 && !cl0 ? exp2_sfu(e0) * (T0 * dif0) : 0.f, c1 && !cl1 ? exp2_sfu(e1) * (T1 * dif1) : 0.f);
        wcol[0] = w0;
        wcol[36] = w1;
    } else {
        term[90] = x2_mul(x2_pack(w0, w1), x2_dup(S.gD));
    }
}

// Backward compositing of one warp's block of a tile from the forward's
// per-pixel blend masks (warp w of the tile's): its 8x4 (or 4x8) block, or in
// tiles of at most 64 sampled pixels pixels 32 w .. 32 w + 31 in row order.
// Mask words past the run where a pixel's warp (or batch) stopped were never
// written: each lane keeps only the bits before its own last blended
// position.
//
// The warp walks its runs of 32 list entries from the last one holding an
// entry one of its pixels blended back to the first.  Per run it stages only
// those entries, one lane each (the record alone: no box, which the masks
// make unnecessary), the last first, into a ring, with the pixels that
// blended each (the run's mask words transposed over the warp).  Steps of
// four entries leave the ring whenever it holds them, across run borders
// (only the last step of a warp is padded); a lane's fragment counts when the
// forward blended it, so both passes take identical decisions by
// construction, and the alpha it recomputes is the forward's (same staged
// values, same arithmetic).
//
// The sums over the pixels go through shared memory: a lane writes each of
// its terms of a pair of entries as one 8-byte word, and a lane a (term, half
// of the block) adds that half's 16 words in packed float32 pairs, as a tree;
// the two halves then exchange an entry's partial sum each.  When mapping,
// the depth and colour sums are products of the entries' weights w with the
// pixels' image gradients: a lane a (channel, entry, half of the block) keeps
// its channel's 16 gradients in registers and reads w.
//
// Every term is formed about the Gaussian's own mean and added in float32, as
// in the kernels without masks.  Moments of h over the block, moved to the
// mean after the sum, need fewer values but lose digits: second moments about
// the block's centre (block / Gaussian)^2 of them (a Gaussian of 0.55 px: 1.6e-6
// relative at stride 1, 2e-5 at 4x4, against 1e-7), and Q sum h d in place
// of sum (Q d) h is three times as far from 64 bits on a needle.
//
// Shared memory bounds it: 107 k wavefronts an SM in 142 k cycles on the
// tracking frame, 275 k in 346 k mapping 1200x680 / 1M, at 57 and 62 %
// issue-active (48.9 M and 129 M warp instructions).  All ten mapping terms
// as eight-byte words, without the weights' part, took 257 us at 1M against
// 229.
//
// They go straight to grad2d, one atomic per (entry, field, warp): the warps
// of a tile share nothing and run as one-warp CTAs that the hardware schedules
// as they free up, heavy tiles first.
template <int DT, int MODE>
__device__ __forceinline__ void bwd_pw(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                       const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                       const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                                       const float* __restrict__ d_rgb, const float* __restrict__ d_depth,
                                       float* __restrict__ grad2d, const uint32_t* __restrict__ bmask, int tile,
                                       int w, PwShared<MODE>& R) {
    constexpr int ROWS = 2 * PW_TERMS;
    const int lane = threadIdx.x & 31;
    const int lt = w * 32 + lane;
    const bool small = g.tw * g.th <= 64;
    PixelMap m;
    if (small) {
        int i, j;
        m.inside = ep_pixel(g, tile, lt, i, j);
        m.i = i;
        m.j = j;
        m.px = i * g.sx;
        m.py = j * g.sy;
    } else {
        m = map_pixel(g, tile, lt);
    }
    const uint32_t start = ranges[2 * tile], end = ranges[2 * tile + 1];
    BackState S;
    const uint32_t own = min(back_start(cfg, g, m, t_final, last_idx, d_rgb, d_depth, S), end - start);
    const uint32_t last = __reduce_max_sync(0xffffffffu, own);
    if (last == 0u) return;  // (warp-uniform) no pixel of the block blended anything
    // this pixel's word of run r at bm[r rs]
    const uint32_t* bm = bmask + (small ? blend_mask_base_ep(tile, start) : blend_mask_base(tile, start)) + lt;
    const size_t rs = small ? 64 : (size_t)tile_threads(g);
    const int r_top = (int)((last + 31u) >> 5) - 1;
    // a run's list ids and mask word are loaded one run ahead (runs below
    // the top one are full: their 32 positions lie inside the list)
    uint32_t id_nx = r_top * 32 + lane < (int)(end - start)
                         ? __ldg(vals + start + (uint32_t)r_top * 32u + (uint32_t)lane)
                         : 0u;
    uint32_t bm_nx = __ldg(bm + (size_t)r_top * rs);
    const float pxc = (float)m.px + 0.5f, pyc = (float)m.py + 0.5f;
    const x2f PXC = x2_dup(pxc), PYC = x2_dup(pyc);
    // where the lane writes its terms, and the half row it sums: half, pair
    // and term; after the halves' exchange entry `ent` of the step
    x2f* const mine_t = &R.term[lane >> 4][0][lane & 15];
    const bool sums = lane < 2 * ROWS;
    const int half = lane >= ROWS ? 1 : 0, row = lane - half * ROWS, term = row % PW_TERMS;
    const int ent = 2 * (row / PW_TERMS) + half, partner = half ? row : row + ROWS;
    const int col = MODE == GS_MAP ? term : field_col<MODE>(term);
    const float scale = field_scale(term);
    // mapping: the lane's entry, half and channel (depth, red, green, blue) of
    // the weighted sums, and that channel's image gradients
    const int we = lane & 3, wh = (lane >> 2) & 1, wc = lane >> 3;
    float gw[16];
    if constexpr (MODE == GS_MAP) {
        R.w[0][lane] = S.gD;
        R.w[1][lane] = S.gC0;
        R.w[2][lane] = S.gC1;
        R.w[3][lane] = S.gC2;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 16; ++k) gw[k] = R.w[wc][16 * wh + k];
        __syncwarp();
    }

    // One step: slots g0 .. g0 + 3 of the ring (g0 a multiple of 4), the
    // first nv of them entries.
    auto step = [&](int g0, int nv) {
        const uint4 pm = *reinterpret_cast<const uint4*>(R.pm + g0);
        const uint32_t bit = 1u << lane;
        float* wcol = nullptr;
        if constexpr (MODE == GS_MAP) wcol = &R.w[0][lane];
        back_pair<MODE>(S, R, g0 >> 1, (pm.x & bit) != 0u, (pm.y & bit) != 0u, PXC, PYC, cfg.alpha_max, mine_t, wcol);
        back_pair<MODE>(S, R, (g0 >> 1) + 1, (pm.z & bit) != 0u, (pm.w & bit) != 0u, PXC, PYC, cfg.alpha_max,
                        mine_t + 18 * PW_TERMS, wcol + (MODE == GS_MAP ? 72 : 0));
        __syncwarp();
        float own = 0.f, other = 0.f;  // this half's sums of the entry kept and of the partner's
        if (sums) {
            const ulonglong2* t = reinterpret_cast<const ulonglong2*>(&R.term[0][0][0] + 18 * lane);
            x2f a[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 v = t[i];
                a[i] = x2_add(v.x, v.y);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < o; ++i) a[i] = x2_add(a[i], a[i + o]);
            float lo, hi;
            x2_unpack(a[0], lo, hi);
            own = half ? hi : lo;
            other = half ? lo : hi;
        }
        float wg = 0.f;
        if constexpr (MODE == GS_MAP) {
            const float4* t = reinterpret_cast<const float4*>(&R.w[we][16 * wh]);
            float a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 v = t[i];
                a[0] = i ? __fmaf_rn(v.x, gw[4 * i], a[0]) : v.x * gw[0];
                a[1] = i ? __fmaf_rn(v.y, gw[4 * i + 1], a[1]) : v.y * gw[1];
                a[2] = i ? __fmaf_rn(v.z, gw[4 * i + 2], a[2]) : v.z * gw[2];
                a[3] = i ? __fmaf_rn(v.w, gw[4 * i + 3], a[3]) : v.w * gw[3];
            }
            wg = (a[0] + a[1]) + (a[2] + a[3]);
        }
        __syncwarp();  // the next step reuses the words
        float f = own + __shfl_sync(0xffffffffu, other, partner & 31);
        if (sums && ent < nv && f != 0.f)
            atomicAdd(grad2d + (size_t)R.id[g0 + ent] * GS_GRAD2D_STRIDE + col, f * scale);
        if constexpr (MODE == GS_MAP) {
            wg += __shfl_xor_sync(0xffffffffu, wg, 4);
            if (wh == 0 && we < nv && wg != 0.f)
                atomicAdd(grad2d + (size_t)R.id[g0 + we] * GS_GRAD2D_STRIDE + (wc == 0 ? 6 : wc + 7), wg);
        }
    };

    int head = 0, tail = 0;  // entries stepped over, entries staged
#pragma unroll 1
    for (int r = r_top; r >= 0; --r) {
        // only bits before the pixel's own last blended position count
        // (this also keeps masks from another forward from sending a load
        // outside the tile's list)
        const uint32_t lim = own > (uint32_t)r * 32u ? min(32u, own - (uint32_t)r * 32u) : 0u;
        const uint32_t mine = bm_nx & (lim == 32u ? ~0u : (1u << lim) - 1u);
        const uint32_t id = id_nx;
        if (r > 0) {
            id_nx = __ldg(vals + start + (uint32_t)(r - 1) * 32u + (uint32_t)lane);
            bm_nx = __ldg(bm + (size_t)(r - 1) * rs);
        }
        // pixels that blended entry 32 r + lane
        const uint32_t pix = warp_transpose(mine);
        const unsigned mw = __ballot_sync(0xffffffffu, pix != 0u);
        if (mw == 0u) continue;
        // stage the run's blended entries, the last first
        if (pix != 0u) {
            const int slot = (tail + __popc(mw & ~((2u << lane) - 1u))) & 63;
            const Splat v = load_splat<DT>(splats, id);
            float* const xy = reinterpret_cast<float*>(R.xy + (slot >> 1)) + (slot & 1);
            float* const ab = reinterpret_cast<float*>(R.ab + (slot >> 1)) + (slot & 1);
            float* const cl = reinterpret_cast<float*>(R.cl + (slot >> 1)) + (slot & 1);
            float* const dr = reinterpret_cast<float*>(R.dr + (slot >> 1)) + (slot & 1);
            float* const gb = reinterpret_cast<float*>(R.gb + (slot >> 1)) + (slot & 1);
            xy[0] = v.x;
            xy[2] = v.y;
            ab[0] = v.ca;
            ab[2] = v.cb;
            cl[0] = v.cc;
            cl[2] = log2_opacity(v.op);
            dr[0] = v.depth;
            dr[2] = v.r;
            gb[0] = v.g;
            gb[2] = v.b;
            R.id[slot] = id;
            R.pm[slot] = pix;
        }
        tail += __popc(mw);
        __syncwarp();
        // at most 3 entries stay behind, so the next run's 32 find room beside
        // them and the four stepped over last, whose fields lanes may still read
#pragma unroll 1
        for (; tail - head >= 4; head += 4) step(head & 63, 4);
    }
    if (tail > head) {  // the last, padded step: no pixel blended the pads
        if (lane < 4 && lane >= tail - head) R.pm[(head & 63) + lane] = 0u;
        __syncwarp();
        step(head & 63, tail - head);
    }
}

// One-warp CTAs of the masked backward per SM: 24 (75 registers, mapping 80).
// us of the kernel, tracking 640x480 / 200k, 1200x680 / 458k at 2x2, mapping
// 1200x680 / 1M and 1920x1080 / 1M f16: 20 a SM 69, 63, 235 and 483; 24 69, 65,
// 224 and 457; 28 72, 67, 227 and 457.  (One float32 butterfly per two to four entries
// instead of the sums through shared memory: 85, 79, 260 and 535.)
#define PW_CTAS 24

// Warps per tile of the masked backward.
__host__ __device__ inline int pw_warps(const Grid& g) { return tile_threads(g) >> 5; }

template <int DT, int MODE>
__global__ void __launch_bounds__(32, PW_CTAS)
    k_render_bwd_pw(gs_config cfg, Grid g, const void* __restrict__ splats, const uint32_t* __restrict__ vals,
                    const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order,
                    const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                    const float* __restrict__ d_rgb, const float* __restrict__ d_depth, float* __restrict__ grad2d,
                    const uint32_t* __restrict__ bmask) {
    __shared__ PwShared<MODE> R;
    const int wpt = pw_warps(g);
    const int t = (int)blockIdx.x / wpt, w = (int)blockIdx.x % wpt;
    const int tile = order ? (int)__ldg(order + t) : t;
    bwd_pw<DT, MODE>(cfg, g, splats, vals, ranges, t_final, last_idx, d_rgb, d_depth, grad2d, bmask, tile, w, R);
}

// ---------------------------------------------------------------------------
// Entry-parallel compositing for the small tiles of downsampled frames
// ---------------------------------------------------------------------------
// With a stride of 2 in both axes or of 4 in one a tile holds at most 64
// sampled pixels but covers the same full-resolution area, hence the same
// list length, as a 16x16 tile: pixel-parallel warps would walk long lists with few (and far apart)
// pixels.  Here one CTA of W warps serves a tile (W = 8 for up to 32
// pixels, else 16) and warp w takes PPW = ceil(pixels / W) of its pixels
// (2 to 4), one at a time.  For its pixel the warp first compacts the staged
// entries whose pixel box contains it (a ballot per 32 entries, in list
// order), then lane l takes the l-th compacted entry.  Front-to-back
// compositing (Eq. 3) becomes a product scan: the transmittance before a
// valid entry is the pixel's T times the product of (1 - alpha) over the
// valid entries before it in the group of 32; the pixel stops at the first
// valid entry that would take T below t_eps.  The backward (Eq. 4, Eq. 5)
// compacts from the pixel's last blended entry back: T before an entry is T
// behind the group divided by the product of (1 - alpha) over it and the
// entries behind it, and the colour behind it is a prefix sum, so
//     dL/dalpha_k = T_k (c_k . g) - (sum_{j>k} w_j c_j . g + T_N bg . g) / (1 - alpha_k)
// with g the pixel's image gradient; each lane adds its entry's gradient to
// the tile's shared accumulators.  Entries are staged as four 16-byte arrays
// (lane l reading element l is conflict-free).

template <int NB>
struct EpStageN {
    float4 a[NB];    // x, y, conic_a, conic_b
    float4 b[NB];    // conic_c, opacity, depth, -
    float4 c[NB];    // r, g, b, -
    int4 box[NB];    // pixel box
};

template <int W>
struct EpFwdBatch {
    static constexpr int N = W == 16 ? 2 * EP_B : EP_B;
};

template <int DT, int W, int NB>
__device__ __forceinline__ void ep_stage(const void* __restrict__ splats, const uint32_t* __restrict__ ids, int n_in,
                                         float alpha_min, EpStageN<NB>& S, uint32_t* sid) {
    for (int e = threadIdx.x; e < n_in; e += W * 32) {
        const uint32_t id = __ldg(ids + e);
        const Splat v = load_splat<DT>(splats, id);
        S.a[e] = make_float4(v.x, v.y, v.ca, v.cb);
        S.b[e] = make_float4(v.cc, v.op, v.depth, log2_opacity(v.op));
        float t2;
        S.box[e] = pixel_box(v, alpha_min, t2);
        S.c[e] = make_float4(v.r, v.g, v.b, 0.f);
        if (sid) sid[e] = id;
    }
}

// Whether staged entry e can blend at full-resolution pixel (px, py): inside
// its pixel box (a superset of the fragments the alpha test accepts, so
// compacting by it changes no result).  Testing the alpha ellipse here as
// well was measured slower: the extra loads cost more than the groups saved.
template <int NB>
__device__ __forceinline__ bool ep_may_blend(const EpStageN<NB>& S, int e, int px, int py) {
    const int4 box = S.box[e];
    return px >= box.x && px <= box.y && py >= box.z && py <= box.w;
}


// Pixel-to-warp assignment of a tile (the pairing of Sec. 5.2's workload
// scheduling unit): the tile's npix = W * ppw pixels are ranked by their
// expected work h (heaviest first, ties by index) and dealt to the W warps
// in snake order, round r going to warps 0..W-1 for even r and W-1..0 for
// odd r, so each warp gets a heavy pixel with a light one in every pair of
// rounds.  h is the pixel's list position of the last blended entry (the
// backward's input, or the previous iteration's for the forward); pixels
// outside the image have h = 0.  perm[w * ppw + j] is warp w's j-th pixel.
// Any h gives a valid permutation; it only changes which warp does what.
template <int W>
__device__ __forceinline__ void ep_pair(const Grid& g, int tile, int npix, const uint32_t* hint,
                                        uint32_t* s_h, uint8_t* perm) {
    const int ppw = (npix + W - 1) / W;
    const int q = (int)threadIdx.x;
    if (q < npix) {
        int i, j;
        uint32_t h = 0;
        if (hint && ep_pixel(g, tile, q, i, j)) h = hint[(size_t)j * g.Ws + i];
        s_h[q] = h;
    }
    __syncthreads();
    if (q < npix) {
        const uint32_t h = s_h[q];
        int r = 0;
        for (int o = 0; o < npix; ++o) {
            const uint32_t v = s_h[o];
            r += (v > h || (v == h && o < q)) ? 1 : 0;
        }
        const int round = r / W, pos = r % W;
        const int w = (round & 1) ? W - 1 - pos : pos;
        perm[w * ppw + round] = (uint8_t)q;
    }
    __syncthreads();
}

// Forward compositing of the pixels of `tile` by the CTA's W warps,
// entry-parallel (S: staging; cbuf_all: W compaction buffers).
template <int DT, int W, int NB>
__device__ __forceinline__ void fwd_ep(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                       const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                       const FwdOut& O, int tile, EpStageN<NB>& S,
                                       int (*cbuf_all)[64], uint32_t* s_h, uint8_t* perm,
                                       uint32_t (*bm_all)[NB / 32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    int* cbuf = cbuf_all[warp];
    const int npix = g.tw * g.th, ppw = (npix + W - 1) / W;
    const uint32_t start = ranges[2 * tile], end = ranges[2 * tile + 1];
    // out_last still holds the previous iteration's positions (read before any write)
    ep_pair<W>(g, tile, npix, cfg.balance ? O.last : nullptr, s_h, perm);
    // lane j < ppw holds the state of the warp's pixel j
    int mi, mj;
    const bool mine = lane < ppw && warp * ppw + lane < npix && ep_pixel(g, tile, perm[warp * ppw + lane], mi, mj);
    float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f, D = 0.f;
    uint32_t last = 0, nb = 0;
    bool done = !mine;
    uint32_t* bmw = bm_all[warp];  // the pixel's blend mask over the batch
    const size_t bm_tile = blend_mask_base_ep(tile, start);
    for (uint32_t b = start; b < end; b += NB) {
        if (__syncthreads_count(!done) == 0) break;
        const int n_in = (int)min((uint32_t)NB, end - b);
        ep_stage<DT, W, NB>(splats, vals + b, n_in, cfg.alpha_min, S, nullptr);
        __syncthreads();
        for (int j = 0; j < ppw; ++j) {
            if (__shfl_sync(0xffffffffu, done, j)) continue;
            int pi, pj;
            ep_pixel(g, tile, perm[warp * ppw + j], pi, pj);
            const int px = pi * g.sx, py = pj * g.sy;
            const float pxc = (float)px + 0.5f, pyc = (float)py + 0.5f;
            float Tj = __shfl_sync(0xffffffffu, T, j);
            float p0 = 0.f, p1 = 0.f, p2 = 0.f, pd = 0.f;
            uint32_t lastj = 0, nbj = 0;
            bool stopped = false;
            if (O.bmask) {
                if (lane < NB / 32) bmw[lane] = 0u;
                __syncwarp();
            }
            // composite the k compacted entries cbuf[0, k), in list order
            auto composite = [&](int k) {
                const int e = lane < k ? cbuf[lane] : -1;
                float alpha = -1.f;
                if (e >= 0) {
                    const float4 A = S.a[e];
                    const float4 Bv = S.b[e];
                    const Quad Qd = quad_form(A.z, A.w, Bv.x, pxc - A.x, pyc - A.y);
                    const float al = fminf(cfg.alpha_max, raw_alpha(Qd.q, Bv.w));
                    if (!(Qd.q < 0.f)) alpha = al;
                }
                const bool valid = alpha >= cfg.alpha_min;
                if (__ballot_sync(0xffffffffu, valid) == 0u) return;
                const float f = valid ? 1.f - alpha : 1.f;
                float P = f;  // inclusive product over lanes 0..l
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float y = __shfl_up_sync(0xffffffffu, P, o);
                    if (lane >= o) P *= y;
                }
                float Tb = __shfl_up_sync(0xffffffffu, P, 1);  // T before this entry
                Tb = lane == 0 ? Tj : Tj * Tb;
                const float Tn = Tb * f;
                const unsigned stop = __ballot_sync(0xffffffffu, valid && Tn < cfg.t_eps);
                const int lstar = stop ? __ffs(stop) - 1 : 32;
                const bool ok = valid && lane < lstar;
                if (ok) {
                    const float w = alpha * Tb;
                    const float4 Cc = S.c[e];
                    p0 += w * Cc.x;
                    p1 += w * Cc.y;
                    p2 += w * Cc.z;
                    pd += w * S.b[e].z;
                }
                const unsigned okm = __ballot_sync(0xffffffffu, ok);
                nbj += __popc(okm);
                if (O.bmask && ok) atomicOr(&bmw[e >> 5], 1u << (e & 31));
                const int ehi = __shfl_sync(0xffffffffu, e, okm ? 31 - __clz(okm) : 0);
                if (okm) lastj = b - start + (uint32_t)ehi + 1u;
                if (lstar < 32) {
                    Tj = __shfl_sync(0xffffffffu, Tb, lstar);
                    stopped = true;
                } else {
                    Tj = __shfl_sync(0xffffffffu, Tn, 31);
                }
            };
            int cnt = 0;
            for (int c = 0; c < n_in && !stopped; c += 32) {
                const int e = c + lane;
                const bool in = e < n_in && ep_may_blend(S, e, px, py);
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (in) cbuf[cnt + __popc(m & lt_mask)] = e;
                cnt += __popc(m);
                __syncwarp();
                if (cnt >= 32) {
                    composite(32);
                    const int rest = cnt - 32;
                    const int v = lane < rest ? cbuf[32 + lane] : 0;
                    __syncwarp();
                    if (lane < rest) cbuf[lane] = v;
                    __syncwarp();
                    cnt = rest;
                }
            }
            if (!stopped && cnt > 0) composite(cnt);
            __syncwarp();
            if (O.bmask && lane < ((n_in + 31) >> 5))
                O.bmask[bm_tile + 64 * (size_t)(((b - start) >> 5) + lane) + perm[warp * ppw + j]] = bmw[lane];
            p0 = warp_sum(p0);
            p1 = warp_sum(p1);
            p2 = warp_sum(p2);
            pd = warp_sum(pd);
            if (lane == j) {
                C0 += p0;
                C1 += p1;
                C2 += p2;
                D += pd;
                T = Tj;
                if (lastj) last = lastj;
                nb += nbj;
                done = stopped;
            }
        }
        __syncthreads();
    }
    float lpart = 0.f;
    if (mine) lpart = write_pixel(cfg, g, O, mi, mj, C0, C1, C2, D, T, last, nb);
    add_loss(O, lpart);
}

// (the batch length decides the summation order, the number of warps does not)
template <int W, int NB = EpFwdBatch<W>::N>
struct EpFwdSmem {
    EpStageN<NB> S;
    int cbuf[W][64];
    uint32_t s_h[64];
    uint8_t perm[64];
    uint32_t bm[W][NB / 32];
};

template <int DT, int W, int NB = EpFwdBatch<W>::N>
__device__ __forceinline__ void fwd_ep_cta(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                           const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                           const uint32_t* __restrict__ order, const FwdOut& O, int blk) {
    extern __shared__ __align__(16) unsigned char r_smem[];
    EpFwdSmem<W, NB>& M = *reinterpret_cast<EpFwdSmem<W, NB>*>(r_smem);
    const int tile = order ? (int)__ldg(order + blk) : blk;
    fwd_ep<DT, W, NB>(cfg, g, splats, vals, ranges, O, tile, M.S, M.cbuf, M.s_h, M.perm, M.bm);
}

template <int DT, int W>
__global__ void __launch_bounds__(W * 32, W == 8 ? 4 : 2)
    k_render_fwd_ep(gs_config cfg, Grid g, const void* __restrict__ splats, const uint32_t* __restrict__ vals,
                    const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order, FwdOut O) {
    fwd_ep_cta<DT, W>(cfg, g, splats, vals, ranges, order, O, (int)blockIdx.x);
}

// Fields merged per entry: GS_TRACK du dv dA dB dC dd, GS_MAP du dv dA dB dC
// dop dd dr dg db; ep_col gives their grad2d columns.
template <int MODE>
struct EpFields {
    static constexpr int N = MODE == GS_MAP ? 10 : 6;
};
template <int MODE>
__device__ __forceinline__ int ep_col(int f) {
    if (MODE == GS_MAP) return f < 7 ? f : f + 1;
    return f < 5 ? f : 6;
}

// Shared memory of the entry-parallel backward (batches of NB entries;
// dynamic: above 48 KB for 16 warps and 512 entries).
template <int MODE, int W, int NB = EpFwdBatch<W>::N>
struct EpBwdSmem {
    EpStageN<NB> S;
    uint32_t sid[NB];
    float acc[EpFields<MODE>::N][NB];
    int cbuf[W][64];
    uint32_t s_h[64];
    uint8_t perm[64];
    uint32_t s_max;
};

// Backward compositing of the pixels of `tile` by the CTA's W warps,
// entry-parallel.  MASKED: from the forward's blend masks (a test inside the
// loops cost the other form 1 to 5 %).
template <int DT, int MODE, int W, bool MASKED>
__device__ __forceinline__ void bwd_ep(const gs_config& cfg, const Grid& g, const void* __restrict__ splats,
                                       const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                       const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                                       const float* __restrict__ d_rgb, const float* __restrict__ d_depth,
                                       float* __restrict__ grad2d, const uint32_t* __restrict__ bmask, int tile,
                                       EpBwdSmem<MODE, W>& M) {
    constexpr int NF = EpFields<MODE>::N;
    constexpr int NB = EpFwdBatch<W>::N;
    EpStageN<NB>& S = M.S;
    uint32_t* sid = M.sid;
    float(&acc)[NF][NB] = M.acc;
    uint32_t& s_max = M.s_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned gt_mask = lane == 31 ? 0u : ~0u << (lane + 1);
    int* cbuf = M.cbuf[warp];
    const int npix = g.tw * g.th, ppw = (npix + W - 1) / W;
    const uint32_t start = ranges[2 * tile], end = ranges[2 * tile + 1];
    uint8_t* perm = M.perm;
    ep_pair<W>(g, tile, npix, last_idx, M.s_h, perm);
    int mi, mj;
    const bool mine = lane < ppw && warp * ppw + lane < npix && ep_pixel(g, tile, perm[warp * ppw + lane], mi, mj);
    // state of pixel `lane`: T after the part already walked, the colour
    // behind it dotted with g, last blended position, image gradient g
    float T = 1.f, sdot = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, gd = 0.f;
    uint32_t last = 0;
    if (mine) {
        const size_t P = (size_t)g.Ws * g.Hs;
        const size_t pix = (size_t)mj * g.Ws + mi;
        T = t_final[pix];
        last = min(last_idx[pix], end - start);
        g0 = d_rgb[pix];
        g1 = d_rgb[P + pix];
        g2 = d_rgb[2 * P + pix];
        gd = d_depth[pix];
        sdot = T * (cfg.bg[0] * g0 + cfg.bg[1] * g1 + cfg.bg[2] * g2);
    }
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    uint32_t wl = last;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wl = max(wl, __shfl_xor_sync(0xffffffffu, wl, o));
    if (lane == 0) atomicMax(&s_max, wl);
    __syncthreads();
    const uint32_t tile_last = s_max;
    const uint32_t* bm_tile = MASKED ? bmask + blend_mask_base_ep(tile, start) : nullptr;
    // batches [start + k NB, start + (k + 1) NB) from the last one holding a
    // blended entry back to the first
    for (int kb = (int)((tile_last + NB - 1) / NB) - 1; kb >= 0; --kb) {
        const uint32_t lo = start + (uint32_t)kb * NB, hi = start + min(tile_last, (uint32_t)(kb + 1) * NB);
        const int n_in = (int)(hi - lo);
        ep_stage<DT, W, NB>(splats, vals + lo, n_in, cfg.alpha_min, S, sid);
        for (int q = threadIdx.x; q < NF * NB; q += W * 32) (&acc[0][0])[q] = 0.f;
        __syncthreads();
        const uint32_t base_pos = lo - start;
        for (int j = 0; j < ppw; ++j) {
            const uint32_t lastj = __shfl_sync(0xffffffffu, last, j);
            if (lastj <= base_pos) continue;  // nothing blended in this batch
            const int nj = (int)min((uint32_t)n_in, lastj - base_pos);
            const int qj = perm[warp * ppw + j];  // the pixel's index in the tile
            int pi, pj;
            ep_pixel(g, tile, qj, pi, pj);
            const int px = pi * g.sx, py = pj * g.sy;
            const float pxc = (float)px + 0.5f, pyc = (float)py + 0.5f;
            // the pixel's blend mask from the forward (entries it blended),
            // else its pixel box, selects the entries to compact
            const uint32_t* bmj = MASKED ? bm_tile + 64 * (size_t)(base_pos >> 5) + qj : nullptr;
            // (lane r takes run r's word, at most 32 a batch: a load a run in
            // the loop below waits for each; 300 tiles of 32 pixels, 50k / 200k
            // Gaussians 47.8 / 68.7 us, now 35.0 / 52.3)
            const uint32_t mw = MASKED && lane < ((nj + 31) >> 5) ? __ldg(bmj + 64 * lane) : 0u;
            float Tj = __shfl_sync(0xffffffffu, T, j);
            float sj = __shfl_sync(0xffffffffu, sdot, j);
            // the pixel's image gradient
            const float h0 = __shfl_sync(0xffffffffu, g0, j), h1 = __shfl_sync(0xffffffffu, g1, j);
            const float h2 = __shfl_sync(0xffffffffu, g2, j), hd = __shfl_sync(0xffffffffu, gd, j);
            // the k compacted entries cbuf[0, k), last first: lane l's entry
            // has the entries of lanes < l behind it
            auto differentiate = [&](int k) {
                const int e = lane < k ? cbuf[lane] : -1;
                float4 Bv = make_float4(0.f, 0.f, 0.f, 0.f), Cc = Bv;
                float dx = 0.f, dy = 0.f, raw = 0.f, alpha = -1.f;
                Quad Qd = {0.f, 0.f, 0.f};
                bool valid = false;
                if (e >= 0) {
                    const float4 A = S.a[e];
                    Bv = S.b[e];
                    Cc = S.c[e];
                    dx = pxc - A.x;
                    dy = pyc - A.y;
                    Qd = quad_form(A.z, A.w, Bv.x, dx, dy);
                    raw = raw_alpha(Qd.q, Bv.w);
                    alpha = fminf(cfg.alpha_max, raw);
                    valid = !(Qd.q < 0.f) && !(alpha < cfg.alpha_min);
                }
                if (__ballot_sync(0xffffffffu, valid) == 0u) return;
                const float f = valid ? 1.f - alpha : 1.f;
                float Q = f;  // inclusive product over lanes 0..l (this entry and those behind it)
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float y = __shfl_up_sync(0xffffffffu, Q, o);
                    if (lane >= o) Q *= y;
                }
                const float Tb = __fdividef(Tj, Q);  // T before this entry (Eq. 5)
                const float w = valid ? alpha * Tb : 0.f;
                const float cg = Cc.x * h0 + Cc.y * h1 + Cc.z * h2 + Bv.z * hd;
                const float wcg = w * cg;
                float Sin = wcg;  // inclusive prefix sum of w (c . g)
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float y = __shfl_up_sync(0xffffffffu, Sin, o);
                    if (lane >= o) Sin += y;
                }
                if (valid) {
                    const float behind = sj + (Sin - wcg);
                    const float dLda = Tb * cg - __fdividef(behind, f);
                    float ga[NF];
#pragma unroll
                    for (int q = 0; q < NF; ++q) ga[q] = 0.f;
                    if (MODE == GS_MAP) {
                        ga[6] = w * hd;
                        ga[7] = w * h0;
                        ga[8] = w * h1;
                        ga[9] = w * h2;
                    } else {
                        ga[5] = w * hd;
                    }
                    if (!(raw > cfg.alpha_max)) {  // the clamp passes no gradient
                        if (MODE == GS_MAP) ga[5] = exp2_sfu(__fmul_rn(Qd.q, R_NEG_HALF_LOG2E)) * dLda;
                        const float dp = alpha * dLda;
                        ga[2] = -0.5f * dx * dx * dp;
                        ga[3] = -dx * dy * dp;
                        ga[4] = -0.5f * dy * dy * dp;
                        ga[0] = Qd.a * dp;
                        ga[1] = Qd.b * dp;
                    }
#pragma unroll
                    for (int q = 0; q < NF; ++q)
                        if (ga[q] != 0.f) atomicAdd(&acc[q][e], ga[q]);
                }
                // state in front of these entries
                Tj = __shfl_sync(0xffffffffu, __fdividef(Tj, Q), 31);
                sj = sj + __shfl_sync(0xffffffffu, Sin, 31);
            };
            int cnt = 0;
            for (int c = (nj - 1) & ~31; c >= 0; c -= 32) {
                const int e = c + lane;
                const uint32_t word = MASKED ? __shfl_sync(0xffffffffu, mw, c >> 5) : 0u;
                const bool in = e < nj && (MASKED ? ((word >> lane) & 1u) != 0u : ep_may_blend(S, e, px, py));
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (in) cbuf[cnt + __popc(m & gt_mask)] = e;
                cnt += __popc(m);
                __syncwarp();
                if (cnt >= 32) {
                    differentiate(32);
                    const int rest = cnt - 32;
                    const int v = lane < rest ? cbuf[32 + lane] : 0;
                    __syncwarp();
                    if (lane < rest) cbuf[lane] = v;
                    __syncwarp();
                    cnt = rest;
                }
            }
            if (cnt > 0) differentiate(cnt);
            __syncwarp();
            if (lane == j) {
                T = Tj;
                sdot = sj;
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < n_in; e += W * 32) {
            float* dst = grad2d + (size_t)sid[e] * GS_GRAD2D_STRIDE;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                const float v = acc[k][e];
                if (v != 0.f) atomicAdd(dst + ep_col<MODE>(k), v);
            }
        }
        __syncthreads();
    }
}

template <int DT, int MODE, int W, bool MASKED>
__global__ void __launch_bounds__(W * 32, W == 8 ? 4 : 2)
    k_render_bwd_ep(gs_config cfg, Grid g, const void* __restrict__ splats, const uint32_t* __restrict__ vals,
                    const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order,
                    const float* __restrict__ t_final, const uint32_t* __restrict__ last_idx,
                    const float* __restrict__ d_rgb, const float* __restrict__ d_depth,
                    float* __restrict__ grad2d, const uint32_t* __restrict__ bmask) {
    extern __shared__ __align__(16) unsigned char r_smem[];
    EpBwdSmem<MODE, W>& M = *reinterpret_cast<EpBwdSmem<MODE, W>*>(r_smem);
    const int tile = order ? (int)__ldg(order + blockIdx.x) : (int)blockIdx.x;
    bwd_ep<DT, MODE, W, MASKED>(cfg, g, splats, vals, ranges, t_final, last_idx, d_rgb, d_depth, grad2d, bmask, tile,
                                M);
}

// ---------------------------------------------------------------------------
// Multi-session waves: forward compositing with the loss and backward
// compositing (GS_TRACK) over every job of a wave, one launch per kernel form
// ---------------------------------------------------------------------------
struct WaveFwdJob {
    Grid g;
    const void* splats;
    const uint32_t* vals;
    const uint32_t* ranges;
    const uint32_t* order;
    FwdOut O;
    int kind;  // wave_render's fwd_kind
};

template <int NW, int CT>
__global__ void __launch_bounds__(R_THREADS, CT)
    k_wave_render_fwd(const gs_config cfg, const __grid_constant__ Wave<WaveFwdJob> W) {
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveFwdJob& J = W.job[j];
    fwd_cta<GS_F32, NW>(cfg, J.g, J.splats, J.vals, J.ranges, J.order, J.O, (int)blockIdx.x - W.start[j]);
}

template <int NW>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 4 : 2)
    k_wave_render_fwd_ep(const gs_config cfg, const __grid_constant__ Wave<WaveFwdJob> W) {
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveFwdJob& J = W.job[j];
    fwd_ep_cta<GS_F32, NW>(cfg, J.g, J.splats, J.vals, J.ranges, J.order, J.O, (int)blockIdx.x - W.start[j]);
}

// Jobs of several forms in one launch, so that they fill each other's tails
// (a wave of six sessions of five forms: 187 us, 246 in five launches).
__global__ void __launch_bounds__(R_THREADS, 4)
    k_wave_render_fwd_mix(const gs_config cfg, const __grid_constant__ Wave<WaveFwdJob> W) {
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveFwdJob& J = W.job[j];
    const int blk = (int)blockIdx.x - W.start[j];
    switch (J.kind) {
        case 0: fwd_cta<GS_F32, 8>(cfg, J.g, J.splats, J.vals, J.ranges, J.order, J.O, blk); break;
        case 1: fwd_cta<GS_F32, 4>(cfg, J.g, J.splats, J.vals, J.ranges, J.order, J.O, blk); break;
        case 2: fwd_ep_cta<GS_F32, 8>(cfg, J.g, J.splats, J.vals, J.ranges, J.order, J.O, blk); break;
        default: fwd_ep_cta<GS_F32, 8, EpFwdBatch<16>::N>(cfg, J.g, J.splats, J.vals, J.ranges, J.order, J.O, blk); break;
    }
}

struct WaveBwdJob {
    Grid g;
    const void* splats;
    const uint32_t* vals;
    const uint32_t* ranges;
    const uint32_t* order;
    const float* t_final;
    const uint32_t* last_idx;
    const float* d_rgb;
    const float* d_depth;
    float* grad2d;
    const uint32_t* bmask;
    int B;
};

template <int KST>
__global__ void __launch_bounds__(R_THREADS, KST == 1 ? 4 : 2)
    k_wave_render_bwd(const gs_config cfg, const __grid_constant__ Wave<WaveBwdJob> W) {
    extern __shared__ __align__(16) unsigned char r_smem[];
    __shared__ uint32_t s_max_all[R_THREADS / 32];
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveBwdJob& J = W.job[j];
    const Group G = make_group(J.g, J.order, J.B, (int)blockIdx.x - W.start[j]);
    if (G.tile < 0) return;
    bwd_pp<GS_F32, GS_TRACK, KST>(cfg, J.g, J.splats, J.vals, J.ranges, J.t_final, J.last_idx, J.d_rgb, J.d_depth,
                                  J.grad2d, G, r_smem, s_max_all);
}

// Jobs with blend masks: one-warp CTAs over (job, tile, warp).
__global__ void __launch_bounds__(32, PW_CTAS) k_wave_render_bwd_pw(const gs_config cfg,
                                                                const __grid_constant__ Wave<WaveBwdJob> W) {
    __shared__ PwRing R;
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveBwdJob& J = W.job[j];
    const int blk = (int)blockIdx.x - W.start[j];
    const int wpt = pw_warps(J.g);
    const int t = blk / wpt, w = blk % wpt;
    const int tile = J.order ? (int)__ldg(J.order + t) : t;
    bwd_pw<GS_F32, GS_TRACK>(cfg, J.g, J.splats, J.vals, J.ranges, J.t_final, J.last_idx, J.d_rgb, J.d_depth,
                                 J.grad2d, J.bmask, tile, w, R);
}

template <int NW>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 4 : 2)
    k_wave_render_bwd_ep(const gs_config cfg, const __grid_constant__ Wave<WaveBwdJob> W) {
    extern __shared__ __align__(16) unsigned char r_smem[];
    EpBwdSmem<GS_TRACK, NW>& M = *reinterpret_cast<EpBwdSmem<GS_TRACK, NW>*>(r_smem);
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveBwdJob& J = W.job[j];
    const int blk = (int)blockIdx.x - W.start[j];
    const int tile = J.order ? (int)__ldg(J.order + blk) : blk;
    if (J.bmask)
        bwd_ep<GS_F32, GS_TRACK, NW, true>(cfg, J.g, J.splats, J.vals, J.ranges, J.t_final, J.last_idx, J.d_rgb,
                                           J.d_depth, J.grad2d, J.bmask, tile, M);
    else
        bwd_ep<GS_F32, GS_TRACK, NW, false>(cfg, J.g, J.splats, J.vals, J.ranges, J.t_final, J.last_idx, J.d_rgb,
                                            J.d_depth, J.grad2d, nullptr, tile, M);
}

}  // namespace gs

using namespace gs;

// Entries a tile stages per batch: R_BATCH, halved while the CTA's tiles
// would need more than `budget` bytes of shared memory.
static int group_batch(int gpc, int bytes_per_entry, int budget) {
    int B = R_BATCH;
    while (B > 32 && gpc * B * bytes_per_entry > budget) B >>= 1;
    return B;
}

// Raises a kernel's dynamic shared-memory limit once per device and
// instantiation (not repeated while a graph is being captured).
static gs_status smem_once(const void* fn, int id, int bytes) {
    static bool done[64][64] = {};  // ids: bwd 6-17, entry-parallel bwd 18-33 (masked 46-61), waves 42-45
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && done[dev][id]) return GS_OK;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
        return set_error(GS_ERR_CUDA, "cudaFuncSetAttribute(render kernel %d)", id);
    if (dev >= 0 && dev < 64) done[dev][id] = true;
    return GS_OK;
}

// Kernel choice per frame.  Forward: tiles of at most 64 pixels (downsampled
// frames) entry-parallel, larger ones pixel-parallel.  (The pixel-parallel
// kernel does less work on large grids of small tiles too -- stride 2x2,
// 100k Gaussians, 300 tiles 117 against 38 us, 1200 62 / 62, 3225 44 / 146 --
// but its products and sums round differently, which moves stops and the
// signs of L1 residuals.)
// Backward with masks, for which both kernels form the same float32 terms: the
// one-warp CTAs do less work, the entry-parallel kernel's 8 or 16 warps a tile
// finish it sooner, which counts while the tiles do not fill the chip.
// One-warp against entry-parallel, us (200k Gaussians; 50k and 600k cross at the
// same numbers of tiles):
//   stride 2x2   384 tiles 72 / 49,  638 63 / 50,  800 62 / 56, 1000 57 / 66
//   stride 4x2  1200 tiles 56 / 44, 1600 58 / 50, 1920 55 / 59, 2160 51 / 63
//   stride 4x4  1200 tiles 49 / 29, 1920 47 / 38, 2160 46 / 41, 2640 45 / 47
static bool fwd_entry_parallel(const Grid& g) { return g.tw * g.th <= 64; }
// On tiles of 64 pixels, lists of a few dozen entries leave the entry-parallel
// kernel's 16 warps a tile without work, and its CTAs, two an SM, go in rounds
// (300 tiles: 1000 Gaussians 4.7 / 10.5, 4000 8.1 / 11.6, 8000 14.1 / 12.9, 16000 26.5
// / 18.3; 638 tiles: 16000 18.5 / 29.0, 50k 41 / 37): it takes 24 Gaussians a tile
// and round.
// tiles, n: of the launch
static bool bwd_entry_parallel(const Grid& g, bool masks, int tiles, int64_t n) {
    const int pixels = g.tw * g.th;
    if (pixels > 64 || !masks) return pixels <= 64;
    if (pixels < 64) return tiles < (pixels == 32 ? 1792 : 2560);
    const int round = 2 * num_sms();
    return tiles < 896 && n >= (int64_t)24 * tiles * ((tiles + round - 1) / round);
}

template <int DT>
static gs_status launch_fwd(const gs_config& cfg, const Grid& g, const void* splats, const uint32_t* vals,
                            const uint32_t* ranges, const uint32_t* order, const FwdOut& O, cudaStream_t st) {
    const int ntiles = g.TX * g.TY;
    if (fwd_entry_parallel(g)) {
        if (g.tw * g.th <= 32)
            k_render_fwd_ep<DT, 8><<<ntiles, 8 * 32, sizeof(EpFwdSmem<8>), st>>>(cfg, g, splats, vals, ranges, order, O);
        else
            k_render_fwd_ep<DT, 16><<<ntiles, 16 * 32, sizeof(EpFwdSmem<16>), st>>>(cfg, g, splats, vals, ranges, order, O);
        return check_launch("k_render_fwd_ep");
    }
    const int nw = tile_threads(g) / 32, gpc = 8 / nw;
    const unsigned nt = (unsigned)((ntiles + gpc - 1) / gpc);
#define GS_FWD(NW, CT) \
    k_render_fwd<DT, NW, CT><<<nt, R_THREADS, sizeof(FwdSmem<NW>), st>>>(cfg, g, splats, vals, ranges, order, O)
    if (nw == 8 && fwd_three(nt)) GS_FWD(8, 3);
    else if (nw == 8) GS_FWD(8, 4);
    else GS_FWD(4, 3);
#undef GS_FWD
    return check_launch("k_render_fwd");
}

static gs_status dispatch_fwd(const gs_config& cfg, const Grid& g, int rec_dtype, const void* splats,
                              const uint32_t* vals, const uint32_t* ranges, const uint32_t* order, const FwdOut& O,
                              cudaStream_t st) {
    if (rec_dtype == GS_F32) return launch_fwd<GS_F32>(cfg, g, splats, vals, ranges, order, O, st);
    if (rec_dtype == GS_BF16) return launch_fwd<GS_BF16>(cfg, g, splats, vals, ranges, order, O, st);
    return launch_fwd<GS_F16>(cfg, g, splats, vals, ranges, order, O, st);
}

template <int DT, int MD>
static gs_status launch_bwd(const gs_config& cfg, const Grid& g, const void* splats, const uint32_t* vals,
                            const uint32_t* ranges, const uint32_t* order, const float* t_final,
                            const uint32_t* last_idx, const float* d_rgb, const float* d_depth, float* grad2d,
                            const uint32_t* bmask, int64_t n, cudaStream_t st) {
    const int ntiles = g.TX * g.TY;
    if (bmask && !bwd_entry_parallel(g, true, ntiles, n)) {  // one-warp CTAs
        k_render_bwd_pw<DT, MD><<<(unsigned)ntiles * (unsigned)pw_warps(g), 32, 0, st>>>(
            cfg, g, splats, vals, ranges, order, t_final, last_idx, d_rgb, d_depth, grad2d, bmask);
        return check_launch("k_render_bwd_pw");
    }
    if (bwd_entry_parallel(g, bmask != nullptr, ntiles, n)) {
        gs_status s;
        const int id = (bmask ? 46 : 18) + 4 * (MD == GS_MAP) + DT;  // + 0 or 8 below: W
#define GS_EP(W, M)                                                                                             \
    {                                                                                                           \
        const int sm = (int)sizeof(EpBwdSmem<MD, W>);                                                           \
        if ((s = smem_once((const void*)k_render_bwd_ep<DT, MD, W, M>, W == 8 ? id : id + 8, sm)) != GS_OK)     \
            return s;                                                                                           \
        k_render_bwd_ep<DT, MD, W, M><<<ntiles, W * 32, sm, st>>>(cfg, g, splats, vals, ranges, order, t_final, \
                                                                   last_idx, d_rgb, d_depth, grad2d, bmask);    \
    }
        if (g.tw * g.th <= 32) { if (bmask) GS_EP(8, true) else GS_EP(8, false) }
        else { if (bmask) GS_EP(16, true) else GS_EP(16, false) }
#undef GS_EP
        return check_launch("k_render_bwd_ep");
    }
    const int gpc = R_THREADS / tile_threads(g);
    const unsigned nt = (unsigned)((ntiles + gpc - 1) / gpc);
    const int per_entry = (int)(sizeof(StagedSplat) + sizeof(uint32_t) + sizeof(float) * Fields<MD>::N);
    const int B = group_batch(gpc, per_entry, R_BWD_SMEM);
    const size_t smem = (size_t)gpc * B * per_entry;
    const int id = 6 + 6 * (MD == GS_MAP) + 2 * DT;
    gs_status s;
    if (gpc == 1) {
        if ((s = smem_once((const void*)k_render_bwd<DT, MD, 1>, id, R_BWD_SMEM)) != GS_OK) return s;
        k_render_bwd<DT, MD, 1><<<nt, R_THREADS, smem, st>>>(cfg, g, splats, vals, ranges, order, t_final,
                                                             last_idx, d_rgb, d_depth, grad2d, B);
    } else {
        if ((s = smem_once((const void*)k_render_bwd<DT, MD, 4>, id + 1, R_BWD_SMEM)) != GS_OK) return s;
        k_render_bwd<DT, MD, 4><<<nt, R_THREADS, smem, st>>>(cfg, g, splats, vals, ranges, order, t_final,
                                                             last_idx, d_rgb, d_depth, grad2d, B);
    }
    return check_launch("k_render_bwd");
}

static gs_status render_checks(const gs_config* cfg, const gs_camera* cam, int rec_dtype, const void* splats,
                               int64_t n) {
    if (!cfg) return set_error(GS_ERR_INVALID_ARG, "config is NULL");
    if (!cam) return set_error(GS_ERR_INVALID_ARG, "camera is NULL");
    if (cam->width <= 0 || cam->height <= 0 || cam->sx < 1 || cam->sy < 1 || cam->width > (1 << 20) ||
        cam->height > (1 << 20))
        return set_error(GS_ERR_INVALID_ARG, "bad camera size or stride");
    if (rec_dtype != GS_F32 && rec_dtype != GS_BF16 && rec_dtype != GS_F16)
        return set_error(GS_ERR_INVALID_ARG, "bad record dtype %d", rec_dtype);
    if (n < 0) return set_error(GS_ERR_INVALID_ARG, "bad Gaussian count");
    if (n > 0 && (!splats || ((uintptr_t)splats & 15)))
        return set_error(GS_ERR_INVALID_ARG, "splats NULL or not 16-byte aligned");
    return GS_OK;
}

extern "C" gs_status gs_render_fwd(const gs_config* cfg, const gs_camera* cam, int rec_dtype, const void* splats,
                                   int64_t n, const uint32_t* vals, const uint32_t* tile_ranges,
                                   const uint32_t* tile_order, float* rgb, float* depth, float* t_final,
                                   uint32_t* last_idx, uint32_t* n_blended, uint32_t* blend_masks,
                                   gs_stream stream) {
    gs_status s;
    if ((s = render_checks(cfg, cam, rec_dtype, splats, n)) != GS_OK) return s;
    if (!tile_ranges || !rgb || !depth || !t_final || !last_idx)
        return set_error(GS_ERR_INVALID_ARG, "an image or range pointer is NULL");
    const FwdOut O = {rgb, depth, t_final, last_idx, n_blended, nullptr, nullptr, nullptr, nullptr, nullptr,
                      blend_masks};
    return dispatch_fwd(*cfg, make_grid(*cam), rec_dtype, splats, vals, tile_ranges, tile_order, O,
                        (cudaStream_t)stream);
}

extern "C" gs_status gs_render_fwd_loss(const gs_config* cfg, const gs_camera* cam, int rec_dtype,
                                        const void* splats, int64_t n, const uint32_t* vals,
                                        const uint32_t* tile_ranges, const uint32_t* tile_order, float* rgb,
                                        float* depth, float* t_final, uint32_t* last_idx, uint32_t* n_blended,
                                        uint32_t* blend_masks, const float* target_rgb, const float* target_depth,
                                        float* d_rgb, float* d_depth, double* loss_out, gs_stream stream) {
    gs_status s;
    if ((s = render_checks(cfg, cam, rec_dtype, splats, n)) != GS_OK) return s;
    if (!tile_ranges || !rgb || !depth || !t_final || !last_idx)
        return set_error(GS_ERR_INVALID_ARG, "an image or range pointer is NULL");
    if (!target_rgb || !target_depth || !d_rgb || !d_depth || !loss_out)
        return set_error(GS_ERR_INVALID_ARG, "a target, gradient or loss pointer is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(loss_out, 0, sizeof(double), st) != cudaSuccess) return set_error(GS_ERR_CUDA, "memset loss");
    const FwdOut O = {rgb, depth, t_final, last_idx, n_blended, target_rgb, target_depth, d_rgb, d_depth, loss_out,
                      blend_masks};
    return dispatch_fwd(*cfg, make_grid(*cam), rec_dtype, splats, vals, tile_ranges, tile_order, O, st);
}

extern "C" size_t gs_blend_mask_words(const gs_camera* cam, int64_t key_capacity) {
    if (!cam || cam->width <= 0 || cam->height <= 0 || cam->sx < 1 || cam->sy < 1 || key_capacity < 0) return 0;
    const Grid g = make_grid(*cam);
    if (g.tw * g.th <= 64)  // entry-parallel tiles: a run per pixel
        return blend_mask_base_ep(g.TX * g.TY, 0) + (size_t)64 * ((size_t)(key_capacity >> 5) + 1);
    return blend_mask_base(g.TX * g.TY, 0) + (size_t)256 * ((size_t)(key_capacity >> 5) + 1);
}

extern "C" gs_status gs_loss_l1(const gs_config* cfg, const gs_camera* cam, const float* rgb, const float* depth,
                                const float* target_rgb, const float* target_depth, float* d_rgb, float* d_depth,
                                double* loss_out, gs_stream stream) {
    if (!cfg || !cam) return set_error(GS_ERR_INVALID_ARG, "config or camera is NULL");
    if (cam->width <= 0 || cam->height <= 0 || cam->sx < 1 || cam->sy < 1)
        return set_error(GS_ERR_INVALID_ARG, "bad camera size or stride");
    if (!rgb || !depth || !target_rgb || !target_depth || !d_rgb || !d_depth || !loss_out)
        return set_error(GS_ERR_INVALID_ARG, "a loss pointer is NULL");
    const Grid g = make_grid(*cam);
    const int64_t P = (int64_t)g.Ws * g.Hs;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(loss_out, 0, sizeof(double), st) != cudaSuccess) return set_error(GS_ERR_CUDA, "memset loss");
    const int64_t want = (P + 255) / 256;
    const int sms = num_sms();
    const unsigned nb = (unsigned)(want < 4 * sms ? want : 4 * sms);
    k_loss_l1<<<nb, 256, 0, st>>>(*cfg, P, rgb, depth, target_rgb, target_depth, d_rgb, d_depth, loss_out);
    return check_launch("k_loss_l1");
}

size_t gs_project_bwd_ws(int64_t n);


extern "C" gs_status gs_render_bwd(const gs_config* cfg, const gs_camera* cam, const gs_gaussians* gsn,
                                   int rec_dtype, const void* splats, const uint32_t* vals,
                                   const uint32_t* tile_ranges, const uint32_t* tile_order, const float* t_final,
                                   const uint32_t* last_idx, const uint32_t* blend_masks, const float* d_rgb,
                                   const float* d_depth, int mode,
                                   float* grad2d, gs_grads* grads, double* pose_grad6, float* score_terms,
                                   void* workspace, size_t* workspace_bytes, gs_stream stream) {
    if (!gsn) return set_error(GS_ERR_INVALID_ARG, "gaussians is NULL");
    gs_status s;
    const int64_t n = gsn->n;
    if ((s = render_checks(cfg, cam, rec_dtype, splats, n)) != GS_OK) return s;
    if (!workspace_bytes) return set_error(GS_ERR_INVALID_ARG, "workspace_bytes is NULL");
    if (mode != GS_TRACK && mode != GS_MAP) return set_error(GS_ERR_INVALID_ARG, "bad mode %d", mode);
    const bool chain = (grads != nullptr) || pose_grad6 || score_terms;
    const size_t need = chain ? gs_project_bwd_ws(n) : 0;
    if (!workspace && need > 0) { *workspace_bytes = need; return GS_OK; }
    if (!workspace) { *workspace_bytes = 0; }
    else if (*workspace_bytes < need) return set_error(GS_ERR_WORKSPACE, "workspace %zu < %zu", *workspace_bytes, need);
    if (!tile_ranges || !t_final || !last_idx || !d_rgb || !d_depth || (n > 0 && !grad2d))
        return set_error(GS_ERR_INVALID_ARG, "an input or grad2d pointer is NULL");
    if (n > 0 && ((uintptr_t)grad2d & 15)) return set_error(GS_ERR_INVALID_ARG, "grad2d not 16-byte aligned");
    cudaStream_t st = (cudaStream_t)stream;
    if (n > 0 && cudaMemsetAsync(grad2d, 0, sizeof(float) * GS_GRAD2D_STRIDE * (size_t)n, st) != cudaSuccess)
        return set_error(GS_ERR_CUDA, "memset grad2d");
    const Grid g = make_grid(*cam);
    if (n > 0) {
#define GS_LB(DT, MD) \
    launch_bwd<DT, MD>(*cfg, g, splats, vals, tile_ranges, tile_order, t_final, last_idx, d_rgb, d_depth, grad2d, \
                       blend_masks, n, st)
        if (mode == GS_MAP)
            s = rec_dtype == GS_F32 ? GS_LB(GS_F32, GS_MAP) : rec_dtype == GS_BF16 ? GS_LB(GS_BF16, GS_MAP)
                                                                                   : GS_LB(GS_F16, GS_MAP);
        else
            s = rec_dtype == GS_F32 ? GS_LB(GS_F32, GS_TRACK) : rec_dtype == GS_BF16 ? GS_LB(GS_BF16, GS_TRACK)
                                                                                     : GS_LB(GS_F16, GS_TRACK);
#undef GS_LB
        if (s != GS_OK) return s;
    }
    if (chain) {
        size_t wb = *workspace_bytes;
        return gs_project_bwd(cfg, cam, gsn, grad2d, grads, pose_grad6, score_terms, workspace, &wb, stream);
    }
    return GS_OK;
}

// ---------------------------------------------------------------------------
// Wave launcher (gs_track_wave): the compositing of every job, grouped by
// kernel form
// ---------------------------------------------------------------------------
namespace gs {

gs_status wave_render(const gs_config& cfg, const gs_track_job* jobs, int n, cudaStream_t st) {
    gs_status s;
    // forward compositing with the fused loss: jobs of one kernel form (warps
    // a tile; or entry-parallel) in its own kernel, of several in the mixed one
    auto fwd_kind = [](const Grid& g) {
        if (fwd_entry_parallel(g)) return g.tw * g.th <= 32 ? 2 : 3;
        return tile_threads(g) == R_THREADS ? 0 : 1;
    };
    int present = 0;
    for (int j = 0; j < n; ++j) present |= 1 << fwd_kind(make_grid(jobs[j].cam));
    const bool mix = (present & (present - 1)) != 0;
    for (int kind = 0; kind < 4; ++kind) {
        if (mix ? kind != 0 : !(present & (1 << kind))) continue;
        Wave<WaveFwdJob> W;
        W.n = 0;
        int blocks = 0;
        for (int j = 0; j < n; ++j) {
            const gs_track_job& t = jobs[j];
            const Grid g = make_grid(t.cam);
            const int kd = fwd_kind(g), gpc = kd == 1 ? 2 : 1;  // tiles per CTA
            const FwdOut O = {t.rgb, t.depth, t.t_final, t.last_idx, t.n_blended, t.target_rgb, t.target_depth,
                              t.d_rgb, t.d_depth, t.loss, t.blend_masks};
            W.start[W.n] = blocks;
            W.job[W.n] = WaveFwdJob{g, t.splats, t.vals, t.tile_ranges, t.tile_order, O, kd};
            ++W.n;
            blocks += (g.TX * g.TY + gpc - 1) / gpc;
        }
        W.start[W.n] = blocks;
        if (mix) {
            const size_t sm = std::max({sizeof(FwdSmem<8>), sizeof(FwdSmem<4>), sizeof(EpFwdSmem<8, EpFwdBatch<16>::N>)});
            k_wave_render_fwd_mix<<<(unsigned)blocks, R_THREADS, sm, st>>>(cfg, W);
            if ((s = check_launch("k_wave_render_fwd")) != GS_OK) return s;
            break;
        }
#define GS_FWD(NW, CT) k_wave_render_fwd<NW, CT><<<(unsigned)blocks, R_THREADS, sizeof(FwdSmem<NW>), st>>>(cfg, W)
        if (kind == 0 && fwd_three(blocks)) GS_FWD(8, 3);
        else if (kind == 0) GS_FWD(8, 4);
        else if (kind == 1) GS_FWD(4, 3);
        else if (kind == 2) k_wave_render_fwd_ep<8><<<(unsigned)blocks, 8 * 32, sizeof(EpFwdSmem<8>), st>>>(cfg, W);
        else k_wave_render_fwd_ep<16><<<(unsigned)blocks, 16 * 32, sizeof(EpFwdSmem<16>), st>>>(cfg, W);
#undef GS_FWD
        if ((s = check_launch("k_wave_render_fwd")) != GS_OK) return s;
    }
    // backward compositing, pose-only fields: one launch per kernel form
    // present (0, 1: without masks, one or several tiles a CTA; 2, 3:
    // entry-parallel tiles of up to 32 or 64 pixels; 4: one-warp CTAs).  The
    // masked sessions' tiles together decide between the last three (they
    // share a launch and so its tail: six sessions 682 us, 740 in three
    // launches by each session's own tiles); both kernels form the same float32
    // terms, so a session's gradients move by their rounding alone.
    int masked = 0;
    int64_t masked_n = 0;
    for (int j = 0; j < n; ++j) {
        const Grid g = make_grid(jobs[j].cam);
        if (jobs[j].blend_masks) {
            masked += g.TX * g.TY;
            masked_n += jobs[j].g.n;
        }
    }
    auto bwd_kind = [masked, masked_n](const gs_track_job& t) {
        const Grid g = make_grid(t.cam);
        if (bwd_entry_parallel(g, t.blend_masks != nullptr, masked, masked_n)) return g.tw * g.th <= 32 ? 2 : 3;
        return t.blend_masks ? 4 : (R_THREADS / tile_threads(g) == 1 ? 0 : 1);
    };
    int kinds = 0;
    for (int j = 0; j < n; ++j) kinds |= 1 << bwd_kind(jobs[j]);
    for (int kind = 0; kind < 5; ++kind) {
        if (!(kinds & (1 << kind))) continue;
        Wave<WaveBwdJob> W;
        W.n = 0;
        int blocks = 0;
        size_t smem = 0;
        const int per_entry = (int)(sizeof(StagedSplat) + sizeof(uint32_t) + sizeof(float) * Fields<GS_TRACK>::N);
        for (int j = 0; j < n; ++j) {
            const gs_track_job& t = jobs[j];
            const Grid g = make_grid(t.cam);
            if (bwd_kind(t) != kind) continue;
            const int ntiles = g.TX * g.TY;
            const int gpc = kind < 2 ? R_THREADS / tile_threads(g) : 1;
            const int B = kind < 2 ? group_batch(gpc, per_entry, R_BWD_SMEM) : 0;
            W.start[W.n] = blocks;
            W.job[W.n] = WaveBwdJob{g, t.splats, t.vals, t.tile_ranges, t.tile_order, t.t_final, t.last_idx, t.d_rgb,
                                    t.d_depth, t.grad2d, t.blend_masks, B};
            ++W.n;
            blocks += kind == 4 ? ntiles * pw_warps(g) : (ntiles + gpc - 1) / gpc;
            if (kind < 2) smem = std::max(smem, (size_t)gpc * B * per_entry);
        }
        W.start[W.n] = blocks;
        if (kind == 0) {
            if ((s = smem_once((const void*)k_wave_render_bwd<1>, 42, R_BWD_SMEM)) != GS_OK) return s;
            k_wave_render_bwd<1><<<(unsigned)blocks, R_THREADS, smem, st>>>(cfg, W);
        } else if (kind == 1) {
            if ((s = smem_once((const void*)k_wave_render_bwd<4>, 43, R_BWD_SMEM)) != GS_OK) return s;
            k_wave_render_bwd<4><<<(unsigned)blocks, R_THREADS, smem, st>>>(cfg, W);
        } else if (kind == 2) {
            const int sm = (int)sizeof(EpBwdSmem<GS_TRACK, 8>);
            if ((s = smem_once((const void*)k_wave_render_bwd_ep<8>, 44, sm)) != GS_OK) return s;
            k_wave_render_bwd_ep<8><<<(unsigned)blocks, 8 * 32, sm, st>>>(cfg, W);
        } else if (kind == 3) {
            const int sm = (int)sizeof(EpBwdSmem<GS_TRACK, 16>);
            if ((s = smem_once((const void*)k_wave_render_bwd_ep<16>, 45, sm)) != GS_OK) return s;
            k_wave_render_bwd_ep<16><<<(unsigned)blocks, 16 * 32, sm, st>>>(cfg, W);
        } else {
            k_wave_render_bwd_pw<<<(unsigned)blocks, 32, 0, st>>>(cfg, W);
        }
        if ((s = check_launch("k_wave_render_bwd")) != GS_OK) return s;
    }
    return GS_OK;
}

}  // namespace gs
