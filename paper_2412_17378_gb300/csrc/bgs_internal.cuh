// bgs_internal.cuh -- shared declarations of the CUDA library (device helpers, the
// plan's control block, per-pair blend rule, kernel launchers).  Not installed.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/bgs.h"

namespace bgs {

// ---- constants of the per-pair rule (Algorithm 5 with standard 3DGS constants) -------
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTMin = 1e-4f;
constexpr float kLog2e = 1.4426950408889634f;  // log2(e): exp(x) = 2^(x log2 e)
constexpr float kLn2 = 0.6931471805599453f;    // ln(2)

constexpr int kMaxViews = 32;  // views of one batched call

// ---- device control block (one per plan) --------------------------------------------
struct DevCtrl {
    unsigned int queue_head;    // pixel-wise queue cursor (starts at num_gauss)
    unsigned int num_items;     // work items in the current list
    unsigned int check_bits;    // BGS_CHECK_* raised by device checks
    unsigned int num_gauss;     // item numbers [0, num_gauss) are Gaussian-wise, the rest pixel-wise
    unsigned long long num_entries;  // K written by binning
    unsigned long long eval_pairs;
    unsigned long long contrib_pairs;
    unsigned long long items_done;
    unsigned int queue_head_g;  // Gaussian-wise queue cursor (starts at 0)
    unsigned int pass_items;    // items the current persistent pass completed
    unsigned long long bin_base;  // binning: entries of the call so far (= num_entries at its end)
    unsigned int warps_done;    // blocks of the current persistent pass that finished
    unsigned int pad1;
    // work-list build: items per sort key, each key's first item, blocks done (the counters
    // return to zero at the end of every build)
    unsigned int wl_cnt[256];
    unsigned int wl_off[256];
    unsigned int wl_done;
    unsigned int gw_first;      // Gaussian-wise segments [0, gw_first) are the tiles' first ones;
                                // the later ones of long lists follow
    unsigned int gw_seg;        // entries per Gaussian-wise segment (0: lists are not split)
    unsigned int gw_wide;       // the segments' items: blocks of pixels (1) or pixel groups (0)
    unsigned long long wl_extra;  // work-list build: later segments (returns to zero)
    // binning: each view's entry count and first point_list slot
    unsigned long long view_k[kMaxViews];
    unsigned long long view_base[kMaxViews];
    unsigned int bin_done[kMaxViews];  // column blocks done (returns to zero)
    unsigned int bin_head[kMaxViews];  // the scatter's queue cursor
};

// End of a persistent pass, per warp (lane 0), for a block of `warps_per_block` warps whose
// shared counters blk[0] (items) and blk[1] (finished warps) start at 0: the block's last
// warp adds the block's completed items to the pass total, and the pass's last block
// (`pass_blocks` in all) compares the total with the queued item count and raises
// BGS_CHECK_QUEUE unless every item ran exactly once.
__device__ __forceinline__ void finish_pass(DevCtrl *ctrl, unsigned long long items, unsigned int *blk,
                                            int warps_per_block, int pass_blocks) {
    atomicAdd(&blk[0], (unsigned int)items);
    __threadfence_block();
    if (atomicAdd(&blk[1], 1u) != (unsigned int)warps_per_block - 1u) return;
    atomicAdd(&ctrl->pass_items, atomicAdd(&blk[0], 0u));
    __threadfence();
    if (atomicAdd(&ctrl->warps_done, 1u) == (unsigned int)pass_blocks - 1u) {
        __threadfence();
        const unsigned int done = atomicAdd(&ctrl->pass_items, 0u);
        if (done != *((volatile unsigned int *)&ctrl->num_items)) atomicOr(&ctrl->check_bits, BGS_CHECK_QUEUE);
    }
}

// Pixel-wise items: Q = pixel rows per lane (the plan's sub-tile knob, 1, 2, 4 or 8).  For
// Q <= 4 an item covers 8 x 4Q pixels of a tile and lane l owns the pixels (l % 8, l / 8 +
// 4 q); for Q = 8 it covers 16 x 16 pixels and lane l owns (l % 16, l / 16 + 2 q), q < Q.
// Either way a lane's pixels share one column (and so their x-offset to a Gaussian).
__host__ __device__ constexpr int pix_item_w(int Q) { return Q == 8 ? 16 : 8; }
__host__ __device__ constexpr int pix_row_step(int Q) { return 32 / pix_item_w(Q); }
__host__ __device__ constexpr int pix_item_h(int Q) { return pix_row_step(Q) * Q; }

// ---- packed per-Gaussian record used by the render kernels (48 bytes) ---------------
//   a = (mx, my, qa, qb), b = (qc, o, lv, odd), c = (r, g, b, depth)
//   with (qa, qb, qc) = -log2(e) (a/2, b, c/2), so that the natural-log power of the
//   pair is ln2 * (qa dx^2 + qb dx dy + qc dy^2) and exp(power) = 2^(qa dx^2 + ...).
//   A pair reaches alpha >= 1/255 only where that exponent is at least -lv (see
//   alpha_level); kernels use it to skip whole records for a block of pixels.  odd is not
//   0 for the records that need the pair rule in full (record_odd).
struct __align__(16) Rec {
    float4 a, b, c;
};

// One pixel-wise work item of the persistent kernels: x = tile id (global over views), y =
// sub-item index inside the tile.  Gaussian-wise tiles have one entry per segment of their
// list instead, (tile id, segment), whose items are numbered arithmetically (gw_items_per):
// kGwBlock x kGwBlock blocks of the tile's pixels, or groups of gw_pixels pixels.
constexpr int kGwBlock = 8;

__host__ __device__ constexpr int gw_blocks_per(int tile_w, int tile_h) {
    return ((tile_w + kGwBlock - 1) / kGwBlock) * ((tile_h + kGwBlock - 1) / kGwBlock);
}

// ---- small device helpers ------------------------------------------------------------
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// hardware reciprocal approximation (a few ulp; used where the backward recovers T_i)
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void raise_check(DevCtrl *ctrl, unsigned int bit) {
    atomicOr(&ctrl->check_bits, bit);
}

// lv = log2(255 o): o 2^p >= 1/255 needs p >= -lv.  -3e38 when o <= 1/255 (no pixel reaches
// it); 3e38 (no block is skipped) when the conic is not positive definite.
__device__ __forceinline__ float alpha_level(float a, float b, float c, float o) {
    const float lo = 255.f * o;
    if (!(lo > 1.f)) return -3.0e38f;
    return a * c - b * b > 0.f ? log2f(lo) : 3.0e38f;
}

// 0 times x is 0, and no product of two such values overflows (false for infinities and NaN).
__device__ __forceinline__ bool tame(float x) { return fabsf(x) < 1e18f; }

// 0 when, at every pixel, the clamp and the sign test of the pair rule decide nothing and a
// masked pair adds nothing: o <= 0.99 (so o G is); the exponent is never above 0 by rounding
// (its float32 error is below 4e-7 of the sum of its square terms, which at det >= 1e-5 a c
// exceed the cross term by 5e-6 of it); and colour and depth are tame.  2 when they are not, 1
// for the other records.
__device__ __forceinline__ float record_odd(float a, float b, float c, float o, float4 rgbd) {
    const float ac = a * c;
    if (!(tame(rgbd.x) && tame(rgbd.y) && tame(rgbd.z) && tame(rgbd.w))) return 2.f;
    return o <= kAlphaMax && a > 0.f && ac < 1e30f && ac - b * b >= 1e-5f * ac ? 0.f : 1.f;
}

// Packs record g into a Rec (the conic is pre-scaled by -log2(e)/2); its colour is
// colour row cg (views of a batched call share the colours of their Gaussians).
__device__ __forceinline__ Rec make_rec(const float *__restrict__ means2D, const float *__restrict__ conic_opacity,
                                        const float *__restrict__ colors, const float *__restrict__ depths,
                                        unsigned int g, unsigned int cg) {
    Rec r;
    const float2 m = reinterpret_cast<const float2 *>(means2D)[g];
    const float4 co = reinterpret_cast<const float4 *>(conic_opacity)[g];
    r.a = make_float4(m.x, m.y, -0.5f * kLog2e * co.x, -kLog2e * co.y);
    r.c = make_float4(colors[3 * cg], colors[3 * cg + 1], colors[3 * cg + 2], depths[g]);
    r.b = make_float4(-0.5f * kLog2e * co.z, co.w, alpha_level(co.x, co.y, co.z, co.w),
                      record_odd(co.x, co.y, co.z, co.w, r.c));
    return r;
}

// true when the record cannot reach alpha >= 1/255 at any pixel whose centre lies within
// (hw, hh) of (cx, cy): the largest exponent over that rectangle is below -lv.  With d = mean
// - pixel, the exponent (a concave quadratic, 0 at d = 0) is largest on the rectangle's edge
// nearest the mean in x (d.x = xn) or in y (d.y = yn), at that edge's own maximum clamped to
// its ends; a mean inside gives xn = yn = 0 and the exponent 0.  The test widens the level by
// 0.01 and by 4e-6 of the sum of the terms' magnitudes at the farthest corner, ten times the
// float32 rounding of a pair's exponent there (which also covers a conic that float32 takes
// for positive definite by rounding alone), so it never drops a pair that pair_oG accepts; a
// NaN keeps the record.
// Against the bounding box of the same level set it keeps 0.51 (4M Gaussians of log-scale
// deviation 1), 0.69 (1M, deviation 0.7) or 0.77-0.84 (deviation 0.5) of an 8x16 block's
// records, where 0.47-0.74 have a pixel that accepts them, for about 40 instructions per 32
// records: the 9-view 4M-Gaussian step 13.89 -> 12.79 ms, a 1080p frame of 600k 640 -> 598 us.
__device__ __forceinline__ bool block_misses(const float4 &a, const float4 &b, float cx, float cy, float hw, float hh) {
    const float ex = a.x - cx, ey = a.y - cy;
    const float xn = copysignf(fmaxf(fabsf(ex) - hw, 0.f), ex), yn = copysignf(fmaxf(fabsf(ey) - hh, 0.f), ey);
    const float h = -0.5f * a.w;
    const float ys = fminf(fmaxf(h * xn * rcp_approx(b.x), ey - hh), ey + hh);
    const float xs = fminf(fmaxf(h * yn * rcp_approx(a.z), ex - hw), ex + hw);
    const float v1 = a.z * xn * xn + ys * (a.w * xn + b.x * ys);
    const float v2 = b.x * yn * yn + xs * (a.w * yn + a.z * xs);
    const float fx = fabsf(ex) + hw, fy = fabsf(ey) + hh;
    const float terms = fabsf(a.z) * fx * fx + fy * (fabsf(a.w) * fx + fabsf(b.x) * fy);
    return fmaxf(v1, v2) + (4e-6f * terms + 0.01f) < -b.z;
}

__device__ __forceinline__ Rec make_rec(const float *__restrict__ means2D, const float *__restrict__ conic_opacity,
                                        const float *__restrict__ colors, const float *__restrict__ depths,
                                        unsigned int g) {
    return make_rec(means2D, conic_opacity, colors, depths, g, g);
}

// power2 = log2(e) * power of the pair (pixel px, py) = qa dx^2 + qb dx dy + qc dy^2,
// evaluated as hx + dy (bx + qc dy) with hx = qa dx^2 and bx = qb dx (shared by pixels of
// one column).  Written with explicit round-to-nearest intrinsics so that no kernel's
// compilation can contract or reorder it: every kernel, forward and backward, takes the
// same skip / stop decisions bit for bit.
struct PairX {
    float dx, hx, bx;
};

__device__ __forceinline__ PairX pair_x(float4 a, float px) {
    PairX r;
    r.dx = __fsub_rn(a.x, px);
    r.hx = __fmul_rn(__fmul_rn(a.z, r.dx), r.dx);
    r.bx = __fmul_rn(a.w, r.dx);
    return r;
}

__device__ __forceinline__ float pair_power2_y(const PairX &x, float ay, float qc, float py, float &dy) {
    dy = __fsub_rn(ay, py);
    return __fmaf_rn(dy, __fmaf_rn(qc, dy, x.bx), x.hx);
}

__device__ __forceinline__ float pair_power2(float4 a, float qc, float px, float py, float &dx, float &dy) {
    const PairX x = pair_x(a, px);
    dx = x.dx;
    return pair_power2_y(x, a.y, qc, py, dy);
}

// Transmittance after a pair, T (1 - alpha), as one fused multiply-add T - T alpha (one
// rounding); the pixel-wise kernels (static, persistent, allocation-free) and the
// backward's T recovery take their stop decision T' < 1e-4 on this value.  The
// Gaussian-wise kernels walk the entries of the stopping chunk with it too, but from a T in
// front of the chunk that is a product of chunk products (reassociated: about 2 ulp per
// 8-entry chunk and composition against this sequential chain), so a decision can only
// flip where T' lies within that rounding of 1e-4: inside the oracle's |T' - 1e-4| < 1e-9
// flag window at the list lengths of the tests.
__device__ __forceinline__ float next_T(float T, float al) { return __fmaf_rn(-T, al, T); }

// o G of a pair.  A pair is accumulated when power2 <= 0 and o G >= 1/255 (the same as
// alpha = min(0.99, o G) >= 1/255, since 1/255 < 0.99); alpha is formed only for those.
__device__ __forceinline__ float pair_oG(float power2, float o) { return __fmul_rn(o, ex2_approx(power2)); }

// ---- pairs of float32 values in one 64-bit register (both halves rounded like the scalar
// instruction; one issue slot for two results) --------------------------------------------
typedef unsigned long long F2;

__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 f2_split(F2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// ---- views ---------------------------------------------------------------------------
// A render call covers V views (1 for the single-view entry points).  Their tiles form
// one global tile space: view v owns tile ids [tile_base[v], tile_base[v+1]).  Record
// (and gradient) index v * n_per_view + g belongs to Gaussian g seen from view v.

struct ViewTable {
    int V;
    int W[kMaxViews], H[kMaxViews], tiles_x[kMaxViews], tiles_y[kMaxViews];
    int tile_base[kMaxViews + 1];
};

// view owning a global tile id (binary search over tile_base)
__device__ __forceinline__ int view_of(const ViewTable &vt, int tile) {
    int lo = 0, hi = vt.V - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (vt.tile_base[mid] <= tile) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

struct ViewOut {  // forward outputs, per view
    float *out_color[kMaxViews], *out_depth[kMaxViews], *out_alpha[kMaxViews], *final_T[kMaxViews];
    int *n_contrib[kMaxViews], *n_eval[kMaxViews];
};

struct ViewGradIn {  // backward inputs, per view
    const float *final_T[kMaxViews];
    const int *n_contrib[kMaxViews];
    const float *dL_dcolor[kMaxViews], *dL_ddepth[kMaxViews], *dL_dalpha[kMaxViews];
};

// ---- launch parameter blocks -----------------------------------------------------------
struct FwdArgs {
    const Rec *recs;             // packed records [V * n_per_view]
    const float *means2D, *conic_opacity, *colors, *depths;  // ABI arrays (static kernel)
    const uint32_t *point_list;
    const uint2 *ranges;         // [total tiles]
    long long N;                 // number of records (V * n_per_view)
    long long num_entries;
    int tile_w, tile_h, num_tiles;
    float bg[3];
    ViewTable vt;
    ViewOut io;
    DevCtrl *ctrl;
    const uint2 *items;          // pixel-wise work list (persistent kernels)
    int pass_blocks;             // blocks of the persistent pass (all forward kernels that run)
    int gw_pixels;
    const uint2 *gw_ent;         // Gaussian-wise segments (tile, segment)
    const uint2 *gw_tile;        // per Gaussian-wise tile: (its first segment's entry, its second's)
    float4 *gw_sum;              // per Gaussian-wise segment, per pixel of a full tile: the summary
    uint32_t *gw_done;           // per (first segment, block): all pixels stopped in it, outputs written
    unsigned int *tile_cost;     // per tile (nullable, zeroed): the largest n_contrib of its pixels
    int pixel_rows;              // Q of the pixel-wise items
    int chunk;
};

// A pixel's record of one Gaussian-wise segment (2 x 16 bytes), per (segment, pixel of the tile).
// Written by the segment's item:
//   cd = colour and depth accumulated with the segment's own transmittance from 1;
//   t  = (transmittance after the segment, last contributor (index in the tile's list, bits;
//        -1: none), contributing pairs (bits), entries up to and including the stop (bits)
//        when the pixel stopped in the segment, else 0).
// Rewritten by the merge, for every segment the pixel reaches when its list has several:
//   cd = colour and depth accumulated behind the segment (with absolute weights, the
//        background's T_f bg included);  t.x = the transmittance behind the segment.
// That is the state a back-to-front walk holds when it enters the segment from behind.
struct GwSum {
    float4 cd;
    float4 t;
};

__device__ __forceinline__ bool tile_is_gauss(int mode, int heavy_threshold, uint32_t n) {
    return mode == BGS_MODE_GAUSSIAN || (mode == BGS_MODE_AUTO && n > (uint32_t)heavy_threshold);
}

struct BwdArgs {
    const Rec *recs;
    const float *means2D, *conic_opacity, *colors, *depths;
    const uint32_t *point_list;
    const uint2 *ranges;
    long long N;
    long long num_entries;
    int tile_w, tile_h, num_tiles;
    float bg[3];
    ViewTable vt;
    ViewGradIn gi;
    float *grad_acc;             // [N][12] accumulators (10 used)
    DevCtrl *ctrl;
    const uint2 *items;
    unsigned int *warp_items;  // per warp of the persistent pass: items it completed
    int pixel_rows;
    int chunk;
    // segmented walk of the tiles the last forward split (bseg_mode: its render mode, -1:
    // none): the forward's per-tile segment item positions and boundary states
    int bseg_mode, heavy_threshold;
    const uint2 *gw_tile;
    const GwSum *gw_sum;
};

// Records a message for bgs_last_error() and returns code.
int set_error(int code, const char *msg);

// ---- launchers (each returns cudaGetLastError() of its launch) ------------------------
// N Gaussians seen from V cameras: record v * N + g (V = 1 for a single view)
cudaError_t launch_preprocess(long long N, int V, const float *means3D, const float *log_scales, const float *quats,
                              const float *opacities, const bgs_camera *cams, int tile_w, int tile_h,
                              float *means2D, float *conic_opacity, float *depths, int *radii,
                              uint32_t *tiles_touched, cudaStream_t s);
// projection backward: dL/d(means2D, conic a b c, depth) of the records [V N] ->
// dL/d(means3D, log_scales, quats) [N] summed over the views (radius-0 records skipped).  With
// dL_dopacities, dL_dconic holds (a, b, c, opacity) rows, whose fourth goes there
cudaError_t launch_preprocess_backward(long long N, int V, const float *means3D, const float *log_scales,
                                       const float *quats, const bgs_camera *cams, const int *radii,
                                       const float *dL_dmeans2D, const float *dL_dconic, const float *dL_ddepths,
                                       float *dL_dmeans3D, float *dL_dlog_scales, float *dL_dquats,
                                       float *dL_dopacities, cudaStream_t s);
// idx[i] = i for i in [lo, hi)
cudaError_t launch_iota(long long lo, long long hi, uint32_t *idx, cudaStream_t s);

cudaError_t launch_touched(long long N, const float *means2D, const int *radii, int W, int H, int tile_w, int tile_h,
                           uint32_t *touched, cudaStream_t s);
cudaError_t launch_gather_u32(long long N, const uint32_t *src, const uint32_t *order, uint32_t *dst, cudaStream_t s);
template <typename KeyT>
cudaError_t launch_duplicate(long long N, const uint32_t *order, const float *means2D, const int *radii,
                             const unsigned long long *offsets, int W, int H, int tile_w, int tile_h, KeyT *keys,
                             uint32_t *vals, long long capacity, cudaStream_t s);
cudaError_t launch_count_total(long long N, const uint32_t *touched, const unsigned long long *offsets,
                               DevCtrl *ctrl, cudaStream_t s);
template <typename KeyT>
cudaError_t launch_ranges(const KeyT *keys, long long K, uint2 *ranges, cudaStream_t s);

// counting-sort binning (binning.cu)
// shared memory of the count kernel (tile counters + one 512-bit mask slice per tile group)
size_t bin_count_smem(int tx, int ty);
int bin_mask_groups(int tx, int ty);
cudaError_t setup_bin_kernels(int tx, int ty);
// also writes each sorted position's record rect[s] = (x0 | w << 16, y0 | h << 16, Gaussian
// index, 0) (both rectangle words 0 when empty) and the (block, tile group) masks, W32
// words each (a multiple of 16)
// blocks [b_lo, b_hi) of the counting pass; skipP (nullable): the exclusive 2D prefix of the
// tiles known to have stopped before b_lo (k_bin_stopped), whose Gaussians are left out
cudaError_t launch_bin_count(long long N, int G, int b_lo, int b_hi, const uint32_t *order, const float *means2D,
                             const int *radii, int W, int H, int tw, int th, uint32_t *Hm, uint4 *rect, uint32_t *masks,
                             int W32, const int *skipP, cudaStream_t s);
// the tiles whose credits over blocks [0, B1) certify that every pixel stopped, as the
// exclusive 2D prefix P [(ty + 1) x (tx + 1)] of their indicator; S [tx ty] holds the per-tile
// sums, zero before and after
cudaError_t launch_bin_stopped(int B1, int tx, int ty, const uint16_t *D, uint32_t *S, int *P, cudaStream_t s);
// What the binning of one view publishes once its tile totals are known (by the last block of
// the column scan, or for one view of several by k_bin_open): each tile's start in the view
// and, from the view's first point_list slot on, its range; the scatter's items per tile group
// (with truncation); for a call's only view the call's entry count, also to host_k (nullable,
// mapped host memory), with the overflow check against capacity.
constexpr int kScatterBlocks = 32;  // single-warp blocks of the scatter per SM
struct BinTiles {
    int T, tx, ty, B, nC, v;
    uint32_t *total, *start;
    uint2 *ranges;
    const uint32_t *bsat;  // nullable: complete lists
    uint32_t *item_start;  // [4 nC + 1], see open_items
    int warps;             // resident warps of the scatter
    bool only;             // the call's only view
    long long capacity;
    unsigned long long *host_k;
    DevCtrl *ctrl;
};
// per tile column: exclusive prefix of H over the blocks and the total; with the credits D
// (nullable) the column is cut after the block b_sat[t] at which they certify that every
// pixel of the tile has stopped (b_sat written when bt.bsat is not null); the last block then
// scans the totals into the starts and stores the view's entry count in ctrl->view_k[v]
cudaError_t launch_bin_colscan(uint32_t *Hm, const uint16_t *D, const BinTiles &bt, cudaStream_t s);
// per block and tile: fixed-point credits toward that certificate (k_bin_credit)
size_t bin_credit_smem(int tx, int ty);
cudaError_t launch_bin_credit(long long N, int G, int b_lo, int b_hi, const uint4 *rect, const float *means2D,
                              const float *conic_opacity, int W, int H, int tw, int th, uint16_t *D, cudaStream_t s);
// a view of several: its ranges from the sum of the entry counts of views 0..v-1 on (stored in
// ctrl->view_base[v] for the scatter) and the scatter's items
cudaError_t launch_bin_open(const BinTiles &bt, cudaStream_t s);
cudaError_t launch_bin_scatter(long long N, int G, int B, int W32, const uint4 *rect, int W, int H, int tw, int th,
                               const uint32_t *Hm, const uint32_t *start, const uint32_t *masks, uint32_t *point_list,
                               long long capacity, const uint32_t *bsat, const uint32_t *item_start, int num_sms,
                               int v, DevCtrl *ctrl, cudaStream_t s);
// num_entries = bin_base = the sum of the V views' counts, also to host_k (nullable); raises
// BGS_CHECK_OVERFLOW past capacity or BGS_MAX_ENTRIES
cudaError_t launch_bin_finish(int V, long long capacity, DevCtrl *ctrl, unsigned long long *host_k, cudaStream_t s);

// view-dependent colour from spherical harmonics (sh.cu); backward: dL_drgb -> dL_dsh,
// dL_dmeans3D (summed over the V <= kMaxViews camera centres campos [V,3], host)
cudaError_t launch_sh(bool backward, long long N, int degree, int stride, const float *sh, const float *means3D,
                      int V, const float *campos, float *rgb, uint8_t *clamped, const float *dL_drgb, float *dL_dsh,
                      float *dL_dmeans3D, cudaStream_t s);

// recs[i] from means2D[i], conic_opacity[i], depths[i] and colors[i % n_colors]
cudaError_t launch_pack(long long N, const float *means2D, const float *conic_opacity, const float *colors,
                        long long n_colors, const float *depths, Rec *recs, cudaStream_t s);

// Work list of the persistent kernels, by bucket counting over the tiles' sort keys:
// k_wl_count gives every tile its place in its key's bucket and (last block) the buckets'
// first items and the ctrl counts; k_wl_emit writes the items (positions past `capacity`
// items raise BGS_CHECK_OVERFLOW and are skipped).  The order of tiles within one key is
// unspecified.
// gw_segment: entries per Gaussian-wise segment (0: no tile is Gaussian-wise); extra_cap: the
// most later segments the list may hold (beyond it the lists are not split).
// bseg_mode >= 0 (a pixel-wise list for the backward): the tiles that the last forward, in
// that render mode, split into segments get their pixel-wise items once per segment
// (ctrl->gw_seg, the forward's segment length, is kept).  gw (null pointers for a list without
// Gaussian-wise tiles): exoff [num_tiles] scratch, the segments' entries ent [ent_cap], per
// tile the entries of its first and second segment, and the cleared flags done.  cost
// [num_tiles] (nullable): the per-tile load that orders the list heaviest first (default: the
// list length).
struct GwLists {
    uint32_t *exoff;
    uint2 *ent;
    long long ent_cap;
    uint2 *tile;
    uint32_t *done;
};
cudaError_t launch_worklist_buckets(const uint2 *ranges, int num_tiles, const ViewTable &vt, int tile_w, int tile_h,
                                    int mode, int heavy_threshold, int lpt, int gw_pixels, int pixel_rows,
                                    int gw_segment, long long extra_cap, uint32_t *slot, uint2 *items,
                                    long long capacity, int bseg_mode, const GwLists &gw, const uint32_t *cost,
                                    int num_sms, DevCtrl *ctrl, cudaStream_t s);

// queue of the current list: rewind for another pass / mark exhausted (fault injection)
cudaError_t launch_rewind_queue(DevCtrl *ctrl, cudaStream_t s);
cudaError_t launch_exhaust_queue(DevCtrl *ctrl, cudaStream_t s);

cudaError_t launch_forward_static(const FwdArgs &a, cudaStream_t s);
cudaError_t launch_forward_gauss(const FwdArgs &a, int grid, cudaStream_t s);
cudaError_t launch_forward_pixel(const FwdArgs &a, int grid, bool after_gauss, cudaStream_t s);
// composes the Gaussian-wise segment summaries per pixel; after the other forward kernels
cudaError_t launch_forward_gw_merge(const FwdArgs &a, int num_sms, cudaStream_t s);
int forward_balanced_block_threads();
const void *forward_pixel_kernel(int pixel_rows);
int forward_gauss_grid(const FwdArgs &a, int num_sms, int max_per_sm);

cudaError_t launch_backward_static(const BwdArgs &a, cudaStream_t s);
cudaError_t launch_backward_balanced(const BwdArgs &a, int grid, cudaStream_t s);
int backward_balanced_block_threads();
const void *backward_balanced_kernel(const BwdArgs &a);  // the instantiation a would launch
// gradients of N records; colours have n_colors rows (n_colors < N: summed over views)
cudaError_t launch_grad_finalize(long long N, long long n_colors, float4 *acc, const float *conic_opacity,
                                 float *dL_dmeans2D, float *dL_dconic, float *dL_dopacity, float *dL_dcolors,
                                 float *dL_ddepths, const unsigned int *warp_items, int n_warps, DevCtrl *ctrl,
                                 cudaStream_t s);

}  // namespace bgs
