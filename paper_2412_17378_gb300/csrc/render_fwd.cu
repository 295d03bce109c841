// render_fwd.cu -- a4/a5: forward render kernels.
//
//  k_forward_static    plain pixel-wise kernel on a static grid (one block per tile, one
//                      thread per pixel, block-wide staging of the tile's records in
//                      shared memory) -- the paper's "naive renderCUDA" (Algorithm 4)
//                      with the shared-memory staging of features and depths of
//                      Sec. 5.2.2.  It is the baseline the balanced kernel is timed against.
//  k_forward_gauss / k_forward_pixel
//                      persistent kernels (Sec. 4.1's inter-block dynamic distribution,
//                      taken down to warp granularity): every warp pulls work items from
//                      a device atomic queue.  The work list holds the Gaussian-wise items
//                      first, then the pixel-wise ones; each kind has its own kernel (and
//                      register budget) and its own queue cursor:
//                        - Gaussian-wise (Sec. 4.2, Algorithm 6, fine-grained per
//                          Sec. 4.3): the segments of a tile's list run on separate warps
//                          and k_forward_gw_merge composes them per pixel; an item is a
//                          segment and an 8x8 block of pixels, or, where the segments are
//                          few, P pixels, the lanes splitting the segment into contiguous
//                          chunks and composing them with a shuffle prefix product;
//                        - pixel-wise: an 8x8 sub-block of a tile, two pixels per lane,
//                          walking the tile's list through a warp-private shared memory
//                          window of 32 records.
//
// All evaluate each (pixel, entry) pair with the same code (pair_power2 / pair_oG), so
// their skip decisions agree bit for bit, and the pixel-wise kernels' stop decisions too;
// the Gaussian-wise kernel's transmittance product is reassociated (see next_T).
// Results of all kernels equal the sequential rule of Algorithm 5 up to float32
// reassociation of the transmittance product (Sec. 4: "without any precision loss").
#include "bgs_internal.cuh"

namespace bgs {

constexpr unsigned kFull = 0xffffffffu;

// The accumulated alpha sum_i alpha_i T_i telescopes to 1 - T (T_i - T_{i+1} summed), so it is
// written from the final T instead of being summed per pair.
__device__ __forceinline__ void write_pixel(const FwdArgs &a, int v, int px, int py, float T, float c0, float c1,
                                            float c2, float D, int last, int neval) {
    const int W = a.vt.W[v];
    const long long HW = (long long)W * a.vt.H[v];
    const long long pid = (long long)py * W + px;
    float *oc = a.io.out_color[v];
    oc[pid] = c0 + T * a.bg[0];
    oc[HW + pid] = c1 + T * a.bg[1];
    oc[2 * HW + pid] = c2 + T * a.bg[2];
    a.io.out_depth[v][pid] = D;
    a.io.out_alpha[v][pid] = 1.f - T;
    a.io.final_T[v][pid] = T;
    a.io.n_contrib[v][pid] = last;
    if (a.io.n_eval[v]) a.io.n_eval[v][pid] = neval;
}

// Validated tile range: an out-of-bounds span raises BGS_CHECK_RANGE and renders empty.
__device__ __forceinline__ uint2 load_range(const FwdArgs &a, int tile) {
    uint2 rg = a.ranges[tile];
    if (rg.y < rg.x || (long long)rg.y > a.num_entries) {
        raise_check(a.ctrl, BGS_CHECK_RANGE);
        rg = make_uint2(0, 0);
    }
    return rg;
}

// =====================================================================================
// plain pixel-wise static kernel
// =====================================================================================
__global__ void __launch_bounds__(1024) k_forward_static(FwdArgs a) {
    extern __shared__ Rec srec[];
    const int nthreads = blockDim.x;
    const int tid = threadIdx.x;
    const int tile = blockIdx.x;  // single view: global tile id = tile of view 0
    const int tx = tile % a.vt.tiles_x[0], ty = tile / a.vt.tiles_x[0];
    const int px = tx * a.tile_w + tid % a.tile_w, py = ty * a.tile_h + tid / a.tile_w;
    const bool inside = px < a.vt.W[0] && py < a.vt.H[0];
    uint2 rg = a.ranges[tile];
    if (rg.y < rg.x || (long long)rg.y > a.num_entries) {
        if (tid == 0) raise_check(a.ctrl, BGS_CHECK_RANGE);
        rg = make_uint2(0, 0);
    }
    const float pxf = (float)px, pyf = (float)py;
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f, D = 0.f;
    int last = 0, neval = (int)(rg.y - rg.x), nacc = 0;
    bool done = !inside;
    for (uint32_t base = rg.x; base < rg.y; base += nthreads) {
        if (__syncthreads_count(done) == nthreads) break;
        const uint32_t j = base + tid;
        if (j < rg.y) {
            const uint32_t g = a.point_list[j];
            if ((long long)g < a.N) {
                srec[tid] = make_rec(a.means2D, a.conic_opacity, a.colors, a.depths, g);
            } else {
                raise_check(a.ctrl, BGS_CHECK_INDEX);
                srec[tid].b = make_float4(0.f, 0.f, 0.f, 0.f);
                srec[tid].a = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        __syncthreads();
        const int cnt = min(nthreads, (int)(rg.y - base));
        for (int k = 0; !done && k < cnt; ++k) {
            const float4 ra = srec[k].a;
            const float4 rb = srec[k].b;
            float dx, dy;
            const float p2 = pair_power2(ra, rb.x, pxf, pyf, dx, dy);
            const float oG = pair_oG(p2, rb.y);
            if (!(p2 <= 0.f && oG >= kAlphaMin)) continue;
            const float al = fminf(kAlphaMax, oG);
            const float tt = next_T(T, al);
            if (tt < kTMin) {
                done = true;
                neval = (int)(base + k + 1 - rg.x);
                break;
            }
            const float4 rc = srec[k].c;
            const float w = al * T;
            c0 += w * rc.x;
            c1 += w * rc.y;
            c2 += w * rc.z;
            D += w * rc.w;
            T = tt;
            last = (int)(base + k + 1 - rg.x);
            ++nacc;
        }
    }
    if (inside) write_pixel(a, 0, px, py, T, c0, c1, c2, D, last, neval);
    // evaluated / contributing pair counters
    unsigned long long e = inside ? (unsigned long long)neval : 0ull, c = inside ? (unsigned long long)nacc : 0ull;
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(kFull, e, o);
        c += __shfl_xor_sync(kFull, c, o);
    }
    if ((tid & 31) == 0) {
        atomicAdd(&a.ctrl->eval_pairs, e);
        atomicAdd(&a.ctrl->contrib_pairs, c);
    }
}

cudaError_t launch_forward_static(const FwdArgs &a, cudaStream_t s) {
    const int threads = a.tile_w * a.tile_h;
    const int tiles = a.vt.tiles_x[0] * a.vt.tiles_y[0];
    if (tiles == 0) return cudaSuccess;
    const size_t smem = sizeof(Rec) * threads;
    k_forward_static<<<tiles, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// =====================================================================================
// balanced persistent kernel
// =====================================================================================
constexpr int kWarpsPerBlock = 8;

struct TileGeom {
    int v;               // view
    int x0, y0, vw, vh;  // tile origin and the part of it inside the view's image
};

__device__ __forceinline__ TileGeom tile_geom(const FwdArgs &a, int tile) {
    TileGeom t;
    t.v = view_of(a.vt, tile);
    const int lt = tile - a.vt.tile_base[t.v];
    const int tx = lt % a.vt.tiles_x[t.v], ty = lt / a.vt.tiles_x[t.v];
    t.x0 = tx * a.tile_w;
    t.y0 = ty * a.tile_h;
    t.vw = min(a.tile_w, a.vt.W[t.v] - t.x0);
    t.vh = min(a.tile_h, a.vt.H[t.v] - t.y0);
    return t;
}

// A record of a window as the pixel-wise items read it: the values that meet two pixels at a
// time stand there twice, the colour and depth negated (they are weighted by -alpha T).
struct __align__(16) Hit {
    float mx, qa, qb;
    uint32_t pos;  // position in the tile's list + 1
    F2 my, qc;
    F2 o, r;
    F2 g, b;
    F2 d;
    float odd, pad;  // record_odd
};

// Gathers the warp's next 32 records (lane's index g, valid: within the list, position pos),
// tests each against the pixel block and packs those that reach it into buf in list order.
// Returns their number; *odd: one of them is (record_odd).
__device__ __forceinline__ int stage_window(const FwdArgs &a, uint32_t g, bool valid, uint32_t pos, float bcx,
                                            float bcy, float hw, float hh, Hit *buf, int lane, bool *odd = nullptr) {
    bool hit = false;
    Rec r;
    if (valid) {
        if ((long long)g < a.N) {
            r = a.recs[g];
            hit = !block_misses(r.a, r.b, bcx, bcy, hw, hh);
        } else {
            raise_check(a.ctrl, BGS_CHECK_INDEX);  // a transparent entry
        }
    }
    const unsigned live = __ballot_sync(kFull, hit);
    if (odd) *odd = __any_sync(kFull, hit && r.b.w != 0.f);
    if (hit) {
        Hit *h = buf + __popc(live & ((1u << lane) - 1u));
        *reinterpret_cast<float4 *>(h) = make_float4(r.a.x, r.a.z, r.a.w, __uint_as_float(pos));
        *reinterpret_cast<float4 *>(&h->my) = make_float4(r.a.y, r.a.y, r.b.x, r.b.x);
        *reinterpret_cast<float4 *>(&h->o) = make_float4(r.b.y, r.b.y, -r.c.x, -r.c.x);
        *reinterpret_cast<float4 *>(&h->g) = make_float4(-r.c.y, -r.c.y, -r.c.z, -r.c.z);
        *reinterpret_cast<float4 *>(&h->d) = make_float4(-r.c.w, -r.c.w, r.b.w, 0.f);
    }
    __syncwarp();
    return __popc(live);
}

// A lane's pixels, two to a pair (rows 2p and 2p + 1 of the lane's column).
template <int Q>
struct PixAcc {
    static constexpr int NP = (Q + 1) / 2;
    F2 npy[NP];  // -y; -infinity once a pixel has stopped (and outside the image): no pair passes
    F2 T[NP], c0[NP], c1[NP], c2[NP], D[NP];
    int last[2 * NP], nacc;
    int *neval;  // the lane's slots in shared memory, 32 apart: written where a pixel stops, read at the end
};

// Where a pixel's t = T (1 - alpha) falls below the stop threshold: the pair is not accumulated.
template <int Q, bool Near>
__device__ __forceinline__ void stop_pixels(F2 *nal, F2 *tt, const F2 *T, bool *v, int pos, int nacc, PixAcc<Q> &s,
                                            bool *near) {
#pragma unroll
    for (int p = 0; p < PixAcc<Q>::NP; ++p) {
        float2 a = f2_split(nal[p]), t = f2_split(tt[p]), y = f2_split(s.npy[p]);
        const float2 T0 = f2_split(T[p]);
        if (Near) {
            const float m = kTMin * 6e-8f * (3.f * (float)nacc + 16.f);
            *near = *near || nacc > 1000 || fabsf(t.x - kTMin) <= m || fabsf(t.y - kTMin) <= m;
        }
        if (t.x < kTMin) {
            a.x = 0.f, t.x = T0.x, y.x = -INFINITY;
            v[2 * p] = false;
            s.neval[32 * (2 * p)] = pos;
        }
        if (t.y < kTMin) {
            a.y = 0.f, t.y = T0.y, y.y = -INFINITY;
            v[2 * p + 1] = false;
            s.neval[32 * (2 * p + 1)] = pos;
        }
        nal[p] = f2(a.x, a.y);
        tt[p] = f2(t.x, t.y);
        s.npy[p] = f2(y.x, y.y);
    }
}

// One record on the lane's pixels: the rule of the scalar kernels, bit for bit, two pixels per
// instruction.  A pair that is not accumulated has alpha = 0, which leaves T and the sums as
// they are, so nothing branches but a pixel's stop.  Odd = false (record_odd): the pair rule
// without its sign test and clamp; Odd = true: in full, a masked pair's colour left out by
// selection.  Against a branch per pair in scalar code the kernel issues 15-23 % fewer
// instructions and takes 2.04 instead of 2.12 ms on the 9-view 4M-Gaussian step, 173-189 instead
// of 207 us on a 720p early-stage view.
template <int Q, bool Odd, bool Near = false>
__device__ __forceinline__ void blend_hit(const Hit &h, float pxf, PixAcc<Q> &s, bool *near = nullptr) {
    constexpr int NP = PixAcc<Q>::NP;
    const float4 h0 = *reinterpret_cast<const float4 *>(&h);
    const ulonglong2 h1 = *reinterpret_cast<const ulonglong2 *>(&h.my);
    const ulonglong2 h2 = *reinterpret_cast<const ulonglong2 *>(&h.o);
    const float dx = __fsub_rn(h0.x, pxf), hx = __fmul_rn(__fmul_rn(h0.y, dx), dx), bx = __fmul_rn(h0.z, dx);
    const int pos = __float_as_int(h0.w);
    const F2 hx2 = f2(hx, hx), bx2 = f2(bx, bx);
    F2 nal[NP], tt[NP];
    bool v[2 * NP];
    float tmin = 1.f;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const F2 dy = f2_add(h1.x, s.npy[p]);
        const F2 pw = f2_fma(dy, f2_fma(h1.y, dy, bx2), hx2);
        const float2 e = f2_split(pw);
        const float2 oG = f2_split(f2_mul(h2.x, f2(ex2_approx(e.x), Q == 1 ? 0.f : ex2_approx(e.y))));
        v[2 * p] = (!Odd || e.x <= 0.f) && oG.x >= kAlphaMin;
        v[2 * p + 1] = Q > 1 && (!Odd || e.y <= 0.f) && oG.y >= kAlphaMin;
        auto neg = [](float x) { return Odd ? fmaxf(-kAlphaMax, -x) : -x; };
        nal[p] = f2(v[2 * p] ? neg(oG.x) : 0.f, v[2 * p + 1] ? neg(oG.y) : 0.f);
        tt[p] = f2_fma(s.T[p], nal[p], s.T[p]);  // next_T
        const float2 t = f2_split(tt[p]);
        tmin = fminf(tmin, fminf(t.x, t.y));
    }
    if (tmin < (Near ? 1.0002f * kTMin : kTMin)) {  // a pixel stops here: the pair is not accumulated
        stop_pixels<Q, Near>(nal, tt, s.T, v, pos, s.nacc, s, near);
    }
    const ulonglong2 h3 = *reinterpret_cast<const ulonglong2 *>(&h.g);
    const F2 h4 = h.d;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const F2 w = f2_mul(nal[p], s.T[p]);
        auto in = [&](F2 c) {
            if (!Odd) return c;
            const float2 u = f2_split(c);
            return f2(v[2 * p] ? u.x : 0.f, v[2 * p + 1] ? u.y : 0.f);
        };
        s.c0[p] = f2_fma(w, in(h2.y), s.c0[p]);
        s.c1[p] = f2_fma(w, in(h3.x), s.c1[p]);
        s.c2[p] = f2_fma(w, in(h3.y), s.c2[p]);
        s.D[p] = f2_fma(w, in(h4), s.D[p]);
        s.T[p] = tt[p];
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        s.last[q] = v[q] ? pos : s.last[q];
        s.nacc += v[q] ? 1 : 0;
    }
}

// The lane's pixels' -alpha T factors of one plain record (record_odd = 0), as blend_hit takes them.
template <int Q>
__device__ __forceinline__ void plain_alpha(const Hit &h, float pxf, const PixAcc<Q> &s, F2 *nal, bool *v) {
    const float4 h0 = *reinterpret_cast<const float4 *>(&h);
    const ulonglong2 h1 = *reinterpret_cast<const ulonglong2 *>(&h.my);
    const F2 o = h.o;
    const float dx = __fsub_rn(h0.x, pxf), hx = __fmul_rn(__fmul_rn(h0.y, dx), dx), bx = __fmul_rn(h0.z, dx);
    const F2 hx2 = f2(hx, hx), bx2 = f2(bx, bx);
#pragma unroll
    for (int p = 0; p < PixAcc<Q>::NP; ++p) {
        const F2 dy = f2_add(h1.x, s.npy[p]);
        const float2 e = f2_split(f2_fma(dy, f2_fma(h1.y, dy, bx2), hx2));
        const float2 oG = f2_split(f2_mul(o, f2(ex2_approx(e.x), Q == 1 ? 0.f : ex2_approx(e.y))));
        v[2 * p] = oG.x >= kAlphaMin;
        v[2 * p + 1] = Q > 1 && oG.y >= kAlphaMin;
        nal[p] = f2(v[2 * p] ? -oG.x : 0.f, v[2 * p + 1] ? -oG.y : 0.f);
    }
}

// Two plain records after one another on the lane's pixels: the arithmetic of blend_hit on each. A
// pixel's alphas do not depend on its transmittance, which alone runs through both, so one
// record's exponentials cover the other's latency (24 warps an SM left 27 % of the issue slots
// empty), and the stop is tested once for both.  A stop is resolved in place, by the lane that
// has it: sent back to blend_hit, the lanes of a warp drift apart by a record (the 9-view step
// 11.84 instead of 11.78 ms), and sent back together they lose the second record's work (11.94).
// Against one record at a time a 600k-Gaussian 1080p frame takes 533 instead of 541 us, a 720p
// early-stage render and backward 545 instead of 559, a 1080p one under the plan's defaults 826
// instead of 867.
template <int Q, bool Near>
__device__ __forceinline__ void blend_two(const Hit &ha, const Hit &hb, float pxf, PixAcc<Q> &s, bool *near) {
    constexpr int NP = PixAcc<Q>::NP;
    F2 na[NP], nb[NP], ta[NP], tb[NP];
    bool va[2 * NP], vb[2 * NP];
    plain_alpha<Q>(ha, pxf, s, na, va);
    plain_alpha<Q>(hb, pxf, s, nb, vb);
    float tmin = 1.f;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        ta[p] = f2_fma(s.T[p], na[p], s.T[p]);  // next_T
        tb[p] = f2_fma(ta[p], nb[p], ta[p]);    // (at most ta)
        const float2 t = f2_split(tb[p]);
        tmin = fminf(tmin, fminf(t.x, t.y));
    }
    const int pa = (int)ha.pos, pb = (int)hb.pos;
    if (tmin < (Near ? 1.0002f * kTMin : kTMin)) {  // a pixel stops, at the first (and meets no second) or the second
        stop_pixels<Q, Near>(na, ta, s.T, va, pa, s.nacc, s, near);
        int nacc = s.nacc;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float2 y = f2_split(s.npy[p]), b = f2_split(nb[p]);
            vb[2 * p] = vb[2 * p] && y.x != -INFINITY;
            vb[2 * p + 1] = vb[2 * p + 1] && y.y != -INFINITY;
            nb[p] = f2(vb[2 * p] ? b.x : 0.f, vb[2 * p + 1] ? b.y : 0.f);
            tb[p] = f2_fma(ta[p], nb[p], ta[p]);
            nacc += (va[2 * p] ? 1 : 0) + (va[2 * p + 1] ? 1 : 0);
        }
        stop_pixels<Q, Near>(nb, tb, ta, vb, pb, nacc, s, near);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const F2 wa = f2_mul(na[p], s.T[p]), wb = f2_mul(nb[p], ta[p]);
        s.c0[p] = f2_fma(wb, hb.r, f2_fma(wa, ha.r, s.c0[p]));
        s.c1[p] = f2_fma(wb, hb.g, f2_fma(wa, ha.g, s.c1[p]));
        s.c2[p] = f2_fma(wb, hb.b, f2_fma(wa, ha.b, s.c2[p]));
        s.D[p] = f2_fma(wb, hb.d, f2_fma(wa, ha.d, s.D[p]));
        s.T[p] = tb[p];
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        s.last[q] = vb[q] ? pb : (va[q] ? pa : s.last[q]);
        s.nacc += (va[q] ? 1 : 0) + (vb[q] ? 1 : 0);
    }
}

// Walks entries [e0, e1) of a tile's list, which starts at e0, for the lane's pixels until all of
// the warp's have stopped.  Near: *near is set when a transmittance comes so close to the stop
// threshold that the same product composed in another order could fall on its other side: two
// such float32 products of n accumulated pairs differ by at most (3 n + 16) 2^-24 of their value.
template <int Q, bool Near>
__device__ __forceinline__ void walk_list(const FwdArgs &a, uint32_t e0, uint32_t e1, float pxf, float bcx, float bcy,
                                          float hw, float hh, Hit *buf, int lane, PixAcc<Q> &s, bool *near) {
    // the point-list index of the lane's next entry, loaded a window ahead
    uint32_t g_next = e1 > e0 + lane ? a.point_list[e0 + lane] : 0u;
    for (uint32_t base = e0; base < e1; base += 32) {
        bool lane_done = true;
#pragma unroll
        for (int p = 0; p < PixAcc<Q>::NP; ++p) {
            const float2 y = f2_split(s.npy[p]);
            lane_done = lane_done && y.x == -INFINITY && y.y == -INFINITY;
        }
        if (__all_sync(kFull, lane_done)) break;
        const uint32_t g = g_next;
        if (e1 - base > 32u + lane) g_next = a.point_list[base + 32u + lane];
        bool odd;
        const Hit *end = buf + stage_window(a, g, base + lane < e1, base + lane + 1u - e0, bcx, bcy, hw, hh, buf, lane,
                                            &odd);
        const Hit *h = buf;
        // (windows are all plain or not: asked per pair of records, the test cost what two gained)
        if (!odd)
            for (; h + 1 < end; h += 2) blend_two<Q, Near>(h[0], h[1], pxf, s, near);
        for (; h < end; ++h) {
            if (h->odd != 0.f) blend_hit<Q, true, Near>(*h, pxf, s, near);
            else blend_hit<Q, false, Near>(*h, pxf, s, near);
        }
        __syncwarp();
    }
}

// Pixel-wise item: an 8 x 4Q sub-block of a tile; lane l owns the pixels (l % 8, l / 8 + 4 q).
// The warp walks the tile's list 32 entries at a time: each lane gathers one record and tests
// it against the item's pixel block, and the records that reach it go to a warp-private
// window in shared memory, from which every lane reads them (broadcast) and applies them to
// its Q pixels, which share dx.
template <int Q>
__device__ __forceinline__ void pixel_item(const FwdArgs &a, int tile, int sub, Hit *buf, int *neval, int lane,
                                           unsigned long long &st_eval, unsigned long long &st_acc) {
    constexpr int kItemW = pix_item_w(Q), kItemH = pix_item_h(Q), kRowStep = pix_row_step(Q);
    const TileGeom tg = tile_geom(a, tile);
    const int cxs = (tg.vw + kItemW - 1) / kItemW;
    const int sx = sub % cxs, sy = sub / cxs;
    const int px = tg.x0 + sx * kItemW + (lane % kItemW);
    const int py0 = tg.y0 + sy * kItemH + (lane / kItemW);
    const uint2 rg = load_range(a, tile);
    const float pxf = (float)px;
    // centre and half-extent of the item's pixel block (for skipping records that miss it)
    const float bcx = (float)(tg.x0 + sx * kItemW) + 0.5f * (kItemW - 1);
    const float bcy = (float)(tg.y0 + sy * kItemH) + 0.5f * (kItemH - 1);
    PixAcc<Q> s;
    s.neval = neval + lane;
    auto inside = [&](int q) { return q < Q && px < tg.x0 + tg.vw && py0 + kRowStep * q < tg.y0 + tg.vh; };
    auto npy_of = [&](int q) { return inside(q) ? -(float)(py0 + kRowStep * q) : -INFINITY; };
#pragma unroll
    for (int p = 0; p < PixAcc<Q>::NP; ++p) {
        s.npy[p] = f2(npy_of(2 * p), npy_of(2 * p + 1));
        s.T[p] = f2(1.f, 1.f);
        s.c0[p] = s.c1[p] = s.c2[p] = s.D[p] = f2(0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        s.last[q] = 0;
        s.neval[32 * q] = (int)(rg.y - rg.x);
    }
    s.nacc = 0;
    walk_list<Q, false>(a, rg.x, rg.y, pxf, bcx, bcy, 0.5f * (kItemW - 1), 0.5f * (kItemH - 1), buf, lane, s, nullptr);
    int mlast = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        if (inside(q)) {
            auto half = [&](F2 x) {
                const float2 u = f2_split(x);
                return q & 1 ? u.y : u.x;
            };
            write_pixel(a, tg.v, px, py0 + kRowStep * q, half(s.T[q / 2]), half(s.c0[q / 2]), half(s.c1[q / 2]),
                        half(s.c2[q / 2]), half(s.D[q / 2]), s.last[q], s.neval[32 * q]);
            st_eval += (unsigned long long)s.neval[32 * q];
            mlast = max(mlast, s.last[q]);
        }
    }
    st_acc += (unsigned long long)s.nacc;
    // the tile's largest n_contrib: the backward's per-tile cost (its work list's order)
    if (a.tile_cost) {
        mlast = __reduce_max_sync(kFull, mlast);
        if (lane == 0 && mlast > 0) atomicMax(a.tile_cost + tile, (unsigned int)mlast);
    }
}

// ---- Gaussian-wise items (Sec. 4.2-4.3, Algorithm 6) ------------------------------------
// The lanes of a warp split a tile's depth-sorted list and combine transmittance with a
// prefix product over lanes, as in Algorithm 6, but at chunk granularity: each lane blends a
// contiguous chunk of kGwChunk entries serially (its own transmittance starts at 1), then a
// prefix product composes the chunks with the over-operator
// (C1, T1) o (C2, T2) = (C1 + T1 C2, T1 T2), once per round instead of once per entry.
// An item covers P pixels: the warp's lanes are PXL pixel-lanes x NCH = 32 / PXL chunk-lanes,
// each lane holding PPL of the item's pixels, so that the PXL lanes of one chunk read the same
// records (one gather serves PXL x PPL pixels) and a round covers NCH chunks.  The list is
// further cut into segments of gw_segment entries handled by separate warps (cross-warp
// splitting of one pixel's list): a segment item walks its segment for its P pixels from
// transmittance 1 and writes each pixel's segment summary (C, D, T, last contributor,
// contributing pairs).  k_forward_gw_merge then composes a pixel's segments in list order
// and, in the segment where the composed transmittance falls below 1e-4, walks the entries
// again one by one from the exact incoming transmittance with Algorithm 5's rule, so the
// stop position, n_contrib and n_eval follow the sequential rule (the composed products
// differ from the sequential chain by float32 reassociation only).
constexpr int kGwChunk = 8;                          // entries a lane blends serially per round
constexpr int kGwIdx = 32 * kGwChunk + 32;           // staged indices of the largest round, skewed

template <int P>
struct GwShape {
    static constexpr int PPL = P >= 2 ? 2 : 1;  // pixels per lane
    static constexpr int PXL = P / PPL;         // pixel-lanes
    static_assert(PXL * PPL == P && 32 % PXL == 0, "pixels per Gaussian-wise item: 1, 2, 4, 8 or 16");
};

// Lanes pl, pl + PXL, pl + 2 PXL, ...: the chunk-lanes of pixel-lane pl.
template <int PXL>
__device__ __forceinline__ unsigned gw_group_mask(int pl) {
    constexpr unsigned pat = PXL == 1 ? 0xffffffffu
                           : PXL == 2 ? 0x55555555u
                           : PXL == 4 ? 0x11111111u
                           : PXL == 8 ? 0x01010101u
                                      : 0x00010001u;
    return pat << pl;
}

__device__ __forceinline__ void gw_item_pixel(const TileGeom &tg, int group, int P, int p, bool &ok, float &pxf,
                                              float &pyf) {
    const int npix = tg.vw * tg.vh;
    const int q = group * P + p;
    ok = q < npix;
    const int qq = ok ? q : 0;
    pxf = (float)(tg.x0 + qq % tg.vw);
    pyf = (float)(tg.y0 + qq / tg.vw);
}

// Walks entries [e0, e1) of a tile's list (which starts at list0) for a lane's PPL pixels of
// a Gaussian-wise item laid out as PXL pixel-lanes x (32 / PXL) chunk-lanes.  Per pixel p, on
// entry: Ts = transmittance in front of e0, live = still walking (both the same on the
// chunk-lanes of a pixel); the lane accumulators (c0, c1, c2, d: this lane's share of colour
// and depth; nacc: its contributing pairs) add to what they hold, last (the same on the
// pixel's lanes) is the latest contributor so far.  Per round each chunk-lane blends kGwChunk
// consecutive entries from a local transmittance of 1; a shuffle prefix product over the
// pixel's chunk-lanes gives the transmittance in front of each chunk.  When the round's
// composed transmittance falls below 1e-4:
//   resolve = true (Ts exact): the chunk-lanes in front of the first one whose product falls
//     below 1e-4 compose as usual, and that lane walks the rest of the round entry by entry
//     with Algorithm 5's rule from the transmittance in front of its chunk; the pixel stops
//     at the first entry whose next transmittance is below 1e-4 (stop = entries up to and
//     including it) -- if none does (float32 reassociation), the walk goes on;
//   resolve = false: the pixel is left saturated (live = false, Ts < 1e-4), for the merge.
template <int PXL, int PPL>
__device__ __forceinline__ void gw_walk(const FwdArgs &a, uint32_t e0, uint32_t e1, uint32_t list0, const float *pxf,
                                        const float *pyf, bool resolve, uint32_t *idx_s, int lane, float *Ts,
                                        float *ca0, float *ca1, float *ca2, float *da, int *last, int *nacc,
                                        int *stop, bool *live) {
    constexpr int NCH = 32 / PXL, RND = NCH * kGwChunk;
    const int pl = lane % PXL, ch = lane / PXL;
    const unsigned gmask = gw_group_mask<PXL>(pl);
    const int src_last = (NCH - 1) * PXL + pl;  // the pixel's last chunk-lane
    for (uint32_t base = e0; base < e1; base += (uint32_t)RND) {
        bool any = false;
#pragma unroll
        for (int p = 0; p < PPL; ++p) any = any || live[p];
        if (!__any_sync(kFull, any)) break;
        const uint32_t rend = (uint32_t)min((unsigned long long)e1, (unsigned long long)base + RND);
        // stage the round's indices (coalesced); entry m of the round sits at m + m / kGwChunk
        __syncwarp();
#pragma unroll
        for (int m = lane; m < RND; m += 32) {
            const uint32_t j = base + (uint32_t)m;
            idx_s[m + m / kGwChunk] = j < rend ? a.point_list[j] : 0u;
        }
        __syncwarp();
        float Tl[PPL], c0[PPL], c1[PPL], c2[PPL], dl[PPL];
        int ll[PPL], nl[PPL];
#pragma unroll
        for (int p = 0; p < PPL; ++p) {
            Tl[p] = 1.f;
            c0[p] = c1[p] = c2[p] = dl[p] = 0.f;
            ll[p] = -1;
            nl[p] = 0;
        }
        const uint32_t jc = base + (uint32_t)(kGwChunk * ch);
        for (int k = 0; k < kGwChunk; ++k) {
            const uint32_t j = jc + (uint32_t)k;
            if (j >= rend) break;
            const uint32_t g = idx_s[kGwChunk * ch + k + ch];
            if ((long long)g >= a.N) {
                raise_check(a.ctrl, BGS_CHECK_INDEX);  // a transparent entry
                continue;
            }
            const Rec r = a.recs[g];
#pragma unroll
            for (int p = 0; p < PPL; ++p) {
                float dx, dy;
                const float p2 = pair_power2(r.a, r.b.x, pxf[p], pyf[p], dx, dy);
                const float oG = pair_oG(p2, r.b.y);
                if (live[p] && p2 <= 0.f && oG >= kAlphaMin) {
                    const float al = fminf(kAlphaMax, oG);
                    const float w = al * Tl[p];
                    c0[p] += w * r.c.x;
                    c1[p] += w * r.c.y;
                    c2[p] += w * r.c.z;
                    dl[p] += w * r.c.w;
                    Tl[p] = next_T(Tl[p], al);
                    ll[p] = (int)(j - list0);
                    ++nl[p];
                }
            }
        }
#pragma unroll
        for (int p = 0; p < PPL; ++p) {
            float incl = Tl[p];
#pragma unroll
            for (int off = 1; off < NCH; off <<= 1) {
                const float v = __shfl_up_sync(kFull, incl, off * PXL);
                if (ch >= off) incl *= v;
            }
            float excl = __shfl_up_sync(kFull, incl, PXL);
            if (ch == 0) excl = 1.f;
            const float Tb = Ts[p] * excl;
            const float Tround = Ts[p] * __shfl_sync(kFull, incl, src_last);
            // the same on the pixel's chunk-lanes
            const bool cross = resolve && live[p] && Tround < kTMin;
            const unsigned bal = __ballot_sync(kFull, cross && Ts[p] * incl < kTMin) & gmask;
            const int lam = cross ? __ffs(bal) - 1 : lane;
            const bool front = live[p] && (!cross || lane < lam);
            if (front) {
                ca0[p] += Tb * c0[p];
                ca1[p] += Tb * c1[p];
                ca2[p] += Tb * c2[p];
                da[p] += Tb * dl[p];
                nacc[p] += nl[p];
            }
            int lmax = front ? ll[p] : -1;
#pragma unroll
            for (int off = PXL; off < 32; off <<= 1) lmax = max(lmax, __shfl_xor_sync(kFull, lmax, off));
            last[p] = max(last[p], lmax);
            // the crossing chunk-lane walks the rest of the round for this pixel
            float T = Tb;
            int st = 0, lw = -1;
            if (cross && lane == lam) {
                for (uint32_t j = jc; j < rend; ++j) {
                    const uint32_t m = j - base;
                    const uint32_t g = idx_s[m + m / kGwChunk];
                    if ((long long)g >= a.N) continue;  // raised above
                    const Rec r = a.recs[g];
                    float dx, dy;
                    const float p2 = pair_power2(r.a, r.b.x, pxf[p], pyf[p], dx, dy);
                    const float oG = pair_oG(p2, r.b.y);
                    if (!(p2 <= 0.f && oG >= kAlphaMin)) continue;
                    const float al = fminf(kAlphaMax, oG);
                    const float tt = next_T(T, al);
                    if (tt < kTMin) {
                        st = (int)(j - list0 + 1u);
                        break;
                    }
                    const float w = al * T;
                    ca0[p] += w * r.c.x;
                    ca1[p] += w * r.c.y;
                    ca2[p] += w * r.c.z;
                    da[p] += w * r.c.w;
                    T = tt;
                    lw = (int)(j - list0);
                    ++nacc[p];
                }
            }
            const float Tn = __shfl_sync(kFull, T, lam);
            const int lwn = __shfl_sync(kFull, lw, lam);
            const int stn = __shfl_sync(kFull, st, lam);
            if (cross) {
                Ts[p] = Tn;
                last[p] = max(last[p], lwn);
                if (stn) {
                    stop[p] = stn;
                    live[p] = false;
                }
            } else if (live[p]) {
                Ts[p] = Tround;
                // a pixel below 1e-4 from a transmittance of at most 1 stops within this
                // segment: the rest of it is not needed
                if (Tround < kTMin) live[p] = false;
            }
        }
    }
}

// Sum over the chunk-lanes of each pixel-lane (xor offsets that keep lane % PXL).
template <int PXL>
__device__ __forceinline__ void gw_group_sum5(float &x0, float &x1, float &x2, float &x3, int &n) {
#pragma unroll
    for (int o = PXL; o < 32; o <<= 1) {
        x0 += __shfl_xor_sync(kFull, x0, o);
        x1 += __shfl_xor_sync(kFull, x1, o);
        x2 += __shfl_xor_sync(kFull, x2, o);
        x3 += __shfl_xor_sync(kFull, x3, o);
        n += __shfl_xor_sync(kFull, n, o);
    }
}

// A Gaussian-wise pixel-group item: P pixels of a tile over one segment of its list (entry
// number `entry`).  The first segment starts from transmittance 1, which is exact, so its stops
// are resolved here; later segments leave saturated pixels to the merge.
template <int P>
__device__ __noinline__ void gw_segment_item(const FwdArgs &a, int tile, int seg, int group, unsigned entry,
                                                uint32_t *idx_s, int lane) {
    constexpr int PPL = GwShape<P>::PPL, PXL = GwShape<P>::PXL;
    const TileGeom tg = tile_geom(a, tile);
    if (group * P >= tg.vw * tg.vh) return;
    const uint2 rg = load_range(a, tile);
    // segment size 0: the list is not split (one segment)
    const unsigned int seg_len = *((volatile unsigned int *)&a.ctrl->gw_seg);
    const unsigned long long L = seg_len ? (unsigned long long)seg_len : (1ull << 32);
    const unsigned long long s0 = (unsigned long long)rg.x + (unsigned long long)seg * L;
    const uint32_t e0 = (uint32_t)min((unsigned long long)rg.y, s0);
    const uint32_t e1 = (uint32_t)min((unsigned long long)rg.y, s0 + L);
    const int pl = lane % PXL;
    float pxf[PPL], pyf[PPL], Ts[PPL], ca0[PPL], ca1[PPL], ca2[PPL], da[PPL];
    int last[PPL], nacc[PPL], stop[PPL];
    bool live[PPL];
#pragma unroll
    for (int p = 0; p < PPL; ++p) {
        bool ok;
        gw_item_pixel(tg, group, P, pl * PPL + p, ok, pxf[p], pyf[p]);
        Ts[p] = 1.f;
        ca0[p] = ca1[p] = ca2[p] = da[p] = 0.f;
        last[p] = -1;
        nacc[p] = stop[p] = 0;
        live[p] = ok;
    }
    gw_walk<PXL, PPL>(a, e0, e1, rg.x, pxf, pyf, seg == 0, idx_s, lane, Ts, ca0, ca1, ca2, da, last, nacc, stop,
                      live);
    GwSum *out = reinterpret_cast<GwSum *>(a.gw_sum) + (size_t)entry * (a.tile_w * a.tile_h) + group * P;
#pragma unroll
    for (int p = 0; p < PPL; ++p) {
        gw_group_sum5<PXL>(ca0[p], ca1[p], ca2[p], da[p], nacc[p]);
        if (lane < PXL) {  // chunk-lane 0 of each pixel-lane
            GwSum sm;
            sm.cd = make_float4(ca0[p], ca1[p], ca2[p], da[p]);
            sm.t = make_float4(Ts[p], __int_as_float(last[p]), __int_as_float(nacc[p]), __int_as_float(stop[p]));
            out[pl * PPL + p] = sm;
        }
    }
}

__device__ __forceinline__ void flush_stats(const FwdArgs &a, int lane, unsigned long long st_eval,
                                            unsigned long long st_acc, unsigned long long st_items) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        st_eval += __shfl_xor_sync(kFull, st_eval, o);
        st_acc += __shfl_xor_sync(kFull, st_acc, o);
    }
    if (lane == 0) {
        atomicAdd(&a.ctrl->eval_pairs, st_eval);
        atomicAdd(&a.ctrl->contrib_pairs, st_acc);
        atomicAdd(&a.ctrl->items_done, st_items);
    }
}

// ---- Gaussian-wise segments by blocks of pixels ---------------------------------------------
// Where a list gives the chip enough (segment, 8 x 8 block) items, a warp takes one: the split
// of a tile's Gaussians is then across warps alone, a lane owns two pixels (8 rows apart by 4)
// and each record is gathered once for 64 pixels and skipped for all of them where its level
// set misses the block -- instead of once per P pixels with every pair evaluated, which kept
// k_forward_gauss at 92 % of the L1 rate.  The transmittances are those of gw_walk bit for bit:
// per pixel, the same chunks of kGwChunk entries each multiplied up from 1, the same rounds
// of nch chunks, composed by the same balanced product (incl_of), hence the same stops.  The
// colours are summed with the transmittance carried from pair to pair.
constexpr int kGwWarps = 4;

struct SegPix {       // a lane's two pixels
    F2 npy, Ts;       // -y (-infinity: not walking); transmittance in front of the round
    F2 X, Tl;         // running transmittance of the round; product of the current chunk
    F2 c0, c1, c2, D;
    int last[2], nacc[2], stop[2];
};

// Per warp: the window of records, the chunk products of a round [nch][32] and, per pixel half,
// its sums at the last window it entered well above 1e-4 [2][7][32].
struct SegShared {
    Hit *buf;
    F2 *cp;
    float *sv;
};

__host__ __device__ constexpr size_t seg_shared_bytes(int nch) {
    return 32 * sizeof(Hit) + (size_t)nch * 32 * sizeof(F2) + 2 * 7 * 32 * sizeof(float);
}

// Chunk-lanes of the pixel-group items of P pixels (GwShape): the chunks of a round.
__host__ __device__ constexpr int gw_chunks(int P) { return P >= 2 ? 64 / P : 32; }

__device__ __forceinline__ SegShared seg_shared(int warp, int nch) {
    extern __shared__ __align__(16) unsigned char seg_smem[];
    unsigned char *p = seg_smem + warp * seg_shared_bytes(nch);
    SegShared r;
    r.buf = reinterpret_cast<Hit *>(p);
    r.cp = reinterpret_cast<F2 *>(p + 32 * sizeof(Hit));
    r.sv = reinterpret_cast<float *>(p + 32 * sizeof(Hit) + (size_t)nch * 32 * sizeof(F2));
    return r;
}

// One record on the lane's two pixels (see blend_hit); Stops: from chunk lam on, a pixel stops
// at the first pair that takes X below 1e-4 (Algorithm 5).
template <bool Odd, bool Stops>
__device__ __forceinline__ void blend_seg(const Hit &h, float pxf, SegPix &s, int c, int lam0, int lam1) {
    const float4 h0 = *reinterpret_cast<const float4 *>(&h);
    const ulonglong2 h1 = *reinterpret_cast<const ulonglong2 *>(&h.my);
    const ulonglong2 h2 = *reinterpret_cast<const ulonglong2 *>(&h.o);
    const ulonglong2 h3 = *reinterpret_cast<const ulonglong2 *>(&h.g);
    const float dx = __fsub_rn(h0.x, pxf), hx = __fmul_rn(__fmul_rn(h0.y, dx), dx), bx = __fmul_rn(h0.z, dx);
    const int pos = __float_as_int(h0.w);
    const F2 dy = f2_add(h1.x, s.npy);
    const float2 e = f2_split(f2_fma(dy, f2_fma(h1.y, dy, f2(bx, bx)), f2(hx, hx)));
    const float2 oG = f2_split(f2_mul(h2.x, f2(ex2_approx(e.x), ex2_approx(e.y))));
    bool v0 = (!Odd || e.x <= 0.f) && oG.x >= kAlphaMin, v1 = (!Odd || e.y <= 0.f) && oG.y >= kAlphaMin;
    auto neg = [](float x) { return Odd ? fmaxf(-kAlphaMax, -x) : -x; };
    F2 nal = f2(v0 ? neg(oG.x) : 0.f, v1 ? neg(oG.y) : 0.f);
    F2 X = f2_fma(s.X, nal, s.X);
    if (Stops) {
        const float2 t = f2_split(X);
        const bool s0 = v0 && c >= lam0 && t.x < kTMin, s1 = v1 && c >= lam1 && t.y < kTMin;
        if (s0 || s1) {
            const float2 x = f2_split(s.X), y = f2_split(s.npy), n = f2_split(nal);
            X = f2(s0 ? x.x : t.x, s1 ? x.y : t.y);
            s.npy = f2(s0 ? -INFINITY : y.x, s1 ? -INFINITY : y.y);
            nal = f2(s0 ? 0.f : n.x, s1 ? 0.f : n.y);
            s.stop[0] = s0 ? pos : s.stop[0];
            s.stop[1] = s1 ? pos : s.stop[1];
            v0 = v0 && !s0;
            v1 = v1 && !s1;
        }
    }
    const F2 w = f2_mul(nal, s.X);
    auto in = [&](F2 x) {
        if (!Odd) return x;
        const float2 u = f2_split(x);
        return f2(v0 ? u.x : 0.f, v1 ? u.y : 0.f);
    };
    s.c0 = f2_fma(w, in(h2.y), s.c0);
    s.c1 = f2_fma(w, in(h3.x), s.c1);
    s.c2 = f2_fma(w, in(h3.y), s.c2);
    s.D = f2_fma(w, in(h.d), s.D);
    s.X = X;
    s.Tl = f2_fma(s.Tl, nal, s.Tl);
    s.last[0] = v0 ? pos - 1 : s.last[0];
    s.last[1] = v1 ? pos - 1 : s.last[1];
    s.nacc[0] += v0 ? 1 : 0;
    s.nacc[1] += v1 ? 1 : 0;
}

// Product of all nch chunk products of the round (mask: the chunks that have one, the others
// are 1), as gw_walk's shuffle prefix product gives it on the last chunk-lane.
__device__ __forceinline__ F2 round_product(const F2 *cp, unsigned mask, int nch, int lane) {
    F2 lv[5], x = f2(1.f, 1.f);
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        if (c >= nch) break;
        x = (mask >> c) & 1u ? cp[c * 32 + lane] : f2(1.f, 1.f);
        int l = 0;
#pragma unroll
        for (; (c >> l) & 1; ++l) x = f2_mul(lv[l], x);
        if (l < 5) lv[l] = x;
    }
    return x;
}

// The prefix product over chunks 0..k of one pixel (half h), as the shuffles give it on
// chunk-lane k: a balanced product over k, k - 1, ..., with 1 in front of chunk 0.
__device__ __noinline__ float incl_of(const F2 *cp, unsigned mask, int nch, int lane, int h, int k) {
    float lv[5], x = 1.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        if (j >= nch) break;
        x = 1.f;
        if (j <= k && (mask >> (k - j)) & 1u) {
            const float2 u = f2_split(cp[(k - j) * 32 + lane]);
            x = h ? u.y : u.x;
        }
        int l = 0;
#pragma unroll
        for (; (j >> l) & 1; ++l) x = lv[l] * x;
        if (l < 5) lv[l] = x;
    }
    return x;
}

// The crossing pixels (low0, low1) of a round [rb, rend) of seg_walk, whose chunk products are in
// sh.cp: finds each one's crossing chunk and walks it again, from its saved window (from0,
// from1) and sums, up to its stop.  Out of line: it runs a few times per item, and its code
// beside the walk's costs instruction fetches (493 -> 719 us for the Gaussian-wise items of a
// 1080p view of 300k).  io: on entry npy as at the round's start; on exit X is the crossing
// pixels' transmittance.
__device__ __noinline__ void resolve_round(const FwdArgs &a, uint32_t e1, uint32_t list0, float pxf, float bcx,
                                           float bcy, int nch, const SegShared sh, int lane, uint32_t rb,
                                           uint32_t rend, unsigned mask, bool low0, bool low1, uint32_t from0,
                                           uint32_t from1, SegPix *io) {
    constexpr float kH = 0.5f * (kGwBlock - 1);
    SegPix s = *io;
    const float2 y = f2_split(s.npy), T0 = f2_split(s.Ts);
    const uint32_t from[2] = {from0, from1}, rpos = rb - list0;
    int cur = -1;
    int lam[2] = {0, 0};
    float Tb[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float Th = h ? T0.y : T0.x;
        Tb[h] = Th;
        if (!(h ? low1 : low0)) continue;
        float P = Th;
        int k = 0;
        for (; k < nch - 1; ++k) {
            if ((mask >> k) & 1u) {
                const float2 u = f2_split(sh.cp[k * 32 + lane]);
                P *= h ? u.y : u.x;
            }
            // the two products differ by far less than 1e-4 of their value
            if (P < 1.0001f * kTMin && Th * incl_of(sh.cp, mask, nch, lane, h, k) < kTMin) break;
        }
        lam[h] = k;
        if (k > 0) Tb[h] = Th * incl_of(sh.cp, mask, nch, lane, h, k - 1);
    }
    // walk again for the crossing pixels, each from its saved window and sums on
    const bool low[2] = {low0, low1};
    float sx[2], s0[2], s1[2], s2[2], sd[2];
    uint32_t w0 = rend;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        auto half = [&](F2 v) {
            const float2 u = f2_split(v);
            return h ? u.y : u.x;
        };
        sx[h] = half(s.X), s0[h] = half(s.c0), s1[h] = half(s.c1), s2[h] = half(s.c2), sd[h] = half(s.D);
        if (!low[h]) continue;
        const float *sv = sh.sv + h * 7 * 32 + lane;
        sx[h] = sv[0], s0[h] = sv[32], s1[h] = sv[64], s2[h] = sv[96], sd[h] = sv[128];
        s.last[h] = __float_as_int(sv[160]), s.nacc[h] = __float_as_int(sv[192]);
        w0 = min(w0, from[h]);
    }
    s.X = f2(sx[0], sx[1]), s.c0 = f2(s0[0], s0[1]), s.c1 = f2(s1[0], s1[1]), s.c2 = f2(s2[0], s2[1]);
    s.D = f2(sd[0], sd[1]);
    s.npy = f2(-INFINITY, -INFINITY);
    bool walked[2] = {!low0, !low1};  // entered its window (and perhaps stopped since)
    for (uint32_t wb = __reduce_min_sync(kFull, w0); wb < rend; wb += 32u) {
        {
            const float2 z = f2_split(s.npy);
            const bool in0 = !walked[0] && wb >= from[0], in1 = !walked[1] && wb >= from[1];
            s.npy = f2(in0 ? y.x : z.x, in1 ? y.y : z.y);
            walked[0] = walked[0] || in0;
            walked[1] = walked[1] || in1;
            const float2 n = f2_split(s.npy);
            const bool todo = !walked[0] || !walked[1] || n.x != -INFINITY || n.y != -INFINITY;
            if (!__any_sync(kFull, todo)) break;  // every crossing pixel has stopped
        }
        const uint32_t g = wb + lane < rend ? a.point_list[wb + lane] : 0u;
        const Hit *end = sh.buf + stage_window(a, g, wb + lane < rend, wb + lane + 1u - list0, bcx, bcy, kH,
                                               kH, sh.buf, lane);
        for (const Hit *h = sh.buf; h != end; ++h) {
            const int c = (int)((h->pos - 1u - rpos) / kGwChunk);
            if (c != cur) {
                const float2 x = f2_split(s.X);
                s.X = f2(cur < lam[0] && c >= lam[0] ? Tb[0] : x.x,
                         cur < lam[1] && c >= lam[1] ? Tb[1] : x.y);
                cur = c;
            }
            blend_seg<true, true>(*h, pxf, s, c, lam[0], lam[1]);
        }
        __syncwarp();
    }
    const float2 z = f2_split(s.npy);
    s.npy = f2(low0 ? z.x : y.x, low1 ? z.y : y.y);
    *io = s;
}

// Walks entries [e0, e1) of a tile's list (which starts at list0) for the lane's two pixels, in
// rounds of nch chunks.  resolve: a pixel whose composed transmittance falls below 1e-4 in a
// round is walked again from the last window it entered well above that, with Algorithm 5's rule
// from its crossing chunk on (the first one whose prefix product takes it below), up to its
// stop; without, it is left saturated (Ts < 1e-4, not walking).
__device__ __forceinline__ void seg_walk(const FwdArgs &a, uint32_t e0, uint32_t e1, uint32_t list0, float pxf,
                                         float bcx, float bcy, int nch, bool resolve, const SegShared &sh, int lane,
                                         SegPix &s) {
    constexpr float kH = 0.5f * (kGwBlock - 1);
    const uint32_t rnd = (uint32_t)(nch * kGwChunk);
    uint32_t g_next = e1 > e0 + lane ? a.point_list[e0 + lane] : 0u;
    for (uint32_t rb = e0; rb < e1;) {
        const float2 y = f2_split(s.npy);
        const bool live0 = y.x != -INFINITY, live1 = y.y != -INFINITY;
        if (!__any_sync(kFull, live0 || live1)) break;
        const uint32_t rend = e1 - rb > rnd ? rb + rnd : e1, rpos = rb - list0;
        s.X = s.Ts;
        s.Tl = f2(1.f, 1.f);
        unsigned mask = 0u;
        int cur = -1;
        uint32_t from[2] = {rb, rb};  // the window of the saved sums
        for (uint32_t wb = rb; wb < rend; wb += 32u) {
            if (resolve) {
                const float2 x = f2_split(s.X), c0 = f2_split(s.c0), c1 = f2_split(s.c1), c2 = f2_split(s.c2);
                const float2 D = f2_split(s.D);
                auto save = [&](int h, float x, float c0, float c1, float c2, float D) {
                    float *sv = sh.sv + h * 7 * 32 + lane;
                    sv[0] = x, sv[32] = c0, sv[64] = c1, sv[96] = c2, sv[128] = D;
                    sv[160] = __int_as_float(s.last[h]), sv[192] = __int_as_float(s.nacc[h]);
                    from[h] = wb;
                };
                if (x.x >= 1.001f * kTMin || wb == rb) save(0, x.x, c0.x, c1.x, c2.x, D.x);
                if (x.y >= 1.001f * kTMin || wb == rb) save(1, x.y, c0.y, c1.y, c2.y, D.y);
            }
            const uint32_t g = g_next;
            if (e1 - wb > 32u + lane) g_next = a.point_list[wb + 32u + lane];
            const Hit *end = sh.buf + stage_window(a, g, wb + lane < rend, wb + lane + 1u - list0, bcx, bcy, kH, kH,
                                                   sh.buf, lane);
            for (const Hit *h = sh.buf; h != end; ++h) {
                const int c = (int)((h->pos - 1u - rpos) / kGwChunk);
                if (c != cur) {  // a new chunk (the same for the whole warp)
                    if (cur >= 0) sh.cp[cur * 32 + lane] = s.Tl, mask |= 1u << cur;
                    s.Tl = f2(1.f, 1.f);
                    cur = c;
                }
                if (h->odd != 0.f) blend_seg<true, false>(*h, pxf, s, c, 0, 0);
                else blend_seg<false, false>(*h, pxf, s, c, 0, 0);
            }
            __syncwarp();
        }
        if (cur >= 0) sh.cp[cur * 32 + lane] = s.Tl, mask |= 1u << cur;
        const float2 T0 = f2_split(s.Ts), Tr = f2_split(f2_mul(s.Ts, round_product(sh.cp, mask, nch, lane)));
        const bool low0 = live0 && Tr.x < kTMin, low1 = live1 && Tr.y < kTMin;
        float2 Tn = make_float2(live0 ? Tr.x : T0.x, live1 ? Tr.y : T0.y);
        if (!resolve) {
            s.npy = f2(low0 ? -INFINITY : y.x, low1 ? -INFINITY : y.y);
        } else if (__any_sync(kFull, low0 || low1)) {
            SegPix t = s;  // a copy: its address is taken
            t.npy = f2(y.x, y.y);
            resolve_round(a, e1, list0, pxf, bcx, bcy, nch, sh, lane, rb, rend, mask, low0, low1, from[0], from[1], &t);
            s = t;
            const float2 x = f2_split(s.X);
            if (low0) Tn.x = x.x;
            if (low1) Tn.y = x.y;
        }
        s.Ts = f2(Tn.x, Tn.y);
        rb = rend;
    }
}

// Where a block item's pixels lie: lane l owns rows l / 8 and l / 8 + 4 of column l % 8.
struct BlockGeom {
    TileGeom tg;
    int px, py0;
    bool in0, in1;
    float bcx, bcy;
};

__device__ __forceinline__ bool block_geom(const FwdArgs &a, int tile, int blk, int lane, BlockGeom &b) {
    const int nbx = (a.tile_w + kGwBlock - 1) / kGwBlock;
    b.tg = tile_geom(a, tile);
    const int ox = (blk % nbx) * kGwBlock, oy = (blk / nbx) * kGwBlock;
    if (ox >= b.tg.vw || oy >= b.tg.vh) return false;  // a block outside the image
    b.px = b.tg.x0 + ox + (lane & 7);
    b.py0 = b.tg.y0 + oy + (lane >> 3);
    const bool col = b.px < b.tg.x0 + b.tg.vw;
    b.in0 = col && b.py0 < b.tg.y0 + b.tg.vh;
    b.in1 = col && b.py0 + 4 < b.tg.y0 + b.tg.vh;
    b.bcx = (float)(b.tg.x0 + ox) + 0.5f * (kGwBlock - 1);
    b.bcy = (float)(b.tg.y0 + oy) + 0.5f * (kGwBlock - 1);
    return true;
}

__device__ __forceinline__ void start_walk(const BlockGeom &b, bool on0, bool on1, float T0, float T1, SegPix &s) {
    s.npy = f2(on0 ? -(float)b.py0 : -INFINITY, on1 ? -(float)(b.py0 + 4) : -INFINITY);
    s.Ts = f2(T0, T1);
    s.c0 = s.c1 = s.c2 = s.D = f2(0.f, 0.f);
    s.last[0] = s.last[1] = -1;
    s.nacc[0] = s.nacc[1] = s.stop[0] = s.stop[1] = 0;
}

// Writes a block's pixels (their final values) and counts them.
__device__ __forceinline__ void write_block(const FwdArgs &a, int tile, const BlockGeom &b, uint32_t n, const float *T,
                                            const float4 *cd, const int *last, const int *nacc, const int *stop,
                                            int lane, unsigned long long &st_eval, unsigned long long &st_acc) {
    int mlast = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!(h ? b.in1 : b.in0)) continue;
        const int neval = stop[h] ? stop[h] : (int)n;
        write_pixel(a, b.tg.v, b.px, b.py0 + 4 * h, T[h], cd[h].x, cd[h].y, cd[h].z, cd[h].w, last[h] + 1, neval);
        st_eval += (unsigned long long)neval;
        st_acc += (unsigned long long)nacc[h];
        mlast = max(mlast, last[h] + 1);
    }
    if (a.tile_cost) {
        mlast = __reduce_max_sync(kFull, mlast);
        if (lane == 0 && mlast > 0) atomicMax(a.tile_cost + tile, (unsigned int)mlast);
    }
}

// A block's segment with the composed transmittances (seg_walk).  A list of one segment, or a
// block whose pixels all stopped in the first, is written; else the summaries are stored.
// Returns whether the block's outputs were written.
__device__ __noinline__ bool block_composed(const FwdArgs &a, unsigned entry, int tile, uint32_t seg, int blk,
                                            const SegShared sh, int nch, int lane, unsigned long long *st) {
    BlockGeom b;
    block_geom(a, tile, blk, lane, b);
    const uint2 rg = load_range(a, tile);
    const uint32_t n = rg.y - rg.x, L = a.ctrl->gw_seg;
    const bool split = L != 0u && n > L;
    const uint32_t e0 = split ? rg.x + seg * L : rg.x;
    const uint32_t e1 = split && rg.y - e0 > L ? e0 + L : rg.y;
    SegPix s;
    start_walk(b, b.in0, b.in1, 1.f, 1.f, s);
    seg_walk(a, e0, e1, rg.x, (float)b.px, b.bcx, b.bcy, nch, seg == 0u, sh, lane, s);
    const float2 T = f2_split(s.Ts), c0 = f2_split(s.c0), c1 = f2_split(s.c1), c2 = f2_split(s.c2), D = f2_split(s.D);
    const float4 cd[2] = {make_float4(c0.x, c1.x, c2.x, D.x), make_float4(c0.y, c1.y, c2.y, D.y)};
    const float Ts[2] = {T.x, T.y};
    if (seg == 0u) {
        const bool open = (b.in0 && !s.stop[0]) || (b.in1 && !s.stop[1]);
        if (!split || !__any_sync(kFull, open)) {
            write_block(a, tile, b, n, Ts, cd, s.last, s.nacc, s.stop, lane, st[0], st[1]);
            return true;
        }
    }
    GwSum *out = reinterpret_cast<GwSum *>(a.gw_sum) + (size_t)entry * (a.tile_w * a.tile_h);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!(h ? b.in1 : b.in0)) continue;
        GwSum sm;
        sm.cd = cd[h];
        sm.t = make_float4(Ts[h], __int_as_float(s.last[h]), __int_as_float(s.nacc[h]), __int_as_float(s.stop[h]));
        out[(b.py0 + 4 * h - b.tg.y0) * b.tg.vw + (b.px - b.tg.x0)] = sm;
    }
    return false;
}

// One (segment, block) item.  The first segment is walked by the pixel-wise rule: where that
// ends every pixel's walk (all stopped, or the list has no other segment) and no
// transmittance came near the stop threshold, the stops are those of the composed products
// too, and the block is written and flagged, which spares its later segments and its merge.
// The other blocks, and the later segments, are walked with the composed products.  (On a 1080p
// view of 300k Gaussians under the plan's defaults: 2464 us with pixel-group items alone, 509
// with the composed walk on every block, 376 with this, 327 with two records at a time.)
__device__ __forceinline__ void block_item(const FwdArgs &a, unsigned entry, int blk, int nb, const SegShared &sh,
                                           int nch, int lane, unsigned long long *st) {
    const uint2 ent = a.gw_ent[entry];
    const int tile = (int)ent.x;
    const uint32_t seg = ent.y;
    uint32_t *done = a.gw_done + (size_t)a.gw_tile[tile].x * nb + blk;
    if (seg != 0u && *((volatile uint32_t *)done)) return;
    BlockGeom b;
    if (!block_geom(a, tile, blk, lane, b)) return;
    bool written = false;
    if (seg == 0u) {
        const uint2 rg = load_range(a, tile);
        const uint32_t n = rg.y - rg.x, L = a.ctrl->gw_seg;
        const bool split = L != 0u && n > L;
        PixAcc<2> s;
        s.npy[0] = f2(b.in0 ? -(float)b.py0 : -INFINITY, b.in1 ? -(float)(b.py0 + 4) : -INFINITY);
        s.T[0] = f2(1.f, 1.f);
        s.c0[0] = s.c1[0] = s.c2[0] = s.D[0] = f2(0.f, 0.f);
        s.last[0] = s.last[1] = 0;
        s.neval = reinterpret_cast<int *>(sh.sv) + lane;  // (free until a round is resolved)
        s.neval[0] = s.neval[32] = (int)n;
        s.nacc = 0;
        bool near = false;
        constexpr float kH = 0.5f * (kGwBlock - 1);
        walk_list<2, true>(a, rg.x, split ? rg.x + L : rg.y, (float)b.px, b.bcx, b.bcy, kH, kH, sh.buf, lane, s, &near);
        const float2 y = f2_split(s.npy[0]);  // -infinity: stopped (or outside the image)
        if (!__any_sync(kFull, near || (split && (y.x != -INFINITY || y.y != -INFINITY)))) {
            const float2 T = f2_split(s.T[0]), c0 = f2_split(s.c0[0]), c1 = f2_split(s.c1[0]), c2 = f2_split(s.c2[0]);
            const float2 D = f2_split(s.D[0]);
            int mlast = 0;
            if (b.in0) {
                write_pixel(a, b.tg.v, b.px, b.py0, T.x, c0.x, c1.x, c2.x, D.x, s.last[0], s.neval[0]);
                st[0] += (unsigned long long)s.neval[0];
                mlast = s.last[0];
            }
            if (b.in1) {
                write_pixel(a, b.tg.v, b.px, b.py0 + 4, T.y, c0.y, c1.y, c2.y, D.y, s.last[1], s.neval[32]);
                st[0] += (unsigned long long)s.neval[32];
                mlast = max(mlast, s.last[1]);
            }
            st[1] += (unsigned long long)s.nacc;
            if (a.tile_cost) {
                mlast = __reduce_max_sync(kFull, mlast);
                if (lane == 0 && mlast > 0) atomicMax(a.tile_cost + tile, (unsigned int)mlast);
            }
            written = true;
        }
    }
    if (!written) {
        unsigned long long t[2] = {0, 0};  // its address is taken
        written = block_composed(a, entry, tile, seg, blk, sh, nch, lane, t);
        st[0] += t[0];
        st[1] += t[1];
    }
    if (written && lane == 0) *((volatile uint32_t *)done) = 1u;
}

// Gaussian-wise items: blocks of pixels (gw_wide = 1) or, on work lists with few segments, pixel
// groups.  Launched first; lets the pixel-wise kernel launch as soon as all its blocks are
// resident (programmatic dependent launch), so that pixel-wise blocks take over SMs as
// Gaussian-wise blocks run out of items.
template <int P>
__global__ void __launch_bounds__(kGwWarps * 32, 5) k_forward_gauss(FwdArgs a) {
    asm volatile("griddepcontrol.launch_dependents;");
    __shared__ unsigned int blk_s[2];
    if (threadIdx.x == 0) blk_s[0] = blk_s[1] = 0u;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kNch = gw_chunks(P);
    const SegShared sh = seg_shared(warp, kNch);
    const bool wide = a.ctrl->gw_wide != 0u;
    const unsigned num_items = a.ctrl->num_gauss, chunk = (unsigned)a.chunk;
    const unsigned per = wide ? (unsigned)gw_blocks_per(a.tile_w, a.tile_h) : (unsigned)(a.tile_w * a.tile_h + P - 1) / P;
    unsigned long long st[2] = {0, 0}, st_items = 0;  // evaluated and contributing pairs
    while (true) {
        unsigned first = 0;
        if (lane == 0) first = atomicAdd(&a.ctrl->queue_head_g, chunk);
        first = __shfl_sync(kFull, first, 0);
        if (first >= num_items) break;
        const unsigned end = min(first + chunk, num_items);
        for (unsigned it = first; it < end; ++it) {
            const unsigned entry = it / per, sub = it - entry * per;
            if (wide) {
                block_item(a, entry, (int)sub, (int)per, sh, kNch, lane, st);
            } else {
                const uint2 ent = a.gw_ent[entry];
                gw_segment_item<P>(a, (int)ent.x, (int)ent.y, (int)sub, entry,
                                   reinterpret_cast<uint32_t *>(sh.buf), lane);
            }
            ++st_items;
        }
    }
    flush_stats(a, lane, st[0], st[1], st_items);
    if (lane == 0) finish_pass(a.ctrl, st_items, blk_s, kGwWarps, a.pass_blocks);
}

// A warp per 8 x 8 block of a Gaussian-wise tile that has no outputs yet: composes its pixels'
// segment summaries in list order with (C1, T1) o (C2, T2) = (C1 + T1 C2, T1 T2) while the
// composed transmittance stays >= 1e-4; a segment in which it would fall below is walked again
// from the exact incoming transmittance with the stop resolved (seg_walk, for the block's
// pixels that cross there together), after which the composition goes on if the walk did not
// stop.  Writes the pixels' outputs and counts their evaluated and contributing pairs.
constexpr int kMergeWarps = 3;  // their 32-chunk regions fit the default 48 KB

__global__ void __launch_bounds__(kMergeWarps * 32) k_forward_gw_merge(FwdArgs a) {
    constexpr int kNch = 32;  // the chunks of a walk for one pixel
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nb = gw_blocks_per(a.tile_w, a.tile_h);
    const SegShared sh = seg_shared(warp, kNch);
    const unsigned num = a.ctrl->gw_first * (unsigned)nb;
    const uint32_t L = a.ctrl->gw_seg;
    const bool wide = a.ctrl->gw_wide != 0u;
    const size_t NP = (size_t)(a.tile_w * a.tile_h);
    unsigned long long st_eval = 0, st_acc = 0;
    for (unsigned it = blockIdx.x * kMergeWarps + warp; it < num; it += gridDim.x * kMergeWarps) {
        if (wide && a.gw_done[it]) continue;
        const int tile = (int)a.gw_ent[it / nb].x;
        BlockGeom b;
        if (!block_geom(a, tile, (int)(it % nb), lane, b)) continue;
        const uint2 rg = load_range(a, tile);
        const uint32_t n = rg.y - rg.x;
        const uint32_t S = (n == 0u || L == 0u) ? 1u : (n - 1u) / L + 1u;
        const uint2 gt = a.gw_tile[tile];
        const bool in[2] = {b.in0, b.in1};
        GwSum *pix[2];  // the pixel's summary in entry 0
#pragma unroll
        for (int h = 0; h < 2; ++h)
            pix[h] = reinterpret_cast<GwSum *>(a.gw_sum) + (b.py0 + 4 * h - b.tg.y0) * b.tg.vw + (b.px - b.tg.x0);
        auto slot = [&](int h, uint32_t sg) { return pix[h] + (size_t)(sg == 0u ? gt.x : gt.y + sg - 1u) * NP; };
        float T[2] = {1.f, 1.f};
        float4 cd[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
        int last[2] = {-1, -1}, nacc[2] = {0, 0}, stop[2] = {0, 0};
        uint32_t s_end[2] = {S - 1u, S - 1u};  // the last segment the pixel reaches
        bool on[2] = {in[0], in[1]};
        GwSum next[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (on[h]) next[h] = *slot(h, 0u);
        for (uint32_t sg = 0; sg < S; ++sg) {
            GwSum sm[2] = {next[0], next[1]};
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (on[h] && sg + 1u < S) next[h] = *slot(h, sg + 1u);
            float4 ab[2];  // the segment's colour and depth with absolute weights
            float T_in[2] = {T[0], T[1]};
            bool cross[2] = {false, false}, wrote[2] = {false, false};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!on[h]) continue;
                const int sst = __float_as_int(sm[h].t.w);
                if (sg == 0u && sst) {  // stopped in the first segment, resolved there
                    T[h] = sm[h].t.x;
                    cd[h] = sm[h].cd;
                    last[h] = __float_as_int(sm[h].t.y);
                    nacc[h] = __float_as_int(sm[h].t.z);
                    stop[h] = sst;
                    s_end[h] = 0u;
                    on[h] = false;
                } else if (T[h] * sm[h].t.x >= kTMin) {
                    const float4 c = sm[h].cd;
                    ab[h] = make_float4(T[h] * c.x, T[h] * c.y, T[h] * c.z, T[h] * c.w);
                    T[h] *= sm[h].t.x;
                    last[h] = max(last[h], __float_as_int(sm[h].t.y));
                    nacc[h] += __float_as_int(sm[h].t.z);
                    wrote[h] = true;
                } else {
                    cross[h] = true;
                }
            }
            if (__any_sync(kFull, cross[0] || cross[1])) {
                const uint32_t e0 = S > 1u ? rg.x + sg * L : rg.x;
                const uint32_t e1 = S > 1u && rg.y - e0 > L ? e0 + L : rg.y;
                SegPix s;
                start_walk(b, cross[0], cross[1], T[0], T[1], s);
                seg_walk(a, e0, e1, rg.x, (float)b.px, b.bcx, b.bcy, kNch, true, sh, lane, s);
                const float2 Tw = f2_split(s.Ts), c0 = f2_split(s.c0), c1 = f2_split(s.c1), c2 = f2_split(s.c2);
                const float2 D = f2_split(s.D);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!cross[h]) continue;
                    ab[h] = h ? make_float4(c0.y, c1.y, c2.y, D.y) : make_float4(c0.x, c1.x, c2.x, D.x);
                    T[h] = h ? Tw.y : Tw.x;
                    last[h] = max(last[h], s.last[h]);
                    nacc[h] += s.nacc[h];
                    wrote[h] = true;
                    if (s.stop[h]) {
                        stop[h] = s.stop[h];
                        s_end[h] = sg;
                        on[h] = false;
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!wrote[h]) continue;
                cd[h].x += ab[h].x, cd[h].y += ab[h].y, cd[h].z += ab[h].z, cd[h].w += ab[h].w;
                // the slot now holds the segment's absolute contribution and entry T (the
                // backward's boundary states are formed from them below)
                if (S > 1u) {
                    GwSum o;
                    o.cd = ab[h];
                    o.t = make_float4(T_in[h], 0.f, 0.f, 0.f);
                    *slot(h, sg) = o;
                }
            }
            if (!__any_sync(kFull, on[0] || on[1])) break;
        }
        // Boundary states for a segmented backward: per segment u the pixel reaches, the
        // transmittance behind it (in front of segment u + 1, or the final T) and the
        // colour and depth accumulated behind it with absolute weights, background
        // included -- summed from the back, so no difference of two sums is formed.
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!in[h] || S == 1u || s_end[h] == 0u) continue;
            float b0 = T[h] * a.bg[0], b1 = T[h] * a.bg[1], b2 = T[h] * a.bg[2], bd = 0.f, Tnext = T[h];
            for (int u = (int)s_end[h]; u >= 0; --u) {
                GwSum *p = slot(h, (uint32_t)u);
                const GwSum sm = *p;
                GwSum o;
                o.cd = make_float4(b0, b1, b2, bd);
                o.t = make_float4(Tnext, 0.f, 0.f, 0.f);
                *p = o;
                b0 += sm.cd.x, b1 += sm.cd.y, b2 += sm.cd.z, bd += sm.cd.w;
                Tnext = sm.t.x;
            }
        }
        write_block(a, tile, b, n, T, cd, last, nacc, stop, lane, st_eval, st_acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        st_eval += __shfl_xor_sync(kFull, st_eval, o);
        st_acc += __shfl_xor_sync(kFull, st_acc, o);
    }
    if (lane == 0 && (st_eval | st_acc)) {
        atomicAdd(&a.ctrl->eval_pairs, st_eval);
        atomicAdd(&a.ctrl->contrib_pairs, st_acc);
    }
}

// Pixel-wise items [num_gauss, num_items) of the work list.
template <int Q>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, Q == 4 ? 3 : 0) k_forward_pixel(FwdArgs a) {
    __shared__ Hit sbuf[kWarpsPerBlock][32];
    __shared__ int neval[kWarpsPerBlock][32 * 2 * PixAcc<Q>::NP];
    __shared__ unsigned int blk[2];
    if (threadIdx.x == 0) blk[0] = blk[1] = 0u;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Hit *buf = sbuf[warp];
    const unsigned num_items = a.ctrl->num_items, num_gauss = a.ctrl->num_gauss;
    const unsigned chunk = (unsigned)a.chunk;
    unsigned long long st_eval = 0, st_acc = 0, st_items = 0;
    while (true) {
        unsigned first = 0;
        if (lane == 0) first = atomicAdd(&a.ctrl->queue_head, chunk);
        first = __shfl_sync(kFull, first, 0);
        if (first >= num_items) break;
        const unsigned end = min(first + chunk, num_items);
        for (unsigned it = first; it < end; ++it) {
            const uint2 item = a.items[it - num_gauss];
            pixel_item<Q>(a, (int)item.x, (int)item.y, buf, neval[threadIdx.x >> 5], lane, st_eval, st_acc);
            ++st_items;
        }
    }
    flush_stats(a, lane, st_eval, st_acc, st_items);
    if (lane == 0) finish_pass(a.ctrl, st_items, blk, kWarpsPerBlock, a.pass_blocks);
    // launched after k_forward_gauss with programmatic serialisation: complete only once the
    // Gaussian-wise grid has (so that whatever follows on the stream, the merge included,
    // sees its summaries); a no-op for an ordinary launch
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

int forward_balanced_block_threads() { return kWarpsPerBlock * 32; }

const void *forward_gauss_kernel(int gw_pixels) {
    switch (gw_pixels) {
        case 1: return (const void *)k_forward_gauss<1>;
        case 2: return (const void *)k_forward_gauss<2>;
        case 4: return (const void *)k_forward_gauss<4>;
        case 8: return (const void *)k_forward_gauss<8>;
        case 16: return (const void *)k_forward_gauss<16>;
        default: return nullptr;
    }
}

const void *forward_pixel_kernel(int pixel_rows) {
    switch (pixel_rows) {
        case 1: return (const void *)k_forward_pixel<1>;
        case 2: return (const void *)k_forward_pixel<2>;
        case 4: return (const void *)k_forward_pixel<4>;
        case 8: return (const void *)k_forward_pixel<8>;
        default: return nullptr;
    }
}

// Shared memory of a block of k_forward_gauss: a warp's regions (above the 48 KB default for
// groups of 1 and 2 pixels, whose rounds have 32 chunks).
static_assert(32 * sizeof(Hit) >= kGwIdx * sizeof(uint32_t), "a pixel group's indices fit the window");

static size_t gauss_smem(int gw_pixels) { return kGwWarps * seg_shared_bytes(gw_chunks(gw_pixels)); }

int forward_gauss_grid(const FwdArgs &a, int num_sms, int max_per_sm) {
    const void *k = forward_gauss_kernel(a.gw_pixels);
    const size_t smem = gauss_smem(a.gw_pixels);
    int per_sm = 0;
    if (!k || (smem > 48 * 1024 &&
               cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kGwWarps * 32, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    if (max_per_sm > 0 && per_sm > max_per_sm) per_sm = max_per_sm;
    return num_sms * per_sm;
}

cudaError_t launch_forward_gauss(const FwdArgs &a, int grid, cudaStream_t s) {
    const void *k = forward_gauss_kernel(a.gw_pixels);
    if (!k) return cudaErrorInvalidValue;
    FwdArgs arg = a;
    void *params[] = {&arg};
    return cudaLaunchKernel(k, dim3(grid), dim3(kGwWarps * 32), params, gauss_smem(a.gw_pixels), s);
}

cudaError_t launch_forward_gw_merge(const FwdArgs &a, int num_sms, cudaStream_t s) {
    k_forward_gw_merge<<<num_sms * 4, kMergeWarps * 32, kMergeWarps * seg_shared_bytes(32), s>>>(a);
    return cudaGetLastError();
}

// after_gauss: launched right after k_forward_gauss on the same stream, with programmatic
// stream serialisation (the two kernels touch disjoint pixels and k_forward_gauss started
// after the work list was complete, so no wait is needed).  Otherwise an ordinary launch:
// the kernel has no grid-dependency wait, so it must not overlap the kernels that build
// its work list.
cudaError_t launch_forward_pixel(const FwdArgs &a, int grid, bool after_gauss, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kWarpsPerBlock * 32);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = after_gauss ? 1 : 0;
    switch (a.pixel_rows) {
        case 1: return cudaLaunchKernelEx(&cfg, k_forward_pixel<1>, a);
        case 2: return cudaLaunchKernelEx(&cfg, k_forward_pixel<2>, a);
        case 4: return cudaLaunchKernelEx(&cfg, k_forward_pixel<4>, a);
        case 8: return cudaLaunchKernelEx(&cfg, k_forward_pixel<8>, a);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bgs
