// render_bwd.cu -- a6: backward render kernels.
//
// The paper describes only the forward kernel; its backward (Sec. 3 cites the L2
// atomic bottleneck of 3DGS gradients) is derived here from Eq. 4.  With
// T_i = prod_{j<i}(1 - alpha_j), R_i the colour accumulated behind entry i normalised by
// T_{i+1} (R starts at the background), and T_f the final transmittance:
//   dL/dc_i      = alpha_i T_i dL/dC
//   dL/dalpha_i  = T_i [ (c_i - R_i) . dL/dC + (d_i - Rd_i) dL/dD ] + T_f/(1-alpha_i) dL/dA
//   R_{i-1}      = alpha_i c_i + (1 - alpha_i) R_i       (same for depth, Rd starts at 0)
// and alpha = min(0.99, o G), G = exp(power): dL/do = G dL/dalpha and dL/dpower =
// o G dL/dalpha where the clamp is inactive (both 0 where o G > 0.99).
// Each pixel walks its tile's list from its last contributor back to the front,
// recovering T_i = T_{i+1} / (1 - alpha_i) from the stored final T (no per-pair state is
// kept by the forward).  All lanes of a warp visit the same list entry at the same step,
// so the per-Gaussian contributions of the warp's pixels are summed with shuffles and added
// to a packed accumulator [N][12] with two red.add instructions (warp-aggregated atomics).
// With gp = dL/dpower2 of a pair, the mean and conic gradients of a Gaussian are sums of
// gp times (dx, dy, dx^2, dx dy, dy^2) combined with the Gaussian's (constant) conic, so a
// lane only sums gp, gp dy and gp dy^2 over its pixels (which share dx), forms the five
// moments once, and the conic is applied after the warp sum.  Two identities shorten the
// per-pair work: R_i enters dL/dalpha only through R_i . dL/dC, so a pixel carries that
// scalar (updated by the same recurrence) instead of R_i; and dL/do = sum G dL/dalpha =
// (sum gp) / o, so the opacity gradient is the gp sum, divided by o once per Gaussian in the
// final pass, which scales and scatters the accumulator into the ABI's gradient arrays.
#include <algorithm>

#include "bgs_internal.cuh"

namespace bgs {

constexpr unsigned kFullB = 0xffffffffu;
constexpr int kBwdWarps = 8;

struct PixState {
    float T, Tf, g0, g1, g2, gD, gA;
    float Rg, Rd;  // R . dL/dC (colour behind the entry, dotted with the pixel's colour gradient), depth behind
    int nc;
};

__device__ __forceinline__ PixState load_pixel(const BwdArgs &a, int v, int px, int py, bool inside) {
    PixState s;
    if (inside) {
        const int W = a.vt.W[v];
        const long long HW = (long long)W * a.vt.H[v];
        const long long pid = (long long)py * W + px;
        s.T = a.gi.final_T[v][pid];
        s.nc = a.gi.n_contrib[v][pid];
        const float *gc = a.gi.dL_dcolor[v];
        s.g0 = gc[pid];
        s.g1 = gc[HW + pid];
        s.g2 = gc[2 * HW + pid];
        s.gD = a.gi.dL_ddepth[v] ? a.gi.dL_ddepth[v][pid] : 0.f;
        s.gA = a.gi.dL_dalpha[v] ? a.gi.dL_dalpha[v][pid] : 0.f;
    } else {
        s.T = 1.f;
        s.nc = 0;
        s.g0 = s.g1 = s.g2 = s.gD = s.gA = 0.f;
    }
    s.Tf = s.T;
    s.Rg = a.bg[0] * s.g0 + a.bg[1] * s.g1 + a.bg[2] * s.g2;
    s.Rd = 0.f;
    return s;
}

// Per-lane sums of one record's pair contributions over the lane's pixels.
struct PairSums {
    float g, gy, gyy;  // sum of gp, gp dy, gp dy^2 (gp = dL/dpower2, power2 the log2 exponent)
    float c0, c1, c2;  // sum of alpha T dL/dC           (-> dL/dcolour)
    float d;           // sum of alpha T dL/dD           (-> dL/ddepth)
};

__device__ __forceinline__ PairSums zero_sums() {
    PairSums a;
    a.g = a.gy = a.gyy = a.c0 = a.c1 = a.c2 = a.d = 0.f;
    return a;
}

// One (pixel, entry) step of the backward walk: adds the pair's contributions to a
// (nothing when the pair is skipped).  dL/dalpha_i = T_i [(c_i - R_i) . dL/dC + (d_i - Rd_i)
// dL/dD] + T_f / (1 - alpha_i) dL/dA; then R_{i-1} = R_i + alpha_i (c_i - R_i), carried as
// Rg = R . dL/dC.  Extra = false: no depth / alpha output gradients (dL/dD = dL/dA = 0), their
// terms are compiled out.
template <bool Extra>
__device__ __forceinline__ bool pair_backward(const Rec &r, const PairX &x, float pyf, bool active, PixState &s,
                                              PairSums &a) {
    float dy;
    const float p2 = pair_power2_y(x, r.a.y, r.b.x, pyf, dy);
    const float oG = pair_oG(p2, r.b.y);
    const bool valid = active && p2 <= 0.f && oG >= kAlphaMin;
    if (valid) {
        const float al = fminf(kAlphaMax, oG);
        const float om = 1.f - al;
        const float io = rcp_approx(om);  // om in [0.01, 1]
        s.T = s.T * io;                   // T_i
        const float w = al * s.T;
        a.c0 += w * s.g0;
        a.c1 += w * s.g1;
        a.c2 += w * s.g2;
        const float diff = (r.c.x * s.g0 + r.c.y * s.g1 + r.c.z * s.g2) - s.Rg;  // (c_i - R_i) . dL/dC
        float dLda = s.T * diff;
        if (Extra) {
            a.d += w * s.gD;
            const float dd = r.c.w - s.Rd;
            dLda += s.T * dd * s.gD + s.Tf * io * s.gA;
            s.Rd += al * dd;
        }
        s.Rg += al * diff;
        // alpha = min(0.99, o G): no gradient through the clamp (branch-free)
        const float gp = oG <= kAlphaMax ? oG * dLda : 0.f;  // dL/dpower2 = o G dL/dalpha
        const float gpy = gp * dy;
        a.g += gp;
        a.gy += gpy;
        a.gyy += gpy * dy;
    }
    return valid;
}

// Adds the lane sums of one record, over the warp's 32 lanes, to the record's accumulator
// row acc[0..9]:
//   acc0..4 = sum gp (dx, dy, dx^2, dx dy, dy^2), acc5 = sum gp (= o sum G dL/dalpha),
//   acc6..8 = colour sums, acc9 = depth sum
// (dx = mean_x - px is shared by the lane's pixels; the final pass applies the Gaussian's
// conic to the first two moments, once per Gaussian).  The eight values (the five moments,
// sum gp, two colour channels) are reduced by recursive halving over lane bits 4, 3, 2
// (4 + 2 + 1 shuffles), leaving in lane l the sum of element (l >> 2) & 7 over the 8 lanes
// that share l's bits 1, 0; the third colour channel (and the depth sum, halved against it
// over bit 4) takes three butterflies.  The four partial sums of every value are then added
// by the atomics themselves: one red.add instruction from all 32 lanes for the eight
// values, one from lanes 0-3 (and 16-19) for colour channel 2 (and depth).  Stopping the
// trees two levels early shortens the per-record dependency chain by two shuffles; L2
// absorbs the extra atomic operations.
template <bool Extra>
__device__ __forceinline__ void warp_reduce_red(const PairSums &s, float dx, float *acc, int lane) {
    const float sdx = dx * s.g;
    float v[8] = {sdx, s.gy, dx * sdx, dx * s.gy, s.gyy, s.g, s.c0, s.c1};
    float h4[4], h2[2];
    {
        const bool hi = (lane & 16) != 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float send = hi ? v[j] : v[j + 4];
            h4[j] = (hi ? v[j + 4] : v[j]) + __shfl_xor_sync(kFullB, send, 16);
        }
    }
    {
        const bool hi = (lane & 8) != 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float send = hi ? h4[j] : h4[j + 2];
            h2[j] = (hi ? h4[j + 2] : h4[j]) + __shfl_xor_sync(kFullB, send, 8);
        }
    }
    float t;
    {
        const bool hi = (lane & 4) != 0;
        t = (hi ? h2[1] : h2[0]) + __shfl_xor_sync(kFullB, hi ? h2[0] : h2[1], 4);
    }
    float u;  // colour channel 2 (lanes with bit 4 clear) / depth (bit 4 set) when Extra
    if (Extra) {
        const bool hi = (lane & 16) != 0;
        u = (hi ? s.d : s.c2) + __shfl_xor_sync(kFullB, hi ? s.c2 : s.d, 16);
    } else {
        u = s.c2 + __shfl_xor_sync(kFullB, s.c2, 16);
    }
    u += __shfl_xor_sync(kFullB, u, 8);
    u += __shfl_xor_sync(kFullB, u, 4);
    if (t != 0.f) atomicAdd(acc + ((lane >> 2) & 7), t);
    const bool ul = Extra ? (lane & 12) == 0 : lane < 4;  // lanes 0-3 (and 16-19)
    if (ul && u != 0.f) atomicAdd(acc + ((Extra && (lane & 16)) ? 9 : 8), u);
}

__device__ __forceinline__ uint2 load_range_bwd(const BwdArgs &a, int tile) {
    uint2 rg = a.ranges[tile];
    if (rg.y < rg.x || (long long)rg.y > a.num_entries) {
        raise_check(a.ctrl, BGS_CHECK_RANGE);
        rg = make_uint2(0, 0);
    }
    return rg;
}

// =====================================================================================
// plain pixel-wise static backward: one block per tile, block-wide staging
// =====================================================================================
__global__ void __launch_bounds__(1024) k_backward_static(BwdArgs a) {
    extern __shared__ Rec srec[];  // [nthreads] records, then [nthreads] indices
    __shared__ int s_max;
    const int nthreads = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    const int tile = blockIdx.x;  // single view
    const int tx = tile % a.vt.tiles_x[0], ty = tile / a.vt.tiles_x[0];
    const int px = tx * a.tile_w + tid % a.tile_w, py = ty * a.tile_h + tid / a.tile_w;
    const bool inside = px < a.vt.W[0] && py < a.vt.H[0];
    uint2 rg = a.ranges[tile];
    if (rg.y < rg.x || (long long)rg.y > a.num_entries) {
        if (tid == 0) raise_check(a.ctrl, BGS_CHECK_RANGE);
        rg = make_uint2(0, 0);
    }
    PixState s = load_pixel(a, 0, px, py, inside);
    if (s.nc > (int)(rg.y - rg.x)) s.nc = (int)(rg.y - rg.x);
    if (tid == 0) s_max = 0;
    __syncthreads();
    atomicMax(&s_max, s.nc);
    __syncthreads();
    const uint32_t hi = rg.x + (uint32_t)s_max;
    const float pxf = (float)px, pyf = (float)py;
    uint32_t *sidx = reinterpret_cast<uint32_t *>(srec + nthreads);
    for (uint32_t top = hi; top > rg.x; top -= min((uint32_t)nthreads, top - rg.x)) {
        const uint32_t lo = top - min((uint32_t)nthreads, top - rg.x);
        const int cnt = (int)(top - lo);
        __syncthreads();
        if (tid < cnt) {
            const uint32_t j = top - 1 - tid;
            const uint32_t g = a.point_list[j];
            Rec r;
            if ((long long)g < a.N) {
                r = make_rec(a.means2D, a.conic_opacity, a.colors, a.depths, g);
            } else {
                raise_check(a.ctrl, BGS_CHECK_INDEX);
                r.a = make_float4(0.f, 0.f, 0.f, 0.f);
                r.b = r.a;
                r.c = r.a;
            }
            srec[tid] = r;
            sidx[tid] = (long long)g < a.N ? g : 0u;
        }
        __syncthreads();
        for (int k = 0; k < cnt; ++k) {
            const Rec r = srec[k];
            const int pos = (int)(top - 1 - k - rg.x);
            const PairX x = pair_x(r.a, pxf);
            PairSums sums = zero_sums();
            const bool valid = pair_backward<true>(r, x, pyf, pos < s.nc, s, sums);
            if (__any_sync(kFullB, valid)) warp_reduce_red<true>(sums, x.dx, a.grad_acc + 12ull * sidx[k], lane);
        }
    }
}

cudaError_t launch_backward_static(const BwdArgs &a, cudaStream_t s) {
    const int threads = a.tile_w * a.tile_h;
    const int tiles = a.vt.tiles_x[0] * a.vt.tiles_y[0];
    if (tiles == 0) return cudaSuccess;
    k_backward_static<<<tiles, threads, (sizeof(Rec) + sizeof(uint32_t)) * threads, s>>>(a);
    return cudaGetLastError();
}

// =====================================================================================
// balanced persistent backward: warps pull pixel-wise items (8x4 sub-blocks)
// =====================================================================================
// A record of a window as the backward items read it: the values that meet two pixels at a
// time stand there twice.
struct __align__(16) HitB {
    float mx, qa, qb;
    int pos;  // position in the tile's list
    F2 my, qc;
    F2 o, r;
    F2 g, b;
    F2 d;
    uint32_t idx;
    float odd;  // record_odd
};

// A lane's pixels, two to a pair (rows 2p and 2p + 1 of the lane's column).  The walk carries
// -R . dL/dC and -Rd, and amin is 1/255 once a pixel takes part (infinity before its last
// contributor, so that none of its pairs passes).
template <int Q, bool Extra>
struct PixGrad {
    static constexpr int NP = (Q + 1) / 2, NE = Extra ? NP : 1;
    F2 npy[NP], T[NP], g0[NP], g1[NP], g2[NP], nRg[NP];
    F2 gD[NE], TfA[NE], nRd[NE];  // depth gradient, T_f dL/dA, -Rd
    float amin[2 * NP];
    int nc[2 * NP];  // one past the last contributor (0 once the pixel takes part)
    int next;        // the largest nc left
};

// One record on the lane's pixels, two pixels per instruction: pair_backward's sums (see
// there) without a branch.  A pair that is not accumulated has alpha = 0 (the pixel's values are
// tame, see bwd_pixel_item).  Odd = false (record_odd): without the sign test and the clamp, so
// that o G is alpha; Odd = true: the pair rule in full, (c - R) . dL/dC and o G selected.  Returns
// whether any pixel accumulated.  28 % fewer instructions than a branch per pair (which the
// latency of the chain, the shuffles among it, turns into 4-8 %: 3.03 instead of 3.17 ms on the
// 9-view 4M-Gaussian step, 330 instead of 359 us on a 720p early-stage view with depth and
// alpha gradients).
template <int Q, bool Extra, bool Odd>
__device__ __forceinline__ bool hit_backward(const HitB &h, const float4 h0, float dx, PixGrad<Q, Extra> &s,
                                             PairSums &sums) {
    constexpr int NP = PixGrad<Q, Extra>::NP;
    const ulonglong2 h1 = *reinterpret_cast<const ulonglong2 *>(&h.my);
    const ulonglong2 h2 = *reinterpret_cast<const ulonglong2 *>(&h.o);
    const ulonglong2 h3 = *reinterpret_cast<const ulonglong2 *>(&h.g);
    const float hx = __fmul_rn(__fmul_rn(h0.y, dx), dx), bx = __fmul_rn(h0.z, dx);
    const F2 hx2 = f2(hx, hx), bx2 = f2(bx, bx), one = f2(1.f, 1.f);
    F2 g = f2(0.f, 0.f), gy = g, gyy = g, c0 = g, c1 = g, c2 = g, d = g;
    bool any = false;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const F2 dy = f2_add(h1.x, s.npy[p]);
        const float2 e = f2_split(f2_fma(dy, f2_fma(h1.y, dy, bx2), hx2));
        const float2 oG = f2_split(f2_mul(h2.x, f2(ex2_approx(e.x), Q == 1 ? 0.f : ex2_approx(e.y))));
        const bool v0 = (!Odd || e.x <= 0.f) && oG.x >= s.amin[2 * p];
        const bool v1 = Q > 1 && (!Odd || e.y <= 0.f) && oG.y >= s.amin[2 * p + 1];
        any = any || v0 || v1;
        auto neg = [](float x) { return Odd ? fmaxf(-kAlphaMax, -x) : -x; };
        const F2 nal = f2(v0 ? neg(oG.x) : 0.f, v1 ? neg(oG.y) : 0.f);
        const float2 om = f2_split(f2_add(one, nal));  // 1 - alpha, in [0.01, 1]
        const F2 io = f2(rcp_approx(om.x), rcp_approx(om.y));  // 1 for a masked pair (measured exact)
        s.T[p] = f2_mul(s.T[p], io);  // T_i
        const F2 nw = f2_mul(nal, s.T[p]);
        c0 = f2_fma(nw, s.g0[p], c0);
        c1 = f2_fma(nw, s.g1[p], c1);
        c2 = f2_fma(nw, s.g2[p], c2);
        // (c_i - R_i) . dL/dC
        const float2 cd = f2_split(f2_fma(h3.y, s.g2[p], f2_fma(h3.x, s.g1[p], f2_fma(h2.y, s.g0[p], s.nRg[p]))));
        const F2 diff = f2(!Odd || v0 ? cd.x : 0.f, !Odd || v1 ? cd.y : 0.f);
        F2 dLda = f2_mul(s.T[p], diff);
        if (Extra) {
            d = f2_fma(nw, s.gD[p], d);
            const float2 de = f2_split(f2_add(h.d, s.nRd[p]));
            const F2 dd = f2(!Odd || v0 ? de.x : 0.f, !Odd || v1 ? de.y : 0.f);
            dLda = f2_fma(f2_mul(s.T[p], dd), s.gD[p], f2_fma(s.TfA[p], io, dLda));
            s.nRd[p] = f2_fma(nal, dd, s.nRd[p]);
        }
        s.nRg[p] = f2_fma(nal, diff, s.nRg[p]);
        // -dL/dpower2 = -o G dL/dalpha, none through the clamp
        const F2 gp = f2_mul(!Odd ? nal
                                  : f2(v0 && oG.x <= kAlphaMax ? -oG.x : 0.f, v1 && oG.y <= kAlphaMax ? -oG.y : 0.f),
                             dLda);
        const F2 gpy = f2_mul(gp, dy);
        g = f2_add(g, gp);
        gy = f2_add(gy, gpy);
        gyy = f2_fma(gpy, dy, gyy);
    }
    auto fold = [](F2 x) {
        const float2 u = f2_split(x);
        return u.x + u.y;
    };
    sums.g = -fold(g), sums.gy = -fold(gy), sums.gyy = -fold(gyy);
    sums.c0 = -fold(c0), sums.c1 = -fold(c1), sums.c2 = -fold(c2);
    sums.d = Extra ? -fold(d) : 0.f;
    return any;
}

// Where a pixel-wise item lies: its tile's visible part, the span of the tile's list that it
// walks (a segment of a tile that the last forward split, seg >= 0; else the whole list) and
// its first pixel.
struct ItemGeom {
    int v, tile, x0, y0, vw, vh, seg, sx, sy;
    uint2 rg;
    uint32_t e0, e1;
};

template <int Q>
__device__ __forceinline__ ItemGeom item_geom(const BwdArgs &a, int tile, int sub, unsigned L) {
    ItemGeom g;
    g.v = view_of(a.vt, tile);
    g.tile = tile;
    const int lt = tile - a.vt.tile_base[g.v];
    g.x0 = (lt % a.vt.tiles_x[g.v]) * a.tile_w;
    g.y0 = (lt / a.vt.tiles_x[g.v]) * a.tile_h;
    g.vw = min(a.tile_w, a.vt.W[g.v] - g.x0);
    g.vh = min(a.tile_h, a.vt.H[g.v] - g.y0);
    const int cxs = (g.vw + pix_item_w(Q) - 1) / pix_item_w(Q);
    g.rg = load_range_bwd(a, tile);
    const uint32_t n = g.rg.y - g.rg.x;
    g.seg = -1;
    g.e0 = g.rg.x;
    g.e1 = g.rg.y;
    if (L != 0u && n > L && tile_is_gauss(a.bseg_mode, a.heavy_threshold, n)) {
        const int per_tile = cxs * ((g.vh + pix_item_h(Q) - 1) / pix_item_h(Q));
        g.seg = sub / per_tile;
        sub -= g.seg * per_tile;
        g.e0 = g.rg.x + (uint32_t)g.seg * L;
        g.e1 = (uint32_t)min((unsigned long long)g.rg.y, (unsigned long long)g.e0 + L);
    }
    g.sx = sub % cxs;
    g.sy = sub / cxs;
    return g;
}

// The state in which a pixel enters the item's span from behind; nc = 0 where it has nothing in it.
__device__ __forceinline__ PixState enter_pixel(const BwdArgs &a, const ItemGeom &g, int px, int py, bool inside) {
    PixState t = load_pixel(a, g.v, px, py, inside);
    t.nc = max(min(t.nc, (int)(g.rg.y - g.rg.x)), 0);
    if (g.seg >= 0) {
        const uint32_t end = g.rg.x + (uint32_t)t.nc;  // one past the last contributor
        if (end <= g.e0) {
            t.nc = 0;  // nothing of this pixel in the segment
        } else if (end >= g.e1 && inside) {
            // enter from behind: the merge's state at the segment's end
            const uint2 gt = a.gw_tile[g.tile];
            const size_t entry = g.seg == 0 ? (size_t)gt.x : (size_t)gt.y + (size_t)(g.seg - 1);
            const GwSum st = a.gw_sum[entry * (size_t)(a.tile_w * a.tile_h) + (py - g.y0) * g.vw + (px - g.x0)];
            const float iT = 1.f / st.t.x;
            t.T = st.t.x;
            t.Rg = (st.cd.x * t.g0 + st.cd.y * t.g1 + st.cd.z * t.g2) * iT;
            t.Rd = st.cd.w * iT;
            t.nc = (int)(g.e1 - g.rg.x);
        }
    }
    return t;
}

// Pixel-wise item: an 8 x 4Q sub-block; lane l owns the pixels (l % 8, l / 8 + 4 q).  The
// lane adds its pixels' contributions before the warp-wide reduction, so one reduction
// serves 32 Q pixels.  In a tile that the last forward split into segments of L entries
// (Gaussian-wise, reading the forward's boundary states), the item walks one segment
// [e0, e1) of the list: a pixel whose last contributor lies behind the segment enters it
// with the state the merge stored for it (T behind the segment, colour and depth behind it
// over that T); one whose last contributor lies inside starts there as usual; the others
// have nothing in it.  Returns false, with nothing done, when a pixel's values are not tame (0
// times them is not 0, see hit_backward): bwd_pixel_item_wild takes the item then.
template <int Q, bool Extra>
__device__ __forceinline__ bool bwd_pixel_item(const BwdArgs &a, const ItemGeom &ig, HitB *buf, int lane) {
    constexpr int kItemW = pix_item_w(Q), kItemH = pix_item_h(Q), kRowStep = pix_row_step(Q);
    const int px = ig.x0 + ig.sx * kItemW + (lane % kItemW);
    const int py0 = ig.y0 + ig.sy * kItemH + (lane / kItemW);
    PixGrad<Q, Extra> s;
    bool wild = false;
    s.next = 0;
#pragma unroll
    for (int p = 0; p < PixGrad<Q, Extra>::NP; ++p) {
        PixState t[2];
        float npy[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int q = 2 * p + k, py = py0 + kRowStep * q;
            t[k] = enter_pixel(a, ig, px, py, q < Q && px < ig.x0 + ig.vw && py < ig.y0 + ig.vh);
            npy[k] = -(float)py;
            s.amin[q] = INFINITY;
            s.nc[q] = t[k].nc;
            s.next = max(s.next, s.nc[q]);
            wild = wild || !(tame(t[k].g0) && tame(t[k].g1) && tame(t[k].g2) && tame(t[k].Rg) && tame(t[k].gD) &&
                             tame(t[k].gA) && tame(t[k].Rd));
        }
        s.npy[p] = f2(npy[0], npy[1]);
        s.T[p] = f2(t[0].T, t[1].T);
        s.g0[p] = f2(t[0].g0, t[1].g0);
        s.g1[p] = f2(t[0].g1, t[1].g1);
        s.g2[p] = f2(t[0].g2, t[1].g2);
        s.nRg[p] = f2(-t[0].Rg, -t[1].Rg);
        if (Extra) {
            s.gD[p] = f2(t[0].gD, t[1].gD);
            s.TfA[p] = f2(t[0].Tf * t[0].gA, t[1].Tf * t[1].gA);
            s.nRd[p] = f2(-t[0].Rd, -t[1].Rd);
        }
    }
    if (__any_sync(kFullB, wild)) return false;
    const uint32_t e0 = ig.e0, first = ig.rg.x, hi = first + (uint32_t)__reduce_max_sync(kFullB, s.next);
    const float pxf = (float)px;
    const float bcx = (float)(ig.x0 + ig.sx * kItemW) + 0.5f * (kItemW - 1);
    const float bcy = (float)(ig.y0 + ig.sy * kItemH) + 0.5f * (kItemH - 1);
    float plain = 0.f;  // the largest record_odd that needs no selection
    // the point-list index of the lane's next entry, loaded a window ahead
    uint32_t g_next = hi > e0 + lane ? a.point_list[hi - 1u - lane] : 0u;
    for (uint32_t top = hi; top > e0; top -= min(32u, top - e0)) {
        const uint32_t g = g_next;
        bool hit = false;
        float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra;
        if (top > e0 + lane) {
            if ((long long)g < a.N) {
                ra = a.recs[g].a;
                rb = a.recs[g].b;
                hit = !block_misses(ra, rb, bcx, bcy, 0.5f * (kItemW - 1), 0.5f * (kItemH - 1));
            } else {
                raise_check(a.ctrl, BGS_CHECK_INDEX);  // a transparent entry
            }
        }
        if (top > e0 + 32u + lane) g_next = a.point_list[top - 33u - lane];
        // back to front over the records that reach the pixel block, packed in that order
        const unsigned live = __ballot_sync(kFullB, hit);
        if (hit) {
            const float4 rc = a.recs[g].c;
            HitB *h = buf + __popc(live & ((1u << lane) - 1u));
            *reinterpret_cast<float4 *>(h) = make_float4(ra.x, ra.z, ra.w, __uint_as_float(top - 1u - lane - first));
            *reinterpret_cast<float4 *>(&h->my) = make_float4(ra.y, ra.y, rb.x, rb.x);
            *reinterpret_cast<float4 *>(&h->o) = make_float4(rb.y, rb.y, rc.x, rc.x);
            *reinterpret_cast<float4 *>(&h->g) = make_float4(rc.y, rc.y, rc.z, rc.z);
            *reinterpret_cast<float4 *>(&h->d) = make_float4(rc.w, rc.w, __uint_as_float(g), rb.w);
        }
        __syncwarp();
        const HitB *end = buf + __popc(live);
        for (const HitB *h = buf; h != end; ++h) {
            const float4 h0 = *reinterpret_cast<const float4 *>(h);
            const int pos = __float_as_int(h0.w);
            if (pos < s.next) {  // a pixel's last contributor: it takes part from here on
                s.next = 0;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    if (pos < s.nc[q]) {
                        s.nc[q] = 0;
                        s.amin[q] = kAlphaMin;
                    }
                    s.next = max(s.next, s.nc[q]);
                }
            }
            const float dx = __fsub_rn(h0.x, pxf);  // shared by the lane's pixels (same column)
            PairSums sums;
            bool any;
            if (h->odd > plain) {
                any = hit_backward<Q, Extra, true>(*h, h0, dx, s, sums);
                if (h->odd > 1.f) plain = -1.f;  // a pixel's carried colour may be anything from here on
            } else {
                any = hit_backward<Q, Extra, false>(*h, h0, dx, s, sums);
            }
            if (__any_sync(kFullB, any)) warp_reduce_red<Extra>(sums, dx, a.grad_acc + 12ull * h->idx, lane);
        }
        __syncwarp();
    }
    return true;
}

// The same item on one row of its pixels after the other (32 pixels, one per lane), one pair at
// a time with a branch: any values.
template <int Q, bool Extra>
__device__ __noinline__ void bwd_pixel_item_wild(const BwdArgs &a, const ItemGeom &ig, int lane) {
    constexpr int kItemW = pix_item_w(Q), kItemH = pix_item_h(Q), kRowStep = pix_row_step(Q);
    const int px = ig.x0 + ig.sx * kItemW + (lane % kItemW);
    for (int q = 0; q < Q; ++q) {
        const int py = ig.y0 + ig.sy * kItemH + (lane / kItemW) + kRowStep * q;
        PixState s = enter_pixel(a, ig, px, py, px < ig.x0 + ig.vw && py < ig.y0 + ig.vh);
        const uint32_t hi = ig.rg.x + (uint32_t)__reduce_max_sync(kFullB, s.nc);
        for (uint32_t top = hi; top > ig.e0; --top) {
            const uint32_t g = a.point_list[top - 1u];
            if ((long long)g >= a.N) {
                raise_check(a.ctrl, BGS_CHECK_INDEX);  // a transparent entry
                continue;
            }
            const Rec r = a.recs[g];
            const PairX x = pair_x(r.a, (float)px);
            PairSums sums = zero_sums();
            const bool any = pair_backward<Extra>(r, x, (float)py, (int)(top - 1u - ig.rg.x) < s.nc, s, sums);
            if (__any_sync(kFullB, any)) warp_reduce_red<Extra>(sums, x.dx, a.grad_acc + 12ull * g, lane);
        }
    }
}

// The item of one pixel a lane (Q = 1), the window walked with the scalar pair rule, which holds for
// every record and gradient: with half of each packed instruction empty the walk of the short
// lists and few warps that such items are chosen for is slower (256 x 256, 10k Gaussians, captured:
// the backward call takes 128 us on complete lists and 113 on truncated ones, packed 140 and 127).
template <bool Extra>
__device__ __forceinline__ void bwd_pixel_item_one(const BwdArgs &a, const ItemGeom &ig, HitB *buf, int lane) {
    constexpr int kItemW = pix_item_w(1), kItemH = pix_item_h(1);
    const int px = ig.x0 + ig.sx * kItemW + (lane % kItemW), py = ig.y0 + ig.sy * kItemH + (lane / kItemW);
    PixState s = enter_pixel(a, ig, px, py, px < ig.x0 + ig.vw && py < ig.y0 + ig.vh);
    const uint32_t e0 = ig.e0, first = ig.rg.x, hi = first + (uint32_t)__reduce_max_sync(kFullB, s.nc);
    const float bcx = (float)(ig.x0 + ig.sx * kItemW) + 0.5f * (kItemW - 1);
    const float bcy = (float)(ig.y0 + ig.sy * kItemH) + 0.5f * (kItemH - 1);
    struct Slot {
        Rec r;
        uint32_t idx;
        int pos;
        float2 pad;
    };
    static_assert(sizeof(Slot) <= sizeof(HitB), "a window slot");
    Slot *win = reinterpret_cast<Slot *>(buf);
    // the point-list index of the lane's next entry, loaded a window ahead
    uint32_t g_next = hi > e0 + lane ? a.point_list[hi - 1u - lane] : 0u;
    for (uint32_t top = hi; top > e0; top -= min(32u, top - e0)) {
        const uint32_t g = g_next;
        bool hit = false;
        Rec r;
        if (top > e0 + lane) {
            if ((long long)g < a.N) {
                r = a.recs[g];
                hit = !block_misses(r.a, r.b, bcx, bcy, 0.5f * (kItemW - 1), 0.5f * (kItemH - 1));
            } else {
                raise_check(a.ctrl, BGS_CHECK_INDEX);  // a transparent entry
            }
        }
        if (top > e0 + 32u + lane) g_next = a.point_list[top - 33u - lane];
        const unsigned live = __ballot_sync(kFullB, hit);
        if (hit) {
            Slot *w = win + __popc(live & ((1u << lane) - 1u));
            w->r = r;
            w->idx = g;
            w->pos = (int)(top - 1u - lane - first);
        }
        __syncwarp();
        const Slot *end = win + __popc(live);
        for (const Slot *w = win; w != end; ++w) {
            const PairX x = pair_x(w->r.a, (float)px);
            PairSums sums = zero_sums();
            const bool any = pair_backward<Extra>(w->r, x, (float)py, w->pos < s.nc, s, sums);
            if (__any_sync(kFullB, any)) warp_reduce_red<Extra>(sums, x.dx, a.grad_acc + 12ull * w->idx, lane);
        }
        __syncwarp();
    }
}

// The walk is latency-bound (dependent FP32 chains, shuffle trees): with colour-only output
// gradients and up to 4 rows per lane the kernel fits 64 registers, so 4 blocks (32 warps)
// stay resident per SM instead of 3.  The other variants would spill there: 3 blocks for
// the depth / alpha gradients at up to 4 rows, no bound at 8 rows.
template <int Q, bool Extra>
__global__ void __launch_bounds__(kBwdWarps * 32, (Q <= 4 && !Extra) ? 4 : (Q <= 4 ? 3 : 1))
    k_backward_balanced(BwdArgs a) {
    __shared__ HitB sbuf[kBwdWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    HitB *buf = sbuf[warp];
    const unsigned num_items = a.ctrl->num_items;
    const unsigned chunk = (unsigned)a.chunk;
    // segment length of the tiles the last forward split (0: no segmented walk)
    const unsigned L = a.bseg_mode >= 0 ? a.ctrl->gw_seg : 0u;
    unsigned long long st_items = 0;
    while (true) {
        unsigned first = 0;
        if (lane == 0) first = atomicAdd(&a.ctrl->queue_head, chunk);
        first = __shfl_sync(kFullB, first, 0);
        if (first >= num_items) break;
        const unsigned end = min(first + chunk, num_items);
        for (unsigned it = first; it < end; ++it) {
            const uint2 item = a.items[it];
            const ItemGeom ig = item_geom<Q>(a, (int)item.x, (int)item.y, L);
            if constexpr (Q == 1) bwd_pixel_item_one<Extra>(a, ig, buf, lane);
            else if (!bwd_pixel_item<Q, Extra>(a, ig, buf, lane)) bwd_pixel_item_wild<Q, Extra>(a, ig, lane);
            ++st_items;
        }
    }
    // the warp's completed items; k_grad_finalize checks their sum (the queue's drain)
    if (lane == 0) a.warp_items[blockIdx.x * kBwdWarps + warp] = (unsigned int)st_items;
}

int backward_balanced_block_threads() { return kBwdWarps * 32; }
static bool has_extra(const BwdArgs &a) {
    for (int v = 0; v < a.vt.V; ++v)
        if (a.gi.dL_ddepth[v] || a.gi.dL_dalpha[v]) return true;
    return false;
}

const void *backward_balanced_kernel(const BwdArgs &a) {
    const bool e = has_extra(a);
    switch (a.pixel_rows) {
        case 1: return e ? (const void *)k_backward_balanced<1, true> : (const void *)k_backward_balanced<1, false>;
        case 2: return e ? (const void *)k_backward_balanced<2, true> : (const void *)k_backward_balanced<2, false>;
        case 4: return e ? (const void *)k_backward_balanced<4, true> : (const void *)k_backward_balanced<4, false>;
        case 8: return e ? (const void *)k_backward_balanced<8, true> : (const void *)k_backward_balanced<8, false>;
        default: return nullptr;
    }
}

cudaError_t launch_backward_balanced(const BwdArgs &a, int grid, cudaStream_t s) {
    const void *k = backward_balanced_kernel(a);
    if (!k) return cudaErrorInvalidValue;
    BwdArgs arg = a;
    void *params[] = {&arg};
    return cudaLaunchKernel(k, dim3(grid), dim3(kBwdWarps * 32), params, 0, s);
}

// ---- accumulator -> ABI gradient arrays ----------------------------------------------
// Record i's accumulator row -> its gradients.  Colours are shared by the views of a
// batched call when n_colors < N (records g, g + n_colors, ... are Gaussian g seen from
// each view): then a thread takes Gaussian g, finalizes its records one view after another
// and writes its colour gradient summed over them, reading each accumulator row once.
__device__ __forceinline__ void finalize_record(long long i, float4 *__restrict__ acc,
                                                const float4 *__restrict__ conic_opacity,
                                                float *__restrict__ dL_dmeans2D, float *__restrict__ dL_dconic,
                                                float *__restrict__ dL_dopacity, float *__restrict__ dL_ddepths,
                                                bool rows, float &cr, float &cg, float &cb) {
    const float4 a0 = acc[3 * i], a1 = acc[3 * i + 1], a2 = acc[3 * i + 2];
    auto bits = [](float4 x) {
        return __float_as_uint(x.x) | __float_as_uint(x.y) | __float_as_uint(x.z) | __float_as_uint(x.w);
    };
    if ((bits(a0) | bits(a1) | bits(a2)) != 0u) {  // leave the accumulators clear
        acc[3 * i] = acc[3 * i + 1] = acc[3 * i + 2] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float4 co = conic_opacity[i];
    // power = ln2 * power2 with power2 = qa dx^2 + qb dx dy + qc dy^2 and (qa, qb, qc) the
    // record's pre-scaled conic; d power / d mean = ln2 (2 qa dx + qb dy, 2 qc dy + qb dx),
    // summed over the pairs from the moments sum gp dx (a0.x) and sum gp dy (a0.y);
    // d power / d(a, b, c) = (-dx^2 / 2, -dx dy, -dy^2 / 2)
    const float qa = -0.5f * kLog2e * co.x, qb = -kLog2e * co.y, qc = -0.5f * kLog2e * co.z;
    dL_dmeans2D[2 * i] = kLn2 * (2.f * qa * a0.x + qb * a0.y);
    dL_dmeans2D[2 * i + 1] = kLn2 * (2.f * qc * a0.y + qb * a0.x);
    // sum gp / o = sum G dL/dalpha (a record with o = 0 has alpha = 0 everywhere: no pair)
    const float go = co.w > 0.f ? a1.y / co.w : 0.f;
    if (rows) {
        reinterpret_cast<float4 *>(dL_dconic)[i] = make_float4(-0.5f * a0.z, -a0.w, -0.5f * a1.x, go);
    } else {
        dL_dconic[3 * i] = -0.5f * a0.z;
        dL_dconic[3 * i + 1] = -a0.w;
        dL_dconic[3 * i + 2] = -0.5f * a1.x;
        dL_dopacity[i] = go;
    }
    if (dL_ddepths) dL_ddepths[i] = a2.y;
    cr += a1.z;
    cg += a1.w;
    cb += a2.x;
}

__global__ void __launch_bounds__(256) k_grad_finalize(long long N, long long n_colors, float4 *__restrict__ acc,
                                                       const float4 *__restrict__ conic_opacity,
                                                       float *__restrict__ dL_dmeans2D, float *__restrict__ dL_dconic,
                                                       float *__restrict__ dL_dopacity, float *__restrict__ dL_dcolors,
                                                       float *__restrict__ dL_ddepths, bool rows,
                                                       const unsigned int *__restrict__ warp_items, int n_warps,
                                                       DevCtrl *ctrl) {
    if (blockIdx.x == 0 && n_warps > 0) {
        // drain check of the persistent backward pass: every queued item ran exactly once
        __shared__ unsigned int part[8];
        unsigned int sum = 0;
        for (int w = threadIdx.x; w < n_warps; w += blockDim.x) sum += warp_items[w];
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned int total = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) total += part[w];
            if (total != ctrl->num_items) atomicOr(&ctrl->check_bits, BGS_CHECK_QUEUE);
        }
    }
    // a thread per record (colours per record), or per Gaussian over its views (shared colours)
    const bool shared = n_colors > 0 && n_colors < N;
    const long long stride = shared ? n_colors : N;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= stride) return;
    float cr = 0.f, cg = 0.f, cb = 0.f;
    for (long long i = g; i < N; i += stride)
        finalize_record(i, acc, conic_opacity, dL_dmeans2D, dL_dconic, dL_dopacity, dL_ddepths, rows, cr, cg, cb);
    if (n_colors > 0) {
        dL_dcolors[3 * g] = cr;
        dL_dcolors[3 * g + 1] = cg;
        dL_dcolors[3 * g + 2] = cb;
    }
}

cudaError_t launch_grad_finalize(long long N, long long n_colors, float4 *acc, const float *conic_opacity,
                                 float *dL_dmeans2D, float *dL_dconic, float *dL_dopacity, float *dL_dcolors,
                                 float *dL_ddepths, const unsigned int *warp_items, int n_warps, DevCtrl *ctrl,
                                 cudaStream_t s) {
    if (N == 0 && n_warps == 0) return cudaSuccess;
    const long long threads = (n_colors > 0 && n_colors < N) ? n_colors : N;
    // an opacity gradient right behind the first conic gradient: the two interleaved, rows of four
    // floats, the layout of conic_opacity, so that no pass has to bring them together (29 us for 3M)
    const bool rows = N > 1 && dL_dopacity == dL_dconic + 3;
    k_grad_finalize<<<(unsigned)std::max<long long>(1, (threads + 255) / 256), 256, 0, s>>>(
        N, n_colors, acc, reinterpret_cast<const float4 *>(conic_opacity), dL_dmeans2D, dL_dconic, dL_dopacity,
        dL_dcolors, dL_ddepths, rows, warp_items, n_warps, ctrl);
    return cudaGetLastError();
}

}  // namespace bgs
