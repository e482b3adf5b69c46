// Coloured-triangle rasteriser fused with the L2 loss (stand-in for the
// Box10 / mesh tasks of Sec. 4.1).  Vertex (x, y) in [0,1]^2 maps to pixel
// coordinates (x W, y H); both windings are drawn (edge coefficients negated
// when the signed area is negative, skipped when it is zero); painter's
// order: the highest covering triangle index wins.
//
// A pixel of row y is covered when it lies in the triangle's pixel box and
// E_i(x) = fma(A_i, x + 1/2, fma(B_i, y + 1/2, C_i)) > th_i for the three
// edges.  Rounding is monotone, so each edge's test is monotone in x along a
// row and a triangle covers one interval of columns.  The loss kernel
// finds the two ends of that interval with the test itself (edge_span below),
// once per row and triangle, and every pixel then needs one range compare per
// candidate instead of three edge functions: the same decisions.
#include <algorithm>

#include "hr_device.cuh"
#include "hr_internal.h"

namespace hr {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxTris = 32;

struct __align__(16) T2Rec {
    float A0, B0, C0, A1;
    float B1, C1, A2, B2;
    float C2, r, g, bl;
    int xlo, xhi, ylo, yhi;
    float th0, th1, th2;      // edge i passes when E_i > th_i (see tl_thr)
    float inv0, inv1, inv2;   // 1 / A_i (guesses of the spans' ends only)
};

// E > 0, or E == 0 on a top-left edge (A > 0, or A == 0 and B > 0), is one
// compare E > th: th = 0, or th = -(smallest subnormal), no float lying
// strictly between the two
__device__ __forceinline__ float tl_thr(float A, float B) {
    return (A > 0.0f || (A == 0.0f && B > 0.0f)) ? -0x1p-149f : 0.0f;
}

__device__ __forceinline__ bool pixel_range2(float mn, float mx, int N, int& lo, int& hi) {
    if (!(mx >= 0.5f) || !(mn <= (float)N - 0.5f)) return false;
    lo = (mn <= 0.5f) ? 0 : (int)ceilf(__fsub_rn(mn, 0.5f));
    hi = (mx >= (float)N - 0.5f) ? N - 1 : (int)floorf(__fsub_rn(mx, 0.5f));
    return lo <= hi;
}

// Set up triangle t from its raw params q[9]; returns false when it covers no pixel.
__device__ bool setup_tri(const float* q, int W, int H, T2Rec& r) {
    const float fW = (float)W, fH = (float)H;
    const float ax = __fmul_rn(q[0], fW), ay = __fmul_rn(q[1], fH);
    const float bx = __fmul_rn(q[2], fW), by = __fmul_rn(q[3], fH);
    const float cx = __fmul_rn(q[4], fW), cy = __fmul_rn(q[5], fH);
    Edge e0 = edge_of(bx, by, cx, cy), e1 = edge_of(cx, cy, ax, ay), e2 = edge_of(ax, ay, bx, by);
    const float D2 = edge_eval(e2.A, e2.B, e2.C, cx, cy);
    if (D2 == 0.0f || D2 != D2) return false;
    if (D2 < 0.0f) {
        e0.A = -e0.A; e0.B = -e0.B; e0.C = -e0.C;
        e1.A = -e1.A; e1.B = -e1.B; e1.C = -e1.C;
        e2.A = -e2.A; e2.B = -e2.B; e2.C = -e2.C;
    }
    const float mnx = fminf(fminf(ax, bx), cx), mxx = fmaxf(fmaxf(ax, bx), cx);
    const float mny = fminf(fminf(ay, by), cy), mxy = fmaxf(fmaxf(ay, by), cy);
    if (!pixel_range2(mnx, mxx, W, r.xlo, r.xhi) || !pixel_range2(mny, mxy, H, r.ylo, r.yhi)) return false;
    r.A0 = e0.A; r.B0 = e0.B; r.C0 = e0.C;
    r.A1 = e1.A; r.B1 = e1.B; r.C1 = e1.C;
    r.A2 = e2.A; r.B2 = e2.B; r.C2 = e2.C;
    r.r = q[6]; r.g = q[7]; r.bl = q[8];
    r.th0 = tl_thr(e0.A, e0.B); r.th1 = tl_thr(e1.A, e1.B); r.th2 = tl_thr(e2.A, e2.B);
    r.inv0 = __fdividef(1.0f, e0.A); r.inv1 = __fdividef(1.0f, e1.A); r.inv2 = __fdividef(1.0f, e2.A);
    return true;
}

// The raw parameters of one render: the scene's, with the optimised subset
// replaced by p(j), j < n.  One CTA; a barrier between the two.
template <class Param>
__device__ __forceinline__ void load_raw(float* dst, const float* raw, const int32_t* pidx, int n_raw, int n, Param p) {
    for (int i = threadIdx.x; i < n_raw; i += blockDim.x) dst[i] = raw[i];
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x) dst[pidx[j]] = p(j);
}

// Squared colour difference of one pixel, in the order the loss has always
// had: fma(d2, d2, fma(d0, d0, d1 d1)).
__device__ __forceinline__ float colour_l2(float d0, float d1, float d2) {
    return __fmaf_rn(d2, d2, __fmaf_rn(d0, d0, __fmul_rn(d1, d1)));
}

// first column x (a whole number) of [lo, hi) with pred(x), hi if none; pred
// false..false true..true
template <class Pred>
__device__ __noinline__ float search_first(float lo, float hi, Pred pred) {
    while (lo < hi) {
        const float mid = floorf(0.5f * (lo + hi));
        if (pred(mid)) hi = mid;
        else lo = mid + 1.0f;
    }
    return lo;
}

// Cuts the columns [lo, hi) of a row (whole numbers, lo < hi) down to those
// where fma(A, x + 1/2, rt) > th (rt the edge's row term).  The end is the
// real-arithmetic crossing -rt / A - 1/2, confirmed by the exact test on both
// sides of it; where the crossing lies within rounding of a pixel centre and
// the test disagrees, a binary search on the test finds it.  A = 0 and NaN:
// the test is the same in every column.
__device__ __forceinline__ void edge_span(float A, float rt, float th, float inv, float& lo, float& hi) {
    auto pass = [=](float x) { return __fmaf_rn(A, __fadd_rn(x, 0.5f), rt) > th; };
    const float xs = __fmaf_rn(-rt, inv, -0.5f);
    if (A > 0.0f) {          // passes from some column on
        const float g = fminf(fmaxf(floorf(xs) + 1.0f, lo), hi);
        const bool sure = (g == hi || pass(g)) && (g == lo || !pass(g - 1.0f));
        lo = sure ? g : search_first(lo, hi, pass);
    } else if (A < 0.0f) {   // passes up to some column
        const float g = fminf(fmaxf(ceilf(xs), lo), hi);
        const bool sure = (g == hi || !pass(g)) && (g == lo || pass(g - 1.0f));
        hi = sure ? g : search_first(lo, hi, [=](float x) { return !pass(x); });
    } else if (!pass(lo)) {
        hi = lo;
    }
}

// Loss of kR consecutive perturbations per CTA, in bands of kBand rows:
//   1. spans: every (render, triangle) in the band's rows, lanes over rows;
//      four lanes (the rows of a row of 8x4 tiles) also give the columns some
//      row covers and those all four cover;
//   2. tiles: a thread per tile finds, for each render, the highest triangle
//      that covers all of the tile (its base), and lists the triangles that
//      meet the tile above the base in some render;
//   3. loss: a warp takes tiles warp, warp + 8, ... in order, one pixel per
//      lane; a lane's winner is the highest listed triangle whose span in its
//      row holds its column, or the base if that is higher.  A tile without
//      either adds the target's own squares, which scene set-up stored.
// Each lane sums its pixels in tile order, then a shuffle tree and the warps
// in order: the order the sum has always had, whatever kR and kBand.
// The target is read as float4 {r, g, b, r^2 + g^2 + b^2} in tile order (one
// coalesced 512-byte load per tile), shared by the kR renders.
//
// Bound by instruction issue (81 % of slots at five CTAs per SM).  The tests
// of three edges per (pixel, candidate) took about 150 instructions per tile
// and render, of which a quarter of the tiles need any: with spans it is 35
// (5.8 of them for the spans, 7 for the lists).  22,528 renders of 256x256,
// 16 triangles: 6.85 ms before, 1.64 ms.  32 rows a band: one span per
// lane, and four renders' spans, lists and records leave room for five CTAs.
constexpr int kBand = 32;

// dynamic shared memory of a CTA: tile lists, tile-row columns and spans
inline size_t loss_bytes(int renders, int n_tris, int W) {
    return (size_t)((W + 7) / 8) * (kBand / 4) * sizeof(uint2) +
           (size_t)renders * ((size_t)(n_tris | 1) * (kBand / 4) * sizeof(uint2) + (size_t)n_tris * kBand * sizeof(uint32_t));
}

template <int kR>
__global__ void __launch_bounds__(kThreads, 5)
tris2d_loss_kernel(RenderBatch b, const float* __restrict__ raw, const int32_t* __restrict__ pidx, int n_tris, int W,
                   int H, const float4* __restrict__ target4) {
    constexpr int kWarps = kThreads / 32, kRows4 = kBand / 4;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ T2Rec s_rec[kR * kMaxTris];
    __shared__ float4 s_col[kR][kMaxTris + 1];   // [0]: background
    __shared__ float s_part[kR][kWarps];
    const int TXn = (W + 7) / 8, TYn = (H + 3) / 4;
    const int pitch = n_tris | 1;   // odd: no bank conflicts over rows or triangles
    uint2* s_tile = reinterpret_cast<uint2*>(s_dyn);         // [TXn kRows4] listed triangles, a byte per render: base + 1
    uint2* s_row = s_tile + TXn * kRows4;                    // [kR][kRows4][pitch]
    uint32_t* s_span = reinterpret_cast<uint32_t*>(s_row + kR * kRows4 * pitch);   // [kR n_tris][kBand] first | length << 16
    float* s_raw = reinterpret_cast<float*>(s_span);                      // [kR][n_tris * 9], before the first span
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * kR;
    const int n_here = min(kR, b.M - m0);
    let_next_start();
#pragma unroll 1
    for (int r = 0; r < n_here; ++r) {
        const Pert pt = resolve(b, m0 + r);
        load_raw(s_raw + r * n_tris * 9, raw, pidx, n_tris * 9, b.n,
                 [&](int j) { return __fadd_rn(pt.theta[j], pt.tau[j]); });
    }
    __syncthreads();
    for (int i = tid; i < kR * n_tris; i += kThreads) {
        const int r = i / n_tris, k = i - r * n_tris;
        T2Rec rec;
        if (r >= n_here || !setup_tri(&s_raw[9 * i], W, H, rec)) {
            rec.ylo = 1;
            rec.yhi = 0;   // no rows
        }
        s_rec[i] = rec;
        s_col[r][k + 1] = make_float4(rec.r, rec.g, rec.bl, 0.0f);
        if (k == 0) s_col[r][0] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    float acc[kR];
#pragma unroll
    for (int r = 0; r < kR; ++r) acc[r] = 0.0f;
    const int dx = lane & 7, dy = lane >> 3;
    // t / TXn = umulhi(t, tx_recip), exactly for t, TXn < 2^16 (Granlund and Montgomery, PLDI 1994)
    const uint32_t tx_recip = TXn > 1 ? (uint32_t)(0xFFFFFFFFu / (uint32_t)TXn) + 1u : 0u;
    int t = warp;   // the warp's next tile, from the band's first
    const float4* tgt = target4 + (size_t)warp * 32 + lane;
    const float4* const tgt_end = target4 + (size_t)TXn * TYn * 32;
    float4 next = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (tgt < tgt_end) next = __ldg(tgt);
    for (int y_band = 0; y_band < H; y_band += kBand) {
        __syncthreads();   // records ready; the previous band's spans no longer read
        for (int i = warp; i < kR * n_tris; i += kWarps) {
            const T2Rec& t = s_rec[i];
            const int r = i / n_tris;
            uint2* row0 = s_row + r * kRows4 * pitch + (i - r * n_tris);
            const int y = y_band + lane;
            float flo = 0.0f, fhi = 0.0f;
            if (y >= t.ylo && y <= t.yhi) {
                const float fy = __fadd_rn((float)y, 0.5f);
                flo = (float)t.xlo;
                fhi = (float)(t.xhi + 1);
                edge_span(t.A0, __fmaf_rn(t.B0, fy, t.C0), t.th0, t.inv0, flo, fhi);
                if (flo < fhi) edge_span(t.A1, __fmaf_rn(t.B1, fy, t.C1), t.th1, t.inv1, flo, fhi);
                if (flo < fhi) edge_span(t.A2, __fmaf_rn(t.B2, fy, t.C2), t.th2, t.inv2, flo, fhi);
            }
            const bool any = flo < fhi;
            if (!__any_sync(0xffffffffu, any)) {   // no row of the band
                s_span[i * kBand + lane] = 0u;
                if (lane < kRows4) row0[lane * pitch] = make_uint2(0u, 0u);
                continue;
            }
            const int lo = any ? (int)flo : 0, hi = any ? (int)fhi : 0;
            s_span[i * kBand + lane] = (uint32_t)lo | ((uint32_t)(hi - lo) << 16);
            // first column and (complemented) end of the union and of the
            // intersection of the four rows, two 16-bit minima or maxima each,
            // then the tiles they meet and the tiles they fill: first | count << 16
            uint32_t u = any ? (uint32_t)lo | ((uint32_t)(0xFFFF - hi) << 16) : 0xFFFFFFFFu, v = u;
            u = __vminu2(u, __shfl_xor_sync(0xffffffffu, u, 1));
            v = __vmaxu2(v, __shfl_xor_sync(0xffffffffu, v, 1));
            u = __vminu2(u, __shfl_xor_sync(0xffffffffu, u, 2));
            v = __vmaxu2(v, __shfl_xor_sync(0xffffffffu, v, 2));
            if ((lane & 3) == 0) {
                const int ulo = (int)(u & 0xFFFFu) >> 3, uhi = (int)(0xFFFFu - (u >> 16) + 7u) >> 3;
                const int vlo = (int)((v & 0xFFFFu) + 7u) >> 3, vhi = (int)(0xFFFFu - (v >> 16)) >> 3;
                row0[(lane >> 2) * pitch] =
                    make_uint2((uint32_t)ulo | ((uint32_t)max(uhi - ulo, 0) << 16),
                               (uint32_t)vlo | ((uint32_t)max(vhi - vlo, 0) << 16));
            }
        }
        __syncthreads();
        const int ty0 = y_band >> 2, ty_end = min(TYn, ty0 + kRows4);
        for (int row = warp; row < ty_end - ty0; row += kWarps) {   // lanes over the tiles of a row
            for (int tx0 = 0; tx0 < TXn; tx0 += 32) {
                const uint32_t tx = (uint32_t)(tx0 + lane);
                uint32_t list = 0u, bases = 0u;
#pragma unroll 1
                for (int r = 0; r < kR; ++r) {
                    const uint2* rw = s_row + (r * kRows4 + row) * pitch;
                    uint32_t part = 0u, base = 0u;
                    for (uint32_t m = __ballot_sync(0xffffffffu, lane < n_tris && (rw[lane].x >> 16) != 0u); m; m &= m - 1) {
                        // ascending: a triangle that fills the tile hides the lower ones
                        const uint32_t bit = m & (0u - m);
                        const int k = 31 - __clz(bit);
                        const uint2 c = rw[k];
                        if (tx - (c.x & 0xFFFFu) < (c.x >> 16)) part |= bit;
                        if (tx - (c.y & 0xFFFFu) < (c.y >> 16)) { part = 0u; base = (uint32_t)k + 1u; }
                    }
                    list |= part;
                    bases |= base << (8 * r);
                }
                if (tx < (uint32_t)TXn) s_tile[row * TXn + tx] = make_uint2(list, bases);
            }
        }
        __syncthreads();
        // this warp's tiles of the band: band tile t is image tile ty0 TXn + t
        const int n_tiles = (ty_end - ty0) * TXn;
        for (; t < n_tiles; t += kWarps) {
            const float4 tg = next;
            tgt += kWarps * 32;
            if (tgt < tgt_end) next = __ldg(tgt);   // one tile ahead
            const uint2 q = s_tile[t];
            if ((q.x | q.y) == 0u) {   // background in every render
#pragma unroll
                for (int r = 0; r < kR; ++r) acc[r] = __fadd_rn(acc[r], tg.w);
                continue;
            }
            uint32_t win[kR];
#pragma unroll
            for (int r = 0; r < kR; ++r) win[r] = (q.y >> (8 * r)) & 0xFFu;
            if (q.x) {
                // a triangle that some render lists is tried in all of them:
                // where it does not meet the tile no span holds the column, where the base hides it the base is higher
                const int row = TXn > 1 ? (int)__umulhi((uint32_t)t, tx_recip) : t;
                const uint32_t x = (uint32_t)((t - row * TXn) * 8 + dx);
                const uint32_t* sp = s_span + row * 4 + dy;
                for (uint32_t m = q.x; m; m &= m - 1) {
                    const uint32_t k = (uint32_t)__ffs(m);   // index + 1
                    const uint32_t* sk = sp + (k - 1u) * kBand;
#pragma unroll
                    for (int r = 0; r < kR; ++r) {
                        const uint32_t w = sk[r * n_tris * kBand];
                        if (x - (w & 0xFFFFu) < (w >> 16)) win[r] = max(win[r], k);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < kR; ++r) {
                const float4 c = s_col[r][win[r]];
                acc[r] = __fadd_rn(acc[r], colour_l2(__fsub_rn(c.x, tg.x), __fsub_rn(c.y, tg.y), __fsub_rn(c.z, tg.z)));
            }
        }
        t -= n_tiles;
    }
#pragma unroll
    for (int r = 0; r < kR; ++r) {
        const float v = warp_sum(acc[r]);
        if (lane == 0) s_part[r][warp] = v;
    }
    __syncthreads();
    if (tid < n_here) {
        float v = 0.0f;
        for (int w = 0; w < kWarps; ++w) v += s_part[tid][w];
        *resolve(b, m0 + tid).loss = v / (float)(W * H * 3);
    }
}

// One image: a thread per pixel tests the triangles from the highest index
// down with the edge functions themselves.
__global__ void __launch_bounds__(kThreads)
tris2d_image_kernel(const float* __restrict__ raw, const int32_t* __restrict__ pidx, int n_tris, int n, int W, int H,
                    const float* __restrict__ params, float* __restrict__ img) {
    __shared__ float s_raw[kMaxTris * 9];
    __shared__ T2Rec s_rec[kMaxTris];
    __shared__ int s_valid[kMaxTris];
    const int tid = threadIdx.x;
    load_raw(s_raw, raw, pidx, n_tris * 9, n, [&](int j) { return params[j]; });
    __syncthreads();
    if (tid < n_tris) s_valid[tid] = setup_tri(&s_raw[9 * tid], W, H, s_rec[tid]) ? 1 : 0;
    __syncthreads();
    const int p = blockIdx.x * kThreads + tid;
    if (p >= W * H) return;
    const int y = p / W, x = p - y * W;
    const float fx = __fadd_rn((float)x, 0.5f), fy = __fadd_rn((float)y, 0.5f);
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f;
    for (int k = n_tris - 1; k >= 0; --k) {
        const T2Rec& r = s_rec[k];
        if (!s_valid[k] || x < r.xlo || x > r.xhi || y < r.ylo || y > r.yhi) continue;
        if (edge_eval(r.A0, r.B0, r.C0, fx, fy) > r.th0 && edge_eval(r.A1, r.B1, r.C1, fx, fy) > r.th1 &&
            edge_eval(r.A2, r.B2, r.C2, fx, fy) > r.th2) {
            c0 = r.r; c1 = r.g; c2 = r.bl;
            break;
        }
    }
    img[3 * (size_t)p] = c0; img[3 * (size_t)p + 1] = c1; img[3 * (size_t)p + 2] = c2;
}

// the target in tile order: lane l of 8x4 tile t holds pixel (l % 8, l / 8) of
// the tile (0 outside the image)
__global__ void tris2d_target_kernel(const float* __restrict__ target, int W, int H, int TXn, int n, float4* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int t = i >> 5, lane = i & 31, ty = t / TXn, tx = t - ty * TXn;
    const int x = tx * 8 + (lane & 7), y = ty * 4 + (lane >> 3);
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (x < W && y < H) {
        const float* p = target + 3 * ((size_t)y * W + x);
        v = make_float4(p[0], p[1], p[2], colour_l2(__fsub_rn(0.0f, p[0]), __fsub_rn(0.0f, p[1]), __fsub_rn(0.0f, p[2])));
    }
    out[i] = v;
}

template <int kR>
void launch_loss(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    // (not launch_after: blocks placed while the sampler's hold parts of the SMs stay
    // unevenly spread; 64x64 Hessian of 1,024 renders 91 us, 105 so)
    tris2d_loss_kernel<kR><<<(b.M + kR - 1) / kR, kThreads, loss_bytes(kR, sc.n_tris, sc.W), s>>>(
        b, sc.raw, sc.pidx, sc.n_tris, sc.W, sc.H, reinterpret_cast<const float4*>(sc.target4));
}

}  // namespace

// Renders per CTA: they share the target's loads and the tile loop but lengthen
// a CTA's work, so more than one only when enough CTAs remain for every SM.
// Measured (256x256, 16 triangles; 1 / 2 / 4 renders per CTA): 99 / 94 / 135 us
// at M = 608 (four per SM), 168 / 135 / 150 at 1,024, 275 / 219 / 221 at 2,048,
// 322 / 244 / 222 at 2,432 (sixteen per SM), 1,023 / 741 / 665 at 8,192; the
// lines lie at the same M for 64x64 to 400x400.
void launch_tris2d_loss(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    const int sms = num_sms();
    if (b.M >= 16 * sms) launch_loss<4>(sc, b, s);
    else if (b.M > 4 * sms) launch_loss<2>(sc, b, s);
    else launch_loss<1>(sc, b, s);
}

size_t tris2d_target_floats(const DevScene& sc) {
    return 4 * 32 * (size_t)((sc.W + 7) / 8) * ((sc.H + 3) / 4);
}

void tris2d_tile_target(const DevScene& sc, cudaStream_t s) {
    const int TXn = (sc.W + 7) / 8, n = 32 * TXn * ((sc.H + 3) / 4);
    tris2d_target_kernel<<<(n + 255) / 256, 256, 0, s>>>(sc.target, sc.W, sc.H, TXn, n,
                                                         reinterpret_cast<float4*>(sc.target4));
}

void launch_tris2d_image(const DevScene& sc, const float* params, float* img, cudaStream_t s) {
    tris2d_image_kernel<<<(sc.W * sc.H + kThreads - 1) / kThreads, kThreads, 0, s>>>(sc.raw, sc.pidx, sc.n_tris, sc.n,
                                                                                      sc.W, sc.H, params, img);
}

}  // namespace hr
