// K5: path tracer of the procedural box (stand-in for the Shadow task of
// Sec. 4.1) fused with the per-pixel L2 loss.  Rendering follows the
// standard Monte Carlo estimator of the rendering equation (Sec. 3.1):
// Lambertian surfaces, next-event estimation to the rectangular light at
// every path vertex, cosine-weighted continuation, fixed depth.
//
// Scene: 12 axis-aligned quads (index 0..11), the light quad (12, horizontal,
// emitting downward), 3 spheres (13..15); 16 primitives staged in shared
// memory, tested brute force per ray (a BVH over 16 primitives costs more
// node tests than it saves).  Rays, hits and all decisions in FP32 with the
// operation order below; radiance in FP32.
//
// Path random numbers: Philox (pixel sample, (k << 8) | (vertex << 4) |
// block, (tag << 24) | sub, request), key = seed; both legs of a pair share
// them (common random numbers).  Vertex 0 = camera jitter; at vertices
// 1..depth block 0 words 0,1 pick the light point, words 2,3 the first disc
// try; blocks 1..3 hold tries 1..6; a cosine-weighted direction comes from a
// unit-disc point (rejection from the square) lifted to the hemisphere.
#include <cmath>
#include <cooperative_groups.h>

#include "hr_device.cuh"
#include "hr_internal.h"

namespace hr {
namespace {

constexpr int kThreads = 256;
constexpr int kLight = 12;
constexpr float kInvPi = 0.318309886183790671538f;

// quad q: {plane, lo_u, lo_v, hi_u} and {hi_v, axis, u, v} as two 16-byte
// loads; sphere i: {centre xyz, r^2}
struct __align__(16) QuadS {
    float plane, lo_u, lo_v, hi_u;
    float hi_v;
    int axis, u, v;
};
struct PtShared {
    QuadS q[13];
    float4 sph[3];
    float alb[16][3];
    float sr[3], isr[3];
    float em[3];
    float box_lo[3], box_hi[3];   // wall planes per axis (procedural box layout)
    int wall_lo[3], wall_hi[3];   // index of the wall quad at box_lo[a] / box_hi[a]
    int light_inside;             // light at least kWallMargin inside every wall plane
};

// Walls (quads 0..5, two per axis) from a ray origin inside the box, i.e.
// box_lo[a] <= o_a <= box_hi[a] on every axis:
//  * the wall behind the ray on axis a (at box_lo[a] when d_a > 0, at
//    box_hi[a] when d_a < 0) has RN(plane - o_a) of the other sign than
//    1/d_a, so t <= 0 and the closest-hit test rejects it: only the forward
//    wall of each axis is tested (still in increasing quad index);
//  * a shadow ray toward a light quad that lies at least kWallMargin inside
//    every wall plane meets a forward wall only beyond the light (its t
//    exceeds the light's by at least the margin over |d_a| <= 1, far above
//    FP32 rounding), so the light is the closest primitive exactly when it
//    is with the walls tested: shadow rays then test no wall.
constexpr float kWallMargin = 1e-3f;

__device__ __forceinline__ float dot3(const float* a, const float* b) {
    return __fmaf_rn(a[2], b[2], __fmaf_rn(a[1], b[1], __fmul_rn(a[0], b[0])));
}

// closest hit with t > 0, ties to the lower primitive index; plane distances
// t = RN(RN(plane - o_a) * RN(1 / d_a)) with the ray's per-axis reciprocals
__device__ int intersect(const PtShared& S, const float o[3], const float d[3], float& t_out) {
    float best = INFINITY;
    int prim = -1;
    const float inv[3] = {__frcp_rn(d[0]), __frcp_rn(d[1]), __frcp_rn(d[2])};
#pragma unroll 1
    for (int q = 0; q <= kLight; ++q) {
        const QuadS Q = S.q[q];
        const int a = Q.axis;
        const float da = a == 0 ? d[0] : (a == 1 ? d[1] : d[2]);
        if (da == 0.0f) continue;
        const float oa = a == 0 ? o[0] : (a == 1 ? o[1] : o[2]);
        const float ia = a == 0 ? inv[0] : (a == 1 ? inv[1] : inv[2]);
        const float t = __fmul_rn(__fsub_rn(Q.plane, oa), ia);
        if (!(t > 0.0f)) continue;
        const float du = Q.u == 0 ? d[0] : d[1], ou = Q.u == 0 ? o[0] : o[1];
        const float dv = Q.v == 1 ? d[1] : d[2], ov = Q.v == 1 ? o[1] : o[2];
        const float hu = __fmaf_rn(t, du, ou);
        const float hv = __fmaf_rn(t, dv, ov);
        if (hu < Q.lo_u || hu > Q.hi_u || hv < Q.lo_v || hv > Q.hi_v) continue;
        if (t < best) { best = t; prim = q; }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float4 sp = S.sph[i];
        const float oc[3] = {__fsub_rn(o[0], sp.x), __fsub_rn(o[1], sp.y), __fsub_rn(o[2], sp.z)};
        const float b = dot3(oc, d);
        const float cc = __fsub_rn(dot3(oc, oc), sp.w);
        const float disc = __fmaf_rn(b, b, -cc);
        if (disc < 0.0f) continue;
        const float sq = __fsqrt_rn(disc);
        float t = __fsub_rn(-b, sq);
        if (!(t > 0.0f)) {
            t = __fsub_rn(sq, b);
            if (!(t > 0.0f)) continue;
        }
        if (t < best) { best = t; prim = 13 + i; }
    }
    t_out = best;
    return prim;
}

// The same closest-hit rule with the quad axes known at compile time: the
// layout the procedural box always has (box walls and block faces two per
// axis, x x y y z z, then the horizontal light).  Fully unrolled and
// predicated: every quad is tested in index order with the same operation
// sequence and the same acceptance (axis direction non-zero, t > 0, hit
// inside the closed rectangle, t < best), so it returns what the general
// loop returns.
// One quad of axis a: accepted when d_a != 0, t > 0, the hit lies in the
// closed rectangle and t < best.
__device__ __forceinline__ void quad_test(const PtShared& S, int q, int a, const float o[3], const float d[3],
                                          const float inv[3], float& best, int& prim) {
    const int u = a == 0 ? 1 : 0, v = a == 2 ? 1 : 2;
    const QuadS Q = S.q[q];
    const float t = __fmul_rn(__fsub_rn(Q.plane, o[a]), inv[a]);
    const float hu = __fmaf_rn(t, d[u], o[u]);
    const float hv = __fmaf_rn(t, d[v], o[v]);
    const bool ok = d[a] != 0.0f && t > 0.0f && !(hu < Q.lo_u || hu > Q.hi_u || hv < Q.lo_v || hv > Q.hi_v) &&
                    t < best;
    best = ok ? t : best;
    prim = ok ? q : prim;
}

// walls: 0 tests all six wall quads, 1 the forward wall of each axis, 2 none
// (see kWallMargin for when 1 and 2 give the result of 0).  A sphere's square
// root and roots are formed only when some lane of the warp has a
// non-negative discriminant (a lane with a negative one rejects it).
__device__ __noinline__ int intersect_canon(const PtShared& S, const float o[3], const float d[3], float& t_out,
                                            int walls) {
    constexpr int kAxis[13] = {0, 0, 1, 1, 2, 2, 0, 0, 1, 1, 2, 2, 1};
    float best = INFINITY;
    int prim = -1;
    const float inv[3] = {__frcp_rn(d[0]), __frcp_rn(d[1]), __frcp_rn(d[2])};
    if (walls == 0) {
#pragma unroll
        for (int q = 0; q < 6; ++q) quad_test(S, q, kAxis[q], o, d, inv, best, prim);
    } else if (walls == 1) {
#pragma unroll
        for (int a = 0; a < 3; ++a) quad_test(S, d[a] > 0.0f ? S.wall_hi[a] : S.wall_lo[a], a, o, d, inv, best, prim);
    }
#pragma unroll
    for (int q = 6; q <= kLight; ++q) quad_test(S, q, kAxis[q], o, d, inv, best, prim);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float4 sp = S.sph[i];
        const float oc[3] = {__fsub_rn(o[0], sp.x), __fsub_rn(o[1], sp.y), __fsub_rn(o[2], sp.z)};
        const float b = dot3(oc, d);
        const float cc = __fsub_rn(dot3(oc, oc), sp.w);
        const float disc = __fmaf_rn(b, b, -cc);
        if (!__any_sync(__activemask(), disc >= 0.0f)) continue;
        const float sq = __fsqrt_rn(fmaxf(disc, 0.0f));
        const float t0 = __fsub_rn(-b, sq), t1 = __fsub_rn(sq, b);
        const float t = t0 > 0.0f ? t0 : t1;
        const bool ok = disc >= 0.0f && t > 0.0f && t < best;   // NaN disc rejects, as in the loop
        best = ok ? t : best;
        prim = ok ? 13 + i : prim;
    }
    t_out = best;
    return prim;
}

__device__ __forceinline__ bool inside_box(const PtShared& S, const float o[3]) {
    return o[0] >= S.box_lo[0] && o[0] <= S.box_hi[0] && o[1] >= S.box_lo[1] && o[1] <= S.box_hi[1] &&
           o[2] >= S.box_lo[2] && o[2] <= S.box_hi[2];
}

template <bool kCanon>
__device__ __forceinline__ int closest_hit(const PtShared& S, const float o[3], const float d[3], float& t_out) {
    return kCanon ? intersect_canon(S, o, d, t_out, inside_box(S, o) ? 1 : 0) : intersect(S, o, d, t_out);
}

// Is the light the closest primitive along a shadow ray?
template <bool kCanon>
__device__ __forceinline__ bool sees_light(const PtShared& S, const float o[3], const float d[3]) {
    float t;
    if (!kCanon) return intersect(S, o, d, t) == kLight;
    const int walls = inside_box(S, o) ? (S.light_inside ? 2 : 1) : 0;
    return intersect_canon(S, o, d, t, walls) == kLight;
}

// work counters of the counting instantiation (kCount): closest-hit rays,
// shadow rays and shaded path vertices
struct PtCount {
    uint32_t hit = 0, shadow = 0, vert = 0;
};

template <bool kCanon, bool kCount>
__device__ void radiance(const PtShared& S, int depth, uint64_t seed, uint32_t request, uint32_t c2, uint32_t k,
                         uint32_t idx, float o[3], float d[3], float L[3], PtCount& cnt) {
    float beta[3] = {1.0f, 1.0f, 1.0f};
    float t;
    if (kCount) ++cnt.hit;
    int prim = closest_hit<kCanon>(S, o, d, t);
    if (prim < 0) return;
    if (prim == kLight) {
        if (d[1] > 0.0f) { L[0] += S.em[0]; L[1] += S.em[1]; L[2] += S.em[2]; }
        return;
    }
    const QuadS& LQ = S.q[kLight];
    const float area = __fmul_rn(__fsub_rn(LQ.hi_u, LQ.lo_u), __fsub_rn(LQ.hi_v, LQ.lo_v));
    for (int v = 1; v <= depth; ++v) {
        if (prim == kLight) return;
        float x[3], n[3], o2[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c] = __fmaf_rn(t, d[c], o[c]);
        if (prim <= kLight) {
            const int a = S.q[prim].axis;
            n[0] = n[1] = n[2] = 0.0f;
            n[a] = d[a] > 0.0f ? -1.0f : 1.0f;
        } else {
            const int i = prim - 13;
            const float4 sp = S.sph[i];
            n[0] = __fmul_rn(__fsub_rn(x[0], sp.x), S.isr[i]);
            n[1] = __fmul_rn(__fsub_rn(x[1], sp.y), S.isr[i]);
            n[2] = __fmul_rn(__fsub_rn(x[2], sp.z), S.isr[i]);
            if (dot3(n, d) > 0.0f) { n[0] = -n[0]; n[1] = -n[1]; n[2] = -n[2]; }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) o2[c] = __fmaf_rn(n[c], 1e-4f, x[c]);
        const float* rho = S.alb[prim];
        if (kCount) ++cnt.vert;
        const uint32_t cbase = (k << 8) | ((uint32_t)v << 4);
        const u32x4 w0 = philox_seed(seed, idx, cbase, c2, request);
        // next-event estimation
        {
            const float ly[3] = {__fmaf_rn(u24f(w0.x), __fsub_rn(LQ.hi_u, LQ.lo_u), LQ.lo_u), LQ.plane,
                                 __fmaf_rn(u24f(w0.y), __fsub_rn(LQ.hi_v, LQ.lo_v), LQ.lo_v)};
            const float wv[3] = {__fsub_rn(ly[0], o2[0]), __fsub_rn(ly[1], o2[1]), __fsub_rn(ly[2], o2[2])};
            const float dist2 = dot3(wv, wv);
            const float idist = __frcp_rn(__fsqrt_rn(dist2));
            float om[3] = {__fmul_rn(wv[0], idist), __fmul_rn(wv[1], idist), __fmul_rn(wv[2], idist)};
            const float cosx = dot3(n, om);
            const float cosl = om[1];
            if (cosx > 0.0f && cosl > 0.0f) {
                if (kCount) ++cnt.shadow;
                if (sees_light<kCanon>(S, o2, om)) {
                    const float geo = cosx * cosl / dist2 * area * kInvPi;
#pragma unroll
                    for (int c = 0; c < 3; ++c) L[c] += beta[c] * rho[c] * S.em[c] * geo;
                }
            }
        }
        if (v == depth) return;
        // cosine-weighted continuation
        float a = 0.0f, b = 0.0f;
        {
            float ta = __fmaf_rn(u24f(w0.z), 2.0f, -1.0f), tb = __fmaf_rn(u24f(w0.w), 2.0f, -1.0f);
            bool found = __fmaf_rn(ta, ta, __fmul_rn(tb, tb)) < 1.0f;
            if (found) { a = ta; b = tb; }
            for (uint32_t blk = 1; blk <= 3 && !found; ++blk) {
                const u32x4 wb = philox_seed(seed, idx, cbase | blk, c2, request);
                ta = __fmaf_rn(u24f(wb.x), 2.0f, -1.0f);
                tb = __fmaf_rn(u24f(wb.y), 2.0f, -1.0f);
                if (__fmaf_rn(ta, ta, __fmul_rn(tb, tb)) < 1.0f) { a = ta; b = tb; found = true; break; }
                ta = __fmaf_rn(u24f(wb.z), 2.0f, -1.0f);
                tb = __fmaf_rn(u24f(wb.w), 2.0f, -1.0f);
                if (__fmaf_rn(ta, ta, __fmul_rn(tb, tb)) < 1.0f) { a = ta; b = tb; found = true; break; }
            }
        }
        const float r2 = __fmaf_rn(a, a, __fmul_rn(b, b));
        const float cz = __fsqrt_rn(__fsub_rn(1.0f, r2));
        // orthonormal basis around n (Duff et al., "Building an Orthonormal
        // Basis, Revisited", JCGT 2017)
        const float sg = copysignf(1.0f, n[2]);
        const float aa = __fdiv_rn(-1.0f, __fadd_rn(sg, n[2]));
        const float bb = __fmul_rn(__fmul_rn(n[0], n[1]), aa);
        const float t1[3] = {__fmaf_rn(__fmul_rn(sg, __fmul_rn(n[0], n[0])), aa, 1.0f), __fmul_rn(sg, bb),
                             -__fmul_rn(sg, n[0])};
        const float t2[3] = {bb, __fmaf_rn(__fmul_rn(n[1], n[1]), aa, sg), -n[1]};
        float nd[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) nd[c] = __fmaf_rn(cz, n[c], __fmaf_rn(b, t2[c], __fmul_rn(a, t1[c])));
#pragma unroll
        for (int c = 0; c < 3; ++c) beta[c] *= rho[c];
        if (kCount) ++cnt.hit;
        prim = closest_hit<kCanon>(S, o2, nd, t);
        if (prim < 0) return;
#pragma unroll
        for (int c = 0; c < 3; ++c) { o[c] = o2[c]; d[c] = nd[c]; }
    }
}

struct PtArgs {
    int32_t qaxis[13];
    float qgeom[13][5];
    float qalb[13][3];
    float sc[3][3], sr[3], salb[3][3];
    float light_half, cam_z, tan_half, pix_scale;
    float em[3];
    int W, H, spp, depth;
    const float* target;
    unsigned long long* stats;   // counting instantiation only: see hr_scene_stats
};

__device__ void load_scene(const PtArgs& A, const float* p, PtShared& S) {
    const int t = threadIdx.x;
    if (t < 12) {
        QuadS& Q = S.q[t];
        Q.axis = A.qaxis[t];
        Q.u = Q.axis == 0 ? 1 : 0;
        Q.v = Q.axis == 2 ? 1 : 2;
        Q.plane = A.qgeom[t][0];
        Q.lo_u = A.qgeom[t][1]; Q.lo_v = A.qgeom[t][2];
        Q.hi_u = A.qgeom[t][3]; Q.hi_v = A.qgeom[t][4];
        S.alb[t][0] = A.qalb[t][0]; S.alb[t][1] = A.qalb[t][1]; S.alb[t][2] = A.qalb[t][2];
    } else if (t >= 13 && t < 16) {
        const int i = t - 13;
        S.sph[i] = make_float4(i == 0 ? p[3] : A.sc[i][0], i == 0 ? p[4] : A.sc[i][1], i == 0 ? p[5] : A.sc[i][2],
                               __fmul_rn(A.sr[i], A.sr[i]));
        for (int c = 0; c < 3; ++c) S.alb[t][c] = A.salb[i][c];
        S.sr[i] = A.sr[i];
        S.isr[i] = __frcp_rn(A.sr[i]);
    } else if (t == 16) {
        QuadS& Q = S.q[kLight];
        Q.axis = 1; Q.u = 0; Q.v = 2;
        Q.plane = p[1];
        Q.lo_u = __fsub_rn(p[0], A.light_half);
        Q.hi_u = __fadd_rn(p[0], A.light_half);
        Q.lo_v = __fsub_rn(p[2], A.light_half);
        Q.hi_v = __fadd_rn(p[2], A.light_half);
        S.alb[kLight][0] = S.alb[kLight][1] = S.alb[kLight][2] = 0.0f;
        S.em[0] = A.em[0]; S.em[1] = A.em[1]; S.em[2] = A.em[2];
        // wall planes (quads 2a, 2a + 1 for axis a in the procedural box layout)
        // and whether the light quad lies kWallMargin inside all of them
        const float lmin[3] = {Q.lo_u, Q.plane, Q.lo_v}, lmax[3] = {Q.hi_u, Q.plane, Q.hi_v};
        bool in = true;
        for (int a = 0; a < 3; ++a) {
            const float p0 = A.qgeom[2 * a][0], p1 = A.qgeom[2 * a + 1][0];
            S.box_lo[a] = fminf(p0, p1);
            S.box_hi[a] = fmaxf(p0, p1);
            S.wall_lo[a] = p0 <= p1 ? 2 * a : 2 * a + 1;
            S.wall_hi[a] = p0 <= p1 ? 2 * a + 1 : 2 * a;
            in = in && lmin[a] >= S.box_lo[a] + kWallMargin && lmax[a] <= S.box_hi[a] - kWallMargin;
        }
        S.light_inside = in ? 1 : 0;
    }
}

template <bool kImage, int kMinBlocks, bool kCanon, bool kCount = false>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
ptbox_kernel(PtArgs A, RenderBatch b, const float* __restrict__ img_params, uint64_t seed_img, uint32_t req_img,
             uint32_t sub_img, uint32_t k_img, uint32_t tag_img, int spp_img, float* __restrict__ img) {
    PtCount cnt;
    __shared__ PtShared S;
    __shared__ float s_p[8];
    __shared__ float s_part[kThreads / 32];
    const int m = blockIdx.x;
    const int tid = threadIdx.x;
    uint64_t seed;
    uint32_t request, sub, k, tag;
    int spp;
    if (kImage) {
        if (tid < 6) s_p[tid] = img_params[tid];
        seed = seed_img; request = req_img; sub = sub_img; k = k_img; tag = tag_img; spp = spp_img;
    } else {
        const Pert pt = resolve(b, m);
        if (tid < 6) s_p[tid] = __fadd_rn(pt.theta[tid], pt.tau[tid]);
        seed = pt.seed;
        request = pt.request;
        const uint2 mt = *pt.meta;
        sub = mt.x; k = mt.y; tag = TAG_PATH; spp = A.spp;
    }
    __syncthreads();
    load_scene(A, s_p, S);
    __syncthreads();
    const uint32_t c2 = (tag << 24) | (sub & 0xFFFFFFu);
    const float inv_spp = 1.0f / (float)spp;
    float acc = 0.0f;
    const int npx = A.W * A.H;
    // (an image's pixels over all blocks, a loss's by one block)
    const int step = kImage ? kThreads * (int)gridDim.x : kThreads;
    for (int px = kImage ? kThreads * (int)blockIdx.x + tid : tid; px < npx; px += step) {
        const int y = px / A.W, x = px - y * A.W;
        float L[3] = {0.0f, 0.0f, 0.0f};
        for (int s = 0; s < spp; ++s) {
            const uint32_t idx = (uint32_t)(px * spp + s);
            const u32x4 wj = philox_seed(seed, idx, k << 8, c2, request);
            const float fx = __fadd_rn((float)x, u24f(wj.x));
            const float fy = __fadd_rn((float)y, u24f(wj.y));
            float d[3] = {__fmaf_rn(fx, A.pix_scale, -A.tan_half), __fmaf_rn(-fy, A.pix_scale, A.tan_half), -1.0f};
            const float il = __frcp_rn(__fsqrt_rn(dot3(d, d)));
            d[0] = __fmul_rn(d[0], il); d[1] = __fmul_rn(d[1], il); d[2] = __fmul_rn(d[2], il);
            float o[3] = {0.0f, 0.0f, A.cam_z};
            radiance<kCanon, kCount>(S, A.depth, seed, request, c2, k, idx, o, d, L, cnt);
        }
        const size_t p3 = 3 * (size_t)px;
        if (kImage) {
            img[p3] = L[0] * inv_spp; img[p3 + 1] = L[1] * inv_spp; img[p3 + 2] = L[2] * inv_spp;
        } else {
            const float d0 = L[0] * inv_spp - A.target[p3];
            const float d1 = L[1] * inv_spp - A.target[p3 + 1];
            const float d2 = L[2] * inv_spp - A.target[p3 + 2];
            acc += d0 * d0 + d1 * d1 + d2 * d2;
        }
    }
    if (kCount && A.stats) {   // [0] renders, [1] closest-hit rays, [2] shadow rays, [3] shaded vertices
        const unsigned long long h = (unsigned long long)warp_sum_i((int)cnt.hit);
        const unsigned long long sh = (unsigned long long)warp_sum_i((int)cnt.shadow);
        const unsigned long long vt = (unsigned long long)warp_sum_i((int)cnt.vert);
        if ((tid & 31) == 0) {
            atomicAdd(&A.stats[1], h);
            atomicAdd(&A.stats[2], sh);
            atomicAdd(&A.stats[3], vt);
        }
        if (tid == 0) atomicAdd(&A.stats[0], 1ull);
    }
    if (!kImage) {
        acc = warp_sum(acc);
        if ((tid & 31) == 0) s_part[tid >> 5] = acc;
        __syncthreads();
        if (tid == 0) {
            float v = 0.0f;
            for (int w = 0; w < kThreads / 32; ++w) v += s_part[w];
            *resolve(b, m).loss = v / (float)(npx * 3);
        }
    }
}

// ---------------------------------------------------------------------------
// Both legs of an antithetic pair by one CTA.  The legs share their path
// random numbers and differ in the light's and sphere 0's centre only, so
// their paths are the same rays until one of them meets the light or
// sphere 0.  A lane follows the common path of its pixel sample for the legs
// still on it (`mask`): the random words, the rays, the tests of the twelve
// quads and spheres 1 and 2 and the surface are formed once, the light,
// sphere 0 and the shadow ray once per leg.  A leg that meets the light ends.
// A leg that meets sphere 0 while the other stays on the common path goes to the
// warp's queue, whose entries are finished 32 at a time, one leg per lane (all
// pending ones before the warp's next sample of a pixel, so that a leg adds its
// contributions in vertex and sample order).
//
// Every value is formed by the operations of `radiance`, and the closest hit is
// the least (t, primitive index) of the accepted ones in either order of tests,
// so losses are the same bits as one render per CTA gives.
//
// Bound by issue and its latencies (71 % of slots busy; the loop's code is about
// as large as the instruction cache holds, so each part of it exists once and
// queued legs run the same loop as camera paths: with separate code for them
// 18.0 ms against 14.2 per 2,048 renders of 128x128, 4 spp).  Of the 4,700
// instructions per pair and path sample 2,000 are shadow rays, 740 queued legs; two
// single renders take 6,150.  8,192 renders of 128x128, 4 spp: 54.6 ms with one
// render per CTA, 41.6 with pairs.  Four CTAs of 64 registers per SM: 4,864
// renders in 27.7 ms, three of 80 registers 31.0.
// ---------------------------------------------------------------------------
constexpr int kQueue = 64;     // 31 left over + one push per lane
constexpr int kQueueWords = 10;
constexpr int kPairWarps = kThreads / 32;

struct PairLeg {
    float4 light;              // lo_u, lo_v, hi_u, hi_v
    float4 sph;                // sphere 0: centre, r^2
    float plane;               // light plane y
    float area;
    int light_inside;
    int pad;
};
struct PairShared {
    float4 rect[12];           // quads: lo_u, lo_v, hi_u, hi_v
    float plane[12];
    float4 sph[2];             // spheres 1, 2
    uint4 keys[5];             // Philox round keys
    float alb[16][3];
    float isr[3];
    float em[3];
    float box_lo[3], box_hi[3];
    int wall_lo[3], wall_hi[3];
    PairLeg leg[2];
    float p[2][8];
    float part[2][kPairWarps];
};
template <int kSlots>   // pixels per lane between two ends of the queue
struct PairWarp {
    float L[kSlots][6][32];    // radiance sums of the slots' pixels: 3 leg + channel
    float q[kQueueWords][kQueue];
    float acc[2][32];          // loss sums of the lanes, by leg
};

struct Hit {
    float t;
    int prim;
};

// philox10 with the key schedule of the pair's seed (ten (k0, k1), read as five float4)
__device__ __forceinline__ u32x4 philox_keyed(const PairShared& S, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) {
#pragma unroll
    for (int r = 0; r < 10; r += 2) {
        const uint4 k = S.keys[r >> 1];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t pa = (uint64_t)0xD2511F53u * c0, pb = (uint64_t)0xCD9E8D57u * c2;
            const uint32_t a = (uint32_t)pa, ha = (uint32_t)(pa >> 32), b = (uint32_t)pb, hb = (uint32_t)(pb >> 32);
            const uint32_t n0 = hb ^ c1 ^ (h ? k.z : k.x), n2 = ha ^ c3 ^ (h ? k.w : k.y);
            c0 = n0; c1 = b; c2 = n2; c3 = a;
        }
    }
    return {c0, c1, c2, c3};
}

__device__ __forceinline__ void quad_hit(float4 R, float plane, int q, int a, const float o[3], const float d[3],
                                         const float inv[3], Hit& h) {
    const int u = a == 0 ? 1 : 0, v = a == 2 ? 1 : 2;
    // d_a = 0: t is infinite or NaN and the last compare rejects it
    const float t = __fmul_rn(__fsub_rn(plane, o[a]), inv[a]);
    const float hu = __fmaf_rn(t, d[u], o[u]);
    const float hv = __fmaf_rn(t, d[v], o[v]);
    const bool ok = t > 0.0f && !(hu < R.x || hu > R.z || hv < R.y || hv > R.w) && t < h.t;
    h.t = ok ? t : h.t;
    h.prim = ok ? q : h.prim;
}

// |o - c|^2 - r^2 of a sphere: the part of its test that depends on the origin only
__device__ __forceinline__ float sphere_cc(float4 sp, const float o[3]) {
    const float oc[3] = {__fsub_rn(o[0], sp.x), __fsub_rn(o[1], sp.y), __fsub_rn(o[2], sp.z)};
    return __fsub_rn(dot3(oc, oc), sp.w);
}

// Distance of the sphere's first root > 0 (see intersect), -1 when it is not
// hit.  With the origin outside (cc > 0) and the sphere behind (b >= 0)
// neither root is positive: disc = fma(b, b, -cc) <= RN(b^2), so its square
// root is at most b.  The roots are formed only when some lane of the warp
// needs them.
__device__ __forceinline__ float sphere_t(float4 sp, float cc, const float o[3], const float d[3], bool live) {
    const float oc[3] = {__fsub_rn(o[0], sp.x), __fsub_rn(o[1], sp.y), __fsub_rn(o[2], sp.z)};
    const float b = dot3(oc, d);
    const float disc = __fmaf_rn(b, b, -cc);
    const bool on = live && disc >= 0.0f && (b < 0.0f || cc <= 0.0f);
    float t = -1.0f;
    if (__any_sync(0xffffffffu, on)) {
        const float sq = __fsqrt_rn(fmaxf(disc, 0.0f));
        const float t0 = __fsub_rn(-b, sq);
        if (on) t = t0 > 0.0f ? t0 : __fsub_rn(sq, b);
    }
    return t;
}

// A ray's origin, with what the tests of several rays from it share.
struct Origin {
    float o[3];
    float cc[2];   // sphere_cc of spheres 1, 2
    bool in;       // inside the walls
};

__device__ __forceinline__ bool in_box(const PairShared& S, const float o[3]) {
    return o[0] >= S.box_lo[0] && o[0] <= S.box_hi[0] && o[1] >= S.box_lo[1] && o[1] <= S.box_hi[1] &&
           o[2] >= S.box_lo[2] && o[2] <= S.box_hi[2];
}

// wall q's distance where its hit lies in the rectangle, else -1 (any axis)
__device__ __noinline__ float any_axis_t(const PairShared& S, int q, float ox, float oy, float oz, float dx, float dy,
                                         float dz) {
    const int a = q >> 1;
    const float oa = a == 0 ? ox : (a == 1 ? oy : oz), da = a == 0 ? dx : (a == 1 ? dy : dz);
    const float ou = a == 0 ? oy : ox, du = a == 0 ? dy : dx;
    const float ov = a == 2 ? oy : oz, dv = a == 2 ? dy : dz;
    const float t = __fmul_rn(__fsub_rn(S.plane[q], oa), __frcp_rn(da));
    const float hu = __fmaf_rn(t, du, ou), hv = __fmaf_rn(t, dv, ov);
    const float4 R = S.rect[q];
    return t > 0.0f && !(hu < R.x || hu > R.z || hv < R.y || hv > R.w) && t < INFINITY ? t : -1.0f;
}

// closest of the primitives both legs share (all but the light and sphere 0)
__device__ __forceinline__ Hit closest_shared(const PairShared& S, const Origin& O, const float d[3],
                                              const float inv[3], bool live) {
    const float* o = O.o;
    Hit h{INFINITY, -1};
    if (O.in) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int q = d[a] > 0.0f ? S.wall_hi[a] : S.wall_lo[a];
            quad_hit(S.rect[q], S.plane[q], q, a, o, d, inv, h);
        }
    } else {
        for (int q = 0; q < 6; ++q) {   // rare: not unrolled, to keep the code small
            const float t = any_axis_t(S, q, o[0], o[1], o[2], d[0], d[1], d[2]);
            if (t > 0.0f && t < h.t) { h.t = t; h.prim = q; }
        }
    }
#pragma unroll
    for (int q = 6; q < 12; ++q) quad_hit(S.rect[q], S.plane[q], q, (q - 6) >> 1, o, d, inv, h);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float t = sphere_t(S.sph[i], O.cc[i], o, d, live);
        const bool ok = t > 0.0f && t < h.t;
        h.t = ok ? t : h.t;
        h.prim = ok ? 14 + i : h.prim;
    }
    return h;
}

// adds one leg's light and sphere 0; equal distances go to the lower index
__device__ __forceinline__ void add_leg(const PairLeg& G, const float o[3], const float d[3], const float inv[3],
                                        bool live, Hit& h) {
    const float t = __fmul_rn(__fsub_rn(G.plane, o[1]), inv[1]);
    const float hu = __fmaf_rn(t, d[0], o[0]);
    const float hv = __fmaf_rn(t, d[2], o[2]);
    const float4 R = G.light;
    if (t > 0.0f && !(hu < R.x || hu > R.z || hv < R.y || hv > R.w) && t < INFINITY &&
        (t < h.t || (t == h.t && h.prim > kLight))) {
        h.t = t;
        h.prim = kLight;
    }
    const float ts = sphere_t(G.sph, sphere_cc(G.sph, o), o, d, live);
    if (ts > 0.0f && (ts < h.t || (ts == h.t && h.prim > 13))) {
        h.t = ts;
        h.prim = 13;
    }
}

// Is the light the closest primitive along a shadow ray?  The light's
// distance first, then any primitive that takes its place: a quad (lower
// index) at most as far, a sphere (higher index) nearer.
__device__ __forceinline__ bool light_seen(const PairShared& S, const PairLeg& G, const Origin& O, const float d[3],
                                           bool live) {
    const float* o = O.o;
    const float inv1 = __frcp_rn(d[1]);
    const float tl = __fmul_rn(__fsub_rn(G.plane, o[1]), inv1);
    const float lu = __fmaf_rn(tl, d[0], o[0]);
    const float lv = __fmaf_rn(tl, d[2], o[2]);
    const float4 R = G.light;
    bool seen = live && tl > 0.0f && !(lu < R.x || lu > R.z || lv < R.y || lv > R.w) && tl < INFINITY;
    auto blocks = [&](float4 Q, float plane, int a, const float* inv) {
        const int u = a == 0 ? 1 : 0, v = a == 2 ? 1 : 2;
        const float t = __fmul_rn(__fsub_rn(plane, o[a]), inv[a]);
        const float hu = __fmaf_rn(t, d[u], o[u]);
        const float hv = __fmaf_rn(t, d[v], o[v]);
        return t > 0.0f && !(hu < Q.x || hu > Q.z || hv < Q.y || hv > Q.w) && t <= tl;
    };
    if (!__any_sync(0xffffffffu, seen)) return false;
    if (!(O.in && G.light_inside)) {
        for (int q = 0; q < 6; ++q) {   // rare: not unrolled, the walls behind an inside origin are rejected too
            const float t = any_axis_t(S, q, o[0], o[1], o[2], d[0], d[1], d[2]);
            seen = seen && !(t > 0.0f && t <= tl);
        }
    }
    __syncwarp();
    {
        const float inv[3] = {__frcp_rn(d[0]), inv1, __frcp_rn(d[2])};
#pragma unroll
        for (int q = 6; q < 12; ++q) seen = seen && !blocks(S.rect[q], S.plane[q], (q - 6) >> 1, inv);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float4 sp = i == 0 ? G.sph : S.sph[i - 1];
        const float t = sphere_t(sp, i == 0 ? sphere_cc(sp, o) : O.cc[i - 1], o, d, seen);
        seen = seen && !(t > 0.0f && t < tl);
    }
    return seen;
}

// surface at the hit: normal against the ray and the offset origin
__device__ __forceinline__ void surface(const PairShared& S, const PairLeg& G, int prim, const float x[3],
                                        const float d[3], float n[3], float o2[3]) {
    if (prim < 12) {
        const int a = prim < 6 ? prim >> 1 : (prim - 6) >> 1;
        const float da = a == 0 ? d[0] : (a == 1 ? d[1] : d[2]);
        const float s = da > 0.0f ? -1.0f : 1.0f;
        n[0] = a == 0 ? s : 0.0f;
        n[1] = a == 1 ? s : 0.0f;
        n[2] = a == 2 ? s : 0.0f;
    } else {
        const float4 sp = prim == 13 ? G.sph : S.sph[prim - 14];
        const float isr = S.isr[prim - 13];
        n[0] = __fmul_rn(__fsub_rn(x[0], sp.x), isr);
        n[1] = __fmul_rn(__fsub_rn(x[1], sp.y), isr);
        n[2] = __fmul_rn(__fsub_rn(x[2], sp.z), isr);
        if (dot3(n, d) > 0.0f) { n[0] = -n[0]; n[1] = -n[1]; n[2] = -n[2]; }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) o2[c] = __fmaf_rn(n[c], 1e-4f, x[c]);
}

// next-event estimation of one leg: adds to its radiance sums L[c][0];
// power: throughput times albedo times emission
__device__ __forceinline__ void add_light(const PairShared& S, const PairLeg& G, bool live, const u32x4& w0,
                                          const float n[3], const Origin& O, const float power[3], float (*L)[32]) {
    const float* o2 = O.o;
    const float4 R = G.light;
    const float ly[3] = {__fmaf_rn(u24f(w0.x), __fsub_rn(R.z, R.x), R.x), G.plane,
                         __fmaf_rn(u24f(w0.y), __fsub_rn(R.w, R.y), R.y)};
    const float wv[3] = {__fsub_rn(ly[0], o2[0]), __fsub_rn(ly[1], o2[1]), __fsub_rn(ly[2], o2[2])};
    const float dist2 = dot3(wv, wv);
    const float idist = __frcp_rn(__fsqrt_rn(dist2));
    const float om[3] = {__fmul_rn(wv[0], idist), __fmul_rn(wv[1], idist), __fmul_rn(wv[2], idist)};
    const float cosx = dot3(n, om);
    const float cosl = om[1];
    live = live && cosx > 0.0f && cosl > 0.0f;
    if (light_seen(S, G, O, om, live)) {
        const float geo = __fmul_rn(__fmul_rn(__fdiv_rn(__fmul_rn(cosx, cosl), dist2), G.area), kInvPi);
#pragma unroll
        for (int c = 0; c < 3; ++c) L[c][0] = __fmaf_rn(power[c], geo, L[c][0]);
    }
    __syncwarp();
}

// cosine-weighted continuation around n (see radiance)
__device__ __forceinline__ void next_direction(const PairShared& S, uint32_t idx, uint32_t cbase, uint32_t c2,
                                               uint32_t request, const u32x4& w0, const float n[3], float nd[3]) {
    float a = 0.0f, b = 0.0f;
    {
        float ta = __fmaf_rn(u24f(w0.z), 2.0f, -1.0f), tb = __fmaf_rn(u24f(w0.w), 2.0f, -1.0f);
        bool found = __fmaf_rn(ta, ta, __fmul_rn(tb, tb)) < 1.0f;
        if (found) { a = ta; b = tb; }
        for (uint32_t blk = 1; blk <= 3 && !found; ++blk) {
            const u32x4 wb = philox_keyed(S, idx, cbase | blk, c2, request);
            ta = __fmaf_rn(u24f(wb.x), 2.0f, -1.0f);
            tb = __fmaf_rn(u24f(wb.y), 2.0f, -1.0f);
            found = __fmaf_rn(ta, ta, __fmul_rn(tb, tb)) < 1.0f;
            if (!found) {
                ta = __fmaf_rn(u24f(wb.z), 2.0f, -1.0f);
                tb = __fmaf_rn(u24f(wb.w), 2.0f, -1.0f);
                found = __fmaf_rn(ta, ta, __fmul_rn(tb, tb)) < 1.0f;
            }
            if (found) { a = ta; b = tb; }
        }
    }
    __syncwarp();
    const float r2 = __fmaf_rn(a, a, __fmul_rn(b, b));
    const float cz = __fsqrt_rn(__fsub_rn(1.0f, r2));
    const float sg = copysignf(1.0f, n[2]);
    const float aa = __fdiv_rn(-1.0f, __fadd_rn(sg, n[2]));
    const float bb = __fmul_rn(__fmul_rn(n[0], n[1]), aa);
    const float t1[3] = {__fmaf_rn(__fmul_rn(sg, __fmul_rn(n[0], n[0])), aa, 1.0f), __fmul_rn(sg, bb),
                         -__fmul_rn(sg, n[0])};
    const float t2[3] = {bb, __fmaf_rn(__fmul_rn(n[1], n[1]), aa, sg), -n[1]};
#pragma unroll
    for (int c = 0; c < 3; ++c) nd[c] = __fmaf_rn(cz, n[c], __fmaf_rn(b, t2[c], __fmul_rn(a, t1[c])));
}

// What the paths of one pair have in common.
struct PairRng {
    uint32_t request, c2, k;
};

__device__ void load_pair(const PtArgs& A, PairShared& S) {
    const int t = threadIdx.x;
    if (t < 12) {
        S.rect[t] = make_float4(A.qgeom[t][1], A.qgeom[t][2], A.qgeom[t][3], A.qgeom[t][4]);
        S.plane[t] = A.qgeom[t][0];
        for (int c = 0; c < 3; ++c) S.alb[t][c] = A.qalb[t][c];
    } else if (t == 12) {
        S.alb[12][0] = S.alb[12][1] = S.alb[12][2] = 0.0f;
    } else if (t < 16) {
        const int i = t - 13;
        if (i > 0) S.sph[i - 1] = make_float4(A.sc[i][0], A.sc[i][1], A.sc[i][2], __fmul_rn(A.sr[i], A.sr[i]));
        for (int c = 0; c < 3; ++c) S.alb[t][c] = A.salb[i][c];
        S.isr[i] = __frcp_rn(A.sr[i]);
        S.em[i] = A.em[i];
        // wall planes of axis i (quads 2 i, 2 i + 1)
        const float p0 = A.qgeom[2 * i][0], p1 = A.qgeom[2 * i + 1][0];
        S.box_lo[i] = fminf(p0, p1);
        S.box_hi[i] = fmaxf(p0, p1);
        S.wall_lo[i] = p0 <= p1 ? 2 * i : 2 * i + 1;
        S.wall_hi[i] = p0 <= p1 ? 2 * i + 1 : 2 * i;
    } else if (t < 18) {
        PairLeg& G = S.leg[t - 16];
        const float* p = S.p[t - 16];
        G.light = make_float4(__fsub_rn(p[0], A.light_half), __fsub_rn(p[2], A.light_half),
                              __fadd_rn(p[0], A.light_half), __fadd_rn(p[2], A.light_half));
        G.plane = p[1];
        G.area = __fmul_rn(__fsub_rn(G.light.z, G.light.x), __fsub_rn(G.light.w, G.light.y));
        G.sph = make_float4(p[3], p[4], p[5], __fmul_rn(A.sr[0], A.sr[0]));
        const float lmin[3] = {G.light.x, G.plane, G.light.y}, lmax[3] = {G.light.z, G.plane, G.light.w};
        bool in = true;
        for (int a = 0; a < 3; ++a) {
            const float p0 = A.qgeom[2 * a][0], p1 = A.qgeom[2 * a + 1][0];
            in = in && lmin[a] >= fminf(p0, p1) + kWallMargin && lmax[a] <= fmaxf(p0, p1) - kWallMargin;
        }
        G.light_inside = in ? 1 : 0;
    }
}

// kSplit: the CTAs of a cluster render one pair, each a round of kSlots x 256
// pixels at a time; rank 0 adds up their pixels in order.
template <int kSlots, bool kSplit>
__global__ void __launch_bounds__(kThreads, 4) ptbox_pair_kernel(PtArgs A, RenderBatch b) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    PairShared& S = *reinterpret_cast<PairShared*>(s_dyn);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    PairWarp<kSlots>& Q = reinterpret_cast<PairWarp<kSlots>*>(s_dyn + ((sizeof(PairShared) + 15) & ~size_t(15)))[warp];
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int parts = kSplit ? (int)cluster.num_blocks() : 1, rank = kSplit ? (int)cluster.block_rank() : 0;
    const int m = 2 * ((int)blockIdx.x / parts);
    PairRng rng;
    {
        const Pert pt = resolve(b, m);
        if (tid == 32) {
            uint32_t k0 = (uint32_t)pt.seed, k1 = (uint32_t)(pt.seed >> 32);
            for (int r = 0; r < 5; ++r) {
                S.keys[r] = make_uint4(k0, k1, k0 + 0x9E3779B9u, k1 + 0xBB67AE85u);
                k0 += 2u * 0x9E3779B9u;
                k1 += 2u * 0xBB67AE85u;
            }
        }
        rng.request = pt.request;
        const uint2 mt = *pt.meta;
        rng.c2 = (TAG_PATH << 24) | (mt.x & 0xFFFFFFu);
        rng.k = mt.y;
        if (tid < 16) {
            const int leg = tid >> 3, j = tid & 7;
            const Pert pl = resolve(b, m + leg);
            if (j < 6) S.p[leg][j] = __fadd_rn(pl.theta[j], pl.tau[j]);
        }
    }
    __syncthreads();
    load_pair(A, S);
    __syncthreads();
    const int spp = A.spp, depth = A.depth, npx = A.W * A.H;
    const float inv_spp = 1.0f / (float)spp;
    Q.acc[0][lane] = Q.acc[1][lane] = 0.0f;
    const uint64_t w_recip = ((1ull << 40) + (uint64_t)A.W - 1) / (uint64_t)A.W;
    for (int first = 0; first < npx; first += parts * kSlots * kThreads) {
        const int px0 = first + rank * kSlots * kThreads + warp * 32;
#pragma unroll
        for (int i = 0; i < kSlots * 6; ++i) (&Q.L[0][0][0])[i * 32 + lane] = 0.0f;
        __syncwarp();
        int s = 0, slot = 0, queued = 0;
        const int slots = max(0, min(kSlots, (npx - px0 + kThreads - 1) / kThreads));
        while (slots > 0) {
            // the next batch of the warp: 32 queued legs (fewer at a sample's
            // end), or the camera paths of the next slot's pixels
            const bool finish = queued >= 32 || (slot == slots && queued > 0);
            if (!finish && slot == slots) {
                slot = 0;
                if (++s == spp) break;
            }
            uint32_t mask;          // legs on this lane's path
            int leg = 0, vert = 1;  // leg: the one leg of a queued path
            int prim = 13;
            float t = 0.0f;
            Origin O;
            float* o = O.o;
            float d[3], beta[3];
            uint32_t idx;
            float (*L)[32];
            if (finish) {
                const int n = min(queued, 32);
                queued -= n;
                const int e = queued + (lane < n ? lane : 0);
                // the hit on sphere 0 is stored as the origin, t = 0
#pragma unroll
                for (int c = 0; c < 3; ++c) { o[c] = Q.q[c][e]; d[c] = Q.q[3 + c][e]; beta[c] = Q.q[6 + c][e]; }
                const uint32_t meta = __float_as_uint(Q.q[9][e]);   // lane | slot << 8 | leg << 16 | vertex << 24
                const int from = (int)((meta >> 8) & 0xFFu), src = (int)(meta & 31u);
                leg = (int)((meta >> 16) & 1u);
                vert = (int)(meta >> 24);
                mask = lane < n ? 1u << leg : 0u;
                idx = (uint32_t)((px0 + from * kThreads + src) * spp + s);
                L = reinterpret_cast<float (*)[32]>(&Q.L[from][0][src]);
                __syncwarp();
            } else {
                const int px = px0 + slot * kThreads + lane;
                mask = px < npx ? 3u : 0u;
                const int y = (int)(((uint64_t)(uint32_t)px * w_recip) >> 40), xp = px - y * A.W;
                idx = (uint32_t)(px * spp + s);
                const u32x4 wj = philox_keyed(S, idx, rng.k << 8, rng.c2, rng.request);
                const float fx = __fadd_rn((float)xp, u24f(wj.x));
                const float fy = __fadd_rn((float)y, u24f(wj.y));
                d[0] = __fmaf_rn(fx, A.pix_scale, -A.tan_half);
                d[1] = __fmaf_rn(-fy, A.pix_scale, A.tan_half);
                d[2] = -1.0f;
                const float il = __frcp_rn(__fsqrt_rn(dot3(d, d)));
                d[0] = __fmul_rn(d[0], il); d[1] = __fmul_rn(d[1], il); d[2] = __fmul_rn(d[2], il);
                o[0] = 0.0f; o[1] = 0.0f; o[2] = A.cam_z;
                beta[0] = beta[1] = beta[2] = 1.0f;
                L = reinterpret_cast<float (*)[32]>(&Q.L[slot][0][lane]);
            }
            O.in = in_box(S, o);
            O.cc[0] = sphere_cc(S.sph[0], o);
            O.cc[1] = sphere_cc(S.sph[1], o);
            const int legs = finish ? 1 : 2;   // a queued path has its own leg, a camera path both
            bool resume = finish;              // queued paths start at their hit
#pragma unroll 1
            for (;;) {
                if (!resume) {
                    // the common ray's closest hit, then each leg's
                    const float inv[3] = {__frcp_rn(d[0]), __frcp_rn(d[1]), __frcp_rn(d[2])};
                    const Hit hs = closest_shared(S, O, d, inv, mask != 0u);
                    uint32_t on_sphere = 0u;
                    float t_sph = 0.0f, t_sph1 = 0.0f;
#pragma unroll 1
                    for (int j = 0; j < legs; ++j) {
                        const int l = finish ? leg : j;
                        const uint32_t bit = 1u << l;
                        Hit h = hs;
                        add_leg(S.leg[l], o, d, inv, (mask & bit) != 0u, h);
                        if (mask & bit) {
                            if (h.prim == 13) {
                                on_sphere |= bit;
                                t_sph1 = h.t;
                                if (on_sphere == bit) t_sph = h.t;
                            } else if (h.prim < 0 || h.prim == kLight) {
                                if (vert == 1 && h.prim == kLight && d[1] > 0.0f)
                                    for (int c = 0; c < 3; ++c) L[3 * l + c][0] = __fadd_rn(L[3 * l + c][0], S.em[c]);
                                mask &= ~bit;
                            }
                        }
                    }
                    // the lane goes on with the legs on the common surface, or
                    // with one leg on sphere 0 when there are none; the other
                    // leg on sphere 0 is queued
                    prim = hs.prim;
                    t = hs.t;
                    uint32_t push = on_sphere;
                    if (on_sphere != 0u && on_sphere == mask) {
                        prim = 13;
                        t = t_sph;   // the first leg's
                        if (!finish) leg = (on_sphere & 1u) ? 0 : 1;
                        push = on_sphere & ~(1u << leg);
                    }
                    if (!finish) {
                        mask &= ~push;
                        const unsigned pushers = __ballot_sync(0xffffffffu, push != 0u);
                        if (pushers) {
                            if (push) {
                                const int e = queued + __popc(pushers & ((1u << lane) - 1u));
#pragma unroll
                                for (int c = 0; c < 3; ++c) {
                                    Q.q[c][e] = __fmaf_rn(t_sph1, d[c], o[c]);
                                    Q.q[3 + c][e] = d[c];
                                    Q.q[6 + c][e] = beta[c];
                                }
                                Q.q[9][e] = __uint_as_float((uint32_t)lane | ((uint32_t)slot << 8) |
                                                            ((push >> 1) << 16) | ((uint32_t)vert << 24));
                            }
                            queued += __popc(pushers);
                            __syncwarp();
                        }
                    }
                    if (!__any_sync(0xffffffffu, mask != 0u)) break;
                    if (mask == 0u) prim = 0;
#pragma unroll
                    for (int c = 0; c < 3; ++c) o[c] = __fmaf_rn(t, d[c], o[c]);
                }
                resume = false;
                float n[3], x[3] = {o[0], o[1], o[2]};
                surface(S, S.leg[leg], prim, x, d, n, o);
                O.in = in_box(S, o);
                O.cc[0] = sphere_cc(S.sph[0], o);
                O.cc[1] = sphere_cc(S.sph[1], o);
                float power[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    beta[c] = __fmul_rn(beta[c], S.alb[prim][c]);
                    power[c] = __fmul_rn(beta[c], S.em[c]);
                }
                const uint32_t cbase = (rng.k << 8) | ((uint32_t)vert << 4);
                const u32x4 w0 = philox_keyed(S, idx, cbase, rng.c2, rng.request);
#pragma unroll 1
                for (int j = 0; j < legs; ++j) {
                    const int l = finish ? leg : j;
                    add_light(S, S.leg[l], ((mask >> l) & 1u) != 0u, w0, n, O, power, L + 3 * l);
                }
                if (vert >= depth) mask = 0u;
                if (!__any_sync(0xffffffffu, mask != 0u)) break;
                next_direction(S, idx, cbase, rng.c2, rng.request, w0, n, d);
                ++vert;
            }
            __syncwarp();
            if (!finish) ++slot;
        }
#pragma unroll
        for (int slot = 0; slot < kSlots; ++slot) {
            const int px = px0 + slot * kThreads + lane;
            if (px < npx) {
                const float* tg = A.target + 3 * (size_t)px;
                const float g0 = tg[0], g1 = tg[1], g2 = tg[2];
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const float d0 = __fmaf_rn(Q.L[slot][3 * l][lane], inv_spp, -g0);
                    const float d1 = __fmaf_rn(Q.L[slot][3 * l + 1][lane], inv_spp, -g1);
                    const float d2 = __fmaf_rn(Q.L[slot][3 * l + 2][lane], inv_spp, -g2);
                    const float v = __fmaf_rn(d2, d2, __fmaf_rn(d0, d0, __fmul_rn(d1, d1)));
                    if (kSplit) Q.L[slot][3 * l][lane] = v;
                    else Q.acc[l][lane] = __fadd_rn(Q.acc[l][lane], v);
                }
            }
        }
        __syncwarp();
        if (kSplit) {
            cluster.sync();
            if (rank == 0) {
                for (int q = 0; q < parts; ++q) {
                    const PairWarp<kSlots>* R = cluster.map_shared_rank(&Q, q);
                    const int qx0 = first + q * kSlots * kThreads + warp * 32 + lane;
#pragma unroll
                    for (int slot = 0; slot < kSlots; ++slot)
                        if (qx0 + slot * kThreads < npx)
                            for (int l = 0; l < 2; ++l) Q.acc[l][lane] = __fadd_rn(Q.acc[l][lane], R->L[slot][3 * l][lane]);
                }
            }
            cluster.sync();
        }
    }
    if (kSplit && rank != 0) return;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        const float v = warp_sum(Q.acc[l][lane]);
        if (lane == 0) S.part[l][warp] = v;
    }
    __syncthreads();
    if (tid < 2) {
        float v = 0.0f;
        for (int w = 0; w < kPairWarps; ++w) v += S.part[tid][w];
        *resolve(b, m + tid).loss = v / (float)(npx * 3);
    }
}

template <int kSlots>
constexpr size_t pair_smem() {
    return ((sizeof(PairShared) + 15) & ~size_t(15)) + kPairWarps * sizeof(PairWarp<kSlots>);
}
constexpr int kWhole = 5;   // slots of a CTA that renders a whole pair

// every two items 2 i, 2 i + 1 of the launch are the legs of one pair
bool in_pairs(const RenderBatch& b) {
    if (b.M & 1) return false;
    if (b.table_rows <= 0) return (b.per_row & 1) == 0;
    for (int r = 0; r < b.table_rows; ++r)
        if ((b.rows[r].start & 1) || (b.rows[r].m_begin & 1)) return false;
    return true;
}

PtArgs make_args(const DevScene& sc) {
    PtArgs a;
    for (int q = 0; q < 13; ++q) {
        a.qaxis[q] = sc.qaxis[q];
        for (int c = 0; c < 5; ++c) a.qgeom[q][c] = sc.qgeom[q][c];
        for (int c = 0; c < 3; ++c) a.qalb[q][c] = sc.qalb[q][c];
    }
    for (int i = 0; i < 3; ++i) {
        for (int c = 0; c < 3; ++c) { a.sc[i][c] = sc.sc_[i][c]; a.salb[i][c] = sc.salb[i][c]; }
        a.sr[i] = sc.sr[i];
    }
    a.light_half = sc.light_half; a.cam_z = sc.cam_z; a.tan_half = sc.tan_half; a.pix_scale = sc.pix_scale;
    for (int c = 0; c < 3; ++c) a.em[c] = sc.emission[c];
    a.W = sc.W; a.H = sc.H; a.spp = sc.spp; a.depth = sc.depth;
    a.target = sc.target;
    a.stats = sc.pt_stats;
    return a;
}

// quad axes of the procedural box (walls, then block faces: x x y y z z)
bool canonical_axes(const DevScene& sc) {
    static const int kAxis[12] = {0, 0, 1, 1, 2, 2, 0, 0, 1, 1, 2, 2};
    for (int q = 0; q < 12; ++q)
        if (sc.qaxis[q] != kAxis[q]) return false;
    return true;
}

template <int kSlots>
void launch_parts(const PtArgs& a, const RenderBatch& b, int parts, cudaStream_t s) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)parts;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)(b.M / 2) * (unsigned)parts);
    c.blockDim = dim3(kThreads);
    c.dynamicSmemBytes = pair_smem<kSlots>();
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, ptbox_pair_kernel<kSlots, true>, a, b);
}

// CTAs that share one pair of renders (1: none) and the pixels per lane of their
// rounds.  Both kernels compute the same bits; the lines come from timing them
// (GB300, 152 SMs; us, one render per CTA / pairs as chosen here):
//   8x8 to 24x24          one render: 46 / 101 at 16x16, 4 spp, M = 64
//   32x32, 4 spp          M 64: 158 / 105; 256: 189 / 212; 1,024: 496 / 557; 4,096: 1,754 / 1,561
//   48x48, 2 spp          M 64: 179 / 116; 256: 210 / 265; 1,024: 556 / 552; 4,096: 1,971 / 1,739
//   64x64, 2 spp          M 256: 364 / 308; 1,024: 975 / 896; 4,096: 3,459 / 3,137
//   128x128, 4 spp        M 64: 2,363 / 750; 1,024: 7,606 / 6,547; 4,096: 27,182 / 23,903
// A pair's lane has a longer serial chain (both legs' shadow rays) than a
// render's, so pairs need images of some size, and below 64x64 either few
// renders, each spread over a cluster, or enough to fill the GPU.
struct PairShape {
    int parts = 0, slots = 4;   // parts 0: one render per CTA
};
PairShape pair_shape(int npx, int pairs, int sms) {
    PairShape p;
    if (npx < 1024) return p;
    if (npx < 4096 && 2 * pairs > sms && 2 * pairs < 13 * sms) return p;
    p.parts = 1;
    // several waves of CTAs even out the end: split while a part keeps two rounds
    while (p.parts < 8 && pairs * p.parts < 16 * sms && 4096 * p.parts <= npx) p.parts *= 2;
    // fewer CTAs than the GPU holds: split on, down to 256 pixels a part
    while (p.parts < 8 && pairs * p.parts < 4 * sms && kThreads * p.parts < npx) p.parts *= 2;
    while (p.slots > 1 && p.slots * kThreads * p.parts >= 2 * npx) p.slots /= 2;
    while (p.slots > 1 && p.slots * kThreads * (p.parts / 2) >= npx) p.slots /= 2;
    return p;
}

// (four CTAs per SM for every scene: 8,192 renders of 128x128, 4 spp take 42 ms,
// 50 with three; a tuner's probe of 2,048 is split over clusters and cannot tell)
void launch_pairs(const PtArgs& a, const RenderBatch& b, const PairShape& p, cudaStream_t s) {
    const int pairs = b.M / 2;
    if (p.parts > 1) {
        if (p.slots == 4) launch_parts<4>(a, b, p.parts, s);
        else if (p.slots == 2) launch_parts<2>(a, b, p.parts, s);
        else launch_parts<1>(a, b, p.parts, s);
        return;
    }
    ptbox_pair_kernel<kWhole, false><<<pairs, kThreads, pair_smem<kWhole>(), s>>>(a, b);
}

template <bool kCanon>
void launch_loss(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    const PtArgs a = make_args(sc);
    if (sc.count_work && a.stats) {   // work counting (diagnostics), default launch shape
        ptbox_kernel<false, 3, kCanon, true><<<b.M, kThreads, 0, s>>>(a, b, nullptr, 0, 0, 0, 0, 0, 0, nullptr);
        return;
    }
    const PairShape p = kCanon && in_pairs(b) ? pair_shape(sc.W * sc.H, b.M / 2, num_sms()) : PairShape{};
    if (p.parts > 0) {
        launch_pairs(a, b, p, s);
        return;
    }
    switch (ptbox_resident(sc.render_variant, b.M, num_sms())) {
        case 2: ptbox_kernel<false, 2, kCanon><<<b.M, kThreads, 0, s>>>(a, b, nullptr, 0, 0, 0, 0, 0, 0, nullptr); break;
        case 3: ptbox_kernel<false, 3, kCanon><<<b.M, kThreads, 0, s>>>(a, b, nullptr, 0, 0, 0, 0, 0, 0, nullptr); break;
        default: ptbox_kernel<false, 4, kCanon><<<b.M, kThreads, 0, s>>>(a, b, nullptr, 0, 0, 0, 0, 0, 0, nullptr); break;
    }
}

}  // namespace

// Launch-shape variants (autotuner) of the kernel of one render per CTA: the same
// 256-thread layout and arithmetic, different register caps through the minimum
// number of resident CTAs per SM (ptbox_resident: by the launch's size, that up to 3,
// up to 2), so the choice never changes a result.  Scenes with the procedural box's
// quad layout use the compile-time-axis intersection, and the pair kernel, which has
// one shape, where it is faster.
void launch_ptbox_loss(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    if (canonical_axes(sc)) launch_loss<true>(sc, b, s);
    else launch_loss<false>(sc, b, s);
}

bool ptbox_variants_apply(const DevScene& sc, int M) {
    if (sc.count_work && sc.pt_stats) return false;
    return !canonical_axes(sc) || (M & 1) || pair_shape(sc.W * sc.H, M / 2, num_sms()).parts == 0;
}

cudaError_t ptbox_prepare() {
    return cudaFuncSetAttribute(ptbox_pair_kernel<kWhole, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)pair_smem<kWhole>());
}

// One thread per pixel over as many blocks as it takes (a 64x64 target of 16 samples
// by one block: 7.6 ms; the whole scene is made in 0.7 ms now).
void launch_ptbox_image(const DevScene& sc, const float* params, uint64_t seed, uint32_t request, uint32_t sub,
                        uint32_t k, uint32_t tag, int spp, float* img, cudaStream_t s) {
    RenderBatch b{};
    const int grid = (sc.W * sc.H + kThreads - 1) / kThreads;
    auto kernel = canonical_axes(sc) ? ptbox_kernel<true, 3, true> : ptbox_kernel<true, 3, false>;
    kernel<<<grid, kThreads, 0, s>>>(make_args(sc), b, params, seed, request, sub, k, tag, spp, img);
}

}  // namespace hr
