// K1: perturbation sampler and kernel weights (Sec. 3.2-3.5).
//
// A block draws a run of antithetic pairs of one sample group: a + leg from
// the positive lobe and a - leg from the negative lobe of the chosen kernel,
// every other dimension N(0, sigma^2) shared by both legs (Sec. 3.2,
// separability; Suppl. "Smooth Gradient Marginalization").  Lobe samples are
// computed in FP64 and rounded once to FP32: that FP32 value is the
// perturbation every renderer sees.  Weights are evaluated in FP64 at the
// FP32 perturbation and stored in FP32.
//
// Philox counter of pair k: (k, block, (1 << 24) | sub, request), key = seed.
// Block 0 = (component word, lobe uniform a, lobe uniform b, sign word);
// block 1 + b holds the Box-Muller uniforms of dims 4b .. 4b + 3.
#include <cmath>
#include <type_traits>

#include "hr_device.cuh"
#include "hr_internal.h"
#include "sample_device.cuh"

namespace hr {
namespace {

constexpr int kSampleThreads = 256;

// What both legs of a pair share.
struct PairDraw {
    int i, j;              // component, -1 without importance sampling
    uint32_t ua, ub, sg;   // Philox words of the lobe uniforms and the sign
};

// The component of pair k (see sample_leg).
__device__ PairDraw draw_component(const SampleArgs& a, const SampleGroup& G, const Lobes& L, int k, uint32_t c2) {
    const int n = a.n;
    const u32x4 w0 = philox_seed(a.seed, (uint32_t)k, 0u, c2, G.request);
    int i, j;
    if (G.comp_i == -3) {
        i = -1; j = -1;
    } else if (G.comp_i >= 0 && G.comp_j == -2) {
        i = G.comp_i;
        j = row_component(a.v, n, i, L, w0.x);
    } else if (G.comp_i >= 0) {
        i = G.comp_i;
        j = G.lobe == 0 ? G.comp_i : G.comp_j;
    } else if (G.lobe == 0) {
        i = (int)(((uint64_t)w0.x * (uint64_t)n) >> 32);
        j = i;
    } else {
        const int e = (int)(((uint64_t)w0.x * (uint64_t)(n * n)) >> 32);
        i = e / n;
        j = e - i * n;
    }
    return {i, j, w0.y, w0.z, w0.w};
}

// (a call, so that the compiler does not run it beside the path that avoids it)
__device__ __noinline__ float off_diagonal_fp64(float x, float y, double is4, double iS) {
    return (float)((double)x * (double)y * is4 * iS);
}

// RN32 of RN64(RN64(RN64(x y) is4) iS), the off-diagonal mixture weight, without
// FP64 where that is certain to give the same bits.  (ch, cl) holds is4 iS in two
// floats.  x y = p + q exactly; (hi, lo) is the product to a relative error
// below 2^-45 (each of q ch, p cl and the sums rounds terms of at most 2^-23
// of the result, ch + cl is within 2^-48 of is4 iS), the FP64 form has one
// below 2^-51, so both round to the same float unless the remainder r lies
// within 2^-43 of half a unit of s (or s is a power of two, whose lower
// neighbour is nearer).  There, and outside the range in which none of the
// terms underflows, FP64 decides.
__device__ __forceinline__ float off_diagonal_weight(float x, float y, float ch, float cl, double is4, double iS) {
    const float p = __fmul_rn(x, y), q = __fmaf_rn(x, y, -p);
    const float hi = __fmul_rn(p, ch);
    const float lo = __fmaf_rn(q, ch, __fmaf_rn(p, cl, __fmaf_rn(p, ch, -hi)));
    const float s = __fadd_rn(hi, lo), r = __fsub_rn(lo, __fsub_rn(s, hi));
    // half a unit of s: 2^(exponent - 24)
    const float half = __int_as_float((__float_as_int(s) & 0x7F800000) - (24 << 23));
    const float as = fabsf(s), ap = fabsf(p);
    if (as > 0x1p-60f && as < 0x1p60f && ap > 0x1p-60f && ap < 0x1p60f && ch > 0x1p-60f && ch < 0x1p60f &&
        (__float_as_int(s) & 0x007FFFFF) != 0 && fabsf(__fsub_rn(fabsf(r), half)) > as * 0x1p-43f)
        return s;
    return off_diagonal_fp64(x, y, is4, iS);
}

// Weights of the Hessian mixture, n (n + 1) / 2 elements a row: thread (e0, r0)
// as below.  The diagonal (a difference) is formed in FP64, by n threads.
__device__ __forceinline__ void hessian_weights(const float* s_t, const double* s_td, const double* s_iS, int rows,
                                                const float2* s_c, int n, int E, double s2, double is4, int e0, int ew,
                                                int r0, int rstep, float* wm) {
    int i = 0, rem = e0;
    for (int e = e0; e < E; e += ew, rem += ew) {
        while (rem >= n - i) { rem -= n - i; ++i; }
        if (rem == 0) continue;
        const int j = i + rem;
        for (int r = r0; r < rows; r += rstep) {
            const float2 c = s_c[r];   // is4 / S in two floats, 0 without a mixture density
            wm[(size_t)r * E + e] =
                c.x != 0.0f ? off_diagonal_weight(s_t[r * n + i], s_t[r * n + j], c.x, c.y, is4, s_iS[r]) : 0.0f;
        }
    }
    for (int x = threadIdx.x; x < rows * n; x += blockDim.x) {
        const int r = x / n, d = x - r * n;
        const double ti = s_td[x], iS = s_iS[r];
        const double c = (ti * ti - s2) * is4;
        wm[(size_t)r * E + upper_index(d, d, n)] = iS != 0.0 ? (float)(c * iS) : 0.0f;
    }
}

// One block: np pairs from pair np blockIdx.x of group blockIdx.y.  The FP64
// chains of a pair (a log or the Lambert-W solve costs thousands of dependent
// cycles on this GPU) do not depend on one another, so they run in different
// warps at the same time, each kind in warps of its own:
//   root units      the diagonal-lobe inverse, one leg per lane;
//   radius units    half-Rayleigh radii, two per pair;
//   Gaussian units  two dims of a pair per lane, once for both legs.
// Then one lane per leg forms the sums over the dims that its weights need
// (in dim order), and all threads write the weights, a row's elements over
// consecutive threads.  Every value is formed by the operations of sample_leg.
//
// Bound by FP64 latency where the launch is small, by the FP64 rate (2 lanes a
// cycle and SM) for many dims.  Stage times between events in us, with one leg
// per thread and this way (both with log(); log_pos takes one to three off): 3 x 1,024
// element-wise 2 x 2: 18.2, 15.6; 4,096 aggregate 2 x 2: 24.6, 18.0; 55 x 64 element-wise
// 10 x 10: 30.3, 16.5; 1,024 aggregate 64 x 64 (2,080 weights each): 671, 34; 16,384
// aggregate HVPs of 64 dims: 169, 95.
__global__ void __launch_bounds__(kSampleThreads) sample_kernel(SampleArgs a, Lobes host_lobes, int np) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ PairDraw s_draw[64];
    __shared__ double s_iS[128], s_tv[128];
    __shared__ float2 s_c[128];
    __shared__ double s_sum[3 * 128];
    __shared__ Lobes s_lobes;
    let_next_start();
    // without these the draws depend on nothing that an earlier kernel writes: they
    // overlap the end of the previous estimate, and only the stores wait for it
    if (a.groups || a.v || a.step || a.sigma_row) wait_for_previous();
    const SampleGroup G = a.groups ? a.groups[blockIdx.y] : a.rule.group((int)blockIdx.y);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x, n = a.n;
    const int kb = blockIdx.x * np;
    if (kb >= G.P) return;
    const int pairs = min(np, G.P - kb), rows = 2 * pairs;
    double* s_td = reinterpret_cast<double*>(s_dyn);       // [rows][n] the perturbations in FP64
    float* s_t = reinterpret_cast<float*>(s_td + 2 * np * n);   // [rows][n]
    const uint32_t sub = G.sub + (a.step ? 64u * (uint32_t)(*a.step) : 0u);
    const uint32_t c2 = (TAG_SAMPLE << 24) | (sub & 0xFFFFFFu);
    if (a.sigma_row) {
        if (tid == 0) s_lobes = lobes_for(a, G, host_lobes);
        __syncthreads();
    }
    const Lobes& L = a.sigma_row ? s_lobes : host_lobes;
    if (tid < pairs) s_draw[tid] = draw_component(a, G, L, kb + tid, c2);
    __syncthreads();
    const double sigma = L.sigma;
    const int leg_units = (rows + 31) >> 5;   // root and radius units: two lanes per pair
    const int half = (n + 1) >> 1, gauss = pairs * half;
    const int units = 2 * leg_units + ((gauss + 31) >> 5);
    for (int u = warp; u < units; u += T >> 5) {
        if (u < leg_units) {
            const int r = u * 32 + lane, leg = r & 1;
            if (r < rows && G.lobe != 0) {
                const PairDraw D = s_draw[r >> 1];
                if (D.i >= 0 && D.i == D.j) {
                    // + leg: the tails (c in (0, 1/4) or (3/4, 1)); - leg: the middle
                    const double ua = u01d(D.ua);
                    const double c = leg ? 0.25 + 0.5 * ua : (ua < 0.5 ? 0.5 * ua : 0.5 + 0.5 * ua);
                    s_t[r * n + D.i] = (float)(sigma * diag_inverse(c));
                }
            }
        } else if (u < 2 * leg_units) {
            const int r = (u - leg_units) * 32 + lane, b = r & 1;   // b: which of the two radii
            if (r < rows) {
                const PairDraw D = s_draw[r >> 1];
                if (D.i >= 0 && (G.lobe == 0 ? b == 0 : D.i != D.j)) {
                    const double x = sigma * sqrt(-2.0 * log_pos(u01d(b ? D.ub : D.ua)));
                    float* t0 = s_t + (r - b) * n;   // the + leg's row; the - leg's follows
                    if (G.lobe == 0) {
                        t0[D.i] = (float)x;
                        t0[n + D.i] = (float)-x;
                    } else {
                        const double sg = (D.sg & 1u) ? -1.0 : 1.0;
                        if (b == 0) {
                            t0[D.i] = (float)(sg * x);
                            t0[n + D.i] = (float)(sg * x);
                        } else {
                            t0[D.j] = (float)(sg * x);
                            t0[n + D.j] = (float)(-sg * x);
                        }
                    }
                }
            }
        } else {
            const int q = (u - 2 * leg_units) * 32 + lane;
            if (q < gauss) {
                const int p = q / half, d = 2 * (q - p * half);
                const PairDraw D = s_draw[p];
                const bool need0 = d != D.i && d != D.j, need1 = d + 1 < n && d + 1 != D.i && d + 1 != D.j;
                if (need0 || need1) {
                    const u32x4 r = philox_seed(a.seed, (uint32_t)(kb + p), (uint32_t)(1 + d / 4), c2, G.request);
                    const double R = sqrt(-2.0 * log_pos(u01d((d & 2) ? r.z : r.x)));
                    const double ph = 2.0 * kPi * u01d((d & 2) ? r.w : r.y);
                    double sn, cs;
                    sincos(ph, &sn, &cs);
                    float* t0 = s_t + 2 * p * n + d;
                    const bool plain = G.comp_i == -3;   // legs +tau and -tau
                    if (need0) {
                        const double g = sigma * (R * cs);
                        t0[0] = (float)g;
                        t0[n] = plain ? (float)(-g) : (float)g;
                    }
                    if (need1) {
                        const double g = sigma * (R * sn);
                        t0[1] = (float)g;
                        t0[n + 1] = plain ? (float)(-g) : (float)g;
                    }
                }
            }
        }
    }
    __syncthreads();
    wait_for_previous();
    if (a.theta_out && blockIdx.x == 0 && blockIdx.y == 0) {
        for (int d = tid; d < a.theta_n; d += T)
            a.theta_out[d] = a.theta_in ? __double2float_rn(a.theta_in[d]) : a.theta_vals[d];
    }
    const int m0 = G.m0 + 2 * kb;
    float* tau = a.tau + (size_t)m0 * n;
    for (int x = tid; x < rows * n; x += T) {
        const float t = s_t[x];
        tau[x] = t;
        s_td[x] = (double)t;
    }
    // With many dims, the three sums of the Hessian mixture's density in lanes of
    // their own: sum |fma(x, m, k)| is sum |x^2 - s^2|, sum |x| or sum x^2
    // (x^2 of a float is exact in FP64), each in dim order.
    const bool split = G.comp_i == -1 && G.quantity != 0 && n >= 16;
    if (split) {
        __syncthreads();
        for (int q = tid; q < 3 * rows; q += T) {
            const int r = q / 3, which = q - 3 * r;
            const double* x = s_td + r * n;
            const double k = which == 0 ? -L.s2 : 0.0;
            double acc = 0.0;
            for (int d = 0; d < n; ++d) acc += fabs(fma(x[d], which == 1 ? 1.0 : x[d], k));
            s_sum[q] = acc;
        }
        __syncthreads();
    }
    for (int r = tid; r < rows; r += T) {
        const float* t = s_t + r * n;
        if (a.meta) a.meta[m0 + r] = make_uint2(sub, (uint32_t)(kb + (r >> 1)));
        double iS = 0.0, tv = 0.0;
        if (G.quantity == 4) {
            iS = row_weight(a.v, n, G.comp_i, L, t);
        } else if (G.comp_i < 0) {
            if (G.comp_i == -1) {
                const double S = G.quantity == 0 ? grad_mixture(t, n, L)
                                 : split ? hess_density(s_sum[3 * r], s_sum[3 * r + 1], s_sum[3 * r + 2], L)
                                         : hess_mixture(t, n, L);
                iS = S > 0.0 ? recip_mixture(S) : 0.0;
            }
            if (G.quantity == 2) tv = dot_dims(t, a.v, n);
        }
        if (G.quantity == 3) a.invS[m0 + r] = (float)iS;
        s_iS[r] = iS;
        s_tv[r] = tv;
        const double c = L.is4 * iS;
        const float ch = (float)c;
        // (0 says that there is no density: a product that leaves FP32 becomes the smallest
        // number instead, with which the weights take their FP64 form)
        s_c[r] = make_float2(ch != 0.0f || iS == 0.0 ? ch : 0x1p-149f, (float)(c - (double)ch));
    }
    if (!a.w || G.quantity == 3) return;
    __syncthreads();
    // weights: thread (e0, r0) takes elements e0, e0 + ew, ... of rows r0, r0 + T / ew, ...
    const int E = a.E;
    int ew = 1;
    while (ew < E && ew < T) ew <<= 1;
    const int e0 = tid & (ew - 1), r0 = tid / ew, rstep = T / ew;
    const double s2 = L.s2, is2 = L.is2, is4 = L.is4;
    float* wm = a.w + (size_t)m0 * E;
    const bool mixture_hessian = G.quantity == 1 && G.comp_i == -1;   // (formed by a loop of its own)
    if (mixture_hessian) hessian_weights(s_t, s_td, s_iS, rows, s_c, n, E, s2, is4, e0, ew, r0, rstep, wm);
    for (int e = e0; e < E; e += ew) {
        if (G.quantity == 4 || G.comp_i >= 0) {   // one element per row
            int hit = G.comp_i;
            double z = G.quantity == 0 ? L.Zg : 0.0;
            if (G.quantity == 1) {
                const int lo = min(G.comp_i, G.comp_j), hi = max(G.comp_i, G.comp_j);
                hit = upper_index(lo, hi, n);
                z = lo == hi ? L.Zd : L.Zo;
            }
            for (int r = r0; r < rows; r += rstep) {
                const double v = G.quantity == 4 ? s_iS[r] : ((r & 1) ? -1.0 : 1.0) * z;
                wm[(size_t)r * E + e] = e == hit ? (float)v : 0.0f;
            }
        } else if (G.quantity == 1) {
            if (mixture_hessian) break;
            int i = 0, rem = e;
            while (rem >= n - i) { rem -= n - i; ++i; }
            const int j = i + rem;
            for (int r = r0; r < rows; r += rstep) {
                const double ti = s_td[r * n + i], tj = s_td[r * n + j];
                const double c = (i == j) ? (ti * ti - s2) * is4 : ti * tj * is4;
                const double iS = s_iS[r];
                wm[(size_t)r * E + e] = G.comp_i == -3 ? (float)c : (iS != 0.0 ? (float)(c * iS) : 0.0f);
            }
        } else if (G.quantity == 0) {
            for (int r = r0; r < rows; r += rstep) {
                const double c = s_td[r * n + e] * is2;
                wm[(size_t)r * E + e] = G.comp_i == -3 ? (float)c : (float)(c * s_iS[r]);
            }
        } else {
            const double v = a.v[e];
            for (int r = r0; r < rows; r += rstep) {
                const double hv = s_td[r * n + e] * s_tv[r] * is4 - v * is2;
                const double iS = s_iS[r];
                wm[(size_t)r * E + e] = G.comp_i == -3 ? (float)hv : (iS != 0.0 ? (float)(hv * iS) : 0.0f);
            }
        }
    }
}

// K6: estimator sums.  Element e sums w[m][e] * loss[m] over its row range in
// a fixed order: 256 contiguous chunks, each a Kahan-compensated FP32 sum,
// then an FP64 tree over the chunks (t, t + o), o = 128 .. 1, times 1/(2P).
constexpr int kChunks = 256;

// Kahan sums of rows [m, end): x and, with kAbs, |x|; the loads of sixteen rows
// go out before their sums, which stay in row order.
template <bool kAbs>
__device__ __forceinline__ void chunk_sums(const float* w, const float* loss, int E, int e, int m, int end,
                                           Kahan& ks, Kahan& ka) {
    auto batch = [&](auto count) {
        constexpr int kN = decltype(count)::value;
        float x[kN];
#pragma unroll
        for (int u = 0; u < kN; ++u) x[u] = __fmul_rn(w[(size_t)(m + u) * E + e], loss[m + u]);
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            ks.add(x[u]);
            if (kAbs) ka.add(fabsf(x[u]));
        }
        m += kN;
    };
    while (m + 15 < end) batch(std::integral_constant<int, 16>{});
    if (m + 7 < end) batch(std::integral_constant<int, 8>{});
    if (m + 3 < end) batch(std::integral_constant<int, 4>{});
    while (m < end) batch(std::integral_constant<int, 1>{});
}

// kEl elements per block of 256 threads: thread (slot, e) holds the chunks
// slot + kSlots j of element e, so that a warp's loads of a row cover kEl
// consecutive weights (one 32-byte sector for 8).  The tree's upper levels add
// chunks of one thread, the others go through shared memory.  With one element
// per block every chunk has its thread.
// kStaged (one element): a chunk's rows lie apart from its neighbour's, so that
// a warp reading its threads' chunks row by row touches 32 lines a load; instead
// sixteen lanes load sixteen rows of one chunk, and the products go through
// shared memory to the chunk's thread.
template <int kEl, bool kAbs, bool kStaged>
__global__ void __launch_bounds__(kChunks) finalize_kernel(FinalizeArgs a) {
    constexpr int kSlots = kChunks / kEl, kJ = kEl;   // kJ chunks per thread
    __shared__ double sh[kEl][kSlots + 1], sa[kAbs ? kEl : 1][kSlots + 1];
    const int el = threadIdx.x % kEl, slot = threadIdx.x / kEl;
    const int e = blockIdx.x * kEl + el;
    const int m0 = (a.elementwise ? e * a.pairs2 : 0) + (int)blockIdx.y * a.row_stride;
    const int cnt = a.pairs2;
    let_next_start();
    wait_for_previous();
    const int chunk = (cnt + kChunks - 1) / kChunks;
    double s[kJ], sb[kAbs ? kJ : 1];
    if constexpr (kStaged) {
        constexpr int kRows = 16;
        __shared__ float sx[kChunks][kRows + 1];
        Kahan ks, ka;
        const int mine = min(cnt, (slot + 1) * chunk) - slot * chunk;   // rows of this thread's chunk (may be <= 0)
        for (int r0 = 0; r0 < chunk; r0 += kRows) {
            __syncthreads();
            float x[kRows];
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                const int q = threadIdx.x + kChunks * k, row = r0 + q % kRows, m = (q / kRows) * chunk + row;
                const bool in = row < chunk && m < cnt;
                x[k] = in ? __fmul_rn(a.w[(size_t)(m0 + m) * a.E + e], a.loss[m0 + m]) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                const int q = threadIdx.x + kChunks * k;
                sx[q / kRows][q % kRows] = x[k];
            }
            __syncthreads();
            const int n_here = min(kRows, mine - r0);
            for (int k = 0; k < n_here; ++k) {
                ks.add(sx[slot][k]);
                if (kAbs) ka.add(fabsf(sx[slot][k]));
            }
        }
        sh[0][slot] = (double)ks.s - (double)ks.c;
        if (kAbs) sa[0][slot] = (double)ka.s - (double)ka.c;
    } else if (e < a.E) {
#pragma unroll
        for (int j = 0; j < kJ; ++j) {
            const int b = m0 + (slot + kSlots * j) * chunk;
            Kahan ks, ka;
            chunk_sums<kAbs>(a.w, a.loss, a.E, e, b, min(m0 + cnt, b + chunk), ks, ka);
            s[j] = (double)ks.s - (double)ks.c;
            if (kAbs) sb[j] = (double)ka.s - (double)ka.c;
        }
#pragma unroll
        for (int o = kJ / 2; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < o; ++j) {
                s[j] += s[j + o];
                if (kAbs) sb[j] += sb[j + o];
            }
        sh[el][slot] = s[0];
        if (kAbs) sa[el][slot] = sb[0];
    }
    __syncthreads();
    if constexpr (kSlots > 32) {
        for (int o = kSlots / 2; o >= 32; o >>= 1) {
            if (slot < o) {
                sh[el][slot] += sh[el][slot + o];
                if (kAbs) sa[el][slot] += sa[el][slot + o];
            }
            __syncthreads();
        }
    }
    // the last five levels by warp shuffles, a warp per element
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= kEl || (int)blockIdx.x * kEl + warp >= a.E) return;
    double vs = sh[warp][lane], va = kAbs ? sa[warp][lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        vs += __shfl_down_sync(0xffffffffu, vs, o);
        if (kAbs) va += __shfl_down_sync(0xffffffffu, va, o);
    }
    if (lane == 0) {
        const int x = blockIdx.x * kEl + warp;
        const double val = a.divide ? vs / (double)cnt : vs * a.inv2P;
        a.out_flat[(size_t)blockIdx.y * a.E + x] = val;
        if (kAbs) a.out_scale[x] = va * a.inv2P;
        if (a.hessian && a.out_full) {
            // x -> (row, col) of the upper triangle
            int r = 0, rem = x;
            while (rem >= a.n - r) { rem -= a.n - r; ++r; }
            const int c = r + rem;
            a.out_full[r * a.n + c] = val;
            a.out_full[c * a.n + r] = val;
        }
    }
}

template <int kEl, bool kStaged>
void launch_finalize_as(const FinalizeArgs& a, cudaStream_t s) {
    const dim3 grid((a.E + kEl - 1) / kEl, a.batches > 0 ? a.batches : 1);
    if (a.out_scale) launch_after(finalize_kernel<kEl, true, kStaged>, grid, dim3(kChunks), 0, s, a);
    else launch_after(finalize_kernel<kEl, false, kStaged>, grid, dim3(kChunks), 0, s, a);
}

}  // namespace

// np pairs per block: a.threads legs (16 pairs unless tuned), fewer where 48 KB
// do not hold their perturbations; a warp for each of the units that the
// block has, at most eight.
void launch_sample(const SampleArgs& a, int n_groups, int max_P, cudaStream_t s) {
    const int legs = (a.threads == 16 || a.threads == 64 || a.threads == 128) ? a.threads : 32;
    const size_t per_pair = 2 * (size_t)a.n * (sizeof(double) + sizeof(float));
    int np = legs / 2;
    while (np > 1 && np * per_pair > 40 * 1024) np /= 2;
    // launches bound by the FP64 rate: enough pairs that the Gaussian units, a lane
    // per two dims of a pair, fill their warps (16 pairs of an odd number of such
    // lanes leave half a warp idle).  131,072 renders, 16 and 32 pairs, us per estimate:
    // plain gradient of 1 dim 76.8, 71.7, aggregate of 9 dims 260, 244, of 13 324, 306.
    if (np == 16 && (((a.n + 1) / 2) & 1) && (int64_t)n_groups * max_P >= 32 * 8 * num_sms() && 32 * per_pair <= 40 * 1024)
        np = 32;
    // many dims: spread few pairs over the SMs
    while (np > 2 && a.n >= 16 && (int64_t)n_groups * ((max_P + np - 1) / np) < num_sms()) np /= 2;
    const int units = 2 * ((2 * np + 31) / 32) + (np * ((a.n + 1) / 2) + 31) / 32;
    const int T = units <= 4 ? 128 : kSampleThreads;
    dim3 grid((max_P + np - 1) / np, n_groups);
    launch_after(sample_kernel, grid, dim3(T), np * per_pair, s, a, make_lobes(a.sigma, a.Zg, a.Zd, a.Zo, a.n), np);
}

// Eight elements per block read whole sectors but give each thread eight times
// the rows: for many elements only (stage times in us, one / eight per block:
// 2,080 elements of 1,024 rows 22.5 / 16.4, 64 of 1,024 8.2 / 12.3, 64 of 16,384
// 22.5 / 41).  Staged where a row's weights are at most a sector and a chunk has
// rows to share (3 elements of 16,384 rows: 22.5 direct, 16.4 staged; 6 of
// 8,192: 14.3, 10.2).
void launch_finalize(const FinalizeArgs& a, cudaStream_t s) {
    const int chunk = (a.pairs2 + kChunks - 1) / kChunks;
    if (a.E >= 1024 && !a.elementwise) launch_finalize_as<8, false>(a, s);
    else if (a.E <= 8 && chunk > 4) launch_finalize_as<1, true>(a, s);
    else launch_finalize_as<1, false>(a, s);
}

}  // namespace hr
