// K2: hard-edged disc renderer fused with the L2 loss (stand-in for the Box2
// plateau task, Sec. 4.1).  One warp renders one perturbation: pixel centre
// ((x + 1/2)/W, (y + 1/2)/H) is inside when fma(dx, dx, dy*dy) < r*r in FP32,
// value 1 inside, 0 outside.  With a 0/1 target every (v - t)^2 is 0 or 1 and
// the FP32 sum is an exact integer count.
#include "disc_device.cuh"
#include "hr.h"
#include "hr_device.cuh"
#include "hr_internal.h"

namespace hr {
namespace {

template <int kW>
__global__ void __launch_bounds__(32 * kW) disc_loss_kernel(RenderBatch b, int W, int H, float radius,
                                                            const float* __restrict__ target,
                                                            const float* __restrict__ centres, DiscBits tb) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m = blockIdx.x * kW + warp;
    let_next_start();
    wait_for_previous();
    if (m >= b.M) return;
    const Pert pt = resolve(b, m);
    const float cx = __fadd_rn(pt.theta[0], pt.tau[0]);
    const float cy = __fadd_rn(pt.theta[1], pt.tau[1]);
    const float loss = disc_loss_warp(target, tb, W, H, radius, centres, centres + W, cx, cy, lane);
    if (lane == 0) *pt.loss = loss;
}

// The same losses against a target that is not binary, for larger images: every
// pixel is visited, so the centres are read from shared memory, and the next
// kernel may start only when this one's work begins (let start at once, the next
// call's renders are placed while these run, unevenly over the SMs: 1,024 renders of
// 333x250 in 152 us instead of 93).  Aggregate Hessians in us, from the table in
// global memory and so: 333x250, 64 renders 179, 90; 1,024 204, 93; 16,384
// 1,173, 984; 512x512, 1,024 renders 355, 205.
template <int kW>
__global__ void __launch_bounds__(32 * kW) disc_grey_kernel(RenderBatch b, int W, int H, float radius,
                                                            const float* __restrict__ target) {
    __shared__ float s_px[HR_MAX_IMAGE_SIDE], s_py[HR_MAX_IMAGE_SIDE];
    centre_tables(s_px, s_py, W, H);
    __syncthreads();
    wait_for_previous();
    let_next_start();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m = blockIdx.x * kW + warp;
    if (m >= b.M) return;
    const Pert pt = resolve(b, m);
    const float cx = __fadd_rn(pt.theta[0], pt.tau[0]);
    const float cy = __fadd_rn(pt.theta[1], pt.tau[1]);
    const float loss = disc_loss_warp(target, DiscBits{}, W, H, radius, s_px, s_py, cx, cy, lane);
    if (lane == 0) *pt.loss = loss;
}

// Bit-packed target rows (bit x % 32 of word x / 32 of row y: pixel (x, y) is
// 1), found[0] raised by any pixel other than 0 or 1, found[1] counting the ones.
__global__ void disc_bits_kernel(const float* __restrict__ target, int W, int H, int words, uint32_t* bits,
                                 int* found) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words * H) return;
    const int y = i / words, j = i - y * words;
    uint32_t b = 0u;
    bool bad = false;
    for (int k = 0; k < 32 && 32 * j + k < W; ++k) {
        const float t = target[(size_t)y * W + 32 * j + k];
        if (t == 1.0f) b |= 1u << k;
        else if (t != 0.0f) bad = true;
    }
    bits[i] = b;
    if (bad) atomicOr(found, 1);
    if (b) atomicAdd(found + 1, __popc(b));
}

// Tables of a disc scene: the pixel centres (columns, then rows) and, a block
// per row, the target's ones by column, pre[y][x] in the first x pixels of row y.
__global__ void disc_tables_kernel(const uint32_t* __restrict__ bits, int W, int H, int words, uint16_t* pre,
                                   float* centres) {
    const int y = blockIdx.x;
    const uint32_t* row = bits + (size_t)y * words;
    for (int x = threadIdx.x; x <= W; x += blockDim.x) {
        int c = 0;
        for (int j = 0; j < (x >> 5); ++j) c += __popc(__ldg(row + j));
        if (x & 31) c += __popc(__ldg(row + (x >> 5)) & ((1u << (x & 31)) - 1u));
        pre[(size_t)y * (W + 1) + x] = (uint16_t)c;
    }
    if (y == 0)
        for (int i = threadIdx.x; i < W; i += blockDim.x) centres[i] = __fdiv_rn(__fadd_rn((float)i, 0.5f), (float)W);
    if (threadIdx.x == 0) centres[W + y] = __fdiv_rn(__fadd_rn((float)y, 0.5f), (float)H);
}

__global__ void disc_image_kernel(const float* params, int W, int H, float radius, float* img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= W * H) return;
    const int y = i / W, x = i - y * W;
    img[i] = disc_value(x, y, W, H, params[0], params[1], __fmul_rn(radius, radius));
}

// Squares (Box2 / Box10): K axis-aligned squares of half-size h; a pixel
// centre is 1 when |px - cx| < h and |py - cy| < h for some square (FP32).
__device__ __forceinline__ float boxes_value(int x, int y, int W, int H, const float* c, int K, float h) {
    const float px = __fdiv_rn(__fadd_rn((float)x, 0.5f), (float)W);
    const float py = __fdiv_rn(__fadd_rn((float)y, 0.5f), (float)H);
    for (int k = 0; k < K; ++k)
        if (fabsf(__fsub_rn(px, c[2 * k])) < h && fabsf(__fsub_rn(py, c[2 * k + 1])) < h) return 1.0f;
    return 0.0f;
}

constexpr int kMaxBoxParams = 64;

template <int kW>
__global__ void __launch_bounds__(32 * kW) boxes_loss_kernel(RenderBatch b, int W, int H, float h,
                                                             const float* __restrict__ target, DiscBits tb) {
    __shared__ float s_c[kW][kMaxBoxParams];
    __shared__ int s_sp[kW][kMaxBoxParams];
    __shared__ float s_px[HR_MAX_IMAGE_SIDE], s_py[HR_MAX_IMAGE_SIDE];
    let_next_start();
    centre_tables(s_px, s_py, W, H);
    __syncthreads();
    wait_for_previous();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m = blockIdx.x * kW + warp;
    if (m >= b.M) return;
    const Pert pt = resolve(b, m);
    for (int d = lane; d < b.n; d += 32) s_c[warp][d] = __fadd_rn(pt.theta[d], pt.tau[d]);
    __syncwarp();
    const float loss = boxes_loss_warp(target, tb, W, H, h, s_px, s_py, s_c[warp], s_sp[warp], b.n / 2, lane);
    if (lane == 0) *pt.loss = loss;
}

__global__ void boxes_image_kernel(const float* params, int K, int W, int H, float h, float* img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= W * H) return;
    const int y = i / W, x = i - y * W;
    img[i] = boxes_value(x, y, W, H, params, K, h);
}

}  // namespace

// Launch-shape variants (autotuner): 8, 4 or 16 warps per CTA; one warp
// renders one perturbation in every shape, so the choice never changes a result.
void launch_boxes_loss(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    const DiscBits tb{sc.tbinary ? sc.tbits : nullptr, sc.tpre, sc.tones};
    switch (sc.render_variant) {
        case 1: launch_after(boxes_loss_kernel<4>, dim3((b.M + 3) / 4), dim3(128), 0, s, b, sc.W, sc.H, sc.radius, sc.target, tb); break;
        case 2: launch_after(boxes_loss_kernel<16>, dim3((b.M + 15) / 16), dim3(512), 0, s, b, sc.W, sc.H, sc.radius, sc.target, tb); break;
        default: launch_after(boxes_loss_kernel<8>, dim3((b.M + 7) / 8), dim3(256), 0, s, b, sc.W, sc.H, sc.radius, sc.target, tb); break;
    }
}

void launch_boxes_image(const DevScene& sc, const float* params, float* img, cudaStream_t s) {
    const int npx = sc.W * sc.H;
    boxes_image_kernel<<<(npx + 255) / 256, 256, 0, s>>>(params, sc.n / 2, sc.W, sc.H, sc.radius, img);
}

template <int kW>
void launch_disc_as(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    const dim3 grid((b.M + kW - 1) / kW), block(32 * kW);
    // up to 64x64 filling the shared tables takes what reading them saves (64x64, 64 / 1,024 /
    // 16,384 renders: 12.0 / 12.9 / 32.7 us from the table, 12.9 / 13.5 / 33.8 so; 80x80: 21.8 / 25.0 /
    // 102.6, 13.8 / 14.4 / 91.2)
    if (!sc.tbinary && sc.W * sc.H > 4096)
        launch_after(disc_grey_kernel<kW>, grid, block, 0, s, b, sc.W, sc.H, sc.radius, sc.target);
    else
        launch_after(disc_loss_kernel<kW>, grid, block, 0, s, b, sc.W, sc.H, sc.radius, sc.target, sc.centres,
                     DiscBits{sc.tbinary ? sc.tbits : nullptr, sc.tpre, sc.tones});
}

void launch_disc_loss(const DevScene& sc, const RenderBatch& b, cudaStream_t s) {
    switch (sc.render_variant) {
        case 1: launch_disc_as<4>(sc, b, s); break;
        case 2: launch_disc_as<16>(sc, b, s); break;
        default: launch_disc_as<8>(sc, b, s); break;
    }
}

// One allocation: packed bits | what the packing found | centres | ones by column.
cudaError_t disc_prepare_target(DevScene& sc, cudaStream_t s) {
    const int words = (sc.W + 31) / 32;
    const bool disc = sc.kind == HR_SCENE_DISC2D;
    const size_t n_bits = (size_t)words * sc.H, n_centres = disc ? (size_t)sc.W + sc.H : 0;
    const size_t n_pre = disc ? (size_t)sc.H * (sc.W + 1) : 0;
    cudaError_t e = cudaMalloc((void**)&sc.tbits, 4 * (n_bits + 2 + n_centres) + 2 * n_pre);
    if (e != cudaSuccess) return e;
    int* d_found = reinterpret_cast<int*>(sc.tbits + n_bits);
    e = cudaMemsetAsync(d_found, 0, 2 * sizeof(int), s);
    if (e == cudaSuccess)
        disc_bits_kernel<<<(words * sc.H + 255) / 256, 256, 0, s>>>(sc.target, sc.W, sc.H, words, sc.tbits, d_found);
    if (e == cudaSuccess && disc) {
        sc.centres = reinterpret_cast<float*>(d_found + 2);
        sc.tpre = reinterpret_cast<uint16_t*>(sc.centres + n_centres);
        disc_tables_kernel<<<sc.H, 128, 0, s>>>(sc.tbits, sc.W, sc.H, words, sc.tpre, sc.centres);
    }
    int found[2] = {1, 0};
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(found, d_found, sizeof(found), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    sc.tbinary = e == cudaSuccess && found[0] == 0;
    sc.tones = found[1];
    return e;
}

void launch_disc_image(const DevScene& sc, const float* params, float* img, cudaStream_t s) {
    const int npx = sc.W * sc.H;
    disc_image_kernel<<<(npx + 255) / 256, 256, 0, s>>>(params, sc.W, sc.H, sc.radius, img);
}

}  // namespace hr
