// Photometric loss of Sec. 4 (Eq. energy) on the smoothed render ("Variance
// Reduction": 3x3 Gaussian, sigma 1): blurred = G * image (replicate border),
// loss = sum |blurred - target| reduced in FP64, and its adjoint
// dloss/dimage = G^T * sign(blurred - target) by gather (no atomics).
// Batched over images through blockIdx.y; arguments travel by value.
//
// The loss sum does not depend on how blocks are scheduled: block b of an
// image always sums the same tiles (tiles b, b + the image's fixed number of
// blocks, ...) in the same order, writes its FP64 partial to its own slot, and
// a block of the second launch adds the partials in block order and stores the
// result.  Repeated calls therefore give bitwise the same loss.
//
// Two launches: the first blurs, compares and sums; the second takes the
// adjoint and the finishing sum.  (They are not one kernel: adj may be the
// image's or the target's own buffer, which the first launch reads.)  Bound by
// launch and load latency at the sizes in use (12.6 MB at 512 x 512, 2 us of
// HBM).  A thread takes a pixel, so its row, column and clamped neighbours are
// found once for three channels, and an interior pixel's adjoint is nine known
// taps; with a thread per channel, divisions by 3 and W, and the adjoint's
// search over 25 pixels x 9 offsets, and the finishing sum a third launch, the
// loss at 512 x 512 took 43 us of GPU time: now 19 us.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int TILE_W = 32, TILE_H = 8, LOSS_THREADS = TILE_W * TILE_H;

FR_D float gw(int dx, int dy) {
    const float e1 = expf(-0.5f), e2 = expf(-1.0f);
    const float z = 1.0f + 4.0f * e1 + 4.0f * e2;
    const int r2 = dx * dx + dy * dy;
    return (r2 == 0 ? 1.0f : (r2 == 1 ? e1 : e2)) / z;
}

FR_HD int loss_tiles(int H, int W) { return ((W + TILE_W - 1) / TILE_W) * ((H + TILE_H - 1) / TILE_H); }

FR_HD int loss_blocks(int H, int W) {
    const int nb = loss_tiles(H, W);
    return nb < FR_LOSS_PARTS ? nb : FR_LOSS_PARTS;
}

// This thread's pixel of tile t; false outside the image.
FR_D bool tile_pixel(int t, int H, int W, int& x, int& y) {
    const int across = (W + TILE_W - 1) / TILE_W;
    x = (t % across) * TILE_W + (threadIdx.x & (TILE_W - 1));
    y = (t / across) * TILE_H + (threadIdx.x / TILE_W);
    return x < W && y < H;
}

__global__ void __launch_bounds__(LOSS_THREADS) k_blur_loss(LossTable t) {
    __shared__ double part[LOSS_THREADS / 32];
    const LossItem& L = t.it[blockIdx.y];
    const int H = L.H, W = L.W, nb = loss_blocks(H, W);
    if ((int)blockIdx.x >= nb) return;                  // block-uniform
    double l = 0.0;
    for (int tile = blockIdx.x; tile < loss_tiles(H, W); tile += nb) {
        int x, y;
        if (!tile_pixel(tile, H, W, x, y)) continue;
        const int xs[3] = {max(x - 1, 0), x, min(x + 1, W - 1)}, ys[3] = {max(y - 1, 0), y, min(y + 1, H - 1)};
        float acc[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const float* q = L.image + 3 * ((size_t)ys[dy + 1] * W + xs[dx + 1]);
#pragma unroll
                for (int k = 0; k < 3; ++k) acc[k] += gw(dx, dy) * q[k];
            }
        const size_t i = 3 * ((size_t)y * W + x);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float r = acc[k] - L.target[i + k];
            l += fabs((double)r);
            L.sign[i + k] = (float)((r > 0.0f) - (r < 0.0f));
            if (L.blurred) L.blurred[i + k] = acc[k];
        }
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < LOSS_THREADS / 32; ++w) s += part[w];
        L.part[blockIdx.x] = s;
    }
}

// loss = sum of the image's block partials in block order (one block)
FR_D void loss_finish(const LossItem& L) {
    __shared__ double part[LOSS_THREADS];
    const int nb = loss_blocks(L.H, L.W);
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += LOSS_THREADS) s += L.part[b];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = LOSS_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *L.loss = part[0];
}

// Block 0 of an image finishes its loss, the others take its tiles:
// adj_q = sum over (p, delta) with clamp(p + delta) == q of w(delta) sgn_p,
// over p in row order, then over delta.
__global__ void __launch_bounds__(LOSS_THREADS) k_blur_adjoint(LossTable t) {
    const LossItem& L = t.it[blockIdx.y];
    if (blockIdx.x == 0) {
        loss_finish(L);
        return;
    }
    if (!L.adj) return;
    const int H = L.H, W = L.W;
    int qx, qy;
    if ((int)blockIdx.x - 1 >= loss_tiles(H, W) || !tile_pixel(blockIdx.x - 1, H, W, qx, qy)) return;
    float acc[3] = {0.0f, 0.0f, 0.0f};
    if (qx > 0 && qx < W - 1 && qy > 0 && qy < H - 1) {        // only p = q - delta
#pragma unroll
        for (int dy = 1; dy >= -1; --dy)
#pragma unroll
            for (int dx = 1; dx >= -1; --dx) {
                const float* g = L.sign + 3 * ((size_t)(qy - dy) * W + qx - dx);
#pragma unroll
                for (int k = 0; k < 3; ++k) acc[k] += gw(dx, dy) * g[k];
            }
    } else {
        for (int py = max(qy - 1, 0); py <= min(qy + 1, H - 1); ++py)
            for (int px = max(qx - 1, 0); px <= min(qx + 1, W - 1); ++px)
                for (int dy = -1; dy <= 1; ++dy) {
                    if (min(max(py + dy, 0), H - 1) != qy) continue;
                    for (int dx = -1; dx <= 1; ++dx) {
                        if (min(max(px + dx, 0), W - 1) != qx) continue;
                        for (int k = 0; k < 3; ++k) acc[k] += gw(dx, dy) * L.sign[3 * ((size_t)py * W + px) + k];
                    }
                }
    }
    for (int k = 0; k < 3; ++k) L.adj[3 * ((size_t)qy * W + qx) + k] = acc[k];
}

}  // namespace

void launch_loss(const LossTable& t, cudaStream_t st) {
    if (t.n <= 0) return;
    int blocks = 0, tiles = 0;
    for (int k = 0; k < t.n; ++k) {
        blocks = std::max(blocks, loss_blocks(t.it[k].H, t.it[k].W));
        if (t.it[k].adj) tiles = std::max(tiles, loss_tiles(t.it[k].H, t.it[k].W));
    }
    k_blur_loss<<<dim3(blocks, t.n), LOSS_THREADS, 0, st>>>(t);
    k_blur_adjoint<<<dim3(1 + tiles, t.n), LOSS_THREADS, 0, st>>>(t);
    fr_count_launches(2);
}

void launch_loss(int H, int W, const float* image, const float* target, double* loss, float* sign, double* part,
                 float* blurred, float* adj_image, cudaStream_t st) {
    LossTable t;
    t.n = 1;
    t.it[0] = LossItem{H, W, image, target, loss, sign, part, blurred, adj_image};
    launch_loss(t, st);
}
