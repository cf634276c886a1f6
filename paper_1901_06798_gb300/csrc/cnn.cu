// cnn.cu -- the per-patch refinement-flag predictor: a learned stand-in for
// the b-cell flag buffer of Sec. 3.2 (regridding).  Three 3x3 convolutions of
// 16 channels with ReLU and a 1x1 head to one logit per cell, over the dense
// planes of a level (5 input features per cell), zero padding at the plane
// edge.  Forward in FP32 (training) or, for inference, one fused kernel on
// the tensor cores with FP16 activations and weights and FP32 accumulation;
// hand-written backward (binary cross-entropy
// with logits, averaged over masked cells) and Adam, all on the device.
//
// Flat parameter vector: for each layer, W (C_out, C_in, k, k) then b (C_out);
// layers (5->16, 3x3), (16->16, 3x3), (16->16, 3x3), (16->1, 1x1).
#include <algorithm>
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include "chain.cuh"
#include "cnn.h"

namespace tsu {

namespace {

constexpr int HID = kCnnHidden;

struct LayerSpec {
    int cin, cout, k, woff, boff;
};

__host__ __device__ inline LayerSpec layer_spec(int l)
{
    const int cin[4] = {kCnnIn, HID, HID, HID}, cout[4] = {HID, HID, HID, 1}, k[4] = {3, 3, 3, 1};
    int off = 0;
    for (int i = 0; i < l; i++) off += cout[i] * cin[i] * k[i] * k[i] + cout[i];
    LayerSpec s{cin[l], cout[l], k[l], off, off + cout[l] * cin[l] * k[l] * k[l]};
    return s;
}

// ---------------------------------------------------------------- FP32 layers
// The 3x3 layers forward, and backward to their inputs, are the same product: a
// sum over the channels and taps of a plane set, in that order.  Each output used
// to re-read its 9 CI inputs from L1 and one weight per multiply (39 us for 16 ->
// 16 on 4 x 128^2 cells); now a CTA of 256 threads stages an 8 x 32 tile of every
// input channel (and the layer's weights, output channel fastest) in shared
// memory, and a thread carries half of the sums of two neighbouring cells, so a
// 16-byte weight read serves eight multiplies, paired (__ffma2_rn) over output
// channels.  The order of every sum is the one before, so the values are too.
// Tiles of 256 cells: 4 x 128^2 cells are 256 CTAs, enough for every SM.
constexpr int kTy = 8, kTx = 32;                       // tile of a CTA
constexpr int kIy = kTy + 2, kIx = kTx + 2;            // its inputs

// a tile of CI planes with its margin, zero outside the plane; plane stride ps floats
template <int CI>
__device__ __forceinline__ void stage_tile(const float *x, float *s, int ps, int H, int W, int ty, int tx)
{
    const long long plane = (long long)H * W;
    for (int e = threadIdx.x; e < CI * kIy * kIx; e += blockDim.x) {
        const int c = e / (kIy * kIx), r = e - c * (kIy * kIx), i = r / kIx, j = r - i * kIx;
        const int yy = ty - 1 + i, xx = tx - 1 + j;
        s[c * ps + r] = yy >= 0 && yy < H && xx >= 0 && xx < W ? x[c * plane + (long long)yy * W + xx] : 0.0f;
    }
}

// BACK = false: y[o] = relu(b[o] + sum_c sum_tap w[o, c, tap] x[c, cell + tap]);
// BACK = true: y[c] = relu'(act[c]) sum_o sum_tap w[o, c, tap] x[o, cell - tap].
// CI planes in, CO planes out; wn, wi: the layer's own output and input channels.
// s: kConvSmem<CI, CO> floats, 16-byte aligned.
template <int CI, int CO> constexpr int kConvSmem = CI * kIy * kIx + CI * 9 * CO;
template <int CI, int CO, bool BACK>
__device__ __forceinline__ void conv3_tile(float *s, int tile, const float *x, const float *theta, int off_w, int off_b,
                                           const float *act, float *y, int H, int W, int tiles_x, int tiles_y)
{
    constexpr int PS = kIy * kIx;
    static_assert(CI * PS % 4 == 0, "the weights are read 16 bytes at a time");
    float *sx = s, *sw = s + CI * PS;
    const int img = tile / (tiles_x * tiles_y), tq = tile - img * (tiles_x * tiles_y);
    const int ty = (tq / tiles_x) * kTy, tx = (tq % tiles_x) * kTx;
    const long long plane = (long long)H * W;
    x += (long long)img * CI * plane;
    y += (long long)img * CO * plane;
    for (int e = threadIdx.x; e < CI * 9 * CO; e += 256) {
        const int o = e % CO, q = e / CO, tap = q % 9, c = q / 9;   // into [c][tap][o]
        sw[e] = theta[off_w + (BACK ? (c * CO + o) : (o * CI + c)) * 9 + tap];
    }
    stage_tile<CI>(x, sx, PS, H, W, ty, tx);
    __syncthreads();
    constexpr int CH = CO / 2;                                     // output channels of a thread
    const int oh = (threadIdx.x >> 7) * CH;                        // the first of them
    const int r = (threadIdx.x >> 4) & 7, c0 = 2 * (threadIdx.x & 15);   // cells (ty + r, tx + c0) and the next
    float2 acc[2][CH / 2];
#pragma unroll
    for (int o = 0; o < CH / 2; o++) {
        const float2 b = BACK ? make_float2(0.0f, 0.0f) : make_float2(theta[off_b + oh + 2 * o], theta[off_b + oh + 2 * o + 1]);
        acc[0][o] = b;
        acc[1][o] = b;
    }
#pragma unroll 1
    for (int c = 0; c < CI; c++) {
        float v[3][4];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const float2 *p = reinterpret_cast<const float2 *>(sx + c * PS + (r + i) * kIx + c0);
            const float2 a = p[0], b = p[1];
            v[i][0] = a.x; v[i][1] = a.y; v[i][2] = b.x; v[i][3] = b.y;
        }
#pragma unroll
        for (int tap = 0; tap < 9; tap++) {
            const int i = BACK ? 2 - tap / 3 : tap / 3, j = BACK ? 2 - tap % 3 : tap % 3;
            const float4 *w4 = reinterpret_cast<const float4 *>(sw + (c * 9 + tap) * CO + oh);
            const float2 v0 = make_float2(v[i][j], v[i][j]), v1 = make_float2(v[i][j + 1], v[i][j + 1]);
#pragma unroll
            for (int o = 0; o < CH / 4; o++) {
                const float4 w = w4[o];
                const float2 wa = make_float2(w.x, w.y), wb = make_float2(w.z, w.w);
                acc[0][2 * o] = __ffma2_rn(wa, v0, acc[0][2 * o]);
                acc[1][2 * o] = __ffma2_rn(wa, v1, acc[1][2 * o]);
                acc[0][2 * o + 1] = __ffma2_rn(wb, v0, acc[0][2 * o + 1]);
                acc[1][2 * o + 1] = __ffma2_rn(wb, v1, acc[1][2 * o + 1]);
            }
        }
    }
    const int yy = ty + r;
    if (yy >= H) return;
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int xx = tx + c0 + q;
        if (xx >= W) continue;
        const long long k = (long long)yy * W + xx;
        float v[CH], a[CH];   // (all loads before the first store: the compiler may not move one past the other)
#pragma unroll
        for (int o = 0; o < CH; o++) {
            v[o] = o & 1 ? acc[q][o / 2].y : acc[q][o / 2].x;
            a[o] = BACK ? act[((long long)img * CO + oh + o) * plane + k] : 0.0f;
        }
#pragma unroll
        for (int o = 0; o < CH; o++) y[(oh + o) * plane + k] = BACK ? (a[o] > 0.0f ? v[o] : 0.0f) : fmaxf(v[o], 0.0f);
    }
}

template <int CI, int CO>
__global__ void __launch_bounds__(256) conv3_kernel(const float *x, const float *theta, int off_w, int off_b, float *y, int H,
                                                    int W, int tiles_x, int tiles_y)
{
    __shared__ __align__(16) float s[kConvSmem<CI, CO>];
    chain_begin();
    conv3_tile<CI, CO, false>(s, blockIdx.x, x, theta, off_w, off_b, nullptr, y, H, W, tiles_x, tiles_y);
}

// The 1x1 head on its own (inference in FP32)
__global__ void head_kernel(const float *__restrict__ a3, const float *__restrict__ theta, int off_w, int off_b,
                            float *__restrict__ z, int n, long long plane)
{
    const long long total = (long long)n * plane;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < total; p += (long long)gridDim.x * blockDim.x) {
        const long long img = p / plane, k = p - img * plane;
        float v = theta[off_b];
#pragma unroll
        for (int c = 0; c < HID; c++) v = fmaf(theta[off_w + c], a3[(img * HID + c) * plane + k], v);
        z[p] = v;
    }
}

// The head, its loss and its backward pass in one pass over the last activations:
// the logit z, g = dL/dz = (sigmoid(z) - t) m / M and the loss, the head's weight
// and bias gradients, and dL/d(a3) times ReLU'.  As four kernels they read a3 three
// times, and the weight gradient alone took 381 us.  A CTA's sums go to its own place
// in part (weights, then the bias) and lpart (grad_sum_kernel adds them up).
__global__ void __launch_bounds__(128) head_loss_kernel(const float *a3, const float *theta, int off_w, int off_b,
                                                        const float *t, const float *m, long long total, long long plane, float inv_count, float *ga, float *part,
                                                        double *lpart)
{
    chain_begin();
    float w[HID], dw[HID], db = 0.0f;
    double ls = 0.0;
#pragma unroll
    for (int c = 0; c < HID; c++) { w[c] = theta[off_w + c]; dw[c] = 0.0f; }
    const float b = theta[off_b];
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < total; p += (long long)gridDim.x * blockDim.x) {
        const long long img = p / plane, k = p - img * plane, q = img * HID * plane + k;
        float a[HID], zz = b;
#pragma unroll
        for (int c = 0; c < HID; c++) { a[c] = a3[q + c * plane]; }
#pragma unroll
        for (int c = 0; c < HID; c++) zz = fmaf(w[c], a[c], zz);
        const float tt = t[p], mm = m[p];
        const float sg = 1.0f / (1.0f + __expf(-zz));
        const float g = (sg - tt) * mm * inv_count;
        const float l = fmaxf(zz, 0.0f) - zz * tt + log1pf(__expf(-fabsf(zz)));
        ls += (double)(l * mm);
        db += g;
#pragma unroll
        for (int c = 0; c < HID; c++) {
            dw[c] = fmaf(g, a[c], dw[c]);
            ga[q + c * plane] = a[c] > 0.0f ? w[c] * g : 0.0f;
        }
    }
    __shared__ float red[4][HID + 1];
    __shared__ double redl[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ls += __shfl_xor_sync(0xffffffffu, ls, o);
        db += __shfl_xor_sync(0xffffffffu, db, o);
#pragma unroll
        for (int c = 0; c < HID; c++) dw[c] += __shfl_xor_sync(0xffffffffu, dw[c], o);
    }
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < HID; c++) red[warp][c] = dw[c];
        red[warp][HID] = db;
        redl[warp] = ls;
    }
    __syncthreads();
    if (threadIdx.x <= HID)
        part[blockIdx.x * (HID + 1) + threadIdx.x] =
            (red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]);
    if (threadIdx.x == 32) lpart[blockIdx.x] = ((redl[0] + redl[1]) + (redl[2] + redl[3])) * (double)inv_count;
}

// Weight and bias gradients of a 3x3 layer: dW[o, c, tap] = sum over cells of g[o,
// cell] a[c, cell + tap], db[o] = sum of g[o].  One thread used to walk 1024 cells
// for each weight, dividing for every index (2.6 ms a 16 -> 16 layer on 4 x 128^2
// cells).  Now a CTA of 256 threads keeps a tile of both operands in shared memory
// (g with the channels together), and a thread owns one input channel and four
// output channels: their 36 sums stay in registers while a 3 x 3 window slides along
// units of 16 cells, 18 paired multiply-adds for one 16-byte and three 4-byte reads.
// The threads that are left over split the units.  A CTA's sums, over several tiles
// where there are more than kGradCtas, go to its own place in part (weights, then
// biases: the layer's slice of the parameter vector); grad_sum_kernel adds them up.
// CTA `block` of `blocks`; s: kGradSmem<CI> floats, 16-byte aligned.
template <int CI> constexpr int kGradSmem = kTy * kTx * HID + CI * (kIy * kIx + 1);
template <int CI>
__device__ __forceinline__ void wgrad3_tiles(float *s, int block, int blocks, const float *g, const float *a, int n, int H, int W, int tiles_x, int tiles_y,
                                             float *part)
{
    constexpr int PS = kIy * kIx + 1;          // odd: channels fall on different banks
    constexpr int NC = 4 * CI;                 // (channel, four outputs) pairs
    constexpr int SUB = 256 / NC;              // threads per pair
    constexpr int UNITS = kTy * kTx / 16;      // units of 16 cells of a row
    float *sg = s, *sa = s + kTy * kTx * HID;
    const long long plane = (long long)H * W;
    const int pair = threadIdx.x % NC, sub = threadIdx.x / NC;
    const int c = pair % CI, og = pair / CI;
    float2 acc[9][2], bs[2];
#pragma unroll
    for (int q = 0; q < 9; q++) { acc[q][0] = make_float2(0.0f, 0.0f); acc[q][1] = make_float2(0.0f, 0.0f); }
    bs[0] = make_float2(0.0f, 0.0f); bs[1] = make_float2(0.0f, 0.0f);
    const int ntile = n * tiles_x * tiles_y;
    for (int tile = block; tile < ntile; tile += blocks) {
        const int img = tile / (tiles_x * tiles_y), q = tile - img * (tiles_x * tiles_y);
        const int ty = (q / tiles_x) * kTy, tx = (q % tiles_x) * kTx;
        __syncthreads();   // the last tile has been used
        stage_tile<CI>(a + (long long)img * CI * plane, sa, PS, H, W, ty, tx);
        for (int e = threadIdx.x; e < kTy * kTx * HID; e += 256) {
            const int o = e / (kTy * kTx), r = e - o * (kTy * kTx), i = r / kTx, j = r - i * kTx;
            const int yy = ty + i, xx = tx + j;
            sg[r * HID + o] = yy < H && xx < W ? g[((long long)img * HID + o) * plane + (long long)yy * W + xx] : 0.0f;
        }
        __syncthreads();
        if (sub < SUB)
            for (int u = sub; u < UNITS; u += SUB) {
                const int i = u / (kTx / 16), j0 = (u % (kTx / 16)) * 16;
                const float *w0 = sa + c * PS + i * kIx + j0;
                const float4 *gp = reinterpret_cast<const float4 *>(sg + (i * kTx + j0) * HID) + og;
                float v[3][3];
#pragma unroll
                for (int d = 0; d < 3; d++) { v[d][1] = w0[d * kIx]; v[d][2] = w0[d * kIx + 1]; }
#pragma unroll 4
                for (int j = 0; j < 16; j++) {
#pragma unroll
                    for (int d = 0; d < 3; d++) { v[d][0] = v[d][1]; v[d][1] = v[d][2]; v[d][2] = w0[d * kIx + j + 2]; }
                    const float4 gg = gp[j * (HID / 4)];
                    const float2 g0 = make_float2(gg.x, gg.y), g1 = make_float2(gg.z, gg.w);
                    bs[0] = __fadd2_rn(bs[0], g0);
                    bs[1] = __fadd2_rn(bs[1], g1);
#pragma unroll
                    for (int t = 0; t < 9; t++) {
                        const float2 x = make_float2(v[t / 3][t % 3], v[t / 3][t % 3]);
                        acc[t][0] = __ffma2_rn(g0, x, acc[t][0]);
                        acc[t][1] = __ffma2_rn(g1, x, acc[t][1]);
                    }
                }
            }
    }
    // the sums of the threads of a pair, through the shared arrays
    __syncthreads();
    float *red = sg;   // [HID][CI][9] and the bias sums: fits in the g tile
    static_assert(HID * CI * 9 + HID <= kTy * kTx * HID, "the sums fit");
    for (int e = threadIdx.x; e < HID * CI * 9 + HID; e += 256) red[e] = 0.0f;
    for (int q = 0; q < SUB; q++) {
        __syncthreads();
        if (sub == q) {
#pragma unroll
            for (int t = 0; t < 9; t++) {
                float *d = red + ((4 * og) * CI + c) * 9 + t;
                d[0] += acc[t][0].x;
                d[CI * 9] += acc[t][0].y;
                d[2 * CI * 9] += acc[t][1].x;
                d[3 * CI * 9] += acc[t][1].y;
            }
            if (c == 0) {
                float *d = red + HID * CI * 9 + 4 * og;
                d[0] += bs[0].x; d[1] += bs[0].y; d[2] += bs[1].x; d[3] += bs[1].y;
            }
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < HID * CI * 9 + HID; e += 256) part[(long long)block * (HID * CI * 9 + HID) + e] = red[e];
}

template <int CI>
__global__ void __launch_bounds__(256) wgrad3_kernel(const float *g, const float *a, int n, int H, int W,
                                                     int tiles_x, int tiles_y, float *part)
{
    __shared__ __align__(16) float s[kGradSmem<CI>];
    chain_begin();
    wgrad3_tiles<CI>(s, blockIdx.x, gridDim.x, g, a, n, H, W, tiles_x, tiles_y, part);
}

// A hidden layer's backward pass in one launch: the first wb CTAs sum its weight
// gradients, the others form the gradient of its input.  Both only read g, and each
// alone leaves an SM waiting most of the time (1.7 CTAs of 8 warps an SM).  With the
// launches of the pass overlapping their starts (chain.cuh), the gradient of four
// 128^2 images takes 261 us where it took 270, the copies from the host included.
__global__ void __launch_bounds__(256) back3_kernel(const float *g, const float *a, const float *theta, int off_w,
                                                    float *gx, int n, int H, int W, int tiles_x, int tiles_y, float *part,
                                                    int wb)
{
    constexpr int S1 = kGradSmem<HID>, S2 = kConvSmem<HID, HID>;
    __shared__ __align__(16) float s[S1 > S2 ? S1 : S2];
    chain_begin();
    if ((int)blockIdx.x < wb) wgrad3_tiles<HID>(s, blockIdx.x, wb, g, a, n, H, W, tiles_x, tiles_y, part);
    else conv3_tile<HID, HID, true>(s, blockIdx.x - wb, g, theta, off_w, 0, a, gx, H, W, tiles_x, tiles_y);
}

// Where the CTAs of the backward pass leave their sums: count[l] slices of layer l's
// parameters in part[l], in CTA order, and count[3] parts of the loss.
struct GradParts {
    float *part[4];
    double *loss;
    int count[4];
};

// The gradient and the loss from the CTAs' sums.  A block takes 32 parameters, eight
// threads each; thread q adds the slices q, q + 8, ... in four interleaved chains, and
// the chains and threads are added as a tree.  The order is fixed and no sum is longer
// than 38 terms: by atomics, 256 to 512 additions one after another in the order of
// arrival, the gradient of 4 x 128^2 cells was off by 2.3e-7 to 2.7e-7 of its norm and
// differed from call to call; now it is off by 0.7e-7.  The whole call takes 258 us (266
// with the atomics and the two fills that cleared their results).
__global__ void __launch_bounds__(256) grad_sum_kernel(GradParts gp, float *grad, double *loss)
{
    chain_begin();
    __shared__ float red[8][32];
    __shared__ double redl[256];
    if (blockIdx.x + 1 == gridDim.x) {
        double v = 0.0;
        for (int b = threadIdx.x; b < gp.count[3]; b += 256) v += gp.loss[b];
        redl[threadIdx.x] = v;
        for (int o = 128; o > 0; o >>= 1) {
            __syncthreads();
            if (threadIdx.x < o) redl[threadIdx.x] += redl[threadIdx.x + o];
        }
        if (threadIdx.x == 0) *loss = redl[0];
        return;
    }
    const int k = blockIdx.x * 32 + (threadIdx.x & 31), q = threadIdx.x >> 5;
    int l = 0, end = 0, np = 0, off = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const LayerSpec S = layer_spec(i);
        end = S.boff + S.cout;
        if (k >= S.woff && k < end) { l = i; off = S.woff; np = end - S.woff; }
    }
    const bool in = k < end;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (in) {
        const float *p = gp.part[l] + (k - off);
        const int n = gp.count[l];
        int b = q;
        for (; b + 24 < n; b += 32) {
#pragma unroll
            for (int i = 0; i < 4; i++) acc[i] += p[(long long)(b + 8 * i) * np];
        }
#pragma unroll
        for (int i = 0; i < 3; i++)
            if (b + 8 * i < n) acc[i] += p[(long long)(b + 8 * i) * np];
    }
    red[q][threadIdx.x & 31] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    __syncthreads();
    if (threadIdx.x < 32 && in) {
        const int c = threadIdx.x;
        grad[k] = ((red[0][c] + red[1][c]) + (red[2][c] + red[3][c])) + ((red[4][c] + red[5][c]) + (red[6][c] + red[7][c]));
    }
}

__global__ void adam_kernel(float *theta, const float *grad, float *m, float *v, int np, float lr, float b1, float b2,
                            float eps, float c1, float c2)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < np; k += gridDim.x * blockDim.x) {
        float gk = grad[k];
        float mk = b1 * m[k] + (1.0f - b1) * gk;
        float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
        m[k] = mk;
        v[k] = vk;
        theta[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    }
}


int blocks_for(long long n, int threads)
{
    long long b = (n + threads - 1) / threads;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}

// ---------------------------------------------------------------- inference on tensor cores
// The FP16 inference path fused into one kernel.  A CTA produces the logits
// of a TH x TW tile of one plane; the tile's inputs and the two hidden
// activations it needs (the tile grown by 2 and by 1 cells) live in shared
// memory as FP16, channels last (24-half pixel stride: ldmatrix rows of 16
// bytes fall on distinct banks).  Each 3x3 layer is an implicit GEMM on the
// warp-level tensor-core MMA (m16n8k16, FP16 inputs, FP32 accumulation): an
// M-block is 16 consecutive pixels of the output region, K runs over the 9
// taps x 16 channels (the 5 input features padded with zeros), N = 16
// channels in two 8-wide blocks.  Activations outside the plane are zero, as
// zero padding of every layer's input requires.  The 1x1 head is a shuffle
// reduction of the last layer's accumulators.

namespace tc {
constexpr int TH = 16, TW = 32;            // output tile
constexpr int PS = 24;                     // halves per pixel in shared memory
constexpr int H0 = TH + 6, W0 = TW + 6;    // input region (3-cell margin)
constexpr int H1 = TH + 4, W1 = TW + 4;    // first hidden layer
constexpr int H2 = TH + 2, W2 = TW + 2;    // second hidden layer
constexpr int N0 = H0 * W0, N1 = H1 * W1, N2 = H2 * W2;
constexpr int NWARP = 4;
// per layer: 9 taps x 2 n-blocks x 32 lanes x 2 registers of packed FP16 weights
constexpr int WFRAG = 9 * 2 * 32 * 2;
constexpr int PACK = 3 * WFRAG + 3 * 16 + 32;   // words of the packed weights: fragments, biases, head and its bias
constexpr size_t smem_bytes()
{
    return (size_t)(N0 > N2 ? N0 : N2) * PS * 2 + (size_t)N1 * PS * 2 + (size_t)PACK * 4;
}
}  // namespace tc

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi)
{
    __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

// One 3x3 layer over an output region of ho x wo pixels (top-left at plane
// row gy, column gx) from an input region of (ho+2) x (wo+2) pixels.  LAST:
// apply the head and write logits instead of storing activations.
template <bool LAST>
__device__ __forceinline__ void tc_layer(const __half *in, int wi, __half *out, int ho, int wo, int gy, int gx, int H,
                                         int W, const uint32_t *wf, const float *bias, const float *whead, float bhead,
                                         float *logits)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    const int npx = ho * wo, nblk = (npx + 15) / 16;
    const uint32_t in_s = (uint32_t)__cvta_generic_to_shared(in);
    // ldmatrix row of this lane: matrix m = lane / 8 -> pixel rows 0-7 / 8-15, channel half 0 / 1
    const int m = lane >> 3, prow = (m & 1) * 8 + (lane & 7), chalf = (m >> 1) * 8;
    for (int blk = warp; blk < nblk; blk += tc::NWARP) {
        int p = blk * 16 + prow;
        p = p < npx ? p : npx - 1;
        const int r = p / wo, c = p - r * wo;
        float acc[2][4];
#pragma unroll
        for (int nb = 0; nb < 2; nb++) {
            const float b0 = bias[nb * 8 + 2 * t4], b1 = bias[nb * 8 + 2 * t4 + 1];
            acc[nb][0] = b0; acc[nb][1] = b1; acc[nb][2] = b0; acc[nb][3] = b1;
        }
#pragma unroll
        for (int tap = 0; tap < 9; tap++) {
            const int di = tap / 3, dj = tap % 3;
            const uint32_t addr = in_s + (uint32_t)(((r + di) * wi + (c + dj)) * tc::PS + chalf) * 2u;
            uint32_t a0, a1, a2, a3;
            ldsm_x4(addr, a0, a1, a2, a3);
#pragma unroll
            for (int nb = 0; nb < 2; nb++) {
                const uint32_t *f = wf + ((tap * 2 + nb) * 32 + lane) * 2;
                mma16816(acc[nb], a0, a1, a2, a3, f[0], f[1]);
            }
        }
        // rows g and g+8 of the block, channels nb*8 + 2*t4, +1
#pragma unroll
        for (int half = 0; half < 2; half++) {
            const int pp = blk * 16 + g + half * 8;
            if (pp >= npx) continue;
            const int rr = pp / wo, cc = pp - rr * wo;
            const int yy = gy + rr, xx = gx + cc;
            const bool inside = yy >= 0 && yy < H && xx >= 0 && xx < W;
            if (!LAST) {
#pragma unroll
                for (int nb = 0; nb < 2; nb++) {
                    const float v0 = inside ? fmaxf(acc[nb][2 * half], 0.0f) : 0.0f;
                    const float v1 = inside ? fmaxf(acc[nb][2 * half + 1], 0.0f) : 0.0f;
                    *reinterpret_cast<uint32_t *>(out + pp * tc::PS + nb * 8 + 2 * t4) = pack_half2(v0, v1);
                }
            }
        }
        if (LAST) {
            // head: activations rounded to FP16 as stored activations are, FP32 dot product
            float part[2] = {0.0f, 0.0f};
#pragma unroll
            for (int half = 0; half < 2; half++)
#pragma unroll
                for (int nb = 0; nb < 2; nb++)
#pragma unroll
                    for (int e = 0; e < 2; e++) {
                        const float v = __half2float(__float2half_rn(fmaxf(acc[nb][2 * half + e], 0.0f)));
                        part[half] = fmaf(whead[nb * 8 + 2 * t4 + e], v, part[half]);
                    }
#pragma unroll
            for (int half = 0; half < 2; half++) {
                part[half] += __shfl_xor_sync(0xffffffffu, part[half], 1);
                part[half] += __shfl_xor_sync(0xffffffffu, part[half], 2);
            }
            if (t4 == 0) {
#pragma unroll
                for (int half = 0; half < 2; half++) {
                    const int pp = blk * 16 + g + half * 8;
                    if (pp >= npx) continue;
                    const int rr = pp / wo, cc = pp - rr * wo;
                    const int yy = gy + rr, xx = gx + cc;
                    if (yy < H && xx < W) logits[(long long)yy * W + xx] = part[half] + bhead;
                }
            }
        }
    }
}

// The weights as the inference kernel's CTAs hold them: MMA fragments b0 =
// (W[o][2t][tap], W[o][2t+1][tap]), b1 = channels 2t+8, 2t+9, o = nb*8 + lane/4;
// biases; the head rounded to FP16 and its bias.  Packed once per call: every CTA
// gathering them from theta itself took longer than its three layers.
__global__ void cnn_pack_kernel(const float *__restrict__ theta, uint32_t *out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < 3 * 9 * 2 * 32) {
        const int l = e / (9 * 2 * 32), rem = e % (9 * 2 * 32);
        const int tap = rem / 64, nb = (rem / 32) % 2, ln = rem % 32;
        const LayerSpec S = layer_spec(l);
        const int o = nb * 8 + ln / 4, k0 = 2 * (ln % 4);
        float w[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int cch = k0 + (q & 1) + (q >> 1) * 8;
            w[q] = cch < S.cin ? theta[S.woff + (o * S.cin + cch) * 9 + tap] : 0.0f;
        }
        uint32_t *f = out + l * tc::WFRAG + ((tap * 2 + nb) * 32 + ln) * 2;
        f[0] = pack_half2(w[0], w[1]);
        f[1] = pack_half2(w[2], w[3]);
    }
    float *tail = reinterpret_cast<float *>(out + 3 * tc::WFRAG);
    if (e < 48) tail[e] = theta[layer_spec(e / 16).boff + e % 16];
    if (e < 32) {
        const LayerSpec S = layer_spec(3);
        tail[48 + e] = e < 16 ? __half2float(__float2half_rn(theta[S.woff + e])) : (e == 16 ? theta[S.boff] : 0.0f);
    }
}

__global__ void __launch_bounds__(tc::NWARP * 32) cnn_infer_tc_kernel(const uint32_t *__restrict__ packed,
                                                                      const float *__restrict__ x, int H, int W,
                                                                      float *__restrict__ logits)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __half *s0 = reinterpret_cast<__half *>(smem);                               // inputs, then layer 2
    __half *s1 = s0 + (size_t)(tc::N0 > tc::N2 ? tc::N0 : tc::N2) * tc::PS;      // layer 1
    uint32_t *wf = reinterpret_cast<uint32_t *>(s1 + (size_t)tc::N1 * tc::PS);    // packed weights
    const float *bias = reinterpret_cast<const float *>(wf + 3 * tc::WFRAG);     // 3 x 16
    const float *whead = bias + 48;                                               // 16, then its bias
    const int img = blockIdx.z;
    const int ty0 = blockIdx.y * tc::TH, tx0 = blockIdx.x * tc::TW;
    const long long plane = (long long)H * W;
    const float *xi = x + (long long)img * kCnnIn * plane;
    static_assert(tc::PACK % 4 == 0 && ((tc::N0 > tc::N2 ? tc::N0 : tc::N2) + tc::N1) * tc::PS % 8 == 0, "16-byte copies");
    for (int e = threadIdx.x; e < tc::PACK / 4; e += blockDim.x)
        reinterpret_cast<uint4 *>(wf)[e] = reinterpret_cast<const uint4 *>(packed)[e];
    // inputs of the 3-cell grown tile, FP16, zero outside the plane and in channels
    // 5..15; a cell's 16 channels are two 16-byte stores
    for (int p = threadIdx.x; p < tc::N0; p += blockDim.x) {
        const int r = p / tc::W0, c = p - r * tc::W0;
        const int yy = ty0 - 3 + r, xx = tx0 - 3 + c;
        float v[kCnnIn];
        const bool in = yy >= 0 && yy < H && xx >= 0 && xx < W;
#pragma unroll
        for (int ch = 0; ch < kCnnIn; ch++) v[ch] = in ? xi[(long long)ch * plane + (long long)yy * W + xx] : 0.0f;
        uint4 *d = reinterpret_cast<uint4 *>(s0 + p * tc::PS);
        d[0] = make_uint4(pack_half2(v[0], v[1]), pack_half2(v[2], v[3]), pack_half2(v[4], 0.0f), 0u);
        d[1] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    tc_layer<false>(s0, tc::W0, s1, tc::H1, tc::W1, ty0 - 2, tx0 - 2, H, W, wf, bias, nullptr, 0.0f, nullptr);
    __syncthreads();
    tc_layer<false>(s1, tc::W1, s0, tc::H2, tc::W2, ty0 - 1, tx0 - 1, H, W, wf + tc::WFRAG, bias + 16, nullptr, 0.0f,
                    nullptr);
    __syncthreads();
    tc_layer<true>(s0, tc::W2, nullptr, tc::TH, tc::TW, ty0, tx0, H, W, wf + 2 * tc::WFRAG, bias + 32, whead,
                   whead[16], logits + (long long)img * plane);
}

}  // namespace


int cnn_n_params()
{
    LayerSpec s = layer_spec(3);
    return s.boff + s.cout;
}

// CTAs that sum the weight gradients of a layer, and of the head: two an SM, eight an SM
constexpr int kGradCtas = 152 * 2, kHeadCtas = 152 * 8;
static long long layer_tiles(int n, int H, int W) { return (long long)n * ((W + kTx - 1) / kTx) * ((H + kTy - 1) / kTy); }

// The workspace of cnn_loss_grad: the activations a1..a3, two gradient plane sets, then
// the CTAs' sums.  Returns its floats (ws null: nothing else).
static size_t grad_workspace(int n, int H, int W, float *ws, GradParts &gp)
{
    const size_t px = (size_t)n * H * W;
    size_t o = px * (size_t)(3 * HID + 2 * HID);   // a multiple of 16 floats: the loss's doubles are aligned
    gp.count[3] = (int)std::min<size_t>((px + 127) / 128, kHeadCtas);
    gp.loss = ws ? reinterpret_cast<double *>(ws + o) : nullptr;
    o += 2 * (size_t)gp.count[3];
    for (int l = 0; l < 4; l++) {
        const LayerSpec S = layer_spec(l);
        if (l < 3) gp.count[l] = (int)std::min<long long>(layer_tiles(n, H, W), kGradCtas);
        gp.part[l] = ws ? ws + o : nullptr;
        o += (size_t)gp.count[l] * (S.boff + S.cout - S.woff);
    }
    return o;
}

size_t cnn_workspace_floats(int n, int H, int W)
{
    GradParts gp;
    return grad_workspace(n, H, W, nullptr, gp);
}

// the three hidden layers in FP32, activations a1, a2, a3 to act
static int hidden_forward(const float *theta, const float *x, int n, int H, int W, float *act, cudaStream_t st)
{
    const long long px = (long long)n * H * W;
    const LayerSpec L0 = layer_spec(0), L1 = layer_spec(1), L2 = layer_spec(2);
    const int txs = (W + kTx - 1) / kTx, tys = (H + kTy - 1) / kTy;
    const long long tiles = (long long)n * txs * tys;
    if (tiles > 0x7fffffffLL) return (int)cudaErrorInvalidValue;
    const unsigned grid = (unsigned)tiles;
    float *a1 = act, *a2 = act + px * HID, *a3 = act + 2 * px * HID;
    int e = launch_chained(conv3_kernel<kCnnIn, HID>, grid, 256, 0, st, x, theta, L0.woff, L0.boff, a1, H, W, txs, tys);
    if (e) return e;
    e = launch_chained(conv3_kernel<HID, HID>, grid, 256, 0, st, a1, theta, L1.woff, L1.boff, a2, H, W, txs, tys);
    if (e) return e;
    return launch_chained(conv3_kernel<HID, HID>, grid, 256, 0, st, a2, theta, L2.woff, L2.boff, a3, H, W, txs, tys);
}

int cnn_forward(const float *theta, const float *x, int n, int H, int W, bool fp16, float *act, float *logits,
                void *half_ws, cudaStream_t st)
{
    const long long px = (long long)n * H * W;
    if (!fp16) {
        const LayerSpec L3 = layer_spec(3);
        const int e = hidden_forward(theta, x, n, H, W, act, st);
        if (e) return e;
        head_kernel<<<blocks_for(px, 128), 128, 0, st>>>(act + 2 * px * HID, theta, L3.woff, L3.boff, logits, n, (long long)H * W);
    } else {
        // FP16 activations and weights, FP32 accumulation: one fused tensor-core kernel
        static bool configured = false;
        const size_t sm = tc::smem_bytes();
        if (!configured) {
            cudaError_t e = cudaFuncSetAttribute(cnn_infer_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
            if (e != cudaSuccess) return (int)e;
            configured = true;
        }
        dim3 grid((W + tc::TW - 1) / tc::TW, (H + tc::TH - 1) / tc::TH, n);
        uint32_t *packed = reinterpret_cast<uint32_t *>(half_ws);
        cnn_pack_kernel<<<(3 * 9 * 2 * 32 + 127) / 128, 128, 0, st>>>(theta, packed);
        cnn_infer_tc_kernel<<<grid, tc::NWARP * 32, sm, st>>>(packed, x, H, W, logits);
    }
    return (int)cudaGetLastError();
}

size_t cnn_half_workspace_bytes(int, int, int)
{
    return (size_t)tc::PACK * 4;   // the packed weights (activations stay in shared memory)
}

int cnn_loss_grad(const float *theta, const float *x, const float *t, const float *m, int n, int H, int W, float mcount,
                  float *ws, float *grad, double *loss, cudaStream_t st)
{
    const long long px = (long long)n * H * W;
    const long long plane = (long long)H * W;
    float *act = ws, *ga = ws + px * 3 * HID, *gb = ga + px * HID;
    const float *a1 = act, *a2 = act + px * HID, *a3 = act + 2 * px * HID;
    const LayerSpec L1 = layer_spec(1), L2 = layer_spec(2), L3 = layer_spec(3);
    GradParts gp;
    grad_workspace(n, H, W, ws, gp);
    const int e = hidden_forward(theta, x, n, H, W, act, st);
    if (e) return e;
    // head (1x1, 16 -> 1)
    int r = launch_chained(head_loss_kernel, gp.count[3], 128, 0, st, a3, theta, L3.woff, L3.boff, t, m, px, plane,
                           mcount > 0 ? 1.0f / mcount : 0.0f, ga, gp.part[3], gp.loss);
    if (r) return r;
    const int txs = (W + kTx - 1) / kTx, tys = (H + kTy - 1) / kTy;
    const int grid = n * txs * tys, wb = gp.count[0];   // hidden_forward has refused grids above 2^31 - 1
    if (grid > 0x7fffffff - wb) return (int)cudaErrorInvalidValue;
    // layer 3 (3x3, 16 -> 16): input a2
    r = launch_chained(back3_kernel, grid + wb, 256, 0, st, ga, a2, theta, L2.woff, gb, n, H, W, txs, tys, gp.part[2], wb);
    if (r) return r;
    // layer 2: input a1
    r = launch_chained(back3_kernel, grid + wb, 256, 0, st, gb, a1, theta, L1.woff, ga, n, H, W, txs, tys, gp.part[1], wb);
    if (r) return r;
    // layer 1: input x (no ReLU before it, no input gradient needed)
    r = launch_chained(wgrad3_kernel<kCnnIn>, wb, 256, 0, st, ga, x, n, H, W, txs, tys, gp.part[0]);
    if (r) return r;
    return launch_chained(grad_sum_kernel, (cnn_n_params() + 31) / 32 + 1, 256, 0, st, gp, grad, loss);
}

int cnn_adam(float *theta, const float *grad, float *m, float *v, int np, float lr, int t, cudaStream_t st)
{
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
    adam_kernel<<<blocks_for(np, 256), 256, 0, st>>>(theta, grad, m, v, np, lr, b1, b2, 1e-8f, c1, c2);
    return (int)cudaGetLastError();
}

}  // namespace tsu
