// Learned warm start for the variable-coefficient Poisson CG: a 4-layer,
// 32-channel, 3x3 (dilated) convolutional network mapping (log k, f) -> u,
// with hand-written forward, backward and Adam kernels.  Not in the paper;
// plain CG to the same tolerance still decides when every solve is done.
//
// Layers: conv(2->C) ReLU, conv(C->C) ReLU, conv(C->C) ReLU, conv(C->1);
// dilation per layer; zero padding.  Activations are stored in bf16 (or
// fp32), every product is accumulated in fp32, master weights are fp32.
// Backward through a layer: the input gradient is a direct convolution with
// the weights flipped and transposed, masked by the ReLU of the forward
// activation; the weight gradient accumulates, per block, over a strided set
// of pixel tiles in registers, and a last kernel adds the blocks' sums.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "internal.h"
#include "warmnet_tc.cuh"

using namespace perks;

namespace {

constexpr int kTile = 16;        // output pixels per block side
constexpr int kConvThreads = kTile * kTile;
constexpr int kMaxC = 32;

template <typename S> __device__ __forceinline__ float ld_f(const S *p) { return to_acc(*p); }
template <> __device__ __forceinline__ float ld_f<float>(const float *p) { return *p; }
template <typename S> __device__ __forceinline__ S st_f(float v) { return from_acc<S>(v); }
template <> __device__ __forceinline__ float st_f<float>(float v) { return v; }
// 16 bytes of a pixel's channels
template <typename S> struct alignas(16) VecC {
    static constexpr int N = 16 / sizeof(S);
    S v[N];
};

// Activations of the hidden layers are NHWC ([img][y][x][32]), so a pixel's
// channels are one 64- or 128-byte run; the two input channels and the output
// are planes.

// First layer, 2 -> 32 channels: one thread per pixel, all 32 outputs in
// registers, weights [ci][tap][co] in shared memory (read by broadcast).
// x1[p][co] = relu(bias[co] + sum_ci sum_tap w[co][ci][tap] x0[ci][p + off])
template <typename S>
__global__ void __launch_bounds__(256, 2) conv_first_kernel(const S *__restrict__ x0, const float *__restrict__ w,
                                                         const float *__restrict__ bias, S *__restrict__ x1, int nimg,
                                                         int H, int W, int dil) {
    __shared__ __align__(16) float s_w[18 * kMaxC];
    for (int e = threadIdx.x; e < 18 * kMaxC; e += blockDim.x) s_w[e] = w[(e % kMaxC) * 18 + e / kMaxC];
    __syncthreads();
    const long long plane = (long long)H * W, total = plane * nimg;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long img = i / plane;
        const int p = (int)(i - img * plane), y = p / W, x = p % W;
        float acc[kMaxC];
#pragma unroll
        for (int co = 0; co < kMaxC; ++co) acc[co] = bias[co];
#pragma unroll 1
        for (int ci = 0; ci < 2; ++ci) {
            const S *in = x0 + (img * 2 + ci) * plane;
#pragma unroll 3
            for (int tap = 0; tap < 9; ++tap) {
                const int yy = y + (tap / 3 - 1) * dil, xx = x + (tap % 3 - 1) * dil;
                const float v = yy >= 0 && yy < H && xx >= 0 && xx < W ? ld_f(in + (long long)yy * W + xx) : 0.f;
                const float *wr = s_w + (ci * 9 + tap) * kMaxC;
#pragma unroll
                for (int co = 0; co < kMaxC; ++co) acc[co] = fmaf(wr[co], v, acc[co]);
            }
        }
        VecC<S> *o = reinterpret_cast<VecC<S> *>(x1 + i * kMaxC);
#pragma unroll
        for (int c = 0; c < kMaxC / VecC<S>::N; ++c) {
            VecC<S> v;
#pragma unroll
            for (int j = 0; j < VecC<S>::N; ++j) v.v[j] = st_f<S>(fmaxf(acc[c * VecC<S>::N + j], 0.f));
            o[c] = v;
        }
    }
}

// Inner layer 32 -> 32 on the CUDA cores (fp32 storage, or bf16 with the
// tensor cores off): a 16 x 16 pixel tile with its halo in shared memory as
// [ci][y][x] (an odd pitch per channel, so a pixel's channels are stored
// without bank conflicts), one thread per pixel.
__host__ __device__ constexpr int conv_mid_pitch(int dil) { return ((kTile + 2 * dil) * (kTile + 2 * dil)) | 1; }
template <typename S>
__global__ void __launch_bounds__(kConvThreads) conv_mid_kernel(const S *__restrict__ in, const float *__restrict__ w,
                                                              const float *__restrict__ bias, S *__restrict__ out,
                                                              int H, int W, int dil, int tiles_x) {
    extern __shared__ __align__(16) float smem[];
    const int TW = kTile + 2 * dil;
    float *s_w = smem;                           // 32 * 9 * 32
    float *s_in = smem + kMaxC * 9 * kMaxC;      // 32 * pitch
    const int pitch = conv_mid_pitch(dil);
    const int tile = blockIdx.x, img = blockIdx.y;
    const int tx0 = (tile % tiles_x) * kTile, ty0 = (tile / tiles_x) * kTile;
    for (int e = threadIdx.x; e < kMaxC * 9 * kMaxC; e += blockDim.x) {
        const int co = e % kMaxC, tap = (e / kMaxC) % 9, ci = e / (9 * kMaxC);
        s_w[e] = w[(co * kMaxC + ci) * 9 + tap];
    }
    const S *inb = in + (long long)img * H * W * kMaxC;
    for (int e = threadIdx.x; e < kMaxC * TW * TW; e += blockDim.x) {
        const int ci = e % kMaxC, q = e / kMaxC, xx = q % TW, yy = q / TW;
        const int gx = tx0 + xx - dil, gy = ty0 + yy - dil;
        s_in[ci * pitch + q] =
            (gx >= 0 && gx < W && gy >= 0 && gy < H) ? ld_f(inb + ((long long)gy * W + gx) * kMaxC + ci) : 0.f;
    }
    __syncthreads();
    const int lx = threadIdx.x % kTile, ly = threadIdx.x / kTile;
    const int gx = tx0 + lx, gy = ty0 + ly;
    float acc[kMaxC];
#pragma unroll
    for (int co = 0; co < kMaxC; ++co) acc[co] = bias[co];
    for (int ci = 0; ci < kMaxC; ++ci) {
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const float v = s_in[ci * pitch + (ly + (tap / 3) * dil) * TW + lx + (tap % 3) * dil];
            const float *wr = s_w + (ci * 9 + tap) * kMaxC;
#pragma unroll
            for (int co = 0; co < kMaxC; ++co) acc[co] = fmaf(wr[co], v, acc[co]);
        }
    }
    if (gx < W && gy < H) {
        VecC<S> *o = reinterpret_cast<VecC<S> *>(out + (((long long)img * H + gy) * W + gx) * kMaxC);
#pragma unroll
        for (int c = 0; c < kMaxC / VecC<S>::N; ++c) {
            VecC<S> v;
#pragma unroll
            for (int j = 0; j < VecC<S>::N; ++j) v.v[j] = st_f<S>(fmaxf(acc[c * VecC<S>::N + j], 0.f));
            o[c] = v;
        }
    }
}

// Last layer, 32 -> 1: one thread per pixel, its nine taps' channels read as
// 16-byte vectors through L1 (8 channels of all taps at a time, so every
// output keeps one fma chain: channel by channel, tap by tap).  With the
// 32 x 32 pixel input window of 32 channels in shared memory (131 KB, one
// block of 256 threads per SM) the same sum took 1790 us for 256 images of
// 64^2; 81 us now.
template <typename S>
__global__ void __launch_bounds__(256) conv_last_kernel(const S *__restrict__ x3, const float *__restrict__ w,
                                                        const float *__restrict__ bias, float *__restrict__ out,
                                                        int nimg, int H, int W, int dil) {
    constexpr int N = VecC<S>::N;
    __shared__ float s_w[kMaxC * 9];
    for (int e = threadIdx.x; e < kMaxC * 9; e += blockDim.x) s_w[e] = w[e];
    __syncthreads();
    const long long plane = (long long)H * W, total = plane * nimg;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int p = (int)(i % plane), y = p / W, x = p % W;
        float acc = bias[0];
#pragma unroll 1
        for (int c = 0; c < kMaxC / N; ++c) {
            VecC<S> v[9];
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int dy = (tap / 3 - 1) * dil, dx = (tap % 3 - 1) * dil;
                const bool inside = y + dy >= 0 && y + dy < H && x + dx >= 0 && x + dx < W;
                if (inside) v[tap] = reinterpret_cast<const VecC<S> *>(x3 + (i + (long long)dy * W + dx) * kMaxC)[c];
                else v[tap] = VecC<S>{};
            }
#pragma unroll
            for (int j = 0; j < N; ++j)
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) acc = fmaf(s_w[(c * N + j) * 9 + tap], to_acc(v[tap].v[j]), acc);
        }
        out[i] = acc;
    }
}

// ------------------------------------------------------------------ backward
//
// Weight gradients: every block sums the pixels it visits in registers,
// writes its sums to its own row of `part` ([block][parameter]) and
// reduce_grad_kernel adds the rows in block order, so a gradient does not
// depend on the order of atomics.

// dg[p][ci] = (x3[p][ci] > 0) sum_tap w[ci][8 - tap] dy[p + off(tap)]   (last layer, 32 <- 1)
template <typename S>
__global__ void __launch_bounds__(256) dgrad_last_kernel(const float *__restrict__ dy, const float *__restrict__ w,
                                                         const S *__restrict__ act, float *__restrict__ dg, int nimg,
                                                         int H, int W, int dil) {
    __shared__ __align__(16) float s_w[9 * kMaxC];  // [tap][ci]
    for (int e = threadIdx.x; e < 9 * kMaxC; e += blockDim.x) s_w[e] = w[(e % kMaxC) * 9 + 8 - e / kMaxC];
    __syncthreads();
    // four threads per pixel, 8 channels each
    const long long plane = (long long)H * W, total = plane * nimg * 4;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long q = i >> 2;
        const int c0 = (int)(i & 3) * 8;
        const int p = (int)(q % plane), y = p / W, x = p % W;
        float acc[8] = {};
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const int oy = (tap / 3 - 1) * dil, ox = (tap % 3 - 1) * dil;
            const bool inside = y + oy >= 0 && y + oy < H && x + ox >= 0 && x + ox < W;
            const float v = inside ? dy[q + (long long)oy * W + ox] : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = fmaf(s_w[tap * kMaxC + c0 + j], v, acc[j]);
        }
        const S *m = act + q * kMaxC + c0;
        float4 *o = reinterpret_cast<float4 *>(dg + q * kMaxC + c0);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = ld_f(m + j) > 0.f ? acc[j] : 0.f;
        o[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        o[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
}

// dx[p][ci] = (act[p][ci] > 0) sum_tap sum_co w[co][ci][8 - tap] dy[p + off(tap)][co]   (32 <- 32)
//
// Bound: the fp32 pipe (9216 fma per pixel).  A block takes 16 x 16 pixels;
// a thread 4 pixels x 8 channels, so that 12 16-byte shared loads (4 of
// pixels, 8 of weights, all without bank conflicts: pixels are padded to 80
// bytes) feed 128 fma, as packed pairs of channels.  dy comes in two halves
// of 16 channels, which keeps three blocks per SM at the default dilations.
// One thread per pixel with all 32 outputs, 9 loads per 32 fma: 89 + 80 us
// for the two layers of 16 images of 64^2, 39 + 38 us now.
constexpr int kDgHalf = 16;                      // dy channels staged at a time
constexpr int kDgPitch = kDgHalf + 4;            // floats per staged pixel
template <typename S>
__global__ void __launch_bounds__(256) dgrad_mid_kernel(const float *__restrict__ dy, const float *__restrict__ w,
                                                        const S *__restrict__ act, float *__restrict__ dx, int H,
                                                        int W, int dil, int tiles_x) {
    extern __shared__ __align__(16) float smem[];
    const int TW = kTile + 2 * dil;
    float *s_w = smem;                            // [tap][co 16][ci 32]
    float *s_d = smem + 9 * kDgHalf * kMaxC;      // [TW * TW][kDgPitch]
    const int tile = blockIdx.x, img = blockIdx.y;
    const int tx0 = (tile % tiles_x) * kTile, ty0 = (tile / tiles_x) * kTile;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = (lane >> 3) * 8, l = lane & 7;  // channels c0..c0+7; pixels x = l, l + 8 of rows 2 warp, 2 warp + 1
    const float *dyb = dy + (long long)img * H * W * kMaxC;
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    for (int half = 0; half < 2; ++half) {
        __syncthreads();
        for (int e = threadIdx.x; e < kDgHalf * kMaxC * 9; e += blockDim.x) {
            const int tap = e % 9, ci = (e / 9) % kMaxC, co = e / (9 * kMaxC);
            s_w[((8 - tap) * kDgHalf + co) * kMaxC + ci] = w[half * kDgHalf * kMaxC * 9 + e];
        }
        for (int e = threadIdx.x; e < TW * TW * (kDgHalf / 4); e += blockDim.x) {
            const int c = e % (kDgHalf / 4), q = e / (kDgHalf / 4);
            const int gx = tx0 + q % TW - dil, gy = ty0 + q / TW - dil;
            const bool inside = gx >= 0 && gx < W && gy >= 0 && gy < H;
            cp_async16_or_zero(s_d + q * kDgPitch + c * 4,
                               inside ? dyb + ((long long)gy * W + gx) * kMaxC + half * kDgHalf + c * 4 : dyb, inside);
        }
        cp_async_wait_all();
        __syncthreads();
#pragma unroll 1
        for (int tap = 0; tap < 9; ++tap) {
            const float *pd = s_d + ((2 * warp + (tap / 3) * dil) * TW + l + (tap % 3) * dil) * kDgPitch;
            const float *pw = s_w + tap * kDgHalf * kMaxC + c0;
#pragma unroll
            for (int k = 0; k < kDgHalf; k += 4) {
                float4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    v[i] = *reinterpret_cast<const float4 *>(pd + ((i >> 1) * TW + (i & 1) * 8) * kDgPitch + k);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float4 wa = *reinterpret_cast<const float4 *>(pw + (k + u) * kMaxC);
                    const float4 wb = *reinterpret_cast<const float4 *>(pw + (k + u) * kMaxC + 4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float x = u == 0 ? v[i].x : u == 1 ? v[i].y : u == 2 ? v[i].z : v[i].w;
                        const float2 xx = make_float2(x, x);
                        acc[i][0] = __ffma2_rn(make_float2(wa.x, wa.y), xx, acc[i][0]);
                        acc[i][1] = __ffma2_rn(make_float2(wa.z, wa.w), xx, acc[i][1]);
                        acc[i][2] = __ffma2_rn(make_float2(wb.x, wb.y), xx, acc[i][2]);
                        acc[i][3] = __ffma2_rn(make_float2(wb.z, wb.w), xx, acc[i][3]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gx = tx0 + l + (i & 1) * 8, gy = ty0 + 2 * warp + (i >> 1);
        if (gx >= W || gy >= H) continue;
        const long long o = (((long long)img * H + gy) * W + gx) * kMaxC + c0;
        float v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) { v[2 * j] = acc[i][j].x; v[2 * j + 1] = acc[i][j].y; }
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = ld_f(act + o + j) > 0.f ? v[j] : 0.f;
        reinterpret_cast<float4 *>(dx + o)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4 *>(dx + o)[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}

// part[block][co][ci][tap] = sum over the block's pixels of dy[p][co] x[p + off(tap)][ci], and the bias sums
// (32 x 32 x 9).
//
// Bound: the fp32 pipe (9216 fma per pixel).  A thread owns 8 co x 4 ci x the
// 3 taps of one kernel row (96 sums, as packed pairs of co): 5 16-byte shared
// loads per pixel feed 96 fma.  A warp is the 4 x 8 grid of (co, ci) groups of
// one kernel row, three warps a pixel stream; a block runs two streams (even
// and odd rows of a 16 x 8 pixel tile), added at the end.  One thread per
// (ci, tap) with all 32 co, 9 loads per 32 fma, and 5.6 M atomics: 114 + 88 us
// for 16 images of 64^2, 48 + 48 us now.
constexpr int kWgX = 16, kWgY = 8, kWgThreads = 192;
template <typename S>
__global__ void __launch_bounds__(kWgThreads, 2) wgrad_mid_kernel(const S *__restrict__ x, const float *__restrict__ dy,
                                                                float *__restrict__ part, int nparams, int off_w,
                                                                int off_b, int nimg, int H, int W, int dil) {
    extern __shared__ __align__(16) float smem[];
    const int TX = kWgX + 2 * dil, TY = kWgY + 2 * dil;
    float *s_dy = smem;                            // [128][32]
    float *s_x = smem + kWgX * kWgY * kMaxC;       // [TX * TY][32]
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int ky = warp % 3, stream = warp / 3;
    const int co0 = (lane >> 3) * 8, ci0 = (lane & 7) * 4;
    float2 acc[4][4][3];                           // [co pair][ci][kx]
    float bacc[8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) acc[i][j][k] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 8; ++i) bacc[i] = 0.f;
    const int tiles_x = (W + kWgX - 1) / kWgX, tiles_y = (H + kWgY - 1) / kWgY;
    const long long tiles_img = (long long)tiles_x * tiles_y, jobs = tiles_img * nimg;
    for (long long job = blockIdx.x; job < jobs; job += gridDim.x) {
        const int img = (int)(job / tiles_img), tile = (int)(job % tiles_img);
        const int tx0 = (tile % tiles_x) * kWgX, ty0 = (tile / tiles_x) * kWgY;
        __syncthreads();
        const float *dyb = dy + (long long)img * H * W * kMaxC;
        for (int e = t; e < kWgX * kWgY * (kMaxC / 4); e += kWgThreads) {
            const int c = e % (kMaxC / 4), p = e / (kMaxC / 4);
            const int gx = tx0 + p % kWgX, gy = ty0 + p / kWgX;
            const bool inside = gx < W && gy < H;
            cp_async16_or_zero(s_dy + p * kMaxC + c * 4, inside ? dyb + ((long long)gy * W + gx) * kMaxC + c * 4 : dyb,
                               inside);
        }
        constexpr int N = VecC<S>::N;
        const S *xb = x + (long long)img * H * W * kMaxC;
#pragma unroll 4
        for (int e = t; e < TX * TY * (kMaxC / N); e += kWgThreads) {
            const int c = e % (kMaxC / N), q = e / (kMaxC / N);
            const int gx = tx0 + q % TX - dil, gy = ty0 + q / TX - dil;
            VecC<S> v{};
            if (gx >= 0 && gx < W && gy >= 0 && gy < H)
                v = *reinterpret_cast<const VecC<S> *>(xb + ((long long)gy * W + gx) * kMaxC + c * N);
            float *d = s_x + q * kMaxC + c * N;
#pragma unroll
            for (int j = 0; j < N; j += 4)
                *reinterpret_cast<float4 *>(d + j) =
                    make_float4(to_acc(v.v[j]), to_acc(v.v[j + 1]), to_acc(v.v[j + 2]), to_acc(v.v[j + 3]));
        }
        cp_async_wait_all();
        __syncthreads();
#pragma unroll 1
        for (int py = stream; py < kWgY; py += 2) {
            const float *pd = s_dy + py * kWgX * kMaxC + co0;
            const float *px = s_x + (py + ky * dil) * TX * kMaxC + ci0;
#pragma unroll 2
            for (int p = 0; p < kWgX; ++p) {
                const float4 da = *reinterpret_cast<const float4 *>(pd + p * kMaxC);
                const float4 db = *reinterpret_cast<const float4 *>(pd + p * kMaxC + 4);
                const float2 d[4] = {make_float2(da.x, da.y), make_float2(da.z, da.w), make_float2(db.x, db.y),
                                     make_float2(db.z, db.w)};
                if (ky == 0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) { bacc[2 * i] += d[i].x; bacc[2 * i + 1] += d[i].y; }
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float4 xv = *reinterpret_cast<const float4 *>(px + (p + k * dil) * kMaxC);
                    const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 xx = make_float2(xs[j], xs[j]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[i][j][k] = __ffma2_rn(d[i], xx, acc[i][j][k]);
                    }
                }
            }
        }
    }
    // the two streams' sums, through shared memory, into the block's row
    float *row = part + (long long)blockIdx.x * nparams;
    float *s_o = smem;                              // 96 threads x 104 sums
    __syncthreads();
    if (stream == 1) {
        float *o = s_o + (warp - 3) * 32 + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    o[(((i * 4 + j) * 3 + k) * 2 + 0) * 96] = acc[i][j][k].x;
                    o[(((i * 4 + j) * 3 + k) * 2 + 1) * 96] = acc[i][j][k].y;
                }
#pragma unroll
        for (int i = 0; i < 8; ++i) o[(96 + i) * 96] = bacc[i];
    }
    __syncthreads();
    if (stream == 0) {
        const float *o = s_o + warp * 32 + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int r = ((i * 4 + j) * 3 + k) * 2;
                    const int a = off_w + ((co0 + 2 * i) * kMaxC + ci0 + j) * 9 + ky * 3 + k;
                    row[a] = acc[i][j][k].x + o[r * 96];
                    row[a + kMaxC * 9] = acc[i][j][k].y + o[(r + 1) * 96];
                }
        if (ky == 0 && ci0 == 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) row[off_b + co0 + i] = bacc[i] + o[(96 + i) * 96];
        }
    }
}

// A block's sums over warps: v[i] of every lane added over the block's warps
// into row[at(i)] by warp 0 (n values per lane).
template <int N, class AT>
__device__ __forceinline__ void sum_over_warps(const float (&v)[N], float *s, float *row, AT &&at) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < N; ++i) s[(warp * N + i) * 32 + lane] = v[i];
    __syncthreads();
    for (int i = warp; i < N; i += nw) {
        float t = 0.f;
        for (int k = 0; k < nw; ++k) t += s[(k * N + i) * 32 + lane];
        const int a = at(i, lane);
        if (a >= 0) row[a] = t;
    }
}

// A warp's walk over the pixels q, q + step, ...: image and pixel
// within the image by additions, where q / plane and q % plane are 64-bit
// divisions of some hundred instructions each.
struct PixelWalk {
    long long q, step;
    int img, p, plane, dimg, dp;
    __device__ __forceinline__ PixelWalk(long long first, long long stride, long long plane_)
        : q(first), step(stride), img((int)(first / plane_)), p((int)(first % plane_)), plane((int)plane_),
          dimg((int)(stride / plane_)), dp((int)(stride % plane_)) {}
    __device__ __forceinline__ void next() {
        q += step;
        img += dimg;
        p += dp;
        if (p >= plane) {
            p -= plane;
            ++img;
        }
    }
};

// Pixels whose loads a warp of the first and last layers' weight gradients has
// in flight: their bound is the latency of a pixel's loads (16 images of 64^2:
// 27 us each with one pixel at a time and two 64-bit divisions per pixel, 14
// and 16 now).
constexpr int kWgAhead = 4;

// Last layer (32 -> 1): part[block][ci][tap] = sum_q dy[q - off(tap)] x3[q][ci]; a warp visits pixels, lane = ci,
// so every activation is read once.  The bias sum rides along.
template <typename S>
__global__ void __launch_bounds__(256) wgrad_last_kernel(const S *__restrict__ x3, const float *__restrict__ dy,
                                                         float *__restrict__ part, int nparams, int off_w, int off_b,
                                                         int nimg, int H, int W, int dil) {
    __shared__ float s[8 * 10 * 32];
    const int lane = threadIdx.x & 31;
    const long long plane = (long long)H * W, total = plane * nimg;
    float acc[10] = {};
    PixelWalk at((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5, ((long long)gridDim.x * blockDim.x) >> 5, plane);
    while (at.q < total) {
        float v[kWgAhead], d[kWgAhead][10];
#pragma unroll
        for (int u = 0; u < kWgAhead; ++u, at.next()) {
            const bool in = at.q < total;
            const int y = at.p / W, x = at.p % W;
            v[u] = in ? ld_f(x3 + at.q * kMaxC + lane) : 0.f;
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int oy = -(tap / 3 - 1) * dil, ox = -(tap % 3 - 1) * dil;
                const bool inside = in && y + oy >= 0 && y + oy < H && x + ox >= 0 && x + ox < W;
                d[u][tap] = inside ? dy[at.q + (long long)oy * W + ox] : 0.f;
            }
            d[u][9] = in ? dy[at.q] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kWgAhead; ++u) {
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) acc[tap] = fmaf(d[u][tap], v[u], acc[tap]);
            if (lane == 0) acc[9] += d[u][9];
        }
    }
    sum_over_warps(acc, s, part + (long long)blockIdx.x * nparams,
                   [&](int i, int l) { return i < 9 ? off_w + l * 9 + i : l == 0 ? off_b : -1; });
}

// First layer (2 -> 32): part[block][co][ci][tap] = sum_p dy[p][co] x0[ci][p + off(tap)]; lane = co.
template <typename S>
__global__ void __launch_bounds__(256) wgrad_first_kernel(const S *__restrict__ x0, const float *__restrict__ dy,
                                                          float *__restrict__ part, int nparams, int off_w, int off_b,
                                                          int nimg, int H, int W, int dil) {
    __shared__ float s[8 * 19 * 32];
    const int lane = threadIdx.x & 31;
    const long long plane = (long long)H * W, total = plane * nimg;
    float acc[19] = {};
    const int ci = lane / 9, oy = (lane % 9 / 3 - 1) * dil, ox = (lane % 3 - 1) * dil;  // lane's input (9 = 3 x 3 taps)
    PixelWalk at((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5, ((long long)gridDim.x * blockDim.x) >> 5, plane);
    while (at.q < total) {
        // lanes 0..17 load the 18 inputs of a pixel, shuffles hand them to every lane
        float d[kWgAhead], mine[kWgAhead];
#pragma unroll
        for (int u = 0; u < kWgAhead; ++u, at.next()) {
            const bool in = at.q < total;
            const int yy = at.p / W + oy, xx = at.p % W + ox;
            d[u] = in ? dy[at.q * kMaxC + lane] : 0.f;
            mine[u] = in && lane < 18 && yy >= 0 && yy < H && xx >= 0 && xx < W
                          ? ld_f(x0 + ((long long)at.img * 2 + ci) * plane + (long long)yy * W + xx) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kWgAhead; ++u) {
#pragma unroll
            for (int i = 0; i < 18; ++i) acc[i] = fmaf(d[u], __shfl_sync(0xffffffffu, mine[u], i), acc[i]);
            acc[18] += d[u];
        }
    }
    sum_over_warps(acc, s, part + (long long)blockIdx.x * nparams,
                   [&](int i, int l) { return i < 18 ? off_w + l * 18 + i : off_b + l; });
}

// grads[i] = sum of part[b][i] over blocks: 32 parameters per block, 8 slices of rows.
__global__ void __launch_bounds__(256) reduce_grad_kernel(const float *__restrict__ part, int nblocks, int nparams,
                                                          float *__restrict__ grads) {
    __shared__ float s[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float t = 0.f;
    if (i < nparams)
#pragma unroll 8
        for (int b = warp; b < nblocks; b += 8) t += part[(long long)b * nparams + i];
    s[warp][lane] = t;
    __syncthreads();
    if (warp == 0 && i < nparams) {
        float v = 0.f;
        for (int k = 0; k < 8; ++k) v += s[k][lane];
        grads[i] = v;
    }
}

// A column's share of a coarse cell's mean log: the product of the values'
// significands (each in [1, 2)), the sum of their exponents, and the
// logarithms of the values that are not normal positive numbers (0, subnormal,
// negative, infinite, NaN), which log itself answers.  The product is a 64-bit
// fixed-point number m 2^-63 2^e, multiplied by the integer units: eleven more
// bits than fp64 carries, without the FP64 pipe.  A factor takes up to one bit
// of m, which normalise() returns after eight of them, so a factor's
// truncation is at most 2^-55 of the product.
struct LogProd {
    unsigned long long m = 1ull << 63;
    double s = 0.0;
    int e = 0;
    __device__ __forceinline__ void mul_significand(unsigned long long sig) {  // sig 2^-63 in [1, 2)
        m = __umul64hi(m, sig);
        e += 1;
    }
    __device__ __forceinline__ void mul(double v) {
        const int hi = __double2hiint(v);
        if ((unsigned)(hi - 0x00100000) < 0x7fe00000u) {
            e += (hi >> 20) - 1023;
            mul_significand(((unsigned long long)__double_as_longlong(v) << 11) | (1ull << 63));
        } else {
            s += log(v);
        }
    }
    __device__ __forceinline__ void normalise() {  // m back into [2^63, 2^64)
        const int n = __clzll((long long)m);
        m <<= n;
        e -= n;
    }
    // no value had a logarithm of its own and the product is within 2^-20 of 1, and not 1; m normalised
    __device__ __forceinline__ bool near_one() const {
        if (__double_as_longlong(s) != 0) return false;
        return e == 0 ? m >> 43 == 1ull << 20 && m != 1ull << 63 : e == -1 && m >> 43 == (1ull << 21) - 1;
    }
    // sum of the logarithms; m normalised
    __device__ __forceinline__ double value() const {
        const double d = __ull2double_rn(m);  // in [2^63, 2^64]
        const double x = __hiloint2double(__double2hiint(d) - (63 << 20), __double2loint(d));
        return fma((double)e, 0.69314718055994530942, log(x)) + s;
    }
};

// Sum of the logarithms of a coarse cell whose product is near 1: LogProd's
// error, 2^-47 at most whatever the sum, would no longer be small beside it
// (coefficients within 1e-9 of 1: 1e-7 of the mean at F = 2, 1e-12: 3e-3).
// Rare, and out of line.
__device__ __noinline__ double log_sum(const double *k, int nx, int F) {
    double s = 0.0;
    for (int dy = 0; dy < F; ++dy)
        for (int dx = 0; dx < F; ++dx) s += log(k[(long long)dy * nx + dx]);
    return s;
}

constexpr int kPoolThreads = 256;
constexpr int kPoolJobs = 8;  // jobs per round, at most

// Dynamic shared memory of a round of nj jobs: every column's sums.
size_t pool_smem(int nj, bool train) { return (size_t)nj * kPoolThreads * (3 * 8 + 4 + (train ? 8 : 0)); }

// Network input: channel 0 = log k, channel 1 = f, each averaged over the
// F x F fine cells of a coarse cell (F = 1: the cells themselves); with u also
// the training target ut, the mean of u over the same cells.
//
// Bound: HBM (16 or 24 B per fine cell) and the FP64 pipe (two operations per
// clock and SM: one addition per fine cell, some 50 per coarse cell), once the
// logarithms are out of the way: a coarse cell's mean log is one log of the
// product of its F^2 significands plus the exponents' sum times ln 2, and the
// product is the integer units'.  A job is a run of whole coarse cells of one
// coarse row: thread t reads fine column t of the F rows (coalesced, 16 loads
// in flight).  After a round of nj jobs one thread per coarse cell combines
// its F columns, so that all warps take part in the logarithms: an fp64
// instruction holds a quarter of the SM for 64 cycles, and with a round per job
// one warp's chain of them held up the other seven.  256 images of 512^2, F = 8:
// 4140 us with a log per fine cell, 548 with fp64 products, a load per use and
// warp 0 combining every job, 270 now (FP64 pipe 74 % busy).
template <typename S>
__global__ void __launch_bounds__(kPoolThreads, 3) features_kernel(const double *__restrict__ k,
                                                                  const double *__restrict__ f,
                                                                  const double *__restrict__ u, S *__restrict__ x0,
                                                                  double *__restrict__ ut, int ny, int nx, int F,
                                                                  int njobs, int nj) {
    extern __shared__ __align__(16) unsigned char pool_raw[];
    unsigned long long *s_m = reinterpret_cast<unsigned long long *>(pool_raw);
    double *s_s = reinterpret_cast<double *>(s_m + nj * kPoolThreads), *s_f = s_s + nj * kPoolThreads;
    double *s_u = s_f + nj * kPoolThreads;        // with u only
    int *s_e = reinterpret_cast<int *>(u ? s_u + nj * kPoolThreads : s_u);
    const int H = ny / F, W = nx / F;
    const long long plane = (long long)H * W;
    const double inv = 1.0 / ((double)F * F);
    const int cells = kPoolThreads / F;           // coarse cells per job
    const int nchunk = (W + cells - 1) / cells;
    const int t = threadIdx.x;
    for (int first = blockIdx.x * nj; first < njobs; first += gridDim.x * nj) {
        const int n = min(nj, njobs - first);
        for (int i = 0; i < n; ++i) {
            const int row = (first + i) / nchunk, X0 = (first + i) % nchunk * cells;  // row: img * H + Y
            if (t < min(cells, W - X0) * F) {
                const long long c0 = (long long)row * F * nx + (long long)X0 * F + t;
                LogProd lp;
                double ff = 0.0, uu = 0.0, kv = 0.0;
                for (int dy0 = 0; dy0 < F; dy0 += 8) {
                    double kr[8], fr[8];          // all eight rows' loads before the first is used
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (dy0 + j < F) {
                            kr[j] = k[c0 + (long long)(dy0 + j) * nx];
                            fr[j] = f[c0 + (long long)(dy0 + j) * nx];
                        }
                    kv = kr[0];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (dy0 + j < F) {
                            if (F > 1) lp.mul(kr[j]);
                            ff += fr[j];
                        }
                    lp.normalise();
                }
                if (u)
#pragma unroll 8
                    for (int dy = 0; dy < F; ++dy) uu += u[c0 + (long long)dy * nx];
                const int q = i * kPoolThreads + t;
                s_m[q] = lp.m;
                s_s[q] = F > 1 ? lp.s : kv;
                s_e[q] = lp.e;
                s_f[q] = ff;
                if (u) s_u[q] = uu;
            }
        }
        __syncthreads();
        for (int c = t; c < n * cells; c += kPoolThreads) {
            const int i = c / cells, cell = c % cells;
            const int row = (first + i) / nchunk, X = (first + i) % nchunk * cells + cell;
            if (X >= W) continue;
            const int q0 = i * kPoolThreads + cell * F;
            double lk, ff = 0.0, uu = 0.0;
            if (F == 1) {
                lk = log(s_s[q0]);
                ff = s_f[q0];
                if (u) uu = s_u[q0];
            } else {
                LogProd lp;
                for (int dx0 = 0; dx0 < F; dx0 += 8) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (dx0 + j < F) {
                            const int q = q0 + dx0 + j;
                            lp.mul_significand(s_m[q]);
                            lp.e += s_e[q];
                            if (__double_as_longlong(s_s[q]) != 0) lp.s += s_s[q];
                            ff += s_f[q];
                            if (u) uu += s_u[q];
                        }
                    lp.normalise();
                }
                if (lp.near_one()) lk = log_sum(k + (long long)row * F * nx + (long long)X * F, nx, F);
                else lk = lp.value();
            }
            const long long img = row / H, p = (long long)(row % H) * W + X;
            x0[(img * 2 + 0) * plane + p] = st_f<S>((float)(lk * inv));
            x0[(img * 2 + 1) * plane + p] = st_f<S>((float)(ff * inv));
            if (u) ut[img * plane + p] = uu * inv;
        }
        __syncthreads();
    }
}

constexpr int kUpThreads = 128;
constexpr int kUpRows = 64;  // fine rows per thread, about

// (double)x and isfinite(x) by the integer units: a conversion or comparison
// of doubles is an instruction of the FP64 pipe.
// The rare cases stay out of line: inlined they are evaluated for every value
// and one of the two results picked.
__device__ __noinline__ double widen_special(float x) { return (double)x; }
__device__ __noinline__ double two_weights(double w, double a, double b) { return (1.0 - w) * a + w * b; }
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
    if (e == 0u ? b << 1 != 0u : e == 0x7f800000u) return widen_special(x);  // subnormal, infinite, NaN
    return __hiloint2double((int)((b & 0x80000000u) | (e == 0u ? 0u : (b >> 3 & 0x0fffffffu) + 0x38000000u)),
                            (int)(b << 29));
}
__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// u = scale * bilinear interpolation of the coarse output at the fine cell
// centres (coarse cell centres at (Y + 1/2) F - 1/2, clamped at the edges).
//
// Bound: the FP64 pipe (HBM writes of 8 B per fine cell take half as long).  A thread owns V neighbouring fine
// columns and walks down a run of rows: the x-interpolation of a coarse row
// is done once for the F fine rows between two coarse centres, so a fine cell
// costs one fma and its share of the store instead of some 20 fp64 operations
// of index arithmetic and weights.  V = 2 (16-byte stores) where nx is even
// and u is 16-byte aligned, else 1; the two columns share the coarse cells'
// conversions and difference where they lie between the same centres.  256
// images of 512^2, F = 8: 6060 us, 325 with conversions, finiteness checks and
// the two-weight form on the FP64 pipe for every value and 2432 blocks walking
// 4096 runs in two uneven turns, 184 now (FP64 pipe 92 % busy, 1.6 operations
// per fine cell).
template <int V>
__global__ void __launch_bounds__(kUpThreads) upsample_kernel(const float *__restrict__ out, float scale, int ny,
                                                             int nx, int F, int nimg, double *__restrict__ u) {
    __shared__ double s_w[32];  // weight of the lower coarse row, i rows below the upper one's centre
    const int H = ny / F, W = nx / F;
    const int odd = F & 1;
    const double dscale = widen(scale);
    if (threadIdx.x < F) s_w[threadIdx.x] = (2.0 * threadIdx.x + (odd ? 0.0 : 1.0)) / (2.0 * F);
    __syncthreads();
    const int ncol = (nx + kUpThreads * V - 1) / (kUpThreads * V);
    const int nrun = (ny + kUpRows - 1) / kUpRows;
    const long long total = (long long)nimg * nrun * ncol;
    for (long long job = blockIdx.x; job < total; job += gridDim.x) {
        const int x = ((int)(job % ncol) * kUpThreads + threadIdx.x) * V;
        const int run = (int)(job / ncol % nrun);
        const long long img = job / ((long long)ncol * nrun);
        if (x >= nx) continue;
        const int ya = run * kUpRows, yb = min(ny, ya + kUpRows);
        // fine cell z lies between coarse centres j and j + 1, j = floor((z + 1/2) / F - 1/2) >= -1
        auto interval = [&](int z) { return (2 * z + 1 + F) / (2 * F) - 1; };
        auto first_of = [&](int j) { return ((2 * j + 1) * F) >> 1; };
        int xl[V], xr[V];
        double wx[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int j = interval(x + v);
            xl[v] = max(j, 0);
            xr[v] = min(j + 1, W - 1);
            wx[v] = j < 0 || j + 1 >= W ? 0.0 : s_w[x + v - first_of(j)];
        }
        const bool same = V > 1 && xl[0] == xl[V - 1] && xr[0] == xr[V - 1];
        const float *o = out + img * (long long)H * W;
        auto coarse_row = [&](int Y, double (&m)[V]) {
            const float *r = o + (long long)min(max(Y, 0), H - 1) * W;
            double a = widen(r[xl[0]]), b = widen(r[xr[0]]), df = b - a;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (v > 0 && !same) {
                    a = widen(r[xl[v]]);
                    b = widen(r[xr[v]]);
                    df = b - a;
                }
                double t;
                if (finite(df)) t = fma(wx[v], df, a);
                else t = two_weights(wx[v], a, b);  // a network that overflowed
                m[v] = t * dscale;
            }
        };
        int y = ya, j = interval(ya);
        double m0[V], m1[V];
        coarse_row(j, m0);
        double *up = u + (img * ny + ya) * (long long)nx + x;
        while (y < yb) {
            coarse_row(j + 1, m1);
            const int y1 = min(yb, first_of(j + 1));
            double d[V];
#pragma unroll
            for (int v = 0; v < V; ++v) d[v] = m1[v] - m0[v];
            int i = y - first_of(j);
            bool fin = true;
#pragma unroll
            for (int v = 0; v < V; ++v) fin = fin && finite(d[v]);
            if (!fin) {
                for (; y < y1; ++y, ++i) {
                    const double w = j < 0 || j + 1 >= H ? 0.0 : s_w[i];
#pragma unroll
                    for (int v = 0; v < V; ++v) up[v] = (1.0 - w) * m0[v] + w * m1[v];
                    up += nx;
                }
            }
            for (; y < y1; ++y, ++i) {
                const double w = s_w[i];
                if constexpr (V == 2) {
                    double2 r;
                    r.x = fma(w, d[0], m0[0]);
                    r.y = fma(w, d[1], m0[1]);
                    *reinterpret_cast<double2 *>(up) = r;
                } else {
                    *up = fma(w, d[0], m0[0]);
                }
                up += nx;
            }
#pragma unroll
            for (int v = 0; v < V; ++v) m0[v] = m1[v];
            ++j;
        }
    }
}

// dout = 2 (out - u/scale) / N; loss += (out - u/scale)^2 / N
__global__ void mse_kernel(const float *__restrict__ out, const double *__restrict__ u, float inv_scale,
                           long long n, float *dout, float *loss) {
    __shared__ float red[32];
    float s = 0.f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = out[i] - (float)u[i] * inv_scale;
        dout[i] = 2.f * d / (float)n;
        s = fmaf(d, d, s);
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
        v = warp_sum(v);
        if (threadIdx.x == 0) atomicAdd(loss, v / (float)n);
    }
}

// sum of u^2 over n values into *acc (fp64)
__global__ void sumsq_kernel(const double *__restrict__ u, long long n, double *acc) {
    __shared__ double red[32];
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s = fma(u[i], u[i], s);
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) atomicAdd(acc, v);
    }
}

__global__ void to_u_kernel(const float *__restrict__ out, float scale, long long n, double *u) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        u[i] = (double)out[i] * scale;
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

size_t conv_mid_smem(int dil) {
    return sizeof(float) * ((size_t)kMaxC * 9 * kMaxC + (size_t)kMaxC * conv_mid_pitch(dil));
}
size_t dgrad_mid_smem(int dil) {
    const int TW = kTile + 2 * dil;
    return sizeof(float) * ((size_t)9 * kDgHalf * kMaxC + (size_t)TW * TW * kDgPitch);
}
size_t wgrad_mid_smem(int dil) {  // operands, and the streams' sums afterwards
    const size_t ops = (size_t)kWgX * kWgY * kMaxC + (size_t)(kWgX + 2 * dil) * (kWgY + 2 * dil) * kMaxC;
    return sizeof(float) * std::max<size_t>(ops, 96 * 104);
}

template <typename K> perks_status set_smem(perks_context *ctx, K kernel, size_t bytes) {
    PERKS_CUDA(ctx, cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return PERKS_OK;
}

}  // namespace

struct perks_warmnet {
    perks_context *ctx = nullptr;
    int device = 0;  // for destroy, which may come after the context is gone
    int C = kMaxC;
    int dil[4] = {1, 2, 4, 8};
    int storage = PERKS_BF16;
    float out_scale = 1.f;
    int pool = 1;                // the network runs on the grid coarsened by this factor
    bool tensor_cores = true;    // bf16 storage: inner layers on tcgen05 (else CUDA cores)
    DevError *err = nullptr;
    double *ut = nullptr;        // pooled training target
    long long cap_ut = 0;
    int nparams = 0;
    int off_w[4], off_b[4];
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    long long adam_t = 0;
    float *loss = nullptr;
    // activations, sized for the largest batch seen
    long long cap_pixels = 0;   // nimg * H * W
    void *x0 = nullptr, *x1 = nullptr, *x2 = nullptr, *x3 = nullptr;
    float *outb = nullptr, *g0 = nullptr, *g1 = nullptr;
    float *part = nullptr;      // [2 x SMs][nparams] partial sums of the weight gradients
};

namespace {

void free_net_bufs(perks_warmnet *n) {
    void *p[] = {n->x0, n->x1, n->x2, n->x3, n->outb, n->g0, n->g1};
    for (void *q : p) if (q) cudaFree(q);
    n->x0 = n->x1 = n->x2 = n->x3 = nullptr;
    n->outb = n->g0 = n->g1 = nullptr;
    n->cap_pixels = 0;
}

perks_status ensure_bufs(perks_warmnet *n, long long pixels) {
    if (pixels <= n->cap_pixels) return PERKS_OK;
    free_net_bufs(n);
    const size_t es = n->storage == PERKS_BF16 ? 2 : 4;
    perks_context *ctx = n->ctx;
    PERKS_CUDA(ctx, cudaMalloc(&n->x0, pixels * 2 * es));
    PERKS_CUDA(ctx, cudaMalloc(&n->x1, pixels * n->C * es));
    PERKS_CUDA(ctx, cudaMalloc(&n->x2, pixels * n->C * es));
    PERKS_CUDA(ctx, cudaMalloc(&n->x3, pixels * n->C * es));
    PERKS_CUDA(ctx, cudaMalloc(&n->outb, pixels * sizeof(float)));
    PERKS_CUDA(ctx, cudaMalloc(&n->g0, pixels * n->C * sizeof(float)));
    PERKS_CUDA(ctx, cudaMalloc(&n->g1, pixels * n->C * sizeof(float)));
    n->cap_pixels = pixels;
    return PERKS_OK;
}

// Forward pass on nimg fine images of ny x nx cells: features pooled to the
// network grid H x W = (ny / pool) x (nx / pool), output left in outb.
template <typename S>
perks_status forward(perks_warmnet *n, int nimg, int ny, int nx, const double *k, const double *f, cudaStream_t s,
                     const double *u = nullptr) {
    perks_context *ctx = n->ctx;
    const int H = ny / n->pool, W = nx / n->pool;
    const int tx = (W + kTile - 1) / kTile, ty = (H + kTile - 1) / kTile;
    const long long pixels = (long long)nimg * H * W;
    const int pgrid = (int)std::min<long long>((pixels + 255) / 256, 16LL * ctx->sm_count);  // thread per pixel
    S *x0 = (S *)n->x0, *x1 = (S *)n->x1, *x2 = (S *)n->x2, *x3 = (S *)n->x3;
    const int cells = kPoolThreads / n->pool;
    // jobs of F fine rows: far below 2^31 for any k that fits in memory.  One round per block of three blocks per SM,
    // as long as that takes no more than kPoolJobs (16 images: rounds of 4 in two turns 44 us, of 5 in one 35)
    const int jobs = (int)((long long)nimg * H * ((W + cells - 1) / cells));
    const int nj = std::min(kPoolJobs, (jobs + 3 * ctx->sm_count - 1) / (3 * ctx->sm_count));
    const size_t fsm = pool_smem(nj, u != nullptr);
    perks_status frc = set_smem(ctx, features_kernel<S>, pool_smem(kPoolJobs, true));
    if (frc) return frc;
    features_kernel<S><<<std::min((jobs + nj - 1) / nj, 3 * ctx->sm_count), kPoolThreads, fsm, s>>>(
        k, f, u, x0, n->ut, ny, nx, n->pool, jobs, nj);
    const float *P = n->params;
    conv_first_kernel<S><<<pgrid, 256, 0, s>>>(x0, P + n->off_w[0], P + n->off_b[0], x1, nimg, H, W, n->dil[0]);
    if (std::is_same<S, __nv_bfloat16>::value && n->tensor_cores) {
        // inner layers as implicit GEMMs on the tensor cores
        const long long ntiles = (long long)nimg * ((W + kTcTX - 1) / kTcTX) * ((H + kTcTY - 1) / kTcTY);
        for (int l = 1; l <= 2; ++l) {
            const size_t sm = tc_conv_smem(n->dil[l]);
            perks_status rc = set_smem(ctx, tc_conv32_kernel, sm);
            if (rc) return rc;
            const int per_sm = std::max(1, std::min(3, (int)(ctx->smem_per_sm / (sm + 1024))));
            const int blocks = (int)std::min<long long>(ntiles, (long long)per_sm * ctx->sm_count);
            tc_conv32_kernel<<<blocks, kTcThreads, sm, s>>>(
                reinterpret_cast<const __nv_bfloat16 *>(l == 1 ? x1 : x2), P + n->off_w[l], P + n->off_b[l],
                reinterpret_cast<__nv_bfloat16 *>(l == 1 ? x2 : x3), nimg, H, W, n->dil[l], n->err);
        }
    } else {
        for (int l = 1; l <= 2; ++l) {
            const size_t sm = conv_mid_smem(n->dil[l]);
            perks_status rc = set_smem(ctx, conv_mid_kernel<S>, sm);
            if (rc) return rc;
            conv_mid_kernel<S><<<dim3(tx * ty, nimg), kConvThreads, sm, s>>>(
                l == 1 ? x1 : x2, P + n->off_w[l], P + n->off_b[l], l == 1 ? x2 : x3, H, W, n->dil[l], tx);
        }
    }
    conv_last_kernel<S><<<pgrid, 256, 0, s>>>(x3, P + n->off_w[3], P + n->off_b[3], n->outb, nimg, H, W, n->dil[3]);
    PERKS_CUDA(ctx, cudaGetLastError());
    return PERKS_OK;
}

template <typename S>
perks_status backward(perks_warmnet *n, int nimg, int H, int W, cudaStream_t s) {
    perks_context *ctx = n->ctx;
    const int tx = (W + kTile - 1) / kTile, ty = (H + kTile - 1) / kTile;
    const dim3 grid(tx * ty, nimg);
    const long long pixels = (long long)nimg * H * W;
    const int pgrid = (int)std::min<long long>((pixels * 4 + 255) / 256, 16LL * ctx->sm_count);
    // rows of partial sums: two blocks per SM, or one per tile where there are fewer
    const long long tiles = (long long)nimg * ((W + kWgX - 1) / kWgX) * ((H + kWgY - 1) / kWgY);
    const int nb = (int)std::min<long long>(tiles, 2LL * ctx->sm_count);
    if (!n->part) PERKS_CUDA(ctx, cudaMalloc(&n->part, sizeof(float) * 2 * ctx->sm_count * (size_t)n->nparams));
    S *x0 = (S *)n->x0, *x1 = (S *)n->x1, *x2 = (S *)n->x2, *x3 = (S *)n->x3;
    const float *P = n->params;
    float *part = n->part;
    const int np = n->nparams;
    // layer 4 (C -> 1): dy = outb-gradient in g1[0..pixels)
    float *dy4 = n->g1;
    wgrad_last_kernel<S><<<nb, 256, 0, s>>>(x3, dy4, part, np, n->off_w[3], n->off_b[3], nimg, H, W, n->dil[3]);
    dgrad_last_kernel<S><<<pgrid, 256, 0, s>>>(dy4, P + n->off_w[3], x3, n->g0, nimg, H, W, n->dil[3]);
    // layers 3 and 2 (C -> C)
    float *dy = n->g0, *dx = n->g1;
    for (int l = 2; l >= 1; --l) {
        S *xin = l == 2 ? x2 : x1;
        const size_t sm = wgrad_mid_smem(n->dil[l]), sd = dgrad_mid_smem(n->dil[l]);
        perks_status rc = set_smem(ctx, wgrad_mid_kernel<S>, sm);
        if (!rc) rc = set_smem(ctx, dgrad_mid_kernel<S>, sd);
        if (rc) return rc;
        wgrad_mid_kernel<S><<<nb, kWgThreads, sm, s>>>(xin, dy, part, np, n->off_w[l], n->off_b[l], nimg, H, W,
                                                       n->dil[l]);
        dgrad_mid_kernel<S><<<grid, 256, sd, s>>>(dy, P + n->off_w[l], xin, dx, H, W, n->dil[l], tx);
        float *t = dy; dy = dx; dx = t;
    }
    // layer 1 (2 -> C): weight gradient only
    wgrad_first_kernel<S><<<nb, 256, 0, s>>>(x0, dy, part, np, n->off_w[0], n->off_b[0], nimg, H, W, n->dil[0]);
    reduce_grad_kernel<<<(np + 31) / 32, 256, 0, s>>>(part, nb, np, n->grads);
    PERKS_CUDA(ctx, cudaGetLastError());
    return PERKS_OK;
}

// SplitMix64 -> normal (Box-Muller) for the He initialisation.
struct Rng {
    uint64_t s;
    uint64_t next() {
        uint64_t z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    }
    double uniform() { return (double)(next() >> 11) * (1.0 / 9007199254740992.0); }
    double normal() {
        const double u1 = std::max(uniform(), 1e-300), u2 = uniform();
        return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
    }
};

perks_status loss_and_grad(perks_warmnet *n, int nimg, int ny, int nx, const double *k, const double *f,
                           const double *u, cudaStream_t s) {
    perks_context *ctx = n->ctx;
    const int H = ny / n->pool, W = nx / n->pool;
    const long long pixels = (long long)nimg * H * W;
    perks_status rc = ensure_bufs(n, pixels);
    if (rc) return rc;
    const double *target = u;
    if (n->pool > 1) {
        if (pixels > n->cap_ut) {
            if (n->ut) cudaFree(n->ut);
            n->ut = nullptr;
            n->cap_ut = 0;
            PERKS_CUDA(ctx, cudaMalloc(&n->ut, sizeof(double) * pixels));
            n->cap_ut = pixels;
        }
        target = n->ut;
    }
    const double *pooled = n->pool > 1 ? u : nullptr;  // pooled into n->ut beside the features
    rc = n->storage == PERKS_BF16 ? forward<__nv_bfloat16>(n, nimg, ny, nx, k, f, s, pooled)
                                  : forward<float>(n, nimg, ny, nx, k, f, s, pooled);
    if (rc) return rc;
    PERKS_CUDA(ctx, cudaMemsetAsync(n->loss, 0, sizeof(float), s));
    mse_kernel<<<1024, 256, 0, s>>>(n->outb, target, 1.f / n->out_scale, pixels, n->g1, n->loss);
    PERKS_CUDA(ctx, cudaGetLastError());
    return n->storage == PERKS_BF16 ? backward<__nv_bfloat16>(n, nimg, H, W, s) : backward<float>(n, nimg, H, W, s);
}

}  // namespace

// ======================================================================= ABI

extern "C" perks_status perks_warmnet_create(perks_context *ctx, const int32_t *dilations, int32_t storage,
                                             uint64_t seed, perks_warmnet **out) {
    if (!ctx) return PERKS_ERR_INVALID_ARG;
    if (!out || (storage != PERKS_BF16 && storage != PERKS_F32))
        return fail(ctx, PERKS_ERR_INVALID_ARG, "warmnet_create: storage must be BF16 or F32");
    *out = nullptr;
    perks_status rc = use_device(ctx);
    if (rc) return rc;
    auto *n = new perks_warmnet();
    n->ctx = ctx;
    n->device = ctx->device;
    n->storage = storage;
    if (dilations)
        for (int l = 0; l < 4; ++l) {
            if (dilations[l] < 1 || dilations[l] > 16) { delete n; return fail(ctx, PERKS_ERR_INVALID_ARG, "warmnet_create: dilation in 1..16"); }
            n->dil[l] = dilations[l];
        }
    const int cins[4] = {2, n->C, n->C, n->C}, couts[4] = {n->C, n->C, n->C, 1};
    int o = 0;
    std::vector<float> h;
    Rng rng{seed};
    for (int l = 0; l < 4; ++l) {
        n->off_w[l] = o;
        const int nw = couts[l] * cins[l] * 9;
        const double sd = std::sqrt(2.0 / (cins[l] * 9.0));
        for (int i = 0; i < nw; ++i) h.push_back((float)(sd * rng.normal()));
        o += nw;
        n->off_b[l] = o;
        for (int i = 0; i < couts[l]; ++i) h.push_back(0.f);
        o += couts[l];
    }
    n->nparams = o;
    cudaError_t e = cudaMalloc(&n->params, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMalloc(&n->grads, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMalloc(&n->m, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMalloc(&n->v, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMalloc(&n->loss, sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->err, sizeof(DevError));
    if (e == cudaSuccess) e = cudaMemset(n->err, 0, sizeof(DevError));
    if (e == cudaSuccess) e = cudaMemcpy(n->params, h.data(), sizeof(float) * o, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, sizeof(float) * o);
    if (e != cudaSuccess) { perks_warmnet_destroy(n); return cuda_fail(ctx, e, "warmnet_create"); }
    *out = n;
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_destroy(perks_warmnet *n) {
    if (!n) return PERKS_OK;
    cudaSetDevice(n->device);
    free_net_bufs(n);
    void *p[] = {n->params, n->grads, n->m, n->v, n->loss, n->ut, n->err, n->part};
    for (void *q : p) if (q) cudaFree(q);
    delete n;
    return PERKS_OK;
}

extern "C" int32_t perks_warmnet_num_params(const perks_warmnet *n) { return n ? n->nparams : 0; }

extern "C" perks_status perks_warmnet_get_params(perks_warmnet *n, float *host) {
    if (!n || !host) return PERKS_ERR_INVALID_ARG;
    PERKS_CUDA(n->ctx, cudaMemcpy(host, n->params, sizeof(float) * n->nparams, cudaMemcpyDeviceToHost));
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_set_params(perks_warmnet *n, const float *host) {
    if (!n || !host) return PERKS_ERR_INVALID_ARG;
    PERKS_CUDA(n->ctx, cudaMemcpy(n->params, host, sizeof(float) * n->nparams, cudaMemcpyHostToDevice));
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_set_scale(perks_warmnet *n, float out_scale) {
    if (!n || !(out_scale > 0.f)) return PERKS_ERR_INVALID_ARG;
    n->out_scale = out_scale;
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_predict(perks_warmnet *n, int32_t nimg, int32_t ny, int32_t nx, const double *k,
                                              const double *f, double *u, perks_stream stream) {
    if (!n) return PERKS_ERR_INVALID_ARG;
    if (nimg < 1 || ny < 1 || nx < 1 || !k || !f || !u) return fail(n->ctx, PERKS_ERR_INVALID_ARG, "warmnet_predict: bad arguments");
    perks_status rc = use_device(n->ctx);
    if (rc) return rc;
    if (ny % n->pool || nx % n->pool)
        return fail(n->ctx, PERKS_ERR_INVALID_ARG, "warmnet_predict: grid not divisible by the pool factor %d", n->pool);
    cudaStream_t s = (cudaStream_t)stream;
    const long long pixels = (long long)nimg * (ny / n->pool) * (nx / n->pool);
    rc = ensure_bufs(n, pixels);
    if (rc) return rc;
    rc = n->storage == PERKS_BF16 ? forward<__nv_bfloat16>(n, nimg, ny, nx, k, f, s) : forward<float>(n, nimg, ny, nx, k, f, s);
    if (rc) return rc;
    if (n->pool == 1) to_u_kernel<<<1024, 256, 0, s>>>(n->outb, n->out_scale, pixels, u);
    else {
        const bool pairs = nx % 2 == 0 && (reinterpret_cast<uintptr_t>(u) & 15) == 0;
        const int V = pairs ? 2 : 1;
        const long long jobs = (long long)nimg * ((ny + kUpRows - 1) / kUpRows) *
                               ((nx + kUpThreads * V - 1) / (kUpThreads * V));
        const int grid = (int)std::min<long long>(jobs, 1 << 30);
        if (pairs) upsample_kernel<2><<<grid, kUpThreads, 0, s>>>(n->outb, n->out_scale, ny, nx, n->pool, nimg, u);
        else upsample_kernel<1><<<grid, kUpThreads, 0, s>>>(n->outb, n->out_scale, ny, nx, n->pool, nimg, u);
    }
    PERKS_CUDA(n->ctx, cudaGetLastError());
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_gradient(perks_warmnet *n, int32_t nimg, int32_t ny, int32_t nx, const double *k,
                                               const double *f, const double *u, float *grad_host, float *loss_host,
                                               perks_stream stream) {
    if (!n) return PERKS_ERR_INVALID_ARG;
    if (nimg < 1 || ny < 1 || nx < 1 || !k || !f || !u || ny % n->pool || nx % n->pool)
        return fail(n->ctx, PERKS_ERR_INVALID_ARG, "warmnet_gradient: bad arguments");
    perks_status rc = use_device(n->ctx);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    rc = loss_and_grad(n, nimg, ny, nx, k, f, u, s);
    if (rc) return rc;
    PERKS_CUDA(n->ctx, cudaStreamSynchronize(s));
    {
        DevError de{};
        PERKS_CUDA(n->ctx, cudaMemcpy(&de, n->err, sizeof(de), cudaMemcpyDeviceToHost));
        if (de.code) return fail(n->ctx, de.code, "warmnet: a tensor-core wait timed out (block %d)", de.block);
    }
    if (grad_host) PERKS_CUDA(n->ctx, cudaMemcpy(grad_host, n->grads, sizeof(float) * n->nparams, cudaMemcpyDeviceToHost));
    if (loss_host) PERKS_CUDA(n->ctx, cudaMemcpy(loss_host, n->loss, sizeof(float), cudaMemcpyDeviceToHost));
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_train_step(perks_warmnet *n, int32_t nimg, int32_t ny, int32_t nx,
                                                 const double *k, const double *f, const double *u, float lr,
                                                 perks_stream stream, float *loss_host) {
    if (!n) return PERKS_ERR_INVALID_ARG;
    if (nimg < 1 || ny < 1 || nx < 1 || !k || !f || !u || !(lr > 0.f) || ny % n->pool || nx % n->pool)
        return fail(n->ctx, PERKS_ERR_INVALID_ARG, "warmnet_train_step: bad arguments");
    perks_status rc = use_device(n->ctx);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    rc = loss_and_grad(n, nimg, ny, nx, k, f, u, s);
    if (rc) return rc;
    ++n->adam_t;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)n->adam_t), c2 = 1.f - std::pow(b2, (float)n->adam_t);
    adam_kernel<<<(n->nparams + 255) / 256, 256, 0, s>>>(n->params, n->grads, n->m, n->v, n->nparams, lr, b1, b2,
                                                         1e-8f, c1, c2);
    PERKS_CUDA(n->ctx, cudaGetLastError());
    if (loss_host) {
        PERKS_CUDA(n->ctx, cudaMemcpyAsync(loss_host, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
        PERKS_CUDA(n->ctx, cudaStreamSynchronize(s));
    }
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_fit(perks_warmnet *n, int32_t nimg, int32_t ny, int32_t nx, const double *k,
                                          const double *f, const double *u, int32_t batch, int32_t epochs, float lr,
                                          int32_t auto_scale, uint64_t seed, perks_stream stream, float *epoch_loss) {
    if (!n) return PERKS_ERR_INVALID_ARG;
    perks_context *ctx = n->ctx;
    if (nimg < 1 || ny < 1 || nx < 1 || !k || !f || !u || batch < 1 || epochs < 0 || !(lr > 0.f) ||
        ny % n->pool || nx % n->pool)
        return fail(ctx, PERKS_ERR_INVALID_ARG, "warmnet_fit: bad arguments");
    perks_status rc = use_device(ctx);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const long long plane = (long long)ny * nx;
    if (auto_scale) {
        double *acc = nullptr;
        PERKS_CUDA(ctx, cudaMalloc(&acc, sizeof(double)));
        cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(double), s);
        if (e == cudaSuccess) {
            sumsq_kernel<<<1024, 256, 0, s>>>(u, plane * nimg, acc);
            e = cudaGetLastError();
        }
        double h = 0.0;
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, acc, sizeof(double), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        cudaFree(acc);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "warmnet_fit: scale");
        const double rms = std::sqrt(h / (double)(plane * nimg));
        n->out_scale = rms > 0.0 ? (float)rms : 1.f;
    }
    const int nb = (nimg + batch - 1) / batch;
    std::vector<int> order(nb);
    Rng rng{seed};
    const float b1 = 0.9f, b2 = 0.999f;
    for (int ep = 0; ep < epochs; ++ep) {
        for (int i = 0; i < nb; ++i) order[i] = i;
        for (int i = nb - 1; i > 0; --i) std::swap(order[i], order[(int)(rng.next() % (uint64_t)(i + 1))]);
        double sum = 0.0;
        for (int bi = 0; bi < nb; ++bi) {
            const int i0 = order[bi] * batch, m = std::min(batch, nimg - i0);
            const long long o = (long long)i0 * plane;
            rc = loss_and_grad(n, m, ny, nx, k + o, f + o, u + o, s);
            if (rc) return rc;
            ++n->adam_t;
            const float c1 = 1.f - std::pow(b1, (float)n->adam_t), c2 = 1.f - std::pow(b2, (float)n->adam_t);
            adam_kernel<<<(n->nparams + 255) / 256, 256, 0, s>>>(n->params, n->grads, n->m, n->v, n->nparams, lr, b1,
                                                                 b2, 1e-8f, c1, c2);
            PERKS_CUDA(ctx, cudaGetLastError());
            if (epoch_loss) {
                float l = 0.f;
                PERKS_CUDA(ctx, cudaMemcpyAsync(&l, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
                PERKS_CUDA(ctx, cudaStreamSynchronize(s));
                sum += (double)l * m;
            }
        }
        if (epoch_loss) epoch_loss[ep] = (float)(sum / nimg);
    }
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_set_tensor_cores(perks_warmnet *n, int32_t enable) {
    if (!n) return PERKS_ERR_INVALID_ARG;
    n->tensor_cores = enable != 0;
    return PERKS_OK;
}

extern "C" perks_status perks_warmnet_set_pool(perks_warmnet *n, int32_t factor) {
    if (!n) return PERKS_ERR_INVALID_ARG;
    if (factor < 1 || factor > 32) return fail(n->ctx, PERKS_ERR_INVALID_ARG, "warmnet_set_pool: factor in 1..32");
    n->pool = factor;
    return PERKS_OK;
}

extern "C" float perks_warmnet_get_scale(const perks_warmnet *n) { return n ? n->out_scale : 0.f; }
