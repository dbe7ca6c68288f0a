// Tensor-core (tcgen05) 3x3 convolution, 32 -> 32 channels, bf16 activations
// (NHWC), fp32 accumulation in tensor memory: the two inner layers of the
// warm-start network, as an implicit GEMM.
//
// A tile is 32 x 16 pixels of one image.  Its input, the tile and a halo of
// the dilation on every side, is staged once in shared memory by 16-byte
// asynchronous copies (zeros outside the image), split by channel chunk:
// chunk c (channels 8c..8c+7) of pixel q sits at c * CS + 16 q, q row-major
// over the halo'd tile.  That is the no-swizzle K-major core-matrix layout
// for any 8 neighbouring pixels of a row, so every tap's A operand is a view
// of the same bytes: an MMA covers 8 x 16 pixels (M = 128: eight pixels of a
// row are one core matrix, the next 8-row group of the operand is the next
// image row, stride offset = the halo'd row), the tap moves the start address
// by (dy * pitch + dx) * 16 bytes, and the leading offset (next channel
// chunk) is CS.  Per MMA tile 9 taps x two K = 16 steps accumulate into 32
// TMEM columns in that order; four MMA tiles share a staged tile.  The
// epilogue reads the accumulators back with tcgen05.ld, adds the bias,
// applies ReLU and stores bf16.
//
// Bound: the L2 -> shared-memory copies (64 B per halo pixel, 1.6 to 1.9 of
// them per output pixel at dilation 2 to 4).  Staging each tap's A operand by
// itself from NCHW planes (9 x 32 two-byte loads per pixel) took 212 us for
// 256 images of 64^2, 56 and 63 us now (dilation 2 and 4).
//
// Waits on the MMA-completion mbarrier are bounded; every exit path frees the
// TMEM it allocated.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace perks {

constexpr int kTcC = 32;                          // channels (MMA N and K)
constexpr int kTcTX = 32, kTcTY = 16;             // output pixels of a tile
constexpr int kTcSub = kTcTX / 8;                 // MMA tiles (8 x 16 pixels, M = 128) per tile
constexpr int kTcWBytes = kTcC * kTcC * 2;        // 2 KB: one tap's B operand
constexpr int kTcThreads = 256;
constexpr int kTcCols = kTcSub * kTcC;            // TMEM columns

__host__ __device__ constexpr int tc_halo_pixels(int dil) { return (kTcTX + 2 * dil) * (kTcTY + 2 * dil); }
__host__ __device__ constexpr size_t tc_conv_smem(int dil) {
    return (size_t)tc_halo_pixels(dil) * kTcC * 2 + 9 * (size_t)kTcWBytes + 16;
}

// Byte offset of element (row, k) of a B operand: no-swizzle K-major, K = 32,
// core matrix of rows 8i.. and channels 8j.. at (4 i + j) * 128.
__device__ __forceinline__ int tc_off(int row, int k) {
    return ((row >> 3) * 4 + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// Shared-memory operand descriptor: leading offset = next core matrix along
// K, stride offset = next 8-row group; no swizzle.
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t addr, uint32_t lead, uint32_t stride) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lead >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((stride >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;                           // descriptor version (tcgen05)
    return d;
}

// kind::f16 instruction descriptor: D fp32, A and B bf16, both K-major,
// N = 32, M = 128.
__host__ __device__ constexpr uint32_t tc_idesc() {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcC >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ bool tc_wait(unsigned long long *bar, unsigned parity, DevError *err) {
    const uint64_t t0 = global_timer_ns();
    for (;;) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (global_timer_ns() - t0 > 1000000000ull) {  // 1 s: the MMAs of one tile take microseconds
            if (err && atomicCAS(&err->code, 0, PERKS_ERR_BARRIER_TIMEOUT) == 0) err->block = blockIdx.x;
            return false;
        }
    }
}

// cp.async of 16 bytes, or of zeros
__device__ __forceinline__ void cp_async16_or_zero(void *smem_dst, const void *gmem_src, bool valid) {
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(smem_dst)), "l"(gmem_src), "r"(n)
                 : "memory");
}

// out[img][y][x][co] = relu(bias[co] + sum_{ci, tap} w[co][ci][tap] in[img][y + dy][x + dx][ci])
// for all images; w is the fp32 layer weight array [32][32][9].
__global__ void __launch_bounds__(kTcThreads) tc_conv32_kernel(const __nv_bfloat16 *__restrict__ in,
                                                             const float *__restrict__ w,
                                                             const float *__restrict__ bias,
                                                             __nv_bfloat16 *__restrict__ out, int nimg, int H, int W,
                                                             int dil, DevError *err) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int PX = kTcTX + 2 * dil, PY = kTcTY + 2 * dil, npx = PX * PY;
    const uint32_t CS = (uint32_t)npx * 16;                    // bytes between channel chunks
    unsigned char *sb = smem;                                  // 9 taps x 2 KB
    unsigned char *sa = smem + 9 * kTcWBytes;                  // 4 chunks x npx x 16 bytes
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(sa + 4 * (size_t)CS);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // B operands (weights) once per block, converted to bf16
#pragma unroll 4
    for (int e = tid; e < 9 * kTcC * kTcC; e += kTcThreads) {
        const int tap = e % 9, k = (e / 9) % kTcC, n = e / (9 * kTcC);
        *reinterpret_cast<__nv_bfloat16 *>(sb + tap * kTcWBytes + tc_off(n, k)) = __float2bfloat16_rn(w[e]);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    constexpr uint32_t idesc = tc_idesc();

    const int tiles_x = (W + kTcTX - 1) / kTcTX, tiles_y = (H + kTcTY - 1) / kTcTY;
    const long long tiles_img = (long long)tiles_x * tiles_y, ntiles = nimg * tiles_img;
    unsigned parity = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int img = (int)(t / tiles_img), tile = (int)(t % tiles_img);
        const int x0 = (tile % tiles_x) * kTcTX, y0 = (tile / tiles_x) * kTcTY;
        const __nv_bfloat16 *inb = in + (long long)img * H * W * kTcC;
        for (int e = tid; e < npx * 4; e += kTcThreads) {
            const int c = e & 3, q = e >> 2;
            const int y = y0 + q / PX - dil, x = x0 + q % PX - dil;
            const bool inside = x >= 0 && x < W && y >= 0 && y < H;
            cp_async16_or_zero(sa + c * CS + q * 16, inside ? inb + ((long long)y * W + x) * kTcC + c * 8 : inb, inside);
        }
        cp_async_wait_all();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (tid == 0) {
            for (int j = 0; j < kTcSub; ++j)
                for (int tap = 0; tap < 9; ++tap)
                    for (int ks = 0; ks < 2; ++ks) {
                        const uint32_t q = (uint32_t)((tap / 3) * dil * PX + (tap % 3) * dil + 8 * j);
                        const uint64_t ad = tc_smem_desc(smem_u32(sa) + 2 * ks * CS + q * 16, CS, (uint32_t)PX * 16);
                        const uint64_t bd = tc_smem_desc(smem_u32(sb + tap * kTcWBytes + ks * 256), 128, 512);
                        tc_mma(tmem + j * kTcC, ad, bd, idesc, tap + ks > 0);
                    }
            tc_commit(bar);
        }
        ok = tc_wait(bar, parity, err);
        parity ^= 1u;
        ok = __syncthreads_and(ok) != 0;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // warps 0-3 read MMA tiles 0 and 1, warps 4-7 tiles 2 and 3; TMEM lane = pixel of the MMA tile
        const int m = (warp & 3) * 32 + lane;
        for (int j = (warp >> 2) * 2; j < (warp >> 2) * 2 + 2; ++j) {
            uint32_t r[32];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                  "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                  "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                : "r"(tmem + j * kTcC + ((uint32_t)((warp & 3) * 32) << 16)));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int x = x0 + 8 * j + (m & 7), y = y0 + (m >> 3);
            if (x < W && y < H) {
                uint4 *o = reinterpret_cast<uint4 *>(out + (((long long)img * H + y) * W + x) * kTcC);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    __align__(16) __nv_bfloat162 v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int k = 8 * c + 2 * i;
                        v[i] = __floats2bfloat162_rn(fmaxf(__uint_as_float(r[k]) + bias[k], 0.f),
                                                     fmaxf(__uint_as_float(r[k + 1]) + bias[k + 1], 0.f));
                    }
                    o[c] = *reinterpret_cast<const uint4 *>(v);
                }
            }
        }
        // the next tile's operand stores and MMAs come after every thread's read of D
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTcCols) : "memory");
}

}  // namespace perks
