// Patch kernel for small 2-D domains: every block keeps its tile of the
// domain in shared memory for the whole run (Sec. 3: D_uncache = 0), together
// with a halo K steps deep.
//
// Between two exchanges a block advances K steps by itself: step s computes
// the tile and the (K - s) R cells around it that the remaining steps need,
// from one shared buffer into the other.  Then it writes the rim its
// neighbours read, K R cells deep, to the field in global memory (the two
// field buffers serve the exchanges in turn), raises its flag and waits for
// the flags of its eight neighbours only.  The neighbours' rim of exchange e
// is overwritten in exchange e + 2, and a block gets there only after its
// neighbours have raised flag e + 1, which they do after reading rim e.
//
// Why: in the resident-tile kernel, which exchanges halos after every step
// through a grid-wide barrier, a small domain's step is mostly that exchange:
// 2d5pt fp64 256^2 spends 0.5 us of the FP64 pipe per step of 3.9 us.  Here one
// exchange (a write, a flag and a read through L2, about 2.5 us) serves four
// steps, and a step takes 2.4 us (fp32 64^2: 1.0, 0.98 M cells of fp64 12): a
// quarter of it the exchange, a third the FP64 work with the recomputed rim,
// the rest short passes (some 780 cells for 512 threads) and a block barrier
// per step.  K = 4 for radius 1, 2 for radius 2: half of that was slower or
// equal at every size (256^2 fp64 2d5pt K = 2 3.4 us; 2d25pt K = 1 7.5 against
// 6.7).  Bound: latency for small tiles, the FP64 pipe and the recomputed rim
// for large fp64 ones.
//
// Cells add their terms in table order with one fma chain from 0 and are
// rounded to the storage type after every step (fp32 / bf16: the same bits as
// every other kernel); the buffers hold the accumulator type.
#pragma once

#include "stencil_vec.cuh"

namespace perks {

constexpr int kPatchThreads = 512;

struct PatchArgs {
    int X, Z;
    int ntx, nty;             // tiles
    int EW, EH;               // shared buffer: tile and halo, at most
    long long steps;
    double boundary;
    float boundary_f;
    double w[25];
    float wf[25];
    void *field[2];
    unsigned long long *flags;  // [tiles] exchanges a tile has published, zero before a launch
    DevError *err;
    long long timeout_ns;
};

using PatchFn = void (*)(PatchArgs);

struct PatchEntry {
    int dtype, shape;
    int k;                    // steps between exchanges
    PatchFn fn;
};

template <typename T, class SH, int K>
__global__ void __launch_bounds__(kPatchThreads, 1) perks_patch_kernel(const __grid_constant__ PatchArgs a) {
    using A = typename AccOf<T>::type;
    constexpr int R = SH::R, H = K * R, NT = kPatchThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    A *cur = reinterpret_cast<A *>(smem_raw), *nxt = cur + a.EW * a.EH;
    const int tid = threadIdx.x, EW = a.EW;
    const int ti = blockIdx.x % a.ntx, tj = blockIdx.x / a.ntx;
    int x0, tx, y0, ty;
    split_axis(a.X, a.ntx, ti, x0, tx);
    split_axis(a.Z, a.nty, tj, y0, ty);
    T bnd_t;
    if constexpr (std::is_same<T, double>::value) bnd_t = a.boundary;
    else bnd_t = from_acc<T>(a.boundary_f);
    const A bnd = to_acc(bnd_t);
    const int org = (H - y0) * EW + H - x0;           // cell (x, y) sits at org + y EW + x
    // the cells within g of the tile and inside the domain
    struct Box {
        int xa, ya, w, h;
    };
    auto box = [&](int g) {
        Box b;
        b.xa = max(x0 - g, 0);
        b.ya = max(y0 - g, 0);
        b.w = min(x0 + tx + g, a.X) - b.xa;
        b.h = min(y0 + ty + g, a.Z) - b.ya;
        return b;
    };
    // f(x, y) over the cells of b, NT at a time
    auto each = [&](const Box &b, auto &&f) {
        const int dj = NT / b.w, di = NT - dj * b.w;
        int j = tid / b.w, i = tid - j * b.w;
        for (; j < b.h;) {
            f(b.xa + i, b.ya + j);
            i += di;
            j += dj;
            if (i >= b.w) { i -= b.w; ++j; }
        }
    };
    for (int e = tid; e < 2 * EW * a.EH; e += NT) cur[e] = bnd;
    __syncthreads();
    each(box(H), [&](int x, int y) {
        cur[org + y * EW + x] = to_acc(__ldcg(static_cast<const T *>(a.field[0]) + (long long)y * a.X + x));
    });
    int n = 0;
    for (long long left = a.steps; left > 0; left -= K, ++n) {
        const int ns = (int)(left < K ? left : K);
        const bool last = left <= K;
        if (n > 0) {
            // the neighbours' rims, published n times
            int fail = 0;
            if (tid < 32) {
                const int ni = ti + tid % 3 - 1, nj = tj + tid / 3 - 1;
                const bool there = tid < 9 && tid != 4 && ni >= 0 && ni < a.ntx && nj >= 0 && nj < a.nty;
                const unsigned long long *flag = a.flags + (there ? nj * a.ntx + ni : 0);
                fail = !warp_wait([&]() { return !there || ld_relaxed_gpu_u64(flag) >= (unsigned long long)n; }, a.err,
                                  a.timeout_ns, n);
                fence_acquire_gpu();
            }
            if (__syncthreads_or(fail)) return;
            const T *in = static_cast<const T *>(a.field[n & 1]);
            // the halo as two runs: the rows above and below the tile, and the ends of its rows
            const Box b = box(ns * R);
            const int up = y0 - b.ya, down = b.ya + b.h - (y0 + ty);
            const int lf = x0 - b.xa, rt = b.xa + b.w - (x0 + tx);
            auto get = [&](int x, int y) { cur[org + y * EW + x] = to_acc(__ldcg(in + (long long)y * a.X + x)); };
            for (int e = tid; e < (up + down) * b.w; e += NT) {
                const int r = e / b.w;
                get(b.xa + e - r * b.w, r < up ? b.ya + r : y0 + ty + r - up);
            }
            const int ends = lf + rt;
            for (int e = tid; e < ends * ty; e += NT) {
                const int r = e / ends, c = e - r * ends;
                get(c < lf ? b.xa + c : x0 + tx + c - lf, y0 + r);
            }
        }
        __syncthreads();
        T *out = static_cast<T *>(a.field[(n & 1) ^ 1]);
        for (int s = 1; s <= ns; ++s) {
            const bool fin = s == ns;
            each(box((ns - s) * R), [&](int x, int y) {
                const A *c = cur + org + y * EW + x;
                A acc = A(0);
                static_for<0, SH::NPTS>([&](auto II) {
                    constexpr int i = decltype(II)::value;
                    A w;
                    if constexpr (std::is_same<A, double>::value) w = a.w[i];
                    else w = a.wf[i];
                    acc = fma(w, c[SH::dz(i) * EW + SH::dx(i)], acc);
                });
                const T t = from_acc<T>(acc);
                nxt[org + y * EW + x] = to_acc(t);
                if (fin && (last || x - x0 < H || x0 + tx - x <= H || y - y0 < H || y0 + ty - y <= H))
                    out[(long long)y * a.X + x] = t;
            });
            __syncthreads();
            A *q = cur;
            cur = nxt;
            nxt = q;
        }
        if (!last && tid == 0)
            asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(a.flags + blockIdx.x),
                         "l"((unsigned long long)(n + 1))
                         : "memory");
    }
}

template <typename T, class SH, int K> PatchEntry patch_entry(int dtype, int shape) {
    PatchEntry e;
    e.dtype = dtype;
    e.shape = shape;
    e.k = K;
    e.fn = perks_patch_kernel<T, SH, K>;
    return e;
}

template <typename T> void patch_entries(std::vector<PatchEntry> &out, int dtype) {
    out.push_back(patch_entry<T, S2d5, 4>(dtype, SH_2D5));
    out.push_back(patch_entry<T, S2d9, 4>(dtype, SH_2D9));
    out.push_back(patch_entry<T, S2ds9, 2>(dtype, SH_2DS9));
    out.push_back(patch_entry<T, S2d25, 2>(dtype, SH_2D25));
}

}  // namespace perks
