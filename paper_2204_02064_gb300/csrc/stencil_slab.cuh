// Slab-streaming kernel for 3-D domains of any row length, no caches.
//
// A block owns a column of the domain, LX * V cells of x by BY rows of y, and
// streams its z planes through a shared-memory ring (cp.async, slab_ahead
// planes ahead).  A row of the tile is a group of LX = 8, 16 or 32 lanes with
// V neighbouring cells each; a thread owns RY consecutive rows, so a row of a
// plane that several of its output rows need is read from shared memory once:
//   * boxes (3d27pt, poisson): the RY + 2 rows of an arriving plane are each
//     read once and feed the running sums of the three output planes they
//     belong to (planes arrive in z order, which is the table order of the
//     terms, so every cell keeps its one fma chain);
//   * stars (3d7pt, 3d13pt): a thread's own columns stay in registers for
//     2R + 1 planes; only the R rows above and below its rows come from
//     shared memory again.
// Row lengths that V divides: a thread's V cells are neighbours (16-byte
// copies, loads and stores), its x-neighbours come from the adjacent lanes by
// warp shuffles and, at the ends of a row, from the row's pad cells.  Other
// row lengths: a thread's V cells lie LX apart, so that every copy, shared
// load and store of a row is one run of LX cells at any alignment, and the
// x-neighbours are read from shared memory the same way.
//
// The blocks' work: where the columns times a whole number of parts nearly
// fill the co-resident grid, every column is cut into that many parts of its
// planes, and the blocks walk them in step, so that the halo rows two columns
// share are in L2 when the second asks; else the columns' planes, laid end to
// end, are cut into one equal share per block.
//
// Why: the plane-streaming body gives a thread one vector of one row, so a
// 27-point cell costs nine shared loads and eighteen shuffles per vector and
// a block barrier comes every two rows' worth of work; 92 us per step for
// 3d27pt fp32 256^3 (182 GCell/s), and domains whose row length no vector
// divides ran one cell per thread (133 us per step for 251 x 246 x 233, 110
// GCell/s).  Here 32 and 33 us (530 and 435 GCell/s), 3d7pt 384^3 fp32 97 -> 74
// us (6.1 TB/s), bf16 66 -> 41 us.  The planes in the middle of a piece run
// without the checks of its first and last ones, and the copies and stores
// walk running pointers: 3d27pt 251 x 246 x 233 took 42 us, 3d13pt bf16 384^3
// 90 (now 56), with a branch per row and the addresses formed anew.
// Bound: HBM (8 B per cell and step in fp32) for stars of large domains, the
// latency of shared loads and block barriers for boxes (issue slots 52 %, FMA
// pipe 38 %), the FP64 pipe for fp64.
#pragma once

#include "stencil_vec.cuh"

namespace perks {

constexpr int kSlabThreads = 256;

struct SlabArgs {
    int X, Y, Z;
    long long XY;
    int loglx;            // log2 of the lanes per row
    int nsx, nsy;         // columns across x and y
    int nz;               // 0: equal shares of the columns' planes laid end to end; else every column cut into nz
                          // parts, one per block, all walked in step
    int PW, plane;        // ring row pitch and cells per ring slot
    long long steps;
    double boundary;
    float boundary_f;
    double w[27];
    float wf[27];
    void *field[2];
    unsigned long long *bar;
    DevError *err;
    long long timeout_ns;
};

using SlabFn = void (*)(SlabArgs);

struct SlabEntry {
    int dtype, shape;
    int v, ry;
    int slots, ahead;     // ring slots, planes in flight
    bool aligned;         // X % V == 0
    SlabFn fn;
};

// 16 bytes per thread and row; rows per thread.  Stars: 3d7pt fp32 with four
// rows instead of two takes 85 us per step at 384^3 (two: 74), 19.7 at 256^3
// (20.2), 4.0 at 50 x 45 x 39 (3.4).  3d27pt: fp32 with two 35.5 us at 251 x 246 x
// 233 (four: 33.2); fp64, bound by the FP64 pipe, with four 59 us at 88 x 96 x
// 100, whose rows fill three quarters of them (two: 54), and equal elsewhere.
template <typename T> __host__ __device__ constexpr int slab_v() { return 16 / sizeof(T); }
template <typename T, class SH> __host__ __device__ constexpr int slab_ry() { return SH::BOX && sizeof(T) == 4 ? 4 : 2; }
// planes in flight, and planes an iteration reads (boxes: the arriving one;
// stars: also those back to the output plane, for its rows above and below)
template <class SH> __host__ __device__ constexpr int slab_ahead() { return SH::BOX || SH::R > 1 ? 3 : 4; }
template <class SH> __host__ __device__ constexpr int slab_slots() { return slab_ahead<SH>() + (SH::BOX ? 1 : SH::R + 1); }

// Cell u of a thread's cells v displaced by DX, its neighbours in side as the
// kernel's sides() leaves them.
template <int DX, bool AL, int R, typename A, int V, int S0, int S1>
__device__ __forceinline__ A slab_at(const A (&v)[V], const A (&side)[S0][S1], int u) {
    if constexpr (DX == 0) {
        return v[u];
    } else if constexpr (!AL) {
        constexpr int k = DX < 0 ? 2 * (-DX - 1) : 2 * DX - 1;
        return side[k][u];
    } else {
        const int x = u + DX;
        return x < 0 ? side[0][x + R < 0 ? 0 : x + R] : x >= V ? side[1][x - V] : v[x];
    }
}

template <typename T, class SH, bool AL>
__global__ void __launch_bounds__(kSlabThreads, 2) perks_slab_kernel(const __grid_constant__ SlabArgs a) {
    using A = typename AccOf<T>::type;
    constexpr int V = slab_v<T>(), RY = slab_ry<T, SH>(), R = SH::R, W = 2 * R + 1, D = slab_ahead<SH>();
    constexpr int S = slab_slots<SH>();
    using VT = VecOf<T, V>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *ring = reinterpret_cast<T *>(smem_raw);
    const int lane = threadIdx.x & 31;
    const int LX = 1 << a.loglx;
    const int pos = lane & (LX - 1);                       // the thread's vector in its row
    const int grp = threadIdx.x >> a.loglx, ngrp = kSlabThreads >> a.loglx;
    T bnd;
    if constexpr (std::is_same<T, double>::value) bnd = a.boundary;
    else bnd = from_acc<T>(a.boundary_f);
    auto wgt = [&](int i) -> A {
        if constexpr (std::is_same<T, double>::value) return a.w[i];
        else return a.wf[i];
    };
    unsigned long long epoch = 0;
    const int cols = a.nsx * a.nsy;
    const long long L = (long long)cols * a.Z;
    long long s_lo = L * blockIdx.x / gridDim.x, s_hi = L * (blockIdx.x + 1) / gridDim.x;
    if (a.nz > 0) {
        const long long c0 = (long long)(blockIdx.x % cols) * a.Z;
        const int part = blockIdx.x / cols;
        s_lo = c0 + (long long)a.Z * part / a.nz;
        s_hi = c0 + (long long)a.Z * (part + 1) / a.nz;
    }
    const bool one_piece = s_lo / a.Z == (s_hi - 1) / a.Z;
    T *const ring_end = ring + S * a.plane;
    bool fresh = true;                                     // the ring's cells outside the domain are not set yet

    for (long long k = 0; k < a.steps; ++k) {
        const T *in = static_cast<const T *>(a.field[k & 1]);
        T *out = static_cast<T *>(a.field[(k & 1) ^ 1]);
        for (long long s0 = s_lo; s0 < s_hi;) {
            const int col = (int)(s0 / a.Z);
            const int z0 = (int)(s0 - (long long)col * a.Z);
            const long long s1 = min(s_hi, (long long)(col + 1) * a.Z);
            const int nz = (int)(s1 - s0);
            s0 = s1;
            int x0, wx, y0, ty;                            // the column's cells of x (wx of them) and rows
            split_axis(AL ? a.X / V : a.X, a.nsx, col % a.nsx, x0, wx);
            if constexpr (AL) { x0 *= V; wx *= V; }
            split_axis(a.Y, a.nsy, col / a.nsx, y0, ty);
            const int xi = AL ? pos * V : pos;             // its first one in the row
            const bool in_row = xi < wx;
            const bool last = AL && xi + V == wx;
            if (fresh || !one_piece) {
                // cells outside the domain keep the boundary value; the copies below never touch them
                __syncthreads();
                for (int e = threadIdx.x; e < S * a.plane / V; e += kSlabThreads) set_vec<T, V>(ring + e * V, bnd);
                __syncthreads();
                fresh = false;
            }
            // the planes of the piece (z = z0 - R on) into the slots in turn, one more per call.  A thread copies every
            // ngrp-th row, from its first one inside the domain on
            int fz = z0 - R;
            const int fz1 = z0 + nz + R;
            T *fslot = ring;
            const int r_lo = max(0, R - y0), r_hi = min(ty + 2 * R, a.Y - y0 + R);
            const int r_first = grp >= r_lo ? grp : grp + (r_lo - grp + ngrp - 1) / ngrp * ngrp;
            const T *fsrc = in + (long long)fz * a.XY + (long long)(y0 - R + r_first) * a.X + x0 + xi;
            const int foff = r_first * a.PW + V + xi;
            const long long fstep = (long long)ngrp * a.X;
            const int fdstep = ngrp * a.PW;
            const bool left = AL ? pos == 0 && x0 > 0 : pos < R && x0 > 0;
            const bool right = AL ? last && x0 + wx < a.X : pos < R && x0 + wx + pos < a.X;
            auto fill = [&]() {
                if (fz < fz1) {
                    if (fz < 0 || fz >= a.Z) {
                        for (int e = threadIdx.x; e < a.plane / V; e += kSlabThreads) set_vec<T, V>(fslot + e * V, bnd);
                    } else {
                        const T *p = fsrc;
                        T *d = fslot + foff;
                        for (int r = r_first; r < r_hi; r += ngrp) {
                            if constexpr (AL) {
                                if (in_row) cp_async<sizeof(T) * V>(d, p);
                                if (left) cp_async<sizeof(T) * V>(d - V, p - V);
                                if (right) cp_async<sizeof(T) * V>(d + V, p + V);
                            } else {
#pragma unroll
                                for (int u = 0; u < V; ++u)
                                    if (xi + LX * u < wx) cp_async<sizeof(T)>(d + LX * u, p + LX * u);
                                if (left) cp_async<sizeof(T)>(d - 2 * pos - 1, p - 2 * pos - 1);
                                if (right) cp_async<sizeof(T)>(d + wx, p + wx);
                            }
                            p += fstep;
                            d += fdstep;
                        }
                    }
                    ++fz;
                    fsrc += a.XY;
                    fslot = fslot + a.plane == ring_end ? ring : fslot + a.plane;
                }
                cp_async_commit();
            };
            const int ry0 = grp * RY;                      // the thread's first row in the tile
            const int toff = ry0 * a.PW + V + xi;
            // row r (from the thread's first one - R) of the slot: the thread's V cells ...
            auto own = [&](const T *slot, int r, A (&v)[V]) {
                const T *row = slot + toff + r * a.PW;
                if constexpr (AL) {
                    const VT c = *reinterpret_cast<const VT *>(row);
#pragma unroll
                    for (int u = 0; u < V; ++u) v[u] = to_acc(c.v[u]);
                } else {
#pragma unroll
                    for (int u = 0; u < V; ++u) v[u] = to_acc(row[LX * u]);
                }
            };
            // ... and their neighbours: AL, R cells on either side of the vector (side[0][j] left, side[1][j]
            // right); else cell u's neighbours at -j - 1 and j + 1 (side[2 j][u], side[2 j + 1][u])
            constexpr int S0 = AL ? 2 : 2 * R, S1 = AL ? R : V;
            auto sides = [&](const T *slot, int r, const A (&v)[V], A (&side)[S0][S1]) {
                const T *row = slot + toff + r * a.PW;
                if constexpr (AL) {
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        side[0][j] = __shfl_up_sync(0xffffffffu, v[V - R + j], 1);
                        side[1][j] = __shfl_down_sync(0xffffffffu, v[j], 1);
                    }
                    if (pos == 0)
#pragma unroll
                        for (int j = 0; j < R; ++j) side[0][j] = to_acc(row[j - R]);
                    if (last)
#pragma unroll
                        for (int j = 0; j < R; ++j) side[1][j] = to_acc(row[V + j]);
                } else {
#pragma unroll
                    for (int j = 0; j < R; ++j)
#pragma unroll
                        for (int u = 0; u < V; ++u) {
                            side[2 * j][u] = to_acc(row[LX * u - j - 1]);
                            side[2 * j + 1][u] = to_acc(row[LX * u + j + 1]);
                        }
                }
            };
            T *oplane = out + (long long)z0 * a.XY + (long long)(y0 + ry0) * a.X + x0 + xi;  // the next output plane
            auto store = [&](int j, const A (&acc)[V]) {   // its row j of the thread
                if (!in_row || ry0 + j >= ty) return;
                T *q = oplane + j * a.X;
                VT o;
                if constexpr (std::is_same<T, __nv_bfloat16>::value) {
                    __nv_bfloat162 *o2 = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
                    for (int u = 0; u < V / 2; ++u) o2[u] = __floats2bfloat162_rn(acc[2 * u], acc[2 * u + 1]);
                } else {
#pragma unroll
                    for (int u = 0; u < V; ++u) o.v[u] = from_acc<T>(acc[u]);
                }
                if constexpr (AL) {
                    *reinterpret_cast<VT *>(q) = o;
                } else {
#pragma unroll
                    for (int u = 0; u < V; ++u)
                        if (xi + LX * u < wx) q[LX * u] = o.v[u];
                }
            };
            // rows of the tile a thread reads: r = ry0 .. ry0 + RY - 1 + 2R in ring rows (ring row = tile row + R);
            // a thread whose rows lie past the tile's end reads rows that exist in the slot, and stores nothing; a
            // warp without a row only copies
            const bool work = __any_sync(0xffffffffu, ry0 < ty);

            const int n = nz + 2 * R;
#pragma unroll
            for (int i = 0; i < D; ++i) fill();
            const T *slot = ring;                          // the arriving plane
            auto next = [&](const T *q) { return q + a.plane == ring_end ? (const T *)ring : q + a.plane; };
            if constexpr (SH::BOX) {
                static_assert(R == 1, "boxes of radius 1");
                A acc[3][RY][V];                           // running sums of output plane t in acc[t % 3]
                // CHK: the first and last planes of a piece, which belong to fewer than three output planes
                auto iteration = [&](auto PI, int i, auto CHK) {
                    constexpr int p = decltype(PI)::value;  // i % 3
                    constexpr bool chk = decltype(CHK)::value;
                    cp_async_wait<D - 1>();
                    __syncthreads();
                    fill();
                    const T *cur = slot;
                    slot = next(slot);
                    // plane i: term dz = -1 of output plane i (new sums), 0 of i - 1, +1 of i - 2 (done)
#pragma unroll
                    for (int j = 0; j < RY; ++j)
#pragma unroll
                        for (int u = 0; u < V; ++u) acc[p][j][u] = A(0);
                    if (!work) return;
                    // the output planes i - 1 - dz that exist
                    const bool use_lo = !chk || i < nz, use_mid = !chk || (i >= 1 && i <= nz), use_hi = !chk || i >= 2;
                    static_for<0, RY + 2>([&](auto QI) {
                        constexpr int q = decltype(QI)::value;
                        A v[V], side[S0][S1];
                        own(cur, q, v);
                        sides(cur, q, v, side);
                        static_for<0, 3>([&](auto ZI) {
                            constexpr int z = decltype(ZI)::value - 1;
                            constexpr int s = (p - 1 - z + 3) % 3;   // output plane i - 1 - z
                            if (!(z < 0 ? use_lo : z > 0 ? use_hi : use_mid)) return;
                            static_for<0, SH::NPTS>([&](auto II) {
                                constexpr int t = decltype(II)::value;
                                constexpr int dx = SH::dx(t), dy = SH::dy(t), dz = SH::dz(t);
                                constexpr int j = q - 1 - dy;        // output row this row is at offset dy of
                                if constexpr (dz == z && j >= 0 && j < RY) {
                                    const A w = wgt(t);
                                    if constexpr (std::is_same<A, float>::value) {
                                        const float2 w2 = make_float2(w, w);
#pragma unroll
                                        for (int u = 0; u < V; u += 2) {
                                            const float2 r = __ffma2_rn(
                                                w2, make_float2(slab_at<dx, AL, R>(v, side, u), slab_at<dx, AL, R>(v, side, u + 1)),
                                                make_float2(acc[s][j][u], acc[s][j][u + 1]));
                                            acc[s][j][u] = r.x;
                                            acc[s][j][u + 1] = r.y;
                                        }
                                    } else {
#pragma unroll
                                        for (int u = 0; u < V; ++u) acc[s][j][u] = fma(w, slab_at<dx, AL, R>(v, side, u), acc[s][j][u]);
                                    }
                                }
                            });
                        });
                    });
                    if (use_hi) {
                        constexpr int s = (p + 1) % 3;      // output plane i - 2
#pragma unroll
                        for (int j = 0; j < RY; ++j) store(j, acc[s][j]);
                        oplane += a.XY;
                    }
                };
                constexpr std::true_type yes{};
                constexpr std::false_type no{};
                for (int i0 = 0; i0 < n; i0 += 3) {
                    if (i0 >= 2 && i0 + 3 <= nz)
                        static_for<0, 3>([&](auto PI) { iteration(PI, i0 + decltype(PI)::value, no); });
                    else
                        static_for<0, 3>([&](auto PI) {
                            if (i0 + decltype(PI)::value < n) iteration(PI, i0 + decltype(PI)::value, yes);
                        });
                }
            } else {
                A c[W][RY][V];                             // the thread's cells of the last 2R + 1 planes
                const T *centre = ring;                    // the plane R before the arriving one, from plane R on
                auto iteration = [&](auto PI, int i) {
                    constexpr int p = decltype(PI)::value;  // i % W
                    cp_async_wait<D - 1>();
                    __syncthreads();
                    fill();
                    const T *cur = slot;
                    slot = next(slot);
                    // output plane i - 2R: its centre plane is i - R
                    const T *mid = centre;
                    if (i >= R) centre = next(centre);
                    if (!work) return;
#pragma unroll
                    for (int j = 0; j < RY; ++j) own(cur, R + j, c[p][j]);
                    if (i < 2 * R) return;
                    constexpr int m = (p - R + W) % W;
                    A up[R][V], dn[R][V];                  // rows above and below the thread's
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        own(mid, j, up[j]);
                        own(mid, R + RY + j, dn[j]);
                    }
                    static_for<0, RY>([&](auto JI) {
                        constexpr int j = decltype(JI)::value;
                        A side[S0][S1];
                        sides(mid, R + j, c[m][j], side);
                        A acc[V];
#pragma unroll
                        for (int u = 0; u < V; ++u) acc[u] = A(0);
                        static_for<0, SH::NPTS>([&](auto II) {
                            constexpr int t = decltype(II)::value;
                            constexpr int dx = SH::dx(t), dy = SH::dy(t), dz = SH::dz(t);
                            constexpr int zs = (p - R + dz + 2 * W) % W;
                            auto cell = [&](int u) -> A {
                                if constexpr (dy != 0) {
                                    constexpr int r = j + dy;
                                    if constexpr (r < 0) return up[r + R][u];
                                    else if constexpr (r >= RY) return dn[r - RY][u];
                                    else return c[m][r][u];
                                } else if constexpr (dx != 0) {
                                    return slab_at<dx, AL, R>(c[m][j], side, u);
                                } else {
                                    return c[zs][j][u];
                                }
                            };
                            const A w = wgt(t);
                            if constexpr (std::is_same<A, float>::value && (!AL || dx % 2 == 0)) {
                                const float2 w2 = make_float2(w, w);
#pragma unroll
                                for (int u = 0; u < V; u += 2) {
                                    const float2 r =
                                        __ffma2_rn(w2, make_float2(cell(u), cell(u + 1)), make_float2(acc[u], acc[u + 1]));
                                    acc[u] = r.x;
                                    acc[u + 1] = r.y;
                                }
                            } else {
#pragma unroll
                                for (int u = 0; u < V; ++u) acc[u] = fma(w, cell(u), acc[u]);
                            }
                        });
                        store(j, acc);
                    });
                    oplane += a.XY;
                };
                for (int i0 = 0; i0 < n; i0 += W)
                    static_for<0, W>([&](auto PI) {
                        if (i0 + decltype(PI)::value < n) iteration(PI, i0 + decltype(PI)::value);
                    });
            }
            cp_async_wait_all();
            if (s0 < s_hi) __syncthreads();                // the next piece refills slots still being read
        }
        if (k + 1 < a.steps && !grid_barrier(a.bar, gridDim.x, epoch, a.err, a.timeout_ns)) return;
    }
}

template <typename T, class SH, bool AL> SlabEntry slab_entry(int dtype, int shape) {
    SlabEntry e;
    e.dtype = dtype;
    e.shape = shape;
    e.v = slab_v<T>();
    e.ry = slab_ry<T, SH>();
    e.slots = slab_slots<SH>();
    e.ahead = slab_ahead<SH>();
    e.aligned = AL;
    e.fn = perks_slab_kernel<T, SH, AL>;
    return e;
}

template <typename T> void slab_entries(std::vector<SlabEntry> &out, int dtype) {
    out.push_back(slab_entry<T, S3d7, true>(dtype, SH_3D7));
    out.push_back(slab_entry<T, S3d27, true>(dtype, SH_3D27));
    out.push_back(slab_entry<T, S3d13, true>(dtype, SH_3D13));
    out.push_back(slab_entry<T, S3d19, true>(dtype, SH_3D19));
    if constexpr (!std::is_same<T, __nv_bfloat16>::value) {
        out.push_back(slab_entry<T, S3d7, false>(dtype, SH_3D7));
        out.push_back(slab_entry<T, S3d27, false>(dtype, SH_3D27));
        out.push_back(slab_entry<T, S3d13, false>(dtype, SH_3D13));
        out.push_back(slab_entry<T, S3d19, false>(dtype, SH_3D19));
    }
}

}  // namespace perks
