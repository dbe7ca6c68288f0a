// Column-strip stencil kernel for 2-D domains: several time steps per sweep,
// all of them in registers.
//
// A warp owns a strip of 32 V cells of x and a run of rows.  It streams the
// rows of the field downwards; row r of time level 0 enters a register window
// of 2R + 1 rows, which gives row r - R of level 1, which enters the next
// window, and so on: after TS windows the warp writes row r - TS R of level
// TS.  The x-neighbours of a lane's cells come from the adjacent lanes by
// warp shuffles, so every level loses R cells at each end of the strip; the
// strips overlap by HL lanes on each side, and the runs of rows by TS R rows,
// and only the cells that are right at level TS are stored.  Warps never meet
// inside a sweep; one grid barrier separates two sweeps.
//
// Why this split: a 2-D domain's step is a few cycles of work per warp and
// row.  One step at a time through a shared-memory row ring (the
// plane-streaming body: one block of 8 warps per SM walking its rows in
// lockstep) ran at 215 GCell/s for 2d5pt fp32 3072^2 (43.9 us per step, 1.7
// TB/s), bound by the latency of that walk; it takes 5.2 us per step here (TS = 4,
// 1.8 TCell/s; 2ds9pt 8.3, 2d9pt 6.7, 2d25pt 15.7).  A sweep of TS steps divides both
// the field's traffic and the grid barriers by TS, and 16 independent warps
// per SM hide the shuffle and load latencies.  Bound: the fp32 / fp64 pipe
// and the redundant cells of the overlaps ((h + R (TS - 1)) / h in rows, 32 /
// (32 - 2 HL) in x).
//
// Every cell adds its terms in table order with one fma chain from 0, rounded
// to the storage type after every step, as the other kernels do: fp32 and
// bf16 results are the same bits.
#pragma once

#include "stencil_vec.cuh"

namespace perks {

constexpr int kStripKDepth = 8;  // rows of level 0 in flight per warp (512 or 256 bytes each)

struct StripKArgs {
    int X, Z;             // row length, rows
    int nsx, nch;         // strips across x, runs of rows
    int sms;              // SMs (blocks from sms on share an SM with an earlier one)
    long long steps;
    double boundary;
    float boundary_f;
    double w[25];
    float wf[25];
    void *field[2];
    unsigned long long *bar;
    DevError *err;
    long long timeout_ns;
};

using StripKFn = void (*)(StripKArgs);

struct StripKEntry {
    int dtype, shape;
    int ts;               // steps per sweep
    int v;                // cells per lane
    int nt;               // threads per block, two blocks per SM
    int hl;               // overlap lanes on each side
    bool aligned;         // rows start on V-cell boundaries (X % V == 0)
    bool rest;            // for the steps left over from whole sweeps only
    StripKFn fn;
};

// Cells per lane: 16 bytes, 8 for bf16 (the fp32 accumulators fill the registers).
template <typename T> __host__ __device__ constexpr int strip_v() { return sizeof(T) == 8 ? 2 : 4; }

template <typename T, class SH, int TS> __host__ __device__ constexpr int strip_hl() {
    return (TS * SH::R + strip_v<T>() - 1) / strip_v<T>();
}

template <typename T> __device__ __forceinline__ typename AccOf<T>::type strip_w(const StripKArgs &a, int i) {
    if constexpr (std::is_same<T, double>::value) return a.w[i];
    else return a.wf[i];
}

// One item: rows [z0, z1) of the strip whose lane 0 starts at cell xs (may be
// negative), advanced by ns <= TS steps from `in` to `out`.
//
// Iteration t takes row r0 + t of level 0 into its window and computes row
// r0 + t - s (R + 1) of every level s from the rows the windows held after
// iteration t - 1 (one row of lag per level), so the TS levels of an
// iteration do not wait for one another.  Iterations where every level's row
// is needed and lies inside the domain -- all but the first and last few of an
// item -- run without a branch between the levels.
template <typename T, class SH, int TS, bool AL, class WF>
__device__ __forceinline__ void strip_sweep(const T *in, T *out, int X, int Z, int xs, int z0, int z1, int ns,
                                            T bnd_t, const WF &wgt, T *ring, int lane) {
    using A = typename AccOf<T>::type;
    constexpr int V = strip_v<T>();
    constexpr int R = SH::R, W = 2 * R + 1, HL = strip_hl<T, SH, TS>(), D = kStripKDepth;
    constexpr int PAD = SH::BOX ? 2 : 0;  // window cells kept left and right of a lane's own (an even number: the
                                          // own cells and the even offsets stay in aligned register pairs)
    using VT = VecOf<T, V>;
    const A bnd = to_acc(bnd_t);
    const int xl = xs + lane * V;
    const bool edge = xs < 0 || xs + 32 * V > X;  // some of the strip's cells lie outside the domain
    const bool store = lane >= HL && lane < 32 - HL && xl < X;
    const int nrows = z1 - z0 + 2 * TS * R;
    const int r0 = z0 - TS * R;

    // row t of level 0 into ring slot t % D: every lane copies the cells it
    // will read back itself; cells outside the domain are left as they are and
    // replaced when the row is taken out
    const T *src = in + (long long)r0 * X + xl;
    auto fetch = [&](int t) {
        const int r = r0 + t;
        if (t < nrows && r >= 0 && r < Z) {
            T *d = ring + (t % D) * 32 * V;
            const T *p = src + (long long)t * X;
            if constexpr (AL) {
                if (xl >= 0 && xl < X) cp_async<sizeof(T) * V>(d, p);
            } else {
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (xl + j >= 0 && xl + j < X) cp_async<sizeof(T)>(d + j, p + j);
            }
        }
        cp_async_commit();
    };
    auto outside = [&](int j) { return AL ? (xl < 0 || xl >= X) : (xl + j < 0 || xl + j >= X); };

    A win[TS][W][V + 2 * PAD];
    // a lane's row of one level, with its box neighbours
    auto enter = [&](A (&dst)[V + 2 * PAD], const A (&v)[V]) {
#pragma unroll
        for (int j = 0; j < V; ++j) dst[PAD + j] = v[j];
        if constexpr (SH::BOX) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                dst[PAD - R + j] = __shfl_up_sync(0xffffffffu, v[V - R + j], 1);
                dst[PAD + V + j] = __shfl_down_sync(0xffffffffu, v[j], 1);
            }
        }
    };

#pragma unroll
    for (int j = 0; j < D; ++j) fetch(j);

    // CHK: with the checks of an item's first and last iterations; EDGE: some
    // of the strip's cells lie outside the domain and keep the boundary value
    auto iteration = [&](auto PI, int t, auto CHK, auto EDGE) {
        constexpr int p = decltype(PI)::value;
        constexpr bool chk = decltype(CHK)::value, at_edge = decltype(EDGE)::value;
        static_for<0, TS>([&](auto QI) {
            constexpr int s = TS - decltype(QI)::value;
            if (chk && (t < s * W || t >= nrows + s)) return;
            constexpr int c = (p - 1 - R + 2 * W) % W;  // window slot of the row being computed
            A acc[V];
            if (!chk || s <= ns) {
                // the row with the neighbours a star needs
                A row[V + 2 * R];
                if constexpr (!SH::BOX) {
#pragma unroll
                    for (int j = 0; j < V; ++j) row[R + j] = win[s - 1][c][j];
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        row[j] = __shfl_up_sync(0xffffffffu, win[s - 1][c][V - R + j], 1);
                        row[R + V + j] = __shfl_down_sync(0xffffffffu, win[s - 1][c][j], 1);
                    }
                }
                auto cell = [&](auto II, int j) -> A {
                    constexpr int i = decltype(II)::value;
                    constexpr int dx = SH::dx(i), dz = SH::dz(i);
                    constexpr int slot = (p - 1 - R + dz + 2 * W) % W;
                    if constexpr (!SH::BOX && dz == 0) return row[R + j + dx];
                    else return win[s - 1][slot][PAD + j + dx];
                };
                if constexpr (std::is_same<A, float>::value) {
                    // a term at an even x offset updates two cells with one packed fma
                    // (__ffma2_rn rounds each lane as fmaf does)
                    float2 a2[V / 2];
#pragma unroll
                    for (int q = 0; q < V / 2; ++q) a2[q] = make_float2(0.f, 0.f);
                    static_for<0, SH::NPTS>([&](auto II) {
                        constexpr int i = decltype(II)::value;
                        const float w = wgt(i);
                        if constexpr (SH::dx(i) % 2 == 0) {
                            const float2 w2 = make_float2(w, w);
#pragma unroll
                            for (int q = 0; q < V / 2; ++q)
                                a2[q] = __ffma2_rn(w2, make_float2(cell(II, 2 * q), cell(II, 2 * q + 1)), a2[q]);
                        } else {
#pragma unroll
                            for (int q = 0; q < V / 2; ++q) {
                                a2[q].x = fmaf(w, cell(II, 2 * q), a2[q].x);
                                a2[q].y = fmaf(w, cell(II, 2 * q + 1), a2[q].y);
                            }
                        }
                    });
#pragma unroll
                    for (int q = 0; q < V / 2; ++q) {
                        acc[2 * q] = a2[q].x;
                        acc[2 * q + 1] = a2[q].y;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j) acc[j] = A(0);
                    static_for<0, SH::NPTS>([&](auto II) {
                        constexpr int i = decltype(II)::value;
                        const A w = wgt(i);
#pragma unroll
                        for (int j = 0; j < V; ++j) acc[j] = fma(w, cell(II, j), acc[j]);
                    });
                }
            } else {  // fewer steps than TS in the last sweep: the row goes through
#pragma unroll
                for (int j = 0; j < V; ++j) acc[j] = win[s - 1][c][PAD + j];
            }
            const int r = r0 + t - s * (R + 1);
            if constexpr (s < TS) {
                if constexpr (std::is_same<T, __nv_bfloat16>::value) {
#pragma unroll
                    for (int q = 0; q < V / 2; ++q) {
                        const float2 f2 = __bfloat1622float2(__floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]));
                        acc[2 * q] = f2.x;
                        acc[2 * q + 1] = f2.y;
                    }
                }
                const bool out_row = chk && (r < 0 || r >= Z);
                if (chk || at_edge) {
#pragma unroll
                    for (int j = 0; j < V; ++j) acc[j] = out_row || outside(j) ? bnd : acc[j];
                }
                enter(win[s < TS ? s : 0][p], acc);
            } else if (store) {
                T *q = out + (long long)r * X + xl;
                VT o;
#pragma unroll
                for (int j = 0; j < V; ++j) o.v[j] = from_acc<T>(acc[j]);
                if constexpr (AL) {
                    *reinterpret_cast<VT *>(q) = o;
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        if (!at_edge && !chk) q[j] = o.v[j];
                        else if (xl + j < X) q[j] = o.v[j];
                }
            }
        });
        if (chk && t >= nrows) return;
        cp_async_wait<D - 1>();
        const VT c = *reinterpret_cast<const VT *>(ring + (t % D) * 32 * V);
        A v[V];
        const bool out_row = chk && (r0 + t < 0 || r0 + t >= Z);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            v[j] = to_acc(c.v[j]);
            if (chk || at_edge) v[j] = out_row || outside(j) ? bnd : v[j];
        }
        fetch(t + D);
        enter(win[0][p], v);
    };

    constexpr std::true_type yes{};
    constexpr std::false_type no{};
    const int total = nrows + TS;
    // every level's row needed and inside the domain
    const int lo = max(TS * W, TS * (R + 1) - r0), hi = ns == TS ? min(nrows, Z - r0) : 0;
    for (int t0 = 0; t0 < total; t0 += W) {
        if (t0 >= lo && t0 + W <= hi) {
            if (edge) static_for<0, W>([&](auto PI) { iteration(PI, t0 + decltype(PI)::value, no, yes); });
            else static_for<0, W>([&](auto PI) { iteration(PI, t0 + decltype(PI)::value, no, no); });
        } else {
            static_for<0, W>([&](auto PI) { iteration(PI, t0 + decltype(PI)::value, yes, yes); });
        }
    }
    cp_async_wait_all();  // the next item starts an empty ring
}

template <typename T, class SH, int TS, bool AL, int NT>
__global__ void __launch_bounds__(NT, 2) perks_strip_kernel(const __grid_constant__ StripKArgs a) {
    constexpr int V = strip_v<T>(), HL = strip_hl<T, SH, TS>();
    __shared__ __align__(16) T rings[NT / 32][kStripKDepth * 32 * V];
    const int lane = threadIdx.x & 31;
    T *ring = rings[threadIdx.x >> 5] + lane * V;
    const long long nwarp = (long long)gridDim.x * (NT / 32);
    const long long items = (long long)a.nsx * a.nch;
    T bnd;
    if constexpr (std::is_same<T, double>::value) bnd = a.boundary;
    else bnd = from_acc<T>(a.boundary_f);
    auto wgt = [&](int i) { return strip_w<T>(a, i); };
    // Fewer items than warps: one warp of every block before a second one of
    // any, the two blocks of an SM starting two warps apart, so that its
    // quarters (warp index mod 4) get the same number.
    const int shift = (int)blockIdx.x >= a.sms ? 2 : 0;
    const long long first = (long long)(((threadIdx.x >> 5) + NT / 32 - shift) % (NT / 32)) * gridDim.x + blockIdx.x;
    unsigned long long epoch = 0;
    int src = 0;
    for (long long left = a.steps; left > 0; left -= TS, src ^= 1) {
        const int ns = (int)(left < TS ? left : TS);
        const T *in = static_cast<const T *>(a.field[src]);
        T *out = static_cast<T *>(a.field[src ^ 1]);
        for (long long q = first; q < items; q += nwarp) {
            const int c = (int)(q / a.nsx), sx = (int)(q % a.nsx);
            const int z0 = (int)((long long)a.Z * c / a.nch), z1 = (int)((long long)a.Z * (c + 1) / a.nch);
            strip_sweep<T, SH, TS, AL>(in, out, a.X, a.Z, sx * (32 - 2 * HL) * V - HL * V, z0, z1, ns, bnd, wgt, ring,
                                        lane);
        }
        if (left > TS && !grid_barrier(a.bar, gridDim.x, epoch, a.err, a.timeout_ns)) return;
    }
}

template <typename T, class SH, int TS, bool AL, int NT> StripKEntry strip_entry(int dtype, int shape, bool rest) {
    StripKEntry e;
    e.dtype = dtype;
    e.shape = shape;
    e.ts = TS;
    e.v = strip_v<T>();
    e.hl = strip_hl<T, SH, TS>();
    e.aligned = AL;
    e.nt = NT;
    e.rest = rest;
    e.fn = perks_strip_kernel<T, SH, TS, AL, NT>;
    return e;
}

template <typename T, class SH, int TS, int NT = 256>
void strip_entries(std::vector<StripKEntry> &out, int dtype, int shape, bool rest = false) {
    out.push_back(strip_entry<T, SH, TS, true, NT>(dtype, shape, rest));
    if constexpr (!std::is_same<T, __nv_bfloat16>::value)
        out.push_back(strip_entry<T, SH, TS, false, NT>(dtype, shape, rest));
}

}  // namespace perks
