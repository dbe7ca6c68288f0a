// Batched variable-coefficient Poisson: -div(k grad u) = f on nx*ny grids
// (5-point finite volumes, h = 1, face coefficient = harmonic mean of the two
// cells' k, Dirichlet 0 through a ghost cell carrying the boundary cell's k),
// solved by CG (the Sec. 2.2.2 recurrence) as ONE persistent launch.
//
// Problems are independent, so the batch needs no grid barrier: each block
// (or group of C blocks) owns one problem at a time, pulling problems from an
// atomic counter, keeps its scalars and partial sums on chip and runs that
// problem's whole CG loop -- SpMV (matrix-free, from precomputed face
// coefficients), dot products and axpys.  With C = 1 the reductions are
// block-level only.  With C > 1 the problem's rows are split over the group's
// blocks, which meet at a bounded barrier of their own after each p update
// and in each dot product (block sums added in rank order, so every block of
// the group takes the same decisions): a batch ends with its hardest problem
// running alone, and a group runs it C times faster.  The true residual is
// recomputed in fp64 on exit and CG restarts while it is above tolerance.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "internal.h"
#include "common.cuh"

using namespace perks;

namespace {

constexpr int kPoiThreads = 256;
constexpr int kPoiMaxGroup = 8;  // blocks per problem, at most

struct PoissonArgs {
    int nx, ny, nprob;
    long long n;                 // cells per problem
    const double *fx;            // [prob][ny][nx+1] x-face coefficients
    const double *fy;            // [prob][ny+1][nx] y-face coefficients
    const double *dg;            // [prob][n] diagonal: (fw + fe) + (fs + fn) of each cell
    const double *b;             // [prob][n]
    double *x, *r, *p, *q;       // [prob][n]
    double rtol;
    int max_iter;
    int max_restarts;
    int *queue;                  // next problem to take
    int *iters;                  // [prob] recurrence iterations
    double *true_rel;            // [prob] ||b - A x|| / ||b||
    int *status;                 // [prob]
    int group;                   // blocks per problem (C)
    unsigned long long *gbar;    // [groups] barrier counter of each block group
    int *gprob;                  // [groups] problem taken by each group
    double *gpart;               // [groups][2][C] block sums, double-buffered
    double *slots;               // [groups][3][C] sums of exchange_sum, all empty before a launch
    double *halo;                // [blocks][2][nx] p of the rows south and north of a block's rows
    int on_chip;                 // each block keeps r of its rows in shared memory
    DevError *err;
    long long timeout_ns;
};

__global__ void poisson_faces_kernel(const double *__restrict__ k, int nx, int ny, long long total_cells,
                                     double *fx, double *fy) {
    // one thread per face; x-faces: (nx+1)*ny per problem, y-faces: nx*(ny+1)
    const long long nfx = (long long)(nx + 1) * ny, nfy = (long long)nx * (ny + 1);
    const long long nprob = total_cells / ((long long)nx * ny);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nprob * (nfx + nfy); t += stride) {
        const long long pb = t / (nfx + nfy), u = t % (nfx + nfy);
        const double *kp = k + pb * (long long)nx * ny;
        if (u < nfx) {
            const int j = (int)(u / (nx + 1)), i = (int)(u % (nx + 1));
            double f;
            if (i == 0) f = kp[(long long)j * nx];
            else if (i == nx) f = kp[(long long)j * nx + nx - 1];
            else {
                const double a = kp[(long long)j * nx + i - 1], c = kp[(long long)j * nx + i];
                f = 2.0 * a * c / (a + c);
            }
            fx[pb * nfx + u] = f;
        } else {
            const long long v = u - nfx;
            const int j = (int)(v / nx), i = (int)(v % nx);
            double f;
            if (j == 0) f = kp[i];
            else if (j == ny) f = kp[(long long)(ny - 1) * nx + i];
            else {
                const double a = kp[(long long)(j - 1) * nx + i], c = kp[(long long)j * nx + i];
                f = 2.0 * a * c / (a + c);
            }
            fy[pb * nfy + v] = f;
        }
    }
}

// Diagonal of every cell, (fw + fe) + (fs + fn), computed once: the matvec
// then needs one multiply and four fused multiply-adds per cell (the FP64
// pipe, not HBM, bounds this CG on GB300).
__global__ void poisson_diag_kernel(const double *__restrict__ fx, const double *__restrict__ fy, int nx, int ny,
                                    long long total_cells, double *dg) {
    const long long n = (long long)nx * ny;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total_cells;
         t += (long long)gridDim.x * blockDim.x) {
        const long long pb = t / n, c = t % n;
        const int j = (int)(c / nx), i = (int)(c % nx);
        const double *fxp = fx + pb * (long long)(nx + 1) * ny;
        const double *fyp = fy + pb * (long long)nx * (ny + 1);
        const double fw = fxp[(long long)j * (nx + 1) + i], fe = fxp[(long long)j * (nx + 1) + i + 1];
        const double fs = fyp[(long long)j * nx + i], fn = fyp[(long long)(j + 1) * nx + i];
        dg[t] = (fw + fe) + (fs + fn);
    }
}

// (A v)_c for cell c = (i, j) of one problem.
__device__ __forceinline__ double apply_cell(const double *__restrict__ fxp, const double *__restrict__ fyp,
                                             const double *__restrict__ dgp, const double *__restrict__ v, int nx,
                                             int ny, int i, int j) {
    const long long c = (long long)j * nx + i;
    const double fw = fxp[(long long)j * (nx + 1) + i], fe = fxp[(long long)j * (nx + 1) + i + 1];
    const double fs = fyp[(long long)j * nx + i], fn = fyp[(long long)(j + 1) * nx + i];
    const double vc = v[c];
    double acc = dgp[c] * vc;
    if (i > 0) acc = fma(-fw, v[c - 1], acc);
    if (i + 1 < nx) acc = fma(-fe, v[c + 1], acc);
    if (j > 0) acc = fma(-fs, v[c - nx], acc);
    if (j + 1 < ny) acc = fma(-fn, v[c + nx], acc);
    return acc;
}

// (A v) for kRows consecutive cells (i, j0..j0+kRows-1) of one column, with
// each value loaded once (v down the column, faces once per row) and the same
// arithmetic, in the same order, as apply_cell.  Rows at or beyond ny are
// skipped.
template <int K>
__device__ __forceinline__ void apply_column(const double *__restrict__ fxp, const double *__restrict__ fyp,
                                             const double *__restrict__ dgp, const double *__restrict__ v, int nx,
                                             int ny, int i, int j0, double (&out)[K], double (&vc)[K]) {
    double col[K + 2];
    double fyv[K + 1];
#pragma unroll
    for (int u = -1; u <= K; ++u) {
        const int j = j0 + u;
        col[u + 1] = (j >= 0 && j < ny) ? v[(long long)j * nx + i] : 0.0;
    }
#pragma unroll
    for (int u = 0; u <= K; ++u) {
        const int j = j0 + u;
        fyv[u] = (j <= ny) ? __ldg(fyp + (long long)j * nx + i) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < K; ++u) {
        const int j = j0 + u;
        if (j < ny) {
            const long long c = (long long)j * nx + i;
            const double *fr = fxp + (long long)j * (nx + 1) + i;
            const double fw = __ldg(fr), fe = __ldg(fr + 1);
            const double fs = fyv[u], fn = fyv[u + 1];
            const double vcen = col[u + 1];
            double acc = __ldg(dgp + c) * vcen;
            if (i > 0) acc = fma(-fw, v[c - 1], acc);
            if (i + 1 < nx) acc = fma(-fe, v[c + 1], acc);
            if (j > 0) acc = fma(-fs, col[u], acc);
            if (j + 1 < ny) acc = fma(-fn, col[u + 2], acc);
            out[u] = acc;
            vc[u] = vcen;
        }
    }
}

__device__ __forceinline__ double bsum(double v, double *red) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        t = l < (int)(blockDim.x >> 5) ? red[l] : 0.0;
        t = warp_sum(t);
        if (l == 0) red[32] = t;
    }
    __syncthreads();
    return red[32];
}

// Row-blocked traversal: each thread takes cell column i of kRows rows at a
// time, so the loads of kRows independent cells (and their neighbours) are in
// flight together instead of one row's worth per memory round trip.
constexpr int kRows = 4;
// Linear traversal unroll for the vector updates.
constexpr int kLin = 2;

// r = b - A x over the whole problem; returns this thread's partial <r,r>
// (and <b,b> through bb); optionally p = r.
template <bool SET_P, int ROWS>
__device__ __forceinline__ double residual_pass(const double *__restrict__ fxp, const double *__restrict__ fyp,
                                                const double *__restrict__ dgp,
                                                const double *__restrict__ b, const double *__restrict__ x,
                                                double *__restrict__ r, double *__restrict__ p, int nx, int ny,
                                                int jb, int je, double &bb) {
    double rr = 0.0;
    for (int j0 = jb; j0 < je; j0 += ROWS)
        for (int i = threadIdx.x; i < nx; i += blockDim.x) {
            double rv[ROWS], bv[ROWS], xc[ROWS];
            apply_column<ROWS>(fxp, fyp, dgp, x, nx, ny, i, j0, rv, xc);
#pragma unroll
            for (int u = 0; u < ROWS; ++u) {
                const int j = j0 + u;
                if (j < ny) {
                    const long long c = (long long)j * nx + i;
                    bv[u] = __ldg(b + c);
                    rv[u] = bv[u] - rv[u];
                }
            }
#pragma unroll
            for (int u = 0; u < ROWS; ++u) {
                const int j = j0 + u;
                if (j < ny) {
                    const long long c = (long long)j * nx + i;
                    r[c] = rv[u];
                    if (SET_P) p[c] = rv[u];
                    bb = fma(bv[u], bv[u], bb);
                    rr = fma(rv[u], rv[u], rr);
                }
            }
        }
    return rr;
}

// Rows [jb, je) of a problem owned by block `rank` of a group of C: row
// blocks of ROWS rows split evenly.
template <int ROWS>
__device__ __forceinline__ void group_rows(int ny, int C, int rank, int &jb, int &je) {
    const int nrb = (ny + ROWS - 1) / ROWS;
    jb = min(ny, (int)((long long)nrb * rank / C) * ROWS);
    je = min(ny, (int)((long long)nrb * (rank + 1) / C) * ROWS);
}

template <int NT, int MINB, int ROWS, int LIN, bool GROUP>
__global__ void __launch_bounds__(NT, MINB) perks_poisson_cg_kernel(const __grid_constant__ PoissonArgs a) {
    __shared__ double red[33];
    __shared__ int s_prob;
    const int nx = a.nx, ny = a.ny;
    const long long n = a.n;
    const int C = GROUP ? a.group : 1;
    const int g = blockIdx.x / C, rank = blockIdx.x % C;
    int jb = 0, je = ny;
    if (GROUP) group_rows<ROWS>(ny, C, rank, jb, je);
    const long long cb = (long long)jb * nx, ce = (long long)je * nx;
    unsigned long long epoch = 0;
    int nred = 0;
    // the group's sum of a per-thread value: block sums, then the group's
    // block sums in rank order (the same value in every block); false if the
    // group barrier gave up
    auto gsum = [&](double v, double &out) -> bool {
        v = bsum(v, red);
        if (!GROUP) { out = v; return true; }
        double *slot = a.gpart + ((long long)g * 2 + (nred & 1)) * C;
        ++nred;
        if (threadIdx.x == 0) slot[rank] = v;
        if (!grid_barrier(a.gbar + g, C, epoch, a.err, a.timeout_ns)) return false;
        double t = 0.0;
        for (int i = 0; i < C; ++i) t += __ldcg(slot + i);
        out = t;
        return true;
    };
    for (;;) {
        if (GROUP) {
            if (rank == 0 && threadIdx.x == 0) a.gprob[g] = atomicAdd(a.queue, 1);
            if (!grid_barrier(a.gbar + g, C, epoch, a.err, a.timeout_ns)) return;
            if (threadIdx.x == 0) s_prob = __ldcg(a.gprob + g);
        } else {
            if (threadIdx.x == 0) s_prob = atomicAdd(a.queue, 1);
        }
        __syncthreads();
        const int pb = s_prob;
        __syncthreads();
        if (pb >= a.nprob) break;
        const double *__restrict__ fxp = a.fx + (long long)pb * (nx + 1) * ny;
        const double *__restrict__ fyp = a.fy + (long long)pb * nx * (ny + 1);
        const double *__restrict__ dgp = a.dg + (long long)pb * n;
        const double *__restrict__ b = a.b + pb * n;
        double *__restrict__ x = a.x + pb * n;
        double *__restrict__ r = a.r + pb * n;
        double *__restrict__ p = a.p + pb * n;
        double *__restrict__ q = a.q + pb * n;
        // r = b - A x, p = r
        double bb = 0.0, rr;
        const double rr_own = residual_pass<true, ROWS>(fxp, fyp, dgp, b, x, r, p, nx, ny, jb, je, bb);
        if (!gsum(bb, bb) || !gsum(rr_own, rr)) return;
        const double tol2 = a.rtol * a.rtol * bb;
        int it = 0, status = PERKS_ERR_NOT_CONVERGED;
        for (int restart = 0;; ++restart) {
            if (rr <= tol2) { status = PERKS_OK; break; }
            bool converged = false;
            while (it < a.max_iter) {
                // q = A p, <p, q>
                double pq = 0.0;
                for (int j0 = jb; j0 < je; j0 += ROWS)
                    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
                        double qv[ROWS], pv[ROWS];
                        apply_column<ROWS>(fxp, fyp, dgp, p, nx, ny, i, j0, qv, pv);
#pragma unroll
                        for (int u = 0; u < ROWS; ++u) {
                            const int j = j0 + u;
                            if (j < je) {
                                q[(long long)j * nx + i] = qv[u];
                                pq = fma(pv[u], qv[u], pq);
                            }
                        }
                    }
                if (!gsum(pq, pq)) return;
                if (!(pq > 0.0) || !isfinite(pq)) { status = PERKS_ERR_BREAKDOWN; break; }
                const double alpha = rr / pq;
                // x += alpha p, r -= alpha q, <r, r>
                double rn = 0.0;
                for (long long c0 = cb + threadIdx.x; c0 < ce; c0 += (long long)blockDim.x * LIN) {
                    double xv[LIN], rv[LIN], pv[LIN], qv[LIN];
#pragma unroll
                    for (int u = 0; u < LIN; ++u) {
                        const long long c = c0 + (long long)u * blockDim.x;
                        if (c < ce) { xv[u] = x[c]; rv[u] = r[c]; pv[u] = p[c]; qv[u] = q[c]; }
                    }
#pragma unroll
                    for (int u = 0; u < LIN; ++u) {
                        const long long c = c0 + (long long)u * blockDim.x;
                        if (c < ce) {
                            x[c] = fma(alpha, pv[u], xv[u]);
                            const double ri = fma(-alpha, qv[u], rv[u]);
                            r[c] = ri;
                            rn = fma(ri, ri, rn);
                        }
                    }
                }
                if (!gsum(rn, rn)) return;
                const double beta = rn / rr;
                // p = r + beta p
                for (long long c0 = cb + threadIdx.x; c0 < ce; c0 += (long long)blockDim.x * LIN) {
                    double rv[LIN], pv[LIN];
#pragma unroll
                    for (int u = 0; u < LIN; ++u) {
                        const long long c = c0 + (long long)u * blockDim.x;
                        if (c < ce) { rv[u] = r[c]; pv[u] = p[c]; }
                    }
#pragma unroll
                    for (int u = 0; u < LIN; ++u) {
                        const long long c = c0 + (long long)u * blockDim.x;
                        if (c < ce) p[c] = fma(beta, pv[u], rv[u]);
                    }
                }
                if (GROUP) {  // the next SpMV reads the neighbouring blocks' edge rows of p
                    if (!grid_barrier(a.gbar + g, C, epoch, a.err, a.timeout_ns)) return;
                } else {
                    __syncthreads();
                }
                rr = rn;
                ++it;
                if (rr <= tol2) { converged = true; break; }
            }
            if (status == PERKS_ERR_BREAKDOWN) break;
            double bdum = 0.0;
            const double rt = residual_pass<true, ROWS>(fxp, fyp, dgp, b, x, r, p, nx, ny, jb, je, bdum);
            if (!gsum(rt, rr)) return;
            if (rr <= tol2) { status = PERKS_OK; break; }
            if (!converged || restart >= a.max_restarts) break;
        }
        if (rank == 0 && threadIdx.x == 0) {
            a.iters[pb] = it;
            a.true_rel[pb] = bb > 0 ? sqrt(rr / bb) : sqrt(rr);
            a.status[pb] = status;
        }
        __syncthreads();
    }
}

// The default solver: the recurrence of perks_poisson_cg_kernel<.., 1, 1, ..>,
// cell by cell the same operations, laid out so that an iteration costs its
// ten fp64 operations per cell and little else (the FP64 pipe, 2 lanes per
// clock and SM, is the bound).
//   * A block's cells are one run, taken NT at a time: with a row of threads
//     per grid row, a 335-cell row left 177 of 512 lanes idle.
//   * Two exchanges per iteration (exchange_sum: sum and barrier in one),
//     where block sum, barrier, partial sums and another barrier took three
//     barriers: p of the two rows next to a block's own is updated by the
//     block itself, from the neighbours' r of those rows, which travels with
//     the <r, r> exchange.
//   * r stays in shared memory where a block's share fits; run_group prefers
//     group sizes that make it fit.
// 64 problems of 512^2, 24 iterations: 11.8 ms with the kernel above, 10.4
// here (the FP64 pipe's time is 6.7 ms); 16 problems of 83 x 368, 2.0 -> 0.5
// ms; 202 problems of 64 x 81 to 1e-8, 61 -> 28 ms.
template <int NT, bool GROUP>
__global__ void __launch_bounds__(NT, 2) perks_poisson_run_kernel(const __grid_constant__ PoissonArgs a) {
    extern __shared__ __align__(16) double poi_smem[];
    double *red = poi_smem;                       // reduce_scratch<NT>()
    double *rs = poi_smem + reduce_scratch<NT>();
    __shared__ int s_prob;
    const int nx = a.nx, ny = a.ny, tid = threadIdx.x;
    const long long n = a.n;
    const int C = GROUP ? a.group : 1;
    const int g = blockIdx.x / C, rank = blockIdx.x % C;
    int jb = 0, je = ny;
    if (GROUP) group_rows<1>(ny, C, rank, jb, je);
    const int cb = jb * nx, ce = je * nx;         // n fits an int: checked by the host
    const bool has_s = GROUP && jb > 0, has_n = GROUP && je < ny;
    double *hs = a.halo + (size_t)blockIdx.x * 2 * nx, *hn = hs + nx;
    unsigned round = 0;
    auto gsum = [&](double v, SumResult &out, auto &&post) -> bool {
        if constexpr (GROUP)
            return exchange_sum<NT>(a.slots + (size_t)g * 3 * C, C, rank, a.err, a.timeout_ns, round, v, red, out, post);
        block_sum4<NT>(v, red, out, post);
        return true;
    };
    auto plain = [](double, double &, int &) {};
    const int di = NT % nx, dj = NT / nx;         // from a thread's cell to its next one
    const int i0 = (cb + tid) % nx, j0 = (cb + tid) / nx;
    // f(c, i, j) for the block's cells c = j nx + i
    auto each_cell = [&](auto &&f) {
        for (int c = cb + tid, i = i0, j = j0; c < ce; c += NT) {
            f(c, i, j);
            i += di;
            j += dj;
            if (i >= nx) { i -= nx; ++j; }
        }
    };
    for (;;) {
        if constexpr (GROUP) {
            double pick = 0.0;
            if (rank == 0 && tid == 0) pick = (double)atomicAdd(a.queue, 1);
            SumResult got;
            if (!gsum(pick, got, plain)) return;
            if (tid == 0) s_prob = (int)got.total;
        } else {
            if (tid == 0) s_prob = atomicAdd(a.queue, 1);
        }
        __syncthreads();
        const int pb = s_prob;
        __syncthreads();
        if (pb >= a.nprob) break;
        const double *__restrict__ fxp = a.fx + (long long)pb * (nx + 1) * ny;
        const double *__restrict__ fyp = a.fy + (long long)pb * nx * (ny + 1);
        const double *__restrict__ dgp = a.dg + (long long)pb * n;
        const double *__restrict__ b = a.b + pb * n;
        double *x = a.x + pb * n, *rg = a.r + pb * n, *p = a.p + pb * n, *q = a.q + pb * n;
        double *r = a.on_chip ? rs - cb : rg;
        // (A v)_c; south / north: v of the cells below and above
        auto apply = [&](int c, int i, int j, double vc, double west, double east, double south, double north) -> double {
            const double fw = __ldg(fxp + c + j), fe = __ldg(fxp + c + j + 1);
            const double fs = __ldg(fyp + c), fn = __ldg(fyp + c + nx);
            double acc = __ldg(dgp + c) * vc;
            if (i > 0) acc = fma(-fw, west, acc);
            if (i + 1 < nx) acc = fma(-fe, east, acc);
            if (j > 0) acc = fma(-fs, south, acc);
            if (j + 1 < ny) acc = fma(-fn, north, acc);
            return acc;
        };
        // r = b - A x, p = r (x from global memory: the neighbours' rows too); the rows the neighbours read of r
        // go to global memory
        auto residual = [&](double &bb, double &rr) {
            each_cell([&](int c, int i, int j) {
                const double west = i > 0 ? __ldcg(x + c - 1) : 0.0, east = i + 1 < nx ? __ldcg(x + c + 1) : 0.0;
                const double south = j > 0 ? __ldcg(x + c - nx) : 0.0, north = j + 1 < ny ? __ldcg(x + c + nx) : 0.0;
                const double bv = __ldg(b + c);
                const double rv = bv - apply(c, i, j, __ldcg(x + c), west, east, south, north);
                r[c] = rv;
                p[c] = rv;
                if (a.on_chip && (j == jb || j == je - 1)) rg[c] = rv;
                bb = fma(bv, bv, bb);
                rr = fma(rv, rv, rr);
            });
        };
        // p of the neighbouring rows, from their r (start: p = r)
        auto halo = [&](bool start, double beta) {
            if (has_s)
                for (int i = tid; i < nx; i += NT) {
                    const double rv = __ldcg(rg + (long long)(jb - 1) * nx + i);
                    hs[i] = start ? rv : fma(beta, hs[i], rv);
                }
            if (has_n)
                for (int i = tid; i < nx; i += NT) {
                    const double rv = __ldcg(rg + (long long)je * nx + i);
                    hn[i] = start ? rv : fma(beta, hn[i], rv);
                }
        };
        SumResult sum;
        double bb = 0.0, rr = 0.0;
        residual(bb, rr);
        if (!gsum(bb, sum, plain)) return;
        bb = sum.total;
        const double tol2 = a.rtol * a.rtol * bb;
        auto small = [&](double t, double &, int &flag) { flag = t <= tol2; };
        if (!gsum(rr, sum, small)) return;
        rr = sum.total;
        int it = 0, status = PERKS_ERR_NOT_CONVERGED;
        for (int restart = 0;; ++restart) {
            if (sum.flag) { status = PERKS_OK; break; }
            halo(true, 0.0);
            __syncthreads();
            bool converged = false;
            while (it < a.max_iter) {
                // q = A p, <p, q>
                double pq = 0.0;
                each_cell([&](int c, int i, int j) {
                    const double pc = p[c];
                    const double west = i > 0 ? p[c - 1] : 0.0, east = i + 1 < nx ? p[c + 1] : 0.0;
                    const double south = j > jb ? p[c - nx] : has_s ? hs[i] : 0.0;
                    const double north = j + 1 < je ? p[c + nx] : has_n ? hn[i] : 0.0;
                    const double qc = apply(c, i, j, pc, west, east, south, north);
                    q[c] = qc;
                    pq = fma(pc, qc, pq);
                });
                if (!gsum(pq, sum, [&](double t, double &ratio, int &flag) {
                        flag = !(t > 0.0) || !isfinite(t);
                        ratio = rr / t;
                    }))
                    return;
                if (sum.flag) { status = PERKS_ERR_BREAKDOWN; break; }
                const double alpha = sum.ratio;
                // x += alpha p, r -= alpha q, <r, r>
                double rn = 0.0;
                for (int c = cb + tid; c < ce; c += NT) {
                    x[c] = fma(alpha, p[c], x[c]);
                    const double rv = fma(-alpha, q[c], r[c]);
                    r[c] = rv;
                    if (GROUP && a.on_chip && (c < cb + nx || c >= ce - nx)) rg[c] = rv;
                    rn = fma(rv, rv, rn);
                }
                if (!gsum(rn, sum, [&](double t, double &ratio, int &flag) { ratio = t / rr; flag = t <= tol2; }))
                    return;
                const double beta = sum.ratio;
                // p = r + beta p
                for (int c = cb + tid; c < ce; c += NT) p[c] = fma(beta, p[c], r[c]);
                halo(false, beta);
                __syncthreads();
                rr = sum.total;
                ++it;
                if (sum.flag) { converged = true; break; }
            }
            if (status == PERKS_ERR_BREAKDOWN) break;
            // true residual: the neighbours' x has to be there
            if (GROUP && !gsum(0.0, sum, plain)) return;
            double bdum = 0.0, rt = 0.0;
            residual(bdum, rt);
            if (!gsum(rt, sum, small)) return;
            rr = sum.total;
            if (sum.flag) { status = PERKS_OK; break; }
            if (!converged || restart >= a.max_restarts) break;
        }
        if (rank == 0 && tid == 0) {
            a.iters[pb] = it;
            a.true_rel[pb] = bb > 0 ? sqrt(rr / bb) : sqrt(rr);
            a.status[pb] = status;
        }
        __syncthreads();
    }
}

// x <- alpha x per problem with alpha = <x, b> / <x, A x>: of all multiples
// of the guess, the one closest to the solution in the A-norm (the energy
// norm CG minimises), so a warm start scaled this way starts CG no farther
// from the solution, in that norm, than a zero start.  Left unchanged where
// <x, A x> is not positive and finite (x = 0, for one).
template <int NT, int ROWS>
__global__ void __launch_bounds__(NT, 1) poisson_scale_guess_kernel(const __grid_constant__ PoissonArgs a,
                                                                   const double *__restrict__ bv,
                                                                   double *__restrict__ xv) {
    __shared__ double red[33];
    const int nx = a.nx, ny = a.ny;
    const long long n = a.n;
    for (int pb = blockIdx.x; pb < a.nprob; pb += gridDim.x) {
        const double *__restrict__ fxp = a.fx + (long long)pb * (nx + 1) * ny;
        const double *__restrict__ fyp = a.fy + (long long)pb * nx * (ny + 1);
        const double *__restrict__ dgp = a.dg + (long long)pb * n;
        const double *__restrict__ b = bv + pb * n;
        double *__restrict__ x = xv + pb * n;
        double xax = 0.0, xb = 0.0;
        for (int j0 = 0; j0 < ny; j0 += ROWS)
            for (int i = threadIdx.x; i < nx; i += blockDim.x) {
                double ax[ROWS], xc[ROWS];
                apply_column<ROWS>(fxp, fyp, dgp, x, nx, ny, i, j0, ax, xc);
#pragma unroll
                for (int u = 0; u < ROWS; ++u) {
                    const int j = j0 + u;
                    if (j < ny) {
                        xax = fma(xc[u], ax[u], xax);
                        xb = fma(xc[u], __ldg(b + (long long)j * nx + i), xb);
                    }
                }
            }
        xax = bsum(xax, red);
        xb = bsum(xb, red);
        if (xax > 0.0 && isfinite(xax) && isfinite(xb)) {
            const double alpha = xb / xax;
            for (long long c = threadIdx.x; c < n; c += blockDim.x) x[c] *= alpha;
        }
        __syncthreads();
    }
}

// y = A v for every problem (one launch; for tests).
__global__ void poisson_apply_kernel(const __grid_constant__ PoissonArgs a, const double *v, double *y) {
    const long long total = (long long)a.nprob * a.n;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long pb = t / a.n, c = t % a.n;
        const double *fxp = a.fx + pb * (a.nx + 1) * a.ny;
        const double *fyp = a.fy + pb * a.nx * (a.ny + 1);
        y[t] = apply_cell(fxp, fyp, a.dg + pb * a.n, v + pb * a.n, a.nx, a.ny, (int)(c % a.nx), (int)(c / a.nx));
    }
}

}  // namespace

struct perks_poisson {
    perks_context *ctx = nullptr;
    int device = 0;  // for destroy, which may come after the context is gone
    int nx = 0, ny = 0, nprob = 0;
    long long n = 0;
    double *fx = nullptr, *fy = nullptr, *dg = nullptr, *b = nullptr, *x = nullptr, *r = nullptr, *p = nullptr,
           *q = nullptr;
    int *queue = nullptr, *iters = nullptr, *status = nullptr;
    double *true_rel = nullptr;
    int block_threads = 512;  // 512 (one block per SM; measured faster) or 256 (two per SM)
    int rows_per_pass = 1;    // 1 (64 registers, 32 warps per SM; measured faster) or kRows (128, 16 warps)
    int group = 0;            // blocks per problem (0: automatic)
    unsigned long long *gbar = nullptr;
    int *gprob = nullptr;
    double *gpart = nullptr;
    double *slots = nullptr;  // [2 x SMs][3]: every group's rounds of exchange_sum
    double *halo = nullptr;   // [blocks of the automatic groups][2][nx]; none where a problem is one block's
    void *small = nullptr;    // the allocation of all of these but halo, and of the counters and results above
    DevError *err = nullptr;
    int max_groups = 0;
};

namespace {
void free_poisson(perks_poisson *P) {
    void *ptrs[] = {P->fx, P->fy, P->dg, P->b, P->x, P->r, P->p, P->q, P->small, P->halo};
    for (void *v : ptrs) if (v) cudaFree(v);
}

// Blocks per problem: as set, or automatically, for problems of 64K cells
// and more, 8 blocks (two per SM, one row per pass) or 4 (one per SM, 4
// rows per pass), and 1 for smaller problems (whose iterations are too short
// to pay for the group barriers).  A batch of 256 problems of 512^2 to 1e-8:
// 4 rows per pass 20.2 s with one block per problem, 16.4 s with 2, 15.9 s
// with 4 or 8; one row per pass 16.3 s with 2, 13.5 s with 4, 13.4 s with 8.
int effective_group(const perks_poisson *P) {
    if (P->group > 0) return P->group;
    if (P->n < 65536) return 1;
    return P->rows_per_pass == 1 ? 8 : 4;
}

PoissonArgs poisson_args(perks_poisson *P) {
    PoissonArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nx = P->nx; a.ny = P->ny; a.nprob = P->nprob; a.n = P->n;
    a.fx = P->fx; a.fy = P->fy; a.dg = P->dg; a.b = P->b; a.x = P->x; a.r = P->r; a.p = P->p; a.q = P->q;
    a.queue = P->queue; a.iters = P->iters; a.true_rel = P->true_rel; a.status = P->status;
    a.group = effective_group(P); a.gbar = P->gbar; a.gprob = P->gprob; a.gpart = P->gpart; a.err = P->err;
    a.slots = P->slots; a.halo = P->halo;
    a.timeout_ns = P->ctx->timeout_ns;
    return a;
}

constexpr int kRunThreads = 512;

// Dynamic shared memory of perks_poisson_run_kernel for groups of C blocks;
// r on chip if the largest share fits in half of an SM.
size_t run_smem(const perks_poisson *P, int C, int &on_chip) {
    const size_t base = sizeof(double) * reduce_scratch<kRunThreads>();
    const size_t rows = (size_t)(P->ny + C - 1) / C, r = sizeof(double) * rows * P->nx;
    const size_t most = (size_t)std::min(P->ctx->smem_optin, P->ctx->smem_per_sm / 2 - 1024) - 64;
    on_chip = base + r <= most;
    return on_chip ? base + r : base;
}

// Blocks per problem of perks_poisson_run_kernel.  The documented group where
// it gives every block at most 8192 cells and all of the batch runs at once;
// otherwise the group that finishes the batch in the fewest cycles by this
// model: a block's iteration takes 6.5 cycles per cell (10 fp64 operations, 2
// lanes per clock and SM, and the rest of an iteration; 7.5 with r in global
// memory), nearly twice that where two blocks share an SM, plus the exchanges;
// the batch takes ceil(problems / groups) of the longest iterations.  Measured
// (ms, the group picked / documented / others): 64 problems of 512^2, 24
// iterations, 19 blocks 10.2 / 8: 12.4 / 25: 10.5; 256 of 355 x 94, 7 blocks
// 3.1 / 1: 3.8 / 19: 4.9; 24 of 332 x 441, 12 blocks 1.4 / 8: 2.1 / 25: 1.4;
// 256 of 146 x 75, one block 1.56 / 2: 1.71.
int run_group(const perks_poisson *P) {
    const int doc = effective_group(P), slots = 2 * P->ctx->sm_count;
    if (P->n <= 8192 || (P->n <= 8192LL * doc && (long long)P->nprob * doc <= slots)) return doc;
    double best = 1e300;
    int bc = doc;
    for (int C = 1; C <= std::min(P->ny, 64); ++C) {
        const int groups = std::min(P->nprob, slots / C);
        if (groups < 1) break;
        int on_chip;
        run_smem(P, C, on_chip);
        const double m = (double)((P->ny + C - 1) / C) * P->nx;
        const double ex = 5000.0 + 3500.0 * std::log2((double)C);
        const double t = groups * C > P->ctx->sm_count ? (on_chip ? 12.3 : 14.5) * m + ex
                                                       : (on_chip ? 6.5 : 7.5) * m + 1.2 * ex;
        const double total = (double)((P->nprob + groups - 1) / groups) * t;
        if (total < best) { best = total; bc = C; }
    }
    return bc;
}
}  // namespace

extern "C" perks_status perks_poisson_create(perks_context *ctx, int32_t nx, int32_t ny, int32_t nprob,
                                             const double *k, int on_device, perks_poisson **out) {
    if (!ctx) return PERKS_ERR_INVALID_ARG;
    if (!out || !k || nx < 1 || ny < 1 || nprob < 1)
        return fail(ctx, PERKS_ERR_INVALID_ARG, "poisson_create: bad arguments");
    *out = nullptr;
    perks_status rc = use_device(ctx);
    if (rc) return rc;
    auto *P = new perks_poisson();
    P->ctx = ctx;
    P->device = ctx->device;
    P->nx = nx; P->ny = ny; P->nprob = nprob;
    P->n = (long long)nx * ny;
    const size_t vb = sizeof(double) * (size_t)P->n * nprob;
    const size_t fxb = sizeof(double) * (size_t)(nx + 1) * ny * nprob;
    const size_t fyb = sizeof(double) * (size_t)nx * (ny + 1) * nprob;
    double *kd = nullptr;
    cudaError_t e = cudaSuccess;
    void **bufs[] = {(void **)&P->b, (void **)&P->x, (void **)&P->r, (void **)&P->p, (void **)&P->q, (void **)&P->dg};
    for (void **bp : bufs) if (e == cudaSuccess) e = cudaMalloc(bp, vb);
    if (e == cudaSuccess) e = cudaMalloc(&P->fx, fxb);
    if (e == cudaSuccess) e = cudaMalloc(&P->fy, fyb);
    if (e == cudaSuccess && !on_device) {
        e = cudaMalloc(&kd, vb);
        if (e == cudaSuccess) e = cudaMemcpy(kd, k, vb, cudaMemcpyHostToDevice);
    }
    // One allocation for counters, results and sums
    P->max_groups = 2 * ctx->sm_count;  // at most two blocks per SM
    const size_t mg = P->max_groups, np = nprob;
    size_t total = 0;
    auto part = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 511) & ~size_t(511);
        return at;
    };
    const size_t queue = part(sizeof(int)), iters = part(sizeof(int) * np), status = part(sizeof(int) * np),
                 rel = part(sizeof(double) * np), gbar = part(sizeof(unsigned long long) * mg),
                 gprob = part(sizeof(int) * mg), gpart = part(sizeof(double) * 2 * kPoiMaxGroup * mg),
                 slots = part(sizeof(double) * 3 * mg), err = part(sizeof(DevError));
    if (e == cudaSuccess) e = cudaMalloc(&P->small, total);
    if (e == cudaSuccess) {
        char *at = static_cast<char *>(P->small);
        P->queue = reinterpret_cast<int *>(at + queue);
        P->iters = reinterpret_cast<int *>(at + iters);
        P->status = reinterpret_cast<int *>(at + status);
        P->true_rel = reinterpret_cast<double *>(at + rel);
        P->gbar = reinterpret_cast<unsigned long long *>(at + gbar);
        P->gprob = reinterpret_cast<int *>(at + gprob);
        P->gpart = reinterpret_cast<double *>(at + gpart);
        P->slots = reinterpret_cast<double *>(at + slots);
        P->err = reinterpret_cast<DevError *>(at + err);
        // halo rows of the blocks that run_group puts to work (two per block: at most two vectors' worth where every block
        // has a row; two rows for each of 2 x SMs blocks took 10 GB for one problem of 1 x 2^21).  A batch that leaves no
        // room for them is solved by the kernel without them.
        const int C = P->n < (1LL << 30) ? run_group(P) : 1;
        if (C > 1 && cudaMalloc(&P->halo, sizeof(double) * 2 * nx * std::min(nprob, P->max_groups / C) * C) != cudaSuccess) {
            P->halo = nullptr;
            (void)cudaGetLastError();
        }
    }
    if (e != cudaSuccess) {
        if (kd) cudaFree(kd);
        free_poisson(P);
        delete P;
        return cuda_fail(ctx, e, "poisson_create");
    }
    poisson_faces_kernel<<<1024, 256>>>(on_device ? k : kd, nx, ny, P->n * nprob, P->fx, P->fy);
    poisson_diag_kernel<<<1024, 256>>>(P->fx, P->fy, nx, ny, P->n * nprob, P->dg);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (kd) cudaFree(kd);
    if (e != cudaSuccess) { free_poisson(P); delete P; return cuda_fail(ctx, e, "poisson_create: faces"); }
    *out = P;
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_destroy(perks_poisson *P) {
    if (!P) return PERKS_OK;
    cudaSetDevice(P->device);
    free_poisson(P);
    delete P;
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_apply(perks_poisson *P, const double *v, double *y, perks_stream stream) {
    if (!P) return PERKS_ERR_INVALID_ARG;
    if (!v || !y) return fail(P->ctx, PERKS_ERR_INVALID_ARG, "poisson_apply: NULL vector");
    perks_status rc = use_device(P->ctx);
    if (rc) return rc;
    poisson_apply_kernel<<<1024, 256, 0, (cudaStream_t)stream>>>(poisson_args(P), v, y);
    PERKS_CUDA(P->ctx, cudaGetLastError());
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_scale_guess(perks_poisson *P, const double *b, double *x,
                                                  perks_stream stream) {
    if (!P) return PERKS_ERR_INVALID_ARG;
    if (!b || !x) return fail(P->ctx, PERKS_ERR_INVALID_ARG, "poisson_scale_guess: NULL vector");
    perks_status rc = use_device(P->ctx);
    if (rc) return rc;
    const int grid = std::max(1, std::min(P->nprob, P->ctx->sm_count));
    poisson_scale_guess_kernel<512, kRows><<<grid, 512, 0, (cudaStream_t)stream>>>(poisson_args(P), b, x);
    PERKS_CUDA(P->ctx, cudaGetLastError());
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_solve(perks_poisson *P, const double *b, double *x, double rtol,
                                            int32_t max_iter, perks_stream stream, perks_poisson_stats *stats) {
    if (!P) return PERKS_ERR_INVALID_ARG;
    perks_context *ctx = P->ctx;
    if (!b || !x || !(rtol >= 0) || max_iter < 0) return fail(ctx, PERKS_ERR_INVALID_ARG, "poisson_solve: bad arguments");
    perks_status rc = use_device(ctx);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t vb = sizeof(double) * (size_t)P->n * P->nprob;
    PERKS_CUDA(ctx, cudaMemcpyAsync(P->b, b, vb, cudaMemcpyDeviceToDevice, s));
    PERKS_CUDA(ctx, cudaMemcpyAsync(P->x, x, vb, cudaMemcpyDeviceToDevice, s));
    PERKS_CUDA(ctx, cudaMemsetAsync(P->queue, 0, sizeof(int), s));
    PoissonArgs a = poisson_args(P);
    a.rtol = rtol;
    a.max_iter = max_iter;
    a.max_restarts = 8;
    // group size and rows per pass by default: the run kernel
    const int own_group = run_group(P);
    const bool run = P->group == 0 && P->rows_per_pass == 1 && P->n < (1LL << 30) && (own_group == 1 || P->halo);
    const int C = run ? own_group : effective_group(P);
    const bool grouped = C > 1;
    const void *kern;
    size_t smem = 0;
    int threads = P->block_threads;
    a.group = C;
    if (run) {
        kern = grouped ? (const void *)perks_poisson_run_kernel<kRunThreads, true>
                       : (const void *)perks_poisson_run_kernel<kRunThreads, false>;
        threads = kRunThreads;
        smem = run_smem(P, C, a.on_chip);
        int budget = 0;
        rc = smem_optin(ctx, kern, &budget);
        if (rc) return rc;
        if (smem > (size_t)budget) {
            a.on_chip = 0;
            smem = sizeof(double) * reduce_scratch<kRunThreads>();
        }
    } else if (P->rows_per_pass == 1)  // two 512-thread blocks per SM, one row per pass
        kern = grouped ? (const void *)perks_poisson_cg_kernel<512, 2, 1, 1, true>
                       : (const void *)perks_poisson_cg_kernel<512, 2, 1, 1, false>;
    else if (P->block_threads == 512)
        kern = grouped ? (const void *)perks_poisson_cg_kernel<512, 1, kRows, kLin, true>
                       : (const void *)perks_poisson_cg_kernel<512, 1, kRows, kLin, false>;
    else
        kern = grouped ? (const void *)perks_poisson_cg_kernel<kPoiThreads, 2, kRows, kLin, true>
                       : (const void *)perks_poisson_cg_kernel<kPoiThreads, 2, kRows, kLin, false>;
    int per_sm = 0;
    PERKS_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (run) per_sm = std::min(per_sm, 2);
    if (per_sm < 1) return fail(ctx, PERKS_ERR_LAUNCH_TOO_LARGE, "poisson_solve: kernel cannot be resident");
    void *kargs[] = {(void *)&a};
    int grid;
    if (!grouped) {
        grid = std::max(1, std::min(P->nprob, per_sm * ctx->sm_count));
        PERKS_CUDA(ctx, cudaLaunchKernel(kern, dim3(grid), dim3(threads), kargs, smem, s));
    } else {
        // groups wait on one another's blocks: every block resident (cooperative launch)
        const int groups = std::min({P->nprob, per_sm * ctx->sm_count / C, P->max_groups});
        if (groups < 1) return fail(ctx, PERKS_ERR_LAUNCH_TOO_LARGE, "poisson_solve: group larger than the GPU");
        grid = groups * C;
        PERKS_CUDA(ctx, cudaMemsetAsync(P->gbar, 0, sizeof(unsigned long long) * groups, s));
        PERKS_CUDA(ctx, cudaMemsetAsync(P->err, 0, sizeof(DevError), s));
        if (run) PERKS_CUDA(ctx, cudaMemsetAsync(P->slots, 0xff, sizeof(double) * 3 * grid, s));
        PERKS_CUDA(ctx, cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(threads), kargs, smem, s));
    }
    PERKS_CUDA(ctx, cudaMemcpyAsync(x, P->x, vb, cudaMemcpyDeviceToDevice, s));
    if (!stats) return PERKS_OK;
    PERKS_CUDA(ctx, cudaStreamSynchronize(s));
    int32_t *it_out = stats->iterations;
    double *tr_out = stats->true_rel_residual;
    const int32_t cap = stats->capacity;
    std::memset(stats, 0, sizeof(*stats));
    stats->iterations = it_out;
    stats->true_rel_residual = tr_out;
    stats->capacity = cap;
    stats->problems = P->nprob;
    stats->grid_blocks = grid;
    int *it = new int[P->nprob];
    int *st = new int[P->nprob];
    double *tr = new double[P->nprob];
    cudaMemcpy(it, P->iters, sizeof(int) * P->nprob, cudaMemcpyDeviceToHost);
    cudaMemcpy(st, P->status, sizeof(int) * P->nprob, cudaMemcpyDeviceToHost);
    cudaMemcpy(tr, P->true_rel, sizeof(double) * P->nprob, cudaMemcpyDeviceToHost);
    perks_status worst = PERKS_OK;
    long long sum_it = 0;
    for (int i = 0; i < P->nprob; ++i) {
        sum_it += it[i];
        stats->max_iterations = std::max(stats->max_iterations, it[i]);
        stats->max_true_rel_residual = std::max(stats->max_true_rel_residual, tr[i]);
        if (st[i] != PERKS_OK && worst == PERKS_OK) worst = st[i];
        if (stats->iterations && i < stats->capacity) {
            stats->iterations[i] = it[i];
            if (stats->true_rel_residual) stats->true_rel_residual[i] = tr[i];
        }
    }
    stats->mean_iterations = (double)sum_it / P->nprob;
    delete[] it;
    delete[] st;
    delete[] tr;
    if (grouped) {
        DevError de{};
        PERKS_CUDA(ctx, cudaMemcpy(&de, P->err, sizeof(DevError), cudaMemcpyDeviceToHost));
        if (de.code != 0)
            return fail(ctx, de.code, "poisson_solve: a block group's barrier gave up (block %d)", de.block);
    }
    if (worst != PERKS_OK) return fail(ctx, worst, "poisson_solve: a problem did not converge (status %d)", worst);
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_set_group(perks_poisson *P, int32_t blocks) {
    if (!P) return PERKS_ERR_INVALID_ARG;
    if (blocks != 0 && blocks != 1 && blocks != 2 && blocks != 4 && blocks != 8)
        return fail(P->ctx, PERKS_ERR_INVALID_ARG, "poisson_set_group: 0 (automatic), 1, 2, 4 or 8 blocks");
    P->group = blocks;
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_set_rows_per_pass(perks_poisson *P, int32_t rows) {
    if (!P) return PERKS_ERR_INVALID_ARG;
    if (rows != 1 && rows != kRows)
        return fail(P->ctx, PERKS_ERR_INVALID_ARG, "poisson_set_rows_per_pass: 1 or %d", kRows);
    P->rows_per_pass = rows;
    return PERKS_OK;
}

extern "C" perks_status perks_poisson_set_block_threads(perks_poisson *P, int32_t threads) {
    if (!P) return PERKS_ERR_INVALID_ARG;
    if (threads != 256 && threads != 512)
        return fail(P->ctx, PERKS_ERR_INVALID_ARG, "poisson_set_block_threads: 256 or 512");
    P->block_threads = threads;
    return PERKS_OK;
}
