// Device helpers shared by the persistent kernels: asynchronous global->shared
// copies, the bounded grid barrier and small numeric utilities.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include "perks.h"

namespace perks {

// ------------------------------------------------------------------ storage

template <typename T> struct AccOf { using type = float; };
template <> struct AccOf<double> { using type = double; };

template <typename T> __device__ __forceinline__ typename AccOf<T>::type to_acc(T v) {
    return static_cast<typename AccOf<T>::type>(v);
}
template <> __device__ __forceinline__ float to_acc<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}
template <typename T> __device__ __forceinline__ T from_acc(typename AccOf<T>::type v) {
    return static_cast<T>(v);
}
template <> __device__ __forceinline__ __nv_bfloat16 from_acc<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}

// ------------------------------------------------------------- async copies

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// cp.async of one 4-, 8- or 16-byte element: 16-byte copies bypass L1
// (.cg); smaller ones can only use .ca.
template <int BYTES>
__device__ __forceinline__ void cp_async(void *smem_dst, const void *gmem_src) {
    static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async size");
    if constexpr (BYTES == 16) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(smem_dst)),
                     "l"(gmem_src)
                     : "memory");
    } else {
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_u32(smem_dst)),
                     "l"(gmem_src), "n"(BYTES)
                     : "memory");
    }
}

__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// ------------------------------------------------------------- grid barrier

__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_relaxed_gpu(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_gpu_add(unsigned long long *p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Device-side error record: word 0 = error code (0 = none), word 1 = the
// block that first failed, word 2 = the barrier epoch at which it failed.
struct DevError {
    int code;
    int block;
    int epoch;
    int pad;
};

__device__ __forceinline__ unsigned long long ld_relaxed_gpu_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void fence_acquire_gpu() {
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

// Grid-wide barrier over `nblocks` co-resident blocks (a cooperative launch
// guarantees co-residency).  `counter` is a monotone 64-bit arrival count,
// zeroed before the launch; the e-th barrier (e = 1, 2, ...) completes when
// the count reaches e * nblocks.  After __syncthreads, thread 0 arrives with
// a gpu-scope release reduction (cumulative over the block's writes ordered
// before it by the bar.sync), polls with relaxed loads and, once the count is
// reached, issues one acquire fence; the closing __syncthreads orders every
// thread's later accesses after it.  No full (sc) fence is needed.  The wait
// is bounded by `timeout_ns` of %globaltimer: on expiry (or when another
// block has already failed) the block records BARRIER_TIMEOUT and the call
// returns false in every thread, so the caller leaves its loop and the whole
// grid winds down without hanging.
__device__ __forceinline__ bool grid_barrier(unsigned long long *counter, unsigned nblocks,
                                             unsigned long long &epoch, DevError *err,
                                             long long timeout_ns) {
    __shared__ int s_fail;
    __syncthreads();
    if (threadIdx.x == 0) {
        int fail = 0;
        ++epoch;
        const unsigned long long target = epoch * (unsigned long long)nblocks;
        red_release_gpu_add(counter, 1ull);
        if (ld_relaxed_gpu_u64(counter) < target) {
            const uint64_t t0 = global_timer_ns();
            unsigned spins = 0;
            for (;;) {
                if (timeout_ns == 0) {  // test hook: give up at the first wait
                    if (atomicCAS(&err->code, 0, PERKS_ERR_BARRIER_TIMEOUT) == 0) {
                        err->block = blockIdx.x;
                        err->epoch = (int)epoch;
                    }
                    fail = 1;
                    break;
                }
                if (ld_relaxed_gpu_u64(counter) >= target) break;
                if ((++spins & 255u) == 0) {
                    if (ld_relaxed_gpu(&err->code) != 0) { fail = 1; break; }
                    if ((long long)(global_timer_ns() - t0) > timeout_ns) {
                        if (atomicCAS(&err->code, 0, PERKS_ERR_BARRIER_TIMEOUT) == 0) {
                            err->block = blockIdx.x;
                            err->epoch = (int)epoch;
                        }
                        fail = 1;
                        break;
                    }
                }
            }
        }
        fence_acquire_gpu();
        s_fail = fail;
    }
    __syncthreads();
    return s_fail == 0;
}

// ----------------------------------------------------------- warp reductions

template <typename T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------------ waits of whole warps
//
// Called by a full warp: polls until ready() holds in every lane, bounded as
// grid_barrier's wait (false, and the error recorded, on expiry).  One loop
// for the warp: lanes that poll words of their own in loops of their own leave
// them one by one, and what follows (an acquire fence among it) runs once per
// lane.
template <class READY>
__device__ __forceinline__ bool warp_wait(READY &&ready, DevError *err, long long timeout_ns, int epoch) {
    if (__all_sync(0xffffffffu, ready())) return true;
    const uint64_t t0 = global_timer_ns();
    unsigned spins = 0;
    for (;;) {
        bool give_up = timeout_ns == 0;  // test hook: give up at the first wait
        if (!give_up) {
            if (__all_sync(0xffffffffu, ready())) return true;
            if ((++spins & 255u) == 0) {
                if (__any_sync(0xffffffffu, ld_relaxed_gpu(&err->code) != 0)) return false;
                give_up = __any_sync(0xffffffffu, (long long)(global_timer_ns() - t0) > timeout_ns);
            }
        }
        if (give_up) {
            if ((threadIdx.x & 31) == 0 && atomicCAS(&err->code, 0, PERKS_ERR_BARRIER_TIMEOUT) == 0) {
                err->block = blockIdx.x;
                err->epoch = epoch;
            }
            return false;
        }
    }
}

// ----------------------------------------------------- sums over many blocks

// Sum of s[0..n), n <= NT; valid in thread 0.  The FP64 pipe takes a quarter
// of an SM 64 cycles per warp addition, so four warps add the values four at a
// time, instead of every warp its own: with two blocks of 512 threads per SM a
// butterfly in all 32 warps takes 2560 cycles, this 500.
template <int NT> __host__ __device__ constexpr int reduce_scratch() { return NT + 16; }  // doubles

template <int NT> __device__ __forceinline__ double reduce4(double *s, int n) {
    static_assert(NT == 512, "four warps, four values each");
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    double *part = s + NT;
    if (w < 4) {
        const int i = w * 32 + l;
        double t = i < n ? s[i] : 0.0;
        const double t1 = i + 128 < n ? s[i + 128] : 0.0;
        if (n > 256) {
            const double t2 = i + 256 < n ? s[i + 256] : 0.0, t3 = i + 384 < n ? s[i + 384] : 0.0;
            t = (t + t1) + (t2 + t3);
        } else if (n > 128) {
            t += t1;
        }
        if (n > 32 || w == 0) t = warp_sum(t);
        if (l == 0) part[w] = t;
    }
    __syncthreads();
    return threadIdx.x == 0 ? (part[0] + part[1]) + (part[2] + part[3]) : 0.0;
}

// The same sum of the threads' v, added in the same order, in 1 KB of scratch
// (128 doubles) for five more block barriers: for kernels that keep their
// data in shared memory up to its limit.
constexpr size_t kSmallReduceBytes = 128 * sizeof(double);

template <int NT> __device__ __forceinline__ double reduce4_small(double v, double *s) {
    static_assert(NT == 512, "four quarters of 128 values");
    const int quarter = threadIdx.x >> 7, i = threadIdx.x & 127;
    __syncthreads();  // the last sum's result has been read
    if (quarter == 1) s[i] = v;
    __syncthreads();
    if (quarter == 0) v += s[i];
    __syncthreads();
    if (quarter == 3) s[i] = v;
    __syncthreads();
    if (quarter == 2) s[i] += v;
    __syncthreads();
    if (quarter == 0) v = warp_sum(v + s[i]);
    __syncthreads();
    if (quarter == 0 && (i & 31) == 0) s[i >> 5] = v;
    __syncthreads();
    return threadIdx.x == 0 ? (s[0] + s[1]) + (s[2] + s[3]) : 0.0;
}

// What every thread of a block needs from a sum: the sum, a ratio formed from
// it and a decision.  Thread 0 forms them and hands them out: an fp64 division
// is some 15 operations of the FP64 pipe, and 32 warps forming the same one
// keep the pipe of an SM busy for 8000 cycles.
struct SumResult {
    double total, ratio;
    int flag;
};

// `total` of thread 0, with post(total, ratio, flag) applied by it, in every
// thread, by way of at[0..2].
template <class POST>
__device__ __forceinline__ void hand_out(double total, double *at, SumResult &out, POST &&post) {
    int *flag = reinterpret_cast<int *>(at + 2);
    if (threadIdx.x == 0) {
        double ratio = 0.0;
        int f = 0;
        post(total, ratio, f);
        at[0] = total;
        at[1] = ratio;
        *flag = f;
    }
    __syncthreads();
    out.total = at[0];
    out.ratio = at[1];
    out.flag = *flag;
}

// Sum of s[0..n) with post(total, ratio, flag) applied by thread 0, in every
// thread.  s[] is complete (a block barrier lies behind its last store).
template <int NT, class POST>
__device__ __forceinline__ void finish_sum(double *s, int n, SumResult &out, POST &&post) {
    hand_out(reduce4<NT>(s, n), s + NT + 8, out, post);
}

// Sum of v over the threads of one block.
template <int NT, class POST>
__device__ __forceinline__ void block_sum4(double v, double *s, SumResult &out, POST &&post) {
    s[threadIdx.x] = v;
    __syncthreads();
    finish_sum<NT>(s, NT, out, post);
}

// Sum of v over the threads of the whole grid and a grid barrier: the blocks'
// sums go to slots[parity][block], and after the barrier every block adds all
// of them in the same order.  (Spinning on the slots themselves saves a trip
// for a few blocks -- exchange_sum -- but with 304 blocks the polls of 304
// words by 304 blocks queue at the L2: 9.5 us a sum.)
// SMALL: s holds kSmallReduceBytes (G at most NT), otherwise reduce_scratch.
template <int NT, bool SMALL, class POST>
__device__ __forceinline__ bool grid_sum4(double *slots, int G, unsigned long long *bar, unsigned long long &epoch,
                                          DevError *err, long long timeout_ns, unsigned &round, double v, double *s,
                                          SumResult &out, POST &&post) {
    double *row = slots + (size_t)(round & 1) * G;
    ++round;
    double sum;
    if constexpr (SMALL) {
        sum = reduce4_small<NT>(v, s);
    } else {
        s[threadIdx.x] = v;
        __syncthreads();
        sum = reduce4<NT>(s, NT);
    }
    if (threadIdx.x == 0) __stcg(row + blockIdx.x, sum);
    if (!grid_barrier(bar, G, epoch, err, timeout_ns)) return false;
    double mine = 0.0;
    for (int i = threadIdx.x; i < G; i += NT) mine = i < NT ? __ldcg(row + i) : mine + __ldcg(row + i);
    if constexpr (SMALL) {
        hand_out(reduce4_small<NT>(mine, s), s + 8, out, post);
    } else {
        s[threadIdx.x] = mine;
        __syncthreads();
        finish_sum<NT>(s, G < NT ? G : NT, out, post);
    }
    return true;
}

// The same among the G blocks (a few dozen at most) of a group, in one
// exchange.  A block publishes its sum in its slot and reads every other
// block's slot until all are there: one trip out and one back, where an
// arrival count, a spin on it and a read of the sums take three.  `slots`
// holds three rounds of G values, all empty before the launch; an empty slot
// holds a NaN pattern no arithmetic gives.  Round e uses row e % 3.  Before
// publishing in it a block empties its slot of the next row, last read in
// round e - 2: every block has left that round, since all have published
// round e - 1; and whoever reads the next row has seen this round's
// publication, which the emptying precedes.  Waits are bounded as in
// grid_barrier; false in every thread when one gave up.
constexpr unsigned long long kSlotEmpty = 0xffffffffffffffffull;

template <int NT, class POST>
__device__ __forceinline__ bool exchange_sum(double *slots, int G, int rank, DevError *err, long long timeout_ns,
                                             unsigned &round, double v, double *s, SumResult &out, POST &&post) {
    const int tid = threadIdx.x;
    double *row = slots + (size_t)(round % 3) * G, *next = slots + (size_t)((round + 1) % 3) * G;
    ++round;
    s[tid] = v;
    __syncthreads();  // ... and every thread's writes come before the publication below
    const double sum = reduce4<NT>(s, NT);
    if (tid == 0) {
        unsigned long long bits = __double_as_longlong(sum);
        if (bits == kSlotEmpty) bits = 0x7ff8000000000000ull;
        reinterpret_cast<volatile unsigned long long *>(next)[rank] = kSlotEmpty;
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(row + rank), "l"(bits) : "memory");
    }
    int fail = 0;
    double mine = 0.0;
    if ((tid & ~31) < G) {  // whole warps
        const unsigned long long *slot = reinterpret_cast<const unsigned long long *>(row + tid);
        unsigned long long bits = 0;
        fail = !warp_wait([&]() { return tid >= G || (bits = ld_relaxed_gpu_u64(slot)) != kSlotEmpty; }, err, timeout_ns,
                          (int)round);
        if (tid < G) mine = __longlong_as_double(bits);
        fence_acquire_gpu();
    }
    s[tid] = mine;  // read by nobody since the barrier inside reduce4
    if (__syncthreads_or(fail)) return false;
    finish_sum<NT>(s, G, out, post);
    return true;
}

}  // namespace perks
