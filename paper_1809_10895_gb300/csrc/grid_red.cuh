// grid_red.cuh -- barriers and reductions over the blocks of a running
// cooperative kernel.
//
// The barrier is one counter, as in CUDA's cooperative-groups grid barrier: block
// 0 adds 2^31 - (blocks - 1) and the others 1, so that the last arrival flips
// the top bit, and nothing is reset between launches.  Here a block arrives with
// an acquire-release atomic and polls with acquire loads, a bounded number of
// times (1.2 us over 152 blocks; adding __threadfence() on
// both sides costs 0.1 us, an all-gather in which every block polls every
// block's slot costs 2-3 us more, and clusters in front of it 0.4 us).  For a
// reduction the blocks publish partials before arriving and each folds all of
// them, in the same order, after it: results are bit-identical in every block.
// Partials alternate between two buffers: a block writes one again only two
// rounds later, when every block has passed the round between.  Each value is
// summed by a warp of its own, on the integer pipes (ix_sum.cuh).  Waits are
// bounded: one that runs out sets the fault flag and the caller's abort flag.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ix_sum.cuh"
#include "rf_reduce.cuh"

namespace rf {

constexpr int GR_NV = 4;             // values of one reduction at most
constexpr int GR_BLOCKS = 1216;      // blocks at most (eight on each of 152 SMs)
constexpr size_t GR_BYTES = 256 + sizeof(double) * 2 * GR_NV * GR_BLOCKS;   // counter, partials
constexpr int GR_POLLS = 1 << 22;    // polls of a wait: seconds

#ifdef __CUDACC__
struct GridRed {
    unsigned int *bar;
    double *part;            // [2][GR_NV][GR_BLOCKS]
    int *fault;
    int polls;
    int buf;
};

__device__ __forceinline__ GridRed grid_red_begin(void *mem, int *fault, int wait_tries)
{
    GridRed R;
    R.bar = static_cast<unsigned int *>(mem);
    R.part = reinterpret_cast<double *>(static_cast<char *>(mem) + 256);
    R.fault = fault;
    // a test limit replaces the default; negative: a single non-blocking test
    R.polls = wait_tries > 0 ? wait_tries : wait_tries < 0 ? 1 : GR_POLLS;
    R.buf = 0;
    return R;
}

// One thread, after a block barrier: arrive and wait for all blocks; false
// when the wait ran out.  Follow with a block barrier.
__device__ __forceinline__ bool grid_red_wait(const GridRed &R)
{
    const unsigned int inc = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1) : 1u;
    unsigned int old, now;
    asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], %2;" : "=r"(old) : "l"(R.bar), "r"(inc) : "memory");
    int polls = 0;
    do {
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(now) : "l"(R.bar) : "memory");
    } while (!((now ^ old) & 0x80000000u) && ++polls < R.polls);
    if (polls < R.polls) return true;
    *R.fault = 1;
    return false;
}

// Maximum of non-negative doubles (and of the all-ones pattern, the largest)
// by their bits.
struct OpMaxBits {
    __device__ static double id() { return 0.0; }
    __device__ static double op(double a, double b)
    {
        return (unsigned long long)__double_as_longlong(a) > (unsigned long long)__double_as_longlong(b) ? a : b;
    }
    __device__ static double warp(double v)
    {
        return __longlong_as_double((long long)ix_warp_max((uint64_t)__double_as_longlong(v)));
    }
};

struct OpIxSum {
    __device__ static double id() { return 0.0; }
    __device__ static double op(double a, double b) { return a + b; }
    __device__ static double warp(double v) { return ix_double(ix_warp_sum(v)); }
};

// Fold value i of the blocks' partials (whole warp; the total on every lane).
template <class Op>
__device__ __forceinline__ double grid_red_fold(const double *part, int i)
{
    const double *src = part + i * GR_BLOCKS;
    double t = Op::id();
    for (int b = threadIdx.x & 31; b < (int)gridDim.x; b += 32) t = Op::op(t, __ldcg(src + b));
    return Op::warp(t);
}

// Block totals (block(i) by warp i < NV, on lane 0 at least) to grid totals in
// tot[0..NV), then fin() on thread 0; everything is visible to the block on
// return.  All threads call it.  abort is a shared flag.
template <class Op, int NV, class Block, class Fin>
__device__ __forceinline__ bool grid_red(GridRed &R, double *tot, int *abort, Block block, Fin fin)
{
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *part = R.part + (size_t)R.buf * GR_NV * GR_BLOCKS;
    if (wid < NV) {
        const double t = block(wid);
        if (lane == 0) {
            if (gridDim.x == 1) tot[wid] = t;
            else part[wid * GR_BLOCKS + blockIdx.x] = t;
        }
    }
    if (NV > 1) __syncthreads();
    if (gridDim.x > 1) {
        if (threadIdx.x == 0 && !grid_red_wait(R)) *abort = 1;
        if (NV > 1) __syncthreads();
        else __syncwarp();
        if (wid < NV) {
            const double t = grid_red_fold<Op>(part, wid);
            if (lane == 0) tot[wid] = t;
        }
        if (NV > 1) __syncthreads();
        R.buf ^= 1;
    }
    if (threadIdx.x == 0) fin();
    __syncthreads();
    return !*abort;
}

// Sum NV FP64 thread values of a block of eight warps over the grid; the rest
// as in grid_red.
template <int NV, class Fin>
__device__ __forceinline__ bool grid_red_sum(GridRed &R, IxSum (*part)[8], double *tot, int *abort,
                                             const double (&v)[NV], Fin fin)
{
#pragma unroll
    for (int i = 0; i < NV; i++) {
        const IxSum w = ix_warp_sum(v[i]);
        if ((threadIdx.x & 31) == 0) part[i][threadIdx.x >> 5] = w;
    }
    __syncthreads();
    return grid_red<OpIxSum, NV>(
        R, tot, abort,
        [&](int i) {
            const int lane = threadIdx.x & 31;
            return ix_fold8(lane < 8 ? part[i][lane] : IxSum{0, {0, 0, 0}});
        },
        fin);
}
#endif

}  // namespace rf
