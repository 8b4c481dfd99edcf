// ff_adjoint.cu -- discrete adjoint of the RK4 / Euler integrator (not part of
// the paper): gradients of a loss of the final states with respect to the
// initial states and the parameters, by reverse sweeps over checkpointed chunks.
//
// One thread per particle walks the chunks in reverse with the adjoint state
// lambda = dL/dx in registers.  A chunk of L <= M*M steps is recomputed from its
// checkpoint twice (once when L <= M): once to place sub-checkpoints every M steps (local memory),
// then per sub-segment (in reverse) to put its <= M states in a shared-memory
// column per thread, which the reverse RK4 steps consume from
// last to first.  The 15-dimensional system is recomputed once per chunk into a
// per-thread scratch area in global memory instead (ff_adjoint_hh3.cu).  Parameter gradients are
// summed per particle in FP32 within a chunk, added to FP64 per chunk, and
// reduced over particles through per-block FP64 partials in fixed order.
//
// This unit holds the dispatch over systems and the fixed-order reductions; the
// kernels themselves are instantiated per family in ff_adjoint_lorenz.cu,
// ff_adjoint_hh3.cu, ff_adjoint_small.cu and ff_adjoint_linear.cu (device code in
// ff_adjoint_impl.cuh).
#include <cstdint>
#include <cuda_runtime.h>

#include "ff.h"
#include "ff_adjoint.h"

namespace ff {

// Column q of the partial rows [r0, r1), summed by one block in a fixed order: thread t adds
// rows r0 + t, r0 + t + 512, ... and the threads' sums meet in a tree over lanes, then warps.
// A chain of one dependent load and FP64 addition per row costs about 0.1 us each, which one
// thread walking all rows paid 1,216 times on a 1M-particle Lorenz sweep (130 us, 4% of the
// training step; 51 us of the 64k-particle HH x 3 one); split over a block both take 5-6 us.
constexpr int kReduceBlock = 512;
__device__ __forceinline__ void block_column_sum(const double* partial, int64_t r0, int64_t r1, int np_stride, int q,
                                                 double* out) {
    __shared__ double warp_sum[kReduceBlock / 32];
    double s = 0.0;
    for (int64_t r = r0 + threadIdx.x; r < r1; r += kReduceBlock) s += partial[r * np_stride + q];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kReduceBlock / 32; ++w) s += warp_sum[w];
        *out = s;
    }
}

// dp[m * np_stride + q] = sum over rows [row0[m], row0[m + 1]) of partial[row][q]: one block per (m, q).
__global__ void __launch_bounds__(kReduceBlock) reduce_member_rows_kernel(const double* partial, const int* row0,
                                                                          int np, int np_stride, double* dp) {
    const int m = blockIdx.x / np, q = blockIdx.x % np;
    block_column_sum(partial, row0[m], row0[m + 1], np_stride, q, dp + (int64_t)m * np_stride + q);
}

// Sum of the per-block (or per-warp) partials: one block per parameter.
__global__ void __launch_bounds__(kReduceBlock) reduce_partials_kernel(const double* partial, int64_t rows,
                                                                       int np_stride, double* out) {
    block_column_sum(partial, 0, rows, np_stride, blockIdx.x, out + blockIdx.x);
}

bool adjoint_supported(int rhs_id) {
    return rhs_id == FF_RHS_LORENZ || rhs_id == FF_RHS_WILSON_COWAN || rhs_id == FF_RHS_HARMONIC ||
           rhs_id == FF_RHS_LINEAR || rhs_id == FF_RHS_HH3;
}

int adjoint_sub_steps(int64_t checkpoint_every) {
    // a chunk of up to 16 steps is one sub-segment (one recomputation); longer chunks take
    // sub-checkpoints every M steps with M * M >= the chunk (two recomputations)
    if (checkpoint_every <= 4) return 4;
    if (checkpoint_every <= 8) return 8;
    if (checkpoint_every <= 16) return 16;
    if (checkpoint_every <= 64) return 8;
    return 16;
}

int64_t adjoint_partial_rows(int num_sms) { return (int64_t)num_sms * 8 * 8; }

int64_t adjoint_scratch_threads(int rhs_id, int method, bool pp, int num_sms, bool batched) {
    return rhs_id == FF_RHS_HH3 ? adjoint_scratch_threads_hh3(method, pp, num_sms, batched) : 0;
}

cudaError_t launch_adjoint(int rhs_id, int method, bool pp, int m, const AdjointArgs& a0, int num_sms,
                           cudaStream_t s, double* dL_dp_dev, int n_params_kernel) {
    AdjointArgs a = a0;
    if (adjoint_task_row(rhs_id, method) > 0) a.np_stride = adjoint_task_row(rhs_id, method);
    const int block = 128;
    int64_t rows = 0;
    cudaError_t e;
    switch (rhs_id) {
    case FF_RHS_LORENZ: e = launch_adjoint_lorenz(method, pp, m, a, block, num_sms, s, &rows); break;
    case FF_RHS_HH3: e = launch_adjoint_hh3(method, pp, m, a, block, num_sms, s, &rows); break;
    case FF_RHS_LINEAR: e = launch_adjoint_linear(method, pp, m, a, block, num_sms, s, &rows); break;
    case FF_RHS_WILSON_COWAN:
    case FF_RHS_HARMONIC: e = launch_adjoint_small(rhs_id, method, pp, m, a, block, num_sms, s, &rows); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    reduce_partials_kernel<<<n_params_kernel, kReduceBlock, 0, s>>>(a.partial, rows, a.np_stride, dL_dp_dev);
    return cudaGetLastError();
}

cudaError_t launch_batch_adjoint(int rhs_id, int method, bool pp, int m, const BatchAdjointArgs& b,
                                 const int* row0_dev, int n_members, int n_params_kernel, int num_sms,
                                 cudaStream_t s, double* dp_dev) {
    cudaError_t e;
    switch (rhs_id) {
    case FF_RHS_LORENZ: e = launch_batch_adjoint_lorenz(method, pp, m, b, num_sms, s); break;
    case FF_RHS_HH3: e = launch_batch_adjoint_hh3(method, pp, m, b, num_sms, s); break;
    case FF_RHS_LINEAR: e = launch_batch_adjoint_linear(method, pp, m, b, num_sms, s); break;
    case FF_RHS_WILSON_COWAN:
    case FF_RHS_HARMONIC: e = launch_batch_adjoint_small(rhs_id, method, pp, m, b, num_sms, s); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int items = n_members * n_params_kernel;
    if (items > 0)
        reduce_member_rows_kernel<<<items, kReduceBlock, 0, s>>>(b.partial, row0_dev, n_params_kernel, b.np_stride,
                                                                 dp_dev);
    return cudaGetLastError();
}

}  // namespace ff
