// Kernels of a lockstep solve of several right-hand sides of one grid.
#include "smpm_device.cuh"
#include "smpm_digits.cuh"

namespace {

#include "smpm_gmres.cuh"
#include "smpm_prepost.cuh"
#include "smpm_refine.cuh"
#include "smpm_lockstep.cuh"

template <typename S>
__global__ void __launch_bounds__(256, 1) k_gmres_lock(LockArgs<S> A0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ LockArgs<S> A;  // the phases are calls: arguments from shared memory
  if (lock_all_done(A0)) return;
  if (threadIdx.x == 0) A = A0;
  __syncthreads();
  unsigned epoch = 0;
  lock_body(A, smraw, epoch);
}

// The right-hand-side and recovery bodies of R columns, one launch each: the
// bodies run one column after another (their barrier epoch carries on), each
// with its own arguments; the scratch vectors they share (t, y, c, c_hat)
// are only touched after a barrier that every CTA passes once it is done with
// the previous column.
__global__ void __launch_bounds__(256, 1) k_pre_cols(const PrePostArgs* __restrict__ Ps, int R) {
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned epoch = 0;
  __shared__ PrePostArgs P;
  for (int c = 0; c < R; ++c) {
    __syncthreads();
    stage16(&P, Ps + c, (int)sizeof(P));
    __syncthreads();
    if (!pre_body(P, smraw, epoch)) return;
  }
}

__global__ void __launch_bounds__(256, 1) k_post_cols(const PrePostArgs* __restrict__ Ps, int R) {
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned epoch = 0;
  __shared__ PrePostArgs P;
  for (int c = 0; c < R; ++c) {
    __syncthreads();
    stage16(&P, Ps + c, (int)sizeof(P));
    __syncthreads();
    if (!post_body(P, smraw, epoch)) return;
  }
}

// One refinement step (refine_body) for every column not yet done, one
// column after another.  A column's done flag is read before its body starts;
// only its own body (rank 0, after a barrier every CTA passed) sets it.
__global__ void __launch_bounds__(256, 1) k_refine_cols(const RefineArgs* __restrict__ Rs, int R) {
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned epoch = 0;
  __shared__ RefineArgs A;
  for (int c = 0; c < R; ++c) {
    if (*((volatile const int*)Rs[c].done)) continue;
    __syncthreads();
    stage16(&A, Rs + c, (int)sizeof(A));
    __syncthreads();
    if (refine_body(A, smraw, epoch) < 0) return;
  }
}

}  // namespace

namespace smpm {

const void* fn_lock64() { return (const void*)k_gmres_lock<double>; }
const void* fn_lock32() { return (const void*)k_gmres_lock<float>; }
const void* fn_pre_cols() { return (const void*)k_pre_cols; }
const void* fn_post_cols() { return (const void*)k_post_cols; }
const void* fn_refine_cols() { return (const void*)k_refine_cols; }
cudaError_t set_spin_lock(long long v) { return cudaMemcpyToSymbol(g_barrier_spin_limit, &v, sizeof(v)); }

}  // namespace smpm
