// Kernels of a solve of one right-hand side (one team spanning the grid).
#include "smpm_device.cuh"
#include "smpm_digits.cuh"

namespace {

#include "smpm_gmres.cuh"
#include "smpm_prepost.cuh"
#include "smpm_refine.cuh"

template <typename S>
__global__ void __launch_bounds__(256, 1) k_gmres(GmresArgs<S> a0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ GmresArgs<S> a;
  if (threadIdx.x == 0) a = a0;
  __syncthreads();
  if (a.skip && *((volatile const int*)a.skip)) return;
  unsigned epoch = 0;
  gmres_body(a, smraw, epoch);
}

__global__ void __launch_bounds__(256, 1) k_pre(PrePostArgs P0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ PrePostArgs P;
  if (threadIdx.x == 0) P = P0;
  __syncthreads();
  unsigned epoch = 0;
  pre_body(P, smraw, epoch);
}

__global__ void __launch_bounds__(256, 1) k_post(PrePostArgs P0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ PrePostArgs P;
  if (threadIdx.x == 0) P = P0;
  __syncthreads();
  unsigned epoch = 0;
  post_body(P, smraw, epoch);
}

__global__ void __launch_bounds__(256, 1) k_refine(RefineArgs R0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ RefineArgs R;
  if (threadIdx.x == 0) R = R0;
  __syncthreads();
  if (*((volatile const int*)R.done)) return;
  unsigned epoch = 0;
  refine_body(R, smraw, epoch);
}

}  // namespace

namespace smpm {

const void* fn_pre() { return (const void*)k_pre; }
const void* fn_post() { return (const void*)k_post; }
const void* fn_gmres64() { return (const void*)k_gmres<double>; }
const void* fn_gmres32() { return (const void*)k_gmres<float>; }
const void* fn_refine() { return (const void*)k_refine; }
cudaError_t set_spin_solve(long long v) { return cudaMemcpyToSymbol(g_barrier_spin_limit, &v, sizeof(v)); }

}  // namespace smpm
