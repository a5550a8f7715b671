// Kernels of a solve of one right-hand side (one team spanning the grid).
#include "smpm_device.cuh"
#include "smpm_digits.cuh"

namespace {

#include "smpm_gmres.cuh"
#include "smpm_prepost.cuh"
#include "smpm_refine.cuh"

// The bodies' phases are calls and take their arguments from shared memory: copied
// from the launch's by all threads (one thread's copy took about a microsecond).
template <typename A>
__device__ __forceinline__ void stage_args(A& a, const A& a0) {
  static_assert(sizeof(A) % 8 == 0 && alignof(A) >= 8, "copied by 8 bytes");
  const long long* src = reinterpret_cast<const long long*>(&a0);
  long long* dst = reinterpret_cast<long long*>(&a);
  for (int i = threadIdx.x; i < (int)(sizeof(A) / 8); i += blockDim.x) dst[i] = src[i];
  __syncthreads();
}

template <typename S>
__global__ void __launch_bounds__(256, 1) k_gmres(const __grid_constant__ GmresArgs<S> a0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ GmresArgs<S> a;
  if (a0.skip && *((volatile const int*)a0.skip)) return;
  stage_args(a, a0);
  unsigned epoch = 0;
  gmres_body(a, smraw, epoch);
}

__global__ void __launch_bounds__(256, 1) k_pre(const __grid_constant__ PrePostArgs P0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ PrePostArgs P;
  stage_args(P, P0);
  unsigned epoch = 0;
  pre_body(P, smraw, epoch);
}

__global__ void __launch_bounds__(256, 1) k_post(const __grid_constant__ PrePostArgs P0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ PrePostArgs P;
  stage_args(P, P0);
  unsigned epoch = 0;
  post_body(P, smraw, epoch);
}

__global__ void __launch_bounds__(256, 1) k_refine(const __grid_constant__ RefineArgs R0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ RefineArgs R;
  if (*((volatile const int*)R0.done)) return;
  stage_args(R, R0);
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
