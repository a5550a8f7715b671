// Constants, solve state and element solves shared by the translation units
// of the persistent kernels (smpm_k_solve.cu, smpm_k_lock.cu, smpm_k_batch.cu)
// and the host side (smpm_solver.cu).
#pragma once
#include <cuda_runtime.h>

// The solve bodies and their phases are calls, not inlined: one kernel with all
// of them inlined spills registers (k_gmres: 1.6 KB per thread) and takes
// minutes to compile.  The kernels stage their arguments in shared memory, so
// that a call's reference to them costs no copy.
#define SMPM_BODY __noinline__
#define SMPM_PHASE __noinline__

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <type_traits>

#include "smpm_internal.h"
#include "smpm_kernels.cuh"

namespace smpm {

// The persistent kernels are compiled in translation units of their own (in
// parallel); the host launches them by address.
const void* fn_pre();
const void* fn_post();
const void* fn_gmres64();
const void* fn_gmres32();
const void* fn_refine();
const void* fn_lock64();
const void* fn_lock32();
const void* fn_pre_cols();
const void* fn_post_cols();
const void* fn_refine_cols();
const void* fn_batch();
// poll limit of the barrier waits of one translation unit's kernels
cudaError_t set_spin_solve(long long v);
cudaError_t set_spin_lock(long long v);
cudaError_t set_spin_batch(long long v);

}  // namespace smpm

using namespace smpm;

namespace {

constexpr int kSlotsPerBlock = 256;   // slots per CTA in the vector kernels
constexpr int kElemThreads = 256;     // threads per element CTA
constexpr int kTraceCap = 1 << 16;    // entries of the optional phase trace
constexpr int kGmresThreads = 256;    // threads per CTA of the persistent GMRES kernel
// per-solve control block (zeroed by one memset): 64 barrier counters, one per
// launch of the solve | (at 256) err, done, nref | 8 accumulators | 32
// refinement residual norms
constexpr size_t kCtlBytes = 720;  // + 32 inner iteration counts
constexpr int kMaxRefine = 8;        // FP64 refinement steps of the mixed-precision path
constexpr double kInnerTol = 1e-4;   // relative tolerance of each FP32 inner GMRES

struct GState {
  double tolabs, beta0, beta, wnorm0sq, resid;
  int j, converged, breakdown, nan;
  double R[(kMaxRestart + 1) * kMaxRestart];  // column j at R[j*(kMaxRestart+1)]
  double h1[kMaxRestart + 2], h2[kMaxRestart + 2];
  double y[kMaxRestart];
  double scal[8];
};



// ------------------------------------------------------- element solves
// U = A_e^-1 B by fast diagonalisation (the Kronecker-sum structure of A_e):
// U = Vy ((Vy^-1 B Vx^-T) ./ (lx_i + ly_j)) Vx^T.  B, U, t1: n*n in shared.
__device__ void elem_solve_dev(int n, const double* __restrict__ fx, const double* __restrict__ fy, const double* B,
                               double* U, double* t1) {
  const double *Vx = fx, *Vxi = fx + n * n, *lx = fx + 2 * n * n;
  const double *Vy = fy, *Vyi = fy + n * n, *ly = fy + 2 * n * n;
  const int nn = n * n;
  for (int q = threadIdx.x; q < nn; q += blockDim.x) {  // t1 = Vyi B
    int j = q / n, a = q % n;
    double s = 0;
    for (int b = 0; b < n; ++b) s += __ldg(Vyi + j * n + b) * B[b * n + a];
    t1[q] = s;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nn; q += blockDim.x) {  // U = t1 Vxi^T ./ (lx + ly)
    int j = q / n, i = q % n;
    double s = 0;
    for (int a = 0; a < n; ++a) s += t1[j * n + a] * __ldg(Vxi + i * n + a);
    U[q] = s / (__ldg(lx + i) + __ldg(ly + j));
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nn; q += blockDim.x) {  // t1 = U Vx^T
    int j = q / n, a = q % n;
    double s = 0;
    for (int i = 0; i < n; ++i) s += U[j * n + i] * __ldg(Vx + a * n + i);
    t1[q] = s;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nn; q += blockDim.x) {  // U = Vy t1
    int b = q / n, a = q % n;
    double s = 0;
    for (int j = 0; j < n; ++j) s += __ldg(Vy + b * n + j) * t1[j * n + a];
    U[q] = s;
  }
  __syncthreads();
}

__device__ __forceinline__ void face_node(int n, int F, int t, int* a, int* b) {
  switch (F) {
    case 0: *a = 0; *b = t; break;
    case 1: *a = n - 1; *b = t; break;
    case 2: *a = t; *b = 0; break;
    default: *a = t; *b = n - 1; break;
  }
}

// n_F . grad U at face node t (U in shared memory, D in global).
// n_F . grad U at face node t of face F (sc = 2/h of the element across F).
__device__ double normal_deriv(const DevGeo& g, const double* __restrict__ D, const double* U, int F, int t,
                               double sc) {
  const int n = g.n;
  double acc = 0;
  switch (F) {
    case 0: for (int c = 0; c < n; ++c) acc += __ldg(D + c) * U[t * n + c]; return -sc * acc;
    case 1: for (int c = 0; c < n; ++c) acc += __ldg(D + (n - 1) * n + c) * U[t * n + c]; return sc * acc;
    case 2: for (int c = 0; c < n; ++c) acc += __ldg(D + c) * U[c * n + t]; return -sc * acc;
    default: for (int c = 0; c < n; ++c) acc += __ldg(D + (n - 1) * n + c) * U[c * n + t]; return sc * acc;
  }
}

// fast-diagonalisation entry: face-type class, or the column / row on a graded grid
__device__ __forceinline__ const double* fd_x(const DevGeo& g, const double* fdx, int e) {
  int ix = e % g.mx;
  int cls = g.graded ? ix : ((ix > 0 ? 1 : 0) | (ix < g.mx - 1 ? 2 : 0));
  return fdx + (size_t)cls * (2 * g.n * g.n + g.n);
}
__device__ __forceinline__ const double* fd_y(const DevGeo& g, const double* fdy, int e) {
  int iy = e / g.mx;
  int cls = g.graded ? iy : ((iy > 0 ? 1 : 0) | (iy < g.my - 1 ? 2 : 0));
  return fdy + (size_t)cls * (2 * g.n * g.n + g.n);
}

}  // namespace
