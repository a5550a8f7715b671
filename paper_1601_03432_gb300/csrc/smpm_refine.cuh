// One step of GMRES-based iterative refinement (mixed precision):
// the inner GMRES (k_gmres<float>) has solved P S M^-1 y = P r in FP32; this
// cooperative kernel turns y into the FP64 correction and the next inner
// right-hand side.  C^+ is the inner solve's own (coarse_solve): the FP64 inverse on
// small grids, else its FP32 copy with FP32 products and sums; c and c_hat are FP64.
//   R1  owner blocks:   t = M^-1 y                        (FP32 operator)
//   R2  white elements: S t on the black slots, c = Z^T S t (FP64 sums)
//   R3  c_hat = C^+ c
//   R4  owner entries:  x_S += t - Z (c_hat - c_hat_r)     (FP64; Eq. deflated_schur
//                       for the correction equation S d = r); y <- 0
//   R5  elements:       r = b_S - S x_S with the FP64 T_e (push form);
//                       ||r||^2 and Z^T r accumulated
//   R6  ||r|| <= tol ||P b_S||: done (all CTAs agree); otherwise
//                       c_hat_r = C^+ Z^T r
//   R7  owner entries:  next inner right-hand side P r = r - S Z c_hat_r (FP32)
#pragma once
// Included inside the anonymous namespace of each translation unit that uses it.

struct alignas(16) RefineArgs {  // 16-byte multiple: staged with 16-byte copies in batched solves
  GmresArgs<float> ga;   // FP32 operator and vectors: x = inner y, t, y, c, chat, rhs (next inner rhs)
  const uint4* T64;      // FP64 T_e per class, packed, and the row exponents (smpm_digits.cuh)
  const short* Te64;
  double* xS;            // kp, FP64 Schur iterate
  const double* bS;      // kp, projected b_S
  double* r;             // kp, FP64 residual
  double* cr;            // d, Z^T r (zero on entry, left zero)
  double* chat_r;        // d, C^+ Z^T r of the current residual
  const double* rgn;     // ||P b_S||^2
  double* rn;            // ||r||^2 accumulator of this step (zero on entry)
  int* done;             // set once converged; later launches return at once
  int* nref;             // refinement steps taken
  float* rhs32;          // kp, next inner right-hand side
  double tol;
};

inline size_t refine_smem_bytes(int m, int M, int n, int ES, int W, long long d, bool w_global = false) {
  return gmres_smem_bytes<float>(m, M, n, ES, W, 0, d, w_global) +
         (size_t)(kGmresThreads / 32 / W) * (sizeof(uint4) * (size_t)digit_bwords<double>(M) + M * sizeof(double));
}

// One refinement step by the CTAs of a team; returns 1 when converged (done
// set), 0 when another inner solve follows, -1 when a barrier timed out.
__device__ SMPM_BODY int refine_body(const RefineArgs& R, unsigned char* smraw, unsigned& epoch) {
  const GmresArgs<float>& a = R.ga;
  const Smem<float> s = carve(a, smraw);
  no_resident(a, s);
  const DevGeo& g = a.g;
  const int n = g.n, M = g.M, G = a.G, rank = team_rank(a), W = a.W_item, kt_n = digit_tiles(M);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W,
            ngrp = kGmresThreads / 32 / W;
  uint4* Bf = reinterpret_cast<uint4*>(s.end + (size_t)grp * (sizeof(uint4) * (size_t)digit_bwords<double>(M) +
                                                              M * sizeof(double)));
  double* rw = reinterpret_cast<double*>(Bf + digit_bwords<double>(M));  // x_S on the element's slots, then its weighted residual entries
  int trace_n = 0;
  // ---- R1-R3: t = M^-1 y, S t, c_hat
  black_phase(a, s, (const float*)a.x, 1.0, (const float*)nullptr);
  if (!apply_op(a, s, a.x, 1.0, true, trace_n, epoch)) return -1;
  // ---- R4: x_S += t - Z (c_hat - c_hat_r); y <- 0 for the next inner solve
  for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
    const int4 en = owned_entry(a, i);
    if (en.x < 0) continue;
    if (en.z >= 0)
      R.xS[en.x] += (double)__ldcg(a.t + en.x) - entry_zw(g, en) * (__ldcg(a.chat + en.z) - R.chat_r[en.z]);
    a.x[en.x] = 0.f;
  }
  if (!team_sync(a, epoch)) return -1;
  // ---- R5: r = b_S - S x_S (FP64), ||r||^2, Z^T r
  double pr = 0;
  for (long long el = rank + (long long)grp * G; el < g.nel; el += (long long)ngrp * G) {
    const int e = (int)el, ct = __ldg(a.dm.tcls + e);
    for (int i = part * 32 + lane; i < M; i += 32 * W) rw[i] = __ldcg(R.xS + el * M + i);
    item_sync(grp, W);
    const int E = pack_one<double>(Bf, rw, M, lane, part, W);
    item_sync(grp, W);
    for (int mt = part; mt < kt_n; mt += W) {
      const int row = tile1_row(mt, lane, M);
      Facing<double> f{};
      if (row >= 0) f = facing_entry(g, e, row, R.xS, R.xS);
      const double z = digits_tile1<double>(R.T64 + (size_t)ct * digit_words<double>(M, M), R.Te64 + (size_t)ct * M, Bf, M,
                                            kt_n, mt, lane, E);
      if (row < 0) continue;
      double rr = 0;
      if (f.sl >= 0) {
        rr = R.bS[f.sl] - (f.t + z);
        R.r[f.sl] = rr;
        pr += rr * rr;
        if (g.zw) rr *= f.w1;  // its weight in Z^T r
      }
      rw[row] = rr;  // (x_S is packed: its place is free)
    }
    item_sync(grp, W);
    if (part == 0) {  // face F summed by the eight lanes 8 F + r
      const int F = lane >> 3, j = dev_iface(g, e, F);
      double sum = 0;
      for (int t = lane & 7; t < n; t += 8) sum += rw[F * n + t];
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if ((lane & 7) == 0 && j >= 0 && sum != 0.0) atomicAdd(R.cr + j, sum);
    }
    item_sync(grp, W);
  }
  pr = warp_sum(pr);
  if ((threadIdx.x & 31) == 0 && pr != 0.0) atomicAdd(R.rn, pr);
  if (!team_sync(a, epoch)) return -1;
  // ---- R6: convergence test (uniform), else c_hat_r = C^+ Z^T r
  const double rho = sqrt(__ldcg(R.rn)), target = R.tol * sqrt(__ldcg(R.rgn));
  if (rank == 0 && threadIdx.x == 0) *R.nref += 1;
  if (rho <= target) {
    if (rank == 0 && threadIdx.x == 0) *R.done = 1;
    return 1;
  }
  if (!coarse_solve(a, s, epoch, R.cr, R.chat_r)) return -1;
  // ---- R7: next inner right-hand side P r (FP32); Z^T r back to zero
  for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
    const int4 en = owned_entry(a, i);
    if (en.x >= 0) R.rhs32[en.x] = (float)deflate_entry(a, (const double*)R.r, R.chat_r, en);
  }
  for (long long j = (long long)rank * blockDim.x + threadIdx.x; j < g.d; j += (long long)G * blockDim.x)
    R.cr[j] = 0.0;
  return 0;
}
