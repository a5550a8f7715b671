// Cooperative kernels around the GMRES kernel (FP64): the right-hand side
// steps before it and the assembly/recovery steps after it, each one launch
// with grid barriers between its phases.  Ownership follows smpm_gmres.cuh:
// CTA c owns the checkerboard blocks and white elements c, c+G, ..., and for
// node-level work the elements e = c, c+G, ...
//
// k_pre (the projections of Sec. 1.4, the Schur right-hand side of
// Eq. schur_complement_system and the GMRES right-hand side P b_S):
//   P1  b = f + tau g on the owned elements; u_L^T b accumulated
//   P2  b <- b - u_L (u_L^T b); w = A_e^-1 b_e (fast diagonalisation); the
//       Robin fluxes of w are pushed into the neighbours' facing slots
//       (b_S = B A^-1 b); the same pass accumulates u_S^T b_S and, per face,
//       the interface sums Z^T b_S
//   P3  b_S <- b_S - u_S (u_S^T b_S) enters through Z^T b_S - (u_S^T b_S) Z^T u_S;
//       c_hat_b = C^+ Z^T b_S (coarse rows)
//   P4  owner entries: b_S projected in place, rhs = P b_S = b_S - S Z c_hat_b
// k_post (the assembly of Eq. deflated_schur, the recovery u = A^-1 (b - E x)
// and the zero-mean normalisation):
//   Q1  t = M^-1 x on the owned blocks
//   Q2  white elements: y = S t, c = Z^T y
//   Q3  c_hat = C^+ c
//   Q4  owner entries: x_S = t - Z (c_hat - c_hat_b)       [Eq. deflated_schur]
//   Q5  owned elements: u_e = A_e^-1 (b_e - E_e x_S); the pushed products
//       T_e x_S also give the true residual ||b_S - S x_S||^2; GLL-weighted
//       mean of u accumulated
//   Q6  u <- u - mean
//
// With `adjoint` set the same kernels run the transposed solve (reverse-mode
// derivative of u(f, g)), on the factors of the slot-swapped S^T (T~ = T^T,
// see the factor step) and with the transposed element operators:
//   P1  y = gbar (= dl/du); 1^T y accumulated
//   P2  y <- y - w^ (1^T y)  (N^T, N the zero-mean map); w = A_e^-T y_e; the
//       face values of w (E^T A^-T y) are pushed into the facing slots
//   P3, P4, Q1-Q4 unchanged (the transposed factors are passed in)
//   Q5  lam_e = A_e^-T (y_e - B_e^T mu_e) with mu_e the element's own slots of
//       the solution; u_L^T lam accumulated
//   Q6  dl/db = lam - u_L (u_L^T lam) written to u; dl/dg on boundary-face
//       slots = tau_F dl/db at the face node (gg, if given)
#pragma once
// Included inside the anonymous namespace of each translation unit that uses it.

// Packed fast-diagonalisation factors (smpm_digits.cuh): per x entry (a
// face-type class, or a column of a graded grid) the digits of V and V^-1 and
// their row exponents, likewise per y entry, and 1 / (lx_i + ly_j) at
// [j n + i] per pair of entries.
struct FdMats {
  const uint4 *x, *y;
  const short *xe, *ye;
  const double* rinv;
  const double *fx, *fy;  // V and V^-1 in FP64, two per class (fd_thread_pass)
  int nx, pad_;
};

struct alignas(16) PrePostArgs {  // 16-byte multiple: staged with 16-byte copies in batched solves
  GmresArgs<double> ga;  // geometry, ownership, operator matrices, t/y/c/chat buffers
  FdMats fd;  // fast diagonalisation (packed)
  const double* D;
  const double* uL;
  const double* uS;
  const double* what;
  const double* ZtuS;  // d : Z^T u_S
  const double* f;
  const double* gn;
  double* b;      // r
  double* bS;     // kp
  double* rg;     // kp
  double* cb;     // d : Z^T b_S (accumulated)
  double* chatb;  // d
  double* xs;     // kp
  double* u;      // r
  double* acc;    // 8 FP64 accumulators
  double* zero[7];  // kp-long buffers zeroed in P1 (x, t, y, vglob, b_S, rhs, x_S)
  double* gacc;     // GMRES accumulators, zeroed in P1
  long long gacc_n;
  float* zero32[4];  // kp-long FP32 buffers zeroed in P1 (mixed precision), or null
  double* cr;        // d, zeroed in P1 (mixed precision), or null
  float* rg32;       // kp, FP32 copy of the GMRES right-hand side (mixed precision), or null
  int W_fd;          // warps per element in the element solves
  int assembled;     // k_post: x_S is given in xs (skip the assembly)
  int adjoint;       // transposed solve (see above)
  double* gg;        // adjoint: kp, dl/dg per padded slot, or null
};

// copy n bytes (a multiple of 16) from global memory into shared memory, all threads
__device__ __forceinline__ void stage16(void* dst, const void* src, int n) {
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* d = reinterpret_cast<int4*>(dst);
  for (int i = threadIdx.x; i < n / 16; i += blockDim.x) d[i] = s[i];
}

// accumulator slots
enum { ACC_ULB = 0, ACC_USBS = 1, ACC_MEAN = 2, ACC_RES = 3, ACC_BSN = 4, ACC_RGN = 5 };

// ---- element solves --------------------------------------------------------
// A group of W warps solves U = A_e^-1 B by fast diagonalisation: U = Vy ((Vy^-1
// B Vx^-T) .* rinv) Vx^T, four n x n products on the tensor cores, the columns
// in tiles of eight shared out over the warps.  B, U, t1: n rows of fd_ld(n)
// doubles; Bf: one packed tile per warp.
__host__ __device__ constexpr int fd_ld(int n) { return (n + 3) / 8 * 8 + 4; }  // 4 modulo 8: rows spread over the banks
// whether a group of W warps forms the products by threads (fd_thread_pass)
__host__ __device__ constexpr bool fd_by_threads(int n, int W) { return n <= 8 || (n <= 12 && n * n <= 64 * W); }
// scratch of a group: three tiles, the slot values (two times 4n), packed tiles
// (none by threads; the element's residual product packs its vector there)
__host__ __device__ inline size_t fd_item_bytes(int n, int W) {
  const size_t tile = fd_by_threads(n, W) ? 0 : sizeof(uint4) * (size_t)digit_bwords<double>(n);
  const size_t vec = sizeof(uint4) * (size_t)digit_bwords<double>(4 * n), bf = W * tile > vec ? W * tile : vec;
  return bf + sizeof(double) * (3 * (size_t)n * fd_ld(n) + 8 * (size_t)n);
}
struct FdItem {
  uint4* Bf;
  double *B, *U, *t1, *p, *q;  // p, q: 4n slot values each
};
__device__ __forceinline__ FdItem fd_item(unsigned char* base, int n, int W, int grp) {
  FdItem f;
  unsigned char* b = base + (size_t)grp * fd_item_bytes(n, W);
  f.B = reinterpret_cast<double*>(b);
  f.U = f.B + (size_t)n * fd_ld(n);
  f.t1 = f.U + (size_t)n * fd_ld(n);
  f.p = f.t1 + (size_t)n * fd_ld(n);
  f.q = f.p + 4 * n;
  f.Bf = reinterpret_cast<uint4*>(f.q + 4 * n);
  return f;
}

// One product: row r, column c of A (packed, n x n) times the columns x[k ldk +
// c ldc], times w[c n + r] where w is given, to out[r ldr + c ldo].
__device__ __noinline__ void fd_pass(const uint4* A, const short* er, uint4* Bw, int n, int lane, int part, int W,
                                     const double* x, int ldk, int ldc, double* out, int ldr, int ldo,
                                     const double* __restrict__ w) {
  const int kt_n = digit_tiles(n);
  for (int c0 = 8 * part; c0 < n; c0 += 8 * W) {
    const int nc = min(8, n - c0), E = pack_cols<double>(Bw, x + c0 * ldc, ldk, ldc, n, nc, lane, 0, 1);
#pragma unroll 1
    for (int mt = 0; mt < kt_n; ++mt) {
      const Tile8<double> t = digits_tile8<double>(A, er, Bw, n, kt_n, mt, lane, E);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int r = mt * 16 + (lane >> 2) + 8 * (v >> 1), c = 2 * (lane & 3) + (v & 1);
        if (r < n && c < nc) out[r * ldr + (c0 + c) * ldo] = w ? t.z[v] * __ldg(w + (c0 + c) * n + r) : t.z[v];
      }
    }
    __syncwarp();
  }
}

// The same by plain FP64 products, a thread per entry of out.  An 8 x 8 product
// takes a warp about 1,500 SM cycles, 256 of them FP64 issue; its packing and
// tile of eight columns (half of it padding) 3,500.  At n = 12 the FP64 products
// alone cost what the tiles do, so there only where the group has a thread for
// every other entry; from n = 16 on the digits win.
__device__ __noinline__ void fd_thread_pass(const double* __restrict__ A, int n, int tid, int nthr, const double* x, int ldk,
                                            int ldc, double* out, int ldr, int ldo, const double* __restrict__ w) {
#pragma unroll 1
  for (int q = tid; q < n * n; q += nthr) {
    const int c = q / n, r = q - c * n;
    double s0 = 0, s1 = 0;
    int k = 0;
#pragma unroll 2
    for (; k + 1 < n; k += 2) {
      s0 += __ldg(A + r * n + k) * x[k * ldk + c * ldc];
      s1 += __ldg(A + r * n + k + 1) * x[(k + 1) * ldk + c * ldc];
    }
    if (k < n) s0 += __ldg(A + r * n + k) * x[k * ldk + c * ldc];
    const double z = s0 + s1;
    out[r * ldr + c * ldo] = w ? z * __ldg(w + q) : z;
  }
}

// U = A_e^-1 B for element e, entered and left with the group in step
__device__ __noinline__ void elem_fd(const FdMats& fd, const DevGeo& g, int e, const FdItem& f, int lane, int part,
                                        int W, int grp) {
  const int n = g.n, ld = fd_ld(n), ix = e % g.mx, iy = e / g.mx;
  const int cx = g.graded ? ix : ((ix > 0 ? 1 : 0) | (ix < g.mx - 1 ? 2 : 0));
  const int cy = g.graded ? iy : ((iy > 0 ? 1 : 0) | (iy < g.my - 1 ? 2 : 0));
  const size_t nw = digit_words<double>(n, n);
  const uint4 *Vx = fd.x + 2 * cx * nw, *Vxi = Vx + nw, *Vy = fd.y + 2 * cy * nw, *Vyi = Vy + nw;
  const short *ex = fd.xe + 2 * cx * n, *exi = ex + n, *ey = fd.ye + 2 * cy * n, *eyi = ey + n;
  const double* ri = fd.rinv + ((size_t)cy * fd.nx + cx) * n * n;
  if (fd_by_threads(n, W)) {
    const size_t nn = (size_t)n * n;
    const double *X = fd.fx + 2 * cx * nn, *Y = fd.fy + 2 * cy * nn;
    fd_thread_pass(Y + nn, n, 32 * part + lane, 32 * W, f.B, ld, 1, f.t1, ld, 1, nullptr);
    item_sync(grp, W);
    fd_thread_pass(X + nn, n, 32 * part + lane, 32 * W, f.t1, 1, ld, f.U, 1, ld, ri);
    item_sync(grp, W);
    fd_thread_pass(X, n, 32 * part + lane, 32 * W, f.U, 1, ld, f.t1, 1, ld, nullptr);
    item_sync(grp, W);
    fd_thread_pass(Y, n, 32 * part + lane, 32 * W, f.t1, ld, 1, f.U, ld, 1, nullptr);
    item_sync(grp, W);
    return;
  }
  uint4* Bw = f.Bf + (size_t)part * digit_bwords<double>(n);
  fd_pass(Vyi, eyi, Bw, n, lane, part, W, f.B, ld, 1, f.t1, ld, 1, nullptr);   // t1 = Vy^-1 B
  item_sync(grp, W);
  fd_pass(Vxi, exi, Bw, n, lane, part, W, f.t1, 1, ld, f.U, 1, ld, ri);         // U = (t1 Vx^-T) .* rinv
  item_sync(grp, W);
  fd_pass(Vx, ex, Bw, n, lane, part, W, f.U, 1, ld, f.t1, 1, ld, nullptr);      // t1 = U Vx^T
  item_sync(grp, W);
  fd_pass(Vy, ey, Bw, n, lane, part, W, f.t1, ld, 1, f.U, ld, 1, nullptr);      // U = Vy t1
  item_sync(grp, W);
}

// n_F . grad U at face node t of face F (rows of ld doubles; sc = 2/h of the element across F)
__device__ __forceinline__ double normal_deriv_ld(const DevGeo& g, const double* __restrict__ D, const double* U, int ld,
                                                  int F, int t, double sc) {
  const int n = g.n, st = F < 2 ? 1 : ld;
  const double* u = F < 2 ? U + t * ld : U + t;
  const double* d = D + ((F & 1) ? (n - 1) * n : 0);
  double a0 = 0, a1 = 0;
  int c = 0;
#pragma unroll 2
  for (; c + 1 < n; c += 2) {
    a0 += __ldg(d + c) * u[c * st];
    a1 += __ldg(d + c + 1) * u[(c + 1) * st];
  }
  if (c < n) a0 += __ldg(d + c) * u[c * st];
  return ((F & 1) ? sc : -sc) * (a0 + a1);
}

__device__ SMPM_BODY bool pre_body(const PrePostArgs& P, unsigned char* smraw, unsigned& epoch) {
  const GmresArgs<double>& a = P.ga;
  const Smem<double> s = carve(a, smraw);
  no_resident(a, s);
  const DevGeo& g = a.g;
  const int n = g.n, nn = n * n, M = g.M, G = a.G, rank = team_rank(a);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = P.W_fd, grp = warp / W, part = warp % W,
            ngrp = kGmresThreads / 32 / W;
  const FdItem f = fd_item(s.end, n, W, grp);
  const int ld = fd_ld(n);
  int trace_n = 0;
  GM_TRACE(50);
  // ---- P1: zero the work vectors; b = f + tau g; u_L^T b
#pragma unroll 1
  for (long long i = (long long)rank * blockDim.x + threadIdx.x; i < g.kp; i += (long long)G * blockDim.x)
    for (int v = 0; v < 7; ++v) P.zero[v][i] = 0.0;
#pragma unroll 1
  for (long long i = (long long)rank * blockDim.x + threadIdx.x; i < P.gacc_n; i += (long long)G * blockDim.x)
    P.gacc[i] = 0.0;
#pragma unroll 1
  for (long long i = (long long)rank * blockDim.x + threadIdx.x; i < g.d; i += (long long)G * blockDim.x) {
    P.cb[i] = 0.0;
    if (P.cr) P.cr[i] = 0.0;
  }
  if (P.zero32[0])
#pragma unroll 1
    for (long long i = (long long)rank * blockDim.x + threadIdx.x; i < g.kp; i += (long long)G * blockDim.x)
      for (int v = 0; v < 4; ++v) P.zero32[v][i] = 0.f;
  if (rank == 0 && threadIdx.x == 0) a.gs->scal[5] = 0.0;  // inner iterations of the solve
  double ulb = 0;
#pragma unroll 1
  for (long long e = rank; e < g.nel; e += G) {
    for (int q = threadIdx.x; q < nn; q += blockDim.x) {
      const int aa = q % n, bb = q / n;
      const long long gq = e * nn + q;
      double v = P.f[gq];
      if (P.gn) {
        const long long s0 = e * M;
        const double tx = face_geo(g, (int)e, 0)[0], ty = face_geo(g, (int)e, 2)[0];
        if (aa == 0 && dev_neighbour(g, (int)e, 0) < 0) v += tx * P.gn[s0 + bb];
        if (aa == n - 1 && dev_neighbour(g, (int)e, 1) < 0) v += tx * P.gn[s0 + n + bb];
        if (bb == 0 && dev_neighbour(g, (int)e, 2) < 0) v += ty * P.gn[s0 + 2 * n + aa];
        if (bb == n - 1 && dev_neighbour(g, (int)e, 3) < 0) v += ty * P.gn[s0 + 3 * n + aa];
      }
      P.b[gq] = v;
      ulb += P.adjoint ? v : P.uL[gq] * v;
    }
  }
  ulb = warp_sum(ulb);
  if ((threadIdx.x & 31) == 0 && ulb != 0.0) atomicAdd(P.acc + ACC_ULB, ulb);
  GM_TRACE(51);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(52);
  // ---- P2: project b; w = A_e^-1 b_e; push fluxes into b_S; u_S^T b_S; Z^T b_S
  const double alpha = __ldcg(P.acc + ACC_ULB);
  double pus = 0;
#pragma unroll 1
  for (long long el = rank + (long long)grp * G; el < g.nel; el += (long long)ngrp * G) {
    const int e = (int)el;
    for (int q = part * 32 + lane; q < nn; q += 32 * W) {
      const long long gq = el * nn + q;
      const double v = P.b[gq] - alpha * (P.adjoint ? P.what[gq] : P.uL[gq]);
      P.b[gq] = v;
      f.B[(q / n) * ld + q % n] = v;
    }
    item_sync(grp, W);
    elem_fd(P.fd, g, e, f, lane, part, W, grp);
    // flux of w into the slot (nbr, opp F, t): -tau' (p' w - n_F . grad w) with
    // tau', p' of the neighbour's face opp F and the gradient in e's own size
#pragma unroll 1
    for (int i = part * 32 + lane; i < M; i += 32 * W) {
      const int F = i / n, t = i - F * n, e2 = dev_neighbour(g, e, F);
      double val = 0;
      if (e2 >= 0) {
        int aa, bb;
        face_node(n, F, t, &aa, &bb);
        const double* fn = face_geo(g, e2, F ^ 1);
        val = P.adjoint ? f.U[bb * ld + aa]
                        : -fn[0] * (fn[1] * f.U[bb * ld + aa] -
                                    normal_deriv_ld(g, P.D, f.U, ld, F, t, face_geo(g, e, F)[2]));
        const size_t sl = (size_t)e2 * M + (F ^ 1) * n + t;
        P.bS[sl] = val;
        pus += P.uS[sl] * val;
        val *= dev_zw(g, e2, F ^ 1);  // its weight in Z^T b_S
      }
      f.p[i] = val;
    }
    item_sync(grp, W);
    if (part == 0) {  // face F summed by the eight lanes 8 F + r
      const int F = lane >> 3, j = dev_iface(g, e, F);
      double sum = 0;
#pragma unroll 1
      for (int t = lane & 7; t < n; t += 8) sum += f.p[F * n + t];
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if ((lane & 7) == 0 && j >= 0) atomicAdd(P.cb + j, sum);
    }
    item_sync(grp, W);
  }
  pus = warp_sum(pus);
  if ((threadIdx.x & 31) == 0 && pus != 0.0) atomicAdd(P.acc + ACC_USBS, pus);
  GM_TRACE(53);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(54);
  // ---- P3: c_hat_b = C^+ Z^T (b_S - beta u_S)
  const double beta = __ldcg(P.acc + ACC_USBS);
  if (a.precond == 2) {
#pragma unroll 1
    for (int j = rank * blockDim.x + threadIdx.x; j < (int)g.d; j += G * blockDim.x)
      a.c[j] = __ldcg(P.cb + j) - beta * P.ZtuS[j];
    GM_TRACE(55);
    if (!team_sync(a, epoch)) return false;
    GM_TRACE(56);
    if (!coarse_solve(a, s, epoch, a.c, a.chat)) return false;  // a.c -> a.chat
    GM_TRACE(58);
#pragma unroll 1
    for (int j = rank * blockDim.x + threadIdx.x; j < (int)g.d; j += G * blockDim.x)
      P.chatb[j] = __ldcg(a.chat + j);
  }
  // ---- P4: owner entries: project b_S, rhs = P b_S
  double bsn = 0, rgn = 0;
#pragma unroll 1
  for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
    const int4 en = owned_entry(a, i);
    const int sl = en.x;
    if (sl < 0) continue;
    if (en.z < 0) {  // slot on the physical boundary
      P.bS[sl] = 0.0;
      P.rg[sl] = 0.0;
      if (P.rg32) P.rg32[sl] = 0.f;
      continue;
    }
    const double v = __ldcg(P.bS + sl) - beta * P.uS[sl];
    P.bS[sl] = v;
    bsn += v * v;
    const double r = deflate_value(a, v, a.precond == 2 ? a.chat : nullptr, en);  // b_S - S Z c_hat_b
    P.rg[sl] = r;
    if (P.rg32) P.rg32[sl] = (float)r;
    rgn += r * r;
  }
  bsn = warp_sum(bsn);
  rgn = warp_sum(rgn);
  if ((threadIdx.x & 31) == 0) {
    if (bsn != 0.0) atomicAdd(P.acc + ACC_BSN, bsn);
    if (rgn != 0.0) atomicAdd(P.acc + ACC_RGN, rgn);
  }
  return true;
}

__device__ SMPM_BODY bool post_body(const PrePostArgs& P, unsigned char* smraw, unsigned& epoch) {
  const GmresArgs<double>& a = P.ga;
  const Smem<double> s = carve(a, smraw);
  no_resident(a, s);
  const DevGeo& g = a.g;
  const int n = g.n, nn = n * n, M = g.M, G = a.G, rank = team_rank(a);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = P.W_fd, grp = warp / W, part = warp % W,
            ngrp = kGmresThreads / 32 / W;
  const FdItem f = fd_item(s.end, n, W, grp);
  const int ld = fd_ld(n), kt_n = digit_tiles(M);
  int trace_n = 0;
  // ---- Q1-Q4: x_S
  if (P.assembled) {
    // x_S given (iterative refinement)
  } else if (a.precond == 0) {
#pragma unroll 1
    for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
      const int sl = entry_slot(a, i);
      if (sl >= 0) P.xs[sl] = __ldcg(a.x + sl);
    }
  } else {
    black_phase(a, s, (const double*)a.x, 1.0, (const double*)nullptr);
    if (a.precond == 1) {
      GM_TRACE(61);
      if (!team_sync(a, epoch)) return false;
      GM_TRACE(62);
#pragma unroll 1
      for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
        const int sl = entry_slot(a, i);
        if (sl >= 0) P.xs[sl] = __ldcg(a.t + sl);
      }
    } else {
      // white step and coarse solve of y = S t, then x_S = t - Z (c_hat - c_hat_b)
      if (!apply_op(a, s, a.x, 1.0, true, trace_n, epoch)) return false;
#pragma unroll 1
      for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
        const int4 en = owned_entry(a, i);
        if (en.x < 0) continue;
        P.xs[en.x] = en.z < 0 ? 0.0 : __ldcg(a.t + en.x) - entry_zw(g, en) * (__ldcg(a.chat + en.z) - P.chatb[en.z]);
      }
    }
  }
  GM_TRACE(63);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(64);
  // ---- Q5: recovery u_e = A_e^-1 (b_e - E_e x_S), residual b_S - S x_S, mean
  double pm = 0, pr = 0;
#pragma unroll 1
  for (long long el = rank + (long long)grp * G; el < g.nel; el += (long long)ngrp * G) {
    const int e = (int)el, ct = __ldg(a.dm.tcls + e);
    for (int q = part * 32 + lane; q < nn; q += 32 * W) f.B[(q / n) * ld + q % n] = P.b[el * nn + q];
    for (int i = part * 32 + lane; i < M; i += 32 * W) f.p[i] = __ldcg(P.xs + el * M + i);
    item_sync(grp, W);
#pragma unroll 1
    for (int F = 0; F < 4; ++F) {  // faces in turn: a corner node takes both slots
      if (dev_neighbour(g, e, F) >= 0) {
        if (!P.adjoint) {
#pragma unroll 1
          for (int t = part * 32 + lane; t < n; t += 32 * W) {
            int aa, bb;
            face_node(n, F, t, &aa, &bb);
            f.B[bb * ld + aa] -= f.p[F * n + t];
          }
        } else {
          // - B_e^T mu: the slot (F, t) feeds, through B, the flux
          // -tau' (p' u(q) - n_F.grad u(q)) at face node q = (F, t), tau' and p'
          // of the neighbour's face opp F; its transpose touches the n nodes
          // on the normal line through q
          const double* fn = face_geo(g, dev_neighbour(g, e, F), F ^ 1);
          const double tau = fn[0], pw = fn[1];
          const double sc = face_geo(g, e, F)[2];
          const int drow = (F & 1) ? n - 1 : 0;   // D row of the face end
          const double sgn = (F & 1) ? 1.0 : -1.0;  // outward normal along the axis
#pragma unroll 1
          for (int idx = part * 32 + lane; idx < nn; idx += 32 * W) {
            const int t = idx / n, k = idx % n;
            const double v = f.p[F * n + t];
            const double dn = sgn * sc * __ldg(P.D + drow * n + k);
            const double coef = -tau * ((k == drow ? pw : 0.0) - dn);
            f.B[F < 2 ? t * ld + k : k * ld + t] -= coef * v;
          }
        }
      }
      item_sync(grp, W);
    }
    elem_fd(P.fd, g, e, f, lane, part, W, grp);
    for (int q = part * 32 + lane; q < nn; q += 32 * W) {
      const double u = f.U[(q / n) * ld + q % n];
      P.u[el * nn + q] = u;
      pm += (P.adjoint ? P.uL[el * nn + q] : P.what[el * nn + q]) * u;
    }
    // (S x_S) on the slots facing e: x_S + T_e x_S,e
    const int E = pack_one<double>(f.Bf, f.p, M, lane, part, W);
    item_sync(grp, W);
#pragma unroll 1
    for (int mt = part; mt < kt_n; mt += W) {
      const int row = tile1_row(mt, lane, M);
      Facing<double> fc{};
      fc.sl = -1;
      if (row >= 0) fc = facing_entry(g, e, row, P.xs, P.xs);
      const double z = digits_tile1<double>(a.dm.T + (size_t)ct * digit_words<double>(M, M), a.dm.Te + (size_t)ct * M, f.Bf,
                                            M, kt_n, mt, lane, E);
      if (fc.sl < 0) continue;
      const double rr = P.bS[fc.sl] - (fc.t + z);
      pr += rr * rr;
    }
    item_sync(grp, W);
  }
  pm = warp_sum(pm);
  pr = warp_sum(pr);
  if ((threadIdx.x & 31) == 0) {
    if (pm != 0.0) atomicAdd(P.acc + ACC_MEAN, pm);
    if (pr != 0.0) atomicAdd(P.acc + ACC_RES, pr);
  }
  GM_TRACE(65);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(66);
  // ---- Q6: zero GLL-weighted mean (adjoint: projection out of u_L, dl/dg)
  const double mean = __ldcg(P.acc + ACC_MEAN);
  if (!P.adjoint) {
#pragma unroll 1
    for (long long e = rank; e < g.nel; e += G)
      for (int q = threadIdx.x; q < nn; q += blockDim.x) P.u[e * nn + q] -= mean;
    return true;
  }
#pragma unroll 1
  for (long long e = rank; e < g.nel; e += G) {
    if (P.gg)
      for (int i = threadIdx.x; i < M; i += blockDim.x) {
        const int F = i / n, t = i % n;
        double v = 0;
        if (dev_neighbour(g, (int)e, F) < 0) {
          int aa, bb;
          face_node(n, F, t, &aa, &bb);
          const long long q = e * nn + bb * n + aa;
          v = face_geo(g, (int)e, F)[0] * (__ldcg(P.u + q) - mean * P.uL[q]);
        }
        P.gg[e * M + i] = v;
      }
    __syncthreads();
    for (int q = threadIdx.x; q < nn; q += blockDim.x) P.u[e * nn + q] -= mean * P.uL[e * nn + q];
  }
  return true;
}

inline size_t prepost_smem_bytes(int m, int M, int n, int ES, int W, int W_fd, long long d, bool w_global = false) {
  return gmres_smem_bytes<double>(m, M, n, ES, W, 0, d, w_global) +
         (size_t)(kGmresThreads / 32 / W_fd) * fd_item_bytes(n, W_fd);
}
