// Lockstep GMRES over R right-hand sides ("columns") of one grid: the R
// Arnoldi processes of Algorithm 2 / 3 (GMRES on S M^-1 or P S M^-1) advance
// together, one step at a time, in ONE persistent cooperative launch, so that
// every operator matrix (G_b, X_b, T_e, the coarse C^+) is read once per step
// for all R columns and the five team barriers of a step (seven with C^+ by strips)
// are shared.  Each element product becomes a small dense GEMM: the M x M matrix
// times a tile of eight columns.
//
// Per column, everything of the single-column kernel is kept: its own basis,
// Hessenberg column, FP64 Givens rotations, residual estimate, convergence,
// breakdown and NaN flags, and its own restarts.  A column that converges
// stops (its scale is set to zero: its later basis vectors are zero and its
// Givens state is frozen); the step loop ends when every column has stopped,
// and a restart cycle restarts only the columns still running.  In exact
// arithmetic the iterates of column rho are those of a single-column solve of that
// right-hand side (same phases, same CGS2, Pythagorean norm and stopping
// criterion).  Rounding differs: v_j is formed at the start of step j, the residual
// norm comes from a rotation per step, the block solves run in stages where a
// single solve may take the whole inverse, and the sums meet in another order.
//
// Layouts: column rho of a kp-vector at base + rho * vs; of a d-vector at
// base + rho * ds.  The basis lives in global memory (L2 / HBM): CTA rank's
// slice of basis vector l, column rho at V + ((rank (m+1) + l) R + rho) ES;
// w likewise (see lk_w); ES is a multiple of 4 here.
// Element work items are (owned element, eight columns); a group of W warps
// takes items grp, grp + ngrp, ...; an item's tiles live in the group's
// shared scratch.
#pragma once
// Included inside the anonymous namespace of each translation unit that uses it,
// after smpm_gmres.cuh.

constexpr int kLockMaxCols = 16;  // columns of one lockstep launch

struct LockColState {  // per column, written by the team's rank 0 at the end
  double beta0, tolabs, resid;
  int its, converged, breakdown, nan, cycles;
  int its_total;  // Arnoldi steps summed over the launches of a solve (zero before the first)
};

template <typename S>
struct LockArgs {
  GmresArgs<S> a;  // geometry, ownership, matrices, team, barrier, err, precond, m, maxit, tol;
                   // rhs, x, t, y, vglob: column 0 (stride vs); c, chat: column 0 (stride ds);
                   // acc: (2m+1) R (m+3) FP64 accumulators (zero on entry)
  int R;           // columns (<= kLockMaxCols)
  int W_item, ngrp;  // warps per element work item (eight columns of an element), groups of that many warps
  size_t wb_bytes;   // shared scratch of the groups
  long long vs, ds;
  S* V;            // basis, G (m+1) R ES
  S* W;            // w (w2 in its place): G R ES, unless w_smem
  int w_smem;
  LockColState* cs;  // R
  double* Rh;        // R m (m+1): Hessenberg R factor per column (written by rank 0)
  double* yv;        // R m: least-squares solution per column
  const int* done;   // per column (stride done_stride ints): nonzero -> the column does not run
  int done_stride;
};

template <typename S>
struct LockSmem {
  double *gcs, *gsn, *gg, *invb, *h1, *h2, *hs1, *hs2, *colv;  // [rho * m3 + l]
  double* misc;                                                // [rho * 8 + k]
  double* scl;                                                 // scale of each column's input
  int* jc;                                                     // steps of the column in this cycle
  int* active;
  int* flags;  // [0]: any column active
  unsigned char* wb;  // group scratch (lock_group_bytes each)
};

// entries from one column of a staged tile to the next: 8 modulo 16, so the
// lanes of a pack (eight columns, consecutive rows) spread over the banks
__host__ __device__ constexpr int lock_ld(int len) { return (len + 7) / 16 * 16 + 8; }
// scratch of a group: packed columns (of M rows, or of the four faces), the
// tiles [p; q] and r1 of eight columns (a white item: contributions to c)
template <typename S>
__host__ __device__ constexpr size_t lock_bf_bytes(int M, int n) {
  const int a = digit_bwords<S>(M), b = 4 * digit_bwords<S>(n);
  return sizeof(uint4) * (size_t)(a > b ? a : b);
}
template <typename S>
__host__ __device__ constexpr size_t lock_group_bytes(int M, int n) {
  const size_t black = 8 * sizeof(S) * (size_t)(lock_ld(2 * M) + lock_ld(M)), white = 8 * (sizeof(double) + sizeof(S)) * (size_t)lock_ld(M);
  return lock_bf_bytes<S>(M, n) + (black > white ? black : white);
}

// shared memory beside the group scratch
inline size_t lock_fixed_bytes(int m, int R) {
  const size_t m3 = m + 3, dbl = 9 * m3 * R + 9 * (size_t)R, ints = 2 * (size_t)R + 4;
  return dbl * sizeof(double) + ints * sizeof(int) + 16 + 128;
}

// Warps per item and groups for `items` items per CTA: every warp busy, as many
// groups as `room` bytes of scratch hold.  Returns the scratch bytes (0: not
// even one group fits).
template <typename S>
inline size_t lock_groups(int M, int n, long long items, size_t room, int* W, int* ngrp) {
  const int warps = kGmresThreads / 32;
  const size_t per = lock_group_bytes<S>(M, n);
  int w = 1;
  while (w < warps && (items * w * 2 <= warps || (warps / w) * per > room)) w *= 2;
  *W = w;
  *ngrp = warps / w;
  return *ngrp * per <= room ? *ngrp * per : 0;
}

template <typename S>
__device__ LockSmem<S> lock_carve(const LockArgs<S>& A, unsigned char* raw) {
  LockSmem<S> s;
  const int m3 = A.a.m + 3, R = A.R;
  double* d = reinterpret_cast<double*>(raw);
  s.gcs = d; d += (size_t)m3 * R;
  s.gsn = d; d += (size_t)m3 * R;
  s.gg = d; d += (size_t)m3 * R;
  s.invb = d; d += (size_t)m3 * R;
  s.h1 = d; d += (size_t)m3 * R;
  s.h2 = d; d += (size_t)m3 * R;
  s.hs1 = d; d += (size_t)m3 * R;
  s.hs2 = d; d += (size_t)m3 * R;
  s.colv = d; d += (size_t)m3 * R;
  s.misc = d; d += 8 * (size_t)R;
  s.scl = d; d += R;
  int* ip = reinterpret_cast<int*>(d);
  s.jc = ip; ip += R;
  s.active = ip; ip += R;
  s.flags = ip; ip += 4;
  s.wb = reinterpret_cast<unsigned char*>((reinterpret_cast<size_t>(ip) + 15) & ~size_t(15));
  return s;
}

template <typename S>
__device__ __forceinline__ S* lk_basis(const LockArgs<S>& A, int l, int rho) {
  return A.V + (((size_t)team_rank(A.a) * (A.a.m + 1) + l) * A.R + rho) * A.a.ES;
}
// w of column rho, then w2 in its place: in the groups' scratch when it fits
// (it lives from the deflation to the next step's v_j, while the element phases
// do not run), else in global memory.
template <typename S>
__device__ __forceinline__ S* lk_w(const LockArgs<S>& A, const LockSmem<S>& s, int rho) {
  return A.w_smem ? reinterpret_cast<S*>(s.wb) + (size_t)rho * A.a.ES
                  : A.W + ((size_t)team_rank(A.a) * A.R + rho) * A.a.ES;
}

// four consecutive entries (16-byte aligned; ES is a multiple of 4)
template <typename S>
struct alignas(16) Quad {
  S v[4];
};
__device__ __forceinline__ Quad<double> ld_quad(const double* p) {  // basis: streamed past L1
  const double2 a = __ldcg(reinterpret_cast<const double2*>(p)), b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
  return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ Quad<float> ld_quad(const float* p) {
  const float4 a = __ldcg(reinterpret_cast<const float4*>(p));
  return {a.x, a.y, a.z, a.w};
}
template <typename S>
__device__ __forceinline__ Quad<S> ld_quad_w(const S* p) {  // w: shared or global, written by this CTA
  return *reinterpret_cast<const Quad<S>*>(p);
}

// Black block solves for all columns: items (owned block k, eight columns), a
// group of W warps each.  Column rho's input is sc[rho] * (the basis slice when
// own, else the global vector src).  t = M^-1 v on the block: r1 = p - X q,
// a = G r1, z = T_e a, t = [a; q - z]; the products run on the tensor cores
// (smpm_digits.cuh), eight columns to a tile.
// Bound by the row tiles' chains (first digits from L2, unpacking, 36 products of
// 8 cycles per k tile in FP64): at M = 96, four blocks and eight columns 116,000 SM
// cycles -- gather 14, X 27, packing 10, G and T 25 each per group of two warps --
// against 492,000 with FP64 FMA.
template <typename S>
__device__ SMPM_PHASE void lk_black(const LockArgs<S>& A, const LockSmem<S>& s, const S* src, const double* sc, int jbasis) {
  const GmresArgs<S>& a = A.a;
  const DevGeo& g = a.g;
  const int M = g.M, n = g.n, G = a.G, rank = team_rank(a), R = A.R, Q = (R + 7) / 8, W = A.W_item;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W;
  const int ldp = lock_ld(2 * M), ldr = lock_ld(M), kt_n = digit_tiles(M), kf_n = digit_tiles(n);
  unsigned char* base = s.wb + (size_t)grp * lock_group_bytes<S>(M, n);
  uint4* Bf = reinterpret_cast<uint4*>(base);
  S* P = reinterpret_cast<S*>(base + lock_bf_bytes<S>(M, n));  // [p; q]: column c at c ldp
  S* Rr = P + 8 * ldp;                                         // r1, then a: column c at c ldr
  for (int it = grp; it < a.nown_b * Q; it += A.ngrp) {
    const int k = it / Q, c0 = (it % Q) * 8, nc = min(8, R - c0);
    const int ib = rank + k * G;
    if (ib >= a.nblack) continue;
    const int e = a.black[ib], cb = a.dm.bcls[ib], ct = a.dm.tcls[e];
    for (int i = part * 32 + lane; i < 2 * M; i += 32 * W) {  // an entry's eight columns together
      S v[8];
      const int sl = jbasis >= 0 ? 0 : block_entry(a, ib, i).x;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int rho = c0 + min(c, nc - 1);
        v[c] = jbasis >= 0 ? lk_basis(A, jbasis, rho)[k * 2 * M + i] : sl >= 0 ? ldcg(src + rho * A.vs + sl) : S(0);
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) P[c * ldp + i] = c < nc ? (S)(sc[c0 + c] * (double)v[c]) : S(0);
    }
    item_sync(grp, W);
    for (int F = part; F < 4; F += W) {  // r1 = p - X q, face by face
      uint4* Bq = Bf + F * digit_bwords<S>(n);
      const S* q = P + M + F * n;
      const int E = pack_cols<S>(Bq, q, 1, ldp, n, 8, lane, 0, 1);
      for (int mt = 0; mt < kf_n; ++mt) {
        const Tile8<S> t = digits_tile8<S>(a.dm.X + ((size_t)cb * 4 + F) * digit_words<S>(n, n),
                                           a.dm.Xe + ((size_t)cb * 4 + F) * n, Bq, n, kf_n, mt, lane, E);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int r = mt * 16 + (lane >> 2) + 8 * (v >> 1), c = 2 * (lane & 3) + (v & 1);
          if (r < n) Rr[c * ldr + F * n + r] = P[c * ldp + F * n + r] - t.z[v];
        }
      }
    }
    item_sync(grp, W);
    for (int stage = 0; stage < 2; ++stage) {  // a = G r1, then z = T_e a and t = q - z on the facing slots
      const int E = pack_cols<S>(Bf, Rr, 1, ldr, M, 8, lane, part, W);
      const uint4* Am = stage == 0 ? a.dm.G + (size_t)cb * digit_words<S>(M, M) : a.dm.T + (size_t)ct * digit_words<S>(M, M);
      const short* er = stage == 0 ? a.dm.Ge + (size_t)cb * M : a.dm.Te + (size_t)ct * M;
      item_sync(grp, W);
      for (int mt = part; mt < kt_n; mt += W) {
        int sl[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = mt * 16 + (lane >> 2) + 8 * h;
          sl[h] = r >= M ? -1 : stage == 0 ? e * M + r : block_entry(a, ib, M + r).x;
        }
        const Tile8<S> t = digits_tile8<S>(Am, er, Bf, M, kt_n, mt, lane, E);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int r = mt * 16 + (lane >> 2) + 8 * (v >> 1), c = 2 * (lane & 3) + (v & 1);
          if (r >= M) continue;
          if (stage == 0) Rr[c * ldr + r] = t.z[v];
          if (c < nc && sl[v >> 1] >= 0)
            a.t[(c0 + c) * A.vs + sl[v >> 1]] = stage == 0 ? t.z[v] : P[c * ldp + M + r] - t.z[v];
        }
      }
      item_sync(grp, W);
    }
  }
  __syncthreads();
}

// White elements for all columns: y = S t on the black slots facing e,
// y = sc * v on e's own slots, c = Z^T y on e's interfaces (with_c).
template <typename S>
__device__ SMPM_PHASE void lk_white(const LockArgs<S>& A, const LockSmem<S>& s, const S* v0, const double* sc, bool with_c) {
  const GmresArgs<S>& a = A.a;
  const DevGeo& g = a.g;
  const int M = g.M, n = g.n, G = a.G, rank = team_rank(a), R = A.R, Q = (R + 7) / 8, W = A.W_item;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W;
  const int kt_n = digit_tiles(M), ldc = lock_ld(M);
  unsigned char* base = s.wb + (size_t)grp * lock_group_bytes<S>(M, n);
  uint4* Bf = reinterpret_cast<uint4*>(base);
  double* ci = reinterpret_cast<double*>(base + lock_bf_bytes<S>(M, n));  // contributions to c: column c at c ldc
  S* Tt = reinterpret_cast<S*>(ci + 8 * ldc);                             // t on e's slots: column c at c ldc
  for (int it = grp; it < a.nown_w * Q; it += A.ngrp) {
    const int k = it / Q, c0 = (it % Q) * 8, nc = min(8, R - c0);
    const int iw = rank + k * G;
    if (iw >= a.nwhite) continue;
    const int e = a.white[iw], ct = a.dm.tcls[e];
    for (int i = part * 32 + lane; i < M; i += 32 * W) {
      S v[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = ldcg(a.t + (c0 + min(c, nc - 1)) * A.vs + (size_t)e * M + i);
#pragma unroll
      for (int c = 0; c < 8; ++c) Tt[c * ldc + i] = v[c];
    }
    item_sync(grp, W);
    const int E = pack_cols<S>(Bf, Tt, 1, ldc, M, nc, lane, part, W);
    item_sync(grp, W);
    for (int mt = part; mt < kt_n; mt += W) {
      Facing<S> f[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int r = min(mt * 16 + (lane >> 2) + 8 * (v >> 1), M - 1), c = min(2 * (lane & 3) + (v & 1), nc - 1);
        f[v] = facing_entry(g, e, r, v0 + (c0 + c) * A.vs, a.t + (c0 + c) * A.vs);
      }
      const Tile8<S> t = digits_tile8<S>(a.dm.T + (size_t)ct * digit_words<S>(M, M), a.dm.Te + (size_t)ct * M, Bf, M, kt_n,
                                         mt, lane, E);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int r = mt * 16 + (lane >> 2) + 8 * (v >> 1), c = 2 * (lane & 3) + (v & 1), rho = c0 + c;
        if (r >= M || c >= nc) continue;
        const S vo = (S)(sc[rho] * (double)f[v].v);
        a.y[rho * A.vs + (size_t)e * M + r] = vo;
        double c1 = 0;
        if (f[v].sl >= 0) {
          const S ys = f[v].t + t.z[v];
          a.y[rho * A.vs + f[v].sl] = ys;
          c1 = facing_c(g, f[v], vo, ys);
        }
        ci[c * ldc + r] = c1;
      }
    }
    item_sync(grp, W);
    if (with_c && part == 0 && lane < 4 * nc) {  // face F of column c summed by lane c * 4 + F
      const int c = lane / 4, F = lane % 4, j = dev_iface(g, e, F);
      if (j >= 0) {
        double sum = 0;
        for (int tt = 0; tt < n; ++tt) sum += ci[c * ldc + F * n + tt];
        a.c[(c0 + c) * A.ds + j] = sum;
      }
    }
    item_sync(grp, W);
  }
  __syncthreads();
}

// c_hat = C^+ c for all columns: the CTA takes a contiguous range of rows,
// one warp per row; lanes read consecutive entries of the row (H row-major)
// and of each column's c, two entries per lane and step, and the loads of the
// next step are issued before the FMAs of this one (software pipelining); the
// R partial sums meet in warp shuffles.
template <typename S, typename HT>
__device__ SMPM_PHASE void lk_coarse_h(const LockArgs<S>& A, const HT* H) {
  const GmresArgs<S>& a = A.a;
  const int d = (int)a.g.d, R = A.R;
  const int per = (d + a.G - 1) / a.G;
  const int r0 = team_rank(a) * per, r1 = min(d, r0 + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  constexpr int U = 2, CG = 8;  // entries per lane and step; columns per pass over the row
  const int nfull = d / (32 * U);
  for (int r = r0 + warp; r < r1; r += nwarps) {
    const HT* hr = H + (size_t)r * ((d + 3) & ~3);
    for (int c0 = 0; c0 < R; c0 += CG) {
      const int nc = min(CG, R - c0);
      const double* cb = a.c + (size_t)c0 * A.ds;
      HT acc[CG];
#pragma unroll
      for (int c = 0; c < CG; ++c) acc[c] = 0;
      HT h[U], cv[CG][U];
      auto load = [&](int st) {
        const int j = st * 32 * U + lane;
#pragma unroll
        for (int u = 0; u < U; ++u) h[u] = __ldg(hr + j + 32 * u);
#pragma unroll
        for (int c = 0; c < CG; ++c)
          if (c < nc)
#pragma unroll
            for (int u = 0; u < U; ++u) cv[c][u] = (HT)__ldcg(cb + c * A.ds + j + 32 * u);
      };
      if (nfull > 0) load(0);
      for (int st = 0; st < nfull; ++st) {
        HT hh[U], cc[CG][U];
#pragma unroll
        for (int u = 0; u < U; ++u) hh[u] = h[u];
#pragma unroll
        for (int c = 0; c < CG; ++c)
#pragma unroll
          for (int u = 0; u < U; ++u) cc[c][u] = cv[c][u];
        if (st + 1 < nfull) load(st + 1);
#pragma unroll
        for (int c = 0; c < CG; ++c)
          if (c < nc)
#pragma unroll
            for (int u = 0; u < U; ++u) acc[c] += hh[u] * cc[c][u];
      }
      for (int j = nfull * 32 * U + lane; j < d; j += 32) {
        const HT hv = __ldg(hr + j);
#pragma unroll
        for (int c = 0; c < CG; ++c)
          if (c < nc) acc[c] += hv * (HT)__ldcg(cb + c * A.ds + j);
      }
#pragma unroll
      for (int c = 0; c < CG; ++c) {
        if (c < nc) {
          const double v = (double)warp_sum(acc[c]);
          if (lane == 0) a.chat[(c0 + c) * A.ds + r] = v;
        }
      }
    }
  }
}

// FP32 columns: the coarse inverse's FP32 copy, FP32 products and sums.  The R
// coarse vectors are converted to FP32 once per CTA, a chunk of dc entries of
// every column at a time, into the groups' idle scratch (converting them on every
// row's pass costs as much as FP64 products); each warp keeps its rows'
// partial sums in c_hat across the chunks.
template <typename S>
__device__ SMPM_PHASE void lk_coarse32_staged(const LockArgs<S>& A, float* cf, int dc) {
  const GmresArgs<S>& a = A.a;
  const int d = (int)a.g.d, R = A.R;
  const int per = (d + a.G - 1) / a.G;
  const int r0 = team_rank(a) * per, r1 = min(d, r0 + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  constexpr int CG = 8;
  for (int j0 = 0; j0 < d; j0 += dc) {
    const int len = min(dc, d - j0);
    for (int i = threadIdx.x; i < R * len; i += blockDim.x) {
      const int c = i / len, j = i - c * len;
      cf[(size_t)c * dc + j] = (float)__ldcg(a.c + (size_t)c * A.ds + j0 + j);
    }
    __syncthreads();
    for (int r = r0 + warp; r < r1; r += nwarps) {
      const float* hr = a.H + (size_t)r * ((d + 3) & ~3) + j0;
      for (int c0 = 0; c0 < R; c0 += CG) {
        const int nc = min(CG, R - c0);
        const float* cc = cf + (size_t)c0 * dc;
        float acc[CG];
#pragma unroll
        for (int c = 0; c < CG; ++c) acc[c] = 0.f;
        int j = lane;
        for (; j + 32 * 7 < len; j += 32 * 8) {  // eight entries per lane per step, loaded first
          float h[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) h[u] = __ldg(hr + j + 32 * u);
#pragma unroll
          for (int c = 0; c < CG; ++c)
            if (c < nc)
#pragma unroll
              for (int u = 0; u < 8; ++u) acc[c] += h[u] * cc[(size_t)c * dc + j + 32 * u];
        }
        for (; j < len; j += 32) {
          const float hv = __ldg(hr + j);
#pragma unroll
          for (int c = 0; c < CG; ++c)
            if (c < nc) acc[c] += hv * cc[(size_t)c * dc + j];
        }
#pragma unroll
        for (int c = 0; c < CG; ++c)
          if (c < nc) {
            const float v = warp_sum(acc[c]);
            double* out = a.chat + (size_t)(c0 + c) * A.ds + r;
            if (lane == 0) *out = (j0 == 0 ? 0.0 : *out) + (double)v;
          }
      }
    }
    __syncthreads();  // the scratch takes the next chunk, or the next phase
  }
}

// As row_dots for NC columns at a time: eight lanes per row or more, as far as
// the rows leave threads; lane l < 8 of a group ends with column l's sum (the
// partial sums are exchanged halving the columns each time: 7 adds per row and
// lane of eight instead of 24).  x: column c of the staged vectors at c * xld.
template <typename T, int NC, typename Get, typename Put>
__device__ __forceinline__ void row_dots_cols(int r0, int r1, int xld, Get&& get, Put&& put) {
  constexpr int V = 16 / (int)sizeof(T);
  int P = 8;
  while (P < 32 && 2 * P * (r1 - r0) <= (int)blockDim.x) P *= 2;
  const int lane = threadIdx.x % P, grp = threadIdx.x / P, ngrp = blockDim.x / P;
  for (int rb = 0; rb < r1 - r0; rb += ngrp) {  // uniform trip count per warp
    const int r = r0 + rb + grp;
    const T* a = nullptr;
    const T* x = nullptr;
    int len = 0;
    if (r < r1) get(r, a, x, len);
    T acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = T(0);
    for (int j = V * lane; j < len; j += 2 * V * P) {
      T h[2][V];
      ld_vec<false>(a + j, h[0]);
      const bool two = j + V * P < len;
      if (two) ld_vec<false>(a + j + V * P, h[1]);
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[c] += h[0][v] * x[(size_t)c * xld + j + v];
      if (two) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[c] += h[1][v] * x[(size_t)c * xld + j + V * P + v];
      }
    }
    // lane keeps the half of the columns that its bit o selects; lanes beyond
    // the columns add the halves that are left
    int w = NC;
    for (int o = P / 2; o >= 8; o >>= 1)  // lanes beyond eight first
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const int half = w > 1 ? w / 2 : 1;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= half) break;
        const T keep = (w > 1 && up) ? acc[(c + half) % NC] : acc[c];
        const T give = (w > 1 && !up) ? acc[(c + half) % NC] : acc[c];
        const T got = __shfl_xor_sync(0xffffffffu, give, o);
        acc[c] = keep + got;
      }
      if (w > 1) w = half;
    }
    // column of this lane: the top log2(NC) bits of lane
    constexpr int S3 = NC == 8 ? 0 : NC == 4 ? 1 : NC == 2 ? 2 : 3;
    if (len > 0 && lane < 8 && (lane & ((1 << S3) - 1)) == 0) put(r, lane >> S3, acc[0]);
  }
}

// C^+ by strips (coarse_strips) for all columns, NC of them at a time staged
// in st (each phase's stretch of every column, xld entries apart).
template <typename S, int NC>
__device__ SMPM_PHASE bool lk_coarse_strips_nc(const LockArgs<S>& A, void* st, unsigned& epoch) {
  using T = typename std::conditional<sizeof(S) == 4, float, double>::type;
  constexpr int V = 16 / (int)sizeof(T);
  const GmresArgs<S>& a = A.a;
  const auto& k = a.strips;
  T* xs = reinterpret_cast<T*>(st);
  const int G = a.G, rank = team_rank(a), d = (int)a.g.d, R = A.R;
  const int srow = k.h * k.row, RS = k.m + 2 * k.mx;
  const size_t gst = 2 * (size_t)k.p * k.mx + 1;  // gsep per column
  {
    const int n1 = k.p * RS, per = (n1 + G - 1) / G, r0 = min(n1, rank * per), r1 = min(n1, r0 + per);
    if (r0 < r1) {
      const int b0 = (r0 / RS) * srow, b1 = min(d, ((r1 - 1) / RS + 1) * srow), xld = b1 - b0 + V;
      for (int c0 = 0; c0 < R; c0 += NC) {
        __syncthreads();
        for (int q = threadIdx.x; q < NC * xld; q += blockDim.x) {
          const int c = q / xld, j = q - c * xld;
          xs[q] = (c0 + c < R && b0 + j < b1) ? (T)__ldcg(a.c + (c0 + c) * A.ds + b0 + j) : T(0);
        }
        __syncthreads();
        row_dots_cols<T, NC>(
            r0, r1, xld,
            [&](int r, const T*& row, const T*& x, int& len) {
              const int i = r / RS, l = r - i * RS, mi = min(k.m, d - i * srow);
              const bool on = l < k.m ? l < mi : (l < k.m + k.mx ? i > 0 : i < k.p - 1);
              row = k.N + (size_t)r * k.ldn;
              x = xs + i * srow - b0;
              len = on ? mi : 0;
            },
            [&](int r, int c, T sum) {
              if (c0 + c >= R) return;
              const int i = r / RS, l = r - i * RS;
              if (l < k.m) a.chat[(c0 + c) * A.ds + i * srow + l] = (double)sum;
              else a.gsep[(c0 + c) * gst + 2 * (size_t)i * k.mx + (l - k.m)] = (double)sum;
            });
      }
    }
    if (!team_sync(a, epoch)) return false;
  }
  {
    const int n2 = k.ns + 1, per = (n2 + G - 1) / G, r0 = min(n2, rank * per), r1 = min(n2, r0 + per);
    if (r0 < r1) {
      const int xld = k.ns + V;
      for (int c0 = 0; c0 < R; c0 += NC) {
        __syncthreads();
        for (int q = threadIdx.x; q < NC * xld; q += blockDim.x) {
          const int c = q / xld, j = q - c * xld;
          T v = T(0);
          if (c0 + c < R && j < k.ns) {
            const int sp = j / k.mx, e = j - sp * k.mx;
            const double* up = a.gsep + (c0 + c) * gst + (2 * (size_t)sp + 1) * k.mx + e;
            v = (T)(__ldcg(a.c + (c0 + c) * A.ds + (sp + 1) * srow - k.mx + e) - __ldcg(up) - __ldcg(up + k.mx));
          }
          xs[q] = v;
        }
        __syncthreads();
        row_dots_cols<T, NC>(
            r0, r1, xld,
            [&](int r, const T*& row, const T*& x, int& len) {
              row = k.Hs + (size_t)r * k.lds;
              x = xs;
              len = k.ns;
            },
            [&](int r, int c, T sum) {
              if (c0 + c >= R) return;
              if (r == k.ns) a.gsep[(c0 + c) * gst + gst - 1] = (double)sum;
              else a.chat[(c0 + c) * A.ds + (r / k.mx + 1) * srow - k.mx + r % k.mx] = (double)sum;
            });
      }
    }
    if (!team_sync(a, epoch)) return false;
  }
  {
    const int n3 = k.p * k.m, per = (n3 + G - 1) / G, r0 = min(n3, rank * per), r1 = min(n3, r0 + per);
    if (r0 < r1) {
      const int i0 = r0 / k.m, i1 = (r1 - 1) / k.m, len0 = (i1 - i0 + 2) * k.mx, xld = len0 + V;
      for (int c0 = 0; c0 < R; c0 += NC) {
        __syncthreads();
        for (int q = threadIdx.x; q < NC * xld; q += blockDim.x) {
          const int c = q / xld, j = q - c * xld, sp = i0 - 1 + j / k.mx;
          xs[q] = (c0 + c < R && sp >= 0 && sp < k.p - 1 && sp <= i1)
                      ? (T)__ldcg(a.chat + (c0 + c) * A.ds + (sp + 1) * srow - k.mx + j % k.mx)
                      : T(0);
        }
        __syncthreads();
        row_dots_cols<T, NC>(
            r0, r1, xld,
            [&](int r, const T*& row, const T*& x, int& len) {
              const int i = r / k.m;
              row = k.W + (size_t)r * k.ldw;
              x = xs + (i - i0) * k.mx;
              len = (r - i * k.m) < min(k.m, d - i * srow) ? 2 * k.mx : 0;
            },
            [&](int r, int c, T sum) {
              if (c0 + c >= R) return;
              const int i = r / k.m;
              double* out = a.chat + (c0 + c) * A.ds + i * srow + (r - i * k.m);
              *out = __ldcg(out) - __ldcg(a.gsep + (c0 + c) * gst + gst - 1) * (double)k.z[r] - (double)sum;
            });
      }
    }
  }
  return team_sync(a, epoch);
}

// longest stretch of a coarse vector that a CTA of a team of G stages
template <typename T>
__host__ __device__ inline int strips_stage(const CoarseStrips<T>& k, int G) {
  const int RS = k.m + 2 * k.mx, per1 = (k.p * RS + G - 1) / G, per3 = (k.p * k.m + G - 1) / G;
  const int s1 = ((per1 + RS - 2) / RS + 1) * k.h * k.row, s3 = ((per3 + k.m - 2) / k.m + 2) * k.mx;
  int m = s1 > s3 ? s1 : s3;
  if (k.ns > m) m = k.ns;
  return m + 16 / (int)sizeof(T);
}

// c_hat = C^+ c for all columns, complete after its last barrier.
template <typename S>
__device__ SMPM_PHASE bool lk_coarse(const LockArgs<S>& A, const LockSmem<S>& s, unsigned& epoch) {
  const int room = (int)(A.wb_bytes / sizeof(S));  // the groups' scratch is idle here
  if (A.a.use_strips) {
    const int nc = room / strips_stage(A.a.strips, A.a.G);
    if (nc >= 8 && A.R > 4) return lk_coarse_strips_nc<S, 8>(A, s.wb, epoch);
    if (nc >= 4 && A.R > 2) return lk_coarse_strips_nc<S, 4>(A, s.wb, epoch);
    if (nc >= 2) return lk_coarse_strips_nc<S, 2>(A, s.wb, epoch);
  }
  bool done = false;
  if constexpr (sizeof(S) == 4) {
    const int dc = (room / A.R) & ~31;  // entries per column and chunk
    if (dc >= 256) {
      lk_coarse32_staged(A, reinterpret_cast<float*>(s.wb), dc);
      done = true;
    }
  }
  if (!done) lk_coarse_h(A, A.a.H);
  return team_sync(A.a, epoch);
}

// op(sc * src) -> y (and c, chat) for all columns; with own_j >= 0 the block
// solves read basis vector own_j (owner slices), else the global src.
template <typename S>
__device__ SMPM_PHASE bool lk_apply(const LockArgs<S>& A, const LockSmem<S>& s, const S* src, const double* sc, int own_j,
                         unsigned& epoch, int& trace_n) {
  const GmresArgs<S>& a = A.a;
  lk_black(A, s, src, sc, own_j);
  GM_TRACE(31);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(32);
  lk_white(A, s, src, sc, a.precond == 2);
  GM_TRACE(33);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(34);
  if (a.precond == 2) {
    if (!lk_coarse(A, s, epoch)) return false;
    GM_TRACE(36);
  }
  return true;
}

// Dot products of the owned basis slices with the columns' vectors w: for each
// pair (l, rho), l < nl, out[l * R + rho] += sum_i basis(l, rho)[i] w(rho)[i],
// with l == nl - 1 giving w.w.  A warp takes four l of a column at a time (over
// all entries, or a chunk of them when there are few items): w is read once
// for the four, lanes keep eight 16-byte loads in flight, and the four sums
// meet in six shuffled additions instead of twenty (an FP64 addition costs as
// much as a product here).  FP32 products are summed in FP32 over 16 entries
// per lane, those in FP64.
template <typename S>
__device__ SMPM_PHASE void lk_dots(const LockArgs<S>& A, const LockSmem<S>& s, int nl, double* out) {
  const int E = A.a.ES, R = A.R, ng = (nl + 3) / 4, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  int nch = 1;  // chunks of the entries: at least two items per warp, 256 entries or more each
  while (ng * R * nch < 2 * nwarps && E / (nch * 2) >= 256) nch *= 2;
  const int clen = (E / 4 + nch - 1) / nch * 4;
  for (int it = warp; it < ng * R * nch; it += nwarps) {
    const int ch = it % nch, pr = it / nch, rho = pr % R, l0 = (pr / R) * 4;
    const S* w = lk_w(A, s, rho);
    const S* v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = lk_basis(A, min(l0 + q, nl - 2), rho);
    const int self = nl - 1 - l0;  // the q that is w itself (0 .. 3), if any
    const int i0 = ch * clen, i1 = min(E, i0 + clen);
    double sum[4] = {0, 0, 0, 0};
    for (int i = i0 + 4 * lane; i < i1; i += 256) {
      const bool two = i + 128 < i1;
      Quad<S> b[2][4], ww[2];
      ww[0] = ld_quad_w(w + i);
      ww[1] = two ? ld_quad_w(w + i + 128) : Quad<S>{};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q == self) {
          b[0][q] = ww[0];
          b[1][q] = ww[1];
        } else {
          b[0][q] = ld_quad(v[q] + i);
          b[1][q] = two ? ld_quad(v[q] + i + 128) : Quad<S>{};
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if constexpr (sizeof(S) == 4) {
          float f = 0.f;
#pragma unroll
          for (int k = 0; k < 8; ++k) f = fmaf(b[k >> 2][q].v[k & 3], ww[k >> 2].v[k & 3], f);
          sum[q] += (double)f;
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k < 4 || two) sum[q] += b[k >> 2][q].v[k & 3] * ww[k >> 2].v[k & 3];
        }
      }
    }
    // lane bits 4 and 3 select the sum a lane keeps
    const bool up = lane & 16, hi = lane & 8;
    double a0 = (up ? sum[2] : sum[0]) + __shfl_xor_sync(0xffffffffu, up ? sum[0] : sum[2], 16);
    double a1 = (up ? sum[3] : sum[1]) + __shfl_xor_sync(0xffffffffu, up ? sum[1] : sum[3], 16);
    double a = (hi ? a1 : a0) + __shfl_xor_sync(0xffffffffu, hi ? a0 : a1, 8);
    for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    const int l = l0 + (up ? 2 : 0) + (hi ? 1 : 0);
    if ((lane & 7) == 0 && l < nl && a != 0.0) atomicAdd(out + l * R + rho, a);
  }
}

// w(rho)[i] - sum_{l < nl} coef[rho * m3 + l] basis(l, rho)[i] for every column
// rho and owned entry i, in place of w (to_basis: into basis vector jdst and the
// column's global vector).  A thread takes U quads of entries at a time through
// l, the next l's loads issued before this l's products (FP32 arithmetic for
// FP32 bases).
template <typename S>
__device__ SMPM_PHASE void lk_combo_pass(const LockArgs<S>& A, const LockSmem<S>& s, const double* coef, int nl, bool to_basis,
                              int jdst) {
  constexpr int U = sizeof(S) == 4 ? 4 : 2;
  const GmresArgs<S>& a = A.a;
  const int E = a.ES, R = A.R, m3 = a.m + 3, E4 = E / 4, NQ = R * E4;
  const size_t lstep = (size_t)R * E;  // from basis vector l to l + 1
  using C = typename std::conditional<sizeof(S) == 4, float, double>::type;
  for (int p0 = threadIdx.x; p0 < NQ; p0 += U * blockDim.x) {
    C acc[U][4];
    const S* b[U];
    const double* cf[U];
    int rho_[U], i_[U];
    Quad<S> cur[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int p = min(p0 + q * (int)blockDim.x, NQ - 1);
      rho_[q] = p / E4;
      i_[q] = 4 * (p - rho_[q] * E4);
      cf[q] = coef + rho_[q] * m3;
      b[q] = lk_basis(A, 0, rho_[q]) + i_[q];
      if (nl > 0) cur[q] = ld_quad(b[q]);
      const Quad<S> w = ld_quad_w(lk_w(A, s, rho_[q]) + i_[q]);
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[q][k] = (C)w.v[k];
    }
    for (int l = 0; l < nl; ++l) {
      Quad<S> nxt[U];
      if (l + 1 < nl) {
#pragma unroll
        for (int q = 0; q < U; ++q) nxt[q] = ld_quad(b[q] + (l + 1) * lstep);
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const C c = (C)cf[q][l];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[q][k] -= c * (C)cur[q].v[k];
      }
      if (l + 1 < nl) {
#pragma unroll
        for (int q = 0; q < U; ++q) cur[q] = nxt[q];
      }
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      if (p0 + q * (int)blockDim.x >= NQ) continue;
      Quad<S> o;
#pragma unroll
      for (int k = 0; k < 4; ++k) o.v[k] = (S)acc[q][k];
      if (!to_basis) {
        *reinterpret_cast<Quad<S>*>(lk_w(A, s, rho_[q]) + i_[q]) = o;
      } else {
        *reinterpret_cast<Quad<S>*>(lk_basis(A, jdst, rho_[q]) + i_[q]) = o;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int sl = entry_slot(a, i_[q] + k);
          if (sl >= 0) a.vglob[rho_[q] * A.vs + sl] = o.v[k];
        }
      }
    }
  }
}

// base - sum_{l < nl} coef[l] basis(l, rho)[i] (FP32 arithmetic for FP32 bases)
template <typename S>
__device__ __forceinline__ double lk_combo(const LockArgs<S>& A, double base, const double* coef, int nl, int rho,
                                           int i) {
  if constexpr (sizeof(S) == 4) {
    float r = (float)base;
    for (int l = 0; l < nl; ++l) r = fmaf(-(float)coef[l], ldcg(lk_basis(A, l, rho) + i), r);
    return (double)r;
  } else {
    double r = base;
    for (int l = 0; l < nl; ++l) r -= coef[l] * ldcg(lk_basis(A, l, rho) + i);
    return r;
  }
}

// The lockstep GMRES by the CTAs of a team; false when a wait timed out.
template <typename S>
__device__ __noinline__ bool lock_body(const LockArgs<S>& A, unsigned char* smraw, unsigned& epoch) {
  const LockSmem<S> s = lock_carve(A, smraw);
  const GmresArgs<S>& a = A.a;
  const int m = a.m, m3 = m + 3, R = A.R;
  const int ES = a.ES, G = a.G, rank = team_rank(a);
  int trace_n = 0;

  // misc per column: 0 ||w||^2, 1 ||w2||^2, 2 residual estimate, 3 state (0 running,
  // 1 converged, 2 breakdown, 3 NaN), 5 Arnoldi steps (all cycles), 6 beta0, 7 tol * beta0
  for (int c = threadIdx.x; c < R; c += blockDim.x) {
    // done flags are written by other CTAs (refinement steps of the same
    // launch in a batch): read from L2, never a stale L1 line
    s.active[c] = (A.done && *((volatile const int*)(A.done + (size_t)c * A.done_stride))) ? 0 : 1;
    s.jc[c] = 0;
    for (int k = 0; k < 8; ++k) s.misc[c * 8 + k] = 0;
  }
  int total = 0, cycle = 0;
  __syncthreads();
  bool any_active = true;
  while (true) {
    double* accN = a.acc + (size_t)(2 * m) * R * m3;
    // ---- cycle start: V[0] = rhs - op(x) for every column
    if (cycle > 0) {
      for (int c = threadIdx.x; c < R; c += blockDim.x) s.scl[c] = 1.0;
      __syncthreads();
      if (!lk_apply(A, s, a.x, s.scl, -1, epoch, trace_n)) return false;
    }
    for (int rho = 0; rho < R; ++rho) {
      S* v0 = lk_basis(A, 0, rho);
      double nn = 0;
      for (int i = threadIdx.x; i < ES; i += blockDim.x) {
        const int4 en = owned_entry(a, i);
        const int sl = en.x;
        S rv = 0;
        if (sl >= 0 && s.active[rho]) {
          double r = (double)ldcg(a.rhs + rho * A.vs + sl);
          if (cycle > 0)
            r -= deflate_entry(a, a.y + rho * A.vs, a.precond == 2 ? a.chat + rho * A.ds : nullptr, en);
          rv = (S)r;
        }
        if (sl >= 0) a.vglob[rho * A.vs + sl] = rv;
        v0[i] = rv;
        nn += (double)rv * (double)rv;
      }
      nn = warp_sum(nn);
      if ((threadIdx.x & 31) == 0 && nn != 0.0) atomicAdd(accN + rho, nn);
    }
    if (!team_sync(a, epoch)) return false;
    if (threadIdx.x < R) {
      const int c = threadIdx.x;
      const double beta = sqrt(__ldcg(accN + c));
      double* mc = s.misc + c * 8;
      if (cycle == 0) {
        mc[6] = beta;
        mc[7] = a.tol * beta;
      }
      s.jc[c] = 0;
      if (s.active[c]) {
        mc[2] = beta;  // residual estimate
        if (!isfinite(beta)) {
          mc[3] = 3;  // nan
          s.active[c] = 0;
        } else if (beta <= mc[7] || beta == 0.0) {
          mc[3] = 1;  // converged
          s.active[c] = 0;
        }
      }
      s.gg[c * m3] = beta;
      s.invb[c * m3] = s.active[c] ? 1.0 / beta : 0.0;
    }
    __syncthreads();
    any_active = false;
    for (int c = 0; c < R; ++c) any_active |= s.active[c] != 0;
    if (!any_active || total >= a.maxit) break;
    int j = 0;
    for (; j < m && total < a.maxit; ++j) {
      double* accD = a.acc + (size_t)(2 * j) * R * m3;
      double* accE = a.acc + (size_t)(2 * j + 1) * R * m3;
      // ---- A: v_j = w2 - V h2 (scaled later) on the owned entries, then block solves
      GM_TRACE(30);
      if (j > 0) {
        lk_combo_pass(A, s, s.hs2, j, true, j);
        __syncthreads();
      }
      for (int c = threadIdx.x; c < R; c += blockDim.x) s.scl[c] = s.invb[c * m3 + j];
      __syncthreads();
      GM_TRACE(37);
      if (!lk_apply(A, s, a.vglob, s.scl, j, epoch, trace_n)) return false;
      // ---- D: w = y - S Z chat on owned entries; V^T w, ||w||^2.  A thread
      // takes an entry through the columns, four at a time: the entry's
      // indices and coefficients are read once
      for (int i = threadIdx.x; i < ES; i += blockDim.x) {
        const int4 en = owned_entry(a, i);
        if (en.z < 0 || a.precond != 2) {
          for (int c = 0; c < R; ++c) lk_w(A, s, c)[i] = en.z < 0 ? S(0) : ldcg(a.y + c * A.vs + en.x);
          continue;
        }
        const int4 J = __ldg(a.if4 + en.y);
        const double2* Rp = reinterpret_cast<const double2*>(a.Rd + 4 * (size_t)en.x);
        const double2 r0 = __ldg(Rp), r1 = __ldg(Rp + 1);
        for (int c0 = 0; c0 < R; c0 += 4) {
          double yv[4], h[4][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = min(c0 + q, R - 1);
            const double* ch = a.chat + c * A.ds;
            yv[q] = (double)ldcg(a.y + c * A.vs + en.x);
            h[q][0] = __ldcg(ch + J.x);
            h[q][1] = __ldcg(ch + J.y);
            h[q][2] = __ldcg(ch + J.z);
            h[q][3] = __ldcg(ch + J.w);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (c0 + q < R)
              lk_w(A, s, c0 + q)[i] =
                  (S)((yv[q] - (r0.x * h[q][0] + r0.y * h[q][1])) - (r1.x * h[q][2] + r1.y * h[q][3]));
        }
      }
      __syncthreads();
      GM_TRACE(38);
      lk_dots(A, s, j + 2, accD);
      GM_TRACE(39);
      if (!team_sync(a, epoch)) return false;
      GM_TRACE(40);
      for (int p = threadIdx.x; p < (j + 2) * R; p += blockDim.x) {
        const int l = p / R, c = p % R;
        double v = __ldcg(accD + p);
        if (l <= j) {
          v *= s.invb[c * m3 + l];
          s.h1[c * m3 + l] = v;
          s.hs1[c * m3 + l] = v * s.invb[c * m3 + l];
        } else {
          s.misc[c * 8 + 0] = v;  // ||w||^2
        }
      }
      __syncthreads();
      // ---- E: w2 = w - V h1; V^T w2, ||w2||^2
      lk_combo_pass(A, s, s.hs1, j + 1, false, 0);
      __syncthreads();
      GM_TRACE(41);
      lk_dots(A, s, j + 2, accE);
      GM_TRACE(42);
      if (!team_sync(a, epoch)) return false;
      GM_TRACE(43);
      for (int p = threadIdx.x; p < (j + 2) * R; p += blockDim.x) {
        const int l = p / R, c = p % R;
        double v = __ldcg(accE + p);
        if (l <= j) {
          v *= s.invb[c * m3 + l];
          s.h2[c * m3 + l] = v;
          s.hs2[c * m3 + l] = v * s.invb[c * m3 + l];
        } else {
          s.misc[c * 8 + 1] = v;  // ||w2||^2
        }
      }
      __syncthreads();
      // ---- Givens update of every running column (thread c), replicated in every CTA
      if (threadIdx.x < R) {
        const int c = threadIdx.x;
        double* mc = s.misc + c * 8;
        if (s.active[c]) {
          const double* h1 = s.h1 + c * m3;
          const double* h2 = s.h2 + c * m3;
          double* col = s.colv + c * m3;
          double* gcs = s.gcs + c * m3;
          double* gsn = s.gsn + c * m3;
          double* gg = s.gg + c * m3;
          double q = 0;
          for (int l = 0; l <= j; ++l) {
            q += h2[l] * h2[l];
            col[l] = h1[l] + h2[l];
          }
          const double bsq = mc[1] - q;
          const double ib = bsq > 0 ? rsqrt(bsq) : 0.0;
          const double bnext = bsq > 0 ? bsq * ib : 0.0;
          double xi = col[0];
          for (int i = 0; i < j; ++i) {
            const double x1 = col[i + 1], cc = gcs[i], sn = gsn[i];
            const double cx1 = cc * x1, sx1 = sn * x1;
            col[i] = fma(cc, xi, sx1);
            xi = fma(-sn, xi, cx1);
          }
          col[j] = xi;
          const double hh = col[j] * col[j] + bnext * bnext;
          const double iden = hh > 0 ? rsqrt(hh) : 0.0;
          const double cs = hh > 0 ? col[j] * iden : 1.0, ss = bnext * iden;
          gcs[j] = cs;
          gsn[j] = ss;
          col[j] = hh * iden;
          gg[j + 1] = -ss * gg[j];
          gg[j] = cs * gg[j];
          s.invb[c * m3 + j + 1] = ib;
          const double resid = fabs(gg[j + 1]);
          mc[2] = resid;
          s.jc[c] = j + 1;
          mc[5] += 1;
          if (rank == 0) {
            double* Rc = A.Rh + ((size_t)c * m + j) * (m + 1);
            for (int l = 0; l <= j; ++l) Rc[l] = col[l];
          }
          if (!isfinite(resid) || !isfinite(bnext)) {
            mc[3] = 3;
            s.active[c] = 0;
          } else if (resid <= mc[7]) {
            mc[3] = 1;
            s.active[c] = 0;
          } else if (bsq <= 1e-28 * mc[0]) {
            mc[3] = 2;  // breakdown
            s.active[c] = 0;
          }
          if (!s.active[c]) s.invb[c * m3 + j + 1] = 0.0;
        } else {
          s.invb[c * m3 + j + 1] = 0.0;
        }
      }
      __syncthreads();
      GM_TRACE(44);
      ++total;
      any_active = false;
      for (int c = 0; c < R; ++c) any_active |= s.active[c] != 0;
      if (!any_active) {
        ++j;
        break;
      }
    }
    // ---- end of cycle: y = R^-1 g per column (team rank 0), x += V diag(invb) y
    if (rank == 0 && threadIdx.x < R) {
      const int c = threadIdx.x, jj = s.jc[c];
      const double* gg = s.gg + c * m3;
      double* y = A.yv + (size_t)c * m;
      for (int i = jj - 1; i >= 0; --i) {
        double sum = gg[i];
        for (int k = i + 1; k < jj; ++k) sum -= A.Rh[((size_t)c * m + k) * (m + 1) + i] * y[k];
        y[i] = sum / A.Rh[((size_t)c * m + i) * (m + 1) + i];
      }
    }
    for (size_t i = (size_t)rank * blockDim.x + threadIdx.x; i < (size_t)(2 * m + 1) * R * m3;
         i += (size_t)G * blockDim.x)
      a.acc[i] = 0.0;
    if (!team_sync(a, epoch)) return false;
    for (int p = threadIdx.x; p < R * m; p += blockDim.x) {
      const int c = p / m, l = p % m;
      s.hs1[c * m3 + l] = l < s.jc[c] ? -__ldcg(A.yv + (size_t)c * m + l) * s.invb[c * m3 + l] : 0.0;
    }
    __syncthreads();
    for (int rho = 0; rho < R; ++rho) {
      const int jj = s.jc[rho];
      if (jj == 0) continue;
      for (int i = threadIdx.x; i < ES; i += blockDim.x) {
        const int sl = entry_slot(a, i);
        if (sl < 0) continue;
        S* xp = a.x + rho * A.vs + sl;
        *xp = (S)lk_combo(A, (double)ldcg(xp), s.hs1 + rho * m3, jj, rho, i);
      }
    }
    if (!team_sync(a, epoch)) return false;
    ++cycle;
    any_active = false;
    for (int c = 0; c < R; ++c) any_active |= s.active[c] != 0;
    if (!any_active || total >= a.maxit) break;
  }
  if (rank == 0 && threadIdx.x < R) {
    const int c = threadIdx.x;
    const double* mc = s.misc + c * 8;
    LockColState st;
    st.beta0 = mc[6];
    st.tolabs = mc[7];
    st.resid = mc[2];
    st.its = (int)mc[5];
    st.converged = (mc[3] == 1 || mc[6] == 0.0) ? 1 : 0;
    st.breakdown = mc[3] == 2 ? 1 : 0;
    st.nan = mc[3] == 3 ? 1 : 0;
    st.cycles = cycle;
    st.its_total = A.cs[c].its_total + st.its;
    A.cs[c] = st;
  }
  return true;
}

// true when every column is marked done (the launch has nothing to do)
template <typename S>
__device__ __forceinline__ bool lock_all_done(const LockArgs<S>& A) {
  if (!A.done) return false;
  for (int c = 0; c < A.R; ++c)
    if (!*((volatile const int*)(A.done + (size_t)c * A.done_stride))) return false;
  return true;
}
