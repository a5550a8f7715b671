// Persistent GMRES kernel for x := GMRES(op, rhs) with op one of
//   S            (Algorithm 1),
//   S M^-1       (Algorithm 2),
//   P S M^-1     (Algorithm 3),
// run as ONE cooperative launch per solve: restarted GMRES(m), classical
// Gram-Schmidt with one re-orthogonalisation (CGS2), the convergence test on
// the least-squares residual, restarts from the true residual.
//
// Work is owned, not redistributed per phase: CTA c owns the checkerboard
// blocks ib = c, c + G, ... (G = grid size) -- the black elements and the
// slots of their blocks, which partition Gamma -- and the white elements
// iw = c, c + G, ...  The matrices are shared per class of elements or blocks,
// packed in digits (smpm_digits.cuh); the class a CTA uses most, its slice of
// the Krylov basis, its entries' table and its rows of C^+ stay in shared
// memory as far as they fit.  One step:
//   A  owner: block solves t = M^-1 v_j on its block slots: a = G (p - X q), b = q - T_e a, in stages
//      (black_phase) or with the whole inverse (black_block)
//   B  white elements: y = S t (y = v on white-owned slots), c = Z^T y
//   C  c_hat = C^+ c (rows over all CTAs, or by element-row strips; Algorithm 3)
//   D  owner: w = y - S Z c_hat; V^T w and ||w||^2, accumulated with FP64
//      atomics in L2
//   E  owner: w2 = w - V h1; V^T w2 and ||w2||^2 likewise; every CTA forms
//      ||v_{j+1}||^2 = ||w2||^2 - ||h2||^2 and the residual norm from its own
//      copy of the Hessenberg column (warp 0), so all CTAs take the same
//      decision, while the other warps form v_{j+1} = w2 - V h2
// Phases are separated by a team barrier (5 per step for Algorithm 3, 7 with
// strips).  The basis is kept unnormalised with the inverse norms replicated
// in every CTA.
//
// What bounds it: on a grid with a block or two per CTA, the chain of one
// step: five barriers (about 3,000 SM cycles each), a dozen dependent loads
// from L2 (about 700 each), FP64 sums at 76 cycles per operation, one packing
// and one product of digits per element phase.  At 16 x 16 elements, n = 16,
// on 128 CTAs the phases and barriers of a step take 55,000 cycles of CTA 0 (57,000 with
// FP64 products and rotations in every step, and a step more per solve).  On large grids, the element products, the
// basis read from L2 and C^+.
//
// Data written by other CTAs inside the kernel is read with ld.global.cg: L1
// is not coherent across SMs.  The barrier spins with a bound and raises an
// error flag instead of hanging.
#pragma once
// Included inside the anonymous namespace of each translation unit that uses it.

// Packed class matrices of the element products (smpm_digits.cuh): T_e per
// element class, G_b and the four X_F per block class, with row exponents,
// and the class of each element / black block.  Elements of one class (face
// types and sizes) share one copy, so a CTA reads its matrices from L1.
struct DigitMats {
  const uint4 *G, *X, *T;
  const short *Ge, *Xe, *Te;
  const int *bcls, *tcls;
  const uint4* B;   // whole block inverses (2M x 2M), or null: see black_block
  const short* Be;
};

template <typename S>
struct GmresArgs {
  DevGeo g;
  const int* black;
  const int* white;
  int nblack, nwhite;
  DigitMats dm;
  // per entry of a black block (2M per block: own slots, then facing slots):
  // {slot or -1, element that pushes into it, its interface or -1, 4 e + F of the slot}
  const int4* bt;
  const int4* if4;   // interfaces of each element (0 where there is none; its weight is 0)
  const double* Rd;  // kp * 4: S Z at each slot, the coefficients of c_hat on the pusher's interfaces
  // coarse inverse, d rows of (d rounded up to a multiple of 4) entries: FP64, or
  // its FP32 copy for the FP32 inner solves of the mixed-precision path
  const typename std::conditional<sizeof(S) == 4, float, double>::type* H;
  const double* H64;  // FP32 solves of small grids: the FP64 inverse, used instead; else null
  S* vglob;         // kp : current basis vector (raw), exchanged between CTAs
  S* vown;          // G * (m+1) * ES : basis slices when not resident in smem
  S* t;             // kp
  S* y;             // kp
  double* c;        // d
  double* chat;     // d
  const S* rhs;     // kp
  S* x;             // kp (zero on entry)
  double* acc;      // (2m + 1) * (m + 3) FP64 accumulators (zero on entry)
  GState* gs;
  unsigned* bar;    // the team's barrier counter
  int* err;
  int precond, m, maxit;
  double tol;
  int nown_b, nown_w;  // blocks / white elements per CTA (ceil)
  int ES;              // entries per CTA in the basis slice (a multiple of 4, >= 2M nown_b)
  int basis_smem;      // 1: basis slice resident in shared memory
  int W_item;          // warps per block / element in the element phases (8 / W_item groups per CTA)
  int res_T, res_G;    // classes whose matrices the CTA keeps in shared memory: T_e (0 .. 2), G_b with X_b (0, 1)
  int tab, res_H;      // 1: the owned entries' table / the CTA's rows of H in shared memory
  int blk;             // 1: black blocks by their whole inverse (dm.B)
  long long* trace;
  int trace_cap;
  const int* skip;  // when non-null and set on entry, the kernel returns at once
  int* its_out;     // when non-null: Arnoldi steps of this launch
  int G;            // CTAs working on this solve (a team; the whole grid for one solve)
  int base;         // first CTA of the team: the CTA's rank is blockIdx.x - base
  S* wscr;          // when non-null: per-CTA global scratch for w (ES per rank)
  // C^+ by element-row strips (strips.p > 0 and use_strips): see coarse_solve
  CoarseStrips<typename std::conditional<sizeof(S) == 4, float, double>::type> strips;
  CoarseStrips<double> strips64;  // where H64 is set
  double* gsep;        // strips: 2 p mx + 1 doubles per column (sums pushed onto the separators, alpha)
  int use_strips;      // 1: the strips are the cheaper form for this team size
};

// rank of this CTA within the team that works on a solve
template <typename S>
__device__ __forceinline__ int team_rank(const GmresArgs<S>& a) {
  return (int)blockIdx.x - a.base;
}

// Phase trace of CTA 0 (SMPM_TRACE); a call, so that the solve's own code stays small.
__device__ __noinline__ void trace_point(long long* trace, int cap, int rank, int tag, int& n) {
  if (rank == 0 && threadIdx.x == 0 && n + 2 <= cap) {
    trace[n++] = tag;
    trace[n++] = clock64();
  }
}
#define GM_TRACE(tag) \
  do {                \
    if (a.trace) trace_point(a.trace, a.trace_cap, team_rank(a), tag, trace_n); \
  } while (0)

template <typename S>
__device__ __forceinline__ S ldcg(const S* p) {
  return __ldcg(p);
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Polls of a barrier wait before it gives up (default 2^28, about a minute
// of polling; smpm_set_barrier_spin_limit lowers it to exercise the timeout).
__device__ long long g_barrier_spin_limit = 1LL << 28;

// Team barrier on a monotonic counter: thread 0 of each CTA adds one with
// release semantics and polls with acquire loads until the counter reaches
// the CTA's next epoch: zero on entry to a kernel, plus the team size G per
// barrier.  Every launch has a counter of its own, zeroed on its stream before
// it.  A cooperative launch does not make its CTAs start together (work on
// another stream can hold an SM back), so the epoch on entry cannot be read from
// a counter that CTAs already running may have advanced.  One flag per CTA,
// polled by a thread each, was four times slower at 152 CTAs (10 k against 2.6 k
// cycles: the polls of all CTAs crowd the flags' L2 slice).  A team of one CTA
// needs no counter.  Bounded spin; err is set on timeout and the caller unwinds.
__device__ __noinline__ bool team_sync_call(unsigned* bar, int* err, unsigned epoch, int G) {
  __syncthreads();
  if (G == 1) return true;
  bool ok = true;
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(1u) : "memory");
    long long spins = 0;
    const long long limit = g_barrier_spin_limit;
    while ((int)(ld_acquire(bar) - epoch) < 0) {
      if (++spins > limit) {  // this CTA's own timeout: code 1 unless a failure is recorded
        atomicCAS(err, 0, 1);
        ok = false;
        break;
      }
      if ((spins & 4095) == 0 && *((volatile int*)err)) {  // another CTA failed: unwind
        ok = false;
        break;
      }
    }
  }
  return __syncthreads_and(ok);
}
template <typename S>
__device__ __forceinline__ bool team_sync(const GmresArgs<S>& a, unsigned& epoch) {
  if (a.G > 1) epoch += (unsigned)a.G;  // the counter stays where it is for a team of one
  return team_sync_call(a.bar, a.err, epoch, a.G);
}

// entry i (< 2M) of black block ib
template <typename S>
__device__ __forceinline__ int4 block_entry(const GmresArgs<S>& a, int ib, int i) {
  return __ldg(a.bt + (size_t)ib * 2 * a.g.M + i);
}

// owned entry i of the CTA: block rank + k G, entry i - 2M k of it
template <typename S>
__device__ __forceinline__ int4 owned_entry(const GmresArgs<S>& a, int i) {
  const int M2 = 2 * a.g.M, k = i / M2, ib = team_rank(a) + k * a.G;
  if (k >= a.nown_b || ib >= a.nblack) return make_int4(-1, 0, -1, 0);
  return block_entry(a, ib, i - k * M2);
}
template <typename S>
__device__ __forceinline__ int entry_slot(const GmresArgs<S>& a, int i) {
  return owned_entry(a, i).x;
}

// ---- shared memory ---------------------------------------------------------
// A group of W warps works on one block or element; its scratch: the packed
// vector (M entries, or n on each of the four faces), the block's values
// [p; q], r1 (then a), and for white elements the contributions to c.
template <typename S>
__host__ __device__ constexpr size_t item_bf_bytes(int M, int n, int blk) {
  const int a = digit_bwords<S>(blk ? 2 * M : M), b = 4 * digit_bwords<S>(n);
  return sizeof(uint4) * (size_t)(a > b ? a : b);
}
template <typename S>
__host__ __device__ constexpr size_t item_bytes(int M, int n, int blk) {
  return item_bf_bytes<S>(M, n, blk) + 3 * (size_t)M * sizeof(double);
}
// warps per item for `items` items per CTA: every warp busy
inline int item_warps(long long items) {
  int w = 1;
  while (w < kGmresThreads / 32 && items * w * 2 <= kGmresThreads / 32) w *= 2;
  return w;
}

// The W warps of a group (named barrier of their own) work on one item.
__device__ __forceinline__ void item_sync(int grp, int W) {
  if (W == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(32 * W) : "memory");
}

// Matrices resident in shared memory: the classes most of the CTA's blocks and
// elements belong to.  L1 does not keep them: the acquiring load of a barrier
// invalidates it (31 % hits measured in k_gmres), so from global memory every
// phase reads its matrices from L2 again.
struct Resident {
  const uint4 *T, *G, *X;
  int clsT[2], clsG;  // -1: none
};

// What the deflation of an owned entry needs besides y and c_hat: its table
// entry, its pusher's interfaces and the row of S Z (a chain of two dependent
// loads from L2, 1,300 cycles of every step, when read from global memory).
struct OwnedEntry {
  int4 en, J;
  double2 r0, r1;
};

template <typename S>
struct Smem {
  double *h1, *h2, *hs1, *hs2, *z, *xi, *gg, *invb, *misc;
  double* cst;  // staged coarse vector c (d, and two entries of padding)
  unsigned char* wb;  // group scratch (item_bytes each)
  Resident* res;
  int4* ob;         // owned blocks: {element or -1, block class, T class}
  int4* ow;         // owned white elements: {element or -1, T class}
  OwnedEntry* tab;  // ES entries, or null
  const typename std::conditional<sizeof(S) == 4, float, double>::type* H;  // the CTA's rows of H, or null
  S* w;     // ES : w, then w2 in its place
  S* V;     // the CTA's slice of the basis, (m+1) * ES: shared or global memory
  unsigned char* end;
};

// bytes of one CTA's rows of H (coarse_rows)
template <typename S>
__host__ __device__ inline size_t coarse_row_bytes(long long d, int G) {
  return (size_t)((d + G - 1) / G) * ((d + 3) & ~3LL) * sizeof(S);
}

template <typename S>
__device__ Smem<S> carve(const GmresArgs<S>& a, unsigned char* raw) {
  Smem<S> s;
  const int m = a.m;
  double* d = reinterpret_cast<double*>(raw);
  s.h1 = d; d += m + 3;
  s.h2 = d; d += m + 3;
  s.hs1 = d; d += m + 3;
  s.hs2 = d; d += m + 3;
  s.z = d; d += m + 3;
  s.xi = d; d += m + 3;
  s.gg = d; d += m + 3;
  s.invb = d; d += m + 3;
  s.misc = d; d += 16;
  s.cst = d; d += a.g.d + 3;
  auto align = [](void* p) { return reinterpret_cast<unsigned char*>((reinterpret_cast<size_t>(p) + 15) & ~size_t(15)); };
  s.res = reinterpret_cast<Resident*>(align(d));
  s.ob = reinterpret_cast<int4*>(align(s.res + 1));
  s.ow = s.ob + a.nown_b;
  s.wb = align(s.ow + a.nown_w);
  S* q = reinterpret_cast<S*>(s.wb + (size_t)(kGmresThreads / 32 / a.W_item) * item_bytes<S>(a.g.M, a.g.n, a.blk));
  if (a.wscr) s.w = a.wscr + (size_t)team_rank(a) * a.ES;
  else { s.w = q; q += a.ES; }
  if (a.basis_smem) { s.V = q; q += (size_t)(m + 1) * a.ES; }
  else s.V = a.vown ? a.vown + (size_t)team_rank(a) * (m + 1) * a.ES : nullptr;
  unsigned char* e = align(q);
  s.tab = nullptr;
  if (a.tab) { s.tab = reinterpret_cast<OwnedEntry*>(e); e += a.ES * sizeof(OwnedEntry); }
  s.H = nullptr;
  if (a.res_H) { s.H = reinterpret_cast<decltype(s.H)>(e); e += coarse_row_bytes<S>(a.g.d, a.G); }
  s.end = e;  // resident matrices, or the scratch of the bodies around GMRES
  return s;
}

template <typename S>
inline size_t resident_bytes(int M, int n, int res_T, int res_G, int blk) {
  return sizeof(uint4) * (res_T * digit_words<S>(M, M) +
                          res_G * (blk ? digit_words<S>(2 * M, 2 * M) : digit_words<S>(M, M) + 4 * digit_words<S>(n, n)));
}

template <typename S>
inline size_t gmres_smem_bytes(int m, int M, int n, int ES, int W, int basis_smem, long long d, bool w_global = false,
                               int res_T = 0, int res_G = 0, int blk = 0, int tab = 0, size_t H_bytes = 0) {
  const size_t dbl = 8 * (size_t)(m + 3) + 16 + (size_t)d + 3;
  size_t sel = w_global ? 0 : ES;
  if (basis_smem) sel += (size_t)(m + 1) * ES;
  return dbl * sizeof(double) + (size_t)(kGmresThreads / 32 / W) * item_bytes<S>(M, n, blk) + sel * sizeof(S) +
         resident_bytes<S>(M, n, res_T, res_G, blk) + sizeof(Resident) +
         (2 * (size_t)(ES / (2 * M)) + 4) * sizeof(int4) + (tab ? ES * sizeof(OwnedEntry) : 0) + H_bytes + 96;
}

// The class that most of the CTA's cnt owned items have other than `skip` (-1:
// none): field f of their tables' entries.  Warp 0; the first 32 items stand for
// all.
__device__ __forceinline__ int main_class(const int4* own, int cnt, int f, int skip) {
  const int lane = threadIdx.x & 31;
  int mine = -1;
  if (lane < cnt && own[lane].x >= 0) mine = f == 1 ? own[lane].y : own[lane].z;
  int n = 0;
  for (int k = 0; k < 32; ++k) n += __shfl_sync(0xffffffffu, mine, k) == mine;
  const int best = __reduce_max_sync(0xffffffffu, mine >= 0 && mine != skip ? n * 32 + lane : -1);
  return best < 0 ? -1 : __shfl_sync(0xffffffffu, mine, best & 31);
}

// The CTA's tables of owned blocks and white elements (all threads; the caller
// synchronises): read in every phase, a dependent load from L2 each.
template <typename S>
__device__ __forceinline__ void load_owned(const GmresArgs<S>& a, const Smem<S>& s) {
  const DigitMats& D = a.dm;
  for (int k = threadIdx.x; k < a.nown_b + a.nown_w; k += blockDim.x) {
    const bool b = k < a.nown_b;
    const int i = team_rank(a) + (b ? k : k - a.nown_b) * a.G;
    const int e = i < (b ? a.nblack : a.nwhite) ? __ldg((b ? a.black : a.white) + i) : -1;
    const int ct = e >= 0 ? __ldg(D.tcls + e) : -1;
    s.ob[k] = b ? make_int4(e, e >= 0 && D.bcls ? __ldg(D.bcls + i) : -1, ct, 0) : make_int4(e, ct, 0, 0);
  }
}

template <typename S>
__device__ __forceinline__ int4 owned_entry(const GmresArgs<S>& a, const Smem<S>& s, int i) {
  return s.tab ? s.tab[i].en : owned_entry(a, i);
}
template <typename S>
__device__ __forceinline__ int entry_slot(const GmresArgs<S>& a, const Smem<S>& s, int i) {
  return owned_entry(a, s, i).x;
}

// Loads the resident matrices and tables (all threads; ends with a barrier).
template <typename S>
__device__ SMPM_PHASE void load_resident(const GmresArgs<S>& a, const Smem<S>& s) {
  const int M = a.g.M, n = a.g.n, rank = team_rank(a);
  const size_t wM = digit_words<S>(M, M), wX = a.blk ? 0 : 4 * digit_words<S>(n, n);
  const size_t wG = a.blk ? digit_words<S>(2 * M, 2 * M) : wM;
  uint4* p = reinterpret_cast<uint4*>(s.end);
  load_owned(a, s);
  __syncthreads();
  if (threadIdx.x < 32) {
    const int t0 = a.res_T > 0 ? main_class(s.ow, a.nown_w, 1, -1) : -1;
    const int t1 = a.res_T > 1 ? main_class(s.ob, a.nown_b, 2, t0) : -1;
    const int g0 = a.res_G > 0 ? main_class(s.ob, a.nown_b, 1, -1) : -1;
    if (threadIdx.x == 0) *s.res = {p, p + a.res_T * wM, p + (a.res_T + 1) * wM, {t0, t1}, g0};
  }
  if (s.tab) {
    for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
      OwnedEntry o = {owned_entry(a, i), make_int4(0, 0, 0, 0), make_double2(0, 0), make_double2(0, 0)};
      if (o.en.z >= 0) {
        const double2* R = reinterpret_cast<const double2*>(a.Rd + 4 * (size_t)o.en.x);
        o.J = __ldg(a.if4 + o.en.y);
        o.r0 = __ldg(R);
        o.r1 = __ldg(R + 1);
      }
      s.tab[i] = o;
    }
  }
  if (s.H && !a.use_strips && a.precond == 2) {
    using T = typename std::conditional<sizeof(S) == 4, float, double>::type;
    const int d = (int)a.g.d, ld = (d + 3) & ~3, per = (d + a.G - 1) / a.G;
    const int r0 = min(d, rank * per), cnt = (min(d, r0 + per) - r0) * ld;
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) const_cast<T*>(s.H)[i] = __ldg(a.H + (size_t)r0 * ld + i);
  }
  __syncthreads();
  const Resident& R = *s.res;
#pragma unroll 1
  for (int k = 0; k < a.res_T; ++k)
    if (R.clsT[k] >= 0)
      for (size_t i = threadIdx.x; i < wM; i += blockDim.x) p[k * wM + i] = __ldg(a.dm.T + R.clsT[k] * wM + i);
  if (R.clsG >= 0) {
    uint4* q = p + a.res_T * wM;
    for (size_t i = threadIdx.x; i < wG; i += blockDim.x) q[i] = __ldg((a.blk ? a.dm.B : a.dm.G) + R.clsG * wG + i);
    for (size_t i = threadIdx.x; i < wX; i += blockDim.x) q[wM + i] = __ldg(a.dm.X + R.clsG * wX + i);
  }
  __syncthreads();
}
// no resident matrices (the bodies around GMRES use their place)
template <typename S>
__device__ __forceinline__ void no_resident(const GmresArgs<S>& a, const Smem<S>& s) {
  __syncthreads();
  load_owned(a, s);
  if (threadIdx.x == 0) *s.res = {nullptr, nullptr, nullptr, {-1, -1}, -1};
  __syncthreads();
}

// packed matrices of a class: resident copy or global memory
template <typename S>
__device__ __forceinline__ const uint4* mat_T(const GmresArgs<S>& a, const Smem<S>& s, int cls) {
  const size_t w = digit_words<S>(a.g.M, a.g.M);
  const Resident& R = *s.res;
  return cls == R.clsT[0] ? R.T : cls == R.clsT[1] ? R.T + w : a.dm.T + cls * w;
}
template <typename S>
__device__ __forceinline__ const uint4* mat_G(const GmresArgs<S>& a, const Smem<S>& s, int cls) {
  return cls == s.res->clsG ? s.res->G : a.dm.G + cls * digit_words<S>(a.g.M, a.g.M);
}
template <typename S>
__device__ __forceinline__ const uint4* mat_B(const GmresArgs<S>& a, const Smem<S>& s, int cls) {
  return cls == s.res->clsG ? s.res->G : a.dm.B + cls * digit_words<S>(2 * a.g.M, 2 * a.g.M);
}
template <typename S>
__device__ __forceinline__ const uint4* mat_X(const GmresArgs<S>& a, const Smem<S>& s, int cls) {  // four of them
  return cls == s.res->clsG ? s.res->X : a.dm.X + cls * 4 * digit_words<S>(a.g.n, a.g.n);
}

// ---- element phases ---------------------------------------------------------
// P = sc * (own slice, or the global src) of block ib, the k-th of this CTA: 2M
// values by the W warps of a group (at: the thread's place in it)
template <typename S>
__device__ __forceinline__ void gather_block(const GmresArgs<S>& a, const S* src, double sc, const S* own, S* P, int ib,
                                             int k, int at) {
  const int M = a.g.M, W = a.W_item;
#pragma unroll 1
  for (int i0 = at; i0 < 2 * M; i0 += 128 * W) {  // four loads in flight per lane
    S v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + 32 * W * u;
      v[u] = S(0);
      if (i >= 2 * M) continue;
      if (own) {
        v[u] = own[k * 2 * M + i];
      } else {
        const int sl = block_entry(a, ib, i).x;
        if (sl >= 0) v[u] = ldcg(src + sl);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + 32 * W * u < 2 * M) P[i0 + 32 * W * u] = (S)(sc * (double)v[u]);
  }
}

// Black block solves of this CTA: block values vb = sc * (own slice, or the
// global src), r1 = p - X q, a = G r1, z = T_e a, t = [a; q - z], the products
// in exact fixed point on the tensor cores.
// Bound by the chain of its stages: one block of M = 64 on a CTA's eight warps takes
// about 14,000 SM cycles (gather 1,300, X 3,900, packing 1,500 twice, G 3,100, T
// 3,200); on CTAs with many blocks, whose groups overlap, by the tiles' issue
// (two instructions to unpack a register of digits, 8 cycles for a product).
template <typename S>
__device__ SMPM_PHASE void black_phase(const GmresArgs<S>& a, const Smem<S>& s, const S* src, double sc, const S* own) {
  const DevGeo& g = a.g;
  const DigitMats& D = a.dm;
  const int M = g.M, n = g.n, W = a.W_item, ngrp = kGmresThreads / 32 / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W;
  const int kt_n = digit_tiles(M), kf_n = digit_tiles(n);
  unsigned char* base = s.wb + (size_t)grp * item_bytes<S>(M, n, a.blk);
  uint4* Bf = reinterpret_cast<uint4*>(base);
  S* P = reinterpret_cast<S*>(base + item_bf_bytes<S>(M, n, a.blk));
  S* Rr = P + 2 * M;
#pragma unroll 1
  for (int k = grp; k < a.nown_b; k += ngrp) {
    const int ib = team_rank(a) + k * a.G, e = s.ob[k].x, cb = s.ob[k].y, ct = s.ob[k].z;
    if (e < 0) break;
    gather_block(a, src, sc, own, P, ib, k, part * 32 + lane);
    item_sync(grp, W);
#pragma unroll 1
    for (int F = part; F < 4; F += W) {  // r1 = p - X q, face by face
      uint4* Bq = Bf + F * digit_bwords<S>(n);
      const S* q = P + M + F * n;
      const int E = pack_one<S>(Bq, q, n, lane, 0, 1);
#pragma unroll 1
      for (int mt = 0; mt < kf_n; ++mt) {
        const S z = digits_tile1<S>(mat_X(a, s, cb) + F * digit_words<S>(n, n), D.Xe + ((size_t)cb * 4 + F) * n,
                                    Bq, n, kf_n, mt, lane, E);
        const int row = tile1_row(mt, lane, n);
        if (row >= 0) Rr[F * n + row] = P[F * n + row] - z;
      }
    }
    item_sync(grp, W);
    for (int stage = 0; stage < 2; ++stage) {  // a = G r1, then z = T_e a and t = q - z on the facing slots
      const int E = pack_one<S>(Bf, Rr, M, lane, part, W);
      const uint4* A = stage == 0 ? mat_G(a, s, cb) : mat_T(a, s, ct);
      const short* er = stage == 0 ? D.Ge + (size_t)cb * M : D.Te + (size_t)ct * M;
      item_sync(grp, W);
#pragma unroll 1
      for (int mt = part; mt < kt_n; mt += W) {
        const int row = tile1_row(mt, lane, M);
        const int sl = row < 0 ? -1 : stage == 0 ? e * M + row : (s.tab ? s.tab[k * 2 * M + M + row].en.x : block_entry(a, ib, M + row).x);
        const S z = digits_tile1<S>(A, er, Bf, M, kt_n, mt, lane, E);
        if (stage == 0 && row >= 0) Rr[row] = z;
        if (sl >= 0) a.t[sl] = stage == 0 ? z : P[M + row] - z;
      }
      item_sync(grp, W);
    }
  }
  __syncthreads();
}

// The same with the whole inverse of a block, t = [G, -G X; -T G, I + T G X] [p; q]
// in one product: twice the products and bytes of the three stages above, but
// one gather, one packing and one product instead of a chain of four (14,000
// SM cycles for one block of M = 64, the stages' latencies).  Taken where a CTA
// owns so few blocks that the chain is what it waits for (see block_pays).
template <typename S>
__device__ SMPM_PHASE void black_block(const GmresArgs<S>& a, const Smem<S>& s, const S* src, double sc, const S* own) {
  const DigitMats& D = a.dm;
  const int M = a.g.M, n = a.g.n, W = a.W_item, ngrp = kGmresThreads / 32 / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W;
  const int kt_n = digit_tiles(2 * M);
  unsigned char* base = s.wb + (size_t)grp * item_bytes<S>(M, n, a.blk);
  uint4* Bf = reinterpret_cast<uint4*>(base);
  S* P = reinterpret_cast<S*>(base + item_bf_bytes<S>(M, n, a.blk));
#pragma unroll 1
  for (int k = grp; k < a.nown_b; k += ngrp) {
    const int ib = team_rank(a) + k * a.G, e = s.ob[k].x, cb = s.ob[k].y;
    if (e < 0) break;
    gather_block(a, src, sc, own, P, ib, k, part * 32 + lane);
    item_sync(grp, W);
    const int E = pack_one<S>(Bf, P, 2 * M, lane, part, W);
    item_sync(grp, W);
#pragma unroll 1
    for (int mt = part; mt < kt_n; mt += W) {
      const int row = tile1_row(mt, lane, 2 * M);
      const int sl = row < 0 ? -1 : row < M ? e * M + row : (s.tab ? s.tab[k * 2 * M + row].en.x : block_entry(a, ib, row).x);
      const S z = digits_tile1<S>(mat_B(a, s, cb), D.Be + (size_t)cb * 2 * M, Bf, 2 * M, kt_n, mt, lane, E);
      if (sl >= 0) a.t[sl] = z;
    }
    item_sync(grp, W);
  }
  __syncthreads();
}

// What a white element's row needs besides its product: v on the own slot, t on
// the facing slot sl (-1 on the physical boundary) and the weights of both in
// the deflation vector.
template <typename S>
struct Facing {
  int sl;
  S v, t;
  double w0, w1;
};
template <typename S>
__device__ __forceinline__ Facing<S> facing_entry(const DevGeo& g, int e, int row, const S* v, const S* t) {
  const int M = g.M, n = g.n, F = row / n, tt = row - F * n, e2 = dev_neighbour(g, e, F);
  Facing<S> f;
  f.sl = e2 >= 0 ? e2 * M + (F ^ 1) * n + tt : -1;
  f.v = ldcg(v + (size_t)e * M + row);
  f.t = e2 >= 0 ? ldcg(t + f.sl) : S(0);
  f.w0 = g.zw && e2 >= 0 ? dev_zw(g, e, F) : 1.0;
  f.w1 = g.zw && e2 >= 0 ? dev_zw(g, e2, F ^ 1) : 1.0;
  return f;
}
// the row's share of c = Z^T y (uniform grids: weights 1, no multiplication)
template <typename S>
__device__ __forceinline__ double facing_c(const DevGeo& g, const Facing<S>& f, S vo, S ys) {
  return g.zw ? f.w0 * (double)vo + f.w1 * (double)ys : (double)vo + (double)ys;
}

// White elements: y = S t on the black slots facing e, y = sc*v on e's slots,
// c = Z^T y on e's interfaces (with_c).
template <typename S>
__device__ SMPM_PHASE void white_phase(const GmresArgs<S>& a, const Smem<S>& s, const S* v, double sc, bool with_c) {
  const DevGeo& g = a.g;
  const DigitMats& D = a.dm;
  const int M = g.M, n = g.n, W = a.W_item, ngrp = kGmresThreads / 32 / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W;
  const int kt_n = digit_tiles(M);
  unsigned char* base = s.wb + (size_t)grp * item_bytes<S>(M, n, a.blk);
  uint4* Bf = reinterpret_cast<uint4*>(base);
  double* ci = reinterpret_cast<double*>(base + item_bf_bytes<S>(M, n, a.blk));  // contributions to c
  S* te = reinterpret_cast<S*>(ci + M);                                   // t on e's slots
#pragma unroll 1
  for (int k = grp; k < a.nown_w; k += ngrp) {
    const int e = s.ow[k].x, ct = s.ow[k].y;
    if (e < 0) break;
    Facing<S> f{};
    if (part < kt_n && tile1_row(part, lane, M) >= 0) f = facing_entry(g, e, tile1_row(part, lane, M), v, a.t);
    for (int i = part * 32 + lane; i < M; i += 32 * W) te[i] = ldcg(a.t + (size_t)e * M + i);
    item_sync(grp, W);
    const int E = pack_one<S>(Bf, te, M, lane, part, W);
    item_sync(grp, W);
#pragma unroll 1
    for (int mt = part; mt < kt_n; mt += W) {
      const int row = tile1_row(mt, lane, M);
      if (row >= 0 && mt != part) f = facing_entry(g, e, row, v, a.t);
      const S z = digits_tile1<S>(mat_T(a, s, ct), D.Te + (size_t)ct * M, Bf, M, kt_n, mt, lane, E);
      if (row < 0) continue;
      const S vo = (S)(sc * (double)f.v);
      a.y[(size_t)e * M + row] = vo;
      double c1 = 0;
      if (f.sl >= 0) {
        const S ys = f.t + z;
        a.y[f.sl] = ys;
        c1 = facing_c(g, f, vo, ys);
      }
      ci[row] = c1;
    }
    item_sync(grp, W);
    if (with_c && part == 0) {  // face F summed by the eight lanes 8 F + r
      const int F = lane >> 3, j = dev_iface(g, e, F);
      double sum = 0;
#pragma unroll 1
      for (int tt = lane & 7; tt < n; tt += 8) sum += ci[F * n + tt];
#pragma unroll 1
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if ((lane & 7) == 0 && j >= 0) a.c[j] = sum;
    }
    item_sync(grp, W);
  }
  __syncthreads();
}

// Push form y = S (sc*v) (Algorithm 1): elements rank, rank + G, ...
template <typename S>
__device__ SMPM_PHASE void push_phase(const GmresArgs<S>& a, const Smem<S>& s, const S* v, double sc) {
  const DevGeo& g = a.g;
  const DigitMats& D = a.dm;
  const int M = g.M, n = g.n, W = a.W_item, ngrp = kGmresThreads / 32 / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / W, part = warp % W;
  const int kt_n = digit_tiles(M);
  unsigned char* base = s.wb + (size_t)grp * item_bytes<S>(M, n, a.blk);
  uint4* Bf = reinterpret_cast<uint4*>(base);
  S* ve = reinterpret_cast<S*>(base + item_bf_bytes<S>(M, n, a.blk));
#pragma unroll 1
  for (long long el = team_rank(a) + (long long)grp * a.G; el < g.nel; el += (long long)ngrp * a.G) {
    const int e = (int)el, ct = __ldg(D.tcls + e);
    for (int i = part * 32 + lane; i < M; i += 32 * W) ve[i] = (S)(sc * (double)ldcg(v + (size_t)e * M + i));
    item_sync(grp, W);
    const int E = pack_one<S>(Bf, ve, M, lane, part, W);
    item_sync(grp, W);
#pragma unroll 1
    for (int mt = part; mt < kt_n; mt += W) {
      const int row = tile1_row(mt, lane, M);
      Facing<S> f{};
      if (row >= 0) f = facing_entry(g, e, row, v, v);
      const S z = digits_tile1<S>(mat_T(a, s, ct), D.Te + (size_t)ct * M, Bf, M, kt_n, mt, lane, E);
      if (row < 0) continue;
      if (f.sl >= 0) a.y[f.sl] = (S)(sc * (double)f.t) + z;
      else a.y[(size_t)e * M + row] = ve[row];
    }
    item_sync(grp, W);
  }
  __syncthreads();
}

// ---- C^+ by strips ----------------------------------------------------------
// C couples two interfaces only when they share an element, so the horizontal
// interfaces between two element rows separate the grid.  With a separator
// every h element rows, c_hat = C^+ c is, for the strips' interiors i and the
// separators s (all factors from the host factor step):
//   P1  y_i = C_ii^-1 c_i, and the sums C_si y_i it pushes onto its separators
//   P2  c_s' = c_s - sum_i C_si y_i;  x_s = H_ss c_s';  alpha = u_C,s . c_s'
//   P3  x_i = y_i - alpha C_ii^-1 u_C,i - C_ii^-1 C_is x_s
// (alpha = u_C . c: the left projection (I - u_C u_C^T); H_ss, the separators'
// block of H, inverts the Schur complement; the result differs from H c by a
// multiple of c0, which S Z maps to zero and the zero mean of u removes).
// About d^2 / 7 products instead of d^2, in three phases of short dot
// products with two more barriers (see strips_pay on when that is less).
template <bool SM>  // SM: from shared memory
__device__ __forceinline__ void ld_vec(const double* p, double (&v)[2]) {
  const double2 t = SM ? *reinterpret_cast<const double2*>(p) : __ldg(reinterpret_cast<const double2*>(p));
  v[0] = t.x; v[1] = t.y;
}
template <bool SM>
__device__ __forceinline__ void ld_vec(const float* p, float (&v)[4]) {
  const float4 t = SM ? *reinterpret_cast<const float4*>(p) : __ldg(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}

// For rows r0 <= r < r1: get(r, &row, &x, &len) names a row (16-byte aligned,
// zero-padded to whole 16-byte groups) and the staged vector (readable to the
// padded length); put(r, sum) takes the dot product (len 0: no call).  P lanes
// per row, P as large as the rows (longest: their greatest length) leave threads
// and entries for, but 4 at least: each
// halving step of the final sums costs as much FP64 time as a product.
template <typename T, bool SM = false, typename Get, typename Put>
__device__ __forceinline__ void row_dots(int r0, int r1, int longest, Get&& get, Put&& put) {
  constexpr int V = 16 / (int)sizeof(T), U = 4;
  const int rows = r1 - r0;
  int P = 32;
  while (P > 4 && (P * rows > (int)blockDim.x || V * P >= 2 * longest)) P >>= 1;
  const int lane = threadIdx.x % P, grp = threadIdx.x / P, ngrp = blockDim.x / P;
#pragma unroll 1
  for (int rb = 0; rb < rows; rb += ngrp) {  // uniform trip count per warp
    const int r = r0 + rb + grp;
    const T* a = nullptr;
    const T* x = nullptr;
    int len = 0;
    if (r < r1) get(r, a, x, len);
    T acc[4] = {T(0), T(0), T(0), T(0)};
    int j = V * lane;
#pragma unroll 1
    for (; j + V * P * (U - 1) < len; j += V * P * U) {
      T h[U][V];
#pragma unroll
      for (int u = 0; u < U; ++u) ld_vec<SM>(a + j + u * V * P, h[u]);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[u] += h[u][v] * x[j + u * V * P + v];
    }
#pragma unroll 1
    for (; j < len; j += V * P) {
      T h[V];
      ld_vec<SM>(a + j, h);
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v & 3] += h[v] * x[j + v];
    }
    T sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll 1
    for (int o = P / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o, P);
    if (lane == 0 && len > 0) put(r, sum);
  }
}

// c_hat = C^+ c, complete after the final barrier; false when a
// barrier timed out.  cst: staging for at least d + 1 entries.
template <typename T, typename S>
__device__ SMPM_PHASE bool coarse_strips(const GmresArgs<S>& a, const CoarseStrips<T>& k, void* cst, unsigned& epoch,
                                         const double* c, double* chat) {
  constexpr int V = 16 / (int)sizeof(T);
  T* xs = reinterpret_cast<T*>(cst);
  const int G = a.G, rank = team_rank(a), d = (int)a.g.d;
  const int srow = k.h * k.row, RS = k.m + 2 * k.mx;  // interfaces of a strip with its upper separator; rows of N
  double* alpha = a.gsep + 2 * (size_t)k.p * k.mx;
  {  // P1
    const int n1 = k.p * RS, per = (n1 + G - 1) / G, r0 = min(n1, rank * per), r1 = min(n1, r0 + per);
    if (r0 < r1) {
      const int b0 = (r0 / RS) * srow, b1 = min(d, ((r1 - 1) / RS + 1) * srow);
      for (int j = threadIdx.x; j < b1 - b0 + V; j += blockDim.x) xs[j] = b0 + j < b1 ? (T)__ldcg(c + b0 + j) : T(0);
      __syncthreads();
      row_dots<T>(
          r0, r1, k.m,
          [&](int r, const T*& row, const T*& x, int& len) {
            const int i = r / RS, l = r - i * RS, mi = min(k.m, d - i * srow);
            const bool on = l < k.m ? l < mi : (l < k.m + k.mx ? i > 0 : i < k.p - 1);
            row = k.N + (size_t)r * k.ldn;
            x = xs + i * srow - b0;
            len = on ? mi : 0;
          },
          [&](int r, T sum) {
            const int i = r / RS, l = r - i * RS;
            if (l < k.m) chat[i * srow + l] = (double)sum;
            else a.gsep[2 * (size_t)i * k.mx + (l - k.m)] = (double)sum;
          });
    }
    if (!team_sync(a, epoch)) return false;
  }
  {  // P2: rows 0 .. ns-1 of H_ss, row ns: u_C on the separators
    const int n2 = k.ns + 1, per = (n2 + G - 1) / G, r0 = min(n2, rank * per), r1 = min(n2, r0 + per);
    if (r0 < r1) {
      for (int j = threadIdx.x; j < k.ns + V; j += blockDim.x) {
        T v = T(0);
        if (j < k.ns) {
          const int sp = j / k.mx, q = j - sp * k.mx;
          const double* up = a.gsep + (2 * (size_t)sp + 1) * k.mx + q;  // strip below; lower sums of the one above
          v = (T)(__ldcg(c + (sp + 1) * srow - k.mx + q) - __ldcg(up) - __ldcg(up + k.mx));
        }
        xs[j] = v;
      }
      __syncthreads();
      row_dots<T>(
          r0, r1, k.ns,
          [&](int r, const T*& row, const T*& x, int& len) {
            row = k.Hs + (size_t)r * k.lds;
            x = xs;
            len = k.ns;
          },
          [&](int r, T sum) {
            if (r == k.ns) *alpha = (double)sum;
            else chat[(r / k.mx + 1) * srow - k.mx + r % k.mx] = (double)sum;
          });
    }
    if (!team_sync(a, epoch)) return false;
  }
  {  // P3: rows of W: 2 mx coefficients of the separators below and above, then C_ii^-1 u_C,i
    const int n3 = k.p * k.m, per = (n3 + G - 1) / G, r0 = min(n3, rank * per), r1 = min(n3, r0 + per);
    if (r0 < r1) {
      const int i0 = r0 / k.m, i1 = (r1 - 1) / k.m;  // separators i0 - 1 .. i1
      for (int j = threadIdx.x; j < (i1 - i0 + 2) * k.mx + V; j += blockDim.x) {
        const int sp = i0 - 1 + j / k.mx;
        xs[j] = (sp >= 0 && sp < k.p - 1 && sp <= i1) ? (T)__ldcg(chat + (sp + 1) * srow - k.mx + j % k.mx) : T(0);
      }
      const double al = __ldcg(alpha);
      __syncthreads();
      row_dots<T>(
          r0, r1, 2 * k.mx,
          [&](int r, const T*& row, const T*& x, int& len) {
            const int i = r / k.m;
            row = k.W + (size_t)r * k.ldw;
            x = xs + (i - i0) * k.mx;
            len = (r - i * k.m) < min(k.m, d - i * srow) ? 2 * k.mx : 0;
          },
          [&](int r, T sum) {
            const int i = r / k.m;
            double* out = chat + i * srow + (r - i * k.m);
            *out = __ldcg(out) - al * (double)k.z[r] - (double)sum;
          });
    }
  }
  return team_sync(a, epoch);
}

// c_hat = H c by rows: the CTA takes a contiguous range of them (own: its rows in
// shared memory, or null), c staged in shared memory, sums in T.
template <typename T, typename S>
__device__ __forceinline__ void coarse_rows_in(const GmresArgs<S>& a, const T* H, const T* own, T* xs, const double* c,
                                               double* chat) {
  const int d = (int)a.g.d, ld = (d + 3) & ~3, per = (d + a.G - 1) / a.G;
  const int r0 = min(d, team_rank(a) * per), r1 = min(d, r0 + per);
  if (r0 >= r1) return;
  for (int j = threadIdx.x; j < d + 16 / (int)sizeof(T); j += blockDim.x) xs[j] = j < d ? (T)__ldcg(c + j) : T(0);
  __syncthreads();
  auto put = [&](int r, T sum) { chat[r] = (double)sum; };
  if (own) {
    row_dots<T, true>(
        r0, r1, d,
        [&](int r, const T*& row, const T*& x, int& len) {
          row = own + (size_t)(r - r0) * ld;
          x = xs;
          len = d;
        },
        put);
  } else {
    row_dots<T>(
        r0, r1, d,
        [&](int r, const T*& row, const T*& x, int& len) {
          row = H + (size_t)r * ld;
          x = xs;
          len = d;
        },
        put);
  }
}
// The FP32 inner solves of the mixed-precision path take the FP64 inverse (or its
// strips) on small grids (H64), where its products are a small part of a step, and
// else its FP32 copy with FP32 products and sums: an inner solve needs only a relative 1e-4, and
// every refinement sweep recomputes the residual in FP64.
template <typename S>
__device__ SMPM_PHASE void coarse_rows(const GmresArgs<S>& a, const Smem<S>& s, const double* c, double* chat) {
  using T = typename std::conditional<sizeof(S) == 4, float, double>::type;
  if constexpr (sizeof(S) == 4)
    if (a.H64) return coarse_rows_in<double>(a, a.H64, (const double*)nullptr, s.cst, c, chat);
  coarse_rows_in<T>(a, a.H, s.H, reinterpret_cast<T*>(s.cst), c, chat);
}

// c_hat = C^+ c by all CTAs of the team (strips or dense rows), complete after
// its last barrier; false when a barrier timed out
template <typename S>
__device__ __forceinline__ bool coarse_solve(const GmresArgs<S>& a, const Smem<S>& s, unsigned& epoch, const double* c,
                                             double* chat) {
  if constexpr (sizeof(S) == 4)
    if (a.use_strips && a.H64) return coarse_strips(a, a.strips64, s.cst, epoch, c, chat);
  if (a.use_strips) return coarse_strips(a, a.strips, s.cst, epoch, c, chat);
  coarse_rows(a, s, c, chat);
  return team_sync(a, epoch);
}

// ys - (S Z chat) at an entry (pull form); 0 on the physical boundary, ys
// itself when chat is null.
template <typename A>
__device__ __forceinline__ double deflate_value(const GmresArgs<A>& a, double ys, const double* chat, int4 en) {
  if (en.z < 0) return 0.0;
  if (!chat) return ys;
  const int4 J = __ldg(a.if4 + en.y);
  const double2* R = reinterpret_cast<const double2*>(a.Rd + 4 * (size_t)en.x);
  const double2 r0 = __ldg(R), r1 = __ldg(R + 1);
  const double c0 = __ldcg(chat + J.x), c1 = __ldcg(chat + J.y), c2 = __ldcg(chat + J.z), c3 = __ldcg(chat + J.w);
  return (ys - (r0.x * c0 + r0.y * c1)) - (r1.x * c2 + r1.y * c3);
}
template <typename S, typename A>
__device__ __forceinline__ double deflate_entry(const GmresArgs<A>& a, const S* y, const double* chat, int4 en) {
  return deflate_value(a, en.x >= 0 ? (double)ldcg(y + en.x) : 0.0, chat, en);
}

// ---- Gram-Schmidt passes over the CTA's slice of the basis ---------------
// Dot products of the owned basis slice with vec (ES entries) for l < nl,
// l == nl - 1 giving vec.vec: P lanes per l (P a power of two <= 32, P*nl <=
// blockDim when possible) read consecutive entries; partial sums meet in warp
// shuffles and are added atomically to out[l] (FP64, in L2).
template <typename S>
__device__ SMPM_PHASE void owned_dots(const GmresArgs<S>& a, const Smem<S>& s, const S* vec, int nl, double* out) {
  const int E = a.ES;
  int P = 32;
  while (P > 1 && P * nl > (int)blockDim.x) P >>= 1;
  const int ngrp = blockDim.x / P, lane = threadIdx.x % P, grp = threadIdx.x / P;
  for (int lb = 0; lb < nl; lb += ngrp) {  // uniform trip count per warp
    const int l = lb + grp;
    double sum = 0;
    if (l < nl) {
      const S* vl = (l == nl - 1) ? vec : (s.V + (size_t)l * a.ES);
      // eight entries per step, loaded before they are used: with the basis
      // in global memory each lane keeps eight independent loads in flight
      if constexpr (sizeof(S) == 4) {
        // FP32 products summed in FP32 over chunks of 16, chunks added in FP64
        int i = lane, cnt = 0;
        float f0 = 0.f;
        for (; i + 7 * P < E; i += 8 * P) {
          float bv[8], wv[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            bv[u] = (float)vl[i + u * P];
            wv[u] = (float)vec[i + u * P];
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) f0 = fmaf(bv[u], wv[u], f0);
          cnt += 8;
          if (cnt == 16) {
            sum += (double)f0;
            f0 = 0.f;
            cnt = 0;
          }
        }
        for (; i < E; i += P) f0 = fmaf((float)vl[i], (float)vec[i], f0);
        sum += (double)f0;
      } else {
        double acc[4] = {0, 0, 0, 0};
        int i = lane;
        for (; i + 7 * P < E; i += 8 * P) {
          double bv[8], wv[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            bv[u] = (double)vl[i + u * P];
            wv[u] = (double)vec[i + u * P];
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) acc[u & 3] += bv[u] * wv[u];
        }
        for (; i < E; i += P) acc[0] += (double)vl[i] * (double)vec[i];
        sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      }
    }
    for (int o = P / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o, P);
    if (l < nl && lane == 0 && sum != 0.0) atomicAdd(out + l, sum);
  }
}

// base[i] - sum_{l < nl} coef[l] * basis(l)[i] for one owned entry; FP32
// arithmetic for FP32 bases (coefficients rounded once), FP64 otherwise.
template <typename S>
__device__ __forceinline__ double basis_combo(const GmresArgs<S>& a, const Smem<S>& s, double base, const double* coef,
                                              int nl, int i) {
  if constexpr (sizeof(S) == 4) {
    float r = (float)base;
    for (int l = 0; l < nl; ++l) r = fmaf(-(float)coef[l], (float)(s.V + (size_t)l * a.ES)[i], r);
    return (double)r;
  } else {
    double r = base;
    for (int l = 0; l < nl; ++l) r -= coef[l] * (double)(s.V + (size_t)l * a.ES)[i];
    return r;
  }
}

// op(sc * src) -> y (and c, chat).  With t_done the owners have already
// written t = M^-1 v for their blocks.
template <typename S>
__device__ SMPM_PHASE bool apply_op(const GmresArgs<S>& a, const Smem<S>& s, const S* src, double sc, bool t_done,
                         int& trace_n, unsigned& epoch) {
  if (a.precond == 0) {
    push_phase(a, s, src, sc);
    return team_sync(a, epoch);
  }
  if (!t_done) {
    if (a.blk) black_block(a, s, src, sc, (const S*)nullptr);
    else black_phase(a, s, src, sc, (const S*)nullptr);
  }
  GM_TRACE(20);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(21);
  white_phase(a, s, src, sc, a.precond == 2);
  GM_TRACE(22);
  if (!team_sync(a, epoch)) return false;
  GM_TRACE(23);
  if (a.precond == 2) {
    if (!coarse_solve(a, s, epoch, a.c, a.chat)) return false;
    GM_TRACE(25);
  }
  return true;
}

// w = y - S Z chat on the owned entries (entries without a slot: 0)
template <typename S>
__device__ SMPM_PHASE void deflate_pass(const GmresArgs<S>& a, const Smem<S>& s, const double* chat) {
#pragma unroll 1
  for (int i = threadIdx.x; i < a.ES; i += blockDim.x) {
    double r;
    if (s.tab) {
      const OwnedEntry o = s.tab[i];
      const bool on = o.en.z >= 0;
      const double ys = on ? (double)ldcg(a.y + o.en.x) : 0.0;
      double c0 = 0, c1 = 0, c2 = 0, c3 = 0;
      if (on && chat) {
        c0 = __ldcg(chat + o.J.x);
        c1 = __ldcg(chat + o.J.y);
        c2 = __ldcg(chat + o.J.z);
        c3 = __ldcg(chat + o.J.w);
      }
      r = (ys - (o.r0.x * c0 + o.r0.y * c1)) - (o.r1.x * c2 + o.r1.y * c3);
    } else {
      r = deflate_entry(a, a.y, chat, owned_entry(a, i));
    }
    s.w[i] = (S)r;
  }
}

// End of a cycle: least squares min ||beta e_1 - H y|| over the j Hessenberg
// columns that CTA 0 stored in gs->R, by Givens rotations, in one warp: each
// rotation meets every later column at once, one column per lane (the loads of
// the next row run ahead of the rotation's chain).  y -> gs->y; returns the
// residual norm.  xi, gg, inv: m + 3 entries of shared memory.
__device__ __noinline__ double hessenberg_lsq(GState* gs, double* xi, double* gg, double* inv, int j, double beta) {
  const int lane = threadIdx.x & 31;
  const size_t m1 = kMaxRestart + 1;
  double* R = gs->R;
#pragma unroll 1
  for (int l = lane; l < j; l += 32) xi[l] = __ldcg(R + l * m1);
  double gcur = beta;
  int l0 = lane;
  double nx = l0 < j ? __ldcg(R + l0 * m1 + 1) : 0.0;
#pragma unroll 1
  for (int i = 0; i < j; ++i) {
    const int l1 = i + 1 + ((lane - i - 1) & 31);
    const double ahead = l1 < j ? __ldcg(R + l1 * m1 + i + 2) : 0.0;
    __syncwarp();
    const double x = xi[i], b = __shfl_sync(0xffffffffu, nx, i & 31);  // h_ii rotated so far, h_i+1,i
    const double hh = x * x + b * b;
    const double iden = hh > 0 ? rsqrt(hh) : 0.0;
    const double cc = hh > 0 ? x * iden : 1.0, ss = b * iden;
#pragma unroll 1
    for (int l = l0; l < j; l += 32) {
      const double x1 = l == l0 ? nx : __ldcg(R + l * m1 + i + 1), xl = xi[l];
      R[l * m1 + i] = l == i ? hh * iden : fma(cc, xl, ss * x1);
      if (l > i) xi[l] = fma(-ss, xl, cc * x1);
    }
    if (lane == 0) {
      gg[i] = cc * gcur;
      inv[i] = hh > 0 ? iden : __longlong_as_double(0x7ff0000000000000LL);
    }
    gcur = -ss * gcur;
    nx = ahead;
    l0 = l1;
  }
  __syncwarp();
  // y = R^-1 g column by column: y_k (1 / R_kk is the rotation's 1 / norm, in inv), then the entries above it lose R_ik y_k; two columns ahead in flight
  auto column = [&](int k) { return k >= 0 && lane < k ? __ldcg(R + k * m1 + lane) : 0.0; };
  double r0 = column(j - 1), r1 = column(j - 2);
  for (int k = j - 1; k >= 0; --k) {
    const double r2 = column(k - 2), yk = gg[k] * inv[k];
    __syncwarp();
    for (int i = lane; i < k; i += 32) gg[i] = fma(-(i == lane ? r0 : __ldcg(R + k * m1 + i)), yk, gg[i]);
    if (lane == 0) gs->y[k] = yk;
    __syncwarp();
    r0 = r1;
    r1 = r2;
  }
  return fabs(gcur);
}

// One GMRES solve by the CTAs of a team (the whole grid for k_gmres).
// epoch: the team barrier's epoch, carried across consecutive bodies.
// Returns false when a barrier or copy wait timed out (err set).
template <typename S>
__device__ SMPM_BODY bool gmres_body(const GmresArgs<S>& a, unsigned char* smraw, unsigned& epoch) {
  const Smem<S> s = carve(a, smraw);
  const DevGeo& g = a.g;
  const int m = a.m;
  const int ES = a.ES, G = a.G, rank = team_rank(a);
  const int m3 = m + 3;
  int trace_n = 0;
  load_resident(a, s);

  // v_{j+1} = w2 - V h2 by the threads `at` of n: on few entries by the warps
  // that have nothing else to do while warp 0 forms the residual norm (never
  // read when the step turns out to be the last), on many (more than about
  // two per thread, where the missing warp would cost more) by all, afterwards
  constexpr int kOverlapEntries = 512;
  auto form_next = [&](int at, int n, int j) {
    if (j + 1 >= m ) return;
    S* vn = s.V + (size_t)(j + 1) * ES;
#pragma unroll 1
    for (int i = at; i < ES; i += n) {
      const S rv = (S)basis_combo(a, s, (double)s.w[i], s.hs2, j + 1, i);
      vn[i] = rv;
      const int sl = entry_slot(a, s, i);
      if (sl >= 0) a.vglob[sl] = rv;
    }
  };
  int total = 0, cycle = 0, jlast = 0;
  bool converged = false, breakdown = false, nan = false;
  double tolabs = 0, beta0 = 0, resid = 0;
  __syncthreads();
  while (true) {
    double* accN = a.acc + (size_t)(2 * m) * m3;
    // ---- cycle start: V[0] = rhs - op(x)
    if (cycle > 0) {
      if (!apply_op(a, s, a.x, 1.0, false, trace_n, epoch)) return false;
    }
    {
      S* v0 = s.V;
      double nn = 0;
      for (int i = threadIdx.x; i < ES; i += blockDim.x) {
        const int4 en = owned_entry(a, i);
        const int sl = en.x;
        S rv = 0;
        if (sl >= 0) {
          double r = (double)ldcg(a.rhs + sl);
          if (cycle > 0) r -= deflate_entry(a, a.y, a.precond == 2 ? a.chat : nullptr, en);
          rv = (S)r;
          a.vglob[sl] = rv;
        }
        v0[i] = rv;
        nn += (double)rv * (double)rv;
      }
      nn = warp_sum(nn);
      if ((threadIdx.x & 31) == 0 && nn != 0.0) atomicAdd(accN, nn);
    }
    if (!team_sync(a, epoch)) return false;
    const double beta = sqrt(__ldcg(accN));
    if (cycle == 0) {
      beta0 = beta;
      tolabs = a.tol * beta;
    }
    resid = beta;
    if (!isfinite(beta)) { nan = true; break; }
    if (beta <= tolabs || beta == 0.0) { converged = true; break; }
    if (threadIdx.x == 0) {
      s.z[0] = s.misc[6] = 1.0;
      s.invb[0] = 1.0 / beta;
    }
    __syncthreads();
    int j = 0;
    const double goal = (beta / tolabs) * (beta / tolabs);
#pragma unroll 1
    for (; j < m && total < a.maxit; ++j) {
      double* accD = a.acc + (size_t)(2 * j) * m3;
      double* accE = a.acc + (size_t)(2 * j + 1) * m3;
      const double ivj = s.invb[j];
      GM_TRACE(1);
      // ---- A: block solves with v_j
      S* vj = s.V + (size_t)j * ES;
      if (a.precond == 0) {
        if (!team_sync(a, epoch)) return false;  // neighbours read v_j
        if (!apply_op(a, s, a.vglob, ivj, false, trace_n, epoch)) return false;
      } else {
        if (a.blk) black_block(a, s, (const S*)nullptr, ivj, vj);
        else black_phase(a, s, (const S*)nullptr, ivj, vj);
        if (!apply_op(a, s, a.vglob, ivj, true, trace_n, epoch)) return false;
      }
      GM_TRACE(4);
      // ---- D: w = y - S Z chat on owned entries; V^T w, ||w||^2
      const double* chat_d = a.precond == 2 ? a.chat : nullptr;
      deflate_pass(a, s, chat_d);
      __syncthreads();
      owned_dots(a, s, s.w, j + 2, accD);
      GM_TRACE(5);
      if (!team_sync(a, epoch)) return false;
      GM_TRACE(6);
#pragma unroll 1
      for (int l = threadIdx.x; l < j + 2; l += blockDim.x) {
        double v = __ldcg(accD + l);
        if (l <= j) {
          v *= s.invb[l];
          s.h1[l] = v;
          s.hs1[l] = v * s.invb[l];
        } else {
          s.misc[0] = v;  // ||w||^2
        }
      }
      __syncthreads();
      // ---- E: w2 = w - V h1; V^T w2, ||w2||^2
#pragma unroll 1
      for (int i = threadIdx.x; i < ES; i += blockDim.x) s.w[i] = (S)basis_combo(a, s, (double)s.w[i], s.hs1, j + 1, i);
      __syncthreads();
      owned_dots(a, s, s.w, j + 2, accE);
      GM_TRACE(8);
      if (!team_sync(a, epoch)) return false;
      GM_TRACE(9);
#pragma unroll 1
      for (int l = threadIdx.x; l < j + 2; l += blockDim.x) {
        double v = __ldcg(accE + l);
        if (l <= j) {
          v *= s.invb[l];
          s.h2[l] = v;
          s.hs2[l] = v * s.invb[l];
        } else {
          s.misc[1] = v;  // ||w2||^2
        }
      }
      __syncthreads();
      GM_TRACE(10);
      // ---- F: ||w2|| (Pythagorean), the breakdown test, and the residual norm
      // from the left null vector z of the Hessenberg matrix, z^T H = 0, z_0 = 1:
      // the least-squares residual is beta z / ||z||^2, so its norm is
      // beta / ||z||, and a new column costs one dot product over the lanes and
      // z_{j+1} = -(z . h_j) / h_{j+1,j}.  (Rotating the column instead is a
      // serial chain of j FP64 steps in one thread: 4,000 cycles of a 57,000
      // cycle step, and hidden behind the next step's barrier it cost a step
      // more per solve.  The rotations are made once, at the end of the cycle.)
      if (threadIdx.x < 32) {
        double q = 0, zd = 0;
        double* Rc = a.gs->R + (size_t)j * (kMaxRestart + 1);
#pragma unroll 1
        for (int l = threadIdx.x; l <= j; l += 32) {
          const double h = s.h1[l] + s.h2[l];
          q += s.h2[l] * s.h2[l];
          zd += s.z[l] * h;
          if (rank == 0) Rc[l] = h;
        }
        q = warp_sum(q);
        zd = warp_sum(zd);
        if (threadIdx.x == 0) {
          const double bsq = s.misc[1] - q;
          const double ib = bsq > 0 ? rsqrt(bsq) : 0.0;
          const double zn = -zd * ib, zz = s.misc[6] + zn * zn;
          s.z[j + 1] = zn;
          s.misc[6] = zz;
          s.invb[j + 1] = ib;
          s.misc[3] = (bsq <= 1e-28 * s.misc[0]) ? 1.0 : 0.0;
          s.misc[4] = bsq > 0 ? bsq * ib : 0.0;  // the new subdiagonal entry
          if (rank == 0) Rc[j + 1] = s.misc[4];
        }
      } else if (ES <= kOverlapEntries) {
        form_next(threadIdx.x - 32, blockDim.x - 32, j);
      }
      __syncthreads();
      GM_TRACE(11);
      ++total;
      // beta / ||z|| <= tolabs (an exact breakdown: residual 0; ||z||^2 beyond the
      // range: below any tolerance).  After a NaN there is no residual to report.
      const double zz = s.misc[6];
      if (isnan(zz) || !isfinite(s.misc[4])) {
        nan = true;
        resid = __longlong_as_double(0x7ff8000000000000LL);
        ++j;
        break;
      }
      if (s.misc[4] == 0.0 || goal <= zz) { converged = true; ++j; break; }
      if (s.misc[3] != 0.0) { breakdown = true; ++j; break; }
      if (ES > kOverlapEntries) {
        form_next(threadIdx.x, blockDim.x, j);
        __syncthreads();
      }
    }
    jlast = j;
    if (nan) break;
    // ---- end of cycle: y by warp 0 of CTA 0, x += V diag(invb) y on owned entries
    if (rank == 0 && threadIdx.x < 32) {
      __syncwarp();
      resid = hessenberg_lsq(a.gs, s.xi, s.gg, s.hs1, j, beta);
    }
    if (!team_sync(a, epoch)) return false;
    // the accumulators are consumed by all CTAs: zero them for the next cycle
#pragma unroll 1
    for (size_t i = (size_t)rank * blockDim.x + threadIdx.x; i < (size_t)(2 * m + 1) * m3;
         i += (size_t)G * blockDim.x)
      a.acc[i] = 0.0;
#pragma unroll 1
    for (int l = threadIdx.x; l < j; l += blockDim.x) s.hs1[l] = -__ldcg(a.gs->y + l) * s.invb[l];
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x; i < ES; i += blockDim.x) {
      const int sl = entry_slot(a, s, i);
      if (sl < 0) continue;
      a.x[sl] = (S)basis_combo(a, s, (double)ldcg(a.x + sl), s.hs1, j, i);
    }
    if (!team_sync(a, epoch)) return false;
    ++cycle;
    if (converged || breakdown || total >= a.maxit) break;
  }
  if (rank == 0 && threadIdx.x == 0) {
    a.gs->beta0 = beta0;
    a.gs->tolabs = tolabs;
    a.gs->resid = resid;
    a.gs->j = total;
    a.gs->converged = converged ? 1 : 0;
    a.gs->breakdown = breakdown ? 1 : 0;
    a.gs->nan = nan ? 1 : 0;
    a.gs->scal[7] = cycle;
    a.gs->scal[6] = jlast;
    a.gs->scal[5] += total;  // iterations over all launches of a solve
    if (a.its_out) *a.its_out = total;
  }
  return true;
}
