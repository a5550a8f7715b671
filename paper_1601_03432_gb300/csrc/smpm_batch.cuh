// Batched solves: many right-hand sides of many independent problems (grids
// of different sizes) in ONE persistent cooperative launch.
//
// The CTAs of the launch are split into teams (contiguous CTA ranges, fixed
// for the launch).  Each team works through its own list of tasks, one task
// = one right-hand side of one problem, all right-hand sides of a problem on
// the same team, and runs for each task the bodies of the single-solve
// kernels in order: pre_body, then gmres_body<double> (FP64) or up to
// kMaxRefine pairs (gmres_body<float>, refine_body) (mixed precision), then
// post_body.  Team barriers replace the grid barriers; a team's barrier epoch
// runs on across its tasks.  The task's arguments are staged in shared
// memory (header of the dynamic buffer) and the bodies carve the rest.
#pragma once
// Included inside the anonymous namespace of each translation unit that uses it.

struct alignas(16) BatchTask {
  PrePostArgs P;          // FP64 pre/post arguments (all-global layout)
  GmresArgs<double> a64;  // FP64 GMRES (its own layout: resident matrices, basis)
  GmresArgs<float> a32;   // FP32 inner GMRES (mixed precision)
  RefineArgs R;           // refinement step (mixed precision)
  int precision;          // 0 FP64, 1 FP32 inner + FP64 refinement
  int has_g;
  long long f_off, g_off, u_off;  // offsets into the packed f, g, u of a call
  unsigned char* ctl;     // the problem's control block (zeroed per task from byte 256)
  int* its;               // inner iterations per refinement step (in ctl)
  double* rn;             // ||r||^2 per refinement step (in ctl)
  // lockstep group (ncols >= 2): ncols right-hand sides of the problem in one
  // lockstep GMRES; per-column arguments live in global memory and are staged
  // one at a time behind this header
  int ncols;
  long long rep0;                // report index of the group's first column
  long long r_len, kp_len;       // node and slot vector lengths of the problem
  LockArgs<double> L64;
  LockArgs<float> L32;
  const PrePostArgs* Pc;         // 2 R: pre (c), post (R + c)
  const RefineArgs* Rc;          // kMaxRefine R: refinement step ref of column c at ref R + c
  unsigned char* lctl;           // column blocks (kLockColBytes each): acc8 | done, nref | rn
};

struct BatchIO {
  const double* f;
  const double* g;
  double* u;
};

struct TaskReport {
  int iterations, restarts, refinements, converged;
  double gmres_num, gmres_den;  // relres = num / den
  double res2, bsn2;            // ||b_S - S x_S||^2, ||b_S||^2
  unsigned long long t_begin, t_end;  // global timer (ns) at the task's start and end on its team's first CTA
  int team, breakdown;  // breakdown: an FP64 solve ended on an Arnoldi breakdown before tol
  int nan, pad_;        // nan: an FP64 solve met a NaN or Inf
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

constexpr size_t kLockColBytes = 256;  // column block of a lockstep solve's control area
constexpr int kBatchTaskBytes = (int)((sizeof(BatchTask) + 127) / 128 * 128);
// header: the task, then staging for one column's pre/post and refinement arguments
constexpr int kBatchHdr = (int)((kBatchTaskBytes + sizeof(PrePostArgs) + sizeof(RefineArgs) + 127) / 128 * 128);

// A lockstep group task: pre bodies of the R columns, the lockstep GMRES
// (FP64, or up to kMaxRefine rounds of FP32 lockstep GMRES and per-column
// refinement), post bodies, reports.  Returns the failing body (0: none).
__device__ __noinline__ int batch_group(BatchTask& T, unsigned char* smraw, unsigned char* body, const BatchIO* io,
                           TaskReport* rep, int team, unsigned& epoch) {
  PrePostArgs& Pst = *reinterpret_cast<PrePostArgs*>(smraw + kBatchTaskBytes);
  RefineArgs& Rst = *reinterpret_cast<RefineArgs*>(smraw + kBatchTaskBytes + sizeof(PrePostArgs));
  const int R = T.ncols;
  const GmresArgs<double>& ga = T.P.ga;
  const int rank = team_rank(ga);
  const unsigned long long t_begin = global_ns();
  auto stage_p = [&](int i, int c) {
    __syncthreads();
    stage16(&Pst, T.Pc + i, (int)sizeof(PrePostArgs));
    __syncthreads();
    if (threadIdx.x == 0) {
      Pst.f = io->f + T.f_off + (size_t)c * T.r_len;
      Pst.u = io->u + T.u_off + (size_t)c * T.r_len;
      Pst.gn = (T.has_g && io->g) ? io->g + T.g_off + (size_t)c * T.kp_len : nullptr;
    }
    __syncthreads();
  };
  // column blocks, lockstep accumulators and column reports start at zero
  if (rank == 0) {
    for (int i = threadIdx.x; i < R * (int)(kLockColBytes / 4); i += blockDim.x) reinterpret_cast<int*>(T.lctl)[i] = 0;
    for (int i = threadIdx.x; i < R * (int)(sizeof(LockColState) / 4); i += blockDim.x)
      reinterpret_cast<int*>(T.precision == 0 ? T.L64.cs : T.L32.cs)[i] = 0;
  }
  {
    const GmresArgs<double>& a = T.P.ga;
    const size_t nacc = (size_t)(2 * a.m + 1) * R * (a.m + 3);
    double* acc = T.precision == 0 ? T.L64.a.acc : T.L32.a.acc;
    for (size_t i = (size_t)rank * blockDim.x + threadIdx.x; i < nacc; i += (size_t)a.G * blockDim.x) acc[i] = 0.0;
    // t starts at zero: the phases never write its physical-boundary slots, which
    // an earlier group of another shape may have used.  They meet zero columns
    // of T_e, but set the scale of the digits that the other slots are cut to.
    const size_t nt = (size_t)R * T.kp_len, i0 = (size_t)rank * blockDim.x + threadIdx.x, di = (size_t)a.G * blockDim.x;
    if (T.precision == 0)
      for (size_t i = i0; i < nt; i += di) T.L64.a.t[i] = 0.0;
    else
      for (size_t i = i0; i < nt; i += di) T.L32.a.t[i] = 0.f;
  }
  if (!team_sync(ga, epoch)) return 1;
  for (int c = 0; c < R; ++c) {
    stage_p(c, c);
    if (!pre_body(Pst, body, epoch)) return 2;
  }
  if (T.precision == 0) {
    if (!lock_body<double>(T.L64, body, epoch)) return 3;
  } else {
    for (int ref = 0; ref < kMaxRefine; ++ref) {
      // every column's done flag was written before the last barrier
      bool all = true;
      for (int c = 0; c < R; ++c)
        all = all && *((volatile const int*)(T.lctl + (size_t)c * kLockColBytes + 64)) != 0;
      if (all) break;
      if (!lock_body<float>(T.L32, body, epoch)) return 3;
      for (int c = 0; c < R; ++c) {
        if (*((volatile const int*)(T.lctl + (size_t)c * kLockColBytes + 64))) continue;
        __syncthreads();
        stage16(&Rst, T.Rc + (size_t)ref * R + c, (int)sizeof(RefineArgs));
        __syncthreads();
        if (refine_body(Rst, body, epoch) < 0) return 4;
      }
      if (!team_sync(ga, epoch)) return 4;
    }
  }
  for (int c = 0; c < R; ++c) {
    stage_p(R + c, c);
    if (!post_body(Pst, body, epoch)) return 5;
  }
  if (!team_sync(ga, epoch)) return 5;
  if (rank == 0 && threadIdx.x < R) {
    const int c = threadIdx.x;
    const unsigned char* blk = T.lctl + (size_t)c * kLockColBytes;
    const double* a8 = reinterpret_cast<const double*>(blk);
    const LockColState& cs = (T.precision == 0 ? T.L64.cs : T.L32.cs)[c];
    TaskReport r{};
    r.res2 = __ldcg(a8 + ACC_RES);
    r.bsn2 = __ldcg(a8 + ACC_BSN);
    r.iterations = cs.its_total;
    if (T.precision == 0) {
      r.restarts = cs.cycles > 1 ? cs.cycles - 1 : 0;
      r.converged = cs.converged;
      r.breakdown = cs.breakdown;
      r.nan = cs.nan;
      r.gmres_num = cs.resid;
      r.gmres_den = cs.beta0;
    } else {
      const int nref = *reinterpret_cast<const int*>(blk + 68);
      const double* rn = reinterpret_cast<const double*>(blk + 128);
      r.refinements = nref;
      r.converged = (*reinterpret_cast<const int*>(blk + 64) != 0 || __ldcg(a8 + ACC_RGN) == 0.0) ? 1 : 0;
      r.gmres_num = nref > 0 ? sqrt(__ldcg(rn + min(nref, kMaxRefine) - 1)) : 0.0;
      r.gmres_den = sqrt(__ldcg(a8 + ACC_RGN));
    }
    r.t_begin = t_begin;
    r.t_end = global_ns();
    r.team = team;
    rep[T.rep0 + c] = r;
  }
  return 0;
}
// stage16 copies these with 16-byte loads and stores
static_assert(sizeof(PrePostArgs) % 16 == 0 && alignof(PrePostArgs) >= 16, "PrePostArgs: 16-byte copies");
static_assert(sizeof(RefineArgs) % 16 == 0 && alignof(RefineArgs) >= 16, "RefineArgs: 16-byte copies");
static_assert(sizeof(BatchTask) % 16 == 0, "BatchTask: 16-byte copies");
