// Integration kernels (PLAIN and QUEUE layouts) and their launch helper,
// instantiated per (species capacity, matrix precision) in the kin_tu_*.cu
// translation units so that the library compiles in parallel.
#pragma once
#include <cuda_runtime.h>

#include "../../include/kin.h"
#include "kin_coop.cuh"
#include "kin_radau.cuh"
#include "kin_team.cuh"
#include "kin_warp.cuh"

namespace kin {

#define KIN_CUDA_TRY(expr)                                                    \
  do {                                                                        \
    cudaError_t e_ = (expr);                                                  \
    if (e_ != cudaSuccess) {                                                  \
      (void)cudaGetLastError();                                               \
      return e_ == cudaErrorMemoryAllocation ? KIN_ERR_NOMEM : KIN_ERR_CUDA; \
    }                                                                         \
  } while (0)

// Shared memory a block may hold, and a kernel opened to it.  The limit is an
// attribute of the kernel in the whole process: set to what a call needs,
// another thread's smaller call could lower it between this call's setting and
// its launch, which is then refused.  So it is always set to the whole.
constexpr size_t BLOCK_SMEM = 227 * 1024;
template <typename K>
inline cudaError_t open_smem(K *kern) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BLOCK_SMEM);
}

__host__ __device__ inline size_t smem_bytes(const MechLayout &L) {
  return sizeof(double) * (size_t)L.nd + sizeof(int) * (size_t)L.ni;
}

// Species capacity of the small-mechanism thread kernels: the per-thread
// workspace is sized for it (a smaller one spills less).
#ifndef KIN_SMALL_MAXN
#define KIN_SMALL_MAXN 16
#endif
constexpr int SMALL_MAXN = KIN_SMALL_MAXN;

struct KernelArgs {
  MechLayout L;
  const double *tab;
  const int *itab;
  double *Y, *T;
  const double *P;
  int32_t *status, *counters;
  unsigned long long *totals;
  RadauParams rp;
  int refill_min;        // QUEUE: idle lanes of a warp that trigger a refill
  const int32_t *order;  // slot -> state permutation or null (identity)
  void *gscratch;        // WARP: per-group Jacobian slots (N x (N+1) doubles each)
  int64_t gslots;        // number of slots in gscratch
  const unsigned char *hot;  // WARP with 32 lanes: the teams' tables (kin_team.cuh)
  int hot_smem;              // copied to shared memory by each block
};

// The state a slot carries: order[slot] when an order is given, else the
// slot itself.  Entries outside [0, n) are skipped (-1) and counted in
// totals[10], so a bad permutation cannot reach memory out of bounds.
__device__ __forceinline__ int64_t state_of(const KernelArgs &a, int64_t slot) {
  if (!a.order) return slot;
  const int32_t s = a.order[slot];
  if (s < 0 || (int64_t)s >= a.rp.n) {
    atomicAdd(a.totals + 10, 1ull);
    return -1;
  }
  return (int64_t)s;
}

template <int MAXN, typename LT>
__device__ void load_state(Work<MAXN, LT> &w, const KernelArgs &a, int N, int64_t i) {
  const int64_t n = a.rp.n;
  w.y[0] = a.T[i];
  for (int k = 0; k < N - 1; ++k) w.y[1 + k] = a.Y[(int64_t)k * n + i];
}

template <int MAXN, typename LT>
__device__ void store_state(const Work<MAXN, LT> &w, const StepState &s, const KernelArgs &a,
                            int N, int64_t i) {
  const int64_t n = a.rp.n;
  a.T[i] = w.y[0];
  double sum = 0.0;
  for (int k = 0; k < N - 1; ++k) {
    a.Y[(int64_t)k * n + i] = w.y[1 + k];
    sum += w.y[1 + k];
  }
  a.Y[(int64_t)(N - 1) * n + i] = 1.0 - sum;
  if (a.status) a.status[i] = s.status;
  if (a.counters) {
    const int32_t c[8] = {s.nstep, s.naccpt, s.nrejct, s.nfcn, s.njac, s.ndec, s.nsol, s.status};
    for (int q = 0; q < 8; ++q) a.counters[(int64_t)q * n + i] = c[q];
  }
  const unsigned long long c7[7] = {(unsigned long long)s.nstep, (unsigned long long)s.naccpt,
                                    (unsigned long long)s.nrejct, (unsigned long long)s.nfcn,
                                    (unsigned long long)s.njac, (unsigned long long)s.ndec,
                                    (unsigned long long)s.nsol};
  for (int q = 0; q < 7; ++q) atomicAdd(a.totals + q, c7[q]);
  if (s.status) atomicAdd(a.totals + 7, 1ull);
  atomicMax(a.totals + 8, (unsigned long long)s.nstep);
}

// Tuning of the thread layouts (measured on 2^18 H2 states; the per-thread
// workspace spills, so latency hiding matters more than spill volume):
//   * 64 threads per block and at least KIN_THREAD_MIN_BLOCKS resident blocks
//     per SM, which caps a thread's registers (20: 48 registers, 40 warps per
//     SM; 0 leaves the allocator free: 168 registers, 12 warps);
//   * the mechanism tables read through L1 rather than staged in shared
//     memory per block (-DKIN_THREAD_TABLES_SMEM stages them), with the
//     unified L1/shared memory split towards L1 (KIN_THREAD_CARVEOUT, percent
//     given to shared memory; -1 = driver default).
// Together: 144k -> 178k states/s (FP32 matrices) and 106k -> 131k (FP64).
#ifndef KIN_THREAD_MIN_BLOCKS
#define KIN_THREAD_MIN_BLOCKS 20
#endif
#if KIN_THREAD_MIN_BLOCKS > 0
#define KIN_THREAD_BOUNDS __launch_bounds__(64, KIN_THREAD_MIN_BLOCKS)
#else
#define KIN_THREAD_BOUNDS __launch_bounds__(64)
#endif
#ifndef KIN_THREAD_CARVEOUT
#define KIN_THREAD_CARVEOUT 0
#endif
#ifdef KIN_THREAD_TABLES_SMEM
#define KIN_THREAD_VIEW(a, smem) stage_tables((a).L, (a).tab, (a).itab, smem)
#else
#define KIN_THREAD_VIEW(a, smem) make_view((a).L, (a).tab, (a).itab)
#endif

// Dynamic shared memory of a thread-layout block: the staged tables (if any),
// then the right-hand side's shared scratch (if any), 8-byte aligned.
__host__ __device__ inline size_t thread_tables_bytes(const MechLayout &L) {
#ifdef KIN_THREAD_TABLES_SMEM
  return (smem_bytes(L) + 7) / 8 * 8;
#else
  (void)L;
  return 0;
#endif
}
template <int MAXN>
__host__ __device__ inline size_t thread_smem_bytes(const MechLayout &L, int block) {
#ifdef KIN_THREAD_SCRATCH_SMEM
  return thread_tables_bytes(L) + ChemScratchS<MAXN>::bytes(L.ns, block);
#else
  (void)block;
  return thread_tables_bytes(L);
#endif
}
template <int MAXN, typename LT>
__device__ __forceinline__ void bind_scratch(Work<MAXN, LT> &w, const KernelArgs &a, double *smem) {
#ifdef KIN_THREAD_SCRATCH_SMEM
  w.cs.bind(smem + thread_tables_bytes(a.L) / 8, a.L.ns);
#else
  (void)w;
  (void)a;
  (void)smem;
#endif
}

// Resident 64-thread blocks per SM that a PLAIN kernel's registers allow.  What
// bounds a batch is the FP64 unit, which a few warps per sub-partition keep
// busy, the spills that fewer registers cost, and the last wave's tail.  A
// batch of many waves takes KIN_THREAD_MIN_BLOCKS (48 registers: the tail is
// short, hiding the spills' latency pays); one of a wave or two takes the
// variant (168, 96 or 72 registers) that was fastest for its blocks per SM.
// Ordered mixed H2 states, ms with 6, 10, 14 and 20 blocks per SM, FP64 at
// dt = 1e-6 s, then FP32 matrices at 1e-4 s:
//    50021 ( 6 blocks per SM)  203 210 211 214    223 230 236 239
//    80000 ( 9)                323 287 338 400    397 365 414 504
//   131072 (14)                471 491 523 705    614 578 644 735
//   160000 (17)                    568 607 739        619 675 776
//   200000 (21)                712 690 687 765    847 879 743 799
//   220000 (23)                    769 737 830        919 854 839
//  1048576 (108), FP32 only                      3986 3758 3565 3337
// and in input order with 10, 14 and 20:
//   160000                         683 791 917        662 683 827
//   180000 (19)                    905 831 942        820 746 836
constexpr int PLAIN_BLOCKS_FEW = 6, PLAIN_BLOCKS_MID = 10, PLAIN_BLOCKS_MANY = 14;
constexpr int PLAIN_USE_FEW = 6, PLAIN_USE_MID = 17, PLAIN_USE_MANY = 21;  // up to, per SM

template <int MAXN, typename LT, bool FDJ, int MINB>
__global__ void __launch_bounds__(64, MINB) k_integrate_plain(KernelArgs a) {
  extern __shared__ double smem[];
  const MechView m = KIN_THREAD_VIEW(a, smem);
  const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (slot >= a.rp.n) return;
  const int64_t i = state_of(a, slot);
  if (i < 0) return;
  Work<MAXN, LT> w;
  bind_scratch(w, a, smem);
  StepState s;
  const int N = m.ns;
  load_state(w, a, N, i);
  integrate_plain<MAXN, LT, FDJ>(m, a.P[i], w, s, a.rp, i);
  store_state(w, s, a, N, i);
}

template <int MAXN, typename LT, bool FDJ>
__global__ void KIN_THREAD_BOUNDS k_integrate_queue(KernelArgs a) {
  extern __shared__ double smem[];
  const MechView m = KIN_THREAD_VIEW(a, smem);
  const int N = m.ns;
  const int64_t n = a.rp.n;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned long long *queue = a.totals + 9;
  Work<MAXN, LT> w;
  bind_scratch(w, a, smem);
  StepState s;
  int64_t idx = -1;
  double P = 0.0;
  bool exhausted = false;  // warp-uniform: the queue has no more states
  // One step attempt per trip for every lane that holds a state.  Idle lanes
  // wait until refill_min of the warp's lanes are idle, then take that many
  // states with one atomic, so refilled lanes start their integrations
  // together.  Every state ends after at most max_steps attempts, so the
  // warp's loop is bounded.
  for (;;) {
    const unsigned idle = __ballot_sync(FULL, idx < 0);
    if (exhausted && idle == FULL) break;
    const int nidle = __popc(idle);
    if (!exhausted && nidle >= a.refill_min) {
      const int leader = __ffs(idle) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(queue, (unsigned long long)nidle);
      base = __shfl_sync(FULL, base, leader);
      if (base + (unsigned long long)nidle >= (unsigned long long)n) exhausted = true;
      if (idx < 0) {
        const unsigned long long t = base + __popc(idle & ((1u << lane) - 1u));
        if (t < (unsigned long long)n) idx = state_of(a, (int64_t)t);
        if (idx >= 0) {
          P = a.P[idx];
          load_state(w, a, N, idx);
          if (radau_init<MAXN, LT, FDJ>(m, P, w, s, a.rp, idx)) {
            store_state(w, s, a, N, idx);
            idx = -1;
          }
        }
      }
    }
    if (idx >= 0 && radau_step<MAXN, LT, FDJ>(m, P, w, s, a.rp, idx)) {
      store_state(w, s, a, N, idx);
      idx = -1;
    }
  }
}

// PLAIN on a small batch: one state per block (kin_coop.cuh).  Eight blocks
// per SM cap the registers at 80; a batch of 1024 is seven states per SM.
template <typename LT, bool FDJ>
__global__ void __launch_bounds__(COOP_NT, 8) k_integrate_coop(KernelArgs a) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  CoopState<LT> &c = *reinterpret_cast<CoopState<LT> *>(coop_smem);
  const MechView m = make_view(a.L, a.tab, a.itab);
  const int nr = m.nr, N = m.ns, tid = threadIdx.x;
  CoopTail<LT> t;
  t.q = reinterpret_cast<double *>(coop_smem + (sizeof(CoopState<LT>) + 15) / 16 * 16);
  t.pkf = reinterpret_cast<LT *>(t.q + 3 * nr);
  t.pkr = t.pkf + nr;
  t.uJ = t.pkf + 2 * nr;
  t.sJ = t.pkf + 3 * nr;
  t.tJ = t.pkf + 4 * nr;
  t.occ = reinterpret_cast<int *>(t.pkf + 5 * nr);
  if (tid == 0) c.outcome = (int)state_of(a, blockIdx.x);
  __syncthreads();
  const int64_t i = c.outcome, n = a.rp.n;
  if (i < 0) return;
  Coop<LT> w{m, c, t, a.P[i]};
  if (tid < N) c.y[tid] = tid == 0 ? a.T[i] : a.Y[(int64_t)(tid - 1) * n + i];
  w.build_lists();  // ends with a barrier
  // every attempt ends the loop or counts a step; max_steps bounds it
  bool done = w.template init<FDJ>(a.rp, i);
  while (!done) done = w.template step<FDJ>(a.rp, i);
  __syncthreads();
  if (tid < N) (tid == 0 ? a.T[i] : a.Y[(int64_t)(tid - 1) * n + i]) = c.y[tid];
  if (tid == 0) {
    const StepState &s = c.s;
    double sum = 0.0;
    for (int k = 0; k < N - 1; ++k) sum += c.y[1 + k];
    a.Y[(int64_t)(N - 1) * n + i] = 1.0 - sum;
    if (a.status) a.status[i] = s.status;
    const int32_t v[8] = {s.nstep, s.naccpt, s.nrejct, s.nfcn, s.njac, s.ndec, s.nsol, s.status};
    for (int q = 0; q < 8; ++q) {
      if (a.counters) a.counters[(int64_t)q * n + i] = v[q];
      if (q < 7) atomicAdd(a.totals + q, (unsigned long long)v[q]);
    }
    if (s.status) atomicAdd(a.totals + 7, 1ull);
    atomicMax(a.totals + 8, (unsigned long long)s.nstep);
  }
}

// PLAIN batches of at most this many states go to k_integrate_coop: its time
// grows with the batch, the per-thread kernel's is flat (a chain of FP64
// latencies) until its warps fill the chip.  H2 (13 species, 27 reactions),
// dt = 1e-6 / 1e-4 s, ms, coop against per thread: FP64 2048: 40 / 60 against
// 150 / 154, 6144: 110 / 169 against 117 / 157, 8192: 145 / 226 against 119 /
// 159; FP32 2048: 26 / 36 against 84 / 116, 6144: 68 / 105 against 86 / 118,
// 8192: 91 / 141 against 87 / 120.  With fewer reactions a thread's chain is
// shorter and the lines cross earlier, depending on how unequal the states are
// (subsets of the H2 species, dt = 1e-6 / 1e-4 s):
//   4 species,   FP64 1216: 0.24 / 0.42 against 0.28 / 0.65
//   1 reaction        2000: 0.42 / 0.61 against 0.28 / 0.65
//   6, 4              5632: 1.7 / 5.0 against 1.7 / 10.8
//   8, 7              4000: 24 / 36 against 27 / 41     5632: 34 / 50 against 27 / 41
//                FP32 4000: 18 / 27 against 21 / 32     5632: 25 / 36 against 21 / 32
//   10, 14       FP64 4000: 58 / 90 against 69 / 91     5632: 81 / 124 against 68 / 90
//                FP32 4000: 37 / 56 against 51 / 66     5632: 51 / 78 against 51 / 66
// More reactions move the line up (16 species, 300 reactions, 20000 states: 747
// against 1020), difference Jacobians too (16 species, 27 reactions, 9000: 194
// against 291); neither raises the limit.  Both kernels give the same bits.
inline int64_t coop_max_n(const MechLayout &L, size_t lt) {
  const bool f64 = lt == sizeof(double);
  if (L.nr < 3) return 1700;
  if (L.nr >= 6 && L.nr < 20) return f64 ? 4400 : 4700;
  return f64 ? 5632 : 6912;
}
// ... and a mechanism whose reaction tail leaves several blocks per SM
constexpr size_t COOP_MAX_SMEM = 64 * 1024;

// a finished state's status and counters, by lane 0 of its group
template <int L>
__device__ __forceinline__ void store_counts(const StepState &s, const KernelArgs &a, int64_t idx) {
  if (Grp<L>::lane() != 0) return;
  const int64_t n = a.rp.n;
  const int32_t c[8] = {s.nstep, s.naccpt, s.nrejct, s.nfcn, s.njac, s.ndec, s.nsol, s.status};
  if (a.status) a.status[idx] = s.status;
  for (int q = 0; q < 8; ++q) {
    if (a.counters) a.counters[(int64_t)q * n + idx] = c[q];
    if (q < 7) atomicAdd(a.totals + q, (unsigned long long)c[q]);
  }
  if (s.status) atomicAdd(a.totals + 7, 1ull);
  atomicMax(a.totals + 8, (unsigned long long)s.nstep);
}

// a finished state's vector, status and counters, from its group of L lanes
template <int L>
__device__ __forceinline__ void store_lanes(const WVecT<Grp<L>::WR> &y, const StepState &s,
                                            const KernelArgs &a, int N, int64_t idx) {
  using G = Grp<L>;
  const int lane = G::lane();
  const int64_t n = a.rp.n;
  double sum = 0.0;
#pragma unroll
  for (int r = 0; r < G::WR; ++r) {
    const int g = lane + L * r;
    if (g == 0) a.T[idx] = y.v[r];
    if (g >= 1 && g < N) {
      a.Y[(int64_t)(g - 1) * n + idx] = y.v[r];
      sum += y.v[r];
    }
  }
  sum = G::sum(sum);
  if (lane == 0) a.Y[(int64_t)(N - 1) * n + idx] = 1.0 - sum;
  store_counts<L>(s, a, idx);
}

// WARP layout: one state per group of L lanes; groups pop states from the
// atomic queue.
// Register cap of the WARP kernels (0: the compiler's choice under the
// 256-thread bound): a build-time tuning knob.
#ifndef KIN_WARP_MAXNREG
#define KIN_WARP_MAXNREG 0
#endif
#if KIN_WARP_MAXNREG > 0
#define KIN_WARP_BOUNDS __maxnreg__(KIN_WARP_MAXNREG)
#else
#define KIN_WARP_BOUNDS __launch_bounds__(256)
#endif

template <int L, typename LT, bool FDJ>
__global__ void KIN_WARP_BOUNDS k_integrate_lanes(KernelArgs a) {
  using G = Grp<L>;
  constexpr int WR = G::WR;
  extern __shared__ double smem[];
  // the mechanism tables are read through L1 from global memory: shared
  // memory holds only the groups' matrices and vectors
  const MechView m = make_view(a.L, a.tab, a.itab);
  const int N = m.ns, lane = G::lane(), grp = (int)(threadIdx.x / L);
  const int64_t n = a.rp.n;
  char *base = reinterpret_cast<char *>(smem) + (size_t)grp * warp_buf_bytes(N, m.nr, sizeof(LT));
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x / L) + grp;  // < gslots (launch)
  LT *Jg = reinterpret_cast<LT *>(a.gscratch) +
           slot * (int64_t)warp_slot_mats(sizeof(LT)) * N * (N + 1);
  const WarpBuf<LT> b = carve_warp_buf<LT>(base, N, m.nr, Jg);
  unsigned long long *queue = a.totals + 9;
  WStateT<WR> w;
  StepState s;
  for (;;) {
    unsigned long long t = 0;
    if (lane == 0) t = atomicAdd(queue, 1ull);
    t = G::bcast(t, 0);
    if (t >= (unsigned long long)n) break;
    int64_t idx = 0;
    if (lane == 0) idx = state_of(a, (int64_t)t);
    idx = G::bcast(idx, 0);
    if (idx < 0) continue;
    const double P = a.P[idx];
#pragma unroll
    for (int r = 0; r < WR; ++r) {
      const int g = lane + L * r;
      w.y.v[r] = (g == 0) ? a.T[idx] : (g < N ? a.Y[(int64_t)(g - 1) * n + idx] : 0.0);
    }
    // every attempt ends the loop or counts a step; max_steps bounds it
    bool done = warp_init<L, LT, FDJ>(m, b, P, w, s, a.rp, idx);
    while (!done) done = warp_step<L, LT, FDJ>(m, b, P, w, s, a.rp, idx);
    store_lanes<L>(w.y, s, a, N, idx);
    G::sync();
  }
}

// Shared memory of one block of `warps` warps for L lanes per state.
__host__ __device__ inline size_t lanes_smem_bytes(const MechLayout &L_, int lanes, size_t lt,
                                                   int warps) {
  return (size_t)warps * (32 / lanes) * warp_buf_bytes(L_.ns, L_.nr, lt);
}

// WARP layout with 32 lanes: a state per team of three warps (kin_team.cuh),
// up to TEAMS teams per block, one block per SM.
template <typename LT, bool FDJ, int TEAMS>
__global__ void __launch_bounds__(TEAMS *TEAM_NT, 1) k_integrate_team(KernelArgs a) {
  using G = Grp<32>;
  extern __shared__ __align__(16) unsigned char team_smem[];
  const MechView m = make_view(a.L, a.tab, a.itab);
  const int N = m.ns, lane = G::lane(), warp = (int)(threadIdx.x / 32);
  const int team = warp / TEAM_WARPS, wt = warp % TEAM_WARPS;
  const int64_t n = a.rp.n;
  const HotTables h = stage_hot(a.L, a.hot, a.hot_smem != 0, team_smem);
  const size_t tb = team_bytes(a.L, N, sizeof(LT));
  const size_t hb = a.hot_smem ? hot_offsets(a.L).bytes : 0;
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x / TEAM_NT) + team;  // < gslots (launch)
  const TeamBuf<LT> t = carve_team<LT>(
      a.L, team_smem + hb + team * tb, team, N,
      reinterpret_cast<unsigned char *>(a.gscratch) +
          slot * (int64_t)warp_slot_mats(sizeof(LT)) * N * (N + 1) * (int64_t)sizeof(LT));
  const TeamMassFrac<LT> f{m, h, t};
  if (wt != 0) {  // workers: a part of each command until the leader is done
    for (;;) {
      named_sync(t.bar, TEAM_NT);
      const int cmd = t.ctl->cmd;
      if (cmd == TEAM_QUIT) return;
      team_exec<LT>(cmd, wt, f);
      named_sync(t.bar, TEAM_NT);
    }
  }
  const TeamSys<LT, TeamMassFrac<LT>> sys{f};
  WarpBuf<LT> b{};
  b.J = t.J;
  unsigned long long *queue = a.totals + 9;
  WStateT<2> w;
  StepState s;
  for (;;) {
    unsigned long long q = 0;
    if (lane == 0) q = atomicAdd(queue, 1ull);
    q = G::bcast(q, 0);
    if (q >= (unsigned long long)n) break;
    int64_t idx = 0;
    if (lane == 0) idx = state_of(a, (int64_t)q);
    idx = G::bcast(idx, 0);
    if (idx < 0) continue;
    const double P = a.P[idx];
    if (lane == 0) t.ctl->P = P;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int g = lane + 32 * r;
      w.y.v[r] = (g == 0) ? a.T[idx] : (g < N ? a.Y[(int64_t)(g - 1) * n + idx] : 0.0);
    }
    // every attempt ends the loop or counts a step; max_steps bounds it
    bool done = warp_init_sys<32, LT, FDJ>(sys, b, P, w, s, a.rp, idx);
    while (!done) done = warp_step_sys<32, LT, FDJ>(sys, b, P, w, s, a.rp, idx);
    store_lanes<32>(w.y, s, a, N, idx);
  }
  sys.post(TEAM_QUIT);
}

struct TeamLaunch {
  unsigned grid, threads;
  size_t smem;
};

// teams per block and blocks for a batch; the tables go to shared memory when
// a team fits beside them.  A team always fits: a mechanism's tables are at
// most 200 KB (build_tables); a reaction takes 64 bytes there and 12 more per
// species that it changes and per collision efficiency, and of a team's buffers
// 24 bytes and 8 per slot and efficiency, beside at most 45 KB of matrices and
// species vectors.  (Only some 2900 reactions of six slots that change no
// species at all would not; they are refused.)
inline bool team_shape(KernelArgs &a, int N, size_t lt, int sms, int most, TeamLaunch &g) {
  const size_t budget = BLOCK_SMEM, tb = team_bytes(a.L, N, lt), hot = hot_offsets(a.L).bytes;
  if (!a.hot || tb > budget) return false;
  a.hot_smem = hot + tb <= budget;
  const size_t fixed = a.hot_smem ? hot : 0;
  int64_t teams = (int64_t)((budget - fixed) / tb);
  teams = teams < most ? teams : most;
  const int64_t want = (a.rp.n + sms - 1) / sms;  // a small batch spreads over the SMs
  teams = teams < want ? teams : want;
  int64_t grid = (a.rp.n + teams - 1) / teams;
  grid = grid < sms ? grid : sms;
  if (grid * teams > a.gslots) grid = a.gslots / teams;  // one slot per team
  if (grid < 1) return false;
  g = TeamLaunch{(unsigned)grid, (unsigned)(teams * TEAM_NT), fixed + teams * tb};
  return true;
}

// most teams per block for n states of N unknowns: the many from two rounds of
// them on (at 1e-4 s 1500 states of 17 to 24 species were 2 % slower with
// seven); difference Jacobians, three right-hand sides at a time, keep every
// warp busy with four (20 species, 10000 states: 283 ms against 288)
inline int team_most(size_t lt, bool fd, int N, int64_t n, int sms) {
  return lt == sizeof(float) && !fd && N <= TEAM_MANY_N && n >= 2ll * TEAM_MANY * sms ? TEAM_MANY
                                                                                    : TEAM_MAX;
}

// workspace slots per SM that teams of N unknowns can use
inline int team_slots(int N) { return N <= TEAM_MANY_N ? TEAM_MANY : TEAM_MAX; }

template <typename LT, bool FDJ>
int launch_team(KernelArgs a, cudaStream_t st, int sms) {
  if (!a.gscratch || a.gslots < 1) return KIN_ERR_UNSUPPORTED;
  TeamLaunch g;
  const int most = team_most(sizeof(LT), FDJ, a.L.ns, a.rp.n, sms);
  if (!team_shape(a, a.L.ns, sizeof(LT), sms, most, g)) return KIN_ERR_UNSUPPORTED;
  auto kern = k_integrate_team<LT, FDJ, TEAM_MAX>;
  if constexpr (sizeof(LT) == sizeof(float) && !FDJ)
    if (most == TEAM_MANY) kern = k_integrate_team<LT, FDJ, TEAM_MANY>;
  KIN_CUDA_TRY(open_smem(kern));
  kern<<<g.grid, g.threads, g.smem, st>>>(a);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

template <int L, typename LT, bool FDJ>
int launch_lanes(const KernelArgs &a, cudaStream_t st, int sms) {
  using G = Grp<L>;
  if (a.L.ns >= G::CAP) return KIN_ERR_UNSUPPORTED;
  if (!a.gscratch || a.gslots < 1) return KIN_ERR_UNSUPPORTED;
  const size_t budget = BLOCK_SMEM;
  auto kern = k_integrate_lanes<L, LT, FDJ>;
  KIN_CUDA_TRY(open_smem(kern));
  // the block size (1 to 8 warps) that keeps the most warps resident per SM
  int warps = 0, per_sm = 0;
  for (int w = 8; w >= 1; w >>= 1) {
    const size_t smw = lanes_smem_bytes(a.L, L, sizeof(LT), w);
    if (smw > budget) continue;
    int b = 0;
    KIN_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, 32 * w, smw));
    if (b * w > per_sm * warps) {
      warps = w;
      per_sm = b;
    }
  }
  if (warps < 1 || per_sm < 1) return KIN_ERR_UNSUPPORTED;
  const size_t sm = lanes_smem_bytes(a.L, L, sizeof(LT), warps);
  int64_t grid = (int64_t)sms * per_sm;
  const int64_t per_block = (int64_t)warps * (32 / L);
  const int64_t need = (a.rp.n + per_block - 1) / per_block;
  if (grid > need) grid = need;
  if (grid * per_block > a.gslots) grid = a.gslots / per_block;  // one J slot per group
  if (grid < 1) return KIN_ERR_UNSUPPORTED;
  kern<<<(unsigned)grid, 32 * warps, sm, st>>>(a);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

template <int MAXN, typename LT, bool FDJ>
int launch_t(const KernelArgs &a, const kin_options &o, cudaStream_t st, int sms) {
  if (o.layout == KIN_LAYOUT_WARP) {
    if constexpr (MAXN == 64) {
      if (a.L.ns > 63) return KIN_ERR_UNSUPPORTED;
      return launch_team<LT, FDJ>(a, st, sms);
    } else {
      return KIN_ERR_UNSUPPORTED;
    }
  }
  const bool plain = o.layout == KIN_LAYOUT_PLAIN;
  const int block = o.block > 0 ? o.block : 64;
  if (block > 64 || block % 32) return KIN_ERR_INVALID_ARG;
  const size_t sm = thread_smem_bytes<MAXN>(a.L, block);
  const int carve = KIN_THREAD_CARVEOUT;  // percent of the unified L1 given to shared memory
  if constexpr (MAXN <= COOP_CAP) {
    const size_t smc = coop_smem_bytes<LT>(a.L.nr);
    if (plain && a.rp.n > 0 && a.rp.n <= coop_max_n(a.L, sizeof(LT)) &&
        smc <= COOP_MAX_SMEM) {
      auto kern = k_integrate_coop<LT, FDJ>;
      KIN_CUDA_TRY(open_smem(kern));
      kern<<<(unsigned)a.rp.n, COOP_NT, smc, st>>>(a);
      KIN_CUDA_TRY(cudaGetLastError());
      return KIN_OK;
    }
  }
  if (plain) {
    // the variant with the fewest registers has the largest frame; an empty
    // batch (reserve_frames) runs one idle block of it
    void (*kern)(KernelArgs) = k_integrate_plain<MAXN, LT, FDJ, KIN_THREAD_MIN_BLOCKS>;
    if constexpr (MAXN <= 16 && !FDJ) {
      const int64_t per_sm = (a.rp.n + 64ll * sms - 1) / (64ll * sms);
      if (per_sm > 0) {
        if (per_sm <= PLAIN_USE_FEW)
          kern = k_integrate_plain<MAXN, LT, FDJ, PLAIN_BLOCKS_FEW>;
        else if (per_sm <= PLAIN_USE_MID)
          kern = k_integrate_plain<MAXN, LT, FDJ, PLAIN_BLOCKS_MID>;
        else if (per_sm <= PLAIN_USE_MANY)
          kern = k_integrate_plain<MAXN, LT, FDJ, PLAIN_BLOCKS_MANY>;
      }
    }
    KIN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    KIN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    const int64_t grid = (a.rp.n + block - 1) / block;
    kern<<<grid > 0 ? (unsigned)grid : 1u, block, sm, st>>>(a);
  } else {
    auto kern = k_integrate_queue<MAXN, LT, FDJ>;
    KIN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    KIN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    int per_sm = o.grid_per_sm;
    if (per_sm <= 0) {
      KIN_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, block, sm));
      if (per_sm < 1) per_sm = 1;
    }
    int64_t grid = (int64_t)sms * per_sm;
    const int64_t need = (a.rp.n + block - 1) / block;
    if (grid > need) grid = need;
    kern<<<(unsigned)grid, block, sm, st>>>(a);
  }
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}


// Per-TU entry points: launch for one (MAXN, LT) pair and upload this TU's
// copy of the Radau constants.
#define KIN_DEFINE_TU(NAME, MAXN, LT)                                                   \
  int kin_launch_##NAME(const KernelArgs &a, const kin_options &o, cudaStream_t st,    \
                        int sms) {                                                     \
    return o.jac_fd ? launch_t<MAXN, LT, true>(a, o, st, sms)                          \
                    : launch_t<MAXN, LT, false>(a, o, st, sms);                        \
  }                                                                                    \
  int kin_consts_##NAME(const RadauConst &rc) {                                        \
    KIN_CUDA_TRY(cudaMemcpyToSymbol(RC, &rc, sizeof rc));                              \
    return KIN_OK;                                                                     \
  }

#define KIN_DECLARE_TU(NAME)                                                            \
  int kin_launch_##NAME(const KernelArgs &a, const kin_options &o, cudaStream_t st,    \
                        int sms);                                                      \
  int kin_consts_##NAME(const RadauConst &rc);

// Groups of 4, 8 or 16 lanes per state (at most 15 species) for one matrix
// precision, in their own translation units.
#define KIN_DEFINE_GROUP_TU(NAME, LT)                                                   \
  int kin_launch_##NAME(const KernelArgs &a, const kin_options &o, cudaStream_t st,    \
                        int sms) {                                                     \
    const bool fd = o.jac_fd != 0;                                                     \
    switch (o.lanes) {                                                                 \
      case 4: return fd ? launch_lanes<4, LT, true>(a, st, sms)                        \
                        : launch_lanes<4, LT, false>(a, st, sms);                      \
      case 8: return fd ? launch_lanes<8, LT, true>(a, st, sms)                        \
                        : launch_lanes<8, LT, false>(a, st, sms);                      \
      case 16: return fd ? launch_lanes<16, LT, true>(a, st, sms)                      \
                         : launch_lanes<16, LT, false>(a, st, sms);                    \
      default: return KIN_ERR_INVALID_ARG;                                             \
    }                                                                                  \
  }                                                                                    \
  int kin_consts_##NAME(const RadauConst &rc) {                                        \
    KIN_CUDA_TRY(cudaMemcpyToSymbol(RC, &rc, sizeof rc));                              \
    return KIN_OK;                                                                     \
  }

KIN_DECLARE_TU(16d)
KIN_DECLARE_TU(16f)
KIN_DECLARE_TU(64d)
KIN_DECLARE_TU(64f)
KIN_DECLARE_TU(grpd)
KIN_DECLARE_TU(grpf)

}  // namespace kin
