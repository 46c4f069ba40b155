// steps.cuh -- several time steps of a batch in one cooperative launch.
//
// A batch that does not fill the device is bound by latency, not by bytes: a
// step of three dependent launches (k_pass, k_collide, k_field) spends its
// time in their prologues, drains and hand-overs (a run of 16,384 particles:
// 28 us per step for 0.1 us of traffic).  k_steps keeps a block on each of its
// SMs for a run of steps.  Every block belongs to one run (its team shares the run's
// particles); the run's tables, grid and field stay in shared memory, real
// collisions are carried out by the pass itself (a thread has two or four
// times the pass kernel's registers), and each block solves the run's field
// for itself, so that a step needs one barrier of the team (1.3 us, bound by
// the round trips to L2) and no hand-over of a result.  Teams never wait for
// one another.  A sample step adds its sums in shared memory as fixed-point
// integers (mom_add4) and shares its moments among the team's blocks.
//
// Measured, us per step of one run with samples every 20 steps and sorts every
// 32 (one launch per phase : here): 16,384 particles on 128 cells 28 : 11; 58,254
// on 114 cells 27 : 12; 524,288 on 1024 cells 38 : 18; 2.1 million on 2048 cells
// 62 : 37.  What is left of the smallest step: the chain of a piece
// (loads, Philox, push, deposit, null-collision test, flush), the barrier and
// the field, about 6, 2 and 4 us.
//
// The particle arithmetic is the phase kernels' own code (step_dev.cuh) and
// the field is formed in the same order, so a trajectory is the same bit for
// bit whichever way a batch takes.
#pragma once
#include "step_dev.cuh"

namespace ecpic {

namespace {

// Polls of a barrier before a block gives up (seconds, where a step takes
// microseconds); the run then fails with ECPIC_ERR_TIMEOUT.
constexpr int kMaxPolls = 1 << 23;

// Threads per block: 512 (128 registers each), or 256 (255 registers) where a
// block has few particles.
constexpr int kStepWarps = 512 / 32;  // at most

struct StepShared {
  RunDev run;
  SegDev seg[kMaxSpecies];
  BatchView b;
  FusedStep fx;
  PassShared pass;
  long long cap[kMaxSpecies], fresh[kMaxSpecies];
  unsigned first[kMaxSpecies + 1];  // the team's blocks of species s: first[s] .. first[s + 1] - 1
  unsigned long long wtot[kMaxSpecies][kStepWarps];
  double owner[kFieldOwners / 8 * 9];  // eight of every nine: no bank conflicts
  double wsm[32];
  double phi0[32];  // electrode potential of 32 levels
  double cs, g0, kc;
  int ok, fail, split, spc;
};

// Dynamic shared memory: StepShared, then dx | background prefix | MC weights
// (doubles per node); C and the deposit (a word per node and species) while
// the field is solved, the sample sums of a piece before it, in one place; the
// field, then what a piece of the pass needs.
constexpr int kMomCells = 1280;  // window of the sample sums: 77 KB
constexpr size_t kStepBase = (sizeof(StepShared) + 15) / 16 * 16;
__host__ __device__ inline int scratch_words(int nmax, int species) {  // of 4 bytes
  const int M = nmax + 1, field = 2 * (1 + species) * M;
  const int sums = 3 * kMomSums * (M < kMomCells ? M : kMomCells);
  return field > sums ? field : sums;
}
__host__ __device__ inline size_t steps_bytes(int nmax, int species, bool weighted, int threads) {
  const size_t M = (size_t)nmax + 1;
  return kStepBase + M * (size_t)(3 * 8 + 4 + 4 * (weighted ? 4 : 3)) + 4 * (size_t)scratch_words(nmax, species) +
         sizeof(int) * (size_t)kRing * (size_t)(threads / 32);
}

// Where everything is.  Every function forms the addresses from the base of
// the dynamic shared memory, so that its accesses are shared-memory
// instructions (a pointer read from memory would make them generic ones).
extern __shared__ __align__(16) unsigned char step_smem[];
__device__ __forceinline__ StepShared& step_shared() { return *reinterpret_cast<StepShared*>(step_smem); }
struct StepArrays {
  double *D, *V, *W, *C;
  unsigned long long* Q;
  float* mom;  // shares C's and Q's place
  float* E;
  uint32_t* dep;
  unsigned char* ring;
};
__device__ __forceinline__ StepArrays step_arrays() {
  const StepShared& sh = step_shared();
  const int M = sh.b.nmax + 1;
  StepArrays a;
  a.D = reinterpret_cast<double*>(step_smem + kStepBase);
  a.V = a.D + M;
  a.W = a.V + M;
  a.C = a.W + M;
  a.Q = reinterpret_cast<unsigned long long*>(a.C + M);
  a.mom = reinterpret_cast<float*>(a.C);
  a.E = a.mom + scratch_words(sh.b.nmax, sh.spc);
  a.dep = reinterpret_cast<uint32_t*>(a.E + M);
  a.ring = reinterpret_cast<unsigned char*>(a.dep + M * (sh.b.weighted ? 4 : 3));
  return a;
}

__device__ __forceinline__ void arrive(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Waits until the team's arrivals reach `want` (thread 0 polls); false when
// the wait gave up.  Every thread calls it.
__device__ __forceinline__ bool await(unsigned* p, unsigned want, StepShared& sh) {
  if (threadIdx.x == 0) {
    unsigned v = 0;
    for (int i = 0; i < kMaxPolls; ++i) {
      asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
      if (v >= want) break;
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    sh.ok = v >= want ? 1 : 0;
  }
  __syncthreads();
  return sh.ok != 0;
}

// FP64 instructions hold a scheduler's FP64 unit for 64 cycles a warp on this
// part (measured; 75 cycles in a dependent chain), so the ones of a rare or
// single-warp branch are written as volatile assembly, which the compiler does
// not hoist out of the branch for every warp to execute.
__device__ __forceinline__ double cvt_f64(long long q) {
  double d;
  asm volatile("cvt.rn.f64.s64 %0, %1;" : "=d"(d) : "l"(q));
  return d;
}
__device__ __forceinline__ float cvt_f32(double d) {
  float f;
  asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(d));
  return f;
}
__device__ __forceinline__ double add64(double a, double b) {
  double d;
  asm volatile("add.rn.f64 %0, %1, %2;" : "=d"(d) : "d"(a), "d"(b));
  return d;
}

// (double)q, formed by integer operations while it is exact
__device__ __forceinline__ double i64_to_f64(long long q) {
  const unsigned long long a = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
  const int lz = __clzll((long long)a);
  if (lz < 11) return cvt_f64(q);  // above 2^53: rounds
  if (a == 0ull) return 0.0;
  // the leading one lands on bit 52 and adds itself to the exponent
  const unsigned long long bits = ((unsigned long long)(1085 - lz) << 52) + (a << (lz - 11));
  return __longlong_as_double((long long)(bits | (q < 0 ? 0x8000000000000000ull : 0ull)));
}

// (float)d, rounded to nearest even by integer operations for results in the
// normal range
__device__ __forceinline__ float f64_to_f32(double d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const unsigned long long a = u & 0x7FFFFFFFFFFFFFFFull;
  if (a < 0x3810000000000000ull || a >= 0x47E0000000000000ull) return cvt_f32(d);  // below 2^-126, from 2^127
  const unsigned long long r = a + 0x0FFFFFFFull + ((a >> 29) & 1ull);
  const unsigned f = (unsigned)(r >> 29) - (896u << 23);
  return __uint_as_float(f | ((unsigned)(u >> 32) & 0x80000000u));
}

// Adds the block's counters to the run's (they are read between launches).
template <int kStepBlock>
__device__ void flush_counters(StepShared& sh, RunState* st, SegState* sst, int ns) {
  const int tid = threadIdx.x, sp = tid >> 5, lane = tid & 31;
  if (sp < ns) {
    const uint32_t v = lane < kNumCtr ? sh.fx.ctr[sp][lane] : 0u;
    if (v) {
      atomicAdd(&st->ctr[sp][lane], (unsigned long long)v);
      sh.fx.ctr[sp][lane] = 0u;
    }
    const bool dead = lane == C_ABS_L || lane == C_ABS_R || lane == C_NAN;
    const uint32_t d = __reduce_add_sync(kFull, dead ? v : 0u);
    if (lane == 0 && d) atomicAdd((unsigned long long*)&sst[sp].n_dead, (unsigned long long)d);
  } else if (tid == kStepBlock - 1 && sh.fx.nlive) {
    atomicAdd(&st->psteps, (unsigned long long)sh.fx.nlive);
    sh.fx.nlive = 0u;
  }
}

// Gives every species its blocks of the team, in proportion to its particles
// and one at least: a block with a piece of two species would take twice the
// time of the others.  A team smaller than the number of species shares every
// species among all its blocks instead (one thread).
__device__ void split_team(StepShared& sh, int ns, unsigned team) {
  if ((int)team < ns) {
    sh.split = 0;
    return;
  }
  sh.split = 1;
  long long all = 0;
  for (int s = 0; s < ns; ++s) all += sh.fx.n[s];
  long long before = 0;
  sh.first[0] = 0;
  for (int s = 0; s < ns; ++s) {
    before += sh.fx.n[s];
    const unsigned at = all > 0 ? (unsigned)((before * (long long)team + all / 2) / all) : (unsigned)(s + 1);
    sh.first[s + 1] = min(max(at, sh.first[s] + 1), team - (unsigned)(ns - 1 - s));
  }
  sh.first[ns] = team;
}

// One piece of the pass.  Functions of their own, like the field's parts: each
// has its own register allocation, and nothing of one is spilled around
// another (a spilled word read again after a barrier comes from L2).
template <int KIND, int kStepBlock, int V>
__device__ __forceinline__ void step_piece(int s, long long k, unsigned beg, unsigned end) {
  StepShared& sh = step_shared();
  const StepArrays a = step_arrays();
  const PieceState ps{sh.fx.cur[s], sh.fx.n[s], k};
  pass_piece<KIND, false, kStepBlock, true, V>(sh.b, &sh.run, sh.seg[s], sh.run.seg0 + s, ps, (long long)beg, (long long)end, MODE_STEP, a.dep, a.mom, a.ring, sh.pass, &sh.fx, a.E,
                                            scratch_words(sh.b.nmax, sh.spc));
}

// This block's share [beg, end) of species s's groups of V particles (every species has its
// blocks; a team smaller than the number of species shares every species among
// all its blocks).
template <int V = 4>
__device__ __forceinline__ bool step_share(const StepShared& sh, int s, unsigned me, unsigned team, unsigned* beg,
                                           unsigned* end) {
  const unsigned first = sh.split ? sh.first[s] : 0u;
  const unsigned count = sh.split ? sh.first[s + 1] - first : team;
  if (me < first || me - first >= count) return false;
  const unsigned T = (unsigned)((sh.fx.n[s] + V - 1) / V);
  const unsigned per = (T + count - 1) / count;
  *beg = min(T, per * (me - first));
  *end = min(T, *beg + per);
  return *beg < *end;
}

template <bool WEIGHTED, int kStepBlock, int V>
__device__ __forceinline__ void step_particles(unsigned me, unsigned team, long long k, bool sample) {
  const StepShared& sh = step_shared();
  const int ns = sh.run.ns;
  for (int s = 0; s < ns; ++s) {
    unsigned beg, end;
    if (!step_share<V>(sh, s, me, team, &beg, &end)) continue;
    if (sh.run.scheme >= ECPIC_SCHEME_EC2)
      step_piece<2, kStepBlock, V>(s, k, beg, end);
    else if (WEIGHTED && sh.run.rb && sample)
      step_piece<WEIGHTED ? 4 : 1, kStepBlock, V>(s, k, beg, end);
    else if (WEIGHTED && sh.run.rb)
      step_piece<WEIGHTED ? 3 : 0, kStepBlock, V>(s, k, beg, end);
    else if (sample)
      step_piece<1, kStepBlock, V>(s, k, beg, end);
    else
      step_piece<0, kStepBlock, V>(s, k, beg, end);
  }
}

// ---- counting sort by cell, between the barriers of a team -----------------
// The cells of a block's share of each species: counted in H (shared memory,
// one array per species, kept for the scatter) and added to the run's
// histogram.
template <int kStepBlock>
__device__ __noinline__ void sort_count(unsigned me, unsigned team) {
  const StepShared& sh = step_shared();
  const int ns = sh.run.ns, N = sh.run.N, M = N + 1;
  int* H = reinterpret_cast<int*>(step_arrays().mom);
  for (int i = threadIdx.x; i < ns * M; i += kStepBlock) H[i] = 0;
  __syncthreads();
  for (int s = 0; s < ns; ++s) {
    unsigned beg, end;
    if (!step_share(sh, s, me, team, &beg, &end)) continue;
    const int32_t* pc = sh.seg[s].cell[sh.fx.cur[s]];
    const long long n = sh.fx.n[s];
    int* h = H + s * M;
    for (unsigned q = beg + threadIdx.x; q < end; q += kStepBlock) {
      int at = -1, run = 0;  // runs of equal cells, one atomic each
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long i = 4ll * q + j;
        const int c = i < n ? pc[i] : -1;
        if (c != at) {
          if (at >= 0) atomicAdd(h + at, run);
          at = c;
          run = 0;
        }
        ++run;
      }
      if (at >= 0) atomicAdd(h + at, run);
    }
  }
  __syncthreads();
  for (int s = 0; s < ns; ++s)
    for (int c = threadIdx.x; c < N; c += kStepBlock)
      if (H[s * M + c]) atomicAdd(sh.b.hist + sh.seg[s].hoff + c, H[s * M + c]);
}

// The share's particles to their cells' places in the other buffer set: a cell
// starts at the prefix of the histogram, a block reserves its part of it with
// one atomic.  fresh[s]: the species' particles after the sort.
template <int kStepBlock>
__device__ __noinline__ void sort_scatter(unsigned me, unsigned team, long long* fresh) {
  StepShared& sh = step_shared();
  const int ns = sh.run.ns, N = sh.run.N, M = N + 1, tid = threadIdx.x;
  int* H = reinterpret_cast<int*>(step_arrays().mom);
  const int per = (N + kStepBlock - 1) / kStepBlock;
  const int cb = min(N, tid * per), ce = min(N, cb + per);
  for (int s = 0; s < ns; ++s) {
    const int* hist = sh.b.hist + sh.seg[s].hoff;
    int* taken = sh.b.rbcnt + sh.seg[s].hoff;
    int loc = 0, total;
    for (int c = cb; c < ce; ++c) loc += hist[c];
    int at = block_excl_scan(loc, reinterpret_cast<int*>(sh.wsm), &total);
    if (tid == 0) fresh[s] = total;
    for (int c = cb; c < ce; ++c) {
      const int mine = H[s * M + c], all = hist[c];
      if (mine) H[s * M + c] = at + atomicAdd(taken + c, mine);
      at += all;
    }
  }
  __syncthreads();
  for (int s = 0; s < ns; ++s) {
    unsigned beg, end;
    if (!step_share(sh, s, me, team, &beg, &end)) continue;
    const SegDev& G = sh.seg[s];
    const int a = sh.fx.cur[s], o = a ^ 1;
    const long long n = sh.fx.n[s];
    int* h = H + s * M;
    for (unsigned q = beg + tid; q < end; q += kStepBlock) {
      int c[4], d[4];
      float x[4], u[4], v[4], w[4];
      uint64_t id[4];
      unsigned kw[4] = {1u, 1u, 1u, 1u};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long i = 4ll * q + j;
        c[j] = i < n ? G.cell[a][i] : -1;
        const bool in = c[j] >= 0;
        x[j] = in ? G.xi[a][i] : 0.0f;
        u[j] = in ? G.vx[a][i] : 0.0f;
        v[j] = in ? G.vy[a][i] : 0.0f;
        w[j] = in ? G.vz[a][i] : 0.0f;
        id[j] = in ? G.id[a][i] : 0ull;
        if (in && G.wt[a]) kw[j] = G.wt[a][i];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // a run of equal cells takes its places with one atomic
        const bool head = j == 0 || c[j] != c[j - 1];
        int run = 1;
        if (head)
          for (int l = j + 1; l < 4; ++l) {
            if (c[l] != c[j]) break;
            ++run;
          }
        d[j] = c[j] < 0 ? -1 : head ? atomicAdd(h + c[j], run) : d[j - 1] + 1;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (d[j] < 0 || !chk(d[j] < G.cap, 35, d[j], G.cap)) continue;
        G.cell[o][d[j]] = c[j];
        G.xi[o][d[j]] = x[j];
        G.vx[o][d[j]] = u[j];
        G.vy[o][d[j]] = v[j];
        G.vz[o][d[j]] = w[j];
        G.id[o][d[j]] = id[j];
        if (G.wt[o]) G.wt[o][d[j]] = kw[j];
      }
    }
  }
}

// The charge prefix C_n (in units of sh.cs) into sh.C for species of one
// weight up to sign: one signed integer sum per node.  A thread owns up to
// kNodes consecutive nodes and reads their deposits itself (the reads of a
// warp's lanes share their lines).
template <int kStepBlock>
__device__ __forceinline__ void prefix_signed(const unsigned long long* S) {
  StepShared& sh = step_shared();
  const StepArrays ar = step_arrays();
  constexpr int kNodes = (kMaxCells + 1 + kStepBlock - 1) / kStepBlock;
  const RunDev* R = &sh.run;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int N = R->N, M = N + 1, ns = R->ns, neg = R->field_neg;
  const int per = (M + kStepBlock - 1) / kStepBlock;
  const int beg = tid * per;
  unsigned long long q[kNodes];
#pragma unroll
  for (int u = 0; u < kNodes; ++u) {
    q[u] = 0ull;
    const int n = beg + u;
    if (u < per && n < M) {
      const unsigned long long a = S[n];
      q[u] = (neg & 1) ? 0ull - a : a;
      if (ns > 1) {
        const unsigned long long c = S[M + n];
        q[u] += (neg & 2) ? 0ull - c : c;
      }
    }
  }
  if (ns > 2)
    for (int s = 2; s < ns; ++s)
#pragma unroll
      for (int u = 0; u < kNodes; ++u) {
        const int n = beg + u;
        if (u < per && n < M) {
          const unsigned long long a = S[(size_t)s * M + n];
          q[u] += ((neg >> s) & 1) ? 0ull - a : a;
        }
      }
  const unsigned long long q0 = q[0];  // (thread 0: node 0, which only enters the total)
  if (tid == 0) q[0] = 0ull;
#pragma unroll
  for (int u = 1; u < kNodes; ++u) q[u] += q[u - 1];
  const unsigned long long loc = q[kNodes - 1];
  const unsigned long long inc = warp_incl_scan(loc);
  if (lane == 31) sh.wtot[0][w] = inc;
  if (tid == 0) {
    sh.wtot[1][0] = q0;
    sh.cs = R->sp[0].cw;
  }
  __syncthreads();
  const unsigned long long t = warp_incl_scan(lane < kStepBlock / 32 ? sh.wtot[0][lane] : 0ull);
  const unsigned long long before = __shfl_sync(kFull, t, w == 0 ? 0 : w - 1);
  const unsigned long long off = (w == 0 ? 0ull : before) + inc - loc;
  double a = 0.0;
  const bool periodic = R->bc == ECPIC_PERIODIC;
  if (periodic) a = i64_to_f64((long long)(__shfl_sync(kFull, t, 31) + sh.wtot[1][0])) * R->inv_L;
#pragma unroll
  for (int u = 0; u < kNodes; ++u) {
    const int n = beg + u;
    if (u < per && n < N) {
      double c = i64_to_f64((long long)(off + q[u]));
      if (periodic) c -= a * ar.V[n];
      ar.C[n] = c;
    }
  }
}

// The same for species of any weights, or where only the totals tell that the
// signed sum is exact (field_solve's decision).
template <int kStepBlock>
__device__ __noinline__ void prefix_species(const unsigned long long* S) {
  StepShared& sh = step_shared();
  const StepArrays ar = step_arrays();
  const RunDev* R = &sh.run;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int N = R->N, M = N + 1, ns = R->ns, neg = R->field_neg;
  for (int n = tid; n < M; n += kStepBlock)
    for (int s = 0; s < ns; ++s) ar.Q[(size_t)s * M + n] = S[(size_t)s * M + n];
  __syncthreads();
  const int per = (M + kStepBlock - 1) / kStepBlock;
  const int beg = min(M, tid * per), end = min(M, beg + per);
  unsigned long long run[kMaxSpecies], tot[kMaxSpecies];
#pragma unroll
  for (int s = 0; s < kMaxSpecies; ++s) {
    run[s] = 0ull;
    if (s < ns) {
      unsigned long long loc = 0ull;
      for (int n = max(beg, 1); n < end; ++n) loc += ar.Q[(size_t)s * M + n];
      const unsigned long long inc = warp_incl_scan(loc);
      if (lane == 31) sh.wtot[s][w] = inc;
      run[s] = inc - loc;
    }
  }
  __syncthreads();
  bool one = R->field_pm != 0;
  unsigned long long sum = 0ull;
#pragma unroll
  for (int s = 0; s < kMaxSpecies; ++s) {
    tot[s] = 0ull;
    if (s < ns) {
      const unsigned long long v = warp_incl_scan(lane < kStepBlock / 32 ? sh.wtot[s][lane] : 0ull);
      const unsigned long long off = __shfl_sync(kFull, v, w == 0 ? 0 : w - 1);
      tot[s] = __shfl_sync(kFull, v, 31) + ar.Q[(size_t)s * M];  // node 0 only enters the total
      run[s] += w == 0 ? 0ull : off;
      one = one && tot[s] < (1ull << 62);
      sum += tot[s] >> 2;
    }
  }
  one = one && sum < (1ull << 61) - 4ull;
  if (tid == 0) sh.cs = one ? R->sp[0].cw : 1.0;
  double a = 0.0;
  const bool periodic = R->bc == ECPIC_PERIODIC;
  if (periodic) {
    double qtot = 0.0;
    unsigned long long qi = 0ull;
#pragma unroll
    for (int s = 0; s < kMaxSpecies; ++s)
      if (s < ns) {
        if (one) qi += ((neg >> s) & 1) ? 0ull - tot[s] : tot[s];
        else qtot += R->sp[s].cw * (double)tot[s];
      }
    if (one) qtot = i64_to_f64((long long)qi);
    a = qtot * R->inv_L;
  }
  for (int n = beg; n < min(end, N); ++n) {
    double c = 0.0;
    unsigned long long qi = 0ull;
#pragma unroll
    for (int s = 0; s < kMaxSpecies; ++s)
      if (s < ns) {
        if (n > 0) run[s] += ar.Q[(size_t)s * M + n];
        if (one) qi += ((neg >> s) & 1) ? 0ull - run[s] : run[s];
        else c += R->sp[s].cw * (double)run[s];
      }
    if (one) c = i64_to_f64((long long)qi);
    if (periodic) c -= a * ar.V[n];
    ar.C[n] = c;
  }
}

// What the first block of a team keeps of a level for the run: the sampled
// potential and the energies.  C holds g.
template <int kStepBlock>
__device__ __noinline__ void keep_level(RunState* st, long long kn, double phi0, bool sample, bool want_fe) {
  StepShared& sh = step_shared();
  const StepArrays ar = step_arrays();
  const RunDev* R = &sh.run;
  __syncthreads();
  double fe_tot = 0.0;
  if (want_fe) {
    double fe = 0.0;
    for (int n = threadIdx.x; n < R->N; n += kStepBlock) fe += ar.C[n] * ar.C[n] * ar.D[n];
    __syncthreads();
    fe_tot = 0.5 * kEps0 * block_sum(fe, sh.wsm);
  }
  if (sample) {
    __syncthreads();
    form_potential<kStepBlock>(R, ar.C, ar.D, phi0, true, sh.wsm);
  }
  if (threadIdx.x == 0) {
    if (sample) {
      st->phi_level = kn;
      close_sample(st, R->ns);
    }
    if (want_fe) st->fe_field = fe_tot;
  }
}

// Field of a level from its deposit S, into sh.E (field_solve says how; the
// sums are formed in the same order).  The first block of the team also
// writes it for the run.
template <int kStepBlock>
__device__ __noinline__ void step_field(const unsigned long long* S, double phi0, bool first) {
  StepShared& sh = step_shared();
  const StepArrays ar = step_arrays();
  const RunDev* R = &sh.run;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int N = R->N, M = N + 1, ns = R->ns;
  const bool face = R->scheme == ECPIC_SCHEME_EC || R->scheme == ECPIC_SCHEME_EC2;
  double *C = ar.C, *D = ar.D;
  // the signed sum stays exact: room for fewer than 2^29 particles (times the
  // largest multiplier) per species, else the totals decide
  bool pm = R->field_pm != 0;
  for (int s = 0; s < ns; ++s) pm = pm && sh.cap[s] < ((1ll << 29) >> (R->rb ? 16 : 0));
  if (pm) prefix_signed<kStepBlock>(S);
  else prefix_species<kStepBlock>(S);
  __syncthreads();
  if (tid < kFieldOwners) {
    const int po = (M + kFieldOwners - 1) / kFieldOwners;
    const int ob = min(M, tid * po), oe = min(N, ob + po);
    double loc = 0.0;
    for (int n = ob; n < oe; ++n) loc += D[n] * C[n];
    sh.owner[tid + (tid >> 3)] = loc;
  }
  __syncthreads();
  // the balanced tree over the owners' sums, and g_0: one warp, eight owners
  // a lane first
  if (w == 0) {
    const double* v = sh.owner + 9 * lane;
    double A = add64(add64(add64(v[7], v[6]), add64(v[5], v[4])), add64(add64(v[3], v[2]), add64(v[1], v[0])));
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) A = add64(A, __shfl_xor_sync(kFull, A, o));
    const double cs = sh.cs;
    A = cs * A;
    const double g0 = (A * kInvEps0 - phi0) * R->inv_L;
    if (lane == 0) {
      sh.g0 = g0;
      sh.kc = cs * kInvEps0;
    }
  }
  __syncthreads();
  const double g0 = sh.g0, kc = sh.kc;
  double* gst = R->g;
  float *E = ar.E, *Eg = R->E;
  for (int n = tid; n < N; n += kStepBlock) {
    const double gn = g0 - C[n] * kc;
    if (face) {
      const float e = f64_to_f32(-gn);
      E[n] = e;
      if (first) Eg[n] = e;
    }
    if (!face || first) C[n] = gn;
    if (first) gst[n] = gn;
  }
  if (!face) {
    __syncthreads();
    const bool periodic = R->bc == ECPIC_PERIODIC;
    const double* W = ar.W;
    for (int n = tid; n <= N; n += kStepBlock) {
      double e;
      if (n > 0 && n < N) {
        e = -(C[n] * W[n] + C[n - 1] * (1.0 - W[n]));
      } else if (periodic) {
        e = -(C[0] * W[0] + C[N - 1] * (1.0 - W[0]));
      } else {
        e = (n == 0) ? -C[0] : -C[N - 1];
      }
      const float ef = f64_to_f32(e);
      E[n] = ef;
      if (first) Eg[n] = ef;
    }
  }
}

template <bool WEIGHTED, int kStepBlock, int V>
__global__ void __launch_bounds__(kStepBlock, 1)
    k_steps(BatchView gb, StepPlan pl, __grid_constant__ const StepTeams tm, int steps, int sort_every,
            int since_sort) {
  StepShared& sh = step_shared();
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int slot = tm.slot[blockIdx.x];
  const unsigned me = tm.index[blockIdx.x], team = tm.size[blockIdx.x];
  const int spc = gb.nseg / gb.max_slots;
  const size_t Mx = (size_t)gb.nmax + 1;
  StepWords* words = pl.words + slot;
  RunState* st = gb.rst + slot;
  {
    if (tid == 0) {
      sh.b = gb;
      sh.spc = spc;
    }
    const uint32_t* src = reinterpret_cast<const uint32_t*>(gb.runs + slot);
    for (int i = tid; i < (int)(sizeof(RunDev) / 4); i += kStepBlock) reinterpret_cast<uint32_t*>(&sh.run)[i] = src[i];
    const uint32_t* sg = reinterpret_cast<const uint32_t*>(gb.segs + (size_t)slot * spc);
    for (int i = tid; i < (int)(sizeof(SegDev) / 4) * spc; i += kStepBlock)
      reinterpret_cast<uint32_t*>(&sh.seg[0])[i] = sg[i];
    for (int i = tid; i < kMaxSpecies * kNumCtr; i += kStepBlock) (&sh.fx.ctr[0][0])[i] = 0u;
  }
  if (tid < spc) {
    const SegState& q = gb.sst[(size_t)slot * spc + tid];
    sh.fx.n[tid] = q.n_proc;
    sh.fx.cur[tid] = q.cur;
  }
  long long k = st->step;
  const long long step_end = st->step_end;
  const int status = st->status;
  __syncthreads();
  const RunDev* R = &sh.run;
  if (!R->active || status != 0 || k >= step_end) return;  // (the whole team)
  const int N = R->N, ns = R->ns, M = N + 1, se = R->sample_every, seg0 = R->seg0;
  SegState* sst = gb.sst + seg0;
  {
    const bool periodic = R->bc == ECPIC_PERIODIC;
    const bool face = R->scheme == ECPIC_SCHEME_EC || R->scheme == ECPIC_SCHEME_EC2;
    if (tid == 0) {
      sh.b.runs = &sh.run - slot;  // indexed by slot and segment like the tables
      sh.b.segs = &sh.seg[0] - seg0;
      sh.fx.S = R->S;
      sh.fx.births = words->births[0];
      sh.fx.imp = words->imp[0];
      sh.fx.fail = &words->fail[0];
      sh.fx.nlive = 0u;
      sh.pass.top[0] = sh.pass.top[1] = 0u;
      sh.pass.lowest = INT_MAX;
      split_team(sh, ns, team);
    }
    const StepArrays ar = step_arrays();
    const int zeros = (int)(ar.ring - reinterpret_cast<unsigned char*>(ar.dep)) / 4;
    for (int i = tid; i < zeros; i += kStepBlock) ar.dep[i] = 0u;
    for (int n = tid; n < M; n += kStepBlock) {
      ar.D[n] = n < N ? R->dx[n] : 0.0;
      ar.V[n] = periodic ? R->cumV[n] : 0.0;
      ar.W[n] = face ? 0.0 : R->mcw[n];
      ar.E[n] = n < N || !face ? R->E[n] : 0.0f;
    }
    if (tid < ns) sh.cap[tid] = sh.seg[tid].cap;
  }
  // three deposits in turn: one is added to, one is being read, one cleared
  unsigned long long* const S1 = pl.deposit + (size_t)slot * 2 * spc * Mx;
  unsigned long long* const S2 = S1 + (size_t)spc * Mx;
  unsigned arrivals = 0;
  // steps to the next sample (the push of level k samples when (k + 1) % se
  // == 0), 0 without samples
  int to_sample = se > 0 ? se - (int)(k % se) : 0;
  int rot = 0;
  __syncthreads();

  for (int t = 0;; ++t) {
    const bool sample = to_sample == 1;
    // (a sine takes as long for one lane as for a warp)
    if ((t & 31) == 0 && w == kStepBlock / 32 - 1) sh.phi0[lane] = electrode(R, k + 1 + lane);
    step_particles<WEIGHTED, kStepBlock, V>(me, team, k, sample);
    const long long kn = k + 1;
    const bool last = t + 1 == steps || kn >= step_end;
    __syncthreads();
    if (tid == 0) arrive(&words->arrive);
    arrivals += team;
    const bool sort = since_sort + 1 == sort_every;
    // the first block of the team closes the launch (the others help with its
    // sample and its sort)
    if (last && me != 0 && !sample && !sort) break;
    const double phi0 = sh.phi0[t & 31];
    if (!await(&words->arrive, arrivals, sh)) {
      if (tid == 0) set_status(st, ECPIC_ERR_TIMEOUT);
      break;
    }

    // ---- field of level kn, solved by every block of the team for itself
    const int rot1 = rot == 2 ? 0 : rot + 1, rot2 = rot == 0 ? 2 : rot - 1;
    unsigned long long* S = rot == 0 ? R->S : rot == 1 ? S1 : S2;
    // the deposit of two steps ahead: nobody reads it now, nobody adds to it
    // before the next barrier
    unsigned long long* Sz = rot2 == 0 ? R->S : rot2 == 1 ? S1 : S2;
    for (int i = tid + kStepBlock * (int)me; i < ns * M; i += kStepBlock * (int)team) Sz[i] = 0ull;
    if (tid >= 32 && tid < 32 + ns) {
      // the step's births are kept up to the capacity
      const int s = tid - 32;
      const long long n = sh.fx.n[s] + (long long)words->births[rot][s];
      if (me == 0) sst[s].n_alloc = n;
      sh.fx.n[s] = min(n, sh.cap[s]);
    } else if (tid == 64) {
      sh.fail = words->fail[rot];
      sh.fx.S = rot1 == 0 ? R->S : rot1 == 1 ? S1 : S2;
      sh.fx.births = words->births[rot1];
      sh.fx.imp = words->imp[rot1];
      sh.fx.fail = &words->fail[rot1];
      if (me == 0) words->fail[rot2] = 0;
    } else if (me == 0 && tid >= 96 && tid < 96 + kMaxSpecies) {
      words->births[rot2][tid - 96] = 0ull;
      words->imp[rot2][tid - 96] = 0ull;
    }
    __syncthreads();
    if (sh.fail) {  // the run stops at level k
      if (me == 0) {
        if (tid == 0) set_status(st, sh.fail);
        for (int i = tid; i < ns * M; i += kStepBlock) R->S[i] = S1[i] = S2[i] = 0ull;
      }
      break;
    }
    if (me == 0 || !last) step_field<kStepBlock>(S, phi0, me == 0);
    // (the moments: a share of the nodes each)
    if (sample) sample_moments<kStepBlock>(R, S, (int)me, (int)team);
    if (me == 0) {
      // the team's first block keeps the run's state; the energy of level kn
      // is sampled by its push
      const bool want_fe = se > 0 && (sample ? se : to_sample - 1) == 1;
      if (sample || want_fe) keep_level<kStepBlock>(st, kn, phi0, sample, want_fe);
      if (tid == 0) {
        st->phi0 = phi0;
        st->step = kn;
      }
      if (tid < ns) sst[tid].n_proc = sst[tid].n_alloc = sh.fx.n[tid];
    }
    __syncthreads();
    since_sort = sort ? 0 : since_sort + 1;
    if (sort) {
      flush_counters<kStepBlock>(sh, st, sst, ns);  // (the sort ends the count of absorbed slots)
      __syncthreads();
      sort_count<kStepBlock>(me, team);
      __syncthreads();
      if (tid == 0) arrive(&words->arrive);
      arrivals += team;
      bool ok = await(&words->arrive, arrivals, sh);
      // the absorbed slots end here: every block has added its own, and adds
      // the next ones after the next barrier
      if (ok && me == 0 && tid < ns) sst[tid].n_dead = 0;
      if (ok) {
        sort_scatter<kStepBlock>(me, team, sh.fresh);
        __syncthreads();
        if (tid == 0) arrive(&words->arrive);
        arrivals += team;
        ok = await(&words->arrive, arrivals, sh);
      }
      if (!ok) {
        if (tid == 0) set_status(st, ECPIC_ERR_TIMEOUT);
        break;
      }
      // the run's cell arrays end at zero
      for (int s = 0; s < ns; ++s)
        for (int c = tid + kStepBlock * (int)me; c < N; c += kStepBlock * (int)team)
          gb.hist[sh.seg[s].hoff + c] = gb.rbcnt[sh.seg[s].hoff + c] = 0;
      if (tid < ns) {
        sh.fx.cur[tid] ^= 1;
        sh.fx.n[tid] = sh.fresh[tid];
        if (me == 0) {
          sst[tid].cur = sh.fx.cur[tid];
          sst[tid].n_proc = sst[tid].n_alloc = sst[tid].n_live = sh.fresh[tid];
        }
      }
      __syncthreads();
    }
    if (last) {
      // every deposit ends at zero, this step's once all have read it
      if (sample && !sort) {
        if (me != 0) {
          if (tid == 0) arrive(&words->arrive);
          break;
        }
        if (!await(&words->arrive, arrivals + team - 1, sh)) {
          if (tid == 0) set_status(st, ECPIC_ERR_TIMEOUT);
          break;
        }
      }
      if (me == 0)
        for (int i = tid; i < ns * M; i += kStepBlock) S[i] = Sz[i] = 0ull;
      break;
    }
    if (sample && se == 1) {
      // the next step samples again: nobody adds to its sums before these are
      // closed (otherwise the next step's barrier comes between)
      if (tid == 0) arrive(&words->arrive);
      arrivals += team;
      if (!await(&words->arrive, arrivals, sh)) {
        if (tid == 0) set_status(st, ECPIC_ERR_TIMEOUT);
        break;
      }
    }
    if ((t & 31) == 31) {  // (32-bit sums)
      flush_counters<kStepBlock>(sh, st, sst, ns);
      __syncthreads();
    }
    k = kn;
    if (se > 0) to_sample = sample ? se : to_sample - 1;
    rot = rot1;
  }
  __syncthreads();
  flush_counters<kStepBlock>(sh, st, sst, ns);
}

constexpr size_t kStepSmem = 226 * 1024;  // dynamic shared memory of a block, at most
size_t steps_smem(const BatchView& b, int threads) {
  return steps_bytes(b.nmax, b.nseg / b.max_slots, b.weighted != 0, threads);
}

template <bool W, int kStepBlock, int V>
cudaError_t launch_w(const BatchView& b, const StepPlan& pl, const StepTeams& tm, int steps, int sort_every,
                     int since_sort, cudaStream_t s) {
  const size_t sm = steps_smem(b, kStepBlock);
  // the same limit on every call: threads with runs of other sizes set it too
  cudaError_t e = cudaFuncSetAttribute(k_steps<W, kStepBlock, V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kStepSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tm.blocks);
  cfg.blockDim = dim3(kStepBlock);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_steps<W, kStepBlock, V>, b, pl, tm, steps, sort_every, since_sort);
}

// The instance for the teams' block size and particles per thread.
template <bool W>
cudaError_t launch_any(const BatchView& b, const StepPlan& pl, const StepTeams& tm, int steps, int sort_every,
                       int since_sort, cudaStream_t s) {
  if (tm.threads == 512) return launch_w<W, 512, 4>(b, pl, tm, steps, sort_every, since_sort, s);
  if (tm.group == 1) return launch_w<W, 256, 1>(b, pl, tm, steps, sort_every, since_sort, s);
  if (tm.group == 2) return launch_w<W, 256, 2>(b, pl, tm, steps, sort_every, since_sort, s);
  return launch_w<W, 256, 4>(b, pl, tm, steps, sort_every, since_sort, s);
}

}  // namespace
}  // namespace ecpic
