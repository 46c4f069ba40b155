// step_dev.cuh -- device code of one time step of one (run, species) segment
// or one run, shared by the kernels that launch a phase at a time (kernels.cu)
// and the one that advances several steps per launch (steps.cu): segment
// prefix sums, fixed-point deposits, the particle pass, real collisions and
// the field solve.
#pragma once
#include <cfloat>
#include <climits>

#include "deposit.cuh"
#include "kernels.h"

namespace ecpic {
namespace {

// Checked builds (-DECPIC_CHECKS): indexed accesses are validated against
// their bounds; the first violation (site, index, bound) and a violation count
// are recorded per translation unit and the access is skipped.  Plain builds
// compile the checks away.
__device__ unsigned long long g_check[4];

#ifdef ECPIC_CHECKS
__device__ __noinline__ bool chk(bool ok, int where, long long idx, long long bound) {
  if (!ok) {
    if (atomicCAS(&g_check[0], 0ull, (unsigned long long)where) == 0ull) {
      g_check[1] = (unsigned long long)idx;
      g_check[2] = (unsigned long long)bound;
    }
    atomicAdd(&g_check[3], 1ull);
  }
  return ok;
}
#else
__device__ __forceinline__ bool chk(bool, int, long long, long long) { return true; }
#endif

constexpr double kEps0 = 8.8541878128e-12;
constexpr double kTwoPi = 6.283185307179586476925286766559;

// ----------------------------------------------------------------- reductions
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// exclusive scan over the block (blockDim a multiple of 32); wsm >= 32 entries
template <typename T>
__device__ T block_excl_scan(T v, T* wsm, T* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const T inc = warp_incl_scan(v);
  if (lane == 31) wsm[w] = inc;
  __syncthreads();
  if (w == 0) {
    T t = lane < nw ? wsm[lane] : T(0);
    t = warp_incl_scan(t);
    if (lane < nw) wsm[lane] = t;
  }
  __syncthreads();
  const T off = w > 0 ? wsm[w - 1] : T(0);
  *total = wsm[nw - 1];
  __syncthreads();
  return off + inc - v;
}

template <typename T>
__device__ T block_sum(T v, T* wsm) {
  T total;
  block_excl_scan(v, wsm, &total);
  return total;
}

// in-place inclusive scan of a[0..n) held in shared memory (fixed partition,
// so the FP64 rounding is deterministic)
template <typename T>
__device__ void block_incl_scan_array(T* a, int n, T* wsm) {
  const int per = (n + blockDim.x - 1) / blockDim.x;
  const int beg = min(n, (int)threadIdx.x * per), end = min(n, beg + per);
  T loc = T(0);
  for (int i = beg; i < end; ++i) loc += a[i];
  T total;
  T run = block_excl_scan(loc, wsm, &total);
  for (int i = beg; i < end; ++i) {
    run += a[i];
    a[i] = run;
  }
  __syncthreads();
}

// ----------------------------------------------------------------- segments
__device__ __forceinline__ bool run_live(const RunDev& R, const RunState& S, int mode, int only,
                                         int slot) {
  if (!R.active) return false;
  if (mode == MODE_REFRESH) return only == kOnlyFresh ? S.fresh != 0 : slot == only;
  if (S.status != 0) return false;
  if (mode == MODE_STEP) return S.step < S.step_end;
  if (mode == MODE_REBAL)  // a rebalancing run at a rebalancing level (once per level)
    return R.rb && (S.rb_force || (R.rb_every > 0 && S.step > 0 && S.step % R.rb_every == 0 &&
                                   S.rb_level != S.step));
  return true;
}

// exclusive prefix of the work of all segments (particles, groups of `unit`
// particles, or recorded real collisions): pre[0..nseg]
// (with meta: per segment its run slot, buffer index and real-collision
// count, meta[3 s .. 3 s + 2], so that the records' consumers need no
// dependent global loads for them)
__device__ long long seg_prefix(const BatchView& b, int mode, int only, long long* pre,
                                long long* wsm, int unit = 1, bool reals = false,
                                int* meta = nullptr) {
  const int per = (b.nseg + blockDim.x - 1) / blockDim.x;
  const int s0 = threadIdx.x * per;
  long long loc = 0;
  for (int k = 0; k < per; ++k) {
    const int s = s0 + k;
    if (s < b.nseg) {
      const int slot = b.segs[s].run;
      const bool live = run_live(b.runs[slot], b.rst[slot], mode, only, slot);
      // records past a list's capacity were never written (the pass failed
      // the run with ECPIC_ERR_CAPACITY): only the stored ones count
      const long long nr = reals ? min(b.sst[s].n_real, b.segs[s].real_cap) : 0;
      const long long c = !live ? 0
                          : reals ? nr + min(b.sst[s].n_imp, b.segs[s].imp_cap)
                                  : (b.sst[s].n_proc + unit - 1) / unit;
      pre[s] = c;
      loc += c;
      if (meta) {
        meta[3 * s] = slot;
        meta[3 * s + 1] = b.sst[s].cur;
        meta[3 * s + 2] = live ? (int)nr : 0;
      }
    }
  }
  long long total;
  long long run = block_excl_scan(loc, wsm, &total);
  for (int k = 0; k < per; ++k) {
    const int s = s0 + k;
    if (s < b.nseg) {
      const long long c = pre[s];
      pre[s] = run;
      run += c;
    }
  }
  if (threadIdx.x == 0) pre[b.nseg] = total;
  __syncthreads();
  return total;
}

// first segment s with pre[s] <= v < pre[s+1]
__device__ __forceinline__ int seg_find(const long long* pre, int nseg, long long v) {
  int lo = 0, hi = nseg;  // pre[lo] <= v, answer in [lo, hi)
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pre[mid] <= v) lo = mid; else hi = mid;
  }
  return lo;
}

// ----------------------------------------------------------------- deposit
// ---- weighted CIC deposit (rebalancing runs) -----------------------------
// A particle of weight multiplier k adds k (2^32 - r) to node c and k r to
// node c+1.  Shared 64-bit atomics are compare-and-swap loops on this part
// and the lanes of a warp share a few cells on sorted data, so the sums stay
// in native 32-bit atomics: with r = rh 2^16 + rl, k rl = a1 2^16 + a0 and
// k rh = b1 2^16 + b0 (k <= 2^16, so every piece is below 2^16), each cell
// keeps K = sum k, A = sum a0, M = sum (a1 + b0), B = sum b1, and
// R = sum k r = 2^32 B + 2^16 M + A.  Flushed at least every
// kFlushParticles / 2 = 2^15 particles, K stays <= 2^31 and M < 2^32.
// Four arrays keep the pass at four CTAs per SM on 1024-cell batches.
struct DepW {
  uint32_t *k, *a, *m, *b;  // (nmax + 1) each
};

template <int V = 4>
__device__ __forceinline__ void depw_add4(const DepW& d, const int c[V], const float f[V],
                                          const unsigned kq[V]) {
  unsigned K[V], A[V], M[V], B[V];
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const bool v = c[j] >= 0;
    const unsigned r = v ? __float2uint_rz(f[j] * 4294967296.0f) : 0u;
    const unsigned k = v ? kq[j] : 0u;
    const unsigned p = k * (r & 0xFFFFu), q = k * (r >> 16);
    K[j] = k;
    A[j] = p & 0xFFFFu;
    M[j] = (p >> 16) + (q & 0xFFFFu);
    B[j] = q >> 16;
  }
#pragma unroll
  for (int j = V - 1; j >= 1; --j) {
    if (c[j] >= 0 && c[j] == c[j - 1]) {
      K[j - 1] += K[j];
      A[j - 1] += A[j];
      M[j - 1] += M[j];
      B[j - 1] += B[j];
      K[j] = 0u;
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) {
    if (K[j]) {
      atomicAdd(d.k + c[j], K[j]);
      atomicAdd(d.a + c[j], A[j]);
      atomicAdd(d.m + c[j], M[j]);
      atomicAdd(d.b + c[j], B[j]);
    }
  }
}

// Adds the sums of cells [a, e) to the node array S (cell c to nodes c and
// c+1) and clears them; every thread of the block calls it, between barriers.
__device__ void depw_flush(const DepW& d, int a, int e, unsigned long long* S) {
  for (int c = a + (int)threadIdx.x; c < e; c += (int)blockDim.x) {
    const uint32_t K = d.k[c];
    if (K) {
      const unsigned long long R = ((unsigned long long)d.b[c] << 32) +
                                   ((unsigned long long)d.m[c] << 16) + d.a[c];
      atomicAdd(S + c, ((unsigned long long)K << 32) - R);
      if (R) atomicAdd(S + c + 1, R);
      d.k[c] = 0u;
      d.a[c] = 0u;
      d.m[c] = 0u;
      d.b[c] = 0u;
    }
  }
}

__device__ __forceinline__ void deposit2_one(unsigned long long* S, int c, float f, int N, bool periodic) {
  int n0;
  unsigned a, b;
  spline2_shares(f, c, &n0, &a, &b);
  atomicAdd(S + node2(n0 - 1, N, periodic), (unsigned long long)a);
  atomicAdd(S + n0, 4294967296ull - a - b);
  atomicAdd(S + node2(n0 + 1, N, periodic), (unsigned long long)b);
}

__device__ __forceinline__ void deposit_one(unsigned long long* S, int c, float f, unsigned k = 1u) {
  const unsigned r = __float2uint_rz(f * 4294967296.0f);
  atomicAdd(S + c, (unsigned long long)k * (4294967296ull - (unsigned long long)r));
  atomicAdd(S + c + 1, (unsigned long long)k * (unsigned long long)r);
}

// ----------------------------------------------------------------- MCC helpers
// Collision frequencies nu_p = n_g sigma_p(E) |g| of a species' processes, in
// process order, from its node-interleaved table: linear interpolation
// between nodes dE apart, the last node's value past the table, zero below a
// process threshold.  Returns the first p whose running sum exceeds Rr (the
// selection of Sec. 2a step 6; -1 for a null collision) and the total in *tot.
__device__ __forceinline__ int select_process(const SpeciesDev* SP, float E, float gm, float ng,
                                              float Rr, float* tot) {
  const int n = SP->ntab, np4 = SP->np4;
  const float u = E * SP->dE_inv;
  const float fi = floorf(u);
  const bool top = fi >= (float)(n - 1);
  int i = top ? n - 1 : (int)fi;
  if (!chk(i >= 0 && i < n, 17, i, n)) i = 0;
  const int i1 = top ? i : i + 1;
  const float t = top ? 0.0f : u - fi;
  const float4* tab = SP->sig4;
  float cum = 0.0f;
  int chosen = -1;
  for (int g = 0; g < np4; ++g) {
    const float4 a = __ldg(tab + (size_t)i * np4 + g);
    const float4 b = __ldg(tab + (size_t)i1 * np4 + g);
    const float sg[4] = {a.x + t * (b.x - a.x), a.y + t * (b.y - a.y), a.z + t * (b.z - a.z),
                         a.w + t * (b.w - a.w)};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p = 4 * g + q;
      const float sig = E < SP->thr_all[p] ? 0.0f : sg[q];
      cum += ng * sig * gm;
      if (chosen < 0 && Rr < cum) chosen = p;
    }
  }
  *tot = cum;
  return chosen;
}

__device__ __forceinline__ void box_muller(float u1, float u2, float& z0, float& z1) {
  const float rad = sqrtf(-2.0f * logf(u1));
  float s, c;
  sincospif(2.0f * u2, &s, &c);
  z0 = rad * c;
  z1 = rad * s;
}

// unit vector uniform on the sphere, polar axis along x
__device__ __forceinline__ void isotropic(float ua, float ub, float& d0, float& d1, float& d2) {
  const float c = 1.0f - 2.0f * ua;
  const float s = sqrtf(fmaxf(0.0f, 1.0f - c * c));
  float sp, cp;
  sincospif(2.0f * ub, &sp, &cp);
  d0 = c;
  d1 = s * cp;
  d2 = s * sp;
}

__device__ __forceinline__ void set_status(RunState* st, int code) {
  atomicCAS(&st->status, 0, code);
}

// write a birth at index idx of a segment; false if the capacity is full
__device__ __forceinline__ bool put_particle(const SegDev& G, long long idx, int cur, int c, float f, float vx,
                                             float vy, float vz, uint64_t id, unsigned k) {
  if (idx >= G.cap) return false;
  G.cell[cur][idx] = c;
  G.xi[cur][idx] = f;
  G.vx[cur][idx] = vx;
  G.vy[cur][idx] = vy;
  G.vz[cur][idx] = vz;
  G.id[cur][idx] = id;
  if (G.wt[cur]) G.wt[cur][idx] = k;
  return true;
}

// cell walk on a non-uniform grid: g = xi + vx dt/dx_c, carried into the
// neighbours with their width ratios; FP32 rounding to 1.0f puts the particle
// on the next face (xi = 0)
__device__ __forceinline__ void walk_nonuniform(int& c, float& f, float g, int N, int bc,
                                                const float* rp, const float* rm) {
  int guard = 0;
  while (g >= 1.0f) {
    if (c == N - 1 && bc != ECPIC_PERIODIC) { c = N; g = 0.0f; break; }
    g = (g - 1.0f) * __ldg(rp + c);
    c = (c == N - 1) ? 0 : c + 1;
    if (++guard > N) { g = 0.0f; break; }
  }
  while (g < 0.0f) {
    if (c == 0 && bc != ECPIC_PERIODIC) { c = -1; g = 0.0f; break; }
    g = 1.0f + g * __ldg(rm + c);
    c = (c == 0) ? N - 1 : c - 1;
    if (g >= 1.0f) {
      c = (c == N - 1) ? 0 : c + 1;
      g = 0.0f;
    }
    if (++guard > N) { g = 0.0f; break; }
  }
  f = g;
}

constexpr int kFarCell = -(1 << 30);
constexpr int kRing = 160;  // candidates (indices) per warp: >= 31 left over + 4 * 32 added

struct PassShared {
  uint32_t ctr[kNumCtr];  // this piece's counters (a piece has < 2^31 particles)
  uint32_t nlive;
  long long wsm[32];
  double dsm[32];
  unsigned top[2];  // k_steps: bounds of a sample's terms (zero between pieces)
  int lowest;       // and the piece's lowest cell (INT_MAX)
};

// A run's step inside k_steps (shared memory): where the particles' phase
// reads its field and leaves its results.  Everything a block may write while
// another block of the run still reads the step before is kept apart here or
// in the rotating words of StepWords.
struct FusedStep {
  unsigned long long* S;                 // this step's deposit (ns * (N + 1))
  unsigned long long* births;            // per species: births of this step
  unsigned long long* imp;               // per species: impacts of this step
  int* fail;                             // first error of this step (ecpic_status)
  long long n[kMaxSpecies];              // particles before this step's births
  int cur[kMaxSpecies];                  // buffer set of each species
  uint32_t ctr[kMaxSpecies][kNumCtr];    // counters not yet added to RunState
  uint32_t nlive;                        // particle-steps not yet added
};

// What a pass reads of a segment's and its run's state: the buffer set, the
// particles to process and the time level.
struct PieceState {
  int cur;
  long long n;
  long long k;
};

template <bool FUSED>
__device__ __forceinline__ void fail_run(FusedStep* fx, RunState* st, int code) {
  if (FUSED) atomicCAS(fx->fail, 0, code);
  else set_status(st, code);
}

// a birth beyond the species' capacity
template <bool FUSED>
__device__ __forceinline__ void lose_birth(FusedStep* fx, RunState* st, int sp) {
  if (FUSED) atomicAdd(&fx->ctr[sp][C_LOST], 1u);
  else atomicAdd(&st->ctr[sp][C_LOST], 1ull);
  fail_run<FUSED>(fx, st, ECPIC_ERR_CAPACITY);
}

// Ionisation of the electron at (c, f) with energy Erem above threshold
// left to share (Sec. 2a step 6): the two electrons split it by a uniform
// fraction, the primary leaving along (d0, d1, d2), the secondary isotropic;
// the ion is drawn from the gas Maxwellian.  The secondary is appended to
// this segment, the ion to its species' segment; both are deposited (and,
// on sample steps, enter the vx moments) in HBM.  Returns the primary's new
// velocity.
template <bool FUSED>
__device__ __noinline__ float3 ionize(const BatchView& b, FusedStep* fx, int s, int chosen, int c, float f,
                                      uint64_t id, long long k, float Erem, bool sample, float d0, float d1,
                                      float d2, unsigned kw) {
  const SegDev& G = b.segs[s];
  const int slot = G.run, sp = G.species;
  const RunDev* R = b.runs + slot;
  RunState* st = b.rst + slot;
  SegState* ss = b.sst + s;
  const SpeciesDev* SP = &R->sp[sp];
  const int N = R->N;
  unsigned long long* Sall = FUSED ? fx->S : R->S;
  const uint64_t seed = R->seed;
  // the indices of both births first: their round trips overlap with the rest
  const int ps = SP->proc[chosen].product_seg;
  const bool ion = chk(ps >= 0 && ps < b.nseg, 18, ps, b.nseg);
  const int pspec = SP->proc[chosen].product_species;
  SegState* is = b.sst + (ion ? ps : s);
  // (in k_steps the segments' own words may still be the ones from before a
  // sort: the team's first block writes them, for the host)
  const int cur_e = FUSED ? fx->cur[sp] : ss->cur, cur_i = FUSED ? fx->cur[ion ? pspec : sp] : is->cur;
  const long long idx_e = (FUSED ? fx->n[sp] : 0) +
                          (long long)atomicAdd(FUSED ? fx->births + sp : (unsigned long long*)&ss->n_alloc, 1ull);
  const long long idx_i =
      !ion ? 0 : (FUSED ? fx->n[pspec] : 0) +
                 (long long)atomicAdd(FUSED ? fx->births + pspec : (unsigned long long*)&is->n_alloc, 1ull);
  const uint4 B = draw(seed, id, (uint32_t)k, ((uint32_t)sp << 8) | 1u);
  const float fr = u24(B.x);
  const float v1 = sqrtf(SP->two_e_over_m * (fr * Erem));
  const float v2 = sqrtf(SP->two_e_over_m * ((1.0f - fr) * Erem));
  float e0, e1, e2;
  isotropic(u24(B.y), u24(B.z), e0, e1, e2);
  const uint4 Cw = draw(seed, id, (uint32_t)k, ((uint32_t)sp << 8) | 2u);
  float z0, z1, z2, z3;
  box_muller(u24_open(Cw.x), u24(Cw.y), z0, z1);
  box_muller(u24_open(Cw.z), u24(Cw.w), z2, z3);
  const float sd = R->vth_gas;
  if (FUSED) atomicAdd(&fx->ctr[sp][C_BIRTHS], 1u);
  else atomicAdd(&st->ctr[sp][C_BIRTHS], 1ull);
  // secondary electron: same segment and species; both products carry the
  // parent's weight multiplier kw (charge conserved)
  const float vb = v2 * e0;
  const float fk = (float)kw;
  if (put_particle(G, idx_e, cur_e, c, f, vb, v2 * e1, v2 * e2, child_id(id, k, 1), kw)) {
    if (R->scheme >= ECPIC_SCHEME_EC2)
      deposit2_one(Sall + (size_t)sp * (N + 1), c, f, N, R->bc == ECPIC_PERIODIC);
    else
      deposit_one(Sall + (size_t)sp * (N + 1), c, f, kw);
    if (sample && SP->charge < 0 && c >= R->eedf_c0 && c <= R->eedf_c1)
      atomicAdd(R->tal + (size_t)sp * R->tal_stride +
                    tally_bin(kin_eV(SP->half_m_over_e, vb, yz2(v2 * e1, v2 * e2)), R->eedf_dEinv, R->eedf_n),
                (unsigned long long)kw);
    if (sample) {
      double* md = R->momd + (size_t)sp * 2 * (N + 1);
      atomicAdd(md + c, (double)(fk * ((1.0f - f) * vb)));
      atomicAdd(md + c + 1, (double)(fk * (f * vb)));
      atomicAdd(md + (N + 1) + c, (double)(fk * ((1.0f - f) * vb * vb)));
      atomicAdd(md + (N + 1) + c + 1, (double)(fk * (f * vb * vb)));
    }
  } else {
    lose_birth<FUSED>(fx, st, sp);
  }
  // ion: the product species' segment
  if (ion) {
    const float ivx = sd * z0;
    if (put_particle(b.segs[ps], idx_i, cur_i, c, f, ivx, sd * z1, sd * z2, child_id(id, k, 2), kw)) {
      if (R->scheme >= ECPIC_SCHEME_EC2)
        deposit2_one(Sall + (size_t)pspec * (N + 1), c, f, N, R->bc == ECPIC_PERIODIC);
      else
        deposit_one(Sall + (size_t)pspec * (N + 1), c, f, kw);
      if (sample) {
        double* md = R->momd + (size_t)pspec * 2 * (N + 1);
        atomicAdd(md + c, (double)(fk * ((1.0f - f) * ivx)));
        atomicAdd(md + c + 1, (double)(fk * (f * ivx)));
        atomicAdd(md + (N + 1) + c, (double)(fk * ((1.0f - f) * ivx * ivx)));
        atomicAdd(md + (N + 1) + c + 1, (double)(fk * (f * ivx * ivx)));
      }
    } else {
      lose_birth<FUSED>(fx, st, pspec);
    }
  }
  return make_float3(v1 * d0, v1 * d1, v1 * d2);
}

// Impact tallies of an ion absorbed at x = 0 this step: energy (eV) and
// angle from the electrode normal (degrees) of the velocity that carried it
// out; the absorbed slot keeps that velocity until the next sort.
__device__ __noinline__ void tally_impact(const BatchView& b, int s, int slot, int cur, int i) {
  const SegDev& G = b.segs[s];
  const RunDev* R = b.runs + slot;
  const int sp = G.species;
  if (!chk(i >= 0 && i < G.cap, 26, i, G.cap)) return;
  const float vx = G.vx[cur][i], yz = yz2(G.vy[cur][i], G.vz[cur][i]);
  const float E = kin_eV(R->sp[sp].half_m_over_e, vx, yz);
  const float th = atan2f(sqrtf(yz), fabsf(vx)) * 57.295779513082323f;
  const unsigned long long kw = G.wt[cur] ? (unsigned long long)G.wt[cur][i] : 1ull;
  unsigned long long* tal = R->tal + (size_t)sp * R->tal_stride + R->eedf_n;
  atomicAdd(tal + tally_bin(E, R->iedf_dEinv, R->iedf_n), kw);
  atomicAdd(tal + R->iedf_n + tally_bin(th, R->iad_binv, R->iad_n), kw);
}

// A real (non-null) collision as recorded by the pass (Sec. 2a step 6):
// process, energy En and relative speed gm of the null-collision test, and
// the particle's pushed state.  Redraws Philox block A (scattering angles)
// and, for heavy species, block B (the target neutral's velocity), scatters
// and writes the new velocity.  On sample steps the pass has already added
// the pre-collision vx moments; the change is added here.
template <bool FUSED>
__device__ __forceinline__ void collide_real(const BatchView& b, FusedStep* fx, int s, int slot, int cur,
                                             long long k, bool sample, const RealRec& rec) {
  const int i = rec.i, chosen = rec.chosen;
  const float En = rec.En, gm = rec.gm;
  const SegDev& G = b.segs[s];
  const int sp = G.species;
  const RunDev* R = b.runs + slot;
  const SpeciesDev* SP = &R->sp[sp];
  const int N = R->N;
  const uint64_t seed = R->seed;
  if (!chk(i >= 0 && i < G.cap && chosen >= 0 && chosen < SP->nproc, 6, i, G.cap)) return;
  const int c = rec.c;
  if (!chk(c >= 0 && c < N, 7, c, N)) return;
  const float f = rec.f;
  float vx = rec.vx, vy = rec.vy, vz = rec.vz;
  const float vx_old = vx;
  const uint64_t id = rec.id;
  const uint4 A = draw(seed, id, (uint32_t)k, (uint32_t)sp << 8);
  float gx = vx, gy = vy, gz = vz, vnx = 0.f, vny = 0.f, vnz = 0.f;
  if (SP->heavy) {
    const uint4 B = draw(seed, id, (uint32_t)k, ((uint32_t)sp << 8) | 1u);
    float z0, z1, z2, z3;
    box_muller(u24_open(B.x), u24(B.y), z0, z1);
    box_muller(u24_open(B.z), u24(B.w), z2, z3);
    const float sd = R->vth_gas;
    vnx = sd * z0;
    vny = sd * z1;
    vnz = sd * z2;
    gx -= vnx;
    gy -= vny;
    gz -= vnz;
  }
  float d0, d1, d2;
  isotropic(u24(A.z), u24(A.w), d0, d1, d2);
  const int kind = SP->proc[chosen].kind;
  const float thr = SP->proc[chosen].thr;
  if (kind == ECPIC_ELASTIC) {
    const float cchi = gm > 0.0f ? (gx * d0 + gy * d1 + gz * d2) / gm : 1.0f;
    const float E1 = En * (1.0f - SP->two_m_over_M * (1.0f - cchi));
    const float v1 = sqrtf(SP->two_e_over_m * E1);
    vx = v1 * d0; vy = v1 * d1; vz = v1 * d2;
  } else if (kind == ECPIC_EXCITATION) {
    const float v1 = sqrtf(SP->two_e_over_m * (En - thr));
    vx = v1 * d0; vy = v1 * d1; vz = v1 * d2;
  } else if (kind == ECPIC_IONIZATION) {
    const float3 v1 = ionize<FUSED>(b, fx, s, chosen, c, f, id, k, En - thr, sample, d0, d1, d2, rec.k);
    vx = v1.x; vy = v1.y; vz = v1.z;
  } else if (kind == ECPIC_ION_ELASTIC) {
    const float h = SP->m_frac * gm;
    vx = SP->mass_frac * vx + SP->m_frac * vnx + h * d0;
    vy = SP->mass_frac * vy + SP->m_frac * vny + h * d1;
    vz = SP->mass_frac * vz + SP->m_frac * vnz + h * d2;
  } else {  // ECPIC_CX
    vx = vnx; vy = vny; vz = vnz;
  }
  G.vx[cur][i] = vx;
  G.vy[cur][i] = vy;
  G.vz[cur][i] = vz;
  if (sample && SP->charge < 0 && c >= R->eedf_c0 && c <= R->eedf_c1) {
    // the pass binned the pre-collision energy of this central particle
    const int b0 = tally_bin(kin_eV(SP->half_m_over_e, rec.vx, yz2(rec.vy, rec.vz)), R->eedf_dEinv, R->eedf_n);
    const int b1 = tally_bin(kin_eV(SP->half_m_over_e, vx, yz2(vy, vz)), R->eedf_dEinv, R->eedf_n);
    if (b0 != b1) {
      unsigned long long* tal = R->tal + (size_t)sp * R->tal_stride;
      atomicAdd(tal + b0, 0ull - (unsigned long long)rec.k);  // minus k, modulo 2^64
      atomicAdd(tal + b1, (unsigned long long)rec.k);
    }
  }
  if (sample) {
    double* md = R->momd + (size_t)sp * 2 * (N + 1);
    const float fk = (float)rec.k;
    const float d1v = vx - vx_old, d2v = vx * vx - vx_old * vx_old;
    atomicAdd(md + c, (double)(fk * ((1.0f - f) * d1v)));
    atomicAdd(md + c + 1, (double)(fk * (f * d1v)));
    atomicAdd(md + (N + 1) + c, (double)(fk * ((1.0f - f) * d2v)));
    atomicAdd(md + (N + 1) + c + 1, (double)(fk * (f * d2v)));
  }
}

// Segmented sums across the lanes of a warp for the sample steps' per-node
// float sums (vx moments, J.E).  Adding every particle's share to shared
// memory made a sample step's pass ten times an ordinary one: float atomics
// on shared memory retry while lanes contend, and on cell-sorted particles
// the 32 lanes of a warp add to the same few cells.  A lane whose particles
// all lie in one cell takes that cell as its key; consecutive lanes with
// equal keys form a segment, their values are summed down the segment in
// five shuffle steps, and the segment's first lane adds the sum to shared
// memory.  A lane whose particles lie in several cells (drifting electrons
// some steps after a sort) has key -1 and adds each of its runs of equal
// cells straight to the run's FP64 sums in HBM.  Called by all lanes.
__device__ __forceinline__ unsigned warp_seg_heads(int key, bool* head) {
  const int lane = threadIdx.x & 31;
  const int prev = __shfl_up_sync(0xFFFFFFFFu, key, 1);
  *head = lane == 0 || key != prev;
  return __ballot_sync(0xFFFFFFFFu, *head);
}

// On return, a segment's first lane holds the segment's sum.
__device__ __forceinline__ float warp_seg_sum(float x, unsigned heads) {
  const int lane = threadIdx.x & 31;
  const unsigned long long hb = heads;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_down_sync(0xFFFFFFFFu, x, o);
    // lanes lane+1 .. lane+o start no segment: lane+o is in this one
    const unsigned long long span = ((1ull << o) - 1ull) << (lane + 1);
    if (lane + o < 32 && (hb & span) == 0ull) x += y;
  }
  return x;
}

// The same sums in k_steps' weighted pieces, whose blocks group the particles
// otherwise: two floats per sum, so that its error does not grow with the
// group (about 2^-45 of the terms' sum of magnitudes).
struct Float2 {
  float hi, lo;
  __device__ __forceinline__ void add(float x, float xlo = 0.0f) {
    const float t = hi + x, z = t - hi;
    lo += ((hi - (t - z)) + (x - z)) + xlo;
    hi = t;
  }
  // adds the product x y without its rounding
  __device__ __forceinline__ void add_product(float x, float y) {
    const float p = __fmul_rn(x, y);
    add(p, __fmaf_rn(x, y, -p));
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

__device__ __forceinline__ Float2 warp_seg_sum(Float2 x, unsigned heads) {
  const int lane = threadIdx.x & 31;
  const unsigned long long hb = heads;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float yh = __shfl_down_sync(0xFFFFFFFFu, x.hi, o), yl = __shfl_down_sync(0xFFFFFFFFu, x.lo, o);
    const unsigned long long span = ((1ull << o) - 1ull) << (lane + 1);
    if (lane + o < 32 && (hb & span) == 0ull) x.add(yh, yl);
  }
  return x;
}

// Sample sums of k_steps' unweighted pieces in shared memory: per cell five
// fixed-point sums (J.E of the old cell; (1 - f) v, f v, (1 - f) v^2, f v^2 of
// the new one), each in three 32-bit words added with native atomics (float
// atomics on shared memory are compare-and-swap loops, and the lanes of a warp
// share a few cells).  With 2^e a bound on a quantity's terms over the piece, a
// float term x of at least 2^(e-24) is the 48-bit integer x 2^(47-e) exactly;
// its signed high and unsigned lower 16-bit parts go to the words.  Smaller
// terms, and cells outside the window that the shared memory holds, are
// added straight to the run's FP64 sums in HBM.  So the sums of the terms are
// exact and the same in any order; the terms, the second moments' products
// included, are the floats that k_pass forms for a particle by itself (products
// without that rounding leave the sums farther from k_pass's: 1.2e-8 against
// 4e-9 with 6 particles per cell).  At most kFlushParticles particles between
// flushes keep every word in range.
constexpr int kMomSums = 5;
struct MomSums {
  int* words;          // [quantity][part][w]
  int w0, w;           // the window's first cell and its cells
  int e[3];            // bounds: J.E, v, v^2
  double *pw, *md;     // the species' FP64 sums
  int N;
};
// e with x < 2^e for 0 <= x < bound
__device__ __forceinline__ int mom_bound(float bound) { return bound > 0.0f ? max(ilogbf(bound) + 1, -100) : -100; }
// one quantity (0: J.E, 1, 2: first moments, 3, 4: second) of V particles,
// runs of equal cells merged (c[j] < 0: none)
template <int Q, int V>
__device__ __forceinline__ void mom_add4(const MomSums& m, const int c[V], const float x[V]) {
  constexpr int kind = (Q + 1) / 2;
  double* far = Q == 0 ? m.pw : m.md + (Q >= 3 ? m.N + 1 : 0) + ((Q & 1) ? 0 : 1);
  int hi[V];
  unsigned mid[V], lo[V];
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const unsigned u = __float_as_uint(x[j]);
    const int sh = (int)((u >> 23) & 0xFFu) - 127 - m.e[kind] + 24;
    const bool in = c[j] >= 0 && sh >= 0 && sh < 24 && (unsigned)(c[j] - m.w0) < (unsigned)m.w;
    if (c[j] >= 0 && !in && (u << 1) != 0u) atomicAdd(far + c[j], (double)x[j]);
    long long t = in ? (long long)((u & 0x7FFFFFu) | 0x800000u) << sh : 0ll;
    t = (int)u < 0 ? -t : t;
    lo[j] = (unsigned)t & 0xFFFFu;
    mid[j] = (unsigned)(t >> 16) & 0xFFFFu;
    hi[j] = (int)(t >> 32);
  }
#pragma unroll
  for (int j = V - 1; j >= 1; --j)
    if (c[j] >= 0 && c[j] == c[j - 1]) {
      hi[j - 1] += hi[j];
      mid[j - 1] += mid[j];
      lo[j - 1] += lo[j];
      hi[j] = 0;
      mid[j] = lo[j] = 0u;
    }
  int* base = m.words + (3 * Q) * m.w - m.w0;
#pragma unroll
  for (int j = 0; j < V; ++j)
    if (hi[j] | (int)(mid[j] | lo[j])) {
      atomicAdd(base + c[j], hi[j]);
      atomicAdd(base + m.w + c[j], (int)mid[j]);
      atomicAdd(base + 2 * m.w + c[j], (int)lo[j]);
    }
}
// Adds the window's sums to the run's FP64 sums in HBM and clears them; every
// thread of the block calls it, between barriers.
template <int BLOCK>
__device__ __forceinline__ void mom_flush(const MomSums& m) {
  for (int c = threadIdx.x; c < m.w && m.w0 + c < m.N; c += BLOCK) {
#pragma unroll
    for (int q = 0; q < kMomSums; ++q) {
      int* h = m.words + (3 * q) * m.w + c;
      if (!(h[0] | h[m.w] | h[2 * m.w])) continue;
      const long long t = (long long)((unsigned long long)(long long)h[0] << 32) +
                          (long long)((unsigned long long)(unsigned)h[m.w] << 16) + (long long)(unsigned)h[2 * m.w];
      h[0] = h[m.w] = h[2 * m.w] = 0;
      const double s = __longlong_as_double((long long)(1023 + m.e[(q + 1) / 2] - 47) << 52);
      atomicAdd(q == 0 ? m.pw + m.w0 + c : m.md + (q >= 3 ? m.N + 1 : 0) + m.w0 + c + ((q & 1) ? 0 : 1),
                (double)t * s);
    }
  }
}

// The key of a lane's valid entries c[j] >= 0: their common cell, -1 if they
// lie in several cells or there are none.
template <int V>
__device__ __forceinline__ int lane_cell_key(const int (&c)[V]) {
  int k = -1;
  bool multi = false;
#pragma unroll
  for (int j = 0; j < V; ++j)
    if (c[j] >= 0) {
      if (k < 0) k = c[j];
      else if (c[j] != k) multi = true;
    }
  return multi ? -1 : k;
}

// L2 prefetch of a byte range (one bulk instruction; 16-byte aligned start,
// size a multiple of 16)
__device__ __forceinline__ void l2_prefetch(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Streaming part of one piece: quads [qbeg, qend) of segment s, four
// particles per thread with 16-byte loads (V: or two, or one, where a block of
// k_steps has few).  Gather (Eq. 6-7 / CIC), leapfrog
// (Eq. 8-9) in cell units, walls, the Philox candidate test, fixed-point
// deposit of X^{k+1} (Eq. 2-3).  Collision candidates (Sec. 2a step 6)
// enter a per-warp ring by their index; the warp drains it 32 at a time (all
// lanes busy): it reads the pushed particle again, redraws its Philox block and
// makes the null-collision test.
// The few real collisions are recorded for k_collide, which scatters them
// with its own register budget.  vy, vz are streamed when a species'
// candidate probability is 1/16 or more (its candidates then touch most
// 32-byte sectors anyway) and on energy-sample steps; otherwise the test
// reads them per candidate.
//
// Compiled five times (KIND): 0 = ordinary steps of the linear schemes (the
// common case), 1 = their energy-sample steps (moments, energy, EEDF, J.E),
// 2 = the EC2 scheme with the sample decision taken at run time, 3 and 4 =
// the linear schemes with per-particle weight multipliers (rebalancing
// runs), ordinary and sample steps.  Keeping the rare code out of the
// common instances keeps their loops small in the instruction cache and
// their registers free of the sample-step state.
//
// FUSED (k_steps): the real collisions are carried out where they are found,
// and impacts tallied, instead of being recorded for k_collide; a block of
// 512 or 256 threads with two or four times the registers of k_pass's.
template <int KIND, bool STAGE, int BLOCK, bool FUSED, int V = 4>
__device__ __forceinline__ void pass_piece(const BatchView& b, const RunDev* R, const SegDev& G, int s,
                           const PieceState& ps, long long qbeg, long long qend, int mode, uint32_t* dep,
                           float* Msm, unsigned char* ring, PassShared& sh, FusedStep* fx = nullptr,
                           const float* field = nullptr, int mom_words = 0) {
  // (indices of the four-particle vector loads, which only V = 4 reaches)
  constexpr int x1 = V > 1 ? 1 : 0, x2 = V > 2 ? 2 : 0, x3 = V > 3 ? 3 : 0;
  const int slot = G.run, sp = G.species;
  RunState* st = b.rst + slot;
  SegState* ss = b.sst + s;
  const int N = R->N, scheme = R->scheme, bc = R->bc, uniform = R->uniform;
  const int cur = ps.cur;
  const long long n = ps.n;
  if (!chk(n <= G.cap && N <= b.nmax && (cur == 0 || cur == 1), 14, n, G.cap)) return;
  int32_t* pc = G.cell[cur];
  float* pxi = G.xi[cur];
  float* pvx = G.vx[cur];
  const float* pvy = G.vy[cur];
  const float* pvz = G.vz[cur];
  const uint64_t* pid = G.id[cur];
  const long long k = ps.k;
  const bool stepping = (mode == MODE_STEP);
  constexpr bool weighted = KIND == 3 || KIND == 4;
  const uint32_t* pwt = weighted ? G.wt[cur] : nullptr;
  const bool sample = KIND == 1 || KIND == 4 ||
                      (KIND == 2 && stepping && R->sample_every > 0 &&
                       ((k + 1) % R->sample_every) == 0);
  const SpeciesDev* SP = &R->sp[sp];
  const float qm_dt = SP->qm_dt, dtdx_u = R->dtdx_u;
  // the run's field staged in shared memory for the gather (after the rings)
  float* Esm = reinterpret_cast<float*>(ring + sizeof(int) * (size_t)kRing * (BLOCK / 32));
  // (launches whose CTAs take only an iteration or two read the field from
  // L1/L2 instead: the staging's barrier and round trip would not pay)
  if (STAGE) {
    const int ne = (scheme == ECPIC_SCHEME_MC || scheme == ECPIC_SCHEME_MC2) ? N + 1 : N;
    for (int q = threadIdx.x; q < ne; q += BLOCK) Esm[q] = R->E[q];
    __syncthreads();
  }
  const float* E = FUSED ? field : STAGE ? Esm : R->E;
  const uint32_t thr24 = SP->thr24;
  const bool mcc = stepping && SP->nproc > 0 && thr24 > 0;
  // (r0 >> 8) < thr24 as one comparison of r0
  const uint32_t thr_last = (thr24 << 8) - 1u;  // 2^32 - 1 for thr24 = 2^24
  const bool heavy = SP->heavy != 0;
  const bool yz_stream = mcc && !heavy && thr24 >= (1u << 20);
  const bool load_yz = sample || yz_stream;
  const bool walls = bc != ECPIC_PERIODIC;
  constexpr bool order2 = KIND == 2;
  const bool eedf_on = sample && SP->charge < 0;
  const bool imp_on = stepping && walls && SP->charge > 0 && G.imp_cap > 0;
  const int ec0 = R->eedf_c0, ec1 = R->eedf_c1;
  unsigned long long* tal = R->tal + (size_t)sp * R->tal_stride;
  float* Psm = Msm + 2 * (b.nmax + 1);
  const uint64_t seed = R->seed;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;

  constexpr bool fixed = FUSED && !weighted;  // fixed-point sample sums
  MomSums mom{};
  if (fixed && sample) {
    // bounds over the piece: |v| after the push is at most |v| + |q/m dt| max|E|
    // (the gathers' weights sum to one); the window starts at its lowest cell
    mom.words = reinterpret_cast<int*>(Msm);
    mom.w = min(N, mom_words / (3 * kMomSums));
    for (int i = threadIdx.x; i < 3 * kMomSums * mom.w; i += BLOCK) mom.words[i] = 0;
    float em = 0.0f, vm = 0.0f;
    int lowest = INT_MAX;
    const int ne = (scheme == ECPIC_SCHEME_MC || scheme == ECPIC_SCHEME_MC2) ? N + 1 : N;
    for (int i = threadIdx.x; i < ne; i += BLOCK) em = fmaxf(em, fabsf(E[i]));
    for (long long q = qbeg + threadIdx.x; q < qend; q += BLOCK) {
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const float a = V * q + j < n ? fabsf(pvx[V * q + j]) : 0.0f;
        vm = a < 3.0e8f ? fmaxf(vm, a) : vm;  // (the others fail the run)
      }
      if (mom.w < N && pc[V * q] >= 0) lowest = min(lowest, pc[V * q]);
    }
    const unsigned eb = __reduce_max_sync(kFull, __float_as_uint(em));
    const unsigned vb = __reduce_max_sync(kFull, __float_as_uint(vm));
    lowest = __reduce_min_sync(kFull, lowest);
    if (lane == 0) {
      atomicMax(&sh.top[0], eb);
      atomicMax(&sh.top[1], vb);
      if (mom.w < N) atomicMin(&sh.lowest, lowest);
    }
    __syncthreads();
    em = __uint_as_float(sh.top[0]);
    vm = (__uint_as_float(sh.top[1]) + fabsf(qm_dt) * em) * 1.0001f;
    // (a margin for the cells that particles moved to since the sort)
    if (mom.w < N) mom.w0 = max(0, min(N - mom.w, (sh.lowest < N ? sh.lowest : 0) - mom.w / 8));
    mom.e[0] = mom_bound(2.0f * vm * em * 1.0001f);
    mom.e[1] = mom_bound(vm);
    mom.e[2] = mom_bound(vm * vm * 1.0001f);
    mom.pw = R->pw + (size_t)sp * N;
    mom.md = R->momd + (size_t)sp * 2 * (N + 1);
    mom.N = N;
    __syncthreads();
    if (threadIdx.x == 0) {
      sh.top[0] = sh.top[1] = 0u;
      sh.lowest = INT_MAX;
    }
  }

  // kinetic energy of sample steps: each quad's four terms in FP32, the
  // quads summed in FP64 (one FP64 add per four particles: FP64 is slow on
  // this part), so the error per particle is a few FP32 roundings whatever
  // the number of particles a thread handles
  double ke = 0.0;
  unsigned ncand = 0, nlive = 0, nabs_l = 0, nabs_r = 0, nnan = 0, nimp_lost = 0;
  // this warp's candidate ring: indices (the test reads the particle again and
  // redraws its Philox block: about one particle in a hundred gets there)
  int* qi = reinterpret_cast<int*>(ring) + (threadIdx.x >> 5) * kRing;
  // a bound on the total collision rate per speed, squared, for the filter of
  // the candidates (2^-16 covers every rounding of the comparison)
  const float nu_max = SP->nu_max, nu_bnd2 = SP->nu_bnd * SP->nu_bnd * (1.0f + 1.0f / 65536.0f);
  int head = 0, wcount = 0;  // warp-uniform
  unsigned ncoll = 0;        // FUSED: lane p counts the collisions of process p
  uint32_t* dcnt = dep;
  uint32_t* dlo = dep + (b.nmax + 1);
  uint32_t* dhi = dep + 2 * (b.nmax + 1);
  // weighted runs: four 32-bit sums per cell (dep holds four arrays when the
  // batch has weighted runs)
  const DepW dw{dep, dep + (b.nmax + 1), dep + 2 * (b.nmax + 1), dep + 3 * (b.nmax + 1)};
  unsigned long long* Sg = (FUSED ? fx->S : R->S) + (size_t)sp * (N + 1);
  int since_flush = 0;

  // block-uniform trip count (warp collectives below need full warps); the
  // pass after the last quad empties both rings
  for (long long base = qbeg;; base += BLOCK) {
    const bool more = base < qend;
    if (more) {
      if (V == 4 && threadIdx.x == 0) {
        // the next iteration's particle records into L2
        const long long nb = base + BLOCK;
        if (nb < qend) {
          const long long p0 = 4 * nb;
          long long p1 = 4 * min(qend, nb + BLOCK);
          p1 = min(p1, n);
          if (p1 > p0) {
            const unsigned b4 = (unsigned)(((p1 - p0) * 4) & ~15ll);
            if (b4) {
              l2_prefetch(pc + p0, b4);
              l2_prefetch(pxi + p0, b4);
              l2_prefetch(pvx + p0, b4);
              if (load_yz) {
                l2_prefetch(pvy + p0, b4);
                l2_prefetch(pvz + p0, b4);
              }
              if (mcc) l2_prefetch(pid + p0, (unsigned)(((p1 - p0) * 8) & ~15ll));
              if (weighted) l2_prefetch(pwt + p0, b4);
            }
          }
        }
      }
      const long long q = base + (long long)threadIdx.x;
      const long long i0 = V * q;
      const bool inq = q < qend && chk(i0 < G.cap, 2, i0, G.cap);
      const bool full = V == 4 && inq && (i0 + 3 < n) && chk(i0 + 3 < G.cap, 3, i0 + 3, G.cap);
      int c[V];
      float f[V], v[V];
      if (full) {
        const int4 c4 = *reinterpret_cast<const int4*>(pc + i0);
        const float4 f4 = *reinterpret_cast<const float4*>(pxi + i0);
        const float4 v4 = *reinterpret_cast<const float4*>(pvx + i0);
        c[0] = c4.x; c[x1] = c4.y; c[x2] = c4.z; c[x3] = c4.w;
        f[0] = f4.x; f[x1] = f4.y; f[x2] = f4.z; f[x3] = f4.w;
        v[0] = v4.x; v[x1] = v4.y; v[x2] = v4.z; v[x3] = v4.w;
      } else {
#pragma unroll
        for (int j = 0; j < V; ++j) {
          const bool in = inq && (i0 + j < n);
          c[j] = in ? pc[i0 + j] : -1;
          f[j] = in ? pxi[i0 + j] : 0.0f;
          v[j] = in ? pvx[i0 + j] : 0.0f;
        }
      }
      // weight multipliers: read here on sample steps (the moments use them),
      // else just before the deposit (a shorter live range)
      unsigned kq[V];
#pragma unroll
      for (int j = 0; j < V; ++j) kq[j] = 1u;
      if (weighted && sample) {
        if (full) {
          const uint4 k4 = *reinterpret_cast<const uint4*>(pwt + i0);
          kq[0] = k4.x; kq[x1] = k4.y; kq[x2] = k4.z; kq[x3] = k4.w;
        } else {
#pragma unroll
          for (int j = 0; j < V; ++j) kq[j] = (inq && i0 + j < n) ? pwt[i0 + j] : 1u;
        }
      }
      bool cand[V] = {};
      unsigned hit = 0u;  // bit j: absorbed at x = 0 (impact tallies)
      int any = c[0];  // negative: some particle is absorbed
#pragma unroll
      for (int j = 1; j < V; ++j) any |= c[j];
      if (any >= 0) {
        nlive += (unsigned)V;
      } else {
        // absorbed particles: far from every cell, wherever the push takes them
#pragma unroll
        for (int j = 0; j < V; ++j) {
          nlive += c[j] >= 0 ? 1u : 0u;
          c[j] = c[j] >= 0 ? c[j] : kFarCell;
        }
      }
      if (stepping) {
        uint64_t id[V] = {};
        if (mcc) {
          if (full) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(pid + i0);
            const ulonglong2 bq = *reinterpret_cast<const ulonglong2*>(pid + i0 + 2);
            id[0] = a.x; id[x1] = a.y; id[x2] = bq.x; id[x3] = bq.y;
          } else {
#pragma unroll
            for (int j = 0; j < V; ++j) id[j] = c[j] >= 0 ? pid[i0 + j] : 0ull;
          }
        }
        // vy^2 + vz^2 (collisions do not change it before the push reads it)
        float yz[V] = {};
        if (load_yz) {
          if (full) {
            const float4 y4 = *reinterpret_cast<const float4*>(pvy + i0);
            const float4 z4 = *reinterpret_cast<const float4*>(pvz + i0);
            yz[0] = yz2(y4.x, z4.x);
            yz[x1] = yz2(y4.y, z4.y);
            yz[x2] = yz2(y4.z, z4.z);
            yz[x3] = yz2(y4.w, z4.w);
          } else {
#pragma unroll
            for (int j = 0; j < V; ++j)
              if (c[j] >= 0) yz[j] = yz2(pvy[i0 + j], pvz[i0 + j]);
          }
        }
        // gather (Eq. 6-7; CIC for MC) and push (Eq. 8), branch-free over the
        // four particles so the loads and arithmetic overlap
        float Ei[V];
#pragma unroll
        for (int j = 0; j < V; ++j) {
          if (!chk(c[j] < N, 4, c[j], N)) c[j] = kFarCell;
          const int cc = max(c[j], 0);
          if (scheme == ECPIC_SCHEME_EC) {
            Ei[j] = E[cc];
          } else if (order2 && scheme == ECPIC_SCHEME_MC2) {
            // the deposit's quadratic weights on the centred node field (its
            // transpose: folded and wrapped nodes read their field)
            const bool up = f[j] >= 0.5f;
            const int n0 = cc + (up ? 1 : 0);
            const float u = up ? f[j] - 1.0f : f[j];
            const float wl = 0.5f * (0.5f - u) * (0.5f - u), wr = 0.5f * (0.5f + u) * (0.5f + u);
            Ei[j] = wl * E[node2(n0 - 1, N, !walls)] + (0.75f - u * u) * E[n0] +
                    wr * E[node2(n0 + 1, N, !walls)];
          } else if (order2) {
            // linear between the faces about the nearest node n0 (faces
            // n0-1 and n0): the derivative of the quadratic-spline potential
            const bool up = f[j] >= 0.5f;
            const int n0 = cc + (up ? 1 : 0);
            const float u = up ? f[j] - 1.0f : f[j];
            float El, Er;
            if (walls) {
              El = n0 >= 1 ? E[n0 - 1] : 0.0f;
              Er = n0 < N ? E[n0] : 0.0f;
            } else {
              El = E[n0 >= 1 ? n0 - 1 : N - 1];
              Er = E[n0 < N ? n0 : 0];
            }
            Ei[j] = (0.5f - u) * El + (0.5f + u) * Er;
          } else {
            const float e0 = E[cc], e1 = E[cc + 1];
            Ei[j] = e0 + f[j] * (e1 - e0);
          }
        }
        float keq = 0.0f;
        Float2 kef{0.0f, 0.0f};  // k_steps: the quad's terms without rounding their sum
        float pje[V] = {};
#pragma unroll
        for (int j = 0; j < V; ++j) {
          const float vnew = v[j] + qm_dt * Ei[j];
          if (sample) {
            const float fk = weighted ? (float)kq[j] : 1.0f;
            if (c[j] >= 0) {
              if (FUSED) kef.add(fk * (v[j] * vnew + yz[j]));
              else keq += fk * (v[j] * vnew + yz[j]);
            }
            // J.E of the push, per cell at level k (scaled by q w / 2 dx later)
            pje[j] = c[j] >= 0 ? fk * ((v[j] + vnew) * Ei[j]) : 0.0f;
          }
          v[j] = vnew;
        }
        if (sample) {
          ke += FUSED ? kef.value() : (double)keq;
          // J.E per cell of level k: per lane, then down each segment
          const int key = lane_cell_key(c);
          double* pwg = R->pw + (size_t)sp * N;
          if (fixed) {
            mom_add4<0, V>(mom, c, pje);
          } else if (FUSED) {
            Float2 pl{0.0f, 0.0f};
#pragma unroll
            for (int j = 0; j < V; ++j) {
              if (c[j] < 0) continue;
              if (key < 0) atomicAdd(pwg + c[j], (double)pje[j]);
              else pl.add(pje[j]);
            }
            bool head;
            const unsigned heads = warp_seg_heads(key, &head);
            pl = warp_seg_sum(pl, heads);
            if (head && key >= 0) atomicAdd(pwg + key, pl.value());
          } else {
          float pl = 0.0f;
          int cc = -1;
#pragma unroll
          for (int j = 0; j < V; ++j) {
            if (c[j] < 0) continue;
            if (key < 0 && c[j] != cc) {
              if (cc >= 0) atomicAdd(pwg + cc, (double)pl);
              cc = c[j];
              pl = 0.0f;
            }
            pl += pje[j];
          }
          if (key < 0 && cc >= 0) {
            atomicAdd(pwg + cc, (double)pl);
            pl = 0.0f;
          }
          bool head;
          const unsigned heads = warp_seg_heads(key, &head);
          pl = warp_seg_sum(pl, heads);
          if (head && key >= 0) atomicAdd(Psm + key, pl);
          }
        }
        // Philox block A of all four: independent chains the scheduler
        // interleaves; A.x decides the candidate, A.y selects the process
        uint32_t r0[V] = {}, ry[V] = {};
        if (mcc) {
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const uint4 A = draw(seed, id[j], (uint32_t)k, (uint32_t)sp << 8);
            r0[j] = A.x;
            ry[j] = A.y;
          }
        }
        // Eq. 9 in cell units, then the walls: absorbed when X <= 0 or X >= L
#pragma unroll
        for (int j = 0; j < V; ++j) cand[j] = mcc && r0[j] <= thr_last;
        if (uniform) {
          int cj[V];
          float g[V];
#pragma unroll
          for (int j = 0; j < V; ++j) {
            g[j] = f[j] + v[j] * dtdx_u;
            const float fl = floorf(g[j]);
            cj[j] = c[j] + (int)fl;
            g[j] -= fl;
          }
          // Nearly every quad stays inside: a live one with cells 0..N-1, off
          // X = 0, offsets that did not round to 1 and finite speeds.  One set
          // of tests per quad sees that (some tests wider than the rule); the
          // others are told apart particle by particle in a rare branch.
          unsigned top = 0u, zero = 0xFFFFFFFFu;
          float gm = 0.0f, vs = 0.0f;
#pragma unroll
          for (int j = 0; j < V; ++j) {
            top = max(top, (unsigned)cj[j]);
            zero = min(zero, (unsigned)cj[j] | __float_as_uint(g[j]));
            gm = fmaxf(gm, g[j]);
            vs += fabsf(v[j]);
          }
          if (top < (unsigned)N && zero != 0u && gm < 1.0f && vs < 3.0e8f) {
#pragma unroll
            for (int j = 0; j < V; ++j) {
              c[j] = cj[j];
              f[j] = g[j];
            }
          } else {
#pragma unroll
            for (int j = 0; j < V; ++j) {
              bool ok = c[j] >= 0;
              if (ok) {
                if (g[j] >= 1.0f) {  // g - floor(g) rounded to 1
                  cj[j] += 1;
                  g[j] = 0.0f;
                }
                if (!walls && (unsigned)cj[j] >= (unsigned)N) {
                  cj[j] %= N;
                  if (cj[j] < 0) cj[j] += N;
                }
                if (!(fabsf(v[j]) < 3.0e8f)) {
                  ++nnan;
                  ok = false;
                } else if (walls && ((unsigned)cj[j] >= (unsigned)N || (cj[j] == 0 && g[j] == 0.0f))) {
                  ok = false;
                  if (cj[j] >= N) {
                    ++nabs_r;
                  } else {
                    ++nabs_l;
                    hit |= imp_on ? 1u << j : 0u;
                  }
                }
              }
              c[j] = ok ? cj[j] : -1;
              f[j] = g[j];
              cand[j] = cand[j] && ok;
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < V; ++j) {
            if (c[j] < 0) {
              c[j] = -1;
              cand[j] = false;
              continue;
            }
            if (!(fabsf(v[j]) < 3.0e8f)) {
              ++nnan;
              c[j] = -1;
              cand[j] = false;
              continue;
            }
            int cj = c[j];
            float fj = f[j];
            walk_nonuniform(cj, fj, fj + v[j] * __ldg(R->dtdx + cj), N, bc, R->rp, R->rm);
            if (walls && (cj < 0 || cj >= N || (cj == 0 && fj == 0.0f))) {
              nabs_r += cj >= N ? 1u : 0u;
              nabs_l += cj >= N ? 0u : 1u;
              hit |= imp_on && cj < N ? 1u << j : 0u;
              c[j] = -1;
              cand[j] = false;
              continue;
            }
            c[j] = cj;
            f[j] = fj;
          }
        }
        if (full) {
          *reinterpret_cast<int4*>(pc + i0) = make_int4(c[0], c[x1], c[x2], c[x3]);
          *reinterpret_cast<float4*>(pxi + i0) = make_float4(f[0], f[x1], f[x2], f[x3]);
          *reinterpret_cast<float4*>(pvx + i0) = make_float4(v[0], v[x1], v[x2], v[x3]);
        } else {
#pragma unroll
          for (int j = 0; j < V; ++j)
            if (inq && i0 + j < n) {
              pc[i0 + j] = c[j];
              pxi[i0 + j] = f[j];
              pvx[i0 + j] = v[j];
            }
        }
        // ions absorbed at x = 0: their indices, for the impact tallies of the
        // collision kernel (the absorbed slot keeps its velocity until the sort)
        if (imp_on && __any_sync(kFull, hit != 0u)) {
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const unsigned m = __ballot_sync(kFull, (hit >> j) & 1u);
            if (m) {
              const int lead = __ffs(m) - 1;
              unsigned long long base = 0ull;
              if (lane == lead) base = atomicAdd(FUSED ? fx->imp + sp : (unsigned long long*)&ss->n_imp,
                                                  (unsigned long long)__popc(m));
              base = __shfl_sync(kFull, base, lead);
              if ((hit >> j) & 1u) {
                const long long idx = (long long)base + __popc(m & lt_mask);
                if (idx >= G.imp_cap) ++nimp_lost;
                else if (FUSED) tally_impact(b, s, slot, cur, (int)(i0 + j));
                else G.imp[idx] = (int)(i0 + j);
              }
            }
          }
        }
        // EEDF of the central cells on sample steps (pre-collision; the
        // collision kernel moves the particles that collide)
        if (eedf_on) {
#pragma unroll
          for (int j = 0; j < V; ++j)
            if (c[j] >= ec0 && c[j] <= ec1)
              atomicAdd(tal + tally_bin(kin_eV(SP->half_m_over_e, v[j], yz[j]), R->eedf_dEinv, R->eedf_n),
                        (unsigned long long)kq[j]);
        }
        if (mcc) {
          // a candidate with Rr >= nu_bnd |g| is a null collision whatever its
          // energy (the total rate never exceeds nu_bnd |g|): where |g| is at
          // hand, only the others go on to the cross-section test.  Compared
          // in squares, with Rr from 23 bits rounded down and the bound
          // rounded up: the test itself decides what this lets through.
          unsigned mine = 0u;
#pragma unroll
          for (int j = 0; j < V; ++j) {
            ncand += cand[j] ? 1u : 0u;
            const float Rl = (__uint_as_float((ry[j] >> 9) | 0x3F800000u) - 1.0f) * nu_max;
            const bool null = yz_stream && Rl * Rl > nu_bnd2 * (v[j] * v[j] + yz[j]);
            mine |= cand[j] && !null ? 1u << j : 0u;
          }
          unsigned m = __ballot_sync(kFull, mine != 0u);
          // one candidate per lane and round (mostly one round, or none)
          while (m) {
            if (mine) {
              int pos = head + wcount + __popc(m & lt_mask);
              if (pos >= kRing) pos -= kRing;
              if (chk(pos >= 0 && pos < kRing, 5, pos, kRing)) qi[pos] = (int)i0 + __ffs((int)mine) - 1;
              mine &= mine - 1u;
            }
            wcount += __popc(m);
            m = __ballot_sync(kFull, mine != 0u);
          }
        }
      }
      // fixed-point CIC deposit of the new positions (Eq. 2-3); vx moments
      // (pre-collision: the collision adds the change)
      if (order2)
        dep2_add4<V>(dlo, dhi, N, !walls, c, f);
      else if (weighted) {
        if (!sample) {
          if (full) {
            const uint4 k4 = *reinterpret_cast<const uint4*>(pwt + i0);
            kq[0] = k4.x; kq[x1] = k4.y; kq[x2] = k4.z; kq[x3] = k4.w;
          } else {
#pragma unroll
            for (int j = 0; j < V; ++j) kq[j] = (inq && i0 + j < n) ? pwt[i0 + j] : 1u;
          }
        }
        depw_add4<V>(dw, c, f, kq);
      }
      else
        dep_add4<V>(dcnt, dlo, dhi, c, f);
      if (sample) {
        // vx moments at the nodes of the new cell (CIC shares): per lane
        // summed where its particles share a cell, then down each segment
        const int Nm = b.nmax + 1;
        int cm[V];
#pragma unroll
        for (int j = 0; j < V; ++j)
          cm[j] = (c[j] >= 0 && chk(c[j] + 1 <= b.nmax, 20, c[j], b.nmax)) ? c[j] : -1;
        const int key = lane_cell_key(cm);
        double* mdg = R->momd + (size_t)sp * 2 * (N + 1);
        if (fixed) {
          float x[V], y[V];
#pragma unroll
          for (int j = 0; j < V; ++j) {
            x[j] = (1.0f - f[j]) * v[j];
            y[j] = x[j] * v[j];
          }
          mom_add4<1, V>(mom, cm, x);
          mom_add4<3, V>(mom, cm, y);
#pragma unroll
          for (int j = 0; j < V; ++j) {
            x[j] = f[j] * v[j];
            y[j] = x[j] * v[j];
          }
          mom_add4<2, V>(mom, cm, x);
          mom_add4<4, V>(mom, cm, y);
        } else if (FUSED) {
          Float2 a1{0.0f, 0.0f}, b1{0.0f, 0.0f}, a2{0.0f, 0.0f}, b2{0.0f, 0.0f};
#pragma unroll
          for (int j = 0; j < V; ++j) {
            if (cm[j] < 0) continue;
            const float fk = weighted ? (float)kq[j] : 1.0f;
            const float lo = fk * ((1.0f - f[j]) * v[j]), hi = fk * (f[j] * v[j]);
            if (key < 0) {
              double* m1 = mdg + cm[j];
              atomicAdd(m1, (double)lo);
              atomicAdd(m1 + 1, (double)hi);
              atomicAdd(m1 + (N + 1), (double)lo * (double)v[j]);
              atomicAdd(m1 + (N + 1) + 1, (double)hi * (double)v[j]);
            } else {
              a1.add(lo);
              b1.add(hi);
              a2.add_product(lo, v[j]);
              b2.add_product(hi, v[j]);
            }
          }
          bool head;
          const unsigned heads = warp_seg_heads(key, &head);
          a1 = warp_seg_sum(a1, heads);
          b1 = warp_seg_sum(b1, heads);
          a2 = warp_seg_sum(a2, heads);
          b2 = warp_seg_sum(b2, heads);
          if (head && key >= 0) {
            atomicAdd(mdg + key, a1.value());
            atomicAdd(mdg + key + 1, b1.value());
            atomicAdd(mdg + (N + 1) + key, a2.value());
            atomicAdd(mdg + (N + 1) + key + 1, b2.value());
          }
        } else {
        float a1 = 0.0f, b1 = 0.0f, a2 = 0.0f, b2 = 0.0f;
        int cc = -1;  // spread lanes: the current run of equal cells
#pragma unroll
        for (int j = 0; j < V; ++j) {
          if (cm[j] < 0) continue;
          const float fk = weighted ? (float)kq[j] : 1.0f;
          const float lo = fk * ((1.0f - f[j]) * v[j]), hi = fk * (f[j] * v[j]);
          if (key < 0 && cm[j] != cc) {
            // spread over cells: each run of equal cells straight to the
            // run's FP64 sums in HBM
            if (cc >= 0) {
              atomicAdd(mdg + cc, (double)a1);
              atomicAdd(mdg + cc + 1, (double)b1);
              atomicAdd(mdg + (N + 1) + cc, (double)a2);
              atomicAdd(mdg + (N + 1) + cc + 1, (double)b2);
            }
            cc = cm[j];
            a1 = b1 = a2 = b2 = 0.0f;
          }
          a1 += lo;
          b1 += hi;
          a2 += lo * v[j];
          b2 += hi * v[j];
        }
        if (key < 0 && cc >= 0) {
          atomicAdd(mdg + cc, (double)a1);
          atomicAdd(mdg + cc + 1, (double)b1);
          atomicAdd(mdg + (N + 1) + cc, (double)a2);
          atomicAdd(mdg + (N + 1) + cc + 1, (double)b2);
          a1 = b1 = a2 = b2 = 0.0f;
        }
        bool head;
        const unsigned heads = warp_seg_heads(key, &head);
        a1 = warp_seg_sum(a1, heads);
        b1 = warp_seg_sum(b1, heads);
        a2 = warp_seg_sum(a2, heads);
        b2 = warp_seg_sum(b2, heads);
        if (head && key >= 0) {
          atomicAdd(Msm + key, a1);
          atomicAdd(Msm + key + 1, b1);
          atomicAdd(Msm + Nm + key, a2);
          atomicAdd(Msm + Nm + key + 1, b2);
        }
        }
      }
    }
    if (mcc) {
      __syncwarp();
      while (wcount >= 32 || (!more && wcount > 0)) {
        // null-collision test of up to 32 candidates
        const int take = min(wcount, 32);
        const bool act = lane < take;
        int pos = head + lane;
        if (pos >= kRing) pos -= kRing;
        int i = 0;
        uint64_t id = 0ull;
        float vx = 0.0f, vy = 0.0f, vz = 0.0f, g2 = 0.0f, Rr = 0.0f;
        if (act) {
          i = qi[pos];
          id = pid[i];
          vx = pvx[i];
          vy = pvy[i];
          vz = pvz[i];
          Rr = u24(draw(seed, id, (uint32_t)k, (uint32_t)sp << 8).y) * nu_max;
          if (heavy) {
            // relative speed to a target neutral drawn from the gas Maxwellian
            const uint4 B = draw(seed, id, (uint32_t)k, ((uint32_t)sp << 8) | 1u);
            float z0, z1, z2, z3;
            box_muller(u24_open(B.x), u24(B.y), z0, z1);
            box_muller(u24_open(B.z), u24(B.w), z2, z3);
            const float sd = R->vth_gas;
            const float gx = vx - sd * z0, gy = vy - sd * z1, gz = vz - sd * z2;
            g2 = gx * gx + gy * gy + gz * gz;
          } else if (yz_stream) {
            g2 = vx * vx + yz2(vy, vz);
          } else {
            g2 = vx * vx + (vy * vy + vz * vz);
          }
        }
        const float gm = sqrtf(g2), En = SP->half_m_over_e * g2;
        float tot = 0.0f;
        int chosen = -1;
        if (act && Rr < SP->nu_bnd * gm) chosen = select_process(SP, En, gm, R->ng, Rr, &tot);
        if (tot > nu_max) atomicAdd(FUSED ? &fx->ctr[sp][C_CLAMPS] : &sh.ctr[C_CLAMPS], 1u);
        const unsigned m = __ballot_sync(kFull, chosen >= 0);
        if (FUSED) {
          if (m) {
            for (int p = 0; p < SP->nproc; ++p) {
              const unsigned mp = __ballot_sync(kFull, chosen == p);
              if (lane == p) ncoll += __popc(mp);
            }
            if (chosen >= 0) {
              RealRec rec;
              rec.id = id;
              rec.i = i;
              rec.chosen = chosen;
              rec.En = En;
              rec.gm = gm;
              rec.vx = vx;
              rec.vy = vy;
              rec.vz = vz;
              rec.c = pc[i];
              rec.f = pxi[i];
              rec.k = weighted ? pwt[i] : 1u;
              collide_real<true>(b, fx, s, slot, cur, k, sample, rec);
            }
          }
        } else if (m) {
          // real collisions: a record each, with the particle's pushed state
          // (still in L1/L2 here), for the collision kernel
          const int lead = __ffs(m) - 1;
          unsigned long long base = 0ull;
          if (lane == lead) base = atomicAdd((unsigned long long*)&ss->n_real, (unsigned long long)__popc(m));
          base = __shfl_sync(kFull, base, lead);
          if (chosen >= 0) {
            const long long idx = (long long)base + __popc(m & lt_mask);
            if (idx < G.real_cap) {
              int4* dst = reinterpret_cast<int4*>(G.real + idx);  // RealRec field order
              dst[0] = make_int4((int)(uint32_t)id, (int)(uint32_t)(id >> 32), i, chosen);
              dst[1] = make_int4(__float_as_int(En), __float_as_int(gm), __float_as_int(vx), __float_as_int(vy));
              dst[2] = make_int4(__float_as_int(vz), pc[i], __float_as_int(pxi[i]),
                                 weighted ? (int)pwt[i] : 1);
            } else {
              set_status(st, ECPIC_ERR_CAPACITY);
            }
          }
        }
        head += take;
        if (head >= kRing) head -= kRing;
        wcount -= take;
        __syncwarp();
      }
    }
    if (!more) break;
    constexpr int iters = kFlushParticles / (V * BLOCK);
    if (++since_flush == (order2 ? iters / 4 : weighted ? iters / 2 : iters)) {
      __syncthreads();
      if (order2)
        dep2_flush(dlo, dhi, 0, N, Sg);
      else if (weighted)
        depw_flush(dw, 0, N, Sg);
      else
        dep_flush(dcnt, dlo, dhi, 0, N, Sg);
      if (fixed && sample) mom_flush<BLOCK>(mom);
      __syncthreads();
      since_flush = 0;
    }
  }

  if (FUSED) {
    // Piece epilogue in k_steps: counters stay in shared memory until the
    // launch ends, the deposit goes to this step's sums.  (The range of cells
    // is not tracked: a block takes few iterations, and its threads look at
    // every cell in two or three reads.)
    ncand = __reduce_add_sync(kFull, ncand);
    nlive = __reduce_add_sync(kFull, nlive);
    nabs_l = __reduce_add_sync(kFull, nabs_l);
    nabs_r = __reduce_add_sync(kFull, nabs_r);
    nnan = __reduce_add_sync(kFull, nnan);
    nimp_lost = __reduce_add_sync(kFull, nimp_lost);
    uint32_t* ctr = fx->ctr[sp];
    if (lane < kMaxProc && ncoll) atomicAdd(ctr + C_COLL0 + lane, ncoll);
    if (lane == 0) {
      if (nlive) atomicAdd(&fx->nlive, nlive);
      if (ncand) atomicAdd(ctr + C_CAND, ncand);
      if (nabs_l) atomicAdd(ctr + C_ABS_L, nabs_l);
      if (nabs_r) atomicAdd(ctr + C_ABS_R, nabs_r);
      if (nimp_lost) atomicAdd(ctr + C_IMP_LOST, nimp_lost);
      if (nnan) {
        atomicAdd(ctr + C_NAN, nnan);
        fail_run<true>(fx, st, ECPIC_ERR_NAN);
      }
    }
    if (sample) {
      const double kes = block_sum(ke, sh.dsm);
      if (threadIdx.x == 0) atomicAdd(&st->ke_acc[sp], 0.5 * SP->m * SP->w * kes);
    }
    __syncthreads();
    if (order2)
      dep2_flush(dlo, dhi, 0, N, Sg);
    else if (weighted)
      depw_flush(dw, 0, N, Sg);
    else
      dep_flush(dcnt, dlo, dhi, 0, N, Sg);
    if (fixed && sample) mom_flush<BLOCK>(mom);
    __syncthreads();
    return;
  }
  // piece epilogue: energy, counters, flush to HBM
  ncand = __reduce_add_sync(kFull, ncand);
  nlive = __reduce_add_sync(kFull, nlive);
  nabs_l = __reduce_add_sync(kFull, nabs_l);
  nabs_r = __reduce_add_sync(kFull, nabs_r);
  nnan = __reduce_add_sync(kFull, nnan);
  nimp_lost = __reduce_add_sync(kFull, nimp_lost);
  if (lane == 0) {
    if (stepping && nlive) atomicAdd(&sh.nlive, nlive);
    if (ncand) atomicAdd(&sh.ctr[C_CAND], ncand);
    if (nabs_l) atomicAdd(&sh.ctr[C_ABS_L], nabs_l);
    if (nabs_r) atomicAdd(&sh.ctr[C_ABS_R], nabs_r);
    if (nimp_lost) atomicAdd(&sh.ctr[C_IMP_LOST], nimp_lost);
    if (nnan) {
      atomicAdd(&sh.ctr[C_NAN], nnan);
      set_status(st, ECPIC_ERR_NAN);
    }
  }
  if (sample) {
    const double kes = block_sum(ke, sh.dsm);
    if (threadIdx.x == 0) atomicAdd(&st->ke_acc[sp], 0.5 * SP->m * SP->w * kes);
  }
  __syncthreads();
  // (every cell: the range that the particles touch is not tracked, which
  // costs the streaming loop more than the few reads of this scan)
  if (order2)
    dep2_flush(dlo, dhi, 0, N, Sg);
  else if (weighted)
    depw_flush(dw, 0, N, Sg);
  else
    dep_flush(dcnt, dlo, dhi, 0, N, Sg);
  if (sample) {
    const int Nm = b.nmax + 1;
    double* md = R->momd + (size_t)sp * 2 * (N + 1);
    double* pwg = R->pw + (size_t)sp * N;
    for (int nn = threadIdx.x; nn <= N; nn += BLOCK) {
      const float m1 = Msm[nn], m2 = Msm[Nm + nn];
      if (m1 != 0.0f) atomicAdd(md + nn, (double)m1);
      if (m2 != 0.0f) atomicAdd(md + (N + 1) + nn, (double)m2);
      Msm[nn] = 0.0f;
      Msm[Nm + nn] = 0.0f;
      if (nn < N) {
        const float pj = Psm[nn];
        if (pj != 0.0f) atomicAdd(pwg + nn, (double)pj);
        Psm[nn] = 0.0f;
      }
    }
  }
  if (threadIdx.x < 32) {  // (kNumCtr < 32)
    const uint32_t val = lane < kNumCtr ? sh.ctr[lane] : lane == kNumCtr ? sh.nlive : 0u;
    if (val) {
      if (lane < kNumCtr) {
        atomicAdd(&st->ctr[sp][lane], (unsigned long long)val);
        sh.ctr[lane] = 0u;
      } else {
        atomicAdd(&st->psteps, (unsigned long long)val);
        sh.nlive = 0u;
      }
    }
    const uint32_t dead = __reduce_add_sync(
        kFull, lane == C_ABS_L || lane == C_ABS_R || lane == C_NAN ? val : 0u);
    if (lane == 0 && dead) atomicAdd((unsigned long long*)&ss->n_dead, (unsigned long long)dead);
  }
  __syncthreads();
}

// ----------------------------------------------------------------- field
// 1/D in FP64 from an FP32 seed and two Newton steps (no FP64 division,
// which is slow on this part); D > 0.
__device__ __forceinline__ double recip(double D) {
  double r = (double)__frcp_rn((float)D);
  r = r * (2.0 - D * r);
  r = r * (2.0 - D * r);
  return r;
}

// Scratch of field_solve in dynamic shared memory: C | dx | every species'
// deposit, N + 1 words of 8 bytes each.
__host__ __device__ inline size_t field_scratch_bytes(int nmax, int species) {
  return sizeof(double) * (size_t)(nmax + 1) * (size_t)(species + 2);
}

struct FieldShared {
  unsigned long long wtot[kFieldOwners / 32][kMaxSpecies];
  double wsum[kFieldOwners / 32];
  double wsm[32];
  double phi0;
};

// Sum of one value per owner thread (tid < kFieldOwners; the others pass
// anything) as a balanced tree over lanes, then over warps: the same
// association whatever the block size, so that the field is bit-identical
// from every kernel that solves it.  One barrier.
__device__ __forceinline__ double owners_sum(double v, double* wsum) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
  if (tid < kFieldOwners && (tid & 31) == 0) wsum[tid >> 5] = v;
  __syncthreads();
  static_assert(kFieldOwners == 256, "eight owner warps");
  return ((wsum[7] + wsum[6]) + (wsum[5] + wsum[4])) + ((wsum[3] + wsum[2]) + (wsum[1] + wsum[0]));
}

constexpr double kInvEps0 = 1.0 / kEps0;

// Moments of a sampled level (Sec. 3a: density and x temperature per node)
// from its deposit S (ns * (N + 1)) and the vx moments, which are cleared; the
// share `part` of `parts` of the nodes.
template <int BLOCK>
__device__ __forceinline__ void sample_moments(const RunDev* R, const unsigned long long* S, int part = 0,
                                               int parts = 1) {
  constexpr double kInvQe = 1.0 / 1.602176634e-19;
  constexpr double k2m32 = 2.3283064365386963e-10;  // 2^-32
  const int N = R->N, ns = R->ns, M = N + 1;
  const bool periodic = (R->bc == ECPIC_PERIODIC);
  double* acc = R->acc;
  for (int n = threadIdx.x + BLOCK * part; n < (periodic ? N : M); n += BLOCK * parts) {
    const bool ends = periodic && n == 0;  // node N is node 0
    for (int s = 0; s < ns; ++s) {
      double* md = R->momd + (size_t)s * 2 * M;
      double Dn, M1, M2;
      if (ends) {
        Dn = (double)(S[(size_t)s * M] + S[(size_t)s * M + N]);
        M1 = md[0] + md[N];
        M2 = md[N + 1] + md[N + 1 + N];
        md[N] = 0.0;
        md[N + 1 + N] = 0.0;
      } else {
        Dn = (double)S[(size_t)s * M + n];
        M1 = md[n];
        M2 = md[N + 1 + n];
      }
      md[n] = 0.0;
      md[N + 1 + n] = 0.0;
      Dn *= k2m32;
      double T = 0.0;
      if (Dn > 0.0) {
        const double iD = recip(Dn);
        const double u = M1 * iD;
        T = R->sp[s].m * (M2 * iD - u * u) * kInvQe;
      }
      for (int q = n; q <= N; q += ends ? N : M) {
        acc[(size_t)s * M + q] += R->sp[s].w * Dn * R->invV[q];
        acc[(size_t)(ns + s) * M + q] += T;
        acc[(size_t)(2 * ns + s) * M + q] += Dn;
        acc[(size_t)(3 * ns + s) * M + q] += M1;
        acc[(size_t)(4 * ns + s) * M + q] += M2;
      }
    }
  }
}

// Potential phi_n = phi_0 + sum_{m<n} g_m dx_m from g in C (shared memory,
// overwritten); summed when sampled.
template <int BLOCK>
__device__ __forceinline__ void form_potential(const RunDev* R, double* C, const double* D, double phi0,
                                               bool sample, double* wsm) {
  const int N = R->N;
  for (int n = threadIdx.x; n < N; n += BLOCK) C[n] *= D[n];
  __syncthreads();
  block_incl_scan_array(C, N, wsm);
  double* phi = R->phi;
  for (int n = threadIdx.x; n <= N; n += BLOCK) {
    double p;
    if (n == 0) p = phi0;
    else if (n == N) p = 0.0;
    else p = phi0 + C[n - 1];
    phi[n] = p;
    if (sample) R->acc[(size_t)(5 * R->ns) * (N + 1) + n] += p;
  }
}

// the energies of a sampled level (one thread)
__device__ __forceinline__ void close_sample(RunState* st, int ns) {
  st->fe = st->fe_field;
  for (int s = 0; s < ns; ++s) {
    st->ke[s] = st->ke_acc[s];
    st->ke_acc[s] = 0.0;
  }
  st->n_samples += 1;
}

// phi_0 of time level kn
__device__ __forceinline__ double electrode(const RunDev* R, long long kn) {
  if (R->bc == ECPIC_PERIODIC) return 0.0;
  const double t = (double)kn * R->dt;
  const double arg = __dadd_rn(__dmul_rn(__dmul_rn(kTwoPi, R->freq), t), R->phase);
  return R->vdc + R->v0 * sin(arg);
}

// Poisson (Eq. 4 in finite-volume form) solved through Gauss's law: with
// g_n = (phi_{n+1}-phi_n)/dx_n, Eq. 4 reads g_n - g_{n-1} = -Q_n/eps0, so
// g_n = g_0 - C_n/eps0 with C_n = sum_{m=1..n} Q_m, and the boundary values
// fix g_0 = (phi_N - phi_0 + sum_n dx_n C_n / eps0) / L.  This is the exact
// solution of the same tridiagonal system that a Thomas sweep solves.  The
// prefix sums of the fixed-point deposit are taken in 64-bit integers (exact),
// so FP64 enters only once per node.  EC field E_j = -g_j (Eq. 5).
//
// One block per run, bound by latency: the deposit, the widths and (periodic)
// the background's prefix are staged in shared memory by coalesced loads that
// travel together, and the deposit is cleared on the way; kFieldOwners threads
// then own a run of consecutive nodes each and scan all species together; the
// per-node results are formed by every thread.  FP64 is slow on this part: the
// node loop keeps its FP64 operations few.  The potential and the field energy
// are formed only on the steps that sample them (and on refresh).  Called by
// every thread of a block of at least kFieldOwners threads; `sm` holds
// field_scratch_bytes.
template <int BLOCK>
__device__ __forceinline__ void field_solve(const BatchView& b, int slot, int advance, unsigned char* sm,
                                            FieldShared& fs) {
  const RunDev* R = b.runs + slot;
  RunState* st = b.rst + slot;
  const long long step0 = st->step;
  const int N = R->N, ns = R->ns, seg0 = R->seg0, M = N + 1;
  const int se = R->sample_every;
  const bool periodic = (R->bc == ECPIC_PERIODIC);
  const bool face = R->scheme == ECPIC_SCHEME_EC || R->scheme == ECPIC_SCHEME_EC2;
  const double* dx = R->dx;
  unsigned long long* Sall = R->S;
  const double inv_L = R->inv_L;
  const int field_pm = R->field_pm, field_neg = R->field_neg;
  double* C = reinterpret_cast<double*>(sm);
  double* D = C + M;
  unsigned long long* Ss = reinterpret_cast<unsigned long long*>(D + M);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool owner = tid < kFieldOwners;
  for (int n = tid; n <= N; n += BLOCK) {
    unsigned long long v[kMaxSpecies];
#pragma unroll
    for (int s = 0; s < kMaxSpecies; ++s) v[s] = s < ns ? Sall[(size_t)s * M + n] : 0ull;
    const double d = n < N ? dx[n] : 0.0;
    const double cv = periodic && n < N ? R->cumV[n] : 0.0;
#pragma unroll
    for (int s = 0; s < kMaxSpecies; ++s)
      if (s < ns) {
        Ss[s * M + n] = v[s];
        Sall[(size_t)s * M + n] = 0ull;
      }
    D[n] = d;
    C[n] = cv;
  }
  // this thread's segment (species tid), for the size update at the end;
  // nothing changes the sizes while the field is solved
  SegState* my_ss = nullptr;
  long long my_cap = 0, my_alloc = 0;
  if (advance && tid < ns) {
    const int sg = seg0 + tid;
    my_ss = b.sst + sg;
    my_cap = b.segs[sg].cap;
    my_alloc = my_ss->n_alloc;
  }
  const long long kn = advance ? step0 + 1 : step0;
  const bool sample = advance && se > 0 && (kn % se) == 0;
  // the push of level kn samples the energy when (kn + 1) % se == 0
  const bool want_fe = !advance || (se > 0 && ((kn + 1) % se) == 0);
  const bool want_phi = !advance || sample;
  // the charge of one deposit share per species (q w 2^-32, formed on the
  // host: FP64 is slow on this part, and every thread would repeat it)
  double cw[kMaxSpecies];
#pragma unroll
  for (int s = 0; s < kMaxSpecies; ++s) cw[s] = s < ns ? R->sp[s].cw : 0.0;
  __syncthreads();

  if (tid == BLOCK - 1) fs.phi0 = electrode(R, kn);

  // C_n = sum_s q_s w_s 2^-32 * sum_{m=1..n} S_s,m, the integer prefix exact:
  // owner t has nodes [beg, end); one block scan for all species
  const int per = (M + kFieldOwners - 1) / kFieldOwners;
  const int beg = owner ? min(M, tid * per) : M, end = min(M, beg + per);
  unsigned long long run[kMaxSpecies];
#pragma unroll
  for (int s = 0; s < kMaxSpecies; ++s) {
    run[s] = 0ull;
    if (s < ns && owner) {
      unsigned long long loc = 0ull;
      for (int n = max(beg, 1); n < end; ++n) loc += Ss[s * M + n];
      const unsigned long long inc = warp_incl_scan(loc);
      if (lane == 31) fs.wtot[w][s] = inc;
      run[s] = inc - loc;
    }
  }
  __syncthreads();
  // Species whose weights q_s w_s are all equal up to sign (electrons and an
  // ion species of the same weight) take the signed integer sum of their
  // prefixes first, so that one conversion to FP64 per node serves them all:
  // C_n = cs * C'_n with cs = 2^-32 q_0 w_0 and C'_n that integer.  The sum is
  // exact while the species' totals stay below 2^63 together.
  unsigned long long tot[kMaxSpecies];
  bool pm = field_pm != 0;
  unsigned long long sum_tot = 0ull;
#pragma unroll
  for (int s = 0; s < kMaxSpecies; ++s) {
    tot[s] = 0ull;
    if (s < ns) {
      unsigned long long off = 0ull, t = 0ull;
#pragma unroll
      for (int q = 0; q < kFieldOwners / 32; ++q) {
        const unsigned long long v = fs.wtot[q][s];
        off += q < w ? v : 0ull;
        t += v;
      }
      run[s] += off;
      tot[s] = t + Ss[s * M];  // node 0 only enters the total
      pm = pm && tot[s] < (1ull << 62);
      sum_tot += tot[s] >> 2;
    }
  }
  pm = pm && sum_tot < (1ull << 61) - 4ull;
  const double cs = pm ? cw[0] : 1.0;
  // total charge (in units of cs) for the uniform neutralising background of
  // a periodic system: Q_n -= V_n Qtot / L
  double a = 0.0;
  if (periodic) {
    double qtot = 0.0;
    if (pm) {
      unsigned long long qi = 0ull;
#pragma unroll
      for (int s = 0; s < kMaxSpecies; ++s)
        if (s < ns) qi += ((field_neg >> s) & 1) ? 0ull - tot[s] : tot[s];
      qtot = (double)(long long)qi;
    } else {
#pragma unroll
      for (int s = 0; s < kMaxSpecies; ++s)
        if (s < ns) qtot += cw[s] * (double)tot[s];
    }
    a = qtot * inv_L;
  }
  double loc = 0.0;
  for (int n = beg; n < end; ++n) {
    double c = 0.0;
    unsigned long long qi = 0ull;
#pragma unroll
    for (int s = 0; s < kMaxSpecies; ++s) {
      if (s < ns) {
        if (n > 0) run[s] += Ss[s * M + n];
        if (pm)
          qi += ((field_neg >> s) & 1) ? 0ull - run[s] : run[s];
        else
          c += cw[s] * (double)run[s];
      }
    }
    if (pm) c = (double)(long long)qi;
    if (n < N) {
      if (periodic) c -= a * C[n];
      C[n] = c;
      loc += D[n] * c;
    }
  }
  const double A = cs * owners_sum(loc, fs.wsum);
  const double phi0 = fs.phi0;
  const double g0 = (A * kInvEps0 - phi0) * inv_L;
  const double kc = cs * kInvEps0;
  double fe = 0.0;
  double* gst = R->g;
  float* E = R->E;
  for (int n = tid; n < N; n += BLOCK) {
    const double gn = g0 - C[n] * kc;
    C[n] = gn;
    gst[n] = gn;
    if (face) E[n] = (float)(-gn);  // face field
    if (want_fe) fe += gn * gn * D[n];
  }
  if (!face) {
    __syncthreads();
    const double* wgt = R->mcw;
    for (int n = tid; n <= N; n += BLOCK) {
      double e;
      if (n > 0 && n < N) {
        e = -(C[n] * wgt[n] + C[n - 1] * (1.0 - wgt[n]));
      } else if (periodic) {
        e = -(C[0] * wgt[0] + C[N - 1] * (1.0 - wgt[0]));
      } else {
        e = (n == 0) ? -C[0] : -C[N - 1];
      }
      E[n] = (float)e;
    }
  }
  if (sample) sample_moments<BLOCK>(R, Ss);
  double fe_tot = 0.0;
  if (want_fe) {
    __syncthreads();  // the C of the node loop, fs.wsm free
    fe_tot = 0.5 * kEps0 * block_sum(fe, fs.wsm);
  }
  if (want_phi) {
    __syncthreads();
    form_potential<BLOCK>(R, C, D, phi0, sample, fs.wsm);
  }
  if (tid == 0) {
    st->phi0 = phi0;
    if (want_phi) st->phi_level = kn;
    if (sample) close_sample(st, ns);
    if (want_fe) st->fe_field = fe_tot;
    if (advance) st->step = kn;
  }
  if (my_ss) {
    // the step's births are kept up to the capacity; the next pass's records start empty
    const long long n = my_alloc < my_cap ? my_alloc : my_cap;
    my_ss->n_proc = n;
    my_ss->n_alloc = n;
    my_ss->n_real = 0;
    my_ss->n_imp = 0;
  }
}

}  // namespace
}  // namespace ecpic
