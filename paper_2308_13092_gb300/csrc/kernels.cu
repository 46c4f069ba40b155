// kernels.cu -- the sm_103a kernels of libecpic.
//
// One time step of every resident run is three launches (batches bound by
// latency take several steps per launch instead: steps.cuh):
//   k_pass   fused gather (Eq. 6-7, or CIC for the MC scheme) -> leapfrog
//            push (Eq. 8-9) in cell-relative FP32 -> wall absorption ->
//            null-collision MCC (Sec. 2a step 6) -> fixed-point CIC deposit
//            (Eq. 2-3) of the new positions, over all (run, species)
//            segments, load-balanced by particle count;
//   k_collide the real collisions and impacts that the pass recorded;
//   k_field  per run: charge from the deposit, Poisson (Eq. 4) in its
//            two-scan form, field (Eq. 5 or centred), potential, sampling.
// Every K steps a counting sort by cell (k_hist, k_scan, k_scatter,
// k_finalize) restores cell order and drops absorbed particles.
#include "loader.cuh"
#include "step_dev.cuh"

namespace ecpic {

namespace {

// WEIGHTED: the batch holds rebalancing runs (weight multipliers).  Their
// instance of the pass is compiled into a kernel of its own so that the
// kernel of unweighted batches keeps its register allocation.
template <bool STAGE, bool WEIGHTED>
__global__ void __launch_bounds__(kPassBlock, 4) k_pass(BatchView b, int mode, int only) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pre = reinterpret_cast<long long*>(smem_raw);
  // deposit sums, 3 (nmax+1): count, lo, hi (linear); -, lo, hi per node (EC2);
  // four when the batch has weighted runs
  uint32_t* dep = reinterpret_cast<uint32_t*>(pre + b.nseg + 1);
  const int ndep = b.weighted ? 4 : 3;
  float* Msm = reinterpret_cast<float*>(dep + ndep * (b.nmax + 1));
  unsigned char* ring = reinterpret_cast<unsigned char*>(Msm + 3 * (b.nmax + 1));  // Msm: M1 | M2 | J.E
  __shared__ PassShared sh;
  for (int i = threadIdx.x; i <= b.nmax; i += kPassBlock) {
    for (int q = 0; q < ndep; ++q) dep[q * (b.nmax + 1) + i] = 0u;
    Msm[i] = 0.0f;
    Msm[b.nmax + 1 + i] = 0.0f;
    Msm[2 * (b.nmax + 1) + i] = 0.0f;
  }
  if (threadIdx.x < kNumCtr) sh.ctr[threadIdx.x] = 0u;
  if (threadIdx.x == 0) sh.nlive = 0u;
  // the work is split in quads of particles, equal quads per CTA
  const long long T = seg_prefix(b, mode, only, pre, sh.wsm, 4);
  if (T == 0) return;
  const long long lo = T * (long long)blockIdx.x / gridDim.x;
  const long long hi = T * (long long)(blockIdx.x + 1) / gridDim.x;
  if (lo >= hi) return;
  for (int s = seg_find(pre, b.nseg, lo); s < b.nseg && pre[s] < hi; ++s) {
    const long long beg = max(lo, pre[s]) - pre[s];
    const long long end = min(hi, pre[s + 1]) - pre[s];
    if (beg >= end) continue;
    if (!chk(b.segs[s].run >= 0 && b.segs[s].run < b.max_slots, 23, s, b.nseg)) continue;
    // which instance: a sampled step of a stepping pass
    const SegDev& G = b.segs[s];
    const RunDev& R = b.runs[G.run];
    const bool stepping = mode == MODE_STEP;
    const long long k = b.rst[G.run].step;
    const bool smp = stepping && R.sample_every > 0 && ((k + 1) % R.sample_every) == 0;
    const PieceState ps{b.sst[s].cur, b.sst[s].n_proc, k};
    if (R.scheme >= ECPIC_SCHEME_EC2)  // EC2, MC2
      pass_piece<2, STAGE, kPassBlock, false>(b, &R, G, s, ps, beg, end, mode, dep, Msm, ring, sh);
    else if (WEIGHTED && R.rb && smp)  // weight multipliers
      pass_piece<WEIGHTED ? 4 : 1, STAGE, kPassBlock, false>(b, &R, G, s, ps, beg, end, mode, dep, Msm, ring, sh);
    else if (WEIGHTED && R.rb)
      pass_piece<WEIGHTED ? 3 : 0, STAGE, kPassBlock, false>(b, &R, G, s, ps, beg, end, mode, dep, Msm, ring, sh);
    else if (smp)
      pass_piece<1, STAGE, kPassBlock, false>(b, &R, G, s, ps, beg, end, mode, dep, Msm, ring, sh);
    else
      pass_piece<0, STAGE, kPassBlock, false>(b, &R, G, s, ps, beg, end, mode, dep, Msm, ring, sh);
  }
}

// Real collisions recorded by this step's pass, then its impact records,
// all segments, equal records per warp.  Process counters are summed over the lanes that share a
// (segment, process) before one atomic each.
__global__ void __launch_bounds__(kCollideBlock) k_collide(BatchView b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pre = reinterpret_cast<long long*>(smem_raw);
  int* meta = reinterpret_cast<int*>(pre + b.nseg + 1);  // slot, buffer, reals per segment
  __shared__ long long wsm[32];
  const long long T = seg_prefix(b, MODE_STEP, -1, pre, wsm, 1, true, meta);
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * kCollideBlock;
  for (long long w0 = (long long)blockIdx.x * kCollideBlock + (threadIdx.x & ~31); w0 < T; w0 += stride) {
    const long long r = w0 + lane;
    const bool valid = r < T;
    int s = 0, slot = 0, cur = 0;
    RealRec rec;
    rec.chosen = -1;
    int imp_i = -1;  // an impact record instead: the absorbed ion's index
    if (valid) {
      s = seg_find(pre, b.nseg, r);
      slot = meta[3 * s];
      cur = meta[3 * s + 1];
      const long long j = r - pre[s];
      const long long nr = meta[3 * s + 2];
      if (j >= nr) {
        const long long ii = j - nr;
        if (ii < b.segs[s].imp_cap) imp_i = b.segs[s].imp[ii];
      } else if (chk(j >= 0 && j < b.segs[s].real_cap, 25, j, b.segs[s].real_cap)) {
        const int4* src = reinterpret_cast<const int4*>(b.segs[s].real + j);  // RealRec field order
        const int4 w0 = src[0], w1 = src[1], w2 = src[2];
        rec.id = (uint64_t)(uint32_t)w0.x | ((uint64_t)(uint32_t)w0.y << 32);
        rec.i = w0.z;
        rec.chosen = w0.w;
        rec.En = __int_as_float(w1.x);
        rec.gm = __int_as_float(w1.y);
        rec.vx = __int_as_float(w1.z);
        rec.vy = __int_as_float(w1.w);
        rec.vz = __int_as_float(w2.x);
        rec.c = w2.y;
        rec.f = __int_as_float(w2.z);
        rec.k = (unsigned)w2.w;
      }
    }
    const bool ok = valid && rec.chosen >= 0 && rec.chosen < kMaxProc;
    const unsigned key = ok ? ((unsigned)s << 4) | (unsigned)rec.chosen : 0xFFFFFFFFu;
    const unsigned grp = __match_any_sync(kFull, key);
    if (ok && lane == __ffs(grp) - 1) {
      const SegDev& G = b.segs[s];
      atomicAdd(&b.rst[slot].ctr[G.species][C_COLL0 + rec.chosen], (unsigned long long)__popc(grp));
    }
    if (ok) {
      const long long k = b.rst[slot].step;
      const int se = b.runs[slot].sample_every;
      collide_real<false>(b, nullptr, s, slot, cur, k, se > 0 && ((k + 1) % se) == 0, rec);
    }
    if (imp_i >= 0) tally_impact(b, s, slot, cur, imp_i);
  }
}

// The field solve (field_solve), one CTA per run.
__global__ void __launch_bounds__(kFieldBlock, 2) k_field(BatchView b, int advance, int only) {
  const int slot = blockIdx.x;
  if (slot >= b.max_slots) return;
  const RunDev* R = b.runs + slot;
  RunState* st = b.rst + slot;
  // every scalar of the decision, loaded before the first branch so that the
  // loads travel together
  const int active = R->active;
  const int status0 = st->status;
  const int fresh = st->fresh;
  const long long step0 = st->step, step_end = st->step_end;
  if (!active) return;
  if (advance) {
    if (status0 != 0 || step0 >= step_end) return;
  } else if ((only >= 0 && slot != only) || (only == kOnlyFresh && !fresh)) {
    return;
  }
  if (only == kOnlyFresh) {
    __syncthreads();  // every thread has read the flag
    if (threadIdx.x == 0) st->fresh = 0;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FieldShared fs;
  field_solve<kFieldBlock>(b, slot, advance, smem_raw, fs);
}

// potential of the current field of one run from the stored g (host reads)
__global__ void __launch_bounds__(kFieldBlock) k_phi(BatchView b, int slot) {
  const RunDev* R = b.runs + slot;
  if (!R->active) return;
  RunState* st = b.rst + slot;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* C = reinterpret_cast<double*>(smem_raw);
  __shared__ double dsm[32];
  const int N = R->N;
  for (int n = threadIdx.x; n < N; n += kFieldBlock) C[n] = R->g[n] * R->dx[n];
  __syncthreads();
  block_incl_scan_array(C, N, dsm);
  const double phi0 = st->phi0;
  for (int n = threadIdx.x; n <= N; n += kFieldBlock)
    R->phi[n] = (n == 0) ? phi0 : (n == N ? 0.0 : phi0 + C[n - 1]);
  if (threadIdx.x == 0) st->phi_level = st->step;
}

// ----------------------------------------------------------------- sort
__global__ void __launch_bounds__(kPassBlock) k_hist(BatchView b, int mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pre = reinterpret_cast<long long*>(smem_raw);
  int* H = reinterpret_cast<int*>(pre + b.nseg + 1);
  __shared__ long long wsm[32];
  __shared__ int lohi[2];
  for (int i = threadIdx.x; i <= b.nmax; i += kPassBlock) H[i] = 0;
  if (threadIdx.x == 0) {
    lohi[0] = INT_MAX;
    lohi[1] = -1;
  }
  // quads of four particles per thread, as in the pass
  const long long T = seg_prefix(b, mode, -1, pre, wsm, 4);
  if (T == 0) return;
  const long long lo = T * (long long)blockIdx.x / gridDim.x;
  const long long hi = T * (long long)(blockIdx.x + 1) / gridDim.x;
  if (lo >= hi) return;
  const int lane = threadIdx.x & 31;
  for (int s = seg_find(pre, b.nseg, lo); s < b.nseg && pre[s] < hi; ++s) {
    const long long beg = max(lo, pre[s]) - pre[s];
    const long long end = min(hi, pre[s + 1]) - pre[s];
    if (beg >= end) continue;
    const SegDev& G = b.segs[s];
    const int32_t* pc = G.cell[b.sst[s].cur];
    const long long n = b.sst[s].n_proc;
    const int Nr = b.runs[G.run].N;
    int my_lo = INT_MAX, my_hi = -1;
    for (long long base = beg + (long long)(threadIdx.x & ~31); base < end; base += kPassBlock) {
      const long long i0 = 4 * (base + lane);
      int c[4];
      if (base + lane < end && i0 + 3 < n && chk(i0 + 3 < G.cap, 26, i0, G.cap)) {
        const int4 c4 = *reinterpret_cast<const int4*>(pc + i0);
        c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = (base + lane < end && i0 + j < n) ? pc[i0 + j] : -1;
      }
      // a thread's consecutive particles in one cell (most quads of sorted
      // data) are counted together: one shared atomic per run of equal cells
      int cur = -1, cnt = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int cj = c[j] < Nr ? c[j] : -1;
        if (cj >= 0) {
          my_lo = min(my_lo, cj);
          my_hi = max(my_hi, cj);
        }
        if (cj != cur) {
          if (cur >= 0 && chk(cur <= b.nmax, 9, cur, b.nmax)) atomicAdd(H + cur, cnt);
          cur = cj;
          cnt = 0;
        }
        ++cnt;
      }
      if (cur >= 0 && chk(cur <= b.nmax, 9, cur, b.nmax)) atomicAdd(H + cur, cnt);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      my_lo = min(my_lo, __shfl_xor_sync(kFull, my_lo, o));
      my_hi = max(my_hi, __shfl_xor_sync(kFull, my_hi, o));
    }
    if (lane == 0 && my_hi >= 0) {
      atomicMin(&lohi[0], my_lo);
      atomicMax(&lohi[1], my_hi);
    }
    __syncthreads();
    const int flo = lohi[0], fhi = lohi[1];
    const int nbeg = flo <= fhi ? flo + (int)threadIdx.x : fhi + 1;  // empty range: skip
    for (int n = nbeg; n <= fhi; n += kPassBlock) {
      const int v = H[n];
      if (v) {
        atomicAdd(b.hist + G.hoff + n, v);
        H[n] = 0;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      lohi[0] = INT_MAX;
      lohi[1] = -1;
    }
    __syncthreads();
  }
}

// per segment: counts -> exclusive cursors; live total
__global__ void __launch_bounds__(kPassBlock) k_scan(BatchView b, int mode) {
  const int s = blockIdx.x;
  if (s >= b.nseg) return;
  const SegDev& G = b.segs[s];
  const int slot = G.run;
  if (!run_live(b.runs[slot], b.rst[slot], mode, -1, slot)) return;
  __shared__ long long wsm[32];
  const int N = b.runs[slot].N;
  int* h = b.hist + G.hoff;
  const int per = (N + kPassBlock - 1) / kPassBlock;
  const int beg = min(N, (int)threadIdx.x * per), end = min(N, beg + per);
  long long loc = 0;
  for (int i = beg; i < end; ++i) loc += h[i];
  long long total;
  long long run = block_excl_scan(loc, wsm, &total);
  for (int i = beg; i < end; ++i) {
    const int c = h[i];
    h[i] = (int)run;
    run += c;
  }
  if (threadIdx.x == 0) b.sst[s].n_live = total;
}

// Counting-sort scatter (the order within a cell is not kept), one CTA
// iteration of kScatQ particles at a time: the chunk's cells are counted in
// shared memory (a range [clo, chi] of its run's cells), each cell present
// reserves its slice of the destination with one global atomic per CTA
// iteration, the records are staged in shared memory in cell order, and
// consecutive threads then write consecutive destinations of each cell, so
// the stores fill whole sectors.  The next iteration's source records are
// prefetched into L2.  Launched as one wave (scatter_grid).
constexpr int kScatQ = 4 * kPassBlock;  // particles per CTA iteration

size_t scatter_smem_bytes(int nseg, int nmax) {
  return sizeof(long long) * (size_t)(nseg + 1) +
         (size_t)kScatQ * (sizeof(unsigned long long) + 6 * sizeof(int)) +
         3 * sizeof(int) * (size_t)(nmax + 1);
}

__global__ void __launch_bounds__(kPassBlock) k_scatter(BatchView b, int mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pre = reinterpret_cast<long long*>(smem_raw);
  unsigned long long* st_id = reinterpret_cast<unsigned long long*>(pre + b.nseg + 1);
  int* st_c = reinterpret_cast<int*>(st_id + kScatQ);
  float* st_x = reinterpret_cast<float*>(st_c + kScatQ);
  float* st_u = st_x + kScatQ;
  float* st_v = st_u + kScatQ;
  float* st_w = st_v + kScatQ;
  uint32_t* st_k = reinterpret_cast<uint32_t*>(st_w + kScatQ);
  const int M = b.nmax + 1;
  int* cnt = reinterpret_cast<int*>(st_k + kScatQ);  // per cell of the chunk's range
  int* lpre = cnt + M;                               // its exclusive prefix
  int* gbase = lpre + M;                             // its reserved destination
  __shared__ long long wsm[32];
  __shared__ int wsi[32];
  __shared__ int lohi[2];
  for (int i = threadIdx.x; i < M; i += kPassBlock) cnt[i] = 0;
  if (threadIdx.x == 0) {
    lohi[0] = INT_MAX;
    lohi[1] = -1;
  }
  const long long T = seg_prefix(b, mode, -1, pre, wsm, 4);  // ends with a barrier
  if (T == 0) return;
  const long long lo = T * (long long)blockIdx.x / gridDim.x;
  const long long hi = T * (long long)(blockIdx.x + 1) / gridDim.x;
  if (lo >= hi) return;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  for (int s = seg_find(pre, b.nseg, lo); s < b.nseg && pre[s] < hi; ++s) {
    const long long beg = max(lo, pre[s]) - pre[s];
    const long long end = min(hi, pre[s + 1]) - pre[s];
    if (beg >= end) continue;
    const SegDev& G = b.segs[s];
    const int src = b.sst[s].cur, dst = src ^ 1;
    const long long n = b.sst[s].n_proc;
    int* cursor = b.hist + G.hoff;
    const int Nr = b.runs[G.run].N;
    const int32_t* sc = G.cell[src];
    const float* sx = G.xi[src];
    const float* su = G.vx[src];
    const float* sv = G.vy[src];
    const float* sw = G.vz[src];
    const uint64_t* si = G.id[src];
    const uint32_t* sk = G.wt[src];  // weight multipliers (rebalancing runs)
    int32_t* dc = G.cell[dst];
    float* dx_ = G.xi[dst];
    float* du = G.vx[dst];
    float* dv = G.vy[dst];
    float* dw = G.vz[dst];
    uint64_t* di = G.id[dst];
    uint32_t* dk = G.wt[dst];
    // block-uniform trip count: the barriers below need every thread
    for (long long base = beg; base < end; base += kPassBlock) {
      if (threadIdx.x == 0) {
        const long long nb = base + kPassBlock;
        if (nb < end) {
          const long long p0 = 4 * nb;
          const long long p1 = min(4 * min(end, nb + kPassBlock), n);
          if (p1 > p0) {
            const unsigned b4 = (unsigned)(((p1 - p0) * 4) & ~15ll);
            if (b4) {
              l2_prefetch(sc + p0, b4);
              l2_prefetch(sx + p0, b4);
              l2_prefetch(su + p0, b4);
              l2_prefetch(sv + p0, b4);
              l2_prefetch(sw + p0, b4);
              l2_prefetch(si + p0, (unsigned)(((p1 - p0) * 8) & ~15ll));
              if (sk) l2_prefetch(sk + p0, b4);
            }
          }
        }
      }
      const long long q = base + threadIdx.x;
      const long long i0 = 4 * q;
      int c[4];
      float x[4], u[4], v[4], w[4];
      uint64_t id[4];
      unsigned kq[4] = {1u, 1u, 1u, 1u};
      if (q < end && i0 + 3 < n && chk(i0 + 3 < G.cap, 27, i0, G.cap)) {
        const int4 c4 = *reinterpret_cast<const int4*>(sc + i0);
        const float4 x4 = *reinterpret_cast<const float4*>(sx + i0);
        const float4 u4 = *reinterpret_cast<const float4*>(su + i0);
        const float4 v4 = *reinterpret_cast<const float4*>(sv + i0);
        const float4 w4 = *reinterpret_cast<const float4*>(sw + i0);
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(si + i0);
        const ulonglong2 a2 = *reinterpret_cast<const ulonglong2*>(si + i0 + 2);
        c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
        x[0] = x4.x; x[1] = x4.y; x[2] = x4.z; x[3] = x4.w;
        u[0] = u4.x; u[1] = u4.y; u[2] = u4.z; u[3] = u4.w;
        v[0] = v4.x; v[1] = v4.y; v[2] = v4.z; v[3] = v4.w;
        w[0] = w4.x; w[1] = w4.y; w[2] = w4.z; w[3] = w4.w;
        id[0] = a.x; id[1] = a.y; id[2] = a2.x; id[3] = a2.y;
        if (sk) {
          const uint4 k4 = *reinterpret_cast<const uint4*>(sk + i0);
          kq[0] = k4.x; kq[1] = k4.y; kq[2] = k4.z; kq[3] = k4.w;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool in = q < end && i0 + j < n && chk(i0 + j < G.cap, 27, i0 + j, G.cap);
          c[j] = in ? sc[i0 + j] : -1;
          x[j] = in ? sx[i0 + j] : 0.f;
          u[j] = in ? su[i0 + j] : 0.f;
          v[j] = in ? sv[i0 + j] : 0.f;
          w[j] = in ? sw[i0 + j] : 0.f;
          id[j] = in ? si[i0 + j] : 0ull;
          if (sk && in) kq[j] = sk[i0 + j];
        }
      }
      // the chunk's cell range (absorbed particles, cell < 0, are dropped)
      int my_lo = INT_MAX, my_hi = -1;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        c[j] = c[j] < Nr ? c[j] : -1;
        if (c[j] >= 0) {
          my_lo = min(my_lo, c[j]);
          my_hi = max(my_hi, c[j]);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        my_lo = min(my_lo, __shfl_xor_sync(kFull, my_lo, o));
        my_hi = max(my_hi, __shfl_xor_sync(kFull, my_hi, o));
      }
      if (lane == 0 && my_hi >= 0) {
        atomicMin(&lohi[0], my_lo);
        atomicMax(&lohi[1], my_hi);
      }
      __syncthreads();
      const int clo = lohi[0], chi = lohi[1];
      const int R = chi >= clo ? chi - clo + 1 : 0;
      // rank of each particle among the chunk's particles of its cell
      int r[4] = {0, 0, 0, 0};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const unsigned grp = __match_any_sync(kFull, c[j] >= 0 ? (unsigned)c[j] : 0xFFFFFFFFu);
        if (c[j] >= 0 && chk(c[j] - clo < M, 28, c[j] - clo, M)) {
          const int leader = __ffs(grp) - 1;
          int b0 = 0;
          if (lane == leader) b0 = atomicAdd(cnt + (c[j] - clo), __popc(grp));
          b0 = __shfl_sync(grp, b0, leader);
          r[j] = b0 + __popc(grp & lt);
        }
      }
      __syncthreads();
      // local prefix of the range's counts; each cell present reserves its
      // destination slice
      const int per = (R + kPassBlock - 1) / kPassBlock;
      const int kb = min(R, (int)threadIdx.x * per), ke = min(R, kb + per);
      int loc = 0;
      for (int k = kb; k < ke; ++k) loc += cnt[k];
      int m;
      int run = block_excl_scan(loc, wsi, &m);
      for (int k = kb; k < ke; ++k) {
        const int ck = cnt[k];
        lpre[k] = run;
        run += ck;
        gbase[k] = ck ? atomicAdd(cursor + clo + k, ck) : 0;
      }
      __syncthreads();
      // stage in cell order
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (c[j] < 0) continue;
        const int p = lpre[c[j] - clo] + r[j];
        if (!chk(p >= 0 && p < kScatQ, 29, p, kScatQ)) continue;
        st_c[p] = c[j];
        st_x[p] = x[j];
        st_u[p] = u[j];
        st_v[p] = v[j];
        st_w[p] = w[j];
        st_id[p] = id[j];
        st_k[p] = kq[j];
      }
      __syncthreads();
      for (int t = threadIdx.x; t < m; t += kPassBlock) {
        const int cc = st_c[t];
        const int k = cc - clo;
        const long long d = (long long)gbase[k] + (t - lpre[k]);
        if (!chk(d >= 0 && d < G.cap, 10, d, G.cap)) continue;
        dc[d] = cc;
        dx_[d] = st_x[t];
        du[d] = st_u[t];
        dv[d] = st_v[t];
        dw[d] = st_w[t];
        di[d] = st_id[t];
        if (dk) dk[d] = st_k[t];
      }
      for (int k = threadIdx.x; k < R; k += kPassBlock) cnt[k] = 0;
      if (threadIdx.x == 0) {
        lohi[0] = INT_MAX;
        lohi[1] = -1;
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(kPassBlock) k_finalize(BatchView b) {
  // (the counting sort's last phase; rebalancing ends with k_rb_finalize)
  const int s = blockIdx.x;
  if (s >= b.nseg) return;
  const SegDev& G = b.segs[s];
  const int slot = G.run;
  if (!run_live(b.runs[slot], b.rst[slot], MODE_SORT, -1, slot)) return;
  const int N = b.runs[slot].N;
  for (int i = threadIdx.x; i < N; i += kPassBlock) b.hist[G.hoff + i] = 0;
  if (threadIdx.x == 0) {
    SegState* ss = b.sst + s;
    ss->cur ^= 1;
    ss->n_proc = ss->n_live;
    ss->n_alloc = ss->n_live;
    ss->n_dead = 0;
  }
}

// ----------------------------------------------------------------- rebalancing
// Particle rebalancing (Sec. 3d proposes keeping the particles per cell near a
// target on non-uniform grids; the rule is this library's design, the same as
// the oracle's).  It runs for the runs due at their current level (after the
// field kernel of that level): a counting sort by cell into the other buffer
// set (k_hist, k_scan, k_scatter in MODE_REBAL), then per (segment, cell):
//   - more than rb_hi particles (at most kRbMaxCell): order them by (vx, id),
//     cut the order into floor(n/4) groups of four, merge the
//     G = min(floor(n/4), ceil((n - target)/2)) groups nearest the middle of
//     the order (ties: the slower), skipping groups heavier than
//     kRbMaxWeight; a group becomes two particles at its weighted centroid
//     with velocities u + sqrt(b/a) d, u - sqrt(a/b) d (u the mean velocity,
//     d the per-component standard deviations with Philox signs for y and z,
//     a = ceil(W/2), b = W - a), taking the group's two smallest ids;
//   - fewer than rb_lo (and some): split the min(target - n, #{k >= 2})
//     heaviest (ties: smallest id) in place into ceil(k/2) (same id) and
//     floor(k/2) (id child_id(id, level, 3));
//   - otherwise copied.
// k_rb_classify lists the cells that merge or split and counts the others,
// k_rb_cells counts each listed cell's output, k_rb_scan places the cells,
// k_rb_copy streams the unchanged cells' particles back into the current
// buffer set and k_rb_cells writes the listed cells there, k_rb_finalize and
// k_rb_mark set the sizes and the run's rebalancing level.
constexpr int kRbBlock = 256;
constexpr int kRbListCells = 4096;  // list entry = segment * kRbListCells + cell
constexpr int kRbGroups = kRbMaxCell / 4;

struct RbSmem {
  unsigned long long k2[kRbMaxCell];  // second key: id
  uint32_t k1[kRbMaxCell];            // first key: monotone vx bits, or ~k
  uint16_t ix[kRbMaxCell];            // index within the cell
  uint16_t pref[kRbGroups];           // eligible groups before each order position
  uint8_t el[kRbGroups];              // group at an order position may merge
  unsigned kmax;                      // the cell's largest weight multiplier
};

// FP32 bits ordered like the values (+0 and -0 as one value)
__device__ __forceinline__ uint32_t rb_fkey(float v) {
  const uint32_t u = __float_as_uint(v == 0.0f ? 0.0f : v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ascending bitonic sort of P (a power of two) entries by (k1, k2)
__device__ void rb_bitonic(RbSmem& sm, int P) {
  for (int size = 2; size <= P; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < (P >> 1); t += blockDim.x) {
        const int i = 2 * stride * (t / stride) + (t % stride);
        const int j = i + stride;
        const bool up = (i & size) == 0;
        const bool gt = sm.k1[i] > sm.k1[j] || (sm.k1[i] == sm.k1[j] && sm.k2[i] > sm.k2[j]);
        if (gt == up) {
          const uint32_t a = sm.k1[i]; sm.k1[i] = sm.k1[j]; sm.k1[j] = a;
          const unsigned long long c = sm.k2[i]; sm.k2[i] = sm.k2[j]; sm.k2[j] = c;
          const uint16_t x = sm.ix[i]; sm.ix[i] = sm.ix[j]; sm.ix[j] = x;
        }
      }
      __syncthreads();
    }
}

// order position of merge group g among ng groups: by distance from the
// middle of the velocity order, the slower group first on a tie
__device__ __forceinline__ int rb_pos(int g, int ng) {
  const int d = 2 * g - (ng - 1);
  return (d < 0 ? -d : d) - (d < 0 ? 1 : 0);
}

__device__ __forceinline__ void rb_copy(const SegDev& G, int in, int out, long long i, long long o) {
  G.cell[out][o] = G.cell[in][i];
  G.xi[out][o] = G.xi[in][i];
  G.vx[out][o] = G.vx[in][i];
  G.vy[out][o] = G.vy[in][i];
  G.vz[out][o] = G.vz[in][i];
  G.id[out][o] = G.id[in][i];
  G.wt[out][o] = G.wt[in][i];
}

// One cell: the particles [start, start + n) of buffer set `in` (sorted by
// cell).  Returns the cell's output count; when write, the output goes to
// buffer set `out` from position obase and the counters are updated.  Every
// thread of the block calls it (block-uniform arguments).
__device__ int rb_cell(const BatchView& b, int s, int c, long long start, int n, bool write,
                       long long obase, RbSmem& sm, long long* wsm) {
  const SegDev& G = b.segs[s];
  const int slot = G.run, sp = G.species;
  const RunDev* R = b.runs + slot;
  RunState* st = b.rst + slot;
  const int out = b.sst[s].cur, in = out ^ 1;
  const int T = R->rb_target;
  int mode = 0;  // 0 copy, 1 merge, 2 split, 3 skip (copy, counted)
  if (n > R->rb_hi) mode = n > kRbMaxCell ? 3 : 1;
  else if (n > 0 && n < R->rb_lo) mode = 2;
  const int tid = threadIdx.x;
  if (mode == 2) {
    long long heavy = 0;
    for (int t = tid; t < n; t += blockDim.x) heavy += G.wt[in][start + t] >= 2u ? 1 : 0;
    heavy = block_sum(heavy, wsm);
    const int S = (int)min((long long)(T - n), heavy);
    if (S <= 0) {
      mode = 0;
    } else {
      if (!write) return n + S;
      int P = 1;
      while (P < n) P <<= 1;
      for (int t = tid; t < P; t += blockDim.x) {
        if (t < n) {
          sm.k1[t] = ~G.wt[in][start + t];  // heaviest first
          sm.k2[t] = G.id[in][start + t];
          sm.ix[t] = (uint16_t)t;
        } else {
          sm.k1[t] = 0xFFFFFFFFu;
          sm.k2[t] = ~0ull;
          sm.ix[t] = 0;
        }
      }
      __syncthreads();
      rb_bitonic(sm, P);
      const long long k_lvl = st->step;
      for (int t = tid; t < n; t += blockDim.x) {
        const long long i = start + sm.ix[t];
        if (t < S) {
          const long long o = obase + 2 * t;
          rb_copy(G, in, out, i, o);
          rb_copy(G, in, out, i, o + 1);
          const unsigned k = G.wt[in][i];
          G.wt[out][o] = (k + 1u) / 2u;
          G.wt[out][o + 1] = k / 2u;
          G.id[out][o + 1] = child_id(G.id[in][i], k_lvl, 3);
        } else {
          rb_copy(G, in, out, i, obase + S + t);
        }
      }
      if (tid == 0) atomicAdd(&st->ctr[sp][C_RB_SPLIT], (unsigned long long)S);
      __syncthreads();
      return n + S;
    }
  }
  if (mode == 0 || mode == 3) {
    // (listed cells only: a split cell with nothing to split)
    if (write)
      for (int t = tid; t < n; t += blockDim.x) rb_copy(G, in, out, start + t, obase + t);
    return n;
  }
  // merge: order by (vx, id), groups of four, the ones nearest the middle
  const int ng = n / 4;
  const int Gw = min(ng, (n - T + 1) / 2);
  if (!write) {
    // with no multiplier above kRbMaxWeight / 4 every group is eligible
    // (W <= kRbMaxWeight), so the count needs no ordering
    if (tid == 0) sm.kmax = 0u;
    __syncthreads();
    unsigned km = 0u;
    for (int t = tid; t < n; t += blockDim.x) km = max(km, G.wt[in][start + t]);
    km = __reduce_max_sync(0xFFFFFFFFu, km);
    if ((tid & 31) == 0) atomicMax(&sm.kmax, km);
    __syncthreads();
    const unsigned kmax = sm.kmax;
    __syncthreads();  // every thread has read it before the next cell resets it
    if (kmax <= kRbMaxWeight / 4u) return n - 2 * Gw;
  }
  int P = 1;
  while (P < n) P <<= 1;
  for (int t = tid; t < P; t += blockDim.x) {
    if (t < n) {
      sm.k1[t] = rb_fkey(G.vx[in][start + t]);
      sm.k2[t] = G.id[in][start + t];
      sm.ix[t] = (uint16_t)t;
    } else {
      sm.k1[t] = 0xFFFFFFFFu;
      sm.k2[t] = ~0ull;
      sm.ix[t] = 0;
    }
  }
  __syncthreads();
  rb_bitonic(sm, P);
  for (int g = tid; g < ng; g += blockDim.x) {
    unsigned W = 0u;
    for (int q = 0; q < 4; ++q) W += G.wt[in][start + sm.ix[4 * g + q]];
    sm.el[rb_pos(g, ng)] = W <= kRbMaxWeight ? 1 : 0;
  }
  __syncthreads();
  // eligible groups before each order position (block scan; ng <= 1024)
  {
    const int per = (ng + blockDim.x - 1) / blockDim.x;
    const int a = min(ng, tid * per), e = min(ng, a + per);
    long long loc = 0;
    for (int q = a; q < e; ++q) loc += sm.el[q];
    long long tot;
    long long run = block_excl_scan(loc, wsm, &tot);
    for (int q = a; q < e; ++q) {
      sm.pref[q] = (uint16_t)run;
      run += sm.el[q];
    }
    __syncthreads();
    const int chosen = (int)min((long long)Gw, tot);
    if (!write) return n - 2 * chosen;
  }
  // output offsets: a chosen group's first particle emits two, its others
  // none, every other particle one.  They are scanned in shared memory (the
  // sort keys are no longer needed), so that consecutive threads take
  // consecutive order positions and their stores coalesce.
  auto emits = [&](int t) -> int {
    const int g = t / 4;
    if (g >= ng) return 1;
    const int ps = rb_pos(g, ng);
    const bool ch = sm.el[ps] && (int)sm.pref[ps] < Gw;
    return ch ? ((t & 3) == 0 ? 2 : 0) : 1;
  };
  long long* opos = reinterpret_cast<long long*>(sm.k2);
  for (int t = tid; t < n; t += blockDim.x) opos[t] = emits(t);
  __syncthreads();
  block_incl_scan_array(opos, n, wsm);
  const long long tot = opos[n - 1];
  const long long k_lvl = st->step;
  unsigned long long merged = 0;
  // single particles: consecutive threads, consecutive positions
  for (int t = tid; t < n; t += blockDim.x)
    if (emits(t) == 1) rb_copy(G, in, out, start + sm.ix[t], obase + opos[t] - 1);
  // chosen groups, one per thread (the FP64 merge arithmetic is a long
  // dependent chain on this part's slow FP64 pipe: spread it over the block)
  for (int g = tid; g < ng; g += blockDim.x) {
    const int t = 4 * g;
    if (emits(t) != 2) continue;
    const long long pos = opos[t] - 2;
    {
      // the group's weighted centroid, mean velocity and spreads (FP64)
      double W = 0.0, X = 0.0, u[3] = {0.0, 0.0, 0.0}, m2[3] = {0.0, 0.0, 0.0};
      unsigned Wi = 0u;
      unsigned long long id0 = ~0ull, id1 = ~0ull;
      long long ii[4];
      for (int q = 0; q < 4; ++q) {
        const long long i = start + sm.ix[t + q];
        ii[q] = i;
        const unsigned k = G.wt[in][i];
        const double kd = (double)k;
        Wi += k;
        W += kd;
        X += kd * (double)G.xi[in][i];
        u[0] += kd * (double)G.vx[in][i];
        u[1] += kd * (double)G.vy[in][i];
        u[2] += kd * (double)G.vz[in][i];
        const unsigned long long id = G.id[in][i];
        if (id < id0) { id1 = id0; id0 = id; } else if (id < id1) { id1 = id; }
      }
      X /= W;
      for (int q = 0; q < 3; ++q) u[q] /= W;
      for (int q = 0; q < 4; ++q) {
        const long long i = ii[q];
        const double kd = (double)G.wt[in][i];
        const double dv[3] = {(double)G.vx[in][i] - u[0], (double)G.vy[in][i] - u[1],
                              (double)G.vz[in][i] - u[2]};
        for (int r = 0; r < 3; ++r) m2[r] += kd * dv[r] * dv[r];
      }
      const uint4 A = draw(R->seed, id0, (uint32_t)k_lvl, ((uint32_t)sp << 8) | 0x10u);
      double d[3] = {sqrt(m2[0] / W), sqrt(m2[1] / W), sqrt(m2[2] / W)};
      if (A.x & 1u) d[1] = -d[1];
      if (A.x & 2u) d[2] = -d[2];
      const unsigned ka = (Wi + 1u) / 2u, kb = Wi - ka;
      const double fa = sqrt((double)kb / (double)ka), fb = sqrt((double)ka / (double)kb);
      float xc = (float)X;
      if (xc >= 1.0f) xc = 0.99999994f;  // the centroid lies in the cell
      const long long o = obase + pos;
      const int cc = G.cell[in][ii[0]];
      G.cell[out][o] = cc;
      G.cell[out][o + 1] = cc;
      G.xi[out][o] = xc;
      G.xi[out][o + 1] = xc;
      G.vx[out][o] = (float)(u[0] + fa * d[0]);
      G.vy[out][o] = (float)(u[1] + fa * d[1]);
      G.vz[out][o] = (float)(u[2] + fa * d[2]);
      G.vx[out][o + 1] = (float)(u[0] - fb * d[0]);
      G.vy[out][o + 1] = (float)(u[1] - fb * d[1]);
      G.vz[out][o + 1] = (float)(u[2] - fb * d[2]);
      G.id[out][o] = id0;
      G.id[out][o + 1] = id1;
      G.wt[out][o] = ka;
      G.wt[out][o + 1] = kb;
      ++merged;
    }
  }
  merged = warp_sum(merged);
  if ((tid & 31) == 0 && merged) atomicAdd(&st->ctr[sp][C_RB_MERGED], merged);
  __syncthreads();
  return (int)tot;
}

// Per (segment, cell) of a due run, one thread: a cell that merges or splits
// (more than rb_hi particles, at most kRbMaxCell; fewer than rb_lo) goes on
// the list for k_rb_cells; the others keep their particles, so their output
// count is their count and k_rb_copy moves them (mode 0; 2: above kRbMaxCell,
// counted as skipped).
__global__ void __launch_bounds__(kPassBlock) k_rb_classify(BatchView b) {
  const int s = blockIdx.y;
  const int c = blockIdx.x * kPassBlock + threadIdx.x;
  if (s >= b.nseg) return;
  const SegDev& G = b.segs[s];
  const int slot = G.run;
  const RunDev& R = b.runs[slot];
  if (!run_live(R, b.rst[slot], MODE_REBAL, -1, slot) || c >= R.N || c >= kRbListCells) return;
  const int* h = b.hist + G.hoff;  // after the scatter: the end of each cell
  const int n = h[c] - (c > 0 ? h[c - 1] : 0);
  const bool listed = (n > R.rb_hi && n <= kRbMaxCell) || (n > 0 && n < R.rb_lo);
  b.rbmode[G.hoff + c] = listed ? 1 : (n > R.rb_hi ? 2 : 0);
  if (listed) {
    // at most one entry per (segment, cell): within nseg * nmax by construction
    const int k = atomicAdd(b.rbnum, 1);
    const bool fits = k < b.nseg * b.nmax;
    chk(fits, 30, k, (long long)b.nseg * b.nmax);
    if (fits) b.rblist[k] = s * kRbListCells + c;
  } else {
    b.rbcnt[G.hoff + c] = n;
  }
}

// write = 0: each listed cell's output count into rbcnt; write = 1: the
// listed cells' particles into the current buffer set at the scanned offsets
__global__ void __launch_bounds__(kRbBlock) k_rb_cells(BatchView b, int write) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RbSmem& sm = *reinterpret_cast<RbSmem*>(smem_raw);
  __shared__ long long wsm[32];
  const int num = *b.rbnum;
  for (int item = blockIdx.x; item < num; item += gridDim.x) {
    const int e = b.rblist[item];
    const int s = e / kRbListCells, c = e % kRbListCells;
    if (!chk(s >= 0 && s < b.nseg, 31, s, b.nseg)) continue;
    const SegDev& G = b.segs[s];
    if (write && b.sst[s].rb_over) continue;
    const int* h = b.hist + G.hoff;
    const long long end = h[c];
    const long long start = c > 0 ? h[c - 1] : 0;
    // (an unconditional guard: the writes below index by this range)
    if (!(start >= 0 && end >= start && end <= G.cap)) continue;
    int* oc = b.rbcnt + G.hoff;
    const int cnt = rb_cell(b, s, c, start, (int)(end - start), write != 0, write ? oc[c] : 0, sm, wsm);
    if (!write && threadIdx.x == 0) oc[c] = cnt;
  }
}

// The particles of the cells that keep them (mode 0 and 2), streamed from the
// sorted buffer set into the current one at their cell's scanned offset:
// consecutive particles of a cell, consecutive positions.  Segments of due
// runs whose plan did not overflow the capacity.
__global__ void __launch_bounds__(kPassBlock) k_rb_copy(BatchView b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pre = reinterpret_cast<long long*>(smem_raw);
  __shared__ long long wsm[32];
  {
    const int per = (b.nseg + blockDim.x - 1) / blockDim.x;
    const int s0 = threadIdx.x * per;
    long long loc = 0;
    for (int k = 0; k < per; ++k) {
      const int sg = s0 + k;
      if (sg < b.nseg) {
        const int slot = b.segs[sg].run;
        const bool due = run_live(b.runs[slot], b.rst[slot], MODE_REBAL, -1, slot) &&
                         !b.sst[sg].rb_over;
        const long long cnt = due ? b.sst[sg].n_live : 0;
        pre[sg] = cnt;
        loc += cnt;
      }
    }
    long long total;
    long long run = block_excl_scan(loc, wsm, &total);
    for (int k = 0; k < per; ++k) {
      const int sg = s0 + k;
      if (sg < b.nseg) {
        const long long cnt = pre[sg];
        pre[sg] = run;
        run += cnt;
      }
    }
    if (threadIdx.x == 0) pre[b.nseg] = total;
    __syncthreads();
  }
  const long long T = pre[b.nseg];
  if (T == 0) return;
  const long long lo = T * (long long)blockIdx.x / gridDim.x;
  const long long hi = T * (long long)(blockIdx.x + 1) / gridDim.x;
  if (lo >= hi) return;
  for (int s = seg_find(pre, b.nseg, lo); s < b.nseg && pre[s] < hi; ++s) {
    const long long beg = max(lo, pre[s]) - pre[s];
    const long long end = min(hi, pre[s + 1]) - pre[s];
    if (beg >= end) continue;
    const SegDev& G = b.segs[s];
    const int out = b.sst[s].cur, in = out ^ 1;
    const int N = b.runs[G.run].N;
    const int* h = b.hist + G.hoff;
    const int* oc = b.rbcnt + G.hoff;
    const uint8_t* md = b.rbmode + G.hoff;
    for (long long i = beg + threadIdx.x; i < end; i += blockDim.x) {
      if (!chk(i < G.cap, 32, i, G.cap)) continue;
      const int c = G.cell[in][i];
      if (!chk(c >= 0 && c < N, 33, c, N)) continue;
      if (md[c] == 1) continue;  // listed: written by k_rb_cells
      const long long o = (long long)oc[c] + (i - (c > 0 ? h[c - 1] : 0));
      // (an unconditional guard, as in k_rb_cells: the writes index by o)
      const bool ok = o >= 0 && o < G.cap;
      chk(ok, 34, o, G.cap);
      if (ok) rb_copy(G, in, out, i, o);
    }
  }
}

// per segment: output counts -> exclusive offsets; the total (capacity check)
__global__ void __launch_bounds__(kPassBlock) k_rb_scan(BatchView b) {
  const int s = blockIdx.x;
  if (s >= b.nseg) return;
  const SegDev& G = b.segs[s];
  const int slot = G.run;
  if (!run_live(b.runs[slot], b.rst[slot], MODE_REBAL, -1, slot)) return;
  __shared__ long long wsm[32];
  const int N = b.runs[slot].N;
  int* h = b.rbcnt + G.hoff;
  const int per = (N + kPassBlock - 1) / kPassBlock;
  const int beg = min(N, (int)threadIdx.x * per), end = min(N, beg + per);
  long long loc = 0;
  for (int i = beg; i < end; ++i) loc += h[i];
  long long total;
  long long run = block_excl_scan(loc, wsm, &total);
  for (int i = beg; i < end; ++i) {
    const int c = h[i];
    h[i] = (int)run;
    run += c;
  }
  if (threadIdx.x == 0) {
    b.sst[s].n_rb = total;
    b.sst[s].rb_over = total > G.cap ? 1 : 0;
  }
}

// per segment: sizes after the rebalancing (or, if the plan overflowed the
// capacity, the sorted particles unchanged); cell arrays cleared
__global__ void __launch_bounds__(kPassBlock) k_rb_finalize(BatchView b) {
  const int s = blockIdx.x;
  if (s >= b.nseg) return;
  const SegDev& G = b.segs[s];
  const int slot = G.run;
  if (!run_live(b.runs[slot], b.rst[slot], MODE_REBAL, -1, slot)) return;
  const int N = b.runs[slot].N;
  const bool over = b.sst[s].rb_over != 0;
  unsigned long long skipped = 0;
  for (int i = threadIdx.x; i < N; i += kPassBlock) {
    b.hist[G.hoff + i] = 0;
    b.rbcnt[G.hoff + i] = 0;
    skipped += (!over && b.rbmode[G.hoff + i] == 2) ? 1ull : 0ull;
    b.rbmode[G.hoff + i] = 0;
  }
  skipped = warp_sum(skipped);
  if ((threadIdx.x & 31) == 0 && skipped)
    atomicAdd(&b.rst[slot].ctr[G.species][C_RB_SKIPPED], skipped);
  __syncthreads();  // every thread has read rb_over
  if (threadIdx.x == 0) {
    SegState* ss = b.sst + s;
    if (ss->rb_over) {
      ss->cur ^= 1;  // the sorted buffer set
      ss->n_proc = ss->n_live;
      ss->n_alloc = ss->n_live;
    } else {
      ss->n_proc = ss->n_rb;
      ss->n_alloc = ss->n_rb;
    }
    ss->n_dead = 0;
  }
}

// per run: the level rebalanced; a capacity overflow fails the run
__global__ void k_rb_mark(BatchView b) {
  const int slot = blockIdx.x * blockDim.x + threadIdx.x;
  if (slot >= b.max_slots) return;
  RunState* st = b.rst + slot;
  const RunDev& R = b.runs[slot];
  if (!run_live(R, *st, MODE_REBAL, -1, slot)) return;
  bool over = false;
  for (int q = 0; q < R.ns; ++q) {
    SegState* ss = b.sst + R.seg0 + q;
    over = over || ss->rb_over;
    ss->rb_over = 0;
  }
  st->rb_level = st->step;
  st->rb_force = 0;
  if (over) {
    set_status(st, ECPIC_ERR_CAPACITY);
  }
}

// ----------------------------------------------------------------- loader
// Uniform positions and Maxwellian velocities (Sec. 2b) from Philox blocks
// (id = i, step word 0xFFFFFFFF, word3 = (s<<8)|0x80 for X, |0x81 for v),
// defined in FP64 so that the cell index matches the FP64 definition exactly.
// Bound by its instructions: in FP64 throughout, some 250 of them per particle
// at 64 cycles per warp.  FP64 only for the position and where loader.cuh cannot
// tell the rounded velocity: 0.13 instead of 0.69 ms for two species of 1e6,
// 0.86 instead of 4.3 ms for 64 runs of 1e4 to 1e6 particles (1.3e7).

// velocities as defined, in FP64
__device__ __noinline__ float3 maxwellian(uint4 B, double sd) {
  const double u1a = __dmul_rn((double)B.x + 1.0, 2.3283064365386963e-10);
  const double u2a = __dmul_rn((double)B.y, 2.3283064365386963e-10);
  const double u1b = __dmul_rn((double)B.z + 1.0, 2.3283064365386963e-10);
  const double u2b = __dmul_rn((double)B.w, 2.3283064365386963e-10);
  const double ra = sqrt(__dmul_rn(-2.0, log(u1a)));
  const double rb = sqrt(__dmul_rn(-2.0, log(u1b)));
  const double aa = __dmul_rn(kTwoPi, u2a), ab = __dmul_rn(kTwoPi, u2b);
  const double z0 = __dmul_rn(ra, cos(aa)), z1 = __dmul_rn(ra, sin(aa));
  const double z2 = __dmul_rn(rb, cos(ab));
  return make_float3(__double2float_rn(__dmul_rn(sd, z0)), __double2float_rn(__dmul_rn(sd, z1)),
                     __double2float_rn(__dmul_rn(sd, z2)));
}

// t / d rounded to FP64 and then to FP32 (t >= 0, d > 0): by a reciprocal good
// to 2^-44 where that decides the float, else by the division
__device__ __forceinline__ float quotient(double t, double d) {
  const float df = (float)d;
  const double r0 = (double)__frcp_rn(df);
  const double q = t * fma(r0, fma(-d, r0, 1.0), r0);
  // the low bits' distance from the middle of two floats
  const int low = (__double2loint(q) & 0x1FFFFFFF) - 0x10000000;
  const float f = __double2float_rn(q);
  if (df > 1e-30f && df < 1e30f && f > 1e-30f && (low > 4096 || low < -4096)) return f;
  return __double2float_rn(__ddiv_rn(t, d));
}

__device__ __forceinline__ void init_run(const BatchView& b, int slot, const InitParams& p) {
  const RunDev* R = b.runs + slot;
  const int sp = blockIdx.y;
  if (sp >= R->ns) return;
  const int s = R->seg0 + sp;
  const SegDev& G = b.segs[s];
  const int cur = b.sst[s].cur;
  const int N = R->N;
  const double L = R->L;
  const double* x = R->x;
  const double* dx = R->dx;
  const double sd = p.sd[sp];
  const Pair sdp{p.sd_hi[sp], p.sd_lo[sp]};
  const long long n = p.n[sp];
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const uint4 A = draw(R->seed, (uint64_t)i, 0xFFFFFFFFu, ((uint32_t)sp << 8) | 0x80u);
    const uint4 B = draw(R->seed, (uint64_t)i, 0xFFFFFFFFu, ((uint32_t)sp << 8) | 0x81u);
    const double u = p.quiet ? __ddiv_rn((double)i + 0.5, (double)n)
                             : (double)A.x * 2.3283064365386963e-10;
    const double X = __dmul_rn(u, L);
    int lo = 0;
    if (R->uniform) {
      // the equal cells' guess, moved to the cell that holds X
      // (compared as integers, which order the doubles of one sign alike)
      lo = p.quiet ? min(N - 1, (int)(u * (double)N)) : (int)__umulhi(A.x, (unsigned)N);
      const long long Xb = __double_as_longlong(X);
      while (lo > 0 && __double_as_longlong(x[lo]) > Xb) --lo;
      while (lo + 1 < N && __double_as_longlong(x[lo + 1]) <= Xb) ++lo;
    } else {
      int hi = N;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (x[mid] <= X) lo = mid; else hi = mid;
      }
    }
    int c = lo;
    float f = quotient(__dsub_rn(X, x[c]), dx[c]);
    if (f >= 1.0f) {
      if (c + 1 < N) {
        c += 1;
        f = 0.0f;
      } else {
        f = 0.99999994f;
      }
    }
    float3 v = make_float3(0.0f, 0.0f, 0.0f);
    bool known = false;
    if (sdp.hi > 1e-15f) {  // (a cold species' zeros take their signs from FP64)
      Pair ca, sa, cb, sb;
      turn(B.y, &ca, &sa);
      turn(B.w, &cb, &sb);
      const Pair ra = radius(B.x + 1u), rb = radius(B.z + 1u);
      known = B.x != 0xFFFFFFFFu && B.z != 0xFFFFFFFFu;  // (u1 = 1: a zero radius)
      known = certain(sdp, ra, ca, &v.x) && known;
      known = certain(sdp, ra, sa, &v.y) && known;
      known = certain(sdp, rb, cb, &v.z) && known;
    }
    if (!known) v = maxwellian(B, sd);
    if (!chk(i < G.cap && c >= 0 && c < N, 11, i, G.cap)) continue;
    G.cell[cur][i] = c;
    G.xi[cur][i] = f;
    G.vx[cur][i] = v.x;
    G.vy[cur][i] = v.y;
    G.vz[cur][i] = v.z;
    G.id[cur][i] = (uint64_t)i;
    if (G.wt[cur]) G.wt[cur][i] = p.rb_m0;
  }
}

__global__ void k_init(BatchView b, int slot, InitParams p) { init_run(b, slot, p); }

// A wave of admitted runs: blockIdx.z indexes the list of slots.
__global__ void k_init_many(BatchView b, const int* slots, const InitParams* ps, int count) {
  if ((int)blockIdx.z >= count) return;
  const int slot = slots[blockIdx.z];
  if (slot < 0 || slot >= b.max_slots) return;
  init_run(b, slot, ps[blockIdx.z]);
}

// ----------------------------------------------------------------- kernel-level entry points
// Deposits of caller-owned arrays: a block takes consecutive quads, so that in
// cell order it meets few cells, sums them in shared memory and adds its sums
// to S.  Bound by HBM (8 bytes per particle) and the warp sums in cell order,
// by the shared atomics in random order: 16.8 million particles on 1024 cells
// in 41 us in cell order up to one cell's drift (scalar loads, 304 blocks and
// lane-by-lane atomics: 85) and 48 in random order (76).
template <bool VEC>
__global__ void __launch_bounds__(kPassBlock) k_deposit_device(int N, long long n, const int* cell, const float* xi,
                                                               unsigned long long* S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* dcnt = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* dlo = dcnt + (N + 1);
  uint32_t* dhi = dcnt + 2 * (N + 1);
  for (int i = threadIdx.x; i < 3 * (N + 1); i += kPassBlock) dcnt[i] = 0u;
  __syncthreads();
  const long long nq = (n + 3) / 4;
  const long long lo = nq * blockIdx.x / gridDim.x, hi = nq * (blockIdx.x + 1) / gridDim.x;
  int since_flush = 0;
  // block-uniform trip count: the periodic flush and the warp sums need every thread
  for (long long base = lo; base < hi; base += kPassBlock) {
    const long long q = base + threadIdx.x;
    int c[4];
    float f[4];
    load_quad<VEC>(cell, xi, q < hi ? q : nq, n, N, c, f);
    dep_add_warp(dcnt, dlo, dhi, c, f);
    if (++since_flush == (kFlushParticles / (4 * kPassBlock))) {
      __syncthreads();
      dep_flush(dcnt, dlo, dhi, 0, N, S);
      __syncthreads();
      since_flush = 0;
    }
  }
  __syncthreads();
  dep_flush(dcnt, dlo, dhi, 0, N, S);
}

// The quadratic deposit (EC2): node N of a periodic system is node 0 here (its
// sums are added there, and mirrored afterwards).  16.8 million particles in 98
// us in cell order (three 64-bit atomics to S per particle: 3.8 ms).
template <bool VEC>
__global__ void __launch_bounds__(kPassBlock) k_deposit2_device(int N, int periodic, long long n, const int* cell,
                                                                const float* xi, unsigned long long* S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* dlo = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* dhi = dlo + (N + 1);
  for (int i = threadIdx.x; i < 2 * (N + 1); i += kPassBlock) dlo[i] = 0u;
  __syncthreads();
  const long long nq = (n + 3) / 4;
  const long long lo = nq * blockIdx.x / gridDim.x, hi = nq * (blockIdx.x + 1) / gridDim.x;
  auto flush = [&]() {
    dep2_flush(dlo, dhi, 0, N - 1, S);
    if (threadIdx.x == 0) {
      const unsigned long long v = ((unsigned long long)dhi[N] << 16) + dlo[N];
      if (v) atomicAdd(S + (periodic ? 0 : N), v);
      dlo[N] = dhi[N] = 0u;
    }
  };
  int since_flush = 0;
  for (long long base = lo; base < hi; base += kPassBlock) {
    const long long q = base + threadIdx.x;
    int c[4];
    float f[4];
    load_quad<VEC>(cell, xi, q < hi ? q : nq, n, N, c, f);
    dep2_add_warp(dlo, dhi, N, periodic != 0, c, f);
    if (++since_flush == kFlushParticles / (16 * kPassBlock)) {
      __syncthreads();
      flush();
      __syncthreads();
      since_flush = 0;
    }
  }
  __syncthreads();
  flush();
}

__global__ void k_mirror_node(int N, unsigned long long* S) { S[N] = S[0]; }

__global__ void k_philox_device(long long n, const uint32_t* ctr, const uint32_t* key,
                                uint32_t* out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 r = philox4x32_10(c, make_uint2(key[2 * i], key[2 * i + 1]));
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
  }
}

}  // namespace

// ----------------------------------------------------------------- launchers
void read_checks(unsigned long long out[4]) {
  cudaMemcpyFromSymbol(out, g_check, sizeof(unsigned long long) * 4);
}

size_t pass_smem_bytes(const BatchView& b) {
  return sizeof(long long) * (size_t)(b.nseg + 1) +
         (b.weighted ? 4 : 3) * sizeof(uint32_t) * (size_t)(b.nmax + 1) +
         sizeof(float) * 3 * (size_t)(b.nmax + 1) +
         sizeof(int) * (size_t)kRing * (kPassBlock / 32) + sizeof(float) * (size_t)(b.nmax + 1);
}

size_t field_smem_bytes(const BatchView& b) { return field_scratch_bytes(b.nmax, b.nseg / b.max_slots); }

static void set_smem_attr(const void* fn, size_t bytes) {
  if (bytes > 48 * 1024) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <bool W>
static int pass_occupancy(size_t sm) {
  set_smem_attr((const void*)k_pass<true, W>, sm);
  set_smem_attr((const void*)k_pass<false, W>, sm);
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pass<true, W>, kPassBlock, sm);
  return n > 0 ? n : 1;
}

int pass_max_ctas_per_sm(const BatchView& b) {
  const size_t sm = pass_smem_bytes(b);
  return b.weighted ? pass_occupancy<true>(sm) : pass_occupancy<false>(sm);
}

template <bool W>
static void launch_pass_w(const BatchView& b, int grid, int mode, int only, cudaStream_t s,
                          bool stage_field, size_t sm) {
  if (stage_field) {
    set_smem_attr((const void*)k_pass<true, W>, sm);
    k_pass<true, W><<<grid, kPassBlock, sm, s>>>(b, mode, only);
  } else {
    set_smem_attr((const void*)k_pass<false, W>, sm);
    k_pass<false, W><<<grid, kPassBlock, sm, s>>>(b, mode, only);
  }
}

void launch_pass(const BatchView& b, int grid, int mode, int only, cudaStream_t s, bool stage_field) {
  const size_t sm = pass_smem_bytes(b);
  if (b.weighted)
    launch_pass_w<true>(b, grid, mode, only, s, stage_field, sm);
  else
    launch_pass_w<false>(b, grid, mode, only, s, stage_field, sm);
}

void launch_collide(const BatchView& b, int grid, cudaStream_t s) {
  const size_t sm = sizeof(long long) * (size_t)(b.nseg + 1) + 3 * sizeof(int) * (size_t)b.nseg;
  set_smem_attr((const void*)k_collide, sm);
  k_collide<<<grid, kCollideBlock, sm, s>>>(b);
}

void launch_field(const BatchView& b, int advance, int only, cudaStream_t s) {
  const size_t sm = field_smem_bytes(b);
  set_smem_attr((const void*)k_field, sm);
  k_field<<<b.max_slots, kFieldBlock, sm, s>>>(b, advance, only);
}

void launch_phi(const BatchView& b, int slot, cudaStream_t s) {
  const size_t sm = field_smem_bytes(b);
  set_smem_attr((const void*)k_phi, sm);
  k_phi<<<1, kFieldBlock, sm, s>>>(b, slot);
}

// The scatter's grid: one wave of as many CTAs as fit on the device at its
// shared-memory size (every CTA takes an equal share of the particles, so a
// partial second wave would leave most SMs idle while it runs).
static int scatter_grid(size_t sms) {
  int dev = 0, nsm = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_scatter, kPassBlock, sms);
  return (occ > 0 ? occ : 1) * (nsm > 0 ? nsm : 1);
}

void launch_sort_phase(const BatchView& b, int grid, int phase, cudaStream_t s) {
  if (phase == 0) {
    const size_t smh = sizeof(long long) * (size_t)(b.nseg + 1) + sizeof(int) * (size_t)(b.nmax + 1);
    set_smem_attr((const void*)k_hist, smh);
    k_hist<<<grid, kPassBlock, smh, s>>>(b, MODE_SORT);
  } else if (phase == 1) {
    k_scan<<<b.nseg, kPassBlock, 0, s>>>(b, MODE_SORT);
  } else if (phase == 2) {
    const size_t sms = scatter_smem_bytes(b.nseg, b.nmax);
    set_smem_attr((const void*)k_scatter, sms);
    k_scatter<<<scatter_grid(sms), kPassBlock, sms, s>>>(b, MODE_SORT);
  } else {
    k_finalize<<<b.nseg, kPassBlock, 0, s>>>(b);
  }
}

void launch_sort(const BatchView& b, int grid, cudaStream_t s) {
  for (int ph = 0; ph < 4; ++ph) launch_sort_phase(b, grid, ph, s);
}

void launch_rebalance(const BatchView& b, int grid, cudaStream_t s) {
  const size_t smh = sizeof(long long) * (size_t)(b.nseg + 1) + sizeof(int) * (size_t)(b.nmax + 1);
  set_smem_attr((const void*)k_hist, smh);
  k_hist<<<grid, kPassBlock, smh, s>>>(b, MODE_REBAL);
  k_scan<<<b.nseg, kPassBlock, 0, s>>>(b, MODE_REBAL);
  const size_t sms = scatter_smem_bytes(b.nseg, b.nmax);
  set_smem_attr((const void*)k_scatter, sms);
  k_scatter<<<scatter_grid(sms), kPassBlock, sms, s>>>(b, MODE_REBAL);
  cudaMemsetAsync(b.rbnum, 0, sizeof(int), s);
  k_rb_classify<<<dim3((unsigned)((b.nmax + kPassBlock - 1) / kPassBlock), (unsigned)b.nseg), kPassBlock, 0,
                  s>>>(b);
  const size_t smr = sizeof(RbSmem);
  set_smem_attr((const void*)k_rb_cells, smr);
  k_rb_cells<<<grid, kRbBlock, smr, s>>>(b, 0);
  k_rb_scan<<<b.nseg, kPassBlock, 0, s>>>(b);
  // (a latency-bound stream: four times the persistent grid in flight)
  const size_t smc = sizeof(long long) * (size_t)(b.nseg + 1);
  set_smem_attr((const void*)k_rb_copy, smc);
  k_rb_copy<<<4 * grid, kPassBlock, smc, s>>>(b);
  k_rb_cells<<<grid, kRbBlock, smr, s>>>(b, 1);
  k_rb_finalize<<<b.nseg, kPassBlock, 0, s>>>(b);
  k_rb_mark<<<(b.max_slots + 127) / 128, 128, 0, s>>>(b);
}

void launch_init(const BatchView& b, int slot, const InitParams& p, cudaStream_t s) {
  long long nmax = 0;
  for (int i = 0; i < kMaxSpecies; ++i) nmax = p.n[i] > nmax ? p.n[i] : nmax;
  long long blocks = (nmax + 255) / 256;
  if (blocks < 1) blocks = 1;
  if (blocks > 4096) blocks = 4096;
  k_init<<<dim3((unsigned)blocks, kMaxSpecies), 256, 0, s>>>(b, slot, p);
}

void launch_init_many(const BatchView& b, const int* slots, const InitParams* ps, int count,
                      long long nmax, cudaStream_t s) {
  if (count <= 0) return;
  // Runs differ in size, so most blocks of a grid cut for the largest would be
  // empty: up to 16 particles per thread as soon as there are thousands of blocks.
  long long blocks = (nmax + 255) / 256;
  if (blocks < 1) blocks = 1;
  long long each = blocks * kMaxSpecies * count / 8192;
  each = each < 1 ? 1 : each > 16 ? 16 : each;
  blocks = (blocks + each - 1) / each;
  if (blocks > 4096) blocks = 4096;
  for (int off = 0; off < count; off += 65535) {
    const int c = count - off < 65535 ? count - off : 65535;
    k_init_many<<<dim3((unsigned)blocks, kMaxSpecies, (unsigned)c), 256, 0, s>>>(b, slots + off, ps + off, c);
  }
}

// Six blocks of 256 threads per SM keep enough loads in flight; a block of
// fewer than two iterations is not worth its flush.
static unsigned deposit_blocks(long long n) {
  const long long blocks = (n + 8 * kPassBlock - 1) / (8 * kPassBlock);
  return (unsigned)(blocks < 1 ? 1 : blocks > 912 ? 912 : blocks);
}
static bool aligned16(const void* a, const void* b) {
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15u) == 0u;
}

void launch_deposit_device(int N, long long n, const int* cell, const float* xi,
                           unsigned long long* S, cudaStream_t s) {
  const size_t sm = 3 * sizeof(uint32_t) * (size_t)(N + 1);
  if (aligned16(cell, xi))
    k_deposit_device<true><<<deposit_blocks(n), kPassBlock, sm, s>>>(N, n, cell, xi, S);
  else
    k_deposit_device<false><<<deposit_blocks(n), kPassBlock, sm, s>>>(N, n, cell, xi, S);
}

void launch_deposit2_device(int N, int periodic, long long n, const int* cell, const float* xi,
                            unsigned long long* S, cudaStream_t s) {
  const size_t sm = 2 * sizeof(uint32_t) * (size_t)(N + 1);
  if (aligned16(cell, xi))
    k_deposit2_device<true><<<deposit_blocks(n), kPassBlock, sm, s>>>(N, periodic, n, cell, xi, S);
  else
    k_deposit2_device<false><<<deposit_blocks(n), kPassBlock, sm, s>>>(N, periodic, n, cell, xi, S);
  if (periodic) k_mirror_node<<<1, 1, 0, s>>>(N, S);
}

void launch_philox_device(long long n, const uint32_t* ctr, const uint32_t* key, uint32_t* out,
                          cudaStream_t s) {
  long long blocks = (n + 255) / 256;
  if (blocks < 1) blocks = 1;
  if (blocks > 4096) blocks = 4096;
  k_philox_device<<<(unsigned)blocks, 256, 0, s>>>(n, ctr, key, out);
}

}  // namespace ecpic
