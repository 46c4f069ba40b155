// deposit.cuh -- fixed-point charge deposits in shared memory (Eq. 2-3), shared
// by the particle pass and the kernel-level entry points.
#pragma once
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>

namespace ecpic {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// ----------------------------------------------------------------- deposit
// Fixed-point CIC deposit (Eq. 2-3) in units of 2^-32 particle: a particle at
// (c, xi) with r = floor(xi 2^32) (xi * 2^32 is exact in FP32; rz truncation
// = floor) adds 2^32 - r to node c and r to node c+1.  In shared memory each
// cell keeps three 32-bit sums, updated with native 32-bit atomics: its
// particle count, and the sums of the low and high 16 bits of r.  The flush
// forms the node values, S[c] += cnt 2^32 - R and S[c+1] += R with
// R = hi 2^16 + lo.  With at most kFlushParticles particles between flushes
// no sum reaches 2^32.
constexpr int kFlushParticles = 65536;

// Adds V particles (cells c[j] < 0 skipped); a thread's consecutive
// particles in the same cell are merged first, so sorted data costs one
// atomic triple per run.
template <int V = 4>
__device__ __forceinline__ void dep_add4(uint32_t* dcnt, uint32_t* dlo, uint32_t* dhi, const int c[V],
                                         const float f[V]) {
  unsigned lo[V], hi[V], cn[V];
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const bool v = c[j] >= 0;
    const unsigned r = v ? __float2uint_rz(f[j] * 4294967296.0f) : 0u;
    lo[j] = r & 0xFFFFu;
    hi[j] = r >> 16;
    cn[j] = v ? 1u : 0u;
  }
#pragma unroll
  for (int j = V - 1; j >= 1; --j) {
    if (c[j] >= 0 && c[j] == c[j - 1]) {
      lo[j - 1] += lo[j];
      hi[j - 1] += hi[j];
      cn[j - 1] += cn[j];
      cn[j] = 0u;
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) {
    if (cn[j]) {
      atomicAdd(dcnt + c[j], cn[j]);
      atomicAdd(dlo + c[j], lo[j]);
      atomicAdd(dhi + c[j], hi[j]);
    }
  }
}

// Adds the shared sums of cells [a, e) to the node array S in HBM and clears
// them.  Every thread of the block calls it, between barriers.
__device__ void dep_flush(uint32_t* dcnt, uint32_t* dlo, uint32_t* dhi, int a, int e,
                          unsigned long long* S) {
  for (int c = a + (int)threadIdx.x; c < e; c += (int)blockDim.x) {
    const uint32_t n = dcnt[c];
    if (n) {
      const unsigned long long R = ((unsigned long long)dhi[c] << 16) + (unsigned long long)dlo[c];
      atomicAdd(S + c, ((unsigned long long)n << 32) - R);
      if (R) atomicAdd(S + c + 1, R);
      dcnt[c] = 0u;
      dlo[c] = 0u;
      dhi[c] = 0u;
    }
  }
}

// ---- quadratic-spline deposit of the EC2 scheme (uniform grids) ----------
// A particle at cell + xi with r = floor(xi 2^32) has its nearest node
// n0 = cell + (r >= 2^31) and offset U = r or r - 2^32 (2^-32 cell units);
// nodes n0-1, n0, n0+1 get a = floor((2^31-U)^2 / 2^33), 2^32 - a - b,
// b = floor((2^31+U)^2 / 2^33): the quadratic B-spline weights to 2^-32,
// exact integers summing to 2^32.
__device__ __forceinline__ void spline2_shares(float f, int c, int* n0, unsigned* a, unsigned* b) {
  const unsigned r = __float2uint_rz(f * 4294967296.0f);
  const bool up = r >= 0x80000000u;
  *n0 = c + (up ? 1 : 0);
  const long long U = up ? (long long)r - 4294967296LL : (long long)r;
  const unsigned long long A = (unsigned long long)(2147483648LL - U);
  const unsigned long long B = (unsigned long long)(2147483648LL + U);
  *a = (unsigned)((__umul64hi(A, A) << 31) | ((A * A) >> 33));
  *b = (unsigned)((__umul64hi(B, B) << 31) | ((B * B) >> 33));
}

// node of a share beyond the cells: folded into the wall node (Dirichlet: the
// ghost node beyond a wall is the wall node), wrapped when periodic (node N
// and node 0 are one node for the field solve)
__device__ __forceinline__ int node2(int n, int N, bool periodic) {
  if (periodic) return n < 0 ? n + N : (n > N ? n - N : n);
  return n < 0 ? 0 : (n > N ? N : n);
}

// Adds V particles to two 32-bit sums per node (the low and high 16 bits
// of the shares it receives, after folding or wrapping); runs of equal
// nearest node merged first.  A wall node can receive two shares of one
// particle, and a run's middle share can reach 2^34, so the EC2 pass flushes
// every kFlushParticles / 4 particles: no sum reaches 2^32.
template <int V = 4>
__device__ __forceinline__ void dep2_add4(uint32_t* dlo, uint32_t* dhi, int N, bool periodic,
                                          const int c[V], const float f[V]) {
  int n0[V];
  unsigned long long A[V], M[V], B[V];
#pragma unroll
  for (int j = 0; j < V; ++j) {
    unsigned a = 0u, b = 0u;
    n0[j] = -1;
    if (c[j] >= 0) spline2_shares(f[j], c[j], &n0[j], &a, &b);
    A[j] = a;
    B[j] = b;
    M[j] = c[j] >= 0 ? 4294967296ull - a - b : 0ull;
  }
#pragma unroll
  for (int j = V - 1; j >= 1; --j) {
    if (n0[j] >= 0 && n0[j] == n0[j - 1]) {
      A[j - 1] += A[j];
      M[j - 1] += M[j];
      B[j - 1] += B[j];
      n0[j] = -1;
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) {
    if (n0[j] >= 0) {
      const int nl = node2(n0[j] - 1, N, periodic), nr = node2(n0[j] + 1, N, periodic);
      atomicAdd(dlo + nl, (unsigned)(A[j] & 0xFFFFu));
      atomicAdd(dhi + nl, (unsigned)(A[j] >> 16));
      atomicAdd(dlo + n0[j], (unsigned)(M[j] & 0xFFFFu));
      atomicAdd(dhi + n0[j], (unsigned)(M[j] >> 16));
      atomicAdd(dlo + nr, (unsigned)(B[j] & 0xFFFFu));
      atomicAdd(dhi + nr, (unsigned)(B[j] >> 16));
    }
  }
}

// Adds the sums of nodes [a, e] to S and clears them; every thread of the
// block calls it, between barriers.
__device__ void dep2_flush(uint32_t* dlo, uint32_t* dhi, int a, int e, unsigned long long* S) {
  for (int n = a + (int)threadIdx.x; n <= e; n += (int)blockDim.x) {
    const unsigned long long v = ((unsigned long long)dhi[n] << 16) + dlo[n];
    if (v) {
      atomicAdd(S + n, v);
      dlo[n] = 0u;
      dhi[n] = 0u;
    }
  }
}

// ---- deposits of caller-owned arrays (kernel-level entry points) ----------
// Particles in cell order put most of a warp's 128 in a few cells, where the
// shared atomics of dep_add4 would queue up on the same words (16.8 million
// particles in cell order up to one cell's drift: 85 us, 0.23 of HBM).  With
// at most kWarpCells cells in the warp its lanes' shares of each cell are
// summed by warp reductions and one lane adds them.  Called by all lanes;
// cells c[j] < 0 are skipped.
constexpr int kWarpCells = 4;
__device__ __forceinline__ void dep_add_warp(uint32_t* dcnt, uint32_t* dlo, uint32_t* dhi, const int c[4],
                                             const float f[4]) {
  int lo = INT_MAX, hi = -1;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    lo = c[j] >= 0 ? min(lo, c[j]) : lo;
    hi = max(hi, c[j]);
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  if (hi < 0) return;
  if (hi - lo >= kWarpCells) {
    dep_add4(dcnt, dlo, dhi, c, f);
    return;
  }
  unsigned r[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) r[j] = c[j] >= 0 ? __float2uint_rz(f[j] * 4294967296.0f) : 0u;
  const unsigned lane = threadIdx.x & 31u;
  for (int k = lo; k <= hi; ++k) {
    // (count, sum of the high parts) in one word: 128 particles of 16 bits
    unsigned a = 0u, b = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c[j] == k) {
        a += (1u << 24) + (r[j] >> 16);
        b += r[j] & 0xFFFFu;
      }
    a = __reduce_add_sync(kFull, a);
    b = __reduce_add_sync(kFull, b);
    if (lane == 0u && a) {
      atomicAdd(dcnt + k, a >> 24);
      atomicAdd(dlo + k, b);
      atomicAdd(dhi + k, a & 0xFFFFFFu);
    }
  }
}

// The same for the quadratic shares, by nearest node.
__device__ __forceinline__ void dep2_add_warp(uint32_t* dlo, uint32_t* dhi, int N, bool periodic, const int c[4],
                                              const float f[4]) {
  int n0[4], lo = INT_MAX, hi = -1;
  unsigned a[4], b[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    n0[j] = -1;
    a[j] = b[j] = 0u;
    if (c[j] >= 0) {
      spline2_shares(f[j], c[j], &n0[j], &a[j], &b[j]);
      lo = min(lo, n0[j]);
      hi = max(hi, n0[j]);
    }
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  if (hi < 0) return;
  if (hi - lo >= kWarpCells) {
    dep2_add4(dlo, dhi, N, periodic, c, f);
    return;
  }
  const int lane = (int)(threadIdx.x & 31u);
  for (int k = lo; k <= hi; ++k) {
    unsigned s[6] = {0u, 0u, 0u, 0u, 0u, 0u};  // left, middle, right: low and high 16 bits
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (n0[j] == k) {
        const unsigned m = 0u - a[j] - b[j];  // 2^32 - a - b, below 2^32 (a + b >= 2^30)
        s[0] += a[j] & 0xFFFFu;
        s[1] += a[j] >> 16;
        s[2] += m & 0xFFFFu;
        s[3] += m >> 16;
        s[4] += b[j] & 0xFFFFu;
        s[5] += b[j] >> 16;
      }
#pragma unroll
    for (int q = 0; q < 6; ++q) s[q] = __reduce_add_sync(kFull, s[q]);
    if (lane < 3) {
      const int node = lane == 1 ? k : node2(k + lane - 1, N, periodic);
      atomicAdd(dlo + node, lane == 0 ? s[0] : lane == 1 ? s[2] : s[4]);
      atomicAdd(dhi + node, lane == 0 ? s[1] : lane == 1 ? s[3] : s[5]);
    }
  }
}

// One thread's four particles of quad q of caller-owned arrays: cells outside
// [0, N) become -1.  VEC: both arrays are 16-byte aligned.
template <bool VEC>
__device__ __forceinline__ void load_quad(const int* cell, const float* xi, long long q, long long n, int N, int c[4],
                                          float f[4]) {
  const long long i = 4 * q;
  if (VEC && i + 3 < n) {
    const int4 a = __ldcs(reinterpret_cast<const int4*>(cell) + q);
    const float4 x = __ldcs(reinterpret_cast<const float4*>(xi) + q);
    c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
    f[0] = x.x; f[1] = x.y; f[2] = x.z; f[3] = x.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      c[j] = i + j < n ? cell[i + j] : -1;
      f[j] = i + j < n ? xi[i + j] : 0.0f;
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) c[j] = (unsigned)c[j] < (unsigned)N ? c[j] : -1;
}

}  // namespace
}  // namespace ecpic
