// noalloc.cu -- fixed-point CIC deposit (Eq. 2-3) that allocates no device
// memory: ecpic_deposit_device_noalloc.
//
// Same result as ecpic_deposit_device, reached another way: instead of
// adding each block's shared-memory sums to S with global atomics, every
// block writes its whole partial row (N+1 sums) into a fixed scratch array
// that is part of this module's image, and a second kernel adds the rows to
// S node by node in row order.  The sums are 64-bit integers, so the order
// does not change the result.
//
// Who needs this: callers that must not allocate device memory while they
// run -- a process that handed all free HBM to its own pool at start-up
// (where a cudaMalloc would fail), or a latency-bound loop in which
// cudaMalloc/cudaFree would stall it by synchronising the device.  So this
// path calls no cudaMalloc, cudaFree or allocating library routine.
#include <cuda_runtime.h>

#include <mutex>

#include "../../include/ecpic.h"
#include "deposit.cuh"

namespace {

constexpr int kNaBlock = 256;
constexpr int kNaMaxRows = 608;  // four blocks per SM on a 152-SM part
constexpr size_t kNaWords = ECPIC_NOALLOC_SCRATCH_BYTES / sizeof(unsigned long long);
constexpr int kMaxDevices = 64;

static_assert((size_t)(ECPIC_NOALLOC_MAX_CELLS + 1) <= kNaWords, "scratch must hold one row");

// Partial rows: row r = block r's sums for nodes 0..N, row-major.  Every entry
// the reduction reads is written by the same call first, so no part of it has
// to start at zero and no call clears it.
static __device__ __align__(256) unsigned long long g_na_scratch[kNaWords];

// scratch address per device, looked up at the first call on that device and
// kept for the life of the process (a device reset makes it stale: see the
// header)
std::mutex g_na_mu;
void* g_na_ptr[kMaxDevices] = {};

// Block-local deposit of a block's consecutive quads, written out as this
// block's row: 32-bit shared sums as in ecpic_deposit_device (deposit.cuh),
// moved into 64-bit ones before they can overflow.  16.8 million particles on
// 1024 cells with the sum of the rows: 61 us in cell order, 53 in random order
// (64-bit shared atomics after a match of the lanes' cells: 340 and 990).
template <bool VEC>
__global__ void __launch_bounds__(kNaBlock) k_na_rows(int N, long long n, const int* __restrict__ cell,
                                                      const float* __restrict__ xi,
                                                      unsigned long long* rows) {
  extern __shared__ __align__(16) unsigned char na_smem[];
  unsigned long long* acc = reinterpret_cast<unsigned long long*>(na_smem);
  uint32_t* dcnt = reinterpret_cast<uint32_t*>(acc + (N + 1));
  uint32_t* dlo = dcnt + (N + 1);
  uint32_t* dhi = dlo + (N + 1);
  for (int i = threadIdx.x; i <= N; i += kNaBlock) {
    acc[i] = 0ull;
    dcnt[i] = dlo[i] = dhi[i] = 0u;
  }
  __syncthreads();
  // node i takes 2^32 - r of its cell and r of the cell before
  auto flush = [&]() {
    __syncthreads();
    for (int i = threadIdx.x; i <= N; i += kNaBlock) {
      const unsigned long long own = ((unsigned long long)dhi[i] << 16) + dlo[i];
      unsigned long long t = ((unsigned long long)dcnt[i] << 32) - own;
      if (i > 0) t += ((unsigned long long)dhi[i - 1] << 16) + dlo[i - 1];
      acc[i] += t;
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= N; i += kNaBlock) dcnt[i] = dlo[i] = dhi[i] = 0u;
    __syncthreads();
  };
  const long long nq = (n + 3) / 4;
  const long long lo = nq * blockIdx.x / gridDim.x, hi = nq * (blockIdx.x + 1) / gridDim.x;
  int since_flush = 0;
  for (long long base = lo; base < hi; base += kNaBlock) {  // block-uniform trip count
    const long long q = base + threadIdx.x;
    int c[4];
    float f[4];
    ecpic::load_quad<VEC>(cell, xi, q < hi ? q : nq, n, N, c, f);
    ecpic::dep_add_warp(dcnt, dlo, dhi, c, f);
    if (++since_flush == ecpic::kFlushParticles / (4 * kNaBlock)) {
      flush();
      since_flush = 0;
    }
  }
  flush();
  unsigned long long* row = rows + (size_t)blockIdx.x * (size_t)(N + 1);
  for (int i = threadIdx.x; i <= N; i += kNaBlock) row[i] = acc[i];
}

// S[i] += sum of the rows' entries i: a warp's lanes take 32 nodes, a block's
// warps every kNaBlock / 32-th row (a serial sum over the rows by one thread
// per node took longer than the rows of 10^5 particles)
__global__ void __launch_bounds__(kNaBlock) k_na_sum(int N, int nrows,
                                                     const unsigned long long* __restrict__ rows,
                                                     unsigned long long* S) {
  constexpr int kWarps = kNaBlock / 32;
  __shared__ unsigned long long part[kWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  unsigned long long s = 0ull;
  if (i <= N) {
#pragma unroll 8
    for (int r = w; r < nrows; r += kWarps) s += rows[(size_t)r * (size_t)(N + 1) + i];
  }
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && i <= N) {
#pragma unroll
    for (int q = 1; q < kWarps; ++q) s += part[q][lane];
    S[i] += s;
  }
}

// The scratch address on the current device; the first call on a device
// looks it up (cudaGetSymbolAddress) with that device current.
int na_scratch(unsigned long long** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ECPIC_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_na_mu);
  if (!g_na_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_na_scratch);
    if (e != cudaSuccess || p == nullptr) return ECPIC_ERR_CUDA;
    g_na_ptr[dev] = p;
  }
  *out = static_cast<unsigned long long*>(g_na_ptr[dev]);
  return ECPIC_OK;
}

}  // namespace

extern "C" int ecpic_deposit_device_noalloc(int N, int64_t n, const int32_t* d_cell, const float* d_xi,
                                            uint64_t* d_S, void* stream) {
  if (N < 1 || n < 0 || (n > 0 && (!d_cell || !d_xi)) || !d_S) return ECPIC_ERR_ARG;
  if (N > ECPIC_NOALLOC_MAX_CELLS) return ECPIC_ERR_CAPACITY;
  unsigned long long* rows = nullptr;
  const int rc = na_scratch(&rows);  // set-up on the first call, even when n == 0
  if (rc != ECPIC_OK) return rc;
  if (n == 0) return ECPIC_OK;
  const long long per_row = (long long)(kNaWords / (size_t)(N + 1));
  long long nrows = (n + 8 * kNaBlock - 1) / (8 * kNaBlock);  // two iterations or more a block
  if (nrows > kNaMaxRows) nrows = kNaMaxRows;
  if (nrows > per_row) nrows = per_row;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // a row of N + 1 sums and three 32-bit ones per node: at most 20 x 2049 =
  // 40,980 B (N = 2048), within the 48 KiB a launch gets without an opt-in
  const size_t smem = (sizeof(unsigned long long) + 3 * sizeof(uint32_t)) * (size_t)(N + 1);
  if (((reinterpret_cast<uintptr_t>(d_cell) | reinterpret_cast<uintptr_t>(d_xi)) & 15u) == 0u)
    k_na_rows<true><<<(unsigned)nrows, kNaBlock, smem, s>>>(N, (long long)n, d_cell, d_xi, rows);
  else
    k_na_rows<false><<<(unsigned)nrows, kNaBlock, smem, s>>>(N, (long long)n, d_cell, d_xi, rows);
  k_na_sum<<<(unsigned)((N + 1 + 31) / 32), kNaBlock, 0, s>>>(
      N, (int)nrows, rows, reinterpret_cast<unsigned long long*>(d_S));
  return cudaGetLastError() == cudaSuccess ? ECPIC_OK : ECPIC_ERR_CUDA;
}
