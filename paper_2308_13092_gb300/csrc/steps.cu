// steps.cu -- k_steps for batches without weight multipliers, and the choice
// between its two translation units (compiled side by side).
#include "steps.cuh"

namespace ecpic {

bool steps_fit(const BatchView& b, int device) {
  int most = 0, coop = 0;
  cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device);
  return coop != 0 && kStepSmem + 1024 <= (size_t)most && steps_smem(b, 512) <= kStepSmem;
}

cudaError_t launch_steps(const BatchView& b, const StepPlan& pl, const StepTeams& tm, int steps, int sort_every,
                         int since_sort, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(pl.words, 0, sizeof(StepWords) * (size_t)b.max_slots, s);
  if (e != cudaSuccess) return e;
  return b.weighted ? launch_steps_weighted(b, pl, tm, steps, sort_every, since_sort, s)
                    : launch_any<false>(b, pl, tm, steps, sort_every, since_sort, s);
}

void read_checks_steps(unsigned long long out[4]) {
  cudaMemcpyFromSymbol(out, g_check, sizeof(unsigned long long) * 4);
}

}  // namespace ecpic
