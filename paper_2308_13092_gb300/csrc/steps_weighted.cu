// steps_weighted.cu -- k_steps for batches that hold rebalancing runs.
#include "steps.cuh"

namespace ecpic {

cudaError_t launch_steps_weighted(const BatchView& b, const StepPlan& pl, const StepTeams& tm, int steps,
                                  int sort_every, int since_sort, cudaStream_t s) {
  return launch_any<true>(b, pl, tm, steps, sort_every, since_sort, s);
}

void read_checks_steps_weighted(unsigned long long out[4]) {
  cudaMemcpyFromSymbol(out, g_check, sizeof(unsigned long long) * 4);
}

}  // namespace ecpic
