// run.cu -- k_run with three CTAs an SM (batches, and what two do not hold).
#include "run.cuh"

namespace qc {

int run_ctas_per_sm(int kc, bool wide) { return wide ? run_wide_ctas_per_sm(kc) : run_occupancy<3>(kc); }

cudaError_t launch_run(const RunJob* jobs, int njobs, int kc, int grid, bool wide, cudaStream_t st) {
  return wide ? launch_run_wide(jobs, njobs, kc, grid, st) : run_launch<3>(jobs, njobs, kc, grid, st);
}

}  // namespace qc
