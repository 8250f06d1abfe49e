// run_wide.cu -- k_run with two CTAs an SM (chunks of up to 2^10 amplitudes).
#include "run.cuh"

namespace qc {

int run_wide_ctas_per_sm(int kc) { return run_occupancy<2>(kc); }

cudaError_t launch_run_wide(const RunJob* jobs, int njobs, int kc, int grid, cudaStream_t st) {
  return run_launch<2>(jobs, njobs, kc, grid, st);
}

}  // namespace qc
