// Instantiation of the drivers' mode-0 step kernel (see tc_k_driver.cuh).
#include "tc_k_driver.cuh"

namespace tcg {

cudaError_t launch_driver0(const DevFields& f, const DevParams& p, double dt, unsigned long long* cursor,
                           long long ntotal, int grid, int block, cudaStream_t st) {
  return launch_driver_kernel<DRIVER + 0, 1>(f, p, dt, cursor, ntotal, grid, block, st);
}
int occupancy_driver0(int block) { return occupancy_driver_kernel<DRIVER + 0, 1>(block); }

}  // namespace tcg
