// Instantiation of the drivers' mode-1 step kernels (see tc_k_driver.cuh).
#include "tc_k_driver.cuh"

namespace tcg {

cudaError_t launch_driver1(const DevFields& f, const DevParams& p, double dt, unsigned long long* cursor,
                           long long ntotal, int grid, int block, cudaStream_t st) {
  return launch_driver_kernel<DRIVER + 1, 1>(f, p, dt, cursor, ntotal, grid, block, st);
}
int occupancy_driver1(int block) { return occupancy_driver_kernel<DRIVER + 1, 1>(block); }

cudaError_t launch_driver1_coop(const DevFields& f, const DevParams& p, double dt, unsigned long long* cursor,
                           long long ntotal, int grid, int block, cudaStream_t st) {
  return launch_driver_kernel<DRIVER + 1, 4>(f, p, dt, cursor, ntotal, grid, block, st);
}
int occupancy_driver1_coop(int block) { return occupancy_driver_kernel<DRIVER + 1, 4>(block); }

}  // namespace tcg
