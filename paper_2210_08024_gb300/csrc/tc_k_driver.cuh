// Step kernels of the equilibrium and PDR drivers in the FP64 modes (tc_eq_curves, tc_pdr).
//
// A driver chains chunks of 1 to 10 Myr from one start state, and cells that pass a thermally
// unstable state on the way multiply any difference, a rounding's too, by up to 1e8: a table's
// result is reproducible only by the same operations in the same order.  So these kernels keep
// one arithmetic whatever the step's kernels do: the plain Newton iteration (its x_e is the last
// iterate's, ~5e-14 off, which the unstable cells carry to 1e-9 of T), and CUDA's exp(), log() and
// division (TCG_PLAIN_FP64).  By the step's own kernels 6 of 80 tables of dense PDR slabs moved by
// more than 1e-9 in T or x_H2 (2-norm; up to 8e-9) and 15 of 40 tables of shielded curves in the
// last chunk's change (up to 6e-7); by their plain iteration still 4 of 120 and 17 of 60.
// The price: 64 curves x 200 densities over 10 chunks 62.0 ms where the step's kernels take 14.0, 48
// slabs x 100 cells over 30 chunks 282 where they take 122.
#pragma once
#define TCG_DRIVER
#include "tc_launch.h"

namespace tcg {

template <int KMODE, int LPC>
inline cudaError_t launch_driver_kernel(const DevFields& f, const DevParams& p, double dt, unsigned long long* cursor,
                                        long long ntotal, int grid, int block, cudaStream_t st) {
  k_step<KMODE, false, LPC><<<grid, block, 0, st>>>(f, nullptr, p, dt, cursor, ntotal, nullptr);
  return cudaGetLastError();
}

template <int KMODE, int LPC>
inline int occupancy_driver_kernel(int block) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_step<KMODE, false, LPC>, block, 0) != cudaSuccess) return 1;
  return nb > 0 ? nb : 1;
}

}  // namespace tcg
