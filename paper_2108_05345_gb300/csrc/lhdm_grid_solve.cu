// lhdm_grid_solve.cu -- the solve kernel of one instance on the whole GPU.
#include "lhdm_kernels.cuh"

using namespace lhdm;

__global__ void __launch_bounds__(NT, 1) lhdm_solve_grid_kernel(Inst I, unsigned int* bar, int* err) {
  extern __shared__ double dyn[];
  solve_on_grid<false>(I, bar, err, dyn);
}
