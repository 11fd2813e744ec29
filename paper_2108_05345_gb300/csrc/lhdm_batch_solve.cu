// lhdm_batch_solve.cu -- the persistent solve kernel of a batch of instances.
#include "lhdm_kernels.cuh"

using namespace lhdm;

__global__ void __launch_bounds__(NT, 1) lhdm_solve_batch_kernel(const BatchItem* items, const int* perm,
                                                                 int batch, int* queue, ScratchLayout L,
                                                                 double* dscr, int* iscr, DevParams prm) {
  extern __shared__ double dyn[];
  solve_queue<false>(items, perm, batch, queue, L, dscr, iscr, prm, dyn);
}
