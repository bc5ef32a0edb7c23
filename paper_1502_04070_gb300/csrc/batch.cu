// batch.cu -- results of the batched solver.
//
// Every instance of a batch runs its refinement steps inside a conditional WHILE node of one CUDA
// graph; the last kernel of a step decides on the device whether the instance goes on (loop_check,
// kernels.cu), so the whole batch runs to convergence in one graph launch without returning to the host.
#include <cuda_runtime.h>

#include "cellops.cuh"
#include "kernels.cuh"

namespace smg {

__global__ void k_batch_store(const double* __restrict__ scal, const int* __restrict__ count,
                              double* __restrict__ out) {
    pdl_wait();
    if (threadIdx.x != 0) return;
    out[0] = scal[0];
    out[1] = scal[2];
    out[2] = (double)*count;
    pdl_trigger();
}

void launch_batch_store(cudaStream_t s, const double* scal, const int* count, double* out) {
    launch_pdl(k_batch_store, 1, 32, 0, s, scal, count, out);
}

}  // namespace smg
