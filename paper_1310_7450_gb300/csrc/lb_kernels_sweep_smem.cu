// Instantiation of the shared-memory resident cluster sweep in FP64 (stress mode A; any width, and the width 4
// as a compile-time constant); lb_kernels_sweep_pair.cu has the FP32 arithmetic.
#include "lb_sweep_smem.cuh"

namespace lbk {
#define LB_SWEEP_SMEM_INST(T, C, NX)                                                                                  \
    template cudaError_t launch_sweep_smem<T, C, 128, 4, NX>(const SweepArgs<T, C>&, int, int, size_t, cudaStream_t); \
    template cudaError_t launch_sweep_smem<T, C, 256, 4, NX>(const SweepArgs<T, C>&, int, int, size_t, cudaStream_t); \
    template cudaError_t launch_sweep_smem_capacity<T, C, 128, 4, NX>(int, size_t, int*);                               \
    template cudaError_t launch_sweep_smem_capacity<T, C, 256, 4, NX>(int, size_t, int*);
LB_SWEEP_SMEM_INST(double, double, 0)
LB_SWEEP_SMEM_INST(double, double, 4)
#undef LB_SWEEP_SMEM_INST
}  // namespace lbk
