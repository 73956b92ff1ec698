// Instantiation of the row-march kernel's fields pass (the fields of the stored state in node order) for
// every variant that steps.
#include "lb_step_march.cuh"

namespace lbk {
#define LB_MARCH_FIELDS(T, SMODE, BND, SCHEME)                                                                        \
    template cudaError_t launch_step_march<T, float, SMODE, BND, SCHEME, true>(const CUtensorMap&, const StepArgs<T, float>&, \
                                                                               const MarchCtl&, int, cudaStream_t);
LB_MARCH_FIELDS_ALL(LB_MARCH_FIELDS)
#undef LB_MARCH_FIELDS
}  // namespace lbk
