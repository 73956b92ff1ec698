// Instantiation of the shared-memory resident sweep in FP32 arithmetic (FP32 / BF16 storage; any width, and the
// width 4 as a compile-time constant).
#include "lb_sweep_pair.cuh"

namespace lbk {
#define X(T, NT, NX) LB_SWEEP_PAIR(, T, NT, NX)
LB_SWEEP_PAIR_VARIANTS(X)
#undef X
}  // namespace lbk
