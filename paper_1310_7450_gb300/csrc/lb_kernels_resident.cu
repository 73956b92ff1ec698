// Instantiation of the resident step (one small channel, many steps per launch).
#include "lb_step_resident.cuh"

namespace lbk {
#define X(T, C, SMODE, NT) LB_RESIDENT(, T, C, SMODE, NT)
LB_RESIDENT_VARIANTS(X)
#undef X
}  // namespace lbk
