// Instantiation of the row-march kernel: BF16 storage, steps, rows of any length (a translation
// unit per storage type, pass and kind of strip, so the library builds in parallel).
#include "lb_step_march.cuh"

namespace lbk {
#define X(T, SMODE, BND, SCHEME) LB_MARCH_STEP(, T, SMODE, BND, SCHEME, kOdd)
LB_MARCH_VARIANTS(X, __nv_bfloat16)
#undef X
}  // namespace lbk
