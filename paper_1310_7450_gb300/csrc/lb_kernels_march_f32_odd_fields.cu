// Instantiation of the row-march kernel: FP32 storage, the fields pass, rows of any length (a translation
// unit per storage type, pass and kind of strip, so the library builds in parallel).
#include "lb_step_march.cuh"

namespace lbk {
#define X(T, SMODE, BND, SCHEME) LB_MARCH_FIELDS(, T, SMODE, BND, SCHEME, kOdd)
LB_MARCH_VARIANTS(X, float)
#undef X
}  // namespace lbk
