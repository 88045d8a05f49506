// Register-FFT field transforms of FP32 boxes.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<float, 12>;
template struct FieldFast<float, 16>;
template struct FieldFast<float, 40>;
template struct FieldFast<float, 48>;
template struct FieldFast<float, 64>;
template struct FieldFast<float, 80>;
template struct FieldFast<float, 128>;
template struct FieldFast<float, 256>;
}  // namespace jdft
