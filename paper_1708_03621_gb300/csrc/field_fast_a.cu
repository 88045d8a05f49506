// Register-FFT field transforms, lengths 12, 16, 24, 128.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 12>;
template struct FieldFast<float, 12>;
template struct HartreeFast<12>;
template struct FieldFast<double, 16>;
template struct FieldFast<float, 16>;
template struct HartreeFast<16>;
template struct FieldFast<double, 24>;
template struct FieldFast<float, 24>;
template struct HartreeFast<24>;
template struct FieldFast<double, 128>;
template struct FieldFast<float, 128>;
template struct HartreeFast<128>;
}  // namespace jdft
