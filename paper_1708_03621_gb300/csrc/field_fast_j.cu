// Register-FFT field transforms, lengths 80, 90.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 80>;
template struct FieldFast<float, 80>;
template struct HartreeFast<80>;
template struct FieldFast<double, 90>;
template struct FieldFast<float, 90>;
template struct HartreeFast<90>;
}  // namespace jdft
