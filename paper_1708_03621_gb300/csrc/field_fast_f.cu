// Register-FFT field transforms, lengths 50, 54.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 50>;
template struct FieldFast<float, 50>;
template struct HartreeFast<50>;
template struct FieldFast<double, 54>;
template struct FieldFast<float, 54>;
template struct HartreeFast<54>;
}  // namespace jdft
