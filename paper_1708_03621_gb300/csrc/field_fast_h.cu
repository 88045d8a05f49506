// Register-FFT field transforms, lengths 60, 81.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 60>;
template struct FieldFast<float, 60>;
template struct HartreeFast<60>;
template struct FieldFast<double, 81>;
template struct FieldFast<float, 81>;
template struct HartreeFast<81>;
}  // namespace jdft
