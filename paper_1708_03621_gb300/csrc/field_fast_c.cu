// Register-FFT field transforms, lengths 32, 36, 75.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 32>;
template struct FieldFast<float, 32>;
template struct HartreeFast<32>;
template struct FieldFast<double, 36>;
template struct FieldFast<float, 36>;
template struct HartreeFast<36>;
template struct FieldFast<double, 75>;
template struct FieldFast<float, 75>;
template struct HartreeFast<75>;
}  // namespace jdft
