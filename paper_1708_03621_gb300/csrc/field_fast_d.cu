// Register-FFT field transforms, lengths 40, 45.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 40>;
template struct FieldFast<float, 40>;
template struct HartreeFast<40>;
template struct FieldFast<double, 45>;
template struct FieldFast<float, 45>;
template struct HartreeFast<45>;
}  // namespace jdft
