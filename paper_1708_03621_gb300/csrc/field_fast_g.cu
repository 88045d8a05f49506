// Register-FFT field transforms, lengths 108, 64.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 108>;
template struct FieldFast<float, 108>;
template struct HartreeFast<108>;
template struct FieldFast<double, 64>;
template struct FieldFast<float, 64>;
template struct HartreeFast<64>;
}  // namespace jdft
