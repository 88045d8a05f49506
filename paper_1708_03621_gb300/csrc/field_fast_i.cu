// Register-FFT field transforms, lengths 72, 96.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 72>;
template struct FieldFast<float, 72>;
template struct HartreeFast<72>;
template struct FieldFast<double, 96>;
template struct FieldFast<float, 96>;
template struct HartreeFast<96>;
}  // namespace jdft
