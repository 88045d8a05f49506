// Register-FFT field transforms of FP64 boxes, lengths 12 16 40.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 12>;
template struct HartreeFast<12>;
template struct FieldFast<double, 16>;
template struct HartreeFast<16>;
template struct FieldFast<double, 40>;
template struct HartreeFast<40>;
}  // namespace jdft
