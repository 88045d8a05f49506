// Register-FFT field transforms of FP64 boxes, lengths 48 64.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 48>;
template struct HartreeFast<48>;
template struct FieldFast<double, 64>;
template struct HartreeFast<64>;
}  // namespace jdft
