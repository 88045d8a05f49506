// Register-FFT field transforms of FP64 boxes, lengths 128 256.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 128>;
template struct HartreeFast<128>;
template struct FieldFast<double, 256>;
template struct HartreeFast<256>;
}  // namespace jdft
