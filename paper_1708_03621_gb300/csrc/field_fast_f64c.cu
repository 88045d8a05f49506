// Register-FFT field transforms of FP64 boxes, lengths 80.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 80>;
template struct HartreeFast<80>;
}  // namespace jdft
