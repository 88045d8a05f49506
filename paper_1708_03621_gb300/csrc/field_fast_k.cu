// Register-FFT field transforms, lengths 100, 256.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 100>;
template struct FieldFast<float, 100>;
template struct HartreeFast<100>;
template struct FieldFast<double, 256>;
template struct FieldFast<float, 256>;
template struct HartreeFast<256>;
}  // namespace jdft
