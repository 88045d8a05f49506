// Register-FFT field transforms, lengths 48, 125.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 48>;
template struct FieldFast<float, 48>;
template struct HartreeFast<48>;
template struct FieldFast<double, 125>;
template struct FieldFast<float, 125>;
template struct HartreeFast<125>;
}  // namespace jdft
