// Register-FFT field transforms, lengths 120.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 120>;
template struct FieldFast<float, 120>;
template struct HartreeFast<120>;
}  // namespace jdft
