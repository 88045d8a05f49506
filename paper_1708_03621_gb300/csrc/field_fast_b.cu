// Register-FFT field transforms, lengths 25, 27, 30.
#include "field_fast_impl.cuh"

namespace jdft {
template struct FieldFast<double, 25>;
template struct FieldFast<float, 25>;
template struct HartreeFast<25>;
template struct FieldFast<double, 27>;
template struct FieldFast<float, 27>;
template struct HartreeFast<27>;
template struct FieldFast<double, 30>;
template struct FieldFast<float, 30>;
template struct HartreeFast<30>;
}  // namespace jdft
