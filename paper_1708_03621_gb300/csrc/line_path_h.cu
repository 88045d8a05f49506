// Line-transform chain, lengths 80, 90.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 80>;
template struct LinePath<float, 80>;
template struct LinePath<double, 90>;
template struct LinePath<float, 90>;
}  // namespace jdft
