// Line-transform chain, lengths 50, 54, 108.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 50>;
template struct LinePath<float, 50>;
template struct LinePath<double, 54>;
template struct LinePath<float, 54>;
template struct LinePath<double, 108>;
template struct LinePath<float, 108>;
}  // namespace jdft
