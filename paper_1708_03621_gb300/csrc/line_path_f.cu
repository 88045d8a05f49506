// Line-transform chain, lengths 60, 64, 81.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 60>;
template struct LinePath<float, 60>;
template struct LinePath<double, 64>;
template struct LinePath<float, 64>;
template struct LinePath<double, 81>;
template struct LinePath<float, 81>;
}  // namespace jdft
