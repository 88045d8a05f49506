// Line-transform chain, lengths 32, 36, 40, 120.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 32>;
template struct LinePath<float, 32>;
template struct LinePath<double, 36>;
template struct LinePath<float, 36>;
template struct LinePath<double, 40>;
template struct LinePath<float, 40>;
template struct LinePath<double, 120>;
template struct LinePath<float, 120>;
}  // namespace jdft
