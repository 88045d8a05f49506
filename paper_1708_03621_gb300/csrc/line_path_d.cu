// Line-transform chain, lengths 45, 48, 125.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 45>;
template struct LinePath<float, 45>;
template struct LinePath<double, 48>;
template struct LinePath<float, 48>;
template struct LinePath<double, 125>;
template struct LinePath<float, 125>;
}  // namespace jdft
