// Line-transform chain, lengths 72, 96.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 72>;
template struct LinePath<float, 72>;
template struct LinePath<double, 96>;
template struct LinePath<float, 96>;
}  // namespace jdft
