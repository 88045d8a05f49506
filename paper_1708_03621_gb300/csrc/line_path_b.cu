// Line-transform chain, lengths 25, 27, 30, 75.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 25>;
template struct LinePath<float, 25>;
template struct LinePath<double, 27>;
template struct LinePath<float, 27>;
template struct LinePath<double, 30>;
template struct LinePath<float, 30>;
template struct LinePath<double, 75>;
template struct LinePath<float, 75>;
}  // namespace jdft
