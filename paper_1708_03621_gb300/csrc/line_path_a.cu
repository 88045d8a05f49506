// Line-transform chain, lengths 12, 16, 24, 128.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 12>;
template struct LinePath<float, 12>;
template struct LinePath<double, 16>;
template struct LinePath<float, 16>;
template struct LinePath<double, 24>;
template struct LinePath<float, 24>;
template struct LinePath<double, 128>;
template struct LinePath<float, 128>;
}  // namespace jdft
