// Line-transform chain, lengths 100, 256.
#include "line_path_impl.cuh"

namespace jdft {
template struct LinePath<double, 100>;
template struct LinePath<float, 100>;
template struct LinePath<double, 256>;
template struct LinePath<float, 256>;
}  // namespace jdft
