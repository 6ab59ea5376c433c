// The operators of degree 4 (kernels and their launches).
#include "operators.cuh"

namespace nhmf {
template struct Operators<4>;
}  // namespace nhmf
