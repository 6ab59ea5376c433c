// The operators of degree 2 (kernels and their launches).
#include "operators.cuh"

namespace nhmf {
template struct Operators<2>;
}  // namespace nhmf
