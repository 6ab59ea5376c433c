// The operators of degree 3 (kernels and their launches).
#include "operators.cuh"

namespace nhmf {
template struct Operators<3>;
}  // namespace nhmf
