// The operators of degree 1 (kernels and their launches).
#include "operators.cuh"

namespace nhmf {
template struct Operators<1>;
}  // namespace nhmf
