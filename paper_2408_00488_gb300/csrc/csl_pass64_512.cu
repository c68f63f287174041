// FP64 instantiation of the sine-transform passes, N = 512.
#include "csl_pass_impl.cuh"

namespace csl {
CSL_INSTANTIATE_PASS(double, 512, 1)
CSL_INSTANTIATE_PASS(double, 512, 2)
}  // namespace csl
