// FP64 instantiation of the sine-transform passes, N <= 64.
#include "csl_pass_impl.cuh"

namespace csl {
CSL_INSTANTIATE_PASS(double, 4, 0)
CSL_INSTANTIATE_PASS(double, 8, 0)
CSL_INSTANTIATE_PASS(double, 16, 0)
CSL_INSTANTIATE_PASS(double, 32, 0)
CSL_INSTANTIATE_PASS(double, 64, 0)
}  // namespace csl
