// FP64 instantiation of the sine-transform passes, N = 128.
#include "csl_pass_impl.cuh"

namespace csl {
CSL_INSTANTIATE_PASS(double, 128, 0)
CSL_INSTANTIATE_PASS(double, 128, 1)
}  // namespace csl
