// FP64 instantiation of the sine-transform passes, N = 256.
#include "csl_pass_impl.cuh"

namespace csl {
CSL_INSTANTIATE_PASS(double, 256, 0)
CSL_INSTANTIATE_PASS(double, 256, 1)
}  // namespace csl
