// FP64 instantiation of the sine-transform passes, N = 1024.
#include "csl_pass_impl.cuh"

namespace csl {
CSL_INSTANTIATE_PASS(double, 1024, 1)
CSL_INSTANTIATE_PASS(double, 1024, 2)
}  // namespace csl
