// FP32 instantiation of the sine-transform passes, N <= 1024.
#include "csl_pass_impl.cuh"

namespace csl {
#define CASE(NN) CSL_INSTANTIATE_PASS(float, NN, 0)
CSL_FOR_EACH_N(CASE)
#undef CASE
CSL_INSTANTIATE_PASS(float, 512, 1)
CSL_INSTANTIATE_PASS(float, 512, 2)
CSL_INSTANTIATE_PASS(float, 1024, 1)
CSL_INSTANTIATE_PASS(float, 1024, 2)
}  // namespace csl
