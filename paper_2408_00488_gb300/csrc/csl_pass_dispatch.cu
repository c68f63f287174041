// Dispatch of the sine-transform passes over the transform lengths; the
// kernels are instantiated by csl_pass32.cu and csl_pass64*.cu.
#include "csl_passes.cuh"

namespace csl {

// the kernels' variant of a requested one (the FP64 form has no variant 0 at N >= 512)
template <typename T, int N, int W>
constexpr int variant_of = sizeof(T) == 8 && N >= 512 && W == 0 ? 1 : W;

template <typename T>
cudaError_t launch_row(int N, int wide, int load, int store, const RowArgs<T>& a, const PassLaunch& L,
                       cudaStream_t s, const RowArgs<T>* batch, int nsys) {
  if (pass_is_big(N)) return launch_row_big<T>(N, load, store, a, L, s, batch, nsys);
  switch (N) {
#define CASE(NN)                                                                       \
  case NN:                                                                             \
    if constexpr (NN >= 512) {                                                         \
      if (wide == 1) return launch_row_n<T, NN, 1>(load, store, a, L, s, batch, nsys); \
      if (wide == 2) return launch_row_n<T, NN, 2>(load, store, a, L, s, batch, nsys); \
    }                                                                                  \
    if constexpr (sizeof(T) == 8 && (NN == 128 || NN == 256)) {                        \
      if (wide == 1) return launch_row_n<T, NN, 1>(load, store, a, L, s, batch, nsys); \
    }                                                                                  \
    return launch_row_n<T, NN, variant_of<T, NN, 0>>(load, store, a, L, s, batch, nsys);
    CSL_FOR_EACH_N(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_strided(int N, int wide, bool mid, const StridedArgs<T>& a, const PassLaunch& L,
                           cudaStream_t s, const StridedArgs<T>* batch, int nsys) {
  if constexpr (sizeof(T) == 4) {
    if (L.tc) return launch_strided_tc(N, L.tc, mid, a, L, s, batch, nsys);
  }
  if (pass_is_big(N)) return launch_strided_big<T>(N, mid, a, L, s, batch, nsys);
  switch (N) {
#define CASE(NN)                                                                    \
  case NN:                                                                          \
    if constexpr (NN >= 512) {                                                      \
      if (wide == 1) return launch_strided_n<T, NN, 1>(mid, a, L, s, batch, nsys);  \
      if (wide == 2) return launch_strided_n<T, NN, 2>(mid, a, L, s, batch, nsys);  \
    }                                                                               \
    if constexpr (sizeof(T) == 8 && (NN == 128 || NN == 256)) {                     \
      if (wide == 1) return launch_strided_n<T, NN, 1>(mid, a, L, s, batch, nsys);  \
    }                                                                               \
    return launch_strided_n<T, NN, variant_of<T, NN, 0>>(mid, a, L, s, batch, nsys);
    CSL_FOR_EACH_N(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t set_pass_attrs() {
  cudaError_t e = cudaSuccess;
#define CASE(NN) \
  if (e == cudaSuccess) e = set_pass_attrs_n<T, NN, variant_of<T, NN, 0>>();
  CSL_FOR_EACH_N(CASE)
#undef CASE
  if (e == cudaSuccess) e = set_pass_attrs_n<T, 512, 1>();
  if (e == cudaSuccess) e = set_pass_attrs_n<T, 512, 2>();
  if (e == cudaSuccess) e = set_pass_attrs_n<T, 1024, 1>();
  if (e == cudaSuccess) e = set_pass_attrs_n<T, 1024, 2>();
  if constexpr (sizeof(T) == 8) {
    if (e == cudaSuccess) e = set_pass_attrs_n<T, 128, 1>();
    if (e == cudaSuccess) e = set_pass_attrs_n<T, 256, 1>();
  }
  if (e == cudaSuccess) e = set_pass_attrs_big<T>();
  return e;
}

#define INSTANTIATE(T)                                                                                           \
  template cudaError_t launch_row<T>(int, int, int, int, const RowArgs<T>&, const PassLaunch&, cudaStream_t,     \
                                     const RowArgs<T>*, int);                                                    \
  template cudaError_t launch_strided<T>(int, int, bool, const StridedArgs<T>&, const PassLaunch&, cudaStream_t, \
                                         const StridedArgs<T>*, int);                                            \
  template cudaError_t set_pass_attrs<T>();
INSTANTIATE(float)
INSTANTIATE(double)

}  // namespace csl
