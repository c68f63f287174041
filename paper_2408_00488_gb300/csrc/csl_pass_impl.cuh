// Launch wrappers of the sine-transform passes for one real type, length and
// variant (launch_*_n).  csl_pass32.cu holds every FP32 length; the FP64 ones are
// spread over csl_pass64*.cu so that they compile in parallel.  The dispatch over
// the lengths is csl_pass_dispatch.cu.
#pragma once
#include "csl_passes.cuh"

namespace csl {

template <typename T, int N, int W>
cudaError_t launch_row_n(int load, int store, const RowArgs<T>& a, const PassLaunch& L, cudaStream_t s,
                         const RowArgs<T>* batch, int nsys) {
  const int grid = batch ? L.blocks * nsys : L.blocks;
  const int bps = L.blocks;
  if constexpr (sizeof(T) == 4) {  // FP32 transform, FP64 vectors
    if (load == LOAD_LANCZOS_V64 && store == STORE_T)
      return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_LANCZOS_V64, STORE_T>, grid, L.threads, L.smem, s, a, batch,
                      bps);
    if (load == LOAD_T && store == STORE_Z_UPDATE_V64)
      return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_T, STORE_Z_UPDATE_V64>, grid, L.threads, L.smem, s, a, batch,
                      bps);
  } else {  // the FP64 form's vectors are FP64 in the plain modes
    if (load == LOAD_LANCZOS_V64) load = LOAD_LANCZOS;
    if (store == STORE_Z_UPDATE_V64) store = STORE_Z_UPDATE;
  }
  if (load == LOAD_V && store == STORE_T)
    return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_V, STORE_T>, grid, L.threads, L.smem, s, a, batch, bps);
  else if (load == LOAD_LANCZOS && store == STORE_T)
    return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_LANCZOS, STORE_T>, grid, L.threads, L.smem, s, a, batch, bps);
  else if (load == LOAD_T && store == STORE_Z)
    return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_T, STORE_Z>, grid, L.threads, L.smem, s, a, batch, bps);
  else if (load == LOAD_T && store == STORE_Z_UPDATE)
    return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_T, STORE_Z_UPDATE>, grid, L.threads, L.smem, s, a, batch, bps);
  else if (load == LOAD_T && store == STORE_D)
    return launch_k(L.pdl != 0, k_row<T, N, W, LOAD_T, STORE_D>, grid, L.threads, L.smem, s, a, batch, bps);
  return cudaErrorInvalidValue;
}

template <typename T, int N, int W>
cudaError_t launch_strided_n(bool mid, const StridedArgs<T>& a, const PassLaunch& L, cudaStream_t s,
                             const StridedArgs<T>* batch, int nsys) {
  const int grid = batch ? L.blocks * nsys : L.blocks;
  if (mid) return launch_k(L.pdl != 0, k_strided<T, N, W, true>, grid, L.threads, L.smem, s, a, batch, L.blocks);
  return launch_k(L.pdl != 0, k_strided<T, N, W, false>, grid, L.threads, L.smem, s, a, batch, L.blocks);
}

template <typename T, int N, int W>
cudaError_t set_pass_attrs_n() {
  cudaError_t e = cudaSuccess;
#define SETA(...) \
  if (e == cudaSuccess) e = allow_dyn_smem((const void*)__VA_ARGS__);
  SETA(k_row<T, N, W, LOAD_V, STORE_T>)
  SETA(k_row<T, N, W, LOAD_LANCZOS, STORE_T>)
  SETA(k_row<T, N, W, LOAD_T, STORE_Z>)
  SETA(k_row<T, N, W, LOAD_T, STORE_Z_UPDATE>)
  SETA(k_row<T, N, W, LOAD_T, STORE_D>)
  SETA(k_strided<T, N, W, true>)
  SETA(k_strided<T, N, W, false>)
  if constexpr (sizeof(T) == 4) {
    SETA(k_row<T, N, W, LOAD_LANCZOS_V64, STORE_T>)
    SETA(k_row<T, N, W, LOAD_T, STORE_Z_UPDATE_V64>)
  }
#undef SETA
  return e;
}

#define CSL_INSTANTIATE_PASS(T, N, W)                                                                            \
  template cudaError_t launch_row_n<T, N, W>(int, int, const RowArgs<T>&, const PassLaunch&, cudaStream_t,       \
                                             const RowArgs<T>*, int);                                            \
  template cudaError_t launch_strided_n<T, N, W>(bool, const StridedArgs<T>&, const PassLaunch&, cudaStream_t,   \
                                                 const StridedArgs<T>*, int);                                    \
  template cudaError_t set_pass_attrs_n<T, N, W>();

}  // namespace csl
