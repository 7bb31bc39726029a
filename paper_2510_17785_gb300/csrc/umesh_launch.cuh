// Definitions of the unstructured-mesh launchers declared in umesh_kern.cuh,
// included only by the explicit-instantiation units umesh_k*.cu.
#pragma once
#include <atomic>

#include "umesh_kern.cuh"

namespace pmg {

template <int DIM, int Q, typename T>
int ucell_apply_q(const T* u, const T* G, const int32_t* cd, const uint8_t* bnd, int64_t nc, T* Y,
                         cudaStream_t s) {
  constexpr int CPB = ucpb(Q);
  constexpr size_t sm = ucell_smem<DIM, Q, T>();
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr[dev & 63]) {
    if (cudaFuncSetAttribute(k_ucell_apply<DIM, Q, T, CPB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) !=
        cudaSuccess)
      return ST_CUDA;
    attr[dev & 63] = true;
  }
  const int64_t grid = (nc + CPB - 1) / CPB;
  k_ucell_apply<DIM, Q, T, CPB><<<(unsigned)grid, 128, sm, s>>>(u, G, cd, bnd, nc, Y);
  return cudaPeekAtLastError() == cudaSuccess ? ST_OK : ST_CUDA;
}

template <int DIM, int P, typename T>
int upatch_launch_P(int mode, const UPatchArgs<T>& a, int grid, cudaStream_t s) {
  constexpr size_t sm0 = upatch_smem<DIM, P, T>();
  if constexpr (sm0 > 227 * 1024) {
    return ST_UNSUPPORTED;
  } else {
    // the workspace slice joins the shared memory when the caller says it fits
    const size_t sm = a.ws_shared ? upatch_smem_aligned<DIM, P, T>() + a.ws_stride * sizeof(T) : sm0;
    if (sm > 227 * 1024) return ST_ARG;
    // the size varies from launch to launch, and contexts may launch from several
    // host threads: the kernel's limit is set to the most a CTA can have, once per
    // device, so that no thread lowers what another one has raised
    constexpr int kMostSmem = 227 * 1024;
    int dev = 0;
    cudaGetDevice(&dev);
    static std::atomic<bool> raised[2][64] = {};
    const bool sweep = mode == MODE_SWEEP;
    if (!raised[sweep][dev & 63].load()) {
      const void* kernel = sweep ? (const void*)k_upatch<DIM, P, T, MODE_SWEEP>
                                 : (const void*)k_upatch<DIM, P, T, MODE_LOCAL>;
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem) != cudaSuccess)
        return ST_CUDA;
      raised[sweep][dev & 63].store(true);
    }
    if (sweep) {
      k_upatch<DIM, P, T, MODE_SWEEP><<<grid, unt(P), sm, s>>>(a);
    } else {
      k_upatch<DIM, P, T, MODE_LOCAL><<<grid, unt(P), sm, s>>>(a);
    }
    return cudaPeekAtLastError() == cudaSuccess ? ST_OK : ST_CUDA;
  }
}

// bytes of dynamic shared memory of the patch kernel without its workspace
template <int DIM, int P, typename T>
size_t upatch_smem_base() {
  return upatch_smem_aligned<DIM, P, T>();
}

template <int DIM, int P>
int ulanczos_launch(const UPatchArgs<double>& a, const ULanczos& z, int grid, cudaStream_t s) {
  constexpr size_t sm = upatch_smem<DIM, P, double>();
  if constexpr (sm > 200 * 1024) {
    return ST_UNSUPPORTED;
  } else {
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (!attr[dev & 63]) {
      if (cudaFuncSetAttribute(k_ulanczos<DIM, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        return ST_CUDA;
      attr[dev & 63] = true;
    }
    k_ulanczos<DIM, P><<<grid, unt(P), sm, s>>>(a, z);
    return cudaPeekAtLastError() == cudaSuccess ? ST_OK : ST_CUDA;
  }
}

#define PMG_UMESH_INSTANTIATE(DIM, P, T)                                                                     \
  template int upatch_launch_P<DIM, P, T>(int, const UPatchArgs<T>&, int, cudaStream_t);                   \
  template int ucell_apply_q<DIM, P, T>(const T*, const T*, const int32_t*, const uint8_t*, int64_t, T*, \
                                        cudaStream_t);
#define PMG_UMESH_INSTANTIATE_LANCZOS(DIM, P) \
  template int ulanczos_launch<DIM, P>(const UPatchArgs<double>&, const ULanczos&, int, cudaStream_t);

}  // namespace pmg
