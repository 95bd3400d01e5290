// Thin-film (2D) persistent kernel for one film on the whole grid, and its launch helpers.
// The method and the device code it runs are in mf_film.cuh.
#include "mf_film.cuh"

namespace mf {

// one film on the whole grid
template <typename T>
__global__ void __launch_bounds__(NT, FILM_CTAS) film_kernel(const Desc* __restrict__ dg, KernelArgs a) {
  film_main<T>(*dg, a, (int)blockIdx.x, gridDim.x);
}

// the core's exchange buffer and twiddle tables
size_t kernel_smem_bytes(const Desc& d) {
  if (d.dim == 2) return film_smem_bytes(d);
  return bulk_smem_bytes(d);
}

int film_max_blocks(int precision, size_t smem) {
  int nb = 0;
  if (precision) {
    cudaFuncSetAttribute(film_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FILM_SMEM_MAX);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, film_kernel<float>, NT, smem);
  } else {
    cudaFuncSetAttribute(film_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FILM_SMEM_MAX);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, film_kernel<double>, NT, smem);
  }
  return nb;
}

cudaError_t film_launch(int precision, const Desc& d, const KernelArgs& a, cudaStream_t s) {
  const Desc* dg = d.dev;
  KernelArgs aa = a;
  void* args[] = {&dg, &aa};
  const size_t smem = kernel_smem_bytes(d);
  const void* fn = precision ? (const void*)film_kernel<float> : (const void*)film_kernel<double>;
  return cudaLaunchCooperativeKernel(fn, dim3(d.grid), dim3(NT), args, smem, s);
}

}  // namespace mf
