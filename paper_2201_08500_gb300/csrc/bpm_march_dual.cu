// Launches of the march with 2 N/16 threads a channel (bpm_dual.cuh).
#include <cuda_runtime.h>

#include "bpm_dual.cuh"

namespace bpm {

namespace {

template <int N, int SPLIT>
__global__ void __launch_bounds__(Dual<N, SPLIT>::kThreads, 1) march_dual_kernel(MarchArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  Dual<N, SPLIT>::run(A, smem);
}

template <int SPLIT>
cudaError_t launch_one(int blocks, const MarchArgs& a, cudaStream_t s) {
  using D = Dual<2048, SPLIT>;
  march_dual_kernel<2048, SPLIT>
      <<<blocks, D::kThreads, share_smem(D::smem_bytes(), a.per_sm), s>>>(a);
  return cudaGetLastError();
}

template <int SPLIT>
cudaError_t attr_one() {
  return cudaFuncSetAttribute(march_dual_kernel<2048, SPLIT>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              int(share_smem(Dual<2048, SPLIT>::smem_bytes(), 1)));
}

}  // namespace

// One block an SM: r channels an SM take r steps' time (in equal shares), the other
// forms the time of two up to r = 2 (us a step: first order 2.64 r against 4.46,
// Strang 3.28 r against 5.14, fourth order 8.4 r against 16.1).
bool march_dual_use(int n, int split_order, int n_ch, int sms) {
  const double r = split_order == 1 ? 1.65 : split_order == 2 ? 1.55 : 1.9;
  return n == 2048 && n_ch <= r * sms;
}

size_t march_dual_smem_bytes(int n) { return n == 2048 ? Dual<2048, 1>::smem_bytes() : 0; }

cudaError_t launch_march_dual(int n, int blocks, const MarchArgs& a, cudaStream_t s) {
  if (n != 2048) return cudaErrorInvalidValue;
  if (a.split_order == 2) return launch_one<2>(blocks, a, s);
  if (a.split_order == 4) return launch_one<4>(blocks, a, s);
  return launch_one<1>(blocks, a, s);
}

cudaError_t march_set_attributes_dual() {
  cudaError_t r[] = {attr_one<1>(), attr_one<2>(), attr_one<4>()};
  for (cudaError_t e : r)
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace bpm
