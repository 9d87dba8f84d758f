// Launches of the march with 8 N/16 threads a channel (bpm_quad.cuh).
#include <cuda_runtime.h>

#include "bpm_quad.cuh"

namespace bpm {

namespace {

template <int N, int SPLIT>
__global__ void __launch_bounds__(Quad<N, SPLIT>::kThreads, 768 / Quad<N, SPLIT>::kThreads)
    march_quad_kernel(MarchArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  Quad<N, SPLIT>::run(A, smem);
}

template <int N, int SPLIT>
cudaError_t launch_one(int blocks, const MarchArgs& a, cudaStream_t s) {
  march_quad_kernel<N, SPLIT><<<blocks, Quad<N, SPLIT>::kThreads,
                                share_smem(Quad<N, SPLIT>::smem_bytes(), a.per_sm), s>>>(a);
  return cudaGetLastError();
}

template <int N>
cudaError_t launch_order(int blocks, const MarchArgs& a, cudaStream_t s) {
  if (a.split_order == 2) return launch_one<N, 2>(blocks, a, s);
  if (a.split_order == 4) return launch_one<N, 4>(blocks, a, s);
  return launch_one<N, 1>(blocks, a, s);
}

}  // namespace

// The step times of the forms for n_ch channels, in us (measured over 1 ... 2500
// channels, 152 SMs).  Up to 3 (256, 512 points) or 1 (1024) channels an SM
// this form ends in 0.6, 1.0 and 1.6 us; beyond, it takes its share of an SM's
// time per channel, and the resident form a whole wave of 16, 8 or 4 channels
// an SM whether full or not.  E.g. first order, 512 points: 201 channels 1.32
// against 3.85, 760 3.1 against 4.05, 1024 4.1 against 4.2.
bool march_quad_use(int n, int split_order, int n_ch, int sms) {
  const int o = split_order == 1 ? 0 : split_order == 2 ? 1 : 2;
  static constexpr double each[3][3] = {{0.25, 0.275, 0.85}, {0.61, 0.66, 2.31}, {1.64, 1.84, 5.24}};
  static constexpr double wave[3][3] = {{2.9, 4.35, 10.3}, {4.2, 5.2, 14.3}, {4.2, 5.2, 14.4}};
  if (n > 1024 || n_ch < 1 || sms < 1) return false;
  const int i = n == 256 ? 0 : n == 512 ? 1 : 2, per = n == 256 ? 16 : n == 512 ? 8 : 4;
  return each[i][o] * ((n_ch + sms - 1) / sms) < wave[i][o] * ((n_ch + per * sms - 1) / (per * sms));
}

size_t march_quad_smem_bytes(int n) {
  return n == 256   ? Quad<256, 1>::smem_bytes()
         : n == 512 ? Quad<512, 1>::smem_bytes()
                    : Quad<1024, 1>::smem_bytes();
}

cudaError_t launch_march_quad(int n, int blocks, const MarchArgs& a, cudaStream_t s) {
  if (n == 256) return launch_order<256>(blocks, a, s);
  if (n == 512) return launch_order<512>(blocks, a, s);
  if (n == 1024) return launch_order<1024>(blocks, a, s);
  return cudaErrorInvalidValue;
}

namespace {
template <int N, int SPLIT>
cudaError_t attr_one() {
  return cudaFuncSetAttribute(march_quad_kernel<N, SPLIT>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              int(share_smem(Quad<N, SPLIT>::smem_bytes(), 1)));
}
}  // namespace

cudaError_t march_set_attributes_quad() {
  cudaError_t r[] = {attr_one<256, 1>(), attr_one<256, 2>(),  attr_one<256, 4>(),
                     attr_one<512, 1>(), attr_one<512, 2>(),  attr_one<512, 4>(),
                     attr_one<1024, 1>(), attr_one<1024, 2>(), attr_one<1024, 4>()};
  for (cudaError_t e : r)
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace bpm
