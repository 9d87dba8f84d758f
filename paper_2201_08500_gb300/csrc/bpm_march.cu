// Resident split-step march of the two-beam BPM (Eq. fov10, first-order
// splitting a1 = b1 = 1 of Eq. split-op), one frequency channel per group of
// T = N/16 threads.  Both envelopes stay in registers for the whole march; per
// step each thread
//   1. prefetches its 16 deformation factors c(x, z_n) = Pi exp(+i h u) for the
//      coupling at the end of the step (coalesced, latency hidden by the FFTs);
//   2. runs the forward FFT of E0 and Eh (radix-16 register butterflies with
//      shared-memory exchanges, see bpm_fft.cuh);
//   3. multiplies the digit-reversed spectra by the tilted propagators
//      p+- = exp(i dz [sqrt(k^2 - (q +- h/2)^2) - k]) (Eq. fov4 with the shifted
//      spectrum after Eq. fov10), stored as FP32 hi + lo pairs that also carry
//      1/N and the FFT round-trip gain correction;
//   4. runs the inverse FFT (exact adjoint of the forward);
//   5. couples the envelopes pointwise (Eq. fov10 with Eq. Authier):
//        E0 <- a E0 + b+ c Eh,   Eh <- a Eh + b- conj(c) E0   inside the crystal.
// At the end of the launch the fields are written back and the per-channel
// reflectivity / transmissivity sums are reduced in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "bpm_march_impl.cuh"

namespace bpm {

int march_threads_per_channel(int n) { return n / 16; }

int march_max_group(int n) {
  switch (n) {
    case 256: return 16;
    case 512: return 8;
    case 1024: return 4;
    case 2048: return 2;
    default: return 1;
  }
}

// Form and channels per block of a plan that names none, over 1 ... 2500
// channels and 152 SMs (us a step, this form against the next best):
//  * 256, 512 points: one channel a block while march_quad_use holds (3.1 against
//    4.6 at 760 channels of 512), then at 256 sixteen (2.9 against 5.3 at 2000);
//  * 1024: one channel a block up to 15/8 an SM, fourth order and Strang up to two
//    (1.7 against 3.1 at 155 channels, 3.26 against 3.07 at 300; fourth order 10.5
//    against 13.2 at 304); beyond, TMEM tables, two channels a block (3.1 against
//    4.6 at 300, 16.7 against 19.1 at 2500), fourth order the parked form (18.7
//    against 23 at 611);
//  * 2048: one channel a block while march_dual_use holds (2.6 against 4.1 at 152),
//    then TMEM tables (13.2 against 16.4 at 1024);
//    fourth order the parked form beyond two channels an SM (21.4 against 29.2
//    at 456, but 16.4 against 16.1 at 304);
//  * 4096: the resident form up to one channel an SM (5.1 against 5.4), then
//    TMEM tables (7.9 against 9.8 at 230, 29.0 against 37.4 at 1024), fourth
//    order parked (27.3 against 34.2 at 230);
//  * 8192: TMEM tables (form 0 is the same kernel).
void march_default_form(int n, int split_order, int n_ch, int sms, int* form, int* group) {
  *form = 0;
  *group = 1;
  const int o = split_order;
  switch (n) {
    case 256:
      if (!march_quad_use(n, o, n_ch, sms)) *group = march_max_group(n);
      break;
    case 1024:
      if (8 * n_ch > (o == 1 ? 15 : 16) * sms) {
        *form = o == 4 ? 2 : 3;
        *group = o == 4 ? 1 : 2;
      }
      break;
    case 2048:
      if (march_dual_use(n, o, n_ch, sms)) break;
      if (o != 4)
        *form = 3;
      else if (n_ch > 2 * sms)
        *form = 2;
      break;
    case 4096:
      if (n_ch > sms) *form = o == 4 ? 2 : 3;
      break;
    default: break;
  }
}

namespace {

// us a step with k = 1, 2, ... blocks on every SM (as many as fit), 152 SMs.
struct StepTimes {
  int n, form, order;  // form 0: bpm_quad.cuh, bpm_dual.cuh
  float t[8];
};
constexpr StepTimes kStepTimes[] = {
    {256, 0, 1, {0.62f, 0.74f, 0.84f, 1.04f, 1.25f, 1.48f}},
    {256, 0, 2, {0.92f, 1.01f, 1.11f, 1.25f, 1.43f, 1.64f}},
    {256, 0, 4, {2.68f, 2.99f, 3.26f, 3.89f, 4.57f, 5.33f}},
    {512, 0, 1, {0.98f, 1.35f, 1.83f}},
    {512, 0, 2, {1.16f, 1.48f, 1.97f}},
    {512, 0, 4, {3.73f, 5.29f, 6.94f}},
    {1024, 0, 1, {1.64f}},
    {1024, 0, 2, {1.84f}},
    {1024, 0, 4, {5.24f}},
    {1024, 2, 1, {2.86f, 3.15f, 4.53f, 4.85f, 5.95f, 6.45f, 7.82f, 8.23f}},
    {1024, 2, 4, {9.46f, 12.1f, 14.8f, 15.7f, 18.9f, 20.2f, 24.2f, 25.4f}},
    {1024, 3, 1, {3.06f, 4.24f, 5.74f, 7.35f}},
    {1024, 3, 2, {3.92f, 4.83f, 6.40f, 8.29f}},
    {2048, 0, 1, {2.64f}},
    {2048, 0, 2, {3.28f}},
    {2048, 0, 4, {8.40f}},
    {2048, 2, 1, {4.12f, 5.30f, 6.85f, 8.71f}},
    {2048, 2, 4, {13.8f, 16.0f, 21.7f, 27.4f}},
    {2048, 3, 1, {4.11f, 4.46f, 6.18f, 7.97f}},
    {2048, 3, 2, {4.91f, 5.14f, 7.13f, 8.91f}},
    {4096, 2, 1, {6.65f, 9.78f}},
    {4096, 2, 4, {18.2f, 28.7f}},
    {4096, 3, 1, {5.27f, 8.72f}},
    {4096, 3, 2, {6.04f, 9.33f}},
    {8192, 0, 1, {10.5f}},
    {8192, 0, 2, {11.6f}},
    {8192, 0, 4, {34.5f}},
};

}  // namespace

// With r blocks' worth of channels an SM, the launch of whole channels takes the
// time of ceil(r) blocks on an SM while they fit and ceil(r) / kmax that of the
// kmax that do beyond; equal shares on k <= r blocks an SM take r / k of theirs.
// E.g. (us a step, whole channels -> shares) 512 channels of 8192 points
// 41.3 -> 35.6; 400 of 4096 13.0 -> 11.5; 700 of 2048 10.1 -> 9.1; 611 of 1024
// 5.7 -> 4.3, 1024 of 1024 7.3 -> 6.4 with three blocks an SM.
// Beyond kmax blocks that end at different times fill some of the gap by
// themselves where several share an SM (1024 of 4096: 29.0, in shares 29.3): 5 %
// has to be expected there.  A share's extra piece costs about a step, so short
// runs take whole channels.
int march_shares(int n, int split_order, int form, int group, int n_ch, int n_steps, int sms) {
  if (n == 8192) form = 0;
  if (n_steps < 16 || sms < 1 || form == 1) return 0;
  if (form == 0 && n != 8192 &&
      (group != 1 || !(march_quad_use(n, split_order, n_ch, sms) ||
                       march_dual_use(n, split_order, n_ch, sms))))
    return 0;
  const StepTimes* s = nullptr;
  for (const StepTimes& row : kStepTimes)
    if (row.n == n && row.form == form && row.order == split_order) s = &row;
  if (!s) return 0;
  int kmax = 1;
  while (kmax < 8 && s->t[kmax] > 0.f) ++kmax;
  const double r = double((n_ch + group - 1) / group) / sms;
  const int up = int(std::ceil(r)), k = std::min(int(r), kmax);
  if (k < 1 || k * sms * group >= n_ch) return 0;
  const double whole = up <= kmax ? s->t[up - 1] : double(up) / kmax * s->t[kmax - 1];
  const double shared = double(n_ch) / (group * sms) / k * s->t[k - 1];
  return whole > (up > kmax && kmax > 1 ? 1.05 : 1.015) * shared ? k : 0;
}

size_t march_smem_bytes(int n, int group) {
#define BPM_SMEM_CASE(NN, GG) \
  if (n == NN && group == GG) return MarchBody<NN, GG, 1, 0>::type::smem_bytes();
  BPM_SMEM_CASE(256, 1) BPM_SMEM_CASE(256, 16)
  BPM_SMEM_CASE(512, 1) BPM_SMEM_CASE(512, 8)
  BPM_SMEM_CASE(1024, 1) BPM_SMEM_CASE(1024, 4)
  BPM_SMEM_CASE(2048, 1) BPM_SMEM_CASE(2048, 2)
  BPM_SMEM_CASE(4096, 1) BPM_SMEM_CASE(8192, 1)
#undef BPM_SMEM_CASE
  return 0;
}

cudaError_t march_set_attributes() {
  cudaError_t e = march_set_attributes_strang();
  if (cudaError_t e4 = march_set_attributes_split4(); e4 != cudaSuccess) e = e4;
  if (cudaError_t eq = march_set_attributes_quad(); eq != cudaSuccess) e = eq;
  if (cudaError_t ed = march_set_attributes_dual(); ed != cudaSuccess) e = ed;
  cudaError_t r[] = {attr_one<256, 1, 1>(),  attr_one<256, 16, 1>(),
                     attr_one<512, 1, 1>(),  attr_one<512, 8, 1>(),
                     attr_one<1024, 1, 1>(), attr_one<1024, 4, 1>(),
                     attr_one<2048, 1, 1>(), attr_one<2048, 2, 1>(),
                     attr_one<4096, 1, 1>(), attr_one<8192, 1, 1>()};
  for (cudaError_t x : r)
    if (x != cudaSuccess) e = x;
  return e;
}

cudaError_t launch_march(int n, int group, int blocks, const MarchArgs& a, cudaStream_t s) {
  int sms = 0;
  if (group == 1 && device_ready(&sms) && march_quad_use(n, a.split_order, a.n_ch, sms))
    return launch_march_quad(n, blocks, a, s);
  if (group == 1 && sms > 0 && a.ext && a.twiddle_p &&  // (not the allocation-free entry)
      march_dual_use(n, a.split_order, a.n_ch, sms))
    return launch_march_dual(n, blocks, a, s);
  if (a.split_order == 2) return launch_march_strang(n, group, blocks, a, s);
  if (a.split_order == 4) return launch_march_split4(n, group, blocks, a, s);
#define BPM_LAUNCH_CASE(NN, GG) \
  if (n == NN && group == GG) return launch_one<NN, GG, 1>(blocks, a, s);
  BPM_LAUNCH_CASE(256, 1) BPM_LAUNCH_CASE(256, 16)
  BPM_LAUNCH_CASE(512, 1) BPM_LAUNCH_CASE(512, 8)
  BPM_LAUNCH_CASE(1024, 1) BPM_LAUNCH_CASE(1024, 4)
  BPM_LAUNCH_CASE(2048, 1) BPM_LAUNCH_CASE(2048, 2)
  BPM_LAUNCH_CASE(4096, 1) BPM_LAUNCH_CASE(8192, 1)
#undef BPM_LAUNCH_CASE
  return cudaErrorInvalidValue;
}

}  // namespace bpm
