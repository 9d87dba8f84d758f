// Work-queue form of the resident march: one persistent launch marches many
// plans (instances of different Nx, z-step counts and channel counts).
//
// Items are (plan, first channel) pairs sorted longest-first on the host.
// Every block repeatedly takes the next item with an atomic counter: at Nx >=
// 1024 one channel in the parked form with tables in tensor memory; below, G =
// 256 / T channels (T = Nx/16 threads each) of the resident form, and single
// channels of what fills no such item with 8 T threads (bpm_quad.cuh).  One
// queue per size, order and kind.  The counters live in global memory and are
// cleared once a round, before its first queue.  No block waits for another's
// items; block 0 of a queue waits, at its end, for the queue before it.
#include <cuda_runtime.h>

#include "bpm_parked.cuh"
#include "bpm_quad.cuh"
#include "bpm_resident.cuh"

namespace bpm {

namespace {

// Queues of a round overlap: a launch that follows another one starts when all
// blocks of that one are running (programmatic dependent launch), and its blocks
// take the SMs that the first queue's empty end leaves, instead of waiting for
// its longest item.  They need nothing of one another.  Block 0 of each launch
// waits for the launch before it to complete, so that completion of the last
// means completion of all (and the others give their SM back at once).  Ten
// uneven instances in four queues: a round of 40.6 ms -> 35.8.
BPM_DEV void chain_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
BPM_DEV void chain_end() {
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kSmallThreads = 256;

template <int N>
constexpr size_t item_smem() {
  return Resident<N, kSmallThreads / (N / 16)>::smem_bytes();
}

constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }

constexpr size_t kSmallSmem = cmax(item_smem<256>(), item_smem<512>());
static_assert(Resident<256, 16, 4>::smem_bytes() <= kSmallSmem &&
                  Resident<256, 16, 2>::smem_bytes() <= kSmallSmem,
              "every order's resident slot fits the first-order bound");

// SPLIT: Eq. split-op order of the queue's plans (1, 2 or 4).  The resident
// body keeps its tables in shared memory only at first and second order, so
// kSmallSmem (first order) bounds every order.
template <int SPLIT>
__global__ void __launch_bounds__(kSmallThreads, 1)
    batch_kernel(const MarchArgs* __restrict__ plans, const BatchItem* __restrict__ items,
                 int n_items, int* counter) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= n_items) break;
    const BatchItem item = items[it];
    const MarchArgs& A = plans[item.plan];
    switch (item.n) {
      case 256: Resident<256, 16, SPLIT>::run_item(A, item.ch0, smem); break;
      case 512: Resident<512, 8, SPLIT>::run_item(A, item.ch0, smem); break;
      default: break;
    }
  }
  chain_end();
}

// Body of the TMEM queues: first order in the narrow layout (fewer spills in
// the work-queue kernel, measured faster), the others in the layout of their
// single-plan kernels (wide at N <= 4096).
template <int N, int SPLIT>
using TmBody = Parked<N, SPLIT, true, SPLIT != 1 && N <= 4096>;

// Items at Nx = 2048, 4096, 8192 in the parked form with tables in tensor
// memory (Parked<N, SPLIT, true>, the fastest single-plan form there): one
// channel per item, N/16 threads per block, 512/(N/16) blocks per SM; every block
// allocates its TMEM columns once and frees them on exit.
template <int N, int SPLIT>
__global__ void __launch_bounds__(N / 16, 512 / (N / 16))
    batch_kernel_tm(const MarchArgs* __restrict__ plans, const BatchItem* __restrict__ items,
                    int n_items, int* counter) {
  chain_begin();
  using P = TmBody<N, SPLIT>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  __shared__ uint32_t s_tbase;
  if (threadIdx.x / 32 == 0) tmem_alloc<P::kCols>(&s_tbase);
  tmem_sync();
  const uint32_t tcol = P::tmem_thread(s_tbase, threadIdx.x);
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= n_items) break;
    const BatchItem item = items[it];
    const MarchArgs& A = plans[item.plan];
    if (item.ch0 < A.n_ch) P::march_channel(A, item.ch0, A.z0, A.n_steps, smem, threadIdx.x, tcol);
  }
  tmem_sync();
  if (threadIdx.x / 32 == 0) tmem_dealloc<P::kCols>(s_tbase);
  chain_end();
}

// Items at Nx = 1024 in the tensor-memory parked form with two channels per
// 128-thread block (Parked<1024, SPLIT, true, true, 2>, the fastest
// single-plan form there): each channel group of 64 threads takes its own
// items (its own slot for the counter's answer, its own named barrier), so
// the two groups march at independent phases; four blocks per SM fill the
// SM's 512 TMEM columns.
template <int N, int SPLIT>
__global__ void __launch_bounds__(2 * (N / 16), 512 / (2 * (N / 16)))
    batch_kernel_tm2(const MarchArgs* __restrict__ plans, const BatchItem* __restrict__ items,
                     int n_items, int* counter) {
  chain_begin();
  using P = Parked<N, SPLIT, true, true, 2>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item[2];
  __shared__ uint32_t s_tbase;
  if (threadIdx.x / 32 == 0) tmem_alloc<P::kCols>(&s_tbase);
  tmem_sync();
  const int grp = threadIdx.x / P::T;
  const int t = threadIdx.x % P::T;
  const uint32_t tcol = P::tmem_thread(s_tbase, threadIdx.x);
  unsigned char* gsmem = smem + size_t(grp) * P::group_bytes();
  for (;;) {
    P::gsync();
    if (t == 0) s_item[grp] = atomicAdd(counter, 1);
    P::gsync();
    const int it = s_item[grp];
    if (it >= n_items) break;
    const BatchItem item = items[it];
    const MarchArgs& A = plans[item.plan];
    if (item.ch0 < A.n_ch) P::march_channel(A, item.ch0, A.z0, A.n_steps, gsmem, t, tcol);
  }
  tmem_sync();  // both groups are done (their TMEM loads waited)
  if (threadIdx.x / 32 == 0) tmem_dealloc<P::kCols>(s_tbase);
  chain_end();
}

// Fourth-order items at Nx = 1024 in the parked form with both table sets read
// from L2, eight blocks per SM: as a single plan 25.1 us a step of 1024
// channels, against 26.1 with two channels a block and one set in TMEM.
__global__ void __launch_bounds__(64, 8)
    batch_kernel_pk1024s4(const MarchArgs* __restrict__ plans, const BatchItem* __restrict__ items,
                          int n_items, int* counter) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= n_items) break;
    const BatchItem item = items[it];
    const MarchArgs& A = plans[item.plan];
    Parked<1024, 4>::march_channel(A, item.ch0, A.z0, A.n_steps, smem, threadIdx.x);
  }
  chain_end();
}

// Single channels at Nx <= 512 with 8 Nx/16 threads each (bpm_quad.cuh).
template <int N, int SPLIT>
__global__ void __launch_bounds__(Quad<N, SPLIT>::kThreads, 768 / Quad<N, SPLIT>::kThreads)
    batch_kernel_quad(const MarchArgs* __restrict__ plans, const BatchItem* __restrict__ items,
                      int n_items, int* counter) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= n_items) break;
    const BatchItem item = items[it];
    const MarchArgs& A = plans[item.plan];
    Quad<N, SPLIT>::march_channel(A, item.ch0, A.z0, A.n_steps, smem);
  }
  chain_end();
}

}  // namespace

// A resident item takes an SM for the time of a full one however few channels
// it has (us a step, first order, Strang, fourth order: 256 points 2.9, 4.4,
// 10.3; 512 points 4.7, 5.8, 15.6), a channel of the other form its share of
// one (0.25, 0.275, 0.85; 0.61, 0.66, 2.31).  One kind for all of a round's plans of
// a size and order: their channels and items are counted together.
bool batch_singles(int n, int split_order, int channels, int items, int sms) {
  if (n > 512 || sms < 1) return false;
  const int i = n == 256 ? 0 : 1, o = split_order == 1 ? 0 : split_order == 2 ? 1 : 2;
  static constexpr double each[2][3] = {{0.25, 0.275, 0.85}, {0.61, 0.66, 2.31}};
  static constexpr double full[2][3] = {{2.9, 4.4, 10.3}, {4.7, 5.8, 15.6}};
  return each[i][o] * ((channels + sms - 1) / sms) < full[i][o] * ((items + sms - 1) / sms);
}

int batch_single_queue(int n, int split_order) {
  if (split_order == 1) return n == 256 ? kQueueQuad256 : kQueueQuad512;
  if (split_order == 2) return n == 256 ? kQueueQuad256s2 : kQueueQuad512s2;
  return n == 256 ? kQueueQuad256s4 : kQueueQuad512s4;
}

int batch_group(int n) { return n == 8192 ? 1 : kSmallThreads / (n / 16); }

int batch_item_channels(int n, int split_order) {
  return n >= 1024 ? 1 : batch_group(n);  // parked forms from 1024 points on
}

int batch_queue(int n, int split_order) {
  if (split_order == 1) {
    if (n == 8192) return kQueueTm8192;
    if (n == 4096) return kQueueTm4096;
    if (n == 2048) return kQueueTm2048;
    if (n == 1024) return kQueueTm1024;
    return kQueueSmall;
  }
  if (split_order == 4) {
    if (n == 8192) return kQueueTm8192s4;
    if (n == 4096) return kQueueTm4096s4;
    if (n == 2048) return kQueueTm2048s4;
    if (n == 1024) return kQueuePk1024s4;
    return kQueueSmall4;
  }
  if (n == 8192) return kQueueTm8192s2;
  if (n == 4096) return kQueueTm4096s2;
  if (n == 2048) return kQueueTm2048s2;
  if (n == 1024) return kQueueTm1024s2;
  return kQueueSmall2;
}

int batch_blocks_per_sm(int queue) {
  switch (queue) {
    case kQueueTm4096:
    case kQueueTm4096s2:
    case kQueueTm4096s4: return 2;
    case kQueueTm2048:
    case kQueueTm2048s2:
    case kQueueTm2048s4:
    case kQueueTm1024:
    case kQueueTm1024s2: return 4;
    case kQueuePk1024s4: return 8;
    case kQueueQuad256:
    case kQueueQuad256s2:
    case kQueueQuad256s4: return 6;
    case kQueueQuad512:
    case kQueueQuad512s2:
    case kQueueQuad512s4: return 3;
    default: return 1;
  }
}

namespace {

using BatchKernel = void (*)(const MarchArgs*, const BatchItem*, int, int*);
struct QueueLaunch {
  BatchKernel kernel;
  int threads;
  size_t smem;
};

template <int N, int SPLIT>
QueueLaunch tm_queue() {
  return {batch_kernel_tm<N, SPLIT>, N / 16, TmBody<N, SPLIT>::smem_bytes()};
}
template <int SPLIT>
QueueLaunch tm2_queue() {
  return {batch_kernel_tm2<1024, SPLIT>, 128, Parked<1024, SPLIT, true, true, 2>::smem_bytes()};
}
template <int N, int SPLIT>
QueueLaunch quad_queue() {
  return {batch_kernel_quad<N, SPLIT>, Quad<N, SPLIT>::kThreads, Quad<N, SPLIT>::smem_bytes()};
}

QueueLaunch queue_launch(int queue) {
  switch (queue) {
    case kQueueTm8192: return tm_queue<8192, 1>();
    case kQueueTm8192s2: return tm_queue<8192, 2>();
    case kQueueTm8192s4: return tm_queue<8192, 4>();
    case kQueueTm4096: return tm_queue<4096, 1>();
    case kQueueTm4096s2: return tm_queue<4096, 2>();
    case kQueueTm4096s4: return tm_queue<4096, 4>();
    case kQueueTm2048: return tm_queue<2048, 1>();
    case kQueueTm2048s2: return tm_queue<2048, 2>();
    case kQueueTm2048s4: return tm_queue<2048, 4>();
    case kQueueTm1024: return tm2_queue<1>();
    case kQueueTm1024s2: return tm2_queue<2>();
    case kQueuePk1024s4: return {batch_kernel_pk1024s4, 64, Parked<1024, 4>::smem_bytes()};
    case kQueueSmall: return {batch_kernel<1>, kSmallThreads, kSmallSmem};
    case kQueueSmall2: return {batch_kernel<2>, kSmallThreads, kSmallSmem};
    case kQueueSmall4: return {batch_kernel<4>, kSmallThreads, kSmallSmem};
    case kQueueQuad512: return quad_queue<512, 1>();
    case kQueueQuad512s2: return quad_queue<512, 2>();
    case kQueueQuad512s4: return quad_queue<512, 4>();
    case kQueueQuad256: return quad_queue<256, 1>();
    case kQueueQuad256s2: return quad_queue<256, 2>();
    case kQueueQuad256s4: return quad_queue<256, 4>();
    default: return {nullptr, 0, 0};
  }
}

}  // namespace

cudaError_t launch_batch(const MarchArgs* plans, const BatchItem* items, int n_items, int* counter,
                         int queue, int blocks, bool follow, cudaStream_t s) {
  if (n_items <= 0) return cudaSuccess;
  const QueueLaunch q = queue_launch(queue);
  if (!q.kernel) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(blocks));
  cfg.blockDim = dim3(unsigned(q.threads));
  cfg.dynamicSmemBytes = q.smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = follow ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, q.kernel, plans, items, n_items, counter);
}

cudaError_t batch_set_attributes() {
  for (int queue = 0; queue < kQueueCount; ++queue) {
    const QueueLaunch q = queue_launch(queue);
    const cudaError_t e =
        cudaFuncSetAttribute(q.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(q.smem));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace bpm
