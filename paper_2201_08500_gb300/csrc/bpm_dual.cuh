// March of one channel by 2 N/16 threads (N = 2048): the form of launches of few
// channels for the chip.
//
// With one channel on an SM nothing covers its exchanges and barriers, and the
// parked march transforms the envelopes one after the other.  Here each half of the
// block has an envelope: both transform at the same time, with the parked march's
// single-envelope transform (a named barrier and two exchange buffers each, the
// envelope's tables in tensor memory), and meet at the coupling, which passes the
// values inside the crystal's extent through shared memory.  Every element's
// operations and their order are those of the parked march, and so are the sums.
// The deformation row's part is prefetched into L1 at the start of a step.
// A step of 152 channels, the best other form -> this one, us: 4.10 -> 2.64, Strang
// 4.93 -> 3.28, fourth order 14.6 -> 8.4 (the other forms' eight warps an SM issue in
// turns; 220 registers a thread let a step's loads go out early).  4096 points have
// half the registers a thread and gain nothing (5.05 against 5.06), 1024 and less the
// form of bpm_quad.cuh.
#pragma once

#include <cuda_runtime.h>

#include "bpm_half.cuh"
#include "bpm_norm.cuh"
#include "bpm_parked.cuh"
#include "bpm_share.cuh"

namespace bpm {

template <int N, int SPLIT>
struct Dual {
  using P = Parked<N, SPLIT, true, true, 2>;  // a "channel group" of P is an envelope
  static constexpr int T = P::T;
  static constexpr int kThreads = 2 * T;
  static constexpr int kSlots = Pad<N>::kSlots;
  static constexpr int kTabs = P::kTabs;

  __host__ __device__ static constexpr size_t smem_bytes() {
    return 4 * size_t(kSlots) * sizeof(float2) + 64 * sizeof(double);
  }

  // own: this envelope's free exchange buffer, oth: the other's.  Before: every
  // read of own by the other envelope's threads has been followed by a barrier.
  static BPM_DEV void couple(float2 (&v)[16], float2* own, const float2* oth, const float2* crow,
                             const HalfCoef& h, unsigned m, int env, int t) {
    if (m == 0u) return;  // no crystal: the same for the block
    float4* q = reinterpret_cast<float4*>(own);
    const float4* p = reinterpret_cast<const float4*>(oth);
    float2 c[16];
#pragma unroll
    for (int k = 0; k < 16; ++k)
      c[k] = (m >> k) & 1u ? __ldg(crow + t + T * k) : make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if ((m >> (2 * i)) & 3u)
        q[P::park_slot(t, i)] = make_float4(v[2 * i].x, v[2 * i].y, v[2 * i + 1].x, v[2 * i + 1].y);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (!((m >> (2 * i)) & 3u)) continue;
      const float4 w = p[P::park_slot(t, i)];
      if (c[2 * i].x != 0.f || c[2 * i].y != 0.f)
        v[2 * i] = half_cell(v[2 * i], make_float2(w.x, w.y), c[2 * i], h, env);
      if (c[2 * i + 1].x != 0.f || c[2 * i + 1].y != 0.f)
        v[2 * i + 1] = half_cell(v[2 * i + 1], make_float2(w.z, w.w), c[2 * i + 1], h, env);
    }
  }

  // March channel ch of plan A by n steps from row z0 (this block).
  static BPM_DEV void march_channel(const MarchArgs& A, int ch, int z0, int n, unsigned char* smem,
                                    uint32_t tcol) {
    const int env = threadIdx.x / T, t = threadIdx.x % T;
    float2* buf = reinterpret_cast<float2*>(smem);
    float2 *x = buf + 2 * env * kSlots, *own = x + kSlots;
    const float2* oth = buf + (2 * (env ^ 1) + 1) * kSlots;
    double* red = reinterpret_cast<double*>(buf + 4 * kSlots) + 32 * env;
    const float4* gtab = A.tables + size_t(ch) * kTabs * 2 * N + env * N;
    const float4* tw = reinterpret_cast<const float4*>(A.twiddle_p);
    float2* field = (env ? A.eh : A.e0) + size_t(ch) * N;
    const int lo = __ldg(A.ext), hi = -__ldg(A.ext + 1);  // crystal cells [lo, hi)
    const unsigned m = lo == kExtNone ? 0u : (2u << ((hi - 1) / T)) - (1u << (lo / T));
    const HalfCoef h0 = half_coef(A.coef[size_t(ch) * kTabs], env);
    const HalfCoef h1 = half_coef(A.coef[size_t(ch) * kTabs + kTabs - 1], env);
    const uint32_t col = tcol + 64u * env;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 tv[2][4];
#pragma unroll
      for (int i = 0; i < 8; ++i) tv[i / 4][i % 4] = __ldg(gtab + (8 * h + i) * T + t);
      tmem_st16(col + uint32_t(32 * h), tv[0]);
      tmem_st16(col + uint32_t(32 * h + 16), tv[1]);
    }
    tmem_wait_st();
    float2 v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = field[t + T * k];
    const float2* crow = A.cfield + size_t(z0) * N;
    for (int step = 0; step < n; ++step, crow += N) {
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if ((m >> k) & 1u) asm volatile("prefetch.global.L1 [%0];" ::"l"(crow + t + T * k));
      if constexpr (SPLIT != 1) {
        __syncthreads();  // the last coupling's reads are done
        couple(v, own, oth, crow, h0, m, env, t);
      }
#pragma unroll 1
      for (int j = 0; j < (SPLIT == 4 ? 3 : 1); ++j) {
        __syncthreads();  // the coupling's reads, and loads of x, are done
        P::propagate(v, x, own, SPLIT == 4 && j == 1 ? gtab + 2 * N : nullptr, col, tw, t);
        couple(v, own, oth, crow, SPLIT != 4 || j == 2 ? h0 : h1, m, env, t);
      }
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      field[t + T * k] = v[k];
      s = add_norm(s, v[k]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
    if ((t & 31) == 0) red[t / 32] = s;
    __syncthreads();
    if (t == 0) {
      s = 0.0;
      for (int i = 0; i < T / 32; ++i) s += red[i];
      (env ? A.refl : A.trans)[ch] = s / A.inc_norm[ch];
    }
    __syncthreads();
  }

  static BPM_DEV void run(const MarchArgs& A, unsigned char* smem) {
    __shared__ uint32_t s_tbase;
    if (threadIdx.x / 32 == 0) tmem_alloc<P::kCols>(&s_tbase);
    tmem_sync();
    const uint32_t tcol = P::tmem_thread(s_tbase, threadIdx.x);
    __shared__ Share share;
    if (threadIdx.x == 0) share_begin(A, blockIdx.x, gridDim.x, &share);
    for (;;) {
      if (threadIdx.x == 0) share_next(A, blockIdx.x, gridDim.x, &share);
      __syncthreads();
      if (share.ch < 0) break;
      march_channel(A, share.ch, share.z0, share.n, smem, tcol);
    }
    tmem_sync();
    if (threadIdx.x / 32 == 0) tmem_dealloc<P::kCols>(s_tbase);
  }
};

}  // namespace bpm
