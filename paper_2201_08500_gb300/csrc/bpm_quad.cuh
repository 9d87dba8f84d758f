// March of one channel by 8 N/16 threads, four values each (N = 256, 512,
// 1024): the form of launches with few channels for the chip.
//
// With N/16 threads a channel, a 512-point channel is one warp, and a step
// lasts as long as that warp needs to issue its ~2400 instructions: 3.1 us
// however idle the chip is.  Here the envelopes go to the two halves of each
// warp and every radix-16 butterfly, as 4 x 4, to four warps: thread (t, q)
// holds the values k = q, q+4, q+8, q+12 of group t of either butterfly layout
// (bpm_fft.cuh).  One transform then exchanges through shared memory three
// times (inside each radix-16 butterfly and between the two), a last stage of
// radix 2 or 4 runs by lane shuffles, and the coupling takes the other
// envelope by a shuffle.  Exchanges alternate between two buffers, so each
// needs one block barrier.  Tables, twiddles and coefficients stay in
// registers.  Every element's operations and their order are those of
// bpm_resident.cuh, so the fields are bitwise the same, and so are the sums of
// the reflectivity.
//
// A step of one channel, first order: 256 points 1.77 -> 0.61 us, 512 points
// 3.1 ... 3.7 -> 0.97, 1024 points 3.2 ... 3.9 -> 1.62 (latency bound: six
// barriers and the chains between them; an SM issues in 22 to 38 % of its
// cycles); 201 channels of 512 points 3.85 -> 1.32; Strang 512 points 4.8 -> 1.15;
// fourth order 11.7 -> 3.7.
#pragma once

#include <cuda_runtime.h>

#include "bpm_half.cuh"
#include "bpm_norm.cuh"
#include "bpm_resident.cuh"
#include "bpm_share.cuh"

namespace bpm {

template <int N, int SPLIT>
struct Quad {
  static_assert(N == 256 || N == 512 || N == 1024, "two radix-16 stages and a last one up to 4");
  using Gm = Geom<N>;
  static constexpr int T = Gm::T;
  static constexpr int kThreads = 8 * T;
  static constexpr int RL = N / 256;                   // radix of the last stage (1: none)
  static constexpr int kSets = SPLIT == 4 ? 2 : 1;     // table and coefficient sets
  static constexpr int kSlots = Pad<N>::kSlots;
  static constexpr int kBuf = 2 * kSlots;              // one exchange buffer: both envelopes

  __host__ __device__ static constexpr size_t smem_bytes() {
    return 2 * size_t(kBuf) * sizeof(float2) + 8 * sizeof(double);
  }

  struct Ctx {
    float2* x0;   // exchange buffers of this thread's envelope
    float2* x1;
    int t, q, env;
    float2 tw0[4], tw1[RL > 1 ? 4 : 1];  // stage twiddles of the thread's values
    float4 tab[kSets][4];                // propagator of the thread's spectrum values
  };

  // Stage-1 position of value k of group t (t = T layout of the second radix-16 stage).
  static BPM_DEV int pos1(int t, int k) { return (t / RL) * T + (t % RL) + RL * k; }

  // Exchange inside a radix-16 butterfly: value i of thread q becomes value q of thread i.
  static BPM_DEV void xchg4(float2 (&v)[4], float2* x, int t, int q) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[(4 * q + i) * T + t] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = x[(4 * i + q) * T + t];
  }
  // Exchange between the stages (padded positions: no bank conflicts either way).
  static BPM_DEV int pad(int p) { return p + (p >> 4); }
  template <bool INV>
  static BPM_DEV void xchg16(float2 (&v)[4], float2* x, int t, int q) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = q + 4 * i;
      x[pad(INV ? pos1(t, k) : t + T * k)] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = q + 4 * i;
      v[i] = x[pad(INV ? t + T * k : pos1(t, k))];
    }
  }

  // 16-point DFT of a group: 4-point DFTs over the thread's own values, the
  // exchange, then 4-point DFTs with the internal twiddles of row q (dft16_fwd
  // and dft16_inv split over the four threads; q is the same in a warp).
  template <bool INV>
  static BPM_DEV void dft16(float2 (&v)[4], float2* x, int t, int q) {
    dft4<INV>(v[0], v[1], v[2], v[3]);
    xchg4(v, x, t, q);
    if (q == 0) {
      dft4<INV>(v[0], v[1], v[2], v[3]);
    } else if (q == 1) {
      v[1] = w16<1, INV>(v[1]);
      v[3] = w16<3, INV>(v[3]);
      dft4_c<2, INV, false>(v[0], v[1], v[2], v[3]);
    } else if (q == 2) {
      v[2] = w16<4, INV>(v[2]);
      dft4_bd<INV, false>(v[0], v[1], v[2], v[3]);
    } else {
      v[1] = w16<3, INV>(v[1]);
      v[3] = w16<9, INV>(v[3]);
      dft4_c<6, INV, false>(v[0], v[1], v[2], v[3]);
    }
  }

  static BPM_DEV float2 shfl(float2 v, int mask) {
    return make_float2(__shfl_xor_sync(0xFFFFFFFFu, v.x, mask),
                       __shfl_xor_sync(0xFFFFFFFFu, v.y, mask));
  }
  // own + other, or (sign -1: the upper lane of a pair) other - own: one rounding
  // either way, and one instruction instead of two and a selection (512 points 1.05
  // -> 0.97 us a step, 1024 points 1.79 -> 1.68).
  static BPM_DEV float2 sumdiff(float2 own, float2 other, float sign) {
    return c_fmas(own, sign, other);
  }

  // Last stage over the RL lanes that share a block of positions (t % RL).
  // Radix 4 leaves outputs 1 and 2 in each other's lane (spectrum_lane), which
  // the tables and the inverse take as it is.
  template <bool INV>
  static BPM_DEV void last(float2 (&v)[4], int t) {
    if constexpr (RL == 2) {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = sumdiff(v[i], shfl(v[i], 1), t & 1 ? -1.f : 1.f);
    } else if constexpr (RL == 4) {
      // forward: sums and differences of lanes 2 apart, then of neighbours;
      // inverse: the other way round.  The pair of differences combines with
      // the quarter turn.
      constexpr int m0 = INV ? 1 : 2, m1 = INV ? 2 : 1;
      const bool turned = t & m0, upper = t & m1;
      const float sg = (upper != INV) ? -1.f : 1.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 a = sumdiff(v[i], shfl(v[i], m0), turned ? -1.f : 1.f);
        const float2 o = shfl(a, m1);
        const float2 d0 = upper ? o : a, d1 = upper ? a : o;
        const float2 plain = sumdiff(a, o, upper ? -1.f : 1.f);
        const float2 quarter = make_float2(fmaf(d1.y, sg, d0.x), fmaf(-d1.x, sg, d0.y));
        v[i] = turned ? quarter : plain;
      }
    }
  }
  static BPM_DEV int spectrum_lane(int t) {
    return RL == 4 ? (t & ~3) | ((t & 1) << 1) | ((t >> 1) & 1) : t;
  }

  // The product by the twiddle of k = 0, which is one, too: at 1024 points cheaper than
  // the branch around it (1.68 -> 1.62 us a step; 512 points 0.97 -> 1.00).
  static constexpr bool kMulAll = N == 1024;

  // Forward FFT, propagator (table set s), inverse FFT of the thread's envelope.
  static BPM_DEV void propagate(float2 (&v)[4], const Ctx& c, int s) {
    dft16<false>(v, c.x0, c.t, c.q);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (kMulAll || i > 0 || c.q > 0) v[i] = c_mul(v[i], c.tw0[i]);
    xchg16<false>(v, c.x1, c.t, c.q);
    dft16<false>(v, c.x0, c.t, c.q);
    if constexpr (RL > 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (kMulAll || i > 0 || c.q > 0) v[i] = c_mul(v[i], c.tw1[i]);
    }
    last<false>(v, c.t);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = c_mul2(v[i], kSets == 2 && s ? c.tab[kSets - 1][i] : c.tab[0][i]);
    last<true>(v, c.t);
    if constexpr (RL > 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (kMulAll || i > 0 || c.q > 0) v[i] = c_mulc(v[i], c.tw1[i]);
    }
    dft16<true>(v, c.x1, c.t, c.q);
    xchg16<true>(v, c.x0, c.t, c.q);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (kMulAll || i > 0 || c.q > 0) v[i] = c_mulc(v[i], c.tw0[i]);
    dft16<true>(v, c.x1, c.t, c.q);
  }

  static BPM_DEV void couple(float2 (&v)[4], const float2 (&cc)[4], const HalfCoef& h, int env) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // both halves of the warp hold the same cells: the vote keeps the shuffles whole
      const bool in = cc[i].x != 0.f || cc[i].y != 0.f;
      if (!__any_sync(0xFFFFFFFFu, in)) continue;
      const float2 o = shfl(v[i], 16);
      if (!in) continue;
      v[i] = half_cell(v[i], o, cc[i], h, env);
    }
  }

  // March channel ch of plan A by n steps from row z0 (this block: kThreads threads).
  static BPM_DEV void march_channel(const MarchArgs& A, int ch, int z0, int n, unsigned char* smem) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    Ctx c;
    c.env = lane >> 4;
    c.q = w / (T / 16);
    c.t = (w % (T / 16)) * 16 + (lane & 15);
    const int t = c.t, q = c.q, env = c.env;
    float2* buf = reinterpret_cast<float2*>(smem);
    c.x0 = buf + env * kSlots;
    c.x1 = c.x0 + kBuf;
    const float4* gtab = A.tables + (size_t(ch) * kSets * 2 + env) * N;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = q + 4 * i;
      c.tw0[i] = __ldg(A.twiddle + t * k);
      if constexpr (RL > 1) c.tw1[i] = __ldg(A.twiddle + 16 * (t % RL) * k);
      const int p = pos1(spectrum_lane(t), k);
#pragma unroll
      for (int s = 0; s < kSets; ++s)
        c.tab[s][i] = __ldg(gtab + size_t(s) * 2 * N + (p % 16) * T + p / 16);
    }
    const HalfCoef h0 = half_coef(A.coef[size_t(ch) * kSets], env);
    const HalfCoef h1 = half_coef(A.coef[size_t(ch) * kSets + kSets - 1], env);
    float2* field = (env ? A.eh : A.e0) + size_t(ch) * N;
    float2 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = field[t + T * (q + 4 * i)];
    const float2* crow = A.cfield + size_t(z0) * N + t + T * q;
    for (int step = 0; step < n; ++step, crow += N) {
      float2 cc[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) cc[i] = __ldg(crow + 4 * T * i);
      if constexpr (SPLIT == 4) {
#pragma unroll 1
        for (int j = 0; j < 3; ++j) {
          couple(v, cc, j == 0 ? h0 : h1, env);
          propagate(v, c, j == 1);
        }
      } else {
        if constexpr (SPLIT == 2) couple(v, cc, h0, env);
        propagate(v, c, 0);
      }
      couple(v, cc, h0, env);
    }
    // fields out, and into shared memory for the sums of |E|^2 in the resident
    // form's order: thread t over its 16 k, then across the threads
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int x = t + T * (q + 4 * i);
      field[x] = v[i];
      c.x0[x] = v[i];
    }
    __syncthreads();
    double* red = reinterpret_cast<double*>(smem + 2 * size_t(kBuf) * sizeof(float2));
    if (threadIdx.x < 2 * T) {
      const int e = threadIdx.x / T, tt = threadIdx.x % T;
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float2 f = buf[e * kSlots + tt + T * k];
        s = add_norm(s, f);
      }
      constexpr int W = T < 32 ? T : 32;
#pragma unroll
      for (int off = W / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      if (tt % W == 0) red[e * (T / W) + tt / W] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      constexpr int nw = T < 32 ? 1 : T / 32;
      double s[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        s[e] = red[e * nw];
        for (int i = 1; i < nw; ++i) s[e] += red[e * nw + i];
      }
      const double inc = A.inc_norm[ch];
      A.trans[ch] = s[0] / inc;
      A.refl[ch] = s[1] / inc;
    }
    __syncthreads();  // shared memory is free for the next channel
  }

  static BPM_DEV void run(const MarchArgs& A, unsigned char* smem) {
    __shared__ Share share;
    if (threadIdx.x == 0) share_begin(A, blockIdx.x, gridDim.x, &share);
    for (;;) {
      if (threadIdx.x == 0) share_next(A, blockIdx.x, gridDim.x, &share);
      __syncthreads();
      if (share.ch < 0) break;
      march_channel(A, share.ch, share.z0, share.n, smem);
    }
  }
};

}  // namespace bpm
