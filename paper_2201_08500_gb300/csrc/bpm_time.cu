// Frequency-to-time assembly (after Eq. ref:tdp):
//   psi_h(t_j) = d_omega sum_i A-(omega_i) exp(-2 pi i (i - n/2) j / n),
// in FP64 for every x, over the n channels of a pulse (n/2 rounded down).
//
// The chip does two FP64 operations a clock and SM (1/64 of FP32), so FP64
// instructions are what bounds this step; shared memory, index arithmetic and
// HBM have room to spare.  Hence transforms instead of sums, at every n:
//  * n = 2^a 3^b 5^c 7^d (up to 4096): Stockham passes of radix 8, 4, 2, 3, 5
//    and 7 through shared memory, about 3.3 FP64 instructions a point and
//    octave (radix 2: 4, a direct sum: 4 n);
//  * any other n up to 2048: Bluestein's chirp transform of the length M >= 2n - 1
//    with the fewest operations, 2^a 3^b 5^c 7^d too, with the same passes (611
//    channels: 1280, not 2048);
//  * beyond that the direct sum.
// Measured against a radix-2 transform (n a power of two up to 1024) and the
// direct sum (the rest): 128 channels x 512 x 512: 2.51 -> 1.55 ms (about 24
// FP64 instructions a point, 85 % of the FP64 rate); 1024 x 4096: 557 -> 310
// us; 24 x 131072: 6.46 ms -> 124 us; 611 = 13 x 47 channels x 1024 (chirp
// form): 32.0 ms -> 236 us (334 at length 2048).
// Twiddles, chirps and the chirp's spectrum are the plan's (time_tables_kernel,
// written once for its n): made in each block they cost as much as a column.
#include <cuda_runtime.h>
#include <math.h>

#include "bpm_internal.h"
#include "bpm_norm.cuh"

namespace bpm {

namespace {

constexpr int kTimeThreads = 256;
constexpr int kTimeMaxLen = 4096;             // two buffers of one column: 192 KB with the twiddles
constexpr size_t kTimeSmem = 200 * 1024;

// Radices of a transform of len points, largest power-of-two radices first;
// false if len has a prime factor above 7.
bool radices(int len, TimeShape* s) {
  s->n_pass = 0;
  auto take = [&](int r) {
    while (len % r == 0) {
      s->radix[s->n_pass++] = (unsigned char)r;
      len /= r;
    }
  };
  int twos = 0;
  for (; len % 2 == 0; len /= 2) ++twos;
  // 4 x 4 instead of 8 x 2: a pass of radix 2 saves no twiddle
  for (; twos >= 3 && twos != 4; twos -= 3) s->radix[s->n_pass++] = 8;
  for (; twos >= 2; twos -= 2) s->radix[s->n_pass++] = 4;
  if (twos) s->radix[s->n_pass++] = 2;
  take(7);
  take(5);
  take(3);
  return len == 1;
}

}  // namespace

bool time_shape(int n, TimeShape* s) {
  *s = TimeShape{};
  if (n < 1) return false;
  s->n = s->len = n;
  if (n <= kTimeMaxLen && radices(n, s)) return true;
  // the chirp form: of the odd parts, each with the power of two that it needs, the
  // one with the fewest FP64 instructions
  if (n > kTimeMaxLen / 2) return false;
  s->chirp = 1;
  double best = 0.0;
  for (int odd : {1, 3, 5, 7, 9, 15, 21, 25, 27, 35, 45, 49}) {
    TimeShape t = *s;
    for (t.len = odd; t.len < 2 * n - 1;) t.len *= 2;
    if (t.len > kTimeMaxLen || !radices(t.len, &t)) continue;
    double cost = 0.0;
    for (int p = 0; p < t.n_pass; ++p) {
      const int r = t.radix[p];
      cost += r == 8 ? 10.0 : r == 4 ? 7.0 : r == 2 ? 4.0 : r == 7 ? 12.9 : r == 5 ? 10.4 : 8.0;
    }
    cost *= t.len;
    if (best == 0.0 || cost < best) {
      best = cost;
      *s = t;
    }
  }
  return best > 0.0;
}

size_t time_table_elems(int n) {
  TimeShape s;
  if (!time_shape(n, &s)) return 0;
  return size_t(s.len) + (s.chirp ? 2 * size_t(n) + s.len : 0);
}

namespace {

__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// a + s b, a + s (-i b)
__device__ __forceinline__ double2 zfma(double s, double2 b, double2 a) {
  return make_double2(fma(s, b.x, a.x), fma(s, b.y, a.y));
}
__device__ __forceinline__ double2 zfmaj(double s, double2 b, double2 a) {
  return make_double2(fma(s, b.y, a.x), fma(-s, b.x, a.y));
}

__device__ __forceinline__ void zdft4(double2& a, double2& b, double2& c, double2& d) {
  const double2 s0 = zadd(a, c), d0 = zsub(a, c), s1 = zadd(b, d), d1 = zsub(b, d);
  a = zadd(s0, s1);
  c = zsub(s0, s1);
  b = make_double2(d0.x + d1.y, d0.y - d1.x);
  d = make_double2(d0.x - d1.y, d0.y + d1.x);
}

// Forward R-point DFT in place, natural order.
template <int R>
__device__ __forceinline__ void zdft(double2 (&v)[R]) {
  if constexpr (R == 2) {
    const double2 s = zadd(v[0], v[1]);
    v[1] = zsub(v[0], v[1]);
    v[0] = s;
  } else if constexpr (R == 4) {
    zdft4(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    constexpr double c8 = 0.7071067811865475244;
    zdft4(v[0], v[2], v[4], v[6]);
    zdft4(v[1], v[3], v[5], v[7]);
    // W8 and W8^3 as c8 times a sum of the parts, the product inside the addition
    const double2 p = make_double2(v[3].x + v[3].y, v[3].y - v[3].x);
    const double2 q = make_double2(v[7].y - v[7].x, -v[7].x - v[7].y);
    const double2 o0 = zadd(v[0], v[1]), o4 = zsub(v[0], v[1]);
    const double2 o1 = zfma(c8, p, v[2]), o5 = zfma(-c8, p, v[2]);
    const double2 o2 = make_double2(v[4].x + v[5].y, v[4].y - v[5].x);
    const double2 o6 = make_double2(v[4].x - v[5].y, v[4].y + v[5].x);
    const double2 o3 = zfma(c8, q, v[6]), o7 = zfma(-c8, q, v[6]);
    v[0] = o0; v[1] = o1; v[2] = o2; v[3] = o3;
    v[4] = o4; v[5] = o5; v[6] = o6; v[7] = o7;
  } else {
    // odd prime: sums and differences of the pairs (k, R - k)
    constexpr int K = (R - 1) / 2;
    constexpr double cs[3] = {R == 3 ? -0.5 : R == 5 ? 0.3090169943749474241 : 0.6234898018587335305,
                              R == 5 ? -0.8090169943749474241 : -0.2225209339563144043,
                              -0.9009688679024191262};
    constexpr double sn[3] = {R == 3   ? 0.8660254037844386468
                              : R == 5 ? 0.9510565162951535721
                                       : 0.7818314824680298087,
                              R == 5 ? 0.5877852522924731292 : 0.9749279121818236070,
                              0.4338837391175581205};
    double2 s[K], d[K], o[R];
    o[0] = v[0];
#pragma unroll
    for (int k = 1; k <= K; ++k) {
      s[k - 1] = zadd(v[k], v[R - k]);
      d[k - 1] = zsub(v[k], v[R - k]);
      o[0] = zadd(o[0], s[k - 1]);
    }
#pragma unroll
    for (int m = 1; m <= K; ++m) {
      double2 a = v[0], b = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 1; k <= K; ++k) {
        const int e = (k * m) % R;  // cos and sin of 2 pi e / R from the first half
        a = zfma(cs[(e <= K ? e : R - e) - 1], s[k - 1], a);
        b = zfma(e <= K ? sn[e - 1] : -sn[R - e - 1], d[k - 1], b);
      }
      o[m] = make_double2(a.x + b.y, a.y - b.x);
      o[R - m] = make_double2(a.x - b.y, a.y + b.x);
    }
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = o[k];
  }
}

// One Stockham pass of radix R over 2^lc columns side by side (element i of
// column c at [i 2^lc + c]); ns = product of the earlier radices.
template <int R>
__device__ void time_pass(const double2* __restrict__ in, double2* __restrict__ out,
                          const double2* __restrict__ tw, int len, int ns, int lc) {
  const int m = len / R, step = m / ns, cols = 1 << lc;
  for (int idx = threadIdx.x; idx < (m << lc); idx += blockDim.x) {
    const int c = idx & (cols - 1), j = idx >> lc;
    const int k = ns == 1 ? 0 : j % ns;
    double2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = in[((j + r * m) << lc) + c];
    if (ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = zmul(v[r], tw[r * k * step]);
    }
    zdft<R>(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) out[((base + r * ns) << lc) + c] = v[r];
  }
}

// All passes; returns the buffer that holds the spectrum (x or y).
__device__ double2* time_passes(const TimeShape& s, double2* x, double2* y, const double2* tw,
                                int lc) {
  int ns = 1;
  for (int p = 0; p < s.n_pass; ++p) {
    const int r = s.radix[p];
    __syncthreads();
    switch (r) {
      case 8: time_pass<8>(x, y, tw, s.len, ns, lc); break;
      case 4: time_pass<4>(x, y, tw, s.len, ns, lc); break;
      case 2: time_pass<2>(x, y, tw, s.len, ns, lc); break;
      case 7: time_pass<7>(x, y, tw, s.len, ns, lc); break;
      case 5: time_pass<5>(x, y, tw, s.len, ns, lc); break;
      default: time_pass<3>(x, y, tw, s.len, ns, lc); break;
    }
    ns *= r;
    double2* t = x;
    x = y;
    y = t;
  }
  __syncthreads();
  return x;
}

// exp(i pi a / n) of an integer a reduced mod 2n
__device__ __forceinline__ double2 half_turns(long long a, int n) {
  double s, c;
  sincospi(double(a % (2LL * n)) / double(n), &s, &c);
  return make_double2(c, s);
}

// Tables of a transform, one block: twiddles exp(-2 pi i k / len) [len] and,
// for the chirp form, exp(-i pi i^2 / n) [n], the same times the output's
// exp(2 pi i (n/2) j / n) [n], and the spectrum of exp(i pi i^2 / n) / len [len].
__global__ void time_tables_kernel(TimeShape s, double2* tt) {
  extern __shared__ __align__(16) double2 sm[];
  double2 *x = sm, *y = sm + s.len, *tw = sm + 2 * s.len;
  for (int k = threadIdx.x; k < s.len; k += blockDim.x) {
    const double2 w = half_turns(-2LL * k, s.len);
    tw[k] = w;
    tt[k] = w;
  }
  if (!s.chirp) return;
  double2 *cin = tt + s.len, *cout = cin + s.n, *filt = cout + s.n;
  for (int i = threadIdx.x; i < s.len; i += blockDim.x) x[i] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int i = threadIdx.x; i < s.n; i += blockDim.x) {
    const long long q = (long long)i * i;
    const double2 w = half_turns(-q, s.n);
    cin[i] = w;
    cout[i] = half_turns(2LL * (s.n / 2) * i - q, s.n);
    const double2 b = make_double2(w.x, -w.y);
    x[i] = b;
    if (i) x[s.len - i] = b;
  }
  const double2* f = time_passes(s, x, y, tw, 0);
  const double inv = 1.0 / double(s.len);
  for (int i = threadIdx.x; i < s.len; i += blockDim.x)
    filt[i] = make_double2(f[i].x * inv, f[i].y * inv);
}

// 2^lc columns x0 .. of the [n][plane] spectrum per block.  The plan holds
// channels first .. first + n_local - 1 of the n (a shard, or all of them); the
// others enter as zeros, so the output is this shard's part of the sum.
// 256 threads and about 2048 points a block (two blocks or more an SM): one
// radix-8 butterfly a thread and pass, and one block's loads under another's
// FP64 work.
template <bool CHIRP>
__global__ void __launch_bounds__(kTimeThreads)
    omega_to_t_kernel(const __grid_constant__ TimeShape s, int lc, int first, int n_local,
                      long long plane, double domega, const double2* __restrict__ tt,
                      const float2* __restrict__ eh, double2* __restrict__ out) {
  extern __shared__ __align__(16) double2 sm[];
  double2 *x = sm, *y = x + (s.len << lc), *tw = y + (s.len << lc);
  const double2 *cin = tt + s.len, *cout = cin + s.n, *filt = cout + s.n;
  const int nc = 1 << lc;
  const long long x0 = (long long)blockIdx.x << lc;
  const int cols = int(min((long long)nc, plane - x0));
  for (int k = threadIdx.x; k < s.len; k += blockDim.x) tw[k] = tt[k];
  for (int idx = threadIdx.x; idx < (s.len << lc); idx += blockDim.x) {
    const int i = idx >> lc, c = idx & (nc - 1), li = i - first;
    double2 v = make_double2(0.0, 0.0);
    if (c < cols && li >= 0 && li < n_local) {
      const float2 f = eh[(long long)li * plane + x0 + c];
      v = make_double2(widen_any(f.x), widen_any(f.y));
      if constexpr (CHIRP) v = zmul(v, cin[i]);
    }
    x[idx] = v;
  }
  double2* r = time_passes(s, x, y, tw, lc);
  if constexpr (CHIRP) {
    // convolution with the chirp: product of the spectra, and the inverse as the
    // conjugate of a forward transform
    for (int idx = threadIdx.x; idx < (s.len << lc); idx += blockDim.x) {
      const double2 v = zmul(r[idx], filt[idx >> lc]);
      r[idx] = make_double2(v.x, -v.y);
    }
    r = time_passes(s, r, r == x ? y : x, tw, lc);
  }
  const int ic = s.n / 2;
  for (int idx = threadIdx.x; idx < (s.n << lc); idx += blockDim.x) {
    const int j = idx >> lc, c = idx & (nc - 1);
    if (c >= cols) continue;
    double2 v = r[idx];
    if constexpr (CHIRP) {
      v = zmul(make_double2(v.x, -v.y), cout[j]);
    } else if (s.n % 2 == 0) {  // exp(2 pi i (n/2) j / n) = (-1)^j
      if (j & 1) v = make_double2(-v.x, -v.y);
    } else {
      const double2 w = tw[int(((long long)ic * j) % s.n)];
      v = zmul(v, make_double2(w.x, -w.y));
    }
    out[(long long)j * plane + x0 + c] = make_double2(domega * v.x, domega * v.y);
  }
}

// Direct FP64 sum for the n that no transform above takes, over this plan's
// channels first .. first + n_local - 1 of the n.
__global__ void omega_to_t_direct_kernel(int n, int first, int n_local, long long plane,
                                         double domega, const float2* __restrict__ eh,
                                         double2* out) {
  const long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (x >= plane) return;
  const int ic = n / 2;
  double re = 0.0, im = 0.0;
  for (int li = 0; li < n_local; ++li) {
    const int i = first + li;
    const long long e = (((long long)(i - ic) * j) % n + n) % n;
    double s, co;
    sincospi(-2.0 * double(e) / double(n), &s, &co);
    const float2 f = eh[(long long)li * plane + x];
    re += double(f.x) * co - double(f.y) * s;
    im += double(f.x) * s + double(f.y) * co;
  }
  out[(long long)j * plane + x] = make_double2(domega * re, domega * im);
}

}  // namespace

cudaError_t time_set_attributes() {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t r[] = {cudaFuncSetAttribute(omega_to_t_kernel<false>, attr, int(kTimeSmem)),
                     cudaFuncSetAttribute(omega_to_t_kernel<true>, attr, int(kTimeSmem)),
                     cudaFuncSetAttribute(time_tables_kernel, attr, int(kTimeSmem))};
  for (cudaError_t e : r)
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t launch_time_tables(int n, double2* tt, cudaStream_t st) {
  TimeShape s;
  if (!time_shape(n, &s)) return cudaSuccess;
  time_tables_kernel<<<1, 512, 3 * size_t(s.len) * sizeof(double2), st>>>(s, tt);
  return cudaGetLastError();
}

cudaError_t launch_omega_to_t(int n_total, int first, int n_local, long long plane, double domega,
                              const double2* tt, const float2* eh, double2* out, cudaStream_t st) {
  if (first < 0 || n_local < 0 || first + n_local > n_total) return cudaErrorInvalidValue;
  TimeShape s;
  if (!time_shape(n_total, &s) || !tt) {
    dim3 grid(unsigned((plane + 127) / 128), unsigned(n_total));
    omega_to_t_direct_kernel<<<grid, 128, 0, st>>>(n_total, first, n_local, plane, domega, eh, out);
    return cudaGetLastError();
  }
  int lc = 0;
  while (lc < 6 && (s.len << (lc + 1)) <= 2560) ++lc;
  // a small plane: fewer columns a block, so that more SMs have one (four columns
  // are still whole 32-byte sectors); 64 channels x 256: 16.7 -> 7.6 us
  while (lc > 2 && (plane >> lc) < 152) --lc;
  const size_t smem = (2 * (size_t(s.len) << lc) + s.len) * sizeof(double2);
  const long long blocks = (plane + (1 << lc) - 1) >> lc;
  if (s.chirp)
    omega_to_t_kernel<true><<<unsigned(blocks), kTimeThreads, smem, st>>>(
        s, lc, first, n_local, plane, domega, tt, eh, out);
  else
    omega_to_t_kernel<false><<<unsigned(blocks), kTimeThreads, smem, st>>>(
        s, lc, first, n_local, plane, domega, tt, eh, out);
  return cudaGetLastError();
}

}  // namespace bpm
