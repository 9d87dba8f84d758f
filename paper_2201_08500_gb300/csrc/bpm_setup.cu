// Per-plan setup kernels of the BPM (FP64 arithmetic, run once per crystal /
// pulse).  The frequency-to-time assembly is in bpm_time.cu.
//
//  deformation_kernel : c(x, z) = Pi(x, z) exp(+i h u(x, z))         (Eq. Authier);
//                       Pi from the crystal's boundaries or a caller's mask
//  tables_kernel      : tilted propagators p+- and coupling coefficients
//                       (Eqs. fov4, fov11, fov12, Zassenhaus-like factor)
//  incident_kernel    : A+ = S g(x, y) exp(i (k sin theta_i - h/2) x), A- = 0
//                       (beam of Section 3.1, spectral amplitude of Eq. ref:tdp)
#include <cuda_runtime.h>
#include <math.h>

#include "bpm_internal.h"
#include "bpm_norm.cuh"

namespace bpm {

namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr double kC = 299792458.0;

struct dc {
  double re, im;
};
__device__ __forceinline__ dc dmk(double r, double i) { return dc{r, i}; }
__device__ __forceinline__ dc dadd(dc a, dc b) { return dc{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ dc dmul(dc a, dc b) {
  return dc{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ dc dscale(dc a, double s) { return dc{a.re * s, a.im * s}; }
__device__ __forceinline__ dc ddiv_real(dc a, double s) { return dc{a.re / s, a.im / s}; }
__device__ __forceinline__ dc dexp(dc z) {
  double s, c;
  sincos(z.im, &s, &c);
  const double m = exp(z.re);
  return dc{m * c, m * s};
}
__device__ __forceinline__ dc drecip(dc z) {
  const double d = z.re * z.re + z.im * z.im;
  return dc{z.re / d, -z.im / d};
}
// principal square root
__device__ __forceinline__ dc dsqrt(dc z) {
  const double r = hypot(z.re, z.im);
  double re = sqrt(0.5 * (r + fabs(z.re)));
  double im = (re > 0.0) ? z.im / (2.0 * re) : 0.0;
  if (z.re < 0.0) {
    const double t = re;
    re = fabs(im);
    im = (z.im >= 0.0) ? t : -t;
  }
  return dc{re, im};
}

__device__ __forceinline__ float2 to_f2(dc z) { return make_float2(float(z.re), float(z.im)); }

// Nearest float (ties to even) of a double whose magnitude is a normal float
// below 2^127, or zero, in integer instructions: the conversion instructions
// between 64 and 32 bits run at the FP64 rate, which the tables are bound by.
__device__ __forceinline__ float round_f32(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned long long a = b & 0x7FFFFFFFFFFFFFFFull;
  const unsigned m = unsigned((a + 0x0FFFFFFFull + ((a >> 29) & 1)) >> 29) - (896u << 23);
  return __uint_as_float((a ? m : 0u) | (unsigned(b >> 32) & 0x80000000u));
}
// v as FP32 hi + lo, each rounded to nearest.
__device__ __forceinline__ void split_f32(double v, float* hi, float* lo) {
  const unsigned e = (unsigned(__double_as_longlong(v) >> 52)) & 0x7FFu;
  if (e - (1023u - 60u) < 100u) {  // 2^-60 <= |v| < 2^40: lo is zero or a normal float too
    *hi = round_f32(v);
    *lo = round_f32(v - widen_f64(*hi));
  } else {
    *hi = float(v);
    *lo = float(v - double(*hi));
  }
}

// Spatial frequency of DFT bin m on an n-point grid of spacing d (Nyquist negative).
__device__ __forceinline__ double qbin(int m, int n, double d) {
  const int mm = (m < n / 2) ? m : m - n;
  return 2.0 * kPi * double(mm) / (double(n) * d);
}

// exp(i dz [sqrt(k^2 - Q^2) - k]) with the evanescent branch decaying.
__device__ __forceinline__ dc tilted_propagator(double k, double Q2, double dz) {
  const double arg = k * k - Q2;
  if (arg >= 0.0) {
    // sqrt(k^2 - Q^2) - k = -Q^2 / (sqrt(k^2 - Q^2) + k): no cancellation
    const double ph = -dz * Q2 / (sqrt(arg) + k);
    double s, c;
    sincos(ph, &s, &c);
    return dc{c, s};
  }
  const double m = exp(-dz * sqrt(-arg));
  double s, c;
  sincos(-dz * k, &s, &c);
  return dc{m * c, m * s};
}

// First cell j of a row whose x_j = j dx (rounded, so that the decision is
// reproducible) is not below (END = false) or not under (END = true: !(x < b))
// the bound b; sa.nx if none is.
template <bool END>
__device__ int first_cell(const SetupArgs& sa, double b) {
  auto past = [&](int j) {
    const double x = __dmul_rn(double(j), sa.dx);
    return END ? !(x < b) : x >= b;
  };
  const double g = ceil(b / sa.dx);
  int j = g >= 0.0 ? (g < double(sa.nx) ? int(g) : sa.nx) : 0;
  while (j > 0 && past(j - 1)) --j;
  while (j < sa.nx && !past(j)) ++j;
  return j;
}

// Crystal cells [lo, hi) of a row at z_n = n dz from the crystal's boundaries
// (they set the geometry, end of Section 2): x_surface + z tan_psi <= x_j <
// x_end + z tan_psi and z_begin <= z_n < z_end.  Products and sums are rounded
// explicitly (no contraction).
__device__ int2 crystal_row(const SetupArgs& sa, int n) {
  const double z = __dmul_rn(double(n), sa.dz);
  if (!(z >= sa.z_begin && z < sa.z_end)) return make_int2(0, 0);
  const double shift = __dmul_rn(z, sa.tan_psi);
  const int lo = first_cell<false>(sa, __dadd_rn(sa.x_surface, shift));
  const int hi = first_cell<true>(sa, __dadd_rn(sa.x_end, shift));
  return lo < hi ? make_int2(lo, hi) : make_int2(0, 0);
}

// Deformation factor c = Pi exp(+i h u) of every row, with the rows' crystal
// extents (span, 3D: the row pass loads c only there) or their union (ext =
// {lo, -hi}, 2D: the parked march couples only there; starts at kExtNone).
// FP64 only where there is crystal: a row's boundaries are found once instead
// of tested in every cell, and vacuum is written without a look at u.
// 2000 x 4096: 230 -> 71 us.
constexpr int kDefRows = 8;
__global__ void __launch_bounds__(256)
    deformation_kernel(SetupArgs sa, const double* __restrict__ u, float2* cfield, int2* span,
                       int* ext) {
  __shared__ int slo[kDefRows], shi[kDefRows];
  const long long rows = (long long)sa.nz * sa.ny;
  const int pairs = sa.nx / 2;
  for (long long r0 = (long long)blockIdx.x * kDefRows; r0 < rows;
       r0 += (long long)gridDim.x * kDefRows) {
    if (threadIdx.x < kDefRows) {
      int2 b = make_int2(sa.nx, 0);  // a mask's extent is found with its cells
      if (!sa.mask && r0 + threadIdx.x < rows) b = crystal_row(sa, int((r0 + threadIdx.x) / sa.ny));
      slo[threadIdx.x] = b.x;
      shi[threadIdx.x] = b.y;
    }
    __syncthreads();
    const int n_rows = int(min((long long)kDefRows, rows - r0));
    for (int i = threadIdx.x; i < n_rows * pairs; i += blockDim.x) {
      const int r = i / pairs, j = 2 * (i % pairs);
      const size_t cell = size_t(r0 + r) * sa.nx + j;
      float2 c[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        bool in;
        if (sa.mask) {
          in = sa.mask[cell + h] != 0;
          if (in) {
            atomicMin(&slo[r], j + h);
            atomicMax(&shi[r], j + h + 1);
          }
        } else {
          in = j + h >= slo[r] && j + h < shi[r];
        }
        if (in) {
          double s = 0.0, co = 1.0;
          if (u) sincos(sa.h * u[cell + h], &s, &co);
          c[h] = make_float2(float(co), float(s));
        }
      }
      *reinterpret_cast<float4*>(cfield + cell) = make_float4(c[0].x, c[0].y, c[1].x, c[1].y);
    }
    __syncthreads();
    if (threadIdx.x < n_rows) {
      const int lo = slo[threadIdx.x], hi = shi[threadIdx.x];
      if (span) span[r0 + threadIdx.x] = lo < hi ? make_int2(lo, hi) : make_int2(0, 0);
      if (ext && lo < hi) {
        atomicMin(ext, lo);
        atomicMin(ext + 1, -hi);
      }
    }
    __syncthreads();
  }
}

// Power series in w^2 of J0(w) (g1 = 0) or G1(w) = 2 J1(w)/w (g1 = 1) (A&S
// 9.1.10).  It ends where neither a term nor any later one (each at most half the
// one before, once |z| <= k^2 / 2) can change the sum: after a few terms of the w
// of thin slices, instead of a serial chain of 39 that took 80 us.
__device__ dc bessel_j0_g1(dc w2, int g1) {
  const dc z = dscale(w2, -0.25);
  const double az = fabs(z.re) + fabs(z.im);
  dc t = dmk(1, 0), s = dmk(1, 0);
  for (int k = 1; k < 40; ++k) {
    t = ddiv_real(dmul(t, z), double(k) * (k + g1));
    s = dadd(s, t);
    const double tiny = (fabs(t.re) + fabs(t.im)) * 0x1p+54;
    if (2.0 * az <= double(k) * k && tiny <= fabs(s.re) && (z.im == 0.0 || tiny <= fabs(s.im)))
      break;
  }
  return s;
}

// The incident field needs nothing of the tables: its launch starts when all of
// theirs run (programmatic dependent launch), and one block waits for them before
// it ends, so that what follows the incident field follows both.
__device__ __forceinline__ void after_tables() {
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void before_incident() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr int kTabThreads = 128;
constexpr int kTabMaxCh = 8;  // channels per block of tables_kernel

// Coupling coefficients of Eq. fov10 for the 32 channels / sets from 32 `blk` on
// (set fastest), fractions cfr of dz: w^2 = (k dz / cos a)^2 chi_h chi_hbar, a =
// J0 e^{i phi} e^{w^2/8} (Zassenhaus), b+ = i G1 e^{i phi} k dz chi_hbar / (2 cos a),
// b- likewise with chi_h; a split into hi + lo.  One lane an item, and a warp for
// each of the four factors, chains of dependent FP64 instructions that took
// 20 us one after the other, the whole kernel's time for a small plan.
__device__ void store_coef(const SetupArgs& sa, const double* omega, int blk, int n_sets,
                           const double (&cfr)[2], ChannelCoef* coef, int* bad) {
  __shared__ dc part[4][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = 32 * blk + lane;
  double kdz = 0.0, cos_a = 1.0;
  bool ok = i < sa.n_ch * n_sets;
  if (ok) {
    const double k = omega[i / n_sets] / kC;
    const double s_ratio = 0.5 * sa.h / k;
    ok = s_ratio < 1.0;
    if (!ok && bad && w == 0) atomicExch(bad, 1);
    cos_a = sqrt(1.0 - s_ratio * s_ratio);  // cos(alpha), Eq. fov3
    kdz = k * sa.dz * cfr[i % n_sets];
  }
  const dc chih = dmk(sa.chih_re, sa.chih_im), chihb = dmk(sa.chihb_re, sa.chihb_im);
  if (ok) {
    const double r = kdz / cos_a;
    if (w == 2) {
      const dc chi0 = dmk(sa.chi0_re, sa.chi0_im);
      part[2][lane] = dexp(dmul(dmk(0, 1), dscale(chi0, kdz / (2.0 * cos_a))));
    } else {
      const dc w2 = dscale(dmul(chih, chihb), r * r);
      part[w][lane] = w < 2            ? bessel_j0_g1(w2, w)
                      : sa.zassenhaus ? dexp(dscale(w2, 0.125))
                                      : dmk(1, 0);
    }
  }
  __syncthreads();
  if (!ok || w > 1) return;
  const dc phase0 = part[2][lane];
  if (w == 0) {
    const dc a = dmul(dmul(part[0][lane], phase0), part[3][lane]);
    const float2 hi = to_f2(a);
    coef[i].a_hi = hi;
    coef[i].a_lo = make_float2(float(a.re - double(hi.x)), float(a.im - double(hi.y)));
  } else {
    const dc ig1p = dmul(dmk(0, 1), dmul(part[1][lane], phase0));
    const double half = kdz / (2.0 * cos_a);
    coef[i].bp = to_f2(dmul(ig1p, dscale(chihb, half)));
    coef[i].bm = to_f2(dmul(ig1p, dscale(chih, half)));
  }
}

// Position of frequency bin f in the digit-reversed spectrum of n points: the
// base-16 digits of f from the lowest, the last one of what remains.
__device__ __forceinline__ int spectrum_position(int f, int n) {
  int p = 0;
  for (int l = n / 16; l >= 1; l /= 16) {
    p += (f & 15) * l;
    f >>= 4;
    if (l < 16) {
      if (l > 1) p += f;
      break;
    }
  }
  return p;
}

// Tables in the march kernel's order: [ch][env][k][t] for the spectrum position
// p = 16 t + k, env 0 = E0 (+h/2), 1 = Eh (-h/2).  FP64 bound (two operations
// a clock and SM), so:
//  * the phase factor of (Eh, q) is that of (E0, -q) bit for bit, (q - h/2)^2 =
//    (-q + h/2)^2, so one square root, division and sincos serve both; only the
//    Nyquist bin, whose -q is not on the grid, has its own;
//  * a thread keeps its bin for up to kTabMaxCh channels: q and the gains'
//    reciprocals are divided out once;
//  * a grid of 128-bin blocks also spreads a single channel over many SMs, and
//    the coefficients (serial chains) run in blocks of their own in front, a lane
//    of four warps per channel.
// 8192 bins x 512 channels: 1600 -> 771 us (about 100 FP64 instructions a pair
// of entries); two sets of 4096 x 256: 660 -> 327 us; 48 plans of 512 x 1, one
// after the other: 91 -> 11.6 us each (20 with the coefficients in one chain).
__global__ void __launch_bounds__(kTabThreads)
    tables_kernel(SetupArgs sa, int coef_blocks, int cpb, const double* __restrict__ omega,
                  const double* __restrict__ gain, const int* __restrict__ rev, float4* tables,
                  ChannelCoef* coef, int* bad) {
  // fractions of dz of the propagations (tables) and couplings (coefficient
  // sets) of Eq. split-op: order 1: (1; 1); order 2: (1; 1/2); order 4:
  // (t, 1-2t; t/2, (1-t)/2) with t = 1/(2 - 2^(1/3))
  before_incident();
  const double t4 = sa.split_order == 4 ? 1.0 / (2.0 - cbrt(2.0)) : 0.0;
  const int n_sets = sa.split_order == 4 ? 2 : 1;
  if (int(blockIdx.x) < coef_blocks) {
    const double cfr[2] = {sa.split_order == 4 ? 0.5 * t4 : (sa.split_order == 2 ? 0.5 : 1.0),
                           0.5 * (1.0 - t4)};
    store_coef(sa, omega, int(blockIdx.x), n_sets, cfr, coef, bad);
    return;
  }
  __shared__ double sk[kTabMaxCh];
  const int n = sa.nx, T = n / 16, chunks = n / kTabThreads;
  const int blk = int(blockIdx.x) - coef_blocks;
  const int ch0 = (blk / chunks) * cpb, nch = min(cpb, sa.n_ch - ch0);
  if (int(threadIdx.x) < nch) {
    const double k = omega[ch0 + threadIdx.x] / kC;
    sk[threadIdx.x] = 0.5 * sa.h / k < 1.0 ? k : -1.0;  // no Bragg solution: no tables
  }
  __syncthreads();
  const int o = (blk % chunks) * kTabThreads + threadIdx.x;  // slot k T + t of env 0
  const int p = 16 * (o % T) + o / T;
  const int f = rev[p];
  const int pm = spectrum_position((n - f) & (n - 1), n);    // where -q lives
  const int om = (pm % 16) * T + pm / 16;
  const double half_h = 0.5 * sa.h, q = qbin(f, n, sa.dx);
  const double sc0 = 1.0 / (double(n) * gain[p]), sc1 = 1.0 / (double(n) * gain[pm]);
  const double Q = q + half_h;
  const bool nyquist = f == n / 2;
  auto put = [](dc P, double scale, float4* dst) {
    P = dscale(P, scale);
    float4 v;
    split_f32(P.re, &v.x, &v.z);
    split_f32(P.im, &v.y, &v.w);
    *dst = v;
  };
  for (int c = 0; c < nch; ++c) {
    const double k = sk[c];
    if (k < 0.0) continue;
    for (int set = 0; set < n_sets; ++set) {
      const double dz = sa.dz * (set ? 1.0 - 2.0 * t4 : sa.split_order == 4 ? t4 : 1.0);
      float4* out = tables + (size_t(ch0 + c) * n_sets + set) * 2 * n;
      dc P = tilted_propagator(k, Q * Q, dz);
      put(P, sc0, out + o);
      if (nyquist) P = tilted_propagator(k, (q - half_h) * (q - half_h), dz);
      put(P, sc1, out + n + om);
    }
  }
}

// 3D: per channel and stored x-frequency column cs (px = 16 (cs % T) + cs / T),
// the anchor exp(i dz (K - k)) / (nx ny g_x(px)), K = sqrt(k^2 - (qx +- h/2)^2),
// as FP32 hi + lo, and the curvature factor -dz / (2 K) of the qy correction.
// Blocks of 128 columns of a channel; coefficients as in tables_kernel.
__global__ void __launch_bounds__(kTabThreads)
    tables3d_kernel(SetupArgs sa, int coef_blocks, const double* __restrict__ omega,
                    const double* __restrict__ gainx, const int* __restrict__ revx, float4* anchor,
                    float* gcorr, ChannelCoef* coef) {
  before_incident();
  if (int(blockIdx.x) < coef_blocks) {
    const double cfr[2] = {sa.coupling_frac, 0.0};
    store_coef(sa, omega, int(blockIdx.x), 1, cfr, coef, nullptr);
    return;
  }
  const int n = sa.nx, T = n / 16, chunks = n / kTabThreads;
  const int blk = int(blockIdx.x) - coef_blocks;
  const int ch = blk / chunks, cs = (blk % chunks) * kTabThreads + threadIdx.x;
  const double k = omega[ch] / kC;
  const double half_h = 0.5 * sa.h;
  const int px = 16 * (cs % T) + cs / T;
  const double qx = qbin(revx[px], n, sa.dx);
  const double scale = 1.0 / (double(n) * double(sa.ny) * gainx[px]);
  for (int env = 0; env < 2; ++env) {
    const double Q = env == 0 ? qx + half_h : qx - half_h;
    const double K2 = k * k - Q * Q;
    dc P = tilted_propagator(k, Q * Q, sa.dz);
    P = dscale(P, scale);
    const float2 hi = to_f2(P);
    const float2 lo = make_float2(float(P.re - double(hi.x)), float(P.im - double(hi.y)));
    const size_t o = (size_t(ch) * 2 + env) * n + cs;
    anchor[o] = make_float4(hi.x, hi.y, lo.x, lo.y);
    gcorr[o] = K2 > 0.0 ? float(-sa.dz / (2.0 * sqrt(K2))) : 0.f;
  }
}

// Incident field A+ = S pref g(x, y) e^{i dq x} and its norm.  FP64 bound like
// the tables, so what is shared is computed once:
//  * the Gaussian is the same for every channel, and in 3D the phase for every
//    row: a block has up to kIncMaxCh channels of its cells;
//  * |A+|^2 = |S pref|^2 |g|^2, so one sum of |g|^2 serves every channel;
//  * cells whose value rounds to zero in FP32 are not computed (a beam of waist
//    w0 fills 20 w0), and the rest is rounded by integer instructions.
// The operations of a cell and their order do not depend on the grouping.
// 4096 x 1024 channels: 895 -> 230 us; 512 x 512 x 128: 7.48 ms -> 493 us;
// 256 x 512 x 24: 3.71 ms -> 165 us.
constexpr int kIncThreads = 256;
constexpr int kIncMaxCh = 8;
constexpr int kIncTile = 64;   // 3D: cells of a block in x
constexpr int kIncRows = 16;   // and in y

__device__ __forceinline__ float narrow_f32(double v) {
  const unsigned e = (unsigned(__double_as_longlong(v) >> 52)) & 0x7FFu;
  return e - (1023u - 120u) < 240u ? round_f32(v) : float(v);  // else zero, denormal, huge or NaN
}

__device__ __forceinline__ dc denominator(const SetupArgs& sa) {
  return dmk(1.0, sa.zR != 0.0 ? sa.zx / sa.zR : 0.0);
}
// Factors of all channels and cells: 1 / denominator, and its square root (2D) or
// itself (3D), which S is multiplied by.  At the waist (denominator 1) they are
// what the general formulas give, without their chains of divisions and roots.
struct Beam {
  dc inv_den, pref;
};
__device__ Beam beam_factors(const SetupArgs& sa) {
  const dc den = denominator(sa);
  if (den.im == 0.0) return Beam{dmk(1.0, -den.im), dmk(1.0, -den.im)};
  const dc inv = drecip(den);
  return Beam{inv, sa.dims == 3 ? inv : drecip(dsqrt(den))};
}
__device__ __forceinline__ dc amplitude(dc pref, double2 w) { return dmul(dmk(w.x, w.y), pref); }
// g at the squared distance r2 from the beam's centre
__device__ __forceinline__ dc gauss(const SetupArgs& sa, dc inv_den, double r2) {
  const double rr = r2 / (sa.w0 * sa.w0);
  if (inv_den.im == 0.0) return dmk(exp(inv_den.re * -rr), 0.0);
  return dexp(dscale(inv_den, -rr));
}
// FP32 bounds that tell where A+ is zero in FP32 (below e^-103.97) without FP64:
// log|S pref| from above, log|g| at r2 (with a margin over their rounding)
__device__ __forceinline__ float log_bound(dc z) {
  return logf(float(fmax(fabs(z.re), fabs(z.im)))) + 0.35f;
}
__device__ __forceinline__ float log_gauss(const SetupArgs& sa, dc inv_den) {
  return -float(inv_den.re / (sa.w0 * sa.w0));
}
constexpr float kLogZero = -106.f;
// |g|^2 below e^-760 is zero in FP64, g below e^-750
constexpr float kLogNormZero = -380.f, kLogGaussZero = -750.f;
// A grid whose cells all have |g| < e^-200 (a beam 14 waists off its edge, or one that
// falls between two cells): the norm's sum is of |kFarScale g|^2, so that |S g|^2 of any
// S is found where |g|^2 alone would be lost.
constexpr float kLogFar = -200.f;
constexpr double kFarScale = 0x1p600;

// Constants of a block's channels, one lane of the first warp each; below the
// log|g| `least` no channel's value is above zero (-inf with a NaN amplitude).
struct IncChannels {
  Beam beam;
  dc sp[kIncMaxCh];
  double dq[kIncMaxCh];
  float bound[kIncMaxCh];
  float least, norm_zero, log_g;  // log_g: log_gauss
  bool far;
};
__device__ void load_channels(const SetupArgs& sa, const double* omega, const double2* weight,
                              int ch0, int nch, IncChannels* s) {
  const int c = threadIdx.x;
  if (c < nch) {
    const double k = omega[ch0 + c] / kC;
    s->dq[c] = k * sin(sa.theta_i) - 0.5 * sa.h;
    const Beam beam = beam_factors(sa);
    s->sp[c] = amplitude(beam.pref, weight[ch0 + c]);
    s->bound[c] = log_bound(s->sp[c]);
    if (c == 0) s->beam = beam;
  }
  __syncthreads();
  if (c == 0) {
    float least = INFINITY;
    for (int i = 0; i < nch; ++i) {
      const float l = kLogZero - s->bound[i];
      least = l == l ? fminf(least, l) : -INFINITY;  // stays: fminf(-inf, l)
    }
    s->least = least;
    // from the beam's centre to a nearest cell (in 3D there is one at y = 0)
    const float j = fminf(fmaxf(rintf(float(sa.x0) / float(sa.dx)), 0.f), float(sa.nx - 1));
    const double d = sa.x0 - double(j) * sa.dx;
    s->log_g = log_gauss(sa, s->beam.inv_den);
    s->far = s->log_g * float(d * d) < kLogFar;
    s->norm_zero = s->far ? kLogGaussZero : kLogNormZero;
  }
  __syncthreads();
}
__device__ __forceinline__ double norm_part(dc g, bool far) {
  if (far) g = dscale(g, kFarScale);
  return g.re * g.re + g.im * g.im;
}

// The last of `blocks` blocks to leave their parts of the sum of |g|^2 adds the
// `parts` parts, in an order that depends on their number alone, and writes every
// channel's norm.
__device__ void finish_norm(const SetupArgs& sa, const double2* weight, dc pref, bool far,
                            int blocks, int parts, NormScratch* scratch, double* inc_norm) {
  __shared__ int last;
  __shared__ double total;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&scratch->arrived, 1) == blocks - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x < 32) {
    double sum = 0.0;
    for (int i = threadIdx.x; i < parts; i += 32) sum += __ldcg(&scratch->part[i]);
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
    if (threadIdx.x == 0) {
      total = sum;
      scratch->arrived = 0;  // for the next pulse
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < sa.n_ch; c += blockDim.x) {
    const dc sp = amplitude(pref, weight[c]);
    double norm = (sp.re * sp.re + sp.im * sp.im) * total;
    if (far) {
      const double m = hypot(sp.re, sp.im) * sqrt(total) / kFarScale;
      norm = m * m;
    }
    inc_norm[c] = norm;
  }
}

// 2D: a block has THREADS cells, one a thread, of up to kIncMaxCh channels; the
// norm's parts are of 32 cells.  A warp's FP64 instruction takes an SM 16 clocks, so
// a small plan has blocks of 64: one channel of 512 points 21.4 -> 9.6 us (with
// the beam's factors once a block, not once a thread), of which most is beside
// the tables.
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    incident_kernel(SetupArgs sa, int cpb, const double* __restrict__ omega,
                    const double2* __restrict__ weight, float2* e0, float2* eh, double* inc_norm,
                    NormScratch* scratch) {
  __shared__ IncChannels sc;
  const int chunks = sa.nx / THREADS;
  const int ch0 = (int(blockIdx.x) / chunks) * cpb, nch = min(cpb, sa.n_ch - ch0);
  const int chunk = int(blockIdx.x) % chunks, j = chunk * THREADS + threadIdx.x;
  load_channels(sa, omega, weight, ch0, nch, &sc);
  const dc inv_den = sc.beam.inv_den;
  const double x = double(j) * sa.dx, d = x - sa.x0, r2 = d * d;
  const float lg = sc.log_g * float(r2);
  dc g = dmk(0.0, 0.0);
  if (!(lg < (ch0 == 0 ? fminf(sc.least, sc.norm_zero) : sc.least))) g = gauss(sa, inv_den, r2);
  for (int c = 0; c < nch; ++c) {
    float2 v = make_float2(0.f, 0.f);
    if (!(lg < kLogZero - sc.bound[c])) {
      double s, co;
      sincos(sc.dq[c] * x, &s, &co);
      const dc a = dmul(dmul(sc.sp[c], g), dmk(co, s));
      v = make_float2(narrow_f32(a.re), narrow_f32(a.im));
    }
    e0[size_t(ch0 + c) * sa.nx + j] = v;
    eh[size_t(ch0 + c) * sa.nx + j] = make_float2(0.f, 0.f);
  }
  if (ch0 == 0) {
    double part = norm_part(g, sc.far);
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, off);
    if (threadIdx.x % 32 == 0) scratch->part[j / 32] = part;
    finish_norm(sa, weight, sc.beam.pref, sc.far, chunks, sa.nx / 32, scratch, inc_norm);
  }
  after_tables();
}

// 3D: a block has a tile of kIncTile x kIncRows cells of up to kIncMaxCh channels,
// the phases of its columns in shared memory.  The beam fills a few tiles and the
// rest is written as zeros, without phases; the low tiles spread the beam's FP64
// work over the SMs (64 rows: the few blocks with the beam took 150 us each, two or
// three of them on an SM).  512 x 512 x 128 channels 490 -> 293 us, 256 x 512 x 24
// 165 -> 106.
__global__ void __launch_bounds__(kIncThreads)
    incident3d_kernel(SetupArgs sa, const double* __restrict__ omega,
                      const double2* __restrict__ weight, float2* e0, float2* eh,
                      double* inc_norm, NormScratch* scratch) {
  __shared__ IncChannels sc;
  __shared__ dc ph[kIncMaxCh][kIncTile];
  __shared__ double red[kIncThreads / 32];
  const int tx = sa.nx / kIncTile, tiles = tx * (sa.ny / kIncRows);
  const int ch0 = (int(blockIdx.x) / tiles) * kIncMaxCh, nch = min(kIncMaxCh, sa.n_ch - ch0);
  const int tile = int(blockIdx.x) % tiles;
  const int jt = (tile % tx) * kIncTile, rt = (tile / tx) * kIncRows;
  load_channels(sa, omega, weight, ch0, nch, &sc);
  const size_t plane = size_t(sa.nx) * sa.ny;
  // two neighbouring cells a thread: 32 threads a row of the tile
  const int jj = 2 * (threadIdx.x % (kIncTile / 2));
  const float lgs = sc.log_g;
  const float least = ch0 == 0 ? fminf(sc.least, sc.norm_zero) : sc.least;
  // no cell of the tile is nearer to the beam's centre than this, and rounding
  // keeps the order
  auto nearest = [](double lo, double hi, double at) {
    return at < lo ? lo - at : at > hi ? hi - at : 0.0;
  };
  const double dx0 = nearest(double(jt) * sa.dx, double(jt + kIncTile - 1) * sa.dx, sa.x0);
  const double dy0 = nearest((double(rt) - double(sa.ny / 2)) * sa.dy,
                             (double(rt + kIncRows - 1) - double(sa.ny / 2)) * sa.dy, 0.0);
  if (lgs <= 0.f && lgs * float(dx0 * dx0 + dy0 * dy0) < least) {
    for (int r = threadIdx.x / (kIncTile / 2); r < kIncRows; r += kIncThreads / (kIncTile / 2))
      for (int c = 0; c < nch; ++c) {
        const size_t at = size_t(ch0 + c) * plane + size_t(rt + r) * sa.nx + jt + jj;
        *reinterpret_cast<float4*>(e0 + at) = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(eh + at) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    if (ch0 == 0) {
      if (threadIdx.x == 0) scratch->part[tile] = 0.0;
      finish_norm(sa, weight, sc.beam.pref, sc.far, tiles, tiles, scratch, inc_norm);
    }
    after_tables();
    return;
  }
  for (int i = threadIdx.x; i < nch * kIncTile; i += kIncThreads) {
    const int c = i / kIncTile, j = i % kIncTile;
    double s, co;
    sincos(sc.dq[c] * (double(jt + j) * sa.dx), &s, &co);
    ph[c][j] = dmk(co, s);
  }
  __syncthreads();
  const dc inv_den = sc.beam.inv_den;
  double acc = 0.0;
  for (int r = threadIdx.x / (kIncTile / 2); r < kIncRows; r += kIncThreads / (kIncTile / 2)) {
    const double y = (double(rt + r) - double(sa.ny / 2)) * sa.dy;
    dc g[2];
    float lg[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double x = double(jt + jj + h) * sa.dx;
      const double r2 = (x - sa.x0) * (x - sa.x0) + y * y;
      lg[h] = lgs * float(r2);
      g[h] = dmk(0.0, 0.0);
      if (!(lg[h] < least)) g[h] = gauss(sa, inv_den, r2);
      acc += norm_part(g[h], sc.far);
    }
    for (int c = 0; c < nch; ++c) {
      float2 v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        v[h] = make_float2(0.f, 0.f);
        if (!(lg[h] < kLogZero - sc.bound[c])) {
          const dc a = dmul(dmul(sc.sp[c], g[h]), ph[c][jj + h]);
          v[h] = make_float2(narrow_f32(a.re), narrow_f32(a.im));
        }
      }
      const size_t at = size_t(ch0 + c) * plane + size_t(rt + r) * sa.nx + jt + jj;
      *reinterpret_cast<float4*>(e0 + at) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
      *reinterpret_cast<float4*>(eh + at) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  if (ch0 == 0) {
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kIncThreads / 32; ++w) acc += red[w];
      scratch->part[tile] = acc;
    }
    finish_norm(sa, weight, sc.beam.pref, sc.far, tiles, tiles, scratch, inc_norm);
  }
  after_tables();
}

}  // namespace

cudaError_t launch_deformation(const SetupArgs& sa, const double* u_dev, float2* cfield,
                               int2* span, int* ext, cudaStream_t s) {
  if (ext) {
    const cudaError_t e = cudaMemsetAsync(ext, kExtNoneByte, 2 * sizeof(int), s);
    if (e != cudaSuccess) return e;
  }
  const long long groups = ((long long)sa.ny * sa.nz + kDefRows - 1) / kDefRows;
  deformation_kernel<<<unsigned(groups < 152 * 32 ? groups : 152 * 32), 256, 0, s>>>(sa, u_dev, cfield,
                                                                                    span, ext);
  return cudaGetLastError();
}

cudaError_t launch_tables(const SetupArgs& sa, const double* omega, const double* gain,
                          const int* rev, float4* tables, ChannelCoef* coef, int* bad,
                          cudaStream_t s) {
  const int sets = sa.split_order == 4 ? 2 : 1, coef_blocks = (sa.n_ch * sets + 31) / 32;
  // as many channels a block as leave eight blocks an SM (16 warps keep FP64 busy)
  const long long chunks = sa.nx / kTabThreads;
  int cpb = kTabMaxCh;
  while (cpb > 1 && chunks * ((sa.n_ch + cpb - 1) / cpb) < 152 * 8) cpb /= 2;
  const long long blocks = coef_blocks + chunks * ((sa.n_ch + cpb - 1) / cpb);
  tables_kernel<<<unsigned(blocks), kTabThreads, 0, s>>>(sa, coef_blocks, cpb, omega, gain, rev,
                                                         tables, coef, bad);
  return cudaGetLastError();
}

cudaError_t launch_tables3d(const SetupArgs& sa, const double* omega, const double* gainx,
                            const int* revx, float4* anchor, float* gcorr, ChannelCoef* coef,
                            cudaStream_t s) {
  const int coef_blocks = (sa.n_ch + 31) / 32;
  tables3d_kernel<<<coef_blocks + sa.n_ch * (sa.nx / kTabThreads), kTabThreads, 0, s>>>(
      sa, coef_blocks, omega, gainx, revx, anchor, gcorr, coef);
  return cudaGetLastError();
}

cudaError_t launch_incident(const SetupArgs& sa, const double* omega, const double2* weight,
                            float2* e0, float2* eh, double* inc_norm, NormScratch* scratch,
                            cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.stream = s;
  cudaLaunchAttribute at{};  // see after_tables
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (sa.dims == 3) {
    const int tiles = (sa.nx / kIncTile) * (sa.ny / kIncRows);
    const int groups = (sa.n_ch + kIncMaxCh - 1) / kIncMaxCh;
    cfg.gridDim = dim3(unsigned(tiles * groups));
    cfg.blockDim = dim3(kIncThreads);
    return cudaLaunchKernelEx(&cfg, incident3d_kernel, sa, omega, weight, e0, eh, inc_norm, scratch);
  }
  // as in launch_tables: several channels a block once every SM has eight warps'
  // work, and small blocks where that is not even so with one
  int threads = kIncThreads;
  auto blocks = [&](int cpb) { return sa.nx / threads * ((sa.n_ch + cpb - 1) / cpb); };
  int cpb = kIncMaxCh;
  while (cpb > 1 && blocks(cpb) < 152 * 2) cpb /= 2;
  if (blocks(cpb) < 152 * 2) threads = 64;
  cfg.gridDim = dim3(unsigned(blocks(cpb)));
  cfg.blockDim = dim3(unsigned(threads));
  return cudaLaunchKernelEx(&cfg, threads == 64 ? incident_kernel<64> : incident_kernel<kIncThreads>,
                            sa, cpb, omega, weight, e0, eh, inc_norm, scratch);
}

}  // namespace bpm
