// Streamed passes of the 3D march (launch form 2; the passes' steps and traffic
// are those of bpm_3d.cu).
//
// Between passes the two envelopes of an element lie side by side: spec
// [ch][c][y]{E0, Eh}, c = (px % E) (NX / E) + px / E for the x-spectrum position
// px, E elements a thread.  In both passes a lane holds one envelope of its
// elements and its neighbour the other, so every access of a warp to shared or
// global memory is a run of 16-byte pairs (no bank conflicts in the tiles, where
// separate planes had 2- to 4-way ones), and the coupling takes the other
// envelope by a shuffle.
//
// A 512-point transform gives a thread 32 elements: its first radix-16 stage on
// two groups, one exchange, then the radix-16 and radix-2 stages of a whole
// block of 32 positions without another.  What bound these passes was the
// shared-memory data path (68 % of its cycles in the row pass) and the stalls
// around exchanges, of which there were two a transform; HBM was half idle.
// 512 x 512 x 128 channels: a column pass 221 -> 202 us (5.3 TB/s, 78 % of the
// copy bandwidth), a row pass 271 -> 232 us (4.6 TB/s, 68 %); a step at 1024 x
// 1024 x 32 644 -> 606 us, 256 x 256 x 128 122 -> 110.  They are now bound by the
// issue of 12 to 16 warps an SM (57 %), the FP32 pipe and the L1 data path (60 %
// each), no one of them full.
// Every element's operations and their order are those of the other forms.
#include <cuda.h>  // CUtensorMap and its encoder's types (the encoder is fetched at run time)
#include <cuda_runtime.h>

#include "bpm_fft.cuh"
#include "bpm_half.cuh"
#include "bpm_internal.h"
#include "bpm_tma.cuh"

namespace bpm {
namespace {

// Transform of N points held by TH threads of E elements, one envelope (pairs of
// neighbouring lanes hold the two).  Element e = 16 h + k of thread t is, in
// space, position t + TH h + (N / 16) k, and in the spectrum E t + (its order
// `spec(e)`).  buf: this lane's half of the group's exchange region, position p
// at buf[2 (p + p / kPad)].
template <int N>
struct FftL {
  static_assert(N == 256 || N == 512 || N == 1024, "3D transforms");
  static constexpr int E = N == 512 ? 32 : 16;
  static constexpr int H = E / 16;
  static constexpr int TH = N / E;
  static constexpr int kThreads = 2 * TH;  // both envelopes
  static constexpr int kPad = E;           // one spare slot per block of a thread: odd strides
  static constexpr int kSlots = N + N / kPad;

  static BPM_DEV void sync(int g) {
    if constexpr (kThreads == 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kThreads) : "memory");
  }
  __host__ __device__ static constexpr int slot(int p) { return 2 * (p + p / kPad); }
  // space position of element e of thread t
  static BPM_DEV int pos(int t, int e) { return t + TH * (e / 16) + (N / 16) * (e % 16); }
  // element that holds spectrum position E t + q
  static BPM_DEV constexpr int elem(int q) { return N == 512 ? 16 * (q & 1) + (q >> 1) : q; }

  template <bool INV, bool PA>
  static BPM_DEV void dft(float2 (&v)[H][16]) {
#pragma unroll
    for (int h = 0; h < H; ++h) {
      if (!PA)
        dft16_sep<INV>(v[h]);
      else if (INV)
        dft16_inv<false, false, true>(v[h]);
      else
        dft16_fwd<false, false, true>(v[h]);
    }
  }
  // A stage twiddle.  With 32 elements a thread (and at 256, with more warps) by
  // plain loads, which the barriers hold where they are used: as read-only ones
  // they are hoisted, out of the whole loop over tiles at worst, and spill (512
  // x 512 x 128 channels: 471 against 447 us a step).  At 1024 points there are
  // registers to keep them (605 against 633 us, 1024 x 1024 x 32).
  static BPM_DEV float2 load_tw(const float2* p) {
    if constexpr (N == 1024)
      return __ldg(p);
    else
      return *p;
  }
  // twiddles of the first stage (thread order: twiddle_order on the host)
  template <bool INV>
  static BPM_DEV void twid0(float2 (&v)[H][16], const float2* tw, int t) {
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int m = 1; m < 16; ++m) {
        const float2 w = load_tw(tw + (m - 1) * (N / 16) + t + TH * h);
        v[h][m] = INV ? c_mulc(v[h][m], w) : c_mul(v[h][m], w);
      }
  }
  // of the second: W_32^m on the odd positions at 512 (immediates), a table at 1024
  template <bool INV>
  static BPM_DEV void twid1(float2 (&v)[H][16], const float2* tw, int t) {
    if constexpr (N == 512) {
#pragma unroll
      for (int m = 1; m < 16; ++m) {
        const float2 w = make_float2(w32_re(m), w32_im(m));
        v[1][m] = INV ? c_mulc(v[1][m], w) : c_mul(v[1][m], w);
      }
    } else if constexpr (N == 1024) {
#pragma unroll
      for (int m = 1; m < 16; ++m) {
        const float2 w = load_tw(tw + 15 * 64 + (m - 1) * 4 + t % 4);
        v[0][m] = INV ? c_mulc(v[0][m], w) : c_mul(v[0][m], w);
      }
    }
  }
  // radix-2 (512: across the halves) or radix-4 (1024: consecutive) last stage
  template <bool INV, bool PA>
  static BPM_DEV void last(float2 (&v)[H][16]) {
    if constexpr (N == 512) {
#pragma unroll
      for (int m = 0; m < 16; ++m) dft2(v[0][m], v[1][m]);
    } else if constexpr (N == 1024) {
      last_stage<4, INV, false, false, true>(v[0]);
    }
  }

  // layout 0: space / first stage; 1: second stage; 2: last stage (1024)
  // (t's part never carries into the next block: a base per thread and constant offsets)
  template <int L>
  __host__ __device__ static constexpr int at(int t, int h, int k) {
    return L == 0                ? t + TH * h + (N / 16) * k
           : L == 1 && N == 512  ? 32 * t + h + 2 * k
           : L == 1 && N == 1024 ? (t / 4) * 64 + t % 4 + 4 * k
                                 : 16 * t + k;
  }
  template <int LF, int LT>
  static BPM_DEV void xchg(float2 (&v)[H][16], float2* buf, int t, int g) {
    float2* st = buf + slot(at<LF>(t, 0, 0));
    const float2* ld = buf + slot(at<LT>(t, 0, 0));
    sync(g);  // the group's reads of the previous exchange are done
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int k = 0; k < 16; ++k) st[slot(at<LF>(0, h, k))] = v[h][k];
    sync(g);
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int k = 0; k < 16; ++k) v[h][k] = ld[slot(at<LT>(0, h, k))];
  }

  template <bool PA>
  static BPM_DEV void fwd(float2 (&v)[H][16], float2* buf, const float2* tw, int t, int g) {
    dft<false, PA>(v);
    twid0<false>(v, tw, t);
    xchg<0, 1>(v, buf, t, g);
    dft<false, PA>(v);
    twid1<false>(v, tw, t);
    if constexpr (N == 1024) xchg<1, 2>(v, buf, t, g);
    last<false, PA>(v);
  }
  // inverse transform up to and with its last exchange, and the rest
  template <bool PA>
  static BPM_DEV void inv_head(float2 (&v)[H][16], float2* buf, const float2* tw, int t, int g) {
    last<true, PA>(v);
    if constexpr (N == 1024) xchg<2, 1>(v, buf, t, g);
    twid1<true>(v, tw, t);
    dft<true, PA>(v);
    xchg<1, 0>(v, buf, t, g);
  }
  template <bool PA>
  static BPM_DEV void inv_tail(float2 (&v)[H][16], const float2* tw, int t) {
    twid0<true>(v, tw, t);
    dft<true, PA>(v);
  }
};

// Passes of a run after the first are programmatic dependents of the pass before:
// their blocks start in its empty end, set themselves up and wait here for it to
// complete (and with it, in turn, every earlier one).  That hides a launch's 2 us
// where the passes are short: us a step 256 x 256 x 1 channel 10.3 -> 8.4, 256 x 512
// x 8 24.7 -> 20.2, 256 x 256 x 64 57.7 -> 53.6, 1024 x 512 x 16 152.3 -> 149.5, 512 x
// 512 x 64 227.0 -> 225.4 (256 x 512 x 24 47.6 -> 48.1: its grids leave no room to start
// in).
BPM_DEV void pass_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... Params, typename... Args>
cudaError_t launch_pass(void (*kernel)(Params...), int blocks, int threads, size_t smem, bool follow,
                        cudaStream_t s, const Args&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(blocks));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = follow ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Column pass: each group of 2 TH lanes walks its share of the n_ch nx columns
// (both envelopes of one, 16 NY contiguous bytes): forward y, propagator,
// inverse y, in place.  A bulk copy brings the next column into the group's
// buffer once the inverse transform's exchange has been read, under its last
// stage and the stores; with 16 warps an SM that covers the copy, and one
// buffer a group is all there is room for.  A wait that gives up records
// kStatusTmaTimeout, waits once more (bounded) and ends the group.
template <int NY>
struct ColStream {
  using F = FftL<NY>;
  static constexpr int kBlock = 128;
  static constexpr int G = kBlock / F::kThreads;
  static constexpr int kBlocksPerSm = NY == 256 ? 5 : 4;
  static constexpr uint32_t kBytes = NY * 16u;
  static constexpr size_t kSmem =
      size_t(G) * F::kSlots * 16 + G * sizeof(uint64_t) + (kBlock / 32) * sizeof(int);
};

template <int NY>
__global__ void __launch_bounds__(ColStream<NY>::kBlock, ColStream<NY>::kBlocksPerSm)
    col_stream_kernel(Pass3DArgs A, int n_ch, int* status) {
  using C = ColStream<NY>;
  using F = typename C::F;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int g = threadIdx.x / F::kThreads, l = threadIdx.x % F::kThreads;
  const int t = l >> 1, env = l & 1;
  float2* area = reinterpret_cast<float2*>(smem_raw) + size_t(g) * 2 * F::kSlots;
  float2* buf = area + env;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + size_t(C::G) * F::kSlots * 16) + g;
  const int lx = 31 - __clz(A.nx), lt = A.nx == 512 ? 4 : lx - 4;  // log2 of nx and of its TH
  const int n_cols = n_ch << lx, stride = int(gridDim.x) * C::G;
  int col = int(blockIdx.x) * C::G + g;
  float2* const spec = A.s0;
  auto issue = [&](int c) {
    mbar_arrive_expect_tx(bar, C::kBytes);
    bulk_load(area, spec + size_t(c) * 2 * NY, C::kBytes, bar);
  };
  if (l == 0) {
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  pass_begin();
  if (l == 0 && col < n_cols) issue(col);
  F::sync(g);
  uint32_t phase = 0;
  for (; col < n_cols; col += stride) {
    // the column's anchor: position px of c in this layout, at (px % 16) (nx / 16) + px / 16
    const int c = col & (A.nx - 1), px = ((c & ((1 << lt) - 1)) << (lx - lt)) + (c >> lt);
    const int ia = (((col >> lx) * 2 + env) << lx) + ((px & 15) << (lx - 4)) + (px >> 4);
    const float4 an = A.anchor[ia];
    const float gc = A.gcorr[ia];
    bool ok = mbar_wait(bar, phase);
    if constexpr (F::kThreads == 32)
      ok = __all_sync(0xFFFFFFFFu, ok);
    else
      ok = __syncthreads_and(ok);  // one group a block
    if (!ok) {
      if (l == 0) atomicExch(status, kStatusTmaTimeout);
      mbar_wait(bar, phase);  // the copy still in flight, bounded
      return;
    }
    phase ^= 1u;
    float2 v[F::H][16];
#pragma unroll
    for (int h = 0; h < F::H; ++h)
#pragma unroll
      for (int k = 0; k < 16; ++k) v[h][k] = buf[2 * F::pos(t, 16 * h + k)];
    F::template fwd<true>(v, buf, A.twy, t, g);
#pragma unroll
    for (int q = 0; q < F::E; ++q) {
      const int py = F::E * t + q;
      const float2 qd = A.qy[(py % 16) * (NY / 16) + py / 16];  // {qy^2, 1/g_y - 1}
      float2& a = v[F::elem(q) / 16][F::elem(q) % 16];
      const float cr = qd.x * gc;
      const float2 w = c_mul2(a, an);
      const float2 f = make_float2(fmaf(-0.5f * cr, cr, qd.y), cr);
      a = make_float2(fmaf(w.x, f.x, fmaf(-w.y, f.y, w.x)), fmaf(w.x, f.y, fmaf(w.y, f.x, w.y)));
    }
    // inverse transform, with the next column's copy after its last exchange
    F::template inv_head<true>(v, buf, A.twy, t, g);
    F::sync(g);  // every read of the buffer is done before it is refilled
    if (l == 0 && col + stride < n_cols) {
      fence_proxy_async_smem();
      issue(col + stride);
    }
    F::template inv_tail<true>(v, A.twy, t);
    float2* out = spec + size_t(col) * 2 * NY + env;
#pragma unroll
    for (int h = 0; h < F::H; ++h)
#pragma unroll
      for (int k = 0; k < 16; ++k) out[2 * F::pos(t, 16 * h + k)] = v[h][k];
  }
}

BPM_DEV float2 shfl2(float2 v, int src) {
  return make_float2(__shfl_sync(0xFFFFFFFFu, v.x, src), __shfl_sync(0xFFFFFFFFu, v.y, src));
}

// Row pass: each block walks tiles (channel, R rows of y).  A tile is the box
// {R 16-byte pairs of y, NX columns} of the spectrum, laid out by the copy engine
// as NX segments of R pairs, the pairs swizzled within the segment; MODE 1
// brings the next tile in while this one is transformed and sends results out
// through the rows' exchange regions.  MODE 0 (first of a run): natural rows
// (e0, eh) in, forward x, tile out; MODE 1: tile in, inverse x, coupling,
// forward x, tile out; MODE 2 (last): tile in, inverse x, coupling, natural rows
// out.
template <int NX, int R>
struct RowStream {
  using F = FftL<NX>;
  static constexpr int kBlock = R * F::kThreads;
  static constexpr int kSeg = R * 16;
  static constexpr int kBoxes = NX / 256;
  static constexpr uint32_t kStage = uint32_t(NX) * kSeg;
  static constexpr uint32_t kXchg = (uint32_t(R) * F::kSlots * 16u + 1023u) / 1024u * 1024u;
  // 1 KB of slack aligns the stage to the swizzle pattern's 1024-byte period
  static constexpr size_t kSmem = 1024 + size_t(kStage) + kXchg + 16;
  static constexpr int kBlocksPerSm = kSmem > 75 * 1024 ? 1 : kBlock == 256 ? 2 : 3;
  static_assert(kSeg == 64 || kSeg == 128, "segment = swizzle span");
  static_assert(kXchg >= kStage, "the output tile fits in the exchange regions");
  static_assert(kSmem <= 227 * 1024, "shared memory of a block");
  // byte offset of pair (t, r); column q TH + t lies q kStep behind (the swizzle
  // repeats every kSeg columns at most)
  static BPM_DEV uint32_t at(int t, int r) {
    const uint32_t lin = uint32_t(t) * uint32_t(kSeg) + uint32_t(r) * 16u;
    return lin ^ (((lin >> 7) & uint32_t(R - 1)) << 4);
  }
  static constexpr int kStep = F::TH * kSeg;
  static_assert(kStep / 128 % R == 0, "a step leaves the swizzle as it is");
};

// Scalar butterfly additions, as in row_pass_kernel: there the compiler fuses the
// c8 products of the inner twiddles into them, which the packed ones never do.
constexpr bool kRowPacked = false;

template <int NX, int R, int MODE>
__global__ void __launch_bounds__(RowStream<NX, R>::kBlock, RowStream<NX, R>::kBlocksPerSm)
    row_stream_kernel(const __grid_constant__ CUtensorMap map, Pass3DArgs A, int n_ch, int* status) {
  using L = RowStream<NX, R>;
  using F = typename L::F;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* stage = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  unsigned char* xreg = stage + L::kStage;  // exchange regions, then the output tile
  uint64_t* bar = reinterpret_cast<uint64_t*>(xreg + L::kXchg);
  const int g = threadIdx.x / F::kThreads;  // row of the tile
  const int l = threadIdx.x % F::kThreads, t = l >> 1, env = l & 1, lane = threadIdx.x & 31;
  float2* buf = reinterpret_cast<float2*>(xreg) + size_t(g) * 2 * F::kSlots + env;
  const uint32_t mine = L::at(t, g) + 8u * env;
  const int tiles_per_ch = A.ny / R, n_tiles = n_ch * tiles_per_ch;
  auto issue = [&](int tile) {  // one thread
    const int cy = (tile / tiles_per_ch) * NX, x = 4 * (tile % tiles_per_ch) * R;
    mbar_arrive_expect_tx(bar, L::kStage);
#pragma unroll
    for (int b = 0; b < L::kBoxes; ++b)
      tma_load_2d(stage + b * 256 * L::kSeg, &map, x, cy + b * 256, bar);
  };
  int tile = blockIdx.x;
  if (MODE != 0 && threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  pass_begin();
  if (MODE != 0 && threadIdx.x == 0 && tile < n_tiles) issue(tile);
  __syncthreads();
  uint32_t phase = 0;
  for (; tile < n_tiles; tile += gridDim.x) {
    const int ch = tile / tiles_per_ch, y0 = (tile % tiles_per_ch) * R, y = y0 + g;
    const size_t row = (size_t(ch) * A.ny + y) * NX;
    float2 v[F::H][16];
    if constexpr (MODE == 0) {
      const float2* in = (env ? A.eh : A.e0) + row;
#pragma unroll
      for (int h = 0; h < F::H; ++h)
#pragma unroll
        for (int k = 0; k < 16; ++k) v[h][k] = in[F::pos(t, 16 * h + k)];
      if (threadIdx.x == 0) bulk_wait_read_all();  // the last tile's stores have read xreg
      __syncthreads();
    } else {
      if (!__syncthreads_and(mbar_wait(bar, phase))) {
        if (threadIdx.x == 0) {
          atomicExch(status, kStatusTmaTimeout);
          mbar_wait(bar, phase);  // the tile still in flight, bounded
          bulk_wait_all();
        }
        return;
      }
      phase ^= 1u;
#pragma unroll
      for (int q = 0; q < F::E; ++q)
        v[F::elem(q) / 16][F::elem(q) % 16] =
            *reinterpret_cast<const float2*>(stage + mine + q * L::kStep);
      if (threadIdx.x == 0) bulk_wait_read_all();  // the last tile's stores have read xreg
      __syncthreads();  // every read of the stage is done; xreg is free
      if (threadIdx.x == 0 && tile + int(gridDim.x) < n_tiles) {
        fence_proxy_async_smem();
        issue(tile + gridDim.x);
      }
      F::template inv_head<kRowPacked>(v, buf, A.twx, t, g);
      // the row's deformation factor, loaded under the last stage (zero outside
      // the row's crystal extent, where the coupling is the identity): each lane
      // of a pair has the values of one half of the elements
      const float2* crow = A.cfield + (size_t(A.z) * A.ny + y) * NX;
      asm volatile("" : "+l"(crow));  // not before the exchange
      const int2 sp = __ldg(A.cspan + size_t(A.z) * A.ny + y);
      float2 cv[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int x = F::pos(t, 16 * (F::H == 2 ? env : 0) + k);
        cv[k] = (x >= sp.x && x < sp.y) ? __ldg(crow + x) : make_float2(0.f, 0.f);
      }
      F::template inv_tail<kRowPacked>(v, A.twx, t);
      const HalfCoef hc = half_coef(A.coef[ch], env);
      // first cell of the warp's run of 16 (times H) cells of value k
      const int xw = (t & ~15);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int xk = xw + (NX / 16) * k;
        if (xk >= sp.y || xk + 16 * F::H <= sp.x) continue;  // the same for the whole warp
#pragma unroll
        for (int h = 0; h < F::H; ++h) {
          const float2 c = F::H == 2 ? shfl2(cv[k], (lane & ~1) | h) : cv[k];
          const float2 o = shfl2(v[h][k], lane ^ 1);
          if (c.x != 0.f || c.y != 0.f) v[h][k] = half_cell(v[h][k], o, c, hc, env);
        }
      }
    }
    if constexpr (MODE == 2) {
      float2* out = (env ? A.eh : A.e0) + row;
#pragma unroll
      for (int h = 0; h < F::H; ++h)
#pragma unroll
        for (int k = 0; k < 16; ++k) out[F::pos(t, 16 * h + k)] = v[h][k];
    } else {
      // (the pointer hidden from the compiler, which would keep the inverse's 30
      // twiddles in registers across the coupling for the forward transform)
      const float2* tw = A.twx;
      asm volatile("" : "+l"(tw));
      F::template fwd<kRowPacked>(v, buf, tw, t, g);
      __syncthreads();  // every row is done with its exchange region
#pragma unroll
      for (int q = 0; q < F::E; ++q)
        *reinterpret_cast<float2*>(xreg + mine + q * L::kStep) =
            v[F::elem(q) / 16][F::elem(q) % 16];
      fence_proxy_async_smem();  // this thread's writes, before the copy engine reads them
      __syncthreads();
      if (threadIdx.x == 0) {
#pragma unroll
        for (int b = 0; b < L::kBoxes; ++b)
          tma_store_2d(&map, 4 * y0, ch * NX + b * 256, xreg + b * 256 * L::kSeg);
        bulk_commit();
      }
    }
  }
  if (MODE != 2 && threadIdx.x == 0) bulk_wait_all();
}

// cuTensorMapEncodeTiled, fetched from the driver through the runtime (no
// link-time dependency on the driver library).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  static const EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return EncodeTiledFn(nullptr);
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

// Tensor map of the spectrum [n_ch * NX][ny] pairs as FP32 quadruples, boxes of
// the row pass's tile.
template <int NX, int R>
bool encode_row_map(CUtensorMap* m, float2* base, int ny, int n_ch) {
  const EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[2] = {cuuint64_t(4) * ny, cuuint64_t(NX) * n_ch};
  const cuuint64_t strides[1] = {cuuint64_t(ny) * 16};
  const cuuint32_t box[2] = {cuuint32_t(4 * R), 256};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE,
            R == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int NX, int R>
cudaError_t row_launch(int mode, const Pass3DArgs& a, int n_ch, int sms, int* status,
                       cudaStream_t s) {
  using L = RowStream<NX, R>;
  if (a.ny % R != 0) return cudaErrorInvalidValue;
  CUtensorMap m;
  if (!encode_row_map<NX, R>(&m, a.s0, a.ny, n_ch)) return cudaErrorInvalidValue;
  const long long tiles = (long long)n_ch * (a.ny / R), cap = (long long)sms * L::kBlocksPerSm;
  const int blocks = int(tiles < cap ? tiles : cap);
  if (blocks == 0) return cudaSuccess;
  auto* kernel = mode == 0   ? row_stream_kernel<NX, R, 0>
                 : mode == 1 ? row_stream_kernel<NX, R, 1>
                             : row_stream_kernel<NX, R, 2>;
  return launch_pass(kernel, blocks, L::kBlock, L::kSmem, mode != 0, s, m, a, n_ch, status);
}

template <int NY>
cudaError_t col_launch(const Pass3DArgs& a, int n_ch, int sms, int* status, cudaStream_t s) {
  using C = ColStream<NY>;
  const long long need = ((long long)n_ch * a.nx + C::G - 1) / C::G;
  const long long cap = (long long)sms * C::kBlocksPerSm;
  return launch_pass(col_stream_kernel<NY>, int(need < cap ? need : cap), C::kBlock, C::kSmem, true, s,
                     a, n_ch, status);
}

template <int NX, int R>
cudaError_t row_attr() {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int smem = int(RowStream<NX, R>::kSmem);
  cudaError_t r[] = {cudaFuncSetAttribute(row_stream_kernel<NX, R, 0>, attr, smem),
                     cudaFuncSetAttribute(row_stream_kernel<NX, R, 1>, attr, smem),
                     cudaFuncSetAttribute(row_stream_kernel<NX, R, 2>, attr, smem)};
  for (cudaError_t e : r)
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

template <int NY>
cudaError_t col_attr() {
  return cudaFuncSetAttribute(col_stream_kernel<NY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              int(ColStream<NY>::kSmem));
}

}  // namespace

cudaError_t stream3d_set_attributes() {
  cudaError_t r[] = {row_attr<256, 8>(), row_attr<512, 4>(), row_attr<512, 8>(), row_attr<1024, 4>(),
                     col_attr<256>(),    col_attr<512>(),    col_attr<1024>()};
  for (cudaError_t e : r)
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

bool row_stream_supported(int nx, int row_threads) {
  return (nx == 256 && row_threads == 128) || (nx == 512 && (row_threads == 128 || row_threads == 256)) ||
         (nx == 1024 && row_threads == 256);
}

cudaError_t launch_row_stream(int mode, int row_threads, const Pass3DArgs& a, int n_ch, int sms,
                              int* status, cudaStream_t s) {
  if (a.nx == 256 && row_threads == 128) return row_launch<256, 8>(mode, a, n_ch, sms, status, s);
  if (a.nx == 512 && row_threads == 128) return row_launch<512, 4>(mode, a, n_ch, sms, status, s);
  if (a.nx == 512 && row_threads == 256) return row_launch<512, 8>(mode, a, n_ch, sms, status, s);
  if (a.nx == 1024 && row_threads == 256) return row_launch<1024, 4>(mode, a, n_ch, sms, status, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_col_stream(const Pass3DArgs& a, int n_ch, int sms, int* status, cudaStream_t s) {
  if (a.ny == 256) return col_launch<256>(a, n_ch, sms, status, s);
  if (a.ny == 512) return col_launch<512>(a, n_ch, sms, status, s);
  if (a.ny == 1024) return col_launch<1024>(a, n_ch, sms, status, s);
  return cudaErrorInvalidValue;
}

}  // namespace bpm
