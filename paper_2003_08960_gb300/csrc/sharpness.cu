// Aberration correction: the reconstruction with a Zernike phase screen in the
// sensor plane, the sharpness of its intensity volume and the gradient of that
// sharpness with respect to the reconstruction distance z and the coefficients
// c_1..c_15, by one hand-written adjoint pass.
//
// Forward (the chain of Eq. 5 - Eq. 7 with the screen P = exp(i sum_j c_j Z_j)
// multiplied into the input chirp c of Eq. 6):
//   rows    u_t = Eq. 5 resample of frame t;  row DFT (+) of c P u_t      -> F[t][y][x]
//   columns column DFT (+), window crop                                  -> sweep-axis intermediate
//   axial   Eq. 7 over t, P_v = |K|^2 |V~_v|^2                            -> volume
//   sums    S1 = sum P_v, S2 = sum P_v^2 (expansions of floats, FP64 between blocks); L = -S2 / S1^2
// Adjoint (W = 2 |K|^2 dL/dP V~, dL/dP = -2 P / S1^2 + 2 S2 / S1^3):
//   axial   V~ recomputed, W formed, sum_q W_q exp(+2 pi i q t / N)      -> intermediate (in place)
//   columns zero outside the window, column DFT (-)                      -> F[t][y][x]
//   rows    row DFT (-) = Y_t; Q = sum_t conj(Y_t) u_t with u_t recomputed from the uint16 frames
//   grad    M = -Im(c P Q); dL/dc_j = sum Z_j M; dL/dz = (pi |K| / z) sum r_pix^2 M
// The DFTs here are the uncentred ones of the lateral kernel, with the centring
// phase (-1)^n folded into c; the unit-modulus factors this moves onto V~ cancel
// in W's round trip, so M is the same as with the centred transform.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "adjoint_share.h"
#include "fft_common.cuh"
#include "float_sums.cuh"
#include "mbarrier.cuh"
#include "pupil_turn.cuh"

namespace ssoct {
namespace {

constexpr int kRowThreads = 256;
constexpr int kGradThreads = 256;

// Split N = N1 x N2 of one axis for these kernels: stage 1 is N2-point DFTs in
// the N1 threads of a transform, stage 2 the N2 N1-point DFTs spread over those
// threads, NI per thread (the last ones idle when N1 does not divide N2, e.g.
// 640 = 32 x 20).  AS is the register array length, TW the width of a column
// tile (16 when 32 N1 threads would exceed 256: at 85 to 128 registers a thread,
// two or more blocks per SM overlap their loads; loss and gradient at 640 x 384 x
// 64 446 -> 420 us against tiles of 32, 384 x 384 x 96 380 -> 365).
template <int N>
struct Lat {
  static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2;
  static constexpr int NI = (N2 + N1 - 1) / N1;
  static constexpr int AS = NI * N1 > N2 ? NI * N1 : N2;
};
// Column-tile width for axis length N (a variable template, instantiated only
// for the column kernels that use it).
template <int N>
constexpr int kLatTW = kTile * Split<N>::N1 <= 256 ? kTile : kTile / 2;

__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }


// Row DFT of sign S over the registers of thread (r, j1) of an N1 x N2 split:
// on entry a[j2] = x[j1 + N1 j2]; on exit a[i N1 + k1] = X[k2 + N2 k1] with
// k2 = j1 + N1 i for the i with k2 < N2.  ex is this row's padded exchange
// block; a row's N1 threads lie in one warp.
template <int N, int S>
__device__ __forceinline__ void row_dft(float2 (&a)[Lat<N>::AS], const float2* tw, float2* ex, int j1) {
  constexpr int N1 = Lat<N>::N1, N2 = Lat<N>::N2, NI = Lat<N>::NI;
  Dft<N2, S>::template run<1, 0>(a);
#pragma unroll
  for (int k2 = 0; k2 < N2; ++k2) {
    const float2 w = ldg2(tw + k2 * N1 + j1);
    a[k2] = cmul(a[k2], S > 0 ? w : conjf2(w));
  }
  __syncwarp();
#pragma unroll
  for (int k2 = 0; k2 < N2; ++k2) ex[k2 * (N1 + 1) + j1] = a[k2];
  __syncwarp();
  static_for<0, NI>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
    if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
      for (int jj = 0; jj < N1; ++jj) a[i * N1 + jj] = ex[k2 * (N1 + 1) + jj];
      Dft<N1, S>::template run<1, i * N1>(a);
    }
  });
}

// Column DFT of sign S over 32-wide tiles: thread (pix, j1), a[j2] = x[j1 + N1 j2]
// on entry, a[i N1 + k1] = X[k2 + N2 k1] (k2 = j1 + N1 i) on exit.  tw holds the
// twiddles of sign TS (conjugated when S differs).
template <int N, int S, int TS, int TW>
__device__ __forceinline__ void col_dft(float2 (&a)[Lat<N>::AS], const float2* tw, float2* ex, int j1, int pix) {
  constexpr int N1 = Lat<N>::N1, N2 = Lat<N>::N2, NI = Lat<N>::NI;
  Dft<N2, S>::template run<1, 0>(a);
#pragma unroll
  for (int k2 = 0; k2 < N2; ++k2) {
    const float2 w = ldg2(tw + k2 * N1 + j1);
    a[k2] = cmul(a[k2], S == TS ? w : conjf2(w));
  }
  __syncthreads();
#pragma unroll
  for (int k2 = 0; k2 < N2; ++k2) ex[(k2 * N1 + j1) * TW + pix] = a[k2];
  __syncthreads();
  static_for<0, NI>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
    if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
      for (int jj = 0; jj < N1; ++jj) a[i * N1 + jj] = ex[(k2 * N1 + jj) * TW + pix];
      Dft<N1, S>::template run<1, i * N1>(a);
    }
  });
}

struct ShParams {
  const uint16_t* frames;  // [nl][ny][nx]
  const Tap* xtab;         // [nl][nx]
  const Tap* ytab;         // [nl][ny]
  const float2* cp;        // [ny][nx] input chirp (with centring) x pupil screen
  const float2* twx;       // [N2x][N1x], sign +
  const float2* twy;       // [N2y][N1y], sign +
  const float2* twl;       // [N2l][N1l], sign -
  float2* F;               // [nl][ny][nx] lateral work frames
  float2* inter;           // [wy][ntx][nl][32] sweep-axis intermediate
  float2* qpart;           // [chunks][ny][nx] partial Q, tpc frames each
  const float* vol;        // [nl][wy][wx] P_v
  double* red;             // [0] S1, [1] S2, [2..18] loss, dL/dz, dL/dc_1..15, [19] float a1, a0, [20] block count, [21] error word
  float sum_scale;         // power of two that keeps the squares of P_v in the float range
  int nx, ny, nl, x0, y0, wx, wy, ntx, tpc;
  int ring_start;          // frame t of the gate is frames[(ring_start + t) mod nl]
  float alpha2;            // |K|^2
  double scale_z;          // pi |K| / z
};

// ----------------------------------------------------------------- forward

template <int NX>
__global__ void __launch_bounds__(kRowThreads) rows_fwd_kernel(const __grid_constant__ ShParams p) {
  after_previous_kernel();
  constexpr int N1 = Lat<NX>::N1, N2 = Lat<NX>::N2, RPI = kRowThreads / N1;
  extern __shared__ __align__(16) unsigned char smem[];
  const int r = threadIdx.x / N1, j1 = threadIdx.x % N1;
  const int y = blockIdx.x * RPI + r, t = blockIdx.y;
  float2* ex = reinterpret_cast<float2*>(smem) + r * N2 * (N1 + 1);
  const uint16_t* fr = p.frames + (size_t)((p.ring_start + t) % p.nl) * p.ny * NX;
  const Tap ty = p.ytab[(size_t)t * p.ny + y];
  const float2* cp = p.cp + (size_t)y * NX;
  float2 a[Lat<NX>::AS];
#pragma unroll
  for (int j2 = 0; j2 < N2; ++j2) {
    const int n = j1 + N1 * j2;
    const float u = rescale_tap_value(fr, NX, p.xtab[(size_t)t * NX + n], ty);
    const float2 c = cp[n];
    a[j2] = make_float2(u * c.x, u * c.y);
  }
  row_dft<NX, 1>(a, p.twx, ex, j1);
  float2* dst = p.F + ((size_t)t * p.ny + y) * NX;
  static_for<0, Lat<NX>::NI>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
    if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) dst[k2 + N2 * k1] = a[i * N1 + k1];
    }
  });
}

template <int NY>
__global__ void __launch_bounds__(kLatTW<NY> * Lat<NY>::N1) cols_fwd_kernel(const __grid_constant__ ShParams p) {
  after_previous_kernel();
  constexpr int N1 = Lat<NY>::N1, N2 = Lat<NY>::N2, TW = kLatTW<NY>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int pix = threadIdx.x % TW, j1 = threadIdx.x / TW;
  const int x = blockIdx.x * TW + pix, t = blockIdx.y;
  const float2* src = p.F + (size_t)t * NY * p.nx + x;
  float2 a[Lat<NY>::AS];
#pragma unroll
  for (int j2 = 0; j2 < N2; ++j2) a[j2] = src[(size_t)(j1 + N1 * j2) * p.nx];
  col_dft<NY, 1, 1, TW>(a, p.twy, reinterpret_cast<float2*>(smem), j1, pix);
  const int kxw = x - p.x0;
  if (kxw < 0 || kxw >= p.wx) return;
  float2* dst = p.inter + ((size_t)(kxw / kTile) * p.nl + t) * kTile + kxw % kTile;
  const size_t row_pitch = (size_t)p.ntx * p.nl * kTile;
  static_for<0, Lat<NY>::NI>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
    if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) {
        const int kyw = k2 + N2 * k1 - p.y0;
        if (kyw >= 0 && kyw < p.wy) dst[(size_t)kyw * row_pitch] = a[i * N1 + k1];
      }
    }
  });
}

// S1 = sum P, S2 = sum P^2 over the volume, and from them the loss and the two
// coefficients of dL/dP = a1 P + a0.  A pass over the volume should be bound by
// its reads (20 us for 512 x 512 x 128); two FP64 operations and a conversion
// per voxel at two FP64 operations per clock and SM took 240.  Each thread sums in
// expansions of floats instead (FloatSums), which meet in FP64, and the last block
// adds the blocks' sums in a fixed order: 42 us.  Relative error of the loss against
// exact sums of the volume at eight sizes, three scenes each: 8e-16 at most, the
// FP64 sums' 3e-15 (their blocks met by atomics); pairs of floats, 9e-15, took 33 us.
// P is scaled by a power of two so that no square leaves the float range.
__global__ void __launch_bounds__(kGradThreads) sums_kernel(const __grid_constant__ ShParams p, size_t n) {
  after_previous_kernel();
  FloatSums sum = {};
  const float k = p.sum_scale;
  const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  const float4* v4 = reinterpret_cast<const float4*>(p.vol);  // the volume is 16-byte aligned
  const size_t n4 = n / 4;
#pragma unroll 4
  for (size_t i = first; i < n4; i += stride) {
    const float4 v = __ldcs(v4 + i);
    sum.add4(v.x * k, v.y * k, v.z * k, v.w * k);
  }
  for (size_t i = n4 * 4 + first; i < n; i += stride) sum.add4(p.vol[i] * k, 0.f, 0.f, 0.f);
  for (int o = 16; o; o >>= 1) {
    auto other = [&](const FloatSum& f) {
      return FloatSum{__shfl_xor_sync(0xffffffffu, f.h, o), __shfl_xor_sync(0xffffffffu, f.l, o),
                      __shfl_xor_sync(0xffffffffu, f.m, o)};
    };
    sum.p.add(other(sum.p));
    sum.q.add(other(sum.q));
  }
  __shared__ double2 sh[kGradThreads / 32];
  __shared__ bool last;
  if (threadIdx.x % 32 == 0) sh[threadIdx.x / 32] = make_double2(sum.p.value(), sum.q.value());
  __syncthreads();
  // the blocks' sums, in the memory of Q's partial sums (not in use before the adjoint row pass)
  double2* const blocks = reinterpret_cast<double2*>(p.qpart);
  if (threadIdx.x == 0) {
    double2 t = make_double2(0.0, 0.0);
    for (int w = 0; w < kGradThreads / 32; ++w) {
      t.x += sh[w].x;
      t.y += sh[w].y;
    }
    __stcg(blocks + blockIdx.x, t);
    __threadfence();
    // the last block to get here sees every sum
    last = atomicAdd(reinterpret_cast<unsigned*>(p.red + 20), 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  double2 t = make_double2(0.0, 0.0);
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kGradThreads) {
    const double2 v = __ldcg(blocks + b);
    t.x += v.x;
    t.y += v.y;
  }
  for (int o = 16; o; o >>= 1) {
    t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
    t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
  }
  __syncthreads();
  if (threadIdx.x % 32 == 0) sh[threadIdx.x / 32] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    t = sh[0];
    for (int w = 1; w < kGradThreads / 32; ++w) {
      t.x += sh[w].x;
      t.y += sh[w].y;
    }
    const double inv = 1.0 / (double)k;  // a power of two: exact
    const double t1 = t.x * inv, t2 = t.y * inv * inv;
    p.red[0] = t1;
    p.red[1] = t2;
    float* c = reinterpret_cast<float*>(p.red + 19);
    c[0] = (float)(-2.0 / (t1 * t1));
    c[1] = (float)(2.0 * t2 / (t1 * t1 * t1));
    p.red[2] = -t2 / (t1 * t1);
  }
}

// ----------------------------------------------------------------- adjoint

template <int NL>
__global__ void __launch_bounds__(kTile * Split<NL>::N1) axial_adj_kernel(const __grid_constant__ ShParams p) {
  after_previous_kernel();
  constexpr int N1 = Split<NL>::N1, N2 = Split<NL>::N2;
  static_assert(N2 % N1 == 0, "sweep lengths split with N1 | N2");
  extern __shared__ __align__(16) unsigned char smem[];
  float2* ex = reinterpret_cast<float2*>(smem);
  const int pix = threadIdx.x % kTile, j1 = threadIdx.x / kTile;
  float2* g = p.inter + ((size_t)blockIdx.y * p.ntx + blockIdx.x) * NL * kTile + pix;
  // dL/dP = a1 P + a0, formed once by sums_kernel: the two FP64 divisions in
  // every thread here took most of this kernel (115 us at 512 x 512 x 128)
  const float a1 = reinterpret_cast<const float*>(p.red + 19)[0], a0 = reinterpret_cast<const float*>(p.red + 19)[1];
  float2 a[N2];
#pragma unroll
  for (int j2 = 0; j2 < N2; ++j2) a[j2] = g[(j1 + N1 * j2) * kTile];
  col_dft<NL, -1, -1, kTile>(a, p.twl, ex, j1, pix);  // V~[q = k2 + N2 k1]
  __syncthreads();
  static_for<0, N2 / N1>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
      const float2 v = a[i * N1 + k1];
      const float pw = p.alpha2 * fmaf(v.x, v.x, v.y * v.y);
      const float s = 2.f * p.alpha2 * fmaf(a1, pw, a0);
      ex[(k2 + N2 * k1) * kTile + pix] = make_float2(s * v.x, s * v.y);  // W in natural order
    }
  });
  __syncthreads();
#pragma unroll
  for (int j2 = 0; j2 < N2; ++j2) a[j2] = ex[(j1 + N1 * j2) * kTile + pix];
  // sum_q W_q exp(+2 pi i q t / NL): the same split with the conjugate twiddles
  col_dft<NL, 1, -1, kTile>(a, p.twl, ex, j1, pix);
  static_for<0, N2 / N1>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) g[(k2 + N2 * k1) * kTile] = a[i * N1 + k1];
  });
}

template <int NY>
__global__ void __launch_bounds__(kLatTW<NY> * Lat<NY>::N1) cols_adj_kernel(const __grid_constant__ ShParams p) {
  after_previous_kernel();
  constexpr int N1 = Lat<NY>::N1, N2 = Lat<NY>::N2, TW = kLatTW<NY>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int pix = threadIdx.x % TW, j1 = threadIdx.x / TW;
  const int x = blockIdx.x * TW + pix, t = blockIdx.y;
  const int kxw = x - p.x0;
  const bool inx = kxw >= 0 && kxw < p.wx;
  const float2* src = p.inter + ((size_t)(inx ? kxw / kTile : 0) * p.nl + t) * kTile + (inx ? kxw % kTile : 0);
  const size_t row_pitch = (size_t)p.ntx * p.nl * kTile;
  float2 a[Lat<NY>::AS];
#pragma unroll
  for (int j2 = 0; j2 < N2; ++j2) {
    const int kyw = j1 + N1 * j2 - p.y0;
    a[j2] = (inx && kyw >= 0 && kyw < p.wy) ? src[(size_t)kyw * row_pitch] : make_float2(0.f, 0.f);
  }
  // the adjoint of the forward column DFT (+) is the column DFT (-), with the forward table conjugated
  col_dft<NY, -1, 1, TW>(a, p.twy, reinterpret_cast<float2*>(smem), j1, pix);
  float2* dst = p.F + (size_t)t * NY * p.nx + x;
  static_for<0, Lat<NY>::NI>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
    if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) dst[(size_t)(k2 + N2 * k1) * p.nx] = a[i * N1 + k1];
    }
  });
}

template <int NX>
__global__ void __launch_bounds__(kRowThreads) rows_adj_kernel(const __grid_constant__ ShParams p) {
  after_previous_kernel();
  constexpr int N1 = Lat<NX>::N1, N2 = Lat<NX>::N2, RPI = kRowThreads / N1, AS = Lat<NX>::AS;
  extern __shared__ __align__(16) unsigned char smem[];
  const int r = threadIdx.x / N1, j1 = threadIdx.x % N1;
  const int y = blockIdx.x * RPI + r, chunk = blockIdx.y;
  float2* ex = reinterpret_cast<float2*>(smem) + r * N2 * (N1 + 1);
  const int t0 = chunk * p.tpc, t1 = min(p.nl, t0 + p.tpc);
  float2 acc[AS];
#pragma unroll
  for (int i = 0; i < AS; ++i) acc[i] = make_float2(0.f, 0.f);
  for (int t = t0; t < t1; ++t) {
    const float2* src = p.F + ((size_t)t * p.ny + y) * NX;
    float2 a[AS];
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) a[j2] = src[j1 + N1 * j2];
    row_dft<NX, -1>(a, p.twx, ex, j1);
    const uint16_t* fr = p.frames + (size_t)((p.ring_start + t) % p.nl) * p.ny * NX;
    const Tap ty = p.ytab[(size_t)t * p.ny + y];
    const Tap* xt = p.xtab + (size_t)t * NX;
    static_for<0, Lat<NX>::NI>([&](auto I) {
      constexpr int i = decltype(I)::value;
      const int k2 = j1 + N1 * i;
      if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
          const float u = rescale_tap_value(fr, NX, xt[k2 + N2 * k1], ty);
          const float2 v = a[i * N1 + k1];
          acc[i * N1 + k1].x = fmaf(v.x, u, acc[i * N1 + k1].x);   // conj(Y) u
          acc[i * N1 + k1].y = fmaf(-v.y, u, acc[i * N1 + k1].y);
        }
      }
    });
  }
  float2* dst = p.qpart + ((size_t)chunk * p.ny + y) * NX;
  static_for<0, Lat<NX>::NI>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1 * i;
    if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) dst[k2 + N2 * k1] = acc[i * N1 + k1];
    }
  });
}

}  // namespace

namespace {

// The same row pass, streamed: one CTA per SM takes an equal, contiguous share of
// the (band of rows, frame) pairs, band by band, and its inputs (the band's rows of
// F, the raw frame rows and the taps of Eq. 5) arrive by bulk copies into two stage
// buffers, one pair ahead.  rows_adj_kernel's accumulators leave room for eight
// warps per SM, which wait for each of these loads in turn.  The exchange is done
// in place in the stage buffer.  Partial sums are those of rows_adj_kernel, eight
// frames in FP32 (see RowsAdjShare).  One per CTA and band instead, 27 to 432 frames
// in one FP32 sum, took 716 us where this took 728 (loss and gradient at 512 x 512 x
// 128), 1298 for 1346 at 1024 x 1024 x 64, 449 for 460 at 256 x 256 x 256; parts of 16
// frames in pairs of floats 730 and 1366 in the first two; rows_adj_kernel 762, 1404
// and 488 (each with the other kernels of its time).  Column and row passes in turn over chunks of frames whose F stays in
// L2 were slower (16 to 96 MiB: 724 to 767 us at 512 x 512 x 128).
template <int NX>
struct RowsAdjStage {
  static constexpr int RPI = kRowThreads / Lat<NX>::N1;
  static constexpr size_t kRows = (size_t)RPI * NX * sizeof(float2);  // then the raw rows, x taps, y taps
  __host__ __device__ static size_t taps_at(int raw_rows) { return kRows + (size_t)raw_rows * NX * sizeof(uint16_t); }
  __host__ __device__ static size_t bytes(int raw_rows) { return taps_at(raw_rows) + NX * sizeof(Tap) + RPI * sizeof(Tap); }
};

constexpr unsigned long long kAdjWaitNs = 4000000000ull;  // 4 s

// Zeroes the slots that two CTAs of rows_adj_stream_kernel add to, 64 KB each at
// most, one a block.  A kernel of its own (4 us): in the column pass it cost 16 us at
// 512 x 512 x 128 and 8 at 1024 x 1024 x 64, beside the sums 32 at the latter.
__global__ void __launch_bounds__(kRowThreads) zero_split_kernel(const __grid_constant__ ShParams p, RowsAdjShare share) {
  after_previous_kernel();
  const int c = blockIdx.x + 1;
  if (!share.splits(c)) return;
  const int i = share.first(c), band_px = p.ny / share.bands * p.nx;
  float4* q = reinterpret_cast<float4*>(p.qpart + (size_t)share.slot(i) * p.ny * p.nx + (size_t)share.band(i) * band_px);
  for (int k = threadIdx.x; k < band_px / 2; k += kRowThreads) q[k] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <int NX>
__global__ void __launch_bounds__(kRowThreads, 1)
    rows_adj_stream_kernel(const __grid_constant__ ShParams p, RowsAdjShare share, int raw_rows, unsigned* err) {
  after_previous_kernel();
  using St = RowsAdjStage<NX>;
  constexpr int N1 = Lat<NX>::N1, N2 = Lat<NX>::N2, NI = Lat<NX>::NI, RPI = St::RPI, AS = Lat<NX>::AS;
  static_assert(32 % N1 == 0, "a row's N1 threads lie in one warp");
  extern __shared__ __align__(1024) unsigned char smem_adj[];
  __shared__ __align__(8) uint64_t full[2];
  const int tid = threadIdx.x;
  const int r = tid / N1, j1 = tid % N1;
  const size_t stage_bytes = (St::bytes(raw_rows) + 127) / 128 * 128;
  const size_t taps_at = St::taps_at(raw_rows);
  const int lo = share.first(blockIdx.x), hi = share.first(blockIdx.x + 1);
  // pair i into stage buffer (i - lo) mod 2, by one thread
  auto fill = [&](int i) {
    const int band = i / share.nt, t = i - band * share.nt;
    unsigned char* buf = smem_adj + (size_t)((i - lo) & 1) * stage_bytes;
    uint64_t* bar = &full[(i - lo) & 1];
    const Tap* yt = p.ytab + (size_t)t * p.ny + band * RPI;
    const int first = yt[0].base, rows = yt[RPI - 1].base + 2 - first;  // at most raw_rows
    const unsigned raw = (unsigned)(rows * NX * sizeof(uint16_t));
    mbar_arrive_tx(bar, (unsigned)St::kRows + raw + (unsigned)((NX + RPI) * sizeof(Tap)));
    tma_load_1d(buf, p.F + ((size_t)t * p.ny + band * RPI) * NX, (unsigned)St::kRows, bar);
    tma_load_1d(buf + St::kRows, p.frames + ((size_t)((p.ring_start + t) % p.nl) * p.ny + first) * NX, raw, bar);
    tma_load_1d(buf + taps_at, p.xtab + (size_t)t * NX, (unsigned)(NX * sizeof(Tap)), bar);
    tma_load_1d(buf + taps_at + NX * sizeof(Tap), yt, (unsigned)(RPI * sizeof(Tap)), bar);
  };
  // bounded wait for the CTA's k-th pair
  auto arrived = [&](int k) {
    uint64_t* bar = &full[k & 1];
    const unsigned parity = (unsigned)(k / 2) & 1u;
    if (mbar_try(bar, parity)) return true;
    const unsigned long long since = global_timer_ns();
    while (!mbar_try(bar, parity))
      if (global_timer_ns() - since > kAdjWaitNs) return false;
    return true;
  };
  if (tid == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = lo; i < hi && i < lo + 2; ++i) fill(i);
  }
  __syncthreads();
  float2 acc[AS];
#pragma unroll
  for (int i = 0; i < AS; ++i) acc[i] = make_float2(0.f, 0.f);
  for (int i = lo; i < hi; ++i) {
    const int k = i - lo;
    const bool ok = arrived(k);
    if (__syncthreads_or(!ok)) {
      // the copies never came: the sums are incomplete, and reported so; what is
      // still in flight lands before the CTA exits
      if (tid == 0) {
        atomicOr(err, kErrAdjoint);
        arrived(k);
        if (i + 1 < hi) arrived(k + 1);
      }
      return;
    }
    unsigned char* buf = smem_adj + (size_t)(k & 1) * stage_bytes;
    float2* row = reinterpret_cast<float2*>(buf) + r * NX;
    const uint16_t* raw = reinterpret_cast<const uint16_t*>(buf + St::kRows);
    const Tap* xt = reinterpret_cast<const Tap*>(buf + taps_at);
    float2 a[AS];
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) a[j2] = row[j1 + N1 * j2];
    Dft<N2, -1>::template run<1, 0>(a);
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) a[k2] = cmul(a[k2], conjf2(ldg2(p.twx + k2 * N1 + j1)));
    __syncwarp();  // the row's values have been read
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) row[k2 * N1 + (j1 ^ (k2 & (N1 - 1)))] = a[k2];
    __syncwarp();
    const Tap ty = xt[NX + r];
    const uint16_t* r0 = raw + (ty.base - xt[NX].base) * NX;
    static_for<0, NI>([&](auto I) {
      constexpr int ii = decltype(I)::value;
      const int k2 = j1 + N1 * ii;
      if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
        for (int jj = 0; jj < N1; ++jj) a[ii * N1 + jj] = row[k2 * N1 + (jj ^ (k2 & (N1 - 1)))];
        Dft<N1, -1>::template run<1, ii * N1>(a);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
          const Tap tx = xt[k2 + N2 * k1];
          const uint16_t* c = r0 + tx.base;
          const float v0 = fmaf(tx.w0, (float)c[0], tx.w1 * (float)c[1]);
          const float v1 = fmaf(tx.w0, (float)c[NX], tx.w1 * (float)c[NX + 1]);
          const float u = fmaf(ty.w0, v0, ty.w1 * v1);
          const float2 v = a[ii * N1 + k1];
          acc[ii * N1 + k1].x = fmaf(v.x, u, acc[ii * N1 + k1].x);   // conj(Y) u
          acc[ii * N1 + k1].y = fmaf(-v.y, u, acc[ii * N1 + k1].y);
        }
      }
    });
    // this thread's accesses to the buffer come before its next fill (async proxy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0 && i + 2 < hi) fill(i + 2);
    if (share.closes(i, hi)) {
      const bool whole = share.whole(i, lo, hi);
      float2* dst = p.qpart + ((size_t)share.slot(i) * p.ny + share.band(i) * RPI + r) * NX;
      static_for<0, NI>([&](auto I) {
        constexpr int ii = decltype(I)::value;
        const int k2 = j1 + N1 * ii;
        if (N2 % N1 == 0 || k2 < N2) {
#pragma unroll
          for (int k1 = 0; k1 < N1; ++k1) {
            float2* d = dst + k2 + N2 * k1;
            const float2 q = acc[ii * N1 + k1];
            if (whole) {
              *d = q;
            } else {
              atomicAdd(&d->x, q.x);
              atomicAdd(&d->y, q.y);
            }
            acc[ii * N1 + k1] = make_float2(0.f, 0.f);
          }
        }
      });
    }
  }
}

}  // namespace

// Z_1..Z_15 (Noll order, RMS-normalised on the unit disk; Noll 1976) at radius
// rho and angle (cos th, sin th).
__host__ __device__ __forceinline__ void zernike15(double rho, double c1, double s1, double (&z)[15]) {
  const double r2 = rho * rho, r3 = r2 * rho, r4 = r2 * r2;
  const double c2 = c1 * c1 - s1 * s1, s2 = 2.0 * s1 * c1;
  const double c3 = c2 * c1 - s2 * s1, s3 = s2 * c1 + c2 * s1;
  const double c4 = c2 * c2 - s2 * s2, s4 = 2.0 * s2 * c2;
  const double q3 = 1.7320508075688772935, q5 = 2.2360679774997896964, q6 = 2.4494897427831780982,
               q8 = 2.8284271247461900976, q10 = 3.1622776601683793320;
  z[0] = 1.0;
  z[1] = 2.0 * rho * c1;
  z[2] = 2.0 * rho * s1;
  z[3] = q3 * (2.0 * r2 - 1.0);
  z[4] = q6 * r2 * s2;
  z[5] = q6 * r2 * c2;
  z[6] = q8 * (3.0 * r3 - 2.0 * rho) * s1;
  z[7] = q8 * (3.0 * r3 - 2.0 * rho) * c1;
  z[8] = q8 * r3 * s3;
  z[9] = q8 * r3 * c3;
  z[10] = q5 * (6.0 * r4 - 6.0 * r2 + 1.0);
  z[11] = q10 * (4.0 * r4 - 3.0 * r2) * c2;
  z[12] = q10 * (4.0 * r4 - 3.0 * r2) * s2;
  z[13] = q10 * r4 * c4;
  z[14] = q10 * r4 * s4;
}

// The same polynomials in the monomials X^a Y^b, a + b <= 4 (X = rho cos, Y =
// rho sin), in the order of mono_a / mono_b: Z_j = sum_i kZernike[j][i] X^a Y^b.
#define SSOCT_ZERNIKE_ROWS \
  {1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0}, \
  {0, 2, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0}, \
  {0, 0, 2, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0}, \
  {-R3, 0, 0, 2 * R3, 0, 2 * R3, 0, 0, 0, 0, 0, 0, 0, 0, 0}, \
  {0, 0, 0, 0, 2 * R6, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0}, \
  {0, 0, 0, R6, 0, -R6, 0, 0, 0, 0, 0, 0, 0, 0, 0}, \
  {0, 0, -2 * R8, 0, 0, 0, 0, 3 * R8, 0, 3 * R8, 0, 0, 0, 0, 0}, \
  {0, -2 * R8, 0, 0, 0, 0, 3 * R8, 0, 3 * R8, 0, 0, 0, 0, 0, 0}, \
  {0, 0, 0, 0, 0, 0, 0, 3 * R8, 0, -R8, 0, 0, 0, 0, 0}, \
  {0, 0, 0, 0, 0, 0, R8, 0, -3 * R8, 0, 0, 0, 0, 0, 0}, \
  {R5, 0, 0, -6 * R5, 0, -6 * R5, 0, 0, 0, 0, 6 * R5, 0, 12 * R5, 0, 6 * R5}, \
  {0, 0, 0, -3 * R10, 0, 3 * R10, 0, 0, 0, 0, 4 * R10, 0, 0, 0, -4 * R10}, \
  {0, 0, 0, 0, -6 * R10, 0, 0, 0, 0, 0, 0, 8 * R10, 0, 8 * R10, 0}, \
  {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, R10, 0, -6 * R10, 0, R10}, \
  {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 4 * R10, 0, -4 * R10, 0}
constexpr double R3 = 1.7320508075688772935, R5 = 2.2360679774997896964, R6 = 2.4494897427831780982,
                 R8 = 2.8284271247461900976, R10 = 3.1622776601683793320;
constexpr int kMono = 15;
static __constant__ double kZernikeDev[15][kMono] = {SSOCT_ZERNIKE_ROWS};
static const double kZernike[15][kMono] = {SSOCT_ZERNIKE_ROWS};
#undef SSOCT_ZERNIKE_ROWS
__host__ __device__ constexpr int mono_a(int i) {  // power of X: 1, X Y, X2 XY Y2, X3 X2Y XY2 Y3, ...
  return i == 0 ? 0 : i < 3 ? 2 - i : i < 6 ? 5 - i : i < 10 ? 9 - i : 14 - i;
}
__host__ __device__ constexpr int mono_b(int i) {
  return i == 0 ? 0 : i < 3 ? i - 1 : i < 6 ? i - 3 : i < 10 ? i - 6 : i - 10;
}

namespace {

// Threads of a block along x in grad_kernel and pupil_table_kernel (nx is a
// multiple of 64).
__host__ __device__ constexpr int grid_tx(int nx) { return nx % 256 == 0 ? 256 : nx % 128 == 0 ? 128 : 64; }

// dL/dz and dL/dc_j: sums over the sensor of M r^2 and M Z_j, M = -Im(c P Q).
// All of them are combinations of the 15 moments sum M X^a Y^b, so a pixel costs
// the moments along y only (five FP64 fused steps); a thread keeps its column x,
// and X^a and the Zernike combinations come in once per thread and per block.
// The chunks of Q are added as pairs of floats (two_sum).  Evaluating the
// polynomials and adding the chunks in FP64 per pixel (two FP64 operations per
// clock and SM) took 98 us at 512 x 512 x 128; 34 us now (with three blocks per SM:
// each thread still ends with some 35 FP64 operations).  The reads of Q alone would
// take 6.
__global__ void __launch_bounds__(kGradThreads) grad_kernel(const __grid_constant__ ShParams p, int chunks,
                                                           const unsigned* queue_err) {
  after_previous_kernel();
  // the call reads one error word back with the loss and gradient
  if (queue_err && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
    atomicOr(reinterpret_cast<unsigned*>(p.red + kShRedErr), *queue_err);
  const int tx = grid_tx(p.nx), ry = kGradThreads / tx;
  const int x = blockIdx.x * tx + threadIdx.x % tx;
  const size_t npix = (size_t)p.nx * p.ny;
  const double inv_radius = 2.0 / (double)min(p.nx, p.ny);  // rho = r_pix / (min(nx, ny) / 2)
  double my[5] = {0.0, 0.0, 0.0, 0.0, 0.0};  // sum_y M Y^b of this column
  for (int y = blockIdx.y * ry + threadIdx.x / tx; y < p.ny; y += gridDim.y * ry) {
    const size_t i = (size_t)y * p.nx + x;
    float qx = 0.f, lx = 0.f, qy = 0.f, ly = 0.f;
#pragma unroll 8
    for (int c = 0; c < chunks; ++c) {
      const float2 q = __ldcs(p.qpart + (size_t)c * npix + i);
      float e;
      qx = two_sum(qx, q.x, e);
      lx += e;
      qy = two_sum(qy, q.y, e);
      ly += e;
    }
    // M = -Im(c P Q), the products and their sum as pairs of floats too
    const float2 cp = p.cp[i];
    const float u = __fmul_rn(cp.x, qy), v = __fmul_rn(cp.y, qx);
    float e;
    const float h = two_sum(u, v, e);
    e += fmaf(cp.x, qy, -u) + fmaf(cp.y, qx, -v) + fmaf(cp.x, ly, cp.y * lx);
    const double m = -((double)h + (double)e);
    const double yy = (double)(y - p.ny / 2) * inv_radius, y2 = yy * yy;
    my[0] += m;
    my[1] = fma(m, yy, my[1]);
    my[2] = fma(m, y2, my[2]);
    my[3] = fma(m, y2 * yy, my[3]);
    my[4] = fma(m, y2 * y2, my[4]);
  }
  const double xx = (double)(x - p.nx / 2) * inv_radius;
  const double xp[5] = {1.0, xx, xx * xx, xx * xx * xx, (xx * xx) * (xx * xx)};
  double mom[16];
#pragma unroll
  for (int i = 0; i < kMono; ++i) mom[i] = mono_a(i) ? my[mono_b(i)] * xp[mono_a(i)] : my[mono_b(i)];
  mom[15] = 0.0;
  // warp sum of the 16 values: each step halves the values a lane holds
  const int lane = threadIdx.x % 32;
#pragma unroll
  for (int h = 8; h; h >>= 1) {
    const bool up = (lane & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double keep = up ? mom[i + h] : mom[i], send = up ? mom[i] : mom[i + h];
      mom[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  // lane l now holds value l % 16, summed over the lanes of its half warp
  double v = mom[0];
  v += __shfl_xor_sync(0xffffffffu, v, 16);
  __shared__ double sh[16][kGradThreads / 32];
  __shared__ double tot[16];
  if (lane < 16) sh[lane][threadIdx.x / 32] = v;
  __syncthreads();
  if (threadIdx.x < 16) {
    double t = 0.0;
    for (int w = 0; w < kGradThreads / 32; ++w) t += sh[threadIdx.x][w];
    tot[threadIdx.x] = t;
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    double t = 0.0;
    if (threadIdx.x == 0) {
      t = (tot[3] + tot[5]) / (inv_radius * inv_radius) * p.scale_z;  // sum M r_pix^2
    } else {
      for (int i = 0; i < kMono; ++i) t += kZernikeDev[threadIdx.x - 1][i] * tot[i];
    }
    atomicAdd(p.red + 3 + threadIdx.x, t);
  }
}

// ----------------------------------------------------------------- launchers

template <class K>
cudaError_t launch_k(K kernel, dim3 grid, int threads, size_t smem, cudaStream_t s, const ShParams& p) {
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_next(kernel, grid, threads, smem, s, p);
}

template <int NX>
size_t row_smem() {
  return (size_t)(kRowThreads / Lat<NX>::N1) * Lat<NX>::N2 * (Lat<NX>::N1 + 1) * sizeof(float2);
}

template <int NX>
cudaError_t rows(bool adjoint, const ShParams& p, int chunks, cudaStream_t s) {
  constexpr int RPI = kRowThreads / Lat<NX>::N1;
  if (adjoint) return launch_k(rows_adj_kernel<NX>, dim3(p.ny / RPI, chunks), kRowThreads, row_smem<NX>(), s, p);
  return launch_k(rows_fwd_kernel<NX>, dim3(p.ny / RPI, p.nl), kRowThreads, row_smem<NX>(), s, p);
}

template <int NY>
cudaError_t cols(bool adjoint, const ShParams& p, cudaStream_t s) {
  constexpr int TW = kLatTW<NY>;
  const size_t smem = (size_t)Lat<NY>::N2 * Lat<NY>::N1 * TW * sizeof(float2);
  const dim3 grid(p.nx / TW, p.nl);
  if (adjoint) return launch_k(cols_adj_kernel<NY>, grid, TW * Lat<NY>::N1, smem, s, p);
  return launch_k(cols_fwd_kernel<NY>, grid, TW * Lat<NY>::N1, smem, s, p);
}

template <int NL>
cudaError_t axial_adj(const ShParams& p, cudaStream_t s) {
  return launch_k(axial_adj_kernel<NL>, dim3(p.ntx, p.wy), kTile * Split<NL>::N1, (size_t)NL * kTile * sizeof(float2),
                  s, p);
}

cudaError_t rows_any(bool adj, const ShParams& p, int chunks, cudaStream_t s) {
  switch (p.nx) {
    case 64: return rows<64>(adj, p, chunks, s);
    case 128: return rows<128>(adj, p, chunks, s);
    case 256: return rows<256>(adj, p, chunks, s);
    case 384: return rows<384>(adj, p, chunks, s);
    case 512: return rows<512>(adj, p, chunks, s);
    case 640: return rows<640>(adj, p, chunks, s);
    case 768: return rows<768>(adj, p, chunks, s);
    case 1024: return rows<1024>(adj, p, chunks, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t cols_any(bool adj, const ShParams& p, cudaStream_t s) {
  switch (p.ny) {
    case 64: return cols<64>(adj, p, s);
    case 128: return cols<128>(adj, p, s);
    case 256: return cols<256>(adj, p, s);
    case 384: return cols<384>(adj, p, s);
    case 512: return cols<512>(adj, p, s);
    case 640: return cols<640>(adj, p, s);
    case 768: return cols<768>(adj, p, s);
    case 1024: return cols<1024>(adj, p, s);
  }
  return cudaErrorInvalidValue;
}

size_t rows_adj_stream_smem(const Plan& pl) {
#define X(n) if (pl.nx == n) return 2 * ((RowsAdjStage<n>::bytes(pl.stage_rows) + 127) / 128 * 128);
  X(64) X(128) X(256) X(384) X(512) X(640) X(768) X(1024)
#undef X
  return SIZE_MAX;
}

cudaError_t rows_adj_stream_any(const ShParams& p, const RowsAdjShare& share, int raw_rows, unsigned* err, cudaStream_t s) {
#define X(n)                                                                                                        \
  if (p.nx == n) {                                                                                                  \
    const size_t smem = 2 * ((RowsAdjStage<n>::bytes(raw_rows) + 127) / 128 * 128);                                 \
    const cudaError_t e = cudaFuncSetAttribute(rows_adj_stream_kernel<n>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                               (int)smem);                                                          \
    if (e != cudaSuccess) return e;                                                                                 \
    return launch_next(rows_adj_stream_kernel<n>, dim3(share.ctas), kRowThreads, smem, s, p, share, raw_rows, err); \
  }
  X(64) X(128) X(256) X(384) X(512) X(640) X(768) X(1024)
#undef X
  return cudaErrorInvalidValue;
}

cudaError_t axial_adj_any(const ShParams& p, cudaStream_t s) {
  switch (p.nl) {
    case 16: return axial_adj<16>(p, s);
    case 32: return axial_adj<32>(p, s);
    case 64: return axial_adj<64>(p, s);
    case 96: return axial_adj<96>(p, s);
    case 128: return axial_adj<128>(p, s);
    case 160: return axial_adj<160>(p, s);
    case 200: return axial_adj<200>(p, s);
    case 256: return axial_adj<256>(p, s);
    case 512: return axial_adj<512>(p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// c P on the sensor grid: the input chirp of Eq. 6 with its centring phase,
// exp(-i pi [alpha (n - N/2)^2 + n]) per axis, times exp(i sum_j c_j Z_j).  Phases
// are reduced in units of pi in float64 before the float32 rounding.
void build_pupil_table(int nx, int ny, double alpha, const double* coeffs, int ncoeffs, std::vector<float2>& out) {
  out.resize((size_t)nx * ny);
  const double pi = 3.14159265358979323846264338327950288;
  const double inv_radius = 2.0 / (double)(nx < ny ? nx : ny);
  for (int l = 0; l < ny; ++l)
    for (int n = 0; n < nx; ++n) {
      const double dx = n - nx / 2.0, dy = l - ny / 2.0;
      double turns = -(std::fmod(alpha * dx * dx, 2.0) + (double)(n & 1)) - (std::fmod(alpha * dy * dy, 2.0) + (double)(l & 1));
      const double rp = std::sqrt(dx * dx + dy * dy);
      double z[15];
      zernike15(rp * inv_radius, rp > 0.0 ? dx / rp : 1.0, rp > 0.0 ? dy / rp : 0.0, z);
      double phi = 0.0;
      for (int j = 0; j < ncoeffs; ++j) phi += coeffs[j] * z[j];
      turns += std::fmod(phi / pi, 2.0);
      out[(size_t)l * nx + n] = make_float2((float)std::cos(pi * turns), (float)std::sin(pi * turns));
    }
}

namespace {

struct PupilParams {
  float2* cp;
  const float4* cis;  // [256] exp(i pi k / 128) as pairs of floats (re hi, re lo, im hi, im lo)
  int nx, ny;
  double c[kMono];    // phase / pi as a polynomial in the pixel offsets from the centre
};

constexpr int kPupilRows = 8;  // rows of a block: their polynomials in x come from the first threads

// c P per sensor pixel, the device twin of build_pupil_table.  The phase over pi
// (chirp and Zernike sum, a polynomial of degree four) is evaluated in float64,
// split into the nearest 1/128 and a remainder, and the remainder turns the
// tabulated exponential (cis_turn): one rounding to float32 and 2^-35, in the place
// of the float64 sine and cosine, square root and fmod per pixel that took 78 us at
// 512 x 512 (two FP64 operations per clock and SM: about 18 per pixel now, 11 us).
__global__ void __launch_bounds__(256) pupil_table_kernel(const __grid_constant__ PupilParams p) {
  after_previous_kernel();
  __shared__ double row[kPupilRows][5];
  __shared__ float4 cis[256];
  const int y0 = blockIdx.y * kPupilRows;
  cis[threadIdx.x] = __ldg(p.cis + threadIdx.x);
  if (threadIdx.x < kPupilRows * 5) {
    const int r = threadIdx.x / 5, a = threadIdx.x % 5;
    const double dy = (double)(y0 + r - p.ny / 2);
    double v = 0.0;  // sum over b of c[a, b] dy^b
    for (int i = kMono - 1; i >= 0; --i)
      if (mono_a(i) == a) v = v * dy + p.c[i];
    row[r][a] = v;
  }
  __syncthreads();
  const int tx = grid_tx(p.nx);
  const int x = blockIdx.x * tx + threadIdx.x % tx;
  const double dx = (double)(x - p.nx / 2);
  for (int r = threadIdx.x / tx; r < kPupilRows && y0 + r < p.ny; r += 256 / tx) {
    const double* k = row[r];
    const double t = (((k[4] * dx + k[3]) * dx + k[2]) * dx + k[1]) * dx + k[0];
    p.cp[(size_t)(y0 + r) * p.nx + x] = cis_turn(t, (x + y0 + r) & 1, cis);  // with the centring phase (-1)^(n + l)
  }
}

}  // namespace

void pupil_cis_table(std::vector<float4>& out) {
  out.resize(256);
  for (int k = 0; k < 256; ++k) {
    const double a = 3.14159265358979323846 * k / 128.0, c = std::cos(a), s = std::sin(a);
    const float ch = (float)c, sh = (float)s;
    out[k] = make_float4(ch, (float)(c - ch), sh, (float)(s - sh));
  }
}

cudaError_t launch_pupil_table(const Plan& pl, cudaStream_t s) {
  PupilParams p;
  p.cp = (float2*)(pl.ws + pl.off_cp);
  p.cis = (const float4*)(pl.ws + pl.off_cis);
  p.nx = pl.nx;
  p.ny = pl.ny;
  const double pi = 3.14159265358979323846, inv_radius = 2.0 / (double)(pl.nx < pl.ny ? pl.nx : pl.ny);
  for (int i = 0; i < kMono; ++i) {
    double v = 0.0;
    for (int j = 0; j < pl.sh_ncoeffs; ++j) v += pl.sh_coeffs[j] * kZernike[j][i];
    p.c[i] = v / pi * std::pow(inv_radius, mono_a(i) + mono_b(i));
  }
  p.c[3] -= pl.sh_alpha;  // the input chirp, -alpha (dx^2 + dy^2)
  p.c[5] -= pl.sh_alpha;
  const int tx = grid_tx(pl.nx);
  return launch_next(pupil_table_kernel, dim3(pl.nx / tx, (pl.ny + kPupilRows - 1) / kPupilRows), 256, 0, s, p);
}

bool generic_lateral_supported(int nx, int ny) {
  auto ok = [](int n) {
    return n == 64 || n == 128 || n == 256 || n == 384 || n == 512 || n == 640 || n == 768 || n == 1024;
  };
  return ok(nx) && ok(ny);
}

bool sharpness_supported(int nx, int ny, int nl) { return generic_lateral_supported(nx, ny) && axial_supported(nl); }

cudaError_t launch_lateral_generic(const Plan& pl, const uint16_t* frames, int ring_start, cudaStream_t s) {
  char* ws = pl.ws;
  ShParams p = {};
  p.frames = frames;
  p.xtab = (const Tap*)(ws + pl.off_xtab);
  p.ytab = (const Tap*)(ws + pl.off_ytab);
  p.cp = (const float2*)(ws + pl.off_cg);
  p.twx = (const float2*)(ws + pl.off_twx);
  p.twy = (const float2*)(ws + pl.off_twy);
  p.twl = (const float2*)(ws + pl.off_twl);
  p.F = (float2*)(ws + pl.off_F);
  p.inter = (float2*)(ws + pl.off_inter);
  p.nx = pl.nx; p.ny = pl.ny; p.nl = pl.nl;
  p.x0 = pl.x0; p.y0 = pl.y0; p.wx = pl.wx; p.wy = pl.wy; p.ntx = pl.ntx;
  p.ring_start = ring_start;
  cudaError_t e = rows_any(false, p, 1, s);
  if (e == cudaSuccess) e = cols_any(false, p, s);
  return e;
}

cudaError_t launch_sharpness(const Plan& pl, const uint16_t* frames, float* vol, bool have_inter, cudaStream_t s) {
  char* ws = pl.ws;
  ShParams p = {};
  p.frames = frames;
  p.xtab = (const Tap*)(ws + pl.off_xtab);
  p.ytab = (const Tap*)(ws + pl.off_ytab);
  p.cp = (const float2*)(ws + pl.off_cp);
  p.twx = (const float2*)(ws + pl.off_twx);
  p.twy = (const float2*)(ws + pl.off_twy);
  p.twl = (const float2*)(ws + pl.off_twl);
  p.F = (float2*)(ws + pl.off_F);
  p.inter = (float2*)(ws + pl.off_inter);
  p.qpart = (float2*)(ws + pl.off_Q);
  p.vol = vol;
  p.red = (double*)(ws + pl.off_red);
  p.nx = pl.nx; p.ny = pl.ny; p.nl = pl.nl;
  p.x0 = pl.x0; p.y0 = pl.y0; p.wx = pl.wx; p.wy = pl.wy; p.ntx = pl.ntx;
  p.tpc = pl.sh_tpc;
  p.alpha2 = (float)(pl.sh_alpha * pl.sh_alpha);
  p.scale_z = 3.14159265358979323846 * pl.sh_alpha / pl.sh_z;
  {
    // sum P <= |K|^2 (65535 nx ny nl)^2 (Parseval), which the scale takes to 2^62:
    // the sum of squares stays under 2^124, and P down to 1e-36 of it counts in full
    int ex = 0;
    const double top = 65535.0 * pl.nx * pl.ny * pl.nl * pl.sh_alpha;
    std::frexp(top * top, &ex);
    p.sum_scale = (float)std::ldexp(1.0, std::max(-126, std::min(126, 62 - ex)));
  }
  const int chunks = (pl.nl + pl.sh_tpc - 1) / pl.sh_tpc;

  // The adjoint row pass is streamed where a CTA's share is longer than a chunk by
  // enough (all chunks but two of a band, on average) and bulk copies can read the
  // frames.
  const RowsAdjShare share{pl.ny * pl.n1x / kRowThreads, pl.nl, pl.num_sms, pl.sh_tpc};
  const bool stream = (uintptr_t)frames % 16 == 0 && share.fits() && share.pairs() >= 2ll * share.ctas &&
                      share.ctas <= (long long)share.bands * (chunks - 2) && rows_adj_stream_smem(pl) <= 226u * 1024u;
  unsigned* const err = (unsigned*)(p.red + kShRedErr);
  cudaError_t e = cudaMemsetAsync(p.red, 0, kShRedDoubles * sizeof(double), s);
  if (e == cudaSuccess && !have_inter) e = rows_any(false, p, chunks, s);
  if (e == cudaSuccess && !have_inter) e = cols_any(false, p, s);
  if (e == cudaSuccess) {
    AxialParams ap = {};
    ap.inter = p.inter;
    ap.vol = vol;
    ap.cplx = nullptr;
    ap.twl = (const float2*)(ws + pl.off_twax);
    ap.ox = (const float2*)(ws + pl.off_ox);
    ap.oy = (const float2*)(ws + pl.off_oy);
    ap.nl = pl.nl; ap.wx = pl.wx; ap.wy = pl.wy; ap.ntx = pl.ntx;
    ap.power_scale = p.alpha2;
    ap.magnitude = 0;
    ap.err = err;
    e = launch_axial(pl, ap, s);
  }
  const size_t nvox = (size_t)pl.nl * pl.wy * pl.wx;
  if (e == cudaSuccess) {
    e = launch_next(sums_kernel, dim3(6 * pl.num_sms), kGradThreads, 0, s, p, nvox);
  }
  if (e == cudaSuccess) e = axial_adj_any(p, s);
  if (e == cudaSuccess && stream && share.ctas > 1)
    e = launch_next(zero_split_kernel, dim3(share.ctas - 1), kRowThreads, 0, s, p, share);
  if (e == cudaSuccess) e = cols_any(true, p, s);
  if (e == cudaSuccess)
    e = stream ? rows_adj_stream_any(p, share, pl.stage_rows, err, s)
               : rows_any(true, p, chunks, s);
  if (e == cudaSuccess) {
    const int tx = grid_tx(p.nx), gx = p.nx / tx, ry = kGradThreads / tx;
    const int gy = std::min((p.ny + ry - 1) / ry, std::max(1, 3 * pl.num_sms / gx));
    e = launch_next(grad_kernel, dim3(gx, gy), kGradThreads, 0, s, p, chunks,
                    (const unsigned*)(have_inter ? &((const Counters*)(ws + pl.off_sctr))->err : nullptr));
  }
  return e;
}

}  // namespace ssoct
