// Frames that one CTA or a pair transforms whole, the lateral kernel's instances
// for square frames up to 512 pixels, and the choice among all lateral kernels.
#include "lateral_kernel.cuh"

namespace ssoct {
namespace {

// ---------------------------------------------------------------- small frames
//
// Frames of up to 128 x 128 pixels fit in the shared memory of one CTA or of a
// pair, which then transforms a whole frame: no queue, no scratch ring, no waits
// on other frames.  The persistent kernel spends such frames in hand-overs
// (publishing a row item and acquiring a column item takes longer than their
// arithmetic).  Event times around this kernel against the persistent one with
// lateral_pick, paper order: 64 x 64 x 32 with a 23 x 17 window 8.9 us against
// 15.3, 64 x 64 x 256 12.4 against 20, 128 x 128 x 64 14.4 against 23, x 256
// 34.7 against 38, x 512 58 against 61.  Eight CTAs for a frame of 256 x 256 are
// slower than the persistent kernel (x 256: 121 against 101 us).
// A frame's rows are split over C CTAs (a pair for 128 x 128 and 64 x 128: one
// CTA of 1024 threads took 19.8 us at 128 x 128 x 64).
//  * the band's raw rows, the frame's x taps, the chirp and the twiddles arrive
//    together, one round trip before the first barrier;
//  * rows: N1x threads per row, each row's exchange in its own block of the
//    band (a row's threads lie in one warp), rows padded by 64 bytes so that
//    the two rows of a half warp fall into different banks;
//  * columns: a warp takes 32 window columns and one j1, so that shared-memory
//    accesses are 256-byte rows and stores are whole tile rows; CTA r takes the
//    column groups r, r + C, ...  The inputs come from all the cluster's bands
//    (distributed shared memory); once all CTAs have read theirs, the exchange
//    between the two stages overwrites the CTA's own band.
template <int NX, int NY, int C>
struct SmallLat {
  static constexpr int kRows = NY / C;                      // rows of a CTA
  static constexpr int kThreadsAll = kRows * Split<NX>::N1;
  static constexpr int kPitch = NX + 8;
  static constexpr int kGroupsAtOnce = kThreadsAll / 32 / Split<NY>::N1;  // 32-column groups per pass and CTA
  static constexpr int kGroups = NX / 32 / C;                             // and of a CTA, at most
  static constexpr size_t kBand = (size_t)kPitch * kRows * sizeof(float2);
  static constexpr size_t kTaps = kBand;
  static constexpr size_t kTables = kTaps + (size_t)NX * sizeof(Tap);
  static constexpr size_t kRaw = kTables + (size_t)(2 * NX + NY) * sizeof(float2);  // raw rows last
  static_assert(C == 1 || (kGroups >= 1 && kGroups <= kGroupsAtOnce && (size_t)NY * 32 * kGroups * sizeof(float2) <= kBand),
                "a cluster's columns go in one pass, their exchange in the band");
  static size_t bytes(int raw_rows) { return kRaw + (size_t)raw_rows * NX * sizeof(uint16_t); }
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// All threads of the cluster: earlier shared-memory accesses are ordered before later ones.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// Address of this CTA's shared-memory address a in the CTA of rank r.
__device__ __forceinline__ unsigned cluster_map(unsigned a, unsigned r) {
  unsigned m;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(m) : "r"(a), "r"(r));
  return m;
}
__device__ __forceinline__ float2 ld_cluster(unsigned a) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}

template <int NX, int NY, int C, bool AF>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(SmallLat<NX, NY, C>::kThreadsAll, C > 1 ? 2 : 1)
    lateral_small_kernel(const __grid_constant__ LateralParams p) {
  after_previous_kernel();
  using L = SmallLat<NX, NY, C>;
  constexpr int T = L::kThreadsAll, PITCH = L::kPitch, RB = L::kRows;
  constexpr int N1x = Split<NX>::N1, N2x = Split<NX>::N2, N1y = Split<NY>::N1, N2y = Split<NY>::N2;
  static_assert(32 % N1x == 0 && N2x % N1x == 0 && N2y % N1y == 0, "a row in one warp, whole second stages");
  static_assert((T / 32) % N1y == 0 && T >= NX && RB % N1y == 0, "whole column groups, one table entry per thread");
  extern __shared__ __align__(1024) unsigned char smem[];
  float2* fr = reinterpret_cast<float2*>(smem);
  Tap* xtaps = reinterpret_cast<Tap*>(smem + L::kTaps);
  float2* cxs = reinterpret_cast<float2*>(smem + L::kTables);
  float2* twx = cxs + NX;
  float2* twy = twx + NX;
  uint16_t* raw = reinterpret_cast<uint16_t*>(smem + L::kRaw);
  const int tid = threadIdx.x;
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int f = blockIdx.x / C;
  const int slot = (p.tab0 + f) % p.nl;
  const int yb = tid / N1x, j1 = tid % N1x;
  const int y = rank * RB + yb;
  float2* row = fr + yb * PITCH;
  constexpr int A = N2x > N2y ? N2x : N2y;
  float2 a[A];
  bool mirrored = false;
  float2 cyv;
  if (tid < NX) {
    cxs[tid] = ldg2((AF ? p.cx2 : p.cx) + tid);
    twx[tid] = ldg2(p.twx + tid);
    if (!AF) xtaps[tid] = p.xtab[(size_t)slot * NX + tid];
  }
  for (int i = tid; i < NY; i += T) twy[i] = ldg2(p.twy + i);
  if constexpr (AF) {
    const int q = af_bin(f, p.nl);
    mirrored = q > p.nl / 2;
    const float2* in = p.aplanes + ((size_t)(mirrored ? p.nl - q : q) * NY + y) * NX;
#pragma unroll
    for (int j2 = 0; j2 < N2x; ++j2) a[j2] = in[j1 + N1x * j2];
    cyv = ldg2(p.cy2 + y);
    __syncthreads();
    if (mirrored) {
      // conj(v) c2, as in row_item
#pragma unroll
      for (int j2 = 0; j2 < N2x; ++j2) {
        const float2 v = a[j2], c = cxs[j1 + N1x * j2];
        a[j2] = make_float2(fmaf(v.x, c.x, v.y * c.y), fmaf(v.x, c.y, -v.y * c.x));
      }
    }
  } else {
    // the band's raw rows: from its first row's base to its last row's base + 1
    const Tap* ytab = p.ytab + (size_t)slot * NY;
    const int lo = ytab[rank * RB].base, hi = ytab[rank * RB + RB - 1].base + 1;
    const Tap ty = ytab[y];
    cyv = ldg2(p.cy + y);
    const uint4* src = reinterpret_cast<const uint4*>(p.frames + ((size_t)((p.ring_start + f) % p.nl) * NY + lo) * NX);
    for (int i = tid; i < (hi - lo + 1) * (NX / 8); i += T) reinterpret_cast<uint4*>(raw)[i] = src[i];
    __syncthreads();
    const uint16_t* r0 = raw + (ty.base - lo) * NX;
    const uint16_t* r1 = r0 + NX;
#pragma unroll
    for (int j2 = 0; j2 < N2x; ++j2) {
      const int n = j1 + N1x * j2;
      const Tap t = xtaps[n];
      const float v0 = fmaf(t.w0, u16_to_f(r0[t.base]), t.w1 * u16_to_f(r0[t.base + 1]));
      const float v1 = fmaf(t.w0, u16_to_f(r1[t.base]), t.w1 * u16_to_f(r1[t.base + 1]));
      const float v = fmaf(ty.w0, v0, ty.w1 * v1);
      const float2 c = cxs[n];
      a[j2] = make_float2(v * c.x, v * c.y);
    }
  }
  Dft<N2x, 1>::template run<1, 0>(a);
  if (AF && !mirrored) {
#pragma unroll
    for (int k2 = 0; k2 < N2x; ++k2) a[k2] = cmul(a[k2], twx[k2 * N1x + j1]);
  } else {
#pragma unroll
    for (int k2 = 0; k2 < N2x; ++k2) a[k2] = cmul(a[k2], cmul(twx[k2 * N1x + j1], cyv));
  }
#pragma unroll
  for (int k2 = 0; k2 < N2x; ++k2) row[xswz<N1x>(k2, j1)] = a[k2];
  __syncwarp();
  static_for<0, N2x / N1x>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const int k2 = j1 + N1x * i;
#pragma unroll
    for (int jj = 0; jj < N1x; ++jj) a[i * N1x + jj] = row[xswz<N1x>(k2, jj)];
    Dft<N1x, 1>::template run<1, i * N1x>(a);
  });
  __syncwarp();
  static_for<0, N2x / N1x>([&](auto I) {
    constexpr int i = decltype(I)::value;
#pragma unroll
    for (int k1 = 0; k1 < N1x; ++k1) row[j1 + N1x * i + N2x * k1] = a[i * N1x + k1];
  });
  if constexpr (C > 1) cluster_sync();
  else __syncthreads();
  // columns of the window, 32 at a time; every thread meets every barrier
  const int lane = tid % 32, k = tid / 32 % N1y;
  const int groups = (p.wx + 31) / 32;  // group g goes to CTA g mod C
  for (int g0 = 0; g0 * C < groups; g0 += L::kGroupsAtOnce) {
    const int g = (g0 + tid / 32 / N1y) * C + rank;
    const int kxw = g * 32 + lane;
    const bool live = g < groups && kxw < p.wx;
    // where this column's exchange goes: the rows it was read from, or (C > 1)
    // its place among the CTA's columns, NY rows in the band
    constexpr int EP = C > 1 ? 32 * L::kGroups : PITCH;
    float2* col = C > 1 ? fr + tid / 32 / N1y * 32 + lane : fr + p.x0 + kxw;
    if (live) {
      if constexpr (C > 1) {
        // row k + N1y j2 lies in the band of rank N1y j2 / RB (k < N1y divides RB)
        const unsigned at = smem_u32(fr + p.x0 + kxw) + (unsigned)(k * PITCH * sizeof(float2));
#pragma unroll
        for (int j2 = 0; j2 < N2y; ++j2)
          a[j2] = ld_cluster(cluster_map(at, (unsigned)(N1y * j2 / RB)) + (unsigned)(N1y * j2 % RB * PITCH * sizeof(float2)));
      } else {
#pragma unroll
        for (int j2 = 0; j2 < N2y; ++j2) a[j2] = col[(k + N1y * j2) * PITCH];
      }
      Dft<N2y, 1>::template run<1, 0>(a);
    }
    if constexpr (C > 1) cluster_sync();  // every band has been read, and no CTA leaves before
    if (live) {
#pragma unroll
      for (int k2 = 0; k2 < N2y; ++k2) col[(k + N1y * k2) * EP] = cmul(a[k2], twy[k2 * N1y + k]);
    }
    __syncthreads();
    if (live) {
      static_for<0, N2y / N1y>([&](auto I) {
        constexpr int i = decltype(I)::value;
        const int k2 = k + N1y * i;
#pragma unroll
        for (int jj = 0; jj < N1y; ++jj) a[i * N1y + jj] = col[(jj + N1y * k2) * EP];
        Dft<N1y, 1>::template run<1, i * N1y>(a);
      });
      if constexpr (AF) {
        const Desc d{kColItem, f, 0, 0, 0, slot};
        if (p.cplx) {
          if (p.magnitude) af_epilogue<NY, false, true, true, NX>(p, d, a, k, kxw);
          else af_epilogue<NY, false, false, true, NX>(p, d, a, k, kxw);
        } else {
          if (p.magnitude) af_epilogue<NY, false, true, false, NX>(p, d, a, k, kxw);
          else af_epilogue<NY, false, false, false, NX>(p, d, a, k, kxw);
        }
      } else {
        float2* dst = p.inter + ((size_t)(kxw / kTile) * p.nl + slot) * kTile + kxw % kTile;
        const size_t row_pitch = (size_t)p.ntx * p.nl * kTile;
        static_for<0, N2y / N1y>([&](auto I) {
          constexpr int i = decltype(I)::value;
          const int k2 = k + N1y * i;
#pragma unroll
          for (int k1 = 0; k1 < N1y; ++k1) {
            const int kyw = k2 + N2y * k1 - p.y0;
            if (kyw >= 0 && kyw < p.wy) dst[(size_t)kyw * row_pitch] = a[i * N1y + k1];
          }
        });
      }
    }
  }
}

// Raw rows that a band of the plan's frames takes, at most, over bands and frames.
inline int small_raw_rows(const Plan& p, int band) {
  int most = 0;
  for (int t = 0; t < p.nl; ++t)
    for (int r = 0; r < p.ny; r += band) {
      const Tap* y = p.ytab.data() + (size_t)t * p.ny + r;
      most = std::max(most, y[band - 1].base + 1 - y[0].base + 1);
    }
  return most;
}

template <int NX, int NY, int C>
cudaError_t launch_small(const Plan& p, const LateralParams& lp, cudaStream_t s) {
  using L = SmallLat<NX, NY, C>;
  auto* kernel = p.axial_first ? lateral_small_kernel<NX, NY, C, true> : lateral_small_kernel<NX, NY, C, false>;
  const size_t smem = L::bytes(p.small_rows);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_next(kernel, dim3(lp.sch.nl * C), L::kThreadsAll, smem, s, lp);
}

}  // namespace

// frame size, CTAs per frame
#define SSOCT_SMALL_SIZES(X) X(64, 64, 1) X(128, 64, 1) X(64, 128, 2) X(128, 128, 2)

int lateral_small_rows(const Plan& p) {
#define X(a, b, c)                                                                     \
  if (p.nx == a && p.ny == b) {                                                        \
    const int rows = small_raw_rows(p, SmallLat<a, b, c>::kRows);                      \
    return SmallLat<a, b, c>::bytes(rows) <= 227u * 1024u ? rows : 0;                  \
  }
  SSOCT_SMALL_SIZES(X)
#undef X
  return 0;
}

// A plan with an injected stall (ssoct_inject_stall) runs the work queue that
// the stall is for.
bool lateral_small(const Plan& p) { return p.small_rows > 0 && !p.inject_skip; }

// Instances of this unit (lateral_large.cu has 640, 768 and 1024)
#define SSOCT_LATERAL_SIZES(X) X(64, 64) X(128, 128) X(256, 256) X(384, 384) X(512, 512) X(128, 64) X(64, 128)

bool lateral_supported(int nx, int ny) {
#define X(a, b) if (nx == a && ny == b) return true;
  SSOCT_LATERAL_SIZES(X) X(640, 640) X(768, 768) X(1024, 1024)
#undef X
  return false;
}

size_t lateral_smem_bytes(const Plan& p) {
  size_t sb, total;
  smem_layout(p, sb, total);
  return total;
}

int lateral_col_band(int ny) { return kThreads / split_n1(ny); }

cudaError_t launch_lateral_with(const Plan& p, const LateralParams& lp, const void* tmap,
                                int num_sms, cudaStream_t s) {
  if (lateral_small(p)) {
#define X(a, b, c) if (p.nx == a && p.ny == b) return launch_small<a, b, c>(p, lp, s);
    SSOCT_SMALL_SIZES(X)
#undef X
  }
#define X(a, b) if (p.nx == a && p.ny == b) return launch_square<a, b>(p, lp, tmap, num_sms, s);
  SSOCT_LATERAL_SIZES(X)
#undef X
  return launch_lateral_large(p, lp, tmap, num_sms, s);
}

cudaError_t launch_lateral_pair(const Plan& p, const LateralParams& lp, int num_sms, cudaStream_t s) {
  if (p.nx <= 256) return launch_lateral_pairs_256(p, lp, p.tmap, num_sms, s);
  if (p.nx <= 512) return launch_lateral_pairs_512(p, lp, p.tmap, num_sms, s);
  return launch_lateral_pairs_1024(p, lp, p.tmap, num_sms, s);
}

cudaError_t launch_lateral(const Plan& p, const LateralParams& lp, cudaStream_t s) {
  return launch_lateral_with(p, lp, p.tmap, p.num_sms, s);
}

}  // namespace ssoct
