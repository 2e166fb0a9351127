// Internal types shared by the host plan code and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/ssoct.h"

namespace ssoct {

constexpr int kThreads = 256;          // threads of a lateral-stage CTA (two CTAs per SM)
constexpr int kTile = 32;              // pixels per sweep-axis tile (one x-run)

// FFT length N = N1 * N2 as the kernels split it: an N2-point DFT per thread,
// a twiddle, an exchange through shared memory, N1-point DFTs (0 = not built).
__host__ __device__ constexpr int split_n1(int n) {
  return n == 16 ? 4 : n == 32 ? 4 : n == 64 ? 8 : n == 96 ? 4 : n == 128 ? 8 : n == 160 ? 4 : n == 200 ? 5
       : n == 256 ? 16 : n == 384 ? 16 : n == 512 ? 16 : n == 640 ? 32 : n == 768 ? 32 : n == 1024 ? 32 : 0;
}

// Stage 2 of a transform of length N = N1 x N2 (N1 = split_n1(N)) in the
// persistent lateral kernel: N2 N1-point DFTs spread over the transform's N1
// threads, NI per thread; where N1 does not divide N2 (384 = 16 x 24,
// 640 = 32 x 20, 768 = 32 x 24) the last one is idle in the threads
// j1 >= N2 - N1 (NI - 1).  A is the register array length.
template <int N, int N1_ = split_n1(N)>
struct Stage2 {
  static constexpr int N1 = N1_, N2 = N / N1_;
  static constexpr int NI = (N2 + N1 - 1) / N1;
  static constexpr int A = NI * N1 > N2 ? NI * N1 : N2;
  // stage-2 DFT i of thread j1 exists (always, for the iterations N1 fills)
  __host__ __device__ static constexpr bool live(int i, int j1) { return (i + 1) * N1 <= N2 || j1 + N1 * i < N2; }
};

// Split of the axial-first first pass's transform over nl frames, N1 x nl/N1
// with a tile of 32 N1 threads: the axial split where it gives 8 to 16 warps,
// and 16 x 6, 16 x 10, 20 x 10 for 96, 160, 200 frames, whose axial splits
// (4 x 24, 4 x 40, 5 x 40) would leave four or five warps per tile.
__host__ __device__ constexpr int ra_split_n1(int nl) {
  return nl == 96 ? 16 : nl == 160 ? 16 : nl == 200 ? 20 : split_n1(nl);
}

// Split of the sweep transform in the axial kernels that write volumes and cuts:
// 8 x 12, 8 x 20 and 10 x 20 for 96, 160 and 200 frames, whose general splits
// (4 x 24, 4 x 40, 5 x 40) would leave four or five warps per tile and 24 or 40
// values per thread.
__host__ __device__ constexpr int ax_split_n1(int nl) {
  return nl == 96 ? 8 : nl == 160 ? 8 : nl == 200 ? 10 : split_n1(nl);
}

// Rows per tensor copy of a lateral column band: the largest divisor of ny up
// to 256 (a box dimension's limit), so that whole boxes cover the column.
__host__ __device__ constexpr int band_box_rows(int ny) {
  int r = ny < 256 ? ny : 256;
  while (r > 1 && ny % r != 0) --r;
  return r;
}

// Separable linear-interpolation tap for one output coordinate of one frame
// (Eq. 5): the value is w0 * in[base] + w1 * in[base + 1]; base is clamped so
// both reads are inside the frame, and a weight is 0 where its tap fell outside.
struct __align__(16) Tap {
  int base;
  float w0;
  float w1;
  float pad;
};

// Eq. 5 along one axis: output pixel i reads the input at u = c + (i - c) s,
// c = n / 2, by linear interpolation; a tap outside [0, n) reads 0.  Host and
// device build the same taps: u is written as the fused step that the device (and
// an Arm host) would make of it, since an x86 host rounds the product too and
// could put a base one row beside the device's, whose rows are staged in buffers
// sized from the host's taps.
__host__ __device__ inline Tap eq5_tap(int i, int n, double s) {
  const double c = n / 2.0;
  const double u = fma(i - c, s, c);
  const double fl = floor(u);
  const double a = u - fl;
  const long long i0 = (long long)fl, i1 = i0 + 1;
  const double w0 = (i0 >= 0 && i0 < n) ? 1.0 - a : 0.0;
  const double w1 = (i1 >= 0 && i1 < n) ? a : 0.0;
  long long b = i0 < 0 ? 0 : i0;
  if (b > n - 2) b = n - 2;
  double wb = 0.0, wb1 = 0.0;
  if (i0 == b) wb += w0; else if (i0 == b + 1) wb1 += w0;
  if (i1 == b) wb += w1; else if (i1 == b + 1) wb1 += w1;
  Tap t;
  t.base = (int)b;
  t.w0 = (float)wb;
  t.w1 = (float)wb1;
  t.pad = 0.f;
  return t;
}

// Eq. 5 along a 64-pixel strip x0 .. x0 + 63 of one frame (axial-first order):
// the position u(x0 + k) = u(x0) + k s_t lies at staged column
// off + k + floor(f + k e) with weight frac(f + k e), where the strip's source
// rows are staged from column xs (a multiple of 8) on.  Built in float64.
struct __align__(16) StripTap {
  int xs;    // first staged source column (multiple of 8; may be negative)
  int off;   // floor(u(x0)) - xs (>= 1)
  float f;   // u(x0) - floor(u(x0))
  float e;   // s_t - 1
};

// Device work-queue counters of the lateral kernel (zeroed before each launch).
struct Counters {
  unsigned ticket;
  unsigned abort;
  unsigned err;
  unsigned pad[29];
  // followed by rows_done[nlambda], cols_done[nlambda]
};

constexpr unsigned kErrTimeout = 1u;      // lateral kernel: a queue wait ran out
constexpr unsigned kErrAxialTc = 2u;      // tensor-core axial kernel: an MMA wait ran out
constexpr unsigned kErrAxial = 4u;        // streaming axial kernel: a stage-buffer wait ran out
constexpr unsigned kErrAdjoint = 8u;      // adjoint row pass: a stage-buffer wait ran out

// Order in which the lateral kernel takes its items.  Step s holds the row
// items of frame s (if s < nl) and then the column items of frame s - lag (if
// s >= lag).  A column item of frame f waits for every row item of f; a row item
// of frame f (f >= slots) waits for every column item of f - slots, whose L2
// scratch slot it reuses.  Both wait on items of earlier tickets, and a ticket
// is only taken by a running CTA, so the queue always drains (requires
// slots > lag).
struct LateralSchedule {
  int nl;
  int n_row;   // row items per frame
  int n_col;   // column items per frame
  int lag;
  int slots;

  __host__ __device__ long long total() const { return (long long)nl * (n_row + n_col); }

  // 32-bit arithmetic: a sweep has at most 512 x 2 x 1024 tickets, and the
  // producer decodes one per item, so 64-bit division would cost it hundreds
  // of cycles.
  __host__ __device__ void decode(unsigned k, int& kind, int& frame, int& item) const {
    const unsigned nr = (unsigned)n_row, nc = (unsigned)n_col;
    const unsigned head = (unsigned)lag * nr;
    if (k < head) {
      kind = 0;
      frame = (int)(k / nr);
      item = (int)(k - (unsigned)frame * nr);
      return;
    }
    k -= head;
    const unsigned per = nr + nc;
    const unsigned both = (unsigned)(nl - lag) * per;
    if (k < both) {
      const unsigned st = k / per;
      const unsigned r = k - st * per;
      if (r < nr) {
        kind = 0;
        frame = lag + (int)st;
        item = (int)r;
      } else {
        kind = 1;
        frame = (int)st;
        item = (int)(r - nr);
      }
      return;
    }
    k -= both;
    kind = 1;
    const unsigned q = k / nc;
    frame = nl - lag + (int)q;
    item = (int)(k - q * nc);
  }
};

// Default lag and ring slots of the lateral kernel for `frames` frames of
// `items` work items each, with at most max_slots scratch slots.  A column item
// waits for every row item of its frame and a row item for the column items of
// the frame whose slot it reuses.  An item is published about 20 us after its
// ticket was taken, and the 304 consumer groups of 152 SMs go through about
// 1200 tickets in that time, so both distances (lag, and slots - lag) span 1200
// items where the ring allows it; a frame count that fits the ring reuses no
// slot.  Measured lateral times, paper order, against lags of 0.7 x 600 items
// with four slots of slack: 256 x 256 x 512 353 -> 203 us, 512 x 512 x 256
// 476 -> 347, 384 x 384 x 96 142 -> 94, 640 x 640 x 160 483 -> 401, 768 x 768 x
// 200 722 -> 675, 1024 x 1024 x 256 1328 -> 1320; 2400 items gave no more.  (Rows of
// 384, 640 and 768 pixels have become faster since, see row_item.)
constexpr int kLateralItemsInFlight = 1200;
struct LateralPick {
  int lag, slots;
};
inline LateralPick lateral_pick(int frames, int items, int max_slots) {
  const int depth = (kLateralItemsInFlight + items - 1) / items;
  LateralPick r;
  r.slots = 2 * depth < max_slots ? 2 * depth : max_slots;
  r.lag = depth;
  if (r.slots < frames && r.lag > r.slots / 2) r.lag = r.slots / 2;
  if (r.slots > frames) r.slots = frames;
  const int most = frames - (frames >= 4 ? 2 : 1);  // frames >= 1; lag < slots always
  if (r.lag > most) r.lag = most;
  return r;
}

// Where the work queue is the faster lateral path for non-square frames, by voxels
// of a sweep.  It saves the two passes their frame buffer, and pays some 15 us for
// filling and draining; the two passes' row and column kernels are slower for 384,
// 640 and 768 (the queue pays earlier there), and the queue's items of frames 64
// pixels wide or high are short (it pays late or, with two powers of two, not at
// all).  Two passes / queue, us a call: 512 x 256 x 32 38 / 45, x 64 88 / 83; 256 x
// 128 x 128 41 / 45, x 256 82 / 76; 384 x 256 x 32 34.0 / 35.0, x 64 69 / 66; 640 x
// 384 x 16 44 / 41, x 160 386 / 333; 1024 x 64 x 128 89 / 98, x 512 315 / 339; 64 x
// 1024 x 64 49 / 57, x 200 147 / 140; 768 x 64 x 256 138 / 131.  A window moves the
// line little (512 x 256 x 32 with 128 x 64: 29 / 31).
inline bool pair_queue_pays(int nx, int ny, long long voxels) {
  auto mixed = [](int n) { return (n & (n - 1)) != 0; };
  if (nx == 64) return ny >= 512 && voxels >= 8000000;
  if (ny == 64) return mixed(nx) && nx >= 640 && voxels >= 6200000;
  if (mixed(nx) && mixed(ny)) return voxels >= 3500000;
  if (mixed(nx) || mixed(ny)) return voxels >= 5000000;
  return voxels >= (nx > ny ? 6500000 : 6000000);
}
// The same for the loss and gradient, where the queue replaces the forward passes
// only: 256 x 256 x 128 267 / 276, x 200 422 / 414; 384 x 384 x 64 348 / 343; 512 x
// 512 x 32 308 / 310, x 64 484 / 450; 640 x 640 x 16 327 / 331; 768 x 768 x 16 426 /
// 405; 1024 x 1024 x 16 621 / 581.
inline bool pupil_queue_pays(int nx, long long voxels) { return voxels >= (nx == 256 ? 12000000 : 8000000); }

// Everything the lateral kernel (rescale + chirp + row FFT, column FFT) reads.
struct LateralParams {
  const uint16_t* frames;  // batch frame f at frames + ((ring_start + f) % nl) * nx * ny
  int ring_start;
  int tab0;                // batch frame f has wavelength / intermediate index (tab0 + f) % nl
  int nx, ny, nl;
  int x0, y0, wx, wy;      // window
  int wxp;                 // scratch row pitch (complex elements)
  int ntx;                 // sweep-axis tiles per window row
  const Tap* xtab;         // [nl][nx]
  const Tap* ytab;         // [nl][ny]
  const float2* cx;        // [nx] input chirp incl. centring phase
  const float2* cy;        // [ny]
  const float2* cx2;       // [nx] squared input chirp (axial-first order, bins above nl/2)
  const float2* cy2;       // [ny]
  const float2* twx;       // [N2x][N1x] row-FFT twiddles
  const float2* twy;       // [N2y][N1y] column-FFT twiddles
  float2* scratch;         // [slots][ny][wxp]
  float2* inter;           // [wy][ntx][nl][32]
  Counters* ctr;
  unsigned* rows_done;     // [nl]
  unsigned* cols_done;     // [nl]
  LateralSchedule sch;
  int stage_rows;          // input rows staged per row item (max over items)
  int stage_bytes;         // bytes of one shared-memory stage buffer (set at launch)
  const float2* cp;        // [ny][nx] chirp x pupil screen in the place of cx, cy, or NULL
  unsigned long long wait_ns;  // limit of every device-side wait (0 = default)
  // axial-first order (SSOCT_FLAG_AXIAL_FIRST): frame f is depth bin af_bin(f);
  // row items read half-spectrum planes, column items write the volume
  const float2* aplanes;   // [nl/2 + 1][ny][nx]
  float* vol;              // [nl][wy][wx]
  float2* cplx;            // optional [nl][wy][wx]
  const float2* ox;        // [wx] output chirp (x)
  const float2* oy;        // [wy] output chirp (y) times K
  float inv_k_abs;         // 1 / |K|: the planes carry |K| (so |V|^2 |K|^2 = |v|^2), oy holds K as well
  int magnitude;
};

struct AxialParams {
  const float2* inter;     // [wy][ntx][nl][32]
  float* vol;              // [nl][wy][wx]
  float2* cplx;            // optional [nl][wy][wx]
  const float2* twl;       // [N2][N1] of ax_split_n1, sign -
  const float2* ox;        // [wx] output chirp (x), incl. centring phase
  const float2* oy;        // [wy] output chirp (y) times the prefactor K
  int nl, wx, wy, ntx;
  float power_scale;       // |K|^2
  int magnitude;           // 1: write |V| instead of |V|^2
  int late;                // launched after the kernel before it, not beside it (see gate_late)
  unsigned* err;           // error word (kErrAxial), the plan's Counters::err
};

struct CutsParams {
  const float* vol;
  float* xy;
  float* xz;
  float* yz;
  int nl, wx, wy, x0, y0, z0;
};

// Host-side plan.
struct Plan {
  int nx, ny, nl;
  int x0, y0, wx, wy;
  unsigned flags;
  double pitch, z, lambda1;
  std::vector<double> lambdas;
  double kre, kim;          // prefactor K
  double alpha;             // d^2 / (lambda_1 z) = |K|
  // host tables
  std::vector<Tap> xtab, ytab;
  std::vector<float2> cx, cy, cx2, cy2, ox, oy, twx, twy, twl, twra, twax;
  std::vector<float2> wq;   // [nl] exp(-2 pi i k / nl), for single-bin transforms
  std::vector<unsigned short> tcb;  // SSOCT_FLAG_TC_AXIAL: BF16 hi / lo 16-point DFT matrix (operand layout)
  // SSOCT_FLAG_PUPIL: input chirp x Zernike screen, its distance z and |K|, frames per Q chunk
  double sh_z = 0.0, sh_alpha = 0.0;
  double sh_coeffs[15] = {};
  int sh_ncoeffs = 0;
  bool sh_dirty = false;     // the device table is built by the next ssoct_sharpness
  int sh_tpc = 8;
  bool sh_ready = false;
  // geometry of the device work
  int n1x, n2x, n1y, n2y, n1l, n2l;
  int rows_per_item, cols_per_item;
  int wxp, ntx;
  int stage_rows;
  int small_rows = 0;        // see lateral_small_rows
  bool pair_queue = false;   // generic plans: launch_lateral_pair takes the plan's frames
  bool pupil_queue = false;  // aberration path: launch_lateral_pupil does
  LateralSchedule sch;
  int slots_alloc = 0;       // scratch-ring slots the workspace holds (sch.slots <= slots_alloc)
  int slots_noalloc = 0;     // ring slots counted in noalloc_bytes
  size_t noalloc_bytes = 0;  // scratch the no-allocation path asks for (its size limit applies to this)
  bool use_tc = false;       // axial pass on the tensor cores (flag, or the autotuner's choice)
  // workspace layout (byte offsets)
  size_t off_ctr, off_xtab, off_ytab, off_cx, off_cy, off_cx2, off_cy2, off_ox, off_oy, off_twx, off_twy, off_twl;
  size_t off_twra = 0;       // twiddles of the tiled first pass's split (ra_split_n1)
  size_t off_twax = 0;       // twiddles of the axial kernels' split (ax_split_n1; off_twl where the splits agree)
  size_t off_cis = 0;        // exp(i pi k / 128) (pupil_cis_table)
  size_t off_sctr = 0;       // the work queue's counters of the aberration path
  // host image of the workspace from off_image on (the tables but the taps), and
  // the rescale ratios lambda_t / lambda_1 in it
  std::vector<unsigned char> image;
  size_t off_image = 0, off_ratio = 0;
  size_t off_tcb, off_wq, off_ring, off_scratch, off_inter, ws_bytes;
  size_t off_cp = 0, off_F = 0, off_Q = 0, off_red = 0;  // SSOCT_FLAG_PUPIL regions
  // Non-square frames other than 128 x 64 and 64 x 128: chirp table and frame buffer
  // of the two passes in sharpness.cu, which pair_queue takes as its scratch ring.
  bool generic = false;
  size_t off_cg = 0;
  // SSOCT_FLAG_AXIAL_FIRST: Eq. 5 + Eq. 7 first (half spectrum of the real
  // rescaled frames), then the lateral kernel on the planes
  bool axial_first = false;  // order of whole-volume reconstructions (the flag's, or the autotuner's choice)
  bool af_forced = false;    // created with SSOCT_FLAG_AXIAL_FIRST: every call runs that order
  bool af_option = false;    // the autotuner may pick the axial-first order (its planes fit the intermediate)
  size_t off_aplanes = 0;
  // tiled first pass (rescale_axial_tiled): strip records [nl][nx / 64] and the
  // staged columns per source row (0: the one-tile-per-CTA kernel instead)
  std::vector<StripTap> xstrip;
  size_t off_xstrip = 0;
  int ra_w = 0;
  char* ws = nullptr;
  int device = -1;
  int noalloc_device = -1;   // device of the plan's last no-allocation call (-1: none)
  int num_sms = 0;
  alignas(64) unsigned char tmap[128];        // CUtensorMap of the scratch ring (column bands)
  // frame ring state
  long long pushed = 0;     // frames in the current gate (capped at nl)
  int ring_head = 0;        // next ring slot to write
  long long next_seq = -1;
  long long stream_count = 0;  // frames pushed since the gate (re)started, uncapped
  long long lat_upto = -1;     // sliding gates: stream index up to which the intermediate holds holograms
  // cuts-only sliding gates: running one-bin transform X(z0) of the gate, valid
  // for the intermediate as it stood at lat_upto == xs_lat; xs_updates frames
  // have been swapped in since it was last summed in full
  size_t off_xys = 0;          // [wy][ntx * 32] complex
  bool xs_valid = false;
  int xs_z0 = 0;
  int xs_updates = 0;
  long long xs_lat = -1;
  std::string last_error;
  // failure injection (ssoct_inject_stall)
  unsigned inject_skip = 0;
  unsigned long long wait_ns = 0;
  // stage timing (ssoct_profile)
  bool profiling = false;
  std::vector<cudaEvent_t> events;  // 3 per recorded call: start, after its first stage, after its second
  std::vector<char> events_af;      // per recorded call: axial-first order (the axial stage is its first)
  size_t events_used = 0;
};

// Kernel launchers (defined in the .cu files).
cudaError_t launch_lateral(const Plan& p, const LateralParams& lp, cudaStream_t s);
cudaError_t launch_axial(const Plan& p, const AxialParams& ap, cudaStream_t s);
cudaError_t launch_cuts(const CutsParams& cp, cudaStream_t s);
// Device copy of a multiple of 16 bytes between 16-byte aligned addresses of the
// current device, and the frames that a push hands to it: memory of the plan's
// own device.  A copy call reaches more than a kernel does (another GPU's memory
// without peer access, and a stream of a device that is not current).
inline bool push_by_kernel(const cudaPointerAttributes& a, int device, int current, const void* frames) {
  return a.type == cudaMemoryTypeDevice && a.device == device && current == device && (uintptr_t)frames % 16 == 0;
}
cudaError_t launch_copy_frames(void* dst, const void* src, size_t bytes, cudaStream_t s);
// The three cuts of the current gate straight from the sweep-axis intermediate
// (xy: one bin per pixel; xz, yz: the axial transform of the cut's tiles).
// xy_state, if not NULL, receives the xy cut's complex X(z0) ([wy][ntx * 32]).
cudaError_t launch_gate_cuts(const Plan& p, int x0, int y0, int z0, float* xy, float* xz, float* yz,
                             float2* xy_state, cudaStream_t s);
// Running xy cut of the sliding gate (one bin of Eq. 7 is linear in the gate's
// holograms): X(z0) += sign * sum over slots slot0 .. slot0 + k - 1 (mod nl) of
// h_t exp(-2 pi i z0 t / nl), then xy = envelope of X if xy is not NULL.
cudaError_t launch_xy_slide(const Plan& p, int slot0, int k, int z0, float sign, float* xy, cudaStream_t s);
// Axial-first order, first pass: Eq. 5 resample of every frame and Eq. 7 over
// the sweep at every pixel, bins 0..nl/2 written as planes [nl/2 + 1][ny][nx].
cudaError_t launch_rescale_axial(const Plan& p, const uint16_t* frames, int ring_start, float2* planes,
                                 cudaStream_t s);
// The tiled first pass: sizes it is built for, and its dynamic shared memory
// for w staged columns per source row.
bool rescale_axial_tiled(int nx, int nl);
size_t rescale_axial_tile_smem(int nl, int w);
// Tensor map over a gate's frames seen as uint16 [nl * ny][nx], boxes of
// box_cols columns x 2 rows (zero fill outside the frame).
bool encode_frames_map(const Plan& p, const uint16_t* frames, int box_cols, void* map_out);
// Tensor map over the sweep-axis intermediate seen as float [rows][64] (one
// row = 32 complex values of one frame of a tile), boxes of box_complex
// complex values x 256 rows.
bool encode_inter_map(const float2* inter, long long rows, int box_complex, void* map_out);
// Tensor map over a volume float [nl][wy][wx] (wx a multiple of 4, vol 16-byte
// aligned), boxes of box_px pixels of one row x nl depth bins (at most 256), whose
// shared-memory rows of 64 bytes (box_px 16) are in the 64-byte swizzle.
bool encode_volume_map(float* vol, int wx, int wy, int nl, int box_px, void* map_out);
bool lateral_supported(int nx, int ny);
// Frames that one CTA or cluster transforms whole, without the work queue: the
// raw rows that a CTA's band takes (0: not such a plan), and whether the next
// launch goes that way.
int lateral_small_rows(const Plan& p);
bool lateral_small(const Plan& p);
// Sliding gates: the kernels that read the intermediate are ordinary launches
// where it does not fit in L2.  Placed beside the kernel before them (launch_next)
// the axial kernel took 28 us more at 1024 x 1024 x 256 and the kernels of a
// cuts-only gate 11 to 23 us more in all (plans in turn, 13 new frames); a gate of
// 256 x 256 x 128 takes 4 us less so.
inline bool gate_late(const Plan& p) {
  return sizeof(float2) * (size_t)p.wy * p.ntx * p.nl * kTile > (128u << 20);
}
bool axial_supported(int nl);
// Tensor-core axial kernel (axial_tc.cu): sweep lengths it handles, its DFT
// operand table, dynamic shared memory, and launcher.  err is the plan's error
// word; the kernel ORs kErrAxialTc into it when an MMA wait runs out.
bool axial_tc_supported(int nl);
void axial_tc_table(std::vector<unsigned short>& out);
size_t axial_tc_smem_bytes();
cudaError_t launch_axial_tc(const Plan& pl, const AxialParams& ap, const unsigned short* bmat, unsigned* err,
                            int num_sms, cudaStream_t s);
// Aberration path (sharpness.cu): sizes it compiles, the c P table, and the
// forward + adjoint launches that leave loss and gradient in the FP64 block at
// off_red ([0] S1, [1] S2, [2] loss, [3] dL/dz, [4..18] dL/dc_1..15, then the
// two coefficients of dL/dP, a block count of the kernels and, in [21], the
// path's error word).  The path's queue has counters of its own (off_sctr): its
// time-outs are the call's status, not ssoct_sync's, and an earlier call's error
// word stays for ssoct_sync.
constexpr int kShRedDoubles = 22;
constexpr int kShRedErr = 21;
bool sharpness_supported(int nx, int ny, int nl);
bool generic_lateral_supported(int nx, int ny);
// Eq. 5 + Eq. 6 as a row pass and a column pass through the frame buffer at
// off_F, for frames[(ring_start + t) mod nl]; writes the sweep-axis intermediate.
cudaError_t launch_lateral_generic(const Plan& pl, const uint16_t* frames, int ring_start, cudaStream_t s);
void build_pupil_table(int nx, int ny, double alpha, const double* coeffs, int ncoeffs, std::vector<float2>& out);
// exp(i pi k / 128), k = 0 .. 255, as pairs of floats (re hi, re lo, im hi, im lo).
void pupil_cis_table(std::vector<float4>& out);
// have_inter: the sweep-axis intermediate already holds the holograms of the frames,
// from the queue with the counters at off_sctr.
cudaError_t launch_sharpness(const Plan& pl, const uint16_t* frames, float* vol, bool have_inter, cudaStream_t s);
cudaError_t launch_pupil_table(const Plan& pl, cudaStream_t s);
// Dynamic shared memory of the lateral kernel for a plan (bytes).
size_t lateral_smem_bytes(const Plan& p);
// The lateral kernel's instances in units of their own: square frames of 640 and
// more; non-square frames by width (paper order); square frames with the table
// lp.cp for the chirp (aberration path).
cudaError_t launch_lateral_large(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms, cudaStream_t s);
cudaError_t launch_lateral_pairs_256(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms, cudaStream_t s);
cudaError_t launch_lateral_pairs_512(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms, cudaStream_t s);
cudaError_t launch_lateral_pairs_1024(const Plan& p, const LateralParams& lp, const void* tmap, int num_sms, cudaStream_t s);
cudaError_t launch_lateral_pair(const Plan& p, const LateralParams& lp, int num_sms, cudaStream_t s);
bool lateral_pupil_supported(int nx, int ny);
cudaError_t launch_lateral_pupil(const Plan& p, const LateralParams& lp, int num_sms, cudaStream_t s);
// Columns per column item of the lateral kernel for a column length ny.
int lateral_col_band(int ny);

// Used by the no-allocation entry point (noalloc.cu): the plan behind a handle,
// a scratch-ring tensor map for `slots` slots at an arbitrary device address,
// and a lateral launch that takes the tensor map and SM count explicitly.
Plan& plan_of(ssoct_plan h);
bool encode_scratch_map_at(const Plan& p, void* scratch_dev, int slots, void* map_out);
cudaError_t launch_lateral_with(const Plan& p, const LateralParams& lp, const void* tmap,
                                int num_sms, cudaStream_t s);
// The axial launch with the SM count given explicitly (the persistent streaming
// form sizes its grid by it); launch_axial passes the plan's own.
cudaError_t launch_axial_with(const Plan& p, const AxialParams& ap, int num_sms, cudaStream_t s);
// Error word of the last no-allocation call made with this plan (0 if none, or
// if that call's kernels met no time-out); read after the caller's stream sync.
cudaError_t noalloc_error_word(Plan& p, unsigned* err);
// Runs the paper's order for one call on a plan whose axial-first order was
// only the autotuner's choice (sliding gates and the no-allocation path keep
// the paper's order); restores the plan's order when it goes out of scope.
struct PaperOrderScope {
  Plan& p;
  bool saved;
  explicit PaperOrderScope(Plan& pl) : p(pl), saved(pl.axial_first) {
    if (!p.af_forced) p.axial_first = false;
  }
  ~PaperOrderScope() { p.axial_first = saved; }
};

// Whole-frame window: the lateral kernel then needs no window bounds checks.
inline bool lateral_full_window(const Plan& p) { return p.x0 == 0 && p.y0 == 0 && p.wx == p.nx && p.wy == p.ny; }

}  // namespace ssoct
