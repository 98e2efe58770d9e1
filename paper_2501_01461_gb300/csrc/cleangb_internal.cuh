// Internal declarations shared by the kernels and the C-ABI host code of
// libcleangb.so.  Nothing here is part of the public ABI (include/cleangb.h).
#pragma once

#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "cleangb.h"

namespace cleangb {

// ---------------------------------------------------------------------------
// Peak keys.  The peak search of Section 3 (first equation) picks the pixel
// of largest |R|, ties to the lowest row-major index.  A pixel is encoded as
// a 64-bit key whose unsigned order is exactly that order:
//   bits 63..32  bit pattern of |R| (monotone in |R| for non-negative floats)
//   bits 31..1   0x7fffffff - index (larger for lower indices)
//   bit  0       sign bit of R, so the signed value is recovered exactly
// Key 0 means "no pixel".  Requires index < 2^31 - 1.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint64_t make_key(float v, int32_t idx) {
  uint32_t bits;
#ifdef __CUDA_ARCH__
  bits = __float_as_uint(v);
#else
  __builtin_memcpy(&bits, &v, 4);
#endif
  uint32_t hi = bits & 0x7fffffffu;
  uint32_t lo = ((0x7fffffffu - (uint32_t)idx) << 1) | (bits >> 31);
  return ((uint64_t)hi << 32) | lo;
}
__host__ __device__ __forceinline__ int32_t key_index(uint64_t k) {
  return (int32_t)(0x7fffffffu - ((uint32_t)k >> 1));
}
__device__ __forceinline__ float key_value(uint64_t k) {
  uint32_t hi = (uint32_t)(k >> 32);
  return __uint_as_float(hi | ((uint32_t)(k & 1u) << 31));
}
__device__ __forceinline__ float key_abs(uint64_t k) {
  return __uint_as_float((uint32_t)(k >> 32));
}

// Tile bounds: tile (i, j) covers rows [floor(i ny / Ty), floor((i+1) ny / Ty))
// and columns likewise (Section 2, Fig. 1; the split of a non-divisible size
// is this library's reading).
struct Rect {
  int32_t y0, y1, x0, x1;
};
__host__ __device__ __forceinline__ Rect tile_rect(int32_t t, int32_t ny,
                                                   int32_t nx, int32_t ty,
                                                   int32_t tx) {
  int32_t i = t / tx, j = t - (t / tx) * tx;
  Rect r;
  r.y0 = (int32_t)(((int64_t)i * ny) / ty);
  r.y1 = (int32_t)(((int64_t)(i + 1) * ny) / ty);
  r.x0 = (int32_t)(((int64_t)j * nx) / tx);
  r.x1 = (int32_t)(((int64_t)(j + 1) * nx) / tx);
  return r;
}

// Status bits (DevState::status).  Sticky for the run.
enum : int32_t {
  ST_NONFINITE_DIRTY = 1,
  ST_NONFINITE_PSF = 2,
  ST_PSF_OFFCENTRE = 4,
  ST_TIMEOUT = 8,
};

// Device-resident control block of a plan.
struct DevState {
  int32_t status;        // ST_* bits
  int32_t active;        // a tile can run in the next round
  uint32_t fb_done;      // feedback blocks finished (last-block pattern)
  int32_t handed;        // the only round's tile waits for the plain loop (see kSelReport)
  int64_t total;         // components in the list
  int64_t n_rounds;      // rounds recorded (>= 1 component)
  int64_t round_comps;   // components of the last closed round
  int64_t max_budget;    // max over tiles of the remaining budget
  int64_t timeout_where; // diagnostic: tile * 2^32 + barrier index of a timeout
  float level;           // flux-trigger level of the next round (0: none)
  int32_t taken_over;   // tiles' rounds that the plain loop took over from the selection
};

// Selection minor loop (minor_select.cu): components a selection may leave
// pending, the control words of a tile's group, and a plan's tables.
constexpr int kSelPending = 64;
// launch_select's flags: leave no component pending; report a hand-over in
// DevState::handed, for a caller that launches the plain loop only then
enum { kSelFlush = 1, kSelReport = 2 };
struct SelCtl {
  unsigned long long key[2];  // peak key of a pass, by the pass's parity
  int64_t k;                  // the posted selection: components of the round so far
  int32_t done;               // the round is over for the tile
  uint32_t cmd, arrived;      // selections posted, CTAs that finished a pass (see
                              // minor_select.cu)
  uint32_t phases;            // passes of the tile so far in this run
  float near;                 // the tile's resolve margin
  int32_t slow;               // selections running that the plain loop would have beaten
  unsigned long long hand_key;  // the peak from which the plain loop takes the round on (0: none)
};
struct SelDev {
  float2* u;            // [T][cell_stride] bounds of R and -R per 8 x 8 cell
  uint2* masks;         // [T][cell_stride] the cells' pixels that are candidates
  const uint32_t* h8;   // PSF range over the windows a cell can meet, by the
                        // cells from the peak's to it (two bf16, see pack_rises)
  const uint32_t* hb;   // the same for a superblock of (1 << lq)^2 cells, by its first
  const uint32_t* lobe; // exact ranges of the 8 x 8 cells around a peak
  SelCtl* ctl;          // [T]
  int64_t cell_stride;  // cells of the largest tile (rows of `pitch`)
  int32_t lq, pitch;
  int32_t oy8, ox8, w8; // h8 and hb: entry of offset 0, row length
  int32_t inside;       // the PSF array holds every offset between two pixels of a tile
  int32_t* handed;      // tiles handed over in the launch (batches; null: not counted)
  float plain_cycles;   // what the launch behind the selection needs for an iteration
                        // (0: no such launch, the selection takes the whole round)
};
struct SelSizes {
  size_t cells, boxes, h8, hb, lobe, ctl;  // bytes
  int smem;                          // dynamic shared memory of the launch
};

// Pointers and sizes every kernel of a plan sees.
struct PlanDev {
  float* R;                 // residual, ny x nx
  float* model;             // model image, ny x nx
  const float* P;           // PSF, pny x pnx
  int32_t ny, nx, pny, pnx, cy, cx;
  int32_t ty, tx, T;        // tile grid and tile count
  float gain, thr;
  int32_t K;                // feedback interval (0 = none)
  float trigger;            // flux trigger (0 = none)
  int32_t cap_round;        // per-tile capacity of the round buffer
  int32_t round0;           // batched runs: the batch round at which this image started
  int64_t* budget;          // [T] remaining iterations per tile
  uint64_t* peak;           // [2][T] peak key per tile, indexed by round parity
  int32_t* rcount;          // [T] components of the current round per tile
  int32_t* rapplied;        // [T] how many of them their own tile's R has had
                            // subtracted (the feedback subtracts the rest)
  clean_component* rcomps;  // [T][cap_round] current round's components
  clean_component* list;    // [niter] all components, list order
  int64_t* round_off;       // [niter + 1] list offset of each recorded round
  uint64_t* gkeys;          // [2][T * G] per-CTA partial keys (grid sync)
  uint32_t* gbar;           // [T] grid-barrier exchanges done per tile in this run
  DevState* st;
  SelDev sel;               // selection minor loop (sel.u null: not in use)
};

// A batched work item: tile `tile` of image `image`.
struct BatchItem {
  int32_t image;
  int32_t tile;
};

// Per-image geometry of a batched feedback launch.
struct BatchImage {
  int32_t block0;    // first flattened block of this image
  int32_t bx, by;    // blocks per tile in x and y
  int32_t nblocks;   // bx * by * T
};

// Minor-loop launch configuration.
struct MinorCfg {
  int32_t G;          // CTAs per tile
  int32_t sync;       // CLEAN_SYNC_CLUSTER or CLEAN_SYNC_GRID
  int32_t resident;   // 1: residual rows live in shared memory for the round
  int32_t threads;    // threads per CTA
  int32_t smem;       // dynamic shared memory bytes
  int64_t spin_limit_ns;
  int32_t force_timeout;
  // bulk-copy pipeline (pipe = 1): rows stream through a ring of `stages`
  // shared-memory buffers, `chunk_rows` rows per buffer
  int32_t pipe;
  int32_t chunk_w;    // columns per chunk (multiple of 4, <= 128)
  int32_t chunk_h;    // rows per chunk
  int32_t box_w;      // TMA box width in floats (chunk_w + 4)
  int32_t stages;
  int32_t res_floats; // resident slab floats (0 when streamed)
  int32_t tmem;       // 1: each CTA's leading full chunks keep their residual
                      // in tensor memory for the launch (streamed pipeline)
  int32_t pair;       // 1: groups of 2G CTAs serve pairs of tiles, alternating
                      // between them (streamed pipeline, grid groups, T even)
  int32_t takeover;   // 1: only tiles that the selection ahead handed over, from
                      // there on (plain loads)
};

// Pipeline geometry and shared-memory size for a minor-loop configuration
// (fills the pipe fields of c; returns false if it does not fit).
// chunk_px: target pixels per chunk (0: 4096); max_stages: ring depth cap
// (0: 8).
bool minor_pipe_geometry(MinorCfg& c, int max_rows, int max_w, int chunk_px = 0,
                         int max_stages = 0);

// Raises a kernel's dynamic shared-memory cap to the device's opt-in maximum.
// The cap is process-wide state of the kernel, so every plan sets the same
// value (setting a plan's own size would break launches of plans that need
// more); each launch still requests only its own size.
inline cudaError_t allow_max_smem(const void* fn) {
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, fn);  // static shared memory counts too
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - (int)fa.sharedSizeBytes);
  return e;
}

// Launchers (return cudaError_t of the launch).
cudaError_t launch_init(const PlanDev& d, const float* dirty, int64_t niter,
                        cudaStream_t s);
cudaError_t launch_validate_psf(const PlanDev& d, cudaStream_t s);
// Flux-trigger level of a run's first round (after launch_init); no-op
// without a trigger.
cudaError_t launch_first_level(const PlanDev& d, cudaStream_t s);
// Whether rounds of this plan end with a feedback.
__host__ __device__ __forceinline__ bool feedback_on(const PlanDev& d) {
  return (d.K > 0 || d.trigger > 0.f) && d.T > 1;
}
// Rounds of several selections, which the plain loop may take over in groups that
// hold their tile in shared memory.  An idle launch costs 10 us: not for rounds that
// a flux trigger ends (3 %), nor for runs of a few selections.  (A plan whose run is
// one round of one tile launches the plain loop only when it has to.)
inline bool takeover_possible(const PlanDev& d, int64_t niter) {
  if (niter / d.T < 256) return false;
  return d.T == 1 ? d.K == 0 || d.K > kSelPending : d.K > kSelPending && !(d.trigger > 0.f);
}
// r_map / p_map: 2-D tensor maps of the residual and the PSF with the box
// (c.box_w x c.chunk_h) of a pipelined configuration (ignored otherwise).
cudaError_t launch_minor(const PlanDev& d, const MinorCfg& c, int parity,
                         const CUtensorMap* r_map, const CUtensorMap* p_map, cudaStream_t s);
// Encodes a 2-D float32 tensor map (rows x cols, row pitch cols floats) with
// the given box; false if the base or pitch is not 16-byte aligned.
bool make_box_tensor_map(CUtensorMap* map, const float* base, int rows, int cols, int box_w,
                         int box_h);
bool encode_tensor_map_2d(CUtensorMap* map, const float* base, int rows, int cols, int box_w,
                          int box_h);
cudaError_t minor_prepare(const MinorCfg& c);  // sets function attributes
// SM cycles of an iteration with plain loads and resident rows, for a tile of h x w
// pixels on the group of c.
float minor_plain_cycles(const MinorCfg& c, int h, int w);
// ---- selection minor loop (minor_select.cu) -----------------------------------
// Table geometry and buffer sizes for an image's tiling; false if a tile is
// too large for the packed positions.
bool select_geometry(SelDev* g, int ny, int nx, int ty, int tx, SelSizes* z);
// The PSF's range tables (after every PSF change); boxes: work area.
cudaError_t select_build_psf(const PlanDev& d, float2* boxes, uint32_t* h8, uint32_t* hb,
                             uint32_t* lobe, cudaStream_t s);
cudaError_t select_prepare();  // kernel attributes
// One round's minor loops, G CTAs a tile (G > 1: a cooperative launch).
cudaError_t launch_select(const PlanDev& d, int G, int smem, int parity, int flags, uint64_t limit_ns,
                          int force_timeout, cudaStream_t s);
// G CTAs per (image, tile) item (G > 1: a cooperative launch, every CTA on an SM of
// its own); direct: tiles without superblocks (SelDev::lq 0).
cudaError_t launch_select_batch(const PlanDev* plans, const BatchItem* items, int n_items,
                                int direct, int G, int smem, int round, uint64_t limit_ns,
                                cudaStream_t s);

// G CTAs per item (G = 1: independent CTAs; G > 1: one thread-block cluster
// per item), each reading its image's plan state from `plans` (device
// arrays); resident: each CTA's rows fit `smem` bytes of shared memory.
// Image i runs its round (round - plans[i].round0).
// takeover: as in MinorCfg.
cudaError_t launch_minor_batch(const PlanDev* plans, const BatchItem* items, int n_items,
                               int G, int resident, int smem, int takeover, int round,
                               cudaStream_t s);
// Clusters of G CTAs of the batched kernel that the device runs at once.
int minor_batch_clusters(int G, int resident, int smem);

// Feedback for many images in one launch (plain loads, or TMA when maps is
// non-NULL: one PSF tensor map per image in device memory, 64-byte aligned).
cudaError_t launch_feedback_batch(const PlanDev* plans, const BatchImage* imgs, int n_images,
                                  int total_blocks, int max_T, const CUtensorMap* maps,
                                  int round, int apply, uint64_t limit_ns, cudaStream_t s);
// Feedback block grid of one image (blocks per tile in x and y).
void feedback_blocks(const PlanDev& d, bool tma, int* bx, int* by);
int minor_max_cluster_ctas(int G, int resident, int smem, int threads);
// psf_map: a 2-D tensor map of the PSF (box 132 x 32 floats) selects the TMA
// kernel; NULL selects the plain-load kernel.
cudaError_t launch_feedback(const PlanDev& d, const CUtensorMap* psf_map, int parity,
                            int apply, uint64_t limit_ns, cudaStream_t s);
cudaError_t feedback_prepare(int T);
// ---- FFT feedback (fft_feedback.cu) -----------------------------------------
// One axis of the 2-D transforms: length L (even, 7-smooth, <= kFftMaxL),
// its radices in stage order and the threads of a block that transforms it
// (every thread holds at most kFftValsPerThread values in a stage).
constexpr int kFftMaxL = 8192;
constexpr int kFftMaxThreads = 512;
constexpr int kFftMaxRadices = 16;
constexpr int kFftValsPerThread = 16;
struct FftAxis {
  int32_t L, nthr, nrad;
  int32_t rad[kFftMaxRadices];
  // twiddle table: entries [0, L) hold exp(-2 pi i t / L); stage s (radix R,
  // Ns = product of the earlier radices) reads exp(-2 pi i r k / (Ns R)) at
  // tw_off[s] + r Ns + k, so neighbouring lanes read neighbouring entries
  int32_t tw_off[kFftMaxRadices];
  int32_t tw_len;
  int32_t p2;  // 1: L is 2048, 4096 or 8192 and takes the radix-16 path (L / 16 threads)
};
// Smallest even n >= m whose prime factors are 2, 3, 5 and 7.
int fft_grid_size(int m);
// Fills *a for length L; false if L is odd, above kFftMaxL or not 7-smooth.
bool fft_axis_init(FftAxis* a, int L);
// The twiddle table of an axis (a.tw_len float2, layout in FftAxis),
// computed in double precision on the host and copied to d_tw; synchronises s.
cudaError_t fft_make_twiddles(float2* d_tw, const FftAxis& a, cudaStream_t s);
// Bytes of the per-round component work area for up to n_max components.
size_t fft_comps_bytes(int64_t n_max);
// Kernel spectrum Kspec[k][m] (k <= Lx / 2, m < Ly) of the PSF kernel image
// K[d mod L] = P[d + c] (|d| < image size), scaled by 1 / (Ly Lx).
cudaError_t fft_build_psf_spectrum(const PlanDev& d, const FftAxis& ay, const FftAxis& ax,
                                   const float2* twy, const float2* twx, float2* Kspec,
                                   cudaStream_t s);
// One FFT feedback: R <- R0 - (round components (*) PSF) on every pixel,
// R0 <- R, next peaks, round close.  Y: (Lx/2 + 1) x (ny rounded up to
// even) float2 work area;
// comps: fft_comps_bytes(T cap_round) bytes of work area.
cudaError_t fft_feedback_round(const PlanDev& d, const FftAxis& ay, const FftAxis& ax,
                               const float2* twy, const float2* twx, const float2* Kspec,
                               float2* Y, int4* comps, float* R0, int parity, cudaStream_t s);
cudaError_t fft_prepare();  // kernel attributes of the FFT feedback
// Encodes the PSF tensor map for the TMA feedback kernel; false if the PSF's
// address or row pitch is not 16-byte aligned (or the driver lacks TMA).
bool make_psf_tensor_map(CUtensorMap* map, const float* psf, int pny, int pnx);
cudaError_t launch_restore_with(const PlanDev& d, float bmaj, float bmin, float bpa,
                                float* beam_buf, int r, float* out, cudaStream_t s);
int minor_threads();

// Accessors the batch code uses on single-image plans (defined with the C ABI).
PlanDev plan_device_state(const clean_plan_s* pl);
bool plan_psf_tensor_map(const clean_plan_s* pl, CUtensorMap* out);
int64_t plan_niter(const clean_plan_s* pl);
// Dynamic shared memory of the plan's selection minor loop (0: not possible).
int plan_select_smem(const clean_plan_s* pl);
// FFT feedback of a plan on the state `d` (a batch job's copy of the plan's
// device state, with its own control block and round phase).
bool plan_uses_fft(const clean_plan_s* pl);
cudaError_t plan_fft_start(clean_plan_s* pl, const PlanDev& d, cudaStream_t s);
cudaError_t plan_fft_round(clean_plan_s* pl, const PlanDev& d, int parity, cudaStream_t s);

}  // namespace cleangb
