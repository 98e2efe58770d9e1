// The selection minor loop's device code (minor_select.cu) on the CPU: a host
// thread a CUDA thread, so that ThreadSanitizer sees the accesses to a block's
// shared memory and to the tile's arrays.  Only __syncthreads and the group's
// release/acquire words order them: warp collectives exchange values, nothing
// else.  A barrier that threads reach from different lines, or that some never
// reach, ends the run.  test_select_emulated.py writes select_device.inc (the
// device code with its PTX loads spelt out) and drives this.
#include <sched.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <cfenv>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda.h>
#include <cuda_runtime.h>
#undef __device__
#undef __global__
#undef __host__
#undef __shared__
#undef __forceinline__
#undef __noinline__
#undef __launch_bounds__
#define __device__
#define __global__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __restrict__
#define __syncthreads() emu_syncthreads(__LINE__)

extern "C" __attribute__((weak)) void AnnotateIgnoreSyncBegin(const char*, int);
extern "C" __attribute__((weak)) void AnnotateIgnoreSyncEnd(const char*, int);

struct Warp {
  std::atomic<uint32_t> slot[2][32] = {};
  std::atomic<int> arrived{0}, gen{0};
};
struct Cta {
  int threads = 0, arrived = 0, line = 0;
  long gen = 0;
  std::mutex m;
  std::condition_variable cv;
  std::vector<Warp> warps;
  std::vector<uint4> smem;
};
static thread_local Cta* cta;
static thread_local unsigned char* sel_smem;
static thread_local dim3 threadIdx(0, 0, 0), blockIdx(0, 0, 0), blockDim(1, 1, 1);
static thread_local int warp_turn;

static void emu_syncthreads(int line) {
  std::unique_lock<std::mutex> l(cta->m);
  if (cta->arrived++ == 0) cta->line = line;
  bool ok = cta->line == line;
  if (ok && cta->arrived == cta->threads) {
    cta->arrived = 0;
    ++cta->gen;
    cta->cv.notify_all();
  } else if (ok) {
    const long g = cta->gen;
    ok = cta->cv.wait_for(l, std::chrono::seconds(60), [&] { return cta->gen != g; });
  }
  if (!ok) {
    std::fprintf(stderr, "barrier divergence: line %d, others at %d\n", line, cta->line);
    _exit(3);
  }
}

// every lane's value, in lane order
static void exchange(unsigned mask, uint32_t v, uint32_t (&all)[32]) {
  if (mask != 0xffffffffu) _exit(4);
  if (AnnotateIgnoreSyncBegin) AnnotateIgnoreSyncBegin(__FILE__, __LINE__);
  Warp& w = cta->warps[threadIdx.x >> 5];
  auto& slot = w.slot[warp_turn ^= 1];
  slot[threadIdx.x & 31] = v;
  const int g = w.gen;
  if (w.arrived.fetch_add(1) == 31) {
    w.arrived = 0;
    ++w.gen;
  } else {
    while (w.gen == g) sched_yield();
  }
  for (int i = 0; i < 32; ++i) all[i] = slot[i];
  if (AnnotateIgnoreSyncEnd) AnnotateIgnoreSyncEnd(__FILE__, __LINE__);
}
static void __syncwarp() {  // (one that does order memory)
  Warp& w = cta->warps[threadIdx.x >> 5];
  const int g = w.gen.load();
  if (w.arrived.fetch_add(1) == 31) {
    w.arrived = 0;
    ++w.gen;
  } else {
    while (w.gen.load() == g) sched_yield();
  }
}
template <class To, class From>
static To bits(From v) {
  static_assert(sizeof(To) == sizeof(From), "");
  To t;
  std::memcpy(&t, &v, sizeof(t));
  return t;
}
static uint32_t __float_as_uint(float v) { return bits<uint32_t>(v); }
static int __float_as_int(float v) { return bits<int>(v); }
static float __uint_as_float(uint32_t v) { return bits<float>(v); }
static float __int_as_float(int v) { return bits<float>(v); }
template <class T>
static T __reduce_max_sync(unsigned m, T v) {
  uint32_t a[32];
  exchange(m, (uint32_t)v, a);
  for (uint32_t o : a) v = std::max(v, (T)o);
  return v;
}
static unsigned __reduce_min_sync(unsigned m, unsigned v) {
  uint32_t a[32];
  exchange(m, v, a);
  return *std::min_element(a, a + 32);
}
static uint32_t __ballot_sync(unsigned m, bool p) {
  uint32_t a[32], b = 0;
  exchange(m, p, a);
  for (int i = 0; i < 32; ++i) b |= a[i] << i;
  return b;
}
template <class T>
static T __shfl_sync(unsigned m, T v, int lane) {
  uint32_t a[32];
  exchange(m, bits<uint32_t>(v), a);
  return bits<T>(a[lane & 31]);
}
template <class T>
static T __shfl_xor_sync(unsigned m, T v, int o) {
  return __shfl_sync(m, v, (int)(threadIdx.x & 31) ^ o);
}
template <class T>
static T __shfl_up_sync(unsigned m, T v, int o) {
  const int l = threadIdx.x & 31;
  return __shfl_sync(m, v, l < o ? l : l - o);
}
template <class F>
__attribute__((noinline)) static float upward(F f) {
  std::fesetround(FE_UPWARD);
  volatile float r = f();
  std::fesetround(FE_TONEAREST);
  return r;
}
static float __fadd_ru(volatile float a, volatile float b) { return upward([&] { return a + b; }); }
static float __fsub_ru(volatile float a, volatile float b) { return upward([&] { return a - b; }); }
static float __fmaf_ru(volatile float a, volatile float b, volatile float c) {
  return upward([&] { return std::fmaf(a, b, c); });
}
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static int __popc(uint32_t v) { return __builtin_popcount(v); }
static uint32_t __byte_perm(uint32_t x, uint32_t y, uint32_t s) {
  const uint64_t v = ((uint64_t)y << 32) | x;
  uint32_t r = 0;
  for (int i = 0; i < 4; ++i) r |= (uint32_t)(v >> (8 * ((s >> (4 * i)) & 7)) & 0xff) << (8 * i);
  return r;
}
template <class T>
static T __ldg(const T* p) { return *p; }
template <class T>
static T __ldcg(const T* p) { return *p; }
template <class T, class V>
static void __stcg(T* p, V v) { *p = v; }
static int atomicAdd(int* p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_RELAXED); }
static uint32_t atomicAdd(uint32_t* p, uint32_t v) {  // (with the fence before it)
  return __atomic_fetch_add(p, v, __ATOMIC_ACQ_REL);
}
static int atomicOr(int* p, int v) { return __atomic_fetch_or(p, v, __ATOMIC_RELAXED); }
static void atomicMax(unsigned long long* p, unsigned long long v) {
  unsigned long long o = __atomic_load_n(p, __ATOMIC_RELAXED);
  while (o < v && !__atomic_compare_exchange_n(p, &o, v, false, __ATOMIC_RELAXED, __ATOMIC_RELAXED)) {
  }
}
static void __threadfence() {}
template <class T>
static T relaxed_load(T* p) {
  T v;
  __atomic_load(p, &v, __ATOMIC_RELAXED);
  return v;
}
static void __nanosleep(unsigned) { sched_yield(); }
static long long clock64() { return std::chrono::steady_clock::now().time_since_epoch().count(); }
using std::max;
using std::min;

#include "cleangb_internal.cuh"
namespace cleangb {
namespace ptx {
static float ld_nc(const float* p) { return *p; }
static uint64_t globaltimer_ns() {
  return std::chrono::steady_clock::now().time_since_epoch() / std::chrono::nanoseconds(1);
}
}  // namespace ptx
}  // namespace cleangb
#include "select_device.inc"

using namespace cleangb;

// `blocks` at once of `threads` each, run(block) by every thread
static void launch(int blocks, int threads, size_t smem, const std::function<void(int)>& run) {
  std::vector<std::unique_ptr<Cta>> ctas;
  std::vector<std::thread> ts;
  for (int b = 0; b < blocks; ++b) {
    ctas.emplace_back(new Cta);
    Cta* c = ctas.back().get();
    c->threads = threads;
    c->warps = std::vector<Warp>((threads + 31) / 32);
    c->smem.assign(smem / sizeof(uint4) + 1, make_uint4(~0u, ~0u, ~0u, ~0u));
    for (int t = 0; t < threads; ++t)
      ts.emplace_back([=, &run] {
        cta = c;
        sel_smem = reinterpret_cast<unsigned char*>(c->smem.data());
        threadIdx.x = t;
        blockDim.x = threads;
        run(b);
      });
  }
  for (auto& t : ts) t.join();
}

int main(int argc, char** argv) {
  // ny nx psf_ny psf_nx tiles_y tiles_x G force_timeout, niter, gain threshold
  // plain_cycles; dirty; PSF
  std::FILE* f = std::fopen(argv[1], "rb");
  int32_t n[8];
  int64_t niter;
  float gt[3];
  if (argc < 3 || !f || std::fread(n, 4, 8, f) != 8 || std::fread(&niter, 8, 1, f) != 1 ||
      std::fread(gt, 4, 3, f) != 3)
    return 2;
  PlanDev d{};
  d.ny = n[0], d.nx = n[1], d.pny = n[2], d.pnx = n[3], d.ty = n[4], d.tx = n[5];
  const int G = n[6];
  d.cy = d.pny / 2, d.cx = d.pnx / 2, d.T = d.ty * d.tx;
  d.gain = gt[0], d.thr = gt[1];
  d.cap_round = (int)(niter / d.T + 1);
  std::vector<float> R((size_t)d.ny * d.nx), P((size_t)d.pny * d.pnx), model(R.size());
  if (std::fread(R.data(), 4, R.size(), f) != R.size() ||
      std::fread(P.data(), 4, P.size(), f) != P.size())
    return 2;
  std::fclose(f);
  std::vector<int64_t> budget(d.T);
  std::vector<uint64_t> peak(2 * d.T);
  std::vector<int32_t> rcount(d.T), rapplied(d.T);
  std::vector<clean_component> rcomps((size_t)d.T * d.cap_round);
  int maxH = 0, maxW = 0;
  for (int t = 0; t < d.T; ++t) {
    const Rect r = tile_rect(t, d.ny, d.nx, d.ty, d.tx);
    maxH = std::max(maxH, r.y1 - r.y0);
    maxW = std::max(maxW, r.x1 - r.x0);
    budget[t] = niter / d.T + (t < niter % d.T ? 1 : 0);
    float a = -1.f;
    for (int y = r.y0; y < r.y1; ++y)
      for (int x = r.x0; x < r.x1; ++x) {
        const float v = R[(size_t)y * d.nx + x];
        if (std::fabs(v) > a) {
          a = std::fabs(v);
          peak[t] = make_key(v, y * d.nx + x);
        }
      }
  }
  DevState st{};
  SelSizes z;
  if (!select_geometry(&d.sel, d.ny, d.nx, d.ty, d.tx, &z)) return 2;
  std::vector<char> u(z.cells, (char)0xff), masks(z.cells, (char)0), boxes(z.boxes), h8(z.h8),
      hb(std::max<size_t>(z.hb, 4)), lobe(z.lobe), ctl(z.ctl, (char)0);
  d.R = R.data(), d.P = P.data(), d.model = model.data(), d.budget = budget.data();
  d.peak = peak.data(), d.rcount = rcount.data(), d.rapplied = rapplied.data();
  d.rcomps = rcomps.data(), d.st = &st;
  d.sel.u = (float2*)u.data(), d.sel.masks = (uint2*)masks.data(), d.sel.ctl = (SelCtl*)ctl.data();
  d.sel.h8 = (uint32_t*)h8.data(), d.sel.hb = (uint32_t*)hb.data(), d.sel.lobe = (uint32_t*)lobe.data();
  d.sel.plain_cycles = gt[2];
  d.sel.inside = d.cy >= maxH - 1 && d.pny - d.cy >= maxH && d.cx >= maxW - 1 && d.pnx - d.cx >= maxW;

  // the PSF's tables (select_build_psf)
  const SelDev& g = d.sel;
  const int rows8 = 2 * g.oy8 + 2, cols8 = 2 * g.ox8 + 2, rows = rows8 - 1, cols = cols8 - 1;
  float2* b8 = (float2*)boxes.data();
  float2* tmp = b8 + (size_t)rows8 * cols8;
  launch(1, 32, 0, [&](int) {
    for (int b = 0; b < rows8 * ((cols8 + 3) / 4); ++b) {
      blockIdx.x = b;
      psf_box_kernel(d, b8, rows8, cols8);
    }
  });
  launch(1, 1, 0, [&](int) {
    for (int q = 0; q < rows8 * cols; ++q) {
      blockIdx.x = q;
      psf_window_kernel(b8, cols8, g.oy8, g.ox8, (uint32_t*)h8.data(), rows, cols);
      if (g.lq) psf_window_x_kernel(b8, rows8, cols8, tmp, cols, 1 << g.lq);
      if (q < 64 * 64) psf_lobe_kernel(d, (uint32_t*)lobe.data());
    }
    for (int q = rows8 * cols; q < 64 * 64; ++q) {
      blockIdx.x = q;
      psf_lobe_kernel(d, (uint32_t*)lobe.data());
    }
    for (int q = 0; g.lq && q < rows * cols; ++q) {
      blockIdx.x = q;
      psf_window_y_kernel(tmp, rows8, cols, (uint32_t*)hb.data(), rows, 1 << g.lq);
    }
  });
  const uint64_t limit = n[7] ? 200000000ull : 60000000000ull;
  for (int t = 0; t < d.T; ++t)
    launch(G, kThreads, z.smem, [&](int rank) {
      blockIdx.x = rank;
      if (g.lq == 0)
        select_body<true>(d, G, 0, 1, limit, n[7], t, rank);
      else
        select_body<false>(d, G, 0, 1, limit, n[7], t, rank);
    });
  f = std::fopen(argv[2], "wb");
  if (!f || st.status)  // (a timeout: its tile in the upper word)
    return st.status == ST_TIMEOUT && st.timeout_where >> 32 == 0 && d.sel.ctl[0].hand_key == 0 ? 5 : 6;
  std::fwrite(R.data(), 4, R.size(), f);
  std::fwrite(model.data(), 4, model.size(), f);
  for (int t = 0; t < d.T; ++t) {
    std::fwrite(&rcount[t], 4, 1, f);
    std::fwrite(&d.sel.ctl[t].hand_key, 8, 1, f);
    std::fwrite(&rcomps[(size_t)t * d.cap_round], sizeof(clean_component), rcount[t], f);
  }
  std::fclose(f);
  return 0;
}
