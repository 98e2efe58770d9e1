// Minor loop by selection: the same components as the iteration-by-iteration
// loop of minor_loop.cu, found on the few pixels that can become the peak.
//
// The plain loop subtracts every component from the whole tile to find the
// next peak, so each iteration costs a pass over the tile and an exchange
// between its CTAs.  Here one CTA per tile keeps the exact values of the
// largest pixels (the candidates, in registers) and, for every 8 x 8 cell of
// the tile, upper bounds of R and of -R over its other pixels.  An iteration
//   1. takes the largest candidate (ties: the lowest index) if no bound
//      reaches it, records the component f = gain * v,
//   2. subtracts f * PSF from the candidates (the same rounded multiply and
//      subtract the pixel gets in the plain loop), and
//   3. raises the bounds by the largest |change| that f * PSF can make in
//      each cell, from a table of the PSF's range over 16 x 16 windows.
// A bound that reaches the best candidate sends its cell to be resolved: its
// 64 pixels are read and every component picked since the last pass is
// subtracted from them in order, which gives their exact values; those near
// the peak join the candidates, the rest give the cell its exact bounds.
// Every pixel thus sees the same operations in the same order as in the plain
// loop, so positions, fluxes and residual are bit for bit the same.
//
// Components picked this way are pending: the feedback launch subtracts a
// tile's own pending components ahead of the other tiles' (the order in which
// the plain loop would have), so a round of K iterations reads and writes the
// residual once, in the feedback.  When a round has more iterations than one
// selection holds (kPending), or the candidates' registers run full, the
// tile's CTAs apply the pending components to the residual, rebuild the cells
// and select again.
//
// Bounds are sound in float32: sums are rounded up, and each step adds
// 2^-22 (|v| + |f P_c|) for a pixel's own two roundings (v the peak, P_c the
// PSF's centre: |R| <= |v| and |PSF| <= P_c, so the product and the difference
// are off by at most 2^-24 |f P_c| and 2^-24 (|v| + |f P_c|)).
//
// Bounds come in two levels so that an iteration touches few of them: a
// superblock of Q x Q cells (Q a power of two, at most kMaxSb superblocks a
// tile) has one offset added to all its cells; only the superblocks around the
// peak, where the PSF varies fast, raise their cells one by one.  The offsets'
// table has an entry for every cell the superblock can lie away from the peak,
// not only for every superblock: windows of (Q + 1)^2 boxes, not (2 Q)^2, rise
// less, and the cells one by one are those of 2 x 2 superblocks (3 x 3 of
// 4 x 4 cells), not of 4 x 4.  It does not fit shared memory and need not: its
// L2 round trip runs beside the candidates'.
//
// Where the residual is flat, most cells come near the peak again and again, and
// the resolves cost more than a pass over a small tile would (256^2 with 250
// sources, 8000 iterations: 4.6 us an iteration against the plain loop's 3.1; with
// 20 sources 2.5).  What decides is the run, not its parameters, so rank 0 times
// its selections: after two running that cost more than the plain loop's
// iterations (SelDev::plain_cycles) the tile's components are applied, the peak
// is left in SelCtl::hand_key, and the launch behind this one goes on from there
// (that field 3.05 us, the sparse one 2.5).
//
// What bounds it: one CTA a tile selects while its group waits (256^2: 4 % of the
// group's issue slots, 0.4 % of the L2 rate; sixteen tiles of 1024^2: a round of 50
// in 0.16 ms and 72 MB).  An iteration is a chain of 1800 cycles with ten clock
// reads in it: 830 to decode the peak, read the cells' ranges and issue the gather
// (one L1 tag a candidate), 430 until its values are subtracted, 340 for a warp's
// reductions, 220 for the barrier and the block's; 3400 with superblocks (the
// gather misses L1 there, and the cells near the peak come after it).  The plain
// loop's were 3.3 us (256^2, cluster of 16) to 12 us (2048^2, and sixteen 1024^2
// tiles at once).  On a flat residual the resolves take as long again (2048^2, 3000
// iterations: 8.9 of 18 ms, 698 of 16 cells).  Code size matters: straight-line
// code beyond the 32 KB that stay near the schedulers ran at a third of the speed,
// so the rare parts are rolled loops.
#include <algorithm>

#include "cleangb_internal.cuh"
#include "ptx.cuh"

namespace cleangb {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kCand = 1024;                    // candidates at most
constexpr int kCandPer = kCand / kThreads;     // candidates a thread holds
constexpr int kCandStart = 700;                // candidates at the start of a selection
constexpr int kPending = kSelPending;          // components of one selection
constexpr int kMaxSb = 1024;
constexpr int kSbPer = kMaxSb / kThreads;      // superblocks a thread keeps
constexpr int kMaxDirect = 4096;               // cells of a tile without superblocks
constexpr int kDirPer = kMaxDirect / kThreads;
constexpr int kBins = 256;                     // 64 an octave
// cells the first candidates come from: few hold enough near bright sources,
// more are taken where large pixels are spread out
constexpr int kStartCells = 128, kMoreCells = 512;
constexpr int kResolveMax = 512;               // cells resolved in one go
constexpr int kResolveBudget = 6000;           // cells resolved in one selection
// cells whose bound is this near the best candidate are resolved together, and
// their pixels this near join the candidates; where that takes more than
// kManyCells, the margin shrinks (a flat residual: thousands of cells lie within
// 7 % of its peak), and widens again under kFewCells
constexpr float kNear = 0.93f;
constexpr int kManyCells = 32, kFewCells = 8;
// a cell whose range depends on the peak's place within a cell: plus the cell's
// place among the 8 x 8 around the peak (a NaN, so no pair that the table holds)
constexpr uint32_t kLobeMark = 0xffc00000u;
// a tile goes to the plain loop after this many selections running that cost
// more than it would, if this many iterations of the round are left (see SelDev)
constexpr int kSlowRuns = 2, kSlowLeft = 32;
constexpr float kFollow = 0.75f;  // see slow_above
constexpr int kUnitRows = 8, kUnitCols = 32;  // pixels a warp takes at a time in a pass

__device__ __forceinline__ uint32_t redux_max(uint32_t v) {
  return __reduce_max_sync(0xffffffffu, v);
}

// Signed integers in the order of the floats.
__device__ __forceinline__ int ord(float v) {
  const int b = __float_as_int(v);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float warp_max_f(float v) {  // (no NaN)
  const int o = __reduce_max_sync(0xffffffffu, ord(v));
  return __int_as_float(o ^ ((o >> 31) & 0x7fffffff));
}
// (a NaN, as an overflow leaves on a pixel, is no bound: the other value)
__device__ __forceinline__ float2 max2(float2 a, float2 b) {
  return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y));
}
__device__ __forceinline__ float2 add_ru(float2 a, float2 b) {
  return make_float2(__fadd_ru(a.x, b.x), __fadd_ru(a.y, b.y));
}

// A tile's pixel as row << 15 | column (tile-local, both < 2^15): ordered
// like the row-major index.  A candidate's key orders by |R|, then by the
// lower index, and carries the sign, as the 64-bit keys of the residual do.
__device__ __forceinline__ uint32_t cand_lo(uint32_t pos, float v) {
  return ((0x3fffffffu - pos) << 1) | (__float_as_uint(v) >> 31);
}
__device__ __forceinline__ uint32_t lo_pos(uint32_t lo) { return 0x3fffffffu - (lo >> 1); }

struct SelShared {
  uint4 red[2][kWarps];       // per warp: its best candidate (|R|, the key's rest) and
                              // largest bound, two buffers
  // superblocks: largest u of their cells, and the offset of their cells;
  // without superblocks the first array holds the cells' bounds
  float2 M[kMaxDirect];
  float2 acc[kMaxSb];
  int4 comp[kPending + 16];    // pending components: row, column (of the tile), flux
                              // bits, PSF offset (SelDev::inside); the loads run past
                              // the last, so every offset is one inside the PSF
  uint32_t lobe[64 * 64];     // SelDev::lobe
  uint32_t cpos[kCand];       // candidates on their way into registers
  float cval[kCand];
  int hist[kBins], more[kBins];
  uint32_t cells[kResolveMax];  // cells, row << 16 | column
  uint32_t sbs[kMaxSb];         // superblocks, row << 16 | column
  int n_cells, n_sbs, n_cand, n_pix, bin;
  unsigned long long key;     // the pass's peak key (this CTA's part)
  long long k_cmd;            // the group's command: components so far, finished
  int done_cmd, abort;
  long long t0;               // when the pass began
  int slow;                   // selections running that the plain loop would have beaten
  // followed by the cells' PSF ranges (SelDev::h8) in tiles without superblocks
};

// The kernel's shared memory.  Every function names it itself, so that the
// compiler knows the address space of what it reads there.
extern __shared__ __align__(16) unsigned char sel_smem[];
__device__ __forceinline__ SelShared& shared_state() {
  return *reinterpret_cast<SelShared*>(sel_smem);
}

// Geometry of one tile.  The largest values that R and -R can have in a cell,
// over the pixels that are no candidates, are u + acc + E: u the cell's, acc its
// superblock's, E the selection's.
struct Geo {
  Rect rc;
  int H, W, ncy, ncx, nsy, nsx, lq;  // lq: log2 of the cells along a superblock's side
  int pitch;       // cells from a row of u and masks to the next (even)
  float2* u;
  uint2* masks;    // which of the 64 pixels are candidates
};

__device__ __forceinline__ Geo make_geo(const PlanDev& d, int t) {
  Geo g;
  g.rc = tile_rect(t, d.ny, d.nx, d.ty, d.tx);
  g.H = g.rc.y1 - g.rc.y0;
  g.W = g.rc.x1 - g.rc.x0;
  g.ncy = (g.H + 7) >> 3;
  g.ncx = (g.W + 7) >> 3;
  g.pitch = d.sel.pitch;
  g.lq = d.sel.lq;
  g.nsy = (g.ncy + (1 << g.lq) - 1) >> g.lq;
  g.nsx = (g.ncx + (1 << g.lq) - 1) >> g.lq;
  const int64_t o = (int64_t)t * d.sel.cell_stride;
  g.u = d.sel.u + o;
  g.masks = d.sel.masks + o;
  return g;
}

// A load of the residual that stays where it is written (see ptx::ld_nc).
__device__ __forceinline__ float ld_res(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ float2 ld_cell(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cells(const float2* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_range(const uint32_t* p) {
  return __float_as_uint(ptx::ld_nc(reinterpret_cast<const float*>(p)));
}

// PSF value at an index of the array, and whether the index lies inside.
__device__ __forceinline__ bool psf_at(const PlanDev& d, int sy, int sx, float* p) {
  const bool in = (unsigned)sy < (unsigned)d.pny && (unsigned)sx < (unsigned)d.pnx;
  *p = in ? __ldg(d.P + (int64_t)sy * d.pnx + sx) : 0.f;
  return in;
}

// The same as one index of the array, below 0 outside.
__device__ __forceinline__ int psf_index(const PlanDev& d, int sy, int sx) {
  return (unsigned)sy < (unsigned)d.pny && (unsigned)sx < (unsigned)d.pnx ? sy * d.pnx + sx : -1;
}

// Two pixels' values less n pending components, in order (up to 32 PSF loads
// in flight; one component at a time, as the clipped PSF had it first, a
// 256 x 256 image with a PSF no larger took 34 ms for 8000 iterations).
__device__ __forceinline__ void less_pending(const PlanDev& d, float (&r)[2],
                                             const uint32_t (&pos)[2], int n) {
  SelShared& s = shared_state();
  const int y0 = (int)(pos[0] >> 15), x0 = (int)(pos[0] & 0x7fffu);
  const int y1 = (int)(pos[1] >> 15), x1 = (int)(pos[1] & 0x7fffu);
  if (d.sel.inside) {
    constexpr int U = 16;
    const float* P0 = d.P + (y0 * d.pnx + x0);
    const float* P1 = d.P + (y1 * d.pnx + x1);
#pragma unroll 1
    for (int j0 = 0; j0 < n; j0 += U) {
      float p[U][2];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int o = s.comp[j0 + u].w;
        p[u][0] = ptx::ld_nc(P0 + o);
        p[u][1] = ptx::ld_nc(P1 + o);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float f = __int_as_float(s.comp[j0 + u].z);
        const float a = __fsub_rn(r[0], __fmul_rn(f, p[u][0]));
        const float b = __fsub_rn(r[1], __fmul_rn(f, p[u][1]));
        if (j0 + u < n) {
          r[0] = a;
          r[1] = b;
        }
      }
    }
  } else {
    // (the array's first value stands in for one off the array)
    constexpr int U = 8;
#pragma unroll 1
    for (int j0 = 0; j0 < n; j0 += U) {
      float p[U][2];
      uint32_t in = 0u;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int4 c = s.comp[j0 + u];
        const int cy = d.cy - c.x, cx = d.cx - c.y;
        const int o0 = psf_index(d, y0 + cy, x0 + cx), o1 = psf_index(d, y1 + cy, x1 + cx);
        in |= (uint32_t)(o0 >= 0 && j0 + u < n) << (2 * u);
        in |= (uint32_t)(o1 >= 0 && j0 + u < n) << (2 * u + 1);
        p[u][0] = ptx::ld_nc(d.P + max(o0, 0));
        p[u][1] = ptx::ld_nc(d.P + max(o1, 0));
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float f = __int_as_float(s.comp[j0 + u].z);
        if ((in >> (2 * u)) & 1u) r[0] = __fsub_rn(r[0], __fmul_rn(f, p[u][0]));
        if ((in >> (2 * u + 1)) & 1u) r[1] = __fsub_rn(r[1], __fmul_rn(f, p[u][1]));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// A pass over the tile (all CTAs of its group): subtract the n pending
// components in order and, with scan, rebuild the cells' exact bounds and the
// peak key.  A warp takes 8 rows x 32 columns at a time: lane = column, so
// the residual and every PSF row are read 32 neighbours at a time whatever
// their alignment, and the loads of four components are in flight together.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tile_pass(const PlanDev& d, const Geo& g, int rank, int G, int n,
                                          bool scan) {
  SelShared& s = shared_state();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ux = (g.W + kUnitCols - 1) / kUnitCols, uy = (g.H + kUnitRows - 1) / kUnitRows;
  unsigned long long best = 0ull;
  const int stride = G * kWarps;
  // the residual of a warp's next unit is on its way while it works on one
  auto load = [&](int v, float (&r)[kUnitRows]) {
    const int ly = (v / ux) * kUnitRows, lx = (v % ux) * kUnitCols + lane;
    const float* Rp = d.R + (int64_t)(g.rc.y0 + ly) * d.nx + g.rc.x0 + lx;
    const int rows = v < ux * uy && lx < g.W ? min(kUnitRows, g.H - ly) : 0;
#pragma unroll
    for (int i = 0; i < kUnitRows; ++i) r[i] = i < rows ? ld_res(Rp + (int64_t)i * d.nx) : 0.f;
  };
  constexpr int A = 2;  // units ahead
  float next[A][kUnitRows];
#pragma unroll
  for (int a = 0; a < A; ++a) load(rank * kWarps + warp + a * stride, next[a]);
#pragma unroll 1
  for (int v = rank * kWarps + warp; v < ux * uy; v += stride) {
    const int ly = (v / ux) * kUnitRows, lx = (v % ux) * kUnitCols + lane;
    const bool xin = lx < g.W;
    const int rows = min(kUnitRows, g.H - ly);
    float r[kUnitRows];
    float* Rp = d.R + (int64_t)(g.rc.y0 + ly) * d.nx + g.rc.x0 + lx;
#pragma unroll
    for (int i = 0; i < kUnitRows; ++i) {
      r[i] = next[0][i];
#pragma unroll
      for (int a = 0; a + 1 < A; ++a) next[a][i] = next[a + 1][i];
    }
    load(v + A * stride, next[A - 1]);
    if (n > 0) {
      if (d.sel.inside) {
        constexpr int U = 4;  // components whose loads are in flight together
        // (columns and rows past the tile read the PSF at the tile's edge)
        const float* Pb = d.P + (int64_t)ly * d.pnx + min(lx, g.W - 1);
        int step[kUnitRows];
#pragma unroll
        for (int i = 0; i < kUnitRows; ++i) step[i] = min(i, rows - 1) * d.pnx;
#pragma unroll 1
        for (int j = 0; j < n; j += U) {
          float p[U][kUnitRows];
#pragma unroll
          for (int c = 0; c < U; ++c) {
            const float* Pp = Pb + s.comp[j + c].w;
#pragma unroll
            for (int i = 0; i < kUnitRows; ++i) p[c][i] = ptx::ld_nc(Pp + step[i]);
          }
#pragma unroll
          for (int c = 0; c < U; ++c) {
            const float f = __int_as_float(s.comp[j + c].z);
            if (j + c < n) {
#pragma unroll
              for (int i = 0; i < kUnitRows; ++i) r[i] = __fsub_rn(r[i], __fmul_rn(f, p[c][i]));
            }
          }
        }
      } else {
        constexpr int U = 4;
#pragma unroll 1
        for (int j = 0; j < n; j += U) {
          float p[U][kUnitRows];
          uint32_t in = 0u;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int4 c = s.comp[j + u];
#pragma unroll
            for (int i = 0; i < kUnitRows; ++i) {
              const int o = psf_index(d, ly + i - c.x + d.cy, lx - c.y + d.cx);
              in |= (uint32_t)(o >= 0 && j + u < n) << (u * kUnitRows + i);
              p[u][i] = ptx::ld_nc(d.P + max(o, 0));
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const float f = __int_as_float(s.comp[j + u].z);
#pragma unroll
            for (int i = 0; i < kUnitRows; ++i)
              if ((in >> (u * kUnitRows + i)) & 1u) r[i] = __fsub_rn(r[i], __fmul_rn(f, p[u][i]));
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kUnitRows; ++i)
        if (xin && i < rows) Rp[(int64_t)i * d.nx] = r[i];
    }
    if (scan) {
      float best_a = -1.f, best_v = 0.f;
      int best_i = 0;
      float2 m = make_float2(-INFINITY, -INFINITY);
#pragma unroll
      for (int i = 0; i < kUnitRows; ++i)
        if (xin && i < rows) {
          m = max2(m, make_float2(r[i], -r[i]));
          if (fabsf(r[i]) > best_a) {  // rows ascend: the first keeps a tie
            best_a = fabsf(r[i]);
            best_v = r[i];
            best_i = i;
          }
        }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1)
        m = max2(m, make_float2(__shfl_xor_sync(0xffffffffu, m.x, o),
                                __shfl_xor_sync(0xffffffffu, m.y, o)));
      if ((lane & 7) == 0 && xin) {
        const int64_t c = (int64_t)(ly >> 3) * g.pitch + (lx >> 3);
        __stcg(&g.u[c], m);
        __stcg(&g.masks[c], make_uint2(0u, 0u));
      }
      if (best_a >= 0.f) {
        const unsigned long long k =
            ((unsigned long long)__float_as_uint(best_a) << 32) |
            cand_lo(((uint32_t)(ly + best_i) << 15) | (uint32_t)lx, best_v);
        best = k > best ? k : best;
      }
    }
  }
  if (scan && n > 0) {
    const uint32_t hi = (uint32_t)(best >> 32);
    const uint32_t m = redux_max(hi);
    const uint32_t l = redux_max(hi == m ? (uint32_t)best : 0u);
    if (lane == 0 && (m | l)) atomicMax(&s.key, ((unsigned long long)m << 32) | l);
  }
}

// Every superblock's largest u: a thread reads a superblock's rows.
__device__ __noinline__ void all_sbs(const Geo g) {
  SelShared& s = shared_state();
  const int Q = 1 << g.lq;
#pragma unroll 1
  for (int b = threadIdx.x; b < g.nsy * g.nsx; b += kThreads) {
    const int by = b / g.nsx, bx = b - by * g.nsx;
    float2 m = make_float2(-INFINITY, -INFINITY);
    if (Q == 1) {
      m = __ldcg(&g.u[(int64_t)by * g.pitch + bx]);
    } else {
#pragma unroll 1
      for (int x = 0; x < Q; x += 2) {
        // (two cells at a time: rows start at even cells, and a last odd one
        // has a neighbour in the padding)
        const bool in = (bx << g.lq) + x < g.ncx;
        const float4* col = reinterpret_cast<const float4*>(&g.u[(bx << g.lq) + x]);
#pragma unroll 4
        for (int y = by << g.lq; y < (by << g.lq) + Q; ++y)
          if (in && y < g.ncy) {
            const float4 c = __ldcg(col + (int64_t)y * (g.pitch >> 1));
            m = max2(m, max2(make_float2(c.x, c.y), make_float2(c.z, c.w)));
          }
      }
    }
    s.M[b] = m;
  }
}

// Largest u of the n superblocks in s.sbs from their cells.  Q lanes (at most a
// warp) take a superblock, a cell column each.
__device__ __forceinline__ void refresh_sbs(const Geo& g, int n) {
  SelShared& s = shared_state();
  const int Q = 1 << g.lq, lw = min(g.lq, 5), L = 1 << lw;
  const int i = threadIdx.x & (L - 1);
#pragma unroll 1
  for (int q0 = 0; q0 < n; q0 += kThreads >> lw) {
    const int q = q0 + (threadIdx.x >> lw);
    const uint32_t sb = s.sbs[min(q, n - 1)];
    const int by = (int)(sb >> 16), bx = (int)(sb & 0xffffu);
    float2 m = make_float2(-INFINITY, -INFINITY);
#pragma unroll 1
    for (int cx = (bx << g.lq) + i; cx < min(g.ncx, (bx + 1) << g.lq); cx += L) {
#pragma unroll 4
      for (int cy = by << g.lq; cy < (by << g.lq) + Q; ++cy)
        if (cy < g.ncy) m = max2(m, __ldcg(&g.u[(int64_t)cy * g.pitch + cx]));
    }
#pragma unroll 1
    for (int o = L >> 1; o > 0; o >>= 1)
      m = max2(m, make_float2(__shfl_xor_sync(0xffffffffu, m.x, o),
                              __shfl_xor_sync(0xffffffffu, m.y, o)));
    if (i == 0 && q < n) s.M[by * g.nsx + bx] = m;
  }
}

// Smallest bin whose suffix holds at most `most` entries, -> s.bin (kBins: the
// top bin alone holds more).  Warp 0; the caller synchronises around it.
__device__ __noinline__ void pick_bin(int most) {
  SelShared& s = shared_state();
  const int lane = threadIdx.x;
  constexpr int per = kBins / 32;
  // lane l holds bins [kBins - per (l + 1), kBins - per l), from the top
  int sum = 0;
  for (int i = 0; i < per; ++i) sum += s.hist[kBins - 1 - (lane * per + i)];
  int run = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += v;
  }
  run -= sum;  // entries above this lane's bins
  int lowest = kBins;
  for (int i = 0; i < per; ++i) {
    run += s.hist[kBins - 1 - (lane * per + i)];
    if (run <= most) lowest = kBins - 1 - (lane * per + i);
  }
  lowest = (int)__reduce_min_sync(0xffffffffu, (unsigned)lowest);
  if (lane == 0) s.bin = lowest;
}

// Histogram bin of |R| = a below a tile's peak (bits abs0): 64 bins an octave,
// four octaves; -1 below them.
__device__ __forceinline__ int bin_of(float a, uint32_t abs0) {
  const int b = kBins - 1 - (int)((abs0 >> 17) - (__float_as_uint(fmaxf(a, 0.f)) >> 17));
  return b < 0 ? -1 : b;
}

// The tile-local positions of a cell's pixels that this lane holds (two of
// the 64): rows lane / 8 and 4 + lane / 8 of the cell, column lane % 8.
__device__ __forceinline__ bool cell_pixel(const Geo& g, uint32_t cell, int half, uint32_t* pos) {
  const int lane = threadIdx.x & 31;
  const int ly = (int)(cell >> 16) * 8 + half * 4 + (lane >> 3);
  const int lx = (int)(cell & 0xffffu) * 8 + (lane & 7);
  *pos = ((uint32_t)ly << 15) | (uint32_t)lx;
  return ly < g.H && lx < g.W;
}
__device__ __forceinline__ float residual_at(const float* R, int nx, const Geo& g, uint32_t pos) {
  return __ldcg(R + (int64_t)(g.rc.y0 + (int)(pos >> 15)) * nx + g.rc.x0 + (int)(pos & 0x7fffu));
}

// Lists the cells whose largest |R| falls in bin `least` or above.
__device__ __forceinline__ void list_cells(const Geo& g, uint32_t abs0, int least) {
  SelShared& s = shared_state();
  const int lane = threadIdx.x & 31, nc = g.ncy * g.pitch;
  constexpr int U = 4;
#pragma unroll 1
  for (int c0 = threadIdx.x; c0 - lane < nc; c0 += kThreads * U) {
    float2 u[U];
#pragma unroll
    for (int j = 0; j < U; ++j)
      u[j] = c0 + j * kThreads < nc ? __ldcg(&g.u[c0 + j * kThreads]) : make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const bool take = bin_of(fmaxf(u[j].x, u[j].y), abs0) >= least;
      const uint32_t m = __ballot_sync(0xffffffffu, take);
      if (m == 0u) continue;
      int i = 0;
      if (lane == 0) i = atomicAdd(&s.n_cells, __popc(m));
      i = __shfl_sync(0xffffffffu, i, 0) + __popc(m & ((1u << lane) - 1u));
      if (take && i < kMoreCells) {
        const int c = c0 + j * kThreads, cy = c / g.pitch;
        s.cells[i] = ((uint32_t)cy << 16) | (uint32_t)(c - cy * g.pitch);
      }
    }
  }
}

// Counts the listed cells' pixels in bin `least` or above by bin, and in s.n_pix.
__device__ __forceinline__ void count_pixels(const PlanDev& d, const Geo& g, uint32_t abs0, int nl,
                                             int least) {
  SelShared& s = shared_state();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int total = 0;
#pragma unroll 4
  for (int i = warp; i < 2 * nl; i += kWarps) {  // half cells
    uint32_t pos;
    const bool in = cell_pixel(g, s.cells[i >> 1], i & 1, &pos);
    const float r = in ? residual_at(d.R, d.nx, g, pos) : 0.f;
    const int b = in ? bin_of(fabsf(r), abs0) : -1;
    if (b >= least) atomicAdd(&s.hist[b], 1);
    total += __popc(__ballot_sync(0xffffffffu, b >= least));
  }
  if (lane == 0 && total) atomicAdd(&s.n_pix, total);
}

// The first candidates: the listed cells' pixels in bin `least` or above (they
// fit); the cells' u over the rest.
__device__ __forceinline__ void start_candidates(const PlanDev& d, const Geo& g, uint32_t abs0,
                                                 int nl, int least) {
  SelShared& s = shared_state();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll 2
  for (int i = warp; i < nl; i += kWarps) {
    const uint32_t cell = s.cells[i];
    uint32_t p0, p1;
    const bool in0 = cell_pixel(g, cell, 0, &p0), in1 = cell_pixel(g, cell, 1, &p1);
    const float v0 = in0 ? residual_at(d.R, d.nx, g, p0) : 0.f;
    const float v1 = in1 ? residual_at(d.R, d.nx, g, p1) : 0.f;
    const bool c0 = in0 && bin_of(fabsf(v0), abs0) >= least;
    const bool c1 = in1 && bin_of(fabsf(v1), abs0) >= least;
    const uint32_t h0 = __ballot_sync(0xffffffffu, c0), h1 = __ballot_sync(0xffffffffu, c1);
    if ((h0 | h1) == 0u) continue;  // as the pass left it
    float2 u = make_float2(-INFINITY, -INFINITY);
    if (in0 && !c0) u = max2(u, make_float2(v0, -v0));
    if (in1 && !c1) u = max2(u, make_float2(v1, -v1));
    u = make_float2(warp_max_f(u.x), warp_max_f(u.y));
    int slot = 0;
    if (lane == 0) {
      slot = atomicAdd(&s.n_cand, __popc(h0) + __popc(h1));
      const int64_t q = (int64_t)(cell >> 16) * g.pitch + (cell & 0xffffu);
      __stcg(&g.u[q], u);
      __stcg(&g.masks[q], make_uint2(h0, h1));
    }
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (c0) {
      const int k = slot + __popc(h0 & below);
      s.cpos[k] = p0;
      s.cval[k] = v0;
    }
    if (c1) {
      const int k = slot + __popc(h0) + __popc(h1 & below);
      s.cpos[k] = p1;
      s.cval[k] = v1;
    }
  }
}

// Resolves the cells whose bound (u + acc + E) reaches `near`: their pixels'
// exact values, the residual less the n pending components, replace the bound;
// those that reach it join s.cpos / s.cval.  Returns the number of cells; -1 if
// the candidates do not fit.  All threads; ends with a barrier.
template <bool DIRECT>
__device__ __forceinline__ int resolve(const PlanDev& d, const Geo& g, int n, float E, float near) {
  SelShared& s = shared_state();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ns = g.nsy * g.nsx, lq = g.lq, Q = 1 << lq;
  int n_sbs = 0;
  if (!DIRECT) {  // (without superblocks the caller has listed the cells)
    auto reaches = [&](float2 u, float2 acc) {
      const float2 b = add_ru(u, acc);
      return __fadd_ru(fmaxf(b.x, b.y), E) >= near;
    };
#pragma unroll 1
    for (int q = tid; q < ns; q += kThreads)
      if (reaches(s.M[q], s.acc[q]))
        s.sbs[atomicAdd(&s.n_sbs, 1)] =
            ((uint32_t)(q / g.nsx) << 16) | (uint32_t)(q - q / g.nsx * g.nsx);
    __syncthreads();
    n_sbs = s.n_sbs;
#pragma unroll 1
    for (int i = tid; i < n_sbs << (2 * lq); i += kThreads) {
      const uint32_t q = s.sbs[i >> (2 * lq)];
      const int by = (int)(q >> 16), bx = (int)(q & 0xffffu), c2 = i & ((1 << (2 * lq)) - 1);
      const int cy = (by << lq) + (c2 >> lq), cx = (bx << lq) + (c2 & (Q - 1));
      if (cy >= g.ncy || cx >= g.ncx) continue;
      if (reaches(__ldcg(&g.u[(int64_t)cy * g.pitch + cx]), s.acc[by * g.nsx + bx])) {
        const int k = atomicAdd(&s.n_cells, 1);
        if (k < kResolveMax) s.cells[k] = ((uint32_t)cy << 16) | (uint32_t)cx;
      }
    }
  }
  __syncthreads();
  const int nl = min(s.n_cells, kResolveMax);
#pragma unroll 1
  for (int i = warp; i < nl; i += kWarps) {
    const uint32_t cell = s.cells[i];
    const int64_t c = (int64_t)(cell >> 16) * g.pitch + (cell & 0xffffu);
    uint32_t pos[2];
    float r[2];
    bool in[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      in[h] = cell_pixel(g, cell, h, &pos[h]);
      if (!in[h]) pos[h] = 0u;  // (any pixel of the tile)
      r[h] = residual_at(d.R, d.nx, g, pos[h]);
    }
    const uint2 was = __ldcg(&g.masks[c]);
    less_pending(d, r, pos, n);
    const uint32_t n0 = __ballot_sync(0xffffffffu, in[0] && fabsf(r[0]) >= near) & ~was.x;
    const uint32_t n1 = __ballot_sync(0xffffffffu, in[1] && fabsf(r[1]) >= near) & ~was.y;
    const uint2 now = make_uint2(was.x | n0, was.y | n1);
    float2 u = make_float2(-INFINITY, -INFINITY);
    if (in[0] && !((now.x >> lane) & 1u)) u = max2(u, make_float2(r[0], -r[0]));
    if (in[1] && !((now.y >> lane) & 1u)) u = max2(u, make_float2(r[1], -r[1]));
    u = make_float2(warp_max_f(u.x), warp_max_f(u.y));
    const int add = __popc(n0) + __popc(n1);
    int slot = 0;
    if (lane == 0) {
      if (add) slot = atomicAdd(&s.n_cand, add);
      if (DIRECT) {
        s.M[(int)(cell >> 16) * g.nsx + (int)(cell & 0xffffu)] =
            make_float2(__fsub_ru(u.x, E), __fsub_ru(u.y, E));
      } else {
        const float2 acc =
            s.acc[(int)(cell >> (16 + lq)) * g.nsx + (int)((cell & 0xffffu) >> lq)];
        __stcg(&g.u[c], make_float2(__fsub_ru(__fsub_ru(u.x, acc.x), E),
                                    __fsub_ru(__fsub_ru(u.y, acc.y), E)));
      }
    }
    if (add == 0) continue;
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (slot + add > kCand) continue;  // the selection ends
    __syncwarp();  // every lane has read the mask
    if (lane == 0) __stcg(&g.masks[c], now);
    const uint32_t below = (1u << lane) - 1u;
    if ((n0 >> lane) & 1u) {
      const int k = slot + __popc(n0 & below);
      s.cpos[k] = pos[0];
      s.cval[k] = r[0];
    }
    if ((n1 >> lane) & 1u) {
      const int k = slot + __popc(n0) + __popc(n1 & below);
      s.cpos[k] = pos[1];
      s.cval[k] = r[1];
    }
  }
  __syncthreads();
  if (s.n_cand > kCand) return -1;
  if (!DIRECT) refresh_sbs(g, n_sbs);
  if (tid == 0) s.n_sbs = s.n_cells = 0;
  __syncthreads();
  return nl;
}

// ---------------------------------------------------------------------------
// One selection (one CTA): components k0, k0 + 1, ... of the round from the
// residual and its cells, starting from the known peak (abs0, lo0).  Returns
// how many were picked (at least one unless the run is over); *done: the
// round is over for this tile.
// ---------------------------------------------------------------------------
template <bool DIRECT>
__device__ __forceinline__ int select_components(const PlanDev& d, const Geo& g, int t,
                                                 uint32_t abs0, uint32_t lo0, int64_t k0,
                                                 int64_t kmax, float level, bool* done) {
  SelShared& s = shared_state();
  uint32_t* const h8s = reinterpret_cast<uint32_t*>(sel_smem + sizeof(SelShared));  // DIRECT
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ns = g.nsy * g.nsx, lq = g.lq, Q = 1 << lq;
  const float stop = fmaxf(d.thr, level);  // threshold, flux trigger
  *done = false;
  if (k0 >= kmax || (abs0 | lo0) == 0u || !(__uint_as_float(abs0) > stop)) {
    *done = true;
    return 0;
  }
  const int room = (int)min((int64_t)kPending, kmax - k0);

  // ---- the first candidates: the pixels above a threshold that at most
  // kStartCells cells reach, or a higher one that at most kCandStart pixels do ----
  for (int i = tid; i < kBins; i += kThreads) s.hist[i] = 0;
  if (!DIRECT)
    for (int b = tid; b < ns; b += kThreads) s.acc[b] = make_float2(0.f, 0.f);
  if (tid == 0) s.n_cells = s.n_sbs = s.n_cand = s.n_pix = 0;
  for (int i = tid; i < 64 * 64 / 4; i += kThreads)
    reinterpret_cast<uint4*>(s.lobe)[i] = __ldg(reinterpret_cast<const uint4*>(d.sel.lobe) + i);
  if (DIRECT) {
    const int n8 = ((2 * d.sel.oy8 + 1) * d.sel.w8 + 1) / 2;  // 8-byte words
#pragma unroll 2
    for (int i = tid; i < n8; i += kThreads)
      reinterpret_cast<uint2*>(h8s)[i] = __ldg(reinterpret_cast<const uint2*>(d.sel.h8) + i);
  }
  __syncthreads();
  if (room > 1) {
    // (16 bytes a load, eight in flight: one cell and four at a time, 65,536 cells
    // took 14 us, now 10.6)
    constexpr int U = 8;
    const int nc2 = (g.ncy * g.pitch) >> 1;
#pragma unroll 1
    for (int c = tid; c < nc2; c += kThreads * U) {
      float4 u[U];
#pragma unroll
      for (int j = 0; j < U; ++j)
        u[j] = c + j * kThreads < nc2 ? ld_cells(&g.u[2 * (c + j * kThreads)])
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int b0 = bin_of(fmaxf(u[j].x, u[j].y), abs0);
        const int b1 = bin_of(fmaxf(u[j].z, u[j].w), abs0);
        if (b0 > 0) atomicAdd(&s.hist[b0], 1);
        if (b1 > 0) atomicAdd(&s.hist[b1], 1);
      }
    }
    __syncthreads();
    int least = 0, nl = 0;
#pragma unroll 1
    for (int most = kStartCells;; most = kMoreCells) {
      if (warp == 0) pick_bin(most);
      __syncthreads();
      least = max(s.bin, 1);
      for (int i = tid; i < kBins; i += kThreads) s.more[i] = s.hist[i];
      __syncthreads();
      for (int i = tid; i < kBins; i += kThreads) s.hist[i] = 0;
      list_cells(g, abs0, least);
      __syncthreads();
      nl = min(s.n_cells, kMoreCells);
      count_pixels(d, g, abs0, nl, least);
      __syncthreads();
      // (no thread writes this count before the block's next barrier)
      if (most == kMoreCells || s.n_pix >= kCandStart / 4 || least == 1) break;
      // too few: back to the cells' counts
      for (int i = tid; i < kBins; i += kThreads) s.hist[i] = s.more[i];
      __syncthreads();
      if (tid == 0) s.n_cells = s.n_pix = 0;
      __syncthreads();
    }
    if (warp == 0) pick_bin(kCandStart);
    __syncthreads();
    start_candidates(d, g, abs0, nl, max(s.bin, least));
    __syncthreads();
    if (!DIRECT) all_sbs(g);
    if (tid == 0) s.n_cells = 0;
    __syncthreads();
  }
  int ncand = s.n_cand;
  // no candidates: more equal pixels than registers; the known peak alone
  const bool alone = ncand == 0;

  // the thread's candidates (an empty slot's NaN stays one and is never the
  // largest) ...
  float r[kCandPer];
  uint32_t pos[kCandPer];
  int at[kCandPer];  // the pixel's place in an array of the PSF's pitch
  auto load_slots = [&](int from, int to) {
#pragma unroll
    for (int i = 0; i < kCandPer; ++i) {
      const int q = tid + i * kThreads;
      if (q >= from && q < to) {
        pos[i] = s.cpos[q];
        r[i] = s.cval[q];
        at[i] = (int)(pos[i] >> 15) * d.pnx + (int)(pos[i] & 0x7fffu);
      }
    }
  };
#pragma unroll
  for (int i = 0; i < kCandPer; ++i) {
    r[i] = NAN;
    pos[i] = 0u;
    at[i] = 0;
  }
  load_slots(0, ncand);
  // ... its superblocks' (DIRECT: cells') places in the table of PSF ranges, and
  // their offsets (bounds; shared memory has the offsets too) ...
  constexpr int kOwn = DIRECT ? kDirPer : kSbPer;
  int hbi[kOwn], sby[DIRECT ? 1 : kOwn], sbx[DIRECT ? 1 : kOwn];
  float2 acc[kOwn];
#pragma unroll
  for (int i = 0; i < kOwn; ++i) {
    const int b = tid + i * kThreads, y = b < ns ? b / g.nsx : 0, x = b < ns ? b - y * g.nsx : 0;
    hbi[i] = ((y << lq) + d.sel.oy8) * d.sel.w8 + (x << lq) + d.sel.ox8;
    if (!DIRECT) {
      sby[i] = y;
      sbx[i] = x;
    }
    acc[i] = make_float2(0.f, 0.f);
    if (DIRECT)
      acc[i] = b < ns ? __ldcg(&g.u[(int64_t)y * g.pitch + x]) : make_float2(-INFINITY, -INFINITY);
  }
  // ... and its cell among the nb x nb superblocks around the peak that its
  // 8 x 8 cells reach (superblocks have 4 x 4 cells at least), nL lanes a
  // superblock (for larger superblocks, its first cell)
  const int nb = lq >= 3 ? 2 : 3;
  const int nlw = min(2 * lq, 5), nL = 1 << nlw;
  const int nq = tid >> nlw, nc0 = tid & (nL - 1), nqy = nq / nb, nqx = nq - nqy * nb;
  const bool near_warp = !DIRECT && (nq & -(32 >> nlw)) < nb * nb;  // (one for the warp)

  uint32_t wabs = abs0, wlo = lo0;
  int n = 0, buf = 0, spent = 0;
  float near = fminf(fmaxf(d.sel.ctl[t].near, kNear), 1.f);  // the margin it ended with
  const float pc = __ldg(d.P + (int64_t)d.cy * d.pnx + d.cx);  // the largest |PSF|
  float E = 0.f;  // the pixels' own roundings so far
#pragma unroll 1
  for (;;) {
    // ---- the component of the accepted peak ----
    const float av = __uint_as_float(wabs);
    if (!(av > stop)) {
      *done = true;
      break;
    }
    const uint32_t p = lo_pos(wlo);
    const int pyl = (int)(p >> 15), pxl = (int)(p & 0x7fffu);
    const float f = __fmul_rn(d.gain, __uint_as_float(wabs | (wlo << 31)));  // first equation
    const int off = (d.cy - pyl) * d.pnx + d.cx - pxl;
    if (tid == kThreads - 32) s.comp[n] = make_int4(pyl, pxl, __float_as_int(f), off);
    ++n;
    // (values that could overflow go one component at a time, as the plain
    // loop sees them)
    const float m = fabsf(f), reach = __fmaf_ru(m, pc, av);
    if (n == room || alone || !(reach < 1e30f)) {
      *done = k0 + n == kmax;
      break;
    }
    E = __fmaf_ru(reach, 0x1p-22f, E);
    // ---- the loads: the PSF ranges (the largest rise of R and of -R for
    // f = 1), then the candidates' PSF values ----
    const int cyl = (pyl + 7) >> 3, cxl = (pxl + 7) >> 3, h0 = -(cyl * d.sel.w8 + cxl);
    // the first of the 8 x 8 cells around the peak, and their ranges for the
    // peak's place within a cell
    const int ly0 = cyl - 4, lx0 = cxl - 4;
    const int nby = ly0 >> lq, nbx = lx0 >> lq;  // the first superblock around it
    const uint32_t* const lobe = s.lobe + (((-pyl & 7) * 8 + (-pxl & 7)) << 6);
    const bool up = f > 0.f;
    float bound = -INFINITY;
    // the cells around the peak first: behind the candidates' loads they would
    // wait for those
    constexpr int kNearU = 2;  // cells at a time
    int no[kNearU];
    float2 nu[kNearU];
    uint32_t nw[kNearU];
    const int nsy = nby + nqy, nsx = nbx + nqx;
    const bool near_in = !DIRECT && nqy < nb && (unsigned)nsy < (unsigned)g.nsy &&
                         (unsigned)nsx < (unsigned)g.nsx;
    auto near_load = [&](int c) {
#pragma unroll
      for (int j = 0; j < kNearU; ++j) {
        const int k = c + j * nL;
        const int cy = (nsy << lq) + (k >> lq), cx = (nsx << lq) + (k & (Q - 1));
        no[j] = near_in && k < (1 << (2 * lq)) && cy < g.ncy && cx < g.ncx ? cy * g.pitch + cx : -1;
        if (no[j] < 0) continue;
        nu[j] = ld_cell(&g.u[no[j]]);
        nw[j] = ld_range(d.sel.h8 + ((cy + d.sel.oy8) * d.sel.w8 + cx + d.sel.ox8 + h0));
      }
    };
    if (near_warp) near_load(nc0);
    uint32_t e16[kOwn];
    float2 mx[DIRECT ? 1 : kOwn];
    bool far[DIRECT ? 1 : kOwn];  // not around the peak (those change below)
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
      if (i * kThreads >= ns) break;
      if (DIRECT) {
        e16[i] = h8s[h0 + hbi[i]];
        if (e16[i] >= kLobeMark) e16[i] = lobe[e16[i] & 63u];
      } else {
        e16[i] = ld_range(d.sel.hb + h0 + hbi[i]);
        far[i] = tid + i * kThreads < ns && !((unsigned)(sby[i] - nby) < (unsigned)nb &&
                                              (unsigned)(sbx[i] - nbx) < (unsigned)nb);
        if (far[i]) mx[i] = s.M[tid + i * kThreads];
      }
    }
    float pv[kCandPer];
    bool ok[kCandPer];
#pragma unroll
    for (int i = 0; i < kCandPer; ++i) {
      ok[i] = i * kThreads < ncand;
      if (!ok[i]) continue;
      if (d.sel.inside)
        pv[i] = ptx::ld_nc(d.P + (off + at[i]));
      else
        ok[i] = psf_at(d, (int)(pos[i] >> 15) - pyl + d.cy, (int)(pos[i] & 0x7fffu) - pxl + d.cx,
                       &pv[i]);
    }
    // ---- the superblocks' offsets, or the cells' bounds ----
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
      const int b = tid + i * kThreads;
      if (i * kThreads >= ns) break;
      const uint32_t w = up ? e16[i] : __byte_perm(e16[i], 0u, 0x1032);
      if (DIRECT) {
        acc[i].x = __fmaf_ru(m, __uint_as_float(w << 16), acc[i].x);
        acc[i].y = __fmaf_ru(m, __uint_as_float(w & 0xffff0000u), acc[i].y);
        bound = fmaxf(bound, fmaxf(acc[i].x, acc[i].y));
      } else if (far[i]) {
        acc[i].x = __fmaf_ru(m, __uint_as_float(w << 16), acc[i].x);
        acc[i].y = __fmaf_ru(m, __uint_as_float(w & 0xffff0000u), acc[i].y);
        s.acc[b] = acc[i];
        const float2 a = add_ru(acc[i], mx[i]);
        bound = fmaxf(bound, fmaxf(a.x, a.y));
      }
    }
    // ---- the cells of the superblocks around the peak one by one ----
    if (near_warp) {
      float2 mm = make_float2(-INFINITY, -INFINITY);
#pragma unroll 1
      for (int c = nc0;;) {
#pragma unroll
        for (int j = 0; j < kNearU; ++j) {
          if (no[j] < 0) continue;
          if (nw[j] >= kLobeMark) nw[j] = lobe[nw[j] & 63u];
          if (!up) nw[j] = __byte_perm(nw[j], 0u, 0x1032);
          nu[j].x = __fmaf_ru(m, __uint_as_float(nw[j] << 16), nu[j].x);
          nu[j].y = __fmaf_ru(m, __uint_as_float(nw[j] & 0xffff0000u), nu[j].y);
          g.u[no[j]] = nu[j];
          mm = max2(mm, nu[j]);
        }
        c += nL * kNearU;
        if (c >= 1 << (2 * lq)) break;
        near_load(c);
      }
      const int b = nsy * g.nsx + nsx;
      if (near_in) {
        const float2 a = add_ru(mm, s.acc[b]);
        bound = fmaxf(bound, fmaxf(a.x, a.y));
      }
      if (nL < 32) {  // 16
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
          mm = max2(mm, make_float2(__shfl_xor_sync(0xffffffffu, mm.x, o),
                                    __shfl_xor_sync(0xffffffffu, mm.y, o)));
      } else {
        mm = make_float2(warp_max_f(mm.x), warp_max_f(mm.y));
      }
      if (near_in && nc0 == 0) s.M[b] = mm;
    }
    bound = fmaxf(__fadd_ru(bound, E), 0.f);
#pragma unroll
    for (int i = 0; i < kCandPer; ++i)
      if (ok[i]) r[i] = __fsub_rn(r[i], __fmul_rn(f, pv[i]));
    bool fail = false;
#pragma unroll 1
    for (;;) {
      // ---- the best candidate and the largest bound ----
      {
        float best = 0.f;
#pragma unroll
        for (int i = 0; i < kCandPer; ++i) best = fmaxf(best, fabsf(r[i]));
        const uint32_t a = __float_as_uint(best), ma = redux_max(a);
        const uint32_t mb = redux_max(__float_as_uint(bound));
        uint32_t l = 0u;
        if (a == ma) {
#pragma unroll
          for (int i = 0; i < kCandPer; ++i)
            if (__float_as_uint(fabsf(r[i])) == ma) l = max(l, cand_lo(pos[i], r[i]));
        }
        l = redux_max(l);
        if (lane == 0) s.red[buf][warp] = make_uint4(ma, l, mb, 0u);
      }
      __syncthreads();
      const uint4 v = s.red[buf][lane & (kWarps - 1)];
      wabs = redux_max(v.x);
      const uint32_t top = redux_max(v.z);
      wlo = redux_max(v.x == wabs ? v.y : 0u);
      buf ^= 1;
      if (top < wabs) break;  // no other pixel reaches the best candidate
      const float reach_to = near * __uint_as_float(wabs);
      uint32_t sent = 0u;  // this thread's cells on the list
      if (DIRECT) {
#pragma unroll
        for (int i = 0; i < kOwn; ++i) {
          const int q = tid + i * kThreads;
          if (!(__fadd_ru(fmaxf(acc[i].x, acc[i].y), E) >= reach_to)) continue;
          const int k = atomicAdd(&s.n_cells, 1);
          if (k >= kResolveMax) continue;
          s.cells[k] = ((uint32_t)(q / g.nsx) << 16) | (uint32_t)(q - q / g.nsx * g.nsx);
          sent |= 1u << i;
        }
      }
      const int cells = resolve<DIRECT>(d, g, n, E, reach_to);
      if (cells == 0) break;  // the best candidate is 0 and no pixel is larger
      spent += cells;
      if (cells > kManyCells)
        near = 1.f - 0.25f * (1.f - near);
      else if (cells < kFewCells)
        near = fmaxf(kNear, 1.f - 1.5f * (1.f - near));
      if (cells < 0 || spent > kResolveBudget) {
        fail = true;
        break;
      }
      const int nn = s.n_cand;
      load_slots(ncand, nn);
      ncand = nn;
      bound = 0.f;
#pragma unroll
      for (int i = 0; i < kOwn; ++i) {
        const int q = tid + i * kThreads;
        if (q >= ns) break;
        float2 a;
        if (DIRECT) {
          if ((sent >> i) & 1u) acc[i] = s.M[q];
          a = acc[i];
        } else {
          a = add_ru(s.M[q], acc[i]);
        }
        bound = fmaxf(bound, __fadd_ru(fmaxf(a.x, a.y), E));
      }
    }
    if (fail) break;
  }
  __syncthreads();
  if (tid == 0) d.sel.ctl[t].near = near;  // (every thread has read it)
  // the records, here and not an iteration at a time (the thread that kept them
  // came to every barrier some 500 cycles after the others): the list, and the
  // model, whose pixels' sums are taken in list order by the thread of the
  // pixel's first component
  float* sum = nullptr;
  float v = 0.f;
  if (tid < n) {
    const int4 c = s.comp[tid];
    clean_component cc;
    cc.y = g.rc.y0 + c.x;
    cc.x = g.rc.x0 + c.y;
    cc.flux = __int_as_float(c.z);
    cc.tile = t;
    d.rcomps[(int64_t)t * d.cap_round + k0 + tid] = cc;
    sum = d.model + (int64_t)cc.y * d.nx + cc.x;
    v = __ldcg(sum);
    bool first = true;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const int4 o = s.comp[j];
      if (o.x != c.x || o.y != c.y) continue;
      first &= j >= tid;
      v = __fadd_rn(v, __int_as_float(o.z));
    }
    if (!first) sum = nullptr;
  }
  __syncthreads();  // every component of a pixel has read it
  if (sum) __stcg(sum, v);
  __syncthreads();
  return n;
}

// ---- the group of a tile ------------------------------------------------------
// The tile's CTAs share its passes; rank 0 selects.  After each pass every
// other rank counts itself in (SelCtl::arrived) and rank 0 waits for the
// count; after each selection rank 0 posts the component count and whether
// the round is over (SelCtl::cmd) and the others wait for the post.  The posts
// count on across launches (base: passes of the tile so far), the arrivals start
// again in each, so that a tile's group may have another size in the next round.
// Waits are bounded by limit_ns; an expired one sets ST_TIMEOUT.

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ bool wait_count(const uint32_t* p, uint32_t want, uint64_t limit_ns,
                                           bool nap) {
  if (ld_acquire(p) == want) return true;
  const uint64_t t0 = ptx::globaltimer_ns();
  for (;;) {
    if (nap) __nanosleep(200);
    if (ld_acquire(p) == want) return true;
    if (ptx::globaltimer_ns() - t0 > limit_ns) return false;
  }
}

// The cycles a component above which the plain loop is preferred.  In a batch its
// launch waits for the last image's selections, so once one has gone over the
// others follow unless they are a good deal faster (32 crowded 200^2 images: 7.8 us
// an iteration on their own account, now 4.8).
__device__ __forceinline__ float slow_above(const PlanDev& d) {
  const bool follow = d.sel.handed && *(volatile int32_t*)d.sel.handed > 0;
  return follow ? kFollow * d.sel.plain_cycles : d.sel.plain_cycles;
}

// CTA `rank` of the G serving tile t for one round.
template <bool DIRECT>
__device__ __forceinline__ void select_body(const PlanDev& d, int G, int parity, int flags,
                                            uint64_t limit_ns, int force_timeout, int t,
                                            int rank) {
  SelShared& s = shared_state();
  const Geo g = make_geo(d, t);
  const uint64_t key = d.peak[parity * d.T + t];
  const int64_t budget = d.budget[t];
  const int64_t kmax = (d.K > 0 && (int64_t)d.K < budget) ? (int64_t)d.K : budget;
  const float level = d.trigger > 0.f ? *(volatile float*)&d.st->level : 0.f;
  const int32_t status = *(volatile int32_t*)&d.st->status;
  SelCtl* ctl = d.sel.ctl + t;
  const uint32_t base = ctl->phases;
  const int slow = ctl->slow;
  // tiles whose rounds the plain loop has taken over (the group reads this
  // before rank 0 can change it: that is behind its wait for their passes)
  const bool hand_all = d.sel.plain_cycles > 0.f && slow >= kSlowRuns;
  const bool idle = kmax <= 0 || key == 0ull || !(key_abs(key) > d.thr) || !(key_abs(key) > level);
  if (threadIdx.x == 0) {
    s.abort = status != 0;  // one thread's for the block
    s.key = 0ull;
    s.slow = slow;
    if (rank == 0) ctl->hand_key = hand_all && !idle ? key : 0ull;
  }
  for (int j = threadIdx.x; j < kPending + 16; j += kThreads) s.comp[j] = make_int4(0, 0, 0, 0);
  int64_t k = 0, applied = 0;  // components of the round; those the residual has
  uint32_t phase = 0;
  bool done = idle;
  __syncthreads();
  if (s.abort) return;
  while (!idle && !hand_all) {
    if (threadIdx.x == 0) s.t0 = clock64();
    // the pending components, then the cells (unless the round is over)
    if (done && (!(flags & kSelFlush) || k == applied)) break;
    tile_pass(d, g, rank, G, (int)(k - applied), !done);
    applied = k;
    if (done) break;
    // all parts of the pass are done
    ++phase;
    __syncthreads();
    if (G > 1 && threadIdx.x == 0) {
      if (rank != 0) {
        if (phase > 1) atomicMax((unsigned long long*)&ctl->key[phase & 1], s.key);
        __threadfence();
        atomicAdd(&ctl->arrived, 1u);
      } else {
        if (!wait_count(&ctl->arrived,
                        phase * (uint32_t)(G - 1) + (force_timeout ? 1u : 0u), limit_ns, false)) {
          atomicOr(&d.st->status, ST_TIMEOUT);
          d.st->timeout_where = ((int64_t)t << 32) | (int64_t)k;
          s.abort = 1;
        }
        if (phase > 1) {
          const unsigned long long o = *(volatile unsigned long long*)&ctl->key[phase & 1];
          s.key = o > s.key ? o : s.key;
        }
        ctl->key[(phase & 1) ^ 1] = 0ull;  // for the next pass (ordered by the post below)
      }
    }
    __syncthreads();
    if (rank == 0 && s.abort) break;  // (the others' threads 0 may be at its next use)
    if (rank == 0) {
      uint32_t abs0 = (uint32_t)(s.key >> 32), lo0 = (uint32_t)s.key;
      if (phase == 1) {  // the round's first peak is known
        const int idx = key_index(key), py = idx / d.nx, px = idx - py * d.nx;
        abs0 = (uint32_t)(key >> 32);
        lo0 = cand_lo(((uint32_t)(py - g.rc.y0) << 15) | (uint32_t)(px - g.rc.x0), key_value(key));
      }
      const bool over = s.slow >= kSlowRuns && kmax - k >= kSlowLeft;
      __syncthreads();
      if (over) {
        // nothing is pending: the plain loop goes on from this peak
        const uint32_t p = lo_pos(lo0);
        if (threadIdx.x == 0) {
          ctl->hand_key = make_key(__uint_as_float(abs0 | (lo0 << 31)),
                                   (g.rc.y0 + (int)(p >> 15)) * d.nx + g.rc.x0 + (int)(p & 0x7fffu));
          if (d.sel.handed) atomicAdd(d.sel.handed, 1);
          if (flags & kSelReport) d.st->handed = 1;
        }
        done = true;
      } else {
        const int n = select_components<DIRECT>(d, g, t, abs0, lo0, k, kmax, level, &done);
        k += n;
        if (threadIdx.x == 0 && d.sel.plain_cycles > 0.f && !done)
          s.slow = (float)(clock64() - s.t0) > slow_above(d) * (float)n ? s.slow + 1 : 0;
      }
      if (threadIdx.x == 0) {
        s.key = 0ull;
        if (G > 1) {
          ctl->k = k;
          ctl->done = done ? 1 : 0;
          st_release(&ctl->cmd, base + phase);
        }
      }
      __syncthreads();
    } else {
      if (threadIdx.x == 0) {
        if (!wait_count(&ctl->cmd, base + phase, limit_ns, true)) {
          atomicOr(&d.st->status, ST_TIMEOUT);
          s.abort = 1;
        }
        s.k_cmd = *(volatile int64_t*)&ctl->k;
        s.done_cmd = *(volatile int32_t*)&ctl->done;
        s.key = 0ull;
      }
      __syncthreads();
      if (s.abort) break;
      k = s.k_cmd;
      done = s.done_cmd != 0;
      if (!done || (flags & kSelFlush))
        for (int j = threadIdx.x; j < (int)(k - applied); j += kThreads) {
          int4 c = __ldcg(reinterpret_cast<const int4*>(
              &d.rcomps[(int64_t)t * d.cap_round + applied + j]));
          c.x -= g.rc.y0;
          c.y -= g.rc.x0;
          c.w = (d.cy - c.x) * d.pnx + d.cx - c.y;
          s.comp[j] = c;
        }
      __syncthreads();
    }
  }
  if (rank == 0 && threadIdx.x == 0) {
    d.peak[(parity ^ 1) * d.T + t] = 0ull;  // the feedback's next peak goes here
    d.rcount[t] = (int32_t)k;
    d.rapplied[t] = (int32_t)applied;
    d.budget[t] = budget - k;
    ctl->phases = base + phase;
    ctl->arrived = 0u;  // (every wait for it is over)
    ctl->slow = s.slow;
    if (s.abort) ctl->hand_key = 0ull;
  }
}

template <bool DIRECT>
__global__ void __launch_bounds__(kThreads, 1)
    select_kernel(PlanDev d, int G, int parity, int flags, uint64_t limit_ns, int force_timeout) {
  select_body<DIRECT>(d, G, parity, flags, limit_ns, force_timeout, (int)blockIdx.x / G,
                      (int)blockIdx.x % G);
}

// G CTAs per (image, tile) item; with G > 1 the launch is cooperative, so they run
// at the same time and may wait for each other.
template <bool DIRECT>
__global__ void __launch_bounds__(kThreads, 1)
    select_batch_kernel(const PlanDev* __restrict__ plans, const BatchItem* __restrict__ items,
                        int G, int round, uint64_t limit_ns) {
  const BatchItem it = items[blockIdx.x / G];
  const PlanDev d = plans[it.image];
  select_body<DIRECT>(d, G, (round - d.round0) & 1, 0, limit_ns, 0, it.tile, blockIdx.x % G);
}

// ---- the PSF's ranges (once per PSF) -------------------------------------------

// Range of the PSF over 8 x 8 boxes of offsets: box (i, j) holds the offsets
// [8 (i - oy), 8 (i - oy) + 8) x ...; offsets off the PSF array count as 0 (those
// pixels do not change).  One warp per four boxes of a row.
__global__ void psf_box_kernel(PlanDev d, float2* __restrict__ g8, int rows, int cols) {
  const int lane = threadIdx.x & 31;
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int per = (cols + 3) / 4;
  if (w >= rows * per) return;
  const int i = w / per, j = (w - i * per) * 4 + (lane >> 3);
  const int y0 = 8 * (i - d.sel.oy8) + d.cy;
  const int x = 8 * ((w - i * per) * 4 - d.sel.ox8) + lane + d.cx;
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    float p;
    psf_at(d, y0 + r, x, &p);
    lo = fminf(lo, p);
    hi = fmaxf(hi, p);
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if ((lane & 7) == 0 && j < cols) g8[(int64_t)i * cols + j] = make_float2(lo, hi);
}

// The rises for a range (minimum, maximum) as two bf16, rounded up.
__device__ __forceinline__ uint32_t pack_rises(float2 m) {
  auto up16 = [](float v) {
    const uint32_t w = __float_as_uint(v);
    return (v > 0.f ? w + 0xffffu : w) >> 16;
  };
  return up16(-m.x) | (up16(m.y) << 16);
}

// Near the peak, where the PSF varies within a window, the exact ranges: entry
// [(sy * 8 + sx) * 64 + i * 8 + j] is that of the 8 x 8 pixels at offsets
// 8 (i - 4) + sy .. + 7 and 8 (j - 4) + sx .. + 7.
__global__ void psf_lobe_kernel(PlanDev d, uint32_t* __restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 64 * 64) return;
  const int y0 = 8 * (((e >> 3) & 7) - 4) + (e >> 9) + d.cy;
  const int x0 = 8 * ((e & 7) - 4) + ((e >> 6) & 7) + d.cx;
  float2 m = make_float2(INFINITY, -INFINITY);
#pragma unroll 8
  for (int i = 0; i < 64; ++i) {
    float p;
    psf_at(d, y0 + (i >> 3), x0 + (i & 7), &p);
    m = make_float2(fminf(m.x, p), fmaxf(m.y, p));
  }
  out[e] = pack_rises(m);
}

// Ranges over windows of 2 x 2 boxes: entry (i, j) is what a cell i - oy8 rows
// and j - ox8 columns of cells from the peak's can meet, wherever in its cell
// the peak lies.  Stored as the largest rises of R and of -R when the PSF is
// subtracted once; kLobeMark for the 8 x 8 around offset 0.
__global__ void psf_window_kernel(const float2* __restrict__ g8, int cols8, int oy8, int ox8,
                                  uint32_t* __restrict__ out, int rows, int cols) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (int64_t)rows * cols) return;
  const int i = (int)(q / cols), j = (int)(q - (int64_t)i * cols);
  const float2* b = g8 + (int64_t)i * cols8 + j;  // (the boxes have a row and a column more)
  const float2 v0 = __ldg(b), v1 = __ldg(b + 1), v2 = __ldg(b + cols8), v3 = __ldg(b + cols8 + 1);
  const float2 m = make_float2(fminf(fminf(v0.x, v1.x), fminf(v2.x, v3.x)),
                               fmaxf(fmaxf(v0.y, v1.y), fmaxf(v2.y, v3.y)));
  const bool lobe = i - oy8 >= -4 && i - oy8 < 4 && j - ox8 >= -4 && j - ox8 < 4;
  out[q] = lobe ? kLobeMark + (uint32_t)((i - oy8 + 4) * 8 + j - ox8 + 4) : pack_rises(m);
}

// The same for superblocks of n x n cells: windows of n + 1 boxes a side as far
// as the boxes go, along the rows first (into tmp, `cols` wide), then down the
// columns.
__global__ void psf_window_x_kernel(const float2* __restrict__ g8, int rows8, int cols8,
                                    float2* __restrict__ tmp, int cols, int n) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (int64_t)rows8 * cols) return;
  const int i = (int)(q / cols), j = (int)(q - (int64_t)i * cols);
  float2 m = make_float2(INFINITY, -INFINITY);
#pragma unroll 4
  for (int x = j; x <= min(j + n, cols8 - 1); ++x) {
    const float2 v = __ldg(&g8[(int64_t)i * cols8 + x]);
    m = make_float2(fminf(m.x, v.x), fmaxf(m.y, v.y));
  }
  tmp[q] = m;
}
__global__ void psf_window_y_kernel(const float2* __restrict__ tmp, int rows8, int cols,
                                    uint32_t* __restrict__ out, int rows, int n) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (int64_t)rows * cols) return;
  const int i = (int)(q / cols), j = (int)(q - (int64_t)i * cols);
  float2 m = make_float2(INFINITY, -INFINITY);
#pragma unroll 4
  for (int y = i; y <= min(i + n, rows8 - 1); ++y) {
    const float2 v = __ldg(&tmp[(int64_t)y * cols + j]);
    m = make_float2(fminf(m.x, v.x), fmaxf(m.y, v.y));
  }
  out[q] = pack_rises(m);
}

}  // namespace

bool select_geometry(SelDev* g, int ny, int nx, int ty, int tx, SelSizes* z) {
  *g = SelDev{};
  *z = SelSizes{};
  int maxH = 0, maxW = 0;
  for (int i = 0; i < ty; ++i)
    maxH = std::max(maxH, (int)(((int64_t)(i + 1) * ny) / ty - ((int64_t)i * ny) / ty));
  for (int j = 0; j < tx; ++j)
    maxW = std::max(maxW, (int)(((int64_t)(j + 1) * nx) / tx - ((int64_t)j * nx) / tx));
  if (maxH < 1 || maxW < 1 || maxH > 32767 || maxW > 32767) return false;
  const int ncy = (maxH + 7) / 8, ncx = (maxW + 7) / 8;
  int lq = 0;
  while ((int64_t)ncy * ncx > kMaxDirect &&
         (int64_t)((ncy + (1 << lq) - 1) >> lq) * ((ncx + (1 << lq) - 1) >> lq) > kMaxSb) ++lq;
  g->lq = lq;
  g->pitch = (ncx + 1) & ~1;
  g->cell_stride = (int64_t)ncy * g->pitch;
  g->oy8 = ncy;
  g->ox8 = ncx;
  g->w8 = 2 * ncx + 1;
  const size_t entries = (size_t)(2 * ncy + 1) * (size_t)(2 * ncx + 1);
  const size_t boxes = (size_t)(2 * ncy + 2) * (size_t)(2 * ncx + 2);
  const size_t table = (sizeof(uint32_t) * (entries + 1)) & ~(size_t)7;  // read 8 bytes at a time
  z->smem = (int)(sizeof(SelShared) + (lq == 0 ? table : 0));
  z->cells = sizeof(float2) * (size_t)g->cell_stride * (size_t)(ty * tx);
  z->boxes = sizeof(float2) * boxes * (lq > 0 ? 2 : 1);  // and the windows' rows
  z->h8 = table;
  z->hb = lq > 0 ? table : 0;
  z->lobe = sizeof(uint32_t) * 64 * 64;
  z->ctl = sizeof(SelCtl) * (size_t)(ty * tx);
  return true;
}

cudaError_t select_build_psf(const PlanDev& d, float2* boxes, uint32_t* h8, uint32_t* hb,
                             uint32_t* lobe, cudaStream_t s) {
  const SelDev& g = d.sel;
  const int rows8 = 2 * g.oy8 + 2, cols8 = 2 * g.ox8 + 2, rows = rows8 - 1, cols = cols8 - 1;
  const int64_t warps = (int64_t)rows8 * ((cols8 + 3) / 4);
  auto blocks = [](int64_t n) { return (unsigned)((n + 127) / 128); };
  psf_box_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(d, boxes, rows8, cols8);
  psf_window_kernel<<<blocks((int64_t)rows * cols), 128, 0, s>>>(boxes, cols8, g.oy8, g.ox8, h8,
                                                                 rows, cols);
  if (g.lq > 0) {
    float2* tmp = boxes + (int64_t)rows8 * cols8;
    psf_window_x_kernel<<<blocks((int64_t)rows8 * cols), 128, 0, s>>>(boxes, rows8, cols8, tmp,
                                                                      cols, 1 << g.lq);
    psf_window_y_kernel<<<blocks((int64_t)rows * cols), 128, 0, s>>>(tmp, rows8, cols, hb, rows,
                                                                     1 << g.lq);
  }
  psf_lobe_kernel<<<32, 128, 0, s>>>(d, lobe);
  return cudaGetLastError();
}

cudaError_t select_prepare() {
  const void* fns[] = {(const void*)select_kernel<true>, (const void*)select_kernel<false>,
                       (const void*)select_batch_kernel<true>,
                       (const void*)select_batch_kernel<false>};
  cudaError_t e = cudaSuccess;
  for (const void* f : fns)
    if (e == cudaSuccess) e = allow_max_smem(f);
  return e;
}

cudaError_t launch_select(const PlanDev& d, int G, int smem, int parity, int flags,
                          uint64_t limit_ns, int force_timeout, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(d.T * G), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = G > 1 ? 1 : 0;  // a group of one waits for nobody
  PlanDev dd = d;
  void* args[] = {&dd, &G, &parity, &flags, &limit_ns, &force_timeout};
  return cudaLaunchKernelExC(
      &cfg, d.sel.lq == 0 ? (const void*)select_kernel<true> : (const void*)select_kernel<false>,
      args);
}

cudaError_t launch_select_batch(const PlanDev* plans, const BatchItem* items, int n_items,
                                int direct, int G, int smem, int round, uint64_t limit_ns,
                                cudaStream_t s) {
  if (n_items <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(n_items * G), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = G > 1 ? 1 : 0;
  void* args[] = {const_cast<PlanDev**>(&plans), const_cast<BatchItem**>(&items), &G, &round,
                  &limit_ns};
  return cudaLaunchKernelExC(&cfg, direct ? (const void*)select_batch_kernel<true>
                                          : (const void*)select_batch_kernel<false>,
                             args);
}

}  // namespace cleangb
