// Set-up, input checks and restoration.
//
// init_kernel      R <- dirty, model <- 0, finiteness of the dirty image, the
//                  first peak key of every tile, and the per-tile budgets
//                  (niter split evenly, the remainder to the lowest tiles).
// validate_psf     finiteness of the PSF and |P| <= P[centre] everywhere.
// restore_kernel   model convolved with a Gaussian clean beam, plus residual.
#include <cmath>

#include "cleangb_internal.cuh"

namespace cleangb {

namespace {

// Set-up: a warp a row, four pixels of a lane in flight.  Small images are
// bound by the latency of a block's few loads (320 x 320 in four tiles: 12 us
// with 16 rows a block one after another, now 5), large ones by memory.  The
// dirty image may be the residual itself (host buffers, runs in place), so its
// loads are ordinary ones: the compiler keeps them ahead of the stores.
constexpr int kInitThreads = 256;
constexpr int kInitRows = kInitThreads / 32;  // tile rows per init block

__device__ __forceinline__ uint64_t umax64(uint64_t a, uint64_t b) {
  return a > b ? a : b;
}

__device__ __forceinline__ uint64_t warp_max_key(uint64_t k) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) k = umax64(k, __shfl_xor_sync(0xffffffffu, k, o));
  return k;
}

__global__ void __launch_bounds__(kInitThreads)
    init_kernel(PlanDev d, const float* dirty, int64_t niter) {
  __shared__ uint64_t s_warp[kInitThreads / 32];
  const int t = blockIdx.y;
  const Rect rc = tile_rect(t, d.ny, d.nx, d.ty, d.tx);
  const int W = rc.x1 - rc.x0;
  const int ya = rc.y0 + blockIdx.x * kInitRows;
  const int yb = min(rc.y1, ya + kInitRows);
  float best_a = -1.f, best_v = 0.f;
  int best_i = 0x7fffffff;
  int bad = 0;
  const int y = ya + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (y < yb) {
    const int64_t row = (int64_t)y * d.nx + rc.x0;
    constexpr int U = 4;
#pragma unroll 1
    for (int c = lane; c < W; c += 32 * U) {
      float v[U];
#pragma unroll
      for (int j = 0; j < U; ++j)
        v[j] = c + 32 * j < W ? dirty[row + c + 32 * j] : 0.f;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (c + 32 * j >= W) break;
        const int64_t gi = row + c + 32 * j;
        d.R[gi] = v[j];
        d.model[gi] = 0.f;
        if (!isfinite(v[j])) bad = 1;
        const float a = fabsf(v[j]);
        if (a > best_a) {  // columns ascend: the first keeps a tie
          best_a = a;
          best_i = (int)gi;
          best_v = v[j];
        }
      }
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&d.st->status, ST_NONFINITE_DIRTY);
  uint64_t k = best_a >= 0.f ? make_key(best_v, best_i) : 0ull;
  k = warp_max_key(k);
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = k;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t m = 0;
    for (int w = 0; w < kInitThreads / 32; ++w) m = umax64(m, s_warp[w]);
    if (m) atomicMax((unsigned long long*)&d.peak[t], (unsigned long long)m);
  }
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    const int64_t T = d.T;
    for (int s = threadIdx.x; s < d.T; s += kInitThreads) {
      d.budget[s] = niter / T + ((int64_t)s < niter % T ? 1 : 0);
      d.rcount[s] = 0;
      d.gbar[s] = 0u;
    }
    if (threadIdx.x == 0) {
      d.st->active = 1;
      d.st->max_budget = niter / T + (niter % T ? 1 : 0);
    }
  }
}

__global__ void validate_psf_kernel(const float* __restrict__ P, int64_t n, int64_t centre,
                                    int32_t* status) {
  const float pc = P[centre];
  int bad = 0, off = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float v = P[i];
    if (!isfinite(v)) bad = 1;
    if (fabsf(v) > pc) off = 1;
  }
  if (!isfinite(pc)) bad = 1;
  bad = __syncthreads_or(bad);
  off = __syncthreads_or(off);
  if (threadIdx.x == 0) {
    if (bad) atomicOr(status, ST_NONFINITE_PSF);
    if (off) atomicOr(status, ST_PSF_OFFCENTRE);
  }
}

// Restore: out[q] = R[q] + sum over offsets o in the disc |o| <= r of
// model[q - o] * B(o), B the clean beam (symmetric, so B(o) = B(-o)).
//
// A CLEAN model is components on few pixels, so a block of output pixels goes
// through the model window that reaches it some rows at a time, from the last
// row and column backwards, and either lists those rows' non-zero pixels and
// adds their beams or, when they are many, sums the rows whole.  Both add a
// pixel's terms in the order of the full sum (descending rows, then columns);
// the terms left out are zeros, so the sums are those of the full convolution
// bit for bit.  Bound by reading the window while sources are few (2048^2, r 28:
// 0.098 ms at 0.2 % of the pixels, 2.97 with every sum whole), by the taps of the
// rows summed whole when they are many (2.2 ms at 20 to 100 %, 0.18 at 256^2; a
// kernel of lists alone took 14.2 and 3.2 at 100 %, one of full sums 2.97 and
// 0.31).
constexpr int kRList = 2048;         // window pixels looked at in one go, whole rows
constexpr int kRCounts = kRList / 32;
// a listed pixel costs about what kRDense taps of a row summed whole cost (between
// 4 and 6 nothing is slower than the full sum at any density, r 12 to 59, 100^2 to
// 2048^2; at 3 lists were, by up to 15 % at 20 %)
constexpr int kRDense = 5;

// images below this many pixels: smaller blocks, to fill the SMs (256^2, r 12, 10 %:
// 0.07 ms, 0.2 with the larger ones; 2048^2, r 59, 0.2 %: 0.19 with those, 0.37)
constexpr int64_t kRSmallPx = 1 << 20;

// RB x RB output pixels, ROWS of a column to a thread
template <int RB, int ROWS>
__global__ void __launch_bounds__(RB * RB / ROWS, 1024 * ROWS / (RB * RB))
    restore_kernel(PlanDev d, const float* __restrict__ beam, int r, float* __restrict__ out) {
  constexpr int kThreads = RB * RB / ROWS, kWarps = kThreads / 32, kPer = kRList / kThreads;
  extern __shared__ __align__(16) float sm[];
  int4* s_src = reinterpret_cast<int4*>(sm);         // row, column, value of each source,
  float* s_rows = sm;                                // or the rows
  float* s_beam = sm + 4 * kRList;                   // (2r+1)^2
  __shared__ int s_first[kRCounts + 1];              // sources before each warp's 32 pixels
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = 2 * r + 1, side = RB + 2 * r, most = kRList / side;
  const int y0 = blockIdx.y * RB, x0 = blockIdx.x * RB;
  const int ylast = y0 + RB - 1 + r, xlast = x0 + RB - 1 + r;
  const int tx = threadIdx.x % RB, ty = threadIdx.x / RB * ROWS;
  for (int i = threadIdx.x; i < n * n; i += kThreads) s_beam[i] = beam[i];
  float acc[ROWS];
#pragma unroll
  for (int k = 0; k < ROWS; ++k) acc[k] = 0.f;
  int pr[kPer], pc[kPer];  // the thread's pixels of the rows
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int i = k * kThreads + (int)threadIdx.x;
    pr[k] = i / side;
    pc[k] = i - pr[k] * side;
  }

  for (int w0 = 0; w0 < side; w0 += most) {
    const int rows = min(most, side - w0);
    float v[kPer];
    uint32_t nz[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int yy = ylast - w0 - pr[k], xx = xlast - pc[k];
      v[k] = pr[k] < rows && yy >= 0 && yy < d.ny && xx >= 0 && xx < d.nx
                 ? d.model[(int64_t)yy * d.nx + xx] : 0.f;
    }
    __syncthreads();  // the last rows have been used
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      nz[k] = __ballot_sync(0xffffffffu, v[k] != 0.f);
      if (lane == 0) s_first[k * kWarps + warp] = __popc(nz[k]);
    }
    __syncthreads();
    if (warp == 0) {  // exclusive prefix of the counts
      int carry = 0;
      for (int b = 0; b < kRCounts; b += 32) {
        const int c = s_first[b + lane];
        int s = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, s, o);
          if (lane >= o) s += t;
        }
        s_first[b + lane] = carry + s - c;
        carry += __shfl_sync(0xffffffffu, s, 31);
      }
      if (lane == 0) s_first[kRCounts] = carry;
    }
    __syncthreads();
    const int ns = s_first[kRCounts];
    if (ns == 0) continue;  // the same for the whole block
    // the image's rows among them
    const int j0 = max(ylast - w0 - (d.ny - 1), 0), j1 = min(ylast - w0 + 1, rows);
    const bool whole = ns * kRDense > (j1 - j0) * n;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      if (whole) {
        if (pr[k] < rows) s_rows[k * kThreads + threadIdx.x] = v[k];
      } else if (v[k] != 0.f) {
        const int at = s_first[k * kWarps + warp] + __popc(nz[k] & ((1u << lane) - 1u));
        s_src[at] = make_int4(ylast - w0 - pr[k], xlast - pc[k], __float_as_int(v[k]), 0);
      }
    }
    __syncthreads();
    if (whole) {
      for (int j = j0; j < j1; ++j) {
        const int oy = y0 + ty - (ylast - w0 - j) + r;  // the first row's; a warp's own
        if (oy + ROWS <= 0 || oy >= n) continue;
        const float* m = s_rows + j * side + RB - 1 - tx;
        const float* bp = s_beam + oy * n;
        if (oy >= 0 && oy + ROWS <= n) {
#pragma unroll 2
          for (int o = 0; o < n; ++o) {
            const float mv = m[o];
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
              const float b = bp[k * n + o];
              if (b != 0.f) acc[k] = fmaf(mv, b, acc[k]);
            }
          }
        } else {
#pragma unroll
          for (int k = 0; k < ROWS; ++k) {
            if ((unsigned)(oy + k) >= (unsigned)n) continue;
#pragma unroll 4
            for (int o = 0; o < n; ++o) {
              const float b = bp[k * n + o];
              if (b != 0.f) acc[k] = fmaf(m[o], b, acc[k]);
            }
          }
        }
      }
    } else {
      for (int j = 0; j < ns; ++j) {
        const int4 c = s_src[j];
        const int oy = y0 + ty - c.x + r, ox = x0 + tx - c.y + r;
        if (oy + ROWS <= 0 || oy >= n || (unsigned)ox >= (unsigned)n) continue;
        const float m = __int_as_float(c.z);
#pragma unroll
        for (int k = 0; k < ROWS; ++k) {
          if ((unsigned)(oy + k) < (unsigned)n) {
            const float b = s_beam[(oy + k) * n + ox];
            if (b != 0.f) acc[k] = fmaf(m, b, acc[k]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < ROWS; ++k) {
    const int y = y0 + ty + k, x = x0 + tx;
    if (y < d.ny && x < d.nx)
      out[(int64_t)y * d.nx + x] = d.R[(int64_t)y * d.nx + x] + acc[k];
  }
}

__global__ void beam_table_kernel(float* beam, int r, float smaj, float smin, float pa) {
  const int n = 2 * r + 1;
  const float c = cosf(pa), s = sinf(pa);
  for (int i = threadIdx.x + blockIdx.x * blockDim.x; i < n * n; i += blockDim.x * gridDim.x) {
    const int oy = i / n - r, ox = i % n - r;
    float v = 0.f;
    if (oy * oy + ox * ox <= r * r) {
      const float u = ox * c + oy * s, w = -ox * s + oy * c;
      v = expf(-0.5f * ((u / smaj) * (u / smaj) + (w / smin) * (w / smin)));
    }
    beam[i] = v;
  }
}

// The flux-trigger level of the first round: trigger x the largest |peak|
// among the tiles that can run (budget left, |peak| > threshold).
__global__ void first_level_kernel(PlanDev d) {
  __shared__ uint32_t s_top;
  if (threadIdx.x == 0) s_top = 0u;
  __syncthreads();
  uint32_t top = 0u;
  for (int s = threadIdx.x; s < d.T; s += blockDim.x) {
    const uint64_t pk = d.peak[s];
    if (d.budget[s] > 0 && pk != 0ull && key_abs(pk) > d.thr) top = max(top, (uint32_t)(pk >> 32));
  }
  if (top) atomicMax(&s_top, top);
  __syncthreads();
  if (threadIdx.x == 0) d.st->level = __fmul_rn(d.trigger, __uint_as_float(s_top));
}

}  // namespace

cudaError_t launch_first_level(const PlanDev& d, cudaStream_t s) {
  if (!(d.trigger > 0.f)) return cudaSuccess;
  first_level_kernel<<<1, 256, 0, s>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_init(const PlanDev& d, const float* dirty, int64_t niter, cudaStream_t s) {
  int maxH = 0;
  for (int i = 0; i < d.ty; ++i)
    maxH = max(maxH, (int)(((int64_t)(i + 1) * d.ny) / d.ty - ((int64_t)i * d.ny) / d.ty));
  dim3 grid((maxH + kInitRows - 1) / kInitRows, d.T, 1);
  init_kernel<<<grid, kInitThreads, 0, s>>>(d, dirty, niter);
  return cudaGetLastError();
}

cudaError_t launch_validate_psf(const PlanDev& d, cudaStream_t s) {
  const int64_t n = (int64_t)d.pny * d.pnx;
  const int64_t centre = (int64_t)d.cy * d.pnx + d.cx;
  int blocks = (int)std::min<int64_t>((n + 255) / 256, 4096);
  validate_psf_kernel<<<blocks, 256, 0, s>>>(d.P, n, centre, &d.st->status);
  return cudaGetLastError();
}

// Beam table scratch: a plan-owned buffer of (2r+1)^2 floats is passed in.
cudaError_t launch_restore_with(const PlanDev& d, float bmaj, float bmin, float bpa,
                                float* beam_buf, int r, float* out, cudaStream_t s) {
  const float k = 1.0f / (2.0f * sqrtf(2.0f * logf(2.0f)));
  beam_table_kernel<<<8, 256, 0, s>>>(beam_buf, r, bmaj * k, bmin * k, bpa);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(int4) * kRList + sizeof(float) * (size_t)(2 * r + 1) * (2 * r + 1);
  auto launch = [&](auto kernel, int side, int threads) {
    const cudaError_t err = allow_max_smem((const void*)kernel);
    if (err != cudaSuccess) return err;
    const dim3 grid((d.nx + side - 1) / side, (d.ny + side - 1) / side, 1);
    kernel<<<grid, threads, smem, s>>>(d, beam_buf, r, out);
    return cudaGetLastError();
  };
  if ((int64_t)d.ny * d.nx < kRSmallPx) return launch(restore_kernel<32, 4>, 32, 256);
  return launch(restore_kernel<64, 8>, 64, 512);
}

}  // namespace cleangb
