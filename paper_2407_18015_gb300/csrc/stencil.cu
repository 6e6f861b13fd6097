// stencil.cu -- minimum / maximum probability fields with the six- or
// eight-neighbour stencil of a 2D grid or the six axis neighbours of a 3D
// grid (the extension named in the paper's Sec. "Conclusion").
//
// The parameters come from the statistics pass (fit_kernel over all D*H*W
// vertices) or from the caller.  Uniform and Epanechnikov: one vertex per
// thread, which reads its own and its K neighbours' parameters through the
// read-only cache, where a neighbour's values are shared by the K+1 threads
// that read them.  Histograms (stencil_hist_tiles): tiles with per-bin rows in
// shared memory, walked as the four-neighbour forward walks them; histograms
// of more bins than the rows' shared memory takes keep tail tables in global
// memory (a table pass, then one vertex per thread).
#include <algorithm>
#include <atomic>

#include "device.cuh"
#include "launch.h"
#include "stencil.cuh"
#include "tile.cuh"

namespace ucp {

namespace {

__device__ __forceinline__ float nanf_() { return __int_as_float(0x7fc00000); }

// tail table of every vertex (one row of hist_table_row(B) floats each)
__global__ void __launch_bounds__(256) hist_table_kernel(const float *__restrict__ params,
                                                         long long V, int B,
                                                         float *__restrict__ tab) {
  const int R = hist_table_row(B);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (long long)gridDim.x * blockDim.x) {
    const float a = params[i], b = params[V + i];
    uint8_t st = (!isfinite(a) || !isfinite(b)) ? V_NONFINITE
                                               : (a > b ? V_BAD : (a == b ? V_DEGENERATE : 0));
    float t = 0.f;
    for (int q = 0; q < B; ++q) {
      const float w = params[(2 + q) * V + i];
      if (!isfinite(w)) st |= V_NONFINITE;
      else if (w < 0.f) st |= V_BAD;
      t += w;
    }
    float *row = tab + i * R;
    const bool point = a == b;
    float c = 0.f;
    for (int q = 0; q < B; ++q) {
      row[q] = point ? 0.f : t - c;
      c += params[(2 + q) * V + i];
    }
    row[B] = 0.f;
    row[B + 1] = 0.f;
    row[B + 2] = t;
    row[B + 3] = (float)st;
  }
}

// status bits of uniform / Epanechnikov parameters (a, b) = (p0, p1)
template <int MODEL>
__device__ __forceinline__ uint8_t check2(float a, float b) {
  if (!isfinite(a) || !isfinite(b)) return V_NONFINITE;
  if (MODEL == kUniform) return a > b ? V_BAD : (a == b ? V_DEGENERATE : 0);
  return b < 0.f ? V_BAD : (b == 0.f ? V_DEGENERATE : 0);
}

template <int MODEL, int ST>
__global__ void __launch_bounds__(128) stencil_kernel(StencilField f) {
  constexpr int K = stencil_k(ST);
  const long long V = f.V, HW = (long long)f.H * f.W;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (long long)gridDim.x * blockDim.x) {
    const int z = (int)(i / HW);
    const long long r = i - (long long)z * HW;
    const int y = (int)(r / f.W), x = (int)(r - (long long)y * f.W);
    long long nidx[K];
    bool present[K];
    int k = 0;
#pragma unroll
    for (int n = 0; n < K; ++n) {
      const int dz = kStencilOff[ST][n][0], dy = kStencilOff[ST][n][1],
                dx = kStencilOff[ST][n][2];
      const int zz = z + dz, yy = y + dy, xx = x + dx;
      present[n] = zz >= 0 && zz < f.D && yy >= 0 && yy < f.H && xx >= 0 && xx < f.W;
      nidx[n] = present[n] ? i + dz * HW + (long long)dy * f.W + dx : i;
      k += present[n];
    }
    const bool zero = f.boundary == 1 && k < K;
    float pmin = 0.f, pmax = 0.f;
    uint8_t st;
    if constexpr (MODEL == kHist) {
      const int B = f.B, R = hist_table_row(B);
      const long long crow = i * R;
      st = (uint8_t)__ldg(f.tab + crow + B + 3);
      float T[K];
#pragma unroll
      for (int n = 0; n < K; ++n) {
        T[n] = 2.f;  // CDF complement 2 - 1 = 1 for an absent neighbour
        if (!present[n]) continue;
        st |= (uint8_t)__ldg(f.tab + nidx[n] * R + B + 3) & (V_NONFINITE | V_BAD);
        T[n] = __ldg(f.tab + nidx[n] * R + B + 2);
      }
      if (st & (V_NONFINITE | V_BAD)) {
        pmin = pmax = nanf_();
      } else if (!zero) {
        const float lo1 = __ldg(f.params + i), hi1 = __ldg(f.params + V + i);
        if (lo1 == hi1) {
          float gm = __ldg(f.tab + crow + B + 2), gM = gm;
#pragma unroll
          for (int n = 0; n < K; ++n) {
            if (!present[n]) continue;
            float gt, lt;
            hist_tails_row(f.tab, nidx[n] * R, B, __ldg(f.params + nidx[n]),
                           __ldg(f.params + V + nidx[n]), T[n], lo1, gt, lt);
            gm *= gt;
            gM *= lt;
          }
          pmin = gm;
          pmax = gM;
        } else {
          HistSegG nw[K];
#pragma unroll
          for (int n = 0; n < K; ++n) {
            HistSegG &h = nw[n];
            if (!present[n]) {
              h.init_absent(crow, (float)B);
              continue;
            }
            const float lo = __ldg(f.params + nidx[n]), hi = __ldg(f.params + V + nidx[n]);
            h.init(f.tab, nidx[n] * R, lo - lo1, lo == hi ? 0.f : (hi - lo) / (float)B, T[n]);
            // move to the segment that contains x = 0
            for (int g = 0; g <= B && h.nx <= 0.f; ++g)
              if (!h.step(f.tab, h.nx, (float)B)) break;
          }
          hist_walk_k<K>(f.tab, crow, B, hi1 - lo1, nw, T, f.cptypes, pmin, pmax);
        }
      }
    } else {
      const float c0 = __ldg(f.params + i), c1 = __ldg(f.params + V + i);
      st = check2<MODEL>(c0, c1);
      float p0[K], p1[K];
#pragma unroll
      for (int n = 0; n < K; ++n) {
        p0[n] = __ldg(f.params + nidx[n]);
        p1[n] = __ldg(f.params + V + nidx[n]);
        if (present[n]) st |= check2<MODEL>(p0[n], p1[n]) & (V_NONFINITE | V_BAD);
      }
      if (st & (V_NONFINITE | V_BAD)) {
        pmin = pmax = nanf_();
      } else if (!zero) {
        if constexpr (MODEL == kUniform) {
          UniParams nb[K];
#pragma unroll
          for (int n = 0; n < K; ++n) nb[n] = UniParams{p0[n], p1[n]};
          uniform_vertex_k<K>(UniParams{c0, c1}, nb, present, f.cptypes, pmin, pmax);
        } else {
          EpanParams nb[K];
#pragma unroll
          for (int n = 0; n < K; ++n) nb[n] = EpanParams{p0[n], p1[n]};
          epan_vertex_k<K>(EpanParams{c0, c1}, nb, present, f.cptypes, pmin, pmax);
        }
      }
    }
    if ((f.cptypes & kMin) && f.out_min) f.out_min[i] = pmin;
    if ((f.cptypes & kMax) && f.out_max) f.out_max[i] = pmax;
    if (f.status) f.status[i] = st;
  }
}

// Tiles of the histogram kernel.  2D stencils: 8 x 32 vertices with a
// one-vertex frame, 10 x 34 staged slots.  3D: 2 x 4 x 32 vertices; staged are
// both slices with their frames (2 x 6 x 34 slots) and the vertices below and
// above (2 x 4 x 32): 664 slots, 106 KB of rows and parameters at 8 bins.
template <int ST>
struct HistTile {
  static constexpr bool flat = ST != kStencil3D6;
  static constexpr int slice = flat ? 340 : 204;  // slots of one slice with its frame
  static constexpr int slots = flat ? slice : 2 * slice + 256;
  static constexpr int RS = hist_r4_stride(slots);
  static constexpr int TY = flat ? 8 : 4, TZ = flat ? 1 : 2;
  static size_t smem(int B) {
    return ((size_t)4 * hist_r4_rows(B) * RS + 4 * slots) * sizeof(float);
  }
};

// Histogram tile: the per-bin rows of every staged vertex from the parameters
// (registers, then shared memory), then one vertex per thread.  Two CTAs per
// SM: the walkers of eight neighbours need the registers.  Bound by
// instruction issue; against tail tables in global memory, where every step
// of every walker read its table through L1 whether it crossed or not: 1024
// x 1024 x 20, 8 bins, eight neighbours 1.02 -> 0.50 ms, fit included.
template <int ST, int RB, int MODE>
__global__ void __launch_bounds__(NTHREADS, 2) stencil_hist_kernel(StencilField f, int tiles_x,
                                                                   int tiles_y) {
  using T_ = HistTile<ST>;
  constexpr int K = stencil_k(ST), HX = 34, SLOTS = T_::slots, RS = T_::RS;
  extern __shared__ __align__(16) float smem[];
  const int B = f.B;
  float4 *R4 = reinterpret_cast<float4 *>(smem);
  float *sm = smem + 4 * hist_r4_rows(B) * RS;  // lo, hi, T, status
  int tile = blockIdx.x;
  const int tx0 = tile % tiles_x * 32;
  tile /= tiles_x;
  const int ty0 = tile % tiles_y * T_::TY, tz0 = tile / tiles_y * T_::TZ;
  const long long HW = (long long)f.H * f.W;
  Field pf{};
  pf.params = f.params;
  pf.plane = f.V;
  for (int l = threadIdx.x; l < SLOTS; l += NTHREADS) {
    int z = tz0, y, x;
    if (T_::flat || l < 2 * T_::slice) {
      const int s = l % T_::slice, r = s / HX;
      z += T_::flat ? 0 : l / T_::slice;
      y = ty0 + r - 1;
      x = tx0 + s - r * HX - 1;
    } else {
      const int s = l - 2 * T_::slice;
      z += s < 128 ? -1 : 2;
      y = ty0 + (s & 127) / 32;
      x = tx0 + (s & 31);
    }
    if (z < 0 || z >= f.D || y < 0 || y >= f.H || x < 0 || x >= f.W) continue;
    HistParamRegs<RB> P;
    const long long gi = z * HW + (long long)y * f.W + x;
    if (B == RB) {
      P.template load<true>(pf, gi, B, false);
      hist_rows_build_regs<SLOTS, RS, RB, true>(P, sm, R4, l, B);
    } else {
      P.template load<false>(pf, gi, B, false);
      hist_rows_build_regs<SLOTS, RS, RB, false>(P, sm, R4, l, B);
    }
  }
  __syncthreads();
  const int v = threadIdx.x, vx = v & 31;
  const int vy = (v >> 5) % T_::TY, vz = (v >> 5) / T_::TY;
  const int x = tx0 + vx, y = ty0 + vy, z = tz0 + vz;
  if (x >= f.W || y >= f.H || z >= f.D) return;
  const int l = vz * T_::slice + (vy + 1) * HX + vx + 1;
  const long long gi = z * HW + (long long)y * f.W + x;
  int nl[K];
  bool present[K];
  int k = 0;
  uint8_t st = (uint8_t)sm[3 * SLOTS + l];
#pragma unroll
  for (int n = 0; n < K; ++n) {
    const int dz = kStencilOff[ST][n][0], dy = kStencilOff[ST][n][1], dx = kStencilOff[ST][n][2];
    const int zz = z + dz, yy = y + dy, xx = x + dx;
    present[n] = zz >= 0 && zz < f.D && yy >= 0 && yy < f.H && xx >= 0 && xx < f.W;
    if (T_::flat || dz == 0) nl[n] = l + dy * HX + dx;
    else if ((vz == 0) == (dz > 0)) nl[n] = l + dz * T_::slice;  // the tile's other slice
    else nl[n] = 2 * T_::slice + (dz > 0 ? 128 : 0) + vy * 32 + vx;
    k += present[n];
    if (present[n]) st |= (uint8_t)sm[3 * SLOTS + nl[n]] & (V_NONFINITE | V_BAD);
  }
  float pmin = 0.f, pmax = 0.f;
  const float lo1 = sm[l], hi1 = sm[SLOTS + l];
  if (st & (V_NONFINITE | V_BAD)) {
    pmin = pmax = nanf_();
  } else if (!(f.boundary == 1 && k < K)) {
    if (lo1 == hi1) {
      float gm = sm[2 * SLOTS + l], gM = gm;
#pragma unroll 1
      for (int n = 0; n < K; ++n) {
        if (!present[n]) continue;
        float gt, lt;
        hist_tails_at_rows(R4 + nl[n], RS, B, sm[nl[n]], sm[SLOTS + nl[n]], sm[2 * SLOTS + nl[n]],
                           lo1, gt, lt);
        gm *= gt;
        gM *= lt;
      }
      pmin = gm;
      pmax = gM;
    } else {
      HistRowWalker nw[K];
#pragma unroll
      for (int n = 0; n < K; ++n) {
        if (!present[n]) {
          nw[n].init_absent();
          continue;
        }
        const float lo = sm[nl[n]], hi = sm[SLOTS + nl[n]];
        nw[n].init(R4 + nl[n], lo - lo1, sm[2 * SLOTS + nl[n]]);
        nw[n].template seek0<RS>(R4 + nl[n], B, lo == hi ? 0.f : (hi - lo) * (1.f / (float)B));
      }
      hist_walk_rows_k<K, RS, MODE>(R4 + l, B, hi1 - lo1, nw, pmin, pmax);
    }
  }
  if ((f.cptypes & kMin) && f.out_min) f.out_min[gi] = pmin;
  if ((f.cptypes & kMax) && f.out_max) f.out_max[gi] = pmax;
  if (f.status) f.status[gi] = st;
}

template <int ST, int RB, int MODE>
cudaError_t launch_hist_tiles_t(const StencilField &f, cudaStream_t s) {
  using T_ = HistTile<ST>;
  // per device: the attribute is set once (host threads may race to set it;
  // setting it twice is harmless, the flag itself is atomic)
  static std::atomic<bool> attr_set[128] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(stencil_hist_kernel<ST, RB, MODE>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T_::smem(RB));
    if (e != cudaSuccess) {
      cudaGetLastError();
      return e;
    }
    attr_set[dev].store(true, std::memory_order_release);
  }
  const long long tx = (f.W + 31) / 32, ty = (f.H + T_::TY - 1) / T_::TY,
                  tz = (f.D + T_::TZ - 1) / T_::TZ;
  if (tx * ty * tz > 0x7fffffffLL) return cudaErrorInvalidValue;
  stencil_hist_kernel<ST, RB, MODE>
      <<<(int)(tx * ty * tz), NTHREADS, T_::smem(f.B), s>>>(f, (int)tx, (int)ty);
  return cudaGetLastError();
}

template <int ST, int RB>
cudaError_t launch_hist_tiles_m(const StencilField &f, cudaStream_t s) {
  if (f.cptypes == kMin) return launch_hist_tiles_t<ST, RB, kWalkMin>(f, s);
  if (f.cptypes == kMax) return launch_hist_tiles_t<ST, RB, kWalkMax>(f, s);
  return launch_hist_tiles_t<ST, RB, kWalkBoth>(f, s);
}

cudaError_t launch_hist_tiles(const StencilField &f, int stencil, cudaStream_t s) {
  switch (stencil) {
    case kStencil6:
      return f.B <= 8 ? launch_hist_tiles_m<kStencil6, 8>(f, s)
                      : launch_hist_tiles_m<kStencil6, 16>(f, s);
    case kStencil8:
      return f.B <= 8 ? launch_hist_tiles_m<kStencil8, 8>(f, s)
                      : launch_hist_tiles_m<kStencil8, 16>(f, s);
    case kStencil3D6: return launch_hist_tiles_m<kStencil3D6, 8>(f, s);
    default: return cudaErrorInvalidValue;
  }
}

int grid_blocks(long long n, int threads, int sm_count, int per_sm) {
  long long b = (n + threads - 1) / threads;
  const long long cap = (long long)sm_count * per_sm;
  if (b > cap) b = cap;
  return (int)(b < 1 ? 1 : b);
}

template <int MODEL>
cudaError_t launch_model(const StencilField &f, int stencil, int blocks, cudaStream_t s) {
  switch (stencil) {
    case kStencil6: stencil_kernel<MODEL, kStencil6><<<blocks, 128, 0, s>>>(f); break;
    case kStencil8: stencil_kernel<MODEL, kStencil8><<<blocks, 128, 0, s>>>(f); break;
    case kStencil3D6: stencil_kernel<MODEL, kStencil3D6><<<blocks, 128, 0, s>>>(f); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_hist_table(const float *params, long long V, int B, float *tab, int sm_count,
                              cudaStream_t s) {
  hist_table_kernel<<<grid_blocks(V, 256, sm_count, 8), 256, 0, s>>>(params, V, B, tab);
  return cudaGetLastError();
}

// Rows of two CTAs per SM: 99 KB at 16 bins for the 2D stencils, 106 KB at 8
// bins for the 3D one (whose tile has more staged vertices).
bool stencil_hist_tiles(int stencil, int B) { return B <= (stencil == kStencil3D6 ? 8 : 16); }

cudaError_t launch_stencil(const StencilField &f, int model, int stencil, int sm_count,
                           cudaStream_t s) {
  if (model == kHist && stencil_hist_tiles(stencil, f.B)) return launch_hist_tiles(f, stencil, s);
  const int blocks = grid_blocks(f.V, 128, sm_count, 16);
  switch (model) {
    case kUniform: return launch_model<kUniform>(f, stencil, blocks, s);
    case kEpan: return launch_model<kEpan>(f, stencil, blocks, s);
    case kHist: return launch_model<kHist>(f, stencil, blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ucp
