// mvn.cu -- multivariate Gaussian model over (X_v, X_e, X_n, X_w, X_s):
// per-vertex mean and covariance (the fit), Cholesky factor, and Monte
// Carlo estimates of P_min / P_max, the approach of the prior work the paper
// compares against (Sec. "Comparison of Parametric Vs. Nonparametric
// Models", multivariate Gaussian with Monte Carlo sampling).
//
// One warp per vertex.  Lanes split the samples, one or two per turn; each sample
// draws two Philox4x32-10 blocks (counter (s, vertex, field, j), key = seed),
// maps the words to uniforms ((r >> 9) + 0.5) 2^-23 (exact in binary32, inside
// (0, 1)), and Box-Muller gives six normals, five of which are used.  The
// comparisons x_v < x_n are evaluated on the differences y_n = x_v - x_n =
// (mu_v - mu_n) + (L_v. - L_n.) z; every lane counts its hits, and the counts
// are added over the warp at the end.
#include "device.cuh"
#include "launch.h"

namespace ucp {

// The two blocks of one sample: counters (s, v, field, 0) and (s, v, field, 1)
// differ only in the last word, so the first round's products are shared.
__device__ __forceinline__ void philox_pair(uint32_t s, uint32_t v, uint32_t field,
                                            const PhiloxKeys &K, uint4 &r0, uint4 &r1) {
  const uint32_t hi0 = __umulhi(0xD2511F53u, s), lo0 = 0xD2511F53u * s;
  const uint32_t hi1 = __umulhi(0xCD9E8D57u, field), lo1 = 0xCD9E8D57u * field;
  const uint32_t a = hi1 ^ v ^ K.k0[0];
  r0 = make_uint4(a, lo1, hi0 ^ K.k1[0], lo0);
  r1 = make_uint4(a, lo1, hi0 ^ 1u ^ K.k1[0], lo0);
#pragma unroll
  for (int r = 1; r < 10; ++r) {
    philox_round(r0, K.k0[r], K.k1[r]);
    philox_round(r1, K.k0[r], K.k1[r]);
  }
}

// Arithmetic of the samples of one lane and turn, every operation rounded
// once: two (PAIR, one per half of a float2) or one, to the same bits.
template <bool PAIR>
struct McOps {
  static constexpr int n = 2;
  using V = float2;
  static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
  static __device__ __forceinline__ V all(float a) { return make_float2(a, a); }
  static __device__ __forceinline__ float &at(V &a, int h) { return h == 0 ? a.x : a.y; }
};
template <>
struct McOps<false> {
  static constexpr int n = 1;
  using V = float;
  static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ V all(float a) { return a; }
  static __device__ __forceinline__ float &at(V &a, int) { return a; }
};

// A Philox word as 1 + m 2^-23, m its upper 23 bits: the uniform is this minus
// 1 - 2^-24, exactly.
__device__ __forceinline__ float word_float(uint32_t r) {
  return __uint_as_float((r >> 9) + 0x3f800000u);
}

// Box-Muller of a turn's samples, wa and wb their words as word_float gives
// them: radius sqrt(-2 ln ua), angle 2 pi ub.  The angle is taken as pi + t with t = 2 pi (ub - 1/2) in [-pi, pi), where the
// hardware sine and cosine are accurate to ~4e-7 absolute: cos(2 pi ub) = -cos
// t, sin(2 pi ub) = -sin t.  ub - 1/2 = (wb - 3/2) + 2^-24 exactly, so one
// multiply-add gives t with the rounding of the product.  The logarithm keeps
// full accuracy (its error is not bounded relative to the radius near ub ->
// 1).  Z1: also the second normal.
template <typename O, bool Z1, typename V>
__device__ __forceinline__ void box_muller(V wa, V wb, V &z0, V &z1) {
  const float twopi = 6.283185307179586f;
  V ua = O::add(wa, O::all(-(1.f - 0x1p-24f))), ln, rs, sn, cs;
#pragma unroll
  for (int h = 0; h < O::n; ++h) O::at(ln, h) = logf(O::at(ua, h));
  V v = O::mul(O::all(-2.f), ln);
#pragma unroll
  for (int h = 0; h < O::n; ++h) O::at(rs, h) = rsqrtf(O::at(v, h));
  V rad = O::mul(v, rs);
  V t = O::fma(O::add(wb, O::all(-1.5f)), O::all(twopi), O::all(twopi * 0x1p-24f));
#pragma unroll
  for (int h = 0; h < O::n; ++h) {
    __sincosf(O::at(t, h), &O::at(sn, h), &O::at(cs, h));
    O::at(rad, h) = -O::at(rad, h);
  }
  z0 = O::mul(rad, cs);
  if constexpr (Z1) z1 = O::mul(rad, sn);
}

// Slots of the variables: 0 = v, 1..4 = e, n, w, s.  Returns the number of
// present variables and their slots in order.
__device__ __forceinline__ int mvn_slots(const Field &f, int y, int x, int *slot,
                                         long long *gidx) {
  int nv = 1;
  slot[0] = 0;
  gidx[0] = (long long)y * f.W + x;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const int yy = y + kDy[d], xx = x + kDx[d];
    if (yy >= 0 && yy < f.H && xx >= 0 && xx < f.W) {
      slot[nv] = 1 + d;
      gidx[nv] = (long long)yy * f.W + xx;
      ++nv;
    }
  }
  return nv;
}

__device__ __forceinline__ int packed(int a, int b) {  // a >= b
  return a * (a + 1) / 2 + b;
}

// Cholesky of the nv x nv matrix A (row-major, 5x5 storage) into L.
__device__ __forceinline__ bool chol5(const float (&A)[5][5], int nv, float (&L)[5][5]) {
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j < 5; ++j) L[i][j] = 0.f;
  bool ok = true;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    if (j >= nv) break;
    float s = A[j][j];
#pragma unroll
    for (int k = 0; k < j; ++k) s = fmaf(-L[j][k], L[j][k], s);
    if (!(s > 0.f)) {
      ok = false;
      break;
    }
    const float d = sqrtf(s);
    L[j][j] = d;
#pragma unroll
    for (int i = j + 1; i < 5; ++i) {
      if (i >= nv) break;
      float t = A[i][j];
#pragma unroll
      for (int k = 0; k < j; ++k) t = fmaf(-L[i][k], L[j][k], t);
      L[i][j] = t / d;
    }
  }
  return ok;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// fit: mean and covariance (N-1) of the present variables, thread per vertex

__global__ void __launch_bounds__(256) mvn_fit_kernel(Field f) {
  float *out = const_cast<float *>(f.params);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < f.plane;
       i += (long long)gridDim.x * blockDim.x) {
    const int y = (int)(i / f.W), x = (int)(i % f.W);
    int slot[5];
    long long g[5];
    const int nv = mvn_slots(f, y, x, slot, g);
    float mu[5] = {0, 0, 0, 0, 0};
    bool nf = false;
    for (int a = 0; a < nv; ++a) {
      float s = 0.f;
      for (int k = 0; k < f.N; ++k) {
        const float v = __ldg(f.ens + (long long)k * f.plane + g[a]);
        nf |= !isfinite(v);
        s += v;
      }
      mu[a] = s / (float)f.N;
    }
    float full_mu[5] = {0, 0, 0, 0, 0};
    for (int a = 0; a < nv; ++a) full_mu[slot[a]] = mu[a];
    for (int q = 0; q < 5; ++q) out[q * f.plane + i] = nf ? __int_as_float(0x7fc00000) : full_mu[q];
    float C[15];
    for (int q = 0; q < 15; ++q) C[q] = 0.f;
    if (f.N > 1) {
      for (int k = 0; k < f.N; ++k) {
        float dv[5];
        for (int a = 0; a < nv; ++a) dv[a] = __ldg(f.ens + (long long)k * f.plane + g[a]) - mu[a];
        for (int a = 0; a < nv; ++a)
          for (int b = 0; b <= a; ++b) C[packed(slot[a], slot[b])] += dv[a] * dv[b];
      }
      for (int q = 0; q < 15; ++q) C[q] /= (float)(f.N - 1);
    }
    for (int q = 0; q < 15; ++q)
      out[(5 + q) * f.plane + i] = nf ? __int_as_float(0x7fc00000) : C[q];
    if (f.status) f.status[i] = nf ? V_NONFINITE : 0;
  }
}

// ---------------------------------------------------------------------------
// Monte Carlo, warp per vertex

// Hits of this lane's samples (lane, lane + 32, ...): minimum and maximum, or
// (SADDLE) the saddle in h0.  D, M: y_n = D[n] + sum_b M[n][b] z_b of the nv
// present variables; FULL: nv = 5 (no test per neighbour).  Bound by
// instruction issue, about 240 a sample, 35 of them 64-bit Philox products
// (four FP32-pipe cycles each): with two samples per turn (PAIR) every FP32
// operation but the logarithms and the special functions is a packed one (the
// same roundings as one by one): 512 x 512 x 40, 10^4 samples 22.2 ->
// 19.4 ms.
template <bool SADDLE, bool FULL, bool PAIR>
__device__ __forceinline__ void mc_count(int S, int lane, uint32_t vid, uint32_t field,
                                         const PhiloxKeys &K, const float *D,
                                         const float (&M)[5][5], int nv, const float *ssg,
                                         bool has_saddle, unsigned &h0, unsigned &h1) {
  using O = McOps<PAIR>;
  using V = typename O::V;
  // samples s and, in a pair, s + 32 (computed, but only counted if `second`)
  auto turn = [&](uint32_t s, bool second) {
    V w[2][4];
#pragma unroll
    for (int h = 0; h < O::n; ++h) {
      uint4 r0, r1;
      philox_pair(s + 32u * h, vid, field, K, r0, r1);
      O::at(w[0][0], h) = word_float(r0.x);
      O::at(w[0][1], h) = word_float(r0.y);
      O::at(w[0][2], h) = word_float(r0.z);
      O::at(w[0][3], h) = word_float(r0.w);
      O::at(w[1][0], h) = word_float(r1.x);
      O::at(w[1][1], h) = word_float(r1.y);
    }
    V z[6];
    box_muller<O, true>(w[0][0], w[0][1], z[0], z[1]);
    box_muller<O, true>(w[0][2], w[0][3], z[2], z[3]);
    box_muller<O, false>(w[1][0], w[1][1], z[4], z[5]);
    // x_v below every neighbour: the largest y_n = x_v - x_n is < 0;
    // above every one: the smallest is > 0
    float ymax[O::n], ymin[O::n];
    bool t1[O::n], t2[O::n];
#pragma unroll
    for (int h = 0; h < O::n; ++h) {
      ymax[h] = -kFar;
      ymin[h] = kFar;
      t1[h] = t2[h] = has_saddle;
    }
#pragma unroll
    for (int n = 1; n < 5; ++n) {
      if (FULL || n < nv) {
        V yv = O::all(D[n]);
#pragma unroll
        for (int b = 0; b <= n; ++b) yv = O::fma(O::all(M[n][b]), z[b], yv);
#pragma unroll
        for (int h = 0; h < O::n; ++h) {
          const float y = O::at(yv, h);
          if constexpr (SADDLE) {
            // t1 wants x_v < x_n where the sign is +1
            const float sy = ssg[n] * y;
            t1[h] &= sy < 0.f;
            t2[h] &= sy > 0.f;
          } else {
            ymax[h] = fmaxf(ymax[h], y);
            ymin[h] = fminf(ymin[h], y);
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < O::n; ++h) {
      const bool count = h == 0 || second;
      if constexpr (SADDLE) {
        h0 += (count && (t1[h] || t2[h])) ? 1u : 0u;
      } else {
        h0 += (count && ymax[h] < 0.f) ? 1u : 0u;
        h1 += (count && ymin[h] > 0.f) ? 1u : 0u;
      }
    }
  };
  constexpr uint32_t step = 32 * O::n;
  const uint32_t whole = (uint32_t)S / step * step;
  for (uint32_t s = 0; s < whole; s += step) turn(s + lane, true);
  const uint32_t s = whole + lane;
  if (s < (uint32_t)S) turn(s, s + 32 < (uint32_t)S);
}

template <bool FROM_MEMBERS, bool SADDLE, bool PAIR>
__global__ void __launch_bounds__(256) mvn_mc_kernel(Field f, int S, uint32_t k0, uint32_t k1,
                                                     uint32_t field) {
  const int lane = threadIdx.x & 31;
  const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long vbeg = (long long)f.y0 * f.W, vend = (long long)f.y1 * f.W;
  for (long long v = vbeg + warp0; v < vend; v += nwarps) {
    const int y = (int)(v / f.W), x = (int)(v % f.W);
    int slot[5];
    long long g[5];
    const int nv = mvn_slots(f, y, x, slot, g);
    float mu[5] = {0, 0, 0, 0, 0};
    float A[5][5];
#pragma unroll
    for (int a = 0; a < 5; ++a)
#pragma unroll
      for (int b = 0; b < 5; ++b) A[a][b] = 0.f;
    bool nf = false;
    if (FROM_MEMBERS) {
      float s[5] = {0, 0, 0, 0, 0};
      for (int k = lane; k < f.N; k += 32)
#pragma unroll
        for (int a = 0; a < 5; ++a)
          if (a < nv) {
            const float t = __ldg(f.ens + (long long)k * f.plane + g[a]);
            nf |= !isfinite(t);
            s[a] += t;
          }
#pragma unroll
      for (int a = 0; a < 5; ++a) mu[a] = warp_sum(s[a]) / (float)f.N;
      nf = __any_sync(0xffffffffu, nf);
      float c[15];
#pragma unroll
      for (int q = 0; q < 15; ++q) c[q] = 0.f;
      for (int k = lane; k < f.N; k += 32) {
        float dv[5];
#pragma unroll
        for (int a = 0; a < 5; ++a)
          dv[a] = (a < nv) ? __ldg(f.ens + (long long)k * f.plane + g[a]) - mu[a] : 0.f;
#pragma unroll
        for (int a = 0; a < 5; ++a)
#pragma unroll
          for (int b = 0; b <= a; ++b) c[packed(a, b)] = fmaf(dv[a], dv[b], c[packed(a, b)]);
      }
      const float inv = f.N > 1 ? 1.f / (float)(f.N - 1) : 0.f;
#pragma unroll
      for (int a = 0; a < 5; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          const float t = warp_sum(c[packed(a, b)]) * inv;
          A[a][b] = t;
          A[b][a] = t;
        }
    } else {
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        if (a >= nv) break;
        mu[a] = __ldg(f.params + (long long)slot[a] * f.plane + v);
      }
#pragma unroll
      for (int a = 0; a < 5; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          if (a < nv) {
            const int sa = slot[a], sb = slot[b];
            const int q = sa >= sb ? packed(sa, sb) : packed(sb, sa);
            const float t = __ldg(f.params + (long long)(5 + q) * f.plane + v);
            A[a][b] = t;
            A[b][a] = t;
          }
        }
    }
    float tr = 0.f;
#pragma unroll
    for (int a = 0; a < 5; ++a) {
      if (a < nv) {
        nf |= !isfinite(mu[a]);
        tr += A[a][a];
#pragma unroll
        for (int b = 0; b < 5; ++b)
          if (b < nv) nf |= !isfinite(A[a][b]);
      }
    }
    uint8_t st = nf ? V_NONFINITE : 0;
    float pmin = 0.f, pmax = 0.f, psad = 0.f;
    // saddle sign of each present variable (+1: t1 wants x_v < x_n); a vertex
    // without a saddle neighbourhood counts no saddle hits
    float ssg[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    const bool line = (f.H == 1 || f.W == 1) && nv == 3;
    const bool has_saddle = (nv == 5) || line;
#pragma unroll
    for (int a = 1; a < 5; ++a)
      if (a < nv) {
        const int sl = slot[a];  // 1 e, 2 n, 3 w, 4 s
        ssg[a] = (nv == 5) ? ((sl == 1 || sl == 3) ? 1.f : -1.f)
                           : ((sl == 1 || sl == 4) ? 1.f : -1.f);
      }
    const bool zero_mm = f.boundary == 1 && nv < 5;
    if (nf) {
      pmin = pmax = psad = __int_as_float(0x7fc00000);
    } else if (tr == 0.f) {
      bool lt = true, gt = true, t1 = has_saddle, t2 = has_saddle;
#pragma unroll
      for (int a = 1; a < 5; ++a)
        if (a < nv) {
          lt &= mu[0] < mu[a];
          gt &= mu[0] > mu[a];
          t1 &= ssg[a] > 0.f ? mu[0] < mu[a] : mu[0] > mu[a];
          t2 &= ssg[a] > 0.f ? mu[0] > mu[a] : mu[0] < mu[a];
        }
      pmin = (lt && !zero_mm) ? 1.f : 0.f;
      pmax = (gt && !zero_mm) ? 1.f : 0.f;
      psad = (t1 || t2) ? 1.f : 0.f;
      st |= V_DEGENERATE;
    } else {
      float L[5][5];
      bool ok = chol5(A, nv, L);
      if (!ok) {
        float eps = 1e-6f * tr / (float)nv;
        for (int r = 0; r < 3 && !ok; ++r) {
          float Aj[5][5];
#pragma unroll
          for (int a = 0; a < 5; ++a)
#pragma unroll
            for (int b = 0; b < 5; ++b) Aj[a][b] = A[a][b] + (a == b ? eps : 0.f);
          ok = chol5(Aj, nv, L);
          eps *= 10.f;
        }
        st |= ok ? V_JITTER : V_CHOLFAIL;
      }
      if (!ok) {
        pmin = pmax = psad = __int_as_float(0x7fc00000);
      } else {
        // y_n = x_0 - x_n = D_n + sum_b M[n][b] z_b
        float D[5], M[5][5];
#pragma unroll
        for (int n = 0; n < 5; ++n) {
          D[n] = mu[0] - mu[n];
#pragma unroll
          for (int b = 0; b < 5; ++b) M[n][b] = (b == 0 ? L[0][0] : 0.f) - L[n][b];
        }
        unsigned h0 = 0, h1 = 0;
        const PhiloxKeys K(k0, k1);
        if (nv == 5)
          mc_count<SADDLE, true, PAIR>(S, lane, (uint32_t)v, field, K, D, M, nv, ssg, has_saddle, h0, h1);
        else
          mc_count<SADDLE, false, PAIR>(S, lane, (uint32_t)v, field, K, D, M, nv, ssg, has_saddle, h0, h1);
        const unsigned cmin = __reduce_add_sync(0xffffffffu, h0), csad = cmin;
        const unsigned cmax = __reduce_add_sync(0xffffffffu, h1);
        pmin = zero_mm ? 0.f : (float)cmin / (float)S;
        pmax = zero_mm ? 0.f : (float)cmax / (float)S;
        psad = (float)csad / (float)S;
      }
    }
    if (lane == 0) {
      // each instance writes its own outputs; the status once (by the
      // minimum / maximum instance when it runs)
      if constexpr (!SADDLE) {
        if ((f.cptypes & kMin) && f.out_min) f.out_min[v] = pmin;
        if ((f.cptypes & kMax) && f.out_max) f.out_max[v] = pmax;
        if (f.status) f.status[v] = st;
      } else {
        if (f.out_saddle) f.out_saddle[v] = psad;
        if (f.status && !(f.cptypes & (kMin | kMax))) f.status[v] = st;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// launchers

cudaError_t launch_mvn_fit(const Field &f, cudaStream_t s) {
  long long b = (f.plane + 255) / 256;
  if (b > (1LL << 30)) b = 1LL << 30;
  mvn_fit_kernel<<<(int)b, 256, 0, s>>>(f);
  return cudaGetLastError();
}

// Two samples per turn take 80 to 93 registers a thread (one: 64) and work on
// 64 samples at a time: few samples go one per turn, for the occupancy of the
// part before the samples.  512 x 512 x 20, one and two per turn: minimum and
// maximum 376 and 459 us at 32 samples, 546 and 559 at 128, 737 and 763 at 224,
// 800 and 769 at 256, 2353 and 2192 at 1000; saddle 401 and 568 at 32, 820 and
// 890 at 256, 1337 and 1351 at 512, 1863 and 1811 at 768.
constexpr int kMcPairs = 225, kMcPairsSaddle = 513;

template <bool SADDLE>
static cudaError_t launch_mc(const Field &f, bool from_members, int samples, uint32_t k0,
                             uint32_t k1, uint32_t field_id, int blocks, cudaStream_t s) {
  const bool pair = samples >= (SADDLE ? kMcPairsSaddle : kMcPairs);
  auto k = from_members ? (pair ? mvn_mc_kernel<true, SADDLE, true> : mvn_mc_kernel<true, SADDLE, false>)
                        : (pair ? mvn_mc_kernel<false, SADDLE, true> : mvn_mc_kernel<false, SADDLE, false>);
  k<<<blocks, 256, 0, s>>>(f, samples, k0, k1, field_id);
  return cudaGetLastError();
}

cudaError_t launch_mvn_mc(const Field &f, bool from_members, int samples, uint64_t seed,
                          uint32_t field_id, cudaStream_t s) {
  // one warp per vertex, 8 warps per CTA, grid-stride over vertices
  const long long nvtx = (long long)(f.y1 - f.y0) * f.W;
  if (nvtx <= 0) return cudaSuccess;
  long long b = (nvtx + 7) / 8;
  if (b > (1LL << 30)) b = 1LL << 30;
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  // minimum / maximum and the saddle are separate instances, so that
  // neither pays for the other's tests in the sample loop
  cudaError_t e = cudaSuccess;
  if (f.cptypes & (kMin | kMax))
    e = launch_mc<false>(f, from_members, samples, k0, k1, field_id, (int)b, s);
  if (e == cudaSuccess && (f.cptypes & kSaddle))
    e = launch_mc<true>(f, from_members, samples, k0, k1, field_id, (int)b, s);
  return e;
}

}  // namespace ucp
