// stencil.cuh -- minimum / maximum probabilities with larger neighbour sets:
// the six-neighbour stencil of a triangulated 2D grid, the eight-neighbour
// stencil, and the six axis neighbours of a 3D grid (the extension named in
// the paper's Sec. "Conclusion").  The integrals are those of Eq.
// localMinimumProb with K <= 8 neighbour factors instead of 4; the piece
// integration is the same as in device.cuh, generalised over K.
#pragma once

#include "device.cuh"

namespace ucp {

constexpr int kStencil4 = 0, kStencil6 = 1, kStencil8 = 2, kStencil3D6 = 3;
constexpr int kMaxK = 8;

__host__ __device__ constexpr int stencil_k(int st) {
  return st == kStencil8 ? 8 : (st == kStencil4 ? 4 : 6);
}

// neighbour offsets (dz, dy, dx) of each stencil, the axis ones (e, n, w, s)
// first; stencil 6 adds ne and sw (every cell cut along its lower-left to
// upper-right diagonal), stencil 8 all four diagonals, the 3D one the
// neighbours below (z - 1) and above (z + 1)
__device__ __constant__ const int kStencilOff[4][kMaxK][3] = {
    {{0, 0, 1}, {0, -1, 0}, {0, 0, -1}, {0, 1, 0}},
    {{0, 0, 1}, {0, -1, 0}, {0, 0, -1}, {0, 1, 0}, {0, -1, 1}, {0, 1, -1}},
    {{0, 0, 1}, {0, -1, 0}, {0, 0, -1}, {0, 1, 0}, {0, -1, 1}, {0, -1, -1}, {0, 1, -1},
     {0, 1, 1}},
    {{0, 0, 1}, {0, -1, 0}, {0, 0, -1}, {0, 1, 0}, {-1, 0, 0}, {1, 0, 0}}};

// integral over [0,1] of (1-t)^(K-j) t^j = 1 / ((K+1) C(K,j))
__host__ __device__ constexpr float bern_w(int K, int j) {
  return 1.0f / float((K + 1) * binom(K, j));
}

// exact mean over [0,1] of a product of K linear factors given by their end
// values (the Bernstein form of bern_mean, for K <= 8)
template <int K>
__device__ __forceinline__ float bern_mean_k(const float *L, const float *R) {
  float e[K + 1];
  e[0] = L[0];
  e[1] = R[0];
#pragma unroll
  for (int i = 1; i < K; ++i) {
    e[i + 1] = e[i] * R[i];
#pragma unroll
    for (int j = i; j >= 1; --j) e[j] = fmaf(e[j - 1], R[i], e[j] * L[i]);
    e[0] = e[0] * L[i];
  }
  float s = 0.f;
#pragma unroll
  for (int j = 0; j <= K; ++j) s = fmaf(e[j], bern_w(K, j), s);
  return s;
}

// bern_mean_k of two products at once, one per half of a float2 (the same
// operations per half, packed FP32 instructions)
template <int K>
__device__ __forceinline__ float2 bern_mean_k_x2(const float2 *L, const float2 *R) {
  float2 e[K + 1];
  e[0] = L[0];
  e[1] = R[0];
#pragma unroll
  for (int i = 1; i < K; ++i) {
    e[i + 1] = __fmul2_rn(e[i], R[i]);
#pragma unroll
    for (int j = i; j >= 1; --j) e[j] = __ffma2_rn(e[j - 1], R[i], __fmul2_rn(e[j], L[i]));
    e[0] = __fmul2_rn(e[0], L[i]);
  }
  float2 s = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j <= K; ++j) s = __ffma2_rn(e[j], make_float2(bern_w(K, j), bern_w(K, j)), s);
  return s;
}

// ascending sort of K keys with NP payload rows (odd-even transposition)
template <int NP>
__device__ __forceinline__ void cswap_k(float *k, float (*p)[kMaxK], int a, int b) {
  const bool sw = k[b] < k[a];
  const float ka = k[a], kb = k[b];
  k[a] = sw ? kb : ka;
  k[b] = sw ? ka : kb;
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const float pa = p[q][a], pb = p[q][b];
    p[q][a] = sw ? pb : pa;
    p[q][b] = sw ? pa : pb;
  }
}
template <int K, int NP>
__device__ __forceinline__ void sort_k(float *k, float (*p)[kMaxK]) {
#pragma unroll
  for (int r = 0; r < K; ++r)
#pragma unroll
    for (int i = r & 1; i + 1 < K; i += 2) cswap_k<NP>(k, p, i, i + 1);
}

// ---------------------------------------------------------------------------
// uniform

// piece J of uniform_side_k: [x[J], x[J+1]], on which the sorted factors
// 0..J-1 have started
template <int J, int K>
__device__ __forceinline__ void uni_pieces(const float *x, const float (*pay)[kMaxK], float *Lv,
                                           float *Rv, Kahan &acc) {
  const float x0 = x[J], x1 = x[J + 1];
#pragma unroll
  for (int i = 0; i < J - 1; ++i) Lv[i] = Rv[i];
  Lv[J - 1] = fmaxf(fmaf(-(x0 - pay[0][J - 1]), pay[1][J - 1], 1.f), 0.f);
#pragma unroll
  for (int i = 0; i < J; ++i) Rv[i] = fmaxf(fmaf(-(x1 - pay[0][i]), pay[1][i], 1.f), 0.f);
  acc.add((x1 - x0) * bern_mean_k<J>(Lv, Rv));
  if constexpr (J < K) uni_pieces<J + 1, K>(x, pay, Lv, Rv, acc);
}

// uniform_side with K factors: int_0^R (1/W1) prod_i (1 - max(0, x - al_i) sl_i)
template <int K>
__device__ __forceinline__ float uniform_side_k(float W1, float R, const float *al,
                                                const float *sl) {
  if (!(R > 0.f)) return 0.f;
  float t[kMaxK], pay[2][kMaxK];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    t[i] = fminf(fmaxf(al[i], 0.f), R);
    pay[0][i] = al[i];
    pay[1][i] = sl[i];
  }
  sort_k<K, 2>(t, pay);
  float x[K + 2];
  x[0] = 0.f;
#pragma unroll
  for (int i = 0; i < K; ++i) x[i + 1] = t[i];
  x[K + 1] = R;
  Kahan acc;
  acc.add(x[1]);  // piece 0: no factor has started
  float Lv[K], Rv[K];
  uni_pieces<1, K>(x, pay, Lv, Rv, acc);
  return acc.get() * frcp(W1);
}

// P_min and P_max of a uniform centre with K neighbours (present[i])
template <int K>
__device__ __forceinline__ void uniform_vertex_k(UniParams c, const UniParams *nb,
                                                 const bool *present, unsigned want,
                                                 float &pmin, float &pmax) {
  if (c.a == c.b) {
    const float v = c.a;
    float gm = 1.f, gM = 1.f;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (!present[i]) continue;
      const float a = nb[i].a, b = nb[i].b;
      float gt, lt;
      if (a == b) {
        gt = a > v ? 1.f : 0.f;
        lt = a < v ? 1.f : 0.f;
      } else {
        const float r = 1.f / (b - a);
        gt = fminf(fmaxf((b - v) * r, 0.f), 1.f);
        lt = fminf(fmaxf((v - a) * r, 0.f), 1.f);
      }
      gm *= gt;
      gM *= lt;
    }
    pmin = gm;
    pmax = gM;
    return;
  }
  const float W1 = c.b - c.a;
  float sl[K];
#pragma unroll
  for (int i = 0; i < K; ++i)
    sl[i] = (present[i] && nb[i].a != nb[i].b) ? frcp(nb[i].b - nb[i].a) : 0.f;
  if (want & kMin) {
    float al[K], R = W1;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (present[i]) {
        al[i] = nb[i].a - c.a;
        R = fminf(R, nb[i].b - c.a);
      } else {
        al[i] = kFar;
      }
    }
    pmin = uniform_side_k<K>(W1, R, al, sl);
  }
  if (want & kMax) {
    // negated variables: -X has support [-b, -a]; origin at -b1
    float al[K], R = W1;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (present[i]) {
        al[i] = c.b - nb[i].b;
        R = fminf(R, c.b - nb[i].a);
      } else {
        al[i] = kFar;
      }
    }
    pmax = uniform_side_k<K>(W1, R, al, sl);
  }
}

// ---------------------------------------------------------------------------
// Epanechnikov: with K neighbours the integrand has degree <= 2 + 3K = 26 on
// a piece; each piece takes the smallest rule of {2, 3, 5, 6, 8, 16} nodes that
// is exact for its degree (EpanNodes; the 16-point rule: to degree 31)

// epan_side with K factors (same frame and arguments)
template <int K>
__device__ __forceinline__ float epan_side_k(float w1, float L, float R, const float *al,
                                             const float *d, const float *iw) {
  if (!(R > L)) return 0.f;
  float t[kMaxK], pay[2][kMaxK];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    t[i] = fminf(fmaxf(al[i], L), R);
    pay[0][i] = d[i];
    pay[1][i] = iw[i];
  }
  sort_k<K, 2>(t, pay);
  float x[K + 2];
  x[0] = L;
#pragma unroll
  for (int i = 0; i < K; ++i) x[i + 1] = t[i];
  x[K + 1] = R;
  const EpanInv iw1(w1);
  Kahan acc;
  epan_pieces<0, K, kMaxK>(x, pay, iw1, acc);
  return not_negative(iw1.times(0.75f * acc.get()));
}

template <int K>
__device__ __forceinline__ void epan_vertex_k(EpanParams c, const EpanParams *nb,
                                              const bool *present, unsigned want, float &pmin,
                                              float &pmax) {
  if (c.w == 0.f) {
    const float v = c.m;
    float gm = 1.f, gM = 1.f;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (!present[i]) continue;
      float gt, lt;
      if (nb[i].w == 0.f) {
        gt = nb[i].m > v ? 1.f : 0.f;
        lt = nb[i].m < v ? 1.f : 0.f;
      } else {
        gt = epan_surv((v - nb[i].m) / nb[i].w);
        lt = epan_surv((nb[i].m - v) / nb[i].w);
      }
      gm *= gt;
      gM *= lt;
    }
    pmin = gm;
    pmax = gM;
    return;
  }
  const float w1 = c.w;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    if (!(want & (side == 0 ? kMin : kMax))) continue;
    // side 1: the negated variables, frame of -m1: d = m1 - m_n
    float al[K], d[K], iw[K], R = w1;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      al[i] = kFar; d[i] = kFar; iw[i] = 0.f;
      if (!present[i]) continue;
      const float dn = side == 0 ? nb[i].m - c.m : c.m - nb[i].m, wn = nb[i].w;
      if (wn == 0.f) {  // point mass: survival 1 below it, and it caps R
        R = fminf(R, dn);
      } else {
        al[i] = dn - wn; d[i] = dn; iw[i] = frcp(wn);
        R = fminf(R, dn + wn);
      }
    }
    const float p = epan_side_k<K>(w1, -w1, R, al, d, iw);
    if (side == 0) pmin = p; else pmax = p;
  }
}

// ---------------------------------------------------------------------------
// histogram of many bins (see stencil_hist_tiles): tail tables in global
// memory, one row of R = B + 4 floats per
// vertex: S_0..S_{B+1} (S_k = T - (m_0 + ... + m_{k-1}), S_B = S_{B+1} = 0,
// all 0 for a point mass), the total mass T, the status bits

__host__ __device__ constexpr int hist_table_row(int B) { return B + 4; }

// HistSeg over a global tail-table row (see HistSeg in device.cuh): the
// read at the next crossing is at tab[addr]; a walker crosses at most B + 1
// edges, so addr stays within its row
struct HistSegG {
  long long addr;
  float kf, lam, h, invh;
  float el, nx, s, sn, sl;
  __device__ __forceinline__ void init_absent(long long a, float Bf) {
    addr = a; kf = Bf + 1.f; lam = h = invh = 0.f;
    el = -kFar; nx = kFar; s = sn = 1.f; sl = 0.f;
  }
  __device__ __forceinline__ void init(const float *tab, long long row, float lam_, float h_,
                                       float T) {
    addr = row + 1; kf = 0.f;
    lam = lam_; h = h_; invh = h_ > 0.f ? frcp(h_) : 0.f;
    el = -kFar; nx = lam_; s = T; sn = __ldg(tab + row); sl = 0.f;
  }
  __device__ __forceinline__ bool step(const float *tab, float x1, float Bf) {
    const bool c = nx <= x1;
    const float t = __ldg(tab + addr);
    s = c ? sn : s;
    sn = c ? t : sn;
    addr += c ? 1 : 0;
    sl = (s - sn) * invh;
    el = c ? x1 : el;
    kf = c ? kf + 1.f : kf;
    nx = c ? (kf <= Bf ? fmaf(kf, h, lam) : kFar) : nx;
    return c;
  }
  __device__ __forceinline__ float G(float x) const { return fmaf(-sl, x - el, s); }
};

// hist_walk with K neighbours (centre row crow of the tail table)
template <int K>
__device__ __forceinline__ void hist_walk_k(const float *tab, long long crow, int B, float W1,
                                            HistSegG *nw, const float *T, unsigned want,
                                            float &pmin, float &pmax) {
  if (!(W1 <= 1e38f)) {
    pmin = pmax = __int_as_float(0x7fc00000);
    return;
  }
  const float Bf = (float)B;
  const float h1 = W1 / Bf, ih1 = frcp(h1);
  long long addr_c = crow + 2;
  float kcf = 1.f;
  float sc = __ldg(tab + crow), scn = __ldg(tab + crow + 1);
  float dens = (sc - scn) * ih1;
  float nxc = B > 1 ? h1 : W1;
  // (G, F) of each factor at the piece's left and right ends
  float2 Pl[K];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const float g = nw[i].G(0.f);
    Pl[i] = make_float2(g, T[i] - g);
  }
  float2 acc = make_float2(0.f, 0.f);
  (void)want;
  float x0 = 0.f;
  const int max_steps = (K + 1) * (B + 2) + 4;
  for (int step = 0; step < max_steps && x0 < W1; ++step) {
    float x1 = nxc;
#pragma unroll
    for (int i = 0; i < K; ++i) x1 = fminf(x1, nw[i].nx);
    x1 = fmaxf(x1, x0);
    float2 Pr[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const float g = nw[i].G(x1);
      Pr[i] = make_float2(g, T[i] - g);
    }
    const float wgt = (x1 - x0) * dens;
    acc = __ffma2_rn(make_float2(wgt, wgt), bern_mean_k_x2<K>(Pl, Pr), acc);
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const bool c = nw[i].step(tab, x1, Bf);
      const float g = c ? nw[i].s : Pr[i].x;
      Pl[i] = make_float2(g, T[i] - g);
    }
    {
      const bool c = nxc <= x1;
      const float t = __ldg(tab + addr_c);
      sc = c ? scn : sc;
      scn = c ? t : scn;
      addr_c += c ? 1 : 0;
      kcf = c ? kcf + 1.f : kcf;
      nxc = c ? (kcf < Bf ? kcf * h1 : (kcf == Bf ? W1 : kFar)) : nxc;
      dens = (sc - scn) * ih1;
    }
    x0 = x1;
  }
  pmin = fmaxf(acc.x, 0.f);
  pmax = fmaxf(acc.y, 0.f);
}

// Mean over [-1, 1] of the product of K = 6 or 8 linear factors m_i - D_i t,
// from their middle values and half falls: pairs of factors are quadratics p -
// b t + e t^2, two pairs a quartic, and the mean of a product of polynomials
// is the sum of its even coefficients over 1, 3, 5, ... .  Every term is a
// product of non-negative numbers.  O: the arithmetic of one or both types
// (HistWalkOps); with both, the odd coefficients of F carry the opposite
// sign, which drops out (they meet in pairs).
template <int K, typename O, typename V>
__device__ __forceinline__ V linear_mean_k(const V *m, const V *D) {
  static_assert(K == 6 || K == 8, "three or four pairs");
  constexpr int P = K / 2;
  V p[P], b[P], e[P];
#pragma unroll
  for (int j = 0; j < P; ++j) {
    p[j] = O::mul(m[2 * j], m[2 * j + 1]);
    e[j] = O::mul(D[2 * j], D[2 * j + 1]);
    b[j] = O::fma(m[2 * j], D[2 * j + 1], O::mul(m[2 * j + 1], D[2 * j]));
  }
  const V c3 = O::all(1.f / 3.f), c5 = O::all(0.2f), c7 = O::all(1.f / 7.f);
  // the quartic of two pairs: coefficients of 1, -t, t^2, -t^3, t^4
  auto quartic = [&](int i, int j, V *q) {
    q[0] = O::mul(p[i], p[j]);
    q[1] = O::fma(p[i], b[j], O::mul(b[i], p[j]));
    q[2] = O::fma(p[i], e[j], O::fma(b[i], b[j], O::mul(e[i], p[j])));
    q[3] = O::fma(b[i], e[j], O::mul(e[i], b[j]));
    q[4] = O::mul(e[i], e[j]);
  };
  V q[5];
  quartic(0, 1, q);
  if constexpr (K == 6) {
    const V u0 = O::fma(e[2], c3, p[2]);
    const V u2 = O::fma(p[2], c3, O::mul(e[2], c5));
    const V u4 = O::fma(p[2], c5, O::mul(e[2], c7));
    const V v = O::fma(q[3], c5, O::mul(q[1], c3));
    return O::fma(q[0], u0, O::fma(q[2], u2, O::fma(q[4], u4, O::mul(v, b[2]))));
  } else {
    V r[5];
    quartic(2, 3, r);
    const V c9 = O::all(1.f / 9.f);
    const V u0 = O::fma(r[2], c3, O::fma(r[4], c5, r[0]));
    const V u2 = O::fma(r[0], c3, O::fma(r[2], c5, O::mul(r[4], c7)));
    const V u4 = O::fma(r[0], c5, O::fma(r[2], c7, O::mul(r[4], c9)));
    const V v1 = O::fma(r[1], c3, O::mul(r[3], c5));
    const V v3 = O::fma(r[1], c5, O::mul(r[3], c7));
    return O::fma(q[0], u0,
                  O::fma(q[2], u2, O::fma(q[4], u4, O::fma(q[1], v1, O::mul(q[3], v3)))));
  }
}

// hist_walk_pieces with K neighbours: the same rows, walkers and steps (every
// lane runs the same instructions, the crossings predicated); MODE kWalkBoth,
// kWalkMin or kWalkMax.
template <int K, int RS, int MODE>
__device__ __forceinline__ void hist_walk_rows_k(const float4 *crow, int B, float W1,
                                                 HistRowWalker *nw, float &pmin, float &pmax) {
  using O = HistWalkOps<MODE>;
  using V = typename O::V;
  if (!(W1 <= 1e38f)) {
    pmin = pmax = __int_as_float(0x7fc00000);
    return;
  }
  uint32_t addr_c = static_cast<uint32_t>(__cvta_generic_to_shared(crow + RS)) + 8u;
  float2 dc;  // (density, next edge) of the centre's current bin
  {
    const float4 t = crow[0];
    dc = make_float2(t.z, t.w);
  }
  V acc = O::all(0.f);
  float x0 = 0.f;
  const int max_steps = (K + 1) * (B + 1) + 4;
#pragma unroll 1
  for (int step = 0; step < max_steps && x0 < W1; ++step) {
    float e[K];
    float x1 = dc.y;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      e[i] = nw[i].nx();
      x1 = fminf(x1, e[i]);
    }
    const float d = x1 - x0, hd = 0.5f * d;
    V m[K], D[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      float4 &r = nw[i].r;
      if constexpr (O::two) {
        const float2 zz = make_float2(r.z, r.z), l = make_float2(r.x, r.y);
        D[i] = __fmul2_rn(zz, make_float2(hd, hd));
        m[i] = __ffma2_rn(zz, make_float2(-hd, hd), l);
        const float2 v = __ffma2_rn(zz, make_float2(-d, d), l);
        r.x = v.x;
        r.y = v.y;
      } else {
        float &l = MODE == kWalkMin ? r.x : r.y;
        D[i] = __fmul_rn(r.z, hd);
        m[i] = __fmaf_rn(r.z, MODE == kWalkMin ? -hd : hd, l);
        l = __fmaf_rn(r.z, MODE == kWalkMin ? -d : d, l);
      }
    }
    acc = O::fma(O::all(__fmul_rn(d, dc.x)), linear_mean_k<K, O>(m, D), acc);
#pragma unroll
    for (int i = 0; i < K; ++i) walker_cross<RS, MODE, true>(e[i], x1, nw[i]);
    lds64_cross<(unsigned)(RS * 16)>(dc.y, x1, addr_c, dc);
    x0 = x1;
  }
  if constexpr (O::two) {
    pmin = fmaxf(acc.x, 0.f);
    pmax = fmaxf(acc.y, 0.f);
  } else {
    (MODE == kWalkMin ? pmin : pmax) = fmaxf(acc, 0.f);
  }
}

// survival and CDF of a histogram neighbour (tail-table row) at a point v
__device__ __forceinline__ void hist_tails_row(const float *tab, long long row, int B, float lo,
                                               float hi, float T, float v, float &gt,
                                               float &lt) {
  if (lo == hi) {
    gt = lo > v ? T : 0.f;
    lt = lo < v ? T : 0.f;
    return;
  }
  if (v <= lo) {
    gt = T; lt = 0.f;
    return;
  }
  if (v >= hi) {
    gt = 0.f; lt = T;
    return;
  }
  const float h = (hi - lo) / (float)B;
  const int j = min(max((int)floorf((v - lo) / h), 0), B - 1);
  const float fr = fminf(fmaxf((v - lo - (float)j * h) / h, 0.f), 1.f);
  const float sj = __ldg(tab + row + j), sj1 = __ldg(tab + row + j + 1);
  gt = fmaxf(fmaf(-fr, sj - sj1, sj), 0.f);
  lt = fmaxf(T - gt, 0.f);
}

}  // namespace ucp
