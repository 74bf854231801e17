// Covariance of log-extinctions by sightline double quadrature (Sect. 3).
//
// For stars i, j at distances s_i, s_j in directions u_i, u_j the density
// covariance is integrated along both sightlines:
//   R_ij = (1 / s_i s_j) int_0^{s_i} int_0^{s_j} g(|t u_i - t' u_j|) dt dt',
// g = expm1(sigma2 phi(r / L0)) (lognormal moment match of rho = exp f) or
// sigma2 phi (first-order form), where phi is the correlation of a
// Kolmogorov spectrum truncated at the outer scale L0 (Sect. 1):
//   phi(x) = 2^(2/3) / Gamma(1/3) x^(1/3) K_(1/3)(x).
// Then K_ij = log1p(R_ij) (or R_ij) times the Wendland taper of the 3-D star
// separation, and m_i = ln(rho_bar s_i) - K_ii / 2.
//
// phi is evaluated once per context on the GPU from the integral
// representation K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt (trapezoid
// rule, exponentially convergent), at the nodes of a log-spaced cubic table
// in x^2 = r^2 / L0^2; each build refits the table of g for the current
// sigma2 and the quadrature kernels interpolate it.  The separation is taken
// in the cancellation-free chord form r^2 = (t - t')^2 + t t' |u_i - u_j|^2.
//
// Two node rules: the Q-node Gauss-Legendre rule on each sightline
// (GM_QUAD_GL), and the band rule of gm_band.cuh (GM_QUAD_BAND), composite
// Gauss-Legendre in d = t - t', m = (t + t')/2 graded towards the cusp of g,
// which converges where s >> L0 (the Q-node rule's nodes are s / Q apart).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "gm_band.cuh"
#include "gm_internal.cuh"

namespace gm {

// ------------------------------------------------------------ phi table
__device__ __forceinline__ double seg_lo(const TableGeom g, int k) {
  int oct = k >> g.m, sub = k & ((1 << g.m) - 1);
  return ldexp(1.0 + (double)sub / (double)(1 << g.m), g.emin + oct);
}

// phi(rho) for rho > 0 by the trapezoid rule with step h = 0.1 in t.
__device__ double phi_of_rho(double rho, double cnorm) {
  const double h = 0.1;
  double sum = 0.5 * exp(-rho);  // t = 0 term: exp(-rho) cosh(0)
  for (int k = 1; k < 4000; ++k) {
    double t = k * h;
    double e = exp(t * (1.0 / 3.0));
    double ei = 1.0 / e;
    double ch3 = 0.5 * (e + ei);                 // cosh(t/3)
    double ch = 0.5 * (e * e * e + ei * ei * ei);  // cosh(t)
    double term = exp(-rho * ch) * ch3;
    sum += term;
    // remaining terms are below 1e-20 of the sum once rho (cosh t - 1)
    // exceeds t/3 + 50
    if (rho * (ch - 1.0) > t * (1.0 / 3.0) + 50.0) break;
  }
  return cnorm * cbrt(rho) * (h * sum);
}

__global__ void k_phi_points(TableGeom g, double cnorm, double* __restrict__ out) {
  const int np = g.n_pts();
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
    int k = p / 3, q = p - 3 * k;
    double x;
    if (k >= g.n_real()) {
      x = ldexp(1.0, g.emax);
    } else {
      double lo = seg_lo(g, k);
      double H = ldexp(1.0 / (double)(1 << g.m), g.emin + (k >> g.m));
      x = lo + H * (double)q / 3.0;
    }
    out[p] = phi_of_rho(sqrt(x), cnorm);
  }
}

// Cubic through g at the four equispaced nodes of each segment (Newton
// forward differences).  FP32 tables hold coefficients of the normalised
// offset v = (x - x_lo) / H in [0, 1) (all O(1)); FP64 tables hold
// coefficients of the absolute offset d = x - x_lo (its range covers 1/H^3).
template <typename T4>
__global__ void k_gtab(TableGeom g, const double* __restrict__ phi, double sigma2, int form,
                       int normalised, T4* __restrict__ tab) {
  const int nr = g.n_real();
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= nr; k += gridDim.x * blockDim.x) {
    T4 o;
    if (k == nr) {
      o.x = o.y = o.z = o.w = 0;
    } else {
      double v[4];
      for (int q = 0; q < 4; ++q) {
        double c = sigma2 * phi[3 * k + q];
        v[q] = form == GM_FORM_LOGNORMAL ? expm1(c) : c;
      }
      double d1 = v[1] - v[0], d2 = v[2] - 2 * v[1] + v[0], d3 = v[3] - 3 * v[2] + 3 * v[1] - v[0];
      // p(w) = c0 + c1 w + c2 w^2 + c3 w^3 with w = 3 v
      double c0 = v[0], c1 = d1 - 0.5 * d2 + d3 / 3.0, c2 = 0.5 * d2 - 0.5 * d3, c3 = d3 / 6.0;
      double H = ldexp(1.0 / (double)(1 << g.m), g.emin + (k >> g.m));
      double sc = normalised ? 3.0 : 3.0 / H;
      o.x = c0;
      o.y = c1 * sc;
      o.z = c2 * sc * sc;
      o.w = c3 * sc * sc * sc;
    }
    tab[k] = o;
  }
}

// ------------------------------------------------------------ g lookup
struct TabF32 {
  int base;      // float bits of 2^emin
  int shift;     // 23 - m
  int last;      // index of the zero segment
  float xmin;
};
struct TabF64 {
  int base;      // high word of 2^emin
  int shift;     // 20 - m
  int last;
  double xmin;
};

// v = position of x inside its segment, in [0, 1): the mantissa bits below
// the segment index, placed in the mantissa of a float in [1, 2), minus 1.
__device__ __forceinline__ float g_lookup(const float4* __restrict__ tab, const TabF32& t, float x) {
  x = fmaxf(x, t.xmin);
  int bits = __float_as_int(x);
  int k = min((bits - t.base) >> t.shift, t.last);
  float v = __int_as_float(((bits << (23 - t.shift)) & 0x007fffff) | 0x3f800000) - 1.0f;
  float4 c = tab[k];
  return fmaf(v, fmaf(v, fmaf(v, c.w, c.z), c.y), c.x);
}

// The FP32 pair kernel keeps a window of the table, from the segment of
// 2^kWinEmin up, in shared memory with every segment stored kRep = 8 times in
// a row (one 128-byte bank row per segment); lane l reads copy l % 8.  The 8
// lanes of a quarter-warp, which share one pass of a 16-byte shared load,
// then always fall in 8 distinct bank groups: the lookups of a warp cost
// four passes whatever segments the lanes hit (a single copy averaged 1.9
// passes per quarter-warp on the 20,000-star field's pairs).  Below 2^kWinEmin
// the argument is clamped: g(x) - g(0) scales as x^(1/3), 2.4e-8 of g(0) there.
constexpr int kWinEmin = -76;
constexpr int kRep = 8;
constexpr int kWinK0 = (kWinEmin - kTabF32.emin) << kTabF32.m;  // first segment kept
constexpr int kWinSegs =  // incl. the zero segment
    ((kTabF32.emax - kTabF32.emin) << kTabF32.m) + 1 - kWinK0;

// tab8 points at copy (lane % 8) of window segment 0.  The window's geometry
// is compile-time, so the segment offset folds into the load's address.
// x must be >= 2^kWinEmin (callers add it to the separation).
constexpr int kWinShift = 23 - kTabF32.m;
constexpr int kWinBaseSeg = (127 + kWinEmin) << kTabF32.m;  // (float bits of 2^kWinEmin) >> shift
constexpr int kWinLast = kWinSegs - 1;
__device__ __forceinline__ float g_lookup_rep(const float4* __restrict__ tab8, float x) {
  const int bits = __float_as_int(x);
  const int k = min((bits >> kWinShift) - kWinBaseSeg, kWinLast);
  const float v = __int_as_float(((bits << (23 - kWinShift)) & 0x007fffff) | 0x3f800000) - 1.0f;
  const float4 c = tab8[k * kRep];
  return fmaf(v, fmaf(v, fmaf(v, c.w, c.z), c.y), c.x);
}

__device__ __forceinline__ double g_lookup(const D4* __restrict__ tab, const TabF64& t,
                                           double x) {
  x = fmax(x, t.xmin);
  int hi = __double2hiint(x);
  int k = min((hi - t.base) >> t.shift, t.last);
  double xlo = __hiloint2double(hi & ~((1 << t.shift) - 1), 0);
  double d = x - xlo;
  const double2* p = reinterpret_cast<const double2*>(tab + k);
  double2 a = __ldg(p), b = __ldg(p + 1);
  return fma(d, fma(d, fma(d, b.y, b.x), a.y), a.x);
}

__device__ __forceinline__ double wendland(double h) {
  if (h >= 1.0) return 0.0;
  double u = 1.0 - h, u2 = u * u;
  return u2 * u2 * (4.0 * h + 1.0);
}
__device__ __forceinline__ float wendland_f(float h) {
  if (h >= 1.0f) return 0.0f;
  const float u = 1.0f - h, u2 = u * u;
  return u2 * u2 * fmaf(4.0f, h, 1.0f);
}

struct QuadParams {
  double inv_L0;
  double inv_cut;
  double log_rho_bar;
  double sigma2;
  int Q;
  int form;
  int taper;
  int symmetric;
};

// Lower-triangle entries copy their transpose (rows are sorted).
template <typename T>
__global__ void k_mirror(int64_t n, const int64_t* __restrict__ row_ptr,
                         const int32_t* __restrict__ col, int64_t nnz, T* __restrict__ val) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = n;
    while (hi - lo > 1) {
      int64_t mid = (lo + hi) >> 1;
      if (row_ptr[mid] <= e) lo = mid; else hi = mid;
    }
    const int32_t i = (int32_t)lo, j = col[e];
    if (j >= i) continue;
    int64_t a = row_ptr[j], b = row_ptr[j + 1];  // search i in row j
    while (b - a > 1) {
      int64_t mid = (a + b) >> 1;
      if (col[mid] <= i) a = mid; else b = mid;
    }
    val[e] = val[a];
  }
}

// Self-covariance k_qq of query points (FP32 form, same rule as the diagonal).
template <int KPL>
__global__ void k_self_quad(QuadParams P, int64_t n_rows, const double* __restrict__ rs,
                            const double* __restrict__ gl_zeta, const double* __restrict__ gl_w,
                            const void* __restrict__ gtab, TabF32 tf, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < n_rows; r += nwarps) {
    const float a = (float)(rs[r] * P.inv_L0);
    float tp[KPL], wp[KPL];
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
      int q = lane + 32 * k;
      bool ok = q < P.Q;
      tp[k] = ok ? a * (float)gl_zeta[q] : 0.f;
      wp[k] = ok ? (float)gl_w[q] : 0.f;
    }
    float acc = 0;
    for (int q = 0; q < P.Q; ++q) {
      const float t = a * (float)gl_zeta[q];
      float inner = 0;
#pragma unroll
      for (int k = 0; k < KPL; ++k) {
        const float d = t - tp[k];
        inner += wp[k] * g_lookup(reinterpret_cast<const float4*>(gtab), tf, d * d);
      }
      acc += (float)gl_w[q] * inner;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) {
      double R = (double)acc;
      double K = P.form == GM_FORM_LOGNORMAL ? log1p(R) : R;
      out[r] = (double)(float)K;
    }
  }
}

// ------------------------------------------------------------ band rule
// The band rule of gm_band.cuh with the warp's lanes holding the pair's
// breakpoints.  What bounds it: about 1,200 evaluations of g a pair (38 per
// lane), so everything around them has to be paid once a pair or once 32
// pairs.  GB300 issues an FP64 instruction every 16 clocks per SM, so
//   * the FP64 work of a pair (distances, chord, difference of the distances,
//     log1p, taper) is done for a batch of up to 32 pairs at once, a lane per
//     pair, and the batch's pairs are then integrated one after another by
//     the whole warp (band_batch);
//   * the graded breakpoints come from a 12-entry table (no pow / log), their
//     clipping, merging with the kink and counting from ballots and shuffles;
//   * the FP32 form places nodes and panels in FP32 (the partition it sums
//     over is a partition whatever its rounding), and reads g from the
//     replicated table window of the 64-node kernel.
// 6,000 stars of the 5-degree field (3.0e6 stored entries, FP32): 199 ms with
// every lane finding its panels by FP64 pow / log, 2.2 ms so (6.7e8 unique
// pairs/s); the carried sums cost 0.2 ms of it and lower the entries' error
// against FP64 from 4.8e-8 to 3.3e-8.
constexpr int kBandPts = 12;  // breakpoints h0 (q^j - 1) / (q - 1), j < 12: 0 .. 88.6 >= kK

struct BandTab {
  double pt[kBandPts];
};

// g by table lookup in the arithmetic type of the sums.
template <typename T>
struct GLook;
template <>
struct GLook<float> {
  const float4* tab8;  // replicated window, this lane's copy
  __device__ float operator()(float x) const {
    return g_lookup_rep(tab8, x + __int_as_float((127 + kWinEmin) << 23));
  }
};
template <>
struct GLook<double> {
  const D4* tab;
  TabF64 t;
  __device__ double operator()(double x) const { return g_lookup(tab, t, x); }
};

// Sum of FP32 terms with its rounding carried along (Knuth's TwoSum), so that
// the few large partial sums of a pair do not round to FP32 on the way.
template <typename T>
struct CarrySum {
  T s = 0;
  __device__ __forceinline__ void add(T x) { s += x; }
  __device__ __forceinline__ double warp_total() {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
  }
};
template <>
struct CarrySum<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    c += __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
    s = t;
  }
  __device__ __forceinline__ double warp_total() {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float so = __shfl_xor_sync(0xffffffffu, s, off);
      const float co = __shfl_xor_sync(0xffffffffu, c, off);
      add(so);
      c += co;
    }
    return (double)s + (double)c;
  }
};

// Node i of this lane in round r (d-node lane + 32 r, i = (lane + 2 r) mod 6):
// the three node and weight values a lane meets.
template <typename T>
struct BandLane {
  T z[3], w[3];
  T pt;  // table breakpoint of this lane (beyond the table: infinity)
};

template <typename T>
__device__ __forceinline__ BandLane<T> band_lane(const BandTab& bt, int lane) {
  BandLane<T> L;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int i = (lane + 2 * r) % gmband::kN;
    L.z[r] = (T)gmband::gl_z(i);
    L.w[r] = (T)gmband::gl_w(i);
  }
  L.pt = (T)INFINITY;
#pragma unroll
  for (int j = 0; j < kBandPts; ++j)
    if (lane == j) L.pt = (T)bt.pt[j];
  return L;
}

// I_ij of one pair (A = s_i / L0, B = s_j / L0, c2 = |u_i - u_j|^2, kink =
// A - B); every lane returns the sum.  Al, Bl: what rounding A and B to T left
// out; the upper end of m adds it to the length of its last panel, so that the
// rounding of the two distances does not scale the whole integral.
template <typename T>
__device__ __forceinline__ double band_I_warp(T A, T B, T Al, T Bl, T c2, T kink, const BandLane<T>& L,
                                         const GLook<T>& g, int lane) {
  constexpr unsigned full = 0xffffffffu;
  const T K = (T)gmband::kK;
  const T Dp = A < K ? A : K, Dn = B < K ? B : K;
  // panels of each side: breakpoints below its extent (0 is one of them)
  const int np = __popc(__ballot_sync(full, L.pt < Dp));
  const int nn = __popc(__ballot_sync(full, L.pt < Dn));
  // base breakpoint of this lane: -side(nn - lane) .. 0 .. side(lane - nn)
  const int t = lane - nn;
  T v = __shfl_sync(full, L.pt, t < 0 ? -t : t);
  const T ext = t < 0 ? Dn : Dp;
  v = v < ext ? v : ext;
  const T base = t < 0 ? -v : v;
  const int nb = nn + np;  // last base index
  const int below = __popc(__ballot_sync(full, lane <= nb && base < kink));
  const T at = __shfl_sync(full, base, below);
  const bool ins = kink > -Dn && kink < Dp && at != kink;
  const T prev = __shfl_up_sync(full, base, 1);
  const T pt = !ins || lane < below ? base : (lane == below ? kink : prev);
  const int npan = nb + (ins ? 1 : 0);
  const T c = sqrt(c2);
  const T sc = c2 > (T)0 ? (T)1 / c : (T)0;
  const T h0 = (T)gmband::kM0 * sc, lim = K * sc;
  const T dsc = (T)1 - (T)0.25 * c2;
  CarrySum<T> acc;
#pragma unroll 1
  for (int r0 = 0; 32 * r0 < npan * gmband::kN; r0 += 3) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int k = lane + 32 * (r0 + r);
      const int pnl = min(k / gmband::kN, 30);
      const T a = __shfl_sync(full, pt, pnl), b = __shfl_sync(full, pt, pnl + 1);
      const T d = a + (b - a) * L.z[r];
      const T wd = (b - a) * L.w[r];
      const T lo = (d < (T)0 ? -d : d) * (T)0.5;
      const T u1 = A - d * (T)0.5, u2 = B + d * (T)0.5;
      const T hi = u1 < u2 ? u1 : u2;
      const T hl = u1 < u2 ? Al : Bl;
      if (k >= npan * gmband::kN || !(hi > lo) || wd == (T)0) continue;
      if (c2 == (T)0) {
        const T gv = g(d * d);
        acc.add(wd * ((hi - lo) * gv + hl * gv));
        continue;
      }
      const T dd = d * d * dsc;
      const T end = hi < lo + lim ? hi : lo + lim;
      T sum = 0, ma = lo, h = h0;
      while (ma < end) {
        const T mb = ma + h < end ? ma + h : end;
        const T len = mb - ma;
        T s6 = 0;
#pragma unroll
        for (int j = 0; j < gmband::kN; ++j) {
          const T m = ma + len * (T)gmband::gl_z(j);
          s6 += (T)gmband::gl_w(j) * g(dd + m * m * c2);
        }
        sum += len * s6;
        if (mb == hi) sum += hl * s6;
        ma = mb;
        h *= (T)gmband::kQ;
      }
      acc.add(wd * sum);
    }
  }
  return acc.warp_total();
}

// Node rules.  A rule integrates up to 32 pairs of a warp, one per active lane
// (A = s_i / L0, B = s_j / L0 and c2 in FP64): the warp takes the active lanes'
// pairs one after another.  Val is the type of the stored entries.
template <typename T>
struct BandRule {
  typedef T Val;
  static constexpr bool kFloatEntry = false;  // log1p and the taper in FP64
  struct Par {
    BandTab bt;
    const void* gtab;
    TabF64 td;
  };
  // FP32: one block of 32 warps per SM around the replicated table window
  static constexpr int kThreads = sizeof(T) == 4 ? 1024 : 256, kBound = kThreads;
  GLook<T> g;
  BandLane<T> L;
  int lane;

  static size_t smem() { return sizeof(T) == 4 ? (size_t)kWinSegs * kRep * sizeof(float4) : 0; }
  __device__ __forceinline__ BandRule(const Par& P, unsigned char* sm) {
    lane = threadIdx.x & 31;
    if constexpr (sizeof(T) == 4) {
      float4* st = reinterpret_cast<float4*>(sm);
      const float4* gt = reinterpret_cast<const float4*>(P.gtab) + kWinK0;
      for (int k = threadIdx.x; k < kWinSegs * kRep; k += blockDim.x) st[k] = gt[k / kRep];
      g.tab8 = st + (threadIdx.x & (kRep - 1));
    } else {
      g.tab = reinterpret_cast<const D4*>(P.gtab);
      g.t = P.td;
    }
    L = band_lane<T>(P.bt, lane);
    __syncthreads();
  }
  __device__ __forceinline__ double R(bool active, double A, double B, double c2) const {
    constexpr unsigned full = 0xffffffffu;
    const T At = (T)A, Bt = (T)B, ct = (T)c2, kt = (T)(A - B);
    const T Al = (T)(A - (double)At), Bl = (T)(B - (double)Bt);
    double mine = 0;
    for (unsigned m = __ballot_sync(full, active); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const double v = band_I_warp<T>(__shfl_sync(full, At, l), __shfl_sync(full, Bt, l),
                                      __shfl_sync(full, Al, l), __shfl_sync(full, Bl, l),
                                      __shfl_sync(full, ct, l), __shfl_sync(full, kt, l), L, g, lane);
      if (lane == l) mine = v;
    }
    return mine / (A * B);
  }
};

// ------------------------------------------------------------ FP64 node sums
// The Q-node rule of FP64 contexts on the FP32 units.  GB300 runs 64 FP32
// instructions in the time of one FP64 instruction, and a node pair takes ten
// of the latter; so the separation, the table cubic and the node sums are
// carried as unevaluated sums of two floats (Dekker 1971, Knuth's TwoSum; 48
// bits), about 70 FP32 instructions.  The table is the cubic of the FP64 table
// re-expanded about the middle of each segment, leading coefficients in two
// floats; its error (2e-12 of g(0)) stays the rule's largest.  It covers
// 2^kDfEmin <= x < 2^11 in shared memory; smaller separations (nodes that
// coincide: the diagonal) use the FP64 table.  Nodes of the same index are s_i - s_j
// times the node apart, taken from the FP64 difference: from the two products, of
// which 48 bits are kept, stars at nearly equal distances lost the separation.
// 2,001 stars, 64 nodes (161,494 unique pairs): 14.2 ms with FP64 instructions
// (Gl64Rule), 2.3 ms so; 4.1 and 0.65 ms at 32 nodes.  Against FP64 Bessel functions
// entries between different stars are 1.0e-12 off (largest 3.6e-12) in both forms, the
// diagonal 1.4e-10 (the table ends at x = 2^-100).
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 f2_of(double x) {
  F2 r;
  r.h = (float)x;
  r.l = (float)(x - (double)r.h);
  return r;
}
__device__ __forceinline__ F2 f2_fast(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ F2 f2_sum(float a, float b) {
  const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z))};
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)));
  return f2_fast(p, e);
}
// acc += a b (both low parts kept, not renormalised)
__device__ __forceinline__ void f2_fma(F2& acc, F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)));
  const F2 s = f2_sum(acc.h, p);
  acc.h = s.h;
  acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, e));
}

constexpr int kDfEmin = -20;
constexpr int kDfSegs = (kTabF64.emax - kDfEmin) << kTabF64.m;  // 3,968: 93 KB
constexpr int kDfShift = 23 - kTabF64.m;
constexpr int kDfBase = (127 + kDfEmin) << kTabF64.m;

// coefficients of v = (x - x_mid) / H in [-1/2, 1/2): c0 and c1 as two floats
// (tab4), c2 and c3 as one (tab2)
__global__ void k_gtab_df(const D4* __restrict__ tab, float4* __restrict__ tab4,
                          float2* __restrict__ tab2) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < kDfSegs; k += gridDim.x * blockDim.x) {
    const D4 d = tab[k + ((kDfEmin - kTabF64.emin) << kTabF64.m)];
    const double H = ldexp(1.0 / (double)(1 << kTabF64.m), kDfEmin + (k >> kTabF64.m));
    const double c1 = d.y * H, c2 = d.z * H * H, c3 = d.w * H * H * H;  // of (x - x_lo) / H
    const F2 a0 = f2_of(d.x + 0.5 * (c1 + 0.5 * (c2 + 0.5 * c3)));
    const F2 a1 = f2_of(c1 + c2 + 0.75 * c3);
    tab4[k] = make_float4(a0.h, a0.l, a1.h, a1.l);
    tab2[k] = make_float2((float)(c2 + 1.5 * c3), (float)c3);
  }
}

template <int KPL>
struct DfRule {
  typedef double Val;
  static constexpr bool kFloatEntry = false;
  struct Par {
    const double* gl_zeta;
    const double* gl_w;
    const D4* gtab;
    TabF64 td;
    const float4* tab4;
    const float2* tab2;
    int Q;
  };
  // launched with 512; up to 64 nodes within the registers of 1,024 (64 a thread), so
  // that two blocks share an SM
  static constexpr int kThreads = 512, kBound = KPL <= 2 ? 1024 : 512;
  static constexpr int kWarps = kThreads / 32;
  const float4* t4;
  const float2* t2;
  const float4* zw;   // nodes and weights (zh, zl, wh, wl), shared memory
  float2* tq;         // this warp's nodes on sightline i
  const D4* gtab;
  TabF64 td;
  int lane, Q;

  static size_t smem() {
    return kDfSegs * (sizeof(float4) + sizeof(float2)) + kMaxNodes * sizeof(float4) +
           kWarps * 32 * KPL * sizeof(float2);
  }
  __device__ __forceinline__ DfRule(const Par& P, unsigned char* sm)
      : gtab(P.gtab), td(P.td), Q(P.Q) {
    lane = threadIdx.x & 31;
    float4* a = reinterpret_cast<float4*>(sm);
    float4* z = a + kDfSegs;
    float2* b = reinterpret_cast<float2*>(z + kMaxNodes);
    tq = b + kDfSegs + (threadIdx.x >> 5) * 32 * KPL;
    for (int k = threadIdx.x; k < kDfSegs; k += blockDim.x) {
      a[k] = P.tab4[k];
      b[k] = P.tab2[k];
    }
    for (int q = threadIdx.x; q < Q; q += blockDim.x) {
      const F2 x = f2_of(P.gl_zeta[q]), w = f2_of(P.gl_w[q]);
      z[q] = make_float4(x.h, x.l, w.h, w.l);
    }
    t4 = a;
    t2 = b;
    zw = z;
    __syncthreads();
  }

  // g at x = xh + xl
  __device__ __forceinline__ F2 g(float xh, float xl) const {
    const int bits = __float_as_int(xh);
    const int k = (bits >> kDfShift) - kDfBase;
    if ((unsigned)k >= (unsigned)kDfSegs) {
      // below the window (coinciding nodes) or beyond the table (zero)
      if (k >= 0) return {0.f, 0.f};
      return f2_of(g_lookup(gtab, td, (double)xh + (double)xl));
    }
    const float4 c = t4[k];
    const float2 d = t2[k];
    // v: the mantissa bits below the segment index, and xl in segment widths
    const float vh = __int_as_float(((bits << kTabF64.m) & 0x007fffff) | 0x3f800000) - 1.5f;
    const float vl =
        xl * __int_as_float(((254 + kTabF64.m) << 23) - (bits & 0x7f800000));
    const float s = __fmaf_rn(vh, d.y, d.x);
    const F2 t = f2_fast(c.z, __fmul_rn(vh, s));
    const float tl = __fmaf_rn(vl, s, __fadd_rn(t.l, c.w));
    const float p = __fmul_rn(vh, t.h);
    const float e = __fmaf_rn(vl, t.h, __fmaf_rn(vh, tl, __fmaf_rn(vh, t.h, -p)));
    const F2 r = f2_fast(c.x, p);
    return {r.h, __fadd_rn(r.l, __fadd_rn(e, c.y))};
  }

  // sum over the nodes of both sightlines; D = A - B
  __device__ __forceinline__ double pair(F2 A, F2 B, F2 D, F2 c2) const {
    F2 tp[KPL], ct[KPL], acc[KPL], dq[KPL];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
      const int q = lane + 32 * k;
      const float4 z = q < Q ? zw[q] : make_float4(0.f, 0.f, 0.f, 0.f);
      const F2 zn = {z.x, z.y};
      tp[k] = f2_mul(B, zn);
      dq[k] = f2_mul(D, zn);
      ct[k] = f2_mul(c2, tp[k]);
      acc[k] = {0.f, 0.f};
      const F2 t = f2_mul(A, zn);
      tq[q] = make_float2(t.h, t.l);
    }
    __syncwarp();
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
      const float2 t = tq[q];
      const float4 z = zw[q];
      const F2 w = {z.z, z.w};
#pragma unroll
      for (int k = 0; k < KPL; ++k) {
        F2 d = f2_sum(t.x, -tp[k].h);
        // where the high parts (nearly) cancel the low ones are all that is left
        d = f2_fast(d.h, __fadd_rn(d.l, __fsub_rn(t.y, tp[k].l)));
        if (q == lane + 32 * k) d = dq[k];
        const float p = __fmul_rn(d.h, d.h);
        const float pe = __fmaf_rn(2.f * d.h, d.l, __fmaf_rn(d.h, d.h, -p));
        const float c = __fmul_rn(t.x, ct[k].h);
        const float ce = __fmaf_rn(t.y, ct[k].h,
                                   __fmaf_rn(t.x, ct[k].l, __fmaf_rn(t.x, ct[k].h, -c)));
        const F2 x = f2_sum(p, c);
        f2_fma(acc[k], w, g(x.h, __fadd_rn(x.l, __fadd_rn(pe, ce))));
      }
    }
    F2 tot = {0.f, 0.f};
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
      const int q = lane + 32 * k;
      const float4 z = q < Q ? zw[q] : make_float4(0.f, 0.f, 0.f, 0.f);
      f2_fma(tot, acc[k], F2{z.z, z.w});
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, tot.h, off);
      const float ol = __shfl_xor_sync(0xffffffffu, tot.l, off);
      const F2 r = f2_sum(tot.h, oh);
      tot.h = r.h;
      tot.l = __fadd_rn(__fadd_rn(tot.l, ol), r.l);
    }
    return (double)tot.h + (double)tot.l;
  }

  __device__ __forceinline__ double R(bool active, double A, double B, double c2) const {
    constexpr unsigned full = 0xffffffffu;
    const F2 a = f2_of(A), b = f2_of(B), e = f2_of(A - B), c = f2_of(c2);
    double mine = 0;
    for (unsigned m = __ballot_sync(full, active); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const F2 al = {__shfl_sync(full, a.h, l), __shfl_sync(full, a.l, l)};
      const F2 bl = {__shfl_sync(full, b.h, l), __shfl_sync(full, b.l, l)};
      const F2 el = {__shfl_sync(full, e.h, l), __shfl_sync(full, e.l, l)};
      const F2 cl = {__shfl_sync(full, c.h, l), __shfl_sync(full, c.l, l)};
      const double v = pair(al, bl, el, cl);
      if (lane == l) mine = v;
    }
    return mine;
  }
};

// The same rule with FP64 instructions: contexts whose g leaves the range in which
// two floats carry its 48 bits (df_fits), and GM_QUAD=fp64.
template <int KPL>
struct Gl64Rule {
  typedef double Val;
  static constexpr bool kFloatEntry = false;
  struct Par {
    const double* gl_zeta;
    const double* gl_w;
    const D4* gtab;
    TabF64 td;
    int Q;
  };
  static constexpr int kThreads = 256, kBound = kThreads;
  const double *z, *w;  // shared memory, padded with zeros
  const D4* gtab;
  TabF64 td;
  int lane, Q;

  static size_t smem() { return 2 * kMaxNodes * sizeof(double); }
  __device__ __forceinline__ Gl64Rule(const Par& P, unsigned char* sm)
      : gtab(P.gtab), td(P.td), Q(P.Q) {
    lane = threadIdx.x & 31;
    double* zs = reinterpret_cast<double*>(sm);
    double* ws = zs + kMaxNodes;
    for (int q = threadIdx.x; q < kMaxNodes; q += blockDim.x) {
      zs[q] = q < Q ? P.gl_zeta[q] : 0.0;
      ws[q] = q < Q ? P.gl_w[q] : 0.0;
    }
    z = zs;
    w = ws;
    __syncthreads();
  }

  __device__ __forceinline__ double pair(double A, double B, double c2) const {
    double acc = 0;
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
      const double t = A * z[q];
      double inner = 0;
#pragma unroll
      for (int k = 0; k < KPL; ++k) {
        const int p = lane + 32 * k;
        const double tp = B * z[p];
        const double d = p == q ? (A - B) * z[q] : t - tp;
        inner += w[p] * g_lookup(gtab, td, d * d + t * (c2 * tp));
      }
      acc += w[q] * inner;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
  }

  __device__ __forceinline__ double R(bool active, double A, double B, double c2) const {
    constexpr unsigned full = 0xffffffffu;
    double mine = 0;
    for (unsigned m = __ballot_sync(full, active); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const double v = pair(__shfl_sync(full, A, l), __shfl_sync(full, B, l),
                            __shfl_sync(full, c2, l));
      if (lane == l) mine = v;
    }
    return mine;
  }
};

// ------------------------------------------------------------ FP32 node sums
// The Q-node rule of FP32 contexts: lanes own the nodes q' of sightline j, loop
// over the nodes q of sightline i, and the warp sums the products.  One 16-byte
// lookup per node pair bounds it (four shared-memory passes a warp: 8 node pairs
// a clock and SM) once the instructions around it are few: the segment's byte
// address is one shift and one mask of x's bits (segments are 128 bytes, the
// lane's copy in the low bits), the in-segment position one mask and one
// subtraction (v / 2^m; the coefficients are scaled by powers of 2^m instead,
// which changes no bit of the cubic), and the clamp to the table's end is left
// out for pairs that cannot reach it.  The FP64 part of 32 pairs runs at once
// (k_pair_entries); a pair's own arithmetic, log1p and the taper included, is
// FP32 as before.
// 20,000 stars (1.58e7 unique pairs x 64 x 64 nodes): 46.7 ms with one pair a warp
// and 22 instructions a node pair, 32.9 ms so (14 instructions; shared memory 88 %
// busy over all SMs, the issue slots 75 %), every entry the same bit for bit.
template <int KPL>
struct Gl32Rule {
  typedef float Val;
  static constexpr bool kFloatEntry = true;
  struct Par {
    const double* gl_zeta;
    const double* gl_w;
    const float4* gtab;
    int Q;
  };
  static constexpr int kThreads = KPL <= 2 ? 1024 : 512, kBound = kThreads;
  const unsigned char* tab;  // segment 0 of the window less the window's first index
  const float4* zw;          // nodes and weights (z, w) of two nodes, padded with w = 0
  int lane, Q;
  unsigned copy;             // byte offset of this lane's copy of a segment

  static size_t smem() {
    return (size_t)kWinSegs * kRep * sizeof(float4) + 2 * kMaxNodes * sizeof(float);
  }
  __device__ __forceinline__ Gl32Rule(const Par& P, unsigned char* sm) : Q(P.Q) {
    lane = threadIdx.x & 31;
    copy = (unsigned)(lane & (kRep - 1)) * sizeof(float4);
    float4* st = reinterpret_cast<float4*>(sm);
    constexpr float s1 = 1 << kTabF32.m, s2 = s1 * s1, s3 = s2 * s1;
    for (int k = threadIdx.x; k < kWinSegs * kRep; k += blockDim.x) {
      float4 c = P.gtab[kWinK0 + k / kRep];
      c.y *= s1;
      c.z *= s2;
      c.w *= s3;
      st[k] = c;
    }
    float2* z = reinterpret_cast<float2*>(st + kWinSegs * kRep);
    for (int q = threadIdx.x; q < kMaxNodes; q += blockDim.x)
      z[q] = q < Q ? make_float2((float)P.gl_zeta[q], (float)P.gl_w[q]) : make_float2(0.f, 0.f);
    zw = reinterpret_cast<const float4*>(z);
    tab = sm;
    __syncthreads();
  }

  // kRep * sizeof(float4) = 128 bytes per segment
  template <bool CLAMP>
  __device__ __forceinline__ float g(float x) const {
    static_assert(kRep * sizeof(float4) == 128 && kWinShift >= 7, "segment address");
    const unsigned bits = (unsigned)__float_as_int(x);
    unsigned off = ((bits >> (kWinShift - 7)) & ~127u) | copy;
    if (CLAMP) off = min(off, (unsigned)(kWinBaseSeg + kWinLast) * 128u + copy);
    const float4 c = *reinterpret_cast<const float4*>(tab + (int)(off - kWinBaseSeg * 128u));
    const float v = __int_as_float((bits & ((1u << kWinShift) - 1u)) | 0x3f800000u) - 1.0f;
    return fmaf(v, fmaf(v, fmaf(v, c.w, c.z), c.y), c.x);
  }

  template <bool CLAMP>
  __device__ __forceinline__ float pair(float a, float b, float c2) const {
    float tp[KPL], ctp[KPL], wp[KPL];
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
      const float2 z = reinterpret_cast<const float2*>(zw)[lane + 32 * k];
      tp[k] = b * z.x;
      ctp[k] = c2 * tp[k];
      wp[k] = z.y;
    }
    float acc = 0;
    auto node = [&](float z, float w) {
      const float t = a * z;
      float inner = 0;
#pragma unroll
      for (int k = 0; k < KPL; ++k) {
        const float d = t - tp[k];
        // x >= 2^kWinEmin by construction: the window's floor is added
        const float x = fmaf(d, d, fmaf(t, ctp[k], __int_as_float((127 + kWinEmin) << 23)));
        inner += wp[k] * g<CLAMP>(x);
      }
      acc += w * inner;
    };
#pragma unroll 1
    for (int q = 0; 2 * q < Q; ++q) {
      // one broadcast load for two nodes; a padding node adds nothing
      const float4 n = zw[q];
      node(n.x, n.y);
      node(n.z, n.w);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
  }

  __device__ __forceinline__ double R(bool active, double A, double B, double c2) const {
    constexpr unsigned full = 0xffffffffu;
    const float a = (float)A, b = (float)B, c = (float)c2;
    // no node pair of this pair reaches the end of the table (2^emax)
    const float top = fmaxf(a, b);
    const bool inside = fmaf(a * b, c, top * top) < 0.99f * (float)(1 << kTabF32.emax);
    const unsigned in = __ballot_sync(full, inside);
    float mine = 0;
    for (unsigned m = __ballot_sync(full, active); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const float al = __shfl_sync(full, a, l), bl = __shfl_sync(full, b, l),
                  cl = __shfl_sync(full, c, l);
      const float v = (in >> l) & 1u ? pair<false>(al, bl, cl) : pair<true>(al, bl, cl);
      if (lane == l) mine = v;
    }
    return (double)mine;
  }
};

// ------------------------------------------------------------ entries
// Entries (i, j) of a CSR by a node rule, with the taper; in symmetric mode
// entries with j < i are left for k_mirror, and the diagonal gives K_ii and
// the prior mean.  A warp takes `batch` entries (a power of two up to 32): the
// FP64 part of a pair (distances, chord, log1p, taper) runs a lane per pair, the
// node sums a warp per pair.  In symmetric mode they lie a batch's share of the list
// apart: consecutive ones are mostly all above or all below the diagonal, and warps
// with several full batches were what a launch waited for (2,441 stars, 64 nodes,
// FP32: 946 us, 695 so; 14,000 stars 16.7 and 14.7 ms; FP64 at 2,441 4.23 and 3.19;
// the band rule 634 and 449 us).
template <typename Rule>
__global__ void __launch_bounds__(Rule::kBound) k_pair_entries(
    QuadParams P, typename Rule::Par rp, int batch, int64_t n_rows, const double* __restrict__ rs,
    const double* __restrict__ rux, const double* __restrict__ ruy, const double* __restrict__ ruz,
    const double* __restrict__ s, const double* __restrict__ ux, const double* __restrict__ uy,
    const double* __restrict__ uz, const int64_t* __restrict__ row_ptr,
    const int32_t* __restrict__ col, int64_t nnz, typename Rule::Val* __restrict__ val,
    double* __restrict__ kdiag, double* __restrict__ prior_m, unsigned* __restrict__ flags,
    const FieldGrid* __restrict__ fg, const int32_t* __restrict__ row_field) {
  typedef typename Rule::Val T;
  extern __shared__ __align__(16) unsigned char smem[];
  const Rule rule(rp, smem);
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t nb = (nnz + batch - 1) / batch;
  for (int64_t b = warp; b < nb; b += nwarps) {
    const int64_t e = P.symmetric ? b + lane * nb : b * batch + lane;
    bool active = lane < batch && e < nnz;
    int64_t i = 0;
    int32_t j = 0;
    if (active) {
      int64_t lo = 0, hi = n_rows;
      while (hi - lo > 1) {
        int64_t mid = (lo + hi) >> 1;
        if (row_ptr[mid] <= e) lo = mid; else hi = mid;
      }
      i = lo;
      j = col[e];
      if (P.symmetric && j < i) active = false;
    }
    double A = 1, B = 1, chord2 = 0, si = 0, sj = 0, inv_cut = 0;
    if (active) {
      const FieldGrid& fgi = fg[row_field ? row_field[i] : 0];
      inv_cut = fgi.inv_cut;
      si = rs[i];
      sj = s[j];
      const double dx = rux[i] - ux[j], dy = ruy[i] - uy[j], dz = ruz[i] - uz[j];
      chord2 = fma(dx, dx, fma(dy, dy, dz * dz));
      A = si * fgi.inv_L0;
      B = sj * fgi.inv_L0;
    }
    const double R = rule.R(active, A, B, chord2);
    if (active) {
      double K;
      if constexpr (Rule::kFloatEntry) {
        // log1p and the taper to ~1e-7 relative; the difference of the distances
        // in FP64: it cancels, and the taper near the cutoff amplifies its error
        const float Rf = (float)R;
        float Kf = P.form == GM_FORM_LOGNORMAL ? log1pf(Rf) : Rf;
        if (P.taper == GM_TAPER_WENDLAND) {
          const float ds = (float)(si - sj);
          const float d = sqrtf(fmaf(ds, ds, (float)si * (float)sj * (float)chord2));
          Kf *= wendland_f(d * (float)inv_cut);
        }
        K = (double)Kf;
      } else {
        K = P.form == GM_FORM_LOGNORMAL ? log1p(R) : R;
        if (P.taper == GM_TAPER_WENDLAND) {
          const double ds = si - sj;
          const double d = sqrt(fma(ds, ds, si * sj * chord2));
          K *= wendland(d * inv_cut);
        }
      }
      if (!isfinite(K)) atomicOr(flags, kFlagNonFinite);
      val[e] = (T)K;
      if (P.symmetric && j == i) {
        kdiag[i] = (double)(T)K;
        prior_m[i] = P.log_rho_bar + log(si) -
                     (P.form == GM_FORM_LOGNORMAL ? 0.5 * (double)(T)K : 0.5 * P.sigma2);
      }
    }
  }
}

// An explicit list of pair geometries (distances si, sj in pc, chord |u_i -
// u_j|): K = log1p(R) (or R) without the taper; sj null: the self-covariance of
// the points si, at the precision of the stored entries.
template <typename Rule>
__global__ void __launch_bounds__(Rule::kBound) k_pair_list(
    QuadParams P, typename Rule::Par rp, int batch, int64_t n, const double* __restrict__ si,
    const double* __restrict__ sj, const double* __restrict__ chord, double* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Rule rule(rp, smem);
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p0 = warp * batch; p0 < n; p0 += nwarps * batch) {
    const int64_t p = p0 + lane;
    const bool active = lane < batch && p < n;
    double A = 1, B = 1, c2 = 0;
    if (active) {
      A = si[p] * P.inv_L0;
      B = sj ? sj[p] * P.inv_L0 : A;
      c2 = sj ? chord[p] * chord[p] : 0.0;
    }
    const double R = rule.R(active, A, B, c2);
    if (active) {
      const double K = P.form == GM_FORM_LOGNORMAL ? log1p(R) : R;
      out[p] = sj ? K : (double)(typename Rule::Val)K;
    }
  }
}

// ------------------------------------------------------------ host side
static TabF32 tab_f32() {
  TabF32 t;
  float xmin = ldexpf(1.0f, kTabF32.emin);
  std::memcpy(&t.base, &xmin, sizeof(int));  // bit pattern of 2^emin
  t.shift = 23 - kTabF32.m;
  t.last = kTabF32.n_real();
  t.xmin = xmin;
  return t;
}

static TabF64 tab_f64() {
  TabF64 t;
  double xmin = std::ldexp(1.0, kTabF64.emin);
  long long bits;
  std::memcpy(&bits, &xmin, sizeof(bits));  // bit pattern of 2^emin
  t.base = (int)(bits >> 32);
  t.shift = 20 - kTabF64.m;
  t.last = kTabF64.n_real();
  t.xmin = xmin;
  return t;
}

static const TableGeom& tab_geom(const gm_ctx* c) {
  return c->cfg.precision == GM_PREC_FP32 ? kTabF32 : kTabF64;
}

gm_status phi_points_init(gm_ctx* c) {
  const TableGeom& g = tab_geom(c);
  c->phi_pts = (double*)dev_alloc(c, g.n_pts() * sizeof(double));
  size_t tb = (size_t)(g.n_real() + 1) * (c->cfg.precision == GM_PREC_FP32 ? 16 : 32);
  c->gtab = dev_alloc(c, tb);
  if (!c->phi_pts || !c->gtab) return set_error(c, GM_E_NOMEM, "phi table");
  if (c->cfg.precision != GM_PREC_FP32) {
    c->gtab_df = dev_alloc(c, kDfSegs * (sizeof(float4) + sizeof(float2)));
    if (!c->gtab_df) return set_error(c, GM_E_NOMEM, "phi table");
  }
  const double cnorm = std::pow(2.0, 2.0 / 3.0) / std::tgamma(1.0 / 3.0);
  int blocks = (int)std::min<int64_t>(ceil_div(g.n_pts(), 128), 4 * sm_count(c));
  GM_PROF(c, "k_phi_points");
  k_phi_points<<<blocks, 128, 0, c->stream>>>(g, cnorm, c->phi_pts);
  GM_LAUNCH_CHECK(c);
  c->gtab_sigma2 = -1;
  return GM_OK;
}

gm_status gtab_update(gm_ctx* c) {
  if (c->gtab_sigma2 == c->cfg.sigma2 && c->gtab_form == c->cfg.form) return GM_OK;
  const TableGeom& g = tab_geom(c);
  int blocks = (int)std::min<int64_t>(ceil_div(g.n_real() + 1, 256), 4 * sm_count(c));
  GM_PROF(c, "k_gtab");
  if (c->cfg.precision == GM_PREC_FP32)
    k_gtab<float4><<<blocks, 256, 0, c->stream>>>(g, c->phi_pts, c->cfg.sigma2, c->cfg.form, 1,
                                                  (float4*)c->gtab);
  else
    k_gtab<D4><<<blocks, 256, 0, c->stream>>>(g, c->phi_pts, c->cfg.sigma2, c->cfg.form, 0,
                                                   (D4*)c->gtab);
  GM_LAUNCH_CHECK(c);
  if (c->cfg.precision != GM_PREC_FP32) {
    float4* t4 = (float4*)c->gtab_df;
    GM_PROF(c, "k_gtab_df");
    k_gtab_df<<<(kDfSegs + 255) / 256, 256, 0, c->stream>>>((const D4*)c->gtab, t4,
                                                            (float2*)(t4 + kDfSegs));
    GM_LAUNCH_CHECK(c);
  }
  c->gtab_sigma2 = c->cfg.sigma2;
  c->gtab_form = c->cfg.form;
  return GM_OK;
}

static QuadParams quad_params(const gm_ctx* c, bool symmetric) {
  QuadParams P;
  P.inv_L0 = 1.0 / c->cfg.outer_scale_pc;
  P.inv_cut = 1.0 / c->cfg.cutoff_pc;
  P.log_rho_bar = std::log(c->cfg.rho_bar);
  P.sigma2 = c->cfg.sigma2;
  P.Q = c->cfg.n_nodes;
  P.form = c->cfg.form;
  P.taper = c->cfg.taper;
  P.symmetric = symmetric ? 1 : 0;
  return P;
}

static BandTab band_tab() {
  BandTab t;
  for (int j = 0; j < kBandPts; ++j)
    t.pt[j] = gmband::kH0 * (std::pow(gmband::kQ, (double)j) - 1.0) / (gmband::kQ - 1.0);
  return t;
}

// Blocks and batch of a rule's kernel over n entries: the resident blocks, and
// the largest batch that still leaves every warp two (small lists: the pairs
// spread over the chip, one per warp in the limit).
template <typename Rule, typename Kern>
static void rule_shape(gm_ctx* c, Kern kern, int64_t n, int* blocks, int* batch) {
  constexpr int nt = Rule::kThreads;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Rule::smem());
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, Rule::smem());
  const int64_t resident = (int64_t)std::max(1, per_sm) * sm_count(c);
  int b = 32;
  while (b > 1 && n < 2 * b * resident * (nt / 32)) b >>= 1;
  *batch = b;
  *blocks = (int)std::min<int64_t>(resident, std::max<int64_t>(1, ceil_div(ceil_div(n, b), nt / 32)));
}

template <typename Rule>
static void launch_entries(gm_ctx* c, const QuadParams& P, const typename Rule::Par& rp,
                           int64_t n_rows, const double* rs, const double* rux, const double* ruy,
                           const double* ruz, const int32_t* row_field, const int64_t* row_ptr,
                           const int32_t* col, int64_t nnz, void* val, const char* name) {
  int blocks, batch;
  auto kern = k_pair_entries<Rule>;
  rule_shape<Rule>(c, kern, nnz, &blocks, &batch);
  GM_PROF(c, name);
  kern<<<blocks, Rule::kThreads, Rule::smem(), c->stream>>>(
      P, rp, batch, n_rows, rs, rux, ruy, ruz, c->s, c->ux, c->uy, c->uz, row_ptr, col, nnz,
      (typename Rule::Val*)val, c->kdiag, c->prior_m, c->d_flags, c->fgrid, row_field);
}

template <typename Rule>
static void launch_list(gm_ctx* c, const QuadParams& P, const typename Rule::Par& rp, int64_t n,
                        const double* si, const double* sj, const double* chord, double* out,
                        const char* name) {
  int blocks, batch;
  auto kern = k_pair_list<Rule>;
  rule_shape<Rule>(c, kern, n, &blocks, &batch);
  GM_PROF(c, name);
  kern<<<blocks, Rule::kThreads, Rule::smem(), c->stream>>>(P, rp, batch, n, si, sj, chord, out);
}

template <typename T>
static typename BandRule<T>::Par band_par(const gm_ctx* c) {
  return {band_tab(), c->gtab, tab_f64()};
}

template <int KPL>
static typename Gl32Rule<KPL>::Par gl32_par(const gm_ctx* c) {
  return {c->gl_zeta, c->gl_w, (const float4*)c->gtab, c->cfg.n_nodes};
}

template <int KPL>
static typename DfRule<KPL>::Par df_par(const gm_ctx* c) {
  const float4* t4 = (const float4*)c->gtab_df;
  return {c->gl_zeta, c->gl_w, (const D4*)c->gtab, tab_f64(), t4, (const float2*)(t4 + kDfSegs),
          c->cfg.n_nodes};
}

template <int KPL>
static typename Gl64Rule<KPL>::Par gl64_par(const gm_ctx* c) {
  return {c->gl_zeta, c->gl_w, (const D4*)c->gtab, tab_f64(), c->cfg.n_nodes};
}

// Whether the node sums of an FP64 context run in pairs of floats: g(0), its largest
// value, between 2^-30 (what it adds to a sum down to 2^-53 of that still has both
// parts above the smallest float) and 2^100 (sums and coefficients below the largest).
// For the lognormal form that is sigma2 up to 69; the FP64 form goes on to 520, where
// its table, g over the cube of a segment, overflows.
static bool df_fits(const gm_ctx* c) {
  const char* e = std::getenv("GM_QUAD");
  if (e && std::strcmp(e, "fp64") == 0) return false;
  const double g0 = c->cfg.form == GM_FORM_LOGNORMAL ? std::expm1(c->cfg.sigma2) : c->cfg.sigma2;
  return g0 >= 0x1p-30 && g0 <= 0x1p100;
}

gm_status pair_quadrature(gm_ctx* c, int64_t n_rows, const double* rs, const double* rux,
                          const double* ruy, const double* ruz, const int32_t* row_field,
                          const int64_t* row_ptr, const int32_t* col, int64_t nnz, void* val,
                          bool symmetric) {
  if (nnz == 0) return GM_OK;
  gm_status st = gtab_update(c);
  if (st != GM_OK) return st;
  QuadParams P = quad_params(c, symmetric);
  const int Q = c->cfg.n_nodes;
  const bool f32 = c->cfg.precision == GM_PREC_FP32;
  const bool df = !f32 && df_fits(c);
#define GM_ENTRIES(RULE, PAR, NAME) \
  launch_entries<RULE>(c, P, PAR, n_rows, rs, rux, ruy, ruz, row_field, row_ptr, col, nnz, val, NAME)
  if (c->cfg.quad_rule == GM_QUAD_BAND) {
    if (f32) GM_ENTRIES(BandRule<float>, band_par<float>(c), "k_pair_quad_band");
    else GM_ENTRIES(BandRule<double>, band_par<double>(c), "k_pair_quad_band");
  } else if (Q <= 32) {
    if (f32) GM_ENTRIES(Gl32Rule<1>, gl32_par<1>(c), "k_pair_quad");
    else if (df) GM_ENTRIES(DfRule<1>, df_par<1>(c), "k_pair_quad");
    else GM_ENTRIES(Gl64Rule<1>, gl64_par<1>(c), "k_pair_quad_fp64");
  } else if (Q <= 64) {
    if (f32) GM_ENTRIES(Gl32Rule<2>, gl32_par<2>(c), "k_pair_quad");
    else if (df) GM_ENTRIES(DfRule<2>, df_par<2>(c), "k_pair_quad");
    else GM_ENTRIES(Gl64Rule<2>, gl64_par<2>(c), "k_pair_quad_fp64");
  } else {
    if (f32) GM_ENTRIES(Gl32Rule<4>, gl32_par<4>(c), "k_pair_quad");
    else if (df) GM_ENTRIES(DfRule<4>, df_par<4>(c), "k_pair_quad");
    else GM_ENTRIES(Gl64Rule<4>, gl64_par<4>(c), "k_pair_quad_fp64");
  }
#undef GM_ENTRIES
  GM_LAUNCH_CHECK(c);
  if (symmetric) {
    int blocks = (int)std::min<int64_t>(ceil_div(nnz, 256), 16 * sm_count(c));
    GM_PROF(c, "k_mirror");
    if (f32) k_mirror<float><<<blocks, 256, 0, c->stream>>>(n_rows, row_ptr, col, nnz, (float*)val);
    else k_mirror<double><<<blocks, 256, 0, c->stream>>>(n_rows, row_ptr, col, nnz, (double*)val);
    GM_LAUNCH_CHECK(c);
  }
  return GM_OK;
}

gm_status mirror_csr(gm_ctx* c, int64_t n, const int64_t* row_ptr, const int32_t* col, int64_t nnz,
                     void* val) {
  if (nnz == 0) return GM_OK;
  int blocks = (int)std::min<int64_t>(ceil_div(nnz, 256), 16 * sm_count(c));
  GM_PROF(c, "k_mirror");
  if (c->cfg.precision == GM_PREC_FP32)
    k_mirror<float><<<blocks, 256, 0, c->stream>>>(n, row_ptr, col, nnz, (float*)val);
  else
    k_mirror<double><<<blocks, 256, 0, c->stream>>>(n, row_ptr, col, nnz, (double*)val);
  GM_LAUNCH_CHECK(c);
  return GM_OK;
}

gm_status self_quadrature(gm_ctx* c, int64_t n_rows, const double* rs, double* kss) {
  if (n_rows == 0) return GM_OK;
  gm_status st = gtab_update(c);
  if (st != GM_OK) return st;
  QuadParams P = quad_params(c, false);
  const int Q = c->cfg.n_nodes;
  const bool f32 = c->cfg.precision == GM_PREC_FP32;
  int blocks = (int)std::min<int64_t>(ceil_div(n_rows * 32, 256), 8 * sm_count(c));
#define GM_SELF32(K)                                                                      \
  k_self_quad<K><<<blocks, 256, 0, c->stream>>>(P, n_rows, rs, c->gl_zeta, c->gl_w, c->gtab, \
                                                tab_f32(), kss)
#define GM_SELF64(K)                                                                             \
  do {                                                                                           \
    if (df_fits(c))                                                                              \
      launch_list<DfRule<K>>(c, P, df_par<K>(c), n_rows, rs, nullptr, nullptr, kss, "k_self_quad"); \
    else                                                                                         \
      launch_list<Gl64Rule<K>>(c, P, gl64_par<K>(c), n_rows, rs, nullptr, nullptr, kss,          \
                               "k_self_quad_fp64");                                              \
  } while (0)
  if (c->cfg.quad_rule == GM_QUAD_BAND) {
    if (f32)
      launch_list<BandRule<float>>(c, P, band_par<float>(c), n_rows, rs, nullptr, nullptr, kss,
                                   "k_self_quad_band");
    else
      launch_list<BandRule<double>>(c, P, band_par<double>(c), n_rows, rs, nullptr, nullptr, kss,
                                    "k_self_quad_band");
  } else if (f32) {
    GM_PROF(c, "k_self_quad");
    if (Q <= 32) GM_SELF32(1);
    else if (Q <= 64) GM_SELF32(2);
    else GM_SELF32(4);
  } else {
    if (Q <= 32) GM_SELF64(1);
    else if (Q <= 64) GM_SELF64(2);
    else GM_SELF64(4);
  }
#undef GM_SELF32
#undef GM_SELF64
  GM_LAUNCH_CHECK(c);
  return GM_OK;
}

}  // namespace gm

namespace gm {

// Sightline quadrature for an explicit list of pair geometries (distances
// si, sj in pc, chord |u_i - u_j|): K = log1p(R) (or R) without the taper.
// FP32 form; same rule and kernel table as the covariance assembly; one warp
// per pair.
template <int KPL>
__global__ void __launch_bounds__(256) k_pairlist_quad(
    QuadParams P, int64_t n, const double* __restrict__ si, const double* __restrict__ sj,
    const double* __restrict__ chord, double* __restrict__ out,
    const double* __restrict__ gl_zeta, const double* __restrict__ gl_w,
    const float4* __restrict__ gtab, TabF32 tf) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* zq = reinterpret_cast<float*>(smem);
  float* wq = zq + kMaxNodes;
  float4* tab = reinterpret_cast<float4*>(smem + 2 * kMaxNodes * sizeof(float));
  for (int k = threadIdx.x; k <= tf.last; k += blockDim.x) tab[k] = gtab[k];
  for (int q = threadIdx.x; q < P.Q; q += blockDim.x) {
    zq[q] = (float)gl_zeta[q];
    wq[q] = (float)gl_w[q];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p = warp; p < n; p += nwarps) {
    const float a = (float)(si[p] * P.inv_L0), b = (float)(sj[p] * P.inv_L0);
    const float c2 = (float)(chord[p] * chord[p]);
    float tp[KPL], ctp[KPL], wp[KPL];
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
      int q = lane + 32 * k;
      bool ok = q < P.Q;
      tp[k] = ok ? b * zq[q] : 0.f;
      ctp[k] = c2 * tp[k];
      wp[k] = ok ? wq[q] : 0.f;
    }
    float acc = 0;
    for (int q = 0; q < P.Q; ++q) {
      const float t = a * zq[q];
      float inner = 0;
#pragma unroll
      for (int k = 0; k < KPL; ++k) {
        const float d = t - tp[k];
        inner += wp[k] * g_lookup(tab, tf, d * d + t * ctp[k]);
      }
      acc += wq[q] * inner;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) {
      const double R = (double)acc;
      out[p] = P.form == GM_FORM_LOGNORMAL ? log1p(R) : R;
    }
  }
}

template <int KPL>
static void launch_pairlist(gm_ctx* c, const QuadParams& P, int64_t n, const double* si,
                            const double* sj, const double* chord, double* out) {
  const size_t smem = 2 * kMaxNodes * sizeof(float) + (size_t)(kTabF32.n_real() + 1) * sizeof(float4);
  auto kern = k_pairlist_quad<KPL>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem);
  int blocks = std::max(1, per_sm) * sm_count(c);
  blocks = (int)std::min<int64_t>(blocks, std::max<int64_t>(1, ceil_div(n * 32, 256)));
  GM_PROF(c, "k_pairlist_quad");
  kern<<<blocks, 256, smem, c->stream>>>(P, n, si, sj, chord, out, c->gl_zeta, c->gl_w,
                                         (const float4*)c->gtab, tab_f32());
}

gm_status pairlist_quadrature(gm_ctx* c, int64_t n, const double* si, const double* sj,
                              const double* chord, double* out) {
  if (n == 0) return GM_OK;
  gm_status st = gtab_update(c);
  if (st != GM_OK) return st;
  QuadParams P = quad_params(c, false);
  const int Q = c->cfg.n_nodes;
  const bool f32 = c->cfg.precision == GM_PREC_FP32;
  const bool df = !f32 && df_fits(c);
#define GM_LIST(RULE, PAR, NAME) launch_list<RULE>(c, P, PAR, n, si, sj, chord, out, NAME)
  if (c->cfg.quad_rule == GM_QUAD_BAND) {
    if (f32) GM_LIST(BandRule<float>, band_par<float>(c), "k_pairlist_quad_band");
    else GM_LIST(BandRule<double>, band_par<double>(c), "k_pairlist_quad_band");
  } else if (Q <= 32) {
    if (f32) launch_pairlist<1>(c, P, n, si, sj, chord, out);
    else if (df) GM_LIST(DfRule<1>, df_par<1>(c), "k_pairlist_quad");
    else GM_LIST(Gl64Rule<1>, gl64_par<1>(c), "k_pairlist_quad_fp64");
  } else if (Q <= 64) {
    if (f32) launch_pairlist<2>(c, P, n, si, sj, chord, out);
    else if (df) GM_LIST(DfRule<2>, df_par<2>(c), "k_pairlist_quad");
    else GM_LIST(Gl64Rule<2>, gl64_par<2>(c), "k_pairlist_quad_fp64");
  } else {
    if (f32) launch_pairlist<4>(c, P, n, si, sj, chord, out);
    else if (df) GM_LIST(DfRule<4>, df_par<4>(c), "k_pairlist_quad");
    else GM_LIST(Gl64Rule<4>, gl64_par<4>(c), "k_pairlist_quad_fp64");
  }
#undef GM_LIST
  GM_LAUNCH_CHECK(c);
  return GM_OK;
}

}  // namespace gm
