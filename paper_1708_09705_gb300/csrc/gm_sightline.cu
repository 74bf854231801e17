// Sightline sampler of the dA/ds >= 0 conditioning (Sect. 5): exact HMC for
// each sightline's truncated Gaussian predictive: a few lanes per sightline up to 32
// points, one thread beyond that.
// The per-sightline arithmetic is in gm_hmc.cuh.
#include <algorithm>
#include <cstdlib>

#include "gm_hmc.cuh"
#include "gm_internal.cuh"

namespace gm {

// Caller layout (sightline-major) -> sightline-fastest scratch:
// mu_t[i * nsl + q] = mean[q * m + i], S_t[e * nsl + q] = cov[q * m * m + e].
__global__ void k_sl_stage(int64_t nsl, int m, const double* __restrict__ mean,
                           const double* __restrict__ cov, double* __restrict__ mu_t,
                           double* __restrict__ S_t, unsigned* __restrict__ flags) {
  const int64_t per = (int64_t)m + (int64_t)m * m;
  const int64_t total = per * nsl;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = k / nsl, q = k - e * nsl;
    double v;
    if (e < m) {
      v = mean[q * m + e];
      mu_t[e * nsl + q] = v;
    } else {
      v = cov[q * (int64_t)m * m + (e - m)];
      S_t[(e - m) * nsl + q] = v;
    }
    if (!isfinite(v)) atomicOr(flags, kFlagNonFinite);
  }
}

__global__ void __launch_bounds__(128)
    k_monotone_hmc(int64_t nsl, int m, int n_burn, int n_samples,
                   const double* __restrict__ mu_t, const double* __restrict__ S_t,
                   double* __restrict__ L_t, double* __restrict__ y_t, double* __restrict__ w_t,
                   const double* __restrict__ mom, double* __restrict__ out,
                   int64_t* __restrict__ hits, unsigned* __restrict__ flags) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= nsl) return;
  const int64_t T = (int64_t)n_burn + n_samples;
  int64_t h = 0;
  const unsigned s = gmhmc::sample_sightline(mu_t + q, S_t + q, L_t + q, y_t + q, w_t + q, nsl,
                                             mom + q * T * m, out + q * (int64_t)n_samples * m,
                                             m, n_burn, n_samples, &h);
  hits[q] = h;
  if (s & gmhmc::kNotPD) atomicOr(flags, kFlagNotSPD);
  if (s & gmhmc::kHitLimit) atomicOr(flags, kFlagHitLimit);
}

// One warp per sightline (m <= 32), two warps per block; the warp's state,
// S and L live in shared memory (gmhmc::WarpState), the phases of a step are
// separated by warp barriers.  Same chain as k_monotone_hmc.
__global__ void __launch_bounds__(64)
    k_monotone_hmc_warp(int64_t nsl, int m, int n_burn, int n_samples,
                        const double* __restrict__ mu_t, const double* __restrict__ S_t,
                        const double* __restrict__ mom, double* __restrict__ out,
                        int64_t* __restrict__ hits, unsigned* __restrict__ flags) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t q = blockIdx.x * 2 + wib;
  if (q >= nsl) return;  // the whole warp
  const size_t per = sizeof(gmhmc::WarpState) + 2 * (size_t)m * m * sizeof(double);
  gmhmc::WarpState& W = *reinterpret_cast<gmhmc::WarpState*>(sm + wib * per);
  if (lane == 0) {
    W.S = reinterpret_cast<double*>(sm + wib * per + sizeof(gmhmc::WarpState));
    W.L = W.S + m * m;
  }
  __syncwarp();
  gmhmc::w_stage(W, lane, m, mu_t + q, S_t + q, nsl);
  __syncwarp();
  if (lane == 0) gmhmc::w_setup(W, m);
  __syncwarp();
  const int64_t T = (int64_t)n_burn + n_samples;
  double* o = out + q * (int64_t)n_samples * m;
  if (W.status) {
    for (int64_t k = lane; k < (int64_t)n_samples * m; k += 32) o[k] = NAN;
    if (lane == 0) {
      hits[q] = 0;
      atomicOr(flags, kFlagNotSPD);
    }
    return;
  }
  unsigned status = 0;
  for (int64_t it = 0; it < T; ++it) {
    gmhmc::w_momentum(W, lane, m, mom + (q * T + it) * m);
    __syncwarp();
    gmhmc::w_velocity(W, lane, m);
    if (lane == 0) W.t_left = gmhmc::kHalfPi;
    __syncwarp();
    int n = 0;
    for (; n < gmhmc::kMaxWallHits; ++n) {
      gmhmc::w_hit(W, lane, m);
      __syncwarp();
      double tb;
      const int j = gmhmc::w_best(W, m, &tb);
      if (j < 0) {
        gmhmc::w_rotate(W, lane, m, W.t_left);
        __syncwarp();
        break;
      }
      gmhmc::w_rotate(W, lane, m, tb);
      __syncwarp();
      if (lane == 0) gmhmc::w_reflect_factor(W, m, j);
      __syncwarp();
      gmhmc::w_reflect(W, lane, m, j);
      __syncwarp();
      if (lane == 0) {
        W.t_left -= tb;
        W.nhits++;
      }
      __syncwarp();
    }
    if (n == gmhmc::kMaxWallHits) status |= gmhmc::kHitLimit;
    if (it >= n_burn && lane < m) o[(it - n_burn) * m + lane] = W.mu[lane] + W.y[lane];
    __syncwarp();
  }
  if (lane == 0) {
    hits[q] = W.nhits;
    if (status & gmhmc::kHitLimit) atomicOr(flags, kFlagHitLimit);
  }
}

// Up to 32 points: LPS lanes per sightline, PPL consecutive points a lane.  The
// chain is the one of gmhmc::sample_sightline, value for value: a chain that
// starts in a narrow wedge between walls amplifies the last bit by 1e8, so the
// times, rotations and reflections keep that routine's expressions.  What
// bounds it is FP64 issue, and nearly all of it was trigonometry of walls that
// are not the next one (hypot, atan2, acos, sin, cos: about 400 instructions a
// wall, one per 16 clocks and SM).  So the walls are screened first: with u =
// tan(t / 2), wall j is met where (c - a) u^2 + 2 b u + (c + a) = 0, and the root
// with the gap closing is algebraic; in FP32 (from FP64 differences) it gives
// each wall's time to 1e-5.  Only walls within the margin of the earliest are
// timed by the full expressions, by the lanes that hold them, all sightlines of
// the warp at once; a wall whose estimate was wrong by more than the margin is
// still found, because the screening repeats without the walls already timed
// until none can be earlier.  The outward root is t = phi + acos(-c / r) unless
// the hit grazes, where the sign of the derivative is evaluated as before.
// The sightlines of a warp do not wait for each other's steps.
// A call of 4,096 sightlines x 16 points x 120 steps: 193 ms with one thread per
// sightline timing every wall, 19.0 ms so (bit for bit the same samples).
constexpr float kHgMargin = 1.02f;    // of the estimate (relative) ...
constexpr float kHgFloor = 4e-6f;     // ... and of u near zero (absolute)

template <int LPS, int PPL>
struct Hg {  // shared doubles per sightline: L, S f_j, momenta, f_j^T S f_j
  static constexpr int M = LPS * PPL;
  static constexpr int doubles = 2 * M * M + 2 * M;
};

// Time of the first outward hit of one wall in (kHitEps, t_left], or -1.
__device__ __forceinline__ double hg_wall_time(double a, double b, double c, double t_left) {
  const double r = hypot(a, b);
  if (r <= fabs(c)) return -1.0;
  const double ph = atan2(b, a);
  const double ac = acos(-c / r);
  // 0 < ac < pi: the derivative -r sin(t - phi) is negative at phi + ac and
  // positive at phi - ac, as computed too unless ac is within rounding of 0
  // or pi
  const bool graze = !(ac > 1e-5 && ac < 3.14158);
  double bt = -1.0;
  for (int s = 0; s < (graze ? 2 : 1); ++s) {
    double t = s == 0 ? ph + ac : ph - ac;
    if (fabs(t) >= gmhmc::kTwoPi) t = fmod(t, gmhmc::kTwoPi);
    if (t < 0.0) t += gmhmc::kTwoPi;
    if (t > gmhmc::kHitEps && t <= t_left) {
      const bool outward = graze ? -a * sin(t) + b * cos(t) < 0.0 : true;
      if (outward && (bt < 0.0 || t < bt)) bt = t;
    }
  }
  return bt;
}

template <int LPS, int PPL>
__global__ void __launch_bounds__(32)
    k_monotone_hmc_group(int64_t nsl, int m, int n_burn, int n_samples,
                         const double* __restrict__ mean, const double* __restrict__ cov,
                         const double* __restrict__ mom, double* __restrict__ out,
                         int64_t* __restrict__ hits, unsigned* __restrict__ flags) {
  constexpr int M = Hg<LPS, PPL>::M;
  constexpr unsigned full = 0xffffffffu;
  extern __shared__ __align__(16) double hg_sm[];
  const int lane = threadIdx.x & 31, sub = lane & (LPS - 1), grp = lane / LPS;
  const unsigned gmask = (LPS == 32 ? full : ((1u << LPS) - 1u)) << (LPS * grp);
  const int64_t q0 = (int64_t)blockIdx.x * (32 / LPS) + grp;
  const bool real = q0 < nsl;
  const int64_t q = real ? q0 : nsl - 1;  // an idle group shadows the last sightline, done at once
  double* L = hg_sm + grp * Hg<LPS, PPL>::doubles;  // L[k * M + i]
  double* D = L + M * M;                            // D[j * M + i] = S[i][j + 1] - S[i][j]
  double* P = D + M * M;
  double* NN = P + M;
  const double* S = cov + q * (int64_t)m * m;
  const double* mu_q = mean + q * m;
  auto Sel = [&](int r, int c) { return r >= c ? S[r * m + c] : S[c * m + r]; };

  // Cholesky factor, the lanes over the rows of a column (sums in the order of
  // gmhmc::cholesky)
  for (int e = sub; e < M * M; e += LPS) L[e] = D[e] = 0.0;
  __syncwarp();
  bool pd = true;
  for (int j = 0; j < m; ++j) {
    double d = Sel(j, j);
    for (int k = 0; k < j; ++k) {
      const double v = L[k * M + j];
      d -= v * v;
    }
    if (!(d > 0.0)) pd = false;  // the same in every lane of the group
    d = sqrt(d);
    for (int i = j + sub; i < m; i += LPS) {
      double v = Sel(i, j);
      for (int k = 0; k < j; ++k) v -= L[k * M + i] * L[k * M + j];
      L[j * M + i] = i == j ? d : v / d;
    }
    __syncwarp();
  }
  for (int j = 0; j + 1 < m; ++j)
    for (int i = sub; i < m; i += LPS) D[j * M + i] = Sel(i, j + 1) - Sel(i, j);
  for (int j = sub; j + 1 < m; j += LPS)
    NN[j] = Sel(j + 1, j + 1) + Sel(j, j) - 2.0 * Sel(j + 1, j);
  __syncwarp();

  double mu[PPL], y[PPL], w[PPL], c[PPL], pn[PPL];
  {
    double run = mu_q[0];
    for (int i = 1; i < sub * PPL && i < m; ++i) run = mu_q[i] > run ? mu_q[i] : run;
#pragma unroll
    for (int k = 0; k < PPL; ++k) {
      const int i = sub * PPL + k;
      mu[k] = y[k] = w[k] = c[k] = 0.0;
      if (i < m) {
        mu[k] = mu_q[i];
        run = mu[k] > run ? mu[k] : run;
        y[k] = (run + 1e-9 * i) - mu[k];
        if (i + 1 < m) c[k] = mu_q[i + 1] - mu[k];
      }
    }
  }
  const int64_t T = (int64_t)n_burn + n_samples;
  const double* mq = mom + q * T * m;
  double* o = out + q * (int64_t)n_samples * m;
  if (real && !pd) {
    for (int64_t k = sub; k < (int64_t)n_samples * m; k += LPS) o[k] = NAN;
    if (sub == 0) {
      hits[q] = 0;
      atomicOr(flags, kFlagNotSPD);
    }
  }
  bool live = real && pd && T > 0;
  int64_t it = 0, n_hits = 0;
  int n = 0;
  double t_left = gmhmc::kHalfPi;
  bool limit = false;
  auto fetch = [&](int64_t step) {
#pragma unroll
    for (int k = 0; k < PPL; ++k) {
      const int i = sub * PPL + k;
      pn[k] = (live && step < T && i < m) ? mq[step * m + i] : 0.0;
    }
  };
  // a new step: momenta to shared memory, w = L p (sums in order)
  auto begin = [&]() {
#pragma unroll
    for (int k = 0; k < PPL; ++k) P[sub * PPL + k] = pn[k];
    __syncwarp(gmask);
#pragma unroll
    for (int k = 0; k < PPL; ++k) w[k] = 0.0;
    for (int l = 0; l < m; ++l) {
      const double pl = P[l];
#pragma unroll
      for (int k = 0; k < PPL; ++k) w[k] += L[l * M + sub * PPL + k] * pl;
    }
    __syncwarp(gmask);
    t_left = gmhmc::kHalfPi;
    n = 0;
    fetch(it + 1);
  };
  fetch(0);
  if (live) begin();
  if (real && pd && T == 0 && sub == 0) hits[q] = 0;

  // every round: the earliest wall of each live sightline, the motion up to it
  // (or to the end of the step), then the reflection or the next step.  At
  // most T (kMaxWallHits + 1) rounds.
  while (__any_sync(full, live)) {
    const double yn = __shfl_down_sync(full, y[0], 1, LPS);
    const double wn = __shfl_down_sync(full, w[0], 1, LPS);
    const float U = tanf(0.5f * (float)t_left) * kHgMargin + kHgFloor;
    // estimate of each wall's u (infinity: not met)
    float ue[PPL];
#pragma unroll
    for (int k = 0; k < PPL; ++k) {
      const int j = sub * PPL + k;
      const double a = (k + 1 < PPL ? y[k + 1 < PPL ? k + 1 : 0] : yn) - y[k];
      const double b = (k + 1 < PPL ? w[k + 1 < PPL ? k + 1 : 0] : wn) - w[k];
      const float cp = (float)(c[k] + a), cm = (float)(c[k] - a), bf = (float)b;
      const float b2 = bf * bf, cc = cm * cp;
      const float disc = b2 - cc, fuzz = 1e-5f * (b2 + fabsf(cc));
      const float s = sqrtf(fmaxf(disc, 0.f));
      // closing: the gap shrinks from cp; opening: it grows, and closes later
      float u = bf < 0.f ? fmaxf(cp, 0.f) / (s - bf) : (bf + s) / -cm;
      // grazing within the estimate's own error: the motion turns at -b / cm
      if (fabsf(disc) <= fuzz) u = fmaxf(0.98f * fminf(u, -bf / cm), 0.f);
      bool met = disc > -fuzz && u >= 0.f && u <= U && !(bf < 0.f && cp < -1e-9f);
      // values whose squares leave the range of floats: timed, whatever they estimate
      const float big = fmaxf(fabsf(bf), fmaxf(fabsf(cp), fabsf(cm)));
      if (!(big > 1e-15f && big < 1e15f)) {
        met = true;
        u = 0.f;
      }
      ue[k] = met && live && j + 1 < m ? u : INFINITY;
    }
    double th = 0.0;
    int bj = M;
    for (;;) {
      float um = ue[0];
#pragma unroll
      for (int k = 1; k < PPL; ++k) um = fminf(um, ue[k]);
#pragma unroll
      for (int off = 1; off < LPS; off <<= 1) um = fminf(um, __shfl_xor_sync(full, um, off));
      const float cut = bj < M ? tanf(0.5f * (float)th) * kHgMargin + kHgFloor : INFINITY;
      const bool more = um < INFINITY && um <= cut;
      if (!__any_sync(full, more)) break;
      // one wall at a time per lane, the smallest estimate first
      double t = -1.0;
      int j = M;
      if (more) {
        float mine = INFINITY;
        double a = 0.0, b = 0.0, cw = 0.0;
#pragma unroll
        for (int k = 0; k < PPL; ++k)
          if (ue[k] < mine) {
            mine = ue[k];
            j = sub * PPL + k;
            a = (k + 1 < PPL ? y[k + 1 < PPL ? k + 1 : 0] : yn) - y[k];
            b = (k + 1 < PPL ? w[k + 1 < PPL ? k + 1 : 0] : wn) - w[k];
            cw = c[k];
          }
        if (mine <= um * kHgMargin + kHgFloor) {
#pragma unroll
          for (int k = 0; k < PPL; ++k)
            if (j == sub * PPL + k) ue[k] = INFINITY;
          t = hg_wall_time(a, b, cw, t_left);
        }
      }
      __syncwarp();
      if (t < 0.0) {
        t = INFINITY;
        j = M;
      }
#pragma unroll
      for (int off = 1; off < LPS; off <<= 1) {
        const double ot = __shfl_xor_sync(full, t, off);
        const int oj = __shfl_xor_sync(full, j, off);
        if (ot < t || (ot == t && oj < j)) {
          t = ot;
          j = oj;
        }
      }
      if (j < M && (bj == M || t < th || (t == th && j < bj))) {
        th = t;
        bj = j;
      }
    }
    const bool hit = bj < M;
    if (live) {
      const double t = hit ? th : t_left;
      const double ct = cos(t), sn = sin(t);
#pragma unroll
      for (int k = 0; k < PPL; ++k) {
        const double yi = y[k], wi = w[k];
        y[k] = yi * ct + wi * sn;
        w[k] = -yi * sn + wi * ct;
      }
    }
    __syncwarp();
    // the rotated velocities of the wall's two points
    const int j0 = hit ? bj : 0, j1 = hit ? bj + 1 : 0;
    double s0 = w[0], s1 = w[0];
#pragma unroll
    for (int k = 1; k < PPL; ++k) {
      if (j0 % PPL == k) s0 = w[k];
      if (j1 % PPL == k) s1 = w[k];
    }
    const double w0 = __shfl_sync(full, s0, j0 / PPL, LPS);
    const double w1 = __shfl_sync(full, s1, j1 / PPL, LPS);
    if (live && hit) {
      const double b = w1 - w0;
      const double f = 2.0 * b / NN[j0];
#pragma unroll
      for (int k = 0; k < PPL; ++k) w[k] -= f * D[j0 * M + sub * PPL + k];
      t_left -= th;
      ++n_hits;
      ++n;
    }
    if (live && (!hit || n == gmhmc::kMaxWallHits)) {
      if (hit) limit = true;
      if (it >= n_burn) {
#pragma unroll
        for (int k = 0; k < PPL; ++k) {
          const int i = sub * PPL + k;
          if (i < m) o[(it - n_burn) * m + i] = mu[k] + y[k];
        }
      }
      ++it;
      if (it < T) {
        begin();
      } else {
        live = false;
        if (sub == 0) {
          hits[q] = n_hits;
          if (limit) atomicOr(flags, kFlagHitLimit);
        }
      }
    }
    __syncwarp();
  }
}

__global__ void k_sl_check(int64_t total, const double* __restrict__ a, unsigned* __restrict__ flags) {
  bool bad = false;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x)
    bad = bad || !isfinite(a[k]);
  if (bad) atomicOr(flags, kFlagNonFinite);
}

template <int LPS, int PPL>
static gm_status launch_group(gm_ctx* c, int64_t nsl, int m, const double* mean, const double* cov,
                              const double* mom, int n_burn, int n_samples, double* out,
                              int64_t* hits, unsigned* flags) {
  const size_t smem = (32 / LPS) * (size_t)Hg<LPS, PPL>::doubles * sizeof(double);
  auto kern = k_monotone_hmc_group<LPS, PPL>;
  GM_CUDA_CHECK(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem));
  kern<<<(unsigned)ceil_div(nsl, 32 / LPS), 32, smem, c->stream>>>(
      nsl, m, n_burn, n_samples, mean, cov, mom, out, hits, flags);
  GM_LAUNCH_CHECK(c);
  return GM_OK;
}

gm_status monotone_sample(gm_ctx* c, int64_t nsl, int m, const double* mean, const double* cov,
                          const double* mom, int n_burn, int n_samples, double* out,
                          int64_t* hits, unsigned* flags) {
  const int64_t mm = (int64_t)m * m;
  // GM_HMC_WARP = 0 / 1 select the one-thread and one-warp kernels (the latter
  // up to 32 points); else from 3 to 32 points a few lanes per sightline, straight
  // from the caller's arrays (two points have one wall, met every other step at
  // most: one thread 0.44 ms, four lanes 1.2 ms for 30,000 x 60 steps)
  const char* e = std::getenv("GM_HMC_WARP");
  const bool warp = m <= gmhmc::kWarpMax && e && e[0] == '1';
  const bool group = m > 2 && m <= 32 && !warp && !(e && e[0] == '0');
  // scratch: mu_t (m), S_t (m^2), L_t (m^2), y_t (m), w_t (m) per sightline
  const size_t bytes = group ? 0 : (size_t)nsl * (3 * m + 2 * mm) * sizeof(double);
  ScopedDev buf(c, std::max<size_t>(bytes, 16));
  double* ws = (double*)buf.p;
  if (!ws) return set_error(c, GM_E_NOMEM, "sampler scratch");
  double *mu_t = ws, *S_t = mu_t + nsl * m, *L_t = S_t + nsl * mm, *y_t = L_t + nsl * mm,
         *w_t = y_t + nsl * m;
  const int64_t per = m + mm;
  const int sb = (int)std::max<int64_t>(
      1, std::min<int64_t>(ceil_div(per * nsl, 256), 8 * sm_count(c)));
  if (group) {
    GM_PROF(c, "k_sl_check");
    k_sl_check<<<sb, 256, 0, c->stream>>>(nsl * m, mean, flags);
    GM_LAUNCH_CHECK(c);
    GM_PROF(c, "k_sl_check");
    k_sl_check<<<sb, 256, 0, c->stream>>>(nsl * mm, cov, flags);
    GM_LAUNCH_CHECK(c);
  } else {
    GM_PROF(c, "k_sl_stage");
    k_sl_stage<<<sb, 256, 0, c->stream>>>(nsl, m, mean, cov, mu_t, S_t, flags);
    GM_LAUNCH_CHECK(c);
  }
  {
    unsigned* h = (unsigned*)c->h_pinned;
    GM_CUDA_CHECK(c, cudaMemcpyAsync(h, flags, sizeof(unsigned), cudaMemcpyDeviceToHost,
                                     c->stream));
    GM_CUDA_CHECK(c, cudaStreamSynchronize(c->stream));
    if (*h & kFlagNonFinite) return GM_OK;  // the caller reads the flag and reports it
  }
  if (group) {
    GM_PROF(c, "k_monotone_hmc");
    // Two points a lane at least (one a lane contracts the rotation's products
    // differently).  Measured (ms for 60 steps, one thread / 4 / 8 / 16 lanes per
    // sightline): 4,096 x 16 points 128 / 15.3 / 14.5 / -, 32,768 x 16 259 / 72 /
    // 84 / -, 2,048 x 32 537 / 61 / 40 / 35, 8,192 x 8 19 / 4.5 / - / -.
    gm_status st;
#define GM_HG(A, B) launch_group<A, B>(c, nsl, m, mean, cov, mom, n_burn, n_samples, out, hits, flags)
    if (m > 16) st = GM_HG(16, 2);
    else if (m > 8) st = nsl <= 8192 ? GM_HG(8, 2) : GM_HG(4, 4);
    else st = GM_HG(4, 2);
#undef GM_HG
    if (st != GM_OK) return st;
  } else if (warp) {
    const size_t per = sizeof(gmhmc::WarpState) + 2 * (size_t)m * m * sizeof(double);
    GM_PROF(c, "k_monotone_hmc_warp");
    k_monotone_hmc_warp<<<(unsigned)ceil_div(nsl, 2), 64, 2 * per, c->stream>>>(
        nsl, m, n_burn, n_samples, mu_t, S_t, mom, out, hits, flags);
    GM_LAUNCH_CHECK(c);
  } else {
    GM_PROF(c, "k_monotone_hmc");
    k_monotone_hmc<<<(unsigned)ceil_div(nsl, 128), 128, 0, c->stream>>>(
        nsl, m, n_burn, n_samples, mu_t, S_t, L_t, y_t, w_t, mom, out, hits, flags);
    GM_LAUNCH_CHECK(c);
  }
  GM_CUDA_CHECK(c, cudaStreamSynchronize(c->stream));
  return GM_OK;
}

}  // namespace gm
