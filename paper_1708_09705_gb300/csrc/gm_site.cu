// EP site update, FP64, one lane per star or several (App. A.2).
//
// For star i with posterior marginal N(mu_i, Sigma_ii) and site (tau_i, nu_i):
//   cavity (eq. cavity):  tau_c = 1/Sigma_ii - tau_i, nu_c = mu_i/Sigma_ii - nu_i,
//     with the cavity variance floored (Sect. 5); tau_c <= 0 skips the star;
//   tilted (eq. tilted):  N(a; mu_c, v_c) * L_i(a), L_i the star's likelihood;
//   moment matching (eq. KL1'): mean mh and variance vh of the tilted give
//     tau_new = 1/vh - tau_c, nu_new = mh/vh - nu_c;
//   damped replacement; an update with tau_new < 0 is skipped.
// Gaussian-in-ln-A likelihood: the tilted is Gaussian (closed form).
// Gaussian-in-A likelihood: mode and curvature of the tilted log-density by
// safeguarded Newton ascent, then a 64-node Gauss-Hermite rule centred at the
// mode and scaled by the curvature.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "gm_internal.cuh"

namespace gm {

struct SiteParams {
  double damping;
  double vc_floor;
};

// Work split.  A group of G lanes (a power of two up to 32) owns a star: every
// lane of the group runs the Newton ascent (the same numbers; FP64 issues per
// warp, so the copies cost nothing while the chip is idle), then lane k of the
// group sums nodes k, k + G, ... of the 64-node rule and shuffles add the three
// sums.  GB300 issues an FP64 warp instruction every ~64 clocks per scheduler,
// so the kernel is bound by the length of a warp's FP64 instruction chain until
// every scheduler has a warp: G is the largest group for which the stars still
// fit one warp per scheduler (site_group).  The ascent evaluates exp once per
// trial point (the accepted trial's value serves the next step) and takes the
// last steps, below 1e-7 where Newton is quadratic, without the line search,
// whose comparison of log-densities is rounding noise there.
// A call of the allocation-free update on 400 stars: 485 us with one thread per
// star and the line search to the end, 80 us so.
__device__ __forceinline__ double log_tilted(double a, double ea, double mc, double vc, double obs,
                                             double s2) {
  const double u = a - mc, w = obs - ea;
  return -0.5 * u * u / vc - 0.5 * w * w / s2;
}

// Mode a of the tilted log-density; h0 its value, sh the scale 1 / sqrt(-h'')
// of the Gauss-Hermite rule.
__device__ __forceinline__ void tilted_mode(double mc, double vc, double obs, double s2,
                                            double* a_out, double* h0_out, double* sh_out) {
  double a;
  if (obs > 0) {
    double aL = log(obs), vL = s2 / (obs * obs);
    a = (mc / vc + aL / vL) / (1.0 / vc + 1.0 / vL);
  } else {
    a = mc;
  }
  const double ivc = 1.0 / vc, is2 = 1.0 / s2;
  double ea = exp(a);
  double h0 = log_tilted(a, ea, mc, vc, obs, s2);
  for (int it = 0; it < 100; ++it) {
    const double gr = -(a - mc) * ivc + (obs - ea) * ea * is2;
    const double H = -ivc + (obs * ea - 2.0 * ea * ea) * is2;
    double step = H < 0 ? -gr / H : gr * vc;
    step = fmax(-1.0, fmin(1.0, step));
    double en = exp(a + step);
    double hn = log_tilted(a + step, en, mc, vc, obs, s2);
    if (fabs(step) > 1e-7 * (1.0 + fabs(a))) {
      for (int k = 0; hn < h0 && k < 60; ++k) {
        step *= 0.5;
        en = exp(a + step);
        hn = log_tilted(a + step, en, mc, vc, obs, s2);
      }
    }
    a += step;
    ea = en;
    h0 = hn;
    if (fabs(step) <= 1e-14 * (1.0 + fabs(a))) break;
  }
  const double H = -ivc + (obs * ea - 2.0 * ea * ea) * is2;
  *a_out = a;
  *h0_out = h0;
  *sh_out = H < 0 ? 1.0 / sqrt(-H) : sqrt(vc);
}

// The same moments with the line search to the last step and the node sums in
// order: what FP32 contexts run (a single lane a star).  Their mean solve stops
// at cg_tol of a residual that a few stars with large site precisions dominate,
// so the last bit of a site can move a posterior mean by 1e-4: the update keeps its
// roundings there until that solve goes further.  It takes 0.39 ms however few the
// stars (the split form 0.08 at 400), 0.2 % of a sweep at 20,000.
__device__ __forceinline__ void tilted_in_order(double mc, double vc, double obs, double s2,
                                                const double* __restrict__ ghx,
                                                const double* __restrict__ ghw, double* mh,
                                                double* vh) {
  double a;
  if (obs > 0) {
    double aL = log(obs), vL = s2 / (obs * obs);
    a = (mc / vc + aL / vL) / (1.0 / vc + 1.0 / vL);
  } else {
    a = mc;
  }
  for (int it = 0; it < 100; ++it) {
    double ea = exp(a);
    double gr = -(a - mc) / vc + (obs - ea) * ea / s2;
    double H = -1.0 / vc + (obs * ea - 2.0 * ea * ea) / s2;
    double step = H < 0 ? -gr / H : gr * vc;
    step = fmax(-1.0, fmin(1.0, step));
    double h0 = log_tilted(a, ea, mc, vc, obs, s2);
    int k = 0;
    while (log_tilted(a + step, exp(a + step), mc, vc, obs, s2) < h0 && k < 60) {
      step *= 0.5;
      ++k;
    }
    a += step;
    if (fabs(step) <= 1e-14 * (1.0 + fabs(a))) break;
  }
  double ea = exp(a);
  double H = -1.0 / vc + (obs * ea - 2.0 * ea * ea) / s2;
  double sh = H < 0 ? 1.0 / sqrt(-H) : sqrt(vc);
  double h0 = log_tilted(a, ea, mc, vc, obs, s2);
  const double sc = 1.4142135623730951 * sh;
  double S0 = 0, S1 = 0, S2 = 0;
  for (int k = 0; k < kGH; ++k) {
    double y = sc * ghx[k];
    double wk = ghw[k] * exp(log_tilted(a + y, exp(a + y), mc, vc, obs, s2) - h0);
    S0 += wk;
    S1 += wk * y;
    S2 += wk * y * y;
  }
  double m1 = S1 / S0;
  *mh = a + m1;
  *vh = S2 / S0 - m1 * m1;
}

constexpr int kSiteThreads = 128;

// What an instantiation computes: the tilted moments split over the group's lanes, or
// in order (Gaussian in A), or the closed form (Gaussian in ln A).  The closed form is
// bound by its FP64 divisions, eleven a star: 1,000,000 stars 267 us a call, 315 as a
// branch of the split form, which took two of them twice and ended in a last block's
// reduction (279 before there was a split form).
enum SiteForm { kSplit, kInOrder, kClosed };

template <int G, SiteForm FORM>
__global__ void __launch_bounds__(kSiteThreads) k_site_update(
    int64_t n, SiteParams P, const double* __restrict__ mu, const double* __restrict__ var,
    const double* __restrict__ obs, const double* __restrict__ sig, double* __restrict__ tau,
    double* __restrict__ nu, const double* __restrict__ gh_x, const double* __restrict__ gh_w,
    double* __restrict__ part_delta, unsigned long long* __restrict__ max_delta,
    unsigned long long* __restrict__ skipped, unsigned* __restrict__ flags) {
  __shared__ double ghx[kGH], ghw[kGH];
  __shared__ double sh[kSiteThreads / 32];
  if (FORM != kClosed) {
    for (int k = threadIdx.x; k < kGH; k += blockDim.x) {
      ghx[k] = gh_x[k];
      ghw[k] = gh_w[k];
    }
    __syncthreads();
  }
  constexpr int kPerBlock = kSiteThreads / G;
  const int sub = threadIdx.x & (G - 1);
  double dmax = 0;
  // the loop count is the same for every thread of a block, so the shuffles
  // below always have whole warps
  for (int64_t i0 = blockIdx.x * (int64_t)kPerBlock; i0 < n; i0 += (int64_t)gridDim.x * kPerBlock) {
    const int64_t i = i0 + threadIdx.x / G;
    const bool star = i < n;
    const double t0 = star ? tau[i] : 0.0, n0 = star ? nu[i] : 0.0;
    const double S = star ? var[i] : 1.0, m = star ? mu[i] : 0.0;
    double tc = 1.0 / S - t0;
    double ncv = m / S - n0;
    bool skip = !star || !(tc > 0) || !isfinite(tc) || !isfinite(ncv);
    double mc = 0, vc = 1, ob = 0, s2 = 1, a = 0, h0 = 0, shw = 0;
    if (!skip) {
      mc = ncv / tc;
      vc = fmax(1.0 / tc, P.vc_floor);
      tc = 1.0 / vc;
      ncv = mc / vc;
      ob = obs[i];
      const double sg = sig[i];
      s2 = sg * sg;
    }
    double mh = 0, vh = 1;
    if (FORM == kClosed) {
      vh = 1.0 / (tc + 1.0 / s2);  // tc = 1 / vc, ncv = mc / vc by now
      mh = vh * (ncv + ob / s2);
    } else if (FORM == kInOrder) {
      if (!skip) tilted_in_order(mc, vc, ob, s2, ghx, ghw, &mh, &vh);
    } else {
      double S0 = 0, S1 = 0, S2 = 0;
      if (!skip) {
        tilted_mode(mc, vc, ob, s2, &a, &h0, &shw);
        // moments about the mode, then shifted
        const double sc = 1.4142135623730951 * shw;
        for (int k = sub; k < kGH; k += G) {
          const double y = sc * ghx[k];
          const double x = a + y;
          const double wk = ghw[k] * exp(log_tilted(x, exp(x), mc, vc, ob, s2) - h0);
          S0 += wk;
          S1 += wk * y;
          S2 += wk * y * y;
        }
      }
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) {
        S0 += __shfl_xor_sync(0xffffffffu, S0, off);
        S1 += __shfl_xor_sync(0xffffffffu, S1, off);
        S2 += __shfl_xor_sync(0xffffffffu, S2, off);
      }
      if (!skip) {
        const double m1 = S1 / S0;
        mh = a + m1;
        vh = S2 / S0 - m1 * m1;
      }
    }
    if (!star || sub != 0) continue;
    const double t_new = 1.0 / vh - tc, n_new = mh / vh - ncv;
    if (!(t_new >= 0) || !isfinite(n_new) || !isfinite(t_new)) skip = true;
    if (skip) {
      atomicAdd(skipped, 1ull);
      continue;
    }
    const double tn = (1.0 - P.damping) * t0 + P.damping * t_new;
    const double nn = (1.0 - P.damping) * n0 + P.damping * n_new;
    tau[i] = tn;
    nu[i] = nn;
    double dt = fabs(tn - t0) / (1.0 + fabs(t0));
    double dn = fabs(nn - n0) / (1.0 + fabs(n0));
    dmax = fmax(dmax, fmax(dt, dn));
  }
  // block max (fixed order)
  for (int off = 16; off > 0; off >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, off));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = dmax;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0;
    for (int w = 0; w < kSiteThreads / 32; ++w) v = fmax(v, sh[w]);
    if (!isfinite(v)) atomicOr(flags, kFlagNonFinite);
    // the blocks' maxima for the caller to reduce, or their maximum (non-negative
    // doubles have their bits in the same order)
    if (part_delta) part_delta[blockIdx.x] = v;
    else atomicMax(max_delta, (unsigned long long)__double_as_longlong(v));
  }
}

// Lanes per star: the largest power of two up to 32 that keeps the update
// within one warp per scheduler (four schedulers per SM; pairs of lanes up to
// 2.25 warps, where they still beat single lanes: 330 against 379 us a call at
// 20,000 stars, 615 against 551 us at 50,000).  Calls of 32 / 16 / 8 / 4 / 2 / 1
// lanes took 82 / 91 / 96 / 117 / 155 / 235 us at 400 stars, 157 / 117 / 102 /
// 117 / 157 / 242 us at 2,400 and 474 / 350 / 254 / 227 / 233 / 231 us at 10,000.
static int site_group(int64_t n, int sms) {
  int g = 32;
  const int64_t room = (int64_t)sms * 4 * 32;
  while (g > 1 && n * g > (g == 2 ? 9 * room / 4 : room)) g >>= 1;
  return g;
}

// blocks: at most max_blocks; the kernel strides over the rest of the stars
static int site_blocks(int64_t n, int group, int64_t max_blocks) {
  return (int)std::min<int64_t>(ceil_div(n * group, kSiteThreads), max_blocks);
}

// group: lanes per star of the split form (the others have one)
static void launch_site(SiteForm form, int group, int blocks, cudaStream_t st, int64_t n,
                        const SiteParams& P, const double* mu, const double* var,
                        const double* obs, const double* sig, double* tau, double* nu,
                        const double* gh_x, const double* gh_w, double* part,
                        unsigned long long* max_delta, unsigned long long* skipped,
                        unsigned* flags) {
#define GM_SITE(G, FORM)                                   \
  k_site_update<G, FORM><<<blocks, kSiteThreads, 0, st>>>( \
      n, P, mu, var, obs, sig, tau, nu, gh_x, gh_w, part, max_delta, skipped, flags)
  if (form == kClosed) GM_SITE(1, kClosed);
  else if (form == kInOrder) GM_SITE(1, kInOrder);
  else if (group == 32) GM_SITE(32, kSplit);
  else if (group == 16) GM_SITE(16, kSplit);
  else if (group == 8) GM_SITE(8, kSplit);
  else if (group == 4) GM_SITE(4, kSplit);
  else if (group == 2) GM_SITE(2, kSplit);
  else GM_SITE(1, kSplit);
#undef GM_SITE
}

gm_status site_update(gm_ctx* c, double* max_delta, int64_t* skipped) {
  const int64_t n = c->n;
  cudaStream_t st = c->stream;
  const int sms = sm_count(c);
  const SiteForm form = c->cfg.likelihood == GM_LIK_GAUSS_IN_LNA ? kClosed
                        : c->cfg.precision == GM_PREC_FP32       ? kInOrder
                                                                 : kSplit;
  const int group = form == kSplit ? site_group(n, sms) : 1;
  const int G = site_blocks(n, group, 4 * sms);
  double* part = (double*)dev_alloc(c, (G + 1) * sizeof(double) + sizeof(unsigned long long));
  if (!part) return set_error(c, GM_E_NOMEM, "site partials");
  unsigned long long* cnt = (unsigned long long*)(part + G);
  GM_CUDA_CHECK(c, cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st));
  SiteParams P{c->cfg.damping, c->cfg.vc_floor};
  GM_PROF(c, "k_site_update");
  launch_site(form, group, G, st, n, P, c->mu, c->var, c->obs, c->obs_sigma, c->tau, c->nu, c->gh_x,
              c->gh_wx, part, nullptr, cnt, c->d_flags);
  GM_LAUNCH_CHECK(c);
  double* hp = (double*)c->h_pinned;
  GM_CUDA_CHECK(c, cudaMemcpyAsync(hp, part, (G + 1) * sizeof(double), cudaMemcpyDeviceToHost, st));
  GM_CUDA_CHECK(c, cudaStreamSynchronize(st));
  double m = 0;
  for (int k = 0; k < G; ++k) m = std::fmax(m, hp[k]);
  unsigned long long sk;
  std::memcpy(&sk, hp + G, sizeof(sk));
  *max_delta = m;
  *skipped = (int64_t)sk;
  dev_free_now(c, part, (G + 1) * sizeof(double) + sizeof(unsigned long long));
  return GM_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free site update (gm_site_update_noalloc).
//
// Some callers cannot allocate device memory while they run: a host
// framework that owns every device allocation through its own pool, code
// running inside a memory-capped or pre-reserved budget, or a service loop
// that must not call cudaMalloc/cudaFree on its latency path.  For them the
// EP site update runs on caller-owned arrays, with its scratch (Gauss-Hermite
// table, skip counter, flags, maximum) in the file-scope array below.  A block
// takes 128 stars or fewer, up to kNaMaxBlocks blocks: n <= kNaMaxStars.  Every GPU that loads the library holds the array
// until the process exits.  All calls share it: concurrent calls on the GPU
// race with one another and must be serialised by the caller.
// ---------------------------------------------------------------------------
constexpr int kNaMaxBlocks = 8192;
constexpr int64_t kNaMaxStars = 128ll * kNaMaxBlocks;  // 1,048,576
constexpr int kNaSlots = 2 * kGH + 3;                  // doubles
constexpr int kNaMaxDevices = 64;

static __device__ __align__(256) double g_na_scratch[kNaSlots];

// Scratch layout (doubles): [0, kGH) nodes, [kGH, 2 kGH) weights * exp(x^2),
// then 64-bit words: the skip counter, the flags, the maximum (bits of a double).
// Per device, the scratch address at which the rule was last uploaded.  The
// address is resolved again on every call, so a module reloaded after a
// device reset (new address) gets its rule uploaded again instead of a stale
// pointer being used.
static double* g_na_ptr[kNaMaxDevices] = {nullptr};

// Device memory of the current device `dev`, or managed memory.  Memory of
// another GPU is refused: without peer access the kernel could not read it.
static bool na_device_ptr(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type == cudaMemoryTypeManaged) return true;
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

// Resolves the device address of the scratch array on the current device
// (the host-side name is only a stand-in) on every call, and uploads the
// Gauss-Hermite rule when that address has not seen it yet (first call on a
// device, or a module reloaded after a device reset).  The upload is a
// synchronous copy followed by a device synchronisation, so the rule is on
// the device before any kernel on any stream (a non-blocking one included)
// can read it; that first call therefore must not run inside a stream
// capture.  Serialised by a mutex.
static gm_status na_setup(int dev, double** out) {
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  double* p = nullptr;
  if (cudaGetSymbolAddress((void**)&p, g_na_scratch) != cudaSuccess || !p) {
    cudaGetLastError();
    return GM_E_CUDA;
  }
  if (g_na_ptr[dev] != p) {
    double rule[2 * kGH];
    gauss_hermite(kGH, rule, rule + kGH);
    if (cudaMemcpy(p, rule, sizeof(rule), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaDeviceSynchronize() != cudaSuccess) {
      cudaGetLastError();
      return GM_E_CUDA;
    }
    g_na_ptr[dev] = p;
  }
  *out = p;
  return GM_OK;
}

}  // namespace gm

extern "C" gm_status gm_site_update_noalloc(int64_t n, const double* mu, const double* var,
                                            const double* obs, const double* obs_sigma,
                                            double* tau, double* nu, int32_t likelihood,
                                            double damping, double vc_floor, void* stream,
                                            double* max_delta_out, int64_t* skipped_out) {
  using namespace gm;
  if (n < 1 || n > kNaMaxStars) return GM_E_INVAL;
  if (!mu || !var || !obs || !obs_sigma || !tau || !nu) return GM_E_INVAL;
  if (likelihood != GM_LIK_GAUSS_IN_A && likelihood != GM_LIK_GAUSS_IN_LNA) return GM_E_INVAL;
  if (!(damping > 0 && damping <= 1) || !(vc_floor >= 0)) return GM_E_INVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices) {
    cudaGetLastError();
    return GM_E_CUDA;
  }
  for (const void* p : {(const void*)mu, (const void*)var, (const void*)obs,
                        (const void*)obs_sigma, (const void*)tau, (const void*)nu})
    if (!na_device_ptr(p, dev)) return GM_E_INVAL;
  double* base = nullptr;
  gm_status st = na_setup(dev, &base);
  if (st != GM_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  double* gh_x = base;
  double* gh_w = base + kGH;
  unsigned long long* skipped = (unsigned long long*)(base + 2 * kGH);
  unsigned* flags = (unsigned*)(skipped + 1);
  // the words keep the previous call's values: clear them
  if (cudaMemsetAsync(skipped, 0, 3 * sizeof(double), s) != cudaSuccess) {
    cudaGetLastError();
    return GM_E_CUDA;
  }
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return GM_E_CUDA;
  }
  const SiteForm form = likelihood == GM_LIK_GAUSS_IN_LNA ? kClosed : kSplit;
  const int group = form == kSplit ? site_group(n, sms > 0 ? sms : 1) : 1;
  SiteParams P{damping, vc_floor};
  launch_site(form, group, site_blocks(n, group, kNaMaxBlocks), s, n, P, mu, var, obs, obs_sigma, tau,
              nu, gh_x, gh_w, nullptr, skipped + 2, skipped, flags);
  if (cudaGetLastError() != cudaSuccess) return GM_E_CUDA;
  unsigned long long h[3];
  if (cudaMemcpyAsync(h, skipped, 3 * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return GM_E_CUDA;
  }
  unsigned fl = (unsigned)(h[1] & 0xffffffffull);
  double md;
  std::memcpy(&md, &h[2], sizeof(md));
  if (max_delta_out) *max_delta_out = md;
  if (skipped_out) *skipped_out = (int64_t)h[0];
  return (fl & kFlagNonFinite) ? GM_E_NONFINITE : GM_OK;
}
