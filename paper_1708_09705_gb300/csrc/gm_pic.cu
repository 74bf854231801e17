// PITC / PIC posterior of the log-extinction at inducing points (Sect. 4.1,
// the simplified case: hyperparameters fixed and each star's observed log-
// extinction Gaussian, a~_n | a_n ~ N(a_n, sigma_n^2)).
//
// The stars are split into sub-catalogues (blocks).  Given the values u at R
// inducing points the blocks are independent (PITC), each with the exact GP
// conditional a_k | u ~ N(m_k + A_k (u - mu_u), K_kk - A_k K_uk),
// A_k = K_ku K_uu^-1, so a~_k | u ~ N(m_k + A_k (u - mu_u), C_k) with
// C_k = K_kk - A_k K_uk + diag(sigma_k^2).  The block-site EP of the paper
// reaches its fixed point in one parallel sweep here (every factor is
// Gaussian), and the posterior of u is
//   P = K_uu^-1 + sum_k A_k^T C_k^-1 A_k,  h = K_uu^-1 mu_u + sum_k A_k^T C_k^-1 y_k,
//   y_k = a~_k - m_k + A_k mu_u,   mean = P^-1 h,   cov = P^-1.
// K_kk are read from the stored covariance, K_ku and K_uu come from the same
// sightline quadrature, cutoff and taper.  The dense algebra (FP64) follows the
// per-output routines of gm_dense.cuh, with a warp per right-hand side and a thread
// block per factorisation.
#include <algorithm>
#include <cmath>
#include <vector>

#include "gm_dense.cuh"
#include "gm_internal.cuh"

namespace gm {

// Lower Cholesky factor in place of each dim[b] x dim[b] row-major matrix at
// base + off[b], mirrored into the upper triangle (column i of L is then a
// contiguous row for the solves); one thread block per matrix, right-looking.
// The chain of columns bounds it: a matrix of up to kCholShared rows stays in
// shared memory (packed lower triangle and the column in work: 229,432 bytes), a larger
// one in global memory; either way the column in work is copied to shared memory
// and the update runs along the rows, a warp per row.  One thread per row on
// global memory took 8 us a column, 1.34 ms at 140 to 170 rows; now 0.42 ms.
constexpr int kCholShared = 238;
constexpr int kCholThreads = 512;

__global__ void __launch_bounds__(kCholThreads) k_pic_chol(double* __restrict__ base,
                                                           const int64_t* __restrict__ off,
                                                           const int32_t* __restrict__ dim,
                                                           unsigned* __restrict__ flags) {
  extern __shared__ double sm[];  // the column, then the matrix if it fits
  __shared__ double d_s[2];
  double* G = base + off[blockIdx.x];
  const int n = dim[blockIdx.x];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5, W = nt >> 5;
  const bool in_sm = n <= kCholShared;
  double* v = sm;
  double* A = in_sm ? sm + n : G;
  auto row = [&](int i) { return A + (in_sm ? (int64_t)i * (i + 1) / 2 : (int64_t)i * n); };
  if (in_sm)
    for (int i = w; i < n; i += W)
      for (int k = lane; k <= i; k += 32) row(i)[k] = G[(int64_t)i * n + k];
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    if (w == 0) {
      const double d = row(j)[j];
      const double r = d > 0.0 ? sqrt(d) : -1.0;
      if (lane == 0) {
        d_s[0] = r;
        d_s[1] = 1.0 / r;
      }
    }
    __syncthreads();
    const double d = d_s[0], rd = d_s[1];
    if (!(d > 0.0)) break;  // uniform
    for (int i = j + tid; i < n; i += nt) {
      double* Ai = row(i);
      const double x = i == j ? d : Ai[j] * rd;
      Ai[j] = x;
      v[i] = x;
    }
    __syncthreads();
    for (int i = j + 1 + w; i < n; i += W) {
      const double x = v[i];
      double* Ai = row(i);
      for (int k = j + 1 + lane; k <= i; k += 32) Ai[k] = fma(-x, v[k], Ai[k]);
    }
    __syncthreads();
  }
  // a matrix that is not positive definite is written back as far as it came
  if (tid == 0 && n > 0 && !(d_s[0] > 0.0)) atomicOr(flags, kFlagNotSPD);
  for (int i = w; i < n; i += W)
    for (int k = lane; k < n; k += 32) {
      const double x = k <= i ? row(i)[k] : row(k)[i];
      if (in_sm || k > i) G[(int64_t)i * n + k] = x;
    }
}

// ------------------------------------------------- solves, a warp per vector
// x (n values in shared memory, of one warp) of L x = b / L^T x = b in place, for a
// mirrored factor M (rows of 256-byte reads in both directions).  Element i is
// final once the steps before it have run, so every lane reads it, divides by the
// diagonal, and the lanes subtract its multiples from their elements.
__device__ __forceinline__ void warp_lower(const double* __restrict__ M, int64_t ld, int n,
                                           double* x, int lane) {
  for (int i0 = 0; i0 < n; i0 += 32) {
    // the diagonal's reciprocals of 32 steps at once
    const int id = i0 + lane;
    const double rd = id < n ? 1.0 / M[(int64_t)id * ld + id] : 0.0;
    const int e = min(32, n - i0);
    // the 32 x 32 triangle in registers: lane holds element i0 + lane
    double y = id < n ? x[id] : 0.0;
#pragma unroll 8
    for (int t = 0; t < e; ++t) {
      const double m = id < n && lane > t ? M[(int64_t)(i0 + t) * ld + id] : 0.0;
      const double xt = __shfl_sync(0xffffffffu, y * rd, t);
      if (lane == t) y = xt;
      y = fma(-m, xt, y);
    }
    if (id < n) x[id] = y;
    __syncwarp();
    // the rows behind it: element k takes all 32 steps at once
    for (int k = i0 + 32 + lane; k < n; k += 32) {
      double a0 = x[k], a1 = 0;
      const double* Mk = M + (int64_t)i0 * ld + k;
#pragma unroll 8
      for (int t = 0; t < 32; t += 2) {
        a0 = fma(-Mk[(int64_t)t * ld], x[i0 + t], a0);
        a1 = fma(-Mk[(int64_t)(t + 1) * ld], x[i0 + t + 1], a1);
      }
      x[k] = a0 + a1;
    }
    __syncwarp();
  }
}

__device__ __forceinline__ void warp_lower_t(const double* __restrict__ M, int64_t ld, int n,
                                             double* x, int lane) {
  for (int i0 = ((n - 1) >> 5) << 5; i0 >= 0; i0 -= 32) {
    const int id = i0 + lane;
    const double rd = id < n ? 1.0 / M[(int64_t)id * ld + id] : 0.0;
    const int e = min(32, n - i0);
    double y = id < n ? x[id] : 0.0;
#pragma unroll 8
    for (int t = e - 1; t >= 0; --t) {
      const double m = lane < t ? M[(int64_t)(i0 + t) * ld + id] : 0.0;
      const double xt = __shfl_sync(0xffffffffu, y * rd, t);
      if (lane == t) y = xt;
      y = fma(-m, xt, y);
    }
    if (id < n) x[id] = y;
    __syncwarp();
    for (int k = lane; k < i0; k += 32) {  // k < i0: whole warps, i0 is a multiple of 32
      double a0 = x[k], a1 = 0;
      const double* Mk = M + (int64_t)i0 * ld + k;
      int t = 0;
#pragma unroll 4
      for (; t + 1 < e; t += 2) {
        a0 = fma(-Mk[(int64_t)t * ld], x[i0 + t], a0);
        a1 = fma(-Mk[(int64_t)(t + 1) * ld], x[i0 + t + 1], a1);
      }
      if (t < e) a0 = fma(-Mk[(int64_t)t * ld], x[i0 + t], a0);
      x[k] = a0 + a1;
    }
    __syncwarp();
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Vectors of one warp: `words` doubles in shared memory, or in the global scratch
// where a block's share of shared memory is too small for them (a sub-catalogue of
// thousands of stars).
__device__ __forceinline__ double* warp_vectors(double* sm, double* scratch, int64_t words) {
  const int w = threadIdx.x >> 5;
  return scratch ? scratch + ((int64_t)blockIdx.x * (blockDim.x >> 5) + w) * words : sm + w * words;
}

// Quadrature inputs of the inducing pairs (a, b), a >= b, diagonal included.
__global__ void k_pic_upairs(int R, const double* __restrict__ us, const double* __restrict__ ux,
                             const double* __restrict__ uy, const double* __restrict__ uz,
                             double* __restrict__ si, double* __restrict__ sj,
                             double* __restrict__ ch) {
  const int64_t np = (int64_t)R * (R + 1) / 2;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np;
       p += (int64_t)gridDim.x * blockDim.x) {
    gmpic::upair(p, us, ux, uy, uz, si, sj, ch);
  }
}

// K_uu (lower triangle, tapered as K) and the prior mean at the inducing
// points from the pairs' untapered values.
__global__ void k_pic_kuu(int R, double inv_cut, int taper, int form, double log_rho_bar,
                          double sigma2, const double* __restrict__ us,
                          const double* __restrict__ ch, const double* __restrict__ kp,
                          double* __restrict__ Kuu, double* __restrict__ mu_u) {
  const int64_t np = (int64_t)R * (R + 1) / 2;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np;
       p += (int64_t)gridDim.x * blockDim.x) {
    gmpic::kuu_entry(p, R, inv_cut, taper == GM_TAPER_WENDLAND ? 0 : 1,
                     form == GM_FORM_LOGNORMAL ? 0 : 1, log_rho_bar, sigma2, us, ch, kp, Kuu,
                     mu_u);
  }
}

// K_ku rows in block order from the inducing points' CSR over the stars.
__global__ void k_pic_kku(int R, const int64_t* __restrict__ qptr,
                          const int32_t* __restrict__ qcol, const double* __restrict__ qval,
                          int64_t qnnz, const int32_t* __restrict__ rowpos,
                          double* __restrict__ Kku) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < qnnz;
       e += (int64_t)gridDim.x * blockDim.x) {
    gmpic::kku_entry(e, R, qptr, qcol, qval, rowpos, Kku);
  }
}

// Rows of A = K_ku K_uu^-1, a warp each.
__global__ void __launch_bounds__(128) k_pic_arow(int64_t n, int R, const double* __restrict__ Lu,
                                                  const double* __restrict__ Kku,
                                                  double* __restrict__ A, double* scratch) {
  extern __shared__ double sm[];
  double* x = warp_vectors(sm, scratch, R);
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  for (int64_t j = blockIdx.x * (int64_t)W + (threadIdx.x >> 5); j < n; j += (int64_t)gridDim.x * W) {
    for (int r = lane; r < R; r += 32) x[r] = Kku[j * R + r];
    __syncwarp();
    warp_lower(Lu, R, R, x, lane);
    warp_lower_t(Lu, R, R, x, lane);
    for (int r = lane; r < R; r += 32) A[j * R + r] = x[r];
    __syncwarp();
  }
}

// Lower triangle of every block's C_k = K_kk - A_k K_uk + diag(sigma^2).
__global__ void k_pic_cmat(int nb, const int64_t* __restrict__ coff,
                           const int64_t* __restrict__ boff, int R,
                           const int64_t* __restrict__ bidx, const int64_t* __restrict__ row_ptr,
                           const int32_t* __restrict__ col, const double* __restrict__ val,
                           const double* __restrict__ A, const double* __restrict__ Kku,
                           const double* __restrict__ sig, double* __restrict__ C) {
  const int64_t total = coff[nb];
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    gmpic::cmat_entry(e, nb, coff, boff, R, bidx, row_ptr, col, val, A, Kku, sig, C);
  }
}

__global__ void k_pic_y(int64_t n, int R, const int64_t* __restrict__ bidx,
                        const double* __restrict__ obs, const double* __restrict__ prior_m,
                        const double* __restrict__ A, const double* __restrict__ mu_u,
                        double* __restrict__ yv) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
       j += (int64_t)gridDim.x * blockDim.x)
    yv[j] = gmdense::y_entry(obs[bidx[j]], prior_m[bidx[j]], A + j * R, mu_u, R);
}

// X_k = L_k^-1 A_k (columns c < R) and yv_k = L_k^-1 y_k (c = R), a warp per column.
__global__ void __launch_bounds__(128) k_pic_fsolve(int nb, int R, int maxN,
                                                    const int64_t* __restrict__ coff,
                                                    const int64_t* __restrict__ boff,
                                                    const double* __restrict__ C,
                                                    double* __restrict__ X, double* __restrict__ yv,
                                                    double* scratch) {
  extern __shared__ double sm[];
  double* x = warp_vectors(sm, scratch, maxN);
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  const int64_t total = (int64_t)nb * (R + 1);
  for (int64_t t = blockIdx.x * (int64_t)W + (threadIdx.x >> 5); t < total;
       t += (int64_t)gridDim.x * W) {
    const int k = (int)(t / (R + 1)), c = (int)(t - (int64_t)k * (R + 1));
    const int N = (int)(boff[k + 1] - boff[k]);
    double* p = c < R ? X + boff[k] * R + c : yv + boff[k];
    const int64_t inc = c < R ? R : 1;
    for (int a = lane; a < N; a += 32) x[a] = p[a * inc];
    __syncwarp();
    warp_lower(C + coff[k], N, N, x, lane);
    for (int a = lane; a < N; a += 32) p[a * inc] = x[a];
    __syncwarp();
  }
}

// Lambda (lower triangle, b <= a) and eta, partial sums over a share of the stars:
// 32 x 32 outputs per block, stars in groups of 32 through shared memory.  The
// right-hand side is column R of [X | yv].  part: split x (R^2 + R).
__global__ void __launch_bounds__(256) k_pic_lambda(int64_t n, int R, int64_t share,
                                                    const double* __restrict__ X,
                                                    const double* __restrict__ yv,
                                                    double* __restrict__ part) {
  __shared__ double sa[32][33], sb[32][33];
  int ta, tb;
  gmpic::tri_index(blockIdx.x, &ta, &tb);  // tiles of rows (of R + 1) and columns
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t j0 = blockIdx.y * share, j1 = min(n, j0 + share);
  double acc[4] = {0, 0, 0, 0};
  auto at = [&](int64_t j, int r) {
    return j < j1 && r <= R ? (r < R ? X[j * R + r] : yv[j]) : 0.0;
  };
  for (int64_t j = j0; j < j1; j += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sa[w + 8 * q][lane] = at(j + w + 8 * q, 32 * ta + lane);
      sb[w + 8 * q][lane] = at(j + w + 8 * q, 32 * tb + lane);
    }
    __syncthreads();
#pragma unroll 8
    for (int t = 0; t < 32; ++t) {
      const double b = sb[t][lane];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fma(sa[t][w + 8 * q], b, acc[q]);
    }
    __syncthreads();
  }
  double* o = part + blockIdx.y * ((int64_t)R * R + R);
  const int b = 32 * tb + lane;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int a = 32 * ta + w + 8 * q;
    if (b >= R) continue;
    if (a < R && b <= a) o[(int64_t)a * R + b] = acc[q];
    if (a == R) o[(int64_t)R * R + b] = acc[q];
  }
}

__global__ void k_pic_lambda_sum(int R, int splits, const double* __restrict__ part,
                                 double* __restrict__ Lam, double* __restrict__ eta) {
  const int64_t RR = (int64_t)R * R, total = RR + R;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (e < RR && e % R > e / R) continue;
    double v = 0.0;
    for (int k = 0; k < splits; ++k) v += part[k * total + e];
    if (e < RR) Lam[e] = v;
    else eta[e - RR] = v;
  }
}

// Columns of (L L^T)^-1, a warp each (it is symmetric: written as rows).
__global__ void __launch_bounds__(128) k_pic_inverse(int R, const double* __restrict__ L,
                                                     double* __restrict__ out, double* scratch) {
  extern __shared__ double sm[];
  double* x = warp_vectors(sm, scratch, R);
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  for (int c = blockIdx.x * W + (threadIdx.x >> 5); c < R; c += gridDim.x * W) {
    for (int r = lane; r < R; r += 32) x[r] = r == c ? 1.0 : 0.0;
    __syncwarp();
    warp_lower(L, R, R, x, lane);
    warp_lower_t(L, R, R, x, lane);
    for (int r = lane; r < R; r += 32) out[(int64_t)r * R + c] = x[r];
    __syncwarp();
  }
}

// P = K_uu^-1 + Lambda (lower triangle) and h = K_uu^-1 mu_u + eta.
__global__ void k_pic_prec(int R, const double* __restrict__ Kinv, const double* __restrict__ Lam,
                           const double* __restrict__ mu_u, const double* __restrict__ eta,
                           double* __restrict__ P, double* __restrict__ h) {
  const int64_t total = (int64_t)R * R + R;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    gmpic::prec_task(e, R, Kinv, Lam, mu_u, eta, P, h);
  }
}

// mean = P^-1 h from the factor of P (one warp).
__global__ void __launch_bounds__(32) k_pic_mean(int R, const double* __restrict__ LP,
                                                 const double* __restrict__ h,
                                                 double* __restrict__ mean, double* scratch) {
  extern __shared__ double sm[];
  double* x = scratch ? scratch : sm;
  const int lane = threadIdx.x;
  for (int r = lane; r < R; r += 32) x[r] = h[r];
  __syncwarp();
  warp_lower(LP, R, R, x, lane);
  warp_lower_t(LP, R, R, x, lane);
  for (int r = lane; r < R; r += 32) mean[r] = x[r];
}

// Warps per block and blocks of a kernel with a warp per item and `words` doubles
// per warp: shared memory while two warps fit half of an SM's, else
// scratch (allocated for the grid).
struct WarpPlan {
  int warps, blocks;
  size_t smem;
  int64_t scratch;  // doubles
};
static WarpPlan warp_plan(gm_ctx* c, int64_t items, int64_t words) {
  WarpPlan p;
  const int64_t room = 96 * 1024 / 8;
  p.scratch = 0;
  if (words * 2 <= room) {
    p.warps = (int)std::min<int64_t>(4, room / words);
    p.smem = (size_t)p.warps * words * sizeof(double);
  } else {
    p.warps = 4;
    p.smem = 0;
  }
  // few items: a block per SM first
  p.warps = (int)std::max<int64_t>(1, std::min<int64_t>(p.warps, ceil_div(items, sm_count(c))));
  if (p.smem) p.smem = (size_t)p.warps * words * sizeof(double);
  p.blocks = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(items, p.warps), 8 * sm_count(c)));
  if (!p.smem) {
    p.blocks = std::min(p.blocks, 2 * sm_count(c));
    p.scratch = (int64_t)p.blocks * p.warps * words;
  }
  return p;
}

static int grid_for(gm_ctx* c, int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 128), 16 * sm_count(c)));
}

// Factors of the last PIC posterior, kept for prediction.
struct PicState {
  int R = 0, nb = 0;
  int64_t n = 0;
  Buffer i64;  // boff (nb + 1), coff (nb + 1), bidx (n)
  Buffer i32;  // dims (nb), block of each star (n)
  Buffer d;    // Lu (R^2), mean (R), cov (R^2), mu_u (R), us, ux, uy, uz (R),
               // A, Kku (n R), C factors (sum N_k^2)
  std::vector<int64_t> h_boff, h_coff;
  int64_t *boff = nullptr, *coff = nullptr, *bidx = nullptr;
  int32_t *dims = nullptr, *blk = nullptr;
  double *Lu = nullptr, *mean = nullptr, *cov = nullptr, *mu_u = nullptr, *us = nullptr,
         *ux = nullptr, *uy = nullptr, *uz = nullptr, *A = nullptr, *Kku = nullptr, *C = nullptr;
  int max_block = 0;
  bool ready = false;  // set once the posterior is complete
};

void pic_free(gm_ctx* c) {
  if (!c->pic) return;
  PicState* P = c->pic;
  for (Buffer* b : {&P->i64, &P->i32, &P->d})
    if (b->p) dev_free_now(c, b->p, b->bytes);
  delete P;
  c->pic = nullptr;
}

bool pic_ready(gm_ctx* c) { return c->pic && c->pic->ready; }
const double* pic_mean(gm_ctx* c) { return c->pic ? c->pic->mean : nullptr; }
const double* pic_cov(gm_ctx* c) { return c->pic ? c->pic->cov : nullptr; }
int pic_blocks(gm_ctx* c) { return c->pic ? c->pic->nb : 0; }
const int32_t* pic_star_blocks(gm_ctx* c) { return c->pic ? c->pic->blk : nullptr; }
int pic_inducing(gm_ctx* c) { return c->pic ? c->pic->R : 0; }

gm_status pic_posterior(gm_ctx* c, int R, const double* us, const double* ux, const double* uy,
                        const double* uz, const int32_t* h_block_int, int nb) {
  const int64_t n = c->n;
  pic_free(c);
  PicState* S = new (std::nothrow) PicState();
  if (!S) return set_error(c, GM_E_NOMEM, "PIC state");
  c->pic = S;
  S->R = R;
  S->nb = nb;
  S->n = n;
  // ---- block lists (host): stars of block k in internal order
  S->h_boff.resize(nb + 1);
  S->h_coff.resize(nb + 1);
  std::vector<int64_t> bidx(n);
  std::vector<int32_t> rowpos(n), dims(nb);
  if (!gmpic::block_lists(n, h_block_int, nb, kMaxPicBlock, S->h_boff.data(), S->h_coff.data(),
                          bidx.data(), rowpos.data(), dims.data())) {
    pic_free(c);
    return set_error(c, GM_E_INVAL, "a sub-catalogue has more than 8192 stars");
  }
  for (int k = 0; k < nb; ++k) S->max_block = std::max(S->max_block, (int)dims[k]);
  const int64_t RR = (int64_t)R * R;
  const int64_t npair = (int64_t)R * (R + 1) / 2;
  const int64_t ncf = S->h_coff[nb];
  if (!ensure(c, S->i64, (size_t)(2 * (nb + 1) + n) * sizeof(int64_t)) ||
      !ensure(c, S->i32, (size_t)(std::max(nb, 1) + n) * sizeof(int32_t)) ||
      !ensure(c, S->d, (size_t)(2 * RR + 7 * R + 2 * n * (int64_t)R + ncf) * sizeof(double))) {
    pic_free(c);
    return set_error(c, GM_E_NOMEM, "PIC state");
  }
  S->boff = (int64_t*)S->i64.p;
  S->coff = S->boff + nb + 1;
  S->bidx = S->coff + nb + 1;
  S->dims = (int32_t*)S->i32.p;
  S->blk = S->dims + std::max(nb, 1);
  S->Lu = (double*)S->d.p;
  S->mean = S->Lu + RR;
  S->cov = S->mean + R;
  S->mu_u = S->cov + RR;
  S->us = S->mu_u + R;
  S->ux = S->us + R;
  S->uy = S->ux + R;
  S->uz = S->uy + R;
  S->A = S->uz + R;
  S->Kku = S->A + n * (int64_t)R;
  S->C = S->Kku + n * (int64_t)R;
  // scratch of this call: Kuu, Kinv, Lam, P (R x R); eta, h (R); pair inputs
  // (4 npair); X (n x R); yv (n); partial sums of Lambda and eta; vectors of the
  // solves where they do not fit shared memory; rowpos (n)
  const WarpPlan rows = warp_plan(c, n, R), cols = warp_plan(c, R, R), one = warp_plan(c, 1, R),
                 fwd = warp_plan(c, (int64_t)nb * (R + 1), std::max(S->max_block, 1));
  const int64_t lt = ceil_div((int64_t)R + 1, 32), lam_tiles = lt * (lt + 1) / 2;
  // shares of at least 256 stars, two blocks per SM
  const int64_t splits = std::max<int64_t>(
      1, std::min<int64_t>(ceil_div(n, 256), 2 * sm_count(c) / lam_tiles));
  const int64_t share = ceil_div(ceil_div(n, splits), 32) * 32;
  const int64_t solve_words =
      std::max(std::max(rows.scratch, cols.scratch), std::max(one.scratch, fwd.scratch));
  ScopedDev b_d(c, (size_t)(4 * RR + 2 * R + 4 * npair + n * (int64_t)R + n + splits * (RR + R) +
                            solve_words) *
                       sizeof(double));
  ScopedDev b_r(c, (size_t)n * sizeof(int32_t));
  ScopedDev b_q(c, (size_t)(R + 1) * sizeof(int64_t));
  ScopedDev b_one(c, sizeof(int64_t) + sizeof(int32_t));
  if (!b_d.p || !b_r.p || !b_q.p || !b_one.p) return set_error(c, GM_E_NOMEM, "PIC arrays");
  double* Kuu = (double*)b_d.p;
  double *Kinv = Kuu + RR, *Lam = Kinv + RR, *P = Lam + RR, *eta = P + RR, *h = eta + R;
  double *psi = h + R, *psj = psi + npair, *pch = psj + npair, *pk = pch + npair;
  double *X = pk + npair, *yv = X + n * (int64_t)R;
  double *lam_part = yv + n, *vecs = lam_part + splits * (RR + R);
  auto sc = [&](const WarpPlan& p) { return p.scratch ? vecs : nullptr; };
  int32_t* d_rowpos = (int32_t*)b_r.p;
  double *Lu = S->Lu, *A = S->A, *Kku = S->Kku, *C = S->C, *mu_u = S->mu_u;
  cudaStream_t st = c->stream;
  GM_CUDA_CHECK(c, cudaMemcpyAsync(S->boff, S->h_boff.data(), (nb + 1) * sizeof(int64_t),
                                   cudaMemcpyHostToDevice, st));
  GM_CUDA_CHECK(c, cudaMemcpyAsync(S->coff, S->h_coff.data(), (nb + 1) * sizeof(int64_t),
                                   cudaMemcpyHostToDevice, st));
  GM_CUDA_CHECK(c, cudaMemcpyAsync(S->bidx, bidx.data(), n * sizeof(int64_t),
                                   cudaMemcpyHostToDevice, st));
  GM_CUDA_CHECK(c, cudaMemcpyAsync(d_rowpos, rowpos.data(), n * sizeof(int32_t),
                                   cudaMemcpyHostToDevice, st));
  GM_CUDA_CHECK(c, cudaMemcpyAsync(S->dims, dims.data(), nb * sizeof(int32_t),
                                   cudaMemcpyHostToDevice, st));
  GM_CUDA_CHECK(c, cudaMemcpyAsync(S->blk, h_block_int, n * sizeof(int32_t),
                                   cudaMemcpyHostToDevice, st));
  for (const double* src : {us, ux, uy, uz}) {
    double* dst = src == us ? S->us : src == ux ? S->ux : src == uy ? S->uy : S->uz;
    GM_CUDA_CHECK(c, cudaMemcpyAsync(dst, src, R * sizeof(double), cudaMemcpyDeviceToDevice, st));
  }
  GM_CUDA_CHECK(c, cudaMemsetAsync(Kku, 0, n * (int64_t)R * sizeof(double), st));
  // ---- K_ku: the inducing points' neighbour CSR over the stars
  int64_t* qptr = (int64_t*)b_q.p;
  Buffer qcol;
  int64_t qnnz = 0;
  gm_status s = neighbour_csr(c, R, us, ux, uy, uz, nullptr, false, qptr, qcol, &qnnz, nullptr);
  if (s != GM_OK) return s;
  ScopedDev b_qc(c, qcol.p, qcol.bytes, ScopedDev::Adopt{});  // released on every return
  ScopedDev b_qv(c, (size_t)std::max<int64_t>(qnnz, 1) * sizeof(double));
  if (!b_qv.p) return set_error(c, GM_E_NOMEM, "PIC cross-covariances");
  s = pair_quadrature(c, R, us, ux, uy, uz, nullptr, qptr, (const int32_t*)qcol.p, qnnz, b_qv.p,
                      false);
  if (s != GM_OK) return s;
  if (qnnz > 0) {
    GM_PROF(c, "k_pic_kku");
    k_pic_kku<<<grid_for(c, qnnz), 128, 0, st>>>(R, qptr, (const int32_t*)qcol.p,
                                                 (const double*)b_qv.p, qnnz, d_rowpos, Kku);
    GM_LAUNCH_CHECK(c);
  }
  // ---- K_uu and the prior mean at the inducing points
  GM_PROF(c, "k_pic_upairs");
  k_pic_upairs<<<grid_for(c, npair), 128, 0, st>>>(R, us, ux, uy, uz, psi, psj, pch);
  GM_LAUNCH_CHECK(c);
  s = pairlist_quadrature(c, npair, psi, psj, pch, pk);
  if (s != GM_OK) return s;
  GM_PROF(c, "k_pic_kuu");
  k_pic_kuu<<<grid_for(c, npair), 128, 0, st>>>(R, 1.0 / c->cfg.cutoff_pc, c->cfg.taper,
                                                c->cfg.form, std::log(c->cfg.rho_bar),
                                                c->cfg.sigma2, us, pch, pk, Kuu, mu_u);
  GM_LAUNCH_CHECK(c);
  // ---- factor K_uu; A = K_ku K_uu^-1
  GM_CUDA_CHECK(c, cudaMemcpyAsync(Lu, Kuu, RR * sizeof(double), cudaMemcpyDeviceToDevice, st));
  {
    const int64_t zero = 0;
    const int32_t dimR = R;
    GM_CUDA_CHECK(c, cudaMemcpyAsync(b_one.p, &zero, sizeof(zero), cudaMemcpyHostToDevice, st));
    GM_CUDA_CHECK(c, cudaMemcpyAsync((char*)b_one.p + sizeof(int64_t), &dimR, sizeof(dimR),
                                     cudaMemcpyHostToDevice, st));
    GM_CUDA_CHECK(c, cudaStreamSynchronize(st));  // the host values above are stack locals
  }
  const int64_t* one_off = (const int64_t*)b_one.p;
  const int32_t* one_dim = (const int32_t*)((char*)b_one.p + sizeof(int64_t));
  // shared memory of a factorisation of up to d rows, and of the solves
  auto chol_smem = [](int64_t d) {
    return (size_t)(d <= kCholShared ? d + d * (d + 1) / 2 : d) * sizeof(double);
  };
  const size_t csm = std::max(chol_smem(std::min(std::max(R, S->max_block), kCholShared)),
                              chol_smem(std::max(R, S->max_block)));
  GM_CUDA_CHECK(c, cudaFuncSetAttribute(k_pic_chol, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)csm));
  auto room = [&](const void* kern, const WarpPlan& p) {
    return p.smem <= 48 * 1024
               ? cudaSuccess
               : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
  };
  GM_CUDA_CHECK(c, room((const void*)k_pic_arow, rows));
  GM_CUDA_CHECK(c, room((const void*)k_pic_fsolve, fwd));
  GM_CUDA_CHECK(c, room((const void*)k_pic_inverse, cols));
  GM_CUDA_CHECK(c, room((const void*)k_pic_mean, one));
  GM_PROF(c, "k_pic_chol");
  k_pic_chol<<<1, kCholThreads, csm, st>>>(Lu, one_off, one_dim, c->d_flags);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_arow");
  k_pic_arow<<<rows.blocks, 32 * rows.warps, rows.smem, st>>>(n, R, Lu, Kku, A, sc(rows));
  GM_LAUNCH_CHECK(c);
  // ---- blocks: C_k, its factor, X_k and yv_k
  if (ncf > 0) {
    GM_PROF(c, "k_pic_cmat");
    k_pic_cmat<<<grid_for(c, ncf), 128, 0, st>>>(nb, S->coff, S->boff, R, S->bidx, c->row_ptr,
                                                 c->col, (const double*)c->val, A, Kku,
                                                 c->obs_sigma, C);
    GM_LAUNCH_CHECK(c);
    GM_PROF(c, "k_pic_chol");
    k_pic_chol<<<nb, kCholThreads, csm, st>>>(C, S->coff, S->dims, c->d_flags);
    GM_LAUNCH_CHECK(c);
  }
  GM_PROF(c, "k_pic_y");
  k_pic_y<<<grid_for(c, n), 128, 0, st>>>(n, R, S->bidx, c->obs, c->prior_m, A, mu_u, yv);
  GM_LAUNCH_CHECK(c);
  GM_CUDA_CHECK(c, cudaMemcpyAsync(X, A, n * (int64_t)R * sizeof(double),
                                   cudaMemcpyDeviceToDevice, st));
  GM_PROF(c, "k_pic_fsolve");
  k_pic_fsolve<<<fwd.blocks, 32 * fwd.warps, fwd.smem, st>>>(nb, R, std::max(S->max_block, 1),
                                                              S->coff, S->boff, C, X, yv, sc(fwd));
  GM_LAUNCH_CHECK(c);
  // ---- posterior of u
  GM_PROF(c, "k_pic_lambda");
  k_pic_lambda<<<dim3((unsigned)lam_tiles, (unsigned)splits), 256, 0, st>>>(n, R, share, X, yv,
                                                                            lam_part);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_lambda_sum");
  k_pic_lambda_sum<<<grid_for(c, RR + R), 128, 0, st>>>(R, (int)splits, lam_part, Lam, eta);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_inverse");
  k_pic_inverse<<<cols.blocks, 32 * cols.warps, cols.smem, st>>>(R, Lu, Kinv, sc(cols));
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_prec");
  k_pic_prec<<<grid_for(c, RR + R), 128, 0, st>>>(R, Kinv, Lam, mu_u, eta, P, h);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_chol");
  k_pic_chol<<<1, kCholThreads, csm, st>>>(P, one_off, one_dim, c->d_flags);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_mean");
  k_pic_mean<<<1, 32, one.smem, st>>>(R, P, h, S->mean, sc(one));
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_pic_inverse");
  k_pic_inverse<<<cols.blocks, 32 * cols.warps, cols.smem, st>>>(R, P, S->cov, sc(cols));
  GM_LAUNCH_CHECK(c);
  GM_CUDA_CHECK(c, cudaStreamSynchronize(st));
  S->ready = true;
  return GM_OK;
}

// ---------------------------------------------------------------- prediction
// Quadrature inputs of the query-inducing pairs p = q R + r within the cutoff: the
// others' tapered covariance is zero, so they need none.  Compact (any order), with
// p in idx and their number in count; K_su of all pairs is zeroed.
__global__ void k_pic_qpairs(int64_t np, int R, double inv_cut, int taper,
                             const double* __restrict__ qs, const double* __restrict__ qx,
                             const double* __restrict__ qy, const double* __restrict__ qz,
                             const double* __restrict__ us, const double* __restrict__ ux,
                             const double* __restrict__ uy, const double* __restrict__ uz,
                             double* __restrict__ si, double* __restrict__ sj,
                             double* __restrict__ ch, int32_t* __restrict__ idx,
                             unsigned long long* __restrict__ count, double* __restrict__ ksu) {
  const int lane = threadIdx.x & 31;
  for (int64_t p0 = blockIdx.x * (int64_t)blockDim.x; p0 < np; p0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = p0 + threadIdx.x;
    double a = 0, b = 0, h = 0;
    bool in = false;
    if (p < np) {
      gmpic::qpair(p, R, qs, qx, qy, qz, us, ux, uy, uz, &a, &b, &h);
      in = gmpic::taper_weight(gmpic::pair_distance(a, b, h), inv_cut, taper) != 0.0;
      ksu[p] = 0.0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, in);
    unsigned long long o = 0;
    if (lane == 0 && m) o = atomicAdd(count, (unsigned long long)__popc(m));
    o = __shfl_sync(0xffffffffu, o, 0) + __popc(m & ((1u << lane) - 1u));
    if (in) {
      si[o] = a;
      sj[o] = b;
      ch[o] = h;
      idx[o] = (int32_t)p;
    }
  }
}

// Tapered K_su of the compact pairs.
__global__ void k_pic_ksu(int64_t m, double inv_cut, int taper, const double* __restrict__ si,
                          const double* __restrict__ sj, const double* __restrict__ ch,
                          const int32_t* __restrict__ idx, const double* __restrict__ kp,
                          double* __restrict__ ksu) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m;
       k += (int64_t)gridDim.x * blockDim.x)
    ksu[idx[k]] =
        gmpic::taper_weight(gmpic::pair_distance(si[k], sj[k], ch[k]), inv_cut, taper) * kp[k];
}

// The predictive (gmpic::pic_point) of the queries [q0, q0 + nc), a warp per query,
// its vectors in shared memory.  FP64 bounds it: 4,400 warp instructions per query at
// 140 inducing points and 170 stars (the products with K_ku and A, four triangular
// solves, the quadratic form), 16 clocks of an SM each, 1.0 ms for 4,000 queries; the
// matrices come from L2.  One thread per query on global scratch took 11.0 ms, now 1.33.
__global__ void __launch_bounds__(128) k_pic_point(
    int64_t q0, int64_t nc, int R, int maxN, const int32_t* __restrict__ qblk,
    const int64_t* __restrict__ boff, const int64_t* __restrict__ coff,
    const int64_t* __restrict__ bidx, const double* __restrict__ Lu, const double* __restrict__ Cf,
    const double* __restrict__ A, const double* __restrict__ Kku, const double* __restrict__ mu_u,
    const double* __restrict__ pmean, const double* __restrict__ pcov,
    const double* __restrict__ obs, const double* __restrict__ prior_m,
    const double* __restrict__ ksu, const double* __restrict__ kss, const double* __restrict__ ms,
    const int64_t* __restrict__ qptr, const int32_t* __restrict__ qcol,
    const double* __restrict__ qval, double* scratch, double* __restrict__ mean,
    double* __restrict__ var) {
  extern __shared__ double sm[];
  double* As = warp_vectors(sm, scratch, 2 * ((int64_t)R + maxN));
  double *Lc = As + R, *D = Lc + R, *g = D + maxN;
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  for (int64_t t = blockIdx.x * (int64_t)W + (threadIdx.x >> 5); t < nc; t += (int64_t)gridDim.x * W) {
    const int64_t q = q0 + t;
    const int k = qblk[q];
    const int64_t b0 = boff[k];
    const int N = (int)(boff[k + 1] - b0);
    const double* ks = ksu + t * R;
    for (int r = lane; r < R; r += 32) As[r] = ks[r];
    __syncwarp();
    warp_lower(Lu, R, R, As, lane);
    warp_lower_t(Lu, R, R, As, lane);
    // D = k_sk - K_ku A_s: 16 rows at once, lanes along them, then a reduction that
    // leaves row a of the group on lane a (and a + 16)
    for (int a0 = 0; a0 < N; a0 += 16) {
      double acc[16];
#pragma unroll
      for (int a = 0; a < 16; ++a) acc[a] = 0.0;
      const int na = min(16, N - a0);
      const double* K0 = Kku + (b0 + a0) * R;
      for (int r = lane; r < R; r += 32) {
        const double x = As[r];
        if (na == 16) {
#pragma unroll
          for (int a = 0; a < 16; ++a) acc[a] = fma(-K0[(int64_t)a * R + r], x, acc[a]);
        } else {
#pragma unroll
          for (int a = 0; a < 16; ++a)
            if (a < na) acc[a] = fma(-K0[(int64_t)a * R + r], x, acc[a]);
        }
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int a = 0; a < o; ++a) {
          const double send = up ? acc[a] : acc[a + o], keep = up ? acc[a + o] : acc[a];
          acc[a] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      double d = acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 16);
      if (lane < na) {
        d += gmpic::row_entry(qcol, qval, qptr[q], qptr[q + 1], bidx[b0 + a0 + lane]);
        D[a0 + lane] = d;
        g[a0 + lane] = d;
      }
    }
    __syncwarp();
    if (N > 0) {
      warp_lower(Cf + coff[k], N, N, g, lane);
      warp_lower_t(Cf + coff[k], N, N, g, lane);
    }
    double m = 0.0, v = 0.0;
    for (int r = lane; r < R; r += 32) {
      double l0 = As[r], l1 = 0.0;
      v = fma(-l0, ks[r], v);
      const double* Ar = A + b0 * R + r;
      int a = 0;
#pragma unroll 4
      for (; a + 1 < N; a += 2) {
        l0 = fma(-g[a], Ar[(int64_t)a * R], l0);
        l1 = fma(-g[a + 1], Ar[(int64_t)(a + 1) * R], l1);
      }
      if (a < N) l0 = fma(-g[a], Ar[(int64_t)a * R], l0);
      l0 += l1;
      Lc[r] = l0;
      m = fma(l0, pmean[r] - mu_u[r], m);
    }
    __syncwarp();
    for (int a = lane; a < N; a += 32) {
      const int64_t j = bidx[b0 + a];
      m = fma(g[a], obs[j] - prior_m[j], m);
      v = fma(-g[a], D[a], v);
    }
    for (int r = lane; r < R; r += 32) {
      double t0 = 0.0, t1 = 0.0;
      const double* Pr = pcov + r;  // symmetric: column r
      int c = 0;
#pragma unroll 4
      for (; c + 1 < R; c += 2) {
        t0 = fma(Pr[(int64_t)c * R], Lc[c], t0);
        t1 = fma(Pr[(int64_t)(c + 1) * R], Lc[c + 1], t1);
      }
      if (c < R) t0 = fma(Pr[(int64_t)c * R], Lc[c], t0);
      v = fma(Lc[r], t0 + t1, v);
    }
    m = warp_sum(m);
    v = warp_sum(v);
    if (lane == 0) {
      mean[q] = ms[q] + m;
      var[q] = kss[q] + v;
    }
    __syncwarp();
  }
}

gm_status pic_predict(gm_ctx* c, int64_t nq, const double* qs, const double* qx,
                      const double* qy, const double* qz, const int32_t* qblk, const double* kss,
                      const double* ms, const int64_t* qptr, const int32_t* qcol,
                      const double* qval, double* mean, double* var) {
  PicState* S = c->pic;
  const int R = S->R;
  const int maxN = std::max(S->max_block, 1);
  // queries per chunk: K_su and its pairs (6 R doubles each: K_su, distances, chord,
  // value, index) within about 1 GB
  const int64_t per = 6 * (int64_t)R;
  const int64_t chunk = std::max<int64_t>(1, std::min<int64_t>(nq, (int64_t)(1 << 27) / per));
  const int64_t words = 2 * ((int64_t)R + maxN);
  const WarpPlan plan = warp_plan(c, chunk, words);
  ScopedDev buf(c, (size_t)(chunk * per + 1 + plan.scratch) * sizeof(double));
  if (!buf.p) return set_error(c, GM_E_NOMEM, "PIC prediction scratch");
  double* si = (double*)buf.p;
  double *sj = si + chunk * R, *ch = sj + chunk * R, *kc = ch + chunk * R, *kp = kc + chunk * R;
  int32_t* idx = (int32_t*)(kp + chunk * R);
  unsigned long long* count = (unsigned long long*)((double*)buf.p + chunk * per);
  double* w = plan.scratch ? (double*)(count + 1) : nullptr;
  cudaStream_t st = c->stream;
  const double inv_cut = 1.0 / c->cfg.cutoff_pc;
  const int taper = c->cfg.taper == GM_TAPER_WENDLAND ? 0 : 1;
  for (int64_t q0 = 0; q0 < nq; q0 += chunk) {
    const int64_t nc = std::min(chunk, nq - q0);
    const int64_t np = nc * R;
    GM_CUDA_CHECK(c, cudaMemsetAsync(count, 0, sizeof(*count), st));
    GM_PROF(c, "k_pic_qpairs");
    k_pic_qpairs<<<grid_for(c, np), 128, 0, st>>>(np, R, inv_cut, taper, qs + q0, qx + q0, qy + q0,
                                                  qz + q0, S->us, S->ux, S->uy, S->uz, si, sj, ch,
                                                  idx, count, kp);
    GM_LAUNCH_CHECK(c);
    unsigned long long* hm = (unsigned long long*)c->h_pinned;
    GM_CUDA_CHECK(c, cudaMemcpyAsync(hm, count, sizeof(*hm), cudaMemcpyDeviceToHost, st));
    GM_CUDA_CHECK(c, cudaStreamSynchronize(st));
    const int64_t m = (int64_t)*hm;
    gm_status s = pairlist_quadrature(c, m, si, sj, ch, kc);
    if (s != GM_OK) return s;
    if (m > 0) {
      GM_PROF(c, "k_pic_ksu");
      k_pic_ksu<<<grid_for(c, m), 128, 0, st>>>(m, inv_cut, taper, si, sj, ch, idx, kc, kp);
      GM_LAUNCH_CHECK(c);
    }
    if (plan.smem > 48 * 1024)
      GM_CUDA_CHECK(c, cudaFuncSetAttribute(k_pic_point, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)plan.smem));
    GM_PROF(c, "k_pic_point");
    k_pic_point<<<plan.blocks, 32 * plan.warps, plan.smem, st>>>(
        q0, nc, R, maxN, qblk, S->boff, S->coff, S->bidx, S->Lu, S->C, S->A, S->Kku, S->mu_u,
        S->mean, S->cov, c->obs, c->prior_m, kp, kss, ms, qptr, qcol, qval, w, mean, var);
    GM_LAUNCH_CHECK(c);
  }
  GM_CUDA_CHECK(c, cudaStreamSynchronize(st));
  return GM_OK;
}

}  // namespace gm
