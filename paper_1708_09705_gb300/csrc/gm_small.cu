// Conjugate gradients of small FP64 problems, one thread block per right-hand side.
//
// Columns of a variance panel do not depend on one another, and up to 2,048 stars
// a column's vectors fit one block (rows in registers, D o P in shared memory).  So
// a block runs its column's whole solve: no launch, reduction kernel or host check
// per iteration, and it stops when its own column has converged.  On a 400-star
// field an iteration of the panel took six launches of 5 to 40 us, latency most of
// them.  Here the FP64 unit bounds it: a warp instruction takes 16 clocks of an SM,
// and a column's iteration has one per 32 stored entries, nine per 32 rows and
// three reductions, 17 us for the three columns that an SM then holds.  Four EP
// solves of 400 stars (15,398 entries, 584 iterations): 17.3 ms in panels, 8.6 ms
// here.
//
// K is read from a sliced ELL copy: slices of 32 rows of similar length, each padded
// to its longest; lanes own rows, so entry e of a slice is one 256-byte access.
// Padding entries point at their own row with value zero.
#include <algorithm>
#include <cstdlib>
#include <string>

#include "gm_internal.cuh"

namespace gm {

constexpr int kSmallRows = 2;           // rows per thread at most
constexpr int64_t kSmallMax = 1024 * kSmallRows;

// Slot of each row, longest row first (ties by index), and the padded size of the
// slice that a slot opens.  n <= kSmallMax: every block counts against all rows.
__global__ void __launch_bounds__(128) k_ell_rank(int n, const int64_t* __restrict__ row_ptr,
                                                  int32_t* __restrict__ slot,
                                                  int32_t* __restrict__ row,
                                                  int64_t* __restrict__ cnt) {
  __shared__ int len[kSmallMax];
  for (int i = threadIdx.x; i < n; i += blockDim.x) len[i] = (int)(row_ptr[i + 1] - row_ptr[i]);
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int li = len[i];
  int r = 0;
  for (int j = 0; j < n; ++j) r += len[j] > li || (len[j] == li && j < i);
  slot[i] = r;
  row[r] = i;
  if ((r & 31) == 0) cnt[r >> 5] = 32 * (int64_t)li;
}

// entry e of the row in slot q at off[q / 32] + 32 e + q % 32, columns as slots
__global__ void __launch_bounds__(128) k_ell_fill(
    int64_t n, int64_t ns, const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
    const double* __restrict__ val, const int32_t* __restrict__ slot,
    const int32_t* __restrict__ row, const int64_t* __restrict__ off, int32_t* __restrict__ ecol,
    double* __restrict__ eval) {
  const int lane = threadIdx.x & 31;
  // warps take the entries of a slice in turn
  const int64_t s = blockIdx.x;
  const int64_t q = 32 * s + lane;
  const int64_t i = q < n ? row[q] : 0;
  const int64_t b = row_ptr[i], len = q < n ? row_ptr[i + 1] - b : 0;
  const int64_t o = off[s], w = (off[s + 1] - o) >> 5;
  for (int64_t e = threadIdx.x >> 5; e < w; e += blockDim.x >> 5) {
    const bool in = e < len;
    ecol[o + 32 * e + lane] = in ? slot[col[b + e]] : (int32_t)(q < n ? q : n - 1);
    eval[o + 32 * e + lane] = in ? val[b + e] : 0.0;
  }
}

struct SmallCg {
  int n;
  const int64_t* off;      // slice offsets
  const int32_t* row;      // row of a slot
  const int32_t* ecol;
  const double* eval;
  const double* dv;        // D
  const double* minv;      // 1 / diag B
  const double* rhs;       // element (row, column) at row * ld + column
  double* x;               // in (warm) and out
  int64_t ld;
  double stop2;            // ||r||^2 <= stop2 ||b||^2
  int warm;
  int max_it;
  double* bb;              // per column: ||b||^2 and the last ||r||^2
  double* rr;
  int* iters;              // largest iteration count (atomic max)
  unsigned* flags;
};

// Sum over the block of NV values per thread, in every thread: the warps'
// values go through shared memory lane by lane, so that the FP64 additions are
// one per warp and sum plus one tree (fixed order).
template <int NV>
__device__ __forceinline__ void small_sum(double (&v)[NV], double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) sh[(k * 32 + w) * 32 + lane] = v[k];
  __syncthreads();
  for (int k = w; k < NV; k += W) {
    const double* s = sh + k * 1024 + lane;
    double a = 0, b = 0;
    for (int q = 0; q < W; q += 2) {
      a += s[32 * q];
      if (q + 1 < W) b += s[32 * (q + 1)];
    }
    a += b;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) sh[NV * 1024 + k] = a;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = sh[NV * 1024 + k];
}

constexpr double kSmallWork = 2.0e5;      // stored entries x columns per SM
constexpr double kSmallMean = 1.6e4;      // stored entries of a mean solve

// T: threads at most; three blocks of 512 share an SM (a warp's chain of loads and
// additions is long, the FP64 unit wants the other columns meanwhile)
template <int RPT, int T>
__global__ void __launch_bounds__(T, T == 512 ? 3 : 1) k_cg_columns(SmallCg A) {
  extern __shared__ double sm[];
  double* pd = sm;                       // n
  double* sh = sm + ((A.n + 31) & ~31);  // 2 x 1024 + 8
  const int64_t c = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  double x[RPT], r[RPT], p[RPT], d[RPT], m[RPT];
  // slots of this thread: a group of four slices over the four schedulers, every
  // other group in reverse, so that each has long and short rows
  int qs[RPT];
  int64_t at[RPT];
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    const int g = (w + k * W) >> 2, l = w & 3;
    qs[k] = 32 * (4 * g + ((g & 1) ? 3 - l : l)) + lane;
    at[k] = qs[k] < A.n ? A.row[qs[k]] * A.ld + c : -1;
  }
  auto product = [&](double (&q)[RPT]) {
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int s = qs[k] >> 5;
      double a0 = 0, a1 = 0;
      if (32 * s < A.n) {
        const int64_t o = A.off[s];
        const int w = (int)((A.off[s + 1] - o) >> 5);
        const int32_t* ec = A.ecol + o + lane;
        const double* ev = A.eval + o + lane;
        int e = 0;
        for (; e + 3 < w; e += 4) {
          const int32_t c0 = ec[32 * e], c1 = ec[32 * e + 32], c2 = ec[32 * e + 64],
                        c3 = ec[32 * e + 96];
          const double v0 = ev[32 * e], v1 = ev[32 * e + 32], v2 = ev[32 * e + 64],
                       v3 = ev[32 * e + 96];
          a0 = fma(v0, pd[c0], a0);
          a1 = fma(v1, pd[c1], a1);
          a0 = fma(v2, pd[c2], a0);
          a1 = fma(v3, pd[c3], a1);
        }
        for (; e < w; ++e) a0 = fma(ev[32 * e], pd[ec[32 * e]], a0);
      }
      q[k] = a0 + a1;
    }
  };
  double s2[2] = {0, 0};
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    x[k] = r[k] = p[k] = d[k] = m[k] = 0.0;
    if (at[k] >= 0) {
      const int i = A.row[qs[k]];
      r[k] = A.rhs[at[k]];
      d[k] = A.dv[i];
      m[k] = A.minv[i];
      if (A.warm) {
        x[k] = A.x[at[k]];
        pd[qs[k]] = d[k] * x[k];
      }
    }
    s2[0] += r[k] * r[k];
  }
  if (A.warm) {  // r = b - B x
    __syncthreads();
    double q[RPT];
    product(q);
#pragma unroll
    for (int k = 0; k < RPT; ++k) r[k] -= x[k] + d[k] * q[k];
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    p[k] = m[k] * r[k];
    s2[1] += r[k] * p[k];
    if (at[k] >= 0) pd[qs[k]] = d[k] * p[k];
  }
  small_sum<2>(s2, sh);
  const double bb = s2[0];
  double rz = s2[1], rr = bb;
  int it = 0;
  if (!isfinite(bb) || !isfinite(rz)) {
    if (threadIdx.x == 0) atomicOr(A.flags, kFlagNonFinite);
  } else if (bb > 0) {
    for (it = 1; it <= A.max_it; ++it) {
      double q[RPT], pq[1] = {0};
      product(q);
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        q[k] = fma(d[k], q[k], p[k]);
        pq[0] = fma(p[k], q[k], pq[0]);
      }
      small_sum<1>(pq, sh);
      double alpha = 0;
      if (pq[0] > 0 && rz > 0) {
        alpha = rz / pq[0];
      } else if (rz > 0) {  // not positive definite (or not finite)
        if (threadIdx.x == 0) atomicOr(A.flags, kFlagNotSPD);
        break;
      }
      double s[2] = {0, 0};
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        x[k] = fma(alpha, p[k], x[k]);
        r[k] = fma(-alpha, q[k], r[k]);
        s[0] = fma(r[k], m[k] * r[k], s[0]);
        s[1] = fma(r[k], r[k], s[1]);
      }
      small_sum<2>(s, sh);
      rr = s[1];
      if (!isfinite(s[0]) || !isfinite(rr)) {
        if (threadIdx.x == 0) atomicOr(A.flags, kFlagNonFinite);
        break;
      }
      if (rr <= A.stop2 * bb || it == A.max_it) break;
      const double beta = rz > 0 ? s[0] / rz : 0.0;
      rz = s[0];
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        p[k] = fma(beta, p[k], m[k] * r[k]);
        if (at[k] >= 0) pd[qs[k]] = d[k] * p[k];
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int k = 0; k < RPT; ++k)
    if (at[k] >= 0) A.x[at[k]] = bb > 0 ? x[k] : 0.0;  // a zero right-hand side: zero
  if (threadIdx.x == 0) {
    A.bb[c] = bb;
    A.rr[c] = rr;
    atomicMax(A.iters, it > A.max_it ? A.max_it : it);
  }
}

// ---------------------------------------------------------------- host
static gm_status small_prepare(gm_ctx* c) {
  const int64_t n = c->n, ns = ceil_div(n, 32);
  cudaStream_t st = c->stream;
  ScopedDev cnt(c, ns * sizeof(int64_t)), slot(c, n * sizeof(int32_t));
  if (!cnt.p || !slot.p || !ensure(c, c->ell_off, (ns + 1) * sizeof(int64_t)) ||
      !ensure(c, c->ell_row, n * sizeof(int32_t)))
    return set_error(c, GM_E_NOMEM, "sliced rows");
  GM_PROF(c, "k_ell_rank");
  k_ell_rank<<<(unsigned)ceil_div(n, 128), 128, 0, st>>>((int)n, c->row_ptr, (int32_t*)slot.p,
                                                         (int32_t*)c->ell_row.p, (int64_t*)cnt.p);
  GM_LAUNCH_CHECK(c);
  gm_status s = scan_i64(c, (const int64_t*)cnt.p, (int64_t*)c->ell_off.p, ns);
  if (s != GM_OK) return s;
  int64_t* h = (int64_t*)c->h_pinned;
  GM_CUDA_CHECK(c, cudaMemcpyAsync(h, (int64_t*)c->ell_off.p + ns, sizeof(int64_t),
                                   cudaMemcpyDeviceToHost, st));
  GM_CUDA_CHECK(c, cudaStreamSynchronize(st));
  const int64_t total = std::max<int64_t>(*h, 1);
  if (!ensure(c, c->ell_col, total * sizeof(int32_t)) ||
      !ensure(c, c->ell_val, total * sizeof(double)))
    return set_error(c, GM_E_NOMEM, "sliced rows");
  GM_PROF(c, "k_ell_fill");
  k_ell_fill<<<(unsigned)ns, 128, 0, st>>>(
      n, ns, c->row_ptr, c->col, (const double*)c->val, (const int32_t*)slot.p,
      (const int32_t*)c->ell_row.p, (const int64_t*)c->ell_off.p, (int32_t*)c->ell_col.p,
      (double*)c->ell_val.p);
  GM_LAUNCH_CHECK(c);
  if (!ensure(c, c->ell_iters, sizeof(int))) return set_error(c, GM_E_NOMEM, "iteration count");
  return GM_OK;
}

void small_release(gm_ctx* c) {
  for (Buffer* b : {&c->ell_off, &c->ell_row, &c->ell_col, &c->ell_val, &c->ell_iters}) {
    if (b->p) dev_free_now(c, b->p, b->bytes);
    *b = Buffer{};
  }
  c->ell_state = -1;
}

// Whether a solve of n_cols FP64 right-hand sides runs here: the rows fit a block,
// an SM's share of the columns is short and the sliced rows fit the memory.  Times of
// a call without its mean solve, stored entries x columns per SM beside it:
//   400 stars, own columns    39,330:  4.4 ms in panels,  2.0 ms here
//   600                      131,448:  7.6,               6.6
//   640                      192,020:  7.4,               7.0
//   700                      211,590:  8.4,               8.4
//   760                      254,280:  8.2,               9.1
//   1,300, 100 queries       144,496: 12.4,               7.9
//   1,500, 100 queries       176,962: 10.3,               9.0
//   1,700, 100 queries       228,742: 11.8,              11.2
//   2,000, 100 queries       297,812: 12.8,              14.5
bool small_cg_fits(gm_ctx* c, int64_t n_cols) {
  if (c->cfg.precision == GM_PREC_FP32 || c->n_fields > 1 || c->n > kSmallMax ||
      c->ell_state < 0)
    return false;
  const char* e = std::getenv("GM_SPMM");  // a pinned product (simt, tc) keeps the panels
  if (e && (e[0] == 's' || e[0] == 't')) return false;
  const double waves = (double)ceil_div(n_cols, (int64_t)sm_count(c));
  if (!((double)c->nnz * waves < kSmallWork)) return false;
  if (c->ell_state == 0) {
    const std::string before = c->last_error;
    if (small_prepare(c) != GM_OK) {
      small_release(c);
      c->last_error = before;
      return false;
    }
    c->ell_state = 1;
  }
  return true;
}

// A mean solve has one column: a block on one SM, against k_cg_run over the chip
// (about 15 us an iteration): 1.1 / 1.2 ms at 14,600 stored entries, 2.5 / 1.3 at
// 43,000, 3.8 / 1.6 at 86,600.
bool small_cg_mean_fits(gm_ctx* c) {
  return (double)c->nnz < kSmallMean && small_cg_fits(c, 1);
}

// Behind small_cg_fits: solves B x = rhs for n_cols columns (leading dimension ld); bb
// and rr: ||b||^2 and ||r||^2 of the columns.  Synchronises.
gm_status small_cg(gm_ctx* c, int64_t n_cols, int64_t ld, const double* dv, const double* minv,
                   const double* rhs, double* x, bool warm, double tol, double* bb, double* rr,
                   int64_t* iters) {
  cudaStream_t st = c->stream;
  int* d_it = (int*)c->ell_iters.p;
  GM_CUDA_CHECK(c, cudaMemsetAsync(d_it, 0, sizeof(int), st));
  // a column goes on to 1e-2 of the tolerance: one iteration in ten, and the stopping
  // error stays out of the results (a panel's columns go on too, to 1e-3 of it, while
  // others need it)
  SmallCg A{(int)c->n, (const int64_t*)c->ell_off.p, (const int32_t*)c->ell_row.p,
            (const int32_t*)c->ell_col.p, (const double*)c->ell_val.p, dv, minv, rhs, x, ld,
            1e-4 * tol * tol,
            warm ? 1 : 0, c->cfg.cg_max_iter, bb, rr, d_it, c->d_flags};
  const int rpt = c->n > 1024 ? 2 : 1;
  const int T = (int)(ceil_div(ceil_div(c->n, rpt), 128) * 128);  // groups of four warps
  const size_t smem = (((c->n + 31) & ~31ll) + 2 * 1024 + 8) * sizeof(double);
  GM_PROF(c, "k_cg_columns");
  auto kern = rpt == 2 ? k_cg_columns<2, 1024>
                       : T > 512 ? k_cg_columns<1, 1024> : k_cg_columns<1, 512>;
  GM_CUDA_CHECK(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kern<<<(unsigned)n_cols, T, smem, st>>>(A);
  GM_LAUNCH_CHECK(c);
  int* h = (int*)c->h_pinned;
  GM_CUDA_CHECK(c, cudaMemcpyAsync(h, d_it, sizeof(int), cudaMemcpyDeviceToHost, st));
  GM_CUDA_CHECK(c, cudaStreamSynchronize(st));
  *iters = *h;
  return GM_OK;
}

}  // namespace gm
