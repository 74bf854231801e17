// FP64 panel product of the variance solves, Q = P + d o (K PD), on the tensor
// cores.
//
// GB300's FP64 units (2 lanes per clock and SM) bound the CUDA-core product: one
// fused multiply-add per stored entry and right-hand side, 1.3 ms for 2,001
// stars.  Here the operands are split into integers that BF16 holds exactly and
// whose products the tensor cores add exactly in FP32 (Ozaki, Ogita, Oishi &
// Rump 2012, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication"):
//   * every row of K is scaled by a power of two to |x| < 1, and v = rint(2^62 x)
//     is written in eight balanced base-256 digits d_0 .. d_7 (|d| <= 128),
//     x = sum_k d_k 2^(-6 - 8 k); the columns of PD likewise;
//   * the digit products d_i e_j with i + j = g <= 7 share the weight
//     2^(-12 - 8 g) and one FP32 accumulator.  At most 8 x 128 products of size
//     2^14 meet in an accumulator between two read-outs (128 columns of K), so
//     every sum is an integer up to 2^24: exact, in any order;
//   * each read-out adds the eight accumulators into two 64-bit integers per
//     element; the result is rounded once, at the end.
// What is left out (i + j >= 8: seven products of up to 2^14 at 2^-76) and the rounding
// of v are below 2^-57 of the row's largest entry times the column's largest, per stored
// entry of the row, where an FP64 sum rounds every partial sum at 2^-53.  The bound is of
// the two maxima, not of each term: an entry keeps 53 bits down to 2^-9 of its column's
// largest, and fewer below that.  Errors of the posteriors against 64-bit references
// did not grow (3.3e-10 at 2,001 stars in both forms).
//
// Layout.  128-row tiles with unions of columns as in the FP32 product, K-steps
// of 16 union columns, eight 4 KB images per K-step.  The panel's digits are
// eight BF16 planes.  A CTA does NC = 64 panel columns (32 where that leaves SMs
// idle): per K-step 36 MMAs of N = NC, digit i of K times digit j of the panel
// into accumulator g = i + j, all of one shape so that those of one accumulator
// stay in order; the eight accumulators take all 512 columns of tensor memory.
//
// Roles: warps 0-2 copy (one bulk copy of K's images and 16-byte asynchronous
// copies of the panel's rows per K-step, a ring of stages), warp 3 issues the
// MMAs, the other warps read the accumulators out after every eight K-steps and
// run the epilogue.  Every wait is bounded and gives up when another thread has.
// 2,001 stars x 2,016 columns (342,585 entries, 295 K-steps): 193 us, with the
// column exponents and digit planes 232 us, against 1,306 us on the FP64 units
// (of which 1,130 us is their rate).  One CTA per SM: the K-steps run at L2's
// rate (48 KB each), the read-outs and the FP64 epilogue (24,000 clocks a CTA)
// are not hidden.
#include <algorithm>
#include <cstdlib>

#include "gm_internal.cuh"
#include "gm_tcgen05.cuh"

namespace gm {

constexpr int kOzDigits = 8;
constexpr int kOzA = 128 * 16 * 2;            // one digit image of a K-step of K
constexpr int kOzB = 16 * 64 * 2;             // one digit of a K-step of the panel
constexpr int kOzPeriod = 8;                  // K-steps between two read-outs
constexpr int kOzRing = 4;

// byte offset of (row, k) in a no-swizzle K-major image with 16 columns
__host__ __device__ __forceinline__ int oz_aoff(int row, int k) {
  return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}
// byte offset of digit j, (k, n), n < 64, in the 128-byte-swizzled MN-major B tile:
// an atom of 8 rows x 64 columns (1 KB) per digit and k-group
__host__ __device__ __forceinline__ int oz_boff(int j, int k, int n) {
  return (k >> 3) * (kOzDigits * 1024) + j * 1024 + (k & 7) * 128 + (((n >> 3) ^ (k & 7)) << 4) +
         (n & 7) * 2;
}

// Exponent e of a double's bits with |x| < 2^e (0 for x = 0, an exponent far
// below any other).
__device__ __forceinline__ int oz_exp(long long bits) {
  return (int)((bits >> 52) & 0x7ff) - 1022;
}

// v = rint(x 2^(62 - e)) for |x| < 2^e, by integer operations (subnormal x: 0).
__device__ __forceinline__ long long oz_fixed(long long bits, int e) {
  const int ex = (int)((bits >> 52) & 0x7ff);
  if (ex == 0) return 0;
  long long m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
  const int s = ex - 1022 - e + 9;  // x = m 2^(ex - 1075): m 2^(ex - 1075 + 62 - e)
  if (s >= 0) m <<= s;
  else if (s >= -54) m = (m + (1ll << (-s - 1))) >> -s;
  else m = 0;
  return bits < 0 ? -m : m;
}

// digits of v, most significant first, as BF16 bit patterns
__device__ __forceinline__ void oz_digits(long long v, uint32_t (&d)[kOzDigits]) {
#pragma unroll
  for (int k = kOzDigits - 1; k >= 0; --k) {
    int q;
    if (k > 0) {
      q = (int)(signed char)(v & 0xff);
      v = (v - q) >> 8;
    } else {
      q = (int)v;
    }
    // |q| <= 128 as a float by the magic-number addition; its high half is BF16
    d[k] = __float_as_uint(__int_as_float(0x4B400000 + q) - 12582912.0f) >> 16;
  }
}

// ---------------------------------------------------------------- K
__global__ void k_oz_row_exp(int64_t n, const int64_t* __restrict__ row_ptr,
                             const double* __restrict__ val, int* __restrict__ erow) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nw) {
    int e = -1022;
    for (int64_t q = row_ptr[i] + lane; q < row_ptr[i + 1]; q += 32)
      e = max(e, oz_exp(__double_as_longlong(val[q])));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) erow[i] = e;
  }
}

// Digit images: entry (i, j) of block b at union position q of j goes to K-step
// kbase[b] + q / 16, column q % 16, row p - brow0 (p = the tile position of i).
__global__ void k_oz_fill(int64_t n, const int64_t* __restrict__ row_ptr,
                          const int32_t* __restrict__ col, const double* __restrict__ val,
                          const int* __restrict__ erow, const int64_t* __restrict__ bptr,
                          const int64_t* __restrict__ kbase, const int32_t* __restrict__ ucol,
                          const int32_t* __restrict__ tpos, unsigned char* __restrict__ img) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nw) {
    const int64_t p = tpos ? tpos[i] : i;
    const int64_t b = p / 128;
    const int t = (int)(p - b * 128);
    const int64_t u0 = bptr[b], u1 = bptr[b + 1];
    const int e = erow[i];
    for (int64_t q0 = row_ptr[i] + lane; q0 < row_ptr[i + 1]; q0 += 32) {
      const int32_t j = col[q0];
      int64_t lo = u0, hi = u1;  // ucol[lo] <= j < ucol[hi]
      while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (ucol[mid] <= j) lo = mid; else hi = mid;
      }
      const int64_t q = lo - u0;
      unsigned char* step = img + (kbase[b] + q / 16) * (int64_t)(kOzDigits * kOzA);
      uint32_t d[kOzDigits];
      oz_digits(oz_fixed(__double_as_longlong(val[q0]), e), d);
      const int off = oz_aoff(t, (int)(q & 15));
#pragma unroll
      for (int k = 0; k < kOzDigits; ++k)
        *reinterpret_cast<uint16_t*>(step + k * kOzA + off) = (uint16_t)d[k];
    }
  }
}

// ---------------------------------------------------------------- panel
__global__ void k_oz_fill_int(int n, int v, int* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = v;
}

// Column exponents of PD: warp-strided rows, lane = column of the chunk.
__global__ void __launch_bounds__(256) k_oz_col_exp(int64_t n, int R, const double* __restrict__ PD,
                                                    int* __restrict__ ecol) {
  __shared__ int sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = blockIdx.y * 32 + lane;
  int e = -1022;
  const int64_t nw = (int64_t)gridDim.x * 8;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * 8 + w; i < n; i += nw)
    e = max(e, oz_exp(__double_as_longlong(PD[i * R + c])));
  sh[w][lane] = e;
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int k = 1; k < 8; ++k) e = max(e, sh[k][lane]);
    atomicMax(ecol + c, e);
  }
}

// Digit planes of PD: thread = (row, 8 columns).
__global__ void __launch_bounds__(256) k_oz_slice(int64_t n, int R, const double* __restrict__ PD,
                                                  const int* __restrict__ ecol,
                                                  uint16_t* __restrict__ planes, int64_t pe) {
  const int64_t total = n * (R / 8);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t at = t * 8;
    const int c = (int)(at % R);
    const double2* src = reinterpret_cast<const double2*>(PD + at);
    uint32_t w[kOzDigits][4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const double2 x = src[h];
      uint32_t a[kOzDigits], b[kOzDigits];
      oz_digits(oz_fixed(__double_as_longlong(x.x), ecol[c + 2 * h]), a);
      oz_digits(oz_fixed(__double_as_longlong(x.y), ecol[c + 2 * h + 1]), b);
#pragma unroll
      for (int k = 0; k < kOzDigits; ++k) w[k][h] = a[k] | (b[k] << 16);
    }
#pragma unroll
    for (int k = 0; k < kOzDigits; ++k)
      *reinterpret_cast<uint4*>(planes + k * pe + at) =
          make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
  }
}

// ---------------------------------------------------------------- product
template <int NC>
struct Oz {
  // 20 warps at 64 columns (five a scheduler: 96 registers a thread)
  static constexpr int kProd = 96;
  static constexpr int kEpiWarps = NC / 4;   // 16 panel columns each, four lane quarters
  static constexpr int kThreads = kProd + 32 + 32 * kEpiWarps;
  static constexpr int kStage = kOzDigits * (kOzA + kOzB);  // 48 KB
  static constexpr int kSmem = kOzRing * kStage + 1024;
};

__device__ __forceinline__ void oz_ld8(uint32_t taddr, uint32_t (&u)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]),
                 "=r"(u[6]), "=r"(u[7])
               : "r"(taddr));
}

// 96-bit two's-complement sum of one element (least significant word first).
struct Oz96 {
  uint32_t w0 = 0, w1 = 0, w2 = 0;
  // += v
  __device__ __forceinline__ void add_low(long long v) {
    const uint32_t a = (uint32_t)v, b = (uint32_t)(v >> 32), s = (uint32_t)((int)b >> 31);
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(w0), "+r"(w1), "+r"(w2)
        : "r"(a), "r"(b), "r"(s));
  }
  // += 2^32 v
  __device__ __forceinline__ void add_high(long long v) {
    const uint32_t a = (uint32_t)v, b = (uint32_t)(v >> 32);
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(w1), "+r"(w2) : "r"(a), "r"(b));
  }
  __device__ __forceinline__ double value() const {
    return fma((double)(long long)(((unsigned long long)w2 << 32) | w1), 0x1p32, (double)w0);
  }
};

// 2^e as a double (e within the normal range)
__device__ __forceinline__ double oz_pow2(int e) {
  return __longlong_as_double((long long)(e + 1023) << 52);
}
// the same for a column: NaN when the column held an infinity or a NaN
__device__ __forceinline__ double oz_col_scale(int e) { return e > 1023 ? NAN : oz_pow2(e); }

template <int NC>
__global__ void __launch_bounds__(Oz<NC>::kThreads, 1) k_panel_spmm_tc64(
    int64_t n, int R, const int64_t* __restrict__ kbase, const int32_t* __restrict__ upad,
    const unsigned char* __restrict__ img, const int* __restrict__ erow,
    const int* __restrict__ ecol, const double* __restrict__ dv, const double* __restrict__ P,
    const uint16_t* __restrict__ planes, int64_t pe, double* __restrict__ Q,
    double* __restrict__ part_pq, const int32_t* __restrict__ trow, unsigned* __restrict__ flags,
    bool expire) {
  typedef Oz<NC> O;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint64_t fullA[kOzRing], fullB[kOzRing], empty[kOzRing], accfull, accempty;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  volatile int* abort_v = &abort_flag;
  unsigned char* smem = smem_raw + ((1024u - (tg::smem(smem_raw) & 1023u)) & 1023u);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int64_t b = blockIdx.y;
  const int c0 = blockIdx.x * NC;
  const int64_t brow0 = b * 128, bend = brow0 + 128 < n ? brow0 + 128 : n;
  const int64_t ks0 = kbase[b], nks = kbase[b + 1] - ks0;
  const int64_t nper = (nks + kOzPeriod - 1) / kOzPeriod;

  if (t == 0) {
    abort_flag = 0;
    for (int q = 0; q < kOzRing; ++q) {
      tg::mbar_init(tg::smem(&fullA[q]), 1);
      tg::mbar_init(tg::smem(&fullB[q]), O::kProd);
      tg::mbar_init(tg::smem(&empty[q]), 1);
    }
    tg::mbar_init(tg::smem(&accfull), 1);
    tg::mbar_init(tg::smem(&accempty), 32 * O::kEpiWarps);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 3) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     tg::smem(&tmem_base)),
                 "n"(kOzDigits * NC));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;

  Oz96 acc[16];

  if (warp < 3) {
    // ---- producers: 16-byte chunks (8 columns of one digit of one row), the
    // chunks of a row's digit in consecutive threads
    constexpr int kPer = NC / 8;  // chunks per row and digit
    int64_t issued = 0;
    for (int64_t ks = 0; ks < nks; ++ks) {
      const int s = (int)(ks % kOzRing);
      const int64_t use = ks / kOzRing;
      if (use > 0 && !tg::wait(tg::smem(&empty[s]), (uint32_t)((use - 1) & 1), abort_v)) {
        abort_flag = 1;
        break;
      }
      unsigned char* sA = smem + s * O::kStage;
      unsigned char* sB = sA + kOzDigits * kOzA;
      if (t == 0) {
        tg::arrive_expect_tx(tg::smem(&fullA[s]), kOzDigits * kOzA);
        tg::bulk_g2s(tg::smem(sA), img + (ks0 + ks) * (int64_t)(kOzDigits * kOzA),
                     kOzDigits * kOzA, tg::smem(&fullA[s]));
        ++issued;
      }
      for (int q = t; q < 16 * kOzDigits * kPer; q += O::kProd) {
        const int ch = q % kPer, j = (q / kPer) % kOzDigits, k = q / (kPer * kOzDigits);
        const int64_t row = __ldg(upad + (ks0 + ks) * 16 + k);
        const int col = c0 + 8 * ch;
        const bool in = col < R;  // R is a multiple of 32
        const uint16_t* src = in ? planes + j * pe + row * R + col : planes;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                         tg::smem(sB) + (uint32_t)oz_boff(j, k, 8 * ch)),
                     "l"(__cvta_generic_to_global(src)), "r"(in ? 16 : 0)
                     : "memory");
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(
                       tg::smem(&fullB[s]))
                   : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (t == 0 && *abort_v) {  // bounded waits for the bulk copies still in flight
      for (int q = 0; q < kOzRing; ++q) {
        const int64_t na = issued > q ? (issued - 1 - q) / kOzRing + 1 : 0;
        if (na > 0) tg::wait(tg::smem(&fullA[q]), (uint32_t)((na - 1) & 1), nullptr);
      }
    }
  } else if (warp == 3) {
    if (lane == 0) {
      // ---- MMA issuer
      int64_t done = 0;
      for (int64_t ks = 0; ks < nks; ++ks) {
        const int s = (int)(ks % kOzRing);
        const uint32_t par = (uint32_t)((ks / kOzRing) & 1);
        const int64_t per = ks / kOzPeriod;
        const bool first = ks % kOzPeriod == 0;
        if (first && per > 0 &&
            !tg::wait(tg::smem(&accempty), (uint32_t)((per - 1) & 1), abort_v)) {
          abort_flag = 1;
          break;
        }
        if (!tg::wait(tg::smem(&fullA[s]), par, abort_v) ||
            !tg::wait(tg::smem(&fullB[s]), par, abort_v)) {
          abort_flag = 1;
          break;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t a = tg::smem(smem + s * O::kStage), bb = a + kOzDigits * kOzA;
        constexpr uint32_t idesc = tg::idesc_bf16(128, NC, false, true);
#pragma unroll
        for (int i = 0; i < kOzDigits; ++i)
#pragma unroll
          for (int j = 0; j < kOzDigits - i; ++j)
            tg::mma(tmem + (uint32_t)(NC * (i + j)), tg::desc(a + i * kOzA, 128, 256, 0),
                    tg::desc(bb + j * 1024, 1024, kOzDigits * 1024, 2), idesc,
                    (i > 0 || !first) ? 1u : 0u);
        tg::commit(tg::smem(&empty[s]));
        ++done;
        if (ks % kOzPeriod == kOzPeriod - 1 || ks == nks - 1) tg::commit(tg::smem(&accfull));
      }
      if (*abort_v && done > 0) {  // bounded wait for the MMAs in flight
        const int64_t last = done - 1;
        tg::wait(tg::smem(&empty[last % kOzRing]), (uint32_t)((last / kOzRing) & 1), nullptr);
      }
    }
    __syncwarp();
  } else {
    // ---- read-outs: warp w reads TMEM lanes 32 (w mod 4) .., panel columns
    // 16 sub .. 16 sub + 15
    const int sub = (warp - 4) >> 2, quad = warp & 3;
    const uint32_t ta = tmem + ((uint32_t)(32 * quad) << 16) + 16u * sub;
    for (int64_t per = 0; per < nper; ++per) {
      bool up = tg::wait(tg::smem(&accfull), (uint32_t)(per & 1), abort_v);
      if (expire && per == nper - 1 && b == 0 && blockIdx.x == 0 && warp == 5 && lane == 7)
        up = false;
      // the warp's lanes leave together: the loads below are for whole warps
      if (!__all_sync(0xffffffffu, up)) {
        abort_flag = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          long long v[8];
#pragma unroll
          for (int g = 0; g < 4; g += 2) {
            uint32_t u[8], x[8];
            oz_ld8(ta + (uint32_t)(NC * (4 * h + g)) + 8u * q, u);
            oz_ld8(ta + (uint32_t)(NC * (4 * h + g + 1)) + 8u * q, x);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              // two groups fit a 64-bit step: |u| 2^8 + |x| < 2^33
              const long long d = ((long long)__float2int_rn(__uint_as_float(u[k])) << 8) +
                                  __float2int_rn(__uint_as_float(x[k]));
              v[k] = g == 0 ? d : (v[k] << 16) + d;
            }
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (h == 0) acc[8 * q + k].add_high(v[k]);
            else acc[8 * q + k].add_low(v[k]);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      tg::arrive(tg::smem(&accempty));
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  const bool ok = !abort_flag;
  double* sh_pq = reinterpret_cast<double*>(smem);  // [4][NC], after the last MMA
  if (ok && warp > 3) {
    const int sub = (warp - 4) >> 2, quad = warp & 3;
    const int64_t pos = brow0 + 32 * quad + lane;
    const bool vrow = pos < bend;
    const int64_t row = (vrow && trow) ? (int64_t)trow[pos] : pos;
    const int cl = 16 * sub;
    double pq[16];
    if (vrow && c0 + cl < R) {
      // times 2^(erow + ecol - 68), the row's part (its d included) once
      const double dr = dv[row] * oz_pow2(max(erow[row], -950) - 68);
      const int64_t at = row * R + c0 + cl;
#pragma unroll
      for (int k = 0; k < 16; k += 2) {
        const double2 p = *reinterpret_cast<const double2*>(P + at + k);
        double2 q;
        q.x = fma(dr, acc[k].value() * oz_col_scale(ecol[c0 + cl + k]), p.x);
        q.y = fma(dr, acc[k + 1].value() * oz_col_scale(ecol[c0 + cl + k + 1]), p.y);
        *reinterpret_cast<double2*>(Q + at + k) = q;
        pq[k] = p.x * q.x;
        pq[k + 1] = p.y * q.y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) pq[k] = 0.0;
    }
    // column sums over the warp's rows: a reduce-scatter of shuffles, fixed
    // order; lanes 2c' and 2c' + 1 end with column c' = bits 4..1 of the lane
#pragma unroll
    for (int w = 8; w >= 1; w >>= 1) {
      const int bit = 2 * w;
#pragma unroll
      for (int j = 0; j < w; ++j) {
        const bool up = lane & bit;
        const double send = up ? pq[j] : pq[j + w];
        const double keep = up ? pq[j + w] : pq[j];
        pq[j] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
      }
    }
    pq[0] += __shfl_xor_sync(0xffffffffu, pq[0], 1);
    const int colw = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 +
                     ((lane >> 1) & 1);
    if ((lane & 1) == 0) sh_pq[quad * NC + cl + colw] = pq[0];
  }
  __syncthreads();
  if (ok) {
    if (t < NC && c0 + t < R)
      part_pq[b * R + c0 + t] = ((sh_pq[t] + sh_pq[NC + t]) + sh_pq[2 * NC + t]) +
                                sh_pq[3 * NC + t];
  } else if (t == 0) {
    atomicOr(flags, kFlagTimeout);
  }
  __syncthreads();
  if (warp == 3) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "n"(kOzDigits * NC));
  }
}

// ---------------------------------------------------------------- host
gm_status tc64_fill(gm_ctx* c, const int64_t* bptr, const int32_t* ucol) {
  const int64_t n = c->n;
  if (!ensure(c, c->tc64_erow, n * sizeof(int)))
    return set_error(c, GM_E_NOMEM, "tile row exponents");
  const int wb = (int)std::min<int64_t>(ceil_div(n * 32, 256), 32 * sm_count(c));
  GM_PROF(c, "k_oz_row_exp");
  k_oz_row_exp<<<wb, 256, 0, c->stream>>>(n, c->row_ptr, (const double*)c->val,
                                          (int*)c->tc64_erow.p);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_oz_fill");
  k_oz_fill<<<wb, 256, 0, c->stream>>>(
      n, c->row_ptr, c->col, (const double*)c->val, (const int*)c->tc64_erow.p, bptr,
      (const int64_t*)c->tc_kbase.p, ucol, c->tc_order ? (const int32_t*)c->tc_tpos.p : nullptr,
      (unsigned char*)c->tc_img.p);
  GM_LAUNCH_CHECK(c);
  return GM_OK;
}

size_t tc64_kstep_bytes() { return (size_t)kOzDigits * kOzA; }

template <int NC>
static gm_status launch_oz(gm_ctx* c, int64_t n, int R, const int* ecol, const double* dv,
                           const double* P, const uint16_t* planes, double* Q, double* part_pq) {
  typedef Oz<NC> O;
  GM_CUDA_CHECK(c, cudaFuncSetAttribute(k_panel_spmm_tc64<NC>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, O::kSmem));
  GM_PROF(c, "k_panel_spmm_tc64");
  k_panel_spmm_tc64<NC><<<dim3((unsigned)ceil_div(R, NC), (unsigned)c->tc_nblk), O::kThreads,
                          O::kSmem, c->stream>>>(
      n, R, (const int64_t*)c->tc_kbase.p, (const int32_t*)c->tc_upad.p,
      (const unsigned char*)c->tc_img.p, (const int*)c->tc64_erow.p, ecol, dv, P, planes,
      n * (int64_t)R, Q, part_pq, c->tc_order ? (const int32_t*)c->tc_trow.p : nullptr,
      c->d_flags, wait_expires("product64"));
  GM_LAUNCH_CHECK(c);
  return GM_OK;
}

bool tc64_panel_room(gm_ctx* c, int64_t n, int64_t R) {
  return ensure(c, c->tc_planes, (size_t)(n * R) * kOzDigits * sizeof(uint16_t)) &&
         ensure(c, c->tc64_ecol, (size_t)R * sizeof(int));
}

gm_status panel_spmm_tc64(gm_ctx* c, int64_t n, int R, const double* dv, const double* P,
                          const double* PD, double* Q, double* part_pq) {
  const int64_t pe = n * (int64_t)R;
  if (!tc64_panel_room(c, n, R)) return set_error(c, GM_E_NOMEM, "digit planes of the panel");
  int* ecol = (int*)c->tc64_ecol.p;
  uint16_t* planes = (uint16_t*)c->tc_planes.p;
  const int sms = sm_count(c);
  k_oz_fill_int<<<(unsigned)ceil_div(R, 256), 256, 0, c->stream>>>(R, -1022, ecol);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_oz_col_exp");
  k_oz_col_exp<<<dim3((unsigned)ceil_div(n, 64), (unsigned)(R / 32)), 256, 0, c->stream>>>(n, R, PD,
                                                                                         ecol);
  GM_LAUNCH_CHECK(c);
  GM_PROF(c, "k_oz_slice");
  k_oz_slice<<<(int)std::min<int64_t>(ceil_div(pe / 8, 256), 16 * sms), 256, 0, c->stream>>>(
      n, R, PD, ecol, planes, pe);
  GM_LAUNCH_CHECK(c);
  // 32 columns a CTA while that leaves SMs idle, else 64
  if (ceil_div(R, 32) * c->tc_nblk <= sms)
    return launch_oz<32>(c, n, R, ecol, dv, P, planes, Q, part_pq);
  return launch_oz<64>(c, n, R, ecol, dv, P, planes, Q, part_pq);
}

}  // namespace gm
