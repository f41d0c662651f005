// l0.cu -- exhaustive L0 search over a listed subspace (Eq. 1 solved exactly
// over the candidates SIS retained: SISSO's sparsifying step).
//
// For every D-subset {p_0 < .. < p_{D-1}} of the n listed candidates, the
// least-squares fit with intercept of y; the best subsets by RMSE.  With the
// candidates' centred columns X (n x N) and the centred target, the fit of a
// subset explains q = b_S^T G_SS^{-1} b_S of Syy (G = X X^T, b = X y), so
// the search is a scan of small Cholesky factorisations over the Gram
// matrix:
//   1. columns, centring, b and raw norms (one block per candidate);
//   2. the Gram matrix G on the tensor cores, error-free up to the slicing
//      (the dense contraction of the step, see k_l0_gram);
//   3. the scan: D = 1 thread per candidate, D = 2 thread per pair, D = 3
//      warp per pair (p_0, p_1) with lanes over p_2 -- an FP32 upper bound of
//      q, then an incremental Cholesky step in FP64 for the subsets it does
//      not exclude -- keeping each warp's 32 best (q, subset) in registers
//      across its lanes, then each block's 32 best;
//   4. the 64 best of all blocks (one block); their Gram entries and q again
//      in plain FP64, sample by sample, the 32 best of those, then an
//      explicit FP64 refit of each (coefficients and the RMSE of the explicit
//      residual) whose order (RMSE, positions) decides.
// The rank rule is that of the refits: a pivot of the centred Cholesky at
// or below 1e-12 of the raw column's norm rejects the subset, with the
// pivots taken in position order (as a QR of [1, X_p0, X_p1, ...] would).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "dse_internal.cuh"
#include "eval64.cuh"
#include "plan.cuh"
#include "tcgen05.cuh"
#include "util.cuh"

namespace dse {

FeatTable table_of(const dse_space *S);

namespace {

constexpr int kTop = 32;        // subsets kept per warp / block / search
constexpr int kMore = 64;       // subsets whose q is taken again in plain FP64
constexpr int kCol = 128;       // threads per column block
constexpr double kRank2 = 1e-24;  // (1e-12)^2: squared pivot / squared raw norm

__device__ __forceinline__ double col_value64(const FeatTable &F, const RungGeom &G, int64_t n_stored, uint64_t gid,
                                              int64_t s) {
  int op;
  int64_t a, b;
  if (gid < (uint64_t)n_stored) {
    op = DSE_OP_PRIMARY;
    a = (int64_t)gid;
    b = -1;
  } else {
    decode_flat(G, gid - (uint64_t)n_stored, &op, &a, &b);
  }
  return eval_op64(op, F.v64[a * F.ld + s], b >= 0 ? F.v64[b * F.ld + s] : 0.0);
}

template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double *sm) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = warp_sum64(v[i]);
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < NV; ++i) sm[w * NV + i] = v[i];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    double t = 0.0;
    for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) t += sm[ww * NV + i];
    v[i] = t;
  }
  __syncthreads();
}

// Centred target and Syy (one block).
__global__ void __launch_bounds__(kCol) k_l0_target(const double *y, int64_t N, double *yc, double *syy,
                                                    double *ymean) {
  pdl_enter();
  __shared__ double sm[(kCol / 32) * 2];
  double s[1] = {0.0};
  for (int64_t i = threadIdx.x; i < N; i += kCol) s[0] += y[i];
  block_sum<1>(s, sm);
  const double my = s[0] / (double)N;
  double q[1] = {0.0};
  for (int64_t i = threadIdx.x; i < N; i += kCol) {
    const double d = y[i] - my;
    yc[i] = d;
    q[0] = fma(d, d, q[0]);
  }
  block_sum<1>(q, sm);
  if (threadIdx.x == 0) {
    *syy = q[0];
    *ymean = my;
  }
}

// Column c: values, centred in X[c], raw sum of squares, b_c = X_c . yc, mean.
// An id outside the space gives a zero column (rejected by the rank rule).
__global__ void __launch_bounds__(kCol) k_l0_columns(FeatTable F, RungGeom G, int64_t n_stored, const uint64_t *ids,
                                                     int64_t n, const double *yc, double *X, double *nrm2, double *b,
                                                     double *mean) {
  pdl_enter();
  __shared__ double sm[(kCol / 32) * 2];
  const int64_t c = blockIdx.x;
  if (c >= n) return;
  const int64_t N = F.N;
  const bool in_space = ids[c] < (uint64_t)n_stored + G.slots;
  double *x = X + c * N;
  double s[2] = {0.0, 0.0};
  for (int64_t i = threadIdx.x; i < N; i += kCol) {
    const double v = in_space ? col_value64(F, G, n_stored, ids[c], i) : 0.0;
    x[i] = v;
    s[0] += v;
    s[1] = fma(v, v, s[1]);
  }
  block_sum<2>(s, sm);
  const double m = s[0] / (double)N;
  double t[1] = {0.0};
  for (int64_t i = threadIdx.x; i < N; i += kCol) {
    const double d = x[i] - m;
    x[i] = d;
    t[0] = fma(d, yc[i], t[0]);
  }
  block_sum<1>(t, sm);
  if (threadIdx.x == 0) {
    nrm2[c] = s[1];
    b[c] = t[0];
    mean[c] = m;
  }
}

// ---------------------------------------------------- Gram matrix, sliced
//
// G = X X^T of the centred columns to FP64 accuracy on the tensor cores.  In
// FP64 instructions the contraction is bound by the FP64 pipe (2 a clock and
// SM: n = 3000, N = 1000 took 7.69 ms).  Here each column is scaled by a power
// of two and cut into eight signed 8-bit digits, x = 2^e sum_k d_k 2^-8(k+1) +
// r with |d_k| <= 128 and |r| <= 2^(e-65), after the error-free splitting of
// Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012).  The digits are BF16 numbers,
// their products integers up to 2^14, and the 36 digit products with
// i + j <= 7 are added by class s = i + j, at most 8 of them a class, over
// blocks of 128 samples (classes 0 to 3: of 256): every partial sum is an
// integer up to 2^24, so the FP32 accumulation in tensor memory is exact in any
// order.  The blocks' sums meet in 64-bit integers; one rounding per entry
// follows at the end.
// What is dropped (r and i + j > 7) is below 2^-62.8 of 2^(e_i + e_j) a sample,
// and each column's norm at least 2^(e-2): below N 2^-58 of the product of the
// norms, where the FP64 sum is within N 2^-53.  A model of the arithmetic against
// extended precision, N = 20000, errors of a diagonal entry: lognormal products
// 2e-17 (FP64 9e-16); 1/normal, whose dropped squares all add, 3e-16 to 8e-16
// (FP64 2e-15 to 4e-15); one value 3000 times the others 7e-16 (FP64 2e-17 to
// 9e-15, by its place).  (Digits of 7 bits, in blocks of 512 samples, left 2e-13
// there, in 286 us against 294.)
namespace sliced {
constexpr int DIG = 8, BITS = 8;
constexpr int RB = 64;                       // columns of X in an image block
constexpr int KC = 16;                       // samples of a stage: one MMA deep
constexpr int TILE = RB * KC * 2;            // bytes of a digit's tile: 2048
constexpr int CHUNK = DIG * TILE;            // bytes of a block's chunk: 16 KB
constexpr int KB = 8;                        // chunks of an exact block: 128 samples
constexpr int64_t PANEL = 1 << 14;           // samples of an image at most: see its epilogue
constexpr int STAGE = 3 * CHUNK, NS = 4;     // A: two blocks (128 columns), B: one
constexpr int EPI = 16, WARPS = 2 + EPI, THREADS = 32 * WARPS;
constexpr uint32_t LBO = 128, SBO = 256;     // K-major 8 x 8 core matrices, no swizzle
constexpr uint32_t kWait = 1u << 22;
struct Shared {
  uint64_t full[NS], empty[NS], acc_full, acc_empty, drain;
  uint32_t tmem;
  int abort;
};
constexpr size_t SMEM = 1024 + (size_t)NS * STAGE;
static_assert(LBO == tc::LBO, "tc::desc_lo");
}  // namespace sliced

// Exponent e of each column: |x| <= 2^(e-1) for every sample (one block per
// column; 0 and nothing to slice for a zero or non-finite column).
__global__ void __launch_bounds__(kCol) k_l0_exponents(const double *X, int64_t N, int *ex) {
  pdl_enter();
  __shared__ unsigned long long sm[kCol / 32];
  const double *x = X + (int64_t)blockIdx.x * N;
  unsigned long long m = 0;  // (the bits of |x| order like the values)
  for (int64_t i = threadIdx.x; i < N; i += kCol) {
    const unsigned long long v = (unsigned long long)__double_as_longlong(x[i]) & 0x7fffffffffffffffull;
    m = v > m ? v : m;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kCol / 32; ++w) m = sm[w] > m ? sm[w] : m;
    const int be = (int)(m >> 52);  // biased exponent of the largest value
    ex[blockIdx.x] = m == 0 || be == 2047 ? INT32_MIN : (be ? be : 1) - 1023 + 2;
  }
}

// Digit images of samples [s0, s0 + ns): block rb, chunk c, digit k at
// ((rb nc + c) DIG + k) TILE, rows (columns of X) x 16 samples in core
// matrices.  A block of 128 threads takes one image block and chunk: thread t
// one row and half of its samples.
__global__ void __launch_bounds__(128) k_l0_slices(const double *X, const int *ex, int64_t n, int64_t N, int64_t s0,
                                                   int64_t ns, int nc, unsigned char *img) {
  pdl_enter();
  using namespace sliced;
  const int c = blockIdx.x, rb = blockIdx.y, row = threadIdx.x & 63, h = threadIdx.x >> 6;
  const int64_t col = (int64_t)rb * RB + row, k0 = (int64_t)c * KC + 8 * h;
  const int e = col < n ? ex[col] : INT32_MIN;
  uint32_t d[DIG][4];
#pragma unroll
  for (int k = 0; k < DIG; ++k) d[k][0] = d[k][1] = d[k][2] = d[k][3] = 0u;
  if (e != INT32_MIN) {
    const double *x = X + col * N + s0 + k0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      // the digits of x 2^(64 - e), an integer below 2^63, lowest first
      long long q = k0 + i < ns ? __double2ll_rn(scalbn(x[i], DIG * BITS - e)) : 0ll;
#pragma unroll
      for (int k = DIG - 1; k >= 0; --k) {
        const int v = k ? (int)((q + 128) & 255) - 128 : (int)q;
        q = (q - v) >> BITS;
        const uint32_t bits = __float_as_uint((float)v) >> 16;  // exact: |v| <= 128
        d[k][i >> 1] |= bits << (16 * (i & 1));
      }
    }
  }
  unsigned char *o = img + ((size_t)rb * nc + c) * CHUNK + (row >> 3) * SBO + h * LBO + (row & 7) * 16;
#pragma unroll
  for (int k = 0; k < DIG; ++k)
    *reinterpret_cast<uint4 *>(o + k * TILE) = make_uint4(d[k][0], d[k][1], d[k][2], d[k][3]);
}

// (h 2^32 + l) 2^e rounded to FP64, for |h| < 2^53 and results in the normal
// range, in integer instructions: the FP64 pipe (2 operations a clock and SM)
// takes 16000 cycles for a tile's entries, after the products and alone (311 us
// a launch for n = 3000, N = 1000; 294 with integers).
__device__ __forceinline__ double wide_to_double(long long h, uint32_t l, int e) {
  const bool neg = h < 0;
  const unsigned long long a = neg ? (unsigned long long)~h + (l == 0u) : (unsigned long long)h;
  const uint32_t b = neg ? 0u - l : l;
  unsigned long long m = a << 32 | b;
  int n;  // significant bits
  if (a >> 21) {
    n = 96 - __clzll((long long)a);
    const int s = n - 53;  // 1 to 32 bits are dropped
    m = a << (32 - s) | (unsigned long long)b >> s;
    const uint32_t rest = b << (32 - s);
    m += rest > 0x80000000u || (rest == 0x80000000u && (m & 1)) ? 1u : 0u;
  } else {
    n = 64 - __clzll((long long)m);
    m = m ? m << (53 - n) : 0ull;
  }
  // (m's leading bit adds the last unit of the exponent field, a carry one more)
  const unsigned long long bits = m ? ((unsigned long long)(1021 + n + e) << 52) + m : 0ull;
  return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}

// One tile of 128 x 64 entries (i-block bi of 128 columns, j-block bj of 64, bj >= 2
// bi) per CTA.  Warp 0: producer; warp 1: tensor memory and the MMAs (36 a
// chunk, accumulators s = 0..7 of 64 columns each: all of tensor memory);
// warps 2-17: the block sums into 64-bit integers, 16 entries a lane, then the
// entries i <= j of the tile, as G[i][j] (upper) or G[j][i] (the other half of
// G is not written), and the scale-free FP32 values the scan's bound reads.
// `add`: onto an earlier panel's.
__global__ void __launch_bounds__(sliced::THREADS, 1) k_l0_gram(const unsigned char *img, const int *ex, int64_t n,
                                                                int nc, int add, int upper, double *Gm, float *G32,
                                                                int *err) {
  pdl_enter();
  using namespace sliced;
  extern __shared__ __align__(1024) unsigned char smem[];
  Shared &sh = *reinterpret_cast<Shared *>(smem);
  unsigned char *stages = smem + 1024;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // tile t: i-block bi has the j-blocks 2 bi .. nb - 1, before it come bi (nb + 1 - bi)
  const int nb = 2 * (int)((n + 127) / 128);
  const int64_t t = blockIdx.x;
  int bi = 0;
  {
    const double h = 0.5 * (nb + 1);
    bi = (int)(h - sqrt(fmax(h * h - (double)t, 0.0)));
    while (bi > 0 && (int64_t)bi * (nb + 1 - bi) > t) --bi;
    while ((int64_t)(bi + 1) * (nb - bi) <= t) ++bi;
  }
  const int bj = 2 * bi + (int)(t - (int64_t)bi * (nb + 1 - bi));
  const int nkb = (nc + KB - 1) / KB;
  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&sh.full[i], 1);
      mbar_init(&sh.empty[i], 1);
    }
    mbar_init(&sh.acc_full, 1);
    mbar_init(&sh.acc_empty, EPI);
    mbar_init(&sh.drain, 1);
    sh.abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = sh.tmem;
  volatile int *abort_flag = &sh.abort;
  auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
    if (mbar_wait_bounded(bar, parity, kWait)) return true;
    atomicExch(err, DSE_ETIMEOUT);
    *abort_flag = 1;
    return false;
  };

  if (warp == 0) {
    if (elect_one()) {
      int c = 0;
      const unsigned char *a0 = img + (size_t)(2 * bi) * nc * CHUNK, *a1 = a0 + (size_t)nc * CHUNK,
                          *b0 = img + (size_t)bj * nc * CHUNK;
      for (; c < nc && !*abort_flag; ++c) {
        const int st = c % NS, u = c / NS;
        if (u >= 1 && !wait(&sh.empty[st], (u - 1) & 1)) break;
        unsigned char *S = stages + (size_t)st * STAGE;
        mbar_arrive_expect_tx(&sh.full[st], STAGE);
        for (int k = 0; k < DIG; ++k) {  // a digit's 128 rows side by side
          bulk_g2s(S + (2 * k) * TILE, a0 + (size_t)c * CHUNK + k * TILE, TILE, &sh.full[st]);
          bulk_g2s(S + (2 * k + 1) * TILE, a1 + (size_t)c * CHUNK + k * TILE, TILE, &sh.full[st]);
        }
        bulk_g2s(S + 2 * CHUNK, b0 + (size_t)c * CHUNK, CHUNK, &sh.full[st]);
      }
      // no copy may still be landing when the CTA exits
      for (int st = 0; st < NS && st < c; ++st) {
        const int last = (c - 1 - st) / NS * NS + st;
        mbar_wait_bounded(&sh.full[st], (last / NS) & 1, kWait);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      for (int kb = 0; kb < nkb && !*abort_flag; ++kb) {
        if (kb >= 1 && !wait(&sh.acc_empty, (kb - 1) & 1)) break;
        tc::fence_after();
        const int c1 = min(nc, (kb + 1) * KB);
        for (int c = kb * KB; c < c1; ++c) {
          const int st = c % NS;
          if (!wait(&sh.full[st], (c / NS) & 1)) break;
          tc::fence_after();
          // operand images as lower descriptor words (offsets in 16 bytes)
          const uint32_t A = tc::desc_lo(smem_u32(stages + (size_t)st * STAGE)), B = A + 2 * CHUNK / 16;
          // digit i of A against the digits j <= 7 - i of B: their tiles lie
          // side by side, as do the accumulators of the classes i + j, so
          // four of them are one MMA of 256 columns
#pragma unroll
          for (int i = 0; i < DIG; ++i) {
#pragma unroll
            for (int j = 0; i + j < DIG; j += 4) {
              // classes 0..3 are read every other block only
              const uint32_t acc = c > kb * KB || i > 0 || (j == 0 && (kb & 1)) ? 1u : 0u;
              const int w = i + j + 4 <= DIG ? 4 : DIG - i - j;
              tc::mma_bf16<tc::desc_hi(SBO)>(tmem + (i + j) * RB, A + 2 * i * TILE / 16, B + j * TILE / 16,
                                             tc::idesc_bf16(128, w * RB), acc);
            }
          }
          tc::mma_commit(&sh.empty[st]);
          if (c == c1 - 1) tc::mma_commit(&sh.acc_full);
        }
      }
      tc::mma_commit(&sh.drain);
      mbar_wait_bounded(&sh.drain, 0, kWait);
    }
  } else {
    const int q = warp & 3, part = (warp - 2) >> 2;
    const uint32_t at = tmem + ((uint32_t)(q * 32) << 16) + part * 16;
    long long hi[16], lo[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) hi[i] = lo[i] = 0;
    bool ok = true;
    for (int kb = 0; kb < nkb && ok; ++kb) {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sh.acc_full, kb & 1, kWait));
      if (!ok) {
        if (lane == 0) {
          atomicExch(err, DSE_ETIMEOUT);
          *abort_flag = 1;
        }
        break;
      }
      tc::fence_after();
      // hi counts in units of 2^-40, lo of 2^-72 (class s: 2^(-8 (s + 2))).
      // Classes 0..3 add at most 4 products a sample: two blocks of them fit.
      // A class is converted while the next one's columns are on their way; the
      // conversions (16 a clock and SM, 4096 cycles for all classes) bound the
      // drain, in which the products wait.  (Eight warps of 32 columns, every
      // class each time: 361 us a launch for n = 3000, N = 1000; 311 so.)
      uint32_t v[2][16];
      const bool all = (kb & 1) || kb + 1 == nkb;
      tc::tmem_ld16_start(at + (all ? 0 : 4 * RB), v[0]);
#pragma unroll
      for (int s = 0; s < DIG; ++s) {
        if (s < 4 && !all) continue;
        tc::tmem_ld16_wait(v[s & 1]);
        if (s + 1 < DIG) tc::tmem_ld16_start(at + (s + 1) * RB, v[(s + 1) & 1]);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int d = __float2int_rn(__uint_as_float(v[s & 1][i])), unit = 1 << (BITS * (3 - (s & 3)));
          long long &sum = s < 4 ? hi[i] : lo[i];
          asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(sum) : "r"(d), "r"(unit));
        }
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.acc_empty);
    }
    const int64_t i = (int64_t)bi * 128 + q * 32 + lane, j0 = (int64_t)bj * RB + part * 16;
    const int ei = i < n ? ex[i] : INT32_MIN;
    if (ok) {
      // A sample adds at most (1 + 2/2^8 + 3/2^16 + ..) 2^38 to hi and (5 +
      // 6/2^8 + ..) 2^38 to lo, which hands over what it holds above 2^32:
      // PANEL samples of hi stay below 2^52.1, as wide_to_double wants it.
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int64_t j = j0 + k;
        if (i < n && j < n && i <= j) {
          const int ej = ex[j];
          // hi takes over what lo holds above its own unit
          const long long h = hi[k] + (lo[k] >> 32);
          const uint32_t l = (uint32_t)lo[k];
          // scaled by the columns' powers of two (a zero column has digits 0)
          const int e = (ei == INT32_MIN ? 0 : ei) + (ej == INT32_MIN ? 0 : ej);
          const bool plain = e > -900 && e < 900;
          double g = wide_to_double(h, l, (plain ? e : 0) - 72);
          if (!plain) g = scalbn(g, e);
          // what l adds is below 2^-40, against 2^-4 for the product of the columns' norms at least
          float f = __ll2float_rn(h) * 0x1p-40f;
          const int64_t at_g = upper ? i * n + j : j * n + i;
          if (add) {
            g += Gm[at_g];
            if (G32) f = (float)(plain ? g * __longlong_as_double((long long)(1023 - e) << 52) : scalbn(g, -e));
          }
          Gm[at_g] = g;
          if (G32) G32[at_g] = f;
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  __syncwarp();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// Per candidate, for the scan: the pivot test, its FP64 root L, z = b / L and
// q = z^2 (valid < 0: the candidate is rejected), and the scale-free FP32
// forms w = 2^e / L (so that G32 w w is the correlation) and cr = z / sqrt(Syy) (0 for a
// constant target: every subset then explains nothing, and all are taken).
struct Cand {
  const double *L, *z, *q;
  const float *w, *cr;
};
__global__ void k_l0_cands(const double *Gm, const int *ex, const double *b, const double *nrm2, int64_t n,
                           const double *syy, double *L, double *z, double *q, float *w, float *cr) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const double g = Gm[p * n + p];
  const bool ok = g > kRank2 * nrm2[p];
  const double l = ok ? sqrt(g) : 1.0, zz = ok ? b[p] / l : 0.0;
  L[p] = l;
  z[p] = zz;
  q[p] = ok ? zz * zz : -1.0;
  w[p] = ok ? (float)scalbn(1.0 / l, ex[p]) : 0.f;
  cr[p] = ok && *syy > 0.0 ? (float)(zz / sqrt(*syy)) : 0.f;
}

// (q, subset) ordering: larger explained q first, then positions ascending
// (packed 21 bits each, lexicographic as one integer).
struct Hit {
  double q;
  uint64_t key;
};
// (q >= 0, or -1 for none: the bits as integers order alike, and FP64 compares
// are slow on this part)
__device__ __forceinline__ bool better(double qa, uint64_t ka, double qb, uint64_t kb) {
  const long long a = __double_as_longlong(qa), b = __double_as_longlong(qb);
  return a > b || (a == b && ka < kb);
}
__device__ __forceinline__ uint64_t pack3(int64_t p0, int64_t p1, int64_t p2) {
  return ((uint64_t)p0 << 42) | ((uint64_t)p1 << 21) | (uint64_t)p2;
}

// A warp's 32 best, one per lane: insert the lanes' candidates in `pass`.
struct WarpTop {
  double q;       // this lane's slot
  uint64_t key;
  double wq;      // the warp's worst slot (broadcast)
  uint64_t wkey;
  int wlane;
  __device__ void init() {
    q = -1.0;
    key = ~0ull;
    wq = -1.0;
    wkey = ~0ull;
    wlane = 0;
  }
  __device__ void worst() {
    // argmin over lanes of the ordering
    double mq = q;
    uint64_t mk = key;
    int ml = threadIdx.x & 31;
    for (int o = 16; o > 0; o >>= 1) {
      const double oq = __shfl_xor_sync(0xffffffffu, mq, o);
      const uint64_t ok = __shfl_xor_sync(0xffffffffu, mk, o);
      const int ol = __shfl_xor_sync(0xffffffffu, ml, o);
      if (better(mq, mk, oq, ok) || (mq == oq && mk == ok && ol < ml)) {
        mq = oq;
        mk = ok;
        ml = ol;
      }
    }
    wq = mq;
    wkey = mk;
    wlane = ml;
  }
  // every lane calls; cq/ck are this lane's candidate, valid if `has`
  __device__ void offer(bool has, double cq, uint64_t ck) {
    const int lane = threadIdx.x & 31;
    unsigned m = __ballot_sync(0xffffffffu, has && better(cq, ck, wq, wkey));
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      const double sq = __shfl_sync(0xffffffffu, cq, src);
      const uint64_t sk = __shfl_sync(0xffffffffu, ck, src);
      if (better(sq, sk, wq, wkey)) {
        if (lane == wlane) {
          q = sq;
          key = sk;
        }
        worst();
      }
    }
  }
};

// Explained sum of squares of the subset, in position order (p0 < p1 < p2):
// incremental Cholesky of the centred Gram submatrix; -1 if a pivot fails
// the rank rule.  g..: the subset's Gram entries.
__device__ __forceinline__ double explained1(double g, double b, double nrm2, double *L11, double *z1) {
  if (!(g > kRank2 * nrm2)) return -1.0;
  *L11 = sqrt(g);
  *z1 = b / *L11;
  return *z1 * *z1;
}
__device__ __forceinline__ double explained2(double q1, double L11, double z1, double g10, double g11, double b1,
                                             double nrm2) {
  const double L21 = g10 / L11;
  const double d = g11 - L21 * L21;
  if (!(d > kRank2 * nrm2)) return -1.0;
  const double z2 = (b1 - L21 * z1) / sqrt(d);
  return q1 + z2 * z2;
}
struct Step2 {  // the state after two pivots
  double L21, z1, z2, q2, i11, i22;
};
__device__ __forceinline__ bool two_pivots(double q1, double L11, double z1, double g10, double g11, double b1,
                                           double nrm2, Step2 *o) {
  o->L21 = g10 / L11;
  const double d2 = g11 - o->L21 * o->L21;
  if (!(d2 > kRank2 * nrm2)) return false;
  const double L22 = sqrt(d2);
  o->z1 = z1;
  o->z2 = (b1 - o->L21 * z1) / L22;
  o->q2 = q1 + o->z2 * o->z2;
  o->i11 = 1.0 / L11;
  o->i22 = 1.0 / L22;
  return true;
}
__device__ __forceinline__ double explained3(const Step2 &s, double g20, double g21, double g22, double b2,
                                             double nrm2) {
  const double L31 = g20 * s.i11;
  const double L32 = (g21 - L31 * s.L21) * s.i22;
  const double d3 = g22 - L31 * L31 - L32 * L32;
  if (!(d3 > kRank2 * nrm2)) return -1.0;
  const double t = b2 - L31 * s.z1 - L32 * s.z2;
  return s.q2 + t * t / d3;
}

// Scan of every D-subset; each block writes its kTop best to out[block].
// An FP32 bound of q / Syy from the candidates' correlations excludes nearly
// every subset.  A correlation G32 w w has five roundings of 2^-24 (G32, both
// w, two products) and what G32 leaves of the entry, 2^-36 of the norms'
// product: within 5e-7.  Pairs: 1 - r^2 is within 1.1e-6 and the numerator
// within 1e-6.  Triples, where 1 - r^2 > 1e-2: its reciprocal root is within
// 5.6e-5 of itself, the second row within 7.3e-5, the last pivot within
// 1.5e-4 and the numerator within 1.4e-4.  The margins below are wider; where
// a pivot is smaller the bound is not used.  The exact evaluation of each
// (about 12 FP64
// operations, two divisions and a root) took 0.96 ms for 4.5 M pairs (0.15 now).
// `floor`: the best 32nd-best q of any warp so far; a subset below it by
// more than 1e-9 cannot be among the kMore best that matter.  Without BOUND
// (little memory: no G32) every subset is evaluated exactly.
template <int D, bool BOUND>
__global__ void __launch_bounds__(256) k_l0_scan(const double *Gm, const float *G32, const double *b,
                                                 const double *nrm2, const Cand C, const double *syy, int64_t n,
                                                 unsigned long long *floor_bits, Hit *out) {
  pdl_enter();
  __shared__ Hit sh[8 * 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WarpTop top;
  top.init();
  // what a bound has to reach, as a share of Syy (one rounding up)
  const double isyy = *syy > 0.0 ? 1.0 / *syy : 0.0;
  float need = -1.f;
  auto renew = [&]() {
    unsigned long long f = 0;
    if (lane == 0) {
      if (top.wq > 0.0) atomicMax(floor_bits, (unsigned long long)__double_as_longlong(top.wq));
      f = *(volatile unsigned long long *)floor_bits;
    }
    f = __shfl_sync(0xffffffffu, f, 0);
    const double q = fmax(top.wq, __longlong_as_double((long long)f));
    need = q > 0.0 && isyy > 0.0 ? (float)(q * isyy) * (1.0f - 1e-6f) : -1.f;
  };
  if (D == 1) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t base0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t base = base0 - lane; base < n; base += stride) {
      const int64_t p = base + lane;
      const double q = p < n ? C.q[p] : -1.0;
      top.offer(q >= 0.0, q, pack3(p, 0, 0));
    }
  } else if (D == 2) {
    const uint64_t npairs = (uint64_t)n * (uint64_t)(n - 1) / 2;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t base0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x - lane;
    int turn = 0;
    for (uint64_t base = base0; base < npairs; base += stride) {
      const uint64_t idx = base + lane;
      if ((++turn & 15) == 0) renew();
      bool maybe = idx < npairs;
      int64_t p0 = 0, p1 = 0;
      if (maybe) {
        uint64_t hi, lo;
        pair_from_index(idx, &hi, &lo);  // lo < hi
        p0 = (int64_t)lo, p1 = (int64_t)hi;
      }
      if (BOUND && maybe) {
        const float r = G32[p1 * n + p0] * C.w[p0] * C.w[p1], c0 = C.cr[p0];
        const float d = fmaf(-r, r, 1.0f), x = fabsf(fmaf(-r, c0, C.cr[p1])) + 2e-6f;
        // (a NaN excludes nothing)
        maybe = !(d > 1e-3f) || !(fmaf(c0, c0, x * x / (d - 4e-6f)) * (1.0f + 1e-5f) + 1e-6f < need);
      }
      if (!__any_sync(0xffffffffu, maybe)) continue;
      double q = -1.0;
      if (maybe && C.q[p0] >= 0.0)
        q = explained2(C.q[p0], C.L[p0], C.z[p0], Gm[p1 * n + p0], Gm[p1 * n + p1], b[p1], nrm2[p1]);
      const double before = top.wq;
      top.offer(q >= 0.0, q, pack3(p0, p1, 0));
      if (top.wq != before) renew();
    }
  } else {
    // warp per pair (p0 < p1); lanes over p2 > p1
    const uint64_t npairs = (uint64_t)n * (uint64_t)(n - 1) / 2;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    int turn = 0;
    for (uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < npairs; w += warps) {
      uint64_t hi, lo;
      pair_from_index(w, &hi, &lo);
      const int64_t p0 = (int64_t)lo, p1 = (int64_t)hi;
      if ((++turn & 7) == 0) renew();
      if (p1 + 1 >= n || C.q[p0] < 0.0) continue;
      // the FP32 forms of the two pivots; the exact ones at the first need
      const float *f0 = G32 + p0 * n, *f1 = G32 + p1 * n;
      const float w0 = C.w[p0], w1 = C.w[p1], c0 = C.cr[p0];
      const float r = BOUND ? f0[p1] * w0 * w1 : 1.0f, d2 = fmaf(-r, r, 1.0f);
      const bool fine = d2 > 1e-2f;
      const float i2 = fine ? rsqrtf(d2) : 0.f, c1 = fmaf(-r, c0, C.cr[p1]) * i2, q2 = fmaf(c0, c0, c1 * c1);
      bool have = false, bad = false;
      Step2 st;
      for (int64_t base = p1 + 1; base < n && !bad; base += 32) {
        const int64_t p2 = base + lane;
        bool maybe = p2 < n;
        if (BOUND && maybe && fine) {
          const float w2 = C.w[p2], l1 = f0[p2] * w0 * w2, l2 = fmaf(-l1, r, f1[p2] * w1 * w2) * i2;
          const float d3 = fmaf(-l2, l2, fmaf(-l1, l1, 1.0f));
          const float x = fabsf(fmaf(-l2, c1, fmaf(-l1, c0, C.cr[p2]))) + 2e-4f;
          maybe = !(d3 > 1e-2f) || !((q2 + x * x / (d3 - 2e-4f)) * (1.0f + 1e-5f) + 3e-4f < need);
        }
        if (!__any_sync(0xffffffffu, maybe)) continue;
        if (!have) {
          have = true;
          bad = !two_pivots(C.q[p0], C.L[p0], C.z[p0], Gm[p0 * n + p1], Gm[p1 * n + p1], b[p1], nrm2[p1], &st);
          if (bad) break;
        }
        double q = -1.0;
        if (maybe) q = explained3(st, Gm[p0 * n + p2], Gm[p1 * n + p2], Gm[p2 * n + p2], b[p2], nrm2[p2]);
        const double before = top.wq;
        top.offer(q >= 0.0, q, pack3(p0, p1, p2));
        if (top.wq != before) renew();
      }
    }
  }
  // the block's kTop best: sort the 8 warps' 256 entries
  sh[warp * 32 + lane] = Hit{top.q, top.key};
  __syncthreads();
  for (int size = 2; size <= 256; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const int i = threadIdx.x, j = i ^ stride;
      if (j > i) {
        const bool up = (i & size) == 0;
        const Hit a = sh[i], c = sh[j];
        const bool sw = up ? better(c.q, c.key, a.q, a.key) : better(a.q, a.key, c.q, c.key);
        if (sw) {
          sh[i] = c;
          sh[j] = a;
        }
      }
      __syncthreads();
    }
  if (threadIdx.x < kTop) out[(size_t)blockIdx.x * kTop + threadIdx.x] = sh[threadIdx.x];
}

// The kMore best of all blocks' lists (one block): each warp's 32 best of its
// share, then a sort of the warps' 1024.  Entries clearly below the floor are
// passed over.  (A sort of all 8192 entries took 0.43 ms; 0.10.)
__global__ void __launch_bounds__(1024) k_l0_merge(const Hit *in, int64_t m, const unsigned long long *floor_bits,
                                                   Hit *best) {
  pdl_enter();
  __shared__ Hit hs[1024];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double floor_q = __longlong_as_double((long long)*floor_bits) * (1.0 - 1e-9);
  WarpTop top;
  top.init();
  for (int64_t base = (int64_t)warp * 32; base < m; base += 1024) {
    const Hit h = base + lane < m ? in[base + lane] : Hit{-1.0, ~0ull};
    top.offer(h.q >= floor_q, h.q, h.key);
  }
  hs[threadIdx.x] = Hit{top.q, top.key};
  __syncthreads();
  for (int size = 2; size <= 1024; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const int i = threadIdx.x, j = i ^ stride;
      if (j > i) {
        const bool up = (i & size) == 0;
        const Hit a = hs[i], c = hs[j];
        const bool sw = up ? better(c.q, c.key, a.q, a.key) : better(a.q, a.key, c.q, c.key);
        if (sw) {
          hs[i] = c;
          hs[j] = a;
        }
      }
      __syncthreads();
    }
  if (threadIdx.x < kMore) best[threadIdx.x] = hs[threadIdx.x];
}

// The kept subsets' Gram entries (00, 10, 11, 20, 21, 22) in plain FP64, the
// samples in order, and their q from them (one warp each): what decides and
// is reported does not depend on the slicing.
__global__ void __launch_bounds__(32) k_l0_exact(Hit *best, int D, const double *X, const double *b,
                                                 const double *nrm2, int64_t N, double *ge) {
  pdl_enter();
  __shared__ double xs[3][64];
  const int lane = threadIdx.x;
  const Hit h = best[blockIdx.x];
  const int64_t p[3] = {(int64_t)((h.key >> 42) & 0x1FFFFF), (int64_t)((h.key >> 21) & 0x1FFFFF),
                        (int64_t)(h.key & 0x1FFFFF)};
  if (!(h.q >= 0.0)) return;
  const int ne = D * (D + 1) / 2, e = lane < ne ? lane : 0;
  const int r = e == 0 ? 0 : e < 3 ? 1 : 2, c = e == 0 || e == 1 || e == 3 ? 0 : e == 5 ? 2 : 1;
  double acc = 0.0;
  for (int64_t s0 = 0; s0 < N; s0 += 64) {
    __syncwarp();
    for (int d = 0; d < D; ++d)
      for (int i = lane; i < 64; i += 32) xs[d][i] = s0 + i < N ? X[p[d] * N + s0 + i] : 0.0;
    __syncwarp();
#pragma unroll 8
    for (int i = 0; i < 64; ++i) acc = fma(xs[c][i], xs[r][i], acc);
  }
  double g[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) g[k] = __shfl_sync(0xffffffffu, acc, k);
  if (lane == 0) {
    for (int k = 0; k < ne; ++k) ge[(size_t)blockIdx.x * 6 + k] = g[k];
    double L11, z1;
    double q = explained1(g[0], b[p[0]], nrm2[p[0]], &L11, &z1);
    if (q >= 0.0 && D == 2) q = explained2(q, L11, z1, g[1], g[2], b[p[1]], nrm2[p[1]]);
    if (q >= 0.0 && D == 3) {
      Step2 st;
      q = two_pivots(q, L11, z1, g[1], g[2], b[p[1]], nrm2[p[1]], &st)
              ? explained3(st, g[3], g[4], g[5], b[p[2]], nrm2[p[2]])
              : -1.0;
    }
    best[blockIdx.x].q = q;
  }
}

// Explicit FP64 refit of each kept subset (one block each): coefficients
// from the centred Cholesky, RMSE of the explicit residual.
__global__ void __launch_bounds__(kCol) k_l0_refit(const Hit *best, int D, const double *X, const double *yc,
                                                   const double *mean, const double *ge, const double *b,
                                                   const double *nrm2, int64_t N, double my, double *rmse,
                                                   double *coef) {
  pdl_enter();
  __shared__ double sm[(kCol / 32) * 2];
  const Hit h = best[blockIdx.x];
  int64_t p[3];
  p[0] = (int64_t)((h.key >> 42) & 0x1FFFFF);
  p[1] = (int64_t)((h.key >> 21) & 0x1FFFFF);
  p[2] = (int64_t)(h.key & 0x1FFFFF);
  bool ok = h.q >= 0.0;
  const double *g = ge + (size_t)blockIdx.x * 6;
  double beta[4] = {0, 0, 0, 0};
  if (ok) {
    double L[3][3] = {}, z[3];
    for (int c = 0; c < D && ok; ++c) {
      double dsum = g[c * (c + 1) / 2 + c];
      for (int k = 0; k < c; ++k) dsum -= L[c][k] * L[c][k];
      if (!(dsum > kRank2 * nrm2[p[c]])) {
        ok = false;
        break;
      }
      L[c][c] = sqrt(dsum);
      for (int r = c + 1; r < D; ++r) {
        double v = g[r * (r + 1) / 2 + c];
        for (int k = 0; k < c; ++k) v -= L[r][k] * L[c][k];
        L[r][c] = v / L[c][c];
      }
    }
    if (ok) {
      for (int c = 0; c < D; ++c) {
        double v = b[p[c]];
        for (int k = 0; k < c; ++k) v -= L[c][k] * z[k];
        z[c] = v / L[c][c];
      }
      for (int c = D - 1; c >= 0; --c) {
        double v = z[c];
        for (int k = c + 1; k < D; ++k) v -= L[k][c] * beta[k + 1];
        beta[c + 1] = v / L[c][c];
      }
      double b0 = my;
      for (int c = 0; c < D; ++c) b0 -= beta[c + 1] * mean[p[c]];
      beta[0] = b0;
    }
  }
  double rss[1] = {0.0};
  if (ok)
    for (int64_t s = threadIdx.x; s < N; s += kCol) {
      double r = yc[s];
      for (int c = 0; c < D; ++c) r = fma(-beta[c + 1], X[p[c] * N + s], r);
      rss[0] = fma(r, r, rss[0]);
    }
  block_sum<1>(rss, sm);
  if (threadIdx.x == 0) {
    rmse[blockIdx.x] = ok ? sqrt(rss[0] / (double)N) : INFINITY;
    for (int c = 0; c < 4; ++c) coef[blockIdx.x * 4 + c] = ok ? beta[c] : 0.0;
  }
}

}  // namespace

dse_status l0_search_impl(dse_space *sp, const dse_l0_desc *d, int64_t *top_pos, double *top_rmse, double *top_coefs,
                          int32_t *n_found) {
  cudaStream_t st = (cudaStream_t)d->stream;
  const int64_t n = d->n_ids, N = sp->N;
  const int D = d->dim;
  const uint64_t total = (uint64_t)sp->n + sp->geom.slots;
  if (!d->ids_on_device)
    for (int64_t i = 0; i < n; ++i)
      if (d->ids[i] >= total) {
        set_error("candidate id %llu out of range", (unsigned long long)d->ids[i]);
        return DSE_ERANGE;
      }
  // digit images: panels of samples, 16 n bytes a sample, 2 GB at most.  Where
  // this and the Gram matrix's FP32 copy do not fit, the shortest panel (one
  // exact block of samples) and no copy.
  const int nblk = 2 * (int)((n + 127) / 128);
  constexpr int64_t kBlock = sliced::KB * sliced::KC;
  const int64_t fit = std::max<int64_t>(kBlock, ((int64_t)2 << 30) / (16 * 64 * (int64_t)nblk) / kBlock * kBlock);
  int64_t panel = std::min<int64_t>(std::min<int64_t>(fit, sliced::PANEL), (N + kBlock - 1) / kBlock * kBlock);
  const int sms = sm_count();
  const int nb = std::min<int64_t>(2 * sms, 8192 / kTop);  // scan blocks (their kTop bests fit the merge)
  // scratch
  double *yd = nullptr, *yc = nullptr, *syy = nullptr, *ym = nullptr, *X = nullptr, *nrm2 = nullptr, *bv = nullptr, *mean = nullptr,
         *Gm = nullptr, *rm = nullptr, *cf = nullptr, *cL = nullptr, *cz = nullptr, *cq = nullptr, *ge = nullptr;
  float *G32 = nullptr, *cw = nullptr, *cc = nullptr;
  int *ex = nullptr, *err = nullptr;
  unsigned char *img = nullptr;
  unsigned long long *floor_bits = nullptr;
  uint64_t *ids = nullptr;
  Hit *part = nullptr, *best = nullptr;
  Scratch sc;
  if (!d->y_on_device) sc.add(&yd, (size_t)N);
  if (!d->ids_on_device) sc.add(&ids, (size_t)n);
  sc.add(&yc, (size_t)N);
  sc.add(&syy, 1);
  sc.add(&ym, 1);
  sc.add(&X, (size_t)n * N);
  sc.add(&nrm2, (size_t)n);
  sc.add(&bv, (size_t)n);
  sc.add(&mean, (size_t)n);
  sc.add(&Gm, (size_t)n * n);
  sc.add(&part, (size_t)nb * kTop);
  sc.add(&best, kMore);
  sc.add(&ex, (size_t)n);
  sc.add(&cL, (size_t)n);
  sc.add(&cz, (size_t)n);
  sc.add(&cq, (size_t)n);
  sc.add(&cw, (size_t)n);
  sc.add(&cc, (size_t)n);
  sc.add(&ge, (size_t)kMore * 6);
  sc.add(&floor_bits, 2);
  sc.add(&rm, kMore);
  sc.add(&cf, (size_t)kMore * 4);
  void *base = nullptr;
  size_t bytes = 0;
  auto allocate = [&](bool copy) {
    Scratch all = sc;
    if (copy) all.add(&G32, (size_t)n * n);
    all.add(&img, (size_t)nblk * (size_t)(panel / sliced::KC) * sliced::CHUNK);
    return all.alloc(&base, &bytes);
  };
  dse_status as = allocate(true);
  if (as == DSE_ENOMEM) {
    clear_error();
    panel = kBlock;
    G32 = nullptr;
    as = allocate(false);
  }
  DSE_TRY(as);
  struct Free {
    void *p;
    ~Free() { dfree(p); }
  } fr{base};
  const double *y = d->y;
  if (!d->y_on_device) {
    DSE_CUDA(cudaMemcpyAsync(yd, d->y, 8 * N, cudaMemcpyHostToDevice, st));
    y = yd;
  }
  const uint64_t *idp = d->ids;
  if (!d->ids_on_device) {
    DSE_CUDA(cudaMemcpyAsync(ids, d->ids, 8 * n, cudaMemcpyHostToDevice, st));
    idp = ids;
  }
  const FeatTable F = table_of(sp);
  err = reinterpret_cast<int *>(floor_bits + 1);
  DSE_CUDA(cudaMemsetAsync(floor_bits, 0, 16, st));
  static bool attr[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr[dev & 63]) {
    DSE_CUDA(cudaFuncSetAttribute(k_l0_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sliced::SMEM));
    attr[dev & 63] = true;
  }
  note_launches(8);
  launch_k(k_l0_target, 1, kCol, 0, st, y, N, yc, syy, ym);
  launch_k(k_l0_columns, (unsigned)n, kCol, 0, st, F, sp->geom, sp->n, idp, n, yc, X, nrm2, bv, mean);
  launch_k(k_l0_exponents, (unsigned)n, kCol, 0, st, X, N, ex);
  const int64_t hb2 = nblk / 2, tiles = hb2 * (nblk + 1 - hb2);  // i-blocks 0..nblk/2 - 1 (see k_l0_gram)
  for (int64_t s0 = 0; s0 < N; s0 += panel) {
    const int64_t ns = std::min(panel, N - s0);
    const int nc = (int)((ns + sliced::KC - 1) / sliced::KC);
    note_launches(2);
    launch_k(k_l0_slices, dim3((unsigned)nc, (unsigned)nblk), 128, 0, st, X, ex, n, N, s0, ns, nc, img);
    launch_k(k_l0_gram, (unsigned)tiles, sliced::THREADS, sliced::SMEM, st, img, ex, n, nc, s0 > 0 ? 1 : 0, D == 3 ? 1 : 0, Gm, G32, err);
  }
  launch_k(k_l0_cands, (unsigned)((n + 127) / 128), 128, 0, st, Gm, ex, bv, nrm2, n, syy, cL, cz, cq, cw, cc);
  const Cand cands{cL, cz, cq, cw, cc};
  auto scan = [&](auto kernel) { launch_k(kernel, nb, 256, 0, st, Gm, G32, bv, nrm2, cands, syy, n, floor_bits, part); };
  if (D == 1) scan(k_l0_scan<1, false>);
  else if (D == 2) G32 ? scan(k_l0_scan<2, true>) : scan(k_l0_scan<2, false>);
  else G32 ? scan(k_l0_scan<3, true>) : scan(k_l0_scan<3, false>);
  launch_k(k_l0_merge, 1, 1024, 0, st, part, (int64_t)nb * kTop, floor_bits, best);
  launch_k(k_l0_exact, kMore, 32, 0, st, best, D, X, bv, nrm2, N, ge);
  launch_k(k_l0_refit, kMore, kCol, 0, st, best, D, X, yc, mean, ge, bv, nrm2, N, 0.0, rm, cf);
  DSE_CUDA(cudaGetLastError());
  // reports: RMSEs, coefficients (intercept without the target's mean), the
  // subsets and the target's mean, one wait
  double *hs = static_cast<double *>(pinned_staging(8 * (kMore * 5 + 2) + sizeof(Hit) * kMore));
  if (!hs) return DSE_ENOMEM;
  Hit *hb = reinterpret_cast<Hit *>(hs + kMore * 5 + 2);
  DSE_CUDA(cudaMemcpyAsync(hs, rm, 8 * kMore, cudaMemcpyDeviceToHost, st));
  DSE_CUDA(cudaMemcpyAsync(hs + kMore, cf, 8 * kMore * 4, cudaMemcpyDeviceToHost, st));
  DSE_CUDA(cudaMemcpyAsync(hs + kMore * 5, ym, 8, cudaMemcpyDeviceToHost, st));
  DSE_CUDA(cudaMemcpyAsync(hs + kMore * 5 + 1, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  DSE_CUDA(cudaMemcpyAsync(hb, best, sizeof(Hit) * kMore, cudaMemcpyDeviceToHost, st));
  DSE_CUDA(cudaStreamSynchronize(st));
  if (*reinterpret_cast<const int *>(hs + kMore * 5 + 1)) {
    set_error("a bounded device wait timed out");
    return DSE_ETIMEOUT;
  }
  const double my = hs[kMore * 5];
  struct Row {
    double q, rmse;
    uint64_t key;
    int64_t p[3];
    double c[4];
  };
  std::vector<Row> rows;
  for (int i = 0; i < kMore; ++i) {
    if (!(hb[i].q >= 0.0)) continue;
    Row r;
    r.q = hb[i].q;
    r.rmse = hs[i];
    r.key = hb[i].key;
    r.p[0] = (int64_t)((hb[i].key >> 42) & 0x1FFFFF);
    r.p[1] = (int64_t)((hb[i].key >> 21) & 0x1FFFFF);
    r.p[2] = (int64_t)(hb[i].key & 0x1FFFFF);
    for (int c = 0; c < 4; ++c) r.c[c] = hs[kMore + i * 4 + c];
    r.c[0] += my;
    rows.push_back(r);
  }
  // the kTop of largest q; of those the full-rank fits, by RMSE
  std::sort(rows.begin(), rows.end(), [](const Row &a, const Row &c) { return a.q > c.q || (a.q == c.q && a.key < c.key); });
  if (rows.size() > (size_t)kTop) rows.resize(kTop);
  rows.erase(std::remove_if(rows.begin(), rows.end(), [](const Row &r) { return !(r.rmse < INFINITY); }), rows.end());
  std::sort(rows.begin(), rows.end(), [&](const Row &a, const Row &c) {
    if (a.rmse != c.rmse) return a.rmse < c.rmse;
    for (int k = 0; k < D; ++k)
      if (a.p[k] != c.p[k]) return a.p[k] < c.p[k];
    return false;
  });
  const int nf = std::min<int>((int)rows.size(), d->n_top);
  for (int i = 0; i < nf; ++i) {
    if (top_pos)
      for (int k = 0; k < D; ++k) top_pos[i * D + k] = rows[i].p[k];
    if (top_rmse) top_rmse[i] = rows[i].rmse;
    if (top_coefs)
      for (int k = 0; k <= D; ++k) top_coefs[i * (D + 1) + k] = rows[i].c[k];
  }
  *n_found = nf;
  return DSE_OK;
}

}  // namespace dse

using namespace dse;

extern "C" dse_status dse_l0_search(dse_space *s, const dse_l0_desc *d, int64_t *top_pos, double *top_rmse,
                                    double *top_coefs, int32_t *n_found) {
  dse::NvtxRange nvtx_range_("dse_l0_search");
  clear_error();
  if (!s || !d || !d->y || !d->ids || !n_found || d->dim < 1 || d->dim > 3 || d->n_ids < d->dim ||
      d->n_ids > (1 << 16) || d->n_top < 1 || d->n_top > 32) {
    set_error("invalid L0 descriptor");
    return DSE_EINVAL;
  }
  *n_found = 0;
  DSE_TRY(check_device());
  AllocStream as((cudaStream_t)d->stream);
  return l0_search_impl(s, d, top_pos, top_rmse, top_coefs, n_found);
}
