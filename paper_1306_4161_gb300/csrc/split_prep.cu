// Split-precision path, the steps around the tensor-core products:
//   1. exponent scan   e_i = ilogb(max_k |A_ik|) + 2, f_j over the columns of B
//   2. slicing         S digits per entry, t_s = RN(r 2^(w s)) - 2^w RN(r 2^(w(s-1))),
//                      r = a 2^-e (round half to even), as int8 (w = 7) or bf16 (w = 9;
//                      8 for S = 7)
//   4. recombination   C_ij = RN(2^(e_i+f_j) sum_d D_d,ij 2^(-w d)), exact sum in
//                      128-bit integers, rounded once to binary64
// Binary64 arithmetic is the slowest unit of this GPU; none of them needs it.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "digits.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "round_scaled.cuh"
#include "../../include/hsumma.h"

namespace hs {
namespace {

// max over |x| by bit pattern (non-negative doubles order like their bits)
__device__ __forceinline__ unsigned long long absbits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// exponent e (ilogb + 2) from the largest |x| bit pattern; flags Inf/NaN
__device__ __forceinline__ int exponent_from_bits(unsigned long long b, bool *nonfinite) {
  const int E = (int)(b >> 52);
  if (E == 0x7FF) {
    *nonfinite = true;
    return 0;
  }
  if (b == 0) return 0;
  int ilogb;
  if (E > 0)
    ilogb = E - 1023;
  else
    ilogb = (63 - __clzll((long long)(b & 0xFFFFFFFFFFFFFull))) - 1074;
  return ilogb + 2;
}

// rows of A: one warp per row
__global__ void exponents_rows_kernel(const double *__restrict__ A, int64_t lda, int64_t M,
                                      int64_t K, int32_t *__restrict__ e, int *status) {
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const double *a = A + row * lda;
  unsigned long long m = 0;
  if ((reinterpret_cast<uintptr_t>(a) & 15) == 0) {
    // 16-byte aligned row: pairs
    const int64_t K2 = K & ~int64_t(1);
    for (int64_t k = 2 * lane; k < K2; k += 64) {
      const double2 v = *reinterpret_cast<const double2 *>(a + k);
      m = max(m, max(absbits(v.x), absbits(v.y)));
    }
    if ((K & 1) && lane == 0) m = max(m, absbits(a[K - 1]));
  } else {
    for (int64_t k = lane; k < K; k += 32) m = max(m, absbits(a[k]));
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    bool nf = false;
    e[row] = exponent_from_bits(m, &nf);
    if (nf) record_error(status, HSUMMA_ERR_NONFINITE, kSiteNonFinite);
  }
}

// columns of B: a block covers 64 columns (32 lanes x 2) and one of the
// gridDim.y slices of k, its 8 warps splitting that slice; the gridDim.y blocks
// of a column group form one cluster (1 x gridDim.y), and its first CTA
// reduces their maxima through distributed shared memory.  Every thread
// reaches both cluster barriers.
__global__ void exponents_cols_kernel(const double *__restrict__ B, int64_t ldb, int64_t K,
                                      int64_t N, int32_t *__restrict__ f, int *status) {
  __shared__ unsigned long long part[8][64];
  __shared__ unsigned long long colmax[64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t j0 = (int64_t)blockIdx.x * 64 + 2 * lane;
  const int64_t kc = (K + gridDim.y - 1) / gridDim.y;
  const int64_t kb = (int64_t)blockIdx.y * kc, ke = kb + kc < K ? kb + kc : K;
  unsigned long long m0 = 0, m1 = 0;
  const bool pairs = ((reinterpret_cast<uintptr_t>(B) | (uintptr_t)(ldb * 8)) & 15) == 0;
  if (j0 + 1 < N && pairs) {
    for (int64_t k = kb + warp; k < ke; k += 8) {
      const double2 v = *reinterpret_cast<const double2 *>(B + k * ldb + j0);
      m0 = max(m0, absbits(v.x));
      m1 = max(m1, absbits(v.y));
    }
  } else {
    for (int64_t k = kb + warp; k < ke; k += 8) {
      if (j0 < N) m0 = max(m0, absbits(B[k * ldb + j0]));
      if (j0 + 1 < N) m1 = max(m1, absbits(B[k * ldb + j0 + 1]));
    }
  }
  part[warp][2 * lane] = m0;
  part[warp][2 * lane + 1] = m1;
  __syncthreads();
  if (threadIdx.x < 64) {
    unsigned long long m = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = max(m, part[w][threadIdx.x]);
    colmax[threadIdx.x] = m;
  }
  const bool split = gridDim.y > 1;
  if (split) cluster_sync();         // every CTA's colmax is written
  if (threadIdx.x < 64 && cluster_ctarank() == 0) {
    unsigned long long m = colmax[threadIdx.x];
    for (uint32_t r = 1; r < gridDim.y; ++r)
      m = max(m, ld_shared_cluster_u64(smem_u32(&colmax[threadIdx.x]), r));
    const int64_t j = (int64_t)blockIdx.x * 64 + threadIdx.x;
    if (j < N) {
      bool nf = false;
      f[j] = exponent_from_bits(m, &nf);
      if (nf) record_error(status, HSUMMA_ERR_NONFINITE, kSiteNonFinite);
    }
  }
  if (split) cluster_sync();         // the first CTA has read every colmax
}

// eight consecutive entries of a row (a) or column (b, step ldb) from k0 on, zeros past K
__device__ __forceinline__ void load_row8(const double *a, int64_t k0, int64_t K, double (&x)[8]) {
  a += k0;
  if (k0 + 7 < K && (reinterpret_cast<uintptr_t>(a) & 15) == 0) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const double2 v = reinterpret_cast<const double2 *>(a)[h];
      x[2 * h] = v.x;
      x[2 * h + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = k0 + u < K ? a[u] : 0.0;
  }
}
__device__ __forceinline__ void load_col8(const double *b, int64_t ldb, int64_t k0, int64_t K,
                                          double (&x)[8]) {
  b += k0 * ldb;
  if (k0 + 7 < K) {
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = __ldg(b + u * ldb);
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = k0 + u < K ? __ldg(b + u * ldb) : 0.0;
  }
}

// The digits of eight values, slice s stored at base + (s - 1) plane: bf16 (16
// bytes) or int8 (8 bytes).  With SQ (bf16) sq[s - 1] is the sum of the squares of
// slice s (exact), and nothing is stored at a null base.
template <bool BYTES, int W, bool SQ, int S>
__device__ __forceinline__ void store_digits(const double (&x)[8], int eb, uint8_t *base,
                                             int64_t plane, float *sq) {
  uint32_t v[S][4];   // slice s of values 2 h, 2 h + 1
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float a[S], b[S];
    digits<W, S>(x[2 * h], eb, a);
    digits<W, S>(x[2 * h + 1], eb, b);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      if (BYTES) {
        // low bytes of the integers
        v[s][h] = __byte_perm(__float_as_uint(a[s] + kRoundMagic),
                              __float_as_uint(b[s] + kRoundMagic), 0x0040);
      } else {
        const __nv_bfloat162 q = __floats2bfloat162_rn(a[s], b[s]);
        v[s][h] = *reinterpret_cast<const uint32_t *>(&q);
      }
      if (SQ) sq[s] = fmaf(b[s], b[s], fmaf(a[s], a[s], sq[s]));
    }
  }
  if (SQ && !base) return;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint8_t *dst = base + s * plane;
    if (BYTES)
      *reinterpret_cast<uint2 *>(dst) = make_uint2(__byte_perm(v[s][0], v[s][1], 0x5410),
                                                   __byte_perm(v[s][2], v[s][3], 0x5410));
    else
      *reinterpret_cast<uint4 *>(dst) = make_uint4(v[s][0], v[s][1], v[s][2], v[s][3]);
  }
}

// N values a lane (a power of two) summed over groups of N lanes, one sum a lane:
// at every step the lanes of a pair split the values they still hold.  With the
// sums then added over the groups, N = 4 over 16 lanes takes 5 shuffles, not 16.
template <int N>
__device__ __forceinline__ float spread_sums(float (&v)[N], int lane) {
  if constexpr (N > 1) {
    float r[N / 2];
    const bool up = lane & (N / 2);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const float keep = up ? v[N / 2 + i] : v[i], give = up ? v[i] : v[N / 2 + i];
      r[i] = keep + __shfl_xor_sync(0xffffffffu, give, N / 2);
    }
    return spread_sums<N / 2>(r, lane);
  } else {
    return v[0];
  }
}

// A slices: As[s][i][k], k < Kp (zero beyond K); each thread 8 consecutive k.
// S is a template parameter so that every digit's bit position is a constant.
template <int KIND, int S>
__global__ void __launch_bounds__(256) slices_rows_kernel(const double *__restrict__ A,
                                                          int64_t lda, int64_t M, int64_t K,
                                                          int64_t Kp,
                                                          const int32_t *__restrict__ e,
                                                          void *__restrict__ out) {
  constexpr int W = slice_width(KIND, S);
  constexpr bool BYTES = KIND == HSUMMA_INT8_SLICES;
  constexpr int EB = BYTES ? 1 : 2;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t groups = Kp / 8;
  if (gid >= M * groups) return;
  const int64_t i = gid / groups, k0 = (gid - i * groups) * 8;
  const int eb = e[i] + 1011;
  double x[8];
  load_row8(A + i * lda, k0, K, x);
  uint8_t *base = reinterpret_cast<uint8_t *>(out) + (i * Kp + k0) * EB;
  store_digits<BYTES, W, false, S>(x, eb, base, M * Kp * EB, nullptr);
}

// B slices, transposed: Bs[t][j][k].  A block covers 32 columns x 64 k; warp
// w takes 16 columns (w & 1) and 16 k (w >> 1), and lanes 2i and 2i + 1 take
// k .. k + 7 and k + 8 .. k + 15 of one column, so that a warp's store of a
// slice fills 16 whole 32-byte sectors (bf16) and its loads read 16
// consecutive doubles of each of 16 rows of B.  One-dimensional grid, column
// blocks fastest (neighbouring blocks read the same rows of B); any product
// whose slices fit in memory has fewer than 2^31 blocks.
template <int KIND, int S>
__global__ void __launch_bounds__(256)
    slices_cols_kernel(const double *__restrict__ B, int64_t ldb, int64_t K, int64_t N,
                       int64_t Kp, const int32_t *__restrict__ f, void *__restrict__ out) {
  constexpr int W = slice_width(KIND, S);
  constexpr bool BYTES = KIND == HSUMMA_INT8_SLICES;
  constexpr int EB = BYTES ? 1 : 2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t njb = (uint32_t)((N + 31) / 32);
  const uint32_t kb = blockIdx.x / njb, jb = blockIdx.x - kb * njb;
  const int64_t j = (int64_t)jb * 32 + (w & 1) * 16 + (lane >> 1);
  const int64_t k0 = (int64_t)kb * 64 + (w >> 1) * 16 + (lane & 1) * 8;
  if (j >= N) return;
  const int eb = f[j] + 1011;
  double x[8];
  load_col8(B + j, ldb, k0, K, x);
  uint8_t *base = reinterpret_cast<uint8_t *>(out) + (j * Kp + k0) * EB;
  store_digits<BYTES, W, false, S>(x, eb, base, N * Kp * EB, nullptr);
}

// Exponents and digits in one kernel, for the product kernel that recombines
// (digits as bf16 whatever the kind).  Both took four launches and read A and B
// twice from memory.  Before and now, with the events around them:
//   512^3, 4 slices 26 / 9 us;  3001 x 2047 x 2500, 5 slices 108 / 70 us;
//   4096^3, 4 slices 179 / 124 us;  16384^3 2.6 / 2.2 ms (1.3 ms for its 8.6 GB)
// It is bound by instruction issue (about 100 a value with 5 slices) and by its
// loads' latency in turn, so that four CTAs an SM (64 registers) are 15 % faster
// than three.
//
// Rows: a CTA of 8 warps takes 8 / wpr rows, wpr warps each; a warp's step is
// 256 k, 8 a lane.  Columns: a cluster takes 16 columns, its CTAs contiguous runs
// of windows of 128 k; a warp takes 16 k of a window, two lanes a column (a
// warp's store of a slice fills whole 32-byte sectors, its loads read 16
// consecutive doubles of 16 rows).  Either scans its part for the largest
// magnitudes, combines them (shared memory, the cluster's shared memory) and
// goes over the part again for the digits, backwards: the last step is still in
// registers, the others come back from the L2 (of 129 MB) as far as it holds what is
// under way: four CTAs on each of 152 SMs have 80 MB of rows or 159 MB of columns at
// 16384^2, so that there a part of the columns' second pass goes to memory.
// With 9-bit digits their squares are summed over windows of 128 k and a sum too
// large sets *big.
struct DigitsParams {
  const double *A, *B;
  int64_t lda, ldb, M, N, K, Kp;
  int64_t m1, n1;                  // this launch ends at row m1, column n1 ..
  int64_t m0, n0;                  // .. and starts at row m0, column n0
  int32_t *e, *f;
  uint8_t *As, *Bs;
  int row_ctas, wpr;               // CTAs for rows; warps a row (2^wlog)
  int wlog;
  int wins, kw;                    // windows of 128 k, and those of a CTA of a cluster
  int *big;
  unsigned long long *counters;    // cleared unless null
  int *status;
};

// What the exponent of a set of values needs: the largest high word of |x|, and
// where that is 0 (it then tells nothing) the leading bit of the low words.
struct Peak {
  uint32_t hi = 0, lo = 0;
  __device__ __forceinline__ void add(uint32_t h, uint32_t l) {
    hi = max(hi, h);
    lo |= l;
  }
  __device__ __forceinline__ void add8(const double (&x)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      add((uint32_t)__double2hiint(x[u]) & 0x7FFFFFFFu, (uint32_t)__double2loint(x[u]));
  }
  __device__ __forceinline__ int exponent(bool *nonfinite) const {
    return exponent_from_bits(hi ? (unsigned long long)hi << 32 : lo, nonfinite);
  }
};

template <int KIND, int S>
__global__ void __launch_bounds__(256, 4) digits_kernel(const __grid_constant__ DigitsParams p) {
  constexpr int W = slice_width(KIND, S);
  constexpr bool SQ = W == 9;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  launch_dependents();
  if (p.counters && blockIdx.x == 0 && threadIdx.x < kCounters) p.counters[threadIdx.x] = 0ull;
  double x[8];
  if ((int)blockIdx.x < p.row_ctas) {
    __shared__ uint2 peaks[8];
    const int part = w & (p.wpr - 1);
    const int64_t row = p.m0 + (((int64_t)blockIdx.x * 8 + w) >> p.wlog);
    const bool valid = row < p.m1;
    const double *a = p.A + (valid ? row : 0) * p.lda;
    const int step = 256 * p.wpr;
    const int steps = valid ? (int)((p.Kp - part * 256 + step - 1) >> (8 + p.wlog)) : 0;
    const int64_t k_first = part * 256 + lane * 8;
    Peak m;
    for (int i = 0; i < steps; ++i) {
      load_row8(a, k_first + (int64_t)i * step, p.K, x);
      m.add8(x);
    }
    m.hi = __reduce_max_sync(0xffffffffu, m.hi);
    m.lo = __reduce_or_sync(0xffffffffu, m.lo);
    if (p.wpr > 1) {
      if (lane == 0) peaks[w] = make_uint2(m.hi, m.lo);
      __syncthreads();
      for (int r = 0; r < p.wpr; ++r) m.add(peaks[w - part + r].x, peaks[w - part + r].y);
    }
    bool nf = false;
    const int ex = m.exponent(&nf);
    if (valid && part == 0 && lane == 0) {
      p.e[row] = ex;
      if (nf) record_error(p.status, HSUMMA_ERR_NONFINITE, kSiteNonFinite);
    }
    // backwards: the last step's values are still here
    for (int i = steps - 1; i >= 0; --i) {
      const int64_t k = k_first + (int64_t)i * step;
      if (i + 1 < steps) load_row8(a, k, p.K, x);
      constexpr int NQ = S <= 1 ? 1 : S <= 2 ? 2 : S <= 4 ? 4 : 8;
      float sq[NQ] = {};
      store_digits<false, W, true, S>(
          x, ex + 1011, k < p.Kp ? p.As + (row * p.Kp + k) * 2 : nullptr, p.M * p.Kp * 2, sq);
      if constexpr (SQ) {
        // a half warp is a window
        float q = spread_sums<NQ>(sq, lane);
#pragma unroll
        for (int o = NQ; o < 16; o <<= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (q > (float)kWindowBound) *p.big = 1;
      }
    }
    return;
  }
  constexpr int NS = S + (S & 1);
  __shared__ uint2 part[8][16];
  __shared__ unsigned long long colmax[16];
  __shared__ int colexp[16];
  __shared__ float win[2][SQ ? 8 : 1][SQ ? NS : 1][16];   // of even and odd windows
  const int cs = (int)cluster_nctas(), rank = (int)cluster_ctarank();
  const int64_t jb = p.n0 + (int64_t)(((int)blockIdx.x - p.row_ctas) / cs) * 16;
  const int64_t j = jb + (lane >> 1);
  const bool valid = j < p.n1;
  const double *b = p.B + (valid ? j : 0);
  const int w0 = rank * p.kw, w1 = min(p.wins, w0 + p.kw);
  const int ko = w * 16 + (lane & 1) * 8;      // in a window
  Peak m;
  for (int wi = w0; wi < w1; ++wi) {
    load_col8(b, p.ldb, (int64_t)wi * kWindow + ko, valid ? p.K : 0, x);
    m.add8(x);
  }
  m.add(__shfl_xor_sync(0xffffffffu, m.hi, 1), __shfl_xor_sync(0xffffffffu, m.lo, 1));
  if ((lane & 1) == 0) part[w][lane >> 1] = make_uint2(m.hi, m.lo);
  __syncthreads();
  if (threadIdx.x < 16) {
    m = Peak();
    for (int r = 0; r < 8; ++r) m.add(part[r][threadIdx.x].x, part[r][threadIdx.x].y);
    colmax[threadIdx.x] = (unsigned long long)m.hi << 32 | m.lo;
  }
  if (cs > 1) cluster_sync();                  // every CTA's colmax is written
  if (threadIdx.x < 16) {
    for (int r = 0; r < cs; ++r) {
      if (r == rank) continue;
      const unsigned long long o = ld_shared_cluster_u64(smem_u32(&colmax[threadIdx.x]), r);
      m.add((uint32_t)(o >> 32), (uint32_t)o);
    }
    bool nf = false;
    const int ex = m.exponent(&nf);
    colexp[threadIdx.x] = ex;
    if (rank == 0 && jb + threadIdx.x < p.n1) {
      p.f[jb + threadIdx.x] = ex;
      if (nf) record_error(p.status, HSUMMA_ERR_NONFINITE, kSiteNonFinite);
    }
  }
  __syncthreads();
  const int eb = colexp[lane >> 1] + 1011;
  for (int wi = w1 - 1; wi >= w0; --wi) {      // backwards likewise
    const int64_t k = (int64_t)wi * kWindow + ko;
    if (wi + 1 < w1) load_col8(b, p.ldb, k, valid ? p.K : 0, x);
    float sq[NS] = {};
    store_digits<false, W, true, S>(
        x, eb, valid && k < p.Kp ? p.Bs + (j * p.Kp + k) * 2 : nullptr, p.N * p.Kp * 2, sq);
    if constexpr (SQ) {
      // a column's window: two lanes of each of the 8 warps; the even lane adds
      // up the first slices, the odd one the others
      const bool up = lane & 1;
#pragma unroll
      for (int s = 0; s < NS / 2; ++s) {
        const float keep = up ? sq[NS / 2 + s] : sq[s], give = up ? sq[s] : sq[NS / 2 + s];
        win[wi & 1][w][up ? NS / 2 + s : s][lane >> 1] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
      }
      __syncthreads();
      if (threadIdx.x < S * 16) {
        float q = 0.f;
#pragma unroll
        for (int r = 0; r < 8; ++r) q += win[wi & 1][r][threadIdx.x >> 4][threadIdx.x & 15];
        if (q > (float)kWindowBound) *p.big = 1;
      }
    }
  }
  if (cs > 1) cluster_sync();                  // every CTA has read this one's colmax
}

// every slice type and count (8 slices exist for int8 only: bf16 stops at 7)
#define HS_KINDS_AND_SLICES(F)                                                             \
  F(HSUMMA_BF16_SLICES, 1);                                                                \
  F(HSUMMA_BF16_SLICES, 2);                                                                \
  F(HSUMMA_BF16_SLICES, 3);                                                                \
  F(HSUMMA_BF16_SLICES, 4);                                                                \
  F(HSUMMA_BF16_SLICES, 5);                                                                \
  F(HSUMMA_BF16_SLICES, 6);                                                                \
  F(HSUMMA_BF16_SLICES, 7);                                                                \
  F(HSUMMA_INT8_SLICES, 1);                                                                \
  F(HSUMMA_INT8_SLICES, 2);                                                                \
  F(HSUMMA_INT8_SLICES, 3);                                                                \
  F(HSUMMA_INT8_SLICES, 4);                                                                \
  F(HSUMMA_INT8_SLICES, 5);                                                                \
  F(HSUMMA_INT8_SLICES, 6);                                                                \
  F(HSUMMA_INT8_SLICES, 7);                                                                \
  F(HSUMMA_INT8_SLICES, 8)

// X = sum_d D_d 2^(w (S+1-d)) by Horner's rule (constant shifts), rounded once.
// Each thread takes four consecutive columns of one row: 16-byte loads from
// every plane when the rows are 16-byte aligned (N a multiple of 4), 16-byte
// stores of C when its row allows, element by element otherwise.  The first
// segment plane of every diagonal is loaded before any arithmetic, so that
// all S loads of a thread are in flight at once; a diagonal's further segment
// planes (np.n[d] of them in all; the planes past those hold zeros and are
// not read) are added in 64 bits.
// X fits in 64 bits whenever |D_2| <= T2: the host derives T2 from the range
// of the other diagonals (np.n[d] int32 planes each), so that
// |D_2| 2^(w (S-1)) + sum_(d>2) n_d 2^31 2^(w (S+1-d)) < 2^63 (every partial
// sum of Horner's rule is bounded by the same sum).  The diagonal sums the
// products give are far inside that bound; other values take the 128-bit path.
// (four resident blocks per SM keep more loads in flight; the kernels of 6 to
// 8 slices need more than the 64 registers that leaves)
struct DiagPlanes {
  int n[8];   // segment planes of diagonal d + 2 that the products can fill
};

template <int W, int S>
__global__ void __launch_bounds__(256, S <= 5 ? 4 : 3) recombine_kernel(const int32_t *__restrict__ D, int nseg,
                                                        DiagPlanes np, int64_t M, int64_t N,
                                                        const int32_t *__restrict__ e,
                                                        const int32_t *__restrict__ f,
                                                        double *__restrict__ C, int64_t ldc,
                                                        int64_t T2) {
  const int64_t j0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  const int64_t i = blockIdx.y;
  if (j0 >= N) return;
  const int64_t plane = M * N, off = i * N + j0;
  const bool full = j0 + 3 < N;
  const bool vec = full && (N & 3) == 0;
  auto load4 = [&](const int32_t *src, int (&v)[4]) {
    if (vec) {
      const int4 q = __ldg(reinterpret_cast<const int4 *>(src));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = j0 + u < N ? __ldg(src + u) : 0;
    }
  };
  int first[S][4];
#pragma unroll
  for (int d = 0; d < S; ++d) load4(D + (int64_t)(d * nseg) * plane + off, first[d]);
  // D_2 whole (its further planes, if any), which decides the width
  long long D2[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) D2[u] = first[0][u];
  for (int g = 1; g < np.n[0]; ++g) {
    int v[4];
    load4(D + (int64_t)g * plane + off, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) D2[u] += v[u];
  }
  int gmax = 1;
#pragma unroll
  for (int d = 1; d < S; ++d) gmax = np.n[d] > gmax ? np.n[d] : gmax;
  // X is linear in the planes: Horner's rule over the first planes, then each
  // further round g adds sum_(d>2) plane_g(D_d) 2^(w (S+1-d)), the round's
  // loads all in flight together (every partial sum is bounded as X is)
  auto round_g = [&](int g, int (&v)[S][4]) {
#pragma unroll
    for (int d = 1; d < S; ++d) {
      if (g < np.n[d]) {
        load4(D + (int64_t)(d * nseg + g) * plane + off, v[d]);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[d][u] = 0;
      }
    }
  };
  const int k = e[i] - W * (S + 1);
  double out[4];
  bool narrow = true;
#pragma unroll
  for (int u = 0; u < 4; ++u) narrow = narrow && llabs(D2[u]) <= T2;
  if (narrow) {
    unsigned long long X[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      X[u] = (unsigned long long)D2[u];
#pragma unroll
      for (int d = 1; d < S; ++d) X[u] = (X[u] << W) + (unsigned long long)(long long)first[d][u];
    }
    for (int g = 1; g < gmax; ++g) {
      int v[S][4];
      round_g(g, v);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        unsigned long long Y = 0;
#pragma unroll
        for (int d = 1; d < S; ++d) Y = (Y << W) + (unsigned long long)(long long)v[d][u];
        X[u] += Y;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      out[u] = j0 + u < N ? round_scaled64((long long)X[u], k + f[j0 + u]) : 0.0;
  } else {
    __int128 X[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      X[u] = D2[u];
#pragma unroll
      for (int d = 1; d < S; ++d) X[u] = (X[u] << W) + (__int128)first[d][u];
    }
    for (int g = 1; g < gmax; ++g) {
      int v[S][4];
      round_g(g, v);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        __int128 Y = 0;
#pragma unroll
        for (int d = 1; d < S; ++d) Y = (Y << W) + (__int128)v[d][u];
        X[u] += Y;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) out[u] = j0 + u < N ? round_scaled(X[u], k + f[j0 + u]) : 0.0;
  }
  double *dst = C + i * ldc + j0;
  if (full && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
    reinterpret_cast<double2 *>(dst)[0] = make_double2(out[0], out[1]);
    reinterpret_cast<double2 *>(dst)[1] = make_double2(out[2], out[3]);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < N) dst[u] = out[u];
  }
}

// T2 of the kernel above: the largest |D_2| for which X stays below 2^63 when
// every other diagonal d holds any sum of np.n[d-2] int32 planes; 2^31 admits
// every int32 plane, and -1 admits none (the other diagonals alone can pass
// 2^63: bf16 with S = 6).
int64_t recombine_narrow_bound(int W, int S, const DiagPlanes &np) {
  long double rest = 0.0L;
  for (int d = 3; d <= S + 1; ++d)
    rest += np.n[d - 2] * ldexpl(2147483648.0L, W * (S + 1 - d));
  const long double room = ldexpl(1.0L, 63) - 1.0L - rest;
  if (room < 0.0L) return -1;
  const long double t = floorl(room / ldexpl(1.0L, W * (S - 1)));
  return t >= 9.0e18L ? (int64_t)9000000000000000000LL : (int64_t)t;
}

template <int W, int S>
void recombine_launch(dim3 grid, cudaStream_t s, const int32_t *D, int nseg, const DiagPlanes &np,
                      int64_t M, int64_t N, const int32_t *e, const int32_t *f, double *C,
                      int64_t ldc) {
  const int64_t T2 = recombine_narrow_bound(W, S, np);
  recombine_kernel<W, S><<<grid, 256, 0, s>>>(D, nseg, np, M, N, e, f, C, ldc, T2);
  count_launch();
}

// the slice count as a template argument; the width follows from kind and S
template <int KIND>
void recombine_dispatch(int S, dim3 grid, cudaStream_t s, const int32_t *D, int nseg,
                        const DiagPlanes &np, int64_t M, int64_t N, const int32_t *e,
                        const int32_t *f, double *C, int64_t ldc) {
#define HS_RECOMBINE(SS)                                                                    \
  recombine_launch<slice_width(KIND, SS), SS>(grid, s, D, nseg, np, M, N, e, f, C, ldc); \
  break
  switch (S) {
    case 1: HS_RECOMBINE(1);
    case 2: HS_RECOMBINE(2);
    case 3: HS_RECOMBINE(3);
    case 4: HS_RECOMBINE(4);
    case 5: HS_RECOMBINE(5);
    case 6: HS_RECOMBINE(6);
    case 7: HS_RECOMBINE(7);
    default: HS_RECOMBINE(8);
  }
#undef HS_RECOMBINE
}

// One slicing launch with kind and slice count as template arguments: rows of A
// (ROWS) or columns of B; X is the operand, L its leading dimension, R its
// rows (A) or columns (B), x the exponents.
template <bool ROWS, int KIND, int S>
void slices_launch(cudaStream_t s, const double *X, int64_t L, int64_t R, int64_t K, int64_t Kp,
                   const int32_t *x, void *out) {
  if (ROWS) {
    slices_rows_kernel<KIND, S>
        <<<(unsigned)ceil_div(R * (Kp / 8), 256), 256, 0, s>>>(X, L, R, K, Kp, x, out);
  } else {
    const int64_t blocks = (Kp / 64) * ceil_div(R, 32);
    slices_cols_kernel<KIND, S><<<(unsigned)blocks, 256, 0, s>>>(X, L, K, R, Kp, x, out);
  }
}

template <bool ROWS>
void slices_dispatch(int kind, int S, cudaStream_t s, const double *X, int64_t L, int64_t R,
                     int64_t K, int64_t Kp, const int32_t *x, void *out) {
#define HS_SLICES(KIND, SS) \
  if (kind == KIND && S == SS) return slices_launch<ROWS, KIND, SS>(s, X, L, R, K, Kp, x, out)
  HS_KINDS_AND_SLICES(HS_SLICES);
#undef HS_SLICES
}

template <int KIND, int S>
cudaError_t digits_launch(const DigitsParams &p, int grid, int cluster, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, digits_kernel<KIND, S>, p);
}

}  // namespace

int launch_split_exponents(int64_t M, int64_t N, int64_t K, const double *A, int64_t lda,
                           const double *B, int64_t ldb, int32_t *e, int32_t *f,
                           cudaStream_t s) {
  int *status = state().d_status;
  if (M > 0) {
    const int64_t blocks = ceil_div(M, 8);
    exponents_rows_kernel<<<(unsigned)blocks, 256, 0, s>>>(A, lda, M, K, e, status);
    count_launch();
  }
  if (N > 0) {
    // k split over a cluster of up to 8 CTAs per column group, enough for
    // about four CTAs per SM (152 SMs) when N is small
    const int64_t nbx = ceil_div(N, 64);
    int ks = (int)ceil_div(4 * 152, nbx);
    ks = ks < 1 ? 1 : (ks > 8 ? 8 : ks);
    if (ks > K) ks = K > 1 ? (int)K : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nbx, (unsigned)ks, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = (unsigned)ks;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e2 = cudaLaunchKernelEx(&cfg, exponents_cols_kernel, B, ldb, K, N, f, status);
    if (e2 != cudaSuccess) return cuda_fail(e2, "launch exponent scan (columns)");
    count_launch();
  }
  cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? HSUMMA_OK : cuda_fail(err, "launch exponent scan");
}

int launch_split_slices(int64_t M, int64_t N, int64_t K, const double *A, int64_t lda,
                        const double *B, int64_t ldb, const int32_t *e, const int32_t *f,
                        int kind, int S, void *As, void *Bs, cudaStream_t s) {
  const int64_t Kp = ceil_div(K, 64) * 64;
  if (Kp == 0) return HSUMMA_OK;
  const int64_t nA = M * (Kp / 8), ncb = N > 0 ? (Kp / 64) * ceil_div(N, 32) : 0;
  if (ceil_div(nA, 256) > 0x7fffffff || ncb > 0x7fffffff) {
    set_error("slicing grid too large (M=%lld N=%lld K=%lld)", (long long)M, (long long)N,
              (long long)K);
    return HSUMMA_ERR_UNSUPPORTED;
  }
  if (M > 0) {
    slices_dispatch<true>(kind, S, s, A, lda, M, K, Kp, e, As);
    count_launch();
  }
  if (N > 0) {
    slices_dispatch<false>(kind, S, s, B, ldb, N, K, Kp, f, Bs);
    count_launch();
  }
  cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? HSUMMA_OK : cuda_fail(err, "launch slicing");
}

int launch_split_digits(int64_t M, int64_t N, int64_t K, const double *A, int64_t lda,
                        const double *B, int64_t ldb, int32_t *e, int32_t *f, int kind, int S,
                        void *As, void *Bs, bool clear_counters, cudaStream_t s) {
  DigitsParams p{};
  p.A = A;
  p.B = B;
  p.lda = lda;
  p.ldb = ldb;
  p.M = M;
  p.N = N;
  p.K = K;
  p.Kp = ceil_div(K, 64) * 64;
  p.e = e;
  p.f = f;
  p.As = static_cast<uint8_t *>(As);
  p.Bs = static_cast<uint8_t *>(Bs);
  p.status = state().d_status;
  p.big = fused_big_digits();
  p.wins = (int)ceil_div(p.Kp, kWindow);
  p.wpr = 1;
  // warps a row: one step each, but at most four where two waves of warps are left
  while (p.wpr < 8 && p.Kp > 256 * p.wpr) p.wpr = 1 << ++p.wlog;
  while (p.wpr > 1 && p.Kp <= 512 * p.wpr && M * (p.wpr / 2) >= 2 * 24 * state().sm_count)
    p.wpr = 1 << --p.wlog;
  int cs = 1;
  while (cs < 8 && p.wins > cs) cs *= 2;
  p.kw = (int)ceil_div(p.wins, cs);
  // A launch takes rows and columns together, up to 1 GiB of operands; more is
  // divided (a launch costs nothing beside the passes it covers), rows first.
  const int64_t limit = int64_t(1) << 27;
  const bool together = (M + N) * K <= limit;
  const int64_t mstep = together ? M : std::max<int64_t>(1, limit / K / 8) * 8;
  const int64_t nstep = together ? N : std::max<int64_t>(1, limit / K / 16) * 16;
  bool first = true;
  for (int64_t m = 0, n = 0; m < M || n < N;) {
    p.m0 = m;
    p.m1 = m = std::min(M, m + mstep);
    p.n0 = p.n1 = n;
    if (p.m0 == p.m1 || together) p.n1 = n = std::min(N, n + nstep);
    const int64_t rows = ceil_div(ceil_div(p.m1 - p.m0, 8 / p.wpr), cs) * cs;
    const int64_t cols = ceil_div(p.n1 - p.n0, 16) * cs;
    if (rows + cols > 0x7fffffff) {
      set_error("slicing grid too large (M=%lld N=%lld K=%lld)", (long long)M, (long long)N,
                (long long)K);
      return HSUMMA_ERR_UNSUPPORTED;
    }
    p.row_ctas = (int)rows;
    p.counters = first && clear_counters ? state().d_counters : nullptr;
    first = false;
    cudaError_t err = cudaErrorInvalidValue;
#define HS_DIGITS(KIND, SS) \
  if (kind == KIND && S == SS) err = digits_launch<KIND, SS>(p, (int)(rows + cols), cs, s)
    HS_KINDS_AND_SLICES(HS_DIGITS);
#undef HS_DIGITS
    if (err != cudaSuccess) return cuda_fail(err, "launch digits_kernel");
    count_launch();
  }
  return HSUMMA_OK;
}

int launch_split_recombine(int64_t M, int64_t N, int64_t K, int kind, int S, const int32_t *D,
                           const int32_t *e, const int32_t *f, double *C, int64_t ldc,
                           cudaStream_t s) {
  const int nseg = split_planes(K, S, kind);
  DiagPlanes np = {};
  for (int d = 2; d <= S + 1 && d - 2 < 8; ++d)
    np.n[d - 2] = split_diagonal_planes(K, S, kind, d - 1);
  // one grid row per matrix row, in bands of at most 65535 rows; a band starts
  // r0 rows in: D, e and C advance by r0 rows, the plane stride stays M N
  for (int64_t r0 = 0; r0 < M; r0 += 65535) {
    const int64_t rows = (M - r0) < 65535 ? (M - r0) : 65535;
    dim3 grid((unsigned)ceil_div(ceil_div(N, 4), 256), (unsigned)rows);
    if (kind == HSUMMA_INT8_SLICES)
      recombine_dispatch<HSUMMA_INT8_SLICES>(S, grid, s, D + r0 * N, nseg, np, M, N, e + r0, f,
                                             C + r0 * ldc, ldc);
    else
      recombine_dispatch<HSUMMA_BF16_SLICES>(S, grid, s, D + r0 * N, nseg, np, M, N, e + r0, f,
                                             C + r0 * ldc, ldc);
  }
  cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? HSUMMA_OK : cuda_fail(err, "launch recombination");
}

}  // namespace hs
