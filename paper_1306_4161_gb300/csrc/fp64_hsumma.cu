// Native binary64 HSUMMA kernel (Section III, Algorithm 1) for sm_103a.
//
// A virtual processor P_(x,y)(i,j) of the P x Q grid owns the C block of rows
// [r Mt, (r+1) Mt) and columns [c Nt, (c+1) Nt) and sweeps it in 128 x 128
// sub-tiles.  For every sub-tile the k loop runs in outer steps of Bouter
// columns and inner steps of b:
//   * outer step: the owner of the outer A block (Algorithm 1's
//     Pivot_group_col) brings A[rows, kB:(k+1)B] into L2 with a TMA prefetch,
//     the owner of the outer B block (Pivot_group_row) brings B[kB:(k+1)B, cols];
//     every group then reads the panels from L2 (the between-group broadcast);
//   * inner step: 16-wide slices of the panels are copied into shared memory
//     by the Tensor Memory Accelerator.  When the group is a thread-block
//     cluster, each A slice is fetched once per cluster row and multicast to the
//     Q/J CTAs of the row (row_comm), each B slice once per cluster column and
//     multicast to the P/I CTAs of the column (col_comm);
//   * local update (Algorithm 1's DGemm): c += a b with the binary64 tensor-core
//     instruction mma.sync.m16n8k4.f64 into register accumulators.
// The outer/inner structure does not change the arithmetic: every C element is
// the k-ascending binary64 sum of its products, so integer inputs give exact
// results for any G, b and Bouter.
//
// Strips.  The DMMA unit is slow (about 1.05 TFLOP/s, 3.5 flops per cycle and SM;
// one warp per SM sub-partition keeps it busy), so nothing but the balance of the
// work over the SMs matters: a 128 x 128 sub-tile of 16 k-columns is 150,000
// cycles of DMMA against 32 KB of copies.  A processor's block is therefore cut
// into strips of RH = 16 rows of a sub-tile, one CTA each (grid dimension z), and
// several CTAs share an SM: their number per SM, not the number of sub-tiles per
// CTA, is what is left to round.  A strip of the same rows of every processor of
// a group is one cluster, so A's rows are multicast as before; each strip brings
// its own copy of the B panel (the counters, which are the processor's, take B
// and the owners' prefetches from its first strip).  Strips past the rows of a
// block are not run, nor warps past its columns.  Same box, one CTA per processor
// sweeping 128 x 128 sub-tiles -> strips of 16 rows (us): 512^3 on 4 x 4, 2 x 2
// clusters 2431 -> 330 (128 strips for 152 SMs); 1024^3 on 8 x 8, flat 4906 ->
// 2370; 2048^3 on 16 x 16, 2 x 2 clusters 19370 -> 16342; 4096^3 on 16 x 16, flat
// 156300 -> 125300 (1.097 TFLOP/s), 2 x 2 clusters 154800 -> 129900, 4 x 4
// clusters 231100 -> 153400 (clusters of 16 do not fill the device); 4096^3 on
// 32 x 32, 2 x 1 clusters 135900 -> 125400.  Strips of 32 rows: 654, 2359, 17123,
// 125260, 133200, 171400, 125300.
//
// Roles (288 threads): warps 0..7 compute (RH x 16 each, the columns rotated by
// CTA so that idle ones fall on different sub-partitions), warp 8 issues the
// copies.  A ring of 16 k-columns a stage (17,700 cycles of DMMA each); "full"
// barriers count the bytes of a stage, "empty" barriers collect the releases of the
// CTA's whole cluster row and column, more than its copies reach (A comes from cluster
// column 0, B from the rows that have a piece).  A barrier can't tell who arrives: this
// is sound where a CTA that releases the next stage has waited, through the copies it
// got, for every release of this one, else its arrival takes the place of a slow CTA's
// and that one's panel is overwritten.  It has where every cluster row sends a piece of
// B (4 NT pieces >= cm rows), or with one column; counts_hold() keeps to that.  Counting
// only the CTAs that the copies reach holds for every shape and takes fewer arrivals,
// but CTAs then drift apart: 4096^3 on 16 x 16, 4 x 4 clusters 153.6 -> 157.7 ms.
// Where CTAs share an SM, two stages (three or four leave fewer CTAs per SM: 4 x 4
// clusters 153.4 / 154.2 / 171.9 ms), and in clusters the warps of a CTA release a
// stage together: each by itself, the shared unit lets some run ahead and the
// cluster waits for the others (153.3 -> 160.1 ms).  A CTA that has its SM to
// itself has nothing to fill the unit while its warps meet: four stages, each warp
// by itself (512^3 on 4 x 4, 2 x 2 clusters: 353 -> 330 us; 304 x 1024 x 4096 on 19 x
// 8, flat: 2670 -> 2454), and so for flat grids, where it costs nothing.
#include "internal.h"
#include "ptx.cuh"
#include "tc05.cuh"
#include "../../include/hsumma.h"

namespace hs {
namespace {

constexpr int TM = 128, TN = 128, BK = 16;
constexpr int MAX_STAGES = 4;
constexpr int RH = 16;                        // rows of a strip
constexpr int NSTRIP = TM / RH;
constexpr int A_STAGE = RH * BK * 8;          // 2 KB pieces of 16 rows x 128 B
__host__ __device__ constexpr int b_stage(int nt) { return BK * nt * 64 * 8; }   // pieces of 16 k x 16 n, 2 KB each
constexpr int NCOMP = 256, NTHREADS = NCOMP + 32;
constexpr int CTAS_PER_SM = 3;                // leaves 72 registers; 56 are used, and four CTAs fit
constexpr int smem_bytes(int stages, int nt) {
  return stages * (A_STAGE + b_stage(nt)) + 2 * MAX_STAGES * 8 + 1024;
}
constexpr int PF_K = 32;                      // k extent of one prefetch box
constexpr int MT = RH / 16;                   // DMMA tiles of a warp: RH x 8 NT, NT = 2 or 1

struct Fp64Params {
  double *C;
  int64_t ldc, M, N, K, Mt, Nt, Kq, Kp;
  int P, Q, cm, cn, nsub_m, nsub_n, Bo, units;
  int stages, free_warps;
  unsigned long long *counters;
  int *status;
};

__device__ __forceinline__ void dmma(double (&c)[4], double a0, double a1, double b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k4.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%0,%1,%2,%3};"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a0), "d"(a1), "d"(b0));
}

__device__ __forceinline__ int64_t clamp_count(int64_t lo, int64_t hi, int64_t a, int64_t b) {
  // |[a, b) ∩ [lo, hi)|
  int64_t x = a > lo ? a : lo, y = b < hi ? b : hi;
  return y > x ? y - x : 0;
}

// Unit u of a processor's sweep: sub-tile (mi, ni), strip st of it, and of the
// strip's columns the part from c0 on (64 NT of them; the first has c0 = 0).
struct Unit {
  int mi, ni, st, c0;
};
template <int NT>
__device__ __forceinline__ Unit unit_of(int u, int nsub_n) {
  constexpr int parts = 2 / NT;
  const int t = u / (NSTRIP * parts), w = u % (NSTRIP * parts);
  return Unit{t / nsub_n, t % nsub_n, w / parts, w % parts * 64};
}

// Whether a cluster's releases are counted soundly (Roles, above).
constexpr bool counts_hold(int cm, int cn, int nt) { return cn == 1 || cm <= 4 * nt; }
static_assert(counts_hold(8, 2, 2) && counts_hold(16, 1, 2), "every cluster of up to 16 CTAs");

// CYC: block-cyclic layout of the grid, else block-checkerboard
template <bool CYC, int NT>
__global__ void __launch_bounds__(NTHREADS, CTAS_PER_SM)
    fp64_hsumma_kernel(const __grid_constant__ CUtensorMap tmA,
                       const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmApf,
                       const __grid_constant__ CUtensorMap tmBpf, const Fp64Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t nst = (uint32_t)p.stages;
  constexpr int B_STAGE = b_stage(NT);
  uint8_t *sA = smem + nst * B_STAGE;
  uint8_t *sB = smem;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + nst * (A_STAGE + B_STAGE));
  uint64_t *empty = full + MAX_STAGES;
  __shared__ int abort_flag;

  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);   // warp-uniform
  const int cx = (int)cluster_ctaid_x(), cy = (int)cluster_ctaid_y();
  const int cn = p.cn, cm = p.cm;
  int r, c;
  raster_proc(cm, cn, cy, cx, 8, &r, &c);

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), (uint32_t)((cn + cm - 1) * (p.free_warps ? NCOMP / 32 : 1)));
    }
    fence_mbar_init();
  }
  cluster_sync();

  const int r0 = r - cy, c0 = c - cx;           // the cluster's first processor row / column
  constexpr bool cyc = CYC;
  const int64_t nk = (p.K + BK - 1) / BK;
  const int64_t nout = p.K > 0 ? (p.K + p.Bo - 1) / p.Bo : 0;
  // whether the cluster skips a unit: a sub-tile wholly outside the matrix in
  // the block-cyclic layout, a strip but a sub-tile's first that holds no row of
  // any of the cluster's blocks (the first one keeps the schedule's copies of B),
  // and a second half without a column of them.  The same answer in every CTA of
  // the cluster.
  auto skipped = [&](const Unit &u) {
    if (tile_skipped(cyc, r0, u.mi, p.P, TM, p.M) || tile_skipped(cyc, c0, u.ni, p.Q, TN, p.N))
      return true;
    int64_t org, lo, hi;
    if (u.c0) {
      tile_rows(cyc, c0, u.ni, p.Q, p.Nt, TN, p.N, &org, &lo, &hi);
      if (org + u.c0 >= hi) return true;
    }
    if (u.st == 0) return false;
    tile_rows(cyc, r0, u.mi, p.P, p.Mt, TM, p.M, &org, &lo, &hi);
    return org + u.st * RH >= hi;
  };

  if (warp == NCOMP / 32) {
    // ---------------- copies: the warp in step, one lane issues ----------------
    const bool el = elect_one();
    const uint16_t row_mask = (uint16_t)(((1u << cn) - 1u) << (cy * cn));
    uint16_t col_mask = 0;
    for (int y = 0; y < cm; ++y) col_mask |= (uint16_t)(1u << (y * cn + cx));
    unsigned long long a_ld = 0, b_ld = 0, pf = 0, nops = 0;
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int ui = blockIdx.z; ui < p.units && ok; ui += gridDim.z) {
      const Unit u = unit_of<NT>(ui, p.nsub_n);
      if (skipped(u)) continue;
      int64_t m0, row_lo, row_hi, n0, col_lo, col_hi;
      tile_rows(cyc, r, u.mi, p.P, p.Mt, TM, p.M, &m0, &row_lo, &row_hi);
      tile_rows(cyc, c, u.ni, p.Q, p.Nt, TN, p.N, &n0, &col_lo, &col_hi);
      const int64_t ms = m0 + u.st * RH;
      // rows of A and columns of B this CTA copies, inside its block and the
      // matrix: piece i of A is issued by cluster column i mod cn, piece j of B
      // by cluster row j mod cm
      for (int i = cx; i < RH / 16 && u.c0 == 0; i += cn)
        a_ld += (unsigned long long)(clamp_count(row_lo, row_hi, ms + i * 16, ms + i * 16 + 16) *
                                     p.K);
      if (u.st == 0)
        for (int j = cy; j < NT * 4; j += cm)
          b_ld += (unsigned long long)(clamp_count(col_lo, col_hi, n0 + u.c0 + j * 16,
                                                   n0 + u.c0 + j * 16 + 16) *
                                       p.K);
      int rem = 0;   // k0 mod B, kept without a 64-bit division per stage
      for (int64_t kt = 0; kt < nk; ++kt) {
        const int64_t k0 = kt * BK;
        const bool outer = rem == 0 && u.st == 0 && u.c0 == 0;
        for (rem += BK; rem >= p.Bo;) rem -= p.Bo;
        if (outer) {
          // outer step o: stage outer panel o (first step) and o + 1 into L2; the
          // owner of an outer block is the processor whose own block of A
          // (columns) / B (rows) contains its first index (block-cyclic: the
          // processor column / row q mod Q / q mod P)
          const int64_t o = k0 / p.Bo;
          for (int64_t q = (o == 0 ? 0 : o + 1); q <= o + 1 && q < nout; ++q) {
            const int64_t kq = q * p.Bo, kend = imin64(p.K, kq + p.Bo);
            if (c == outer_owner(cyc, q, kq, p.Kq, p.Q)) {
              if (el)
                for (int64_t kk = kq; kk < kend; kk += PF_K)
                  tma_prefetch_2d(&tmApf, (int32_t)kk, (int32_t)m0);
              pf += 1;
            }
            if (r == outer_owner(cyc, q, kq, p.Kp, p.P)) {
              if (el)
                for (int64_t kk = kq; kk < kend; kk += PF_K)
                  tma_prefetch_2d(&tmBpf, (int32_t)n0, (int32_t)kk);
              pf += 1;
            }
          }
        }
        if (!__all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&empty[stage]), phase ^ 1u))) {
          record_error(p.status, HSUMMA_ERR_TIMEOUT, kSiteEmpty);
          ok = false;
          break;
        }
        const uint32_t fb = smem_u32(&full[stage]);
        const uint32_t a_dst = smem_u32(sA + stage * A_STAGE), b_dst = smem_u32(sB + stage * B_STAGE);
        if (el) {
          mbar_arrive_expect_tx(fb, A_STAGE + B_STAGE);
          for (int i = cx; i < RH / 16; i += cn) {
            if (cn > 1)
              tma_load_2d_mc(a_dst + i * 2048, &tmA, (int32_t)k0, (int32_t)(ms + i * 16), fb,
                             row_mask);
            else
              tma_load_2d(a_dst + i * 2048, &tmA, (int32_t)k0, (int32_t)(ms + i * 16), fb);
            nops += 1;
          }
          for (int j = cy; j < NT * 4; j += cm) {
            const int32_t nj = (int32_t)(n0 + u.c0 + j * 16);
            if (cm > 1)
              tma_load_2d_mc(b_dst + j * 2048, &tmB, nj, (int32_t)k0, fb, col_mask);
            else
              tma_load_2d(b_dst + j * 2048, &tmB, nj, (int32_t)k0, fb);
            nops += 1;
          }
        }
        __syncwarp();
        if (++stage == nst) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok) atomicExch(&abort_flag, 1);
    if (el) {
      atomicAdd(&p.counters[0], a_ld);
      atomicAdd(&p.counters[1], a_ld * cn);
      atomicAdd(&p.counters[2], b_ld);
      atomicAdd(&p.counters[3], b_ld * cm);
      atomicAdd(&p.counters[4], pf);
      atomicAdd(&p.counters[5], nops);
    }
  } else {
    // ---------------- rank-16 updates with DMMA ----------------
    // a warp's columns: rotated by CTA, so that the warps without columns in
    // short blocks sit on different SM sub-partitions in the CTAs that share an SM
    const int wn = (warp + (int)(blockIdx.x + blockIdx.y + blockIdx.z)) & 7;
    const int g = lane >> 2, t = lane & 3;
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int ui = blockIdx.z; ui < p.units && ok; ui += gridDim.z) {
      const Unit u = unit_of<NT>(ui, p.nsub_n);
      if (skipped(u)) continue;
      int64_t m0, row_lo, row_hi, n0, col_lo, col_hi;
      tile_rows(cyc, r, u.mi, p.P, p.Mt, TM, p.M, &m0, &row_lo, &row_hi);
      tile_rows(cyc, c, u.ni, p.Q, p.Nt, TN, p.N, &n0, &col_lo, &col_hi);
      const int64_t ms = m0 + u.st * RH, ns = n0 + u.c0 + wn * (8 * NT);
      const bool busy = ms < row_hi && ns < col_hi;   // else nothing of C is here
      double acc[MT][NT][4];
#pragma unroll
      for (int a = 0; a < MT; ++a)
#pragma unroll
        for (int b = 0; b < NT; ++b)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[a][b][e] = 0.0;
      for (int64_t kt = 0; kt < nk; ++kt) {
        const bool bad = !__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[stage]), phase));
        if (bad) record_error(p.status, HSUMMA_ERR_TIMEOUT, kSiteFull);
        if (busy) {
          const uint8_t *a_base = sA + stage * A_STAGE;
          // (a warp's columns: a piece of 16, or half of one)
          const uint8_t *b_base = sB + stage * B_STAGE + wn * NT / 2 * 2048;
          const int nw = NT == 1 ? (wn & 1) * 8 : 0;
#pragma unroll
          for (int kk = 0; kk < BK / 4; ++kk) {
            const int k = kk * 4 + t;
            double af[MT][2], bf[NT];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
              const int row = mt * 16 + g;
              af[mt][0] = *reinterpret_cast<const double *>(a_base + swz128(row, k * 8));
              af[mt][1] = *reinterpret_cast<const double *>(a_base + swz128(row + 8, k * 8));
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
              bf[nt] = *reinterpret_cast<const double *>(b_base + swz128(k, (nw + nt * 8 + g) * 8));
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
              for (int nt = 0; nt < NT; ++nt) dmma(acc[mt][nt], af[mt][0], af[mt][1], bf[nt]);
          }
        }
        // done with the stage, go on or stop: the warps together, or each by itself
        if (p.free_warps) {
          __syncwarp();
          ok = !bad;
        } else {
          ok = !named_barrier_or(1, NCOMP, bad);
        }
        if (!ok) break;
        // release it to every CTA that delivers into it
        if (p.free_warps ? lane == 0 : threadIdx.x == 0) {
          const uint32_t eb = smem_u32(&empty[stage]);
          for (int x = 0; x < cn; ++x) mbar_arrive_cluster(eb, (uint32_t)(cy * cn + x));
          for (int y = 0; y < cm; ++y)
            if (y != cy) mbar_arrive_cluster(eb, (uint32_t)(y * cn + cx));
        }
        if (++stage == nst) { stage = 0; phase ^= 1u; }
      }
      if (!ok || !busy) continue;
      // epilogue: C := the strip (beta = 0), rows/cols inside the block
      // (block-cyclic: inside the tile and the matrix)
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int64_t row = ms + mt * 16 + g + h * 8;
          if (row >= row_hi) continue;
          double *crow = p.C + row * p.ldc;
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const int64_t col = ns + nt * 8 + 2 * t;
            const double v0 = acc[mt][nt][2 * h], v1 = acc[mt][nt][2 * h + 1];
            if (col + 1 < col_hi && ((reinterpret_cast<uintptr_t>(crow + col) & 15) == 0)) {
              *reinterpret_cast<double2 *>(crow + col) = make_double2(v0, v1);
            } else {
              if (col < col_hi) crow[col] = v0;
              if (col + 1 < col_hi) crow[col + 1] = v1;
            }
          }
        }
      }
    }
    if (!ok) atomicExch(&abort_flag, 1);
  }
  __syncthreads();
  // an aborted CTA may still have copies in flight into its shared memory:
  // give them a bounded moment to land before leaving
  if (abort_flag) bounded_sleep(2000000ull);
  // no CTA leaves while a peer may still deliver into its shared memory or
  // arrive on its barriers
  cluster_sync();
}

}  // namespace

int fp64_cluster_limit(int *limit) {
  cudaError_t e = cudaFuncSetAttribute(fp64_hsumma_kernel<false, 2>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem_bytes(2, 2));
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(smem)");
  e = cudaFuncSetAttribute(fp64_hsumma_kernel<false, 2>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(non-portable cluster)");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16, 1, 1);
  cfg.blockDim = dim3(NTHREADS, 1, 1);
  cfg.dynamicSmemBytes = smem_bytes(2, 2);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxPotentialClusterSize(&n, fp64_hsumma_kernel<false, 2>, &cfg);
  if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxPotentialClusterSize");
  *limit = n;
  return HSUMMA_OK;
}

int launch_fp64_hsumma(const GridPlan &g, const double *A, int64_t lda, const double *B,
                       int64_t ldb, double *C, int64_t ldc, cudaStream_t s) {
  CUtensorMap tA, tB, tApf, tBpf;
  const auto F64 = CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
  if (!encode_tmap_2d(&tA, F64, 8, A, g.K, g.M, lda, 16, 16, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_tmap_2d(&tB, F64, 8, B, g.N, g.K, ldb, 16, 16, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_tmap_2d(&tApf, F64, 8, A, g.K, g.M, lda, PF_K, TM, CU_TENSOR_MAP_SWIZZLE_NONE) ||
      !encode_tmap_2d(&tBpf, F64, 8, B, g.N, g.K, ldb, TN, PF_K, CU_TENSOR_MAP_SWIZZLE_NONE))
    return HSUMMA_ERR_ARG;
  Fp64Params p;
  p.C = C;
  p.ldc = ldc;
  p.M = g.M;
  p.N = g.N;
  p.K = g.K;
  p.Mt = g.Mt;
  p.Nt = g.Nt;
  p.Kq = g.Kq;
  p.Kp = g.Kp;
  p.P = g.P;
  p.Q = g.Q;
  p.cm = g.cm;
  p.cn = g.cn;
  p.nsub_m = (int)(g.cyc ? ceil_div(ceil_div(g.M, TM), g.P) : ceil_div(g.Mt, TM));
  p.nsub_n = (int)(g.cyc ? ceil_div(ceil_div(g.N, TN), g.Q) : ceil_div(g.Nt, TN));
  p.Bo = g.Bo;
  // Strips of half the columns where the busiest SM then has 5 % less: n CTAs take
  // the time of ceil(n / SMs).  256^3 on 2 x 2, flat (32 / 64 CTAs) 162 / 90 us; 1024^3 on 8 x
  // 8 (512 / 1024) flat 2352 / 2059, 2 x 2 clusters 2381 / 2186; not for less (2048^3
  // on 16 x 16, 2 x 2 clusters, 2 %: 16.33 / 16.41 ms).  Not in clusters of more
  // than four rows: some of those rows would have no piece of B (see Roles; such
  // products gave wrong sums).
  const int64_t whole = (int64_t)p.nsub_m * p.nsub_n * NSTRIP, procs = (int64_t)g.P * g.Q;
  const int sms = state().sm_count;
  const int nt =
      g.cm <= 4 && ceil_div(procs * whole * 2, sms) * 20 <= ceil_div(procs * whole, sms) * 38 ? 1 : 2;
  if (!counts_hold(g.cm, g.cn, nt)) {   // (no cluster of 16 CTAs)
    set_error("clusters of %d x %d are not supported", g.cm, g.cn);
    return HSUMMA_ERR_UNSUPPORTED;
  }
  const int64_t units = whole * (2 / nt);
  if (units > 0x7fffffff) {
    set_error("blocks of %d x %d sub-tiles are not supported", p.nsub_m, p.nsub_n);
    return HSUMMA_ERR_UNSUPPORTED;
  }
  p.units = (int)units;
  const int64_t ctas = procs * (units < 65535 ? units : 65535);
  const bool alone = ctas <= sms;
  p.free_warps = alone || g.cm * g.cn == 1;
  p.stages = alone ? 4 : 2;
  const int smem = smem_bytes(p.stages, nt);
  p.counters = state().d_counters;
  p.status = state().d_status;
  auto kern = nt == 2 ? (g.cyc ? fp64_hsumma_kernel<true, 2> : fp64_hsumma_kernel<false, 2>)
                      : (g.cyc ? fp64_hsumma_kernel<true, 1> : fp64_hsumma_kernel<false, 1>);
  cudaError_t e = cudaFuncSetAttribute(kern,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem_bytes(MAX_STAGES, nt));
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(smem)");
  if (g.cm * g.cn > 8) {
    e = cudaFuncSetAttribute(kern,
                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(non-portable cluster)");
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)g.Q, (unsigned)g.P, (unsigned)(units < 65535 ? units : 65535));
  cfg.blockDim = dim3(NTHREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)g.cn;
  at[0].val.clusterDim.y = (unsigned)g.cm;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, tA, tB, tApf, tBpf, p);
  if (e != cudaSuccess) return cuda_fail(e, "launch fp64_hsumma_kernel");
  count_launch();
  return HSUMMA_OK;
}

}  // namespace hs
