// Host side of the product kernel that recombines (split_fused.cuh), and its
// instances with tiles of 128 columns.
#include "internal.h"

namespace hs {
namespace {
constexpr int TN = 128;
}
}  // namespace hs
#include "split_fused.cuh"

namespace hs {

// Whether the products of (g, kind, S) can run on this kernel: every pass's sum
// fits a signed 64-bit integer whatever the digits.
bool split_fused_ok(const GridPlan &g, int kind, int S) {
  const int w = slice_width(kind, S), top = S + 1;
  const int low = S <= 4 ? top : (S == 5 ? 4 : 5);
  for (int ps = 0; ps < 2; ++ps) {
    const int dlo = ps ? low + 1 : 2, dhi = ps ? top : low;
    long double sum = 0.0L;
    for (int x = dlo; x <= dhi; ++x)
      sum += (long double)(x - 1) * (long double)g.K * ldexpl(1.0L, 2 * w - 2 + w * (dhi - x));
    if (sum >= 4.5e18L) return false;   // and the guard bit
  }
  const int64_t rt = ceil_div(g.M, 128) + g.P, ct = ceil_div(g.N, 128) + g.Q;
  return rt * ct < (1ll << 30) && kFusedClusters * ceil_div(g.K, 128) < (1ll << 31);
}

// The panel-load counters of the schedule (every processor's copies, once per
// slice pair): closed forms over the nominal sub-tiles of both layouts.
static void schedule_counters(const GridPlan &g, int tn, int64_t npairs, unsigned long long *out) {
  const int64_t nout = ceil_div(g.K, g.Bo);
  int64_t sm, sn, pf;   // row (column) sweeps summed over the processor rows (columns)
  if (g.cyc) {
    const int64_t Tm = ceil_div(g.M, TM), Tn = ceil_div(g.N, tn);
    sm = sn = pf = 0;
    int64_t om = 0, on = 0;   // sweeps weighted by the outer blocks the processor owns
    for (int r = 0; r < g.P; ++r) {
      const int64_t r0 = r - r % g.cm, a = r0 < Tm ? ceil_div(Tm - r0, g.P) : 0;
      sm += a;
      om += a * (r < nout ? ceil_div(nout - r, g.P) : 0);
    }
    for (int c = 0; c < g.Q; ++c) {
      const int64_t c0 = c - c % g.cn, a = c0 < Tn ? ceil_div(Tn - c0, g.Q) : 0;
      sn += a;
      on += a * (c < nout ? ceil_div(nout - c, g.Q) : 0);
    }
    pf = sm * on + sn * om;
  } else {
    const int64_t nsm = ceil_div(g.Mt, TM), nsn = ceil_div(g.Nt, tn);
    sm = g.P * nsm;
    sn = g.Q * nsn;
    pf = nsm * nsn * nout * (g.P + g.Q);
  }
  out[0] = (unsigned long long)(npairs * g.M * g.K * (sn / g.cn));
  out[1] = (unsigned long long)(npairs * g.M * g.K * sn);
  out[2] = (unsigned long long)(npairs * g.K * g.N * (sm / g.cm));
  out[3] = (unsigned long long)(npairs * g.K * g.N * sm);
  out[4] = (unsigned long long)(npairs * pf);
}

// Partial sums, what large chunks add, low words, arrival counts: one buffer, allocated on
// first use and kept until hsumma_finalize; behind them a count of finished CTAs, the
// "large digits" word and a word that a launch sets when it gives up.  All but the
// sums and the low words are at zero between products.
constexpr size_t kSumBytes = (size_t)kFusedClusters * kParts * 2 * kPartWords * 8;
constexpr size_t kMissedBytes = (size_t)kFusedClusters * 2 * kTileWords * 8;
constexpr size_t kLowBytes = kMissedBytes / 2;
constexpr int kCounts = kFusedClusters * 2 * NEPI;
constexpr size_t kCountsAt = kSumBytes + kMissedBytes + kLowBytes;
constexpr size_t kBufBytes = kCountsAt + (kCounts + 3) * 4;

int *fused_big_digits() {
  return reinterpret_cast<int *>(static_cast<uint8_t *>(state().fused_buf) + kCountsAt) +
         kCounts + 1;
}

static int fused_zero() {
  cudaError_t e = cudaMemset(state().fused_buf, 0, kBufBytes);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return e == cudaSuccess ? HSUMMA_OK : cuda_fail(e, "clear the partial sums");
}

int fused_clear() {
  if (!state().fused_buf) return HSUMMA_OK;
  int gave_up = 0;
  cudaError_t e = cudaDeviceSynchronize();   // no product is at work on another stream
  if (e == cudaSuccess)
    e = cudaMemcpy(&gave_up, fused_big_digits() + 1, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "read whether a product gave up");
  return gave_up ? fused_zero() : HSUMMA_OK;
}

int fused_reserve() {
  DeviceState &st = state();
  if (st.fused_buf) return HSUMMA_OK;
  cudaError_t e = cudaMalloc(&st.fused_buf, kBufBytes);
  if (e != cudaSuccess) {
    st.fused_buf = nullptr;
    return cuda_fail(e, "cudaMalloc(partial sums)");
  }
  return fused_zero();
}

int launch_split_fused(const GridPlan &g, int kind, int S, const void *As, const void *Bs,
                       const int32_t *e, const int32_t *f, double *C, int64_t ldc, bool last_use,
                       cudaStream_t s) {
  const int64_t Kpad = ceil_div(g.K, BK) * BK;
  const auto BF16 = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  int res = 0;
  int st = fused_resident<9, 1>(&res);   // as every kernel of the family: one CTA an SM
  if (st == HSUMMA_OK) st = fused_reserve();
  if (st != HSUMMA_OK) return st;
  if (res > kFusedClusters) res = kFusedClusters;
  // Tiles of 64 columns where all of them fit the device at once and the estimate
  // has them ahead: adding the parts and the rounding, which one cluster does for
  // a tile whatever the number of its parts, are halved, but the MMAs of a block
  // take nearly as long.  64 / 128 columns, kernel alone (us): 4 slices 128^3 14.8
  // / 18.5, 512^3 20.6 / 25.0, 1024^3 31.0 / 33.0, 512 x 512 x 8192 53.4 / 51.5; int8
  // with 8 slices 512^3 29 / 45; 3 slices 1000 x 1000 x 4000 62 / 57.5 (not taken).
  auto col_tiles = [&](int tn) {
    return (int)(g.cyc ? ceil_div(g.N, tn)
                       : g.N / g.Nt * ceil_div(g.Nt, tn) + ceil_div(g.N % g.Nt, tn));
  };
  const int nsub = (int)ceil_div(g.Mt, TM);
  // (blocks: the processors' that hold rows or columns, the last one short)
  const int ntr = (int)(g.cyc ? ceil_div(g.M, TM)
                              : g.M / g.Mt * nsub + ceil_div(g.M % g.Mt, TM));
  const int kblocks = (int)(Kpad / BK);
  const int64_t wide_tiles = (int64_t)((ntr + 1) / 2) * col_tiles(TN),
                narrow_tiles = (int64_t)((ntr + 1) / 2) * col_tiles(64);
  const bool narrow = narrow_tiles <= res &&
                      split_remainder((int)narrow_tiles, kblocks, res, S, 64).cycles <
                          split_remainder((int)wide_tiles, kblocks, res, S, TN).cycles;
  const int width = narrow ? 64 : TN;
  CUtensorMap tA, tB;
  if (!encode_tmap_3d(&tA, BF16, 2, As, Kpad, g.M, S, BK, TM, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_tmap_3d(&tB, BF16, 2, Bs, Kpad, g.N, S, BK, width / 2, CU_TENSOR_MAP_SWIZZLE_128B))
    return HSUMMA_ERR_ARG;
  FusedParams p{};
  uint8_t *buf = static_cast<uint8_t *>(state().fused_buf);
  p.part = reinterpret_cast<unsigned long long *>(buf);
  p.missed = reinterpret_cast<unsigned long long *>(buf + kSumBytes);
  p.low = reinterpret_cast<uint32_t *>(buf + kSumBytes + kMissedBytes);
  p.arrived = reinterpret_cast<int *>(buf + kCountsAt);
  p.finished = last_use ? p.arrived + kCounts : nullptr;
  const int w = slice_width(kind, S), tn = kind == HSUMMA_BF16_SLICES ? 256 : 128;
  p.C = C;
  p.ldc = ldc;
  p.e = e;
  p.f = f;
  p.M = g.M;
  p.N = g.N;
  p.Mt = g.Mt;
  p.Nt = g.Nt;
  p.cyc = g.cyc;
  p.nsub = nsub;
  p.ncol = (int)ceil_div(g.Nt, width);
  p.ntr = ntr;
  p.ntc = col_tiles(width);
  p.kblocks = kblocks;
  p.expo = -w * (S + 1);
  schedule_counters(g, tn, (int64_t)S * (S + 1) / 2, p.sched);
  p.counters = state().d_counters;
  p.big = fused_big_digits();
  p.status = state().d_status;
  // Bands of whole rounds, one launch each: long products of many rounds come
  // back into step at every launch (resident clusters drift apart along k, and
  // past what the L2 holds of the panels they share each reads its own).
  const int policy = state().pair_launch & 0xf;
  const bool bands = policy == HSUMMA_PAIR_LAUNCH_PER_DIAGONAL ||
                     (policy == HSUMMA_PAIR_LAUNCH_AUTO &&
                      wide_tiles >= 48ll * (state().sm_count / 2) &&
                      (int64_t)(S * (S + 1) / 2) * Kpad >= 10 * 16384);
  const int nbands = bands ? S + 1 : 1;
  return narrow ? launch_fused_narrow(w, S, tA, tB, p, nbands, s)
                : launch_fused_kernel(w, S, tA, tB, p, nbands, s);
}

}  // namespace hs
