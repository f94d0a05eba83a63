// Split-precision HSUMMA, steps 3 and 4 in one kernel on CTA pairs: the kept
// slice-pair products of a tile, summed exactly and rounded once into C.
//
// A CTA pair (tcgen05 cta_group::2) computes a tile of 256 rows (two row tiles
// of 128, one per SM) by TN = 128 columns of C (64 for products of few tiles).  Per block of 64 k-columns each SM
// loads its 128 rows of every A slice and half (64 columns) of every B slice
// once, and the pair MMAs (256 x 128 x 16) run every kept slice pair of the
// block from those panels: S (S + 1) / 2 products from 2 S panels, where a
// launch per slice pair or per diagonal copies 2 panels for every pair.  At
// S = 4 an SM takes in 96 KB per 40 MMAs (2560 tensor cycles), 38 B per cycle,
// against 64 B for one pair at a time with twice the tile width.
//
// Sums.  Every diagonal d = s + t has its own accumulator of 128 columns of
// tensor memory (four of them fill it).  A chunk of at most 2^(26-2w) products
// is exact in fp32 (256 for 9-bit digits: 16 MMAs; 1024 for 8-bit, 4096 for
// 7-bit ones); a diagonal with more MMAs than that in one block is dealt to two
// accumulators, one with fewer keeps its accumulator open over several blocks.
// While one diagonal's accumulator is drained the MMAs run on the others, so
// four single accumulators do what two pairs of buffers would.  The drain warps
// add each chunk, shifted by its diagonal's weight, into one 64-bit integer per
// element, X = sum_d D_d 2^(w (dmax - d)) (one multiply-add each): the diagonal
// sums are never stored, and C = RN(2^(e_i + f_j - w (S+1)) X) leaves the kernel.
// Where four accumulators or 64 bits are not enough (S >= 5) a tile takes two
// passes over k, the low diagonals' sum (largest weights) second; the first
// pass's X goes on into it divided by their weights' ratio, and the bits below
// (at most 28) wait in memory for the rounding.
//
// Work.  One persistent cluster per resident slot sweeps whole tiles round
// robin (walked down columns of 8 tile pairs); the tiles past the last whole
// round are cut along k into equal parts for as many clusters as take least time
// by an estimate.  Each part's X goes to memory, and warp by warp the last part to
// arrive adds the others' to its own (integers: the order does not matter) and
// rounds.  (64-bit atomics into one place took 60,000 cycles at 512^3, where
// storing, arriving and adding three other parts take 14,000.)
//
// Roles (640 threads): warp 0 issues the copies, warp 1 the MMAs (leader CTA
// only), warps 2 and 3 idle, warps 4..19 drain: a warp reads the tensor-memory
// lanes of its quarter (warp mod 4) and a quarter of the 128 columns, 32 sums of
// 64 bits a thread.  The issuing warpgroup gives registers to the draining ones.
// The ring has 9 slots of one slice each (A 128 x 64 and B 64 x 64, 24 KB), more
// than two blocks at S = 4; a slot is released by its slice's last pair.
//
// What bounds it: the MMAs where K is large (16384^3 with 4 slices: the power
// limit); otherwise the rounding of a tile, 16384 entries a CTA, during which the
// MMAs get no further than the four accumulators.  It is bound by the integer
// units and the 64-bit conversion: 10,000 cycles with one pass, 16,000 with two
// (33,000 with 128-bit sums and a trip of both passes' X through memory).
// Every wait is bounded (4 s) and ends in an error status.
//
// The including file sets TN, a tile's columns.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "internal.h"
#include "ptx.cuh"
#include "round_scaled.cuh"
#include "tc05.cuh"
#include "../../include/hsumma.h"

namespace hs {

struct FusedParams {
  double *C;
  const int32_t *e, *f;
  int64_t ldc, M, N, Mt, Nt;
  int cyc, nsub, ncol;           // block layout: row / column tiles per processor
  int ntr, ntc, kblocks;         // row tiles, column tiles, blocks of 64 k
  int expo;                      // exponent offset -w (S + 1)
  int L0, L1;                    // whole tiles of this launch
  int R0, nrem, nc;              // first remainder tile, their number, clusters sharing them
  uint32_t bound[kFusedClusters + 1];   // cluster c's windows [bound[c], bound[c + 1])
  unsigned long long *part;      // [cluster][item][CTA]: X [COLS / 2][512][2], low words [COLS][512]
  int *arrived;                  // [tile][CTA][warp] parts that have arrived, zero between
                                 // launches
  unsigned long long *missed;    // [CTA of the grid]: what large chunks add [COLS][512], zero
                                 // between tiles (apart from all else: its place depends on TN)
  uint32_t *low;                 // [CTA of the grid]: low words [COLS][512]
  unsigned long long sched[5];   // the schedule's panel-load counters
  unsigned long long *counters;
  int *big;                      // non-zero: digits too large for chunks of twice the length;
                                 // beside it a word that a launch which gives up sets
  int *finished;                 // CTAs that are done, where the last one clears *big (else null)
  int *status;
};


// The clusters that share nrem tiles of tn columns, and the estimated cycles: a
// window of two blocks of MMAs (256 cycles a slice pair and block; 232 with 64
// columns, which issue and the copies of A bound), rounding a tile, and where tiles are cut storing a
// part and loading those of a tile.
struct RemainderSplit {
  int clusters;
  int64_t cycles;
};
inline RemainderSplit split_remainder(int nrem, int kblocks, int res, int S, int tn) {
  const int npairs = S * (S + 1) / 2, npass = S <= 4 ? 1 : 2;
  const int64_t window = tn == 128 ? 512 : 464, round = tn * (npass == 1 ? 100 : 150);
  const int64_t store = tn * 60 * npass, load = tn * 26 * npass;
  const int64_t T = (int64_t)nrem * ((kblocks + 1) / 2), most = T < res ? T : res;
  RemainderSplit best{nrem, INT64_MAX};
  for (int64_t n = nrem; n <= most; ++n) {
    const int64_t t = ceil_div(T, n) * window * npairs + round +
                      (n == nrem ? 0 : store + load * (ceil_div(n, nrem) - 1));
    if (t < best.cycles) best = {(int)n, t};
  }
  return best;
}
int launch_fused_narrow(int w, int S, const CUtensorMap &tA, const CUtensorMap &tB, FusedParams &p,
                        int nbands, cudaStream_t s);

namespace {

constexpr int TM = 128, HN = TN / 2, BK = 64;
constexpr int A_BYTES = TM * BK * 2, B_BYTES = HN * BK * 2;
constexpr int UNIT_BYTES = A_BYTES + B_BYTES;          // one slice of A and half of B
constexpr int SLOTS = 9;
constexpr int NEPI = 16, NDRAIN = NEPI * 32;           // draining warps and threads
constexpr int COLS = 4 * TN / NEPI;                    // columns of a drain warp
constexpr int EPI = 8;                                 // entries of C a thread rounds at a time
static_assert(COLS % EPI == 0 && COLS <= 32, "a lane holds one column's exponent");
constexpr int NTHREADS = (4 + NEPI) * 32;             // copy, MMA, two idle warps; drain warps
constexpr int ISSUE_REGS = 64, DRAIN_REGS = 104;       // 128 x 64 + 512 x 104 = 640 x 96
constexpr int MAXACC = 4;
constexpr uint32_t TMEM_COLS = 512;
constexpr int SMEM_BYTES = SLOTS * UNIT_BYTES + 1024 + 256;
constexpr uint32_t IDESC = idesc_bf16_f32(2 * TM, TN);
constexpr int kMaxOps = 36;                            // S = 8: 36 slice pairs
constexpr int kTileWords = TM * TN;                    // X of one CTA's half of a tile
// A part of a tile's half: 64-bit X and 32-bit low words.
constexpr int kPartWords = kTileWords + kTileWords / 2;
constexpr int kParts = 2;                              // partial tiles a cluster holds at most

// One slice pair of a pass: 4 MMAs per block.
struct PairOp {
  int s, t;            // slices of A and B, as units of the block
  int rel0, rel1;      // units whose last use this is (-1: none)
  int ready;           // units of the block that the pairs up to this one need
  int acc;             // its accumulator
  bool first, last;    // of its accumulator's pairs in the block
};
struct Pass {
  int ns, na;                    // slices (units per block), accumulators
  int nops;
  PairOp op[kMaxOps];
  int slice[8];                  // the slice (0-based) of each unit, in order of first use
  int blocks[MAXACC];            // blocks per chunk of an accumulator
  int longer[MAXACC];            // and where the digits allow twice the chunk
  int shift[MAXACC];             // weight w (dmax - d) of its diagonal, in bits
  int alt[MAXACC];               // a second buffer for every other chunk (-1: none)
};

// Diagonals dlo..dhi of slices of w bits as one pass.  The schedule is a
// compile-time table: the MMA warp's loop over a block is straight-line code
// (read at run time from the launch parameters it cost about 600 cycles a pair,
// against the 256 of its MMAs).
//
// Order of the pairs.  The copies run ahead by what the ring holds beyond a block,
// so with many slices a slot should be free early and needed late: outer slices
// first, (ns, 1), (1, ns), (ns-1, 1), .., which frees the slots one after the
// other (by diagonals, most are free only at the block's end).  With five slices
// or fewer the ring holds nearly two blocks, and what counts is the time from an
// accumulator's last pair in a block to its first in the next, the more the
// shorter its chunks are: diagonal by diagonal.  1024 x 2432 x 8192 (one tile a
// cluster), by diagonals / by slices: int8 S = 8 744 / 651 us, S = 6 402 / 388,
// S = 5 291 / 291; bf16 S = 6 (9-bit digits, chunks of two blocks) 438 / 451.
//
// Accumulators are numbered by their last pair in the block, the order in which
// they are drained.  One that nothing uses serves as a second buffer of the one
// whose pairs come round soonest.
__host__ __device__ constexpr Pass make_pass(int dlo, int dhi, int w) {
  Pass p{};
  const int cap = bf16_chunk_products(w) / 16;   // MMAs of an exact chunk
  const int per = BK / 16;                       // MMAs of a pair per block
  p.ns = dhi - 1;
  int s[kMaxOps] = {}, t[kMaxOps] = {};
  if (w < 9 && p.ns > 5) {
    for (int hi = p.ns; hi >= 1; --hi)
      for (int lo = 1; lo <= hi; ++lo) {
        if (hi + lo < dlo || hi + lo > dhi) continue;
        s[p.nops] = hi, t[p.nops++] = lo;
        if (lo < hi) s[p.nops] = lo, t[p.nops++] = hi;
      }
  } else {
    for (int d = dlo; d <= dhi; ++d)
      for (int lo = 1; 2 * lo <= d; ++lo) {
        // outer pairs first: in the last diagonal they free the outer slices
        s[p.nops] = lo, t[p.nops++] = d - lo;
        if (2 * lo < d) s[p.nops] = d - lo, t[p.nops++] = lo;
      }
  }
  // units in order of first use, and the pairs that use one last
  int unit[9] = {}, nu = 0;
  for (int o = 0; o < p.nops; ++o) {
    PairOp &op = p.op[o];
    for (int x : {s[o], t[o]})
      if (unit[x] == 0) {
        p.slice[nu] = x - 1;
        unit[x] = ++nu;
      }
    op.s = unit[s[o]] - 1;
    op.t = unit[t[o]] - 1;
    op.ready = nu;
    op.rel0 = op.rel1 = -1;
  }
  bool used[8] = {};
  for (int o = p.nops - 1; o >= 0; --o) {
    PairOp &op = p.op[o];
    if (!used[op.s]) op.rel0 = op.s;
    used[op.s] = true;
    if (!used[op.t]) op.rel1 = op.t;
    used[op.t] = true;
  }
  // a diagonal's pairs dealt to as many accumulators as its block of MMAs needs
  int acc[kMaxOps] = {}, diag[MAXACC] = {}, size[MAXACC] = {}, end[MAXACC] = {}, begin[MAXACC] = {};
  for (int d = dlo; d <= dhi; ++d) {
    const int np = d - 1, parts = (np * per + cap - 1) / cap;
    int i = 0, n = 0;   // part, pairs of the diagonal so far
    for (int o = 0; o < p.nops; ++o) {
      if (s[o] + t[o] != d) continue;
      while (n >= np * (i + 1) / parts) ++i;
      const int x = p.na + i;
      acc[o] = x;
      diag[x] = d;
      if (size[x]++ == 0) begin[x] = o;
      end[x] = o;
      ++n;
    }
    p.na += parts;
  }
  int rank[MAXACC] = {};
  for (int x = 0; x < p.na; ++x)
    for (int y = 0; y < p.na; ++y) rank[x] += end[y] < end[x] ? 1 : 0;
  int slack[MAXACC] = {};
  for (int x = 0; x < p.na; ++x) {
    const int a = rank[x], d = diag[x];
    // the leading slices' product may have one sign: at half the chunk its sums
    // stay below the drain's quick bound for digits of half the largest
    p.blocks[a] = cap / (size[x] * per * (d == 2 && cap >= 2 * per ? 2 : 1));
    // twice the chunk (see fused_big_digits): whole windows of two blocks, half as
    // many again where one pair has the accumulator for itself
    p.longer[a] = p.blocks[a];
    if (cap == 16) {
      const int b = 8 / size[x] / 2 * 2;
      p.longer[a] = d == 2 && b > 4 ? 4 : b;
    }
    p.shift[a] = w * (dhi - d);
    p.alt[a] = -1;
    slack[a] = p.nops - end[x] + begin[x];
  }
  for (int o = 0; o < p.nops; ++o) {
    p.op[o].acc = rank[acc[o]];
    p.op[o].first = o == begin[acc[o]];
    p.op[o].last = o == end[acc[o]];
  }
  for (int spare = p.na; spare < MAXACC; ++spare) {
    int best = -1;
    for (int a = 0; a < p.na; ++a)
      if (p.alt[a] < 0 && (best < 0 || slack[a] < slack[best])) best = a;
    if (best >= 0) p.alt[best] = spare;
  }
  return p;
}

template <int DLO, int DHI, int W>
struct PassTable {
  static constexpr Pass p = make_pass(DLO, DHI, W);
};

// f(integral_constant<int, I>) for I in [I, N)
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F &&f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// S slices of W bits: up to four diagonals share one pass; from five on the low
// diagonals (largest weights) take a second one.
template <int W, int S>
struct Plan {
  static constexpr int top = S + 1;
  static constexpr int npass = S <= 4 ? 1 : 2;
  static constexpr int low = S <= 4 ? top : (S == 5 ? 4 : 5);   // top diagonal of the last pass
  __host__ __device__ static constexpr int dlo(int ps) { return npass == 2 && ps == 0 ? low + 1 : 2; }
  __host__ __device__ static constexpr int dhi(int ps) { return npass == 2 && ps == 0 ? top : low; }
  // a pass's slices in the order of its units, four bits each
  __host__ __device__ static constexpr uint32_t units(int ps) {
    const Pass p = make_pass(dlo(ps), dhi(ps), W);
    uint32_t v = 0;
    for (int u = 0; u < p.ns; ++u) v |= (uint32_t)p.slice[u] << (4 * u);
    return v;
  }
  static constexpr int hi_shift = npass == 2 ? W * (top - low) : 1;   // weight of the last pass
};

__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity,
                                              volatile int *abort_flag) {
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if (*abort_flag) return false;
    if (globaltimer() - t0 > kWaitLimitNs) return false;
  }
}

// one answer for the warp's 32 lanes; the first try needs no clock
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity,
                                          volatile int *abort_flag) {
  if (__all_sync(0xffffffffu, mbar_try_wait_cluster(bar, parity))) return true;
  return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort_flag));
}

// Work item i of cluster cid: tile L, blocks [k0, k1); false past the last one.
__device__ __forceinline__ bool work_item(const FusedParams &p, int cid, int ncl, int i, int *L,
                                          int *k0, int *k1) {
  const int n = p.L1 - p.L0;
  const int nw = n > cid ? (n - cid + ncl - 1) / ncl : 0;
  if (i < nw) {
    *L = p.L0 + cid + i * ncl;
    *k0 = 0;
    *k1 = p.kblocks;
    return true;
  }
  if (cid >= p.nc) return false;
  const int ku = (p.kblocks + 1) / 2;        // parts are whole windows of two blocks
  const uint32_t lo = p.bound[cid], hi = p.bound[cid + 1];
  const uint32_t t = lo / ku + (i - nw), b = t * ku;
  if (b >= hi) return false;
  *L = p.R0 + (int)t;
  *k0 = 2 * (int)(max(lo, b) - b);
  *k1 = min(p.kblocks, 2 * (int)(min(hi, b + ku) - b));
  return true;
}

// The part of remainder tile t that cluster c holds is item t - first tile of
// c's range; a cluster has at most kParts.
__device__ __forceinline__ int part_item(const FusedParams &p, int c, int t) {
  return t - (int)(p.bound[c] / (uint32_t)((p.kblocks + 1) / 2));
}

// tile L -> row tile of this CTA and column tile: tile pairs walked down
// columns of 8
__device__ __forceinline__ void tile_place(const FusedParams &p, int L, int ry, int *rt, int *ct) {
  const int rows = 8, nrp = (p.ntr + 1) / 2;
  const int group = L / (rows * p.ntc);
  const int in_group = min(rows, nrp - group * rows);
  const int idx = L - group * rows * p.ntc;
  *rt = (group * rows + idx % in_group) * 2 + ry;
  *ct = idx / in_group;
}

__device__ __forceinline__ void tile_origin(bool cyc, int i, int per, int width, int64_t blk,
                                            int64_t len, int64_t *org, int64_t *hi) {
  if (cyc) {
    *org = (int64_t)i * width;
    *hi = len;
  } else {
    const int r = i / per;
    *org = r * blk + (int64_t)(i - r * per) * width;
    *hi = imin64(len, (r + 1) * blk);
  }
}

// 16 drained fp32 sums added into 64-bit X with weight 2^SH.  A value below 2^22
// in magnitude converts by one add of 1.5 2^23 (its bits are then those of the
// constant plus the value); each X takes the constant's bits too, which the
// caller subtracts once at the end (`bias`).  With a constant SH > 0 the shift
// and the 64-bit add are one multiply-add (a weight of 1 takes two adds on the
// busier pipe, so every pass carries X doubled, kGuard, and halves it at the
// end).
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr int kGuard = 1;
template <int SH>
__device__ __forceinline__ void add_chunk16(unsigned long long *X, const uint32_t (&v)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint32_t y = __float_as_uint(__uint_as_float(v[i]) + 12582912.f);
    X[i] += (unsigned long long)y << SH;
  }
}
// the largest magnitude
__device__ __forceinline__ void max_chunk16(const uint32_t (&v)[16], float &mx) {
#pragma unroll
  for (int i = 0; i < 16; i += 2)
    asm("max.f32 %0, %1, %2, %0;"
        : "+f"(mx)
        : "f"(fabsf(__uint_as_float(v[i]))), "f"(fabsf(__uint_as_float(v[i + 1]))));
}

// What those adds missed of a chunk that holds larger values: the warp's columns at
// `ta` are read again, and the difference goes to the sums' memory (not to X:
// a second, rare definition of X would cost the common path a move per word).
static __device__ __noinline__ void add_missed(uint32_t ta, unsigned long long *sums, int shift) {
#pragma unroll 1
  for (int j = 0; j < COLS; j += 16) {
    uint32_t v[16];
    tmem_ld16(ta + j, v);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float x = __uint_as_float(v[i]);
      const long long miss = (long long)__float2int_rn(x) + (long long)kMagicBits -
                             (long long)__float_as_uint(x + 12582912.f);
      if (miss) atomicAdd(sums + (j + i) * NDRAIN, (unsigned long long)miss << shift);
    }
  }
}

struct MmaState {
  uint32_t ring, bars;   // shared-memory addresses: slots; full barriers
  uint32_t tmem;
  int base;              // ring slot of the block's first unit
  uint32_t phase;        // parity of its full barrier
  uint32_t acc_ph;       // parity bits of the accumulators' hand-backs
  bool el;
};
// full[SLOTS], empty[SLOTS], acc_full[MAXACC], acc_empty[MAXACC], 8 bytes each
constexpr uint32_t kEmptyOff = 8 * SLOTS, kAccFullOff = 16 * SLOTS,
                   kAccEmptyOff = kAccFullOff + 8 * MAXACC;

__device__ __forceinline__ uint64_t desc_from(uint32_t lo) {
  // sdesc_k128 with its address field and the two constant halves formed apart
  constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
  return ((uint64_t)hi << 32) | lo;
}

// The pair MMAs of blocks [k0, k1) of one pass; false when a wait ran out.
template <int DLO, int DHI, int W>
__device__ __forceinline__ bool mma_pass(MmaState &m, int k0, int k1, bool twice, int *status,
                                         volatile int *abort_flag) {
  using PS = PassTable<DLO, DHI, W>;
  constexpr int ns = PS::p.ns;
  int cnt[MAXACC] = {}, buf[MAXACC] = {0, 1, 2, 3};
  bool ok = true;
  for (int kb = k0; kb < k1 && ok; ++kb) {
    uint32_t lo[8], bar[8];   // descriptor word and full barrier of each unit
    static_for<0, ns>([&](auto iu) {
      constexpr int u = iu.value;
      const int x = m.base + u, sl = x >= SLOTS ? x - SLOTS : x;
      lo[u] = ((m.ring + sl * UNIT_BYTES) >> 4) | (1u << 16);
      bar[u] = m.bars + 8 * sl;
    });
    static_for<0, PS::p.nops>([&](auto io) {
      constexpr int o = io.value;
      constexpr PairOp op = PS::p.op[o];
      constexpr int a = op.acc, b1 = PS::p.blocks[a], b2 = PS::p.longer[a], alt = PS::p.alt[a];
      if (!ok) return;
      uint32_t accum = 1;
      if (op.first && cnt[a] == 0) {
        if (!warp_wait(m.bars + kAccEmptyOff + 8 * buf[a], ((m.acc_ph >> buf[a]) & 1u) ^ 1u,
                       abort_flag)) {
          if (!*abort_flag) record_error(status, HSUMMA_ERR_TIMEOUT, kSiteAccEmpty);
          ok = false;
          return;
        }
        m.acc_ph ^= 1u << buf[a];
        accum = 0;
        tc_fence_after();
      }
      // units that an earlier pair has not waited for
      constexpr int ready = o ? PS::p.op[o ? o - 1 : 0].ready : 0, need = op.ready;
      static_for<ready, need>([&](auto iu) {
        constexpr int u = iu.value;
        ok = ok && warp_wait(bar[u], m.phase ^ (m.base + u >= SLOTS ? 1u : 0u), abort_flag);
      });
      if constexpr (need > ready) {
        if (!ok && !*abort_flag) record_error(status, HSUMMA_ERR_TIMEOUT, kSiteFull);
        tc_fence_after();
      }
      if (!ok) return;
      if (m.el) {
        const uint32_t dt = m.tmem + (uint32_t)(buf[a] * TN);
        const uint32_t al = lo[op.s], bl = lo[op.t] + (A_BYTES >> 4);
#pragma unroll
        for (int k = 0; k < BK / 16; ++k)
          mma2_bf16(dt, desc_from(al + 2 * k), desc_from(bl + 2 * k), IDESC, k ? 1u : accum);
        if constexpr (op.rel0 >= 0) mma2_commit_mc(bar[op.rel0] + kEmptyOff, (uint16_t)3u);
        if constexpr (op.rel1 >= 0) mma2_commit_mc(bar[op.rel1] + kEmptyOff, (uint16_t)3u);
      }
      __syncwarp();
      if constexpr (op.last) {
        if (++cnt[a] == (twice ? b2 : b1) || kb + 1 == k1) {
          if (m.el) mma2_commit_mc(m.bars + kAccFullOff + 8 * buf[a], (uint16_t)3u);
          __syncwarp();
          cnt[a] = 0;
          if constexpr (alt >= 0) buf[a] ^= a ^ alt;
        }
      }
    });
    m.base += ns;
    if (m.base >= SLOTS) {
      m.base -= SLOTS;
      m.phase ^= 1u;
    }
  }
  return ok;
}

struct DrainState {
  uint32_t bars, tmem;   // barriers; this warp's lanes and columns of accumulator 0
  uint32_t full_ph;      // parity bits of the accumulators
  bool leader;
};

// Adds blocks [k0, k1) of one pass to X of this thread's elements; what large
// chunks add goes through `sums`, at zero before and after.
template <int DLO, int DHI, int W>
__device__ __forceinline__ bool drain_pass(DrainState &t, int k0, int k1, bool twice, int lane,
                                           unsigned long long (&X)[COLS],
                                           unsigned long long *sums, volatile int *abort_flag) {
  using PS = PassTable<DLO, DHI, W>;
  constexpr int na = PS::p.na;
  int cnt[MAXACC] = {}, buf[MAXACC] = {0, 1, 2, 3};
  unsigned long long bias = 0;
#pragma unroll
  for (int i = 0; i < COLS; ++i) X[i] <<= kGuard;
  bool ok = true, missed = false;
  for (int kb = k0; kb < k1 && ok; ++kb) {
    static_for<0, na>([&](auto ia) {
      constexpr int a = ia.value;
      constexpr int b1 = PS::p.blocks[a], b2 = PS::p.longer[a], alt = PS::p.alt[a];
      const int blocks = twice ? b2 : b1;
      if (!ok || (++cnt[a] != blocks && kb + 1 != k1)) return;
      cnt[a] = 0;
      if (!warp_wait(t.bars + kAccFullOff + 8 * buf[a], (t.full_ph >> buf[a]) & 1u, abort_flag)) {
        ok = false;
        return;
      }
      t.full_ph ^= 1u << buf[a];
      tc_fence_after();
      const uint32_t ta = t.tmem + buf[a] * TN;
      constexpr int sh = PS::p.shift[a] + kGuard;
      float mx = 0.f;
      uint32_t v[16];
      tmem_ld16(ta, v);
      tmem_ld_wait();
      max_chunk16(v, mx);
      if constexpr (COLS == 32) {
        add_chunk16<sh>(X, v);
        tmem_ld16(ta + 16, v);
        tmem_ld_wait();
        max_chunk16(v, mx);
      }
      if (__any_sync(0xffffffffu, !(mx < kFastDrainBound))) {
        add_missed(ta, sums, sh);
        missed = true;
        tmem_ld16(ta + COLS - 16, v);        // not kept over the call
        tmem_ld_wait();
      }
      // hand the accumulator back (nothing was written, so no release ordering
      // is needed), then add the rest
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        const uint32_t eb = t.bars + kAccEmptyOff + 8 * buf[a];
        if (t.leader)
          mbar_arrive(eb);
        else
          mbar_arrive_cluster_relaxed(eb, 0u);
      }
      if constexpr (alt >= 0) buf[a] ^= a ^ alt;
      add_chunk16<sh>(X + COLS - 16, v);
      bias += (unsigned long long)kMagicBits << sh;
    });
  }
  if (!ok) return false;
  // what large chunks add comes before the halving: without it X may be past 64 bits
  // (a chunk below -1.5 2^23 first counts as about 2^31), with it X is twice the sum
  if (missed) {
#pragma unroll
    for (int i = 0; i < COLS; ++i) {
      X[i] += __ldcg(sums + i * NDRAIN);
      sums[i * NDRAIN] = 0;
    }
  }
#pragma unroll
  for (int i = 0; i < COLS; ++i) X[i] = (unsigned long long)((long long)(X[i] - bias) >> kGuard);
  return true;
}

// C entry i of a thread from its exact sum, X 2^HS + low with two passes: any
// exponent, and exponents from kScaleLo to kScaleHi - 32
template <int NPASS, int HS>
static __device__ __noinline__ double entry_any(unsigned long long X, uint32_t low, int k) {
  return NPASS == 1 ? round_scaled64((long long)X, k)
                    : round_scaled(((__int128)(long long)X << HS) + low, k);
}
template <int NPASS, int HS>
__device__ __forceinline__ double entry(unsigned long long X, uint32_t low, int k, int i) {
  if constexpr (NPASS == 2) return round_scaled_ext<HS>(X, low, k);
  // one entry of four in integers: both units are busy as long (4096 x 4096 x 64
  // with 4 slices takes 63.8 us, 65.8 with half of them, 71.4 with all)
  return i % 4 == 1 ? round_scaled_int((long long)X, k) : round_scaled_cvt((long long)X, k);
}

// Transposes a 4 x 4 block over four neighbouring lanes (lane's c[u] to lane u's
// c[lane]).
__device__ __forceinline__ void transpose4(double (&c)[4], int lane) {
#pragma unroll
  for (int d = 1; d <= 2; d *= 2) {
    const bool up = lane & d;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (u & d) continue;
      const double other = __shfl_xor_sync(0xffffffffu, up ? c[u] : c[u + d], d);
      if (up) c[u] = other;
      else c[u + d] = other;
    }
  }
}

template <int W, int S>
__global__ void __launch_bounds__(NTHREADS, 1)
    split_fused_kernel(const __grid_constant__ CUtensorMap tmA,
                       const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ FusedParams p) {
  using PL = Plan<W, S>;
  constexpr int NPASS = PL::npass;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + SLOTS * UNIT_BYTES);
  uint64_t *empty = full + SLOTS;
  uint64_t *acc_full = empty + SLOTS, *acc_empty = acc_full + MAXACC;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + MAXACC);
  __shared__ volatile int abort_flag;
  // whether the chunks are of twice the length, and a barrier that says it is known
  __shared__ int twice_word;
  __shared__ uint64_t twice_known;

  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);   // warp-uniform
  const int ry = (int)cluster_ctarank();          // member of the pair
  const bool leader = ry == 0;
  const int ncl = (int)gridDim.x / 2, cid = (int)blockIdx.x / 2;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int a = 0; a < MAXACC; ++a) {
      mbar_init(smem_u32(&acc_full[a]), 1);
      mbar_init(smem_u32(&acc_empty[a]), 2 * NEPI);
    }
    mbar_init(smem_u32(&twice_known), 32);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc2(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish2();
  }
  if (threadIdx.x == 0) {
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  cluster_sync();
  // everything above overlaps the end of the digits' kernel (512^3: 1.7 us of 28.8);
  // from here on its results are read and C is written
  wait_for_primary();
  // the digits' answer, from one load for the pair: all who count blocks get the same.
  // The warp in step (a branch of some lanes here cost the roles registers and 2 % of
  // 3001 x 2047 x 2500 with 5 slices), the MMA warp's wait here (in its role it cost
  // 24576 x 16384 x 32768 with 5 slices 2-4 %) and the draining warps' in theirs: 512^3
  // with 4 slices 22.4 us where all wait here, 21.3 so (21.5 where every thread loads
  // the word by itself).
  if (W == 9 && leader && warp == 2) {
    const uint32_t word = *p.big == 0;
    for (uint32_t r = 0; r < 2; ++r) {
      st_shared_cluster_u32(smem_u32(&twice_word), r, word);
      mbar_arrive_cluster(smem_u32(&twice_known), r);
    }
  }
  if (W == 9 && warp == 1 && leader &&
      !__all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&twice_known), 0u))) {
    record_error(p.status, HSUMMA_ERR_TIMEOUT, kSiteFull);
    abort_flag = 1;
  }
  const bool twice = W == 9 && __all_sync(0xffffffffu, twice_word != 0);   // of the MMA warp

  if (warp < 4) {
    regs_dec<ISSUE_REGS>();
    if (warp == 0) {
      // ---------------- copies (both CTAs): the warp in step, one lane issues ----------------
      const bool el = elect_one();
      int slot = 0;
      uint32_t phase = 0;
      unsigned long long nops = 0;
      bool ok = true;
      int L, k0, k1;
      for (int it = 0; ok && work_item(p, cid, ncl, it, &L, &k0, &k1); ++it) {
        int rt, ct;
        tile_place(p, L, ry, &rt, &ct);
        int64_t m0, mhi, n0, nhi;
        tile_origin(p.cyc, rt, p.nsub, TM, p.Mt, p.M, &m0, &mhi);
        tile_origin(p.cyc, ct, p.ncol, TN, p.Nt, p.N, &n0, &nhi);
        if (rt >= p.ntr) m0 = p.M;                  // no such row tile: zero-filled copies
#pragma unroll 1
        for (int ps = 0; ps < NPASS && ok; ++ps) {
          constexpr uint32_t units0 = PL::units(0), units1 = PL::units(NPASS - 1);
          const uint32_t units = ps ? units1 : units0;
          const int ns = PL::dhi(ps) - 1;
          for (int kb = k0; kb < k1 && ok; ++kb) {
            const int64_t kk = (int64_t)kb * BK;
            for (int u = 0; u < ns; ++u) {
              const int s = (int)(units >> (4 * u)) & 15;
              if (!warp_wait(smem_u32(&empty[slot]), phase ^ 1u, &abort_flag)) {
                if (!abort_flag) record_error(p.status, HSUMMA_ERR_TIMEOUT, kSiteEmpty);
                abort_flag = 1;
                ok = false;
                break;
              }
              const uint32_t a_dst = smem_u32(smem + slot * UNIT_BYTES), b_dst = a_dst + A_BYTES;
              if (el) {
                // the leader's barrier counts the bytes of both CTAs
                const uint32_t fb = smem_u32(&full[slot]);
                if (leader) {
                  mbar_arrive_expect_tx(fb, 2 * UNIT_BYTES);
                  tma_load_3d(a_dst, &tmA, (int32_t)kk, (int32_t)m0, s, fb);
                  tma_load_3d(b_dst, &tmB, (int32_t)kk, (int32_t)n0, s, fb);
                } else {
                  const uint32_t lb = cluster_addr(fb, 0);
                  tma_load_3d_pair(a_dst, &tmA, (int32_t)kk, (int32_t)m0, s, lb);
                  tma_load_3d_pair(b_dst, &tmB, (int32_t)kk, (int32_t)n0 + HN, s, lb);
                }
              }
              __syncwarp();
              nops += 2;
              if (++slot == SLOTS) { slot = 0; phase ^= 1u; }
            }
          }
        }
      }
      // every release of the last slots has landed before leaving
      for (int i = 0; i < SLOTS && ok; ++i) {
        if (!warp_wait(smem_u32(&empty[slot]), phase ^ 1u, &abort_flag)) {
          if (!abort_flag) record_error(p.status, HSUMMA_ERR_TIMEOUT, kSiteEmpty);
          abort_flag = 1;
          ok = false;
        }
        if (++slot == SLOTS) { slot = 0; phase ^= 1u; }
      }
      if (el) {
        if (blockIdx.x == 0)
          for (int i = 0; i < 5; ++i)
            if (p.sched[i]) atomicAdd(&p.counters[i], p.sched[i]);
        atomicAdd(&p.counters[5], nops);
      }
    } else if (warp == 1 && leader) {
      // ---------------- pair MMAs: the warp in step, one lane issues ----------------
      MmaState m{smem_u32(smem), smem_u32(full), tmem_base, 0, 0u, 0u, elect_one()};
      bool ok = true;
      int L, k0, k1;
      for (int it = 0; ok && work_item(p, cid, ncl, it, &L, &k0, &k1); ++it) {
        ok = mma_pass<PL::dlo(0), PL::dhi(0), W>(m, k0, k1, twice, p.status, &abort_flag);
        if constexpr (NPASS == 2)
          ok = ok && mma_pass<PL::dlo(1), PL::dhi(1), W>(m, k0, k1, twice, p.status, &abort_flag);
        if (!ok) abort_flag = 1;
      }
    }
  } else {
    regs_inc<DRAIN_REGS>();
    // ---------------- drain, recombination, C (both CTAs) ----------------
    constexpr uint32_t kLowMask = (1u << PL::hi_shift) - 1;
    const int q = warp & 3;                 // tensor-memory lane quarter of this warp
    const int h = (warp - 4) >> 2;          // quarter of the tile's columns
    const int tid = (int)threadIdx.x - 128;
    unsigned long long *mine = p.missed + (int64_t)blockIdx.x * kTileWords + tid;
    uint32_t *const mylow = p.low + (int64_t)blockIdx.x * kTileWords + tid;
    DrainState dr{smem_u32(full), tmem_base + ((uint32_t)(q * 32) << 16) + h * COLS, 0u, leader};
    bool ok = true;
    if (W == 9 && !warp_wait(smem_u32(&twice_known), 0u, &abort_flag)) ok = false;
    const bool twice = W == 9 && __all_sync(0xffffffffu, twice_word != 0);
    int L, k0, k1;
    for (int it = 0; ok && work_item(p, cid, ncl, it, &L, &k0, &k1); ++it) {
      int rt, ct;
      tile_place(p, L, ry, &rt, &ct);
      int64_t m0, row_hi, t0, col_hi;
      tile_origin(p.cyc, rt, p.nsub, TM, p.Mt, p.M, &m0, &row_hi);
      tile_origin(p.cyc, ct, p.ncol, TN, p.Nt, p.N, &t0, &col_hi);
      if (rt >= p.ntr) row_hi = 0;
      const int64_t row = m0 + q * 32 + lane;
      const int64_t n0 = t0 + h * COLS;
      const bool whole = k0 == 0 && k1 == p.kblocks;
      const int tt = L - p.R0;               // remainder tile
      // where cluster c keeps its part of this tile's half: X, and the low bits of
      // the first pass's
      auto part_of = [&](int c) {
        return p.part + ((int64_t)(c * kParts + part_item(p, c, tt)) * 2 + ry) * kPartWords;
      };
      auto x_of = [&](int c) { return part_of(c) + 2 * tid; };
      auto low_of = [&](int c) {
        return reinterpret_cast<uint32_t *>(part_of(c) + kTileWords) + tid;
      };
      const int nvalid = row < row_hi ? (int)imax64(0, imin64(COLS, col_hi - n0)) : 0;
      const int k = nvalid > 0 ? p.e[row] + p.expo : 0;
      const int fj = n0 + lane < col_hi ? __ldcg(p.f + n0 + lane) : 0;   // of column `lane`
      double *const crow = p.C + row * p.ldc + n0;
      unsigned long long X[COLS];
#pragma unroll
      for (int i = 0; i < COLS; ++i) X[i] = 0;
      auto pass = [&](auto ips) {
        constexpr int ps = ips.value;
        ok = ok && drain_pass<PL::dlo(ps), PL::dhi(ps), W>(dr, k0, k1, twice, lane, X, mine,
                                                           &abort_flag);
        if (!ok) return;
        if (ps + 1 < NPASS) {
          // the last pass goes on from the sum's high part; the low HS bits wait
          uint32_t *const dst = whole ? mylow : low_of(cid);
#pragma unroll
          for (int i = 0; i < COLS; ++i) {
            dst[i * NDRAIN] = (uint32_t)X[i] & kLowMask;
            X[i] = (unsigned long long)((long long)X[i] >> PL::hi_shift);
          }
        }
      };
      static_for<0, NPASS>(pass);
      if (!ok) break;
      if (!whole) {
        ulonglong2 *const dst = reinterpret_cast<ulonglong2 *>(x_of(cid));
#pragma unroll
        for (int i = 0; i < COLS; i += 2)
          dst[i / 2 * NDRAIN] = make_ulonglong2(X[i], X[i + 1]);
        // the last part of this warp's entries to arrive adds the others' sums to
        // its own and rounds (no part waits for another; warp by warp, the parts
        // share that work)
        int c0 = cid, c1 = cid;              // the clusters that share the tile
        const uint32_t ku = (p.kblocks + 1) / 2;
        while (p.bound[c0] > tt * ku) --c0;
        while (p.bound[c1 + 1] < (tt + 1) * ku) ++c1;
        __threadfence();
        __syncwarp();
        int last = 0;
        if (lane == 0) {
          int *const cnt = p.arrived + (tt * 2 + ry) * NEPI + warp - 4;
          last = atomicAdd(cnt, 1) == c1 - c0;
          if (last) *cnt = 0;
        }
        if (!__shfl_sync(0xffffffffu, last, 0)) continue;
        __threadfence();
        if constexpr (NPASS == 2) {
          // the low parts first, their carries into X
          uint32_t low[COLS], carry[COLS];
#pragma unroll
          for (int i = 0; i < COLS; ++i) low[i] = carry[i] = 0;
#pragma unroll 1
          for (int c = c0; c <= c1; ++c) {
            const uint32_t *const src = low_of(c);
#pragma unroll
            for (int i = 0; i < COLS; ++i) {
              low[i] += __ldcg(src + i * NDRAIN);
              carry[i] += low[i] >> PL::hi_shift;
              low[i] &= kLowMask;
            }
          }
#pragma unroll
          for (int i = 0; i < COLS; ++i) {
            mylow[i * NDRAIN] = low[i];
            X[i] = carry[i];
          }
        }
#pragma unroll 1
        for (int c = c0; c <= c1; ++c) {
          if (NPASS == 1 && c == cid) continue;   // X is this part's
          const ulonglong2 *const src = reinterpret_cast<const ulonglong2 *>(x_of(c));
#pragma unroll
          for (int i = 0; i < COLS; i += 2) {
            const ulonglong2 v = __ldcg(src + i / 2 * NDRAIN);
            X[i] += v.x;
            X[i + 1] += v.y;
          }
        }
      }
      // C, a few entries at a time.  A short loop over X, which moves down that
      // many places each time: it runs once a tile, and unrolled its instructions
      // took longer to fetch than to run (as did a trip of X through memory).
      // Exponents that keep every result normal, the common case, take the
      // quick forms.
      const int fl = __reduce_min_sync(0xffffffffu, fj), fh = __reduce_max_sync(0xffffffffu, fj);
      const bool quick =
          __all_sync(0xffffffffu, nvalid == 0 || (k + fl >= kScaleLo && k + fh + 32 <= kScaleHi));
      // 32-byte stores where every row allows them; else four lanes store a row's
      // 32 bytes together, in a quarter of the transactions of a lane a row
      const bool vec =
          __all_sync(0xffffffffu, nvalid == COLS && (reinterpret_cast<uintptr_t>(crow) & 31) == 0);
      // of row (lane & ~3), column (lane & 3) of the warp's
      double *const trow = p.C + (row - (lane & 3)) * p.ldc + n0 + (lane & 3);
#pragma unroll 1
      for (int i = 0; i < COLS; i += EPI) {
        uint32_t fx[EPI] = {};
        if constexpr (NPASS == 2) {
#pragma unroll
          for (int u = 0; u < EPI; ++u) fx[u] = __ldcg(mylow + (i + u) * NDRAIN);
        }
#pragma unroll
        for (int g = 0; g < EPI; g += 4) {
          double c[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int kj = k + __shfl_sync(0xffffffffu, fj, i + g + u);
            c[u] = quick ? entry<NPASS, PL::hi_shift>(X[g + u], fx[g + u], kj, g + u)
                         : entry_any<NPASS, PL::hi_shift>(X[g + u], fx[g + u], kj);
          }
          if (vec) {
            st_global_v4(crow + i + g, c[0], c[1], c[2], c[3]);
          } else {
            transpose4(c, lane);
            const int rows = (int)(row_hi - row) + (lane & 3);   // valid ones from trow on
            if (n0 + i + g + (lane & 3) < col_hi) {
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (u < rows) trow[u * p.ldc + i + g] = c[u];
            }
          }
        }
#pragma unroll
        for (int j = 0; j < COLS - EPI; ++j) X[j] = X[j + EPI];
      }
    }
    if (!ok) {
      if (!abort_flag) record_error(p.status, HSUMMA_ERR_TIMEOUT, kSiteAccFull);
      abort_flag = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (abort_flag) {
    if (threadIdx.x == 0) p.big[1] = 1;        // counts and sums stay behind
    bounded_sleep(2000000ull);                 // in-flight copies and MMAs land
  }
  // both CTAs of the pair are done with tensor memory before it is released
  cluster_sync();
  if (p.finished && threadIdx.x == 0 && atomicAdd(p.finished, 1) == (int)gridDim.x - 1) {
    *p.finished = 0;
    *p.big = 0;
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc2(tmem_base, TMEM_COLS);
  }
  cluster_sync();
}

}  // namespace

template <int W, int S>
static int fused_resident(int *clusters) {
  auto kern = split_fused_kernel<W, S>;
  int &res = state().fused_resident[TN == 128 ? 0 : 1][W == 7 ? 1 : 0][S - 1];
  if (res == 0) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         SMEM_BYTES);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(fused smem)");
    cudaLaunchConfig_t q = {};
    q.gridDim = dim3(2, 1, 1);
    q.blockDim = dim3(NTHREADS, 1, 1);
    q.dynamicSmemBytes = SMEM_BYTES;
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeClusterDimension;
    qa[0].val.clusterDim.x = 2;
    qa[0].val.clusterDim.y = 1;
    qa[0].val.clusterDim.z = 1;
    q.attrs = qa;
    q.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, kern, &q);
    if (e != cudaSuccess || n < 1) {
      set_error("cudaOccupancyMaxActiveClusters(fused kernel): %s (%d clusters)",
                cudaGetErrorString(e), n);
      return HSUMMA_ERR_CUDA;
    }
    res = n;
  }
  *clusters = res;
  return HSUMMA_OK;
}

template <int W, int S>
static int launch_fused(const CUtensorMap &tA, const CUtensorMap &tB, FusedParams &p, int nbands,
                        cudaStream_t s) {
  int res = 0;
  int st = fused_resident<W, S>(&res);
  if (st != HSUMMA_OK) return st;
  if (res > kFusedClusters) res = kFusedClusters;
  const int ntiles = ((p.ntr + 1) / 2) * p.ntc;
  int *const finished = p.finished;
  const int rounds = ntiles / res;
  const int nrem = ntiles - rounds * res;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(NTHREADS, 1, 1);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (nbands > rounds) nbands = rounds > 0 ? rounds : 1;
  for (int b = 0; b < nbands; ++b) {
    const bool last = b + 1 == nbands;
    p.L0 = (int)((int64_t)rounds * b / nbands) * res;
    p.L1 = (int)((int64_t)rounds * (b + 1) / nbands) * res;
    p.R0 = rounds * res;
    p.nrem = last ? nrem : 0;
    p.nc = 0;
    if (p.nrem) {
      const int64_t T = (int64_t)p.nrem * ((p.kblocks + 1) / 2);
      p.nc = split_remainder(p.nrem, p.kblocks, res, S, TN).clusters;
      for (int c = 0; c <= p.nc; ++c) p.bound[c] = (uint32_t)(c * T / p.nc);
    }
    if (b) std::fill(p.sched, p.sched + 5, 0ull);
    p.finished = last ? finished : nullptr;
    const int ncl = p.L1 > p.L0 ? res : p.nc;
    cfg.gridDim = dim3((unsigned)(2 * ncl), 1, 1);
    cudaError_t e = cudaLaunchKernelEx(&cfg, split_fused_kernel<W, S>, tA, tB, p);
    if (e != cudaSuccess) return cuda_fail(e, "launch split_fused_kernel");
    count_launch();
  }
  return HSUMMA_OK;
}


// the kernel of S slices of w bits
static int launch_fused_kernel(int w, int S, const CUtensorMap &tA, const CUtensorMap &tB,
                               FusedParams &p, int nbands, cudaStream_t s) {
#define HS_FUSED(W, SS) \
  if (w == W && S == SS) return launch_fused<W, SS>(tA, tB, p, nbands, s)
  HS_FUSED(9, 1);
  HS_FUSED(9, 2);
  HS_FUSED(9, 3);
  HS_FUSED(9, 4);
  HS_FUSED(9, 5);
  HS_FUSED(9, 6);
  HS_FUSED(8, 7);
  HS_FUSED(7, 1);
  HS_FUSED(7, 2);
  HS_FUSED(7, 3);
  HS_FUSED(7, 4);
  HS_FUSED(7, 5);
  HS_FUSED(7, 6);
  HS_FUSED(7, 7);
  HS_FUSED(7, 8);
#undef HS_FUSED
  set_error("no product kernel for %d slices of %d bits", S, w);
  return HSUMMA_ERR_UNSUPPORTED;
}

}  // namespace hs
