// Learned cost model: a 10 -> 64 -> 64 -> 64 -> 1 MLP with exact GELU,
// trained in fp32 (forward, backpropagation, Adam) and run in bf16 to score the
// candidate configurations of a product.  Not in the paper, which picks the
// group count by sampling a few runs (Section V-A-1, Section VI); this model
// proposes (P, Q, G, b, B) from the features of a shape instead.
//
// Parameter vector layout (row-major W[out][in]):
//   W1[64][10] b1[64] W2[64][64] b2[64] W3[64][64] b3[64] W4[1][64] b4[1]
// Every kernel keeps the weights in shared memory (36 KB).  The scoring ones give
// one sample to each warp (lane j computes neurons j and j + 32); the backward
// pass takes 16 samples a block, and a second kernel sums the blocks' partial
// gradients in a fixed order.
#include <cuda_bf16.h>
#include <cstring>
#include <mutex>

#include "internal.h"
#include "../../include/hsumma.h"

namespace hs {
namespace {

constexpr int NIN = 10, NH = 64;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH,
              OFF_B2 = OFF_W2 + NH * NH, OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH * NH,
              OFF_W4 = OFF_B3 + NH, OFF_B4 = OFF_W4 + NH, NPARAM = OFF_B4 + 1;
static_assert(NPARAM == 9089, "parameter count");
constexpr int WARPS = 8;

__device__ __forceinline__ float gelu(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
// h_out[j] = W[j][:] . h_in + b[j] for this lane's two neurons (j, j + 32);
// h_in lives in shared memory, one row per warp.
template <int NI>
__device__ __forceinline__ void dense2(const float *W, const float *b, const float *h_in,
                                       int lane, float &z0, float &z1) {
  float a0 = b[lane], a1 = b[lane + 32];
#pragma unroll 8
  for (int i = 0; i < NI; ++i) {
    const float x = h_in[i];
    a0 = fmaf(W[lane * NI + i], x, a0);
    a1 = fmaf(W[(lane + 32) * NI + i], x, a1);
  }
  z0 = a0;
  z1 = a1;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(WARPS * 32) mlp_forward_kernel(int batch, const float *theta,
                                                                  const float *X, float *y,
                                                                  float *cache) {
  __shared__ float w[NPARAM];
  __shared__ float h[WARPS][3][NH];
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) w[i] = theta[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int smp = blockIdx.x * WARPS + warp; smp < batch; smp += gridDim.x * WARPS) {
    float *hin = h[warp][0];
    if (lane < NIN) hin[lane] = X[(int64_t)smp * NIN + lane];
    __syncwarp();
    float z0, z1;
    dense2<NIN>(w + OFF_W1, w + OFF_B1, hin, lane, z0, z1);
    if (cache) {
      cache[(int64_t)smp * 192 + lane] = z0;
      cache[(int64_t)smp * 192 + lane + 32] = z1;
    }
    h[warp][1][lane] = gelu(z0);
    h[warp][1][lane + 32] = gelu(z1);
    __syncwarp();
    dense2<NH>(w + OFF_W2, w + OFF_B2, h[warp][1], lane, z0, z1);
    if (cache) {
      cache[(int64_t)smp * 192 + 64 + lane] = z0;
      cache[(int64_t)smp * 192 + 96 + lane] = z1;
    }
    h[warp][2][lane] = gelu(z0);
    h[warp][2][lane + 32] = gelu(z1);
    __syncwarp();
    dense2<NH>(w + OFF_W3, w + OFF_B3, h[warp][2], lane, z0, z1);
    if (cache) {
      cache[(int64_t)smp * 192 + 128 + lane] = z0;
      cache[(int64_t)smp * 192 + 160 + lane] = z1;
    }
    const float out = warp_sum(w[OFF_W4 + lane] * gelu(z0) + w[OFF_W4 + lane + 32] * gelu(z1));
    if (lane == 0) y[smp] = out + w[OFF_B4];
    __syncwarp();
  }
}

// Per-block partial gradient of mean_i (f(x_i) - t_i)^2 (and partial loss).
//
// A block takes TILE samples at a time through small matrix products in shared
// memory: 2 x 33 K multiply-adds a sample with one sample a warp were bound by
// 32-way bank conflicts on the weights and by shared-memory atomics on the
// gradient (229 us for 2400 samples on 300 blocks).  Here the weights' rows are
// padded to an odd stride, activations are [neuron][sample] (four samples of a
// neuron in one load), and each thread keeps its part of the gradient, 4 x 4
// entries of each 64 x 64 matrix, in registers over all the block's tiles.  TILE =
// 16 makes one tile a block and one block an SM of 2400 samples; what is left is
// latency: loading the weights, ten short products in turn, the partials' store.
// A step of this kernel, the sum below and Adam takes 22.6 us for 2400 samples
// (246 before), 21 for 64.
constexpr int TILE = 16;
constexpr int LDW = NH + 1, LDW1 = NIN + 1;   // odd: lanes on rows hit different banks
constexpr int LDH = TILE + 4;                 // 16-byte rows, eight lanes' rows on all banks
struct TrainSmem {
  float x[NIN * LDH], h1[NH * LDH], h2[NH * LDH], h3[NH * LDH];   // [neuron][sample]
  float d1[NH * LDH], d2[NH * LDH], d3[NH * LDH];                 // d loss / d z
  float w2[NH * LDW], w3[NH * LDW], w1[NH * LDW1];
  float b1[NH], b2[NH], b3[NH], w4[NH];
  float gy[TILE], loss[TILE], b4;
};

// z[u] = W[j][:] . h[:][s0 + u] + b[j], the terms in the order of i
template <int NI, int LD>
__device__ __forceinline__ void dense4(const float *W, float b, const float *h, int j, int s0,
                                       float (&z)[4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) z[u] = b;
#pragma unroll 16
  for (int i = 0; i < NI; ++i) {
    const float w = W[j * LD + i];
    const float4 v = *reinterpret_cast<const float4 *>(h + i * LDH + s0);
    z[0] = fmaf(w, v.x, z[0]);
    z[1] = fmaf(w, v.y, z[1]);
    z[2] = fmaf(w, v.z, z[2]);
    z[3] = fmaf(w, v.w, z[3]);
  }
}
// z[u] = sum_o W[o][j] d[o][s0 + u]
__device__ __forceinline__ void dense4_t(const float *W, const float *d, int j, int s0,
                                         float (&z)[4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) z[u] = 0.f;
#pragma unroll 16
  for (int o = 0; o < NH; ++o) {
    const float w = W[o * LDW + j];
    const float4 v = *reinterpret_cast<const float4 *>(d + o * LDH + s0);
    z[0] = fmaf(w, v.x, z[0]);
    z[1] = fmaf(w, v.y, z[1]);
    z[2] = fmaf(w, v.z, z[2]);
    z[3] = fmaf(w, v.w, z[3]);
  }
}
// h = gelu(z) stored, g = gelu'(z) kept
__device__ __forceinline__ void activate4(const float (&z)[4], float *h, float (&g)[4]) {
  float v[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float e = erff(z[u] * 0.70710678118654752f);
    v[u] = 0.5f * z[u] * (1.0f + e);
    g[u] = 0.5f * (1.0f + e) + z[u] * 0.39894228040143268f * expf(-0.5f * z[u] * z[u]);
  }
  *reinterpret_cast<float4 *>(h) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ float dot4(float4 a, float4 b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}
// acc[a][b] += sum_s d[o + a][s] h[i + 16 b][s]
__device__ __forceinline__ void outer4(const float *d, const float *h, int o, int i,
                                       float (&acc)[4][4]) {
#pragma unroll
  for (int s = 0; s < TILE; s += 4) {
    float4 dv[4], hv[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      dv[a] = *reinterpret_cast<const float4 *>(d + (o + a) * LDH + s);
      hv[a] = *reinterpret_cast<const float4 *>(h + (i + 16 * a) * LDH + s);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = dot4(dv[a], hv[b], acc[a][b]);
  }
}

__global__ void __launch_bounds__(WARPS * 32)
    mlp_backward_kernel(int batch, const float *theta, const float *X, const float *target,
                        float *partial, float *partial_loss) {
  extern __shared__ __align__(16) unsigned char train_raw[];
  TrainSmem &m = *reinterpret_cast<TrainSmem *>(train_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
  for (int i = tid; i < NH * NH; i += WARPS * 32) {
    const int at = (i / NH) * LDW + i % NH;
    m.w2[at] = theta[OFF_W2 + i];
    m.w3[at] = theta[OFF_W3 + i];
  }
  for (int i = tid; i < NH * NIN; i += WARPS * 32)
    m.w1[(i / NIN) * LDW1 + i % NIN] = theta[OFF_W1 + i];
  if (tid < NH) {
    m.b1[tid] = theta[OFF_B1 + tid];
    m.b2[tid] = theta[OFF_B2 + tid];
    m.b3[tid] = theta[OFF_B3 + tid];
    m.w4[tid] = theta[OFF_W4 + tid];
  }
  if (tid == 0) m.b4 = theta[OFF_B4];
  // neuron j of samples s0 .. s0 + 3; gradient entries (o4 + a, i4 + 16 b)
  const int j = tid & (NH - 1), s0 = (tid >> 6) * 4, at = j * LDH + s0;
  const int o4 = (tid >> 4) * 4, i4 = tid & 15;
  float gw2[4][4] = {}, gw3[4][4] = {}, gw1[3] = {}, gvec = 0.f, gb4 = 0.f, loss = 0.f;
  for (int64_t first = (int64_t)blockIdx.x * TILE; first < batch;
       first += (int64_t)gridDim.x * TILE) {
    const int n = (int)min((int64_t)TILE, batch - first);
    // a short tile is filled up with its first sample, whose error then counts as 0
    // (values that are finite for a sample stay finite beside it)
    for (int i = tid; i < TILE * NIN; i += WARPS * 32)
      m.x[(i % NIN) * LDH + i / NIN] = X[first * NIN + (i < n * NIN ? i : i % NIN)];
    __syncthreads();
    float z[4], g1[4], g2[4], g3[4];
    dense4<NIN, LDW1>(m.w1, m.b1[j], m.x, j, s0, z);
    activate4(z, m.h1 + at, g1);
    __syncthreads();
    dense4<NH, LDW>(m.w2, m.b2[j], m.h1, j, s0, z);
    activate4(z, m.h2 + at, g2);
    __syncthreads();
    dense4<NH, LDW>(m.w3, m.b3[j], m.h2, j, s0, z);
    activate4(z, m.h3 + at, g3);
    __syncthreads();
    for (int s = warp; s < TILE; s += WARPS) {
      const float out = warp_sum(m.w4[lane] * m.h3[lane * LDH + s] +
                                 m.w4[lane + 32] * m.h3[(lane + 32) * LDH + s]) +
                        m.b4;
      if (lane == 0) {
        const float diff = s < n ? out - target[first + s] : 0.f;
        m.gy[s] = 2.0f * diff / (float)batch;
        m.loss[s] = diff * diff;
      }
    }
    __syncthreads();
    // layer 3: dz3 = W4 gy gelu'(z3)
#pragma unroll
    for (int u = 0; u < 4; ++u) z[u] = m.w4[j] * m.gy[s0 + u] * g3[u];
    *reinterpret_cast<float4 *>(m.d3 + at) = make_float4(z[0], z[1], z[2], z[3]);
    __syncthreads();
    // layer 2: dz2 = (W3^T dz3) gelu'(z2)
    dense4_t(m.w3, m.d3, j, s0, z);
    *reinterpret_cast<float4 *>(m.d2 + at) =
        make_float4(z[0] * g2[0], z[1] * g2[1], z[2] * g2[2], z[3] * g2[3]);
    outer4(m.d3, m.h2, o4, i4, gw3);
    __syncthreads();
    // layer 1: dz1 = (W2^T dz2) gelu'(z1)
    dense4_t(m.w2, m.d2, j, s0, z);
    *reinterpret_cast<float4 *>(m.d1 + at) =
        make_float4(z[0] * g1[0], z[1] * g1[1], z[2] * g1[2], z[3] * g1[3]);
    outer4(m.d2, m.h1, o4, i4, gw2);
    __syncthreads();
    // W4 and the biases, one vector of 64 for each quarter of the threads; W1
    const int which = tid >> 6;
    const float *const vec = which == 0 ? m.h3 : which == 1 ? m.d3 : which == 2 ? m.d2 : m.d1;
#pragma unroll
    for (int s = 0; s < TILE; ++s)
      gvec = fmaf(which == 0 ? m.gy[s] : 1.f, vec[j * LDH + s], gvec);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const int i = tid + e * WARPS * 32;
      if (i < NH * NIN) {
        const float *d = m.d1 + (i / NIN) * LDH, *x = m.x + (i % NIN) * LDH;
#pragma unroll
        for (int s = 0; s < TILE; s += 4)
          gw1[e] = dot4(*reinterpret_cast<const float4 *>(d + s),
                        *reinterpret_cast<const float4 *>(x + s), gw1[e]);
      }
    }
    if (tid == 0)
      for (int s = 0; s < TILE; ++s) {
        gb4 += m.gy[s];
        loss += m.loss[s];
      }
    __syncthreads();                 // all read before the next tile's samples
  }
  float *out = partial + (int64_t)blockIdx.x * NPARAM;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      out[OFF_W2 + (o4 + a) * NH + i4 + 16 * b] = gw2[a][b];
      out[OFF_W3 + (o4 + a) * NH + i4 + 16 * b] = gw3[a][b];
    }
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (tid + e * WARPS * 32 < NH * NIN) out[OFF_W1 + tid + e * WARPS * 32] = gw1[e];
  const int which = tid >> 6;
  out[(which == 0 ? OFF_W4 : which == 1 ? OFF_B3 : which == 2 ? OFF_B2 : OFF_B1) + j] = gvec;
  if (tid == 0) {
    out[OFF_B4] = gb4;
    partial_loss[blockIdx.x] = loss;
  }
}

// The partials summed: a block takes 32 parameters, its eight warps every eighth
// partial each (one thread a parameter, 300 loads in turn, took 20 us), and adds
// the eight sums in order.
__global__ void __launch_bounds__(256)
    mlp_reduce_kernel(int nblocks, int batch, const float *partial, const float *partial_loss,
                      float *grad, float *loss) {
  __shared__ float part[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // the loss is one parameter more
  const int i = blockIdx.x * 32 + lane;
  const float *src = i < NPARAM ? partial + i : partial_loss;
  const int64_t step = i < NPARAM ? NPARAM : 1;
  float s = 0.f;
  if (i <= NPARAM) {
#pragma unroll 8
    for (int b = w; b < nblocks; b += 8) s += src[b * step];
  }
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && i <= NPARAM) {
    s = part[0][lane];
#pragma unroll
    for (int r = 1; r < 8; ++r) s += part[r][lane];
    if (i < NPARAM)
      grad[i] = s;
    else if (loss)
      *loss = s / (float)batch;
  }
}

__global__ void mlp_adam_kernel(int n, float *theta, const float *grad, float *m, float *v,
                                float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float g = grad[i];
  const float mi = b1 * m[i] + (1.f - b1) * g;
  const float vi = b2 * v[i] + (1.f - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// bf16 inference: weights and activations rounded to bf16, fp32 accumulation.
__global__ void __launch_bounds__(WARPS * 32) mlp_bf16_kernel(int n, const float *theta,
                                                               const float *X, float *pred) {
  __shared__ __nv_bfloat16 w[NPARAM + 1];
  __shared__ float h[WARPS][2][NH];
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) w[i] = __float2bfloat16_rn(theta[i]);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto W = [&](int i) { return __bfloat162float(w[i]); };
  auto rb = [](float x) { return __bfloat162float(__float2bfloat16_rn(x)); };
  for (int smp = blockIdx.x * WARPS + warp; smp < n; smp += gridDim.x * WARPS) {
    float a0 = W(OFF_B1 + lane), a1 = W(OFF_B1 + lane + 32);
    for (int i = 0; i < NIN; ++i) {
      const float x = rb(X[(int64_t)smp * NIN + i]);
      a0 = fmaf(W(OFF_W1 + lane * NIN + i), x, a0);
      a1 = fmaf(W(OFF_W1 + (lane + 32) * NIN + i), x, a1);
    }
    h[warp][0][lane] = rb(gelu(a0));
    h[warp][0][lane + 32] = rb(gelu(a1));
    __syncwarp();
    for (int layer = 0; layer < 2; ++layer) {
      const int ow = layer == 0 ? OFF_W2 : OFF_W3, ob = layer == 0 ? OFF_B2 : OFF_B3;
      const float *hi = h[warp][layer & 1];
      a0 = W(ob + lane);
      a1 = W(ob + lane + 32);
      for (int i = 0; i < NH; ++i) {
        a0 = fmaf(W(ow + lane * NH + i), hi[i], a0);
        a1 = fmaf(W(ow + (lane + 32) * NH + i), hi[i], a1);
      }
      __syncwarp();
      h[warp][(layer + 1) & 1][lane] = rb(gelu(a0));
      h[warp][(layer + 1) & 1][lane + 32] = rb(gelu(a1));
      __syncwarp();
    }
    const float out = warp_sum(W(OFF_W4 + lane) * h[warp][0][lane] +
                               W(OFF_W4 + lane + 32) * h[warp][0][lane + 32]) +
                      W(OFF_B4);
    if (lane == 0) pred[smp] = out;
    __syncwarp();
  }
}

// argmin with ties to the smaller index, one block
__global__ void argmin_kernel(int n, const float *pred, int32_t *best) {
  __shared__ float bv[256];
  __shared__ int bi[256];
  float v = INFINITY;
  int idx = 0x7fffffff;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float p = pred[i];
    if (p < v || (p == v && i < idx)) {
      v = p;
      idx = i;
    }
  }
  bv[threadIdx.x] = v;
  bi[threadIdx.x] = idx;
  __syncthreads();
  for (int s = blockDim.x / 2; s; s >>= 1) {
    if (threadIdx.x < s) {
      const float ov = bv[threadIdx.x + s];
      const int oi = bi[threadIdx.x + s];
      if (ov < bv[threadIdx.x] || (ov == bv[threadIdx.x] && oi < bi[threadIdx.x])) {
        bv[threadIdx.x] = ov;
        bi[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *best = bi[0] == 0x7fffffff ? -1 : bi[0];
}

// blocks of the backward pass: a tile each, up to two blocks an SM
int train_grid(int n) {
  const int b = (n + TILE - 1) / TILE;
  const int cap = state().sm_count > 0 ? state().sm_count * 2 : 256;
  return b < cap ? b : cap;
}

int grid_for(int n) {
  const int b = (n + WARPS - 1) / WARPS;
  const int cap = state().sm_count > 0 ? state().sm_count * 4 : 512;
  return b < 1 ? 1 : (b < cap ? b : cap);
}

}  // namespace

// loaded model for hsumma_gemm's automatic choice
struct LoadedModel {
  bool loaded = false;
  float theta[NPARAM];
  float mean[NIN], stdv[NIN];
};
LoadedModel g_model;

const float *loaded_model(float *mean, float *stdv) {
  if (!g_model.loaded) return nullptr;
  for (int i = 0; i < NIN; ++i) {
    mean[i] = g_model.mean[i];
    stdv[i] = g_model.stdv[i];
  }
  return g_model.theta;
}

int mlp_pick_device(int n, const float *d_theta, const float *d_X, float *d_pred,
                    int32_t *d_best, cudaStream_t s) {
  mlp_bf16_kernel<<<grid_for(n), WARPS * 32, 0, s>>>(n, d_theta, d_X, d_pred);
  argmin_kernel<<<1, 256, 0, s>>>(n, d_pred, d_best);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? HSUMMA_OK : cuda_fail(e, "launch mlp pick");
}

// Scratch of hsumma_mlp_backward_noalloc: the per-block gradient partials
// (kNoAllocBlocks x NPARAM floats) followed by the per-block loss partials
// (kNoAllocBlocks floats), 9.3 MB in all.  It lives in the library's own
// device image, so every device that loads the library holds it until the
// process exits; nothing is allocated when the entry point runs.
constexpr int kNoAllocBlocks = (HSUMMA_MLP_NOALLOC_MAX_BATCH + TILE - 1) / TILE;
constexpr int kNoAllocDevices = 64;
static __device__ __align__(256) float g_noalloc_scratch[(size_t)kNoAllocBlocks * (NPARAM + 1)];

// Device address of g_noalloc_scratch on each device (host-side, filled on the
// first call made with that device current; emptied by hsumma_finalize, since a
// cudaDeviceReset in between leaves a stale address).
static std::mutex g_noalloc_mutex;
static float *g_noalloc_addr[kNoAllocDevices] = {};

void forget_noalloc_scratch() {
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  for (auto &p : g_noalloc_addr) p = nullptr;
}

}  // namespace hs

using namespace hs;

extern "C" {

int hsumma_mlp_forward(int batch, const float *theta, const float *X, float *y, float *cache,
                       void *stream) {
  if (batch < 0 || (batch > 0 && (!theta || !X || !y))) {
    set_error("bad MLP arguments");
    return HSUMMA_ERR_ARG;
  }
  if (batch == 0) return HSUMMA_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  mlp_forward_kernel<<<grid_for(batch), WARPS * 32, 0, s>>>(batch, theta, X, y, cache);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? HSUMMA_OK : cuda_fail(e, "launch mlp forward");
}

int hsumma_mlp_backward(int batch, const float *theta, const float *X, const float *target,
                        float *grad, float *loss, void *stream) {
  if (batch <= 0 || !theta || !X || !target || !grad) {
    set_error("bad MLP arguments");
    return HSUMMA_ERR_ARG;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int nb = train_grid(batch);
  // partial gradients of every block, reduced in block order (deterministic),
  // in a buffer of this call only, taken from and returned to the current
  // device's stream-ordered pool on `s`: calls on different devices, streams or
  // threads never share it, and growing it synchronises nothing
  float *partial = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(&partial),
                                  (size_t)nb * (NPARAM + 1) * sizeof(float), s);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync(mlp partials)");
  float *ploss = partial + (size_t)nb * NPARAM;
  const int smem = (int)sizeof(TrainSmem);
  e = cudaFuncSetAttribute(mlp_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           smem);
  if (e == cudaSuccess) {
    mlp_backward_kernel<<<nb, WARPS * 32, smem, s>>>(batch, theta, X, target, partial, ploss);
    mlp_reduce_kernel<<<NPARAM / 32 + 1, 256, 0, s>>>(nb, batch, partial, ploss, grad, loss);
    e = cudaGetLastError();
  }
  const cudaError_t ef = cudaFreeAsync(partial, s);
  if (e != cudaSuccess) return cuda_fail(e, "launch mlp backward");
  return ef == cudaSuccess ? HSUMMA_OK : cuda_fail(ef, "cudaFreeAsync(mlp partials)");
}

// Same gradient and loss as hsumma_mlp_backward, with the block partials kept
// in the fixed scratch above instead of a buffer grown with cudaMalloc.  Every
// slot the reduction reads (blocks 0..nb-1) is written by the backward kernel
// earlier in the same call, so nothing has to be cleared between calls.
int hsumma_mlp_backward_noalloc(int batch, const float *theta, const float *X,
                                const float *target, float *grad, float *loss, void *stream) {
  if (batch <= 0 || !theta || !X || !target || !grad) {
    set_error("bad MLP arguments");
    return HSUMMA_ERR_ARG;
  }
  if (batch > HSUMMA_MLP_NOALLOC_MAX_BATCH) {
    set_error("hsumma_mlp_backward_noalloc: batch %d exceeds its fixed scratch of "
              "HSUMMA_MLP_NOALLOC_MAX_BATCH = %d samples",
              batch, HSUMMA_MLP_NOALLOC_MAX_BATCH);
    return HSUMMA_ERR_ARG;
  }
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kNoAllocDevices) {
    set_error("hsumma_mlp_backward_noalloc: device ordinal beyond 63");
    return HSUMMA_ERR_UNSUPPORTED;
  }
  float *partial = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
      void *addr = nullptr;
      e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(mlp scratch)");
      g_noalloc_addr[dev] = static_cast<float *>(addr);
    }
    partial = g_noalloc_addr[dev];
  }
  const int nb = train_grid(batch);  // <= ceil(batch / TILE) = kNoAllocBlocks at most
  float *ploss = partial + (size_t)kNoAllocBlocks * NPARAM;
  const int smem = (int)sizeof(TrainSmem);
  e = cudaFuncSetAttribute(mlp_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(mlp backward)");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  mlp_backward_kernel<<<nb, WARPS * 32, smem, s>>>(batch, theta, X, target, partial, ploss);
  mlp_reduce_kernel<<<NPARAM / 32 + 1, 256, 0, s>>>(nb, batch, partial, ploss, grad, loss);
  e = cudaGetLastError();
  return e == cudaSuccess ? HSUMMA_OK : cuda_fail(e, "launch mlp backward (no-alloc)");
}

int hsumma_mlp_adam(int n, float *theta, const float *grad, float *m, float *v, int t, float lr,
                    float beta1, float beta2, float eps, void *stream) {
  if (n <= 0 || t < 1 || !theta || !grad || !m || !v) {
    set_error("bad Adam arguments");
    return HSUMMA_ERR_ARG;
  }
  const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
  mlp_adam_kernel<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, theta, grad, m, v, lr, beta1, beta2, eps, c1, c2);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? HSUMMA_OK : cuda_fail(e, "launch adam");
}

int hsumma_mlp_pick(int n, const float *theta, const float *X, float *pred, int32_t *best,
                    void *stream) {
  if (n <= 0 || !theta || !X || !pred || !best) {
    set_error("bad MLP arguments");
    return HSUMMA_ERR_ARG;
  }
  return mlp_pick_device(n, theta, X, pred, best, reinterpret_cast<cudaStream_t>(stream));
}

int hsumma_mlp_load(const float *theta, const float *mean, const float *stdv) {
  forget_model_range();
  if (!theta) {
    g_model.loaded = false;
    forget_choices();
    return HSUMMA_OK;
  }
  if (!mean || !stdv) {
    set_error("model needs feature means and standard deviations");
    return HSUMMA_ERR_ARG;
  }
  memcpy(g_model.theta, theta, sizeof(g_model.theta));
  memcpy(g_model.mean, mean, sizeof(g_model.mean));
  memcpy(g_model.stdv, stdv, sizeof(g_model.stdv));
  g_model.loaded = true;
  forget_choices();
  return HSUMMA_OK;
}

}  // extern "C"
