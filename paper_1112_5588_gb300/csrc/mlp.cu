// Cost model of the learned tuner (include/pjds_mlp.h): training and
// inference kernels for a 15 -> 64 -> 64 -> 1 ReLU perceptron, the host
// training loop, the matrix features / candidate encoding, and the choice of
// a launch configuration (the model inside its feature range, the exhaustive
// sweep outside it).
//
// The kernels take tiles of 16 samples, one CTA of 256 threads each, with every
// parameter (5121) and activation of a tile in shared memory. A thread computes
// one unit for four samples, or a 4 x 4 block of the weights' gradient, so that
// one or two shared-memory loads feed four or sixteen multiply-adds. An epoch is
// one cooperative launch: per step the CTAs write the gradients of their samples,
// and after a grid barrier each CTA adds up its share of the parameters, over the
// CTAs in their order, and updates it.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "common.h"
#include "cooperative.h"
#include "gridsum.cuh"
#include "pjds_mlp.h"
#include "pjds_tune.h"

namespace pjds {
namespace mlp {

using kry::GridBarrier;
using kry::GridSlots;
using kry::GridSum;

constexpr int IN = PJDS_MLP_IN, H = PJDS_MLP_HID, NT = 256;
constexpr int TS = 16;  // samples of a tile
constexpr int O_W1 = 0, O_B1 = O_W1 + H * IN, O_W2 = O_B1 + H, O_B2 = O_W2 + H * H, O_W3 = O_B2 + H,
              O_B3 = O_W3 + H, NP = O_B3 + 1;
constexpr int NP4 = (NP + 3) & ~3;
static_assert(H == 64 && IN < 16 && NT == 4 * H && TS == 16, "the kernels' thread mapping");

// Shared memory. The strides keep the accesses free of bank conflicts: H + 1 for
// the transpose of W2, whose rows are filled by columns, 20 floats for four
// samples of each of 8 units in one 16-byte access.
constexpr int XP = 16, LT = H + 1, LS = 20;
struct __align__(16) Sm {
  float w1t[IN * H], b1[H];              // [input][unit]
  float w2[H * H], b2[H], w3[H];         // [unit][input]
  float xs[TS * XP], xt[XP * TS];        // [sample][input], [input][sample]
  float a1[TS * H], a1t[H * LS];         // relu(z1): [sample][unit], [unit][sample]
  float a2[TS * H];                      // relu(z2)
  float dz2[TS * H], dz2t[H * LS];
  float dz1[TS * H];
  float red[4][3][H];                    // dw3, db2, db1 by quarters of the samples
  float out[TS], d[TS];
  float w2t[H * LT];                     // [input][unit]
  float b3, db3;
};

__device__ __forceinline__ void load_parameters(Sm &m, const float *P) {
  for (int q = threadIdx.x; q < H * IN; q += NT) m.w1t[q % IN * H + q / IN] = __ldcg(P + O_W1 + q);
  if (threadIdx.x < H) {
    m.b1[threadIdx.x] = __ldcg(P + O_B1 + threadIdx.x);
    m.b2[threadIdx.x] = __ldcg(P + O_B2 + threadIdx.x);
    m.w3[threadIdx.x] = __ldcg(P + O_W3 + threadIdx.x);
  }
  if (threadIdx.x == 0) m.b3 = __ldcg(P + O_B3);
#pragma unroll
  for (int r = 0; r < H * H / 4 / NT; ++r) {
    const int q = 4 * (threadIdx.x + r * NT), h = q / H, k = q % H;
    const float4 w = __ldcg(reinterpret_cast<const float4 *>(P + O_W2 + q));
    *reinterpret_cast<float4 *>(m.w2 + q) = w;
    m.w2t[k * LT + h] = w.x, m.w2t[(k + 1) * LT + h] = w.y;
    m.w2t[(k + 2) * LT + h] = w.z, m.w2t[(k + 3) * LT + h] = w.w;
  }
}

// Forward pass of samples idx[0 .. cnt) (rows first .. first + cnt if idx is
// NULL), cnt at most TS; absent ones read as zeros. Leaves the activations and
// outputs in m; a1, z2: this thread's unit (threadIdx.x % H) for its four samples.
__device__ __forceinline__ void forward_tile(Sm &m, const float *__restrict__ X, const int32_t *idx, int64_t first,
                                             int cnt, float (&a1)[4], float (&z2)[4]) {
  const int h = threadIdx.x % H, sg = threadIdx.x / H * 4;
  {
    const int s = threadIdx.x / XP, i = threadIdx.x % XP;
    float v = 0.0f;
    if (s < cnt && i < IN) v = X[(idx ? (int64_t)idx[s] : first + s) * IN + i];
    m.xs[s * XP + i] = v;
    m.xt[i * TS + s] = v;
  }
  __syncthreads();
  {  // z1 = x W1^T + b1
    float a[4] = {m.b1[h], m.b1[h], m.b1[h], m.b1[h]};
#pragma unroll
    for (int i = 0; i < IN; ++i) {
      const float w = m.w1t[i * H + h];
      const float4 x = *reinterpret_cast<const float4 *>(m.xt + i * TS + sg);
      a[0] = fmaf(x.x, w, a[0]), a[1] = fmaf(x.y, w, a[1]), a[2] = fmaf(x.z, w, a[2]), a[3] = fmaf(x.w, w, a[3]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) m.a1[(sg + j) * H + h] = a1[j] = fmaxf(a[j], 0.0f);
    *reinterpret_cast<float4 *>(m.a1t + h * LS + sg) = make_float4(a1[0], a1[1], a1[2], a1[3]);
  }
  __syncthreads();
  {  // z2 = relu(z1) W2^T + b2
    float a[4] = {m.b2[h], m.b2[h], m.b2[h], m.b2[h]};
#pragma unroll 16
    for (int k = 0; k < H; ++k) {
      const float w = m.w2t[k * LT + h];
      const float4 x = *reinterpret_cast<const float4 *>(m.a1t + k * LS + sg);
      a[0] = fmaf(x.x, w, a[0]), a[1] = fmaf(x.y, w, a[1]), a[2] = fmaf(x.z, w, a[2]), a[3] = fmaf(x.w, w, a[3]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      z2[j] = a[j];
      m.a2[(sg + j) * H + h] = fmaxf(a[j], 0.0f);
    }
  }
  __syncthreads();
  {  // out = relu(z2) w3 + b3: one warp per sample, lanes over units
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int s = w; s < TS; s += NT / 32) {
      float a = m.a2[s * H + l] * m.w3[l] + m.a2[s * H + l + 32] * m.w3[l + 32];
      for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
      if (l == 0) m.out[s] = a + m.b3;
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(NT)
    forward_kernel(const float *__restrict__ P, const float *__restrict__ X, int32_t n, float *__restrict__ out) {
  extern __shared__ unsigned char raw[];
  Sm &m = *reinterpret_cast<Sm *>(raw);
  load_parameters(m, P);
  float a1[4], z2[4];
  for (int64_t first = (int64_t)blockIdx.x * TS; first < n; first += (int64_t)gridDim.x * TS) {
    const int cnt = (int)min((int64_t)TS, n - first);
    __syncthreads();
    forward_tile(m, X, nullptr, first, cnt, a1, z2);
    if (threadIdx.x < cnt) out[first + threadIdx.x] = m.out[threadIdx.x];
  }
}

// One CTA's gradient sums, in registers over its tiles.
struct Grad {
  float w2[4][4];  // units 4 (t / 16) .., inputs 4 (t % 16) ..
  float w1[4];     // unit t % H, inputs 4 (t / H) ..
  float w3, b2, b1;  // unit t % H, this thread's samples
  float b3;
};

// Adds the gradient of inv_n sum (out - y)^2 over a tile's samples.
__device__ __forceinline__ void gradient_tile(Sm &m, const float *__restrict__ X, const float *__restrict__ Y,
                                              const int32_t *idx, int cnt, float inv_n, Grad &g) {
  const int t = threadIdx.x, h = t % H, sg = t / H * 4;
  float a1[4], z2[4];
  forward_tile(m, X, idx, 0, cnt, a1, z2);
  if (t < TS) m.d[t] = t < cnt ? 2.0f * (m.out[t] - Y[idx[t]]) * inv_n : 0.0f;
  __syncthreads();
  {
    float dz[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float d = m.d[sg + j];
      dz[j] = z2[j] > 0.0f ? d * m.w3[h] : 0.0f;
      g.w3 = fmaf(fmaxf(z2[j], 0.0f), d, g.w3);
      g.b2 += dz[j];
      m.dz2[(sg + j) * H + h] = dz[j];
    }
    *reinterpret_cast<float4 *>(m.dz2t + h * LS + sg) = make_float4(dz[0], dz[1], dz[2], dz[3]);
    if (t == 0)
      for (int s = 0; s < TS; ++s) g.b3 += m.d[s];
  }
  __syncthreads();
  {  // dW2[h][k] += sum_s dz2[s][h] relu(z1[s][k])
    const int hq = t / 16 * 4, kq = t % 16 * 4;
#pragma unroll
    for (int s = 0; s < TS; ++s) {
      const float4 z = *reinterpret_cast<const float4 *>(m.dz2 + s * H + hq);
      const float4 a = *reinterpret_cast<const float4 *>(m.a1 + s * H + kq);
      const float zz[4] = {z.x, z.y, z.z, z.w}, aa[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) g.w2[r][c] = fmaf(zz[r], aa[c], g.w2[r][c]);
    }
  }
  {  // dz1 = (dz2 W2) where z1 > 0
    float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 16
    for (int u = 0; u < H; ++u) {
      const float w = m.w2[u * H + h];
      const float4 z = *reinterpret_cast<const float4 *>(m.dz2t + u * LS + sg);
      a[0] = fmaf(z.x, w, a[0]), a[1] = fmaf(z.y, w, a[1]), a[2] = fmaf(z.z, w, a[2]), a[3] = fmaf(z.w, w, a[3]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v = a1[j] > 0.0f ? a[j] : 0.0f;
      g.b1 += v;
      m.dz1[(sg + j) * H + h] = v;
    }
  }
  __syncthreads();
  {  // dW1[h][i] += sum_s dz1[s][h] x[s][i]
    const int ig = t / H * 4;
#pragma unroll
    for (int s = 0; s < TS; ++s) {
      const float z = m.dz1[s * H + h];
      const float4 x = *reinterpret_cast<const float4 *>(m.xs + s * XP + ig);
      g.w1[0] = fmaf(z, x.x, g.w1[0]), g.w1[1] = fmaf(z, x.y, g.w1[1]);
      g.w1[2] = fmaf(z, x.z, g.w1[2]), g.w1[3] = fmaf(z, x.w, g.w1[3]);
    }
  }
  __syncthreads();
}

__device__ __forceinline__ void store_gradient(Sm &m, const Grad &g, float *dst) {
  const int t = threadIdx.x, h = t % H, q = t / H;
  m.red[q][0][h] = g.w3, m.red[q][1][h] = g.b2, m.red[q][2][h] = g.b1;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    *reinterpret_cast<float4 *>(dst + O_W2 + (t / 16 * 4 + r) * H + t % 16 * 4) =
        make_float4(g.w2[r][0], g.w2[r][1], g.w2[r][2], g.w2[r][3]);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (q * 4 + j < IN) dst[O_W1 + h * IN + q * 4 + j] = g.w1[j];
  if (t == 0) dst[O_B3] = g.b3;
  __syncthreads();
  if (t < 3 * H) {
    const int what = t / H, u = t % H;
    const float v = ((m.red[0][what][u] + m.red[1][what][u]) + m.red[2][what][u]) + m.red[3][what][u];
    dst[(what == 0 ? O_W3 : what == 1 ? O_B2 : O_B1) + u] = v;
  }
}

// One epoch of mini-batches idx[0 .. batch), idx[batch .. 2 batch), ..., each with
// an Adam step (Kingma & Ba 2015, Algorithm 1; c[step] = {1 - beta1^t, 1 -
// beta2^t}), then, if loss is not NULL, the mean squared error over all samples.
// Bound by latency: a step is a tile's passes through shared memory (1.4 us for
// the 64 CTAs of a batch of 1024), two grid barriers (1.2 us each) and the reads
// behind them. 2,709 -> 954 us for two epochs of 21,600 samples in batches of
// 1024, against one launch each for the gradient (16 CTAs of 64 samples, 36 us),
// its sum and the update.
struct TrainArgs {
  float *P, *m, *v, *partial;  // partial: a row of NP4 per CTA
  const float *X, *Y;
  const int32_t *idx;
  const float2 *c;
  float *loss;
  GridSlots *slots;
  int32_t n, batch;
  float lr;
  uint32_t arrived, sums;  // barrier arrivals and grid sums of the launches before
};

__global__ void __launch_bounds__(NT) train_kernel(const __grid_constant__ TrainArgs a) {
  extern __shared__ unsigned char raw[];
  Sm &sm = *reinterpret_cast<Sm *>(raw);
  __shared__ float part[NT / 32][32];
  const int t = threadIdx.x, w = t >> 5, l = t & 31;
  GridBarrier barrier{a.slots, a.arrived};
  const int32_t share = (NP + gridDim.x - 1) / gridDim.x;  // of the parameters
  const int32_t p0 = min((int32_t)(blockIdx.x * share), NP), p1 = min(p0 + share, NP);
  for (int32_t b0 = 0, step = 0; b0 < a.n; b0 += a.batch, ++step) {
    const int32_t cnt = min(a.batch, a.n - b0), tiles = (cnt + TS - 1) / TS;
    if ((int32_t)blockIdx.x < tiles) {
      load_parameters(sm, a.P);
      Grad g{};
      for (int32_t k = blockIdx.x; k < tiles; k += gridDim.x)
        gradient_tile(sm, a.X, a.Y, a.idx + b0 + (int64_t)k * TS, min(TS, cnt - k * TS), 1.0f / (float)cnt, g);
      store_gradient(sm, g, a.partial + (int64_t)blockIdx.x * NP4);
    }
    if (!barrier()) return;
    const int32_t rows = min(tiles, (int32_t)gridDim.x);
    const float2 c = a.c[step];
    for (int32_t q0 = p0; q0 < p1; q0 += 32) {  // 32 parameters: warps over the rows, lanes over the parameters
      const int32_t q = q0 + l;
      const bool on = q < p1;
      float mq = 0.0f, vq = 0.0f, pq = 0.0f, s = 0.0f;
      if (on && w == 0) mq = a.m[q], vq = a.v[q], pq = __ldcg(a.P + q);
#pragma unroll 8
      for (int32_t r = w; r < rows; r += NT / 32)
        if (on) s += __ldcg(a.partial + (int64_t)r * NP4 + q);
      part[w][l] = s;
      __syncthreads();
      if (w == 0 && on) {
        float g = 0.0f;
#pragma unroll
        for (int k = 0; k < NT / 32; ++k) g += part[k][l];
        mq = 0.9f * mq + 0.1f * g;
        vq = 0.999f * vq + 0.001f * g * g;
        a.m[q] = mq;
        a.v[q] = vq;
        a.P[q] = pq - a.lr * (mq / c.x) / (sqrtf(vq / c.y) + 1e-8f);
      }
      __syncthreads();
    }
    if (!barrier()) return;
  }
  if (!a.loss) return;
  load_parameters(sm, a.P);
  double e = 0.0;
  float a1[4], z2[4];
  for (int64_t first = (int64_t)blockIdx.x * TS; first < a.n; first += (int64_t)gridDim.x * TS) {
    const int cnt = (int)min((int64_t)TS, a.n - first);
    __syncthreads();
    forward_tile(sm, a.X, nullptr, first, cnt, a1, z2);
    if (t < cnt) {
      const double d = (double)sm.out[t] - (double)a.Y[first + t];
      e += d * d;
    }
  }
  GridSum sum{a.slots, a.sums};
  double total;
  if (!sum.operator()<false>(e, total)) return;
  if (blockIdx.x == 0 && t == 0) *a.loss = (float)(total / a.n);
}

// Standardise the inputs (and targets) in place.
struct Scale {
  float mean[IN], std[IN], out_mean, out_std;
};
__global__ void standardise_kernel(const __grid_constant__ Scale f, float *X, float *Y, int64_t n) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n * IN) {
    const int i = (int)(q % IN);
    X[q] = (X[q] - f.mean[i]) / f.std[i];
  }
  if (Y && q < n) Y[q] = (Y[q] - f.out_mean) / f.out_std;
}

static inline size_t a256(size_t b) { return (b + 255) & ~(size_t)255; }

// At most one CTA per SM, and no more than there are tiles.
constexpr int MAX_CTAS = kry::GS_MAX_CTAS;
static int32_t parts_of(int32_t n, int32_t batch) {
  const int32_t tiles = (int32_t)(((int64_t)std::max(1, std::min(batch, n)) + TS - 1) / TS);
  return std::min(tiles, MAX_CTAS);
}

struct Work {
  float *P, *m, *v, *partial, *X, *Y, *out;
  int32_t *idx;
  float2 *c;
  GridSlots *slots;
};

// train: with what only a training run uses (its steps' constants and the slots of
// its grid-wide waits); prediction takes any training workspace of as many samples.
static size_t carve(void *w, int32_t n, int32_t batch, bool train, Work *k) {
  char *const base = static_cast<char *>(w);
  size_t at = 0;
  auto take = [&](size_t bytes) {
    char *q = base + at;
    at += a256(bytes);
    return q;
  };
  const int64_t steps = ((int64_t)n + std::max(1, batch) - 1) / std::max(1, batch);
  k->P = reinterpret_cast<float *>(take(sizeof(float) * NP4));
  k->m = reinterpret_cast<float *>(take(sizeof(float) * NP));
  k->v = reinterpret_cast<float *>(take(sizeof(float) * NP));
  k->partial = reinterpret_cast<float *>(take(sizeof(float) * NP4 * (size_t)parts_of(n, batch)));
  k->X = reinterpret_cast<float *>(take(sizeof(float) * IN * (size_t)n));
  k->Y = reinterpret_cast<float *>(take(sizeof(float) * (size_t)n));
  k->out = reinterpret_cast<float *>(take(sizeof(float) * (size_t)n));
  k->idx = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * (size_t)n));
  if (!train) return at;
  k->c = reinterpret_cast<float2 *>(take(sizeof(float2) * (size_t)steps));
  k->slots = reinterpret_cast<GridSlots *>(take(sizeof(GridSlots)));
  return at;
}

static size_t work_bytes(int32_t n, int32_t batch, bool train) {
  Work k;
  return carve(nullptr, n, batch, train, &k);
}

static void pack(const pjds_mlp &m, float *P) {
  memcpy(P + O_W1, m.w1, sizeof(m.w1));
  memcpy(P + O_B1, m.b1, sizeof(m.b1));
  memcpy(P + O_W2, m.w2, sizeof(m.w2));
  memcpy(P + O_B2, m.b2, sizeof(m.b2));
  memcpy(P + O_W3, m.w3, sizeof(m.w3));
  P[O_B3] = m.b3;
}

static void unpack(const float *P, pjds_mlp &m) {
  memcpy(m.w1, P + O_W1, sizeof(m.w1));
  memcpy(m.b1, P + O_B1, sizeof(m.b1));
  memcpy(m.w2, P + O_W2, sizeof(m.w2));
  memcpy(m.b2, P + O_B2, sizeof(m.b2));
  memcpy(m.w3, P + O_W3, sizeof(m.w3));
  m.b3 = P[O_B3];
}

static inline uint64_t mix64(uint64_t z) {  // splitmix64 output function
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

static int set_smem_limits() {
  cudaError_t e = cudaFuncSetAttribute(train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sm));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sm));
  return e == cudaSuccess ? PJDS_OK : set_error(PJDS_ECUDA, "shared memory attribute: %s", cudaGetErrorString(e));
}

static int sm_count(int *sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return e == cudaSuccess ? PJDS_OK : set_error(PJDS_ECUDA, "device query: %s", cudaGetErrorString(e));
}

// Raw samples to the device, standardised there.
static cudaError_t upload(const pjds_mlp &m, const float *X, const float *y, int32_t n, const Work &w, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(w.X, X, sizeof(float) * IN * (size_t)n, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && y) e = cudaMemcpyAsync(w.Y, y, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  Scale f;
  memcpy(f.mean, m.in_mean, sizeof(f.mean));
  memcpy(f.std, m.in_std, sizeof(f.std));
  f.out_mean = m.out_mean, f.out_std = m.out_std;
  standardise_kernel<<<(unsigned)(((int64_t)n * IN + 255) / 256), 256, 0, s>>>(f, w.X, y ? w.Y : nullptr, n);
  return cudaGetLastError();
}

static unsigned forward_grid(int32_t n) { return (unsigned)std::min<int64_t>(((int64_t)n + TS - 1) / TS, 4096); }

}  // namespace mlp
}  // namespace pjds

using namespace pjds;
using namespace pjds::mlp;

extern "C" int pjds_mlp_init(pjds_mlp *m, uint64_t seed) {
  clear_error();
  if (!m) return set_error(PJDS_EINVAL, "m is NULL");
  memset(m, 0, sizeof(*m));
  uint64_t c = 0;
  auto u = [&](float lim) {
    const uint64_t r = mix64(mix64(seed * 0x9E3779B97F4A7C15ULL + 77) + (c++) * 0xD1B54A32D192ED03ULL);
    return (float)(((double)(r >> 11) * 0x1.0p-53 * 2.0 - 1.0) * lim);
  };
  const float l1 = sqrtf(6.0f / IN), l2 = sqrtf(6.0f / H);
  for (float &w : m->w1) w = u(l1);
  for (float &w : m->w2) w = u(l2);
  for (float &w : m->w3) w = u(l2);
  for (int i = 0; i < IN; ++i) m->in_std[i] = 1.0f;
  m->out_std = 1.0f;
  for (int i = 0; i < PJDS_MLP_FEATURES; ++i) {
    m->feat_lo[i] = 1.0f;
    m->feat_hi[i] = -1.0f;
  }
  return PJDS_OK;
}

extern "C" int pjds_mlp_fit_range(pjds_mlp *m, const float *feat, int32_t n) {
  clear_error();
  if (!m || !feat || n <= 0) return set_error(PJDS_EINVAL, "bad arguments");
  for (int i = 0; i < PJDS_MLP_FEATURES; ++i) {
    float lo = feat[i], hi = feat[i];
    for (int64_t k = 1; k < n; ++k) {
      lo = std::min(lo, feat[k * PJDS_MLP_FEATURES + i]);
      hi = std::max(hi, feat[k * PJDS_MLP_FEATURES + i]);
    }
    m->feat_lo[i] = lo;
    m->feat_hi[i] = hi;
  }
  return PJDS_OK;
}

extern "C" int pjds_mlp_fit_scaling(pjds_mlp *m, const float *X, const float *y, int32_t n) {
  clear_error();
  if (!m || !X || !y || n <= 0) return set_error(PJDS_EINVAL, "bad arguments");
  for (int i = 0; i < IN; ++i) {
    double s = 0.0, s2 = 0.0;
    for (int64_t k = 0; k < n; ++k) s += X[k * IN + i];
    const double mu = s / n;
    for (int64_t k = 0; k < n; ++k) s2 += (X[k * IN + i] - mu) * (X[k * IN + i] - mu);
    const double sd = sqrt(s2 / n);
    m->in_mean[i] = (float)mu;
    m->in_std[i] = sd > 1e-12 ? (float)sd : 1.0f;
  }
  double s = 0.0, s2 = 0.0;
  for (int64_t k = 0; k < n; ++k) s += y[k];
  const double mu = s / n;
  for (int64_t k = 0; k < n; ++k) s2 += (y[k] - mu) * (y[k] - mu);
  const double sd = sqrt(s2 / n);
  m->out_mean = (float)mu;
  m->out_std = sd > 1e-12 ? (float)sd : 1.0f;
  return PJDS_OK;
}

extern "C" int pjds_mlp_workspace_bytes(int32_t n, int32_t batch, size_t *bytes) {
  clear_error();
  if (n <= 0 || batch <= 0 || !bytes) return set_error(PJDS_EINVAL, "bad arguments");
  *bytes = work_bytes(n, batch, true);
  return PJDS_OK;
}

extern "C" int pjds_mlp_train(pjds_mlp *m, const float *X, const float *y, int32_t n, int32_t epochs, int32_t batch,
                              float lr, uint64_t seed, float *loss_hist, void *work, size_t wbytes, void *stream) {
  clear_error();
  if (!m || !X || !y || !work || n <= 0 || epochs < 0 || batch <= 0 || !(lr > 0.0f))
    return set_error(PJDS_EINVAL, "bad arguments");
  if (wbytes < work_bytes(n, batch, true)) return set_error(PJDS_EINVAL, "workspace too small");
  int rc = set_smem_limits();
  if (rc) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int sms = 0;
  if ((rc = sm_count(&sms))) return rc;
  const int32_t bsz = std::min(batch, n);
  Work w;
  carve(work, n, batch, true, &w);
  std::vector<float> P(NP);
  pack(*m, P.data());
  cudaError_t e = upload(*m, X, y, n, w, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(w.P, P.data(), sizeof(float) * NP, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.m, 0, sizeof(float) * NP, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.v, 0, sizeof(float) * NP, s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp upload: %s", cudaGetErrorString(e));
  const int32_t steps = (int32_t)(((int64_t)n + bsz - 1) / bsz);
  // CTAs: one on each SM as far as there are tiles (of all samples: the losses
  // need them too; a step's tiles may be fewer)
  int32_t grid = (int32_t)std::min<int64_t>(((int64_t)n + TS - 1) / TS, std::min(sms, MAX_CTAS));
  // the next epoch's order is drawn while an epoch runs, into the other buffer
  std::vector<int32_t> order[2];
  std::vector<float2> c[2];
  for (int k = 0; k < 2; ++k) {
    order[k].resize((size_t)n);
    c[k].resize((size_t)steps);
  }
  e = cudaMemsetAsync(w.slots, 0, sizeof(GridSlots), s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp upload: %s", cudaGetErrorString(e));
  TrainArgs a{w.P, w.m, w.v, w.partial, w.X, w.Y, w.idx, w.c, nullptr, w.slots, n, bsz, lr, 0u, 0u};
  int64_t t = 0;
  int32_t kept = 0;  // losses on the device, from epoch ep - kept
  for (int32_t ep = 0; ep < epochs; ++ep) {
    std::vector<int32_t> &o = order[ep & 1];
    std::vector<float2> &cs = c[ep & 1];
    if (bsz < n || ep == 0)
      for (int32_t i = 0; i < n; ++i) o[(size_t)i] = i;
    if (bsz < n) {  // Fisher-Yates with a counter-based generator
      const uint64_t base = mix64(seed + 0x51ED2701ULL * (uint64_t)(ep + 1));
      for (int32_t i = n - 1; i > 0; --i)
        std::swap(o[(size_t)i], o[(size_t)(mix64(base + (uint64_t)i) % (uint64_t)(i + 1))]);
    }
    for (int32_t k = 0; k < steps; ++k) {
      ++t;
      cs[(size_t)k] = make_float2((float)(1.0 - pow(0.9, (double)t)), (float)(1.0 - pow(0.999, (double)t)));
    }
    // the epoch before has ended, and so have the copies from its buffers
    if (ep > 0) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && (bsz < n || ep == 0))
      e = cudaMemcpyAsync(w.idx, o.data(), sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(w.c, cs.data(), sizeof(float2) * (size_t)steps, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp epoch upload: %s", cudaGetErrorString(e));
    a.loss = loss_hist ? w.out + kept : nullptr;
    void *args[] = {&a};
    e = launch_cooperative((const void *)train_kernel, (unsigned)grid, NT, args, sizeof(Sm), s);
    while (e == cudaErrorCooperativeLaunchTooLarge && grid > 1) {  // (a context limited to some of the SMs)
      grid /= 2;
      e = launch_cooperative((const void *)train_kernel, (unsigned)grid, NT, args, sizeof(Sm), s);
    }
    if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp training launch: %s", cudaGetErrorString(e));
    a.arrived += 2u * (uint32_t)steps * (uint32_t)grid;
    a.sums += loss_hist ? 1u : 0u;
    if (++kept == n || ep + 1 == epochs) {
      unsigned long long error = 0;
      if (loss_hist)
        e = cudaMemcpyAsync(loss_hist + (ep + 1 - kept), w.out, sizeof(float) * (size_t)kept, cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(&error, &w.slots->error, sizeof(error), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp loss: %s", cudaGetErrorString(e));
      if (error) return set_error(PJDS_ECUDA, "mlp training: a wait between CTAs ran out");
      kept = 0;
    }
  }
  e = cudaMemcpyAsync(P.data(), w.P, sizeof(float) * NP, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp download: %s", cudaGetErrorString(e));
  unpack(P.data(), *m);
  return PJDS_OK;
}

extern "C" int pjds_mlp_predict(const pjds_mlp *m, const float *X, int32_t n, float *out, void *work, size_t wbytes,
                                void *stream) {
  clear_error();
  if (!m || !X || !out || !work || n <= 0) return set_error(PJDS_EINVAL, "bad arguments");
  if (wbytes < work_bytes(n, 1, false)) return set_error(PJDS_EINVAL, "workspace too small");
  int rc = set_smem_limits();
  if (rc) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Work w;
  carve(work, n, 1, false, &w);
  std::vector<float> P(NP);
  pack(*m, P.data());
  cudaError_t e = upload(*m, X, nullptr, n, w, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(w.P, P.data(), sizeof(float) * NP, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp upload: %s", cudaGetErrorString(e));
  forward_kernel<<<forward_grid(n), NT, sizeof(Sm), s>>>(w.P, w.X, n, w.out);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, w.out, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "mlp predict: %s", cudaGetErrorString(e));
  for (int32_t i = 0; i < n; ++i) out[i] = out[i] * m->out_std + m->out_mean;
  return PJDS_OK;
}

extern "C" int pjds_features(int32_t n_rows, int32_t n_cols, const int64_t *row_ptr, const int32_t *col_idx,
                             float out[PJDS_MLP_FEATURES]) {
  clear_error();
  if (n_rows <= 0 || n_cols < 1 || !row_ptr || !out) return set_error(PJDS_EINVAL, "bad arguments");
  const int64_t nnz = row_ptr[n_rows];
  if (nnz > 0 && !col_idx) return set_error(PJDS_EINVAL, "col_idx is NULL");
  double s1 = 0.0, s2 = 0.0, s3 = 0.0, mx = 0.0;
  const double mean = (double)nnz / n_rows;
  for (int32_t i = 0; i < n_rows; ++i) {
    const double l = (double)(row_ptr[i + 1] - row_ptr[i]), d = l - mean;
    s1 += l;
    s2 += d * d;
    s3 += d * d * d;
    mx = std::max(mx, l);
  }
  const double var = s2 / n_rows, sd = sqrt(var);
  double band = 0.0, near = 0.0;
#pragma omp parallel for schedule(static) reduction(+ : band, near)
  for (int32_t i = 0; i < n_rows; ++i)
    for (int64_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) {
      const double d = fabs((double)col_idx[k] - (double)i);
      band += d;
      near += d <= 64.0 ? 1.0 : 0.0;
    }
  out[0] = (float)log10((double)n_rows);
  out[1] = (float)log10((double)std::max<int64_t>(nnz, 1));
  out[2] = (float)log2(1.0 + mean);
  out[3] = mean > 0.0 ? (float)(sd / mean) : 0.0f;
  out[4] = sd > 0.0 ? (float)((s3 / n_rows) / (sd * sd * sd)) : 0.0f;
  out[5] = (float)log2(1.0 + mx);
  out[6] = nnz > 0 ? (float)(band / nnz / n_rows) : 0.0f;
  out[7] = nnz > 0 ? (float)(near / nnz) : 0.0f;
  (void)s1;
  return PJDS_OK;
}

extern "C" int pjds_tune_encode(const float feat[PJDS_MLP_FEATURES], const pjds_candidate *cands, int32_t n,
                                float *out) {
  clear_error();
  if (!feat || !cands || !out || n <= 0) return set_error(PJDS_EINVAL, "bad arguments");
  for (int32_t c = 0; c < n; ++c) {
    float *o = out + (int64_t)c * IN;
    for (int i = 0; i < PJDS_MLP_FEATURES; ++i) o[i] = feat[i];
    const bool plan = cands[c].plan == 1;
    const int32_t t = !plan && cands[c].threads_per_row > 0 ? cands[c].threads_per_row : 1;
    o[8] = (float)log2((double)cands[c].b / 32.0);
    o[9] = (float)log2((double)t);
    o[10] = cands[c].dtype == PJDS_F64 ? 1.0f : 0.0f;
    o[11] = cands[c].dtype == PJDS_F32 ? 1.0f : 0.0f;
    o[12] = cands[c].dtype == PJDS_BF16 ? 1.0f : 0.0f;
    o[13] = plan ? 1.0f : 0.0f;
    o[14] = !plan && cands[c].tile_order == 1 ? 1.0f : 0.0f;
  }
  return PJDS_OK;
}

extern "C" int pjds_tune_pick(int32_t n_rows, int32_t n_cols, const int64_t *row_ptr, const int32_t *col_idx,
                              const double *val, const pjds_mlp *model, const pjds_candidate *cands, int32_t n_cands,
                              int32_t reps, void *work, size_t work_bytes, void *arena, size_t arena_bytes,
                              void *flush, size_t flush_bytes, pjds_pick *out, void *stream) {
  clear_error();
  if (!out || !cands || n_cands <= 0 || !row_ptr || n_rows <= 0 || n_cols < 1)
    return set_error(PJDS_EINVAL, "bad arguments");
  memset(out, 0, sizeof(*out));
  float feat[PJDS_MLP_FEATURES];
  int rc = pjds_features(n_rows, n_cols, row_ptr, col_idx, feat);
  if (rc) return rc;
  int32_t outside = 0;
  if (model) {
    for (int i = 0; i < PJDS_MLP_FEATURES; ++i) {
      const float lo = model->feat_lo[i], hi = model->feat_hi[i];
      if (lo > hi) continue;  // no range: trusted
      const float tol = 0.02f * (hi - lo);
      outside += feat[i] < lo - tol || feat[i] > hi + tol;
    }
  }
  out->n_outside = outside;
  if (model && outside == 0) {
    std::vector<float> X((size_t)n_cands * IN), pred((size_t)n_cands);
    if ((rc = pjds_tune_encode(feat, cands, n_cands, X.data()))) return rc;
    if ((rc = pjds_mlp_predict(model, X.data(), n_cands, pred.data(), work, work_bytes, stream))) return rc;
    int32_t best = 0;
    for (int32_t c = 1; c < n_cands; ++c)
      if (pred[(size_t)c] < pred[(size_t)best]) best = c;
    out->cand = cands[best];
    out->index = best;
    out->source = PJDS_PICK_MODEL;
    out->us = exp((double)pred[(size_t)best]);
    return PJDS_OK;
  }
  if (!arena) return set_error(PJDS_EINVAL, "the matrix lies outside the model's range and no sweep arena was given");
  std::vector<pjds_tune_entry> e((size_t)n_cands);
  int32_t best = -1;
  rc = pjds_tune_sweep(n_rows, n_cols, row_ptr, col_idx, val, cands, n_cands, reps, arena, arena_bytes, flush,
                       flush_bytes, e.data(), &best, stream);
  if (rc) return rc;
  if (best < 0) return set_error(PJDS_EINVAL, "no candidate ran");
  out->cand = cands[best];
  out->index = best;
  out->source = PJDS_PICK_SWEEP;
  out->us = e[(size_t)best].us;
  clear_error();
  return PJDS_OK;
}
