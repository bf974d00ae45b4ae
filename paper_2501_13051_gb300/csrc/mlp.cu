// The learned join-size estimator (an addition of this library; the paper
// sizes every join exactly, Algorithm 1's count pass).  A 16 -> 64 -> 64 -> 1
// ReLU network predicts log2(1 + join output size) from 16 features of the
// join; the engine sizes the output buffer from the prediction, writes the
// join in a single pass, and falls back to the exact three-pass join when
// the prediction was too small.  Tuple results never depend on the network.
//
// Training runs in FP32 on these kernels: forward, backward and each block's
// share of the parameter gradients in one kernel, the shares summed in a
// fixed order by a second (deterministic: no atomics), pinball (quantile)
// loss at level tau, Adam update (Kingma & Ba, 2015).  Inference runs with BF16 weights and
// activations and FP32 accumulation.
//
// Parameters: one flat FP32 vector W1 (64x16 row-major), b1, W2 (64x64
// row-major), b2, w3 (64), b3: 5313 values.
#include <cuda_bf16.h>

#include <cmath>

#include "kernels.h"

namespace cdl {

namespace {

constexpr int kIn = kMlpIn, kH = kMlpHidden;
constexpr int oW1 = 0, ob1 = oW1 + kH * kIn, oW2 = ob1 + kH, ob2 = oW2 + kH * kH, ow3 = ob2 + kH,
              ob3 = ow3 + kH;
static_assert(ob3 + 1 == kMlpParams, "parameter layout");

__device__ __forceinline__ float block64_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  const float s = red[0] + red[1];
  __syncthreads();
  return s;
}

// One pass over the batch: forward, backward and this block's share of every
// parameter gradient, nothing but the predictions and the shares stored.
// Tiny arithmetic (3 x 5313 multiply-adds per sample), so what bounds it is
// latency: the network sits in shared memory once per block, a block takes
// kTileS samples at a time (thread = one hidden unit of kSPT samples, rows
// padded by one word so that W2 is read without bank conflicts by rows
// (forward) and by columns (backward)), and a thread then adds a 4 x 4 patch
// of dW2 and a 1 x 4 patch of dW1 over the tile from shared memory.  Before,
// one thread per parameter walked the whole batch in global memory:
// a gradient call of 3,000 samples took 228 us and takes 56 (most of it the
// caller's), one of 100,000 samples 12.9 ms and 0.146 ms.
constexpr int kGT = 256;                  // threads
constexpr int kTileS = 32;                // samples per tile
constexpr int kSPT = kTileS * kH / kGT;   // samples per thread in a tile
constexpr int kP1 = kIn + 1, kP2 = kH + 1;  // padded rows of W1, W2
constexpr int kGradBlocks = 304;          // at most two blocks per SM
constexpr int kGradSamples = 21;          // samples a block takes at least (mlp_gradient)

struct MlpTile {
  float w1[kH * kP1], w2[kH * kP2], b1[kH], b2[kH], w3[kH];
  alignas(16) float x[kTileS * kIn];
  alignas(16) float h1[kTileS * kH], h2[kTileS * kH];  // activations
  alignas(16) float g1[kTileS * kH], g2[kTileS * kH];  // dL/dZ1, dL/dZ2
  float go[kTileS];                                    // dL/dprediction
};

template <bool GRAD>
__global__ void __launch_bounds__(kGT) k_mlp_batch(const float* __restrict__ th,
                                                   const float* __restrict__ X,
                                                   const float* __restrict__ y, uint64_t n,
                                                   float tau, float* __restrict__ out,
                                                   float* __restrict__ part) {
  extern __shared__ __align__(16) char raw[];
  MlpTile& m = *reinterpret_cast<MlpTile*>(raw);
  const int t = threadIdx.x, h = t & (kH - 1), q = t / kH, lane = t & 31, warp = t >> 5;
  // this block's samples: an even share of the batch
  const uint64_t s_lo = n * blockIdx.x / gridDim.x, s_hi = n * (blockIdx.x + 1) / gridDim.x;
  for (int i = t; i < kH * kIn; i += kGT) m.w1[i / kIn * kP1 + i % kIn] = th[oW1 + i];
#pragma unroll
  for (int i = t; i < kH * kH; i += kGT) m.w2[i / kH * kP2 + i % kH] = th[oW2 + i];
  if (t < kH) {
    m.b1[t] = th[ob1 + t];
    m.b2[t] = th[ob2 + t];
    m.w3[t] = th[ow3 + t];
  }
  const float b3 = th[ob3];
  float aw2[4][4] = {}, aw1[4] = {}, av = 0.f;
  for (uint64_t s0 = s_lo; s0 < s_hi; s0 += kTileS) {
    const int ns = s_hi - s0 < (uint64_t)kTileS ? (int)(s_hi - s0) : kTileS;
    __syncthreads();  // weights staged; the last tile's sums are done
    for (int i = t; i < kTileS * kIn; i += kGT) m.x[i] = i < ns * kIn ? X[s0 * kIn + i] : 0.f;
    __syncthreads();
    const int sq = q * kSPT;  // this thread's samples of the tile
    const bool live = sq < ns;  // (whole warps)
    float z[kSPT];
    if (live) {
#pragma unroll
      for (int u = 0; u < kSPT; ++u) z[u] = m.b1[h];
#pragma unroll
      for (int k = 0; k < kIn; ++k) {
        const float w = m.w1[h * kP1 + k];
#pragma unroll
        for (int u = 0; u < kSPT; ++u) z[u] += w * m.x[(sq + u) * kIn + k];
      }
#pragma unroll
      for (int u = 0; u < kSPT; ++u) m.h1[(sq + u) * kH + h] = fmaxf(z[u], 0.f);
    }
    __syncthreads();
    if (live) {
#pragma unroll
      for (int u = 0; u < kSPT; ++u) z[u] = m.b2[h];
#pragma unroll 4
      for (int i = 0; i < kH; i += 4) {
        float w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = m.w2[h * kP2 + i + r];
#pragma unroll
        for (int u = 0; u < kSPT; ++u) {
          const float4 v = *reinterpret_cast<const float4*>(&m.h1[(sq + u) * kH + i]);
          z[u] += w[0] * v.x;
          z[u] += w[1] * v.y;
          z[u] += w[2] * v.z;
          z[u] += w[3] * v.w;
        }
      }
#pragma unroll
      for (int u = 0; u < kSPT; ++u) m.h2[(sq + u) * kH + h] = fmaxf(z[u], 0.f);
    }
    __syncthreads();
    // predictions: a warp takes every eighth sample
    for (int s = warp; s < ns; s += kGT / 32) {
      float v0 = m.w3[lane] * m.h2[s * kH + lane], v1 = m.w3[32 + lane] * m.h2[s * kH + 32 + lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
      }
      if (lane == 0) {
        const float p = v0 + v1 + b3;
        out[s0 + s] = p;
        if (GRAD) m.go[s] = (y[s0 + s] > p ? -tau : 1.f - tau) / (float)n;
      }
    }
    if constexpr (GRAD) {
      __syncthreads();
      if (live) {
#pragma unroll
        for (int u = 0; u < kSPT; ++u)
          m.g2[(sq + u) * kH + h] =
              sq + u < ns && m.h2[(sq + u) * kH + h] > 0.f ? m.go[sq + u] * m.w3[h] : 0.f;
      }
      __syncthreads();
      if (live) {
#pragma unroll
        for (int u = 0; u < kSPT; ++u) z[u] = 0.f;
#pragma unroll 4
        for (int j = 0; j < kH; j += 4) {
          float w[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) w[r] = m.w2[(j + r) * kP2 + h];
#pragma unroll
          for (int u = 0; u < kSPT; ++u) {
            const float4 v = *reinterpret_cast<const float4*>(&m.g2[(sq + u) * kH + j]);
            z[u] += v.x * w[0];
            z[u] += v.y * w[1];
            z[u] += v.z * w[2];
            z[u] += v.w * w[3];
          }
        }
#pragma unroll
        for (int u = 0; u < kSPT; ++u)
          m.g1[(sq + u) * kH + h] = m.h1[(sq + u) * kH + h] > 0.f ? z[u] : 0.f;
      }
      __syncthreads();
      // this thread's parameters, summed over the tile's samples in order
      const int j4 = (t >> 4) * 4, i4 = (t & 15) * 4, r1 = t >> 2, k4 = (t & 3) * 4;
#pragma unroll 4
      for (int s = 0; s < ns; ++s) {
        const float4 g = *reinterpret_cast<const float4*>(&m.g2[s * kH + j4]);
        const float4 a = *reinterpret_cast<const float4*>(&m.h1[s * kH + i4]);
        const float4 x = *reinterpret_cast<const float4*>(&m.x[s * kIn + k4]);
        const float gv[4] = {g.x, g.y, g.z, g.w}, hv[4] = {a.x, a.y, a.z, a.w},
                    xv[4] = {x.x, x.y, x.z, x.w}, g1 = m.g1[s * kH + r1];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
#pragma unroll
          for (int c = 0; c < 4; ++c) aw2[r][c] += gv[r] * hv[c];
          aw1[r] += g1 * xv[r];
        }
        if (q == 0)
          av += m.g1[s * kH + h];
        else if (q == 1)
          av += m.g2[s * kH + h];
        else if (q == 2)
          av += m.go[s] * m.h2[s * kH + h];
        else if (h == 0)
          av += m.go[s];
      }
    }
  }
  if constexpr (GRAD) {
    float* g = part + (uint64_t)blockIdx.x * kMlpParams;
    const int j4 = (t >> 4) * 4, i4 = (t & 15) * 4, r1 = t >> 2, k4 = (t & 3) * 4;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int c = 0; c < 4; ++c) g[oW2 + (j4 + r) * kH + i4 + c] = aw2[r][c];
      g[oW1 + r1 * kIn + k4 + r] = aw1[r];
    }
    if (q < 3)
      g[(q == 0 ? ob1 : q == 1 ? ob2 : ow3) + h] = av;
    else if (h == 0)
      g[ob3] = av;
  }
}

// The blocks' shares of every gradient, summed in a fixed order (no atomics):
// a block takes 32 parameters, each warp an eighth of the shares.
__global__ void __launch_bounds__(kGT) k_mlp_reduce(const float* __restrict__ part, int nparts,
                                                    float* __restrict__ grad) {
  constexpr int kW = kGT / 32;
  __shared__ float red[kW][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float acc = 0.f;
  if (p < kMlpParams) {
#pragma unroll 8
    for (int b = warp; b < nparts; b += kW) acc += part[(uint64_t)b * kMlpParams + p];
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && p < kMlpParams) {
#pragma unroll
    for (int w = 1; w < kW; ++w) acc += red[w][lane];
    grad[p] = acc;
  }
}

// b1, b2 and their complements ob1 = 1 - b1, ob2 = 1 - b2 come rounded
// from double (1 - 0.999f in float would be 1.3e-5 off 0.001).
__global__ void k_adam(float* __restrict__ th, const float* __restrict__ grad,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                       float ob1, float ob2, float eps, float c1, float c2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kMlpParams) return;
  const float g = grad[p];
  const float mm = b1 * m[p] + ob1 * g;
  const float vv = b2 * v[p] + ob2 * g * g;
  m[p] = mm;
  v[p] = vv;
  th[p] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

__global__ void k_to_bf16(const float* __restrict__ th, __nv_bfloat16* __restrict__ tb) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kMlpParams) tb[p] = __float2bfloat16_rn(th[p]);
}

// BF16 weights and activations, FP32 accumulation.
__global__ void __launch_bounds__(kH) k_mlp_infer_bf16(const __nv_bfloat16* __restrict__ tb,
                                                       const float* __restrict__ X, uint64_t n,
                                                       float* __restrict__ out) {
  __shared__ __nv_bfloat16 x[kIn], h1[kH];
  __shared__ float red[2];
  const uint64_t s = blockIdx.x;
  const int t = threadIdx.x;
  if (t < kIn) x[t] = __float2bfloat16_rn(X[s * kIn + t]);
  __syncthreads();
  float z1 = __bfloat162float(tb[ob1 + t]);
#pragma unroll
  for (int k = 0; k < kIn; ++k) z1 += __bfloat162float(tb[oW1 + t * kIn + k]) * __bfloat162float(x[k]);
  h1[t] = __float2bfloat16_rn(fmaxf(z1, 0.f));
  __syncthreads();
  float z2 = __bfloat162float(tb[ob2 + t]);
#pragma unroll 16
  for (int i = 0; i < kH; ++i) z2 += __bfloat162float(tb[oW2 + t * kH + i]) * __bfloat162float(h1[i]);
  const float h2 = __bfloat162float(__float2bfloat16_rn(fmaxf(z2, 0.f)));
  const float o = block64_sum(__bfloat162float(tb[ow3 + t]) * h2, red);
  if (t == 0) out[s] = o + __bfloat162float(tb[ob3]);
}

// ---------------------------------------------------------------- features
constexpr int kFT = 1024;
constexpr int kSample = 2048;  // deterministic stride sample per side
constexpr int kSet = 4096;     // open-addressing set of sampled key hashes

__device__ __forceinline__ uint32_t key_hash(const uint32_t* k0, const uint32_t* k1, uint64_t i) {
  const uint32_t h = hash_key(__ldg(k0 + i), k1 ? __ldg(k1 + i) : 0u);
  return h == 0xFFFFFFFFu ? 0xFFFFFFFEu : h;
}

// Inserts h; returns true when it was not yet in the set.
__device__ __forceinline__ bool set_insert(uint32_t* set, uint32_t h) {
  uint32_t s = mix32(h) & (kSet - 1);
  for (int probe = 0; probe < kSet; ++probe) {
    const uint32_t prev = atomicCAS(set + s, 0xFFFFFFFFu, h);
    if (prev == 0xFFFFFFFFu) return true;
    if (prev == h) return false;
    s = (s + 1) & (kSet - 1);
  }
  return false;
}

// Writes the 16 features of one join (see JoinFeatureHost for the host part).
__global__ void __launch_bounds__(kFT) k_join_features(const uint32_t* pk0, const uint32_t* pk1,
                                                       uint64_t np, const uint32_t* bk0,
                                                       const uint32_t* bk1, uint64_t nb,
                                                       JoinFeatureHost hf, float* __restrict__ f) {
  __shared__ uint32_t setP[kSet], setB[kSet];
  __shared__ uint32_t hP[32], hB[32], dB[32], dist[2];
  for (int i = threadIdx.x; i < kSet; i += kFT) setP[i] = setB[i] = 0xFFFFFFFFu;
  if (threadIdx.x < 32) hP[threadIdx.x] = hB[threadIdx.x] = dB[threadIdx.x] = 0;
  if (threadIdx.x < 2) dist[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t sp = np < kSample ? (uint32_t)np : kSample;
  const uint32_t sb = nb < kSample ? (uint32_t)nb : kSample;
  for (uint32_t s = threadIdx.x; s < sp; s += kFT) {
    const uint32_t h = key_hash(pk0, pk1, (uint64_t)s * np / sp);
    atomicAdd(&hP[h >> 27], 1u);
    if (set_insert(setP, h)) atomicAdd(&dist[0], 1u);
  }
  for (uint32_t s = threadIdx.x; s < sb; s += kFT) {
    const uint32_t h = key_hash(bk0, bk1, (uint64_t)s * nb / sb);
    atomicAdd(&hB[h >> 27], 1u);
    if (set_insert(setB, h)) {
      atomicAdd(&dist[1], 1u);
      atomicAdd(&dB[h >> 27], 1u);
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const float fp = sp ? (float)np / sp : 0.f, fb = sb ? (float)nb / sb : 0.f;
  const float ub_scale = dist[1] ? (float)hf.build_distinct / dist[1] : 0.f;
  float est = 0.f, maxp = 0.f, maxb = 0.f, entp = 0.f, entb = 0.f, dot = 0.f, np2 = 0.f, nb2 = 0.f;
  for (int b = 0; b < 32; ++b) {
    const float cp = hP[b] * fp, cb = hB[b] * fb, db = fmaxf(1.f, dB[b] * ub_scale);
    est += cp * cb / db;
    const float qp = sp ? (float)hP[b] / sp : 0.f, qb = sb ? (float)hB[b] / sb : 0.f;
    maxp = fmaxf(maxp, qp);
    maxb = fmaxf(maxb, qb);
    if (qp > 0.f) entp -= qp * log2f(qp);
    if (qb > 0.f) entb -= qb * log2f(qb);
    dot += qp * qb;
    np2 += qp * qp;
    nb2 += qb * qb;
  }
  f[0] = log2f(1.f + (float)np);
  f[1] = log2f(1.f + (float)nb);
  f[2] = log2f(1.f + hf.probe_full);
  f[3] = log2f(1.f + (float)dist[0]);
  f[4] = log2f(1.f + (float)dist[1]);
  f[5] = log2f(1.f + (float)nb / fmaxf(1.f, hf.build_distinct));
  f[6] = log2f(1.f + est);
  f[7] = maxp;
  f[8] = maxb;
  f[9] = entp;
  f[10] = entb;
  f[11] = (np2 > 0.f && nb2 > 0.f) ? dot * rsqrtf(np2 * nb2) : 0.f;
  f[12] = hf.round;
  f[13] = log2f(1.f + hf.prev_output);
  f[14] = log2f(1.f + hf.prev_delta);
  f[15] = hf.filtered;
}

}  // namespace

cudaError_t mlp_forward(Ctx& c, const float* th, const float* X, uint64_t n, float* out) {
  if (n == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_mlp_batch<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(MlpTile));
  if (e != cudaSuccess) return e;
  ProfScope p(c, kMlp, 0.0);
  const uint64_t blocks = (n + kSPT - 1) / kSPT;
  k_mlp_batch<false><<<(unsigned)(blocks < kGradBlocks ? blocks : kGradBlocks), kGT, sizeof(MlpTile),
                       c.st>>>(th, X, nullptr, n, 0.f, out, nullptr);
  return cudaGetLastError();
}

cudaError_t mlp_gradient(Ctx& c, const float* th, const float* X, const float* y, uint64_t n,
                         float tau, float* out, float* grad, void* ws) {
  if (n == 0) return cudaMemsetAsync(grad, 0, sizeof(float) * kMlpParams, c.st);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_batch<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(MlpTile));
  if (e != cudaSuccess) return e;
  // a block for every kGradSamples samples: the shares then fit the
  // workspace (257 floats per sample, 5313 per share); one block's share is
  // the gradient itself
  static_assert((4 * kH + 1) * kGradSamples >= kMlpParams, "shares fit the workspace");
  uint64_t blocks = n / kGradSamples;
  blocks = blocks < 1 ? 1 : blocks < kGradBlocks ? blocks : kGradBlocks;
  float* part = blocks == 1 ? grad : static_cast<float*>(ws);
  ProfScope p(c, kMlp, 0.0);
  k_mlp_batch<true><<<(unsigned)blocks, kGT, sizeof(MlpTile), c.st>>>(th, X, y, n, tau, out, part);
  if (blocks > 1)
    k_mlp_reduce<<<(kMlpParams + 31) / 32, kGT, 0, c.st>>>(part, (int)blocks, grad);
  return cudaGetLastError();
}

cudaError_t mlp_adam(Ctx& c, float* th, const float* grad, float* m, float* v, uint64_t step,
                     float lr) {
  const double b1 = 0.9, b2 = 0.999;
  const float c1 = (float)(1.0 - std::pow(b1, (double)step));
  const float c2 = (float)(1.0 - std::pow(b2, (double)step));
  ProfScope p(c, kMlp, 0.0);
  k_adam<<<(kMlpParams + 255) / 256, 256, 0, c.st>>>(th, grad, m, v, lr, (float)b1, (float)b2,
                                                      (float)(1.0 - b1), (float)(1.0 - b2), 1e-8f,
                                                      c1, c2);
  return cudaGetLastError();
}

cudaError_t mlp_to_bf16(Ctx& c, const float* th, void* tb) {
  k_to_bf16<<<(kMlpParams + 255) / 256, 256, 0, c.st>>>(th, static_cast<__nv_bfloat16*>(tb));
  return cudaGetLastError();
}

cudaError_t mlp_infer_bf16(Ctx& c, const void* tb, const float* X, uint64_t n, float* out) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kMlp, 0.0);
  k_mlp_infer_bf16<<<(unsigned)n, kH, 0, c.st>>>(static_cast<const __nv_bfloat16*>(tb), X, n, out);
  return cudaGetLastError();
}

cudaError_t join_features(Ctx& c, const uint32_t* pk0, const uint32_t* pk1, uint64_t np,
                          const uint32_t* bk0, const uint32_t* bk1, uint64_t nb,
                          const JoinFeatureHost& hf, float* f) {
  ProfScope p(c, kMlp, 4.0 * (np < kSample ? np : kSample) + 4.0 * (nb < kSample ? nb : kSample));
  k_join_features<<<1, kFT, 0, c.st>>>(pk0, pk1, np, bk0, bk1, nb, hf, f);
  return cudaGetLastError();
}

}  // namespace cdl
