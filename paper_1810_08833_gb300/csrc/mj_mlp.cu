// Learned first-pass band: candidate features and an FP32 MLP (8 -> 64 -> 64
// -> 1, ReLU) with hand-written forward, backward and Adam kernels.  Nothing
// here is in the MinJoin paper; the band it proposes only narrows a first
// verification pass, and every pair that pass does not settle is verified
// again with band K, so the join's output does not depend on the model.
#include <algorithm>

#include "mj_internal.cuh"

namespace mj {
namespace {

constexpr int F = kBandFeatures;
constexpr int H = kBandHidden;
constexpr int OFF_W1 = 0;               // [H][F]
constexpr int OFF_B1 = OFF_W1 + H * F;  // [H]
constexpr int OFF_W2 = OFF_B1 + H;      // [H][H]
constexpr int OFF_B2 = OFF_W2 + H * H;  // [H]
constexpr int OFF_W3 = OFF_B2 + H;      // [H]
constexpr int OFF_B3 = OFF_W3 + H;      // [1]
static_assert(OFF_B3 + 1 == kBandParams, "parameter layout");

__device__ __forceinline__ float relu(float v) { return v > 0.f ? v : 0.f; }

// Features of candidate u (see kBandFeatures in mj_internal.cuh).
__global__ void features_kernel(const uint32_t* __restrict__ ci, const uint32_t* __restrict__ cj,
                                const uint32_t* __restrict__ mult, const uint32_t* __restrict__ parts,
                                const int64_t* __restrict__ offsets, uint64_t m, uint32_t K, uint32_t T,
                                float* __restrict__ X) {
  for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < m; u += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t x = ci[u], y = cj[u];
    const int64_t lx = offsets[x + 1] - offsets[x], ly = offsets[y + 1] - offsets[y];
    const float n = (float)(lx < ly ? lx : ly), d0 = (float)(lx < ly ? ly - lx : lx - ly);
    const float c = (float)mult[u];
    const float pa = (float)parts[x], pb = (float)parts[y];
    const float pmin = fminf(pa, pb) > 1.f ? fminf(pa, pb) : 1.f;
    const float t1 = (float)T + 1.f;
    float* o = X + u * F;
    o[0] = log2f(1.f + n) / 16.f;
    o[1] = d0 / (float)(K ? K : 1);
    o[2] = c / t1;
    o[3] = pa / t1;
    o[4] = pb / t1;
    o[5] = c / pmin;
    o[6] = log2f(1.f + c) / 8.f;
    o[7] = (float)K / (float)(K + 100);
  }
}

__device__ __forceinline__ uint64_t mix(uint64_t z) {  // splitmix64 finaliser (Steele, Lea, Flood 2014)
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// The network runs on chunks of 64 samples, a block of 256 threads each, as
// 64 x 64 x 64 products in shared memory: thread t holds the 16 outputs of rows
// t / 16 + 16 i and columns t % 16 + 16 j.  Operands are rows along the summed
// index, read 16 bytes at a time: 8 loads feed 64 multiply-adds, and rows
// kLd = 68 words apart keep the 8 lanes of a load phase in different banks.
// Sums run in ascending order from the bias in FP32, as in a plain loop.
constexpr int kSB = 64;
constexpr int kNetThreads = 256;
constexpr int kLd = H + 4;
constexpr int kTile = kSB * kLd;
static_assert(kSB == H, "the products are square");

// acc[i][j] += sum over k of A[row i][k] B[column j][k]
__device__ __forceinline__ void product(const float* __restrict__ A, const float* __restrict__ B, int tr, int tc,
                                        float (&acc)[4][4]) {
#pragma unroll 4
  for (int k = 0; k < H; k += 4) {
    float4 a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(A + (tr + 16 * i) * kLd + k);
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(B + (tc + 16 * j) * kLd + k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
        acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
        acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
        acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
      }
  }
}

// The first layer of the chunk's samples xs[s][f]: units tc + 16 j of samples
// tr + 16 i.
__device__ __forceinline__ void first_layer(const float* __restrict__ w, const float* __restrict__ xs, int tr, int tc,
                                            float (&h)[4][4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4* wj = reinterpret_cast<const float4*>(w + OFF_W1 + (tc + 16 * j) * F);
    const float4 p = wj[0], q = wj[1];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4* xi = reinterpret_cast<const float4*>(xs + (tr + 16 * i) * F);
      const float4 x = xi[0], y = xi[1];
      float z = w[OFF_B1 + tc + 16 * j];
      z = fmaf(p.x, x.x, z);
      z = fmaf(p.y, x.y, z);
      z = fmaf(p.z, x.z, z);
      z = fmaf(p.w, x.w, z);
      z = fmaf(q.x, y.x, z);
      z = fmaf(q.y, y.y, z);
      z = fmaf(q.z, y.z, z);
      z = fmaf(q.w, y.w, z);
      h[i][j] = relu(z);
    }
  }
}

// Output of sample s from the second layer h2t[c][s].
__device__ __forceinline__ float last_layer(const float* __restrict__ w, const float* __restrict__ h2t, int s) {
  float y = w[OFF_B3];
#pragma unroll 16
  for (int c = 0; c < H; ++c) y = fmaf(w[OFF_W3 + c], h2t[c * kLd + s], y);
  return y;
}

// The parameters into shared memory: w as they are but W2, whose rows go to w2
// (and its columns to w2t, when given).
__device__ __forceinline__ void load_params(const float* __restrict__ P, float* __restrict__ w, float* __restrict__ w2,
                                            float* __restrict__ w2t) {
  for (int i = threadIdx.x; i < kBandParams; i += kNetThreads) {
    const float v = P[i];
    if (i >= OFF_W2 && i < OFF_B2) {
      const int c = (i - OFF_W2) / H, a = (i - OFF_W2) % H;
      w2[c * kLd + a] = v;
      if (w2t) w2t[a * kLd + c] = v;
    } else {
      w[i] = v;
    }
  }
}

constexpr int kParamPad = (kBandParams + 3) / 4 * 4;
constexpr size_t kForwardSmem = sizeof(float) * (kParamPad + kSB * F + 3 * kTile);

// y of every sample.  Bound by the FP32 multiply-adds (4,672 a sample):
// 65,536 samples 76 us with one sample per thread and a shared load for every
// one to four of them, 32 us so (300,000: 290, 83).
__global__ void __launch_bounds__(kNetThreads) forward_kernel(const float* __restrict__ P, const float* __restrict__ X,
                                                              uint64_t m, float* __restrict__ out) {
  extern __shared__ __align__(16) float sm[];
  float* w = sm;
  float* xs = w + kParamPad;
  float* w2 = xs + kSB * F;
  float* h1 = w2 + kTile;    // [s][a]
  float* h2t = h1 + kTile;   // [c][s]
  load_params(P, w, w2, nullptr);
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
  for (uint64_t base = (uint64_t)blockIdx.x * kSB; base < m; base += (uint64_t)gridDim.x * kSB) {
    __syncthreads();   // the parameters are there, the previous chunk's rows are read
    for (int i = threadIdx.x; i < kSB * F; i += kNetThreads) xs[i] = base * F + i < m * F ? X[base * F + i] : 0.f;
    __syncthreads();
    float h[4][4];
    first_layer(w, xs, tr, tc, h);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h1[(tr + 16 * i) * kLd + tc + 16 * j] = h[i][j];
        h[i][j] = w[OFF_B2 + tr + 16 * i];
      }
    __syncthreads();
    product(w2, h1, tr, tc, h);   // unit c = row, sample = column
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) h2t[(tr + 16 * i) * kLd + tc + 16 * j] = relu(h[i][j]);
    __syncthreads();
    if (threadIdx.x < kSB && base + threadIdx.x < m) out[base + threadIdx.x] = last_layer(w, h2t, threadIdx.x);
  }
}

constexpr size_t kGradSmem = sizeof(float) * (kParamPad + 2 * kSB * F + 2 * kSB + 6 * kTile);

// Loss and parameter gradient of a batch: every block's sums over its chunks
// to part[block][kBandParams + 1] (the loss last), summed by grad_sum_kernel.
//  samples: batch index b, or with seed != 0 the sample mix(seed + b) % m.
//  target:  y from Y, or from ed as min(ed, K+1) / K.
//  loss:    tau == 0: mean squared error; else pinball loss at quantile tau.
// Sums are taken in a fixed order, so that a call's result does not depend on
// the blocks' timing.  Bound by the FP32 multiply-adds (13,400 a sample):
// 65,536 samples with two warps per chunk and atomic sums 267 us, so 133 (the
// call with its readback); a training step of 1,024 samples 65 us, 30 so.  The
// loss of 300,000 samples was 2e-5 off the sum in 64 bits, and is 1e-8 off.
__global__ void __launch_bounds__(kNetThreads, 2) grad_kernel(const float* __restrict__ P, const float* __restrict__ X,
                                                              const float* __restrict__ Y,
                                                              const uint32_t* __restrict__ ed, uint32_t K, uint64_t m,
                                                              uint64_t batch, uint64_t seed, float tau,
                                                              float* __restrict__ part) {
  extern __shared__ __align__(16) float sm[];
  float* w = sm;
  float* xs = w + kParamPad;       // [s][f]
  float* xt = xs + kSB * F;        // [f][s]
  float* dys = xt + kSB * F;       // dy of every sample
  float* ls = dys + kSB;           // its loss
  float* w2 = ls + kSB;            // [c][a]
  float* w2t = w2 + kTile;         // [a][c]
  float* h1 = w2t + kTile;         // [s][a], then d2 [s][c]
  float* h1t = h1 + kTile;         // [a][s]
  float* h2t = h1t + kTile;        // [c][s], then d1 [a][s]
  float* d2t = h2t + kTile;        // [c][s]
  float* d2 = h1;
  float* d1t = h2t;
  load_params(P, w, w2, w2t);
  const int t = threadIdx.x, tr = t >> 4, tc = t & 15;
  const float inv = 1.f / (float)batch;
  float g2[4][4] = {};             // W2[tr + 16 i][tc + 16 j]
  float g1[2] = {0.f, 0.f};        // W1 entries t and t + 256
  float gv = 0.f;                  // t < 64: b1, < 128: b2, < 192: W3, = 192: b3
  float loss = 0.f;                // t = 224
  for (uint64_t base = (uint64_t)blockIdx.x * kSB; base < batch; base += (uint64_t)gridDim.x * kSB) {
    __syncthreads();
    for (int i = t; i < kSB * F; i += kNetThreads) {
      const uint64_t b = base + i / F;
      const uint64_t u = seed ? mix(seed + b) % m : b;
      const float x = b < batch ? X[u * F + i % F] : 0.f;
      xs[i] = x;
      xt[(i % F) * kSB + i / F] = x;
    }
    __syncthreads();
    float h[4][4];
    first_layer(w, xs, tr, tc, h);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h1[(tr + 16 * i) * kLd + tc + 16 * j] = h[i][j];
        h1t[(tc + 16 * j) * kLd + tr + 16 * i] = h[i][j];
        h[i][j] = w[OFF_B2 + tr + 16 * i];
      }
    __syncthreads();
    product(w2, h1, tr, tc, h);   // unit c = tr + 16 i, sample = tc + 16 j
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h[i][j] = relu(h[i][j]);
        h2t[(tr + 16 * i) * kLd + tc + 16 * j] = h[i][j];
      }
    __syncthreads();
    if (t < kSB) {
      float dy = 0.f, l = 0.f;
      const uint64_t b = base + t;
      if (b < batch) {
        const uint64_t u = seed ? mix(seed + b) % m : b;
        const float y = Y ? Y[u] : (float)(ed[u] < K + 1 ? ed[u] : K + 1) / (float)(K ? K : 1);
        const float r = y - last_layer(w, h2t, t);
        if (tau == 0.f) {
          l = r * r;
          dy = -2.f * r;
        } else {
          l = r > 0.f ? tau * r : (tau - 1.f) * r;
          dy = r > 0.f ? -tau : (1.f - tau);
        }
        dy *= inv;
        l *= inv;
      }
      dys[t] = dy;
      ls[t] = l;
    }
    __syncthreads();
    // back through layer 3 and the second ReLU (samples past the batch have dy = 0)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float v = h[i][j] > 0.f ? dys[tc + 16 * j] * w[OFF_W3 + tr + 16 * i] : 0.f;
        d2[(tc + 16 * j) * kLd + tr + 16 * i] = v;
        d2t[(tr + 16 * i) * kLd + tc + 16 * j] = v;
        h[i][j] = 0.f;
      }
    if (t >= 128 && t < 192) {
      const float* row = h2t + (t - 128) * kLd;
      float g = 0.f;
#pragma unroll 16
      for (int q = 0; q < kSB; ++q) g = fmaf(dys[q], row[q], g);
      gv += g;
    } else if (t == 192) {
      float g = 0.f;
      for (int q = 0; q < kSB; ++q) g += dys[q];
      gv += g;
    } else if (t == 224) {
      float g = 0.f;
      for (int q = 0; q < kSB; ++q) g += ls[q];
      loss += g;
    }
    __syncthreads();
    product(w2t, d2, tr, tc, h);   // unit a = tr + 16 i, sample = tc + 16 j
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int at = (tr + 16 * i) * kLd + tc + 16 * j;
        d1t[at] = h1t[at] > 0.f ? h[i][j] : 0.f;
        h[i][j] = 0.f;
      }
    product(d2t, h1t, tr, tc, h);   // c = tr + 16 i, a = tc + 16 j, summed over the chunk's samples
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) g2[i][j] += h[i][j];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 2; ++e) {   // W1[a][f]
      const int p = t + kNetThreads * e;
      const float* row = d1t + (p / F) * kLd;
      const float* col = xt + (p % F) * kSB;
      float g = 0.f;
#pragma unroll 16
      for (int q = 0; q < kSB; ++q) g = fmaf(row[q], col[q], g);
      g1[e] += g;
    }
    if (t < 128) {
      const float* row = t < 64 ? d1t + t * kLd : d2t + (t - 64) * kLd;
      float g = 0.f;
#pragma unroll 16
      for (int q = 0; q < kSB; ++q) g += row[q];
      gv += g;
    }
  }
  float* o = part + (uint64_t)blockIdx.x * (kBandParams + 1);
#pragma unroll
  for (int e = 0; e < 2; ++e) o[OFF_W1 + t + kNetThreads * e] = g1[e];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) o[OFF_W2 + (tr + 16 * i) * H + tc + 16 * j] = g2[i][j];
  if (t < 64) o[OFF_B1 + t] = gv;
  else if (t < 128) o[OFF_B2 + t - 64] = gv;
  else if (t < 192) o[OFF_W3 + t - 128] = gv;
  else if (t == 192) o[OFF_B3] = gv;
  else if (t == 224) o[kBandParams] = loss;
}

// grad[p] and *loss = the blocks' partial sums: eight interleaved sums, then
// their pairwise sum.
__global__ void grad_sum_kernel(const float* __restrict__ part, int blocks, float* __restrict__ grad,
                                float* __restrict__ loss) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p > kBandParams) return;
  float s[8] = {};
  int b = 0;
  for (; b + 8 <= blocks; b += 8) {
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] += part[(uint64_t)(b + k) * (kBandParams + 1) + p];
  }
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (b + k < blocks) s[k] += part[(uint64_t)(b + k) * (kBandParams + 1) + p];
  const float v = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
  if (p == kBandParams) *loss = v;
  else grad[p] = v;
}

// Adam (Kingma & Ba 2015) with bias correction.
__global__ void adam_kernel(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ M,
                            float* __restrict__ V, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kBandParams) return;
  const float g = G[i];
  const float mm = b1 * M[i] + (1.f - b1) * g;
  const float vv = b2 * V[i] + (1.f - b2) * g * g;
  M[i] = mm;
  V[i] = vv;
  P[i] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

// First-pass band of candidate u from ŷ: the widest band that still fits in
// the fewest 32-bit words holding ceil(ŷ K) + margin (and at least the
// length difference); pairs that would need as many words as band K get K.
__global__ void band_rule_kernel(const float* __restrict__ yhat, const uint32_t* __restrict__ ci,
                                 const uint32_t* __restrict__ cj, const int64_t* __restrict__ offsets, uint64_t m,
                                 uint32_t K, uint32_t margin, uint32_t* __restrict__ kband) {
  const uint32_t wK = (K + 1 + 31) / 32;
  for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < m; u += (uint64_t)gridDim.x * blockDim.x) {
    const float y = yhat[u];
    uint32_t kb = K;
    if (y == y && y < 1.f) {   // not NaN, predicted within K
      const uint32_t x = ci[u], z = cj[u];
      const int64_t lx = offsets[x + 1] - offsets[x], lz = offsets[z + 1] - offsets[z];
      const uint32_t d0 = (uint32_t)(lx > lz ? lx - lz : lz - lx);
      float want = ceilf(fmaxf(y, 0.f) * (float)K) + (float)margin;
      uint32_t kw = want > (float)K ? K : (uint32_t)want;
      if (kw < d0) kw = d0;
      const uint32_t w = (kw + 1 + 31) / 32;
      kb = w < wK ? 32 * w - 1 : K;
    }
    kband[u] = kb;
  }
}

// Network output for one feature row (weights in shared memory).
__device__ __forceinline__ float mlp_eval(const float* s, const float* xf) {
  float h1[H];
#pragma unroll
  for (int a = 0; a < H; ++a) {
    float zz = s[OFF_B1 + a];
#pragma unroll
    for (int f = 0; f < F; ++f) zz = fmaf(s[OFF_W1 + a * F + f], xf[f], zz);
    h1[a] = relu(zz);
  }
  float y = s[OFF_B3];
#pragma unroll 4
  for (int cc = 0; cc < H; ++cc) {
    float zz = s[OFF_B2 + cc];
#pragma unroll
    for (int a = 0; a < H; ++a) zz = fmaf(s[OFF_W2 + cc * H + a], h1[a], zz);
    y = fmaf(s[OFF_W3 + cc], relu(zz), y);
  }
  return y;
}

constexpr int kQueue = 128;   // threads per block of the fused band kernel

// Features, network and band rule in one pass over the candidates (learned
// joins).  Candidates from fewer than min_mult matched partition pairs keep
// band K without running the network; the others are gathered in a block
// queue and evaluated 128 at a time, so a sparse gate does not leave lanes
// idle during the network.
__global__ void __launch_bounds__(kQueue) band_fused_kernel(const float* __restrict__ P, const uint32_t* __restrict__ ci,
                                                            const uint32_t* __restrict__ cj,
                                                            const uint32_t* __restrict__ run_start, uint64_t raw,
                                                            const uint32_t* __restrict__ parts,
                                                            const int64_t* __restrict__ offsets, uint64_t m, uint32_t K,
                                                            uint32_t T, uint32_t margin, uint32_t min_mult,
                                                            const uint8_t* __restrict__ rejected,
                                                            uint32_t* __restrict__ kband) {
  __shared__ float s[kBandParams];
  __shared__ uint32_t q_u[2 * kQueue];
  __shared__ uint32_t q_c[2 * kQueue];
  __shared__ uint32_t qn;
  for (int i = threadIdx.x; i < kBandParams; i += blockDim.x) s[i] = P[i];
  if (threadIdx.x == 0) qn = 0;
  __syncthreads();
  const uint32_t wK = (K + 1 + 31) / 32;
  auto evaluate = [&](uint64_t u, uint32_t c) {
    const uint32_t x = ci[u], z = cj[u];
    const int64_t lx = offsets[x + 1] - offsets[x], lz = offsets[z + 1] - offsets[z];
    const uint32_t d0 = (uint32_t)(lx > lz ? lx - lz : lz - lx);
    const float n = (float)(lx < lz ? lx : lz);
    const float pa = (float)parts[x], pb = (float)parts[z];
    const float pmin = fminf(pa, pb) > 1.f ? fminf(pa, pb) : 1.f;
    const float t1 = (float)T + 1.f;
    const float xf[F] = {log2f(1.f + n) / 16.f, (float)d0 / (float)(K ? K : 1), (float)c / t1, pa / t1, pb / t1,
                         (float)c / pmin, log2f(1.f + (float)c) / 8.f, (float)K / (float)(K + 100)};
    const float y = mlp_eval(s, xf);
    uint32_t kb = K;
    if (y == y && y < 1.f) {
      const float want = ceilf(fmaxf(y, 0.f) * (float)K) + (float)margin;
      uint32_t kw = want > (float)K ? K : (uint32_t)want;
      if (kw < d0) kw = d0;
      const uint32_t w = (kw + 1 + 31) / 32;
      if (w < wK) kb = 32 * w - 1;
    }
    kband[u] = kb;
  };
  const uint64_t stride = (uint64_t)gridDim.x * kQueue;
  for (uint64_t base = (uint64_t)blockIdx.x * kQueue; base < m; base += stride) {
    const uint64_t u = base + threadIdx.x;
    if (u < m) {
      const uint64_t e = u + 1 < m ? run_start[u + 1] : raw;
      const uint32_t c = (uint32_t)(e - run_start[u]);
      kband[u] = K;
      if (c >= min_mult && !(rejected && rejected[u])) {   // a rejected pair needs no pass at all
        const uint32_t slot = atomicAdd(&qn, 1u);
        q_u[slot] = (uint32_t)u;
        q_c[slot] = c;
      }
    }
    __syncthreads();
    const uint32_t n_q = qn;
    const bool last = base + stride >= m;
    if (n_q >= kQueue || (last && n_q > 0)) {
      // evaluate the first min(n_q, kQueue) entries, keep the rest queued
      const uint32_t take = n_q < kQueue ? n_q : kQueue;
      if (threadIdx.x < take) evaluate(q_u[threadIdx.x], q_c[threadIdx.x]);
      __syncthreads();
      const uint32_t left = n_q - take;
      const bool mv = threadIdx.x < left;
      uint32_t qa = 0, qb = 0;
      if (mv) {
        qa = q_u[take + threadIdx.x];
        qb = q_c[take + threadIdx.x];
      }
      __syncthreads();
      if (mv) {
        q_u[threadIdx.x] = qa;
        q_c[threadIdx.x] = qb;
      }
      if (threadIdx.x == 0) qn = left;
      __syncthreads();
      if (last && left > 0) {
        if (threadIdx.x < left) evaluate(q_u[threadIdx.x], q_c[threadIdx.x]);
        __syncthreads();
        if (threadIdx.x == 0) qn = 0;
        __syncthreads();
      }
    }
  }
}

// Gate for the learned band from training samples: the 1st percentile of the
// multiplicity c (recovered from feature 6 = log2(1+c)/8) among samples whose
// band-K result fits a band narrower than K's word count, written to *out.
__global__ void gate_hist_kernel(const float* __restrict__ X, const uint32_t* __restrict__ ed, uint64_t m, uint32_t K,
                                 unsigned int* __restrict__ hist) {
  const uint32_t wK = (K + 1 + 31) / 32;
  const uint32_t kmax1 = wK > 1 ? 32 * (wK - 1) - 1 : 0;
  for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < m; u += (uint64_t)gridDim.x * blockDim.x) {
    if (wK <= 1 || ed[u] > kmax1) continue;
    const float c = exp2f(8.f * X[u * F + 6]) - 1.f;
    uint32_t ci = (uint32_t)(c + 0.5f);
    if (ci > 255) ci = 255;
    atomicAdd(hist + ci, 1u);
  }
}

unsigned grid1(uint64_t n, int threads) {
  uint64_t g = (n + threads - 1) / threads;
  uint64_t cap = (uint64_t)kNumSMsHint * 16;
  return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

int launch_band_features(const uint32_t* ci, const uint32_t* cj, const uint32_t* mult, const uint32_t* parts,
                         const int64_t* offsets, uint64_t m, uint32_t K, uint32_t T, float* X, cudaStream_t s) {
  if (!m) return MJ_OK;
  features_kernel<<<grid1(m, 256), 256, 0, s>>>(ci, cj, mult, parts, offsets, m, K, T, X);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_band_forward(const float* P, const float* X, uint64_t m, float* out, cudaStream_t s) {
  if (!m) return MJ_OK;
  MJ_CUDA_TRY(cudaFuncSetAttribute(forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kForwardSmem));
  const uint64_t blocks = std::min<uint64_t>((m + kSB - 1) / kSB, (uint64_t)kNumSMsHint * 3);
  forward_kernel<<<(unsigned)blocks, kNetThreads, kForwardSmem, s>>>(P, X, m, out);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

static uint64_t grad_blocks(uint64_t batch) {
  return std::min<uint64_t>((batch + kSB - 1) / kSB, (uint64_t)kNumSMsHint * 2);
}

size_t band_grad_part_bytes(uint64_t batch) { return sizeof(float) * grad_blocks(batch) * (kBandParams + 1); }

int launch_band_grad(const float* P, const float* X, const float* Y, const uint32_t* ed, uint32_t K, uint64_t m,
                     uint64_t batch, uint64_t seed, float tau, float* part, float* grad, float* loss, cudaStream_t s) {
  if (!batch) return MJ_OK;
  MJ_CUDA_TRY(cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem));
  const unsigned blocks = (unsigned)grad_blocks(batch);
  grad_kernel<<<blocks, kNetThreads, kGradSmem, s>>>(P, X, Y, ed, K, m, batch, seed, tau, part);
  MJ_KERNEL_DONE();
  grad_sum_kernel<<<(kBandParams + 1 + 127) / 128, 128, 0, s>>>(part, (int)blocks, grad, loss);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_band_adam(float* P, const float* G, float* M, float* V, float lr, float b1, float b2, float eps, int step,
                     cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  adam_kernel<<<(kBandParams + 255) / 256, 256, 0, s>>>(P, G, M, V, lr, b1, b2, eps, c1, c2);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_band_fused(const float* P, const uint32_t* ci, const uint32_t* cj, const uint32_t* run_start, uint64_t raw,
                      const uint32_t* parts, const int64_t* offsets, uint64_t m, uint32_t K, uint32_t T, uint32_t margin,
                      uint32_t min_mult, const uint8_t* rejected, uint32_t* kband, cudaStream_t s) {
  if (!m) return MJ_OK;
  band_fused_kernel<<<grid1(m, kQueue), kQueue, 0, s>>>(P, ci, cj, run_start, raw, parts, offsets, m, K, T, margin,
                                                       min_mult, rejected, kband);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_gate_hist(const float* X, const uint32_t* ed, uint64_t m, uint32_t K, unsigned int* hist, cudaStream_t s) {
  MJ_CUDA_TRY(cudaMemsetAsync(hist, 0, 256 * sizeof(unsigned int), s));
  if (!m) return MJ_OK;
  gate_hist_kernel<<<grid1(m, 256), 256, 0, s>>>(X, ed, m, K, hist);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_band_rule(const float* yhat, const uint32_t* ci, const uint32_t* cj, const int64_t* offsets, uint64_t m,
                     uint32_t K, uint32_t margin, uint32_t* kband, cudaStream_t s) {
  if (!m) return MJ_OK;
  band_rule_kernel<<<grid1(m, 256), 256, 0, s>>>(yhat, ci, cj, offsets, m, K, margin, kband);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

}  // namespace mj
