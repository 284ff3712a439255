// a13: learned candidate scorer (not in the paper; Section 2.4 keeps or drops
// triggers by threshold alone).  A multilayer perceptron 1600 -> 128 -> 32 -> 1
// with GELU hidden units scores 64-channel x 5 x 5-pixel cutouts of the
// high-passed standardised cube around a trigger.  Weights are served in BF16
// and every product is accumulated in FP32; training keeps FP32 master weights
// and Adam moments.  The inputs are FP32, so the contractions stay on the FP32
// pipe (packed multiply-adds).  They are small (a few hundred MFLOP per step)
// and a step is bound by launches and latency: the forward pass is two kernels
// and the gradient a third, with the long sums (1600 inputs, the batch) split
// over CTAs and thread groups so that a batch of 256 fills the chip.  Before, in
// 12 launches of 32 x 32 tiles -> now, gradient and Adam step of 256 samples:
// 197 -> 36 us (layer 1 forward 101 -> 7 us, weight gradients 47 -> 8 us).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace ovro {
namespace {

constexpr int kIn = 1600, kH1 = 128, kH2 = 32;
constexpr int kCutCh = 64, kCutPix = 5;
constexpr int kNParams = kH1 * kIn + kH1 + kH2 * kH1 + kH2 + kH2 + 1;
// parameter offsets, layer by layer (W row-major [out][in], then b)
constexpr int kW1 = 0, kB1 = kW1 + kH1 * kIn, kW2 = kB1 + kH1, kB2 = kW2 + kH2 * kH1, kW3 = kB2 + kH2,
              kB3 = kW3 + kH2;

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

template <bool BF16>
__device__ __forceinline__ float ldw(const void* w, long long i) {
  if (BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(w)[i]);
  return static_cast<const float*>(w)[i];
}

// ---------------------------------------------------------------- cutouts
// x[t][i][dr][dc] = zp[k - 32 + i][r - 2 + dr][c - 2 + dc], 0 outside the
// trigger's coarse channel or the image.
__global__ void k_cutouts(const float* __restrict__ zp, int n_chan, int n, const int* __restrict__ chan0,
                          int n_coarse, const int* __restrict__ trig, int n_trig, float* __restrict__ x) {
  const long long total = static_cast<long long>(n_trig) * kIn;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int t = static_cast<int>(e / kIn);
    const int j = static_cast<int>(e - static_cast<long long>(t) * kIn);
    const int i = j / (kCutPix * kCutPix), rc = j - i * kCutPix * kCutPix;
    const int dr = rc / kCutPix, dc = rc - dr * kCutPix;
    const int k = trig[3 * t], r = trig[3 * t + 1], c = trig[3 * t + 2];
    int lo = 0, hi = n_chan;
    for (int q = 0; q < n_coarse; ++q)
      if (k >= chan0[q] && k < chan0[q + 1]) { lo = chan0[q]; hi = chan0[q + 1]; }
    const int kk = k - kCutCh / 2 + i, rr = r - kCutPix / 2 + dr, cc = c - kCutPix / 2 + dc;
    float v = 0.f;
    if (kk >= lo && kk < hi && rr >= 0 && rr < n && cc >= 0 && cc < n)
      v = zp[(static_cast<long long>(kk) * n + rr) * n + cc];
    x[e] = v;
  }
}

// ------------------------------------------------------------ dense layers
// acc + (w, w) . (a, b) packed
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long dup2(float x) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 z;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(z.x), "=f"(z.y) : "l"(v));
  return z;
}

// Layer 1's products: part[split][b][o] = sum over the split's inputs of
// x[b][i] w[o][i], 64 samples x all 128 outputs per CTA, 32 inputs staged at a
// time (the next ones already in registers), 4 samples x 8 outputs per thread.
// A batch of few tiles is split along the inputs until the CTAs fill the chip
// (fwd_splits): 256 samples take 100 CTAs of two 32-input steps, where 32 CTAs
// walked all 50 steps before.  x16, w16: the buffers start on 16 bytes (their
// rows are multiples of 16).
constexpr int kFB = 64, kFK = 32;
template <bool BF16>
__global__ void __launch_bounds__(256)
k_dense_fwd(const float* __restrict__ x, const void* __restrict__ w, int B, int steps, bool x16, bool w16,
            float* __restrict__ part) {
  __shared__ __align__(16) float xs[kFK][kFB];
  __shared__ __align__(16) float ws[kFK][kH1];
  const int t = threadIdx.x;
  const int b0 = blockIdx.x * kFB;
  const int k0 = blockIdx.y * steps * kFK, k1 = min(kIn, k0 + steps * kFK);
  // loads: 8 inputs of a sample, 16 weights of an output per thread
  const int lb = t & 63, lk = (t >> 6) * 8, lo = t & 127, lw = (t >> 7) * 16;
  const float* xp = x + static_cast<long long>(min(b0 + lb, B - 1)) * kIn + lk;
  float xq[8], wq[16];
  auto fetch = [&](int k) {
    const long long o = kW1 + static_cast<long long>(lo) * kIn + k + lw;
    if (x16) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(xp + k) + u);
        xq[4 * u] = v.x; xq[4 * u + 1] = v.y; xq[4 * u + 2] = v.z; xq[4 * u + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) xq[u] = __ldg(xp + k + u);
    }
    if (!w16) {
#pragma unroll
      for (int u = 0; u < 16; ++u) wq[u] = ldw<BF16>(w, o + u);
    } else if constexpr (BF16) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(w) + o) + u);
        const uint32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {                     // a bf16 is the upper half of its float
          wq[8 * u + 2 * q] = __uint_as_float(r[q] << 16);
          wq[8 * u + 2 * q + 1] = __uint_as_float(r[q] & 0xffff0000u);
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(w) + o) + u);
        wq[4 * u] = v.x; wq[4 * u + 1] = v.y; wq[4 * u + 2] = v.z; wq[4 * u + 3] = v.w;
      }
    }
  };
  const int tb = (t >> 4) * 4, to = (t & 15) * 4;           // outputs to .. to + 3 and to + 64 ..
  unsigned long long acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  fetch(k0);
  for (int k = k0; k < k1; k += kFK) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) xs[lk + u][lb] = xq[u];
#pragma unroll
    for (int u = 0; u < 16; ++u) ws[lw + u][lo] = wq[u];
    __syncthreads();
    if (k + kFK < k1) fetch(k + kFK);
#pragma unroll 8
    for (int i = 0; i < kFK; ++i) {
      const float4 xv = *reinterpret_cast<const float4*>(&xs[i][tb]);
      const ulonglong2 wa = *reinterpret_cast<const ulonglong2*>(&ws[i][to]);
      const ulonglong2 wb = *reinterpret_cast<const ulonglong2*>(&ws[i][to + 64]);
      const float xr[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const unsigned long long d = dup2(xr[q]);
        acc[q][0] = fma2(d, wa.x, acc[q][0]);
        acc[q][1] = fma2(d, wa.y, acc[q][1]);
        acc[q][2] = fma2(d, wb.x, acc[q][2]);
        acc[q][3] = fma2(d, wb.y, acc[q][3]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int b = b0 + tb + q;
    if (b >= B) continue;
    float* o = part + (static_cast<long long>(blockIdx.y) * B + b) * kH1;
    const float2 z0 = unpack2(acc[q][0]), z1 = unpack2(acc[q][1]), z2 = unpack2(acc[q][2]), z3 = unpack2(acc[q][3]);
    *reinterpret_cast<float4*>(o + to) = make_float4(z0.x, z0.y, z1.x, z1.y);
    *reinterpret_cast<float4*>(o + to + 64) = make_float4(z2.x, z2.y, z3.x, z3.y);
  }
}

// The rest of the network for kMB samples per CTA: layer 1's sums, bias and
// GELU, layers 2 and 3; with targets also the loss of each sample and the
// gradients with respect to the logits (d3) and the pre-activations (d2, d1),
// dL/dlogit = (sigma(z) - y) / B.
constexpr int kMB = 4;
template <bool BF16>
__global__ void __launch_bounds__(256)
k_dense_mid(const float* __restrict__ part, int n_split, const void* __restrict__ w, const float* __restrict__ y,
            int B, float* __restrict__ logit, float* __restrict__ h1, float* __restrict__ h2, float* __restrict__ d1,
            float* __restrict__ d2, float* __restrict__ d3, float* __restrict__ loss) {
  __shared__ float w2[kH2][kH1 + 1];
  __shared__ float z1s[kMB][kH1], h1s[kMB][kH1], z2s[kMB][kH2], d2s[kMB][kH2];
  __shared__ float w3[kH2];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int b0 = blockIdx.x * kMB;
  for (int i = t; i < kH2 * kH1; i += 256) w2[i / kH1][i % kH1] = ldw<BF16>(w, kW2 + i);
  if (t < kH2) w3[t] = ldw<BF16>(w, kW3 + t);
  for (int e = t; e < kMB * kH1; e += 256) {
    const int q = e / kH1, o = e % kH1, b = min(b0 + q, B - 1);
    float s = 0.f;
#pragma unroll 5
    for (int p = 0; p < n_split; ++p) s += __ldg(part + (static_cast<long long>(p) * B + b) * kH1 + o);
    const float z = s + ldw<BF16>(w, kB1 + o), h = gelu(z);
    z1s[q][o] = z;
    h1s[q][o] = h;
    if (h1 && b0 + q < B) h1[static_cast<long long>(b) * kH1 + o] = h;
  }
  __syncthreads();
  {
    // two threads a sum: 4 samples x 32 outputs
    const int q = t >> 6, o = (t >> 1) & 31, half = t & 1;
    float s = 0.f;
#pragma unroll 8
    for (int k = 0; k < kH1 / 2; ++k) s = fmaf(h1s[q][2 * k + half], w2[o][2 * k + half], s);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (half == 0) z2s[q][o] = s + ldw<BF16>(w, kB2 + o);
  }
  __syncthreads();
  if (warp < kMB) {
    const int q = warp, b = b0 + q;
    const float z2 = z2s[q][lane], h = gelu(z2);
    float s = h * w3[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float z = s + ldw<BF16>(w, kB3);
    if (lane == 0 && b < B && logit) logit[b] = z;
    if (y) {
      const float tgt = y[min(b, B - 1)];
      const float g = (1.0f / (1.0f + expf(-z)) - tgt) / static_cast<float>(B);
      const float v = g * w3[lane] * gelu_grad(z2);
      d2s[q][lane] = v;
      if (b < B) {
        h2[static_cast<long long>(b) * kH2 + lane] = h;
        d2[static_cast<long long>(b) * kH2 + lane] = v;
        if (lane == 0) {
          d3[b] = g;
          loss[b] = fmaxf(z, 0.f) - tgt * z + log1pf(expf(-fabsf(z)));
        }
      }
    }
  }
  if (!y) return;
  __syncthreads();
  for (int e = t; e < kMB * kH1; e += 256) {
    const int q = e / kH1, k = e % kH1, b = b0 + q;
    float s = 0.f;
#pragma unroll 8
    for (int o = 0; o < kH2; ++o) s = fmaf(d2s[q][o], w2[o][k], s);
    if (b < B) d1[static_cast<long long>(b) * kH1 + k] = s * gelu_grad(z1s[q][k]);
  }
}

// All parameter gradients in one launch.  CTAs 0 .. kW1Tiles - 1: tiles of
// dW1[o][i] = sum_b d1[b][o] x[b][i], 64 outputs x 32 inputs; then the tiles of
// dW2 (d2, h1); then the sums over the batch that are single numbers (dW3,
// biases, the mean loss), a warp each.  A tile's CTA has four groups of 128
// threads, each taking every fourth 16 samples into sums of its own, which are
// added in group order at the end.
constexpr int kGO = 64, kGI = 32, kGB = 16, kGGroups = 4;
constexpr int kW1Tiles = (kH1 / kGO) * (kIn / kGI), kW2Tiles = kH1 / kGI;
constexpr int kSums = kH2 + kH1 + kH2 + 1 + 1;            // dW3, db1, db2, db3, loss
constexpr int kSumCtas = (kSums + 15) / 16;
__global__ void __launch_bounds__(128 * kGGroups)
k_grads(const float* __restrict__ x, const float* __restrict__ h1, const float* __restrict__ h2,
        const float* __restrict__ d1, const float* __restrict__ d2, const float* __restrict__ d3,
        const float* __restrict__ loss, int B, bool x16, float* __restrict__ grad, float* __restrict__ loss_out) {
  __shared__ __align__(16) float ds[kGGroups][kGB][kGO];
  __shared__ __align__(16) float xs[kGGroups][kGB][kGI];
  const int tid = threadIdx.x, lane = tid & 31;
  if (static_cast<int>(blockIdx.x) >= kW1Tiles + kW2Tiles) {
    int o = (blockIdx.x - kW1Tiles - kW2Tiles) * 16 + (tid >> 5);
    if (o >= kSums) return;
    // the o-th sum: sum_b a[b sa] c[b sc]
    const float *a, *c = nullptr;
    int sa, sc = 0;
    float* out;
    if (o < kH2) { a = h2 + o; sa = kH2; c = d3; sc = 1; out = grad + kW3 + o; }
    else if ((o -= kH2) < kH1) { a = d1 + o; sa = kH1; out = grad + kB1 + o; }
    else if ((o -= kH1) < kH2) { a = d2 + o; sa = kH2; out = grad + kB2 + o; }
    else if ((o -= kH2) < 1) { a = d3; sa = 1; out = grad + kB3; }
    else { a = loss; sa = 1; out = loss_out; }
    float s = 0.f;
    for (int b = lane; b < B; b += 32) {
      const float v = a[static_cast<long long>(b) * sa];
      s = c ? fmaf(c[static_cast<long long>(b) * sc], v, s) : s + v;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0 && out) *out = a == loss ? s / static_cast<float>(B) : s;
    return;
  }
  const bool second = static_cast<int>(blockIdx.x) >= kW1Tiles;
  const int tile = second ? blockIdx.x - kW1Tiles : blockIdx.x;
  const int in = second ? kH1 : kIn, out = second ? kH2 : kH1;
  const float* dz = second ? d2 : d1;
  const float* xv = second ? h1 : x;
  float* dw = grad + (second ? kW2 : kW1);
  const int i0 = tile % (in / kGI) * kGI, o0 = tile / (in / kGI) * kGO;
  const int grp = tid >> 7, t = tid & 127;
  const int to = (t >> 3) * 4, ti = (t & 7) * 4;              // 4 outputs x 4 inputs per thread
  unsigned long long acc[4][2];
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[q][0] = acc[q][1] = 0ull;
  const int lo = t & 63, lb = t >> 6, xi = (t & 7) * 4, xb = t >> 3;   // loads
  // every group runs the same number of steps: the barriers are the CTA's
  for (int s0 = 0; s0 < B; s0 += kGB * kGGroups) {
    const int s = s0 + grp * kGB;
    float dq[8];
    float4 xq = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int b = s + lb + 2 * u;
      dq[u] = b < B && o0 + lo < out ? __ldg(dz + static_cast<long long>(b) * out + o0 + lo) : 0.f;
    }
    if (s + xb < B) {
      const float* xp = xv + static_cast<long long>(s + xb) * in + i0 + xi;
      if (x16 || second) xq = __ldg(reinterpret_cast<const float4*>(xp));
      else xq = make_float4(__ldg(xp), __ldg(xp + 1), __ldg(xp + 2), __ldg(xp + 3));
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) ds[grp][lb + 2 * u][lo] = dq[u];
    *reinterpret_cast<float4*>(&xs[grp][xb][xi]) = xq;
    __syncthreads();
#pragma unroll
    for (int b = 0; b < kGB; ++b) {
      const float4 d = *reinterpret_cast<const float4*>(&ds[grp][b][to]);
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&xs[grp][b][ti]);
      const float dr[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const unsigned long long dd = dup2(dr[q]);
        acc[q][0] = fma2(dd, v.x, acc[q][0]);
        acc[q][1] = fma2(dd, v.y, acc[q][1]);
      }
    }
  }
  // the groups' sums, through ds (64 x 32 a group fills two of its 16 x 64)
  __syncthreads();
  float* red = &ds[0][0][0];
  for (int g = 1; g < kGGroups; ++g) {
    if (grp == g)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 a = unpack2(acc[q][0]), c = unpack2(acc[q][1]);
        *reinterpret_cast<float4*>(red + (to + q) * kGI + ti) = make_float4(a.x, a.y, c.x, c.y);
      }
    __syncthreads();
    if (grp == 0)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(red + (to + q) * kGI + ti);
        const float2 a = unpack2(acc[q][0]), c = unpack2(acc[q][1]);
        const float2 p = make_float2(a.x + v.x, a.y + v.y), r = make_float2(c.x + v.z, c.y + v.w);
        asm("mov.b64 %0, {%1, %2};" : "=l"(acc[q][0]) : "f"(p.x), "f"(p.y));
        asm("mov.b64 %0, {%1, %2};" : "=l"(acc[q][1]) : "f"(r.x), "f"(r.y));
      }
    __syncthreads();
  }
  if (grp == 0)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (o0 + to + q < out) {
        const float2 a = unpack2(acc[q][0]), c = unpack2(acc[q][1]);
        float* p = dw + static_cast<long long>(o0 + to + q) * in + i0 + ti;
        p[0] = a.x;                                         // (the caller's gradient may start anywhere)
        p[1] = a.y;
        p[2] = c.x;
        p[3] = c.y;
      }
}

// 1 - b is passed on its own (1 - 0.999f in FP32 is 1.3e-5 off) and the bias
// corrections c = 1 - b^t come from the host in FP64.
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, int n, float lr, float b1, float omb1, float b2, float omb2,
                       float eps, float c1, float c2, __nv_bfloat16* __restrict__ wb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + omb1 * gi;
  const float vi = b2 * v[i] + omb2 * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  w[i] = wi;
  if (wb) wb[i] = __float2bfloat16_rn(wi);
}

__global__ void k_to_bf16(const float* __restrict__ w, int n, __nv_bfloat16* __restrict__ wb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) wb[i] = __float2bfloat16_rn(w[i]);
}

struct ScorerWs {
  float *part, *h1, *h2, *d3, *d2, *d1, *loss;
  int* chan0;
};

// Splits of layer 1's sum: CTAs for about every SM when the batch has few tiles
// (at least two 32-input steps each), none beyond.
constexpr int kFwdSteps = kIn / kFK;                        // 50
int fwd_steps(int B) {
  const int tiles = (B + kFB - 1) / kFB;
  const int splits = std::max(1, std::min(kFwdSteps / 2, 152 / std::max(1, tiles)));
  return (kFwdSteps + splits - 1) / splits;
}
int fwd_splits(int B) { return (kFwdSteps + fwd_steps(B) - 1) / fwd_steps(B); }
// partial sums of a batch of B, and of every smaller one (a workspace sized for
// a batch serves them): splits * B <= min(25 B, max(152 tiles, B))
size_t part_rows(int B) {
  return std::min<size_t>(static_cast<size_t>(B) * (kFwdSteps / 2), std::max<size_t>(152 * kFB, static_cast<size_t>(B)));
}
bool on16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

ScorerWs carve_scorer(void* ws, size_t bytes, int B, int n_coarse, size_t* need) {
  Carver c(ws, bytes);
  ScorerWs w;
  w.part = c.take<float>(part_rows(B) * kH1);
  w.h1 = c.take<float>(static_cast<size_t>(B) * kH1);
  w.h2 = c.take<float>(static_cast<size_t>(B) * kH2);
  w.d3 = c.take<float>(B);
  w.d2 = c.take<float>(static_cast<size_t>(B) * kH2);
  w.d1 = c.take<float>(static_cast<size_t>(B) * kH1);
  w.loss = c.take<float>(B);
  w.chan0 = c.take<int>(n_coarse + 1);
  *need = c.used;
  return w;
}

// logits, and with targets y what k_grads needs
template <bool BF16>
int forward_impl(const void* w, const float* x, const float* y, int B, const ScorerWs& s, float* logit,
                 cudaStream_t st) {
  const int splits = fwd_splits(B);
  k_dense_fwd<BF16><<<dim3((B + kFB - 1) / kFB, splits), 256, 0, st>>>(x, w, B, fwd_steps(B), on16(x),
                                                                            on16(w), s.part);
  OVRO_LAUNCH_CHECK();
  k_dense_mid<BF16><<<(B + kMB - 1) / kMB, 256, 0, st>>>(s.part, splits, w, y, B, logit, y ? s.h1 : nullptr, s.h2,
                                                          s.d1, s.d2, s.d3, s.loss);
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

template <bool BF16>
int grad_impl(const void* w, const float* x, const float* y, int B, const ScorerWs& s, float* grad,
              float* loss_out, cudaStream_t st) {
  if (int e = forward_impl<BF16>(w, x, y, B, s, nullptr, st)) return e;
  k_grads<<<kW1Tiles + kW2Tiles + kSumCtas, 128 * kGGroups, 0, st>>>(x, s.h1, s.h2, s.d1, s.d2, s.d3, s.loss, B,
                                                                     on16(x), grad, loss_out);
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

}  // namespace
}  // namespace ovro

extern "C" {

int ovro_scorer_n_params(void) { return ovro::kNParams; }

size_t ovro_scorer_workspace_size(int batch, int n_coarse) {
  if (batch <= 0) return 0;
  size_t need = 0;
  ovro::carve_scorer(nullptr, 0, batch, n_coarse > 0 ? n_coarse : 1, &need);
  return need;
}

int ovro_scorer_cutouts(const float* d_zp, int n_chan, int image_size, int n_coarse, const int32_t* h_nfft,
                        const int32_t* d_trig, int n_trig, float* d_x, void* d_ws, size_t ws_bytes,
                        void* stream) {
  using namespace ovro;
  if (!d_zp || !h_nfft || !d_x || n_chan <= 0 || image_size <= 0 || n_coarse <= 0 || n_trig < 0)
    return OVRO_ERR_INVALID_ARG;
  if (n_trig == 0) return OVRO_OK;
  if (!d_trig) return OVRO_ERR_INVALID_ARG;
  size_t need = 0;
  ScorerWs s = carve_scorer(d_ws, ws_bytes, 1, n_coarse, &need);
  if (int e = check_workspace(d_ws, ws_bytes, need)) return e;
  std::vector<int> c0(n_coarse + 1, 0);
  for (int c = 0; c < n_coarse; ++c) {
    if (h_nfft[c] <= 0) return OVRO_ERR_INVALID_ARG;
    c0[c + 1] = c0[c] + h_nfft[c];
  }
  if (c0[n_coarse] != n_chan) return OVRO_ERR_INVALID_ARG;
  cudaStream_t st = as_stream(stream);
  OVRO_CUDA_TRY(cudaMemcpyAsync(s.chan0, c0.data(), c0.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  const long long total = static_cast<long long>(n_trig) * kIn;
  const int blocks = static_cast<int>(std::min<long long>((total + 255) / 256, 8LL * num_sms()));
  k_cutouts<<<blocks, 256, 0, st>>>(d_zp, n_chan, image_size, s.chan0, n_coarse, d_trig, n_trig, d_x);
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

int ovro_scorer_forward(const void* d_w_bf16, const float* d_x, int batch, float* d_logit, void* d_ws,
                        size_t ws_bytes, void* stream) {
  using namespace ovro;
  if (!d_w_bf16 || !d_x || !d_logit || batch <= 0) return OVRO_ERR_INVALID_ARG;
  size_t need = 0;
  ScorerWs s = carve_scorer(d_ws, ws_bytes, batch, 1, &need);
  if (int e = check_workspace(d_ws, ws_bytes, need)) return e;
  OVRO_PROF("k_scorer_fwd", as_stream(stream));
  return forward_impl<true>(d_w_bf16, d_x, nullptr, batch, s, d_logit, as_stream(stream));
}

int ovro_scorer_grad(const void* d_w, int w_is_bf16, const float* d_x, const float* d_y, int batch,
                     float* d_grad, float* d_loss_or_null, void* d_ws, size_t ws_bytes, void* stream) {
  using namespace ovro;
  if (!d_w || !d_x || !d_y || !d_grad || batch <= 0) return OVRO_ERR_INVALID_ARG;
  size_t need = 0;
  ScorerWs s = carve_scorer(d_ws, ws_bytes, batch, 1, &need);
  if (int e = check_workspace(d_ws, ws_bytes, need)) return e;
  cudaStream_t st = as_stream(stream);
  return w_is_bf16 ? grad_impl<true>(d_w, d_x, d_y, batch, s, d_grad, d_loss_or_null, st)
                   : grad_impl<false>(d_w, d_x, d_y, batch, s, d_grad, d_loss_or_null, st);
}

int ovro_scorer_adam(float* d_master, float* d_m, float* d_v, const float* d_grad, int step, float lr,
                     void* d_w_bf16_or_null, void* stream) {
  using namespace ovro;
  if (!d_master || !d_m || !d_v || !d_grad || step <= 0 || !(lr > 0.f)) return OVRO_ERR_INVALID_ARG;
  const double b1 = 0.9, b2 = 0.999;
  const float c1 = static_cast<float>(1.0 - std::pow(b1, step));
  const float c2 = static_cast<float>(1.0 - std::pow(b2, step));
  k_adam<<<(kNParams + 255) / 256, 256, 0, as_stream(stream)>>>(
      d_master, d_m, d_v, d_grad, kNParams, lr, static_cast<float>(b1), static_cast<float>(1.0 - b1),
      static_cast<float>(b2), static_cast<float>(1.0 - b2), 1e-8f, c1, c2,
      static_cast<__nv_bfloat16*>(d_w_bf16_or_null));
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

int ovro_scorer_to_bf16(const float* d_master, void* d_w_bf16, void* stream) {
  using namespace ovro;
  if (!d_master || !d_w_bf16) return OVRO_ERR_INVALID_ARG;
  k_to_bf16<<<(kNParams + 255) / 256, 256, 0, as_stream(stream)>>>(d_master, kNParams,
                                                                   static_cast<__nv_bfloat16*>(d_w_bf16));
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

}  // extern "C"
