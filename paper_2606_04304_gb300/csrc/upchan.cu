// a1-a3: unpack 4+4-bit voltages, FFT upchannelizer, 8-bit requantisation.
//
// Section 2.1 of the paper: each ~24 kHz coarse channel is upchannelized by an
// FFT over its time samples, and the fine-channel voltages are correlated by an
// 8-bit X-engine.  One CTA handles one spectrum (N consecutive samples) of a
// group of G adjacent inputs: it transposes the G-byte-wide rows of packed samples
// into a tile of one row per input in shared memory, runs F FFTs at a time
// (Stockham auto-sort, radix-16 passes through a padded exchange buffer, 16 complex
// values per thread in registers), requantises the bins from registers into the
// room of the samples they came from, and writes the int8 spectra for all G inputs
// with row-contiguous stores, so the output for fine channel k' is one 2G-byte run
// in [k'][spectrum][input] order -- the layout the X-engine reads.  (N < 16: a
// thread an FFT, samples and bins staged side by side.)
#include <cmath>
#include <mutex>
#include <numeric>
#include <vector>

#include "common.cuh"
#include "fft.cuh"
#include "tune.h"
#include "upchan_impl.h"

namespace ovro {
namespace {

constexpr int kMaxLog2N = 14;
constexpr int kMaxN = 1 << kMaxLog2N;

// ---------------------------------------------------------------- power pass
// Exact sum over the used samples of re^2 + im^2 per (coarse, input).
__device__ __forceinline__ uint32_t sample_power(uint32_t b) {
  int re = static_cast<int>(static_cast<int8_t>(b)) >> 4;
  int im = static_cast<int>(static_cast<int8_t>(b << 4)) >> 4;
  return static_cast<uint32_t>(re * re + im * im);
}

// `fold` rows of n_input bytes laid end to end are one row of nvec VW-byte columns:
// with fold = VW / gcd(n_input, VW) every such row starts on a VW-byte word and has
// a whole number of them, so any width is read in full words.  Thread = one column
// of R such rows at a time (blockDim.x = R columns of rows), a CTA reads
// consecutive bytes, and the sums of one input meet in shared memory.  Bound by the
// read: 169 MB in rows of 704 took 122 us with one row per 64-thread CTA step, now
// 62; the same in rows of 574, read a byte at a time, cost another 0.5 ms.
template <int VW>
__global__ void __launch_bounds__(256)
k_power(const uint8_t* __restrict__ volt, int n_input, int fold, long long n_rows, int nvec, int col0,
        unsigned long long* __restrict__ power) {
  extern __shared__ uint32_t sum[];                     // [inputs of this CTA's columns]
  const int first = blockIdx.y * col0;
  const int cols = min(nvec - first, col0);
  const int n_sum = min(n_input, cols * VW);
  const int rows = blockDim.x / col0;
  const int cv = threadIdx.x % col0, r0 = threadIdx.x / col0;
  for (int i = threadIdx.x; i < n_sum; i += blockDim.x) sum[i] = 0u;
  __syncthreads();
  if (cv < cols && r0 < rows) {
    uint32_t acc[VW];
#pragma unroll
    for (int j = 0; j < VW; ++j) acc[j] = 0;
    const long long step = static_cast<long long>(gridDim.x) * rows;
    const long long pitch = static_cast<long long>(n_input) * fold;
    const uint8_t* at = volt + static_cast<long long>(first + cv) * VW;
#pragma unroll 8
    for (long long r = static_cast<long long>(blockIdx.x) * rows + r0; r < n_rows; r += step) {
      const uint8_t* p = at + r * pitch;
      if (VW == 16) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(p));
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[q * 4 + b] += sample_power((ws[q] >> (8 * b)) & 0xffu);
      } else if (VW == 4) {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(p));
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[b] += sample_power((w >> (8 * b)) & 0xffu);
      } else {
        acc[0] += sample_power(*p);
      }
    }
    int in = cv * VW % n_input;
#pragma unroll
    for (int j = 0; j < VW; ++j) {
      if (acc[j]) atomicAdd(&sum[in], acc[j]);
      if (++in == n_input) in = 0;
    }
  }
  __syncthreads();
  const int in0 = static_cast<int>(static_cast<long long>(first) * VW % n_input);
  for (int i = threadIdx.x; i < n_sum; i += blockDim.x)
    if (sum[i])
      atomicAdd(power + (in0 + i < n_input ? in0 + i : in0 + i - n_input), static_cast<unsigned long long>(sum[i]));
}

// s = 8 sqrt(2) / sqrt(W P), P = power / n_used, in FP64; rounded to FP32.
// W = N for the plain FFT, the sum of the squared taps (*h2) for a PFB.
__global__ void k_scale(const unsigned long long* __restrict__ power, const double* __restrict__ user,
                        int n, int nfft, long long n_used, const double* __restrict__ h2,
                        float* __restrict__ scale) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s;
  if (user) {
    s = user[i];
  } else {
    const double w = h2 ? *h2 : static_cast<double>(nfft);
    double pbar = static_cast<double>(power[i]) / static_cast<double>(n_used);
    s = pbar > 0.0 ? (8.0 * sqrt(2.0)) / sqrt(w * pbar) : 0.0;
  }
  scale[i] = static_cast<float>(s);
}

// *out = sum of h[i]^2 in FP64 (each square exact), one CTA of 256 threads.
__global__ void __launch_bounds__(256) k_sumsq(const float* __restrict__ h, int n, double* __restrict__ out) {
  __shared__ double part[256];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) {
    const double x = static_cast<double>(h[i]);
    acc += x * x;
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = part[0];
}

// omega_N^k = exp(-2 pi i k / N) for the largest N in the call, FP64 -> FP32.
__global__ void k_twiddle(float2* tw, int n) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  double s, c;
  sincospi(-2.0 * static_cast<double>(k) / static_cast<double>(n), &s, &c);
  tw[k] = make_float2(static_cast<float>(c), static_cast<float>(s));
}

// --------------------------------------------------------- FFT + requantise


// N = 2, 4, 8: one thread per FFT (the whole transform in registers), 256
// inputs of the group at a time.
template <int LOG2N>
__global__ void __launch_bounds__(256)
k_upchan(UpchanArgs a) {
  constexpr int N = 1 << LOG2N;
  static_assert(N < 16, "short transforms only");
  extern __shared__ __align__(16) unsigned char smem[];
  const int G = a.group;
  uint8_t* raw = smem;                                                          // [N][G]
  int8_t* stg = reinterpret_cast<int8_t*>(raw + static_cast<size_t>(N) * G);    // [N][G][2]
  float* sc = reinterpret_cast<float*>(
      stg + ((static_cast<size_t>(N) * G * 2 + 15) & ~static_cast<size_t>(15)));  // [G]
  const int tid = threadIdx.x;
  const int T = blockDim.x;
  const int s = blockIdx.y;
  const int i0 = blockIdx.x * G;
  const int gv = min(G, a.n_input - i0);
  const long long row0 = static_cast<long long>(s) * N;
  {
    const uint8_t* src = a.volt + row0 * a.n_input + i0;
    for (int idx = tid; idx < N * G; idx += T) {
      const int n = idx / G, g = idx - n * G;
      raw[idx] = g < gv ? src[static_cast<long long>(n) * a.n_input + g] : 0;
    }
    for (int g = tid; g < G; g += T) sc[g] = g < gv ? a.scale[i0 + g] : 0.0f;
  }
  __syncthreads();
  for (int g = tid; g < gv; g += T) {
    float2 v[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const uint32_t byte = raw[n * G + g];
      v[n].x = static_cast<float>(static_cast<int>(static_cast<int8_t>(byte)) >> 4);
      v[n].y = static_cast<float>(static_cast<int>(static_cast<int8_t>(byte << 4)) >> 4);
    }
    dft_reg<N>(v);
    const float s_g = sc[g];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int kp = (k + N / 2) & (N - 1);
      float qr = rintf(__fmul_rn(s_g, v[k].x));
      float qi = rintf(__fmul_rn(s_g, v[k].y));
      qr = fminf(fmaxf(qr, -127.f), 127.f);
      qi = fminf(fmaxf(qi, -127.f), 127.f);
      char2 q2;
      q2.x = static_cast<signed char>(qr);
      q2.y = static_cast<signed char>(qi);
      reinterpret_cast<char2*>(stg)[kp * G + g] = q2;
      if (a.out_f) {
        const long long o = ((static_cast<long long>(kp) * a.n_spec + s) * a.n_input + i0 + g);
        reinterpret_cast<float2*>(a.out_f)[o] = v[k];
      }
    }
  }
  __syncthreads();
  int8_t* dst0 = a.out_q + (static_cast<long long>(s) * a.n_input + i0) * 2;
  const long long row_stride = static_cast<long long>(a.n_spec) * a.n_input * 2;
  for (int idx = tid; idx < N * gv; idx += T) {
    const int kp = idx / gv, g = idx - kp * gv;
    *reinterpret_cast<char2*>(dst0 + kp * row_stride + 2 * g) = reinterpret_cast<const char2*>(stg)[kp * G + g];
  }
}

// Radix-16 Stockham kernel for N = 2^LOG2N >= 16 (fft.cuh's row passes): F FFTs of
// the group in flight (F N = 8192 points, 16 per thread; one FFT of 16384), exchange
// rows padded by one slot per 16 so the stride-16 writes of a pass hit distinct
// banks, every index split a shift.  The first pass unpacks the staged 4+4-bit
// samples; the last one requantises its bins straight from registers.
//
// What bounds it is the load pipe, shared memory first, so every access is made to
// be one wavefront:
//  - a tile row per input (2 N bytes: first its packed samples, then, once they have
//    been read, its int8 bins, fftshifted), so the threads of a pass touch
//    consecutive bytes.  Rows are transposed four samples of four inputs at a time
//    on the way in and two bins of four inputs on the way out; the row pitch spreads
//    both over the banks.  With the inputs of a sample side by side half of all
//    wavefronts were conflicts.
//  - the twiddles of the passes after 16 and 256 points in shared memory, [m][k] =
//    omega_N^(k 2^m N / (NS R)), as a warp reads them; from the global table they
//    were scattered 8-byte reads.
// With the samples in the bins' room two CTAs of 64 registers a thread share an SM;
// from 2048 points they would hold too few inputs each for the rows to coalesce
// (and spill), so there it is one with 128.  704 inputs x 240000 samples: 8192
// points 1.40 -> 1.09 ms, 4096 1.06 -> 0.76, 1024 1.05 -> 0.61, 16384 3.0 -> 1.8 (the
// power pass left out).
template <int LOG2N>
struct P2Plan {
  static constexpr int N = 1 << LOG2N;
  static constexpr int F = N >= 8192 ? 1 : 8192 / N;
  static constexpr int THREADS = F * N / 16;
  static constexpr int CTAS = LOG2N < 11 ? 2 : 1;    // per SM
  static constexpr int LDP = N + N / 16;             // pad16(x) < LDP for x < N
  static constexpr int TW16 = LOG2N > 4 ? 16 * (LOG2N < 8 ? LOG2N - 4 : 4) : 0;
  static constexpr int TW256 = LOG2N > 8 ? 256 * (LOG2N < 12 ? LOG2N - 8 : 4) : 0;
};

// Bytes from one input's row of the tile to the next: lanes of four (or two) inputs
// side by side and consecutive words of their rows hit distinct banks.
__host__ __device__ inline int tile_pitch(int n, int G) { return 2 * n + 4 * (G < 32 ? 32 / G : 1); }

// Packed samples of the inputs of one CTA, sizeof(W) inputs and four rows of them at a
// time, transposed into the tile.
template <class W>
__device__ __forceinline__ void stage_samples(const uint8_t* __restrict__ src, long long row, int n, int lg, int gv,
                                              uint8_t* tile, int pitch) {
  constexpr int I = sizeof(W), LI = I == 4 ? 2 : I == 2 ? 1 : 0, U = 2;
  const int sh = lg - LI, items = n / 4 << sh, T = blockDim.x;
  for (int i1 = threadIdx.x; i1 < items; i1 += U * T) {
    uint32_t v[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = i1 + u * T, q = idx >> sh, g = (idx & ((1 << sh) - 1)) << LI;
      const uint8_t* p = src + 4 * q * row + g;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[u][j] = idx < items && g < gv ? static_cast<uint32_t>(*reinterpret_cast<const W*>(p + j * row)) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = i1 + u * T, q = idx >> sh, g = (idx & ((1 << sh) - 1)) << LI;
      if (idx >= items) continue;
#pragma unroll
      for (int i = 0; i < I; ++i) {
        const uint32_t lo = __byte_perm(v[u][0], v[u][1], i | (4 + i) << 4);
        const uint32_t hi = __byte_perm(v[u][2], v[u][3], i | (4 + i) << 4);
        *reinterpret_cast<uint32_t*>(tile + (g + i) * pitch + 4 * q) = __byte_perm(lo, hi, 0x5410);
      }
    }
  }
}

// The tile's bins to rows of 2 G bytes, I inputs of two bins at a time.
template <int I>
__device__ __forceinline__ void write_bins(const uint8_t* tile, int pitch, int n, int lg, int gv, int8_t* dst,
                                           long long row) {
  constexpr int LI = I == 4 ? 2 : I == 2 ? 1 : 0;
  const int sh = lg - LI, items = n / 2 << sh, T = blockDim.x;
#pragma unroll 4
  for (int idx = threadIdx.x; idx < items; idx += T) {
    const int p = idx >> sh, g = (idx & ((1 << sh) - 1)) << LI;
    if (g >= gv) continue;
    uint32_t b[I];
#pragma unroll
    for (int i = 0; i < I; ++i) b[i] = *reinterpret_cast<const uint32_t*>(tile + (g + i) * pitch + 4 * p);
    int8_t* d = dst + 2 * p * row + 2 * g;
    if constexpr (I == 1) {
      *reinterpret_cast<uint16_t*>(d) = static_cast<uint16_t>(b[0]);
      *reinterpret_cast<uint16_t*>(d + row) = static_cast<uint16_t>(b[0] >> 16);
    } else if constexpr (I == 2) {
      *reinterpret_cast<uint32_t*>(d) = __byte_perm(b[0], b[1], 0x5410);
      *reinterpret_cast<uint32_t*>(d + row) = __byte_perm(b[0], b[1], 0x7632);
    } else {
      *reinterpret_cast<uint2*>(d) = make_uint2(__byte_perm(b[0], b[1], 0x5410), __byte_perm(b[2], b[3], 0x5410));
      *reinterpret_cast<uint2*>(d + row) = make_uint2(__byte_perm(b[0], b[1], 0x7632), __byte_perm(b[2], b[3], 0x7632));
    }
  }
}

// F32: FP32 spectra are asked for as well; known when compiled, as the test in the
// last pass cost the transforms without them 2 to 4%.
template <int LOG2N, bool F32>
__global__ void __launch_bounds__(P2Plan<LOG2N>::THREADS, P2Plan<LOG2N>::CTAS)
k_upchan_p2(UpchanArgs a) {
  using P = P2Plan<LOG2N>;
  constexpr int N = P::N, F = P::F;
  // FP32 rows leave by F inputs at a time, in full sectors from F = 4 (1024 points x
  // 574 inputs x 303090 samples: 2.5 -> 1.02 ms); one slot more, so that those hit
  // distinct banks
  constexpr bool wide = F32 && F > 1;
  constexpr int LDP = P::LDP + (wide ? 1 : 0);
  extern __shared__ __align__(16) unsigned char smem[];
  const int G = a.group, lg = 31 - __clz(G);    // G is a power of two
  const int pitch = tile_pitch(N, G);
  float2* buf = reinterpret_cast<float2*>(smem);                                 // [F][LDP]
  float2* tws = buf + F * LDP;
  float* sc = reinterpret_cast<float*>(tws + P::TW16 + P::TW256);                // [G]
  uint8_t* tile = reinterpret_cast<uint8_t*>(sc + G);                            // [G][pitch]
  const int tid = threadIdx.x;
  const int T = blockDim.x;
  const int s = blockIdx.y;
  const int i0 = blockIdx.x * G;
  const int gv = min(G, a.n_input - i0);        // valid inputs in this group
  const int tw_stride = a.tw_n / N;
  for (int i = tid; i < P::TW16 + P::TW256; i += T) {
    const int NS = i < P::TW16 ? 16 : 256, x = i < P::TW16 ? i : i - P::TW16;
    const int left = N / NS;                    // points left: a pass of radix 16, or the last one
    tws[i] = __ldg(a.tw + ((x & (NS - 1)) * (left >= 16 ? left / 16 : 1) << (x / NS)) * tw_stride);
  }
  for (int g = tid; g < G; g += T) sc[g] = g < gv ? a.scale[i0 + g] : 0.0f;
  {
    const uint8_t* src = a.volt + static_cast<long long>(s) * N * a.n_input + i0;
    const uintptr_t al = reinterpret_cast<uintptr_t>(a.volt) | a.n_input | G;   // where rows and groups start
    if ((al & 3) == 0)
      stage_samples<uint32_t>(src, a.n_input, N, lg, gv, tile, pitch);
    else if ((al & 1) == 0)
      stage_samples<uint16_t>(src, a.n_input, N, lg, gv, tile, pitch);
    else
      stage_samples<uint8_t>(src, a.n_input, N, lg, gv, tile, pitch);
  }
  __syncthreads();
  auto tw = [&](int i, auto ns, int m, int k) {
    if constexpr (decltype(ns)::value == 16) return tws[m * 16 + k];
    if constexpr (decltype(ns)::value == 256) return tws[P::TW16 + m * 256 + k];
    return __ldg(a.tw + i * tw_stride);
  };
  for (int f0 = 0; f0 < gv; f0 += F) {
    auto sample = [&](int f, int x, int) {
      // high nibble real, low nibble imaginary (two's complement)
      float2 v = make_float2(0.f, 0.f);
      const int g = f0 + f;
      if (g < G) {
        const uint32_t byte = tile[g * pitch + x];
        v.x = static_cast<float>(static_cast<int>(static_cast<int8_t>(byte)) >> 4);
        v.y = static_cast<float>(static_cast<int>(static_cast<int8_t>(byte << 4)) >> 4);
      }
      return v;
    };
    auto bin = [&](int f, int k, float2 X) {
      const int g = f0 + f;
      if (g >= gv) return;
      const float s_g = sc[g];
      const int kp = (k + N / 2) & (N - 1);
      float qr = rintf(__fmul_rn(s_g, X.x));
      float qi = rintf(__fmul_rn(s_g, X.y));
      qr = fminf(fmaxf(qr, -127.f), 127.f);
      qi = fminf(fmaxf(qi, -127.f), 127.f);
      char2 q2;
      q2.x = static_cast<signed char>(qr);
      q2.y = static_cast<signed char>(qi);
      *reinterpret_cast<char2*>(tile + g * pitch + 2 * kp) = q2;
      if constexpr (F32) {
        const long long o = ((static_cast<long long>(kp) * a.n_spec + s) * a.n_input + i0 + g);
        reinterpret_cast<float2*>(a.out_f)[o] = X;
      }
    };
    if constexpr (wide) {
      // through the exchange buffer: F neighbouring inputs make a row of 8 F bytes
      fft_rows_io<LOG2N, false>(buf, LDP, true, sample, tw,
                                [&](int f, int k, float2 X) { buf[f * LDP + pad16(k)] = X; });
#pragma unroll 8
      for (int idx = tid; idx < F * N; idx += P::THREADS) {
        const int f = idx % F, k = idx / F;
        bin(f, k, buf[f * LDP + pad16(k)]);
      }
    } else {
      // one pass alone: its bins overlap its samples
      fft_rows_io<LOG2N, true>(buf, LDP, LOG2N == 4, sample, tw, bin);
    }
    __syncthreads();       // buf reused by the next F inputs, the bins complete
  }
  int8_t* dst = a.out_q + (static_cast<long long>(s) * a.n_input + i0) * 2;
  const long long row = static_cast<long long>(a.n_spec) * a.n_input * 2;
  const uintptr_t al = reinterpret_cast<uintptr_t>(a.out_q) | 2 * a.n_input | 2 * G;
  if ((al & 7) == 0)
    write_bins<4>(tile, pitch, N, lg, gv, dst, row);
  else if ((al & 3) == 0)
    write_bins<2>(tile, pitch, N, lg, gv, dst, row);
  else
    write_bins<1>(tile, pitch, N, lg, gv, dst, row);
}

size_t smem_p2(int log2n, int G) {
  const int N = 1 << log2n;
  const int F = N >= 8192 ? 1 : 8192 / N;
  return static_cast<size_t>(F) * (N + N / 16 + (F > 1 ? 1 : 0)) * 8 + (log2n > 8 ? 1088 : 64) * sizeof(float2) + 4 * G +
         static_cast<size_t>(G) * tile_pitch(N, G);
}

size_t smem_for(int log2n, int G);

int group_for(int log2n, int n_input) {
  // G inputs per CTA: the most that leave room for the CTAs planned per SM, at least F (wider groups coalesce the G-byte
  // row reads and 2G-byte row writes)
  const int F = log2n >= 13 ? 1 : (log2n < 4 ? 256 : (8192 >> log2n));
  const size_t budget = (log2n >= 4 && log2n < 11 ? 112 : 224) * 1024;
  int G = 1;
  while (G < 64 && smem_for(log2n, 2 * G) <= budget) G *= 2;
  if (G < F) G = F;
  int np2 = 1;
  while (np2 < n_input) np2 *= 2;
  if (G > np2) G = np2;
  return G;
}

size_t smem_for(int log2n, int G) {
  if (log2n >= 4) return smem_p2(log2n, G);
  const int N = 1 << log2n;
  return static_cast<size_t>(N) * G + ((static_cast<size_t>(N) * G * 2 + 15) & ~static_cast<size_t>(15)) + 4 * G +
         16;
}

template <int L>
int launch_upchan_t(const UpchanArgs& a, cudaStream_t st) {
  const size_t sm = smem_for(L, a.group);
  dim3 grid((a.n_input + a.group - 1) / a.group, a.n_spec);
  if constexpr (L >= 4) {
    auto kern = a.out_f ? k_upchan_p2<L, true> : k_upchan_p2<L, false>;
    OVRO_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm)));
    OVRO_PROF("k_upchan", st);
    kern<<<grid, P2Plan<L>::THREADS, sm, st>>>(a);
  } else {
    auto kern = k_upchan<L>;
    OVRO_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm)));
    OVRO_PROF("k_upchan", st);
    kern<<<grid, 256, sm, st>>>(a);
  }
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

int launch_upchan(int log2n, const UpchanArgs& a, cudaStream_t st) {
  switch (log2n) {
    case 1: return launch_upchan_t<1>(a, st);
    case 2: return launch_upchan_t<2>(a, st);
    case 3: return launch_upchan_t<3>(a, st);
    case 4: return launch_upchan_t<4>(a, st);
    case 5: return launch_upchan_t<5>(a, st);
    case 6: return launch_upchan_t<6>(a, st);
    case 7: return launch_upchan_t<7>(a, st);
    case 8: return launch_upchan_t<8>(a, st);
    case 9: return launch_upchan_t<9>(a, st);
    case 10: return launch_upchan_t<10>(a, st);
    case 11: return launch_upchan_t<11>(a, st);
    case 12: return launch_upchan_t<12>(a, st);
    case 13: return launch_upchan_t<13>(a, st);
    case 14: return launch_upchan_t<14>(a, st);
    default: return OVRO_ERR_UNSUPPORTED;
  }
}

// G inputs per CTA from the autotuner: every G with F <= G <= 64 whose shared
// memory fits (results do not depend on G).  Untuned, the widest, halved while the
// CTAs still fit the SMs one each: a call of few spectra of few inputs is a chain of
// the G / F transforms of a CTA (9 spectra of 8192 points: 16 inputs 57 us with G = 8,
// 24 with 1, and 104 and 28 with FP32 spectra; 40 inputs 57 with G = 8, 34 with 4).
int launch_upchan_tuned(int l, UpchanArgs a, cudaStream_t st) {
  const int F = l >= 13 ? 1 : (l < 4 ? 256 : (8192 >> l));
  int np2 = 1;
  while (np2 < a.n_input) np2 *= 2;
  int g0 = group_for(l, a.n_input);
  auto ctas = [&](int g) { return static_cast<long long>((a.n_input + g - 1) / g) * a.n_spec; };
  while (l >= 4 && g0 / 2 >= F && ctas(g0 / 2) <= num_sms()) g0 /= 2;
  std::vector<int> cands;
  for (int g = F; g <= 64; g *= 2) {
    if (g > np2 && g > F) break;
    if (smem_for(l, g) <= (size_t(227) << 10)) cands.push_back(g);
  }
  auto run = [&](int g) -> int {
    a.group = g;
    return launch_upchan(l, a, st);
  };
  const std::string key = tune_key("k_upchan", {l, a.n_input});
  int g = tuned(key, g0);
  if (tuning(st) && cands.size() > 1)
    if (int e = tune_pick(key, cands, run, st, &g)) return e;
  if (l >= 4 && (g <= 0 || (g & (g - 1)) || smem_for(l, g) > (size_t(227) << 10))) g = g0;
  return run(g);
}

struct UpchanWs {
  unsigned long long* power;
  float* scale;
  double* user;
  double* h2;
  float2* tw;
};

UpchanWs carve_upchan(void* ws, size_t bytes, int n_input, int n_coarse, size_t* need) {
  Carver c(ws, bytes);
  UpchanWs w;
  w.power = c.take<unsigned long long>(static_cast<size_t>(n_input) * n_coarse);
  w.scale = c.take<float>(static_cast<size_t>(n_input) * n_coarse);
  w.user = c.take<double>(static_cast<size_t>(n_input) * n_coarse);
  w.h2 = c.take<double>(static_cast<size_t>(n_coarse));
  w.tw = c.take<float2>(kMaxN);
  *need = c.used;
  return w;
}

}  // namespace
}  // namespace ovro

extern "C" {

size_t ovro_upchan_workspace_size(int n_input, int n_coarse) {
  if (n_input <= 0 || n_coarse <= 0) return 0;
  size_t need = 0;
  ovro::carve_upchan(nullptr, 0, n_input, n_coarse, &need);
  return need;
}

int ovro_upchan_ex(const uint8_t* d_volt, int n_input, int n_coarse, int64_t n_time,
                   const int32_t* h_nfft, const double* h_scale_or_null, const ovro_upchan_options* opt,
                   int8_t* d_fine_q, float* d_fine_f32_or_null, void* d_ws, size_t ws_bytes, void* stream) {
  using namespace ovro;
  if (!d_volt || !h_nfft || !d_fine_q || n_input <= 0 || n_coarse <= 0 || n_time <= 0)
    return OVRO_ERR_INVALID_ARG;
  const bool taps = opt && opt->h_taps;
  const int n_tap = opt ? opt->n_taps : 1;
  const int lo = opt ? opt->chan_lo : 0;
  const int cnt_opt = opt ? opt->chan_count : 0;
  if (n_tap < 1 || (n_tap > 1 && !taps) || lo < 0 || cnt_opt < 0) return OVRO_ERR_INVALID_ARG;
  struct Coarse {
    int n, cnt, k;
    bool mixed;
    MrPlan plan;                     // mixed only
  };
  std::vector<Coarse> cs(n_coarse);
  int max_pow2 = 2;
  for (int c = 0; c < n_coarse; ++c) {
    Coarse& e = cs[c];
    e.n = h_nfft[c];
    if (e.n <= 0) return OVRO_ERR_INVALID_ARG;
    if (taps && !opt->h_taps[c]) return OVRO_ERR_INVALID_ARG;
    const long long blocks = n_time / e.n;
    const long long k = blocks - n_tap + 1;
    if (k < 1 || k > INT32_MAX) return OVRO_ERR_UNSUPPORTED;
    e.k = static_cast<int>(k);
    e.cnt = cnt_opt ? cnt_opt : e.n;
    if (static_cast<long long>(lo) + e.cnt > e.n) return OVRO_ERR_INVALID_ARG;
    e.mixed = taps || lo != 0 || e.cnt != e.n || !is_pow2(e.n) || e.n > kMaxN || k > 65535;
    if (e.mixed) {
      int group = 0;
      size_t smem = 0;
      if (!mr_plan(e.n, n_input, taps ? n_tap : 1, e.cnt, &e.plan, &group, &smem)) return OVRO_ERR_UNSUPPORTED;
    } else {
      if (e.n < 2) return OVRO_ERR_UNSUPPORTED;
      max_pow2 = std::max(max_pow2, e.n);
    }
  }
  size_t need = 0;
  UpchanWs w = carve_upchan(d_ws, ws_bytes, n_input, n_coarse, &need);
  if (int e = check_workspace(d_ws, ws_bytes, need)) return e;
  cudaStream_t st = as_stream(stream);

  const size_t nsc = static_cast<size_t>(n_input) * n_coarse;
  if (h_scale_or_null) {
    OVRO_CUDA_TRY(cudaMemcpyAsync(w.user, h_scale_or_null, nsc * sizeof(double),
                                  cudaMemcpyHostToDevice, st));
  } else {
    OVRO_CUDA_TRY(cudaMemsetAsync(w.power, 0, nsc * sizeof(unsigned long long), st));
  }
  int table_n = 0;   // length of the table in w.tw
  bool table_mr = false;   // by passes, else omega_{table_n}^k
  long long q_off = 0;
  for (int c = 0; c < n_coarse; ++c) {
    const Coarse& e = cs[c];
    const int n = e.n;
    const long long n_used = (n_time / n) * n;
    if (!h_scale_or_null) {
      const uint8_t* vc = d_volt + static_cast<long long>(c) * n_time * n_input;
      unsigned long long* pc = w.power + static_cast<size_t>(c) * n_input;
      // bytes a thread reads at a time: the widest word the samples start on that
      // whole numbers of rows make up, if the rows come out even
      int vw = 16, fold = 1;
      for (; vw > 1; vw /= 4) {
        fold = vw / std::gcd(n_input, vw);
        if (reinterpret_cast<uintptr_t>(vc) % vw == 0 && n_used % fold == 0) break;
      }
      if (vw == 1) fold = 1;
      const long long n_rows = n_used / fold;
      const int nvec = static_cast<int>(static_cast<long long>(n_input) * fold / vw), ny = (nvec + 255) / 256;
      const int col0 = (nvec + ny - 1) / ny, rows = 256 / col0;
      const long long blocks = std::min<long long>((n_rows + rows - 1) / rows, (vw == 16 ? 4LL : 8LL) * num_sms());
      // a CTA's 32-bit sums: at most 128 a sample over its share of the rows
      const long long share = (n_rows + blocks - 1) / blocks * fold;
      dim3 grid(static_cast<unsigned>(share < (1LL << 24) ? blocks : (n_used + (1LL << 24) - 1) >> 24), ny);
      auto kern = vw == 16 ? k_power<16> : vw == 4 ? k_power<4> : k_power<1>;
      kern<<<grid, col0 * rows, static_cast<size_t>(std::min(n_input, col0 * vw)) * 4, st>>>(vc, n_input, fold, n_rows,
                                                                                              nvec, col0, pc);
      OVRO_LAUNCH_CHECK();
      if (taps) {
        k_sumsq<<<1, 256, 0, st>>>(opt->h_taps[c], n_tap * n, w.h2 + c);
        OVRO_LAUNCH_CHECK();
      }
    }
    k_scale<<<(n_input + 255) / 256, 256, 0, st>>>(
        w.power + static_cast<size_t>(c) * n_input,
        h_scale_or_null ? w.user + static_cast<size_t>(c) * n_input : nullptr, n_input, n,
        n_used, taps ? w.h2 + c : nullptr, w.scale + static_cast<size_t>(c) * n_input);
    OVRO_LAUNCH_CHECK();

    // twiddles: those of the plan's passes for the mixed-radix kernel; any
    // power-of-two table at least N long for the radix-16 kernel
    const bool ok = table_mr == e.mixed && (e.mixed ? table_n == n : table_n >= n);
    if (!ok) {
      table_n = e.mixed ? n : max_pow2;
      table_mr = e.mixed;
      if (e.mixed) {
        if (int err = launch_twiddle_mr(w.tw, e.plan, st)) return err;
      } else {
        k_twiddle<<<(table_n + 255) / 256, 256, 0, st>>>(w.tw, table_n);
        OVRO_LAUNCH_CHECK();
      }
    }

    UpchanArgs a;
    a.volt = d_volt + static_cast<long long>(c) * n_time * n_input;
    a.tw = w.tw;
    a.scale = w.scale + static_cast<size_t>(c) * n_input;
    a.out_q = d_fine_q + q_off;
    a.out_f = d_fine_f32_or_null ? d_fine_f32_or_null + q_off : nullptr;
    a.n_input = n_input;
    a.n_spec = e.k;
    a.tw_n = table_n;
    a.taps = taps ? opt->h_taps[c] : nullptr;
    a.n_tap = taps ? n_tap : 1;
    a.chan_lo = lo;
    a.chan_cnt = e.cnt;
    if (e.mixed) {
      if (int err = launch_upchan_mr(a, a.n_tap, st)) return err;
    } else {
      if (int err = launch_upchan_tuned(ilog2(n), a, st)) return err;
    }
    q_off += static_cast<long long>(e.cnt) * e.k * n_input * 2;
  }
  return OVRO_OK;
}

int ovro_upchan(const uint8_t* d_volt, int n_input, int n_coarse, int64_t n_time,
                const int32_t* h_nfft, const double* h_scale_or_null, int8_t* d_fine_q,
                float* d_fine_f32_or_null, void* d_ws, size_t ws_bytes, void* stream) {
  return ovro_upchan_ex(d_volt, n_input, n_coarse, n_time, h_nfft, h_scale_or_null, nullptr, d_fine_q,
                        d_fine_f32_or_null, d_ws, ws_bytes, stream);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free variant of ovro_upchan.
//
// Some callers cannot call cudaMalloc at all: a plugin hosted by a framework
// that owns the whole device heap, or a real-time acquisition loop where an
// allocation (which may synchronise the device) would stall the other streams.
// They get ovro_upchan_noalloc, whose scratch (the per-input power sums and
// scales, and the twiddle table) lives in the fixed array below.  Every GPU
// that loads this library holds the array until the process exits.
namespace ovro {
namespace {

constexpr size_t kNoAllocScratchBytes = 1u << 20;   // 1 MiB
static __device__ __align__(256) unsigned char g_upchan_scratch[kNoAllocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_ptr[kMaxDevices];     // device address per device, once found

// Device address of the scratch array for the current device (host code must
// not use the symbol itself as a device address).  Only a successful lookup
// is kept: after a failure (say, a first call made during a stream capture)
// the next call looks again.
int noalloc_scratch(void** out) {
  int dev = 0;
  OVRO_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return OVRO_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (g_scratch_ptr[dev] == nullptr) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_upchan_scratch);
    if (e != cudaSuccess) {
      set_last_error("cudaGetSymbolAddress(g_upchan_scratch)", e);
      return OVRO_ERR_CUDA;
    }
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return OVRO_OK;
}

}  // namespace
}  // namespace ovro

extern "C" {

int ovro_upchan_noalloc(const uint8_t* d_volt, int n_input, int n_coarse, int64_t n_time,
                        const int32_t* h_nfft, const double* h_scale_or_null, int8_t* d_fine_q,
                        float* d_fine_f32_or_null, void* stream) {
  using namespace ovro;
  if (n_input <= 0 || n_coarse <= 0) return OVRO_ERR_INVALID_ARG;
  const size_t need = ovro_upchan_workspace_size(n_input, n_coarse);
  if (need > kNoAllocScratchBytes) {
    snprintf_last_error("ovro_upchan_noalloc: n_input * n_coarse needs %zu bytes of scratch, "
                        "more than the fixed %zu", need, kNoAllocScratchBytes);
    return OVRO_ERR_CAPACITY;
  }
  void* scratch = nullptr;
  if (int e = noalloc_scratch(&scratch)) return e;
  return ovro_upchan(d_volt, n_input, n_coarse, n_time, h_nfft, h_scale_or_null, d_fine_q,
                     d_fine_f32_or_null, scratch, kNoAllocScratchBytes, stream);
}

}  // extern "C"
