// In-register radix-R DFTs and a shared-memory Stockham FFT used by the
// upchannelizer and the imaging kernels.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace ovro {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

template <int R>
struct BitRev {
  static __device__ __forceinline__ constexpr int of(int x) {
    int r = 0;
    for (int b = 1, m = R >> 1; b < R; b <<= 1, m >>= 1)
      if (x & b) r |= m;
    return r;
  }
};

// V[k] = sum_r v[r] exp(-2 pi i r k / R), natural order in and out.
template <int R>
__device__ __forceinline__ void dft_reg(float2 (&v)[R]) {
  float2 t[R];
#pragma unroll
  for (int i = 0; i < R; ++i) t[i] = v[BitRev<R>::of(i)];
#pragma unroll
  for (int h = 1; h < R; h <<= 1) {
#pragma unroll
    for (int b = 0; b < R; b += 2 * h) {
#pragma unroll
      for (int j = 0; j < h; ++j) {
        float2 x = t[b + j + h];
        if (j != 0) {
          // w = exp(-2 pi i j / (2h)) = exp(-2 pi i (j * 8 / h) / 16)
          const int q = j * (8 / h);
          float cw, sw;
          switch (q) {
            case 1: cw = 0.92387953251128674f; sw = -0.38268343236508977f; break;
            case 2: cw = 0.70710678118654752f; sw = -0.70710678118654752f; break;
            case 3: cw = 0.38268343236508977f; sw = -0.92387953251128674f; break;
            case 4: cw = 0.0f; sw = -1.0f; break;
            case 5: cw = -0.38268343236508977f; sw = -0.92387953251128674f; break;
            case 6: cw = -0.70710678118654752f; sw = -0.70710678118654752f; break;
            default: cw = -0.92387953251128674f; sw = -0.38268343236508977f; break;
          }
          if (q == 4) {
            x = make_float2(x.y, -x.x);           // multiply by -i
          } else {
            x = cmul(x, make_float2(cw, sw));
          }
        }
        const float2 a = t[b + j];
        t[b + j] = make_float2(a.x + x.x, a.y + x.y);
        t[b + j + h] = make_float2(a.x - x.x, a.y - x.y);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = t[i];
}

// Shared-memory index with one pad slot per 16 elements: Stockham writes at
// stride 16 become conflict-free.
__device__ __forceinline__ int pad16(int x) { return x + (x >> 4); }

// One radix-R butterfly of the pass after NS points, in registers: x[r] omega_G^(k r
// G / (NS R)), then the DFT.
template <int R, int NS, int G, class Tw>
__device__ __forceinline__ void stockham_butterfly(float2 (&x)[R], int k, Tw&& tw) {
  if (NS > 1) {
    // twiddles w^r, w = omega_G^base: w^(2^m) read, the others products of
    // those (at most three roundings deep), so a pass reads log2 R of them
    const int base = k * (G / (NS * R));
    float2 t[R];
    constexpr std::integral_constant<int, NS> ns{};
    t[1] = tw(base, ns, 0, k);
    if (R >= 4) t[2] = tw(2 * base, ns, 1, k);
    if (R >= 8) t[4] = tw(4 * base, ns, 2, k);
    if (R >= 16) t[8] = tw(8 * base, ns, 3, k);
#pragma unroll
    for (int r = 3; r < R; ++r) {
      if ((r & (r - 1)) == 0) continue;
      const int hb = 1 << (31 - __clz(r));            // highest power of two in r (compile-time)
      t[r] = cmul(t[hb], t[r - hb]);
    }
#pragma unroll
    for (int r = 1; r < R; ++r) x[r] = cmul(x[r], t[r]);
  }
  dft_reg<R>(x);
}

// One Stockham pass over rows of G points, the first NS-point transforms
// already done (G, R and NS are compile-time, so every index split is a shift).
// load(f, x, slot) gives element x of row f of the pass's input, slot (0 .. 15,
// compile-time) being which of the thread's 16 values it is; store(f, x, v) takes
// element x of its output.  in_place: the output may overlap the input (every
// read completes before the first write) and is complete for the CTA when the
// pass returns.  tw(i, ns, m, k) = omega_G^i, i = k (G / (NS R)) 2^m: where it lies in
// a table by passes, for tables laid out so.
template <int R, int NS, int G, class Load, class Tw, class Store>
__device__ __forceinline__ void stockham_pass(bool in_place, Load&& load, Tw&& tw, Store&& store) {
  // every thread holds exactly 16 values: 16 / R butterflies of radix R
  constexpr int NB = 16 / R;
  constexpr int per = G / R;
  const int T = blockDim.x;
  float2 v[16];
  int fj[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int gb = threadIdx.x + b * T;
    const int f = gb / per, j = gb - f * per;
    fj[b] = gb;
#pragma unroll
    for (int r = 0; r < R; ++r) v[b * R + r] = load(f, j + r * per, b * R + r);
  }
  if (in_place) __syncthreads();
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int f = fj[b] / per, j = fj[b] - f * per;
    const int k = j & (NS - 1);
    float2 x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = v[b * R + r];
    stockham_butterfly<R, NS, G>(x, k, tw);
    const int o = (j / NS) * NS * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) store(f, o + r * NS, x[r]);
  }
  if (in_place) __syncthreads();
}

// The last two passes at once, of radix 16 after NS points and of radix R after
// 16 NS = G / R: the R butterflies whose outputs meet in the last pass are given to
// lanes 32 / R apart and swap them by shuffles, which saves a trip through the
// exchange buffer and its barriers (of radix 8 the outputs of a warp lie so far apart
// that they cost as much).  The same arithmetic as the two passes.
template <int R, int NS, int G, class Load, class Tw, class Store>
__device__ __forceinline__ void stockham_tail(Load&& load, Tw&& tw, Store&& store) {
  constexpr int per = G / 16, KK = 32 / R;
  static_assert(per == NS * R && NS % KK == 0, "whole warps per row");
  const int f = threadIdx.x / per, jj = threadIdx.x % per;
  const int g = (jj & 31) / KK, k = (jj >> 5) * KK + (jj & (KK - 1)), j = g * NS + k;
  float2 v[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) v[r] = load(f, j + r * per, r);
  stockham_butterfly<16, NS, G>(v, k, tw);
  // R x R transposes: of v[i R + c] lane g keeps c = g, from every lane
#pragma unroll
  for (int bit = 1; bit < R; bit <<= 1) {
    const bool up = (g & bit) != 0;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      if (r & bit) continue;
      const float2 send = up ? v[r] : v[r + bit];
      const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, send.x, bit * KK),
                                     __shfl_xor_sync(0xffffffffu, send.y, bit * KK));
      if (up) v[r] = got;
      else v[r + bit] = got;
    }
  }
#pragma unroll
  for (int i = 0; i < 16 / R; ++i) {
    const int k2 = k + (i * R + g) * NS;
    float2 x[R];
#pragma unroll
    for (int c = 0; c < R; ++c) x[c] = v[i * R + c];
    stockham_butterfly<R, 16 * NS, G>(x, k2, tw);
#pragma unroll
    for (int c = 0; c < R; ++c) store(f, k2 + c * 16 * NS, x[c]);
  }
}

// Forward FFTs of rows of G = 2^LOG2G points, 16 <= G <= 16384, by the whole CTA
// with blockDim.x * 16 == rows * G: radix-16 passes, then one of radix 2, 4 or
// 8, exchanging through `a` (row f at a[f * ldp], element x at pad16(x)).  The
// first pass reads its input through load0(f, x, slot) and may overlap `a`; the
// last one hands its results to store(f, x, v): in_place when they overlap `a`, which
// TAIL (the last two passes at once, where there are two and a shorter one) rules out.
template <int LOG2G, bool TAIL, class Load, class Tw, class Store>
__device__ __forceinline__ void fft_rows_io(float2* a, int ldp, bool in_place, Load&& load0, Tw&& tw, Store&& store) {
  constexpr int G = 1 << LOG2G;
  constexpr int n16 = LOG2G / 4;
  constexpr int rem = LOG2G % 4;
  constexpr int NSR = 1 << (4 * n16);                 // transforms done before the last radix-2/4/8 pass
  static_assert(n16 >= 1 && n16 <= 3, "16 <= G <= 16384");
  auto get = [&](int f, int x, int) { return a[f * ldp + pad16(x)]; };
  auto put = [&](int f, int x, float2 v) { a[f * ldp + pad16(x)] = v; };
  if constexpr (n16 == 1 && rem == 0) {
    stockham_pass<16, 1, G>(in_place, load0, tw, store);
  } else {
    stockham_pass<16, 1, G>(true, load0, tw, put);
    if constexpr (n16 == 2 && rem == 0) {
      stockham_pass<16, 16, G>(in_place, get, tw, store);
    } else {
      if constexpr (n16 == 3) stockham_pass<16, 16, G>(true, get, tw, put);
      if constexpr (n16 == 3 && rem == 0) {
        stockham_pass<16, 256, G>(in_place, get, tw, store);
      } else if constexpr (n16 >= 2 && rem <= 2 && TAIL) {
        stockham_tail<1 << rem, NSR / 16, G>(get, tw, store);
      } else {
        if constexpr (n16 >= 2) stockham_pass<16, NSR / 16, G>(true, get, tw, put);
        stockham_pass<1 << rem, NSR, G>(in_place, get, tw, store);
      }
    }
  }
}

// The same in place.
template <int LOG2G, class Load, class Tw>
__device__ void fft_rows_inplace_f(float2* a, int ldp, Load&& load0, Tw&& tw) {
  fft_rows_io<LOG2G, false>(
      a, ldp, true, [&](int f, int x, int) { return load0(f, x); },
      [&](int i, auto, int, int) { return tw(i); },
      [&](int f, int x, float2 v) { a[f * ldp + pad16(x)] = v; });
}

}  // namespace ovro
