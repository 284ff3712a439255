// a5-a7: uvw, prolate-spheroidal gridding and dirty imaging per fine channel.
//
// Section 2.2 of the paper images every fine channel over the visible
// hemisphere; the dirty images are the search product.  Per channel:
//
//  a5  u = (x_a - x_b) s_nu in grid cells with s_nu = nu / (c du): one
//      correctly rounded FP64 multiply per coordinate, then rounded to 1/Q
//      cell.  GB300's FP64 pipe is narrow, so the kernels evaluate it as a
//      float-float product and only falls back to a real FP64 multiply when
//      the float-float bound cannot decide rint(u Q) (|frac - 1/2| within the
//      error bound) -- the integer result equals the FP64 definition exactly.
//  a6  Stokes I = (XX + YY)/2 of each kept cross baseline is gridded once (the
//      mirror conj(V) at (-u, -v) is accounted for by taking 2 Re of the
//      transform, which is exact because the mirror's footprint is the point
//      reflection), with a separable 7 x 7 prolate-spheroidal kernel.  The uv
//      position of a baseline moves by a fraction of a cell across a call's
//      channels, so the k_plan_* kernels list, once per call, the baselines that
//      can touch each 4 x 4-cell tile of the grid; k_grid_tiles gives every tile
//      to one warp whose 32 lanes are 32 adjacent channels: each lane takes
//      the tile's records for its own channel (exact uv, keep test, weights)
//      and accumulates the tile in registers, so no cell is written by two
//      threads and there are no atomics.  k_fft_rows transforms the rows.
//  a7  The uv grid is padded by 2 (G = 2N cells a side, du = 1 / (G cell)) and
//      the image is the central N x N of its transform, as padded imagers do:
//      the horizon then sits where the kernel's transform is still > 0.25, so
//      the grid correction does not amplify FP32 round-off.  The image is
//      the real part of the transform, i.e. the transform of the grid's
//      Hermitian part, whose row transforms come in conjugate pairs: k_fft_rows
//      forms that part, transforms rows 0 .. G/2 only and keeps the N central
//      columns; k_fft_cols
//      transforms those columns, keeps the N central rows, and applies the
//      (-1)^(r+c) centring sign, normalisation, grid correction and horizon
//      mask while writing the image.  The (-1)^(ku+kv) centring sign is
//      applied at gridding time, and the exp(+) transform is a forward
//      transform of the conjugated grid.  Channel batches keep the
//      intermediate half-transformed grids L2-sized.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "fft.cuh"
#include "pswf.h"
#include "stages.h"
#include "tune.h"

namespace ovro {
namespace {

constexpr double kCLight = 299792458.0;
constexpr int kQ = kOversample;
constexpr int kHalfTab = kSupport * kOversample / 2;
constexpr int kHalfSup = kSupport / 2;
constexpr int kPad = 2;              // uv grid cells per image pixel, per axis
// storage of the half-transformed grid between the row and column passes
constexpr int kStoreF32 = OVRO_STORE_FP32, kStoreBF16 = OVRO_STORE_BF16, kStoreF16 = OVRO_STORE_FP16;

struct Baseline {
  double dx, dy;
  float dxh, dxl, dyh, dyl;
  long long bl;
};

struct ChanScale {
  double s;          // s_nu * Q
  double nu_c;       // nu / c (wavelengths per metre)
  float sh, sl;      // float-float split of s
};

__host__ __device__ __forceinline__ long long bl_index(int a, int b, int n) {
  return static_cast<long long>(a) * n - static_cast<long long>(a) * (a - 1) / 2 + (b - a);
}

// rint(fl64(x * s)) decided in FP32: a float-float product, exact unless the
// fractional part is within the error bound (1.2e-7) of 1/2 or |x s| >= 2^21;
// returns false in those (rare) cases, where the FP64 product must be taken.
__device__ __forceinline__ bool fast_rint_prod(float xh, float xl, const ChanScale& s, long long* p) {
  const float hi = __fmul_rn(xh, s.sh);
  if (!(fabsf(hi) < 2097152.0f)) return false;
  const float e = __fmaf_rn(xh, s.sh, -hi);           // exact error of hi
  const float t = __fmaf_rn(xh, s.sl, __fmaf_rn(xl, s.sh, e));
  const float n = rintf(hi);
  const float f = __fadd_rn(hi - n, t);              // x s - n, |error| < 1.2e-7
  if (fabsf(fabsf(f) - 0.5f) <= 2.5e-7f) return false;
  long long q = static_cast<long long>(n);
  if (f > 0.5f) ++q;
  else if (f < -0.5f) --q;
  *p = q;
  return true;
}

__device__ __forceinline__ long long exact_rint_prod(double x, float xh, float xl, const ChanScale& s) {
  long long p;
  if (fast_rint_prod(xh, xl, s, &p)) return p;
  return __double2ll_rn(__dmul_rn(x, s.s));
}

// The same decision in 32-bit integers (|x s| < 2^21 is required anyway).
__device__ __forceinline__ bool fast_rint_prod32(float xh, float xl, const ChanScale& s, int* p) {
  const float hi = __fmul_rn(xh, s.sh);
  if (!(fabsf(hi) < 2097152.0f)) return false;
  const float e = __fmaf_rn(xh, s.sh, -hi);
  const float t = __fmaf_rn(xh, s.sl, __fmaf_rn(xl, s.sh, e));
  const float n = rintf(hi);
  const float f = __fadd_rn(hi - n, t);
  if (fabsf(fabsf(f) - 0.5f) <= 2.5e-7f) return false;
  *p = __float2int_rn(n) + (f > 0.5f ? 1 : 0) - (f < -0.5f ? 1 : 0);   // n is integral, |n| < 2^21
  return true;
}

static_assert(kQ == 1024, "centre_cell32 divides by shifting");
__device__ __forceinline__ void centre_cell32(int p, int& c0, int& off) {
  const int c = (abs(p) + kQ / 2) >> 10;
  c0 = p < 0 ? -c : c;
  off = p - c0 * kQ;
}

// a5 on its own: rounded positions p_u, p_v (1/Q cells) of every cross baseline.
__global__ void k_uvw(const Baseline* __restrict__ base, int n_cross, const ChanScale* __restrict__ cs,
                      int32_t* __restrict__ pu, int32_t* __restrict__ pv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int f = blockIdx.y;
  if (i >= n_cross) return;
  const Baseline B = base[i];
  const ChanScale s = cs[f];
  const long long u = exact_rint_prod(B.dx, B.dxh, B.dxl, s);
  const long long v = exact_rint_prod(B.dy, B.dyh, B.dyl, s);
  const long long lim = 1LL << 30;
  const long long o = static_cast<long long>(f) * n_cross + i;
  pu[o] = static_cast<int32_t>(u > lim ? lim : (u < -lim ? -lim : u));
  pv[o] = static_cast<int32_t>(v > lim ? lim : (v < -lim ? -lim : v));
}

// device counters of one call's plan (ImgWs::counts)
constexpr int kCountListed = 0, kCountRows = 1, kCountSlots = 2, kCountHeavy = 3, kCounts = 4;

struct GridEntry {
  int bl;            // baseline index in the visibility record
  int cross;         // cross-baseline index (FP64 fallback, baseline length)
  int a;             // antennas a < b
  int bf;            // b | kCheckUv when the uv range must be decided per channel
  float dxh, dxl, dyh, dyl;
};
constexpr int kCheckUv = 1 << 16;

// Calibration and baseline-selection options of one gridding call.
struct GridOpts {
  const float2* gains;      // [n_chan][n_input] corrections or nullptr
  int n_input;
  const double* blen;       // [n_cross] baseline lengths, metres (FP64)
  double uv_min, uv_max;    // wavelengths, [uv_min, uv_max)
};

// Row pitch of a shared-memory grid band: G + G/16 pad slots, rounded so the
// pitch is 7 (mod 16) float2 -- consecutive rows then start 14 banks apart and
// 16 consecutive transposed columns hit distinct banks.
__host__ __device__ constexpr int band_pitch(int g) { return (g + g / 16) + ((7 - (g + g / 16) % 16) + 16) % 16; }

// Gridding tiles.  A warp owns a kTileV x kTileU tile of grid cells for 32
// consecutive channels, one channel per lane, and keeps the tile's 32 complex
// accumulators of its channel in registers.  Every lane of a warp takes the
// same visibility record at the same time; across 32 adjacent fine channels a
// baseline's uv position moves by far less than a cell, so the lanes' centre
// cells agree (or differ by one) and their table reads hit the same words.
// No two warps write the same (cell, channel): there are no atomics.
constexpr int kTileV = 4, kTileU = 4;          // cells per warp tile (rows, columns)
constexpr int kLanes = 32;                     // channels per warp

// Tiles cover the rows G/2 .. G-1 (v >= 0) of the grid's Hermitian part only
// (the rows below are the conjugate reflection).
__host__ __device__ constexpr int n_tiles_u(int g) { return g / kTileU; }
__host__ __device__ constexpr int n_tiles(int g) { return (g / 2 / kTileV) * (g / kTileU); }

// Weights of the separable kernel indexed by (d, off): a tap d cells from the
// centre cell of a position whose offset from that cell is off / Q weighs
// C(d - off / Q) when |d| <= 3 and 0 otherwise.  The table holds every d in
// [-kTabD, kTabD] at stride Q + 1, so (d, off) -> (d + kTabD) (Q + 1) + Q / 2 - off
// is one-to-one over off in [-Q/2, Q/2] (d = 3 at off = -Q/2 and d = 4 at
// off = Q/2 land on different entries) and a tile's weights are plain loads at
// fixed strides from one base, with no range tests.  Offsets a tile column
// can take when the footprint touches the tile lie in [-(3 + kTileU - 1), 3];
// the kTabMargin rows beyond them (zeros) let a lane whose centre is up to
// kTabMargin cells from a tile it is listed for read zeros there.
constexpr int kTabMargin = 4;
constexpr int kTabD = kHalfSup + kTileU - 1 + kTabMargin;   // 10
constexpr int kTabStride = kQ + 1;
constexpr int kTabXLen = (2 * kTabD + 1) * kTabStride;
constexpr int kTabBytes = 8;         // the tile kernel holds every weight twice, for packed arithmetic

// Per-channel record of one listed baseline, prepared once per channel group
// by k_grid_prep: its exact rounded position p = rint(u Q), rint(v Q) and its
// value in the Hermitian part of the grid, conj(Stokes I) / 2, or V = 0 when
// the visibility is not gridded in that channel.  Layout [group][listed][32].
// With table bases (a call whose footprints move by less than kTabMargin
// cells over its channels), pu and pv hold instead the byte offsets of the
// position in the tile kernel's table (8 bytes an entry): column c's weight is
// entry pu / 8 + c (Q + 1), row r's pv / 8 + r (Q + 1) (r, c grid indices), zero
// beyond the footprint.
struct PrepRec {
  int pu, pv;
  float vr, vi;
};
constexpr int kMirror = 1 << 31;    // tile list flag: grid the record's mirror (-u, -v, conj V)

// Table offset of a position with centre cell c and offset off (1/Q cells)
// on an axis of G cells; the mirror position (-c, -off) has offset
// tab_mirror(G) - tab_base(G, c, off).
__host__ __device__ constexpr int tab_base(int g, int c, int off) {
  return (kTabD - g / 2 - c) * kTabStride + kQ / 2 - off;
}
__host__ __device__ constexpr int tab_mirror(int g) { return 2 * (kTabD - g / 2) * kTabStride + kQ; }

// a5 and the Stokes I of a6 for one channel group and kPrepBl listed
// baselines per CTA: for each (channel, baseline) a thread decides the exact
// rounded position (float-float, FP64 when that cannot decide), the keep test
// (centre cell inside the grid's margin; the uv range when it must be decided
// per channel), reads XX and YY and forms the record -- the image is the real
// part of the transform, i.e. the transform of the grid's Hermitian part
// H = (G + conj G(-u, -v)) / 2, so the record carries half of
// conj(Stokes I) = conj(XX + YY) / 4 (the exp(+) transform is a forward FFT of
// the conjugated grid); calibration corrections c_a conj(c_b) are applied per
// polarisation in FP32 when given.  Lanes are baselines while the
// visibilities are read (a warp reads consecutive baselines of one channel:
// nearly sequential 32-byte records), and the records are turned around in
// shared memory so each baseline's 32 channel records are stored as one
// 512-byte run ([group][listed][lane], n_cross listed slots per group).  Kept visibilities are counted per
// channel.
constexpr int kPrepBl = 64;          // listed baselines per CTA of k_grid_prep
constexpr int kPrepCh = kLanes / 8;  // channels per warp (8 warps)

template <int LOG2G, bool CAL, bool BASES>
__global__ void __launch_bounds__(256, CAL ? 1 : 4)
k_grid_prep(const GridEntry* __restrict__ listed, const unsigned long long* __restrict__ counts, long long n_cross,
            const int32_t* __restrict__ vis, long long n_bl, const Baseline* __restrict__ base,
            const ChanScale* __restrict__ cs, int ch0, int nb, int* __restrict__ kept, PrepRec* __restrict__ prep,
            GridOpts opt) {
  constexpr int G = 1 << LOG2G;
  // [baseline][channel] records, rows padded by one record so that the lanes'
  // 16-byte stores (lanes = baselines) fall in distinct banks
  __shared__ int4 tile[kPrepBl][kLanes + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int group = blockIdx.y;
  const int i0 = blockIdx.x * kPrepBl;
  const int nbl = min(kPrepBl, static_cast<int>(counts[kCountListed]) - i0);
  if (nbl <= 0) return;                                // the grid covers every cross baseline
  const int cmax = G / 2 - kHalfSup - 1;
  const int lim = (cmax + 1) * kQ;                     // < 2^21
  // this lane's two baselines (i0 + lane, i0 + lane + 32)
  GridEntry en[2];
  bool has[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int bi = lane + 32 * h;
    has[h] = bi < nbl;
    en[h] = listed[i0 + (has[h] ? bi : 0)];
  }
  // every visibility read of the thread (kPrepCh channels x 2 baselines) is
  // issued before any is used
  int2 xx[kPrepCh][2], yy[kPrepCh][2];
#pragma unroll
  for (int cc = 0; cc < kPrepCh; ++cc) {
    const int cb = group * kLanes + warp * kPrepCh + cc;
    const long long chan = ch0 + (cb < nb ? cb : nb - 1);
    const int2* vis2 = reinterpret_cast<const int2*>(vis) + chan * n_bl * 4;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      xx[cc][h] = __ldg(vis2 + static_cast<long long>(en[h].bl) * 4);
      yy[cc][h] = __ldg(vis2 + static_cast<long long>(en[h].bl) * 4 + 3);
    }
  }
#pragma unroll
  for (int cc = 0; cc < kPrepCh; ++cc) {
    const int cl = warp * kPrepCh + cc;              // channel within the group
    const int cb = group * kLanes + cl;
    const bool active = cb < nb;
    const long long chan = ch0 + (active ? cb : nb - 1);
    const ChanScale sc = cs[chan];
    const float2* gc = (CAL && opt.gains != nullptr) ? opt.gains + chan * opt.n_input : nullptr;
    int n_kept = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const GridEntry& e = en[h];
      int pu, pv;
      if (!fast_rint_prod32(e.dxh, e.dxl, sc, &pu)) {
        const long long pl = __double2ll_rn(__dmul_rn(base[e.cross].dx, sc.s));
        pu = static_cast<int>(pl > lim ? lim : (pl < -lim ? -lim : pl));
      }
      if (!fast_rint_prod32(e.dyh, e.dyl, sc, &pv)) {
        const long long pl = __double2ll_rn(__dmul_rn(base[e.cross].dy, sc.s));
        pv = static_cast<int>(pl > lim ? lim : (pl < -lim ? -lim : pl));
      }
      bool keep = pu > -lim && pu < lim && pv > -lim && pv < lim;
      if (keep) {
        int cu, cv, o;
        centre_cell32(pu, cu, o);
        centre_cell32(pv, cv, o);
        keep = cu <= cmax && cu >= -cmax && cv <= cmax && cv >= -cmax;
      }
      if (CAL && (e.bf & kCheckUv)) {
        const double lam = __dmul_rn(opt.blen[e.cross], sc.nu_c);
        keep = keep && lam >= opt.uv_min && lam < opt.uv_max;
      }
      PrepRec r{lim, lim, 0.0f, 0.0f};
      if (BASES) {
        // the position's table offsets, kept or not (a record is only read for
        // tiles within kTabMargin cells of its footprint)
        int cu, cv, ou, ov;
        centre_cell32(pu, cu, ou);
        centre_cell32(pv, cv, ov);
        r.pu = kTabBytes * tab_base(G, cu, ou);
        r.pv = kTabBytes * tab_base(G, cv, ov);
      }
      if (keep) {
        float vr, vi;
        if (!CAL || gc == nullptr) {
          vr = 0.25f * static_cast<float>(xx[cc][h].x + yy[cc][h].x);
          vi = -0.25f * static_cast<float>(xx[cc][h].y + yy[cc][h].y);
        } else {
          const int a = e.a, b = e.bf & 0xffff;
          float pr = 0.f, pi = 0.f;
#pragma unroll
          for (int pol = 0; pol < 2; ++pol) {
            const float2 ca = __ldg(gc + 2 * a + pol), cbv = __ldg(gc + 2 * b + pol);
            const int2 q = pol ? yy[cc][h] : xx[cc][h];
            const float qr = static_cast<float>(q.x), qi = static_cast<float>(q.y);
            const float gr = ca.x * cbv.x + ca.y * cbv.y, gi = ca.y * cbv.x - ca.x * cbv.y;
            pr += gr * qr - gi * qi;
            pi += gr * qi + gi * qr;
          }
          vr = 0.25f * pr;
          vi = -0.25f * pi;
        }
        if (!BASES) {
          r.pu = pu;
          r.pv = pv;
        }
        r.vr = vr;
        r.vi = vi;
        if (has[h]) ++n_kept;
      }
      tile[lane + 32 * h][cl] = make_int4(r.pu, r.pv, __float_as_int(r.vr), __float_as_int(r.vi));
    }
    // the channel's kept visibilities over the warp's 64 baselines
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n_kept += __shfl_xor_sync(0xffffffffu, n_kept, o);
    if (lane == 0 && active && n_kept) atomicAdd(kept + chan, n_kept);
  }
  __syncthreads();
  // one baseline's 32 channel records per warp store: 512 contiguous bytes
  int4* out = reinterpret_cast<int4*>(prep) + (static_cast<long long>(group) * n_cross + i0) * kLanes;
  for (int bi = warp; bi < nbl; bi += 8) out[static_cast<long long>(bi) * kLanes + lane] = tile[bi][lane];
}

// Rows of the half-transformed grid kept per channel: the gridded plane is the
// Hermitian part H of the grid on its rows j = G/2 .. G-1; the row transforms
// of H satisfy R(G - j, k) = conj R(j, k), and row 0 is empty (no footprint
// reaches it), so these G/2 rows carry everything the column pass needs.
__host__ __device__ constexpr int half_rows(int g) { return g / 2; }

// A row-pass CTA transforms row_lines(G) lines (8192 points; every row of the
// smallest grids): row_chans(G) channels of as many rows each as fit, whose
// values of four cells are 256 (128 at 2048 points) contiguous bytes of the grid.
__host__ __device__ constexpr int row_lines(int g) { return 8192 / g < 4 * g ? 8192 / g : 4 * g; }
__host__ __device__ constexpr int row_chans(int g) { return row_lines(g) < 8 ? row_lines(g) : 8; }
__host__ __device__ constexpr int row_rows(int g) { return row_lines(g) / row_chans(g); }

// Gridding of one channel batch into the Hermitian part of the grid, rows
// G/2 .. G-1 (v >= 0; a record whose footprint lies below is listed as its
// mirror, one straddling row G/2 as both).  Work items are (warp tile, group of
// 32 channels) pairs, the tiles of kHeavy entries and more first and the others
// as they lie: from the middle rows of the plane, where the lists are long,
// outwards, and neighbours together, whose records and lines of the grid then
// meet in L2 (from the longest list to the shortest, the stores of a sparse
// grid went to DRAM line by line: 0.53 against 0.35 ms at 64 channels of
// 1024^2).  The warps of the persistent grid (one CTA of kGridWarps warps per
// SM) draw items from a counter, the next one while they work on the last.  The
// gap-indexed weight table sits in shared memory with
// every weight twice, so that one 8-byte load gives both factors of a packed
// multiply-add on a cell's (re, im): a record costs a lane one 16-byte load,
// 8 table loads, 4 + 16 packed multiply(-add)s and its decoding, where scalar
// arithmetic took 8 + 32.  kRing records are in flight per warp, a quad of
// list entries ahead of them; whole quads run without a branch, so the loads
// of one record overlap the arithmetic of the last.
//   BASES: the record holds the table offsets of its position, so the weights
//     are 8 loads at fixed strides from (offset + tile origin) and a lane off
//     the footprint reads the table's zero rows;
//   otherwise the lane takes the centre cells from the position and adds
//     zeros when its footprint misses the tile.
// The tile is written with the (-1)^(row + col) centring sign to grid
// [group][G/2][G/4][32 channels][4 cells] (row j - G/2): a row of the tile and
// channel is one 32-byte store, 1 KB a warp.  With a plane per channel every lane
// wrote halves of sectors of its own, and that bounded sparse grids; with planes
// of 4 or 8 channels the lines went to DRAM in pieces.  Before (scalar, plane per channel,
// static items) -> now, 352 antennas: 1000 channels of 256^2 1.16 -> 0.69 ms,
// 300 of 512^2 1.32 -> 0.46 ms, 64 of 1024^2 1.97 -> 0.35 ms.
constexpr int kGridWarps = 20;
constexpr int kHeavy = 256;        // list entries of a tile that is taken first
constexpr int kRing = 4;           // records in flight per warp: one quad of list entries
constexpr size_t kTileSmem = static_cast<size_t>(kTabXLen) * kTabBytes;

// (a.x b.x, a.y b.y) and (a.x b.x + c.x, a.y b.y + c.y), each rounded once
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long pack2(int lo, int hi) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}

template <int LOG2G, bool BASES>
__global__ void __launch_bounds__(kGridWarps * 32, 1)
k_grid_tiles(const int4* __restrict__ tile_idx, const int2* __restrict__ tile_rng, const int* __restrict__ heavy,
             const unsigned long long* __restrict__ counts, const PrepRec* __restrict__ prep, long long n_cross, const float* __restrict__ tabx_g, int nb,
             unsigned* __restrict__ next_item, float2* __restrict__ grid) {
  constexpr int G = 1 << LOG2G;
  constexpr int NTU = n_tiles_u(G);
  constexpr int NT = n_tiles(G);
  constexpr int STEP = kTabStride * kTabBytes;        // bytes from one grid cell's weight to the next
  extern __shared__ __align__(16) unsigned char smem[];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kTabXLen; i += blockDim.x) {
    const float w = __ldg(tabx_g + i);
    reinterpret_cast<float2*>(smem)[i] = make_float2(w, w);
  }
  __syncthreads();
  const unsigned n_groups = static_cast<unsigned>((nb + kLanes - 1) / kLanes);
  const unsigned n_first = static_cast<unsigned>(counts[kCountHeavy]) * n_groups;
  const unsigned n_items = n_first + n_groups * NT;
  auto draw = [&]() {
    unsigned i = 0;
    if (lane == 0) i = atomicAdd(next_item, 1u);
    return i;
  };
  unsigned item = __shfl_sync(full, draw(), 0);
#pragma unroll 1
  while (item < n_items) {
    const unsigned after = draw();                     // broadcast once this item is done
    const bool first = item < n_first;
    const unsigned at = first ? item : item - n_first;
    const int g = static_cast<int>(at % n_groups);
    const int tile = first ? __ldg(heavy + at / n_groups) : static_cast<int>(at / n_groups);
    const int2 rng = __ldg(tile_rng + tile);
    if (!first && rng.y - rng.x >= kHeavy) {           // done among the first
      item = __shfl_sync(full, after, 0);
      continue;
    }
    const PrepRec* pg = prep + static_cast<long long>(g) * n_cross * kLanes + lane;
    const int tv = tile / NTU, tu = tile - tv * NTU;
    const int r0 = G / 2 + tv * kTileV, c0 = tu * kTileU;
    unsigned long long acc[kTileV][kTileU];            // (re, im)
#pragma unroll
    for (int i = 0; i < kTileV; ++i)
#pragma unroll
      for (int j = 0; j < kTileU; ++j) acc[i][j] = 0ull;
    auto load_rec = [&](int ent) {
      return __ldg(reinterpret_cast<const int4*>(pg + static_cast<long long>(ent & ~kMirror) * kLanes));
    };
    // bu, bv: byte offsets of the tile's first column's and row's weights
    auto accumulate = [&](int bu, int bv, unsigned long long v) {
      unsigned long long wv[kTileV], wu[kTileU];
#pragma unroll
      for (int i = 0; i < kTileV; ++i) wv[i] = *reinterpret_cast<const unsigned long long*>(smem + bv + i * STEP);
#pragma unroll
      for (int j = 0; j < kTileU; ++j) wu[j] = *reinterpret_cast<const unsigned long long*>(smem + bu + j * STEP);
#pragma unroll
      for (int i = 0; i < kTileV; ++i) {
        const unsigned long long b = mul2(wv[i], v);
#pragma unroll
        for (int j = 0; j < kTileU; ++j) acc[i][j] = fma2(b, wu[j], acc[i][j]);
      }
    };
    // one list entry: the record (mirrored if flagged) decoded here, at its use
    auto grid_one = [&](int4 v, int ent) {
      const int s = ent >> 31;                         // -1: the mirror (-u, -v, conj V)
      const unsigned long long val = pack2(v.z, v.w ^ (s & kMirror));
      if (BASES) {
        // the mirror's offset is tab_mirror - offset = tab_mirror + 1 + ~offset
        const int m = s & (kTabBytes * tab_mirror(G) + 1);
        accumulate((v.x ^ s) + m + c0 * STEP, (v.y ^ s) + m + r0 * STEP, val);
        return;
      }
      int cu, offu, cv, offv;
      centre_cell32(s ? -v.x : v.x, cu, offu);
      centre_cell32(s ? -v.y : v.y, cv, offv);
      int dv0 = r0 - (G / 2 + cv), du0 = c0 - (G / 2 + cu);   // offsets of the tile's first row / column
      const bool touch = dv0 <= kHalfSup && dv0 >= -(kHalfSup + kTileV - 1) && du0 <= kHalfSup &&
                         du0 >= -(kHalfSup + kTileU - 1);
      if (__any_sync(full, touch)) {
        // a lane whose footprint misses the tile adds zeros; its table reads
        // stay inside the table
        if (!touch) dv0 = du0 = offu = offv = 0;
        accumulate(((du0 + kTabD) * kTabStride + kQ / 2 - offu) * kTabBytes,
                   ((dv0 + kTabD) * kTabStride + kQ / 2 - offv) * kTabBytes, touch ? val : 0ull);
      }
    };
    if (rng.y > rng.x) {
      // lists start on a quad and are padded to whole quads (entry 0)
      const int last = (rng.y - 1) >> 2;
      int q = rng.x >> 2;
      int4 e = __ldg(tile_idx + q), en = __ldg(tile_idx + min(q + 1, last));
      int4 rec[kRing] = {load_rec(e.x), load_rec(e.y), load_rec(e.z), load_rec(e.w)};
#pragma unroll 1
      for (const int whole = rng.y >> 2; q < whole; ++q) {
        const int4 ahead = __ldg(tile_idx + min(q + 2, last));
        grid_one(rec[0], e.x);
        rec[0] = load_rec(en.x);
        grid_one(rec[1], e.y);
        rec[1] = load_rec(en.y);
        grid_one(rec[2], e.z);
        rec[2] = load_rec(en.z);
        grid_one(rec[3], e.w);
        rec[3] = load_rec(en.w);
        e = en;
        en = ahead;
      }
      const int rest = rng.y & 3;
      if (rest > 0) grid_one(rec[0], e.x);
      if (rest > 1) grid_one(rec[1], e.y);
      if (rest > 2) grid_one(rec[2], e.z);
    }
    // ---- the tile, with the centring sign (r0 and c0 are even)
    if (g * kLanes + lane < nb) {
      float2* out = grid + ((static_cast<long long>(g) * (G / 2) + r0 - G / 2) * G + c0) * kLanes + lane * kTileU;
#pragma unroll
      for (int i = 0; i < kTileV; ++i) {
        unsigned long long z[kTileU];
#pragma unroll
        for (int j = 0; j < kTileU; ++j) z[j] = (i + j) & 1 ? acc[i][j] ^ 0x8000000080000000ull : acc[i][j];
        asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(out + i * G * kLanes), "l"(z[0]), "l"(z[1]),
                     "l"(z[2]), "l"(z[3])
                     : "memory");
      }
    }
    item = __shfl_sync(full, after, 0);
  }
}

// The central N columns of the CTA's row transforms (line f = channel
// f / row_rows, row f % row_rows) in 16-bit storage.
template <int G, int LDP, int S>
__device__ __forceinline__ void store_band(const float2* band, int cb0, int row0, int nb, int n_img, void* h,
                                           float* hs) {
  constexpr int R = row_rows(G);
  const int offc = G / 2 - n_img / 2;
  const int lines = min(row_chans(G), nb - cb0) * R;    // the channels of the batch
  auto row_of = [&](int f) { return static_cast<long long>(cb0 + f / R) * half_rows(G) + row0 + f % R; };
  if constexpr (S == kStoreBF16) {
    for (int i = threadIdx.x; i < lines * n_img; i += blockDim.x) {
      const int f = i / n_img, c = i - f * n_img;
      static_cast<__nv_bfloat162*>(h)[row_of(f) * n_img + c] = __float22bfloat162_rn(band[f * LDP + pad16(offc + c)]);
    }
  } else {
    // FP16 with a power-of-two scale per row: the row's largest component
    // lands in [2^13, 2^14), far from FP16 overflow; scaling is exact
    const int lane = threadIdx.x & 31, n_w = blockDim.x >> 5;
    for (int f = threadIdx.x >> 5; f < lines; f += n_w) {
      const long long row = row_of(f);
      float m = 0.f;
      for (int c = lane; c < n_img; c += 32) {
        const float2 v = band[f * LDP + pad16(offc + c)];
        m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      int e = 0;
      if (m > 0.f) frexpf(m, &e);
      const float sc = m > 0.f ? ldexpf(1.0f, 14 - e) : 1.0f;
      if (lane == 0) hs[row] = m > 0.f ? ldexpf(1.0f, e - 14) : 0.0f;
      for (int c = lane; c < n_img; c += 32) {
        const float2 v = band[f * LDP + pad16(offc + c)];
        static_cast<__half2*>(h)[row * n_img + c] = __float22half2_rn(make_float2(v.x * sc, v.y * sc));
      }
    }
  }
}

// ------------------------------------------------------------ line FFTs
// Forward FFTs of G = 2^LOG2G points (32 .. 2048) along lines in shared memory:
// a radix-16 pass, one of radix 2 .. 16 (16 points done) and, from 512 points
// on, one of radix 2, 4 or 8 (256 done).  Every thread holds 16 values.  The
// passes are issue bound, so the additions are packed (re, im), the twiddles
// of a pass are read from a table of its own laid out [factor][k] (a warp's
// reads are consecutive; from one table of powers they met in few banks, which
// had to be traded against products of powers), the first pass reads wherever
// the lines come from and the last one hands its values to a functor instead
// of another trip through shared memory.  Against the shared passes of
// fft.cuh with staged input and output, 352 antennas: 1000 channels of 256^2
// rows 0.60 -> 0.46 ms, columns 0.42 -> 0.31 ms; 300 of 512^2 0.72 -> 0.52 and
// 0.54 -> 0.39 ms.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 p, q, r;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tadd.rn.f32x2 r, p, q;\n\t"
      "mov.b64 {%0, %1}, r;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
// a + s b for a pair of signs or factors s
__device__ __forceinline__ float2 axpy2(float2 a, float s, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 p, q, r;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tmov.b64 r, {%6, %6};\n\t"
      "fma.rn.f32x2 r, q, r, p;\n\tmov.b64 {%0, %1}, r;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(s));
  return d;
}

// (a, b) <- (a + w b, a - w b), w = exp(-2 pi i Q / 16)
template <int Q>
__device__ __forceinline__ void bfly(float2& a, float2& b) {
  constexpr float r2 = 0.70710678118654752f;
  if constexpr (Q == 0) {
    const float2 x = b;
    b = axpy2(a, -1.0f, x);
    a = add2(a, x);
  } else if constexpr (Q == 4) {
    const float2 x = b, y = a;                          // -i x = (x.y, -x.x)
    a = make_float2(y.x + x.y, y.y - x.x);
    b = make_float2(y.x - x.y, y.y + x.x);
  } else if constexpr (Q == 2 || Q == 6) {
    // r2 (1 - i) x and r2 (-1 - i) x: the factor goes into the sums
    const float2 u = Q == 2 ? make_float2(b.x + b.y, b.y - b.x) : make_float2(b.y - b.x, -b.x - b.y);
    const float2 y = a;
    a = axpy2(y, r2, u);
    b = axpy2(y, -r2, u);
  } else {
    constexpr float cw = Q == 1 ? 0.92387953251128674f : Q == 3 ? 0.38268343236508977f
                         : Q == 5 ? -0.38268343236508977f : -0.92387953251128674f;
    constexpr float sw = Q == 1 || Q == 7 ? -0.38268343236508977f : -0.92387953251128674f;
    const float2 x = cmul(b, make_float2(cw, sw));
    b = axpy2(a, -1.0f, x);
    a = add2(a, x);
  }
}

// V[k] = sum_r v[r] exp(-2 pi i r k / R), in natural order; R = 2, 4, 8, 16.
template <int R>
__device__ __forceinline__ void dft_line(float2* v) {
  float2 t[R];
#pragma unroll
  for (int i = 0; i < R; ++i) t[i] = v[BitRev<R>::of(i)];
#pragma unroll
  for (int i = 0; i < R; i += 2) bfly<0>(t[i], t[i + 1]);
  if constexpr (R >= 4) {
#pragma unroll
    for (int i = 0; i < R; i += 4) {
      bfly<0>(t[i], t[i + 2]);
      bfly<4>(t[i + 1], t[i + 3]);
    }
  }
  if constexpr (R >= 8) {
#pragma unroll
    for (int i = 0; i < R; i += 8) {
      bfly<0>(t[i], t[i + 4]);
      bfly<2>(t[i + 1], t[i + 5]);
      bfly<4>(t[i + 2], t[i + 6]);
      bfly<6>(t[i + 3], t[i + 7]);
    }
  }
  if constexpr (R >= 16) {
    bfly<0>(t[0], t[8]);
    bfly<1>(t[1], t[9]);
    bfly<2>(t[2], t[10]);
    bfly<3>(t[3], t[11]);
    bfly<4>(t[4], t[12]);
    bfly<5>(t[5], t[13]);
    bfly<6>(t[6], t[14]);
    bfly<7>(t[7], t[15]);
  }
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = t[i];
}

// Twiddle tables of the second and third pass: [R2][16] with R2 = min(G / 16, 16)
// of exp(-2 pi i r k / (16 R2)), then, from 512 points on, [G / 256][256] of
// exp(-2 pi i r k / G).  Behind them omega_G^k, k < G, for 16-bit storage.
__host__ __device__ constexpr int tw_entries(int g) { return g <= 256 ? g : 256 + g; }
__host__ __device__ constexpr int tw_all(int g) { return tw_entries(g) + g; }

// One pass of radix R over `NS` done points: load(f, x) gives point x of line f
// and store(f, x, v) takes point x of its result; split(i, f, j) the line and
// index of butterfly i (all of the CTA's, in the order the threads take them).
// in_place: the results overwrite the input.
template <int R, int NS, int G, class Split, class Load, class Store>
__device__ __forceinline__ void line_pass(const float2* tw, bool in_place, Split&& split, Load&& load, Store&& store) {
  constexpr int NB = 16 / R;
  float2 v[16];
  int f[NB], j[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    split(static_cast<int>(threadIdx.x + b * blockDim.x), f[b], j[b]);
#pragma unroll
    for (int r = 0; r < R; ++r) v[b * R + r] = load(f[b], j[b] + r * (G / R));
  }
  if (in_place) __syncthreads();                        // every read before the first write
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int k = j[b] & (NS - 1);
    if constexpr (NS > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[b * R + r] = cmul(v[b * R + r], tw[r * NS + k]);
    }
    dft_line<R>(v + b * R);
    const int o = (j[b] / NS) * NS * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) store(f[b], o + r * NS, v[b * R + r]);
  }
  if (in_place) __syncthreads();
}

// load0(f, x), split0: the first pass's input and item order; store(f, x, v),
// split1: the last pass's output and item order.
// Lines lie at a[f * ldp], element x at pad16(x), in between; blockDim.x * 16 ==
// lines * G.
template <int LOG2G, class Split0, class Load0, class Split1, class Store>
__device__ __forceinline__ void fft_lines(float2* a, int ldp, const float2* tw, Split0&& split0, Load0&& load0,
                                          Split1&& split1, Store&& store) {
  constexpr int G = 1 << LOG2G;
  constexpr int R2 = G / 16 < 16 ? G / 16 : 16;
  static_assert(G >= 32 && G <= 2048, "two or three passes");
  auto put = [&](int f, int x, float2 v) { a[f * ldp + pad16(x)] = v; };
  auto get = [&](int f, int x) { return a[f * ldp + pad16(x)]; };
  line_pass<16, 1, G>(tw, true, split0, load0, put);
  if constexpr (G <= 256) {
    line_pass<R2, 16, G>(tw, false, split1, get, store);
  } else {
    auto split = [&](int i, int& f, int& j) {
      f = i / (G / 16);
      j = i % (G / 16);
    };
    line_pass<16, 16, G>(tw, true, split, get, put);
    line_pass<G / 256, 256, G>(tw + 256, false, split1, get, store);
  }
}

// The row transforms' last butterflies have radix last_radix(G).
__host__ __device__ constexpr int last_radix(int g) { return g <= 256 ? g / 16 : g / 256; }

// Row transforms of the gridded half planes: a CTA copies its channels' rows in
// (64 KB) and transforms them; the central N columns go to h
// ([batch][G/2][N], row j - G/2), straight from the last pass.  With 16-bit
// storage the rows go through fft_rows_inplace_f instead: rounding to 16 bits
// turns a last-bit difference of a row into one of 2^-9 or 2^-12, and images
// keep the bits they had.
template <int LOG2G, int S>
__global__ void __launch_bounds__(512, 2)
k_fft_rows(const float2* __restrict__ grid, const float2* __restrict__ tw_g, int nb, int n_img,
           void* __restrict__ h, float* __restrict__ hs) {
  constexpr int G = 1 << LOG2G;
  constexpr int LDP = band_pitch(G);
  constexpr int CH = row_chans(G), R = row_rows(G);
  extern __shared__ __align__(16) unsigned char smem[];
  float2* band = reinterpret_cast<float2*>(smem);     // [row_lines][LDP]; first the input [R][G/4][CH][4]
  float2* tw = band + row_lines(G) * LDP;
  // the CTAs of one row's channels run next to one another: they share its lines
  const int cb0 = blockIdx.x * CH, row0 = blockIdx.y * R;
  const float4* src = reinterpret_cast<const float4*>(grid) +
                      (static_cast<long long>(cb0 / kLanes) * half_rows(G) + row0) * (G / 4) * (2 * kLanes) +
                      cb0 % kLanes * 2;
  float4 q[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = threadIdx.x + u * blockDim.x;       // ((row, col / 4), 16-byte piece)
    q[u] = __ldg(src + i / (2 * CH) * (2 * kLanes) + i % (2 * CH));
  }
  constexpr int TW0 = S == kStoreF32 ? 0 : tw_entries(G), TWN = S == kStoreF32 ? tw_entries(G) : G;
  for (int i = threadIdx.x; i < TWN; i += blockDim.x) tw[i] = __ldg(tw_g + TW0 + i);
#pragma unroll
  for (int u = 0; u < 8; ++u) reinterpret_cast<float4*>(band)[threadIdx.x + u * blockDim.x] = q[u];
  __syncthreads();
  // the first pass takes four cells and the channels in adjacent lanes, as
  // they lie in shared memory
  constexpr int J = G / 16 < 4 ? G / 16 : 4;
  auto split0 = [&](int i, int& f, int& j) {
    const int x = i / (J * CH);                       // (row, group of J butterflies)
    f = (i / J % CH) * R + x / (G / 16 / J);
    j = x % (G / 16 / J) * J + i % J;
  };
  auto load0 = [&](int f, int x) { return band[(((f % R) * (G / 4) + x / 4) * CH + f / R) * 4 + x % 4]; };
  if constexpr (S == kStoreF32) {
    constexpr int PER = G / last_radix(G);
    const int offc = G / 2 - n_img / 2;
    fft_lines<LOG2G>(
        band, LDP, tw, split0, load0,
        [&](int i, int& f, int& j) {
          f = i / PER;
          j = i % PER;
        },
        [&](int f, int x, float2 v) {
          const int cb = cb0 + f / R, c = x - offc;
          if (cb < nb && static_cast<unsigned>(c) < static_cast<unsigned>(n_img))
            static_cast<float2*>(h)[(static_cast<long long>(cb) * half_rows(G) + row0 + f % R) * n_img + c] = v;
        });
  } else {
    fft_rows_inplace_f<LOG2G>(band, LDP, load0, [&](int i) { return tw[i]; });
    store_band<G, LDP, S>(band, cb0, row0, nb, n_img, h, hs);
  }
}

// Two adjacent values (idx even) of the half-transformed grid in FP32.
template <int S>
__device__ __forceinline__ void load_h2(const void* h, const float* hs, long long row, long long idx, float2& v0,
                                        float2& v1) {
  if constexpr (S == kStoreF32) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(static_cast<const float2*>(h) + idx));
    v0 = make_float2(q.x, q.y);
    v1 = make_float2(q.z, q.w);
  } else {
    const uint2 raw = __ldg(reinterpret_cast<const uint2*>(static_cast<const unsigned*>(h) + idx));
    if constexpr (S == kStoreBF16) {
      __nv_bfloat162 b0, b1;
      memcpy(&b0, &raw.x, sizeof(b0));
      memcpy(&b1, &raw.y, sizeof(b1));
      v0 = __bfloat1622float2(b0);
      v1 = __bfloat1622float2(b1);
    } else {
      __half2 b0, b1;
      memcpy(&b0, &raw.x, sizeof(b0));
      memcpy(&b1, &raw.y, sizeof(b1));
      const float sc = __ldg(hs + row);
      v0 = __half22float2(b0);
      v1 = __half22float2(b1);
      v0 = make_float2(v0.x * sc, v0.y * sc);
      v1 = make_float2(v1.x * sc, v1.y * sc);
    }
  }
}

// Column transforms of the N central columns and the image itself.
//
// The row transforms are of the Hermitian part of the grid, so every column c
// satisfies c(-k) = conj c(k) and its DFT is real: two columns c1, c2 share
// one complex FFT of d = c1 + i c2, whose DFT is DFT(c1) + i DFT(c2).  Rows
// G/2 .. G-1 are read; rows G/2 - r are their conjugates and row 0 is empty.
// d is formed doubled and the output scale takes the factor 1/2 back.  C
// columns per CTA, C / 2 transforms.  IMG8: the image starts on 8 bytes (its rows
// are of even length), so a thread's two columns leave as one word; the caller's
// image may start on any float.  (Known when compiled: the test at every store
// cost 7 us of the 320 of 1000 channels of 256^2.)
template <int LOG2G, int S, bool IMG8>
__global__ void __launch_bounds__(512, 2)
k_fft_cols(const void* __restrict__ h, const float* __restrict__ hs, int n_img, int cols_per_cta, int ch0,
           const float2* __restrict__ tw_g, const float* __restrict__ inv_corr,
           const uint8_t* __restrict__ mask, const int* __restrict__ kept, float* __restrict__ img) {
  constexpr int G = 1 << LOG2G;
  constexpr int LDP = band_pitch(G);
  extern __shared__ __align__(16) unsigned char smem[];
  const int C = cols_per_cta, CP = C / 2;             // powers of two
  const int cp_shift = __ffs(CP) - 1;
  float2* A = reinterpret_cast<float2*>(smem);        // [C / 2][LDP]: packed column pairs
  float2* tw = A + CP * LDP;
  const int cb = blockIdx.y;
  const int c0 = blockIdx.x * C;
  const long long hrow0 = static_cast<long long>(cb) * half_rows(G);
  for (int i = threadIdx.x; i < tw_entries(G); i += blockDim.x) tw[i] = __ldg(tw_g + i);
  // U items per thread in flight: the reads come from L2 and would otherwise
  // wait one round trip each
  constexpr int U = 8;
  const int n_items = half_rows(G) * CP;
  for (int p = threadIdx.x; p < CP; p += blockDim.x) A[p * LDP] = make_float2(0.0f, 0.0f);   // row 0: empty
  for (int i0 = threadIdx.x; i0 < n_items; i0 += U * blockDim.x) {
    float2 a[U], e[U];                                // c1, c2 at row j = G/2 + r
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < n_items) {
        const int r = i >> cp_shift, p = i & (CP - 1);
        load_h2<S>(h, hs, hrow0 + r, (hrow0 + r) * n_img + c0 + 2 * p, a[u], e[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < n_items) {
        const int r = i >> cp_shift, p = i & (CP - 1);
        const int j = G / 2 + r, jm = G / 2 - r;      // rows j and G - j
        // d = 2 (c1 + i c2); at G - j the columns are conjugated
        A[p * LDP + pad16(j)] = make_float2(2.0f * (a[u].x - e[u].y), 2.0f * (a[u].y + e[u].x));
        if (r > 0) A[p * LDP + pad16(jm)] = make_float2(2.0f * (a[u].x + e[u].y), 2.0f * (e[u].x - a[u].y));
      }
    }
  }
  __syncthreads();
  const long long chan = ch0 + cb;
  const int k = kept[chan];
  const float norm = k > 0 ? 0.5f / static_cast<float>(k) : 0.0f;
  const int off = G / 2 - n_img / 2;
  float* out = img + chan * n_img * n_img + c0;
  // the last pass takes the column pairs in adjacent lanes, so a warp writes
  // whole pieces of image rows; a thread keeps its pair
  const int pair = threadIdx.x & (CP - 1);
  const float2 ic = __ldg(reinterpret_cast<const float2*>(inv_corr + c0) + pair);
  fft_lines<LOG2G>(
      A, LDP, tw, [&](int i, int& f, int& j) {
        f = i / (G / 16);
        j = i % (G / 16);
      },
      [&](int f, int x) { return A[f * LDP + pad16(x)]; },
      [&](int i, int& f, int& j) {
        f = i & (CP - 1);
        j = i >> cp_shift;
      },
      [&](int, int x, float2 z) {
        const int r = x - off;
        if (static_cast<unsigned>(r) >= static_cast<unsigned>(n_img)) return;
        const uchar2 m = *reinterpret_cast<const uchar2*>(mask + r * n_img + c0 + 2 * pair);
        const float ir = __ldg(inv_corr + r);
        float2 v = make_float2(z.x * norm * ir * ic.x, z.y * norm * ir * ic.y);
        // centring sign: (r + col) odd, c0 and the pair's first column even
        if (r & 1) v.x = -v.x;
        else v.y = -v.y;
        if (!m.x) v.x = 0.0f;
        if (!m.y) v.y = 0.0f;
        float* o = out + static_cast<long long>(r) * n_img + 2 * pair;
        if constexpr (IMG8) {
          *reinterpret_cast<float2*>(o) = v;
        } else {
          o[0] = v.x;
          o[1] = v.y;
        }
      });
}

__global__ void k_counts_out(const int* __restrict__ kept, int n_chan, int32_t* __restrict__ out) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f < n_chan) out[f] = 2 * kept[f];
}

// ---------------------------------------------------------- per-call tables and lists
// Everything one geometry and frequency axis needs is made on the device from
// the antenna positions, the frequencies and the kernel table, in five
// launches without a synchronisation.  Made by one host core (7169 N cosines
// for the grid correction, a list push per tile and baseline) it took 13.5, 26
// and 61 ms at 352 antennas and 256^2, 512^2 and 1024^2 images, five to twenty
// times the gridding itself; these kernels take 0.10, 0.11 and 0.17 ms.

// Half of the even kernel table, C(m / Q) for m = 0 .. S Q / 2, passed by
// value: the tables are built from it without a copy through memory.
struct KernelHalf {
  double c[kHalfTab + 1];
};

// The tables: the first n/2 + 1 CTAs form the reciprocal grid correction
// 1 / C^(d), C^(d) = (1/Q) sum_m C(m/Q) cos(2 pi m d / (Q G)), one |d| each
// (the table is even, and so is C^; m = 64 a + b, and 57 + 64 cosines and sines,
// their phases reduced in integers, give all 3585 by the angle sum: a cosine a
// term took 166 us at 1024^2); the others fill the gap-indexed weights, the
// twiddles, the horizon mask and the channel scales, one element a thread.
constexpr int kTabThreads = 256;
constexpr int kCorrB = 64, kCorrA = kHalfTab / kCorrB + 1;
__global__ void __launch_bounds__(kTabThreads)
k_img_tables(const __grid_constant__ KernelHalf kh, int n, int g, double cell, const double* __restrict__ freq,
             int n_chan, float* __restrict__ inv_corr, float* __restrict__ tabx, float2* __restrict__ tw,
             uint8_t* __restrict__ mask, ChanScale* __restrict__ cs) {
  const int n_corr = n / 2 + 1;
  if (static_cast<int>(blockIdx.x) < n_corr) {
    __shared__ double part[kTabThreads / 32];
    __shared__ double2 ca[kCorrA], cb[kCorrB];         // (cos, sin) of the angles of kCorrB a and of b
    const int d = blockIdx.x;
    const int period = kQ * g;                         // a power of two, <= 2^21
    if (threadIdx.x < kCorrA + kCorrB) {
      const int i = threadIdx.x;
      const long long m = i < kCorrA ? static_cast<long long>(kCorrB) * i : i - kCorrA;
      const int r = static_cast<int>((m * d) & (period - 1));
      double si, co;
      sincospi(2.0 * static_cast<double>(r) / static_cast<double>(period), &si, &co);
      (i < kCorrA ? ca[i] : cb[i - kCorrA]) = make_double2(co, si);
    }
    __syncthreads();
    double s = 0.0;
    for (int m = threadIdx.x; m <= kHalfTab; m += kTabThreads) {
      const double2 x = ca[m / kCorrB], y = cb[m % kCorrB];
      const double t = kh.c[m] * (x.x * y.x - x.y * y.y);
      s += m ? 2.0 * t : t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kTabThreads / 32; ++w) s += part[w];
      const float v = static_cast<float>(1.0 / (s / kQ));
      inv_corr[n / 2 - d] = v;                         // pixel offsets -d and d
      if (d < n / 2) inv_corr[n / 2 + d] = v;
    }
    return;
  }
  long long i = static_cast<long long>(blockIdx.x - n_corr) * kTabThreads + threadIdx.x;
  if (i < kTabXLen) {
    const int d = static_cast<int>(i) / kTabStride - kTabD, off = kQ / 2 - static_cast<int>(i) % kTabStride;
    tabx[i] = abs(d) <= kHalfSup ? static_cast<float>(kh.c[abs(d * kQ - off)]) : 0.0f;
    return;
  }
  i -= kTabXLen;
  if (i < tw_all(g)) {
    // exp(-2 pi i r k / len): the second pass's table, the third's, omega_G^k
    const bool powers = i >= tw_entries(g), third = i >= 256;
    const int e = static_cast<int>(third ? i - 256 : i);
    const int rk = powers ? static_cast<int>(i) - tw_entries(g) : third ? (e >> 8) * (e & 255) : (e >> 4) * (e & 15);
    const int len = powers || third ? g : min(g, 256);
    double si, co;
    sincospi(-2.0 * static_cast<double>(rk) / static_cast<double>(len), &si, &co);
    tw[i] = make_float2(static_cast<float>(co), static_cast<float>(si));
    return;
  }
  i -= tw_all(g);
  if (i < static_cast<long long>(n) * n) {
    const int r = static_cast<int>(i) / n, c = static_cast<int>(i) - r * n;
    const double l = static_cast<double>(c - n / 2) * cell;
    const double m = static_cast<double>(r - n / 2) * cell;
    mask[i] = __dadd_rn(__dmul_rn(l, l), __dmul_rn(m, m)) < 1.0 ? 1 : 0;
    return;
  }
  i -= static_cast<long long>(n) * n;
  if (i < n_chan) {
    const double du = 1.0 / (static_cast<double>(g) * cell);
    const double sn = freq[i] / (kCLight * du);
    ChanScale c;
    c.s = sn * static_cast<double>(kQ);                // exact: Q is a power of two
    c.nu_c = freq[i] / kCLight;
    c.sh = static_cast<float>(c.s);
    c.sl = static_cast<float>(c.s - static_cast<double>(c.sh));
    cs[i] = c;
  }
}

// The frequency axis of a call as the lists need it: the extreme scales s_nu Q
// and wavelengths per metre, and the uv range.
struct PlanAxis {
  double s_lo, s_hi;          // cells / Q per metre
  double w_lo, w_hi;          // wavelengths per metre
  double uv_min, uv_max;
  int uv_cut;
  // a baseline of l0 .. l1 wavelengths is outside the uv range in every channel,
  // or inside in every one, with a relative margin
  static constexpr double kEps = 1e-9;
  __host__ __device__ bool uv_outside(double l0, double l1) const {
    return l1 < uv_min * (1.0 - kEps) || l0 >= uv_max * (1.0 + kEps);
  }
  __host__ __device__ bool uv_inside(double l0, double l1) const {
    return l0 >= uv_min * (1.0 + kEps) && l1 < uv_max * (1.0 - kEps);
  }
};

// Centre cells of a cross baseline over the call's channels, and whether the
// uv range must be decided per channel; u0 > u1: never gridded.
struct PlanRange {
  short u0, u1, v0, v1;
  int check;
};

// Centre cell of a rounded position p (1/Q cells): p / Q rounded half away from zero.
__device__ __forceinline__ long long centre_cell64(long long p) {
  const long long c = (llabs(p) + kQ / 2) / kQ;
  return p < 0 ? -c : c;
}

// Per cross baseline (a < b, row-major): its FP64 difference, length, and the
// range of centre cells -- p = rint(dx s) is monotone in s, so every channel's
// centre cells lie between those at the smallest and the largest scale.
// blk[CTA] counts the CTA's baselines that can be gridded in some channel.
constexpr int kPlanThreads = 256;
__global__ void __launch_bounds__(kPlanThreads)
k_plan_baselines(const double* __restrict__ ant, int n_ant, long long n_cross, int cmax, PlanAxis ax,
                 Baseline* __restrict__ base, double* __restrict__ blen, PlanRange* __restrict__ rng,
                 int* __restrict__ blk) {
  const long long i = static_cast<long long>(blockIdx.x) * kPlanThreads + threadIdx.x;
  bool live = false;
  if (i < n_cross) {
    // row a holds the pairs a (2n - a - 1) / 2 .. ; the root is exact to a row
    const double q = 2.0 * n_ant - 1.0;
    int a = static_cast<int>((q - sqrt(q * q - 8.0 * static_cast<double>(i))) * 0.5);
    auto first = [&](long long r) { return r * (2LL * n_ant - r - 1) / 2; };
    while (a > 0 && first(a) > i) --a;
    while (first(a + 1) <= i) ++a;
    const int b = static_cast<int>(i - first(a)) + a + 1;
    Baseline B;
    B.dx = __dsub_rn(ant[3 * a], ant[3 * b]);
    B.dy = __dsub_rn(ant[3 * a + 1], ant[3 * b + 1]);
    B.dxh = static_cast<float>(B.dx);
    B.dxl = static_cast<float>(B.dx - static_cast<double>(B.dxh));
    B.dyh = static_cast<float>(B.dy);
    B.dyl = static_cast<float>(B.dy - static_cast<double>(B.dyh));
    B.bl = bl_index(a, b, n_ant);
    base[i] = B;
    const double L = __dsqrt_rn(__dadd_rn(__dmul_rn(B.dx, B.dx), __dmul_rn(B.dy, B.dy)));
    blen[i] = L;
    auto cells = [&](double d, short& lo, short& hi) {
      const long long x = centre_cell64(__double2ll_rn(__dmul_rn(d, ax.s_lo)));
      const long long y = centre_cell64(__double2ll_rn(__dmul_rn(d, ax.s_hi)));
      const long long l = max(min(x, y), static_cast<long long>(-cmax)), h = min(max(x, y), static_cast<long long>(cmax));
      lo = static_cast<short>(l <= h ? l : 0);
      hi = static_cast<short>(l <= h ? h : -1);
      return l <= h;
    };
    PlanRange r;
    live = cells(B.dx, r.u0, r.u1);
    live = cells(B.dy, r.v0, r.v1) && live;
    r.check = 0;
    if (live && ax.uv_cut) {
      // decided here when every channel of the call agrees (with a relative
      // margin), per channel when the records are prepared otherwise
      const double l0 = __dmul_rn(L, ax.w_lo), l1 = __dmul_rn(L, ax.w_hi);
      if (ax.uv_outside(l0, l1)) live = false;
      r.check = !ax.uv_inside(l0, l1);
    }
    if (!live) {
      r.u0 = 0;
      r.u1 = -1;
    }
    rng[i] = r;
  }
  const int c = __syncthreads_count(live);
  if (threadIdx.x == 0) blk[blockIdx.x] = c;
}

// The listed baselines in cross order (a compaction: each CTA sums the counts
// before its own), their ranges beside them, and how many there are.
__global__ void __launch_bounds__(kPlanThreads)
k_plan_list(int n_ant, long long n_cross, const Baseline* __restrict__ base, const PlanRange* __restrict__ rng,
            const int* __restrict__ blk, GridEntry* __restrict__ listed, PlanRange* __restrict__ lrng,
            unsigned long long* __restrict__ counts) {
  __shared__ int wsum[kPlanThreads / 32];
  __shared__ int wlive[kPlanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int before = 0;
  for (int j = threadIdx.x; j < static_cast<int>(blockIdx.x); j += kPlanThreads) before += blk[j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  const long long i = static_cast<long long>(blockIdx.x) * kPlanThreads + threadIdx.x;
  PlanRange r;
  r.u0 = 0;
  r.u1 = -1;
  if (i < n_cross) r = rng[i];
  const bool live = r.u0 <= r.u1;
  const unsigned m = __ballot_sync(0xffffffffu, live);
  if (lane == 0) {
    wsum[warp] = before;
    wlive[warp] = __popc(m);
  }
  __syncthreads();
  int pos = __popc(m & ((1u << lane) - 1u));
  for (int w = 0; w < kPlanThreads / 32; ++w) pos += wsum[w] + (w < warp ? wlive[w] : 0);
  if (live) {
    const Baseline B = base[i];
    GridEntry e;
    e.bl = static_cast<int>(B.bl);
    e.cross = static_cast<int>(i);
    // the antennas: cross = bl - a - 1, b from a
    const int a = static_cast<int>(B.bl - i) - 1;
    e.a = a;
    e.bf = static_cast<int>(B.bl - bl_index(a, a, n_ant)) + a;
    if (r.check) e.bf |= kCheckUv;
    e.dxh = B.dxh;
    e.dxl = B.dxl;
    e.dyh = B.dyh;
    e.dyl = B.dyl;
    listed[pos] = e;
    lrng[pos] = r;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kPlanThreads - 1)
    counts[kCountListed] = static_cast<unsigned long long>(pos + (live ? 1 : 0));
}

// Tile rows a listed baseline's footprint (centre rows v0 .. v1 over the
// call's channels, 3 cells to each side) touches among the gridded rows
// G/2 .. G-1; the mirror's range is the negated one.
__device__ __forceinline__ bool touches_row(int v0, int v1, int tv) {
  return v1 + kHalfSup >= tv * kTileV && v0 - kHalfSup < (tv + 1) * kTileV;
}

// Per tile row, the records and mirrors that touch it, in listed order (a
// record before its own mirror), each with its range of tile columns.  One CTA
// per row: every warp counts its share of the list, the CTA reserves its range
// of the buffer, every warp writes its share.  (A tile then scans its row's
// few hundred entries, where it would scan tens of thousands of baselines.)
constexpr int kRowWarps = 32;
__global__ void __launch_bounds__(kRowWarps * 32)
k_plan_rows(const PlanRange* __restrict__ lrng, int g, unsigned long long* __restrict__ counts,
            int2* __restrict__ row_ent, long long cap, int2* __restrict__ row_rng) {
  __shared__ int wcnt[kRowWarps];
  __shared__ int start;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tv = blockIdx.x;
  const unsigned lt = (1u << lane) - 1u;
  const int n = static_cast<int>(counts[kCountListed]);
  const int per = ((n + kRowWarps - 1) / kRowWarps + 31) & ~31;
  const int i0 = min(n, warp * per), i1 = min(n, i0 + per);
  auto hits = [&](int i, PlanRange& r, bool& rec, bool& mir) {
    rec = mir = false;
    if (i < i1) {
      r = lrng[i];
      rec = touches_row(r.v0, r.v1, tv);
      mir = touches_row(-r.v1, -r.v0, tv);
    }
  };
  int c = 0;
#pragma unroll 4
  for (int i = i0; i < i1; i += 32) {
    PlanRange r;
    bool rec, mir;
    hits(i + lane, r, rec, mir);
    c += (rec ? 1 : 0) + (mir ? 1 : 0);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) wcnt[warp] = c;
  __syncthreads();
  int off = 0, total = 0;
  for (int w = 0; w < kRowWarps; ++w) {
    off += w < warp ? wcnt[w] : 0;
    total += wcnt[w];
  }
  if (threadIdx.x == 0) {
    // (a plan that does not fit was refused on the host: the test only keeps
    // every store inside the buffer)
    const unsigned long long s = atomicAdd(counts + kCountRows, static_cast<unsigned long long>(total));
    start = s + total <= static_cast<unsigned long long>(cap) ? static_cast<int>(s) : -1;
    row_rng[tv] = start < 0 ? make_int2(0, 0) : make_int2(start, start + total);
  }
  __syncthreads();
  if (start < 0) return;
  off += start;
#pragma unroll 2
  for (int i = i0; i < i1; i += 32) {
    PlanRange r;
    bool rec, mir;
    hits(i + lane, r, rec, mir);
    const unsigned mr = __ballot_sync(0xffffffffu, rec), mm = __ballot_sync(0xffffffffu, mir);
    int pos = off + __popc(mr & lt) + __popc(mm & lt);
    const int half = g / 2;
    if (rec)
      row_ent[pos++] = make_int2(i + lane, ((half + r.u0 - kHalfSup) / kTileU) | (((half + r.u1 + kHalfSup) / kTileU) << 16));
    if (mir)
      row_ent[pos] = make_int2((i + lane) | kMirror,
                               ((half - r.u1 - kHalfSup) / kTileU) | (((half - r.u0 + kHalfSup) / kTileU) << 16));
    off += __popc(mr) + __popc(mm);
  }
}

// Per tile, its list in listed order: one warp per kTilesPerWarp adjacent tiles
// scans their row's entries twice (count, then write to a range reserved by one
// atomic).  Ranges are whole quads, the last one filled with entry 0.  Tiles of
// kHeavy entries and more are listed in heavy, in any order.
constexpr int kTileListWarps = 8, kTilesPerWarp = 8;
static_assert(32 / kTileU % kTilesPerWarp == 0, "a warp's tiles lie in one row of the smallest grid");
__global__ void __launch_bounds__(kTileListWarps * 32)
k_plan_tiles(const int2* __restrict__ row_ent, const int2* __restrict__ row_rng, int ntu, int nt,
             unsigned long long* __restrict__ counts, int* __restrict__ tile_idx, long long cap,
             int2* __restrict__ tile_rng, int* __restrict__ heavy) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int tile0 = (blockIdx.x * kTileListWarps + (threadIdx.x >> 5)) * kTilesPerWarp;
  if (tile0 >= nt) return;
  const int tv = tile0 / ntu, tu0 = tile0 - tv * ntu;
  const int2 rr = row_rng[tv];
  // columns of entry i, relative to the warp's first tile (none: an empty range)
  auto range = [&](int i, int& ent, int& lo, int& hi) {
    int2 e = make_int2(0, 0);
    const bool in = i < rr.y;
    if (in) e = __ldg(row_ent + i);
    ent = e.x;
    lo = (e.y & 0xffff) - tu0;
    hi = in ? (e.y >> 16) - tu0 : -1;
  };
  int c[kTilesPerWarp];
#pragma unroll
  for (int u = 0; u < kTilesPerWarp; ++u) c[u] = 0;
#pragma unroll 2
  for (int i = rr.x; i < rr.y; i += 32) {
    int ent, lo, hi;
    range(i + lane, ent, lo, hi);
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) c[u] += __popc(__ballot_sync(full, u >= lo && u <= hi));
  }
  int start[kTilesPerWarp], slots = 0;
#pragma unroll
  for (int u = 0; u < kTilesPerWarp; ++u) {
    start[u] = slots;
    slots += (c[u] + 3) & ~3;
  }
  int base = 0;
  if (lane == 0 && slots) {
    const unsigned long long s = atomicAdd(counts + kCountSlots, static_cast<unsigned long long>(slots));
    base = s + slots <= static_cast<unsigned long long>(cap) ? static_cast<int>(s) : -1;
  }
  base = __shfl_sync(full, base, 0);
#pragma unroll
  for (int u = 0; u < kTilesPerWarp; ++u) {
    start[u] += base;
    if (lane == u) {
      const int n = base < 0 ? 0 : c[u];
      tile_rng[tile0 + u] = make_int2(start[u], start[u] + n);
      if (n >= kHeavy) heavy[atomicAdd(counts + kCountHeavy, 1ull)] = tile0 + u;
    }
  }
  if (base < 0) return;
#pragma unroll 1
  for (int i = rr.x; i < rr.y; i += 32) {
    int ent, lo, hi;
    range(i + lane, ent, lo, hi);
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) {
      const bool h = u >= lo && u <= hi;
      const unsigned m = __ballot_sync(full, h);
      if (h) tile_idx[start[u] + __popc(m & ((1u << lane) - 1u))] = ent;
      start[u] += __popc(m);
    }
  }
#pragma unroll
  for (int u = 0; u < kTilesPerWarp; ++u)
    if (lane < (4 - (c[u] & 3)) % 4) tile_idx[start[u] + lane] = 0;
}

// ---------------------------------------------------------------- planning
struct ImgPlan {
  int n, g, log2g, batch, cols_per_cta, storage;
  long long n_cross;
};

ImgPlan make_plan(int n_ant, int n_chan, int n, int storage) {
  ImgPlan p;
  p.n = n;
  p.storage = storage;
  p.g = kPad * n;
  p.log2g = ilog2(p.g);
  p.n_cross = static_cast<long long>(n_ant) * (n_ant - 1) / 2;
  // channels per launch: whole groups of 32 (one per lane of a tile warp);
  // the gridded half planes, the prepared records and the half-transformed
  // grids of a batch together up to about 256 MB (the autotuner picks among
  // this and its halves down to 32 channels)
  const long long per = 4LL * p.g * p.g + 4LL * p.g * n + 16LL * std::max<long long>(1, p.n_cross);
  long long b = ((256LL << 20) / per) / kLanes * kLanes;
  if (b < kLanes) b = kLanes;
  if (b > 256) b = 256;
  if (b > n_chan) b = n_chan;
  p.batch = static_cast<int>(b);
  // an even number of columns per CTA (the column pass pairs them)
  int c = 8192 / p.g;
  // at least 8 columns per CTA, so each row segment the column pass reads (4
  // bytes a value in 16-bit storage) and writes is a whole 32-byte sector
  if (c < 8) c = 8;
  if (c > n) c = n;
  p.cols_per_cta = c;
  return p;
}

struct ImgWs {
  float* tabx;       // [kTabXLen] weights by (tap offset, position offset)
  float* inv_corr;
  float2* tw;
  uint8_t* mask;
  double* axis;      // antenna positions [n_ant][3], then frequencies [n_chan]
  Baseline* base;
  ChanScale* cs;
  int* kept;         // [n_chan] kept visibilities, then an item counter per batch (at most n_chan)
  PlanRange* rng;    // [n_cross] centre-cell ranges
  int* blk;          // listed baselines per CTA of k_plan_baselines
  GridEntry* listed; // baselines that can be gridded in some channel of the call
  PlanRange* lrng;   // their ranges
  int2* row_ent;     // per tile row: (listed index | kMirror, first | last << 16 tile column)
  int2* row_rng;     // [tile rows] their ranges in row_ent
  int2* tile_rng;    // [n_tiles] ranges in tile_idx
  int* heavy;        // [n_tiles] tiles of kHeavy entries and more
  int* tile_idx;     // per tile: indices into listed | kMirror
  unsigned long long* counts;   // [kCounts]
  double* blen;      // [n_cross] baseline lengths (metres)
  PrepRec* prep;     // [batch groups][n_cross][32] prepared records (the listed ones first)
  float2* grid;      // [batch groups][G/2][G/4][32][4] gridded half planes
  void* h;           // [batch][G][N] complex in the storage format
  float* hs;         // [batch][G] row scales (FP16 storage)
  bool bases = false;  // records carry weight-table offsets (footprints move < kTabMargin cells)
};

// Tile list entries: each listed baseline once per warp tile its footprint, or
// its mirror's, can touch in the gridded half plane in some channel of the
// call.  Over a coarse channel a footprint moves by at most a cell, so a
// baseline touches 6 to 9 tiles of 4 x 4 (a footprint straddling row G/2 up to
// as many more through its mirror).
constexpr int kEntriesPerBaseline = 24;
long long entry_capacity(const ImgPlan& p) { return std::max<long long>(1, p.n_cross * kEntriesPerBaseline); }
// list slots: the entries, and up to 3 per tile to fill its last quad
long long slot_capacity(const ImgPlan& p) { return entry_capacity(p) + 3LL * n_tiles(p.g); }

ImgWs carve_img(void* ws, size_t bytes, const ImgPlan& p, int n_ant, int n_chan, size_t* need) {
  Carver c(ws, bytes);
  ImgWs w;
  const size_t nx = p.n_cross > 0 ? static_cast<size_t>(p.n_cross) : 1;
  w.tabx = c.take<float>(kTabXLen);
  w.inv_corr = c.take<float>(p.n);
  w.tw = c.take<float2>(tw_all(p.g));
  w.mask = c.take<uint8_t>(static_cast<size_t>(p.n) * p.n);
  w.axis = c.take<double>(static_cast<size_t>(n_ant) * 3 + n_chan);
  w.base = c.take<Baseline>(nx);
  w.cs = c.take<ChanScale>(n_chan);
  w.kept = c.take<int>(2 * static_cast<size_t>(n_chan));
  w.rng = c.take<PlanRange>(nx);
  w.blk = c.take<int>((nx + kPlanThreads - 1) / kPlanThreads);
  w.listed = c.take<GridEntry>(nx);
  w.lrng = c.take<PlanRange>(nx);
  w.row_ent = c.take<int2>(entry_capacity(p));
  w.row_rng = c.take<int2>(half_rows(p.g) / kTileV);
  w.tile_rng = c.take<int2>(n_tiles(p.g));
  w.heavy = c.take<int>(n_tiles(p.g));
  w.tile_idx = c.take<int>(slot_capacity(p));
  w.counts = c.take<unsigned long long>(kCounts);
  w.blen = c.take<double>(nx);
  w.prep = c.take<PrepRec>(static_cast<size_t>((p.batch + kLanes - 1) / kLanes) * nx * kLanes);
  w.grid = c.take<float2>(static_cast<size_t>((p.batch + kLanes - 1) / kLanes) * kLanes * half_rows(p.g) * p.g);
  w.h = c.take<float2>(static_cast<size_t>(p.batch) * half_rows(p.g) * p.n);
  w.hs = c.take<float>(static_cast<size_t>(p.batch) * half_rows(p.g));
  *need = c.used;
  return w;
}

template <int L, int S>
int launch_batch(const ImgPlan& p, const ImgWs& w, const GridOpts& o, const int32_t* vis, long long n_bl, int ch0,
                 int nb, unsigned* next_item, float* img, cudaStream_t st) {
  constexpr int G = 1 << L;
  constexpr int LDP = band_pitch(G);
  {
    // calibration corrections or a uv range select the variant that applies them
    const bool cal = o.gains != nullptr || o.uv_min > 0.0 || std::isfinite(o.uv_max);
    const int n_groups = (nb + kLanes - 1) / kLanes;
    if (p.n_cross > 0) {
      dim3 grid(static_cast<unsigned>((p.n_cross + kPrepBl - 1) / kPrepBl), n_groups);
      OVRO_PROF("k_grid_prep", st);
      auto prep = cal ? (w.bases ? k_grid_prep<L, true, true> : k_grid_prep<L, true, false>)
                      : (w.bases ? k_grid_prep<L, false, true> : k_grid_prep<L, false, false>);
      prep<<<grid, 256, 0, st>>>(w.listed, w.counts, p.n_cross, vis, n_bl, w.base, w.cs, ch0, nb, w.kept, w.prep,
                                o);
      OVRO_LAUNCH_CHECK();
    }
    auto tiles = w.bases ? k_grid_tiles<L, true> : k_grid_tiles<L, false>;
    OVRO_CUDA_TRY(cudaFuncSetAttribute(tiles, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kTileSmem)));
    const long long items = static_cast<long long>(n_groups) * n_tiles(G);
    const long long ctas = std::min<long long>(num_sms(), (items + kGridWarps - 1) / kGridWarps);
    OVRO_PROF("k_grid_tiles", st);
    tiles<<<static_cast<unsigned>(ctas), kGridWarps * 32, kTileSmem, st>>>(
        reinterpret_cast<const int4*>(w.tile_idx), w.tile_rng, w.heavy, w.counts, w.prep, p.n_cross, w.tabx, nb,
        next_item, w.grid);
    OVRO_LAUNCH_CHECK();
  }
  {
    const size_t sm = (static_cast<size_t>(row_lines(G)) * LDP + tw_entries(G)) * sizeof(float2);
    OVRO_CUDA_TRY(cudaFuncSetAttribute(k_fft_rows<L, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm)));
    dim3 grid((nb + row_chans(G) - 1) / row_chans(G), half_rows(G) / row_rows(G));
    OVRO_PROF("k_fft_rows", st);
    k_fft_rows<L, S><<<grid, row_lines(G) * G / 16, sm, st>>>(w.grid, w.tw, nb, p.n, w.h, w.hs);
    OVRO_LAUNCH_CHECK();
  }
  {
    const size_t sm = (static_cast<size_t>(p.cols_per_cta / 2) * LDP + tw_entries(G)) * sizeof(float2);
    auto cols = reinterpret_cast<uintptr_t>(img) % 8 == 0 ? k_fft_cols<L, S, true> : k_fft_cols<L, S, false>;
    OVRO_CUDA_TRY(cudaFuncSetAttribute(cols, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm)));
    const int threads = p.cols_per_cta * G / 32;
    dim3 grid(p.n / p.cols_per_cta, nb);
    OVRO_PROF("k_fft_cols", st);
    cols<<<grid, threads, sm, st>>>(w.h, w.hs, p.n, p.cols_per_cta, ch0, w.tw, w.inv_corr, w.mask, w.kept, img);
    OVRO_LAUNCH_CHECK();
  }
  return OVRO_OK;
}

template <int L>
int launch_storage(const ImgPlan& p, const ImgWs& w, const GridOpts& o, const int32_t* vis, long long n_bl, int ch0,
                   int nb, unsigned* next_item, float* img, cudaStream_t st) {
  switch (p.storage) {
    case kStoreF32: return launch_batch<L, kStoreF32>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case kStoreBF16: return launch_batch<L, kStoreBF16>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case kStoreF16: return launch_batch<L, kStoreF16>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    default: return OVRO_ERR_INVALID_ARG;
  }
}

int run_batch(const ImgPlan& p, const ImgWs& w, const GridOpts& o, const int32_t* vis, long long n_bl, int ch0,
              int nb, unsigned* next_item, float* img, cudaStream_t st) {
  switch (p.log2g) {
    case 5: return launch_storage<5>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case 6: return launch_storage<6>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case 7: return launch_storage<7>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case 8: return launch_storage<8>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case 9: return launch_storage<9>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case 10: return launch_storage<10>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    case 11: return launch_storage<11>(p, w, o, vis, n_bl, ch0, nb, next_item, img, st);
    default: return OVRO_ERR_UNSUPPORTED;
  }
}

// What a call over a wide band needs to know before anything is launched: the
// most cells a listed footprint moves over the channels, and the tile list
// entries there will be.  FP64 as in k_plan_baselines, k_plan_rows and
// k_plan_tiles (host code is built without FMA contraction), so the two agree.
struct PlanExtent {
  int move = 0;
  long long entries = 0;
};

PlanExtent plan_extent(int g, int n_ant, const double* ant, const PlanAxis& ax) {
  PlanExtent out;
  const int half = g / 2, cmax = half - kHalfSup - 1;
  // a baseline that reaches past the grid at the smallest scale is never listed
  const double reach = ax.s_lo > 0.0 ? (cmax + 1.0) * kQ / ax.s_lo : HUGE_VAL;
  // centre cell of a product d s: rint by the addition of 1.5 2^52 (products far off
  // the grid are held at 2^40), then half away from zero
  auto centre = [](double v) {
    constexpr double kRint = 6755399441055744.0, kFar = 1099511627776.0;
    const double p = ((v < kFar ? std::max(v, -kFar) : kFar) + kRint) - kRint;
    return static_cast<int>((p + std::copysign(kQ / 2.0, p)) * (1.0 / kQ));
  };
  // tiles of the rows kept that centre rows v0 .. v1 and columns u0 .. u1 touch
  auto tiles = [&](int v0, int v1, int u0, int u1) -> long long {
    if (v1 + kHalfSup < 0) return 0;
    const unsigned r = static_cast<unsigned>(v1 + kHalfSup) / kTileV - static_cast<unsigned>(std::max(0, v0 - kHalfSup)) / kTileV + 1;
    const unsigned c = static_cast<unsigned>(half + u1 + kHalfSup) / kTileU - static_cast<unsigned>(half + u0 - kHalfSup) / kTileU + 1;
    return r * c;
  };
  std::vector<double> x(n_ant), y(n_ant);
  for (int a = 0; a < n_ant; ++a) {
    x[a] = ant[3 * a];
    y[a] = ant[3 * a + 1];
  }
  for (int a = 0; a < n_ant; ++a)
    for (int b = a + 1; b < n_ant; ++b) {
      const double dx = x[a] - x[b], dy = y[a] - y[b];
      if (!(std::fabs(dx) <= reach && std::fabs(dy) <= reach)) continue;
      const int ua = centre(dx * ax.s_lo), ub = centre(dx * ax.s_hi), va = centre(dy * ax.s_lo), vb = centre(dy * ax.s_hi);
      const int u0 = std::max(std::min(ua, ub), -cmax), u1 = std::min(std::max(ua, ub), cmax);
      const int v0 = std::max(std::min(va, vb), -cmax), v1 = std::min(std::max(va, vb), cmax);
      if (u0 > u1 || v0 > v1) continue;
      if (ax.uv_cut) {
        const double x2 = dx * dx, y2 = dy * dy, len = std::sqrt(x2 + y2);
        if (ax.uv_outside(len * ax.w_lo, len * ax.w_hi)) continue;
      }
      out.move = std::max(out.move, std::max(std::abs(ub - ua), std::abs(vb - va)));
      out.entries += tiles(v0, v1, u0, u1) + tiles(-v1, -v0, -u1, -u0);
    }
  return out;
}

// The call's tables and lists, made on the device without a synchronisation.
// bases: the prepared records may hold weight-table offsets, because no listed
// footprint moves by kTabMargin cells over the call's channels (one cell of
// slack for a rounding of u Q that differs from the exact one) and every frequency
// is a number: with NaN among them the range spans the other channels alone, and the
// offsets of that channel would lie outside the table.  A listed
// |d| s is below (cmax + 1) Q at the smallest scale, so no centre moves by more
// than (cmax + 1) (s_hi / s_lo - 1) + 1 cells; a footprint that moves by at most
// two touches 3 x 3 tiles, its mirror as many: 18 entries, within the capacity
// of 24, and there is nothing more to know.  Over a wider band (60 kHz at 1024^2
// and 60 MHz) the array itself decides, on the host: waiting for the device's
// counts took the call's asynchrony, and the bound alone kept compact arrays from
// the faster records.  352 antennas, 512 channels over 512 kHz at 256^2: the call
// returns after 0.5 ms and is done after 1.7 (with the wait 1.4); the same array
// ten times smaller 6.6 ms (general records 8.4).
int upload_common(const ImgPlan& p, ImgWs& w, int n_ant, const double* h_ant,
                  const double* h_freq, int n_chan, double cell, cudaStream_t st,
                  double uv_min = 0.0, double uv_max = HUGE_VAL) {
  const KernelTables& kt = kernel_tables();
  KernelHalf kh;
  std::copy(kt.table64.begin() + kHalfTab, kt.table64.end(), kh.c);
  std::vector<double> axis(h_ant, h_ant + 3 * static_cast<size_t>(n_ant));
  axis.insert(axis.end(), h_freq, h_freq + n_chan);
  // the scales s_nu Q exactly as the device computes them
  const double du = 1.0 / (static_cast<double>(p.g) * cell);
  PlanAxis ax;
  ax.s_lo = HUGE_VAL;
  ax.s_hi = -HUGE_VAL;
  double fmin = h_freq[0], fmax = h_freq[0];
  bool finite = true;                                  // a channel without a position has no table offset
  for (int f = 0; f < n_chan; ++f) {
    const double sq = (h_freq[f] / (kCLight * du)) * static_cast<double>(kQ);
    finite = finite && std::isfinite(sq);
    ax.s_lo = std::min(ax.s_lo, sq);
    ax.s_hi = std::max(ax.s_hi, sq);
    fmin = std::min(fmin, h_freq[f]);
    fmax = std::max(fmax, h_freq[f]);
  }
  ax.w_lo = fmin / kCLight;
  ax.w_hi = fmax / kCLight;
  ax.uv_min = uv_min;
  ax.uv_max = uv_max;
  ax.uv_cut = uv_min > 0.0 || std::isfinite(uv_max);
  const int cmax = p.g / 2 - kHalfSup - 1;
  double move = ax.s_lo > 0.0 ? (cmax + 1) * (ax.s_hi / ax.s_lo - 1.0) + 1.0 : HUGE_VAL;
  if (!(move <= 2.0)) {
    const PlanExtent e = plan_extent(p.g, n_ant, h_ant, ax);
    if (e.entries > entry_capacity(p)) return OVRO_ERR_CAPACITY;
    move = e.move;
  }
  w.bases = finite && move + 1.0 <= kTabMargin;
  const double* d_ant = w.axis;
  const double* d_freq = w.axis + 3 * static_cast<size_t>(n_ant);
  // a copy from pageable memory is staged before cudaMemcpyAsync returns, so
  // the vector may go out of scope
  OVRO_CUDA_TRY(cudaMemcpyAsync(w.axis, axis.data(), axis.size() * sizeof(double), cudaMemcpyHostToDevice, st));
  OVRO_CUDA_TRY(cudaMemsetAsync(w.counts, 0, kCounts * sizeof(unsigned long long), st));
  const long long elems = kTabXLen + static_cast<long long>(tw_all(p.g)) + static_cast<long long>(p.n) * p.n + n_chan;
  k_img_tables<<<static_cast<unsigned>(p.n / 2 + 1 + (elems + kTabThreads - 1) / kTabThreads), kTabThreads, 0, st>>>(
      kh, p.n, p.g, cell, d_freq, n_chan, w.inv_corr, w.tabx, w.tw, w.mask, w.cs);
  OVRO_LAUNCH_CHECK();
  const int rows = half_rows(p.g) / kTileV, nt = n_tiles(p.g);
  if (p.n_cross > 0) {
    const unsigned blocks = static_cast<unsigned>((p.n_cross + kPlanThreads - 1) / kPlanThreads);
    k_plan_baselines<<<blocks, kPlanThreads, 0, st>>>(d_ant, n_ant, p.n_cross, cmax, ax, w.base, w.blen, w.rng, w.blk);
    OVRO_LAUNCH_CHECK();
    k_plan_list<<<blocks, kPlanThreads, 0, st>>>(n_ant, p.n_cross, w.base, w.rng, w.blk, w.listed, w.lrng, w.counts);
    OVRO_LAUNCH_CHECK();
  }
  k_plan_rows<<<rows, kRowWarps * 32, 0, st>>>(w.lrng, p.g, w.counts, w.row_ent, entry_capacity(p), w.row_rng);
  OVRO_LAUNCH_CHECK();
  constexpr int per_cta = kTileListWarps * kTilesPerWarp;
  k_plan_tiles<<<(nt + per_cta - 1) / per_cta, kTileListWarps * 32, 0, st>>>(
      w.row_ent, w.row_rng, n_tiles_u(p.g), nt, w.counts, w.tile_idx, slot_capacity(p), w.tile_rng, w.heavy);
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

int validate(int n_ant, const double* h_ant, const double* h_freq, int n_chan, int n, double cell) {
  if (!h_ant || !h_freq || n_ant <= 0 || n_chan <= 0) return OVRO_ERR_INVALID_ARG;
  if (!(cell > 0.0)) return OVRO_ERR_INVALID_ARG;
  if (!is_pow2(n) || n < 16 || n > 1024) return OVRO_ERR_UNSUPPORTED;
  if (n_ant > 4096) return OVRO_ERR_UNSUPPORTED;
  return OVRO_OK;
}

}  // namespace

struct GridCtx {
  ImgPlan p;
  ImgWs w;
  int n_ant = 0, n_chan = 0;
  double cell = 0.0;
  const float2* gains = nullptr;      // calibration corrections [n_chan][2 n_ant]
  double uv_min = 0.0, uv_max = HUGE_VAL;
};

size_t grid_ctx_workspace(int n_ant, int n_chan, int image_size, int storage) {
  if (n_ant <= 0 || n_chan <= 0 || !is_pow2(image_size) || image_size < 16 || image_size > 1024) return 0;
  if (storage != OVRO_STORE_FP32 && storage != OVRO_STORE_BF16 && storage != OVRO_STORE_FP16) return 0;
  const ImgPlan p = make_plan(n_ant, n_chan, image_size, storage);
  size_t need = 0;
  carve_img(nullptr, 0, p, n_ant, n_chan, &need);
  return need;
}

int grid_ctx_init(GridCtx** out, int n_ant, int n_chan, int image_size, double cell, int storage, void* d_ws,
                  size_t ws_bytes, const void* d_gains, double uv_min, double uv_max) {
  if (!out) return OVRO_ERR_INVALID_ARG;
  *out = nullptr;
  if (n_ant <= 0 || n_chan <= 0 || !(cell > 0.0)) return OVRO_ERR_INVALID_ARG;
  if (storage != OVRO_STORE_FP32 && storage != OVRO_STORE_BF16 && storage != OVRO_STORE_FP16)
    return OVRO_ERR_INVALID_ARG;
  if (!is_pow2(image_size) || image_size < 16 || image_size > 1024 || n_ant > 4096) return OVRO_ERR_UNSUPPORTED;
  GridCtx* g = new GridCtx;
  g->p = make_plan(n_ant, n_chan, image_size, storage);
  size_t need = 0;
  g->w = carve_img(d_ws, ws_bytes, g->p, n_ant, n_chan, &need);
  if (int e = check_workspace(d_ws, ws_bytes, need)) {
    delete g;
    return e;
  }
  g->n_ant = n_ant;
  g->n_chan = n_chan;
  g->cell = cell;
  g->gains = static_cast<const float2*>(d_gains);
  g->uv_min = uv_min;
  g->uv_max = uv_max;
  *out = g;
  return OVRO_OK;
}

int grid_ctx_upload(GridCtx* g, const double* h_ant_enu_m, const double* h_chan_freq_hz, cudaStream_t st) {
  if (!g) return OVRO_ERR_INVALID_ARG;
  if (int e = validate(g->n_ant, h_ant_enu_m, h_chan_freq_hz, g->n_chan, g->p.n, g->cell)) return e;
  return upload_common(g->p, g->w, g->n_ant, h_ant_enu_m, h_chan_freq_hz, g->n_chan, g->cell, st, g->uv_min,
                       g->uv_max);
}

int grid_ctx_enqueue(GridCtx* g, const int32_t* d_vis, float* d_img, int32_t* d_counts_or_null, cudaStream_t st) {
  if (!g || !d_vis || !d_img) return OVRO_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(d_vis) % 16 != 0) return OVRO_ERR_INVALID_ARG;
  const ImgPlan& p = g->p;
  const long long n_bl = static_cast<long long>(g->n_ant) * (g->n_ant + 1) / 2;
  GridOpts o;
  o.gains = g->gains;
  o.n_input = 2 * g->n_ant;
  o.blen = g->w.blen;
  o.uv_min = g->uv_min;
  o.uv_max = g->uv_max;
  // channels per launch pair (at most the workspace's batch): every choice
  // gives the same images and counts
  auto all = [&](int batch) -> int {
    OVRO_CUDA_TRY(cudaMemsetAsync(g->w.kept, 0, 2 * static_cast<size_t>(g->n_chan) * sizeof(int), st));
    unsigned* next_item = reinterpret_cast<unsigned*>(g->w.kept + g->n_chan);
    for (int ch0 = 0; ch0 < g->n_chan; ch0 += batch) {
      const int nb = g->n_chan - ch0 < batch ? g->n_chan - ch0 : batch;
      if (int e = run_batch(p, g->w, o, d_vis, n_bl, ch0, nb, next_item++, d_img, st)) return e;
    }
    return OVRO_OK;
  };
  const std::string key = tune_key("grid_batch", {g->n_ant, g->n_chan, p.n, p.storage});
  int batch = std::min(p.batch, std::max(1, tuned(key, p.batch)));
  if (tuning(st)) {
    std::vector<int> cands;
    // whole groups of 32 channels (or the call's channels, if fewer)
    for (int b = p.batch; cands.size() < 4; b /= 2) {
      const int c = b >= kLanes ? b / kLanes * kLanes : b;
      if (cands.empty() || c < cands.back()) cands.push_back(c);
      if (c <= kLanes) break;
    }
    if (int e = tune_pick(key, cands, all, st, &batch)) return e;
  }
  if (int e = all(batch)) return e;
  if (d_counts_or_null) {
    k_counts_out<<<(g->n_chan + 255) / 256, 256, 0, st>>>(g->w.kept, g->n_chan, d_counts_or_null);
    OVRO_LAUNCH_CHECK();
  }
  return OVRO_OK;
}

int grid_ctx_gridded(GridCtx* g, long long* total, cudaStream_t st) {
  if (!g || !total) return OVRO_ERR_INVALID_ARG;
  std::vector<int> k(g->n_chan);
  OVRO_CUDA_TRY(cudaMemcpyAsync(k.data(), g->w.kept, g->n_chan * sizeof(int), cudaMemcpyDeviceToHost, st));
  OVRO_CUDA_TRY(cudaStreamSynchronize(st));
  long long s = 0;
  for (int v : k) s += v;
  *total = s;
  return OVRO_OK;
}

void grid_ctx_free(GridCtx* g) { delete g; }

}  // namespace ovro

extern "C" {

size_t ovro_grid_image_workspace_size(int n_ant, int n_chan, int image_size, int storage) {
  return ovro::grid_ctx_workspace(n_ant, n_chan, image_size, storage);
}

int ovro_grid_image(const int32_t* d_vis, int n_ant, const double* h_ant_enu_m,
                    const double* h_chan_freq_hz, int n_chan, int image_size, double cell_dircos,
                    int storage, float* d_img, int32_t* d_n_gridded_or_null, void* d_ws,
                    size_t ws_bytes, void* stream) {
  ovro_grid_options o;
  o.storage = storage;
  o.d_gains_or_null = nullptr;
  o.uv_min_lambda = 0.0;
  o.uv_max_lambda = 0.0;
  return ovro_grid_image_ex(d_vis, n_ant, h_ant_enu_m, h_chan_freq_hz, n_chan, image_size, cell_dircos, &o, d_img,
                            d_n_gridded_or_null, d_ws, ws_bytes, stream);
}

int ovro_grid_image_ex(const int32_t* d_vis, int n_ant, const double* h_ant_enu_m, const double* h_chan_freq_hz,
                       int n_chan, int image_size, double cell_dircos, const ovro_grid_options* opt, float* d_img,
                       int32_t* d_n_gridded_or_null, void* d_ws, size_t ws_bytes, void* stream) {
  using namespace ovro;
  if (!d_vis || !d_img || !opt) return OVRO_ERR_INVALID_ARG;
  if (int e = validate(n_ant, h_ant_enu_m, h_chan_freq_hz, n_chan, image_size, cell_dircos)) return e;
  const int storage = opt->storage;
  if (storage != OVRO_STORE_FP32 && storage != OVRO_STORE_BF16 && storage != OVRO_STORE_FP16)
    return OVRO_ERR_INVALID_ARG;
  if (!(opt->uv_min_lambda >= 0.0) || std::isnan(opt->uv_max_lambda)) return OVRO_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(d_vis) % 16 != 0) return OVRO_ERR_INVALID_ARG;
  if (opt->d_gains_or_null && reinterpret_cast<uintptr_t>(opt->d_gains_or_null) % 8 != 0) return OVRO_ERR_INVALID_ARG;
  const double uv_max = opt->uv_max_lambda > 0.0 ? opt->uv_max_lambda : HUGE_VAL;
  GridCtx* g = nullptr;
  if (int e = grid_ctx_init(&g, n_ant, n_chan, image_size, cell_dircos, storage, d_ws, ws_bytes,
                            opt->d_gains_or_null, opt->uv_min_lambda, uv_max))
    return e;
  cudaStream_t st = as_stream(stream);
  int e = grid_ctx_upload(g, h_ant_enu_m, h_chan_freq_hz, st);
  if (!e) e = grid_ctx_enqueue(g, d_vis, d_img, d_n_gridded_or_null, st);
  grid_ctx_free(g);
  return e;
}

// a5 alone: rounded uv positions p = rint(u Q), Q = 1024, of every cross
// baseline (a < b, row-major) in every channel: int32 [n_chan][n_cross]
// (saturated at +-2^30).  Workspace as for ovro_grid_image.
int ovro_uvw(const double* h_ant_enu_m, int n_ant, const double* h_chan_freq_hz, int n_chan,
             int image_size, double cell_dircos, int32_t* d_pu, int32_t* d_pv, void* d_ws,
             size_t ws_bytes, void* stream) {
  using namespace ovro;
  if (!d_pu || !d_pv) return OVRO_ERR_INVALID_ARG;
  if (int e = validate(n_ant, h_ant_enu_m, h_chan_freq_hz, n_chan, image_size, cell_dircos)) return e;
  const ImgPlan p = make_plan(n_ant, n_chan, image_size, OVRO_STORE_FP32);
  size_t need = 0;
  ImgWs w = carve_img(d_ws, ws_bytes, p, n_ant, n_chan, &need);
  if (int e = check_workspace(d_ws, ws_bytes, need)) return e;
  cudaStream_t st = as_stream(stream);
  if (int e = upload_common(p, w, n_ant, h_ant_enu_m, h_chan_freq_hz, n_chan, cell_dircos, st)) return e;
  if (p.n_cross == 0) return OVRO_OK;
  dim3 g(static_cast<unsigned>((p.n_cross + 255) / 256), n_chan);
  k_uvw<<<g, 256, 0, st>>>(w.base, static_cast<int>(p.n_cross), w.cs, d_pu, d_pv);
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

}  // extern "C"
