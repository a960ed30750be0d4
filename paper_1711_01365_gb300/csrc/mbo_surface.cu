// Closed-surface path of the MBO step (Sec. 5.2 and Algorithm 2 of Osting &
// Wang, arXiv:1711.01365), declared in include/mbo_surface.h.
//
// The diffusion of Algorithm 2 is the double sum
//   A~(x_t) = (h/2pi)^3 Re sum_m e^{-h^2 tau |m|^2} e^{i h m.x_t} sum_q w_q A(x_q^c) e^{-i h m.x_q}
// over m in {-M..M-1}^3.  With theta = h (x - centre) every point lies in
// [-pi/2, pi/2]^3, and the two non-uniform sums are computed on a periodic grid
// of nf points per axis (spacing 2 pi / nf, nf >= 4M) with the "exponential
// of semicircle" kernel phi(z) = exp(beta (sqrt(1 - z^2) - 1)) of width W grid
// points (Barnett, Magland, af Klinteberg, SIAM J. Sci. Comput. 41, 2019):
//   k_spread   type-1 spreading: source q adds w_q A(x_q^c) phi(2 (j - u_q) / W) to
//              the W^3 grid points j around its grid coordinate u_q (phi of a
//              vector: the product of its three coordinates' factors).
//   (3-D FFT diffusion with the per-axis multiplier
//              nf (h / 2 pi) win(k) e^{-k^2 h^2 tau} / psi(k)^2, psi the kernel's
//              Fourier transform: forward FFT, multiplier, inverse FFT; FP32 on
//              the box of the points, mbo_box.cuh, FP64 one call of the torus path)
//   k_interp   type-2 interpolation: target t sums the phi-weighted grid values
//              around its coordinate.
//   k_sproject projection of every target (Lemma 1.1) with the step statistics.
// win(k) = 1 for |k| < M, 1/2 at |k| = M (the real part of the sum over
// -M..M-1), 0 beyond.  The volume-preserving step (Sec. 7, Algorithm 3) runs
// the diffusion into the caller's point order, the flat-torus dE keys and
// class assignment (k_vp_delta / k_vp_assign) on the points, and between them
// a weighted radix selection (k_wselect_*).
//
// Points whose footprints (the W^3 grid points spread to or read from) start
// at the same grid point share their footprint, and the plan sorts them into
// such groups once (the geometry is fixed).  Spreading (k_spread): one warp per
// group of sources, a lane per footprint column (x, y) holding the W points along
// z for CG channels in registers; the group's sources are summed there and added
// once to a shared-memory tile of the group's bin of kBin^3 cells, which goes to
// the grid at the end.  FP32 at width 7 (k_spread7): the groups of a column slide
// along z and what falls out goes straight to the grid.  Interpolation: one block
// per group of targets stages the footprint values in shared memory once and
// evaluates every target of the group from them (k_interp a target per thread,
// k_interp7 two).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <type_traits>
#include <vector>

#include "../../include/mbo_surface.h"
#include "mbo_internal.h"
#include "mbo_kernels.cuh"

#include "mbo_box.cuh"

namespace mbo {
namespace {

constexpr int kBin = 8;         // spreading bin: kBin^3 grid cells
constexpr int kMaxW = 8;        // kernel width limit (register arrays)
constexpr int kMinW = 4;
constexpr int kSpreadThreads = 512;
constexpr int kProjThreads = 256;

template <typename T> struct V4 { T x, y, z, w; };

struct SurfStats {
  unsigned long long maxd_bits;  // max |delta| as double bits (non-negative)
  unsigned long long flips, fallback, nonfinite;
};

template <typename T> __device__ __forceinline__ T es_kernel(T z, T beta) {
  const T a = T(1) - z * z;
  return a > T(0) ? exp(beta * (sqrt(a) - T(1))) : T(0);
}

template <typename T> struct SpreadArgs {
  const T* A;            // surface field, C x nq
  const V4<T>* su;       // sources sorted by (bin, group): d per axis, weight w_q
  const int* sidx;       // source -> field point
  const int* gsrc;       // group -> first source (ngroups + 1)
  const int* gt0;        // group -> footprint start in the bin tile, t0x | t0y << 4 | t0z << 8
  const int* bgrp;       // bin -> first group (nbins + 1)
  // k_spread7: groups over the whole grid instead of per bin
  const int4* g0;        // group -> footprint start on the grid (x, y even; z)
  const int* seg;        // segment -> first group (nseg + 1)
  int nseg;
  const int* bid;        // bin -> bin id (bz nb + by) nb + bx
  T* F;                  // grid box, C channels
  GridBox box;
  long long nq;
  int C, nf, nb, W;
  T beta;
};

// One block per (non-empty bin, group of CG channels); one warp per point
// group.  A group holds the sources of a bin whose footprints start at the
// same z and within a 2 x 2 block in (x, y), so its footprint is
// (W + 1) x (W + 1) x W points (a source's weights vanish outside its own W^3).
// The warp stages chunk_of<T>() sources at a time in shared memory, lane l the
// l-th source (its one-dimensional weights, z first, and strengths w_q A, in
// 16-byte vectors; the per-source stride makes the vector stores of a quarter
// warp hit distinct banks); then lane p of round rd owns footprint column
// (x, y) = (p % (W+1), p / (W+1)), p = lane + 32 rd, sums it over the chunk, W
// points along z for CG channels in registers, and adds it to the bin tile.
// WT: the kernel width as a compile-time constant (the width of eps = 1e-6,
// the paper's choice, has its own instantiation), or 0 for the runtime width.
template <typename T> __host__ __device__ constexpr int chunk_of() { return sizeof(T) == 4 ? 32 : 16; }
// Tile column of x in tile row y.  At width 7 (FP64 only: FP32 has k_spread7) the rows
// are 16 wide, 128 bytes: x ^ 8 on rows with bit 1 of y set spreads the 4 rows x 8
// columns that a flush writes over the banks.
template <int WT> __device__ __forceinline__ int swz(int x, int y) {
  if constexpr (WT == 7) return x ^ (((y >> 1) & 1) << 3);
  return x;
}
// Add a block's tile ([c][z][y][x]) to the grid box.
template <typename T, int WT>
__device__ __forceinline__ void spread_flush(const SpreadArgs<T>& a, const T* tile, int c0, int cg, int W,
                                             int TX, int TZ, int threads) {
  const int b = a.bid[blockIdx.x];
  const int bx = b % a.nb, by = (b / a.nb) % a.nb, bz = b / (a.nb * a.nb);
  const int nf = a.nf;
  const long long P = a.box.points();
  const int lx = (bx * kBin - W / 2 + nf) % nf, ly = (by * kBin - W / 2 + nf) % nf,
            lz = (bz * kBin - W / 2 + nf) % nf;
  const int TV = TX * TX * TZ;
  // sixteen lanes per tile row (TX is at most 17)
  const int half = threadIdx.x & 15;
  for (int row = threadIdx.x >> 4; row < cg * TZ * TX; row += threads / 16) {
    const int c = row / (TZ * TX), zy = row - c * TZ * TX, z = zy / TX, y = zy - z * TX;
    int gy = ly + y, gz = lz + z;
    gy -= gy >= nf ? nf : 0;
    gz -= gz >= nf ? nf : 0;
    gy -= a.box.b0[1];
    gz -= a.box.b0[2];
    // tile rows outside the box hold zeros
    if ((unsigned)gy >= (unsigned)a.box.bn[1] || (unsigned)gz >= (unsigned)a.box.bn[2]) continue;
    T* Frow = a.F + (long long)(c0 + c) * P + ((long long)gz * a.box.bn[1] + gy) * a.box.bn[0];
    const T* trow = tile + c * TV + zy * TX;
    for (int x = half; x < TX; x += 16) {
      const T v = trow[swz<WT>(x, y)];
      if (v == T(0)) continue;
      int gx = lx + x;
      gx -= gx >= nf ? nf : 0;
      gx -= a.box.b0[0];
      if ((unsigned)gx < (unsigned)a.box.bn[0]) atomicAdd(&Frow[gx], v);
    }
  }
}

constexpr int kWS = 9;     // weight slots of x and of y per source (>= W + 1)
constexpr int kWSrc = 28;  // per source: z[8] | x[kWS] | y[kWS] | 2 pad, then strengths
template <typename T> __host__ __device__ constexpr int src_stride() { return sizeof(T) == 4 ? 44 : 34; }
template <typename T, int CG, int WT>
__global__ void __launch_bounds__(kSpreadThreads) k_spread(SpreadArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int CH = chunk_of<T>(), SRC = src_stride<T>();
  constexpr int VW = 16 / sizeof(T);  // elements per 16-byte vector
  constexpr int CGP = (CG + VW - 1) / VW * VW;
  static_assert(kWSrc + CGP <= SRC, "strengths must fit the source stride");
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  const int W = WT ? WT : a.W, FW = W + 1, TX = kBin + FW, TZ = kBin + W, TV = TX * TX * TZ;
  T* tile = reinterpret_cast<T*>(smem_raw);  // [c][z][y][x], TX x TX x TZ
  const int c0 = blockIdx.y * CG;
  const int cg = min(CG, a.C - c0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T* stg = tile + ((CG * TV + VW - 1) / VW) * VW + warp * CH * SRC;  // 16-byte aligned
  for (int i = tid; i < CG * TV; i += kSpreadThreads) tile[i] = T(0);
  __syncthreads();

  const int F2 = FW * FW;
  const T sc2 = T(2) / T(W);
  const int g0 = a.bgrp[blockIdx.x], g1 = a.bgrp[blockIdx.x + 1];
  for (int g = g0 + warp; g < g1; g += kSpreadThreads / 32) {
    const int pk = a.gt0[g];
    const int tx = pk & 15, ty = (pk >> 4) & 15, tz = (pk >> 8) & 15;
    const int s0 = a.gsrc[g], s1 = a.gsrc[g + 1];
    for (int cs = s0; cs < s1; cs += CH) {
      const int ns = min(CH, s1 - cs);
      __syncwarp();
      if (lane < ns) {
        const V4<T> u = a.su[cs + lane];  // distance past the group footprint start
        const long long src = a.sidx[cs + lane];
        T r[SRC];
#pragma unroll
        for (int k = 0; k < 8; ++k) r[k] = (k < W) ? es_kernel((T(k) - u.z) * sc2, a.beta) : T(0);
#pragma unroll
        for (int i = 0; i < kWS; ++i) {
          r[8 + i] = (i < FW) ? es_kernel((T(i) - u.x) * sc2, a.beta) : T(0);
          r[8 + kWS + i] = (i < FW) ? es_kernel((T(i) - u.y) * sc2, a.beta) : T(0);
        }
#pragma unroll
        for (int e = 8 + 2 * kWS; e < kWSrc; ++e) r[e] = T(0);
#pragma unroll
        for (int c = 0; c < SRC - kWSrc; ++c)
          r[kWSrc + c] = (c < cg) ? a.A[(long long)(c0 + c) * a.nq + src] * u.w : T(0);
        V* dst = reinterpret_cast<V*>(stg + lane * SRC);
#pragma unroll
        for (int v = 0; v < SRC / VW; ++v) {
          if constexpr (VW == 4) dst[v] = make_float4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
          else dst[v] = make_double2(r[2 * v], r[2 * v + 1]);
        }
      }
      __syncwarp();
      for (int rd = 0; rd * 32 < F2; ++rd) {
        const int p = lane + 32 * rd;
        const bool ok = p < F2;
        const int j = ok ? p / FW : 0, i = ok ? p - j * FW : 0;
        T acc[kMaxW][CG];
#pragma unroll
        for (int k = 0; k < kMaxW; ++k)
#pragma unroll
          for (int c = 0; c < CG; ++c) acc[k][c] = T(0);
        for (int q = 0; q < ns; ++q) {
          const T* wq = stg + q * SRC;
          const T wxy = wq[8 + i] * wq[8 + kWS + j];
          T wz[8], str[CGP];
#pragma unroll
          for (int v = 0; v < 8 / VW; ++v) {
            const V x = reinterpret_cast<const V*>(wq)[v];
            if constexpr (VW == 4) { wz[4 * v] = x.x; wz[4 * v + 1] = x.y; wz[4 * v + 2] = x.z; wz[4 * v + 3] = x.w; }
            else { wz[2 * v] = x.x; wz[2 * v + 1] = x.y; }
          }
#pragma unroll
          for (int v = 0; v < CGP / VW; ++v) {
            const V x = reinterpret_cast<const V*>(wq + kWSrc)[v];
            if constexpr (VW == 4) { str[4 * v] = x.x; str[4 * v + 1] = x.y; str[4 * v + 2] = x.z; str[4 * v + 3] = x.w; }
            else { str[2 * v] = x.x; str[2 * v + 1] = x.y; }
          }
#pragma unroll
          for (int k = 0; k < kMaxW; ++k) {
            if (k < W) {
              const T w = wz[k] * wxy;
#pragma unroll
              for (int c = 0; c < CG; ++c) acc[k][c] += w * str[c];
            }
          }
        }
        if (ok) {
          int addr = (tz * TX + ty + j) * TX + swz<WT>(tx + i, ty + j);
#pragma unroll
          for (int k = 0; k < kMaxW; ++k) {
            if (k < W) {
#pragma unroll
              for (int c = 0; c < CG; ++c)  // channels past cg add their zeros
                atomicAdd(&tile[c * TV + addr], acc[k][c]);
            }
            addr += TX * TX;
          }
        }
      }
    }
  }
  __syncthreads();

  spread_flush<T, WT>(a, tile, c0, cg, W, TX, TZ, kSpreadThreads);
}

// FP32, width 7 (eps = 1e-6, the paper's choice).  The work is the rank-one
// update of a group's 64 footprint columns by 7 x CG values per source: FMA
// work, so the kernel is laid out to keep the FMA pipe the limit.
//   - Groups hold about 18 sources on the paper's sphere, so adding a group's
//     7 x 8 x 8 x CG sums anywhere costs more than making them.  A warp takes a
//     segment of a column of groups (one footprint start in x and y over the
//     whole grid, z ascending, up to kSegSources sources) and slides its seven
//     accumulator planes along z: only the plane that falls out leaves, straight
//     to the grid box by reductions in L2 (eight neighbours along x share a
//     sector), with no tile in shared memory and no block to wait for.
//   - Two warps share a segment, one for each half of the 64 columns, and stage
//     64 sources together: 16 warps per SM at 128 registers (one warp with both
//     halves in its registers, 8 per SM, waited on instruction latency: 1.09 ms).
//   - Packed two-lane multiply-adds over channel pairs: the z weights are stored
//     twice so that a 16-byte load brings two packed operands; (w_x w_y) scales
//     the strengths once per column.  54 instructions per source and half instead
//     of 84.  The next source's operands are loaded while this one is summed.
// Unit sphere of the paper (3.3M points, n = 3): 1.71 ms with a group per warp and a
// shared-memory tile per bin, 0.84 ms (segments of 512 sources 0.86, 1024 0.94).
constexpr int kSpread7Threads = 64;
constexpr int kSegSources = 256;
template <int CG> struct Spread7 {
  static constexpr int NP = (CG + 1) / 2;                 // channel pairs
  static constexpr int SP = (2 * NP + 3) / 4 * 4;         // strengths, padded to vectors
  static constexpr int OX = 16 + SP, OY = OX + 8;         // z (twice, 14 + 2) | strengths | x | y
  static constexpr int SRC = (OY + 8) / 4 % 2 ? OY + 8 : OY + 12;  // odd number of vectors: no bank conflicts
};
// Coordinate of the box from a footprint coordinate in [-W, nf + W).
__device__ __forceinline__ int box_coord(int g, int nf, int b0) {
  g += g < 0 ? nf : 0;
  g -= g >= nf ? nf : 0;
  return g - b0;
}
template <int CG>
__global__ void __launch_bounds__(kSpread7Threads, 8) k_spread7(SpreadArgs<float> a) {
  using S = Spread7<CG>;
  constexpr int NP = S::NP;
  __shared__ __align__(16) float stg[kSpread7Threads * S::SRC];
  const int c0 = blockIdx.y * CG;
  const int cg = min(CG, a.C - c0);
  const int tid = threadIdx.x;
  const int i = tid & 7, j = tid >> 3;  // footprint column
  int g = a.seg[blockIdx.x];
  const int ge = a.seg[blockIdx.x + 1];
  const int4 start = a.g0[g];
  int tz = start.z;
  const long long P = a.box.points(), plane = (long long)a.box.bn[0] * a.box.bn[1];
  const int gx = box_coord(start.x + i, a.nf, a.box.b0[0]);
  float* F = a.F + c0 * P + (long long)box_coord(start.y + j, a.nf, a.box.b0[1]) * a.box.bn[0] + gx;
  float2 acc[7][NP];
#pragma unroll
  for (int k = 0; k < 7; ++k)
#pragma unroll
    for (int c = 0; c < NP; ++c) acc[k][c] = make_float2(0.f, 0.f);
  // the lowest plane to the grid, the others down by one
  auto slide = [&]() {
    const long long at = box_coord(tz, a.nf, a.box.b0[2]) * plane;
#pragma unroll
    for (int c = 0; c < CG; ++c) {
      if (c < cg) atomicAdd(F + c * P + at, c % 2 ? acc[0][c / 2].y : acc[0][c / 2].x);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k)
#pragma unroll
      for (int c = 0; c < NP; ++c) acc[k][c] = acc[k + 1][c];
#pragma unroll
    for (int c = 0; c < NP; ++c) acc[6][c] = make_float2(0.f, 0.f);
    ++tz;
  };
  const int s1 = a.gsrc[ge];
  int gend = a.gsrc[g + 1];  // the end of the group in work
  for (int cs = a.gsrc[g]; cs < s1; cs += kSpread7Threads) {
    const int ns = min(kSpread7Threads, s1 - cs);
    __syncthreads();
    if (tid < ns) {
      const V4<float> u = a.su[cs + tid];  // distance past the group footprint start
      const long long src = a.sidx[cs + tid];
      float st[S::SP];
#pragma unroll
      for (int c = 0; c < S::SP; ++c) st[c] = c < CG && c < cg ? a.A[(long long)(c0 + c) * a.nq + src] * u.w : 0.f;
      float4* dst = reinterpret_cast<float4*>(stg + tid * S::SRC);
      constexpr float sc2 = 2.f / 7.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float za = es_kernel((float(2 * k) - u.z) * sc2, a.beta);
        const float zb = 2 * k + 1 < 7 ? es_kernel((float(2 * k + 1) - u.z) * sc2, a.beta) : 0.f;
        dst[k] = make_float4(za, za, zb, zb);
      }
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        float x[4], y[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          x[e] = es_kernel((float(4 * v + e) - u.x) * sc2, a.beta);
          y[e] = es_kernel((float(4 * v + e) - u.y) * sc2, a.beta);
        }
        dst[S::OX / 4 + v] = make_float4(x[0], x[1], x[2], x[3]);
        dst[S::OY / 4 + v] = make_float4(y[0], y[1], y[2], y[3]);
      }
#pragma unroll
      for (int v = 0; v < S::SP / 4; ++v) dst[4 + v] = make_float4(st[4 * v], st[4 * v + 1], st[4 * v + 2], st[4 * v + 3]);
    }
    __syncthreads();
    float4 z[4], sv[S::SP / 4];
    float wx, wy;
    auto fetch = [&](int q) {
      const float4* r = reinterpret_cast<const float4*>(stg + q * S::SRC);
#pragma unroll
      for (int v = 0; v < 4; ++v) z[v] = r[v];
#pragma unroll
      for (int v = 0; v < S::SP / 4; ++v) sv[v] = r[4 + v];
      const float* w = stg + q * S::SRC;
      wx = w[S::OX + i];
      wy = w[S::OY + j];
    };
    fetch(0);
    int q = 0;
    while (q < ns) {
      if (cs + q == gend) {  // the next group of the column, some planes up
        ++g;
        gend = a.gsrc[g + 1];
        const int up = a.g0[g].z;
#pragma unroll 1
        while (tz < up) slide();
      }
      const int qe = min(ns, gend - cs);
      for (; q < qe; ++q) {
        const float2 zz[7] = {{z[0].x, z[0].y}, {z[0].z, z[0].w}, {z[1].x, z[1].y}, {z[1].z, z[1].w},
                              {z[2].x, z[2].y}, {z[2].z, z[2].w}, {z[3].x, z[3].y}};
        const float w = wx * wy;
        float2 pc[NP];
#pragma unroll
        for (int c = 0; c < NP; ++c) {
          const float4 v = sv[c / 2];
          const float2 t = c % 2 ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
          pc[c] = __fmul2_rn(t, make_float2(w, w));
        }
        if (q + 1 < ns) fetch(q + 1);
#pragma unroll
        for (int k = 0; k < 7; ++k)
#pragma unroll
          for (int c = 0; c < NP; ++c) acc[k][c] = __ffma2_rn(zz[k], pc[c], acc[k][c]);
      }
    }
  }
#pragma unroll 1
  for (int k = 0; k < 7; ++k) slide();
}

template <typename T> struct InterpArgs {
  const T* F;          // grid box, C channels
  GridBox box;
  const V4<T>* tu;     // targets sorted by group: d per axis
  const int* tidx;     // target -> field point
  const int* tgrp;     // group -> first target (ngroups + 1)
  const int4* tg0;     // group -> first footprint point on the grid (gx, gy, gz)
  T* dst;              // C x nq, the caller's order: the passes that follow stream it
  long long nq;
  int nf, W;
  T beta;
};

// Offset of a grid point of the box.
__device__ __forceinline__ long long box_at(const GridBox& b, int gx, int gy, int gz) {
  return ((long long)(gz - b.b0[2]) * b.bn[1] + (gy - b.b0[1])) * b.bn[0] + (gx - b.b0[0]);
}

// One block per target group: the group's W^3 footprint values (C channels
// padded to CP, point-major) are staged in shared memory once; each thread
// evaluates one target from them (all lanes of a warp read the same values:
// broadcast), with its 3W one-dimensional weights in registers.
constexpr int kInterpBlock = 128;
template <typename T, int C> __host__ __device__ constexpr int padded_channels() {
  return C == 1 ? 1 : (sizeof(T) == 4 ? (C + 3) / 4 * 4 : (C + 1) / 2 * 2);
}
template <typename T, int NM, int WT>
__global__ void __launch_bounds__(kInterpBlock) k_interp(InterpArgs<T> a) {
  constexpr int C = NM * NM, CP = padded_channels<T, C>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* fp = reinterpret_cast<T*>(smem_raw);  // [W^3][CP]
  const int W = WT ? WT : a.W, W2 = W * W, W3 = W2 * W, nf = a.nf;
  const long long P = a.box.points();
  const int g = blockIdx.x;
  const int4 g0 = a.tg0[g];
  for (int e = threadIdx.x; e < CP * W3; e += kInterpBlock) {
    const int c = e / W3, p = e - c * W3;
    T v = T(0);
    if (c < C) {
      const int k = p / W2, r = p - k * W2, j = r / W, i = r - j * W;
      int gx = g0.x + i, gy = g0.y + j, gz = g0.z + k;
      gx -= gx >= nf ? nf : 0;
      gy -= gy >= nf ? nf : 0;
      gz -= gz >= nf ? nf : 0;
      v = __ldg(&a.F[c * P + box_at(a.box, gx, gy, gz)]);
    }
    fp[p * CP + c] = v;
  }
  __syncthreads();
  const int t1 = a.tgrp[g + 1];
  const T sc2 = T(2) / T(W);
  for (int t = a.tgrp[g] + threadIdx.x; t < t1; t += kInterpBlock) {
    const V4<T> u = a.tu[t];
    T wx[kMaxW], wy[kMaxW];
#pragma unroll
    for (int i = 0; i < kMaxW; ++i) {
      wx[i] = (i < W) ? es_kernel((T(i) - u.x) * sc2, a.beta) : T(0);
      wy[i] = (i < W) ? es_kernel((T(i) - u.y) * sc2, a.beta) : T(0);
    }
    T acc[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = T(0);
    for (int k = 0; k < W; ++k) {
      const T wz = es_kernel((T(k) - u.z) * sc2, a.beta);
      const T* plane = fp + k * W2 * CP;
#pragma unroll
      for (int j = 0; j < kMaxW; ++j) {
        if (j < W) {
          const T wyz = wz * wy[j];
#pragma unroll
          for (int i = 0; i < kMaxW; ++i) {
            if (i < W) {
              const T w = wyz * wx[i];
              const T* pt = plane + (j * W + i) * CP;
              if constexpr (CP % 4 == 0 && sizeof(T) == 4) {
#pragma unroll
                for (int v = 0; v < CP / 4; ++v) {
                  const float4 x = reinterpret_cast<const float4*>(pt)[v];
                  acc[4 * v] += w * x.x;
                  acc[4 * v + 1] += w * x.y;
                  acc[4 * v + 2] += w * x.z;
                  acc[4 * v + 3] += w * x.w;
                }
              } else if constexpr (CP % 2 == 0 && sizeof(T) == 8) {
#pragma unroll
                for (int v = 0; v < CP / 2; ++v) {
                  const double2 x = reinterpret_cast<const double2*>(pt)[v];
                  acc[2 * v] += w * x.x;
                  acc[2 * v + 1] += w * x.y;
                }
              } else {
#pragma unroll
                for (int c = 0; c < CP; ++c) acc[c] += w * pt[c];
              }
            }
          }
        }
      }
    }
    const long long q = a.tidx[t];
#pragma unroll
    for (int c = 0; c < C; ++c) a.dst[c * a.nq + q] = acc[c];
  }
}

// FP32, width 7, n = 2 and 3: a lane evaluates two targets at once, so a
// footprint point (broadcast from shared memory, whose bandwidth bounds this
// kernel: a 16-byte broadcast moves 512 bytes to the warp) serves both; channels
// in pairs, by packed multiply-adds.  A warp takes 64 targets of its group at a
// time, or 32 where no more are left.  Unit sphere of the paper: one target per lane
// 0.79 ms, two 0.645 ms.
template <int NM> struct Interp7 {
  static constexpr int C = NM * NM, NP = (C + 1) / 2, ST = (2 * NP + 3) / 4 * 4;  // floats per point
};
template <int NM, int NT>
__device__ __forceinline__ void interp7_targets(const InterpArgs<float>& a, const float* fp, int t, int t1) {
  using S = Interp7<NM>;
  constexpr float sc2 = 2.f / 7.f;
  float2 wx[NT][7], acc[NT][S::NP];
  float wy[NT][7], uz[NT];
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const V4<float> u = a.tu[min(t + 32 * n, t1 - 1)];
    uz[n] = u.z;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      const float w = es_kernel((float(i) - u.x) * sc2, a.beta);
      wx[n][i] = make_float2(w, w);
      wy[n][i] = es_kernel((float(i) - u.y) * sc2, a.beta);
    }
#pragma unroll
    for (int c = 0; c < S::NP; ++c) acc[n][c] = make_float2(0.f, 0.f);
  }
#pragma unroll 1
  for (int k = 0; k < 7; ++k) {
    const float* plane = fp + k * 49 * S::ST;
    float wz[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) wz[n] = es_kernel((float(k) - uz[n]) * sc2, a.beta);
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      float2 row[NT][S::NP];  // sum over x of this footprint row
#pragma unroll
      for (int i = 0; i < 7; ++i) {
        float2 v[(S::NP + 1) / 2 * 2];
#pragma unroll
        for (int c = 0; c < S::NP / 2; ++c) {
          const float4 x = reinterpret_cast<const float4*>(plane + (j * 7 + i) * S::ST)[c];
          v[2 * c] = make_float2(x.x, x.y);
          v[2 * c + 1] = make_float2(x.z, x.w);
        }
        if constexpr (S::NP % 2) v[S::NP - 1] = reinterpret_cast<const float2*>(plane + (j * 7 + i) * S::ST)[S::NP - 1];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
#pragma unroll
          for (int c = 0; c < S::NP; ++c)
            row[n][c] = i ? __ffma2_rn(wx[n][i], v[c], row[n][c]) : __fmul2_rn(wx[n][0], v[c]);
        }
      }
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const float w = wz[n] * wy[n][j];
#pragma unroll
        for (int c = 0; c < S::NP; ++c) acc[n][c] = __ffma2_rn(make_float2(w, w), row[n][c], acc[n][c]);
      }
    }
  }
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    if (t + 32 * n >= t1) continue;
    const long long q = a.tidx[t + 32 * n];
#pragma unroll
    for (int c = 0; c < S::C; ++c) a.dst[c * a.nq + q] = c % 2 ? acc[n][c / 2].y : acc[n][c / 2].x;
  }
}
template <int NM>
__global__ void __launch_bounds__(kInterpBlock) k_interp7(InterpArgs<float> a) {
  using S = Interp7<NM>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* fp = reinterpret_cast<float*>(smem_raw);  // [343][ST]
  const int g = blockIdx.x, nf = a.nf;
  const long long P = a.box.points();
  const int4 g0 = a.tg0[g];
  for (int p = threadIdx.x; p < 343; p += kInterpBlock) {
    const int k = p / 49, r = p - k * 49, j = r / 7, i = r - j * 7;
    int gx = g0.x + i, gy = g0.y + j, gz = g0.z + k;
    gx -= gx >= nf ? nf : 0;
    gy -= gy >= nf ? nf : 0;
    gz -= gz >= nf ? nf : 0;
    const float* src = a.F + box_at(a.box, gx, gy, gz);
    float v[S::ST];
#pragma unroll
    for (int c = 0; c < S::ST; ++c) v[c] = c < S::C ? __ldg(src + c * P) : 0.f;
#pragma unroll
    for (int c = 0; c < S::ST / 4; ++c)
      reinterpret_cast<float4*>(fp + p * S::ST)[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
  }
  __syncthreads();
  const int t1 = a.tgrp[g + 1], lane = threadIdx.x & 31;
  for (int t = a.tgrp[g] + (threadIdx.x >> 5) * 64; t < t1; t += kInterpBlock / 32 * 64) {
    if (t + 32 < t1) interp7_targets<NM, 2>(a, fp, t + lane, t1);
    else interp7_targets<NM, 1>(a, fp, t + lane, t1);
  }
}

template <typename T> struct ProjArgs {
  const T* At;        // C x nq diffused values
  T* A;               // field, C x nq (read: previous; written: projected)
  SurfStats* st;
  long long nq;
  T fb;
};

// Add a block's statistics to the step's: integer warp reductions (the bits of
// non-negative doubles order like them; a butterfly of FP64 maxima in every warp
// took a quarter of the projection), and a maximum that does not raise the
// recorded one is not sent.
template <typename T> __device__ __forceinline__ void surf_stats(const PointStats<T>& ps, SurfStats* st) {
  __shared__ unsigned long long s_mx[kProjThreads / 32];
  unsigned long long mx;
  if constexpr (sizeof(T) == 4) {
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(ps.maxd));
    mx = (unsigned long long)__double_as_longlong((double)__uint_as_float(m));
  } else {
    mx = warp_max_u64((unsigned long long)__double_as_longlong(ps.maxd));
  }
  const bool lead = (threadIdx.x & 31) == 0;
  if (__any_sync(0xffffffffu, ps.flips | ps.nonfinite | ps.fallback)) {
    const unsigned fl = __reduce_add_sync(0xffffffffu, (unsigned)ps.flips);
    const unsigned nf = __reduce_add_sync(0xffffffffu, (unsigned)ps.nonfinite);
    const unsigned fb = __reduce_add_sync(0xffffffffu, (unsigned)ps.fallback);
    if (lead && fl) atomicAdd(&st->flips, (unsigned long long)fl);
    if (lead && nf) atomicAdd(&st->nonfinite, (unsigned long long)nf);
    if (lead && fb) atomicAdd(&st->fallback, (unsigned long long)fb);
  }
  if (lead) s_mx[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kProjThreads / 32; ++w) mx = s_mx[w] > mx ? s_mx[w] : mx;
    if (mx > *reinterpret_cast<volatile unsigned long long*>(&st->maxd_bits)) atomicMax(&st->maxd_bits, mx);
  }
}

// Projection of every target (Lemma 1.1) and the step statistics.
template <typename T, int NM>
__global__ void __launch_bounds__(kProjThreads) k_sproject(ProjArgs<T> a) {
  constexpr int C = NM * NM;
  const long long t = (long long)blockIdx.x * kProjThreads + threadIdx.x;
  PointStats<T> ps;
  if (t < a.nq) {
    T m[C], old[C], bb[C], sg;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      m[c] = a.At[c * a.nq + t];
      old[c] = a.A[c * a.nq + t];
    }
    bool fin = true;
#pragma unroll
    for (int c = 0; c < C; ++c) fin = fin && isfinite(m[c]);
    ps.nonfinite += fin ? 0 : 1;
    if (!project_point<NM>(m, bb, sg, a.fb)) {
      sg = project_point_f64<NM>(m, bb);
      ps.fallback += 1;
    }
    T d = T(0);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      d = fmax(d, fabs(bb[c] - old[c]));
      a.A[c * a.nq + t] = bb[c];
    }
    ps.maxd = d;
    ps.flips = (det_sign<NM>(old) != sg) ? 1 : 0;
  }
  surf_stats(ps, a.st);
}

// Step statistics of the volume-preserving step: compare the previous field
// with the assigned one, point by point (both in the caller's order).
template <typename T, int NM>
__global__ void __launch_bounds__(kProjThreads) k_sdelta(const T* old, const T* A, long long nq, SurfStats* st) {
  constexpr int C = NM * NM;
  const long long q = (long long)blockIdx.x * kProjThreads + threadIdx.x;
  PointStats<T> ps;
  if (q < nq) {
    T o[C], b[C];
    bool fin = true;
    T d = T(0);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      o[c] = old[c * nq + q];
      b[c] = A[c * nq + q];
      fin = fin && isfinite(b[c]);
      d = fmax(d, fabs(b[c] - o[c]));
    }
    ps.maxd = d;
    ps.nonfinite = fin ? 0 : 1;
    ps.flips = (det_sign<NM>(o) != det_sign<NM>(b)) ? 1 : 0;
  }
  surf_stats(ps, st);
}

// Weighted selection of Algorithm 3 (Sec. 7 on surfaces): with points ordered
// by decreasing dE (ascending key, lower index first on equal keys), the
// smallest prefix whose weight reaches the target volume V.  Weights are
// fixed-point integers (the plan scales every w_q so that all of them sum to
// 2^62), so the sums are exact and independent of the summation order.  Twelve
// MSB-first passes over 8-bit digits of the 96-bit (key, index) composite, as
// in the count-based selection, with weight sums per digit instead of counts;
// the result goes into a SelectState for the class assignment (a point takes
// SO(n) iff its (key, index) <= (hi, lo) and the target is positive).
struct WSelect {
  unsigned long long hi;      // key part of the prefix / result
  unsigned int lo;            // index part
  int all;                    // the target exceeds the total weight: select every point
  unsigned long long vrem;    // weight still to reach inside the current prefix
  unsigned long long target;  // V
  unsigned long long hist[256];
};

__device__ __forceinline__ unsigned wdigit(unsigned long long key, unsigned idx, int d) {
  return d < 8 ? (unsigned)((key >> (56 - 8 * d)) & 0xffu) : ((idx >> (24 - 8 * (d - 8))) & 0xffu);
}

__device__ __forceinline__ bool wprefix(unsigned long long key, unsigned idx, unsigned long long hi,
                                        unsigned lo, int d) {
  if (d == 0) return true;
  if (d <= 8) {
    const int sh = 64 - 8 * d;
    return (key >> sh) == (hi >> sh);
  }
  if (key != hi) return false;
  const int sh = 32 - 8 * (d - 8);
  return (idx >> sh) == (lo >> sh);
}

// V = the weight of the points with det A > 0 (the input's own volume).
template <typename T, int NM>
__global__ void __launch_bounds__(256) k_wvolume(const T* A, const unsigned long long* w, long long nq,
                                                 WSelect* ws) {
  constexpr int C = NM * NM;
  __shared__ unsigned long long part[8];
  unsigned long long v = 0;
  for (long long q = blockIdx.x * 256LL + threadIdx.x; q < nq; q += (long long)gridDim.x * 256) {
    T m[C];
#pragma unroll
    for (int c = 0; c < C; ++c) m[c] = A[c * nq + q];
    if (det_sign<NM>(m) > T(0)) v += w[q];
  }
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int i = 0; i < 8; ++i) t += part[i];
    atomicAdd(&ws->target, t);
  }
}

__global__ void k_wselect_init(WSelect* ws, unsigned long long target, int use_given) {
  if (threadIdx.x == 0) {
    if (use_given) ws->target = target;
    ws->hi = 0;
    ws->lo = 0;
    ws->all = 0;
    ws->vrem = ws->target;
  }
  for (int i = threadIdx.x; i < 256; i += blockDim.x) ws->hist[i] = 0;
}

__global__ void __launch_bounds__(256) k_wselect_hist(const unsigned long long* __restrict__ keys,
                                                      const unsigned long long* __restrict__ w, long long nq,
                                                      WSelect* ws, int d) {
  __shared__ unsigned long long h[256];
  for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
  __syncthreads();
  const unsigned long long hi = ws->hi;
  const unsigned lo = ws->lo;
  const bool active = ws->target > 0 && !ws->all;
  if (active) {
    for (long long x = blockIdx.x * 256LL + threadIdx.x; x < nq; x += (long long)gridDim.x * 256) {
      const unsigned long long key = keys[x];
      if (wprefix(key, (unsigned)x, hi, lo, d)) atomicAdd(&h[wdigit(key, (unsigned)x, d)], w[x]);
    }
  }
  __syncthreads();
  if (active)
    for (int i = threadIdx.x; i < 256; i += blockDim.x)
      if (h[i]) atomicAdd(&ws->hist[i], h[i]);
}

__global__ void k_wselect_pick(WSelect* ws, SelectState* ss, int d) {
  if (threadIdx.x != 0) return;
  if (ws->target > 0 && !ws->all) {
    const unsigned long long v = ws->vrem;
    unsigned long long cum = 0;
    int b = 0;
    for (; b < 256; ++b) {
      if (cum + ws->hist[b] >= v) break;
      cum += ws->hist[b];
    }
    if (b == 256) {  // only on the first pass: V exceeds the total weight
      ws->all = 1;
      ws->hi = ~0ull;
      ws->lo = ~0u;
    } else {
      ws->vrem = v - cum;
      if (d < 8) ws->hi |= ((unsigned long long)b) << (56 - 8 * d);
      else ws->lo |= ((unsigned)b) << (24 - 8 * (d - 8));
    }
  }
  for (int i = 0; i < 256; ++i) ws->hist[i] = 0;
  if (d == 11) {
    ss->hi = ws->hi;
    ss->lo = ws->lo;
    ss->n_plus = ws->target > 0 ? 1 : 0;
  }
}

// ----------------------------------------------------------------------------
// host-side geometry (Algorithm 2, step 1) and plan parameters
// ----------------------------------------------------------------------------

double tail_T(double x) { return 2.0 * x / std::sqrt(M_PI) * std::exp(-x * x) + std::erfc(x); }

// Gauss-Legendre nodes and weights on [-1, 1] (Newton iteration on the
// three-term recurrence of P_n, starting from the Chebyshev-like guesses
// cos(pi (i - 1/4) / (n + 1/2))).
void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w) {
  x.assign(n, 0.0);
  w.assign(n, 0.0);
  for (int i = 0; i < (n + 1) / 2; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    x[i] = -z;
    x[n - 1 - i] = z;
    w[i] = w[n - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

// Band cells and quadrature points (Algorithm 2, step 1): the cells
// x_g + [0, dx]^3 of the grid dx Z^3 with |i| <= li, |j|, |k| <= lr whose corner
// x_g is in the band, each with p^3 points (the tensor product of the Chebyshev
// nodes cos((2k - 1) pi / (2p)) mapped to [0, dx], with Fejer's first-rule
// weights) and their closest points.  Order: cells (i, j, k) lexicographic, k
// fastest, then the nodes (a, b, c), c fastest.  With any output NULL only the
// count is produced.
template <typename InBand, typename Closest>
mbo_status emit_band(double dx, int p, long long li, long long lr, InBand in_band, Closest closest,
                     double* xq, double* wq, double* xc, int64_t capacity, int64_t* count) {
  std::vector<double> off(p), wc(p);
  for (int k = 0; k < p; ++k) {
    const double th = (2.0 * (k + 1) - 1.0) * M_PI / (2.0 * p);
    double s = 0.0;
    for (int j = 1; j <= p / 2; ++j) s += std::cos(2.0 * j * th) / (4.0 * j * j - 1.0);
    off[k] = dx * (1.0 + std::cos(th)) / 2.0;
    wc[k] = (2.0 / p) * (1.0 - 2.0 * s) * dx / 2.0;
  }
  const long long per = (long long)p * p * p;
  int64_t n = 0;
  const bool fill = xq && wq && xc;
  for (long long i = -li; i <= li; ++i)
    for (long long j = -lr; j <= lr; ++j)
      for (long long k = -lr; k <= lr; ++k) {
        const double gx = dx * i, gy = dx * j, gz = dx * k;
        if (!in_band(gx, gy, gz)) continue;
        if (fill && n + per <= capacity) {
          for (int a = 0; a < p; ++a)
            for (int b = 0; b < p; ++b)
              for (int c = 0; c < p; ++c) {
                const int64_t q = n + ((int64_t)a * p + b) * p + c;
                xq[3 * q] = gx + off[a];
                xq[3 * q + 1] = gy + off[b];
                xq[3 * q + 2] = gz + off[c];
                wq[q] = wc[a] * wc[b] * wc[c];
                closest(xq[3 * q], xq[3 * q + 1], xq[3 * q + 2], xc + 3 * q);
              }
        }
        n += per;
      }
  *count = n;
  if (fill && n > capacity) return MBO_ERR_INVALID_ARG;
  return MBO_OK;
}

// Generating curve of the peanut surface (Sec. 6.3), t in [-1, 1]: x = 3t - t^3
// and rho = sqrt((1 + x^2)(4 - x^2)) / 2, written as (1 - t^2) sqrt((1 + x^2)(4 - t^2)) / 2
// (4 - x^2 = (1 - t^2)^2 (4 - t^2)), which stays real to the ends.
void peanut_curve(double t, double& x, double& rho) {
  x = 3.0 * t - t * t * t;
  rho = 0.5 * (1.0 - t * t) * std::sqrt((1.0 + x * x) * (4.0 - t * t));
}

// Closest point c on the peanut surface to (x, y, z) and its distance.  The
// surface is one of revolution about the x axis, so the closest point is that of
// (x, |(y, z)|) on the generating curve, turned into the point's meridian (the
// +y meridian on the axis): a scan of 257 values of t, then a golden-section
// search between the neighbours of the nearest one.
double peanut_closest(double px, double py, double pz, double* c) {
  const double r = std::sqrt(py * py + pz * pz);
  auto D = [&](double t) {
    double x, rho;
    peanut_curve(t, x, rho);
    return (x - px) * (x - px) + (rho - r) * (rho - r);
  };
  constexpr int kScan = 257;
  int best = 0;
  double dbest = D(-1.0);
  for (int i = 1; i < kScan; ++i) {
    const double d = D(-1.0 + 2.0 * i / (kScan - 1));
    if (d < dbest) {
      dbest = d;
      best = i;
    }
  }
  const double step = 2.0 / (kScan - 1);
  double lo = std::max(-1.0, -1.0 + step * (best - 1)), hi = std::min(1.0, -1.0 + step * (best + 1));
  const double g = 0.5 * (std::sqrt(5.0) - 1.0);
  double a = hi - g * (hi - lo), b = lo + g * (hi - lo), fa = D(a), fb = D(b);
  for (int it = 0; it < 80; ++it) {
    if (fa < fb) {
      hi = b;
      b = a;
      fb = fa;
      a = hi - g * (hi - lo);
      fa = D(a);
    } else {
      lo = a;
      a = b;
      fa = fb;
      b = lo + g * (hi - lo);
      fb = D(b);
    }
  }
  const double t = 0.5 * (lo + hi);
  double x, rho;
  peanut_curve(t, x, rho);
  const double uy = r > 0 ? py / r : 1.0, uz = r > 0 ? pz / r : 0.0;
  c[0] = x;
  c[1] = rho * uy;
  c[2] = rho * uz;
  return std::sqrt(D(t));
}

bool smooth23(int N) {
  while (N % 2 == 0) N /= 2;
  while (N % 3 == 0) N /= 3;
  return N == 1;
}

}  // namespace
}  // namespace mbo

using namespace mbo;

struct mbo_surface_ctx {
  int dev = 0;
  mbo_dtype dtype = MBO_F32;
  int n = 0, C = 0;
  long long nq = 0;
  double tau = 0, eps = 0;
  mbo_surface_params prm{};
  int nb = 0;        // bins per axis
  int nbins = 0;     // non-empty source bins
  int sgroups = 0;   // source groups
  int tgroups = 0;   // target groups
  int cg = 1, chgroups = 1;  // channels per spreading block, channel groups
  size_t tile_bytes = 0;
  GridBox box{};              // FP32: the box of all footprints; FP64: the whole grid
  BoxDiffusion bd{};          // FP32: diffusion between points of the box
  mbo_handle fine = nullptr;  // FP64: 3-D FFT diffusion on the nf^3 grid
  void* F = nullptr;          // grid values of the box, C channels
  void* At = nullptr;         // diffused values, C x nq
  // volume-preserving step (allocated on first use)
  void* Au = nullptr;                      // diffused values in the caller's order, C x nq
  unsigned long long* vkeys = nullptr;     // one selection key per point
  SelectState* vss = nullptr;
  WSelect* vws = nullptr;
  unsigned long long* vw = nullptr;        // fixed-point weights (caller's order), sum 2^62
  double wscale = 0;                       // fixed-point units per unit of w_q
  std::vector<double> hw;                  // the weights w_q (host copy)
  void* su = nullptr;         // V4<T> sources
  int* sidx = nullptr;
  int* gsrc = nullptr;
  int* gt0 = nullptr;
  int4* sg0 = nullptr;        // FP32, width 7: source group -> footprint start on the grid
  int* seg = nullptr;         // FP32, width 7: segment -> first group
  int nseg = 0;
  int* bgrp = nullptr;
  int* bid = nullptr;
  void* tu = nullptr;         // V4<T> targets
  int* tidx = nullptr;
  int* tgrp = nullptr;
  int4* tg0 = nullptr;
  SurfStats* st = nullptr;
  SurfStats* h_st = nullptr;  // pinned
  size_t bytes = 0;
  // per-pass timing (mbo_surface_profile_*)
  bool prof = false;
  struct Pending { int pass; cudaEvent_t a, b; };
  std::vector<Pending> pending;
  std::vector<cudaEvent_t> ev_free;
  double prof_ms[MBO_SURFACE_PROFILE_PASSES] = {0};
  long long prof_n[MBO_SURFACE_PROFILE_PASSES] = {0};
  char err[512] = {0};
};

namespace {

cudaEvent_t take_event(mbo_surface_ctx* s) {
  if (!s->ev_free.empty()) {
    cudaEvent_t e = s->ev_free.back();
    s->ev_free.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

// Run f (a launch sequence on stream st); when profiling, bracket it with events.
template <typename Fn> cudaError_t timed(mbo_surface_ctx* s, int pass, cudaStream_t st, Fn&& f) {
  if (!s->prof) return f();
  cudaEvent_t a = take_event(s), b = take_event(s);
  cudaEventRecord(a, st);
  const cudaError_t e = f();
  cudaEventRecord(b, st);
  s->pending.push_back({pass, a, b});
  return e;
}

mbo_status sfail(mbo_surface_ctx* s, mbo_status rc, const char* fmt, const char* what = "") {
  if (s) snprintf(s->err, sizeof(s->err), fmt, what);
  return rc;
}

#define SCK(call)                                                                           \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return sfail(s, e_ == cudaErrorMemoryAllocation ? MBO_ERR_OOM : MBO_ERR_CUDA,         \
                   "%s", cudaGetErrorString(e_));                                           \
  } while (0)

// Shared bytes of a spreading block: the tile and the per-warp staging.
size_t spread_smem(int cg, size_t elem, size_t tv) {
  const size_t vw = 16 / elem;
  const size_t chunk = elem == 4 ? chunk_of<float>() : chunk_of<double>();
  const size_t stride = elem == 4 ? src_stride<float>() : src_stride<double>();
  return (((size_t)cg * tv + vw - 1) / vw * vw + (size_t)(kSpreadThreads / 32) * chunk * stride) * elem;
}

// Channels per spreading block for n*n channels: the largest instantiated
// group that fits in `limit` shared bytes (0 if none fits).
int spread_cg(int C, size_t elem, size_t tv, size_t limit) {
  const int cand[] = {9, 8, 4, 3, 1};
  for (int cg : cand) {
    if (cg > C || (elem == 8 && cg > 4)) continue;  // FP64: at most 4 (registers)
    if (spread_smem(cg, elem, tv) <= limit) return cg;
  }
  return 0;
}

template <typename T, int CG> cudaError_t spread_run(const SpreadArgs<T>& a, dim3 grid, size_t smem,
                                                     cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    if (a.W == 7) {
      k_spread7<CG><<<dim3(a.nseg, grid.y), kSpread7Threads, 0, st>>>(a);
      return cudaGetLastError();
    }
  }
  const bool w7 = sizeof(T) == 8 && a.W == 7;
  auto k = w7 ? k_spread<T, CG, sizeof(T) == 8 ? 7 : 0> : k_spread<T, CG, 0>;
  static SmemLimit limit[2];
  const cudaError_t e = raise_smem(k, smem, limit[w7]);
  if (e != cudaSuccess) return e;
  k<<<grid, kSpreadThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_spread(mbo_surface_ctx* s, const void* A, cudaStream_t st) {
  SpreadArgs<T> a;
  a.A = static_cast<const T*>(A);
  a.su = static_cast<const V4<T>*>(s->su);
  a.sidx = s->sidx;
  a.gsrc = s->gsrc;
  a.gt0 = s->gt0;
  a.bgrp = s->bgrp;
  a.g0 = s->sg0;
  a.seg = s->seg;
  a.nseg = s->nseg;
  a.bid = s->bid;
  a.F = static_cast<T*>(s->F);
  a.box = s->box;
  a.nq = s->nq;
  a.C = s->C;
  a.nf = s->prm.nf;
  a.nb = s->nb;
  a.W = s->prm.width;
  a.beta = (T)s->prm.beta;
  const dim3 grid(s->nbins, s->chgroups);
  switch (s->cg) {
    case 1: return spread_run<T, 1>(a, grid, s->tile_bytes, st);
    case 3: return spread_run<T, 3>(a, grid, s->tile_bytes, st);
    case 4: return spread_run<T, 4>(a, grid, s->tile_bytes, st);
    default: break;
  }
  if constexpr (sizeof(T) == 4) {  // FP64 groups stop at 4 channels (registers)
    if (s->cg == 8) return spread_run<T, 8>(a, grid, s->tile_bytes, st);
    if (s->cg == 9) return spread_run<T, 9>(a, grid, s->tile_bytes, st);
  }
  return cudaErrorInvalidValue;
}

template <typename T, int NM> cudaError_t interp_run(const InterpArgs<T>& a, int groups, size_t smem,
                                                      cudaStream_t st) {
  if constexpr (sizeof(T) == 4 && (NM == 2 || NM == 3)) {
    if (a.W == 7) {
      k_interp7<NM><<<groups, kInterpBlock, 343 * Interp7<NM>::ST * sizeof(float), st>>>(a);
      return cudaGetLastError();
    }
  }
  constexpr int W7 = sizeof(T) == 4 && (NM == 2 || NM == 3) ? 0 : 7;
  auto k = a.W == 7 ? k_interp<T, NM, W7> : k_interp<T, NM, 0>;
  static SmemLimit limit[2];
  const cudaError_t e = raise_smem(k, smem, limit[a.W == 7 && W7]);
  if (e != cudaSuccess) return e;
  k<<<groups, kInterpBlock, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_interp(mbo_surface_ctx* s, void* dst, cudaStream_t st) {
  InterpArgs<T> a;
  a.F = static_cast<const T*>(s->F);
  a.box = s->box;
  a.tu = static_cast<const V4<T>*>(s->tu);
  a.tidx = s->tidx;
  a.tgrp = s->tgrp;
  a.tg0 = s->tg0;
  a.dst = static_cast<T*>(dst);
  a.nq = s->nq;
  a.nf = s->prm.nf;
  a.W = s->prm.width;
  a.beta = (T)s->prm.beta;
  const int W3 = s->prm.width * s->prm.width * s->prm.width;
  const int CP = s->C == 1 ? 1 : (sizeof(T) == 4 ? (s->C + 3) / 4 * 4 : (s->C + 1) / 2 * 2);
  const size_t smem = (size_t)W3 * CP * sizeof(T);
  switch (s->n) {
    case 1: return interp_run<T, 1>(a, s->tgroups, smem, st);
    case 2: return interp_run<T, 2>(a, s->tgroups, smem, st);
    case 3: return interp_run<T, 3>(a, s->tgroups, smem, st);
    default: return interp_run<T, 4>(a, s->tgroups, smem, st);
  }
}

template <typename T> cudaError_t launch_project(mbo_surface_ctx* s, void* A, cudaStream_t st) {
  ProjArgs<T> a;
  a.At = static_cast<const T*>(s->At);
  a.A = static_cast<T*>(A);
  a.st = s->st;
  a.nq = s->nq;
  a.fb = T(0);
  const unsigned blocks = (unsigned)((s->nq + kProjThreads - 1) / kProjThreads);
  switch (s->n) {
    case 1: k_sproject<T, 1><<<blocks, kProjThreads, 0, st>>>(a); break;
    case 2: k_sproject<T, 2><<<blocks, kProjThreads, 0, st>>>(a); break;
    case 3: k_sproject<T, 3><<<blocks, kProjThreads, 0, st>>>(a); break;
    default: k_sproject<T, 4><<<blocks, kProjThreads, 0, st>>>(a); break;
  }
  return cudaGetLastError();
}

mbo_status surface_diffusion(mbo_surface_ctx* s, const void* A, void* dst, cudaStream_t st) {
  const size_t elem = s->dtype == MBO_F32 ? 4 : 8;
  SCK(cudaMemsetAsync(s->F, 0, (size_t)s->C * s->box.points() * elem, st));
  SCK(timed(s, 0, st, [&] {
    return s->dtype == MBO_F32 ? launch_spread<float>(s, A, st) : launch_spread<double>(s, A, st);
  }));
  if (s->dtype == MBO_F32) {
    SCK(timed(s, 1, st, [&] { return box_diffuse(s->bd, static_cast<float*>(s->F), st); }));
  } else {
    mbo_status rc = MBO_OK;
    timed(s, 1, st, [&] {
      rc = mbo_diffuse(s->fine, s->F, s->F, st);
      return cudaSuccess;
    });
    if (rc != MBO_OK) return sfail(s, rc, "grid diffusion: %s", mbo_last_error(s->fine));
  }
  SCK(timed(s, 2, st, [&] {
    return s->dtype == MBO_F32 ? launch_interp<float>(s, dst, st) : launch_interp<double>(s, dst, st);
  }));
  return MBO_OK;
}

template <typename T> void upload_points(const std::vector<V4<double>>& in, void* dst) {
  std::vector<V4<T>> v(in.size());
  for (size_t i = 0; i < in.size(); ++i) v[i] = V4<T>{(T)in[i].x, (T)in[i].y, (T)in[i].z, (T)in[i].w};
  cudaMemcpy(dst, v.data(), v.size() * sizeof(V4<T>), cudaMemcpyHostToDevice);
}

}  // namespace

extern "C" {

double mbo_surface_band_width(double eps, double tau) {
  if (!(eps > 0 && eps < 1) || !(tau > 0) || !std::isfinite(tau)) return -1.0;
  double lo = 0.0, hi = 1.0;
  while (tail_T(hi) > eps) hi *= 2.0;
  for (int i = 0; i < 200 && hi - lo > 0; ++i) {
    const double mid = 0.5 * (lo + hi);
    (tail_T(mid) > eps ? lo : hi) = mid;
  }
  return 2.0 * std::sqrt(tau) * hi;
}

mbo_status mbo_surface_heat_modes(double eps, double tau, double R, double* h, int* M) {
  if (!(eps > 0 && eps < 0.5) || !(tau > 0) || !(R > 0) || !std::isfinite(tau) || !std::isfinite(R))
    return MBO_ERR_INVALID_ARG;
  const double hh = std::min(M_PI / R, M_PI / (2.0 * std::sqrt(tau * std::fabs(std::log(eps)))));
  const double lg = std::log(2.0 * hh * std::sqrt(tau) / (std::sqrt(M_PI) * eps));
  const double mm = std::ceil(std::sqrt(std::max(lg, 0.0) / tau) / hh);
  if (h) *h = hh;
  if (M) *M = (int)std::max(1.0, std::min(mm, 1e9));
  return MBO_OK;
}

mbo_status mbo_surface_sphere_band(double radius, double dx, double wb, int p, double* xq,
                                   double* wq, double* xc, int64_t capacity, int64_t* count) {
  if (!(radius > 0) || !(dx > 0) || !(wb > 0) || p < 1 || p > 16 || !count) return MBO_ERR_INVALID_ARG;
  const long long lim = (long long)std::ceil((radius + wb) / dx) + 1;
  auto in_band = [&](double x, double y, double z) {
    return std::fabs(std::sqrt(x * x + y * y + z * z) - radius) < wb;
  };
  auto closest = [&](double x, double y, double z, double* c) {
    const double r = std::sqrt(x * x + y * y + z * z);
    if (r > 0) {
      c[0] = radius * x / r;
      c[1] = radius * y / r;
      c[2] = radius * z / r;
    } else {
      c[0] = 0.0;
      c[1] = 0.0;
      c[2] = radius;
    }
  };
  return emit_band(dx, p, lim, lim, in_band, closest, xq, wq, xc, capacity, count);
}

mbo_status mbo_surface_peanut_band(double dx, double wb, int p, double* xq, double* wq, double* xc,
                                   int64_t capacity, int64_t* count) {
  if (!(dx > 0) || !(wb > 0) || p < 1 || p > 16 || !count) return MBO_ERR_INVALID_ARG;
  double rho_max = 0.0;
  for (int i = 0; i <= 4096; ++i) {
    double x, rho;
    peanut_curve(-1.0 + 2.0 * i / 4096, x, rho);
    rho_max = std::max(rho_max, rho);
  }
  const long long lx = (long long)std::ceil((2.0 + wb) / dx) + 1;
  const long long lr = (long long)std::ceil((rho_max + wb) / dx) + 1;
  auto in_band = [&](double x, double y, double z) {
    double c[3];
    return peanut_closest(x, y, z, c) < wb;
  };
  auto closest = [&](double x, double y, double z, double* c) { peanut_closest(x, y, z, c); };
  return emit_band(dx, p, lx, lr, in_band, closest, xq, wq, xc, capacity, count);
}

mbo_status mbo_surface_destroy(mbo_surface s) {
  if (!s) return MBO_ERR_INVALID_ARG;
  int prev = -1;
  if (cudaGetDevice(&prev) == cudaSuccess && prev != s->dev) cudaSetDevice(s->dev);
  else prev = -1;
  cudaDeviceSynchronize();
  if (s->fine) mbo_destroy(s->fine);
  void* bufs[] = {s->bd.tabs, s->bd.W1, s->bd.W2, s->F, s->At, s->su, s->sidx, s->gsrc, s->gt0, s->bgrp, s->bid, s->sg0, s->seg,
                  s->tu, s->tidx, s->tgrp, s->tg0, s->st, s->Au, s->vkeys, s->vss, s->vws, s->vw};
  for (void* b : bufs)
    if (b) cudaFree(b);
  if (s->h_st) cudaFreeHost(s->h_st);
  for (auto& p : s->pending) {
    cudaEventDestroy(p.a);
    cudaEventDestroy(p.b);
  }
  for (cudaEvent_t e : s->ev_free) cudaEventDestroy(e);
  if (prev >= 0) cudaSetDevice(prev);
  delete s;
  return MBO_OK;
}

mbo_status mbo_surface_create(mbo_surface* out, int64_t nq, const double* xq, const double* wq,
                              const double* xc, int n, double tau, double eps, mbo_dtype dtype) {
  if (!out) return MBO_ERR_INVALID_ARG;
  *out = nullptr;
  if (nq < 1 || nq >= (1LL << 31) || !xq || !wq || !xc || n < 1 || n > 4 || !(tau > 0) ||
      !std::isfinite(tau) || !(eps > 1e-12 && eps < 0.5) || (dtype != MBO_F32 && dtype != MBO_F64))
    return MBO_ERR_INVALID_ARG;
  for (int64_t i = 0; i < 3 * nq; ++i)
    if (!std::isfinite(xq[i]) || !std::isfinite(xc[i])) return MBO_ERR_INVALID_ARG;
  for (int64_t i = 0; i < nq; ++i)
    if (!std::isfinite(wq[i])) return MBO_ERR_INVALID_ARG;

  mbo_surface_ctx* s = new mbo_surface_ctx();
  cudaGetDevice(&s->dev);
  s->dtype = dtype;
  s->n = n;
  s->C = n * n;
  s->nq = nq;
  s->tau = tau;
  s->eps = eps;
  s->hw.assign(wq, wq + nq);
  mbo_surface_params& prm = s->prm;

  // extent and centre of all points
  double lo[3], hi[3];
  for (int a = 0; a < 3; ++a) lo[a] = hi[a] = xq[a];
  for (int64_t i = 0; i < nq; ++i)
    for (int a = 0; a < 3; ++a) {
      lo[a] = std::min(lo[a], std::min(xq[3 * i + a], xc[3 * i + a]));
      hi[a] = std::max(hi[a], std::max(xq[3 * i + a], xc[3 * i + a]));
    }
  prm.R = 0;
  for (int a = 0; a < 3; ++a) {
    prm.center[a] = 0.5 * (lo[a] + hi[a]);
    prm.R = std::max(prm.R, hi[a] - lo[a]);
  }
  if (!(prm.R > 0)) prm.R = 1.0;  // a single point: any radius
  mbo_surface_heat_modes(eps, tau, prm.R, &prm.h, &prm.M);
  int W = (int)std::ceil(std::log10(1.0 / eps)) + 1;
  W = std::max(kMinW, std::min(W, kMaxW));
  prm.width = W;
  prm.beta = 2.30 * W;
  int nf = std::max(std::max(4 * prm.M, 2 * W), 8);
  while (!smooth23(nf)) ++nf;
  prm.nf = nf;
  if (nf > 2048) {
    mbo_surface_destroy(s);
    return MBO_ERR_UNSUPPORTED_SIZE;
  }
  const int nb = (nf + kBin - 1) / kBin;
  s->nb = nb;

  // grid coordinates u = (h (x - centre) + pi) nf / (2 pi); the footprint of a
  // point starts at g = ceil(u - W/2) on each axis (W points), and d = u - g
  const double sc = (double)nf / (2.0 * M_PI);
  auto grid_coord = [&](const double* x, double* u) {
    for (int a = 0; a < 3; ++a) {
      const double v = (prm.h * (x[a] - prm.center[a]) + M_PI) * sc;
      u[a] = std::min(std::max(v, 0.0), std::nextafter((double)nf, 0.0));
    }
  };
  // sources: key (bin, footprint start in the bin tile), or for k_spread7 the
  // footprint start on the grid, z fastest; targets: footprint start
  const bool columns = dtype == MBO_F32 && W == 7;
  std::vector<char> bin_used((size_t)nb * nb * nb, 0);
  std::vector<long long> skey(nq), tkey(nq);
  std::vector<V4<double>> sd(nq), td(nq);
  // extent of all footprints (unwrapped): sources cover W + 1 points from an
  // even start in x and y, everything else W
  int ext_lo[3] = {nf, nf, nf}, ext_hi[3] = {-nf, -nf, -nf};
  auto cover = [&](int a, int from, int count) {
    ext_lo[a] = std::min(ext_lo[a], from);
    ext_hi[a] = std::max(ext_hi[a], from + count);
  };
  for (int64_t i = 0; i < nq; ++i) {
    double u[3];
    int b[3], t0[3], g[3];
    grid_coord(xq + 3 * i, u);
    for (int a = 0; a < 3; ++a) {
      b[a] = std::min((int)(u[a] / kBin), nb - 1);
      // footprint start relative to the tile origin b kBin - W/2, kept in [0, kBin];
      // the group start rounds it down to even in x and y
      t0[a] = (int)std::ceil(u[a] - 0.5 * W) - (b[a] * kBin - W / 2);
      t0[a] = std::min(std::max(t0[a], 0), kBin);
      if (a < 2) t0[a] &= ~1;
      g[a] = b[a] * kBin - W / 2 + t0[a];
      if (columns) {
        g[a] = (int)std::ceil(u[a] - 0.5 * W);
        if (a < 2) g[a] -= g[a] & 1;
      }
      cover(a, g[a], a < 2 ? W + 1 : W);
    }
    const long long bin = ((long long)b[2] * nb + b[1]) * nb + b[0];
    bin_used[bin] = 1;
    skey[i] = columns ? (((long long)(g[1] + kMaxW) << 12 | (g[0] + kMaxW)) << 12 | (g[2] + kMaxW))
                      : bin * 4096 + (t0[2] << 8 | t0[1] << 4 | t0[0]);
    sd[i] = V4<double>{u[0] - g[0], u[1] - g[1], u[2] - g[2], wq[i]};
    grid_coord(xc + 3 * i, u);
    for (int a = 0; a < 3; ++a) {
      g[a] = (int)std::ceil(u[a] - 0.5 * W);
      cover(a, g[a], W);
    }
    // wrapped start on the periodic grid (u >= 0, so g >= -W/2)
    const int gx = (g[0] + nf) % nf, gy = (g[1] + nf) % nf, gz = (g[2] + nf) % nf;
    tkey[i] = ((long long)gz * nf + gy) * nf + gx;
    td[i] = V4<double>{u[0] - g[0], u[1] - g[1], u[2] - g[2], 0.0};
  }
  std::vector<int> sperm(nq), tperm(nq);
  std::iota(sperm.begin(), sperm.end(), 0);
  std::iota(tperm.begin(), tperm.end(), 0);
  std::stable_sort(sperm.begin(), sperm.end(), [&](int x, int y) { return skey[x] < skey[y]; });
  std::stable_sort(tperm.begin(), tperm.end(), [&](int x, int y) { return tkey[x] < tkey[y]; });
  std::vector<int> gsrc, gt0, bgrp, bid, tgrp, seg;
  std::vector<int4> sg0;
  std::vector<int4> tg0;
  std::vector<V4<double>> sds(nq), tds(nq);
  for (int64_t r = 0; r < nq; ++r) {
    const int i = sperm[r];
    sds[r] = sd[i];
    if (r == 0 || skey[i] != skey[sperm[r - 1]]) {
      const long long bin = skey[i] / 4096;
      if (columns) {
        sg0.push_back(make_int4((int)(skey[i] >> 12 & 4095) - kMaxW, (int)(skey[i] >> 24) - kMaxW,
                                (int)(skey[i] & 4095) - kMaxW, 0));
      } else if (r == 0 || bin != skey[sperm[r - 1]] / 4096) {
        bid.push_back((int)bin);
        bgrp.push_back((int)gsrc.size());
      }
      gsrc.push_back((int)r);
      gt0.push_back((int)(skey[i] % 4096));
    }
    const int j = tperm[r];
    tds[r] = td[j];
    if (r == 0 || tkey[j] != tkey[tperm[r - 1]]) {
      tgrp.push_back((int)r);
      const long long k = tkey[j];
      tg0.push_back(make_int4((int)(k % nf), (int)((k / nf) % nf), (int)(k / ((long long)nf * nf)), 0));
    }
  }
  gsrc.push_back((int)nq);
  tgrp.push_back((int)nq);
  bgrp.push_back((int)gt0.size());
  // segments: runs of a column's groups, up to kSegSources sources where a group
  // does not hold more, without gaps of a whole footprint in z
  for (size_t g = 0; g < sg0.size(); ++g) {
    const bool run = g > 0 && sg0[g].x == sg0[g - 1].x && sg0[g].y == sg0[g - 1].y &&
                     sg0[g].z - sg0[g - 1].z < W && gsrc[g + 1] - gsrc[seg.back()] <= kSegSources;
    if (!run) seg.push_back((int)g);
  }
  s->nseg = (int)seg.size();
  seg.push_back((int)sg0.size());
  s->nbins = (int)bid.size();
  s->sgroups = (int)gsrc.size() - 1;
  s->tgroups = (int)tg0.size();
  prm.bins = std::count(bin_used.begin(), bin_used.end(), 1);

  // channel groups of the spreading tile
  const size_t elem = dtype == MBO_F32 ? 4 : 8;
  const size_t tv = (size_t)(kBin + W + 1) * (kBin + W + 1) * (kBin + W);
  int maxsm = 0;
  cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->dev);
  s->cg = spread_cg(s->C, elem, tv, (size_t)maxsm);
  s->chgroups = s->cg ? (s->C + s->cg - 1) / s->cg : 0;
  s->tile_bytes = spread_smem(s->cg, elem, tv);
  if (s->cg == 0) {
    mbo_surface_destroy(s);
    return MBO_ERR_UNSUPPORTED_SIZE;
  }

  // the grid's FFT diffusion with the deconvolved heat factor
  mbo_status rc = MBO_OK;
  for (int a = 0; a < 3; ++a) {
    // an axis whose footprints wrap keeps all of it
    const bool inside = dtype == MBO_F32 && ext_lo[a] >= 0 && ext_hi[a] <= nf;
    s->box.b0[a] = inside ? ext_lo[a] : 0;
    s->box.bn[a] = inside ? ext_hi[a] - ext_lo[a] : nf;
  }
  if (dtype == MBO_F64) {
    const int64_t dims[3] = {nf, nf, nf};
    rc = mbo_create(&s->fine, 3, dims, n, 1.0, dtype, nullptr);
    if (rc != MBO_OK) {
      snprintf(s->err, sizeof(s->err), "grid plan: %s", mbo_status_string(rc));
      mbo_surface_destroy(s);
      return rc;
    }
  }
  std::vector<double> gx, gwt, mult(nf);
  gauss_legendre(128, gx, gwt);
  for (int k = 0; k < nf; ++k) {
    const int kf = (2 * k <= nf) ? k : k - nf;
    const int ak = std::abs(kf);
    const double win = ak < prm.M ? 1.0 : (ak == prm.M ? 0.5 : 0.0);
    if (win == 0.0) {
      mult[k] = 0.0;
      continue;
    }
    // psi(k) = (W/2) int_{-1}^{1} phi(z) cos(pi k W z / nf) dz
    double psi = 0.0;
    for (size_t i = 0; i < gx.size(); ++i) {
      const double z = gx[i];
      psi += gwt[i] * std::exp(prm.beta * (std::sqrt(1.0 - z * z) - 1.0)) * std::cos(M_PI * kf * W * z / nf);
    }
    psi *= 0.5 * W;
    mult[k] = nf * (prm.h / (2.0 * M_PI)) * win * std::exp(-(double)kf * kf * prm.h * prm.h * tau) / (psi * psi);
  }
  const double* mm[3] = {mult.data(), mult.data(), mult.data()};
  if (dtype == MBO_F64 && !set_axis_multipliers(s->fine, mm)) {
    snprintf(s->err, sizeof(s->err), "grid multipliers: %s", cudaGetErrorString(cudaGetLastError()));
    mbo_surface_destroy(s);
    return MBO_ERR_CUDA;
  }
  if (dtype == MBO_F32) {
    rc = box_create(s->bd, s->box, nf, n, prm.M, mult.data(), maxsm, s->bytes);
    if (rc != MBO_OK) {
      snprintf(s->err, sizeof(s->err), "grid plan: %s", mbo_status_string(rc));
      mbo_surface_destroy(s);
      return rc;
    }
  }

  // device tables
  const long long P = s->box.points();
  auto alloc = [&](void** p, size_t b) {
    if (cudaMalloc(p, std::max<size_t>(b, 16)) != cudaSuccess) return false;
    s->bytes += b;
    return true;
  };
  const size_t v4 = dtype == MBO_F32 ? sizeof(V4<float>) : sizeof(V4<double>);
  if (!alloc(&s->F, (size_t)s->C * P * elem) || !alloc(&s->At, (size_t)s->C * nq * elem) ||
      !alloc(&s->su, nq * v4) || !alloc((void**)&s->sidx, nq * sizeof(int)) ||
      !alloc((void**)&s->gsrc, gsrc.size() * sizeof(int)) || !alloc((void**)&s->gt0, gt0.size() * sizeof(int)) ||
      !alloc((void**)&s->sg0, sg0.size() * sizeof(int4)) || !alloc((void**)&s->seg, seg.size() * sizeof(int)) ||
      !alloc((void**)&s->bgrp, bgrp.size() * sizeof(int)) || !alloc((void**)&s->bid, bid.size() * sizeof(int)) ||
      !alloc(&s->tu, nq * v4) || !alloc((void**)&s->tidx, nq * sizeof(int)) ||
      !alloc((void**)&s->tgrp, tgrp.size() * sizeof(int)) || !alloc((void**)&s->tg0, tg0.size() * sizeof(int4)) ||
      !alloc((void**)&s->st, sizeof(SurfStats)) ||
      cudaMallocHost((void**)&s->h_st, sizeof(SurfStats)) != cudaSuccess) {
    mbo_surface_destroy(s);
    return MBO_ERR_OOM;
  }
  if (dtype == MBO_F32) {
    upload_points<float>(sds, s->su);
    upload_points<float>(tds, s->tu);
  } else {
    upload_points<double>(sds, s->su);
    upload_points<double>(tds, s->tu);
  }
  cudaMemcpy(s->sidx, sperm.data(), nq * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->gsrc, gsrc.data(), gsrc.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->gt0, gt0.data(), gt0.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->bgrp, bgrp.data(), bgrp.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->sg0, sg0.data(), sg0.size() * sizeof(int4), cudaMemcpyHostToDevice);
  cudaMemcpy(s->seg, seg.data(), seg.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->bid, bid.data(), bid.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->tidx, tperm.data(), nq * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->tgrp, tgrp.data(), tgrp.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(s->tg0, tg0.data(), tg0.size() * sizeof(int4), cudaMemcpyHostToDevice);
  const cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    snprintf(s->err, sizeof(s->err), "table upload: %s", cudaGetErrorString(e));
    mbo_surface_destroy(s);
    return MBO_ERR_CUDA;
  }
  *out = s;
  return MBO_OK;
}

mbo_status mbo_surface_get_params(mbo_surface s, mbo_surface_params* p) {
  if (!s || !p) return MBO_ERR_INVALID_ARG;
  *p = s->prm;
  return MBO_OK;
}

mbo_status mbo_surface_diffuse(mbo_surface s, const void* A, void* A_tilde, void* stream) {
  if (!s || !A || !A_tilde || ((uintptr_t)A & 15) || ((uintptr_t)A_tilde & 15)) return MBO_ERR_INVALID_ARG;
  return surface_diffusion(s, A, A_tilde, static_cast<cudaStream_t>(stream));
}

mbo_status mbo_surface_step(mbo_surface s, void* A, mbo_stats* stats, void* stream) {
  if (!s || !A || ((uintptr_t)A & 15)) return MBO_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  mbo_status rc = surface_diffusion(s, A, s->At, st);
  if (rc != MBO_OK) return rc;
  SCK(cudaMemsetAsync(s->st, 0, sizeof(SurfStats), st));
  SCK(timed(s, 3, st, [&] {
    return s->dtype == MBO_F32 ? launch_project<float>(s, A, st) : launch_project<double>(s, A, st);
  }));
  if (stats) {
    SCK(cudaMemcpyAsync(s->h_st, s->st, sizeof(SurfStats), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    double md;
    std::memcpy(&md, &s->h_st->maxd_bits, sizeof(md));
    stats->energy = NAN;
    stats->max_delta = md;
    stats->det_flips = (int64_t)s->h_st->flips;
    stats->fallback_points = (int64_t)s->h_st->fallback;
    stats->nonfinite = (int64_t)s->h_st->nonfinite;
    if (stats->nonfinite) {
      snprintf(s->err, sizeof(s->err), "non-finite values in the projected field");
      return MBO_ERR_NUMERIC;
    }
  }
  return MBO_OK;
}

mbo_status mbo_surface_step_volume(mbo_surface s, void* A, double volume, mbo_stats* stats, void* stream) {
  if (!s || !A || ((uintptr_t)A & 15) || std::isnan(volume)) return MBO_ERR_INVALID_ARG;
  if (s->n > 3) return sfail(s, MBO_ERR_UNSUPPORTED_SIZE, "%s", "the volume-preserving step supports n <= 3");
  const size_t elem = s->dtype == MBO_F32 ? 4 : 8;
  const size_t fbytes = (size_t)s->C * (size_t)s->nq * elem;
  if (!s->Au) {
    // fixed-point weights: w_q scaled so that all of them sum to 2^62
    long double tot = 0;
    for (double w : s->hw) {
      if (!(w >= 0)) return sfail(s, MBO_ERR_INVALID_ARG, "%s", "the volume step needs weights w_q >= 0");
      tot += w;
    }
    if (!(tot > 0)) return sfail(s, MBO_ERR_INVALID_ARG, "%s", "the volume step needs a positive total weight");
    s->wscale = (double)(std::ldexp(1.0L, 62) / tot);
    std::vector<unsigned long long> wf(s->nq);
    for (long long q = 0; q < s->nq; ++q) wf[q] = (unsigned long long)((long double)s->hw[q] * s->wscale);
    // all buffers or none: a failed call leaves the plan as it was
    void* au = nullptr;
    void* keys = nullptr;
    void* ss = nullptr;
    void* ws = nullptr;
    void* w = nullptr;
    cudaError_t e = cudaMalloc(&au, fbytes);
    if (e == cudaSuccess) e = cudaMalloc(&keys, (size_t)s->nq * sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMalloc(&ss, sizeof(SelectState));
    if (e == cudaSuccess) e = cudaMalloc(&ws, sizeof(WSelect));
    if (e == cudaSuccess) e = cudaMalloc(&w, (size_t)s->nq * sizeof(unsigned long long));
    if (e == cudaSuccess)
      e = cudaMemcpy(w, wf.data(), (size_t)s->nq * sizeof(unsigned long long), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      void* bufs[] = {au, keys, ss, ws, w};
      for (void* b : bufs)
        if (b) cudaFree(b);
      return sfail(s, e == cudaErrorMemoryAllocation ? MBO_ERR_OOM : MBO_ERR_CUDA, "%s", cudaGetErrorString(e));
    }
    s->Au = au;
    s->vkeys = static_cast<unsigned long long*>(keys);
    s->vss = static_cast<SelectState*>(ss);
    s->vws = static_cast<WSelect*>(ws);
    s->vw = static_cast<unsigned long long*>(w);
    s->bytes += fbytes + (size_t)s->nq * 16 + sizeof(SelectState) + sizeof(WSelect);
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the diffused field in the caller's order; the previous field kept for the statistics
  mbo_status rc = surface_diffusion(s, A, s->Au, st);
  if (rc != MBO_OK) return rc;
  SCK(cudaMemcpyAsync(s->At, A, fbytes, cudaMemcpyDeviceToDevice, st));
  // dE keys (the flat-torus volume step's kernels, on the nq points), the
  // weighted selection of Algorithm 3, class assignment
  Geom g{};
  g.P = s->nq;
  g.n = s->n;
  g.C = s->C;
  const StatsPtrs none{};
  const int blocks = (int)std::min<long long>((s->nq + 255) / 256, 152 * 16);
  auto vol = [&](VolumePass which) {
    return s->dtype == MBO_F32
               ? launch_volume<float>(which, g, static_cast<const float*>(s->Au), static_cast<float*>(A),
                                      s->vkeys, s->vss, none, 0.0, blocks, st)
               : launch_volume<double>(which, g, static_cast<const double*>(s->Au), static_cast<double*>(A),
                                       s->vkeys, s->vss, none, 0.0, blocks, st);
  };
  SCK(vol(VP_DELTA));
  if (volume < 0) {
    SCK(cudaMemsetAsync(&s->vws->target, 0, sizeof(unsigned long long), st));
#define MBO_WVOL(T, NM)                                                                              \
  k_wvolume<T, NM><<<blocks, 256, 0, st>>>(static_cast<const T*>(A), s->vw, s->nq, s->vws)
    if (s->dtype == MBO_F32) {
      if (s->n == 1) MBO_WVOL(float, 1); else if (s->n == 2) MBO_WVOL(float, 2); else MBO_WVOL(float, 3);
    } else {
      if (s->n == 1) MBO_WVOL(double, 1); else if (s->n == 2) MBO_WVOL(double, 2); else MBO_WVOL(double, 3);
    }
#undef MBO_WVOL
    k_wselect_init<<<1, 256, 0, st>>>(s->vws, 0, 0);
  } else {
    const long double t = std::min((long double)volume * s->wscale, std::ldexp(1.0L, 63));
    k_wselect_init<<<1, 256, 0, st>>>(s->vws, (unsigned long long)std::llround((double)t), 1);
  }
  for (int d = 0; d < 12; ++d) {
    k_wselect_hist<<<blocks, 256, 0, st>>>(s->vkeys, s->vw, s->nq, s->vws, d);
    k_wselect_pick<<<1, 32, 0, st>>>(s->vws, s->vss, d);
  }
  SCK(cudaGetLastError());
  SCK(vol(VP_ASSIGN));
  SCK(cudaMemsetAsync(s->st, 0, sizeof(SurfStats), st));
  const unsigned pb = (unsigned)((s->nq + kProjThreads - 1) / kProjThreads);
#define MBO_SDELTA(T, NM)                                                                   \
  k_sdelta<T, NM><<<pb, kProjThreads, 0, st>>>(static_cast<const T*>(s->At), static_cast<const T*>(A), s->nq, s->st)
  if (s->dtype == MBO_F32) {
    if (s->n == 1) MBO_SDELTA(float, 1); else if (s->n == 2) MBO_SDELTA(float, 2); else MBO_SDELTA(float, 3);
  } else {
    if (s->n == 1) MBO_SDELTA(double, 1); else if (s->n == 2) MBO_SDELTA(double, 2); else MBO_SDELTA(double, 3);
  }
#undef MBO_SDELTA
  SCK(cudaGetLastError());
  if (stats) {
    SCK(cudaMemcpyAsync(s->h_st, s->st, sizeof(SurfStats), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    double md;
    std::memcpy(&md, &s->h_st->maxd_bits, sizeof(md));
    stats->energy = NAN;
    stats->max_delta = md;
    stats->det_flips = (int64_t)s->h_st->flips;
    stats->fallback_points = 0;
    stats->nonfinite = (int64_t)s->h_st->nonfinite;
    if (stats->nonfinite) {
      snprintf(s->err, sizeof(s->err), "non-finite values in the assigned field");
      return MBO_ERR_NUMERIC;
    }
  }
  return MBO_OK;
}

mbo_status mbo_surface_profile_enable(mbo_surface s, int enable) {
  if (!s) return MBO_ERR_INVALID_ARG;
  for (auto& p : s->pending) {
    cudaEventSynchronize(p.b);
    s->ev_free.push_back(p.a);
    s->ev_free.push_back(p.b);
  }
  s->pending.clear();
  for (int i = 0; i < MBO_SURFACE_PROFILE_PASSES; ++i) {
    s->prof_ms[i] = 0;
    s->prof_n[i] = 0;
  }
  s->prof = enable != 0;
  return MBO_OK;
}

mbo_status mbo_surface_profile_read(mbo_surface s, double* ms, int64_t* launches, int npass) {
  if (!s || npass < 0) return MBO_ERR_INVALID_ARG;
  for (auto& p : s->pending) {
    SCK(cudaEventSynchronize(p.b));
    float t = 0.f;
    SCK(cudaEventElapsedTime(&t, p.a, p.b));
    s->prof_ms[p.pass] += t;
    s->prof_n[p.pass] += 1;
    s->ev_free.push_back(p.a);
    s->ev_free.push_back(p.b);
  }
  s->pending.clear();
  for (int i = 0; i < npass && i < MBO_SURFACE_PROFILE_PASSES; ++i) {
    if (ms) ms[i] = s->prof_ms[i];
    if (launches) launches[i] = s->prof_n[i];
  }
  return MBO_OK;
}

int64_t mbo_surface_workspace_bytes(mbo_surface s) {
  if (!s) return -1;
  return (int64_t)s->bytes + (s->fine ? mbo_workspace_bytes(s->fine) : 0);
}

const char* mbo_surface_last_error(mbo_surface s) { return s ? s->err : "null plan"; }

}  // extern "C"
