// FP32 diffusion on the oversampled grid of the closed-surface path (Algorithm 2,
// steps 4 and 5, between the non-uniform sums): forward FFT of the nf^3 grid,
// per-axis multiplier, inverse FFT.
//
// Two thirds of every axis take no part: by the choice of h all points lie in
// the middle half of an axis, so the grid is zero outside a box of about
// (nf/2 + W)^3 points and only its values are read back; and the multiplier is
// zero beyond the M modes, half of an axis again (nf >= 4M).  So a pass transforms
// only the lines that cross the box on the axes still in space and the modes on
// the axes already transformed, reads the part of a line that is not zero, and
// writes the part the next pass uses:
//   box_row  fwd   rows of the box in x         -> modes kx      W1[q][z][y][kx]
//   box_axis FWD   y lines of the box's z       -> modes ky      W2[q][z][ky][kx]
//   box_axis FGI   z lines of every (kx, ky): forward, multiplier, inverse, in place
//   box_axis INV   y lines back                                  W1
//   box_row  inv   rows back to the box
// About a quarter of the lines of the full grid per pass, and with compact
// arrays (box and modes only) the 192^3 grid of the paper's sphere takes 40 MB
// and its two workspaces 45 MB each, within L2, instead of 255 and 283 MB:
// 1.23 ms for the whole grid, 0.254 ms.  The line transforms are the in-place
// network of mbo_dev.cuh; spectra leave it digit-reversed, and the passes store
// mode a (natural order: 0 .. M, -M .. -1) from position kpos[a].
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/mbo.h"
#include "mbo_kernels.cuh"

namespace mbo {
namespace {

// The part of the periodic nf^3 grid that holds every footprint: points
// b0 .. b0 + bn - 1 per axis (x, y, z; wrapping only where it is the whole
// axis), x fastest.
struct GridBox {
  int b0[3], bn[3];
  __host__ __device__ long long points() const { return (long long)bn[0] * bn[1] * bn[2]; }
};

struct BoxDiffusion {
  GridBox box;
  int nf, C, Q;
  int na, NA;         // modes per axis, and the row pitch of W1 and W2 (a multiple of 8)
  int xlast;          // modes kx the last plane keeps (its x spectrum is Hermitian for odd C)
  Plan plan;
  const float2* tw;   // stage twiddles
  const int* kpos;    // mode a -> position in the digit-reversed spectrum
  const float* mult;  // multiplier of mode a
  const float* multp; // multiplier by position
  float inv_p;        // 1 / nf^3
  float2 *W1, *W2;
  void* tabs;
  int row_threads;
};

// One row (y, z) of the box, all complex planes.
template <int NM, bool INV>
__global__ void __launch_bounds__(256) k_box_row(BoxDiffusion b, float* F) {
  constexpr int C = NM * NM, Q = (C + 1) / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  const RowLayout lay{row_pad(b.nf)};
  const int tid = threadIdx.x, T = blockDim.x;
  const int bx = b.box.bn[0], x0 = b.box.b0[0];
  const long long P = b.box.points();
  const long long row = blockIdx.x;  // z * by + y
  const long long rows = (long long)b.box.bn[1] * b.box.bn[2];
  float* f = F + row * bx;
  float2* w = b.W1 + row * b.NA;
  const long long wq = rows * b.NA;
  if (!INV) {
#pragma unroll
    for (int q = 0; q < Q; ++q)
      for (int x = tid; x < b.nf; x += T) {
        const int i = x - x0;
        float2 z = make_float2(0.f, 0.f);
        if ((unsigned)i < (unsigned)bx) {
          z.x = f[(2 * q) * P + i];
          if (2 * q + 1 < C) z.y = f[(2 * q + 1) * P + i];
        }
        s[lay.addr(q, x)] = z;
      }
    __syncthreads();
    fft_fwd(s, lay, b.nf, Q, b.plan, b.tw);
    for (int a = tid; a < b.na; a += T) {
      const int p = b.kpos[a];
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (q < Q - 1 || a < b.xlast) w[q * wq + a] = s[lay.addr(q, p)];
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < Q; ++q)
    for (int x = tid; x < b.nf; x += T) s[lay.addr(q, x)] = make_float2(0.f, 0.f);
  __syncthreads();
  for (int a = tid; a < b.na; a += T) {
    const int p = b.kpos[a];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float2 z;
      if (q < Q - 1 || a < b.xlast) {
        z = w[q * wq + a];
      } else {  // mode -k of a real channel's row
        z = w[q * wq + (b.na - a)];
        z.y = -z.y;
      }
      s[lay.addr(q, p)] = z;
    }
  }
  __syncthreads();
  fft_inv(s, lay, b.nf, Q, b.plan, b.tw);
  for (int i = tid; i < bx; i += T) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const float2 z = s[lay.addr(q, x0 + i)];
      f[(2 * q) * P + i] = z.x;
      if (2 * q + 1 < C) f[(2 * q + 1) * P + i] = z.y;
    }
  }
}

// A tile of eight kx columns along y (FWD, INV; outer index z of the box) or z
// (FGI; outer index ky).
constexpr int kBoxTx = 8, kBoxLtx = 3, kBoxThreads = 128;
template <int MODE> __global__ void __launch_bounds__(kBoxThreads) k_box_axis(BoxDiffusion b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  const ColLayout lay{kBoxLtx};
  const int by = b.box.bn[1], bz = b.box.bn[2], NA = b.NA, nf = b.nf;
  const int nouter = MODE == AXIS_FGI ? b.na : bz;
  const int xt = NA / kBoxTx, xtl = (b.xlast + kBoxTx - 1) / kBoxTx;
  const int full = (b.Q - 1) * nouter * xt;
  int t = blockIdx.x, q, o, x;
  if (t < full) {
    q = t / (nouter * xt);
    t -= q * nouter * xt;
    o = t / xt;
    x = (t - o * xt) * kBoxTx;
  } else {
    q = b.Q - 1;
    t -= full;
    o = t / xtl;
    x = (t - o * xtl) * kBoxTx;
  }
  const int tid = threadIdx.x, c = tid & (kBoxTx - 1), p0 = tid >> kBoxLtx;
  constexpr int DP = kBoxThreads / kBoxTx;
  x += c;
  const long long pl1 = (long long)bz * by * NA, pl2 = (long long)bz * b.na * NA;  // plane strides
  // lines: element p of the box part, or mode a
  float2* y1 = b.W1 + q * pl1 + ((long long)o * by) * NA + x;    // + p NA (y of the box)
  float2* y2 = b.W2 + q * pl2 + ((long long)o * b.na) * NA + x;  // + a NA (modes ky)
  float2* zl = b.W2 + q * pl2 + (long long)o * NA + x;           // + p na NA (z of the box)
  const long long zs = (long long)b.na * NA;
  if (MODE == AXIS_INV) {
    for (int p = p0; p < nf; p += DP) s[lay.addr(c, p)] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int a = p0; a < b.na; a += DP) s[lay.addr(c, b.kpos[a])] = y2[(long long)a * NA];
  } else {
    const int l0 = MODE == AXIS_FGI ? b.box.b0[2] : b.box.b0[1];
    const int ln = MODE == AXIS_FGI ? bz : by;
    for (int p = p0; p < nf; p += DP) {
      const int i = p - l0;
      const bool in = (unsigned)i < (unsigned)ln;
      float2 z = make_float2(0.f, 0.f);
      if (in) z = MODE == AXIS_FGI ? zl[i * zs] : y1[(long long)i * NA];
      s[lay.addr(c, p)] = z;
    }
  }
  __syncthreads();
  if (MODE != AXIS_INV) fft_fwd(s, lay, nf, kBoxTx, b.plan, b.tw);
  if (MODE == AXIS_FWD) {
    for (int a = p0; a < b.na; a += DP) y2[(long long)a * NA] = s[lay.addr(c, b.kpos[a])];
    return;
  }
  if (MODE == AXIS_FGI) {
    const float fo = (x < b.na ? b.mult[x] : 0.f) * b.mult[o] * b.inv_p;
    for (int p = p0; p < nf; p += DP) {
      const int e = lay.addr(c, p);
      const float2 z = s[e];
      const float f = fo * b.multp[p];
      s[e] = make_float2(z.x * f, z.y * f);
    }
    __syncthreads();
  }
  fft_inv(s, lay, nf, kBoxTx, b.plan, b.tw);
  if (MODE == AXIS_FGI) {
    for (int i = p0; i < bz; i += DP) zl[i * zs] = s[lay.addr(c, b.box.b0[2] + i)];
  } else {
    for (int i = p0; i < by; i += DP) y1[(long long)i * NA] = s[lay.addr(c, b.box.b0[1] + i)];
  }
}

inline cudaError_t box_axis_smem(size_t bytes) {
  static SmemLimit axis[3];
  cudaError_t e = raise_smem(k_box_axis<AXIS_FWD>, bytes, axis[0]);
  if (e == cudaSuccess) e = raise_smem(k_box_axis<AXIS_FGI>, bytes, axis[1]);
  if (e == cudaSuccess) e = raise_smem(k_box_axis<AXIS_INV>, bytes, axis[2]);
  return e;
}

template <int NM> cudaError_t box_run(const BoxDiffusion& b, float* F, cudaStream_t st) {
  const size_t rs = (size_t)b.Q * row_pad(b.nf) * sizeof(float2);
  const size_t as = (size_t)row_pad(b.nf) * kBoxTx * sizeof(float2);
  static SmemLimit row[2];
  cudaError_t e = raise_smem(k_box_row<NM, false>, rs, row[0]);
  if (e == cudaSuccess) e = raise_smem(k_box_row<NM, true>, rs, row[1]);
  if (e == cudaSuccess) e = box_axis_smem(as);
  if (e != cudaSuccess) return e;
  const unsigned rows = (unsigned)(b.box.bn[1] * b.box.bn[2]);
  const unsigned cols = (unsigned)((b.Q - 1) * (b.NA / kBoxTx) + (b.xlast + kBoxTx - 1) / kBoxTx);
  k_box_row<NM, false><<<rows, b.row_threads, rs, st>>>(b, F);
  k_box_axis<AXIS_FWD><<<cols * b.box.bn[2], kBoxThreads, as, st>>>(b);
  k_box_axis<AXIS_FGI><<<cols * b.na, kBoxThreads, as, st>>>(b);
  k_box_axis<AXIS_INV><<<cols * b.box.bn[2], kBoxThreads, as, st>>>(b);
  k_box_row<NM, true><<<rows, b.row_threads, rs, st>>>(b, F);
  return cudaGetLastError();
}

// F <- the diffused values at the box's points (C channels, as GridBox lays them out).
inline cudaError_t box_diffuse(const BoxDiffusion& b, float* F, cudaStream_t st) {
  switch (b.C) {
    case 1: return box_run<1>(b, F, st);
    case 4: return box_run<2>(b, F, st);
    case 9: return box_run<3>(b, F, st);
    default: return box_run<4>(b, F, st);
  }
}

// Tables and workspaces; mult: nf values in natural frequency order, zero beyond
// |k| = M.  maxsm: shared bytes a block may have; bytes: device bytes, added to.
inline mbo_status box_create(BoxDiffusion& b, const GridBox& box, int nf, int n, int M, const double* mult,
                             int maxsm, size_t& bytes) {
  b.box = box;
  b.nf = nf;
  b.C = n * n;
  b.Q = (b.C + 1) / 2;
  b.na = std::min(2 * M + 1, nf);
  b.NA = (b.na + kBoxTx - 1) / kBoxTx * kBoxTx;
  b.xlast = (b.C & 1) && b.na == 2 * M + 1 ? M + 1 : b.na;
  b.plan = make_plan(nf);
  b.inv_p = (float)(1.0 / ((double)nf * nf * nf));
  // a thread per butterfly of a radix-12 stage
  b.row_threads = std::max(64, std::min(256, (b.Q * nf / 12 + 31) / 32 * 32));
  if ((size_t)b.Q * row_pad(nf) * sizeof(float2) > (size_t)maxsm ||
      (size_t)row_pad(nf) * kBoxTx * sizeof(float2) > (size_t)maxsm)
    return MBO_ERR_UNSUPPORTED_SIZE;
  const int ntw = std::max(plan_twiddles(b.plan), 1);
  std::vector<float> tab(2 * (size_t)ntw + 2 * (size_t)nf, 0.f);  // twiddles | mult of mode a | by position
  std::vector<int> kpos(nf, 0);
  for (int i = 0; i < b.plan.nst; ++i) {
    const Stage& s = b.plan.st[i];
    if (s.m <= 1) continue;
    for (int n1 = 0; n1 < s.m; ++n1)
      for (int j = 1; j < s.rad; ++j) {
        const double ang = 2.0 * M_PI * (double)(((long long)n1 * j) % s.lb) / (double)s.lb;
        const size_t at = 2 * ((size_t)s.tw + (size_t)(j - 1) * s.m + n1);
        tab[at] = (float)std::cos(ang);
        tab[at + 1] = (float)(-std::sin(ang));
      }
  }
  std::vector<int> pos;
  digit_positions(b.plan, nf, pos);
  float* ma = &tab[2 * (size_t)ntw];
  float* mp = ma + nf;
  for (int k = 0; k < nf; ++k) mp[pos[k]] = (float)mult[k];
  for (int a = 0; a < b.na; ++a) {
    const int k = b.na < nf && a > M ? a - b.na + nf : a;
    kpos[a] = pos[k];
    ma[a] = (float)mult[k];
  }
  const size_t w1 = (size_t)b.Q * box.bn[2] * box.bn[1] * b.NA * sizeof(float2);
  const size_t w2 = (size_t)b.Q * box.bn[2] * b.na * b.NA * sizeof(float2);
  const size_t tb = tab.size() * sizeof(float) + kpos.size() * sizeof(int);
  if (cudaMalloc(&b.tabs, tb) != cudaSuccess || cudaMalloc((void**)&b.W1, w1) != cudaSuccess ||
      cudaMalloc((void**)&b.W2, w2) != cudaSuccess)
    return MBO_ERR_OOM;
  bytes += w1 + w2 + tb;
  // the padding columns past the modes are transformed with the others: start them at zero
  if (cudaMemset(b.W1, 0, w1) != cudaSuccess || cudaMemset(b.W2, 0, w2) != cudaSuccess ||
      cudaMemcpy(b.tabs, tab.data(), tab.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy((char*)b.tabs + tab.size() * sizeof(float), kpos.data(), kpos.size() * sizeof(int),
                 cudaMemcpyHostToDevice) != cudaSuccess)
    return MBO_ERR_CUDA;
  const float* d = static_cast<const float*>(b.tabs);
  b.tw = reinterpret_cast<const float2*>(d);
  b.mult = d + 2 * (size_t)ntw;
  b.multp = b.mult + nf;
  b.kpos = reinterpret_cast<const int*>(d + tab.size());
  return MBO_OK;
}

}  // namespace
}  // namespace mbo
