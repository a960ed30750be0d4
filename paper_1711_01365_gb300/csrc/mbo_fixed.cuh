// FP64 transforms in 64-bit fixed point.
//
// GB300 issues FP64 at 1/64 of the FP32 rate (measured: 1.96 DFMA lanes per
// clock and SM), and integers at half of it (50 64-bit additions per clock and
// SM, 22 32x32 -> 64 multiply-adds).  A transform is two thirds additions, so the
// FP64 passes run it on integers: the in-place network of mbo_dev.cuh with
// complex elements of two int64 on a common power-of-two scale.
//
//   Scale.  Every partial sum of a DFT is at most the L1 norm of its input, so
//   a sequence scaled to an L1 norm just under 2^62 cannot overflow, whatever it
//   holds.  A flat sequence of N points then keeps 62 - log2 N bits over its RMS
//   at the input and gains half a bit per doubling on the way, so the first
//   stage is where rounding would show; a stage of radix r needs room for r
//   times the largest entry only, so the input takes the scale of that and the
//   first stage shifts its results down to the norm's.  The relative error of a
//   transform is then below the FP64 network's (RMS, flat input: 1024 points
//   0.6e-16 against 2.0e-16, 2048 points 0.9e-16 against 2.3e-16).  Norm and largest
//   entry are taken in FP32 (a scale needs an exponent), one scale per
//   sequence: per (row, plane) in the x pass and per column in the strided
//   passes, which take a second one between multiplier and inverse.  Fields that
//   come from the projection have entries in [-1, 1]: their forward transform
//   takes a fixed scale.
//   Products.  Twiddles are Q60 in limbs of 29 + 31 bits, elements are split
//   into 31 + 31 bits, so a real product is a high product, two cross products
//   and the upper word of the low one; a complex product sums the cross terms
//   of both parts before the one rounding shift.
//   Range.  Any finite input is accepted, subnormals included: norms outside the
//   FP32 range take a slower pass that scales by the largest exponent first, and
//   results below 2^-1022 are rounded to subnormals as FP64 does.  A sequence with a
//   non-finite entry gives NaN throughout, as a floating-point DFT does.
//   W stays in FP64 between the passes.
#pragma once
#include <cmath>

#include "mbo_kernels.cuh"

namespace mbo {

struct alignas(16) fx2 {
  long long x, y;
};
// Limbs of an element part, |x| < 2^62.
struct FxL {
  int h;       // x >> 31
  unsigned l;  // low 31 bits
};
__device__ __forceinline__ FxL fx_limbs(long long x) { return FxL{(int)(x >> 31), (unsigned)x & 0x7fffffffu}; }

// round((a . c)) for the Q60 constant c = (ch 2^31 + cl) / 2^60
__device__ __forceinline__ long long fx_mul(FxL a, int ch, int cl) {
  const long long hh = (long long)a.h * ch;
  const long long mid = (long long)a.h * cl + (long long)(int)a.l * ch +
                        (long long)(unsigned)__umulhi(a.l, (unsigned)cl << 1);
  return (hh << 2) + ((mid + (1ll << 28)) >> 29);
}

// round(a f 2^e) for f in Q60, where the result stays below 2^62: for e > 0 the
// shift takes in the bits a plain product would round away
__device__ __forceinline__ long long fx_mul_shift(FxL a, long long f, int e) {
  const int ch = (int)(f >> 31), cl = (int)(f & 0x7fffffff);
  const long long hh = (long long)a.h * ch;
  const long long mid = (long long)a.h * cl + (long long)(int)a.l * ch +
                        (long long)(unsigned)__umulhi(a.l, (unsigned)cl << 1);
  if (e <= 0) {
    const long long r = (hh << 2) + ((mid + (1ll << 28)) >> 29);
    return e < -62 ? 0 : e == 0 ? r : (r + (1ll << (-e - 1))) >> -e;
  }
  if (e < 29) return (hh << (2 + e)) + ((mid + (1ll << (28 - e))) >> (29 - e));
  return e > 92 ? 0 : ((hh << 31) + mid) << (e - 29);  // beyond 92 only zeros have room
}

// a t, t = (c, s): (x c - y s, x s + y c).  With |(x, y)| < 2^62 the cross terms
// of both products sum to less than 2^63 (2^31 (|xh| + |yh|) <= sqrt(2) 2^62 and
// 2^29 (xl + yl) <= 2^61).
__device__ __forceinline__ fx2 fx_cmul(fx2 a, int ch, int cl, int sh, int sl) {
  const FxL x = fx_limbs(a.x), y = fx_limbs(a.y);
  const unsigned cl2 = (unsigned)cl << 1, sl2 = (unsigned)sl << 1;
  const int lre = (int)__umulhi(x.l, cl2) - (int)__umulhi(y.l, sl2);
  const unsigned lim = __umulhi(x.l, sl2) + __umulhi(y.l, cl2);
  const long long hre = (long long)x.h * ch + (long long)y.h * -sh;
  const long long him = (long long)x.h * sh + (long long)y.h * ch;
  const long long mre = (long long)x.h * cl + (long long)(int)x.l * ch + (long long)y.h * -sl +
                        (long long)(int)y.l * -sh + (long long)lre;
  const long long mim = (long long)x.h * sl + (long long)(int)x.l * sh + (long long)y.h * cl +
                        (long long)(int)y.l * ch + (long long)lim;
  return fx2{(hre << 2) + ((mre + (1ll << 28)) >> 29), (him << 2) + ((mim + (1ll << 28)) >> 29)};
}

// Constants in Q60, round(2^60 cos or sin).
constexpr long long kFxC8 = 815238614083298888ll;     // cos(pi/4)
constexpr long long kFxC16 = 1065160580698383124ll;   // cos(pi/8)
constexpr long long kFxS16 = 441203958630471860ll;    // sin(pi/8)
constexpr long long kFxS3 = 998459311558907194ll;     // sin(pi/3)
constexpr long long kFxC9a = 883189111956446361ll, kFxS9a = 741083658102443606ll;     // 2 pi/9
constexpr long long kFxC9b = 200202718267994420ll, kFxS9b = 1135406036351323053ll;    // 4 pi/9
constexpr long long kFxC9d = -1083391830224440781ll, kFxS9d = 394322378248879447ll;   // 8 pi/9

// a exp(-i angle) for constants c = cos, s = sin of it
__device__ __forceinline__ fx2 fx_rot(fx2 a, long long c, long long s) {
  const FxTw t = fx_tw(c, -s);
  return fx_cmul(a, t.ch, t.cl, t.sh, t.sl);
}
// a exp(-i pi/4) and a exp(-3 i pi/4)
__device__ __forceinline__ fx2 fx_rot8(fx2 a) {
  const FxTw t = fx_tw(kFxC8, 0);
  const long long x = fx_mul(fx_limbs(a.x), t.ch, t.cl), y = fx_mul(fx_limbs(a.y), t.ch, t.cl);
  return fx2{x + y, y - x};
}
__device__ __forceinline__ fx2 fx_rot83(fx2 a) {
  const FxTw t = fx_tw(kFxC8, 0);
  const long long x = fx_mul(fx_limbs(a.x), t.ch, t.cl), y = fx_mul(fx_limbs(a.y), t.ch, t.cl);
  return fx2{y - x, -x - y};
}

// The register DFTs of mbo_dev.cuh that multiply, forward.
template <int DIR> __device__ __forceinline__ void dft3(fx2* v) {
  static_assert(DIR < 0, "forward");
  const fx2 s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
  const fx2 t1 = fx2{v[0].x - ((s.x + 1) >> 1), v[0].y - ((s.y + 1) >> 1)};
  const FxTw t = fx_tw(kFxS3, 0);
  const fx2 hd = fx2{fx_mul(fx_limbs(d.x), t.ch, t.cl), fx_mul(fx_limbs(d.y), t.ch, t.cl)};
  v[0] = cadd(v[0], s);
  v[1] = cadd_i<-1>(t1, hd);
  v[2] = csub_i<-1>(t1, hd);
}
template <int DIR> __device__ __forceinline__ void dft8(fx2* v) {
  static_assert(DIR < 0, "forward");
  fx2 e[4] = {v[0], v[2], v[4], v[6]};
  fx2 o[4] = {v[1], v[3], v[5], v[7]};
  dft4<-1>(e);
  dft4<-1>(o);
  o[1] = fx_rot8(o[1]);
  o[3] = fx_rot83(o[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (k == 2) {
      v[2] = cadd_i<-1>(e[2], o[2]);
      v[6] = csub_i<-1>(e[2], o[2]);
    } else {
      v[k] = cadd(e[k], o[k]);
      v[k + 4] = csub(e[k], o[k]);
    }
  }
}
template <int DIR> __device__ __forceinline__ void dft16(fx2* v) {
  static_assert(DIR < 0, "forward");
  fx2 e[8], o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    e[k] = v[2 * k];
    o[k] = v[2 * k + 1];
  }
  dft8<-1>(e);
  dft8<-1>(o);
  o[1] = fx_rot(o[1], kFxC16, kFxS16);
  o[2] = fx_rot8(o[2]);
  o[3] = fx_rot(o[3], kFxS16, kFxC16);
  o[5] = fx_rot(o[5], -kFxS16, kFxC16);
  o[6] = fx_rot83(o[6]);
  o[7] = fx_rot(o[7], -kFxC16, kFxS16);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    if (k == 4) {
      v[4] = cadd_i<-1>(e[4], o[4]);
      v[12] = csub_i<-1>(e[4], o[4]);
    } else {
      v[k] = cadd(e[k], o[k]);
      v[k + 8] = csub(e[k], o[k]);
    }
  }
}
template <int DIR> __device__ __forceinline__ void dft9(fx2* v) {
  static_assert(DIR < 0, "forward");
  fx2 u[3][3];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) u[n2][n1] = v[n2 + 3 * n1];
    dft3<-1>(u[n2]);
  }
  u[1][1] = fx_rot(u[1][1], kFxC9a, kFxS9a);
  u[1][2] = fx_rot(u[1][2], kFxC9b, kFxS9b);
  u[2][1] = fx_rot(u[2][1], kFxC9b, kFxS9b);
  u[2][2] = fx_rot(u[2][2], kFxC9d, kFxS9d);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    fx2 a[3] = {u[0][k1], u[1][k1], u[2][k1]};
    dft3<-1>(a);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = a[k2];
  }
}

// One stage of the network (see radix_stage in mbo_dev.cuh).  An inverse
// transform works on elements with their parts swapped: swapping the parts
// before and after turns a forward DFT into an inverse one, so both directions
// share the forward butterflies and twiddles, and only the twiddles' place
// differs (after the butterfly, or in the transposed inverse before it).  The
// two-turn loop keeps one copy of either in the instruction cache, which a
// small field's step otherwise spends its time filling.  drop (first stage
// only): bits the results are shifted down by, per sequence.
template <int RAD, class L>
__device__ __forceinline__ void radix_stage_fx(fx2* s, const L& lay, int N, int M, const Stage& sd,
                                               const FxTw* __restrict__ tw, bool inv, const int* drop) {
  const int NR = N / RAD;
  const int m = sd.m, lb = sd.lb, ps = sd.pstride;
  const unsigned B = (unsigned)(NR * M);
  const FxTw* __restrict__ tws = tw + sd.tw;
  const int da = lay.at(0, ps);  // the affine stride in layout units
  for (unsigned u = threadIdx.x; u < B; u += blockDim.x) {
    int seq, w;
    if constexpr (L::kColumns) {
      seq = (int)(u & ((1u << lay.ltx) - 1));
      w = (int)(u >> lay.ltx);
    } else {
      seq = (int)fdiv(sd.dnr, u);
      w = (int)u - seq * NR;
    }
    const int b = (int)fdiv(sd.dm, (unsigned)w);
    const int n1 = w - b * m;
    const int base = b * lb + n1;
    int a[RAD];
    if (ps) {
      const int a0 = lay.addr(seq, base);
#pragma unroll
      for (int j = 0; j < RAD; ++j) a[j] = a0 + j * da;
    } else {
#pragma unroll
      for (int j = 0; j < RAD; ++j) a[j] = lay.addr(seq, base + j * m);
    }
    fx2 v[RAD];
#pragma unroll
    for (int j = 0; j < RAD; ++j) v[j] = s[a[j]];
#pragma unroll 1
    for (int turn = 0; turn < 2; ++turn) {
      if ((turn == 0) != inv) {
        dft<-1, RAD>(v);
      } else if (m > 1) {
        const FxTw* t = tws + n1;
#pragma unroll
        for (int j = 1; j < RAD; ++j) {
          const int4 c = __ldg(reinterpret_cast<const int4*>(&t[(j - 1) * m]));
          v[j] = fx_cmul(v[j], c.x, c.y, c.z, c.w);
        }
      }
    }
    if (drop) {
      const int d = drop[seq];
      const long long half = (1ll << d) >> 1;
#pragma unroll
      for (int j = 0; j < RAD; ++j) v[j] = fx2{(v[j].x + half) >> d, (v[j].y + half) >> d};
    }
#pragma unroll
    for (int j = 0; j < RAD; ++j) s[a[j]] = v[j];
  }
  __syncthreads();
}

// Forward transform, or inverse of a digit-reversed spectrum with swapped parts
// (both unnormalised); the inverse's first stage is the plan's last.
template <class L>
__device__ __noinline__ void fft_fx(fx2* s, L lay, int N, int M, const Plan& pl, const FxTw* __restrict__ tw,
                                    bool inv, const int* drop) {
#pragma unroll 1
  for (int i = 0; i < pl.nst; ++i) {
    const Stage& sd = pl.st[inv ? pl.nst - 1 - i : i];
    const int* d = i ? nullptr : drop;
    switch (sd.rad) {
      case 16: radix_stage_fx<16>(s, lay, N, M, sd, tw, inv, d); break;
      case 12: radix_stage_fx<12>(s, lay, N, M, sd, tw, inv, d); break;
      case 9: radix_stage_fx<9>(s, lay, N, M, sd, tw, inv, d); break;
      case 8: radix_stage_fx<8>(s, lay, N, M, sd, tw, inv, d); break;
      case 6: radix_stage_fx<6>(s, lay, N, M, sd, tw, inv, d); break;
      case 4: radix_stage_fx<4>(s, lay, N, M, sd, tw, inv, d); break;
      case 3: radix_stage_fx<3>(s, lay, N, M, sd, tw, inv, d); break;
      default: radix_stage_fx<2>(s, lay, N, M, sd, tw, inv, d); break;
    }
  }
}

// ---------------------------------------------------------------------------
// Conversions, in integer instructions (the FP64 unit converts a 64-bit integer
// at its own rate: two conversions cost as much as two FP64 operations).
// ---------------------------------------------------------------------------

// round(d 2^k) for |d| 2^k < 2^62 and d zero or normal; k as the scale functions give it.
__device__ __forceinline__ long long fx_from(double d, int k) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const int e = (int)(u >> 52) & 0x7ff;
  // mantissa << 10: 63 bits; the value is mant 2^(e - 1075), so shift right by
  // 10 - (e - 1075 + k) >= 1
  const unsigned long long m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
  const int r = 1085 - e - k;
  if (e == 0 || r > 63) return 0;
  const long long v = (long long)((m + (1ull << (r - 1))) >> r);
  return (long long)u < 0 ? -v : v;
}

// v 2^e rounded to FP64 (overflow to infinity; zero below 2^-1022)
__device__ __forceinline__ double fx_to(long long v, int e) {
  if (v == 0) return 0.0;
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << lz;  // bit 63 set
  const int ex = 63 - lz + e + 1022;     // biased exponent less one: the leading bit adds it
  unsigned long long b = (m >> 11) + ((m >> 10) & 1) + ((unsigned long long)(unsigned)ex << 52);
  if (ex < 0) b = 0;
  if (ex > 2045) b = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull)));
}

// Subnormals occur only in sequences whose scale k is large.  There the values
// are lifted by 2^600 before fx_from and lowered again after fx_to (an FP64 multiply,
// which rounds results below 2^-1022 as FP64 does), each in a loop of its own, so
// that the conversions of ordinary sequences do not test for them (per element
// that took 1 to 4% of a step).
constexpr int kFxBad = 0x7fffffff;  // scale of a sequence with a non-finite entry
constexpr int kFxUp = 600;
__device__ __forceinline__ int fx_lift(int k) { return k > 960 && k != kFxBad ? kFxUp : 0; }
__device__ __forceinline__ void fx_scale2(double2& z, double f) { z = double2{z.x * f, z.y * f}; }

// A part in FP32.
__device__ __forceinline__ float fx_float(long long v) {
  return (float)(int)(v >> 32) * 4294967296.f + (float)(unsigned)v;
}

// A bound of |z| in FP32, without squares (which would leave the FP32 range)
// (at most 8% above, never below; NaN where a part is NaN, so that the sum shows it)
__device__ __forceinline__ float fx_mod(float x, float y) {
  float big;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(big) : "f"(fabsf(x)), "f"(fabsf(y)));
  return big + 0.4142136f * fminf(fabsf(x), fabsf(y));
}

__device__ __forceinline__ bool fx_nonzero(double d) {
  return (((unsigned)__double2hiint(d) << 1) | (unsigned)__double2loint(d)) != 0;
}
// The bound of an entry that norms are summed from: positive for every entry but
// zero, so that a norm is 0 for a sequence of zeros only.  Those are common (dead
// columns of a ragged tile, constant channels, grid outside a surface's points)
// and need no scale.
constexpr float kFxTiny = 1.4e-45f;
__device__ __forceinline__ float fx_norm(double2 z) {
  const float a = fx_mod((float)z.x, (float)z.y);
  return a == 0.f && (fx_nonzero(z.x) || fx_nonzero(z.y)) ? kFxTiny : a;
}

// k such that a bound of s 2^e becomes less than 2^62, with room for the
// roundings of the sum and of the transform (s finite, positive and normal).
__device__ __forceinline__ int fx_scale(float s, int e) { return 61 - ilogbf(s * 1.002f) - e; }
// The scale of a sequence of L1 norm l1 and largest entry mx (both 2^e), and of
// its input where a stage of radix r comes first.
struct FxScale {
  int k, in;
};
__device__ __forceinline__ FxScale fx_scales(float l1, float mx, int e, int r) {
  if (l1 == 0.f) return FxScale{0, 0};
  const int k = fx_scale(l1, e);
  return FxScale{k, max(k, fx_scale(mx * (float)r, e))};
}
// Whether the FP32 norm gives the scale.
__device__ __forceinline__ bool fx_plain(float s) { return s == 0.f || (s > 1e-30f && s < 1e37f); }

constexpr int kFxZero = -2000;  // below every exponent
// floor(log2 |d|) of any d: kFxZero for zeros, 1024 for infinities and NaN
__device__ __forceinline__ int fx_exponent(double d) {
  const unsigned hi = (unsigned)__double2hiint(d) & 0x7fffffffu, lo = (unsigned)__double2loint(d);
  if (hi >= 0x00100000u) return (int)(hi >> 20) - 1023;
  return hi ? -1011 - __clz((int)hi) : lo ? -1043 - __clz((int)lo) : kFxZero;
}

// Scales of one sequence whose FP32 norm is out of range (all threads of the
// block call it; `each(f)` runs f over this thread's entries of the sequence).
// red: 32 words.
template <class Each> __device__ FxScale fx_scale_slow(Each each, int r, unsigned* red) {
  int e = kFxZero;
  each([&](double2 z) { e = max(e, max(fx_exponent(z.x), fx_exponent(z.y))); });
  e = __reduce_max_sync(0xffffffffu, e);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (unsigned)e;
  __syncthreads();
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) e = max(e, (int)red[w]);
  if (e == 1024) return FxScale{kFxBad, 0};
  if (e == kFxZero) return FxScale{0, 0};
  float s = 0.f;
  each([&](double2 z) { s += fx_mod((float)scalbn(z.x, -e), (float)scalbn(z.y, -e)); });
  s = warp_sum(s);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = __float_as_uint(s);
  __syncthreads();
  s = 0.f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += __uint_as_float(red[w]);
  return fx_scales(s, 3.f, e, r);  // parts below 2
}

// ---------------------------------------------------------------------------
// x pass
// ---------------------------------------------------------------------------

// Fixed scale of a projected field's forward transform: parts in [-1, 1], so
// |z| <= sqrt(2) and the sum of N of them stays below 2^(ceil(log2 N) + 1/2).
__device__ __forceinline__ int fx_unit_scale(int N) { return 61 - (32 - __clz(N - 1)); }

// SHORT: the form for few rows of at most 64 points.  There a block's own chain of
// instructions is the time (32^2, n = 3: 2800 a warp, one after another in the one
// warp that a row has points for, each fetched for the first time), so the planes
// are spread over groups of warps, and each group runs one copy of a plane's
// conversions.  Long rows unroll the planes instead: their conversions overlap
// (96^3, n = 3, diffusion: 831 us, 892 with the planes in turn).
template <int NM, int MODE, bool SHORT>
__global__ void __launch_bounds__(kMaxThreads, 1)
k_row_fx(Geom g, Tables<double> t, const double* __restrict__ Ain, double* A, double2* W, StatsPtrs sp) {
  constexpr int C = NM * NM, Q = (C + 1) / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double redd[MODE == ROW_FWD ? 32 : 1];
  __shared__ StatsShared<double, MODE == ROW_INV_PROJECT_FWD ? kMaxThreads : 1> sh;
  __shared__ float rs[2][12][Q];
  __shared__ int drops[Q];
  __shared__ int ks[Q], kins[Q];  // scale exponents of the planes whose norm is out of the FP32 range (SHORT: all)
  __shared__ unsigned slow[32];
  __shared__ int s_flag, s_bad;
  if (sp.respect_stop && *(volatile int*)&sp.st->stop) return;

  double2* sd = reinterpret_cast<double2*>(smem_raw);
  fx2* s = reinterpret_cast<fx2*>(smem_raw);
  const int nx = g.nx;
  const RowLayout lay{row_pad(nx)};
  const long long P = g.P;
  const int T = blockDim.x, tid = threadIdx.x;
  const FxTw* tw = static_cast<const FxTw*>(t.tw[0]);
  // scale exponent of each plane's sequence (SHORT: in ks), less the lift of the planes in `lifted`
  int k[Q] = {};
  unsigned lifted = 0;
  // SHORT: group `grp` of `ng` groups of `gthreads` threads takes planes grp, grp + ng, ...;
  // threads past the last group take none
  const int wpp = (nx + 31) >> 5, ng = SHORT ? max(1, min(Q, (T >> 5) / wpp)) : 1;
  const int gthreads = SHORT ? (ng == 1 ? T : wpp << 5) : T;
  const int grp = SHORT ? tid / gthreads : 0, gt = tid - grp * gthreads;
  // f(q, x) over this thread's share of the planes' entries
  auto visit = [&](auto f) {
    if constexpr (SHORT) {
      if (grp < ng) {
#pragma unroll 1
        for (int q = grp; q < Q; q += ng)
          for (int x = gt; x < nx; x += gthreads) f(q, x);
      }
    } else {
      for (int x = tid; x < nx; x += T) {
#pragma unroll
        for (int q = 0; q < Q; ++q) f(q, x);
      }
    }
  };
  auto scale_of = [&](int q) {
    if constexpr (SHORT) return ks[q];
    else return k[q];
  };

  // scales of the Q sequences in sd, and the sequences converted in place, for
  // a transform whose first stage has radix r (inverse: parts swapped)
  // The slow scales of the planes in `todo` (all threads call it; it ends in a barrier).
  auto slow_scales = [&](unsigned todo, int r) {
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
      if (!(todo >> q & 1)) continue;
      auto points = [&](auto each) {
        for (int x = tid; x < nx; x += T) each(sd[lay.addr(q, x)]);
      };
      const FxScale f = fx_scale_slow(points, r, slow);
      const int up = fx_lift(f.in), down = fx_lift(f.k);
      if (up) points([](double2& z) { fx_scale2(z, 0x1p600); });
      if (down) lifted |= 1u << q;
      if (tid == 0) {
        ks[q] = f.k == kFxBad ? kFxBad : f.k - down;
        kins[q] = f.in - up;
        drops[q] = f.k == kFxBad ? 0 : f.in - f.k;
      }
    }
    __syncthreads();
  };
  auto to_fixed_short = [&](int r, bool swap) {
    const int gw = gthreads >> 5;  // warps of a group
    if (grp < ng) {
#pragma unroll 1
      for (int q = grp; q < Q; q += ng) {
        float n = 0.f, mx = 0.f;
        for (int x = gt; x < nx; x += gthreads) {
          const float a = fx_norm(sd[lay.addr(q, x)]);
          n += a;
          mx = fmaxf(mx, a);
        }
        n = warp_sum(n);
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
        if ((tid & 31) == 0) {
          rs[0][gt >> 5][q] = n;
          rs[1][gt >> 5][q] = __uint_as_float(m);
        }
      }
    }
    __syncthreads();
    // the scales, a thread per plane
    bool plain = true;
    if (tid < Q) {
      float sum = 0.f, top = 0.f;
      for (int w = 0; w < gw; ++w) {
        sum += rs[0][w][tid];
        top = fmaxf(top, rs[1][w][tid]);
      }
      plain = fx_plain(sum);
      const FxScale f = plain ? fx_scales(sum, top, 0, r) : FxScale{0, 0};
      ks[tid] = f.k;
      kins[tid] = f.in;
      drops[tid] = f.in - f.k;
      slow[tid] = plain ? 0u : 1u;
    }
    lifted = 0;
    if (!__syncthreads_and(plain)) {
      unsigned todo = 0;
      for (int q = 0; q < Q; ++q) todo |= slow[q] << q;
      slow_scales(todo, r);
    }
    visit([&](int q, int x) {
      const int a = lay.addr(q, x), kin = kins[q];
      const double2 z = sd[a];
      const long long re = fx_from(z.x, kin), im = fx_from(z.y, kin);
      s[a] = ks[q] == kFxBad ? fx2{0, 0} : swap ? fx2{im, re} : fx2{re, im};
    });
    __syncthreads();
  };
  auto to_fixed_long = [&](int r, bool swap) {
    float n[Q], mx[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) n[q] = mx[q] = 0.f;
    for (int x = tid; x < nx; x += T) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float a = fx_norm(sd[lay.addr(q, x)]);
        n[q] += a;
        mx[q] = fmaxf(mx[q], a);
      }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      n[q] = warp_sum(n[q]);
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx[q]));
      if ((tid & 31) == 0) {
        rs[0][tid >> 5][q] = n[q];
        rs[1][tid >> 5][q] = __uint_as_float(m);
      }
    }
    __syncthreads();
    int kin[Q];
    unsigned todo = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float sum = 0.f, top = 0.f;
      for (int w = 0; w < (T >> 5); ++w) {
        sum += rs[0][w][q];
        top = fmaxf(top, rs[1][w][q]);
      }
      const bool plain = fx_plain(sum);  // the same in every thread
      const FxScale f = plain ? fx_scales(sum, top, 0, r) : FxScale{0, 0};
      todo |= plain ? 0u : 1u << q;
      k[q] = f.k;
      kin[q] = f.in;
      if (tid == 0) drops[q] = f.in - f.k;
    }
    lifted = 0;
    if (todo) {
      slow_scales(todo, r);
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (todo >> q & 1) {
          k[q] = ks[q];
          kin[q] = kins[q];
        }
    }
    for (int x = tid; x < nx; x += T) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int a = lay.addr(q, x);
        const double2 z = sd[a];
        const long long re = fx_from(z.x, kin[q]), im = fx_from(z.y, kin[q]);
        s[a] = k[q] == kFxBad ? fx2{0, 0} : swap ? fx2{im, re} : fx2{re, im};
      }
    }
    __syncthreads();
  };
  auto to_fixed = [&](int r, bool swap) {
    if constexpr (SHORT) to_fixed_short(r, swap);
    else to_fixed_long(r, swap);
  };
  auto from_fixed = [&](fx2 v, int kk) {
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    return kk == kFxBad ? double2{nan, nan} : double2{fx_to(v.x, -kk), fx_to(v.y, -kk)};
  };

  long long off = (long long)blockIdx.x * nx;
  if (MODE == ROW_FWD) {
    double defect = 0.0;
    for (int x = tid; x < nx; x += T) {
      double sq = 0.0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const double re = Ain[(2 * q) * P + off + x];
        const double im = (2 * q + 1 < C) ? Ain[(2 * q + 1) * P + off + x] : 0.0;
        sd[lay.addr(q, x)] = double2{re, im};
        if (sp.do_stats) sq += re * re + im * im;
      }
      defect += (double)NM - sq;
    }
    __syncthreads();
    to_fixed(t.plan[0].st[0].rad, false);
    fft_fx(s, lay, nx, Q, t.plan[0], tw, false, drops);
    visit([&](int q, int x) { W[q * P + off + x] = from_fixed(s[lay.addr(q, x)], scale_of(q)); });
    if (lifted) {
      visit([&](int q, int x) {
        if (lifted >> q & 1) fx_scale2(W[q * P + off + x], 0x1p-600);
      });
    }
    if (sp.do_stats) {
      const double tot = block_sum(defect, redd);
      double all;
      if (grid_sum(tot, sp.rb, redd, &s_flag, &all) && tid == 0) sp.st->defect = all;
    }
    return;
  }

  PointStats<double> ps;
  bool last = false;
  const long long gstride = (long long)gridDim.x * nx;
  for (;; off += gstride) {
#pragma unroll
    for (int q = 0; q < Q; ++q)
      for (int x = tid; x < nx; x += T) cp_async_elem(&sd[lay.addr(q, x)], &W[q * P + off + x]);
    if (MODE == ROW_INV_PROJECT_FWD && tid == 0) s_bad = 0;
    cp_async_wait_all();
    __syncthreads();
    to_fixed(t.plan[0].st[t.plan[0].nst - 1].rad, true);
    fft_fx(s, lay, nx, Q, t.plan[0], tw, true, drops);

    if (MODE == ROW_INV_OUT) {
      visit([&](int q, int x) {
        const double2 z = from_fixed(s[lay.addr(q, x)], scale_of(q));  // swapped
        A[(2 * q) * P + off + x] = z.y;
        if (2 * q + 1 < C) A[(2 * q + 1) * P + off + x] = z.x;
      });
      if (lifted) {
        visit([&](int q, int x) {
          if (!(lifted >> q & 1)) return;
          A[(2 * q) * P + off + x] *= 0x1p-600;
          if (2 * q + 1 < C) A[(2 * q + 1) * P + off + x] *= 0x1p-600;
        });
      }
      return;
    }

    // ROW_INV_PROJECT_FWD.  The projected entries lie in [-1, 1] (they are
    // parts of an orthogonal matrix): fixed scale, with room for the first
    // stage only; it shifts its results down to the room the others need.
    const int ku = fx_unit_scale(nx);
    const int kin = t.plan[0].nst > 1 ? 61 - (32 - __clz(t.plan[0].st[0].rad - 1)) : ku;
    int bad = 0;
    // the polar factor does not depend on the scale: where every plane is lifted or zero, m
    // stays so
    bool all = true;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      k[q] = scale_of(q);
      all = all && ((lifted >> q & 1) || k[q] == 0);
    }
    if (!all) {
#pragma unroll
      for (int q = 0; q < Q; ++q) k[q] += lifted >> q & 1 ? kFxUp : 0;
    }
    for (int x = tid; x < nx; x += T) {
      double old[C], m[C], b[C], sg;
#pragma unroll
      for (int c = 0; c < C; ++c) old[c] = A[c * P + off + x];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const double2 z = from_fixed(s[lay.addr(q, x)], k[q]);
        m[2 * q] = z.y;  // swapped
        if (2 * q + 1 < C) m[2 * q + 1] = z.x;
      }
      bool fin = true;
#pragma unroll
      for (int c = 0; c < C; ++c) fin = fin && isfinite(m[c]);
      ps.nonfinite += fin ? 0 : 1;
      project_point<NM>(m, b, sg, 0.0);
      double2 pt[Q];
      finish_point<NM>(A, P, off, x, old, b, sg, pt, 1, ps);
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        // not an orthogonal matrix's entry (NaN included): the plane's spectrum is NaN
        if (!(fabsf((float)pt[q].x) < 1.25f && fabsf((float)pt[q].y) < 1.25f)) bad |= 1 << q;
        else s[lay.addr(q, x)] = fx2{fx_from(pt[q].x, kin), fx_from(pt[q].y, kin)};
      }
    }
    if (bad) atomicOr(&s_bad, bad);
    if (tid < Q) drops[tid] = kin - ku;
    const bool end = off + gstride >= P;
    if (end && sp.do_stats) stats_park(ps, sh);
    __syncthreads();
    const int planes_bad = s_bad;
    if (end && sp.do_stats) last = stats_arrive(sp, sh);
    fft_fx(s, lay, nx, Q, t.plan[0], tw, false, drops);
    visit([&](int q, int x) {
      W[q * P + off + x] = from_fixed(s[lay.addr(q, x)], (planes_bad >> q & 1) ? kFxBad : ku);
    });
    if (end) break;
    __syncthreads();  // the row is in W: its slots are free
  }
  if (!sp.do_stats) return;
  stats_finish(g.P, g.tau, sp, last, sh);
}

// ---------------------------------------------------------------------------
// strided passes
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(kMaxThreads, 1)
k_axis_fx(Geom g, Tables<double> t, double2* W, StatsPtrs sp, int axis, int ltx) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double redd[32];
  __shared__ float rs[2][12][16];
  __shared__ int drops[16];
  __shared__ unsigned slow[32];
  __shared__ int s_flag;
  if (sp.respect_stop && *(volatile int*)&sp.st->stop) return;

  double2* sd = reinterpret_cast<double2*>(smem_raw);
  fx2* s = reinterpret_cast<fx2*>(smem_raw);
  const int tx = 1 << ltx;
  const int L = (axis == 1) ? g.ny : g.nz;
  const long long es = (axis == 1) ? (long long)g.nx : (long long)g.nx * g.ny;
  const int nouter = (axis == 1) ? g.nz : g.ny;
  const long long ostride = (axis == 1) ? (long long)g.nx * g.ny : (long long)g.nx;
  int q, o, x0;
  col_tile(g, nouter, tx, blockIdx.x, q, o, x0);
  double2* base = W + (long long)q * g.P + (long long)o * ostride + x0;
  const ColLayout lay{ltx};
  const int T = blockDim.x, tid = threadIdx.x;
  const FxTw* tw = static_cast<const FxTw*>(t.tw[axis]);
  const int mcol = tid & (tx - 1);
  const int p0 = tid >> ltx, dp = T >> ltx;
  const long long gstep = (long long)dp * es;
  const bool live = x0 + mcol < g.nx;
  {
    const double2* src = base + mcol + (long long)p0 * es;
    for (int p = p0; p < L; p += dp, src += gstep) {
      if (live) cp_async_elem(&sd[lay.addr(mcol, p)], src);
      else sd[lay.addr(mcol, p)] = double2{0.0, 0.0};
    }
  }
  cp_async_wait_all();
  __syncthreads();

  // sum and maximum over the threads of this thread's column
  auto col_fold = [&](float& v, float& m) {
    for (int d = tx; d < 32; d <<= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, d);
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
    }
    __syncthreads();
    if ((tid & 31) < tx) {
      rs[0][tid >> 5][tid & 31] = v;
      rs[1][tid >> 5][tid & 31] = m;
    }
    __syncthreads();
    v = m = 0.f;
    for (int w = 0; w < (T >> 5); ++w) {
      v += rs[0][w][mcol];
      m = fmaxf(m, rs[1][w][mcol]);
    }
  };
  const int r_fwd = t.plan[axis].st[0].rad, r_inv = t.plan[axis].st[t.plan[axis].nst - 1].rad;
  int k;
  {
    const int r0 = MODE == AXIS_INV ? r_inv : r_fwd;
    float n = 0.f, mx = 0.f;
    for (int p = p0; p < L; p += dp) {
      const double2 z = sd[lay.addr(mcol, p)];
      const float a = fx_norm(z);
      n += a;
      mx = fmaxf(mx, a);
    }
    col_fold(n, mx);
    const bool plain = fx_plain(n);
    FxScale f = plain ? fx_scales(n, mx, 0, r0) : FxScale{0, 0};
    int up = 0;
    if (!__syncthreads_and(plain)) {
      for (int c = 0; c < tx; ++c) {
        float nc = 0.f;  // column c's norm, as col_fold left its parts
        for (int w = 0; w < (T >> 5); ++w) nc += rs[0][w][c];
        if (fx_plain(nc)) continue;
        const FxScale fc = fx_scale_slow(
            [&](auto each) {
              if (mcol == c)
                for (int p = p0; p < L; p += dp) each(sd[lay.addr(mcol, p)]);
            },
            r0, slow);
        if (mcol == c) f = fc;
      }
      up = fx_lift(f.in);
      if (up)
        for (int p = p0; p < L; p += dp) fx_scale2(sd[lay.addr(mcol, p)], 0x1p600);
    }
    k = f.k;
    if (tid < tx) drops[tid] = k == kFxBad ? 0 : f.in - k;  // thread tid owns column tid
    f.in -= up;
    for (int p = p0; p < L; p += dp) {
      const int a = lay.addr(mcol, p);
      const double2 z = sd[a];
      const long long re = fx_from(z.x, f.in), im = fx_from(z.y, f.in);
      s[a] = k == kFxBad ? fx2{0, 0} : MODE == AXIS_INV ? fx2{im, re} : fx2{re, im};
    }
  }
  __syncthreads();
  fft_fx(s, lay, L, tx, t.plan[axis], tw, MODE == AXIS_INV, drops);

  double acc = 0.0;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  if (MODE == AXIS_FGI || MODE == AXIS_ENERGY) {
    // the last axis applies g(k) = g_x g_y (g_z); in 3-D the y frequency is
    // the outer index o of this tile (the y pass ran before).
    double go = 1.0, omo = 0.0;
    if (g.ndim == 3) {
      go = t.g[1][o];
      omo = t.om[1][o];
    }
    const int x = live ? x0 + mcol : 0;
    const double gxx = t.g[0][x], omx = t.om[0][x];
    if (sp.do_stats && live) {
      // sum (1 - g) |X|^2 with 1 - g = (omx + gx omo) + gx go om[p], without cancellation
      const double b0 = omx + gxx * omo, b1 = gxx * go;
      const double* omL = t.om[axis];
      double a0 = 0.0, a1 = 0.0;
      for (int p = p0; p < L; p += dp) {
        const fx2 v = s[lay.addr(mcol, p)];
        const double vx = fx_to(v.x, -62), vy = fx_to(v.y, -62);
        const double n2 = vx * vx + vy * vy;
        a0 += n2;
        a1 += omL[p] * n2;
      }
      // the scale back in two exact steps (its square may leave the FP64 range)
      const double w = (double)col_weight(g, q, x) * (b0 * a0 + b1 * a1);
      acc = k == kFxBad ? nan : scalbn(scalbn(w, 62 - k), 62 - k);
    }
    if (MODE == AXIS_FGI) {
      // the multiplier of entry p, gcol gL[p] in FP64, and a new scale for the
      // inverse from the norm of the products
      const double gcol = gxx * go * t.inv_p;
      const double* gL = t.g[axis];
      int ge = 0;
      const double gm = frexp(gcol, &ge);  // the norm in units of 2^ge: FP32 holds it
      float n = 0.f, mx = 0.f;
      for (int p = p0; p < L; p += dp) {
        const fx2 v = s[lay.addr(mcol, p)];
        const double gp = gm * gL[p];
        float a = fx_mod(fx_float(v.x), fx_float(v.y)) * fabsf((float)gp);
        if (a == 0.f && (v.x | v.y) != 0 && fx_nonzero(gp)) a = kFxTiny;
        n += a;
        mx = fmaxf(mx, a);
      }
      col_fold(n, mx);
      FxScale f = n > 1e-20f ? fx_scales(n, mx, ge, r_inv) : FxScale{0, 0};
      if (!__syncthreads_and(n > 1e-20f || n == 0.f || k == kFxBad)) {
        // products below the FP32 range: the norm in FP64
        double nd = 0.0;
        for (int p = p0; p < L; p += dp) {
          const fx2 v = s[lay.addr(mcol, p)];
          nd += (fabs((double)v.x) + fabs((double)v.y)) * fabs(gm * gL[p]);
        }
        for (int c = 0; c < tx; ++c) {
          const double sum = block_sum(mcol == c ? nd : 0.0, redd);
          __syncthreads();
          if (tid == 0) redd[31] = sum;
          __syncthreads();
          const double all = redd[31];
          if (mcol == c && !(n > 1e-20f) && all > 1e-290) f.k = f.in = 61 - ilogb(all * 1.002) - ge;
          __syncthreads();
        }
      }
      if (tid < tx) drops[tid] = f.in - f.k;
      const int sft = f.in + ge;
      for (int p = p0; p < L; p += dp) {
        const int a = lay.addr(mcol, p);
        const fx2 v = s[a];
        // v f 2^sft, f in units of 2^ge: its 53-bit mantissa as Q60 in [1/2, 1), its exponent
        // joins the shift, so that small products keep their digits
        const unsigned long long u = (unsigned long long)__double_as_longlong(gm * gL[p]);
        const int fe = (int)(u >> 52) & 0x7ff;
        long long mt = (long long)(((u & 0xfffffffffffffull) | 0x10000000000000ull) << 7);
        if ((long long)u < 0) mt = -mt;
        if (fe == 0) mt = 0;
        const int e = fe - 1022 + sft;
        // for the inverse: parts swapped
        s[a] = fx2{fx_mul_shift(fx_limbs(v.y), mt, e), fx_mul_shift(fx_limbs(v.x), mt, e)};
      }
      if (k != kFxBad) k += f.k;
    }
    __syncthreads();
  }
  if (MODE == AXIS_FGI) fft_fx(s, lay, L, tx, t.plan[axis], tw, true, drops);
  if (MODE != AXIS_ENERGY && live) {
    double2* dst = base + mcol + (long long)p0 * es;
    const int up = fx_lift(k), e = up - k;
    for (int p = p0; p < L; p += dp, dst += gstep) {
      const fx2 v = s[lay.addr(mcol, p)];
      const double re = fx_to(MODE == AXIS_FWD ? v.x : v.y, e), im = fx_to(MODE == AXIS_FWD ? v.y : v.x, e);
      *dst = k == kFxBad ? double2{nan, nan} : double2{re, im};
    }
    if (up) {
      dst = base + mcol + (long long)p0 * es;
      for (int p = p0; p < L; p += dp, dst += gstep) fx_scale2(*dst, 0x1p-600);
    }
  }
  if ((MODE == AXIS_FGI || MODE == AXIS_ENERGY) && sp.do_stats) {
    const double tot = block_sum(acc, redd);
    if (MODE == AXIS_FGI && sp.epart) {  // the x pass's finaliser adds these up
      if (tid == 0) {
        sp.epart[blockIdx.x] = tot;
        if (blockIdx.x == 0) sp.st->nep = gridDim.x;
      }
      return;
    }
    double all;
    if (grid_sum(tot, sp.rb, redd, &s_flag, &all)) {
      if (tid == 0) {
        RunState* st = sp.st;
        const double Pd = (double)g.P;
        const double E_tau = (all / Pd + st->defect) / (Pd * g.tau);
        st->energy_last = E_tau;
        sp.hist.energy[st->step & (kRing - 1)] = E_tau;
      }
    }
  }
}

}  // namespace mbo
