// FP32 x pass of the MBO step (Algorithm 1 of Osting & Wang,
// arXiv:1711.01365) for x axes whose plan is the warp-cooperative four-step
// transform (mbo_wfft.cuh): lengths 256, 512 and 1024, and 768 = 3 x 256,
// 1536 = 3 x 512, 2048 = 2 x 1024 through a radix-3 / radix-2 stage across
// groups of lanes.  Instantiated in k_warp.cu, the
// small-grid form in k_wsmall.cu; the strided passes are in k_wcol.cu.
//
//   k_wrow  x axis: one sequence (row, complex plane) per LQ lanes.  Inverse
//           transform in registers, exchange through shared memory so that one
//           thread sees all n*n channels of a point, projection (Lemma 1.1) and
//           step statistics, exchange back, forward transform of the new field.
// Data layout in HBM is that of the generic passes (mbo_kernels.cuh); spectra
// along these axes are in natural order.
#pragma once
#include "mbo_kernels.cuh"
#include "mbo_tma.cuh"
#include "mbo_wfft.cuh"
#include "mbo_wshape.cuh"

namespace mbo {
namespace {

// HX > 1 (one row group per block, lengths of one lane group): HX times the
// threads the transforms take; the extra warps share the points of the
// projection.  For grids of at most two blocks per SM, where the block's own
// chain of steps is the time: a thread projects 8 points in turn at 256^2, n = 2
// with the transforms' 64 threads, 2 with 256.
template <int NM, int MODE, int N, bool PERS, int HX>
__global__ void __launch_bounds__(wrow_threads(N, NM) * HX, HX > 1 ? 2 : wrow_minb(N, NM))
k_wrow(Geom g, Tables<float> t, const float* __restrict__ Ain, float* A, float2* W, StatsPtrs sp,
       float fb_sigma, int ahead) {
  constexpr int R = w_r(N), M = w_m(N), LQ = w_lq(N), RB = wrow_rb(N);
  using F = WarpFFTR<M, LQ, R>;
  constexpr int C = NM * NM, Q = (C + 1) / 2, E = F::E, RS = F::RS, NT = wrow_threads(N, NM) * HX;
  static_assert(HX == 1 || (R == 1 && !PERS), "helper warps skip the transforms, which must not hold block barriers");
  constexpr int PS = R * RS;  // slots of one (row, plane): R group regions, >= N
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double redd[MODE == ROW_FWD ? 32 : 1];
  __shared__ StatsShared<float, MODE == ROW_INV_PROJECT_FWD ? NT : 1> sh;
  __shared__ int s_flag, s_nfb;
  pdl_wait();  // the previous pass's spectrum and run state are complete
  if (sp.respect_stop && *(volatile int*)&sp.st->stop) return;
  pdl_release();

  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const int tid = threadIdx.x;
  const int grp = tid / LQ, l = tid - grp * LQ;  // group = (row, plane, r)
  const int seq = grp / R, r = grp - seq * R;
  const int row = seq / Q, q = seq - row * Q;
  const long long P = g.P;
  const long long rows = P / N;
  const long long ngroups = (rows + RB - 1) / RB;  // row groups: RB rows each
  float2* base = sm + seq * PS;  // this (row, plane)'s regions
  const float2* tw = static_cast<const float2*>(t.tw[0]);
  const float2* twr = tw + M;
  float* fbM = reinterpret_cast<float*>(sm + wrow_nseq(N, NM) * PS);
  int* fbX = reinterpret_cast<int*>(fbM + kFallbackCap * C);
  const bool mirror = q == Q - 1 && g.xh < N;
  const bool fft = HX == 1 || tid < wrow_threads(N, NM);  // warp-uniform
  float2 v[E];
  PointStats<float> ps;  // projection mode: over all of the block's rows
  bool last = false;     // projection mode, thread 0: this block arrived last
  double defect = 0.0;   // forward mode

  // Row groups of this block: its own index, or with PERS the groups
  // blockIdx.x, blockIdx.x + gridDim.x, ... (a grid of one wave).
  const long long gstep = PERS ? (long long)gridDim.x : ngroups;
  auto do_group = [&](long long gi) {
    const long long row0 = gi * RB;
    const bool live = seq < RB * Q && row0 + row < rows;  // a whole sequence is live or not
    const long long off = (row0 + row) * N;
    // the forward spectrum of this sequence to W; the last plane of an odd
    // channel count is Hermitian: columns k < xh only
    auto store_spectrum = [&](const float2(&u)[E]) {
      if (!live) return;
      float2* wdst = W + q * P + off;
      if (q < Q - 1 || g.xh == N) {
#pragma unroll
        for (int j = 0; j < E; ++j) wdst[l + M * r + LQ * j] = u[j];
      } else {
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int k = l + LQ * j + M * r;
          if (k < g.xh) wdst[k] = u[j];
        }
      }
    };

    if (MODE == ROW_FWD) {
      // The rows straight into registers (one address per element, constant
      // offsets): lane (q, r, l) takes channels 2q and 2q + 1 of its own points,
      // so nothing is exchanged before the transform.  sum n - |A|^2: the plane
      // that comes first brings the n of its points, every lane takes off its
      // squares, summed in two FP32 words (TwoSum) and joined in FP64.
      const float* a0 = Ain + (2 * q) * P + off + r;
      const float* a1 = a0 + P;
      const bool pair = 2 * q + 1 < C;
      if (!live) {
#pragma unroll
        for (int j = 0; j < E; ++j) v[j] = float2{0.f, 0.f};
      } else {
#pragma unroll
        for (int j = 0; j < E; ++j) v[j].x = a0[R * (l + LQ * j)];
#pragma unroll
        for (int j = 0; j < E; ++j) v[j].y = pair ? a1[R * (l + LQ * j)] : 0.f;
        if (sp.do_stats) {
          float hi = 0.f, lo = 0.f;
#pragma unroll
          for (int j = 0; j < E; ++j) {
            const float t2 = v[j].x * v[j].x + v[j].y * v[j].y;
            const float sm2 = hi + t2, bb = sm2 - hi;
            lo += (hi - (sm2 - bb)) + (t2 - bb);
            hi = sm2;
          }
          defect += ((q == 0 ? (double)(NM * E) : 0.0) - (double)hi) - (double)lo;
        }
      }
      F::fwd(v, base, r, tw, twr, l);
      store_spectrum(v);
      return;
    }

    if (MODE == ROW_INV_PROJECT_FWD && tid < C) {
      // the old field of this group's rows, wanted after the inverse transform
      const long long nr = rows - row0 < RB ? rows - row0 : RB;
      bulk_prefetch_l2(A + tid * P + row0 * N, (unsigned)(nr * N * sizeof(float)));
    } else if (tid >= 32 && tid < 32 + RB * Q && (PERS || ahead > 0)) {
      // the spectrum rows of the group this block (or a block of a later
      // wave) takes next
      const long long rn = (PERS ? row0 + gstep * RB : row0 + (long long)ahead * RB) + (tid - 32) / Q;
      const int qq = (tid - 32) % Q;
      if (rn < rows) {
        const int cols = qq == Q - 1 ? g.xh : N;
        bulk_prefetch_l2(W + qq * P + rn * N, (unsigned)((cols * sizeof(float2) + 15) & ~15u));
      }
    }

    // inverse modes: the spectrum rows straight into registers (coalesced); a
    // Hermitian last plane supplies columns k > N/2 as conj(column N - k)
    const float2* wrow = W + q * P + off;  // this sequence's spectrum row
    if (!live) {
#pragma unroll
      for (int j = 0; j < E; ++j) v[j] = float2{0.f, 0.f};
    } else if (!mirror) {  // warp-uniform: one address per element, constant offsets
#pragma unroll
      for (int j = 0; j < E; ++j) v[j] = wrow[l + M * r + LQ * j];
    } else {
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const int k = l + LQ * j + M * r;
        const bool up = 2 * k > N;
        float2 z = wrow[up ? N - k : k];
        z.y = up ? -z.y : z.y;
        v[j] = z;
      }
    }
    if (fft) F::inv(v, base, r, tw, twr, l);

    if (MODE == ROW_INV_OUT) {
      if (live) {
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int x = R * (l + LQ * j) + r;
          A[(2 * q) * P + off + x] = v[j].x;
          if (2 * q + 1 < C) A[(2 * q + 1) * P + off + x] = v[j].y;
        }
      }
      return;
    }

    // ROW_INV_PROJECT_FWD
    if constexpr (R > 1) __syncthreads();  // every group's transposes are done: the regions hold points now
    if (fft) {
#pragma unroll
      for (int j = 0; j < E; ++j) base[R * (l + LQ * j) + r] = v[j];
    }
    if (tid == 0) s_nfb = 0;
    __syncthreads();
    for (int p = tid; p < RB * N; p += NT) {
      const int rw = p / N, x = p - rw * N;
      if (row0 + rw >= rows) continue;
      // issued first, used last: the loads overlap the projection (the rows
      // were prefetched to L2 at the start of the group)
      float old[C];
      {
        const float* src = A + (row0 + rw) * N + x;
#pragma unroll
        for (int c = 0; c < C; ++c, src += P) old[c] = *src;
      }
      const long long ro = (row0 + rw) * N;
      float2* pt = sm + rw * Q * PS + x;
      float m[C];
#pragma unroll
      for (int qq = 0; qq < Q; ++qq) {
        const float2 z = pt[qq * PS];
        m[2 * qq] = z.x;
        if (2 * qq + 1 < C) m[2 * qq + 1] = z.y;
      }
      // finite entries have a finite sum of squares (up to overflow, which
      // the entry-wise test below settles)
      float nx = 0.f;
#pragma unroll
      for (int c = 0; c < C; ++c) nx += m[c] * m[c];
      bool fin = isfinite(nx);
      if (!fin) {
        fin = true;
#pragma unroll
        for (int c = 0; c < C; ++c) fin = fin && isfinite(m[c]);
      }
      ps.nonfinite += fin ? 0 : 1;
      float b[C];
      float sg;
      if (!project_point<NM>(m, b, sg, fb_sigma) && fin) {
        const int slot = atomicAdd(&s_nfb, 1);
        if (slot < kFallbackCap) {
          fbX[slot] = p;
#pragma unroll
          for (int c = 0; c < C; ++c) fbM[slot * C + c] = m[c];
          continue;
        }
        sg = project_point_f64<NM>(m, b);
        ps.fallback += 1;
      }
      finish_point<NM>(A, P, ro, x, old, b, sg, pt, PS, ps);
    }
    if (NM >= 2) {
      // the FP64 re-projections collected above, spread over the block
      __syncthreads();
      const int nf = min(s_nfb, kFallbackCap);
      for (int k = tid; k < nf; k += NT) {
        const int p = fbX[k];
        const int rw = p / N, x = p - rw * N;
        const long long ro = (row0 + rw) * N;
        float m[C], b[C], old[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          m[c] = fbM[k * C + c];
          old[c] = A[c * P + ro + x];
        }
        const float sg = project_point_f64<NM>(m, b);
        ps.fallback += 1;
        finish_point<NM>(A, P, ro, x, old, b, sg, sm + rw * Q * PS + x, PS, ps);
      }
    }
    // one row group per block: its statistics are complete, and the arrival at
    // the grid's counter overlaps the forward transform below (a block that
    // walks several groups arrives after its loop: the test for the last one
    // cost the 2048-point rows 1%)
    if (!PERS && sp.do_stats) stats_park(ps, sh);
    __syncthreads();
    if (!PERS && sp.do_stats) last = stats_arrive(sp, sh);
    if (!fft) return;
#pragma unroll
    for (int j = 0; j < E; ++j) v[j] = base[R * (l + LQ * j) + r];
    if constexpr (R > 1) __syncthreads();
    else __syncwarp();
    F::fwd(v, base, r, tw, twr, l);
    store_spectrum(v);
  };
  if constexpr (PERS) {
    for (long long gi = blockIdx.x; gi < ngroups; gi += gstep) {
      if (gi != blockIdx.x) __syncthreads();  // the previous group's regions are free
      do_group(gi);
    }
  } else {
    do_group(blockIdx.x);
  }

  if (!sp.do_stats || MODE == ROW_INV_OUT) return;
  if (MODE == ROW_FWD) {
    const double tot = block_sum(defect, redd);
    double all;
    if (grid_sum(tot, sp.rb, redd, &s_flag, &all) && tid == 0) sp.st->defect = all;
    return;
  }
  if constexpr (PERS) {
    stats_park(ps, sh);
    __syncthreads();
    last = stats_arrive(sp, sh);
  }
  stats_finish(g.P, g.tau, sp, last, sh);
}

}  // namespace
}  // namespace mbo
