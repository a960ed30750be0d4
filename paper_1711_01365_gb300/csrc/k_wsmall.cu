// FP32 x pass over warp-plan axes (mbo_wrow.cuh): the form with helper warps,
// for grids of at most two blocks per SM.
#include "mbo_wrow.cuh"

namespace mbo {
namespace {

template <int NM, int N>
cudaError_t small_nm(const Geom& g, const Tables<float>& t, float* A, void* W, const StatsPtrs& sp, float fb,
                     int blocks, size_t smem, cudaStream_t s, bool prepare_only) {
  constexpr int HX = wrow_helpers(N, NM);
  if constexpr (HX > 1) {
    auto k = k_wrow<NM, ROW_INV_PROJECT_FWD, N, false, HX>;
    static SmemLimit limit;
    const cudaError_t e = raise_smem(k, smem, limit);
    if (e != cudaSuccess || prepare_only) return e;
    return launch_pdl(k, blocks, wrow_threads(N, NM) * HX, smem, s, g, t, (const float*)nullptr, A,
                      static_cast<float2*>(W), sp, fb, 0);
  }
  return cudaErrorInvalidValue;
}

template <int N>
cudaError_t small_n(const Geom& g, const Tables<float>& t, float* A, void* W, const StatsPtrs& sp, float fb,
                    int blocks, size_t smem, cudaStream_t s, bool prep) {
  switch (g.n) {
    case 1: return small_nm<1, N>(g, t, A, W, sp, fb, blocks, smem, s, prep);
    case 2: return small_nm<2, N>(g, t, A, W, sp, fb, blocks, smem, s, prep);
    case 3: return small_nm<3, N>(g, t, A, W, sp, fb, blocks, smem, s, prep);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_wrow_small(const Geom& g, const Tables<float>& t, float* A, void* W, const StatsPtrs& sp,
                              float fb, int blocks, size_t smem, cudaStream_t s, bool prepare_only) {
  switch (g.nx) {
    case 256: return small_n<256>(g, t, A, W, sp, fb, blocks, smem, s, prepare_only);
    case 512: return small_n<512>(g, t, A, W, sp, fb, blocks, smem, s, prepare_only);
    case 1024: return small_n<1024>(g, t, A, W, sp, fb, blocks, smem, s, prepare_only);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mbo
