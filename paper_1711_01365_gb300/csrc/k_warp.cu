// FP32 x pass over warp-plan axes (mbo_wrow.cuh): launchers.
#include "mbo_wrow.cuh"

namespace mbo {
namespace {

template <int NM, int MODE, int N>
cudaError_t wrow_nm(const Geom& g, const Tables<float>& t, const float* Ain, float* A, void* W,
                    const StatsPtrs& sp, float fb, cudaStream_t s, bool prepare_only) {
  // the one-wave form is instantiated for the projecting pass only
  constexpr bool CAN_PERS = MODE == ROW_INV_PROJECT_FWD;
  auto k = k_wrow<NM, MODE, N, false, 1>;
  auto kp = k_wrow<NM, MODE, N, CAN_PERS, 1>;
  static SmemLimit limit, limit_p;
  static DeviceCount fits;
  const size_t smem = wrow_smem_bytes(g, N, MODE == ROW_INV_PROJECT_FWD);
  cudaError_t e = raise_smem(k, smem, limit);
  if (e == cudaSuccess && CAN_PERS) e = raise_smem(kp, smem, limit_p);
  if (e != cudaSuccess) return e;
  const int dev = current_device(), sms = device_sms(dev);
  const int resident = fits.get(dev, [&] {  // blocks of this kernel that fit on the device at once
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, wrow_threads(N, NM), smem);
    return sms * (per_sm > 0 ? per_sm : 1);
  });
  constexpr bool CAN_HELP = MODE == ROW_INV_PROJECT_FWD && wrow_helpers(N, NM) > 1;
  if constexpr (CAN_HELP) {
    if (prepare_only && (e = launch_wrow_small(g, t, A, W, sp, fb, 0, smem, s, true)) != cudaSuccess) return e;
  }
  if (prepare_only) return cudaSuccess;
  constexpr int RB = wrow_rb(N);
  const long long rows = g.P / N;
  const int blocks = (int)((rows + RB - 1) / RB);
  if constexpr (CAN_HELP) {
    if (wrow_helpers_flag() && blocks <= 2 * sms) return launch_wrow_small(g, t, A, W, sp, fb, blocks, smem, s, false);
  }
  // a block prefetches the spectrum rows of the block one wave later
  const int ahead = blocks > resident ? resident : 0;
  // persistent: one wave of blocks walks the row groups with a stride of the grid
  // (also wherever the last block would have too many records to sum)
  if (CAN_PERS && blocks > resident && (wrow_persistent_flag() || blocks > (int)kReduceOneLevel))
    return launch_pdl(kp, resident, wrow_threads(N, NM), smem, s, g, t, Ain, A, static_cast<float2*>(W),
                      sp, fb, 0);
  return launch_pdl(k, blocks, wrow_threads(N, NM), smem, s, g, t, Ain, A, static_cast<float2*>(W), sp,
                    fb, ahead);
}

template <int N>
cudaError_t wrow_n(RowMode mode, const Geom& g, const Tables<float>& t, const float* Ain, float* A,
                   void* W, const StatsPtrs& sp, float fb, cudaStream_t s, bool prep) {
#define MBO_WROW_CASE(NM)                                                                        \
  if (g.n == NM) {                                                                               \
    if (mode == ROW_FWD) return wrow_nm<NM, ROW_FWD, N>(g, t, Ain, A, W, sp, fb, s, prep);       \
    if (mode == ROW_INV_OUT) return wrow_nm<NM, ROW_INV_OUT, N>(g, t, Ain, A, W, sp, fb, s, prep); \
    return wrow_nm<NM, ROW_INV_PROJECT_FWD, N>(g, t, Ain, A, W, sp, fb, s, prep);                \
  }
  MBO_WROW_CASE(1)
  MBO_WROW_CASE(2)
  MBO_WROW_CASE(3)
  MBO_WROW_CASE(4)
#undef MBO_WROW_CASE
  return cudaErrorInvalidValue;
}

}  // namespace

bool warp_plan_length(int N) {
  return N == 256 || N == 512 || N == 768 || N == 1024 || N == 1536 || N == 2048;
}
int warp_plan_radix(int N) { return w_r(N); }

size_t wrow_smem_bytes(const Geom& g, int N, bool fallback) {
  const int LQ = w_lq(N), RB = wrow_rb(N), R = w_r(N);
  const size_t rs = (size_t)(LQ + 1) * (w_m(N) / LQ);
  const int threads = (RB * g.Q * R * LQ + 31) / 32 * 32;
  const int nseq = (threads + R * LQ - 1) / (R * LQ);  // wrow_nseq(N, g.n)
  size_t b = (size_t)nseq * R * rs * sizeof(float2);
  if (fallback) b += (size_t)kFallbackCap * ((size_t)g.C * sizeof(float) + sizeof(int));
  return (b + 15) & ~(size_t)15;
}

namespace {
template <int NM, int N> double wrow_waves_nm(const Geom& g) {
  auto k = k_wrow<NM, ROW_INV_PROJECT_FWD, N, false, 1>;
  const int sms = device_sms(current_device());
  int per_sm = 0;
  const size_t smem = wrow_smem_bytes(g, N, true);
  // a shape that does not fit is rejected by the caller; leave no error behind
  if ((smem > 48 * 1024 &&
       cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, wrow_threads(N, NM), smem) != cudaSuccess) {
    (void)cudaGetLastError();
    return 1e9;
  }
  const double blocks = (double)((g.P / N + wrow_rb(N) - 1) / wrow_rb(N));
  return blocks / ((double)sms * (per_sm > 0 ? per_sm : 1));
}
template <int N> double wrow_waves_n(const Geom& g) {
  switch (g.n) {
    case 1: return wrow_waves_nm<1, N>(g);
    case 2: return wrow_waves_nm<2, N>(g);
    case 3: return wrow_waves_nm<3, N>(g);
    default: return wrow_waves_nm<4, N>(g);
  }
}
}  // namespace

double wrow_waves(const Geom& g) {
  switch (g.nx) {
    case 2048: return wrow_waves_n<2048>(g);
    case 1536: return wrow_waves_n<1536>(g);
    case 1024: return wrow_waves_n<1024>(g);
    case 768: return wrow_waves_n<768>(g);
    case 512: return wrow_waves_n<512>(g);
    case 256: return wrow_waves_n<256>(g);
    default: return 0.0;
  }
}

bool& wrow_persistent_flag() {
  thread_local bool on = false;
  return on;
}

bool& wrow_helpers_flag() {
  thread_local bool on = true;
  return on;
}

bool& pdl_flag() {
  thread_local bool on = true;
  return on;
}

cudaError_t launch_wrow(RowMode mode, const Geom& g, const Tables<float>& t, const float* Ain,
                        float* A, void* W, const StatsPtrs& sp, double fb, cudaStream_t s,
                        bool prepare_only) {
  const float f = (float)fb;
  switch (g.nx) {
    case 2048: return wrow_n<2048>(mode, g, t, Ain, A, W, sp, f, s, prepare_only);
    case 1536: return wrow_n<1536>(mode, g, t, Ain, A, W, sp, f, s, prepare_only);
    case 1024: return wrow_n<1024>(mode, g, t, Ain, A, W, sp, f, s, prepare_only);
    case 768: return wrow_n<768>(mode, g, t, Ain, A, W, sp, f, s, prepare_only);
    case 512: return wrow_n<512>(mode, g, t, Ain, A, W, sp, f, s, prepare_only);
    case 256: return wrow_n<256>(mode, g, t, Ain, A, W, sp, f, s, prepare_only);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mbo
