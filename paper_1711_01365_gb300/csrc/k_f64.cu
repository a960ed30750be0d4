// FP64 passes: the transforms in 64-bit fixed point (mbo_fixed.cuh), the
// pointwise kernels instantiated from mbo_kernels.cuh.
#include "mbo_fixed.cuh"

namespace mbo {

namespace {

template <int NM, int MODE, bool SHORT>
cudaError_t row_fx_form(const Geom& g, const Tables<double>& t, const double* Ain, double* A, void* W,
                   const StatsPtrs& sp, int threads, cudaStream_t s, bool prepare_only = false) {
  auto k = k_row_fx<NM, MODE, SHORT>;
  static SmemLimit limit;
  const size_t smem = row_smem_bytes(g, sizeof(double), false);
  const cudaError_t e = raise_smem(k, smem, limit);
  if (e != cudaSuccess || prepare_only) return e;
  int rows = g.nz * g.ny;
  if (MODE == ROW_INV_PROJECT_FWD) {
    static std::atomic<unsigned long long> fits{0};
    rows = std::min(rows, resident_blocks(k, threads, smem, fits));
  }
  k<<<rows, threads, smem, s>>>(g, t, Ain, A, static_cast<double2*>(W), sp);
  return cudaGetLastError();
}

template <int NM, int MODE>
cudaError_t row_fx(const Geom& g, const Tables<double>& t, const double* Ain, double* A, void* W,
                   const StatsPtrs& sp, int threads, cudaStream_t s, bool prepare_only = false) {
  if (fx_short_rows(g)) return row_fx_form<NM, MODE, true>(g, t, Ain, A, W, sp, threads, s, prepare_only);
  return row_fx_form<NM, MODE, false>(g, t, Ain, A, W, sp, threads, s, prepare_only);
}

template <int NM>
cudaError_t row_fx_mode(RowMode mode, const Geom& g, const Tables<double>& t, const double* Ain, double* A,
                        void* W, const StatsPtrs& sp, int threads, cudaStream_t s, bool prep) {
  switch (mode) {
    case ROW_FWD: return row_fx<NM, ROW_FWD>(g, t, Ain, A, W, sp, threads, s, prep);
    case ROW_INV_OUT: return row_fx<NM, ROW_INV_OUT>(g, t, Ain, A, W, sp, threads, s, prep);
    default: return row_fx<NM, ROW_INV_PROJECT_FWD>(g, t, Ain, A, W, sp, threads, s, prep);
  }
}

cudaError_t row_fx_n(RowMode mode, const Geom& g, const Tables<double>& t, const double* Ain, double* A,
                     void* W, const StatsPtrs& sp, int threads, cudaStream_t s, bool prep) {
  switch (g.n) {
    case 1: return row_fx_mode<1>(mode, g, t, Ain, A, W, sp, threads, s, prep);
    case 2: return row_fx_mode<2>(mode, g, t, Ain, A, W, sp, threads, s, prep);
    case 3: return row_fx_mode<3>(mode, g, t, Ain, A, W, sp, threads, s, prep);
    case 4: return row_fx_mode<4>(mode, g, t, Ain, A, W, sp, threads, s, prep);
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE>
cudaError_t axis_fx(const Geom& g, const Tables<double>& t, void* W, const StatsPtrs& sp, int axis, int tx,
                    int threads, cudaStream_t s, bool prepare_only = false) {
  auto k = k_axis_fx<MODE>;
  static SmemLimit limit;
  const size_t smem = axis_smem_bytes(axis == 1 ? g.ny : g.nz, tx, sizeof(double));
  const cudaError_t e = raise_smem(k, smem, limit);
  if (e != cudaSuccess || prepare_only) return e;
  int ltx = 0;
  while ((1 << ltx) < tx) ++ltx;
  const int tiles = col_tiles(g, axis == 1 ? g.nz : g.ny, tx);
  k<<<tiles, threads, smem, s>>>(g, t, static_cast<double2*>(W), sp, axis, ltx);
  return cudaGetLastError();
}

cudaError_t axis_fx_mode(AxisMode mode, const Geom& g, const Tables<double>& t, void* W, const StatsPtrs& sp,
                         int axis, int tx, int threads, cudaStream_t s, bool prep) {
  switch (mode) {
    case AXIS_FWD: return axis_fx<AXIS_FWD>(g, t, W, sp, axis, tx, threads, s, prep);
    case AXIS_INV: return axis_fx<AXIS_INV>(g, t, W, sp, axis, tx, threads, s, prep);
    case AXIS_FGI: return axis_fx<AXIS_FGI>(g, t, W, sp, axis, tx, threads, s, prep);
    default: return axis_fx<AXIS_ENERGY>(g, t, W, sp, axis, tx, threads, s, prep);
  }
}

}  // namespace

template <>
cudaError_t launch_row<double>(RowMode mode, const Geom& g, const Tables<double>& t, const double* A_in,
                               double* A_out, void* W, const StatsPtrs& sp, double, int threads,
                               cudaStream_t s) {
  return row_fx_n(mode, g, t, A_in, A_out, W, sp, threads, s, false);
}

template <>
cudaError_t launch_axis<double>(AxisMode mode, int axis, const Geom& g, const Tables<double>& t, void* W,
                                const StatsPtrs& sp, int tx, int threads, cudaStream_t s, const CUtensorMap*,
                                int, const void*, long long) {
  return axis_fx_mode(mode, g, t, W, sp, axis, tx, threads, s, false);
}

template <>
cudaError_t prepare_kernels<double>(const Geom& g, const Tables<double>& t, int, int net_tx, int) {
  StatsPtrs sp{};
  cudaError_t e = cudaSuccess;
  for (int m = ROW_FWD; m <= ROW_INV_PROJECT_FWD && e == cudaSuccess; ++m)
    e = row_fx_n((RowMode)m, g, t, nullptr, nullptr, nullptr, sp, 32, 0, true);
  for (int axis = 1; axis <= (g.ndim == 3 ? 2 : 1); ++axis)
    for (int m = AXIS_FWD; m <= AXIS_ENERGY && e == cudaSuccess; ++m)
      e = axis_fx_mode((AxisMode)m, g, t, nullptr, sp, axis, net_tx, 64, 0, true);
  return e;
}

MBO_INSTANTIATE_POINTS(double)

}  // namespace mbo
