// FP64 middle pass of the preconditioner and the last pass of the mixed
// solver's outer loop (block fixed-point transforms).
#include "dht_fx.cuh"

namespace psd {

template <>
cudaError_t launch_mid<double>(double* data, const KParams& kp, Ctrl* ctrl, double* partials, double* xi,
                               double* dspec, const AxisTables<double>& tb, cudaStream_t st) {
  const int n = kp.dim == 2 ? kp.ny : kp.nz;
  const bool small = fx_short((long long)kp.nx * kp.ny * kp.nz, tb.nsm);
  PSD_DISPATCH_N(n, (small ? mid_fx_impl<NN, kFxShort<NN>>(data, kp, ctrl, partials, xi, dspec, tb, st)
                           : mid_fx_impl<NN, 8>(data, kp, ctrl, partials, xi, dspec, tb, st)));
}

cudaError_t launch_dht_last(const double* data, double* theta, float* out32, const KParams& kp, Ctrl* ctrl,
                            double* partials, const AxisTables<double>& tb, cudaStream_t st, double* dc,
                            const int* skip) {
  const int n = kp.dim == 3 ? kp.nz : kp.ny;
  const bool small = fx_short((long long)kp.nx * kp.ny * kp.nz, tb.nsm);
  PSD_DISPATCH_N(n, (small ? last_fx_impl<NN, kFxShort<NN>>(data, theta, out32, kp, ctrl, partials, tb, st, dc, skip)
                           : last_fx_impl<NN, 8>(data, theta, out32, kp, ctrl, partials, tb, st, dc, skip)));
}

namespace {
template <int N, int RM>
void set_attrs_mid_fx_radix() {
  constexpr size_t np = kFxThreads / LineFFT<fx, N, RM>::TS;
  constexpr int line = (int)(np * fx_pair_smem<N, RM, false>()), stage = (int)(np * N * sizeof(double2));
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaFuncSetAttribute(k_mid_fx<N, RM, 4, true>, attr, line);
  cudaFuncSetAttribute(k_mid_fx<N, RM, 6, true>, attr, line + 2 * stage);
  cudaFuncSetAttribute(k_mid_fx<N, RM, 4, false>, attr, line);
  cudaFuncSetAttribute(k_mid_fx<N, RM, 6, false>, attr, line + 2 * stage);
  cudaFuncSetAttribute(k_last_fx<N, RM, EPI_THETA>, attr, line + stage);
  cudaFuncSetAttribute(k_last_fx<N, RM, EPI_RESID>, attr, line + stage);
}
template <int N>
cudaError_t set_attrs_mid_fx() {
  set_attrs_mid_fx_radix<N, 8>();
  if constexpr (kFxShort<N> != 8) set_attrs_mid_fx_radix<N, kFxShort<N>>();
  return cudaSuccess;
}
}  // namespace

cudaError_t init_dht_attributes_f32(int n);

cudaError_t init_dht_attributes(int n) {
  const cudaError_t e = init_dht_attributes_f32(n);
  if (e != cudaSuccess) return e;
  PSD_DISPATCH_N(n, (set_attrs_mid_fx<NN>()));
}

}  // namespace psd
