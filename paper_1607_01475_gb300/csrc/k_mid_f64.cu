// FP64 middle pass of the preconditioner and the last pass of the mixed
// solver's outer loop (block fixed-point transforms).
#include "dht_fx.cuh"

namespace psd {

template <>
cudaError_t launch_mid<double>(double* data, const KParams& kp, Ctrl* ctrl, double* partials, double* xi,
                               double* dspec, const AxisTables<double>& tb, cudaStream_t st) {
  const int n = kp.dim == 2 ? kp.ny : kp.nz;
  PSD_DISPATCH_N(n, (mid_fx_impl<NN>(data, kp, ctrl, partials, xi, dspec, tb, st)));
}

cudaError_t launch_dht_last(const double* data, double* theta, float* out32, const KParams& kp, Ctrl* ctrl,
                            double* partials, const AxisTables<double>& tb, cudaStream_t st, double* dc,
                            const int* skip) {
  const int n = kp.dim == 3 ? kp.nz : kp.ny;
  PSD_DISPATCH_N(n, (last_fx_impl<NN>(data, theta, out32, kp, ctrl, partials, tb, st, dc, skip)));
}

namespace {
template <int N>
void set_attrs_mid_fx() {
  constexpr size_t np = kFxThreads / LineFFT<fx, N, 8>::TS;
  constexpr int line = (int)(np * fx_pair_smem<N, false>()), stage = (int)(np * N * sizeof(double2));
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaFuncSetAttribute(k_mid_fx<N, 4>, attr, line);
  cudaFuncSetAttribute(k_mid_fx<N, 6>, attr, line + 2 * stage);
  cudaFuncSetAttribute(k_last_fx<N, EPI_THETA>, attr, line + stage);
  cudaFuncSetAttribute(k_last_fx<N, EPI_RESID>, attr, line + stage);
}
}  // namespace

void init_dht_attributes_f32();

void init_dht_attributes() {
  init_dht_attributes_f32();
  set_attrs_mid_fx<8>();
  set_attrs_mid_fx<16>();
  set_attrs_mid_fx<32>();
  set_attrs_mid_fx<64>();
  set_attrs_mid_fx<128>();
  set_attrs_mid_fx<256>();
  set_attrs_mid_fx<512>();
  set_attrs_mid_fx<1024>();
}

}  // namespace psd
