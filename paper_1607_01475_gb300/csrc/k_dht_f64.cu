// FP64 Hartley transform passes along x and along a strided axis (block
// fixed point), and the spectral helpers.
#include "dht_fx.cuh"

namespace psd {

template <>
cudaError_t launch_dht_rows<double>(const double* src, double* dst, int nx, int nrows, double scale, const int* done,
                                    const AxisTables<double>& tb, cudaStream_t st, unsigned int* dmax_hi) {
  PSD_DISPATCH_N(nx, (fx_short((long long)nx * nrows, tb.nsm) ? rows_fx_impl<NN, kFxShort<NN>, double>(src, src, nullptr, dst, nrows, scale, done, tb, st, dmax_hi)
                                                              : rows_fx_impl<NN, 8, double>(src, src, nullptr, dst, nrows, scale, done, tb, st, dmax_hi)));
}

cudaError_t launch_dht_rows_from_f32(const float* src, const float* src_odd, const int* iter, double* dst, int nx,
                                     int nrows, const AxisTables<double>& tb, cudaStream_t st, const int* skip) {
  PSD_DISPATCH_N(nx, (fx_short((long long)nx * nrows, tb.nsm) ? rows_fx_impl<NN, kFxShort<NN>, float>(src, src_odd, iter, dst, nrows, 1.0, skip, tb, st, nullptr)
                                                              : rows_fx_impl<NN, 8, float>(src, src_odd, iter, dst, nrows, 1.0, skip, tb, st, nullptr)));
}

template <>
cudaError_t launch_dht_cols<double>(double* data, const KParams& kp, int ax, double scale, const int* done,
                                    const AxisTables<double>& tb, cudaStream_t st) {
  const int n = ax == 1 ? kp.ny : kp.nz;
  const size_t plane = (size_t)kp.nx * kp.ny;
  const size_t line_stride = ax == 1 ? (size_t)kp.nx : plane;
  const size_t outer_stride = ax == 1 ? plane : (size_t)kp.nx;
  const int nouter = ax == 1 ? kp.nz : kp.ny;
  const bool small = fx_short((long long)plane * kp.nz, tb.nsm);
  PSD_DISPATCH_N(n, (small ? cols_fx_impl<NN, kFxShort<NN>>(data, kp.nx, nouter, line_stride, outer_stride, scale, done,
                                                 tb.fxtw[ax], tb.nsm, st)
                           : cols_fx_impl<NN, 8>(data, kp.nx, nouter, line_stride, outer_stride, scale, done,
                                                 tb.fxtw[ax], tb.nsm, st)));
}

#define PSD_INST_SPEC(T)                                                                               \
  template cudaError_t launch_spec6_combine<T>(T*, const T*, const KParams&, const AxisTables<T>&,      \
                                               cudaStream_t);                                          \
  template cudaError_t launch_spec_apply_T<T>(T*, T, const KParams&, const AxisTables<T>&, cudaStream_t);
PSD_INST_SPEC(double)
#undef PSD_INST_SPEC
template cudaError_t launch_spec_quad<double>(const double*, const KParams&, Ctrl*, double*, const AxisTables<double>&,
                                              cudaStream_t);

}  // namespace psd
