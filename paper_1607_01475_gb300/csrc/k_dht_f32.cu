// FP32 Hartley transform passes and the middle pass (the mixed solver's
// inner iteration).
#include "dht_kernels.cuh"

namespace psd {

template <>
cudaError_t launch_dht_rows<float>(const float* src, float* dst, int nx, int nrows, float scale, const int* done,
                                   const AxisTables<float>& tb, cudaStream_t st, unsigned int*) {
  PSD_DISPATCH_N(nx, (rows_impl<float, NN>(src, dst, nrows, scale, done, tb.twc[0], tb.tws[0], st, tb.nsm,
                                           tb.tile_cap[0])));
}

template <>
cudaError_t launch_dht_cols<float>(float* data, const KParams& kp, int ax, float scale, const int* done,
                                   const AxisTables<float>& tb, cudaStream_t st) {
  const int n = ax == 1 ? kp.ny : kp.nz;
  const size_t plane = (size_t)kp.nx * kp.ny;
  const size_t line_stride = ax == 1 ? (size_t)kp.nx : plane;
  const size_t outer_stride = ax == 1 ? plane : (size_t)kp.nx;
  const int nouter = ax == 1 ? kp.nz : kp.ny;
  PSD_DISPATCH_N(n, (cols_impl<float, NN>(data, kp.nx, nouter, line_stride, outer_stride, scale, done, tb.twc[ax],
                                          tb.tws[ax], st, tb.nsm, tb.tile_cap[1])));
}

template <>
cudaError_t launch_mid<float>(float* data, const KParams& kp, Ctrl* ctrl, double* partials, float* xi, float* dspec,
                              const AxisTables<float>& tb, cudaStream_t st) {
  const int n = kp.dim == 2 ? kp.ny : kp.nz;
  PSD_DISPATCH_N(n, (mid_impl<float, NN>(data, kp, ctrl, partials, xi, dspec, tb, st)));
}

cudaError_t init_dht_attributes_f32(int n) { PSD_DISPATCH_N(n, (set_attrs_T<float, NN>())); }

}  // namespace psd
