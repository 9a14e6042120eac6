// Launch geometry of the residual and line-search kernels, shared by the
// translation units that instantiate them (one per kind of vertex factor)
// and by the dispatching launchers.
#pragma once

#include "kernels.h"

namespace psd {

constexpr int BX = 32;   // tile width (x)
constexpr int BY3 = 8;   // tile height (y), 3D
constexpr int kWarps2D = 4;  // most marches (warps) per block, 2D
constexpr int NT = 256;  // threads per block
// 3D FP32 marches: most warps (four rows each) per CTA, CTAs per SM
constexpr int kMarchWarps = 4, kMarchResCtas = 2, kMarchLsCtas = 5;

enum ResKind { RK_2D, RK_SMALL3D, RK_COL, RK_RB4, RK_MARCH };
struct ResGeom {
  int kind;
  dim3 grid;
  int zc;  // general 3D kernel: planes per CTA; 2D: rows per march (negative: two cells per lane)
  int threads;
};
// linesearch: the strips of the 2D line search; pairs: 2D FP32 fields aligned to
// 8 bytes (two cells per lane on wide grids).  Geometry for a kernel whose __launch_bounds__ guarantee ctas_per_sm
// resident CTAs per SM (defined in k_stencil.cu).
ResGeom res_geometry(const KParams& kp, bool fp32, int ctas_per_sm, bool linesearch = false, bool pairs = true);
// The residual launch: k_res3d_rb keeps 2 CTAs per SM resident, k_res3d_col 3.
ResGeom residual_geometry(const KParams& kp, bool fp32, bool pairs = true);

namespace detail {
// Residual and line-search launchers for one vertex-factor kind PK (PK_4,
// PK_3, PK_6 or PK_GEN), explicitly instantiated by k_res_p3.cu, k_res_p4.cu, k_res_p6.cu and
// k_res_pgen.cu.
template <typename T, int PK, int MODE>
cudaError_t res_impl(const ResArgs<T>& a, const KParams& kp, Ctrl* ctrl, double* partials, cudaStream_t st);
template <typename T, int PK, bool INNER>
cudaError_t ls_impl(const T* u, const T* ubase, const T* d, const KParams& kp, Ctrl* ctrl, double* partials,
                    cudaStream_t st);
}  // namespace detail

}  // namespace psd
