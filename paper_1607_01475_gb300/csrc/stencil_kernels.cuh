// Residual and line-search kernels of the PSD iteration (included by the
// per-vertex-factor translation units k_res_p3.cu, k_res_p4.cu, k_res_p6.cu
// and k_res_pgen.cu, each of which instantiates one kind):
//   r = f - N_h[u],  N_h[u] = cu u - s d.(|D u|^{p-2} D u) + s eps^2 Delta_h^2 u
// (Eq. "discrete-4th-order", Sec. 5.3; the local part of the sixth-order
// operator of Sec. 5.4 / 6.2 with cu = s lambda), fused with the deferred
// update u <- u + alpha d (Eq. "eq:psd4"); and the line-search reduction that
// gives the step size alpha as the root of q(alpha) = (N_h[u + alpha d] - f, d)_2
// (Eq. "eqn-search", Sec. 6.1).
//
// D is the centre-to-vertex gradient and d. the vertex-to-centre divergence
// of Sec. 5.1; in 3D the tensor extension (D_x A_y A_z, d_x a_y a_z).  A CTA
// owns a TX x TY column of cells and marches along z keeping rolling planes
// of u (5, halo 2 in x/y), of Delta_h u (3, halo 1) and of the vertex fluxes
// (2 vertex planes) in shared memory.  Every vertex flux and every Laplacian
// value is computed once per CTA.
#pragma once

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <type_traits>

#include "fx_line.cuh"
#include "stencil_geom.h"

namespace psd {
namespace {

// |g|^{p-2} from g2 = |g|^2: g2 (p = 4), g2^2 (p = 6), its root (p = 3), else
// pow.
template <int PK, typename T>
__device__ __forceinline__ T vfactor(T g2, T beta) {
  if (PK == PK_4) return g2;
  if (PK == PK_6) return g2 * g2;
  if (PK == PK_3) return sqrt(g2);
  return pow(g2, beta);  // beta = (p-2)/2; pow(0, 0) = 1, pow(0, b>0) = 0
}

// Flux difference F(a + e) - F(a), F(g) = |g|^{p-2} g, in a form whose
// rounding error scales with |e| (no cancellation of F(a) against itself).
template <int PK, typename T>
__device__ __forceinline__ void flux_diff(const T (&a)[3], const T (&e)[3], T beta, T (&out)[3]) {
  const T a2 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2];
  // |a+e|^2 - |a|^2 = (2a + e).e, formed from e
  const T dl = (T(2) * a[0] + e[0]) * e[0] + (T(2) * a[1] + e[1]) * e[1] + (T(2) * a[2] + e[2]) * e[2];
  const T c2 = a2 + dl;  // |a+e|^2
  if (PK == PK_4) {
    // |a+e|^2 (a+e) - |a|^2 a = |a+e|^2 e + (|a+e|^2 - |a|^2) a
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = c2 * e[c] + dl * a[c];
  } else if (PK == PK_6) {
    // |a+e|^4 (a+e) - |a|^4 a = |a+e|^4 e + (|a+e|^2 - |a|^2)(|a+e|^2 + |a|^2) a
    const T c4 = c2 * c2, w = dl * (c2 + a2);
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = c4 * e[c] + w * a[c];
  } else if (PK == PK_3) {
    // |a+e| e + (|a+e| - |a|) a, the difference of the roots from dl
    const T na = sqrt(a2), nc = sqrt(c2 > T(0) ? c2 : T(0)), den = na + nc;
    const T w = den > T(0) ? dl / den : T(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = nc * e[c] + w * a[c];
  } else {
    const T fc = pow(c2 > T(0) ? c2 : T(0), beta);
    T dfac;  // |a+e|^{p-2} - |a|^{p-2}
    if (a2 > T(0))
      dfac = pow(a2, beta) * expm1(beta * log1p(dl / a2));
    else
      dfac = fc;
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = fc * e[c] + dfac * a[c];
  }
}

template <int PK, typename T>
__device__ __forceinline__ void flux(const T (&g)[3], T beta, T (&out)[3]) {
  const T g2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
  const T f = vfactor<PK>(g2, beta);
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c] = f * g[c];
}

// Linearised flux W(a) e = |a|^{p-2} e + (p-2)|a|^{p-4} (a.e) a (the second
// variation of Sec. 5.3; the (p-2)-term is 0 where a = 0 for p < 4).
template <int PK, typename T>
__device__ __forceinline__ void flux_lin(const T (&a)[3], const T (&e)[3], T beta, T (&out)[3]) {
  const T a2 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2];
  const T ae = a[0] * e[0] + a[1] * e[1] + a[2] * e[2];
  if (PK == PK_4) {
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = a2 * e[c] + T(2) * ae * a[c];
  } else if (PK == PK_6) {
    // |a|^4 e + 4 |a|^2 (a.e) a
    const T a4 = a2 * a2, w = T(4) * a2 * ae;
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = a4 * e[c] + w * a[c];
  } else if (PK == PK_3) {
    // |a| e + (a.e) / |a| a
    const T na = sqrt(a2), w = na > T(0) ? ae / na : T(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = na * e[c] + w * a[c];
  } else {
    const T f = pow(a2, beta);
    const T w = (a2 > T(0)) ? T(2) * beta * pow(a2, beta - T(1)) * ae : T(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = f * e[c] + w * a[c];
  }
}

// Store a residual value (FP64 plain: or, for the mixed solver, its FP32 rounding
// twice).
template <int MODE, typename T>
__device__ __forceinline__ void store_r(const ResArgs<T>& a, size_t i, T r) {
  if constexpr (sizeof(T) == 8 && MODE == RM_PLAIN) {
    if (a.r32 != nullptr) {
      a.r32[i] = (float)r;
      a.r32b[i] = (float)r;
      return;
    }
  }
  a.r[i] = r;
}

// Last-block bookkeeping of the residual kernel.
__device__ void residual_epilogue(Ctrl* ctrl, const KParams& kp, double sum2, double maxabs, int norm,
                                  int update_iter, bool hvp = false) {
  if (hvp) {
    const double pq = sum2 * kp.hd;  // (v, H v)_2
    ctrl->c1 = pq;
    ctrl->c2 = maxabs;
    if (ctrl->cg) {
      // CG step length alpha = (r, z) / (p, H p); H is positive definite
      // (the second variation, Sec. 5.3), so pq <= 0 means a breakdown
      if (pq > 0.0 && isfinite(pq)) {
        ctrl->alpha = ctrl->rz / pq;
      } else {
        ctrl->status = 7;
        ctrl->done = 1;
      }
    }
    ctrl->counter[CS_RES] = 0;
    return;
  }
  if (update_iter) {
    const int it = ctrl->iter;
    if (ctrl->hist_alpha != nullptr && it < ctrl->hist_cap) ctrl->hist_alpha[it] = ctrl->alpha;
    ctrl->iter = it + 1;
  }
  if (norm) {
    const double res = sqrt(sum2 * kp.hd);
    ctrl->res_l2 = res;
    ctrl->res_linf = maxabs;
    const int it = ctrl->iter;
    if (ctrl->hist_res != nullptr && it < ctrl->hist_cap) ctrl->hist_res[it] = res;
    if (!isfinite(res)) {
      ctrl->status = 7;
      ctrl->done = 1;
    } else if (res < ctrl->tol) {
      ctrl->status = 0;
      ctrl->done = 1;
    } else if (it >= ctrl->max_iter) {
      ctrl->status = 4;
      ctrl->done = 1;
    }
  }
  ctrl->counter[CS_RES] = 0;
}

// ------------------------------------------------------------- 3D residual
template <typename T, int PK, int MODE>
__global__ void __launch_bounds__(NT)
    k_res3d(ResArgs<T> a, KParams kp, Ctrl* ctrl, double* partials, int zc) {
  if (ctrl->done) return;
  constexpr int SXM = BX + 4, SYM = BY3 + 4;
  constexpr int NB = (MODE != RM_PLAIN) ? 2 : 1;
  __shared__ T su[5][SYM][SXM];
  __shared__ T sb[NB][SYM][SXM];
  __shared__ T sl[3][BY3 + 2][BX + 2];
  __shared__ T sf[2][3][BY3 + 1][BX + 1];
  __shared__ T sred[red_size<T>(2)];
  __shared__ int sflag;

  const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
  const int TX = nx < BX ? nx : BX, TY = ny < BY3 ? ny : BY3;
  const int SX = TX + 4, SY = TY + 4;
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * zc;
  const size_t plane = (size_t)nx * ny;
  const bool upd = a.d != nullptr;
  const T alpha = upd ? (T)ctrl->alpha : T(0);
  const KConst<T>& C = kconst<T>(kp);
  const T ih = C.inv_h, ih2 = ih * ih, q4 = T(0.25) * ih;
  const T s = C.s, se2 = C.se2, cu = C.cu;
  const T beta = C.beta;

  auto uslot = [&](int zz) { return (zz - z0 + 2) % 5; };
  auto lslot = [&](int zz) { return (zz - z0 + 1) % 3; };
  auto fslot = [&](int zz) { return (zz - z0 + 1) & 1; };  // vertex plane zz + 1/2
  auto bslot = [&](int zz) { return (zz - z0 + 2) & 1; };

  auto load_plane = [&](int zz) {
    const int sl_ = uslot(zz);
    const size_t gz = (size_t)wrapi(zz, nz) * plane;
    const bool own = (zz >= z0) && (zz < z0 + zc);
    for (int idx = tid; idx < SX * SY; idx += NT) {
      const int ly = idx / SX, lx = idx - ly * SX;
      const int gx = wrapi(x0 + lx - 2, nx), gy = wrapi(y0 + ly - 2, ny);
      const size_t g = gz + (size_t)gy * nx + gx;
      T v = a.u_in[g];
      if (upd) {
        v = v + alpha * a.d[g];
        if (own && lx >= 2 && lx < TX + 2 && ly >= 2 && ly < TY + 2) a.u_out[g] = v;
      }
      su[sl_][ly][lx] = v;
    }
  };
  auto load_base = [&](int zz) {
    if (MODE == RM_PLAIN) return;
    const int sl_ = bslot(zz);
    const size_t gz = (size_t)wrapi(zz, nz) * plane;
    for (int idx = tid; idx < SX * SY; idx += NT) {
      const int ly = idx / SX, lx = idx - ly * SX;
      const int gx = wrapi(x0 + lx - 2, nx), gy = wrapi(y0 + ly - 2, ny);
      sb[sl_ % NB][ly][lx] = a.ubase[gz + (size_t)gy * nx + gx];
    }
  };
  auto comp_lap = [&](int zz) {
    const int cm = uslot(zz - 1), c0 = uslot(zz), cp = uslot(zz + 1), ls = lslot(zz);
    const int LX = TX + 2, LY = TY + 2;
    for (int idx = tid; idx < LX * LY; idx += NT) {
      const int ly = idx / LX, lx = idx - ly * LX;
      const T c = su[c0][ly + 1][lx + 1];
      const T sum = (su[c0][ly + 1][lx] + su[c0][ly + 1][lx + 2]) + (su[c0][ly][lx + 1] + su[c0][ly + 2][lx + 1]) +
                    (su[cm][ly + 1][lx + 1] + su[cp][ly + 1][lx + 1]);
      sl[ls][ly][lx] = (sum - T(6) * c) * ih2;
    }
  };
  auto grad8 = [&](T (&fld)[SYM][SXM], T (&fld1)[SYM][SXM], int vy, int vx, T (&g)[3]) {
    const T u000 = fld[vy + 1][vx + 1], u001 = fld[vy + 1][vx + 2];
    const T u010 = fld[vy + 2][vx + 1], u011 = fld[vy + 2][vx + 2];
    const T u100 = fld1[vy + 1][vx + 1], u101 = fld1[vy + 1][vx + 2];
    const T u110 = fld1[vy + 2][vx + 1], u111 = fld1[vy + 2][vx + 2];
    g[0] = q4 * (((u001 - u000) + (u011 - u010)) + ((u101 - u100) + (u111 - u110)));
    g[1] = q4 * (((u010 - u000) + (u011 - u001)) + ((u110 - u100) + (u111 - u101)));
    g[2] = q4 * (((u100 - u000) + (u101 - u001)) + ((u110 - u010) + (u111 - u011)));
  };
  auto comp_flux = [&](int zz) {  // vertex plane zz + 1/2
    const int c0 = uslot(zz), c1 = uslot(zz + 1), fs = fslot(zz);
    const int VX = TX + 1, VY = TY + 1;
    for (int idx = tid; idx < VX * VY; idx += NT) {
      const int vy = idx / VX, vx = idx - vy * VX;
      T g[3], F[3];
      grad8(su[c0], su[c1], vy, vx, g);
      if (MODE != RM_PLAIN) {
        T ab[3];
        grad8(sb[bslot(zz) % NB], sb[bslot(zz + 1) % NB], vy, vx, ab);
        if (MODE == RM_INNER)
          flux_diff<PK>(ab, g, beta, F);
        else
          flux_lin<PK>(ab, g, beta, F);
      } else {
        flux<PK>(g, beta, F);
      }
      sf[fs][0][vy][vx] = F[0];
      sf[fs][1][vy][vx] = F[1];
      sf[fs][2][vy][vx] = F[2];
    }
  };

  T acc2 = T(0), accm = T(0);
  auto comp_out = [&](int zz) {
    const int lm = lslot(zz - 1), l0 = lslot(zz), lp = lslot(zz + 1);
    const int fm = fslot(zz - 1), fp = fslot(zz), c0 = uslot(zz);
    const size_t gz = (size_t)wrapi(zz, nz) * plane;
    for (int idx = tid; idx < TX * TY; idx += NT) {
      const int ty = idx / TX, tx = idx - ty * TX;
      const T bih = (((sl[l0][ty + 1][tx] + sl[l0][ty + 1][tx + 2]) + (sl[l0][ty][tx + 1] + sl[l0][ty + 2][tx + 1])) +
                     (sl[lm][ty + 1][tx + 1] + sl[lp][ty + 1][tx + 1]) - T(6) * sl[l0][ty + 1][tx + 1]) *
                    ih2;
      const T dx = q4 * (((sf[fm][0][ty][tx + 1] - sf[fm][0][ty][tx]) + (sf[fm][0][ty + 1][tx + 1] - sf[fm][0][ty + 1][tx])) +
                         ((sf[fp][0][ty][tx + 1] - sf[fp][0][ty][tx]) + (sf[fp][0][ty + 1][tx + 1] - sf[fp][0][ty + 1][tx])));
      const T dy = q4 * (((sf[fm][1][ty + 1][tx] - sf[fm][1][ty][tx]) + (sf[fm][1][ty + 1][tx + 1] - sf[fm][1][ty][tx + 1])) +
                         ((sf[fp][1][ty + 1][tx] - sf[fp][1][ty][tx]) + (sf[fp][1][ty + 1][tx + 1] - sf[fp][1][ty][tx + 1])));
      const T dz = q4 * (((sf[fp][2][ty][tx] - sf[fm][2][ty][tx]) + (sf[fp][2][ty][tx + 1] - sf[fm][2][ty][tx + 1])) +
                         ((sf[fp][2][ty + 1][tx] - sf[fm][2][ty + 1][tx]) + (sf[fp][2][ty + 1][tx + 1] - sf[fm][2][ty + 1][tx + 1])));
      const T div = dx + dy + dz;
      const T uc = su[c0][ty + 2][tx + 2];
      const size_t g = gz + (size_t)(y0 + ty) * nx + (x0 + tx);
      T r;
      if (MODE == RM_INNER)
        r = (a.f ? a.f[g] : T(0)) - ((cu * uc + se2 * bih) - s * div);
      else if (MODE == RM_HVP)
        r = (cu * uc + se2 * bih) - s * div;
      else
        r = (a.f ? a.f[g] : T(0)) - cu * uc + s * div - se2 * bih;
      store_r<MODE>(a, g, r);
      acc2 += (MODE == RM_HVP) ? uc * r : r * r;
      accm = max_abs(accm, r);
    }
  };

  // prologue: planes z0-2 .. z0+1, Laplacians at z0-1, z0, fluxes at z0-1/2
  for (int zz = z0 - 2; zz <= z0 + 1; ++zz) load_plane(zz);
  load_base(z0 - 1);
  load_base(z0);
  __syncthreads();
  comp_lap(z0 - 1);
  comp_lap(z0);
  comp_flux(z0 - 1);
  // base slot of z0 - 1, read just above, is the one the first step refills
  if (MODE != RM_PLAIN) __syncthreads();
  for (int z = z0; z < z0 + zc; ++z) {
    load_plane(z + 2);
    load_base(z + 1);
    __syncthreads();
    comp_lap(z + 1);
    comp_flux(z);
    __syncthreads();
    comp_out(z);
  }

  T v[2] = {acc2, accm};
  block_reduce<T, 2, true>(v, sred);
  if (publish_and_check_last<T>(v, 2, reinterpret_cast<T*>(partials), &ctrl->counter[CS_RES], &sflag)) {
    T tt[2];
    gather_partials<T, 2, true>(tt, reinterpret_cast<const T*>(partials), sred);
    double tot[2];
    for (int m_ = 0; m_ < 2; ++m_) tot[m_] = (double)tt[m_];
    if (tid == 0) residual_epilogue(ctrl, kp, tot[0], tot[1], a.norm, a.update_iter, MODE == RM_HVP);
  }
}

// The fixed-point variants' bookkeeping (see fx_decide).  track_publish: the
// block's bounds on |u| and |G|^2 (um, gm: largest high words, of integers in
// units of 2^-fxs and of the flux's |G|^2 when fxs is a scale, of FP64 values
// otherwise) into the running maxima of ctrl; scanned: ctrl->umax is the bound of this
// very iterate, from its scan, and 0 there leaves both at 0 (the integers' unit would
// bound it by 2^-23, and the next scales would be too coarse for a solution much
// smaller than that).  track_collect, in the last block: the maxima become the
// iterate's bounds.
__device__ __forceinline__ void track_publish(unsigned um, unsigned gm, int fxs, int fxg, bool scanned, Ctrl* ctrl,
                                              unsigned* smax) {
  block_max2(um, gm, smax);
  if (threadIdx.x == 0 && !(scanned && ctrl->umax == 0.0)) {
    const bool fx = fxs != kFxOff;
    const double ub = fx ? ((double)um + 1.0) * fx_unit(fxs - 32) : __hiloint2double((int)um, -1);
    const double g2 = fx ? ((double)gm + 1.0) * fx_unit(2 * (fxs + fxg) - 96) : __hiloint2double((int)gm, -1);
    atomicMax(&ctrl->umax_hi, (unsigned)__double2hiint(ub) + 1u);
    atomicMax(&ctrl->gmax2_hi, (unsigned)__double2hiint(g2) + 1u);
  }
}
__device__ __forceinline__ void track_collect(Ctrl* ctrl) {
  ctrl->umax = __hiloint2double((int)atomicExch(&ctrl->umax_hi, 0u), 0);
  ctrl->gmax = fx_sqrt_above(atomicExch(&ctrl->gmax2_hi, 0u));
}

// ------------------------------------------------------------ line search
// alpha = root of q(alpha) = -rd + lin alpha + sum_{j=1..5} c_j alpha^j, the
// polynomial form of q(alpha) = (N_h[u + alpha d] - f, d)_2 for p = 4 (a
// cubic) and p = 6 (a quintic) of Sec. 6.1, with the s factor folded into
// c_j.  q(0) = -rd < 0 and q is strictly increasing (Sec. 2.3), so the root
// is unique; Newton's method with a bisection safeguard on a bracket.
//
// One thread runs this at the end of the line search, where every dependent
// FP64 operation takes 65 clocks and a division about 1000 (the plain FP64 Newton
// iteration took 7 us of the 1024^2 line search's 11).  So the iteration is done
// in FP32 on x = alpha / alpha_0, alpha_0 = rd / q'(0), where Q(x) = q / rd = -1 + x
// + e_1 x^2 + .. is of order one, and finished by two FP64 Newton steps with FP32
// quotients: the first leaves about 1e-13, the second is below rounding.
// newton_x: false when that does not settle (then the plain iteration decides).
// K: the coefficients e_1 .. e_{K-1}.
template <int K>
__device__ __forceinline__ bool newton_x(const double (&e)[4], double* x_out) {
  float f[K - 1];
#pragma unroll
  for (int j = 0; j < K - 1; ++j) f[j] = (float)e[j];
  auto qf = [&](float x) {
    float v = f[K - 2];
#pragma unroll
    for (int j = K - 3; j >= 0; --j) v = fmaf(x, v, f[j]);
    return fmaf(x, fmaf(x, v, 1.0f), -1.0f);
  };
  auto df = [&](float x) {
    float v = (float)K * f[K - 2];
#pragma unroll
    for (int j = K - 3; j >= 0; --j) v = fmaf(x, v, (float)(j + 2) * f[j]);
    return fmaf(x, v, 1.0f);
  };
  float lo = 0.0f, hi = 1.0f;
  for (int i = 0; i < 40 && !(qf(hi) > 0.0f); ++i) {
    lo = hi;
    hi *= 2.0f;
  }
  float xf = hi;
  for (int it = 0; it < 40; ++it) {
    const float q = qf(xf);
    if (q < 0.0f)
      lo = xf;
    else
      hi = xf;
    float nx = xf - __fdividef(q, df(xf));
    if (!(lo < nx && nx < hi)) nx = 0.5f * (lo + hi);
    const bool settled = fabsf(nx - xf) <= 4e-7f * nx;
    xf = nx;
    if (settled) break;
  }
  double x = (double)xf;
  float step = 0.0f;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    double v = e[K - 2];
#pragma unroll
    for (int j = K - 3; j >= 0; --j) v = fma(x, v, e[j]);
    step = __fdividef((float)fma(x, fma(x, v, 1.0), -1.0), df((float)x));
    x -= (double)step;
  }
  *x_out = x;
  return x > 0.0 && fabsf(step) <= 1e-9f * (float)x && df((float)x) > 0.0f;
}
// K: the degree of q.
template <int K>
__device__ double solve_poly_alpha(double rd, double lin, const double (&c)[5], int* status) {
  auto q = [&](double al) { return -rd + al * (lin + c[0] + al * (c[1] + al * (c[2] + al * (c[3] + al * c[4])))); };
  auto dq = [&](double al) {
    return lin + c[0] + al * (2.0 * c[1] + al * (3.0 * c[2] + al * (4.0 * c[3] + al * 5.0 * c[4])));
  };
  const double d0 = dq(0.0);
  if (!(rd > 0.0) || !(d0 > 0.0) || !isfinite(rd) || !isfinite(d0)) {
    *status = (isfinite(rd) && isfinite(d0)) ? 0 : 7;
    return 0.0;
  }
  {
    const double r0 = recip_pos(d0), a0 = rd * r0, a2 = a0 * a0;
    double e[4] = {c[1] * (a0 * r0), c[2] * (a2 * r0), 0.0, 0.0};
    if (K == 5) {
      e[2] = c[3] * (a2 * a0 * r0);
      e[3] = c[4] * (a2 * a2 * r0);
    }
    double x;
    // FP32 range: |e| below 2^60
    const unsigned top = max(max((unsigned)__double2hiint(e[0]) & 0x7FFFFFFFu, (unsigned)__double2hiint(e[1]) & 0x7FFFFFFFu),
                             max((unsigned)__double2hiint(e[2]) & 0x7FFFFFFFu, (unsigned)__double2hiint(e[3]) & 0x7FFFFFFFu));
    if (top < (1083u << 20) && newton_x<K>(e, &x)) return a0 * x;
  }
  double lo = 0.0, hi = -1.0;
  double alpha = rd / d0;
  double b = alpha;
  for (int i = 0; i < 200; ++i) {
    if (q(b) > 0.0) {
      hi = b;
      break;
    }
    lo = b;
    b *= 2.0;
  }
  if (hi < 0.0) {
    *status = 7;
    return alpha;
  }
  alpha = fmin(fmax(alpha, lo), hi);
  for (int it = 0; it < 200; ++it) {
    const double qa = q(alpha);
    if (qa == 0.0) return alpha;
    if (qa < 0.0)
      lo = alpha;
    else
      hi = alpha;
    const double step = qa / dq(alpha);
    if (fabs(step) <= 4e-16 * fabs(alpha)) return alpha - step;  // Newton step below rounding
    double nw = alpha - step;
    if (!(lo < nw && nw < hi)) nw = 0.5 * (lo + hi);
    if (hi - lo <= 4e-16 * hi) return nw;
    alpha = nw;
  }
  return alpha;
}

// Whether the line search of this vertex-factor kind is one pass (p = 4, 6:
// the coefficients of a polynomial q) or one pass per Newton step (general
// p: P(alpha) - P(0) and P'(alpha) at a trial alpha), and how many vertex
// sums a pass reduces.
template <int PK>
__host__ __device__ constexpr bool ls_closed_form() {
  return PK == PK_4 || PK == PK_6;
}
template <int PK>
__host__ __device__ constexpr int ls_nsums() {
  return PK == PK_6 ? 5 : (PK == PK_4 ? 3 : 2);
}

// Whether 2 x < y for x, y >= 0 (FP64: from the high words, an FP64 comparison takes
// the slot of an addition).
__device__ __forceinline__ bool below_half(float x, float y) { return 2.0f * x < y; }
__device__ __forceinline__ bool below_half(double x, double y) {
  return __double2hiint(x) + 0x100000 < __double2hiint(y);
}

// Vertex sums for one vertex with a = grad u (+ grad ubase), b = grad d.
// With A = |a|^2, B = a.b, C = |b|^2, the vertex term of P(alpha) =
// sum_v |a + alpha b|^{p-2} (a + alpha b).b is (A + 2 alpha B + alpha^2 C)^k
// (B + alpha C) for p = 2k + 2; its alpha^j coefficients (j >= 1) are summed:
//   p = 4: AC + 2B^2, 3BC, C^2;
//   p = 6: A^2 C + 4AB^2, 6ABC + 4B^3, 8B^2 C + 2AC^2, 5BC^2, C^3.
template <int PK, typename T>
__device__ __forceinline__ void ls_accumulate(const T (&av)[3], const T (&bv)[3], T trial, T beta, T pm2,
                                              T (&acc)[ls_nsums<PK>()]) {
  if (PK == PK_4 || PK == PK_6) {
    const T A = av[0] * av[0] + av[1] * av[1] + av[2] * av[2];
    const T B = av[0] * bv[0] + av[1] * bv[1] + av[2] * bv[2];
    const T C = bv[0] * bv[0] + bv[1] * bv[1] + bv[2] * bv[2];
    if (PK == PK_4) {
      acc[0] += A * C + T(2) * B * B;
      acc[1] += T(3) * B * C;
      acc[2] += C * C;
    } else {
      const T B2 = B * B, C2 = C * C;
      acc[0] += A * (A * C + T(4) * B2);
      acc[1] += B * (T(6) * A * C + T(4) * B2);
      acc[ls_nsums<PK>() - 3] += C * (T(8) * B2 + T(2) * A * C);
      acc[ls_nsums<PK>() - 2] += T(5) * B * C2;
      acc[ls_nsums<PK>() - 1] += C * C2;
    }
  } else {
    // with e = trial b, c = a + e: (F(c) - F(a)).b = |c|^{p-2} trial C + (|c|^{p-2} -
    // |a|^{p-2}) B, and its derivative |c|^{p-2} C + (p-2) |c|^{p-4} (c.b)^2
    const T A = av[0] * av[0] + av[1] * av[1] + av[2] * av[2];
    const T B = av[0] * bv[0] + av[1] * bv[1] + av[2] * bv[2];
    const T C = bv[0] * bv[0] + bv[1] * bv[1] + bv[2] * bv[2];
    const T c[3] = {av[0] + trial * bv[0], av[1] + trial * bv[1], av[2] + trial * bv[2]};
    const T c2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
    const T cb = B + trial * C, dl = trial * (B + cb);  // |c|^2 - |a|^2
    T fc, dfac, w;  // |c|^{p-2}, its difference from |a|^{p-2}, (p-2) |c|^{p-4}
    if (PK == PK_3) {
      const T na = sqrt(A);
      fc = sqrt(c2);
      dfac = na + fc > T(0) ? dl / (na + fc) : T(0);
      w = fc > T(0) ? T(1) / fc : T(0);
    } else {
      fc = pow(c2, beta);
      // from dl where |c| is close to |a|; where it is much smaller, dl / A + 1 has lost it,
      // and with it |c|^{p-2}, up to eps^{(p-2)/2} |a|^{p-2}
      const T fa = pow(A, beta);
      dfac = below_half(c2, A) ? fc - fa : (A > T(0) ? fa * expm1(beta * log1p(fmax(dl / A, T(-1)))) : fc);
      w = c2 > T(0) ? pm2 * fc / c2 : T(0);
    }
    acc[0] += fc * trial * C + dfac * B;
    acc[1] += fc * C + w * cb * cb;
  }
}

// p = 4 with the coefficients' constant factors (2, 3) left to the sums: AC, BC,
// C^2 into acc, B^2 into sbb.  Returns the high word of C.
template <typename T, int M>
__device__ __forceinline__ unsigned ls_accumulate4(const T (&av)[3], const T (&bv)[3], T (&acc)[M], T& sbb) {
  const T A = fma(av[2], av[2], fma(av[1], av[1], av[0] * av[0]));
  const T B = fma(av[2], bv[2], fma(av[1], bv[1], av[0] * bv[0]));
  const T C = fma(bv[2], bv[2], fma(bv[1], bv[1], bv[0] * bv[0]));
  acc[0] = fma(A, C, acc[0]);
  sbb = fma(B, B, sbb);
  acc[1] = fma(B, C, acc[1]);
  acc[2] = fma(C, C, acc[2]);
  return (unsigned)__double2hiint(C);
}
// The same from integer gradients a, b (moduli below 2^61): A, B and C are
// integer products of the gradients shifted to full length, each within a few
// 2^-57 of |a||a|, |a||b|, |b||b|; only the four accumulations are FP64.
template <int M>
__device__ __forceinline__ unsigned fx_ls_accumulate(long long a0, long long a1, long long a2, long long b0,
                                                     long long b1, long long b2, double (&acc)[M], double& sbb) {
  // leading zeros of the largest component, by the ones' complement magnitudes
  auto shift = [](long long x, long long y, long long z) {
    const unsigned long long m = (unsigned long long)((x ^ (x >> 63)) | (y ^ (y >> 63)) | (z ^ (z >> 63))) | 1ULL;
    return __clzll((long long)m) - 4;  // components below 2^60, moduli below 2^61 after the shift
  };
  const int sa = shift(a0, a1, a2), sb = shift(b0, b1, b2);
  const fx_halves x0 = fx_split(fx_shl(a0, sa)), x1 = fx_split(fx_shl(a1, sa)), x2 = fx_split(fx_shl(a2, sa));
  const fx_halves y0 = fx_split(fx_shl(b0, sb)), y1 = fx_split(fx_shl(b1, sb)), y2 = fx_split(fx_shl(b2, sb));
  auto square = [](const fx_halves& p, const fx_halves& q, const fx_halves& r) {
    const long long t = fx_wide(p.h, p.l) + (fx_wide(q.h, q.l) + (fx_wide(r.h, r.l) + (1LL << 30)));
    return fx_wide(p.h, p.h) + (fx_wide(q.h, q.h) + (fx_wide(r.h, r.h) + (t >> 31)));
  };
  const long long ia = square(x0, x1, x2), ic = square(y0, y1, y2);
  const long long t0 = fx_wide(x0.h, y0.l) + (fx_wide(x1.h, y1.l) + (fx_wide(x2.h, y2.l) + (1LL << 31)));
  const long long t1 = fx_wide(x0.l, y0.h) + (fx_wide(x1.l, y1.h) + fx_wide(x2.l, y2.h));
  const long long ib = fx_wide(x0.h, y0.h) + (fx_wide(x1.h, y1.h) + (fx_wide(x2.h, y2.h) + ((t0 + t1) >> 32)));
  const double A = fx_result(ia, 64 - 2 * sa), B = fx_result(ib, 64 - sa - sb), C = fx_result(ic, 64 - 2 * sb);
  acc[0] = fma(A, C, acc[0]);
  sbb = fma(B, B, sbb);
  acc[1] = fma(B, C, acc[1]);
  acc[2] = fma(C, C, acc[2]);
  return (unsigned)__double2hiint(C);
}
// Scales of u and d for the fixed-point line search from the bounds in ctrl.
__device__ __forceinline__ bool ls_scales(const Ctrl* ctrl, int* Su, int* Sd) {
  return ctrl->umax >= 0.0 && fx_scale_of(ctrl->umax, Su) && fx_scale_of(__hiloint2double((int)ctrl->dmax_hi, 0), Sd);
}
// The p = 4 sums with their factors and units, and the block's bound on |grad d|^2.
template <typename T, int M>
__device__ __forceinline__ void ls_track(T (&acc)[M], T sbb, unsigned gm, bool fixed, int Su, int Sd, Ctrl* ctrl,
                                         unsigned* smax) {
  acc[0] = acc[0] + T(2) * sbb;
  acc[1] = T(3) * acc[1];
  if (fixed) {  // powers of two
    acc[0] *= (T)fx_unit(2 * (Su + Sd));
    acc[1] *= (T)fx_unit(Su + 3 * Sd);
    acc[2] *= (T)fx_unit(4 * Sd);
  }
  unsigned none = 0u;
  block_max2(gm, none, smax);
  if (threadIdx.x == 0) {
    const double g2 = __hiloint2double((int)gm, -1) * (fixed ? fx_unit(2 * Sd) : 1.0);
    atomicMax(&ctrl->gmax2_hi, (unsigned)__double2hiint(g2) + 1u);
  }
}

// Whether the Newton step `step` from `trial` (both moduli) is the general-p line
// search's last: what it leaves has to be below rounding.  For p >= 3, q' is
// Lipschitz and the step after one of length e is M e^2, M = step / prev^2 from the last
// two (prev: the move before, 0 on the first pass, where trial stands for it), so
// step^3 / prev^2 is left.  For 2 < p < 3, q' is only Hoelder continuous: where the
// gradients vanish at the root, Newton contracts by up to (p - 2) / (p - 1) a pass,
// and step^2 / prev bounds what is left at every rate.  A limit on the step alone
// (5e-9) left alpha 1e-10 off there.  Steps that stop contracting are rounding.  FP32
// sums give an alpha that is used rounded to FP32.
__device__ __forceinline__ bool newton_settled(double step, double trial, double prev, bool smooth, bool f32) {
  if (!(step <= (f32 ? 1e-4 : 5e-9) * trial)) return false;
  if (step <= (f32 ? 2e-7 : 4e-16) * trial) return true;
  if (prev > 0.0 && step >= 0.7 * prev) return true;
  const double left = (f32 ? 1e-8 : 1e-16) * trial;
  if (!smooth) return step * step <= left * prev;
  const double e = prev > 0.0 ? prev : trial;
  return step * step * step <= left * (e * e);
}

// Last-block logic of the line search (f32: the sums are FP32's).
template <int PK>
__device__ void linesearch_epilogue(Ctrl* ctrl, const KParams& kp, const double (&tot)[ls_nsums<PK>()], bool f32) {
  const double lin = ctrl->lin;
  if (ls_closed_form<PK>()) {
    int st = 0;
    // the kernels sum unscaled vertex gradients G = g / q: s g^p-terms = cdiv G^p-terms
    double c[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int j = 0; j < ls_nsums<PK>(); ++j) c[j] = kp.cdiv * kp.hd * tot[j];
    const double al = solve_poly_alpha<ls_nsums<PK>()>(ctrl->rd, lin, c, &st);
    ctrl->c1 = c[0];
    ctrl->c2 = c[1];
    ctrl->c3 = c[2];
    ctrl->alpha = al;
    if (st != 0) {
      ctrl->status = st;
      ctrl->done = 1;
    }
  } else {
    // one safeguarded Newton step per launch; state in c1 (lo), c2 (hi), c3 (done
    // flag); the first trial is the previous iteration's step size.
    const double trial = f32 ? (double)(float)ctrl->trial : ctrl->trial;
    const double qv = -ctrl->rd + trial * lin + kp.cdiv * kp.hd * tot[0];
    const double dqv = lin + kp.cdiv * kp.hd * tot[1];
    double lo = ctrl->c1, hi = ctrl->c2;
    if (qv < 0.0)
      lo = trial;
    else if (qv > 0.0)
      hi = trial;
    const double step = (dqv > 0.0) ? qv * recip_pos(dqv) : 0.0;
    double nw = (dqv > 0.0) ? trial - step : 0.5 * (lo + hi);
    const bool tiny = (dqv > 0.0) && newton_settled(fabs(step), fabs(trial), ctrl->ls_step, kp.p >= 3.0, f32);
    if (!tiny) {
      if (hi > 0.0) {
        if (!(lo < nw && nw < hi)) nw = 0.5 * (lo + hi);
      } else if (!(nw > lo)) {
        nw = 2.0 * (lo > 0.0 ? lo : 1.0);
      }
    }
    if (qv == 0.0 || tiny || (hi > 0.0 && hi - lo <= 4e-16 * hi)) {
      ctrl->c3 = 1.0;  // converged
      nw = (qv == 0.0) ? trial : nw;
    }
    ctrl->c1 = lo;
    ctrl->c2 = hi;
    ctrl->ls_step = fabs(nw - trial);
    ctrl->alpha = nw;
    ctrl->trial = nw;
    if (!isfinite(nw) || !isfinite(qv)) {
      ctrl->status = 7;
      ctrl->done = 1;
    }
  }
  ctrl->counter[CS_LS] = 0;
}

// Block and grid reduction of a line-search pass (fixed order; the last
// block runs the epilogue).  track: the scales of the residual that
// follows are chosen from the bounds in ctrl (fx_decide).  sred:
// red_size<T>(ls_nsums<PK>()) shared elements.
template <typename T, int PK>
__device__ __forceinline__ void ls_finish(T (&acc)[ls_nsums<PK>()], T* sred, double* partials, Ctrl* ctrl,
                                          const KParams& kp, int* sflag, bool track = false) {
  constexpr int M = ls_nsums<PK>();
  block_reduce<T, M, false>(acc, sred);
  if (publish_and_check_last<T>(acc, M, reinterpret_cast<T*>(partials), &ctrl->counter[CS_LS], sflag)) {
    T tt[M];
    gather_partials<T, M, false>(tt, reinterpret_cast<const T*>(partials), sred);
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    if (tid == 0) {
      double tot[M];
#pragma unroll
      for (int m = 0; m < M; ++m) tot[m] = (double)tt[m];
      linesearch_epilogue<PK>(ctrl, kp, tot, sizeof(T) == 4);
      if (track) {
        // the next iterate u + alpha d: |u| and |G| are at most these
        const double al = fabs(ctrl->alpha), gd = fx_sqrt_above(atomicExch(&ctrl->gmax2_hi, 0u));
        fx_decide(ctrl, kp, ctrl->umax + al * __hiloint2double((int)ctrl->dmax_hi, 0), ctrl->gmax + al * gd, 0.0);
      }
    }
  }
}

}  // namespace
}  // namespace psd
#include "stencil2d.cuh"
#include "stencil3d_col.cuh"
#include "stencil3d_march.cuh"
#include "stencil3d_rb.cuh"
namespace psd {
namespace {

template <typename T, int PK, bool INNER>
__global__ void __launch_bounds__(NT)
    k_ls3d(const T* __restrict__ u, const T* __restrict__ ubase, const T* __restrict__ d, KParams kp, Ctrl* ctrl,
           double* partials, int zc) {
  if (ctrl->done) return;
  if (!ls_closed_form<PK>() && ctrl->c3 != 0.0) return;  // Newton already converged
  constexpr int SXM = BX + 1, SYM = BY3 + 1;
  __shared__ T su[2][SYM][SXM];
  __shared__ T sd[2][SYM][SXM];
  __shared__ T sred[red_size<T>(ls_nsums<PK>())];
  __shared__ int sflag;
  const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
  const int TX = nx < BX ? nx : BX, TY = ny < BY3 ? ny : BY3;
  const int SX = TX + 1, SY = TY + 1;
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * zc;
  const size_t plane = (size_t)nx * ny;
  const T beta = kconst<T>(kp).beta, pm2 = kconst<T>(kp).pm2;
  const T trial = ls_closed_form<PK>() ? T(0) : (T)ctrl->trial;
  auto load = [&](int zz) {
    const int sl_ = (zz - z0) & 1;
    const size_t gz = (size_t)wrapi(zz, nz) * plane;
    for (int idx = tid; idx < SX * SY; idx += NT) {
      const int ly = idx / SX, lx = idx - ly * SX;
      const size_t g = gz + (size_t)wrapi(y0 + ly, ny) * nx + wrapi(x0 + lx, nx);
      T v = u[g];
      if (INNER) v += ubase[g];
      su[sl_][ly][lx] = v;
      sd[sl_][ly][lx] = d[g];
    }
  };
  auto grad = [&](T (&f0)[SYM][SXM], T (&f1)[SYM][SXM], int vy, int vx, T (&g)[3]) {
    const T u000 = f0[vy][vx], u001 = f0[vy][vx + 1], u010 = f0[vy + 1][vx], u011 = f0[vy + 1][vx + 1];
    const T u100 = f1[vy][vx], u101 = f1[vy][vx + 1], u110 = f1[vy + 1][vx], u111 = f1[vy + 1][vx + 1];
    g[0] = ((u001 - u000) + (u011 - u010)) + ((u101 - u100) + (u111 - u110));
    g[1] = ((u010 - u000) + (u011 - u001)) + ((u110 - u100) + (u111 - u101));
    g[2] = ((u100 - u000) + (u101 - u001)) + ((u110 - u010) + (u111 - u011));
  };
  T acc[ls_nsums<PK>()] = {};
  load(z0);
  for (int z = z0; z < z0 + zc; ++z) {
    load(z + 1);
    __syncthreads();
    const int s0 = (z - z0) & 1, s1 = (z + 1 - z0) & 1;
    for (int idx = tid; idx < TX * TY; idx += NT) {
      const int vy = idx / TX, vx = idx - vy * TX;
      T av[3], bv[3];
      grad(su[s0], su[s1], vy, vx, av);
      grad(sd[s0], sd[s1], vy, vx, bv);
      ls_accumulate<PK>(av, bv, trial, beta, pm2, acc);
    }
    __syncthreads();
  }
  ls_finish<T, PK>(acc, sred, partials, ctrl, kp, &sflag);
}

}  // namespace

namespace detail {

// Whether every pointer is 8-byte aligned.
template <typename... P>
bool aligned8(const P*... p) {
  return ((reinterpret_cast<unsigned long long>(p) | ...) & 7ull) == 0;
}

template <typename T, int PK, int MODE>
cudaError_t res_impl(const ResArgs<T>& a, const KParams& kp, Ctrl* ctrl, double* partials, cudaStream_t st) {
  const ResGeom g = residual_geometry(kp, sizeof(T) == 4, aligned8(a.u_in, a.d, a.u_out, a.f, a.ubase, a.r));
  switch (g.kind) {
    case RK_MARCH:
      if constexpr (sizeof(T) == 4) k_res3d_march<T, PK, MODE><<<g.grid, g.threads, 0, st>>>(a, kp, ctrl, partials);
      break;
    case RK_RB4:
      if constexpr (sizeof(T) == 4) k_res3d_rb<T, PK, MODE, 4><<<g.grid, NT, 0, st>>>(a, kp, ctrl, partials);
      break;
    case RK_COL:
      if constexpr (sizeof(T) == 8) k_res3d_col<T, PK, MODE><<<g.grid, NT, 0, st>>>(a, kp, ctrl, partials);
      break;
    case RK_SMALL3D:
      if constexpr (sizeof(T) == 8) k_res3d<T, PK, MODE><<<g.grid, NT, 0, st>>>(a, kp, ctrl, partials, g.zc);
      break;
    default:
      if constexpr (sizeof(T) == 4) {
        if (g.zc < 0) {  // two cells per lane
          k_res2d<T, PK, MODE, 2><<<g.grid, g.threads, 0, st>>>(a, kp, ctrl, partials, -g.zc);
          break;
        }
      }
      k_res2d<T, PK, MODE, 1><<<g.grid, g.threads, 0, st>>>(a, kp, ctrl, partials, g.zc);
  }
  return cudaGetLastError();
}

template <typename T, int PK, bool INNER>
cudaError_t ls_impl(const T* u, const T* ubase, const T* d, const KParams& kp, Ctrl* ctrl, double* partials,
                    cudaStream_t st) {
  // the same tiles as the residual; __launch_bounds__(256, 3)
  const ResGeom g = res_geometry(kp, sizeof(T) == 4, 3, true, aligned8(u, ubase, d));
  switch (g.kind) {
    case RK_MARCH:
      if constexpr (sizeof(T) == 4)
        k_ls3d_march<T, PK, INNER><<<g.grid, g.threads, 0, st>>>(u, ubase, d, kp, ctrl, partials);
      break;
    case RK_RB4:
      if constexpr (sizeof(T) == 4) k_ls3d_rb<T, PK, INNER, 4><<<g.grid, NT, 0, st>>>(u, ubase, d, kp, ctrl, partials);
      break;
    case RK_COL:
      if constexpr (sizeof(T) == 8) k_ls3d_col<T, PK, INNER><<<g.grid, NT, 0, st>>>(u, ubase, d, kp, ctrl, partials);
      break;
    case RK_SMALL3D:
      if constexpr (sizeof(T) == 8) k_ls3d<T, PK, INNER><<<g.grid, NT, 0, st>>>(u, ubase, d, kp, ctrl, partials, g.zc);
      break;
    default:
      if constexpr (sizeof(T) == 4) {
        if (g.zc < 0) {
          k_ls2d<T, PK, INNER, 2><<<g.grid, g.threads, 0, st>>>(u, ubase, d, kp, ctrl, partials, -g.zc);
          break;
        }
      }
      k_ls2d<T, PK, INNER, 1><<<g.grid, g.threads, 0, st>>>(u, ubase, d, kp, ctrl, partials, g.zc);
  }
  return cudaGetLastError();
}


}  // namespace detail
}  // namespace psd
