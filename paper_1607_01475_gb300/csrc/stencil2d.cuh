// 2D residual and line-search kernels: a warp owns a strip of 32 V cells along
// x (V per lane) and marches along y, with everything in registers and the
// x-neighbours by shuffle: no shared tiles, no barriers, no index divisions.
// Same unscaled arithmetic as the 3D column kernels (vertex-gradient sums
// G = g / q, Laplacian sums h^2 Delta_h).
//
// Window cell i of a strip is the grid cell x0 - 2 + i (periodic).  Per row, with
// D = u[i+1] - u[i] and A = u[i+1] + u[i]:
//   vertex (i + 1/2, y + 1/2):  G_x = D(y) + D(y+1),  G_y = A(y+1) - A(y);
//   lap'(i, y) = (D[i] - D[i-1]) + ((u(y-1) + u(y+1)) - 2 u(y));
//   with S = Phi_x(y-1/2) + Phi_x(y+1/2), E = Phi_y(y+1/2) - Phi_y(y-1/2):
//   div' = (S[i] - S[i-1]) + (E[i] + E[i-1]).
// Cells 2 .. 32 V - 3 of the window are the strip's outputs.  A march of TY rows
// reads 4 more for its start; TY is chosen so that every SM has several marches
// (res_geometry).  These grids live in L2, and the
// kernels are bound by the latency of a row's chain of shuffles and
// arithmetic.  The tiled kernels they replace took (event-timed) 18.6 us
// (residual) and 15 us (line search) on 1024^2 in FP32, and 23 us each on 64^2
// in FP64.
#pragma once

namespace psd {
namespace {

// Task of this warp: strip and march; false when there is none.
struct March2D {
  int x0, y0, ny;  // first output cell of the strip, rows y0 .. y0 + ny - 1
};
__device__ __forceinline__ bool march2d(const KParams& kp, int outputs, int ty, March2D& m) {
  const int task = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int nstrip = (kp.nx + outputs - 1) / outputs;
  const int chunk = task / nstrip;
  m.x0 = (task - chunk * nstrip) * outputs;
  m.y0 = chunk * ty;
  m.ny = ty;
  return m.y0 < kp.ny;
}

// V consecutive values of a row (8-byte aligned for V = 2).
template <int V>
__device__ __forceinline__ void load_row(const float* p, float (&v)[V]) {
  if constexpr (V == 2) {
    const float2 a = *reinterpret_cast<const float2*>(p);
    v[0] = a.x;
    v[1] = a.y;
  } else {
    v[0] = *p;
  }
}
template <int V>
__device__ __forceinline__ void load_row(const double* p, double (&v)[V]) {
#pragma unroll
  for (int k = 0; k < V; ++k) v[k] = p[k];
}
template <int V>
__device__ __forceinline__ void store_row(float* p, const float (&v)[V]) {
  if constexpr (V == 2)
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  else
    *p = v[0];
}
template <int V>
__device__ __forceinline__ void store_row(double* p, const double (&v)[V]) {
#pragma unroll
  for (int k = 0; k < V; ++k) p[k] = v[k];
}

// The value at the window cell after (before) each of this lane's cells.
template <int V, typename L>
__device__ __forceinline__ void right_of(const L (&v)[V], L (&out)[V]) {
#pragma unroll
  for (int k = 0; k + 1 < V; ++k) out[k] = v[k + 1];
  out[V - 1] = __shfl_down_sync(0xffffffffu, v[0], 1);
}
template <int V, typename L>
__device__ __forceinline__ void left_of(const L (&v)[V], L (&out)[V]) {
#pragma unroll
  for (int k = 1; k < V; ++k) out[k] = v[k - 1];
  out[0] = __shfl_up_sync(0xffffffffu, v[V - 1], 1);
}

// One march of the residual; FX and TRACK as in res3d_col.
template <typename T, int PK, int MODE, int V, bool FX>
__device__ __forceinline__ void res2d_march(const ResArgs<T>& a, const KParams& kp, const Ctrl* ctrl,
                                            const March2D& m, int fxs, int fxg, T& acc2, T& accm, unsigned& um,
                                            unsigned& gm) {
  constexpr bool INNER = MODE == RM_INNER, HVP = MODE == RM_HVP, BASE = MODE != RM_PLAIN;
  constexpr bool TRACK = sizeof(T) == 8 && MODE == RM_PLAIN && PK == PK_4;
  using L = typename std::conditional<FX, long long, T>::type;
  const int lane = threadIdx.x & 31;
  const int nx = kp.nx, ny = kp.ny;
  const bool upd = a.d != nullptr;
  const T alpha = upd ? (T)ctrl->alpha : T(0);
  const KConst<T>& C = kconst<T>(kp);
  const T cu = C.cu, cdiv = C.cdiv, cbih = C.cbih, beta = C.beta;
  const T cuq = FX ? cu * (T)fx_unit(fxs) : cu, cbihq = FX ? cbih * (T)fx_unit(fxs) : cbih;
  const T cdivq = FX ? cdiv * (T)fx_unit(3 * (fxs + fxg) - 125) : cdiv;
  const int i0 = lane * V;  // first window cell of this lane
  const int gx = (m.x0 + i0 - 2) & (nx - 1);
  const bool out = i0 >= 2 && i0 < 32 * V - 2 && m.x0 + i0 - 2 < nx;

  T pu[V], pd[V], pb[V], pf[V];  // rows in flight: u and d of row k, base of row k - 1, f of row k - 2
  auto fetch = [&](int k) {
    const size_t row = (size_t)(k & (ny - 1)) * nx + gx;
    load_row(a.u_in + row, pu);
    if (upd) load_row(a.d + row, pd);
    if (BASE) load_row(a.ubase + (size_t)((k - 1) & (ny - 1)) * nx + gx, pb);
    if (a.f != nullptr && k >= m.y0 + 2) load_row(a.f + (size_t)(k - 2) * nx + gx, pf);
  };
#pragma unroll
  for (int v = 0; v < V; ++v) pu[v] = pd[v] = pb[v] = pf[v] = T(0);
  L u0[V], u1[V], D0[V], D1[V], A0[V], A1[V], Lm[V], L0[V];
  T Db0[V], Ab0[V];
  L F0[2][V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    u0[v] = u1[v] = D0[v] = D1[v] = A0[v] = A1[v] = Lm[v] = L0[v] = F0[0][v] = F0[1][v] = L(0);
    Db0[v] = Ab0[v] = T(0);
  }
  fetch(m.y0 - 2);
  for (int k = m.y0 - 2; k < m.y0 + m.ny + 2; ++k) {
    // row k arrives: u2, its differences and sums along x
    T x[V], b[V], fc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      x[v] = upd ? pu[v] + alpha * pd[v] : pu[v];
      b[v] = pb[v];
      fc[v] = pf[v];
    }
    const bool own = out && k >= m.y0 && k < m.y0 + m.ny;
    if (upd && own) store_row(a.u_out + (size_t)k * nx + gx, x);
    if (k + 1 < m.y0 + m.ny + 2) fetch(k + 1);
    L u2[V], un[V], D2[V], A2[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if constexpr (FX)
        u2[v] = fx_quantise((unsigned)__double2hiint(x[v]), (unsigned)__double2loint(x[v]), 1077 - fxs, 55).v;
      else
        u2[v] = x[v];
      if constexpr (TRACK) {
        const int hi = FX ? (int)(fx_bits(u2[v]) >> 32) : (int)((unsigned)(fx_bits(u2[v]) >> 32) & 0x7FFFFFFFu);
        if (own) um = max(um, (unsigned)(hi < 0 ? -hi : hi));
      }
    }
    right_of<V>(u2, un);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      D2[v] = un[v] - u2[v];
      A2[v] = un[v] + u2[v];
    }
    T Db1[V], Ab1[V];
    if (BASE) {
      T bn[V];
      right_of<V>(b, bn);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        Db1[v] = bn[v] - b[v];
        Ab1[v] = bn[v] + b[v];
      }
    }
    // lap'(k - 1)
    L Dl[V], Lp[V];
    left_of<V>(D1, Dl);
#pragma unroll
    for (int v = 0; v < V; ++v) Lp[v] = (D1[v] - Dl[v]) + ((u0[v] + u2[v]) - (u1[v] + u1[v]));
    if (k > m.y0) {
      // flux at the vertices of row k - 3/2, and S, E with row k - 5/2
      L F[2][V], S[V], E[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        if constexpr (FX) {
          using ull = unsigned long long;
          const long long g0 = (long long)(((ull)D0[v] + (ull)D1[v]) << fxg);
          const long long g1 = (long long)(((ull)A1[v] - (ull)A0[v]) << fxg);
          long long Fv[3];
          const unsigned top = fx_flux(g0, g1, 0LL, Fv);
          if (i0 + v < 32 * V - 1) gm = max(gm, top);  // the window's last cell has no right neighbour
          F[0][v] = Fv[0];
          F[1][v] = Fv[1];
        } else {
          const T G[3] = {D0[v] + D1[v], A1[v] - A0[v], T(0)};
          T Fv[3];
          if constexpr (BASE) {
            const T Ab[3] = {Db0[v] + Db1[v], Ab1[v] - Ab0[v], T(0)};
            if (INNER)
              flux_diff<PK>(Ab, G, beta, Fv);
            else
              flux_lin<PK>(Ab, G, beta, Fv);
          } else if constexpr (TRACK) {
            const T g2 = G[0] * G[0] + G[1] * G[1];
            if (i0 + v < 32 * V - 1) gm = max(gm, (unsigned)__double2hiint(g2));
            Fv[0] = g2 * G[0];
            Fv[1] = g2 * G[1];
          } else {
            flux<PK>(G, beta, Fv);
          }
          F[0][v] = Fv[0];
          F[1][v] = Fv[1];
        }
        S[v] = F0[0][v] + F[0][v];
        E[v] = F[1][v] - F0[1][v];
        F0[0][v] = F[0][v];
        F0[1][v] = F[1][v];
      }
      if (k >= m.y0 + 2) {
        // residual of row y = k - 2
        L Sl[V], El[V], Ll[V], Lr[V];
        left_of<V>(S, Sl);
        left_of<V>(E, El);
        left_of<V>(L0, Ll);
        right_of<V>(L0, Lr);
        T r[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const L divl = (S[v] - Sl[v]) + (E[v] + El[v]);
          const L bihl = ((Ll[v] + Lr[v]) + (Lm[v] + Lp[v])) - (L(2) * L0[v] + L(2) * L0[v]);
          T uc, bih, div;
          if constexpr (FX) {
            uc = fx_result(u0[v], 0);
            bih = fx_result(bihl, 0);
            div = fx_result(divl, 0);
          } else {
            uc = u0[v];
            bih = bihl;
            div = divl;
          }
          if (INNER)
            r[v] = fc[v] - ((cu * uc + cbih * bih) - cdiv * div);
          else if (HVP)
            r[v] = (cu * uc + cbih * bih) - cdiv * div;
          else
            r[v] = FX ? fma(cdivq, div, fma(-cbihq, bih, fma(-cuq, uc, fc[v])))
                      : (fc[v] - cuq * uc) + (cdivq * div - cbihq * bih);
          if (out) {
            acc2 += HVP ? uc * r[v] : r[v] * r[v];
            accm = max_abs(accm, r[v]);
          }
        }
        if constexpr (V == 1) {
          if (out) store_r<MODE>(a, (size_t)(k - 2) * nx + gx, r[0]);
        } else {
          if (out) store_row(a.r + (size_t)(k - 2) * nx + gx, r);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      Lm[v] = L0[v];
      L0[v] = Lp[v];
      u0[v] = u1[v];
      u1[v] = u2[v];
      D0[v] = D1[v];
      D1[v] = D2[v];
      A0[v] = A1[v];
      A1[v] = A2[v];
      if (BASE) {
        Db0[v] = Db1[v];
        Ab0[v] = Ab1[v];
      }
    }
  }
}

template <typename T, int PK, int MODE, int V>
__global__ void __launch_bounds__(kWarps2D * 32)
    k_res2d(ResArgs<T> a, KParams kp, Ctrl* ctrl, double* partials, int ty) {
  if (ctrl->done) return;
  constexpr bool TRACK = sizeof(T) == 8 && MODE == RM_PLAIN && PK == PK_4;
  __shared__ T sred[red_size<T>(2)];
  __shared__ unsigned smax[2];
  __shared__ int sflag;
  March2D m;
  T acc2 = T(0), accm = T(0);
  unsigned um = 0u, gm = 0u;
  int fxs = kFxOff, fxg = 0;
  if (TRACK && a.fixed) {
    fxs = ctrl->fx_s;
    fxg = ctrl->fx_g;
  }
  if (march2d(kp, 32 * V - 4, ty, m)) {
    bool fixed = false;
    if constexpr (TRACK) {
      if (fxs != kFxOff) {
        res2d_march<T, PK, MODE, V, true>(a, kp, ctrl, m, fxs, fxg, acc2, accm, um, gm);
        fixed = true;
      }
    }
    if (!fixed) res2d_march<T, PK, MODE, V, false>(a, kp, ctrl, m, 0, 0, acc2, accm, um, gm);
  }
  if constexpr (TRACK) track_publish(um, gm, fxs, fxg, fxs != kFxOff && a.d == nullptr, ctrl, smax);
  T v[2] = {acc2, accm};
  block_reduce<T, 2, true>(v, sred);
  if (publish_and_check_last<T>(v, 2, reinterpret_cast<T*>(partials), &ctrl->counter[CS_RES], &sflag)) {
    T tt[2];
    gather_partials<T, 2, true>(tt, reinterpret_cast<const T*>(partials), sred);
    if (threadIdx.x == 0) {
      if constexpr (TRACK) track_collect(ctrl);
      residual_epilogue(ctrl, kp, (double)tt[0], (double)tt[1], a.norm, a.update_iter, MODE == RM_HVP);
    }
  }
}

// Line search: the vertices (x + 1/2, y + 1/2) of the strip's first 32 V - V cells.
template <typename T, int PK, bool INNER, int V, bool FX>
__device__ __forceinline__ void ls2d_march(const T* __restrict__ u, const T* __restrict__ ubase,
                                           const T* __restrict__ d, const KParams& kp, T trial, const March2D& m,
                                           int Su, int Sd, T (&acc)[ls_nsums<PK>()], T& sbb, unsigned& gm) {
  constexpr bool TRACK = sizeof(T) == 8 && PK == PK_4 && !INNER;
  using L = typename std::conditional<FX, long long, T>::type;
  const T beta = kconst<T>(kp).beta, pm2 = kconst<T>(kp).pm2;
  const int lane = threadIdx.x & 31, nx = kp.nx, ny = kp.ny;
  const int i0 = lane * V;
  const int gx = (m.x0 + i0) & (nx - 1);
  const bool out = lane < 31 && m.x0 + i0 < nx;
  T pu[V], pb[V], pd[V];
#pragma unroll
  for (int v = 0; v < V; ++v) pb[v] = T(0);
  auto fetch = [&](int k) {
    const size_t row = (size_t)(k & (ny - 1)) * nx + gx;
    load_row(u + row, pu);
    if (INNER) load_row(ubase + row, pb);
    load_row(d + row, pd);
  };
  auto enter = [&](T x, int S) -> L {
    if constexpr (FX)
      return fx_quantise((unsigned)__double2hiint(x), (unsigned)__double2loint(x), 1077 - S, 55).v;
    else
      return x;
  };
  L Du0[V], Au0[V], Dd0[V], Ad0[V];
#pragma unroll
  for (int v = 0; v < V; ++v) Du0[v] = Au0[v] = Dd0[v] = Ad0[v] = L(0);
  fetch(m.y0);
  for (int k = m.y0; k <= m.y0 + m.ny; ++k) {
    L uc[V], dc[V], un[V], dn[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      uc[v] = enter(INNER ? pu[v] + pb[v] : pu[v], Su);
      dc[v] = enter(pd[v], Sd);
    }
    if (k < m.y0 + m.ny) fetch(k + 1);
    right_of<V>(uc, un);
    right_of<V>(dc, dn);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const L Du = un[v] - uc[v], Au = un[v] + uc[v], Dd = dn[v] - dc[v], Ad = dn[v] + dc[v];
      if (out && k > m.y0) {
        if constexpr (FX) {
          gm = max(gm, fx_ls_accumulate(Du0[v] + Du, Au - Au0[v], 0LL, Dd0[v] + Dd, Ad - Ad0[v], 0LL, acc, sbb));
        } else {
          const T av[3] = {Du0[v] + Du, Au - Au0[v], T(0)}, bv[3] = {Dd0[v] + Dd, Ad - Ad0[v], T(0)};
          if constexpr (TRACK)
            gm = max(gm, ls_accumulate4(av, bv, acc, sbb));
          else
            ls_accumulate<PK>(av, bv, trial, beta, pm2, acc);
        }
      }
      Du0[v] = Du;
      Au0[v] = Au;
      Dd0[v] = Dd;
      Ad0[v] = Ad;
    }
  }
}

template <typename T, int PK, bool INNER, int V>
__global__ void __launch_bounds__(kWarps2D * 32)
    k_ls2d(const T* __restrict__ u, const T* __restrict__ ubase, const T* __restrict__ d, KParams kp, Ctrl* ctrl,
           double* partials, int ty) {
  if (ctrl->done) return;
  if (!ls_closed_form<PK>() && ctrl->c3 != 0.0) return;  // Newton already converged
  constexpr bool TRACK = sizeof(T) == 8 && PK == PK_4 && !INNER;
  __shared__ T sred[red_size<T>(ls_nsums<PK>())];
  __shared__ unsigned smax[2];
  __shared__ int sflag;
  const T trial = ls_closed_form<PK>() ? T(0) : (T)ctrl->trial;
  T acc[ls_nsums<PK>()] = {};
  T sbb = T(0);
  unsigned gm = 0u;
  int Su = 0, Sd = 0;
  bool fixed = false;
  if constexpr (TRACK) fixed = ls_scales(ctrl, &Su, &Sd);
  March2D m;
  if (march2d(kp, 31 * V, ty, m)) {
    if constexpr (TRACK) {
      if (fixed) ls2d_march<T, PK, INNER, V, true>(u, ubase, d, kp, trial, m, Su, Sd, acc, sbb, gm);
    }
    if (!fixed) ls2d_march<T, PK, INNER, V, false>(u, ubase, d, kp, trial, m, 0, 0, acc, sbb, gm);
  }
  if constexpr (TRACK) ls_track(acc, sbb, gm, fixed, Su, Sd, ctrl, smax);
  ls_finish<T, PK>(acc, sred, partials, ctrl, kp, &sflag, TRACK);
}

}  // namespace
}  // namespace psd
