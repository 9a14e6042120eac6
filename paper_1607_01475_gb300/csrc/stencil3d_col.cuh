// Column-owning 3D kernels (tiles of 32 x 8; nx >= 32, ny >= 8): the
// residual and the line-search reduction, organised for a low operation
// count (GB300 issues FP64 at 1/64 of the FP32 rate, so the FP64 variants
// are bound by their operation count).
//
// Arithmetic (same operators as Sec. 5.1 with the tensor reading in 3D):
//  * vertex gradient g = q G, q = 1/(4h), from per-cell z-pair sums
//    P = u(z) + u(z+1) and differences M = u(z+1) - u(z) of the two cell
//    planes around the vertex plane:
//      G_x = (P[x+1,y] - P[x,y]) + (P[x+1,y+1] - P[x,y+1])
//      G_y = (P[x,y+1] - P[x,y]) + (P[x+1,y+1] - P[x+1,y])
//      G_z = (M[x,y] + M[x+1,y]) + (M[x,y+1] + M[x+1,y+1]);
//  * flux Phi = |G|^{p-2} G (|g|^{p-2} g = q^{p-1} Phi);
//  * divergence from per-vertex z-sums S_c = Phi_c(z-1/2) + Phi_c(z+1/2)
//    (c = x, y) and D_z = Phi_z(z+1/2) - Phi_z(z-1/2), so that
//    s d.(|g|^{p-2} g) = cdiv * div', cdiv = s q^p;
//  * Laplacian sums lap' = h^2 Delta_h u, bih' = h^4 Delta_h^2 u.
//
// Each thread owns one (x, y) column and marches in z; z-neighbours are
// kept in registers, xy-neighbours go through shared memory, and the next
// plane's global loads are issued a step ahead.
//
// Residual, per step z (output plane z):
//   P/M of the vertex plane z+1/2 from the register history of U(z),
//   U(z+1) (and of the base field B); store U(z+2)          -> sync
//   prefetch U(z+3), B(z+2), f(z+1)
//   lap'(z+1) over tile + halo 1 -> sL ring
//   Phi(z+1/2) at own (+ halo) vertex; S/D with Phi(z-1/2) -> sS
//   -> sync -> residual at plane z.
// U = u_in + alpha d (the fused update; the owner writes it to u_out);
// B = the base field of the correction form (RM_INNER only).
#pragma once

namespace psd {
namespace {

// Shared memory of the column residual (one set for both of its variants).
template <typename T, int MODE>
struct ResColSmem {
  static constexpr int TX = 32, TY = 8;
  static constexpr bool BASE = MODE != RM_PLAIN;
  T sU[3][TY + 4][TX + 4];
  T sL[2][TY + 2][TX + 2];
  T sP[TY + 2][TX + 2];
  T sM[TY + 2][TX + 2];
  T sPb[BASE ? TY + 2 : 1][BASE ? TX + 2 : 1];
  T sMb[BASE ? TY + 2 : 1][BASE ? TX + 2 : 1];
  T sS[3][TY + 1][TX + 1];
  T sred[red_size<T>(2)];
  unsigned smax[2];
  int sflag;
};

// FX (FP64, plain mode, p = 4): no FP64 arithmetic before the final
// combination but the update u + alpha d.  Each u enters as the 64-bit integer
// q = round(u 2^S), |q| < 2^55 (S from a bound on |u|), and the z-pair sums,
// vertex gradients and both Laplacian passes are exact integer sums
// (|h^4 Delta_h^2 q| <= 144 2^55 < 2^63).  The z-pair sums are stored shifted left
// by g, modulo 2^64, so that the gradients G 2^(S+g), whose modulus is below
// 2^61 by a bound on |G|, use all 64 bits; the flux |G|^2 G is two rounds of
// products kept to their high 64 bits (units of 2^-58 of the largest flux), its
// z-sums and divergence are integer sums below 2^63.  Only
// r = (f - cu u) + (cdiv div - cbih bih) and the norms are FP64.
// The linear part is that of u rounded to 2^-56 of max|u|, below the rounding
// of the FP64 Laplacian sums it replaces; the variant runs when the flux part's
// worst-case error is below those roundings too (fx_decide).  FP64 issues at
// 1/64 of the FP32 rate: at 256^3 the all-FP64 kernel takes 1.88 ms, this one
// 0.53 ms (0.57 with the maximum as an FP64 comparison and four operations in r).
//
// TRACK (both variants of that case): the largest |u| and |G| of the new
// iterate go to ctrl for the next scales.
template <typename T, int PK, int MODE, bool FX>
__device__ __forceinline__ void res3d_col(const ResArgs<T>& a, const KParams& kp, Ctrl* ctrl, double* partials,
                                          ResColSmem<T, MODE>& sm, int fxs, int fxg) {
  constexpr bool TRACK = sizeof(T) == 8 && MODE == RM_PLAIN && PK == PK_4;
  static_assert(!FX || TRACK, "FX: FP64 plain p = 4 only");
  using LT = typename std::conditional<FX, long long, T>::type;  // arithmetic of the linear part and the flux
  constexpr int TX = 32, TY = 8;
  constexpr int UX = TX + 4, UY = TY + 4, UN = UX * UY;  // U tile, halo 2
  constexpr int LX = TX + 2, LY = TY + 2, LN = LX * LY;  // halo-1 tile (Laplacian, P/M)
  constexpr int VX = TX + 1, VY = TY + 1;                // vertex tile
  constexpr bool INNER = MODE == RM_INNER;
  constexpr bool HVP = MODE == RM_HVP;
  constexpr bool BASE = MODE != RM_PLAIN;  // a base field B enters the flux
  constexpr int NLH = 2 * LX + 2 * TY;                   // Laplacian halo cells (84)
  constexpr int NVH = VY + TX;                           // vertex halo (41)
  // FX: the tiles hold 64-bit integers in the 8 bytes of an FP64 value
  LT(*sU)[UY][UX] = reinterpret_cast<LT(*)[UY][UX]>(&sm.sU[0][0][0]);
  LT(*sL)[LY][LX] = reinterpret_cast<LT(*)[LY][LX]>(&sm.sL[0][0][0]);
  LT(*sP)[LX] = reinterpret_cast<LT(*)[LX]>(&sm.sP[0][0]);
  LT(*sM)[LX] = reinterpret_cast<LT(*)[LX]>(&sm.sM[0][0]);
  LT(*SS)[VY][VX] = reinterpret_cast<LT(*)[VY][VX]>(&sm.sS[0][0][0]);
  auto& sPb = sm.sPb;
  auto& sMb = sm.sMb;

  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
  const size_t plane = (size_t)nx * ny;
  const bool upd = a.d != nullptr;
  const T alpha = upd ? (T)ctrl->alpha : T(0);
  const KConst<T>& C = kconst<T>(kp);
  const T cdiv = C.cdiv, cbih = C.cbih, cu = C.cu;
  const T beta = C.beta;
  // FX: cu, cbih and cdiv carry the units of q, of h^4 Delta_h^2 q and of the
  // divergence (flux units of 2^(125 - 3 (S + g)))
  const T cuq = FX ? cu * (T)fx_unit(fxs) : cu, cbihq = FX ? cbih * (T)fx_unit(fxs) : cbih;
  const T cdivq = FX ? cdiv * (T)fx_unit(3 * (fxs + fxg) - 125) : cdiv;
  const int fxE = 1077 - fxs;  // biased exponent of 2^(55 - S)
  unsigned um = 0u, gm = 0u;   // TRACK: largest |u| and |G|^2, high words (FX: of the integers)

  // One wave of CTAs: the column-planes (w = column * nz + z) are split
  // into equal contiguous shares, each marched as one or more z-segments
  // with their own prologue; columns map to tiles in lockstep order
  // (lockstep_tile).
  const int gx = nx / TX;
  const int ncol = gx * (ny / TY);
  const int wtot = ncol * nz;
  const int wend = (int)((long long)wtot * (blockIdx.x + 1) / gridDim.x);
  const int mls = lockstep_classes(gridDim.x, ncol);
  T acc2 = T(0), accm = T(0);
  for (int w = (int)((long long)wtot * blockIdx.x / gridDim.x); w < wend;) {
    const int col = w / nz, z0 = w - col * nz;
    const int zc = min(nz - z0, wend - w);
    w += zc;
    const int tile = lockstep_tile(col, mls, ncol);
    const int x0 = (tile % gx) * TX, y0 = (tile / gx) * TY;

    // this thread's U-tile elements (flattened e = tid, tid + 256) and where
    // they land in the halo-1 P/M tile
    int uoff[2], upm[2];
    bool uval[2], uown[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int e = tid + 256 * k;
      uval[k] = e < UN;
      const int ly = e / UX, lx = e - ly * UX;
      uoff[k] = ((y0 + ly - 2) & (ny - 1)) * nx + ((x0 + lx - 2) & (nx - 1));
      uown[k] = uval[k] && lx >= 2 && lx < TX + 2 && ly >= 2 && ly < TY + 2;
      upm[k] = (uval[k] && ly >= 1 && ly <= LY && lx >= 1 && lx <= LX) ? (ly - 1) * LX + (lx - 1) : -1;
    }
    int boff[2];
    bool bval[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int e = tid + 256 * k;
      bval[k] = BASE && e < LN;
      const int ly = e / LX, lx = e - ly * LX;
      boff[k] = ((y0 + ly - 1) & (ny - 1)) * nx + ((x0 + lx - 1) & (nx - 1));
    }
    const int gown = (y0 + ty) * nx + x0 + tx;

    T pu[2] = {T(0), T(0)}, pd[2] = {T(0), T(0)}, pb[2] = {T(0), T(0)};
    LT h1[2] = {LT(0), LT(0)}, h0[2] = {LT(0), LT(0)};  // U history: h1 newest stored plane, h0 the one before
    T bprev[2] = {T(0), T(0)};
    auto fetchU = [&](int zz) {
      const size_t gz = (size_t)(zz & (nz - 1)) * plane;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (uval[k]) {
          pu[k] = a.u_in[gz + uoff[k]];
          if (upd) pd[k] = a.d[gz + uoff[k]];
        }
    };
    // store the prefetched plane zz into ring slot `slot` and shift the
    // register history (h0 <- h1 <- new)
    auto storeU = [&](int zz, int slot) {
      const size_t gz = (size_t)(zz & (nz - 1)) * plane;
      const bool ownplane = zz >= z0 && zz < z0 + zc;
      LT* dst = &sU[slot][0][0];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (uval[k]) {
          T x = pu[k];
          if (upd) {
            x = x + alpha * pd[k];
            if (ownplane && uown[k]) a.u_out[gz + uoff[k]] = x;
          }
          LT v;
          if constexpr (FX) {
            const unsigned hi = (unsigned)__double2hiint(x);
            v = fx_quantise(hi, (unsigned)__double2loint(x), fxE, 55).v;
          } else {
            v = x;
          }
          if constexpr (TRACK) {
            const int hi = FX ? (int)(fx_bits(v) >> 32) : (int)((unsigned)(fx_bits(v) >> 32) & 0x7FFFFFFFu);
            if (ownplane && uown[k]) um = max(um, (unsigned)(hi < 0 ? -hi : hi));
          }
          dst[tid + 256 * k] = v;
          h0[k] = h1[k];
          h1[k] = v;
        }
    };
    // P/M of the vertex plane between the two newest history planes
    auto storePM = [&]() {
      LT* P = &sP[0][0];
      LT* M = &sM[0][0];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (upm[k] >= 0) {
          if constexpr (FX) {  // modulo 2^64: only the gradients need to fit
            P[upm[k]] = (long long)((unsigned long long)(h0[k] + h1[k]) << fxg);
            M[upm[k]] = (long long)((unsigned long long)(h1[k] - h0[k]) << fxg);
          } else {
            P[upm[k]] = h0[k] + h1[k];
            M[upm[k]] = h1[k] - h0[k];
          }
        }
    };
    auto fetchB = [&](int zz) {
      if (!BASE) return;
      const size_t gz = (size_t)(zz & (nz - 1)) * plane;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (bval[k]) pb[k] = a.ubase[gz + boff[k]];
    };
    // base P/M between bprev and the prefetched plane (first: only record)
    auto storeB = [&](bool first) {
      if (!BASE) return;
      T* P = &sPb[0][0];
      T* M = &sMb[0][0];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (bval[k]) {
          if (!first) {
            P[tid + 256 * k] = bprev[k] + pb[k];
            M[tid + 256 * k] = pb[k] - bprev[k];
          }
          bprev[k] = pb[k];
        }
    };
    // h^2 Delta_h U at halo-1 cell (ly, lx) of the plane in slot s0
    auto lap_at = [&](int ly, int lx, int sm, int s0, int sp) -> LT {
      const LT c = sU[s0][ly + 1][lx + 1];
      const LT sum = (sU[s0][ly + 1][lx] + sU[s0][ly + 1][lx + 2]) + (sU[s0][ly][lx + 1] + sU[s0][ly + 2][lx + 1]) +
                     (sU[sm][ly + 1][lx + 1] + sU[sp][ly + 1][lx + 1]);
      return sum - LT(6) * c;
    };
    auto halo_lap_cell = [&](int h, int& ly, int& lx) {
      if (h < LX) {
        ly = 0;
        lx = h;
      } else if (h < 2 * LX) {
        ly = LY - 1;
        lx = h - LX;
      } else if (h < 2 * LX + TY) {
        ly = 1 + h - 2 * LX;
        lx = 0;
      } else {
        ly = 1 + h - 2 * LX - TY;
        lx = LX - 1;
      }
    };
    auto lap_plane = [&](int sm, int s0, int sp, int ls) -> LT {
      const LT own = lap_at(ty + 1, tx + 1, sm, s0, sp);
      sL[ls][ty + 1][tx + 1] = own;
      const int h = tid - (256 - NLH);
      if (h >= 0) {
        int ly, lx;
        halo_lap_cell(h, ly, lx);
        sL[ls][ly][lx] = lap_at(ly, lx, sm, s0, sp);
      }
      return own;
    };
    // Phi at vertex (vy, vx) of the current vertex plane (from sP/sM)
    auto vphi = [&](int vy, int vx, LT (&F)[3]) {
      if constexpr (FX) {
        using ull = unsigned long long;
        auto P = [&](int y, int x) { return (ull)sP[y][x]; };
        auto M = [&](int y, int x) { return (ull)sM[y][x]; };
        const long long g0 = (long long)((P(vy, vx + 1) - P(vy, vx)) + (P(vy + 1, vx + 1) - P(vy + 1, vx)));
        const long long g1 = (long long)((P(vy + 1, vx) - P(vy, vx)) + (P(vy + 1, vx + 1) - P(vy, vx + 1)));
        const long long g2 = (long long)((M(vy, vx) + M(vy, vx + 1)) + (M(vy + 1, vx) + M(vy + 1, vx + 1)));
        gm = max(gm, fx_flux(g0, g1, g2, F));
        return;
      } else {
        T G[3];
        G[0] = (sP[vy][vx + 1] - sP[vy][vx]) + (sP[vy + 1][vx + 1] - sP[vy + 1][vx]);
        G[1] = (sP[vy + 1][vx] - sP[vy][vx]) + (sP[vy + 1][vx + 1] - sP[vy][vx + 1]);
        G[2] = (sM[vy][vx] + sM[vy][vx + 1]) + (sM[vy + 1][vx] + sM[vy + 1][vx + 1]);
        if (BASE) {
          T A[3];
          A[0] = (sPb[vy][vx + 1] - sPb[vy][vx]) + (sPb[vy + 1][vx + 1] - sPb[vy + 1][vx]);
          A[1] = (sPb[vy + 1][vx] - sPb[vy][vx]) + (sPb[vy + 1][vx + 1] - sPb[vy][vx + 1]);
          A[2] = (sMb[vy][vx] + sMb[vy][vx + 1]) + (sMb[vy + 1][vx] + sMb[vy + 1][vx + 1]);
          if (INNER)
            flux_diff<PK>(A, G, beta, F);
          else
            flux_lin<PK>(A, G, beta, F);
        } else if constexpr (TRACK) {
          const T g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
          gm = max(gm, (unsigned)__double2hiint(g2));
#pragma unroll
          for (int c = 0; c < 3; ++c) F[c] = g2 * G[c];
        } else {
          flux<PK>(G, beta, F);
        }
      }
    };
    // own vertex (ty+1, tx+1) and, for tid < NVH, one halo vertex
    const bool hv = tid < NVH;
    const int hvy = tid < VY ? tid : 0;
    const int hvx = tid < VY ? 0 : tid - VY + 1;
    LT Fo[3] = {LT(0), LT(0), LT(0)}, Fh[3] = {LT(0), LT(0), LT(0)};  // Phi of the previous vertex plane
    auto phi_plane = [&](bool first) {
      LT F[3];
      vphi(ty + 1, tx + 1, F);
      if (!first) {
        SS[0][ty + 1][tx + 1] = Fo[0] + F[0];
        SS[1][ty + 1][tx + 1] = Fo[1] + F[1];
        SS[2][ty + 1][tx + 1] = F[2] - Fo[2];
      }
      Fo[0] = F[0];
      Fo[1] = F[1];
      Fo[2] = F[2];
      if (hv) {
        vphi(hvy, hvx, F);
        if (!first) {
          SS[0][hvy][hvx] = Fh[0] + F[0];
          SS[1][hvy][hvx] = Fh[1] + F[1];
          SS[2][hvy][hvx] = F[2] - Fh[2];
        }
        Fh[0] = F[0];
        Fh[1] = F[1];
        Fh[2] = F[2];
      }
    };

    // ---- prologue
    // ring slots 0, 1, 2 hold U(z0-2), U(z0-1), U(z0); P/M of vertex plane z0-1/2
    fetchU(z0 - 2);
    storeU(z0 - 2, 0);
    fetchU(z0 - 1);
    storeU(z0 - 1, 1);
    fetchU(z0);
    storeU(z0, 2);
    storePM();  // from (U(z0-1), U(z0))
    fetchB(z0 - 1);
    storeB(true);
    fetchB(z0);
    storeB(false);  // base P/M of plane z0 - 1/2
    __syncthreads();
    LT Lm = lap_at(ty + 1, tx + 1, 0, 1, 2);  // lap'(z0 - 1), own column only
    phi_plane(true);                         // Phi(z0 - 1/2) into registers
    __syncthreads();
    fetchU(z0 + 1);
    storeU(z0 + 1, 0);  // history now (U(z0), U(z0+1))
    __syncthreads();
    int lz = 0;
    LT L0 = lap_plane(1, 2, 0, lz);  // lap'(z0)
    __syncthreads();  // lap'(z0) read slot 1, which the first loop step overwrites
    // loop convention: um = slot of U(z-1), u0 = U(z), u1 = U(z+1)
    int um = 1, u0 = 2, u1 = 0;
    fetchU(z0 + 2);
    fetchB(z0 + 1);
    T fr = a.f ? a.f[(size_t)(z0 & (nz - 1)) * plane + gown] : T(0);

    for (int z = z0; z < z0 + zc; ++z) {
      const int u2 = um;
      storePM();        // vertex plane z + 1/2 from (U(z), U(z+1))
      storeU(z + 2, u2);
      storeB(false);    // base P/M of plane z + 1/2
      __syncthreads();  // (A)
      const T fcur = fr;
      fetchU(z + 3);
      fetchB(z + 2);
      fr = a.f ? a.f[(size_t)((z + 1) & (nz - 1)) * plane + gown] : T(0);
      const LT Lp = lap_plane(u0, u1, u2, lz ^ 1);  // lap'(z+1)
      phi_plane(false);                             // S/D for the cells of plane z
      const LT ucl = sU[u0][ty + 2][tx + 2];
      __syncthreads();  // (B)
      const LT bihl = (((sL[lz][ty + 1][tx] + sL[lz][ty + 1][tx + 2]) + (sL[lz][ty][tx + 1] + sL[lz][ty + 2][tx + 1])) +
                       (Lm + Lp)) -
                      LT(6) * L0;
      const LT dx = (SS[0][ty][tx + 1] - SS[0][ty][tx]) + (SS[0][ty + 1][tx + 1] - SS[0][ty + 1][tx]);
      const LT dy = (SS[1][ty + 1][tx] - SS[1][ty][tx]) + (SS[1][ty + 1][tx + 1] - SS[1][ty][tx + 1]);
      const LT dz = (SS[2][ty][tx] + SS[2][ty][tx + 1]) + (SS[2][ty + 1][tx] + SS[2][ty + 1][tx + 1]);
      const LT divl = (dx + dy) + dz;
      T uc, bih, div;
      if constexpr (FX) {
        uc = fx_result(ucl, 0);
        bih = fx_result(bihl, 0);
        div = fx_result(divl, 0);
      } else {
        uc = ucl;
        bih = bihl;
        div = divl;
      }
      T r;
      if (INNER)
        r = fcur - ((cu * uc + cbih * bih) - cdiv * div);
      else if (HVP)
        r = (cu * uc + cbih * bih) - cdiv * div;
      else
        r = FX ? fma(cdivq, div, fma(-cbihq, bih, fma(-cuq, uc, fcur))) : (fcur - cuq * uc) + (cdivq * div - cbihq * bih);
      store_r<MODE>(a, (size_t)(z & (nz - 1)) * plane + gown, r);
      acc2 += HVP ? uc * r : r * r;
      accm = max_abs(accm, r);
      Lm = L0;
      L0 = Lp;
      lz ^= 1;
      um = u0;
      u0 = u1;
      u1 = u2;
    }
    __syncthreads();  // the next segment's prologue refills the shared tiles
  }

  if constexpr (TRACK) {
    track_publish(um, gm, FX ? fxs : kFxOff, fxg, FX && a.d == nullptr, ctrl, sm.smax);
  }
  T v[2] = {acc2, accm};
  block_reduce<T, 2, true>(v, sm.sred);
  if (publish_and_check_last<T>(v, 2, reinterpret_cast<T*>(partials), &ctrl->counter[CS_RES], &sm.sflag)) {
    T tt[2];
    gather_partials<T, 2, true>(tt, reinterpret_cast<const T*>(partials), sm.sred);
    if (tid == 0) {
      if constexpr (TRACK) {
        track_collect(ctrl);
      }
      residual_epilogue(ctrl, kp, (double)tt[0], (double)tt[1], a.norm, a.update_iter, HVP);
    }
  }
}

template <typename T, int PK, int MODE>
__global__ void __launch_bounds__(256, 3)  // 80 registers, 3 CTAs per SM
    k_res3d_col(ResArgs<T> a, KParams kp, Ctrl* ctrl, double* partials) {
  if (ctrl->done) return;
  __shared__ __align__(16) ResColSmem<T, MODE> sm;
  if constexpr (sizeof(T) == 8 && MODE == RM_PLAIN && PK == PK_4) {
    if (a.fixed && ctrl->fx_s != kFxOff) {
      res3d_col<T, PK, MODE, true>(a, kp, ctrl, partials, sm, ctrl->fx_s, ctrl->fx_g);
      return;
    }
  }
  res3d_col<T, PK, MODE, false>(a, kp, ctrl, partials, sm, 0, 0);
}

// Column-owning 3D line-search reduction (tiles of 32 x 8 vertices).  Each
// thread owns a vertex column; the z-pair sums / differences of u (+ base)
// and d are formed from a per-element register history as each plane
// arrives, double-buffered in shared memory (one barrier per plane).  The
// sums use the unscaled gradients A = a/q, B = b/q; the epilogue applies q^p.
//
// FX (FP64, p = 4): u and d enter as 64-bit integers (scales from the bounds
// on |u| and |d| in ctrl), so the gradients are exact sums; |a|^2, a.b and |b|^2
// are integer products (fx_ls_accumulate), four FP64 operations per vertex
// accumulate instead of about 40 in all.  TRACK: the bounds of the next iterate, from
// alpha and the largest |grad d|, choose the residual's scales.
template <typename T>
struct LsColSmem {
  T P[2][2][9][33], M[2][2][9][33];  // [u, d][buffer][y][x]
  unsigned smax[2];
  int sflag;
};
template <typename T, int PK, bool INNER, bool FX>
__device__ __forceinline__ void ls3d_col(const T* __restrict__ u, const T* __restrict__ ubase,
                                         const T* __restrict__ d, const KParams& kp, Ctrl* ctrl, double* partials,
                                         LsColSmem<T>& sm, T* sred, int Su, int Sd) {
  constexpr bool TRACK = sizeof(T) == 8 && PK == PK_4 && !INNER;
  static_assert(!FX || TRACK, "FX: FP64 p = 4 without a base only");
  using LT = typename std::conditional<FX, long long, T>::type;
  constexpr int TX = 32, TY = 8;
  constexpr int SX = TX + 1, SY = TY + 1, SN = SX * SY;  // cells x0..x0+TX, y0..y0+TY
  using Tile = LT(*)[SY][SX];
  Tile sPu = reinterpret_cast<Tile>(&sm.P[0][0][0][0]), sPd = reinterpret_cast<Tile>(&sm.P[1][0][0][0]);
  Tile sMu = reinterpret_cast<Tile>(&sm.M[0][0][0][0]), sMd = reinterpret_cast<Tile>(&sm.M[1][0][0][0]);
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
  const size_t plane = (size_t)nx * ny;
  const T beta = kconst<T>(kp).beta, pm2 = kconst<T>(kp).pm2;
  const T trial = ls_closed_form<PK>() ? T(0) : (T)ctrl->trial;
  // one wave of CTAs, each marching an equal share of the column-planes (as
  // the residual column kernel)
  const int gx = nx / TX;
  const int ncol = gx * (ny / TY);
  const int wtot = ncol * nz;
  const int wend = (int)((long long)wtot * (blockIdx.x + 1) / gridDim.x);
  const int mls = lockstep_classes(gridDim.x, ncol);
  int off[2], ely[2], elx[2];
  bool val[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int e = tid + 256 * k;
    val[k] = e < SN;
    ely[k] = e / SX;
    elx[k] = e - ely[k] * SX;
    off[k] = 0;
  }
  // prefetched plane: u, base and d kept apart until used a step later
  T pu[2] = {T(0), T(0)}, pbv[2] = {T(0), T(0)}, pdv[2] = {T(0), T(0)};
  LT hu[2] = {LT(0), LT(0)}, hdd[2] = {LT(0), LT(0)};
  auto fetch = [&](int zz) {
    const size_t gz = (size_t)(zz & (nz - 1)) * plane;
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (val[k]) {
        pu[k] = u[gz + off[k]];
        if (INNER) pbv[k] = ubase[gz + off[k]];
        pdv[k] = d[gz + off[k]];
      }
  };
  auto enter = [&](T x, int S) -> LT {
    if constexpr (FX)
      return fx_quantise((unsigned)__double2hiint(x), (unsigned)__double2loint(x), 1077 - S, 55).v;
    else
      return x;
  };
  auto store = [&](int buf, bool first) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (val[k] && INNER) pu[k] += pbv[k];
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (val[k]) {
        const LT un = enter(pu[k], Su), dn = enter(pdv[k], Sd);
        if (!first) {
          (&sPu[buf][0][0])[tid + 256 * k] = hu[k] + un;
          (&sMu[buf][0][0])[tid + 256 * k] = un - hu[k];
          (&sPd[buf][0][0])[tid + 256 * k] = hdd[k] + dn;
          (&sMd[buf][0][0])[tid + 256 * k] = dn - hdd[k];
        }
        hu[k] = un;
        hdd[k] = dn;
      }
  };
  auto grad = [&](LT (&P)[SY][SX], LT (&M)[SY][SX], LT (&g)[3]) {
    g[0] = (P[ty][tx + 1] - P[ty][tx]) + (P[ty + 1][tx + 1] - P[ty + 1][tx]);
    g[1] = (P[ty + 1][tx] - P[ty][tx]) + (P[ty + 1][tx + 1] - P[ty][tx + 1]);
    g[2] = (M[ty][tx] + M[ty][tx + 1]) + (M[ty + 1][tx] + M[ty + 1][tx + 1]);
  };
  T acc[ls_nsums<PK>()] = {};
  T sbb = T(0);      // TRACK: sum (a.b)^2, kept apart from sum |a|^2 |b|^2
  unsigned gm = 0u;  // TRACK: largest |b|^2, high word
  for (int w = (int)((long long)wtot * blockIdx.x / gridDim.x); w < wend;) {
    const int col = w / nz, z0 = w - col * nz;
    const int zc = min(nz - z0, wend - w);
    w += zc;
    const int tile = lockstep_tile(col, mls, ncol);
    const int x0 = (tile % gx) * TX, y0 = (tile / gx) * TY;
#pragma unroll
    for (int k = 0; k < 2; ++k) off[k] = ((y0 + ely[k]) & (ny - 1)) * nx + ((x0 + elx[k]) & (nx - 1));
    fetch(z0);
    store(0, true);
    fetch(z0 + 1);
    for (int z = z0; z < z0 + zc; ++z) {
      const int buf = (z - z0) & 1;
      store(buf, false);  // vertex plane z + 1/2
      __syncthreads();
      fetch(z + 2);
      LT av[3], bv[3];
      grad(sPu[buf], sMu[buf], av);
      grad(sPd[buf], sMd[buf], bv);
      if constexpr (FX)
        gm = max(gm, fx_ls_accumulate(av[0], av[1], av[2], bv[0], bv[1], bv[2], acc, sbb));
      else if constexpr (TRACK)
        gm = max(gm, ls_accumulate4(av, bv, acc, sbb));
      else
        ls_accumulate<PK>(av, bv, trial, beta, pm2, acc);
    }
    __syncthreads();  // the next segment writes the shared buffers again
  }
  if constexpr (TRACK) {
    ls_track(acc, sbb, gm, FX, Su, Sd, ctrl, sm.smax);
  }
  ls_finish<T, PK>(acc, sred, partials, ctrl, kp, &sm.sflag, TRACK);
}

template <typename T, int PK, bool INNER>
__global__ void __launch_bounds__(256, 3)
    k_ls3d_col(const T* __restrict__ u, const T* __restrict__ ubase, const T* __restrict__ d, KParams kp,
               Ctrl* ctrl, double* partials) {
  if (ctrl->done) return;
  if (!ls_closed_form<PK>() && ctrl->c3 != 0.0) return;  // Newton already converged
  __shared__ __align__(16) LsColSmem<T> sm;
  __shared__ T sred[red_size<T>(ls_nsums<PK>())];
  if constexpr (sizeof(T) == 8 && PK == PK_4 && !INNER) {
    int Su, Sd;
    if (ls_scales(ctrl, &Su, &Sd)) {
      ls3d_col<T, PK, INNER, true>(u, ubase, d, kp, ctrl, partials, sm, sred, Su, Sd);
      return;
    }
  }
  ls3d_col<T, PK, INNER, false>(u, ubase, d, kp, ctrl, partials, sm, sred, 0, 0);
}

}  // namespace
}  // namespace psd
