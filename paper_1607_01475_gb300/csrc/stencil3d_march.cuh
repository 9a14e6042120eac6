// 3D FP32 residual and line search as warp marches: a warp owns a strip of 32
// cells along x and RY rows along y and marches along z, with everything in
// registers and the x-neighbours by shuffle -- no shared tiles and no barriers.
// The arithmetic is that of the column kernels (unscaled vertex-gradient sums
// G = g / q, Laplacian sums h^2 Delta_h), arranged for few instructions:
//
// Per plane and row, D = u[x+1] - u[x], A = u[x+1] + u[x] (one shuffle).  At the
// vertex plane between two planes, a = D + D', b = A + A', c = A' - A per row, and
// at the vertex between rows v and v + 1: G = (a_v + a_{v+1}, b_{v+1} - b_v, c_v +
// c_{v+1}).  lap' = (D - D[x-1]) + ((y-neighbours) + (z-neighbours)) - 4 u (one
// shuffle).  With the flux sums S over the two vertex planes of a cell plane, T1
// = Sx_{j-1} + Sx_j and T2 = (Sy_j - Sy_{j-1}) + (Sz_{j-1} + Sz_j):
//   div' = (T1 + T2) + (T2 - T1)[x-1],
// so that the x - 1/2 vertices and lap'[x-1] reach a cell by one shuffle of
// cdiv (T2 - T1) - cbih lap', and lap'[x+1] by another: 26 shuffles per step of
// 4 rows, where the shared-memory kernel this replaces read 17 words and wrote
// 10 per cell.  The window's outer two cells on each side are not outputs (28 of
// 32); a strip reads 2 rows above and below.
//
// The kernels are bound by instruction issue (about 190 instructions per cell in
// the residual, with 20% of the lanes outside the grid at nx = 256).  Grids with at
// least 2 x 152 tiles of 32 x 32 x 16 cells take the shared-memory kernels of
// stencil3d_rb.cuh, whose tiles waste no lanes (256^3 residual: 132 us there, 156
// here; line search 65.5 and 67); on smaller grids these replace the 32 x 8 column tiles and the general
// tiles (128^3, traced launches: residual 46 -> 27.5 us, line search 27 -> 19 us).  One
// wave of CTAs takes equal shares of the (column, plane) pairs, a column being a
// strip of the CTA's warps, four rows each, one below the other, which share
// their halo rows in L1.
#pragma once

namespace psd {
namespace {

constexpr int kMarchRows = 4;  // rows per warp

// The share of column-planes of this CTA, one z-segment at a time.
struct March3D {
  int w, wend, m, ncol, nstrip, nz;
  int x0, y0, z0, zc;
  __device__ __forceinline__ March3D(const KParams& kp, int outputs) {
    nstrip = (kp.nx + outputs - 1) / outputs;
    nz = kp.nz;
    ncol = nstrip * (kp.ny / ((int)(blockDim.x >> 5) * kMarchRows));
    const long long wtot = (long long)ncol * nz;
    w = (int)(wtot * blockIdx.x / gridDim.x);
    wend = (int)(wtot * (blockIdx.x + 1) / gridDim.x);
    m = lockstep_classes(gridDim.x, ncol);
  }
  __device__ __forceinline__ bool next(int outputs) {
    if (w >= wend) return false;
    const int col = w / nz;
    z0 = w - col * nz;
    zc = min(nz - z0, wend - w);
    w += zc;
    const int tile = lockstep_tile(col, m, ncol);
    x0 = (tile % nstrip) * outputs;
    y0 = ((tile / nstrip) * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5)) * kMarchRows;
    return true;
  }
};

template <typename T>
__device__ __forceinline__ T lane_right(T v) {
  return __shfl_down_sync(0xffffffffu, v, 1);
}
template <typename T>
__device__ __forceinline__ T lane_left(T v) {
  return __shfl_up_sync(0xffffffffu, v, 1);
}

// Element at byte offset off of a plane: a uniform base and a 32-bit offset per
// lane, one instruction (planes have at most 2^20 cells).
template <typename T>
__device__ __forceinline__ T at(const T* plane, unsigned off) {
  return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(plane) + off);
}
template <typename T>
__device__ __forceinline__ void put(T* plane, unsigned off, T v) {
  *reinterpret_cast<T*>(reinterpret_cast<char*>(plane) + off) = v;
}

// What a march keeps of one plane: u (rows 0 .. RY + 3 of the strip), D and A and
// lap' (rows 1 .. RY + 2), and for the base field D and A.
template <typename T, bool BASE>
struct MarchPlane {
  static constexpr int RY = kMarchRows;
  T U[RY + 4], D[RY + 2], A[RY + 2], L[RY + 2];
  T Db[BASE ? RY + 2 : 1], Ab[BASE ? RY + 2 : 1];
  T F[RY + 1][3];  // flux of the vertex plane below
};

template <typename T, int PK, int MODE>
__global__ void __launch_bounds__(32 * kMarchWarps, kMarchResCtas)
    k_res3d_march(ResArgs<T> p, KParams kp, Ctrl* ctrl, double* partials) {
  if (ctrl->done) return;
  constexpr int RY = kMarchRows, NU = RY + 4, NR = RY + 2, NV = RY + 1;  // rows of u, of lap' / base, of vertices
  constexpr bool INNER = MODE == RM_INNER, HVP = MODE == RM_HVP, BASE = MODE != RM_PLAIN;
  using Plane = MarchPlane<T, BASE>;
  __shared__ T sred[red_size<T>(2)];
  __shared__ int sflag;
  const int lane = threadIdx.x & 31;
  const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
  const size_t plane = (size_t)nx * ny;
  const bool upd = p.d != nullptr, has_f = p.f != nullptr, sums = HVP || p.norm != 0;
  // without an update u + 0 u: no branch in the march
  const T alpha = upd ? (T)ctrl->alpha : T(0);
  const T* dir = upd ? p.d : p.u_in;
  const T cdiv = kconst<T>(kp).cdiv, cbih = kconst<T>(kp).cbih, cu = kconst<T>(kp).cu, beta = kconst<T>(kp).beta;
  T acc2 = T(0), accm = T(0);
  March3D ms(kp, 28);
  while (ms.next(28)) {
    const int z0 = ms.z0, zend = ms.z0 + ms.zc;
    const int gx = (ms.x0 + lane - 2) & (nx - 1);
    const bool out = lane >= 2 && lane < 30 && ms.x0 + lane - 2 < nx;
    unsigned off[NU];  // byte offset of row y0 - 2 + j within a plane
#pragma unroll
    for (int j = 0; j < NU; ++j) off[j] = (unsigned)(((ms.y0 + j - 2) & (ny - 1)) * nx + gx) * (unsigned)sizeof(T);
    T pu[NU], pd[NU], pb[NR];  // u and d of the next plane, base of the plane before it
    auto fetch = [&](int k) {
      const size_t g = (size_t)(k & (nz - 1)) * plane;
#pragma unroll
      for (int j = 0; j < NU; ++j) {
        pu[j] = at(p.u_in + g, off[j]);
        pd[j] = at(dir + g, off[j]);
      }
      if (BASE) {
        const T* b = p.ubase + (size_t)((k - 1) & (nz - 1)) * plane;
#pragma unroll
        for (int j = 0; j < NR; ++j) pb[j] = at(b, off[j + 1]);
      }
    };
    Plane P0, P1, P2;  // planes in rotation; of plane k - 1 lap' and the base are formed at step k
    auto clear = [&](Plane& q) {
#pragma unroll
      for (int j = 0; j < NU; ++j) q.U[j] = T(0);
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        q.D[j] = q.A[j] = q.L[j] = T(0);
        if (BASE) q.Db[j] = q.Ab[j] = T(0);
      }
#pragma unroll
      for (int j = 0; j < NV; ++j) q.F[j][0] = q.F[j][1] = q.F[j][2] = T(0);
    };
    clear(P0);
    clear(P1);
    clear(P2);
#pragma unroll
    for (int j = 0; j < NU; ++j) pu[j] = pd[j] = T(0);
    // Step k: a, b, c hold planes k - 2, k - 1, k (u, D, A); lap' is known for
    // planes k - 3 (in c, before it is overwritten) and k - 2, the base for k - 2;
    // the flux of the vertex plane k - 5/2 is in a, that of k - 3/2 goes to b.
    auto step = [&](int k, Plane& a, Plane& b, Plane& c) {
      T base[NR];
#pragma unroll
      for (int j = 0; j < NU; ++j) c.U[j] = pu[j] + alpha * pd[j];
      if (BASE) {
#pragma unroll
        for (int j = 0; j < NR; ++j) base[j] = pb[j];
      }
      if (upd && out && k >= z0 && k < zend) {
        T* uo = p.u_out + (size_t)k * plane;
#pragma unroll
        for (int j = 0; j < RY; ++j) put(uo, off[j + 2], c.U[j + 2]);
      }
      if (k + 1 < zend + 2) fetch(k + 1);
      const bool emit = k >= z0 + 2;
      T f[RY];
#pragma unroll
      for (int j = 0; j < RY; ++j) f[j] = T(0);
      if (has_f && emit) {
        const T* fp = p.f + (size_t)(k - 2) * plane;
#pragma unroll
        for (int j = 0; j < RY; ++j) f[j] = at(fp, off[j + 2]);
      }
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        const T r = lane_right(c.U[j + 1]);
        c.D[j] = r - c.U[j + 1];
        c.A[j] = r + c.U[j + 1];
        b.L[j] = ((b.D[j] - lane_left(b.D[j])) + ((b.U[j] + b.U[j + 2]) + (a.U[j + 1] + c.U[j + 1]))) -
                 T(4) * b.U[j + 1];
        if (BASE) {
          const T rb = lane_right(base[j]);
          b.Db[j] = rb - base[j];
          b.Ab[j] = rb + base[j];
        }
      }
      if (k <= z0) return;
      T S[NV][3];
      T a0 = a.D[0] + b.D[0], b0 = a.A[0] + b.A[0], c0 = b.A[0] - a.A[0];
      T e0 = T(0), g0 = T(0), h0 = T(0);
      if (BASE) {
        e0 = a.Db[0] + b.Db[0];
        g0 = a.Ab[0] + b.Ab[0];
        h0 = b.Ab[0] - a.Ab[0];
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const T a1 = a.D[v + 1] + b.D[v + 1], b1 = a.A[v + 1] + b.A[v + 1], c1 = b.A[v + 1] - a.A[v + 1];
        const T G[3] = {a0 + a1, b1 - b0, c0 + c1};
        if constexpr (BASE) {
          const T e1 = a.Db[v + 1] + b.Db[v + 1], g1 = a.Ab[v + 1] + b.Ab[v + 1], h1 = b.Ab[v + 1] - a.Ab[v + 1];
          const T Gb[3] = {e0 + e1, g1 - g0, h0 + h1};
          if (INNER)
            flux_diff<PK>(Gb, G, beta, b.F[v]);
          else
            flux_lin<PK>(Gb, G, beta, b.F[v]);
          e0 = e1;
          g0 = g1;
          h0 = h1;
        } else {
          flux<PK>(G, beta, b.F[v]);
        }
        a0 = a1;
        b0 = b1;
        c0 = c1;
        S[v][0] = a.F[v][0] + b.F[v][0];
        S[v][1] = a.F[v][1] + b.F[v][1];
        S[v][2] = b.F[v][2] - a.F[v][2];
      }
      if (!emit) return;
      T* rp = p.r + (size_t)(k - 2) * plane;
#pragma unroll
      for (int j = 0; j < RY; ++j) {
        const T T1 = S[j][0] + S[j + 1][0];
        const T T2 = (S[j + 1][1] - S[j][1]) + (S[j][2] + S[j + 1][2]);
        const T lap = a.L[j + 1];
        const T ql = lane_left(cdiv * (T2 - T1) - cbih * lap), lr = lane_right(lap);
        // -cbih bih' + cdiv div' without the terms of ql
        const T bih = ((a.L[j] + a.L[j + 2]) + (c.L[j + 1] + b.L[j + 1]) + lr) - T(6) * lap;
        const T nl = (cdiv * (T1 + T2) - cbih * bih) + ql;
        const T uc = a.U[j + 2];
        T r;
        if (INNER)
          r = f[j] - (cu * uc - nl);
        else if (HVP)
          r = cu * uc - nl;
        else
          r = (f[j] - cu * uc) + nl;
        if (out) put(rp, off[j + 2], r);
        if (sums && out) {
          acc2 += HVP ? uc * r : r * r;
          accm = fmax(accm, fabs(r));
        }
      }
    };
    fetch(z0 - 2);
    for (int k = z0 - 2;;) {
      step(k, P0, P1, P2);
      if (++k >= zend + 2) break;
      step(k, P1, P2, P0);
      if (++k >= zend + 2) break;
      step(k, P2, P0, P1);
      if (++k >= zend + 2) break;
    }
  }
  T v[2] = {acc2, accm};
  block_reduce<T, 2, true>(v, sred);
  if (publish_and_check_last<T>(v, 2, reinterpret_cast<T*>(partials), &ctrl->counter[CS_RES], &sflag)) {
    T tt[2];
    gather_partials<T, 2, true>(tt, reinterpret_cast<const T*>(partials), sred);
    if (threadIdx.x == 0) residual_epilogue(ctrl, kp, (double)tt[0], (double)tt[1], p.norm, p.update_iter, HVP);
  }
}

// Line search: the vertices (x + 1/2, y + 1/2, z + 1/2) of the strip's first 31
// cells and RY rows; one row more of u (+ base) and d.
template <typename T, int PK, bool INNER>
__global__ void __launch_bounds__(32 * kMarchWarps, kMarchLsCtas)
    k_ls3d_march(const T* __restrict__ u, const T* __restrict__ ubase, const T* __restrict__ d, KParams kp, Ctrl* ctrl,
                 double* partials) {
  if (ctrl->done) return;
  if (!ls_closed_form<PK>() && ctrl->c3 != 0.0) return;  // Newton already converged
  constexpr int RY = kMarchRows, NR = RY + 1;
  __shared__ T sred[red_size<T>(ls_nsums<PK>())];
  __shared__ int sflag;
  const int lane = threadIdx.x & 31;
  const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
  const size_t plane = (size_t)nx * ny;
  const T beta = kconst<T>(kp).beta, pm2 = kconst<T>(kp).pm2;
  const T trial = ls_closed_form<PK>() ? T(0) : (T)ctrl->trial;
  T acc[ls_nsums<PK>()] = {};
  March3D ms(kp, 31);
  while (ms.next(31)) {
    const int z0 = ms.z0, zc = ms.zc;
    const int gx = (ms.x0 + lane) & (nx - 1);
    const bool out = lane < 31 && ms.x0 + lane < nx;
    unsigned off[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) off[j] = (unsigned)(((ms.y0 + j) & (ny - 1)) * nx + gx) * (unsigned)sizeof(T);
    T pu[NR], pb[NR], pd[NR];
    auto fetch = [&](int k) {
      const size_t g = (size_t)(k & (nz - 1)) * plane;
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        pu[j] = at(u + g, off[j]);
        pb[j] = INNER ? at(ubase + g, off[j]) : T(0);
        pd[j] = at(d + g, off[j]);
      }
    };
    struct Plane {
      T Du[NR], Au[NR], Dd[NR], Ad[NR];
    } P0, P1;
#pragma unroll
    for (int j = 0; j < NR; ++j) P1.Du[j] = P1.Au[j] = P1.Dd[j] = P1.Ad[j] = T(0);
    // step k: a holds plane k - 1, b receives plane k
    auto step = [&](int k, const Plane& a, Plane& b) {
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        const T w = INNER ? pu[j] + pb[j] : pu[j], q = pd[j];
        const T wr = lane_right(w), qr = lane_right(q);
        b.Du[j] = wr - w;
        b.Au[j] = wr + w;
        b.Dd[j] = qr - q;
        b.Ad[j] = qr + q;
      }
      if (k < z0 + zc) fetch(k + 1);
      if (k > z0 && out) {
        T a0 = a.Du[0] + b.Du[0], b0 = a.Au[0] + b.Au[0], c0 = b.Au[0] - a.Au[0];
        T e0 = a.Dd[0] + b.Dd[0], g0 = a.Ad[0] + b.Ad[0], h0 = b.Ad[0] - a.Ad[0];
#pragma unroll
        for (int v = 0; v < RY; ++v) {
          const T a1 = a.Du[v + 1] + b.Du[v + 1], b1 = a.Au[v + 1] + b.Au[v + 1], c1 = b.Au[v + 1] - a.Au[v + 1];
          const T e1 = a.Dd[v + 1] + b.Dd[v + 1], g1 = a.Ad[v + 1] + b.Ad[v + 1], h1 = b.Ad[v + 1] - a.Ad[v + 1];
          const T av[3] = {a0 + a1, b1 - b0, c0 + c1}, bv[3] = {e0 + e1, g1 - g0, h0 + h1};
          ls_accumulate<PK>(av, bv, trial, beta, pm2, acc);
          a0 = a1;
          b0 = b1;
          c0 = c1;
          e0 = e1;
          g0 = g1;
          h0 = h1;
        }
      }
    };
    fetch(z0);
    for (int k = z0;;) {
      step(k, P1, P0);
      if (++k > z0 + zc) break;
      step(k, P0, P1);
      if (++k > z0 + zc) break;
    }
  }
  ls_finish<T, PK>(acc, sred, partials, ctrl, kp, &sflag);
}

}  // namespace
}  // namespace psd
