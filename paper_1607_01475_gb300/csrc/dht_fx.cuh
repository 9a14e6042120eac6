// Hartley transform passes of FP64 fields in 64-bit block fixed point (the
// line FFT of fx_line.cuh): the x pass, the strided pass, the middle pass of
// the preconditioner and the last pass of the mixed solver's outer loop.
// Data in memory is FP64 before and after every pass.
//
// At 256^3 a pass moves 268 MB (40 us at the measured copy rate) and takes 88
// us (rows, columns), bound by integer issue; with FP64 butterflies it took 547
// us.  The sixth-order middle pass takes 535 us instead of 1711, bound by the
// 13 FP64 operations per element of the symbol division, the Parseval sums and the
// output conversions (about 410 us at 1.74 per clock and SM) and by integer issue.
#pragma once

#include <algorithm>
#include <cmath>

#include "dht_kernels.cuh"
#include "fx_line.cuh"

namespace psd {
namespace {

constexpr int kFxThreads = 256;

// Elements between the real arrays of consecutive line pairs in shared
// memory, in 8-byte points (each pair holds its real and imaginary line of
// F::L): the smallest LS >= F::L with LS = r (mod M), so that a warp's accesses
// in every pass spread over the banks.  Row passes (a warp spans 32/TS
// pairs): r = m/2, M = m for m = TS/2 (odd LS when m < 2, free when m >= 32);
// strided passes (a warp spans `pairs` pairs): r = 16/k, M = 32/k for k =
// min(2 pairs, 16).
template <int N, int RM, bool ROWS>
__host__ __device__ constexpr int fx_line_stride() {
  constexpr int L = LineFFT<fx, N, RM>::L, TS = LineFFT<fx, N, RM>::TS;
  int r = 0, M = 1;
  if (ROWS) {
    const int m = TS / 2;
    if (m >= 32) return L;
    r = m < 2 ? 1 : m / 2;
    M = m < 2 ? 2 : m;
  } else {
    const int k = (kFxThreads / TS) * 2 < 16 ? (kFxThreads / TS) * 2 : 16;
    r = 16 / k;
    M = 32 / k;
  }
  return L + (((r - L) % M) + M) % M;
}
template <int N, int RM, bool ROWS>
constexpr size_t fx_pair_smem() {
  return 2 * (size_t)fx_line_stride<N, RM, ROWS>() * sizeof(fx);
}

// The common exponent and scale of a line pair from its team's values.  ROWS:
// the team is TS consecutive threads; otherwise the team of pair p is the
// threads tid = p (mod pairs).  share() reduces the largest exponent and the squared
// 2-norm relative to it within the warp; a team of several warps leaves them in
// scr, and after a barrier line() combines the warps in a fixed order.
struct FxLine {
  int E, B;  // largest biased exponent (at least 1), scale
};
template <int N, int RM, bool ROWS>
struct FxTeam {
  static constexpr int R = FxPlan<N, RM>::R, TS = N / R;
  static constexpr bool kOneWarp = ROWS && TS <= 32;
  int p, pairs;
  int E;       // of this warp
  unsigned l;  // bound on the squared 2-norm of this warp's points, in units of 2^(2 (E - 1032))

  __device__ __forceinline__ void share(const double (&xr)[R], const double (&xi)[R], uint2 (*scr)[32]) {
    const int nthr = (int)blockDim.x;
    const unsigned mask = nthr >= 32 ? 0xffffffffu : (1u << nthr) - 1u;
    const int o0 = ROWS ? 1 : pairs, o1 = ROWS ? (TS < 32 ? TS : 32) : (nthr < 32 ? nthr : 32);
    unsigned e = 0u;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      e = max(e, (unsigned)__double2hiint(xr[q]) & 0x7FFFFFFFu);
      e = max(e, (unsigned)__double2hiint(xi[q]) & 0x7FFFFFFFu);
    }
    for (int o = o0; o < o1; o <<= 1) e = max(e, __shfl_xor_sync(mask, e, o));
    E = (int)(e >> 20);
    l = 0u;
#pragma unroll
    for (int q = 0; q < R; ++q)
      l += fx_square((unsigned)__double2hiint(xr[q]), E) + fx_square((unsigned)__double2hiint(xi[q]), E);
    for (int o = o0; o < o1; o <<= 1) l += __shfl_xor_sync(mask, l, o);
    const int lane = threadIdx.x & 31;
    if (!kOneWarp && (ROWS ? lane == 0 : lane < pairs)) scr[threadIdx.x >> 5][lane] = make_uint2((unsigned)E, l);
  }
  __device__ __forceinline__ FxLine line(const uint2 (*scr)[32]) const {
    if (kOneWarp) return {max(E, 1), fx_scale<FxPlan<N, RM>>(l)};
    // the team's warps: w0, w0 + step, ..
    const int nw = ROWS ? p * (TS / 32) + TS / 32 : ((int)blockDim.x + 31) >> 5;
    const int step = !ROWS && pairs > 32 ? pairs >> 5 : 1;
    const int w0 = ROWS ? p * (TS / 32) : p >> 5, lane = ROWS ? 0 : p & 31;
    int Em = 0;
    for (int w = w0; w < nw; w += step) Em = max(Em, (int)scr[w][lane].x);
    unsigned lm = 0u;
    for (int w = w0; w < nw; w += step) {
      const uint2 v = scr[w][lane];
      lm += (v.y >> min(2 * (Em - (int)v.x), 31)) + 1u;
    }
    return {max(Em, 1), fx_scale<FxPlan<N, RM>>(lm)};
  }
};

// Twiddle source of the fixed-point passes (see TwPair): Q62 products divide
// by 4, so the points a pass does not rotate are divided too.
struct TwFx {
  const fx_tw* __restrict__ tab;
  __device__ __forceinline__ void rotate(int t, fx& a, fx& b, bool odd) const {
    const int4 w = __ldg(reinterpret_cast<const int4*>(tab + t));
    fx_rotate(a, b, fx_tw{w.x, w.y, w.z, w.w}, odd);
  }
  __device__ __forceinline__ void untwiddled(fx& a, fx& b) const {
    a = fx_quarter(a);
    b = fx_quarter(b);
  }
};

// The bits of an FP64 value, or of an FP32 value as FP64.
__device__ __forceinline__ double fx_load(double x) { return x; }
__device__ __forceinline__ double fx_load(float x) {
  const unsigned b = __float_as_uint(x), E = (b >> 23) & 0xFFu, m = b & 0x7FFFFFu;
  if (E == 0u && m != 0u) return (double)x;  // subnormal
  const unsigned e = E == 0u ? 0u : (E == 0xFFu ? 0x7FFu : E + 896u);
  const unsigned f = E == 0u ? 0u : m;
  return __hiloint2double((int)((b & 0x80000000u) | (e << 20) | (f >> 3)), (int)(f << 29));
}

// A line pair's points as integers of the line's scale (0 where it is not
// finite).  Lines below the smallest exponent, whose zeros and subnormals have no place in
// fx_quantise, enter 2^512 times as large (a branch that no ordinary line takes: at most
// 0.5% of a solve of L_h in order 4, 1.7% in order 6 at 256^3).
template <int N, int RM>
__device__ __forceinline__ void fx_enter(double (&xr)[FxPlan<N, RM>::R], double (&xi)[FxPlan<N, RM>::R],
                                         const FxLine& ln, fx (&vr)[FxPlan<N, RM>::R], fx (&vi)[FxPlan<N, RM>::R]) {
  int E = ln.E;
  if (E < kFxMinExp) {
    E += 512;
#pragma unroll
    for (int q = 0; q < FxPlan<N, RM>::R; ++q) {
      xr[q] *= 0x1p512;
      xi[q] *= 0x1p512;
    }
  }
#pragma unroll
  for (int q = 0; q < FxPlan<N, RM>::R; ++q) {
    vr[q] = fx_quantise((unsigned)__double2hiint(xr[q]), (unsigned)__double2loint(xr[q]), E, ln.B);
    vi[q] = fx_quantise((unsigned)__double2hiint(xi[q]), (unsigned)__double2loint(xi[q]), E, ln.B);
    if (E > kFxMaxExp) vr[q].v = vi[q].v = 0;
  }
}
// A Hartley output from the split sum w; subnormal ones give 0 (rounding them here took 3%
// of a solve of L_h).
template <int N, int RM>
__device__ __forceinline__ double fx_leave(fx w, const FxLine& ln, int scale_e) {
  return ln.E > kFxMaxExp ? __longlong_as_double(0x7FF8000000000000LL)
                          : fx_result(w.v, ln.E - ln.B + FxPlan<N, RM>::kOut + scale_e);
}
// The same by the hardware conversion and an addition to the exponent, for the
// passes whose FP64 pipe is otherwise idle (one FP64-rate operation instead of
// about 20 integer ones; 256^3 row pass 107 -> 94 us when it was taken).  Lines whose outputs
// could leave the normal range take fx_leave.
template <int N, int RM>
__device__ __forceinline__ double fx_leave_hw(fx w, const FxLine& ln, int scale_e) {
  const int e = ln.E - ln.B + FxPlan<N, RM>::kOut + scale_e;
  if (ln.E > kFxMaxExp || (unsigned)(e + 1000) >= 1900u) return fx_leave<N, RM>(w, ln, scale_e);
  const double v = __ll2double_rn(w.v);
  const int hi = __double2hiint(v);
  return __hiloint2double(hi == 0 ? 0 : hi + (e << 20), __double2loint(v));
}

// -------------------------------------------------------------- x (rows)
template <int N, int RM, typename SI>
__global__ void __launch_bounds__(kFxThreads, 3)
    k_rows_fx(const SI* src, const SI* src_odd, const int* iter, double* dst, int nrows, int scale_e, const int* done,
              const fx_tw* __restrict__ tab, unsigned int* dmax_hi) {
  using F = LineFFT<fx, N, RM>;
  constexpr int R = F::R, TS = F::TS;
  if (done != nullptr && *done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint2 scr[kFxThreads / 32][32];
  const int tid = threadIdx.x;
  const int pairs = blockDim.x / TS;
  const int p = tid / TS, j = tid - p * TS;
  const int row0 = 2 * (blockIdx.x * pairs + p);
  const bool valid = row0 < nrows;
  constexpr int LS = fx_line_stride<N, RM, true>();
  fx* sr = reinterpret_cast<fx*>(smem_raw) + (size_t)p * 2 * LS;
  fx* si = sr + LS;
  FxTeam<N, RM, true> team{p, pairs};
  double xr[R], xi[R];
  const SI* s0 = (iter != nullptr && (*iter & 1) ? src_odd : src) + (size_t)row0 * N;
#pragma unroll
  for (int q = 0; q < R; ++q) {
    xr[q] = valid ? fx_load(s0[j + q * TS]) : 0.0;
    xi[q] = valid ? fx_load(s0[N + j + q * TS]) : 0.0;
  }
  team.share(xr, xi, scr);
  if (!team.kOneWarp) __syncthreads();
  const FxLine ln = team.line(scr);
  fx vr[R], vi[R];
  fx_enter<N, RM>(xr, xi, ln, vr, vi);
  double* d0 = dst + (size_t)row0 * N;
  unsigned top = 0u;  // largest magnitude written, high word
  auto put = [&](int k, fx h1, fx h2) {
    const double a = fx_leave_hw<N, RM>(h1, ln, scale_e), b = fx_leave_hw<N, RM>(h2, ln, scale_e);
    d0[k] = a;
    d0[N + k] = b;
    top = max(top, max((unsigned)__double2hiint(a) & 0x7FFFFFFFu, (unsigned)__double2hiint(b) & 0x7FFFFFFFu));
  };
  if constexpr (FxTeam<N, RM, true>::kOneWarp) {
    // the last pass ends in registers, the split by shuffle
    F::run_tw_regs(vr, vi, j, sr, si, TwFx{tab});
    fx h1[R], h2[R];
    dht_split_regs<fx, N, R, TS>(vr, vi, j, h1, h2);
    if (valid) {
#pragma unroll
      for (int q = 0; q < R; ++q) put(j + q * TS, h1[q], h2[q]);
    }
  } else {
    F::run_tw(vr, vi, j, sr, si, TwFx{tab});
    if (valid) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        fx h1, h2;
        dht_split(sr, si, j + q * TS, N, h1, h2);
        put(j + q * TS, h1, h2);
      }
    }
  }
  if (dmax_hi != nullptr) {
    const unsigned nthr = blockDim.x;
    for (int o = 16; o > 0; o >>= 1)
      if (o < (int)nthr) top = max(top, __shfl_xor_sync(nthr >= 32 ? 0xffffffffu : (1u << nthr) - 1u, top, o));
    if ((tid & 31) == 0) scr[tid >> 5][0].x = top;
    __syncthreads();
    if (tid == 0) {
      for (unsigned w = 1; w < (nthr + 31) / 32; ++w) top = max(top, scr[w][0].x);
      atomicMax(dmax_hi, top + 1u);
    }
  }
}

// ------------------------------------------------------ strided lines (y, z)
// The transform of a strided kernel's line pairs from the points (xr, xi) to
// the spectrum in sr / si.  Block: `pairs` pairs of adjacent x-columns packed
// as re/im, thread (p, j) = (tid % pairs, tid / pairs), so that a warp reads
// whole row segments.  The line buffers are written after the first barrier.
template <int N, int RM>
__device__ __forceinline__ FxLine fx_cols_transform(double (&xr)[FxPlan<N, RM>::R], double (&xi)[FxPlan<N, RM>::R],
                                                    int p, int j, int pairs, fx* sr, fx* si, uint2 (*scr)[32],
                                                    const fx_tw* __restrict__ tab) {
  FxTeam<N, RM, false> team{p, pairs};
  team.share(xr, xi, scr);
  __syncthreads();
  const FxLine ln = team.line(scr);
  fx vr[FxPlan<N, RM>::R], vi[FxPlan<N, RM>::R];
  fx_enter<N, RM>(xr, xi, ln, vr, vi);
  LineFFT<fx, N, RM>::run_tw(vr, vi, j, sr, si, TwFx{tab});
  return ln;
}

template <int N, int RM>
__global__ void __launch_bounds__(kFxThreads, 3)
    k_cols_fx(double* data, size_t line_stride, size_t outer_stride, int scale_e, const int* done,
              const fx_tw* __restrict__ tab) {
  using F = LineFFT<fx, N, RM>;
  constexpr int R = F::R, TS = F::TS;
  if (done != nullptr && *done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint2 scr[kFxThreads / 32][32];
  const int tid = threadIdx.x;
  const int pairs = blockDim.x / TS;
  const int p = tid % pairs, j = tid / pairs;
  const size_t base = (size_t)blockIdx.y * outer_stride + (size_t)blockIdx.x * 2 * pairs + 2 * p;
  constexpr int LS = fx_line_stride<N, RM, false>();
  fx* sr = reinterpret_cast<fx*>(smem_raw) + (size_t)p * 2 * LS;
  fx* si = sr + LS;
  double xr[R], xi[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const double2 v = *reinterpret_cast<const double2*>(data + base + (size_t)(j + q * TS) * line_stride);
    xr[q] = v.x;
    xi[q] = v.y;
  }
  const FxLine ln = fx_cols_transform<N, RM>(xr, xi, p, j, pairs, sr, si, scr, tab);
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int kk = j + q * TS;
    fx h1, h2;
    dht_split(sr, si, kk, N, h1, h2);
    *reinterpret_cast<double2*>(data + base + (size_t)kk * line_stride) =
        make_double2(fx_leave_hw<N, RM>(h1, ln, scale_e), fx_leave_hw<N, RM>(h2, ln, scale_e));
  }
}

// ------------------------------------ last axis with a fused epilogue
// The last 1D DHT (z in 3D, y in 2D) of FP64 lines; the transformed values h
// are not stored but consumed:
//   EPI_THETA:  theta += h / mu            (theta = DHT(T_h v) accumulates)
//   EPI_RESID:  out32 = h - theta (FP32), and sum of (h - theta)^2 into
//               ctrl->res_l2 = (h^d / N sum)^{1/2} (Parseval)
// with mu the symbol of -Delta_h at the element; the zero mode gives 0
// (mean-zero projection).  Same thread mapping as k_cols_fx.
enum { EPI_THETA = 0, EPI_RESID = 1 };
template <int N, int RM, int EPI>
__global__ void __launch_bounds__(kFxThreads, 3)
    k_last_fx(const double* data, double* theta, float* out32, size_t line_stride, size_t outer_stride, KParams kp,
              Ctrl* ctrl, double* partials, const fx_tw* __restrict__ tab, const double* __restrict__ symx,
              const double* __restrict__ symo, const double* __restrict__ syml, double* dc, const int* skip) {
  using F = LineFFT<fx, N, RM>;
  constexpr int R = F::R, TS = F::TS;
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint2 scr[kFxThreads / 32][32];
  __shared__ float sred[red_size<float>(1)];
  __shared__ int sflag;
  const int tid = threadIdx.x;
  const int pairs = blockDim.x / TS;
  const int p = tid % pairs, j = tid / pairs;
  const int x = blockIdx.x * 2 * pairs + 2 * p;
  const size_t base = (size_t)blockIdx.y * outer_stride + x;
  constexpr int LS = fx_line_stride<N, RM, false>();
  fx* sr = reinterpret_cast<fx*>(smem_raw) + (size_t)p * 2 * LS;
  fx* si = sr + LS;
  // theta of this thread's elements, copied asynchronously while the
  // transform runs: [q][j][p] (each thread reads what it copied)
  double2* pre = reinterpret_cast<double2*>(smem_raw + (size_t)pairs * 2 * LS * sizeof(fx));
  double xr[R], xi[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const size_t idx = base + (size_t)(j + q * TS) * line_stride;
    const double2 v = *reinterpret_cast<const double2*>(data + idx);
    cp_async_16(pre + ((size_t)(q * TS + j) * pairs + p), theta + idx);
    xr[q] = v.x;
    xi[q] = v.y;
  }
  const FxLine ln = fx_cols_transform<N, RM>(xr, xi, p, j, pairs, sr, si, scr, tab);
  cp_async_wait_all();
  const double mo = symo != nullptr ? symo[blockIdx.y] : 0.0;
  const double mx[2] = {symx[x] + mo, symx[x + 1] + mo};
  float acc = 0.0f;
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int kk = j + q * TS;
    fx w[2];
    dht_split(sr, si, kk, N, w[0], w[1]);
    const double ml = syml[kk];
    const size_t idx = base + (size_t)kk * line_stride;
    const double2 th = pre[(size_t)(q * TS + j) * pairs + p];
    const double thv[2] = {th.x, th.y};
    double outv[2];
    float o32[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const double h = fx_leave<N, RM>(w[c], ln, 0);
      const bool live = !(x + c == 0 && blockIdx.y == 0 && kk == 0);  // mu > 0: every mode but the zero one
      if (EPI == EPI_THETA) {
        if (!live && dc != nullptr) *dc = h;
        outv[c] = live ? fma(h, recip_pos(mx[c] + ml), thv[c]) : thv[c];
      } else {
        o32[c] = live ? (float)(h - thv[c]) : 0.0f;
        acc = fmaf(o32[c], o32[c], acc);
      }
    }
    if (EPI == EPI_THETA) {
      *reinterpret_cast<double2*>(theta + idx) = make_double2(outv[0], outv[1]);
    } else {
      *reinterpret_cast<float2*>(out32 + idx) = make_float2(o32[0], o32[1]);
    }
  }
  if (EPI == EPI_RESID) {
    float v[1] = {acc};
    block_reduce<float, 1, false>(v, sred);
    if (publish_and_check_last<float>(v, 1, reinterpret_cast<float*>(partials), &ctrl->counter[CS_MID], &sflag)) {
      float tt[1];
      gather_partials<float, 1, false>(tt, reinterpret_cast<const float*>(partials), sred);
      if (tid == 0) {
        ctrl->res_l2 = sqrt((double)tt[0] * kp.hd * kp.inv_ntot);
        ctrl->res_linf = -1.0;
        ctrl->counter[CS_MID] = 0;
      }
    }
  }
}

// ------------------------------------------------------------- middle pass
// FP64 form of k_mid (dht_kernels.cuh), lines along the last axis.  The symbol
// division and the Parseval sums are FP64; both transforms are fixed point, each with
// its own line exponents.  MIRROR (3D): the two lines of a thread's pair mirror each
// other in y (y and ny - y; lines 0 and ny / 2, which mirror themselves, make one
// pair), so that mu and the reciprocal of the symbol are formed once for two modes:
// the FP64 pipe, with 11 (order 4) and 16 (order 6) operations a mode at 1.74 per
// clock and SM, was 50 to 80% of the pass.  Otherwise they are x and x + 1.
template <int N, int RM, int ORDER, bool MIRROR>
__global__ void __launch_bounds__(kFxThreads, 2)
    k_mid_fx(double* data, unsigned line_stride, unsigned outer_stride, int ntx, KParams kp, Ctrl* ctrl,
             double* partials, double* xi_, double* dspec, const double* __restrict__ symx,
             const double* __restrict__ symo, const double* __restrict__ syml, const fx_tw* __restrict__ tab,
             int scale_e) {
  using F = LineFFT<fx, N, RM>;
  constexpr int R = F::R, TS = F::TS;
  if (ctrl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint2 scr[kFxThreads / 32][32];
  __shared__ double sred[red_size<double>(3)];
  __shared__ int sflag;
  const int tid = threadIdx.x;
  const int pairs = blockDim.x / TS;
  const int p = tid % pairs, j = tid / pairs;
  constexpr int LS = fx_line_stride<N, RM, false>();
  fx* sr = reinterpret_cast<fx*>(smem_raw) + (size_t)p * 2 * LS;
  fx* si = sr + LS;
  // order 6: xi and dspec of the tile, copied while the transform runs
  double2* pre_x = reinterpret_cast<double2*>(smem_raw + (size_t)pairs * 2 * LS * sizeof(fx));
  double2* pre_d = pre_x + (size_t)N * pairs;
  const int x = ((int)blockIdx.x % ntx * pairs + p) * (MIRROR ? 1 : 2), yo = (int)blockIdx.x / ntx;
  const int y1 = !MIRROR ? yo : (yo == 0 ? kp.ny >> 1 : kp.ny - yo);  // of the second line
  const bool self = !MIRROR || yo == 0;                               // each line has its own mu
  const unsigned base0 = (unsigned)yo * outer_stride + (unsigned)x;   // every grid has fewer than 2^32 cells
  const unsigned base1 = (unsigned)y1 * outer_stride + (unsigned)x;   // MIRROR
  double xr[R], xi[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const unsigned off = (unsigned)(j + q * TS) * line_stride;
    if (ORDER == 6) {
      const unsigned e = (unsigned)(q * TS + j) * pairs + p;
      if (MIRROR) {
        cp_async_8(&pre_x[e].x, xi_ + base0 + off);
        cp_async_8(&pre_x[e].y, xi_ + base1 + off);
        cp_async_8(&pre_d[e].x, dspec + base0 + off);
        cp_async_8(&pre_d[e].y, dspec + base1 + off);
      } else {
        cp_async_16(pre_x + e, xi_ + base0 + off);
        cp_async_16(pre_d + e, dspec + base0 + off);
      }
    }
    if (MIRROR) {
      xr[q] = data[base0 + off];
      xi[q] = data[base1 + off];
    } else {
      const double2 v = *reinterpret_cast<const double2*>(data + base0 + off);
      xr[q] = v.x;
      xi[q] = v.y;
    }
  }
  FxLine ln = fx_cols_transform<N, RM>(xr, xi, p, j, pairs, sr, si, scr, tab);
  if (ORDER == 6) cp_async_wait_all();
  const KConst<double>& C = kp.c64;
  const double s = C.s, se2 = C.se2, sl = C.sl;
  const double alpha_prev = ORDER == 6 ? ctrl->alpha : 0.0;
  const double mo = symo != nullptr ? symo[yo] : 0.0;
  const double mxa = symx[x] + mo, mxb = MIRROR ? symx[x] + symo[y1] : symx[x + 1] + mo;
  double acc[mid_nsums<double, ORDER>()] = {};
  auto put = [&](double* f, unsigned off, double a, double b) {
    if (MIRROR) {
      f[base0 + off] = a;
      f[base1 + off] = b;
    } else {
      *reinterpret_cast<double2*>(f + base0 + off) = make_double2(a, b);
    }
  };
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int kk = j + q * TS;
    fx w[2];
    dht_split(sr, si, kk, N, w[0], w[1]);
    const double ml = syml[kk];
    double mu = 0.0, ip = 0.0, wl = 0.0, dv[2];  // wl: the symbol without its s mu (order 6: s mu^2) term
    if (ORDER == 4) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const double h = fx_leave<N, RM>(w[c], ln, 0);
        if (c == 0 || self) {
          mu = (c ? mxb : mxa) + ml;
          wl = fma(se2 * mu, mu, 1.0);
          ip = recip_pos(fma(s, mu, wl));
        }
        const double d = h * ip;
        dv[c] = d;
        acc[0] = fma(h, d, acc[0]);
        acc[1] = fma(wl * d, d, acc[1]);
      }
    } else {
      // xi advances with the previous step and is added to the transformed
      // local residual; d = mu rt / P and T_h d = rt / P, P = 1 + mu (lam s +
      // mu (s + s eps^2 mu)) (see k_mid), formed as wl + s mu^2
      const unsigned off = (unsigned)kk * line_stride, e = (unsigned)(q * TS + j) * pairs + p;
      const double2 xv = pre_x[e], dp = pre_d[e];
      const double xs[2] = {xv.x, xv.y}, ds[2] = {dp.x, dp.y};
      double xn[2], tn[2];
      double mus[2], ips[2], wls[2];
      auto symbol = [&](double m, double& w) {
        const double m2 = m * m;
        w = fma(fma(se2, m2, sl), m, 1.0);
        return recip_pos(fma(s, m2, w));
      };
      if (MIRROR) {  // both before the conversions: 187 us for a solve of L_h at 128^3, else 191
        mus[0] = mxa + ml;
        mus[1] = self ? mxb + ml : mus[0];
        ips[0] = symbol(mus[0], wls[0]);
        ips[1] = ips[0];
        wls[1] = wls[0];
        if (self) ips[1] = symbol(mus[1], wls[1]);
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const double h = fx_leave<N, RM>(w[c], ln, 0);
        double rt = 0.0, d = 0.0, xc = 0.0, td = 0.0;
        if (MIRROR) {
          mu = mus[c];
          ip = ips[c];
          wl = wls[c];
        } else {
          mu = (c ? mxb : mxa) + ml;
          ip = symbol(mu, wl);
        }
        if (!(c == 0 && yo == 0 && x == 0 && kk == 0)) {  // mu > 0: every mode but the zero one
          xc = fma(-alpha_prev, ds[c], xs[c]);
          rt = h + xc;
          td = rt * ip;
          d = mu * td;
        }
        xn[c] = xc;
        tn[c] = td;
        dv[c] = d;
        acc[0] = fma(rt, d, acc[0]);
        acc[1] = fma(wl * td, d, acc[1]);
        acc[mid_nsums<double, ORDER>() - 1] = fma(rt, rt, acc[mid_nsums<double, ORDER>() - 1]);
      }
      put(xi_, off, xn[0], xn[1]);
      put(dspec, off, tn[0], tn[1]);
    }
    xr[q] = dv[0];
    xi[q] = dv[1];
  }
  // the barrier inside, before the line buffers are written again, comes
  // after every thread has read the forward spectrum
  ln = fx_cols_transform<N, RM>(xr, xi, p, j, pairs, sr, si, scr, tab);
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int kk = j + q * TS;
    fx h1, h2;
    dht_split(sr, si, kk, N, h1, h2);
    put(data, (unsigned)kk * line_stride, fx_leave_hw<N, RM>(h1, ln, scale_e), fx_leave_hw<N, RM>(h2, ln, scale_e));
  }
  mid_finish<double, ORDER>(acc, sred, partials, ctrl, kp, &sflag);
}

// ------------------------------------------------------------ launch helpers
// Line pairs per block: as many as fill 256 threads, fewer while the grid
// would leave SMs without a block (down to one warp; strided passes keep two
// pairs, whole 32-byte sectors).  total: line pairs of the pass.  On a 64^2 grid
// (eight blocks of one warp instead of one of 256 threads, on one SM) a row pass
// takes 7.6 us instead of 21 and the middle pass 15.5 instead of 59, fixed point,
// narrowing and radix 4 together.
template <int N, int RM, bool ROWS>
int fx_pairs(long long total, int avail, int nsm) {
  constexpr int TS = LineFFT<fx, N, RM>::TS;
  int pairs = kFxThreads / TS;
  while (pairs > 1 && pairs > avail) pairs >>= 1;
  while (pairs > (ROWS ? 1 : 2) && pairs * TS > 32 && total / pairs < nsm) pairs >>= 1;
  return pairs;
}
// Whether a pass over a field of `cells` takes radix 4 instead of 8: with 16
// points per thread (8 of each line of the pair) the grid would have fewer than
// eight warps per SM, and a thread's chain of integer and FP64 work is the time.
// Lines of 512 and more keep radix 8: with two more passes dividing by 4, decaying
// lines would lose more than FP64 does.
template <int N>
constexpr int kFxShort = N <= 256 ? 4 : 8;
inline bool fx_short(long long cells, int nsm) { return cells / 16 < 256LL * nsm; }
// The exponent of a power-of-two scale (every pass scales by 1 or 1/N).
inline bool fx_scale_exp(double scale, int* e) {
  const double m = std::frexp(scale, e);
  *e -= 1;
  return m == 0.5;
}

template <int N, int RM, typename SI>
cudaError_t rows_fx_impl(const SI* src, const SI* src_odd, const int* iter, double* dst, int nrows, double scale, const int* done,
                         const AxisTables<double>& tb, cudaStream_t st, unsigned int* dmax_hi) {
  constexpr int TS = LineFFT<fx, N, RM>::TS;
  int se;
  if (!fx_scale_exp(scale, &se)) return cudaErrorInvalidValue;
  const int np = (nrows + 1) / 2;
  const int pairs = fx_pairs<N, RM, true>(np, 1 << 30, tb.nsm);
  k_rows_fx<N, RM, SI><<<(np + pairs - 1) / pairs, pairs * TS, pairs * fx_pair_smem<N, RM, true>(), st>>>(src, src_odd, iter, dst, nrows, se,
                                                                                                 done, tb.fxtw[0], dmax_hi);
  return cudaGetLastError();
}

template <int N, int RM>
cudaError_t cols_fx_impl(double* data, int nx, int nouter, size_t line_stride, size_t outer_stride, double scale,
                         const int* done, const fx_tw* tab, int nsm, cudaStream_t st) {
  constexpr int TS = LineFFT<fx, N, RM>::TS;
  int se;
  if (!fx_scale_exp(scale, &se)) return cudaErrorInvalidValue;
  const int pairs = fx_pairs<N, RM, false>((long long)(nx / 2) * nouter, nx / 2, nsm);
  k_cols_fx<N, RM><<<dim3(nx / (2 * pairs), nouter), pairs * TS, pairs * fx_pair_smem<N, RM, false>(), st>>>(
      data, line_stride, outer_stride, se, done, tab);
  return cudaGetLastError();
}

// Line and outer strides of the last axis (y in 2D, z in 3D).
struct LastAxis {
  size_t line_stride, outer_stride;
  int nouter, ax;
};
inline LastAxis last_axis(const KParams& kp) {
  if (kp.dim == 2) return {(size_t)kp.nx, 0, 1, 1};
  return {(size_t)kp.nx * kp.ny, (size_t)kp.nx, kp.ny, 2};
}

template <int N, int RM, bool MIRROR>
cudaError_t mid_fx_launch(double* data, const KParams& kp, Ctrl* ctrl, double* partials, double* xi, double* dspec,
                          const AxisTables<double>& tb, cudaStream_t st) {
  constexpr int TS = LineFFT<fx, N, RM>::TS;
  const LastAxis a = last_axis(kp);
  int se;
  if (!fx_scale_exp(kp.inv_ntot, &se)) return cudaErrorInvalidValue;
  const int cols = MIRROR ? kp.nx : kp.nx / 2, nout = MIRROR ? kp.ny / 2 : a.nouter;
  const int pairs = fx_pairs<N, RM, false>((long long)cols * nout, cols, tb.nsm);
  const int ntx = cols / pairs;
  const double* symo = kp.dim == 2 ? nullptr : tb.sym[1];
  const size_t sm = pairs * fx_pair_smem<N, RM, false>() + (kp.order == 6 ? 2 : 0) * (size_t)N * pairs * sizeof(double2);
  if (kp.order == 4)
    k_mid_fx<N, RM, 4, MIRROR><<<ntx * nout, pairs * TS, sm, st>>>(
        data, (unsigned)a.line_stride, (unsigned)a.outer_stride, ntx, kp, ctrl, partials, xi, dspec, tb.sym[0], symo,
         tb.sym[a.ax], tb.fxtw[a.ax], se);
  else
    k_mid_fx<N, RM, 6, MIRROR><<<ntx * nout, pairs * TS, sm, st>>>(
        data, (unsigned)a.line_stride, (unsigned)a.outer_stride, ntx, kp, ctrl, partials, xi, dspec, tb.sym[0], symo,
         tb.sym[a.ax], tb.fxtw[a.ax], se);
  return cudaGetLastError();
}
// Mirrored pairs of lines where a block reads whole 32-byte sectors of a row (four
// columns; shorter blocks are those of 1024-point lines and of the smallest grids).
// Solve of L_h at 64x256x128, order 4: 156 -> 142 us; middle pass of order 6 at 256^3: 582 -> 534 us,
// of order 4 at 128^3: 92 -> 76.5 us.
// In 2D, where x is the axis to mirror, it loses: the rows' sectors are split between
// blocks (1024^2, order 6, whole solve of L_h: 107 us adjacent, 127 us mirrored).
template <int N, int RM>
cudaError_t mid_fx_impl(double* data, const KParams& kp, Ctrl* ctrl, double* partials, double* xi, double* dspec,
                        const AxisTables<double>& tb, cudaStream_t st) {
  if (kp.dim == 3 && fx_pairs<N, RM, false>((long long)kp.nx * (kp.ny / 2), kp.nx, tb.nsm) >= 4)
    return mid_fx_launch<N, RM, true>(data, kp, ctrl, partials, xi, dspec, tb, st);
  return mid_fx_launch<N, RM, false>(data, kp, ctrl, partials, xi, dspec, tb, st);
}

template <int N, int RM>
cudaError_t last_fx_impl(const double* data, double* theta, float* out32, const KParams& kp, Ctrl* ctrl,
                         double* partials, const AxisTables<double>& tb, cudaStream_t st, double* dc,
                         const int* skip) {
  constexpr int TS = LineFFT<fx, N, RM>::TS;
  const LastAxis a = last_axis(kp);
  const int pairs = fx_pairs<N, RM, false>((long long)(kp.nx / 2) * a.nouter, kp.nx / 2, tb.nsm);
  const dim3 grid(kp.nx / (2 * pairs), a.nouter);
  const size_t sm = pairs * fx_pair_smem<N, RM, false>() + (size_t)N * pairs * sizeof(double2);
  const double* symo = kp.dim == 2 ? nullptr : tb.sym[1];
  if (out32 == nullptr)
    k_last_fx<N, RM, EPI_THETA><<<grid, pairs * TS, sm, st>>>(data, theta, out32, a.line_stride, a.outer_stride, kp, ctrl,
                                                          partials, tb.fxtw[a.ax], tb.sym[0], symo, tb.sym[a.ax], dc,
                                                          skip);
  else
    k_last_fx<N, RM, EPI_RESID><<<grid, pairs * TS, sm, st>>>(data, theta, out32, a.line_stride, a.outer_stride, kp, ctrl,
                                                          partials, tb.fxtw[a.ax], tb.sym[0], symo, tb.sym[a.ax],
                                                          nullptr, skip);
  return cudaGetLastError();
}

}  // namespace
}  // namespace psd
