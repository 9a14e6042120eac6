// Shared device-side definitions of the PSD library: parameter blocks, the
// device-resident control block, and deterministic grid reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace psd {

// Kinds of the vertex factor |g|^{p-2}: specialised p = 3 (|g|), p = 4 (|g|^2)
// and p = 6 (|g|^4 = (|g|^2)^2), and a general p (pow).
enum PKind { PK_GEN = 0, PK_3 = 3, PK_4 = 4, PK_6 = 6 };
inline int pkind_of(double p) { return p == 3.0 ? PK_3 : p == 4.0 ? PK_4 : p == 6.0 ? PK_6 : PK_GEN; }

// Slots of the "last block" counters in the control block.
enum CounterSlot { CS_RES = 0, CS_MID = 1, CS_LS = 2, CS_MISC = 3, CS_COUNT = 8 };

// Device-resident state of one PSD run.  Written only by the last block of
// a reducing kernel (or by the host between runs).
struct Ctrl {
  int done;        // 1: converged, failed or stopped -> later kernels return
  int iter;        // completed PSD iterations
  int status;      // psd_status of the run
  int max_iter;    // iteration limit for this run
  double alpha;    // step size of the current iteration
  double tol;      // stop when res_l2 < tol
  double res_l2;   // ||r||_2 of the current iterate
  double res_linf; // max |r| of the current iterate (-1 if not formed)
  double rd;       // (r, d)_2 of the current direction, by Parseval
  double dd, lapdd, tdd;  // sums of the discrete energies (psd_energy)
  double lin;      // cu (d, d)_2 + (T_h d, d)_2 + s eps^2 (Delta_h d, Delta_h d)_2: q's linear part
  // line search: the first three polynomial coefficients of q (p = 4, 6;
  // weighted by h^d and s), or the general-p Newton state (c1, c2 = bracket,
  // c3 = converged flag)
  double c1, c2, c3;
  double trial;    // general p: the step size at which the next Newton pass evaluates q
  // inner (mixed-precision) stop on the preconditioned residual norm
  // (r, L_h^{-1} r)^{1/2} = ||d||_L (Eq. "RRT-1"): done when it drops below
  // pre_eta times its first value pre_ref (pre_eta <= 0 disables).
  double pre_eta;
  double pre_ref;
  double pre_win;  // value at the start of the current stall window
  int pre_stall;   // iterations without halving pre_win
  int pre_stall_max;
  // conjugate gradients (the adjoint solve): cg = 1 switches the middle pass
  // and the Hessian-vector kernel to their CG bookkeeping -- the middle pass
  // forms beta = (r, z) / rz into alpha and stores rz = (r, z); the
  // Hessian-vector kernel forms alpha = rz / (p, H p)
  int cg;
  int cg_pad_;
  double rz;
  // device-side loop control of graph-driven solves (WHILE nodes)
  int guard;        // body executions of the current loop (a hard cap)
  int ls_pass;      // general-p line search: Newton passes of this iteration
  int outer;        // mixed solve: FP64 outer residual evaluations
  int inner_total;  // mixed solve: inner iterations so far
  int max_outer;
  int cfg_pad_;
  double last_alpha;
  unsigned int counter[CS_COUNT];
  // FP64 p = 4 stencils (fixed-point variants): bounds on |u| and on the
  // vertex gradient sums |G| of the last residual's iterate (umax < 0: none),
  // the high word of a bound on |d| (the x pass that ends the preconditioner),
  // the scales of the next residual (fx_s = kFxOff: the FP64 variant), and
  // running maxima (high words of bounds, zero between kernels)
  double umax, gmax;
  unsigned int dmax_hi, umax_hi, gmax2_hi;
  int fx_s, fx_g;
  int hist_cap;
  double* hist_alpha;  // device arrays of length hist_cap (or null)
  double* hist_res;
  double ls_step;  // general p: how far the last Newton pass moved trial (0: first pass of the iteration)
};

// Problem scalars passed by value to the kernels.
// Constants of the operator in a kernel's arithmetic type, formed once on
// the host.  (Formed in a kernel from the FP64 parameters, a value such as
// (float)(s * eps2) may be recomputed inside unrolled loops when registers
// are short, and GB300 issues FP64 at 1/64 of the FP32 rate.)
template <typename T>
struct KConst {
  T s, se2, sl, cu;  // s, s eps^2, s lambda, coefficient of u
  T cdiv, cbih;      // see KParams
  T inv_h, inv_ntot;
  T beta, pm2;       // (p - 2) / 2, p - 2
};

struct KParams {
  int nx, ny, nz;       // cells per axis (nz = 1 in 2D)
  int dim;
  double h, inv_h;      // spacing
  double s, eps2, lam;  // s, eps^2, lambda
  double p;             // exponent
  double cu;            // coefficient of u in N_h: 1 (order 4) or s*lambda (6)
  double hd;            // h^d (cell volume)
  double inv_ntot;      // 1 / (nx ny nz)
  int order;
  double fx_lin;        // 64 2^-53 cbih and |Omega|^{1/2}: the error rule of the fixed-point residual
  double sqrt_vol;
  int nsm;              // SMs of the current device (finish_kparams; sizes one-wave grids)
  // derived constants (set by finish_kparams): the column kernels work with
  // unscaled vertex-gradient sums G = g / q and Laplacian sums h^2 Delta_h.
  double q;             // 1 / (2^(d-1) h): g = q G
  double cdiv;          // s q^p: s d.(|g|^{p-2} g) = cdiv * (sum of differences of |G|^{p-2} G)
  double cbih;          // s eps^2 / h^4: s eps^2 Delta_h^2 u = cbih * (h^4 Delta_h^2 u)
  KConst<double> c64;   // the constants in FP64 and FP32 (finish_kparams)
  KConst<float> c32;
};

template <typename T>
__device__ __forceinline__ const KConst<T>& kconst(const KParams& kp);
template <>
__device__ __forceinline__ const KConst<double>& kconst<double>(const KParams& kp) {
  return kp.c64;
}
template <>
__device__ __forceinline__ const KConst<float>& kconst<float>(const KParams& kp) {
  return kp.c32;
}

// Fill the derived constants of KParams (host side).
inline void finish_kparams(KParams& kp) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      sms <= 0)
    sms = 152;
  kp.nsm = sms;
  kp.q = kp.inv_h / (kp.dim == 3 ? 4.0 : 2.0);
  const double qp = (kp.p == 4.0) ? kp.q * kp.q * kp.q * kp.q : std::pow(kp.q, kp.p);
  kp.cdiv = kp.s * qp;
  kp.cbih = kp.s * kp.eps2 * kp.inv_h * kp.inv_h * kp.inv_h * kp.inv_h;
  kp.fx_lin = 64.0 * std::ldexp(1.0, -53) * kp.cbih;
  kp.sqrt_vol = std::sqrt(kp.hd / kp.inv_ntot);
  KConst<double>& d = kp.c64;
  d.s = kp.s;
  d.se2 = kp.s * kp.eps2;
  d.sl = kp.s * kp.lam;
  d.cu = kp.cu;
  d.cdiv = kp.cdiv;
  d.cbih = kp.cbih;
  d.inv_h = kp.inv_h;
  d.inv_ntot = kp.inv_ntot;
  d.beta = 0.5 * (kp.p - 2.0);
  d.pm2 = kp.p - 2.0;
  KConst<float>& f = kp.c32;
  f.s = (float)d.s;
  f.se2 = (float)d.se2;
  f.sl = (float)d.sl;
  f.cu = (float)d.cu;
  f.cdiv = (float)d.cdiv;
  f.cbih = (float)d.cbih;
  f.inv_h = (float)d.inv_h;
  f.inv_ntot = (float)d.inv_ntot;
  f.beta = (float)d.beta;
  f.pm2 = (float)d.pm2;
}

// -------------------------------------------- scales of the fixed-point stencils
constexpr int kFxOff = -10000;

// These run in one thread at the end of a reduction, where a dependent FP64
// operation takes 65 clocks: exponents are taken from the bits.
//
// e with v (1 + 2^-20) < 2^e, from the bits of a finite v >= 0 (zero: -1022).
__device__ __forceinline__ int fx_exp_above(double v) {
  const unsigned h = (unsigned)__double2hiint(v) + 2u;  // at least v (1 + 2^-20)
  return (int)(h >> 20) - 1022;
}
__device__ __forceinline__ bool fx_finite(double v) { return ((unsigned)__double2hiint(v) & 0x7FFFFFFFu) < 0x7FE00000u; }
// The scale S with |v| 2^S < 2^55 for |v| <= vmax (1 + 2^-20) (zero: 55); false
// when vmax is not finite or S is outside [-200, 200].
__device__ __forceinline__ bool fx_scale_of(double vmax, int* S) {
  if (!fx_finite(vmax)) return false;
  *S = vmax > 0.0 ? 55 - fx_exp_above(vmax) : 55;
  return *S >= -200 && *S <= 200;
}
// Choose the scales of a fixed-point residual for |u| <= umax, |G| <= gmax into
// c: S, and the shift g of the gradient sums with |G| 2^(S+g) < 2^61 (|G| < 16
// max|u|, so g >= 2).  With 2^ge = 2^(61-S-g) >= |G|, the flux error is at most cdiv
// 2^-51 2^(3 ge) per cell (24 fluxes of a few units of 2^-58 of the cube of 2^ge);
// the variant runs when that is below the FP64 rounding of the Laplacian sums,
// about 64 units 2^-53 of cbih max|u|.  Otherwise (gradients steeper than any smooth
// field on the grid) the FP64 variant runs.  tol > 0, for the outer residuals of 3D
// mixed solves only: also when the error is below tol / 20 in the 2-norm.
template <class C, class K>
__device__ __forceinline__ void fx_decide(C* c, const K& kp, double umax, double gmax, double tol) {
  int S = kFxOff, g = 60;
  if (!(umax >= 0.0) || !fx_finite(gmax) || !fx_scale_of(umax, &S)) {
    c->fx_s = kFxOff;
    return;
  }
  if (gmax > 0.0) g = 61 - S - fx_exp_above(gmax);
  g = g < 2 ? 2 : (g > 60 ? 60 : g);
  const int e3 = 3 * (61 - S - g) - 51;
  const double err = kp.cdiv * __hiloint2double((e3 < -1000 ? 23 : e3 + 1023) << 20, 0);
  const bool ok = umax == 0.0 || err <= kp.fx_lin * umax || err * kp.sqrt_vol < 0.05 * tol;
  c->fx_s = ok ? S : kFxOff;
  c->fx_g = g;
}
// An upper bound of sqrt(v) (within 2^-20) from the high word of v >= 0.
__device__ __forceinline__ double fx_sqrt_above(unsigned hi) {
  if (hi == 0u) return 0.0;
  const int e = ((int)(hi >> 20) - 1023) & ~1;  // even exponent: v = m 2^e, m in [1, 4)
  const float m = __uint_as_float((((hi >> 20) - 1023u - (unsigned)e + 127u) << 23) | ((hi & 0xFFFFFu) << 3));
  const float r = sqrtf(m) * (1.0f + 0x1p-20f);  // in [1, 2]
  const unsigned b = __float_as_uint(r);
  return __hiloint2double((int)((((b >> 23) - 127u + (unsigned)(e / 2) + 1023u) << 20) | ((b >> 3) & 0xFFFFFu)),
                          (int)(b << 29));
}

// ------------------------------------------------------------------ reductions

// fmax(m, |x|) for m >= 0 (a NaN leaves m).  FP64 as integers: the bits of
// non-negative values are ordered, and an FP64 comparison takes the slot of an addition.
__device__ __forceinline__ float max_abs(float m, float x) { return fmaxf(m, fabsf(x)); }
__device__ __forceinline__ double max_abs(double m, double x) {
  const long long b = __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL;
  return b > __double_as_longlong(m) && b <= 0x7FF0000000000000LL ? __longlong_as_double(b) : m;
}

// Block maxima of two values, for every thread (one-dimensional blocks of
// whole warps); sh: two words of shared memory.
__device__ __forceinline__ void block_max2(unsigned& a, unsigned& b, unsigned* sh) {
  if (threadIdx.x < 2) sh[threadIdx.x] = 0u;
  __syncthreads();
  a = __reduce_max_sync(0xffffffffu, a);
  b = __reduce_max_sync(0xffffffffu, b);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&sh[0], a);
    atomicMax(&sh[1], b);
  }
  __syncthreads();
  a = sh[0];
  b = sh[1];
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Shared words of block_reduce over m values of type A in a block of up to
// 256 threads.
template <typename A>
__host__ __device__ constexpr int red_size(int m) {
  return (sizeof(A) == 8 ? 256 : 32) * m;
}

// Reduce M values of type A over the block in a fixed order; the result is
// valid in thread 0.  The last value is reduced with max when LASTMAX is set,
// every value when ALLMAX is.  FP32 kernels reduce in float, by warp
// butterflies and then warp 0 over the warp results.  FP64 kernels reduce in
// double through shared memory, each value summed by a group of up to 32
// lanes: an FP64 instruction occupies the pipe for 16 clocks and its warp for
// 65 whatever the lanes it needs, so the butterflies' 5 (M + M nthr / 32) adds
// (225 for 5 values of 256 threads) cost 2 us, the groups' 12 M adds a third.
// Requires blockDim to be a power of two (below 32: thread 0 sums serially);
// sh: red_size<A>(M).
template <typename A, int M, bool LASTMAX, bool ALLMAX = false>
__device__ __forceinline__ void block_reduce(A (&v)[M], A* sh) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int nthr = blockDim.x * blockDim.y * blockDim.z;
  auto op = [](int m, A x, A y) { return (ALLMAX || (LASTMAX && m == M - 1)) ? fmax(x, y) : x + y; };
  if (nthr < 32) {
    __syncthreads();
#pragma unroll
    for (int m = 0; m < M; ++m) sh[tid * M + m] = v[m];
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        A acc = sh[m];
        for (int t = 1; t < nthr; ++t) acc = op(m, acc, sh[t * M + m]);
        v[m] = acc;
      }
    }
    __syncthreads();
    return;
  }
  if constexpr (sizeof(A) == 8) {
    int P = 32;  // lanes per value
    while (P * M > nthr) P >>= 1;
    __syncthreads();
#pragma unroll
    for (int m = 0; m < M; ++m) sh[m * nthr + tid] = v[m];
    __syncthreads();
    if ((tid & ~31) < P * M) {  // the warps that hold a group
      const int m = tid / P, l = tid - m * P;
      A x = A(0);
      if (m < M) {
        x = sh[m * nthr + l];
        for (int t = l + P; t < nthr; t += P) x = op(m, x, sh[m * nthr + t]);
      }
      for (int o = P >> 1; o > 0; o >>= 1) x = op(m, x, __shfl_xor_sync(0xffffffffu, x, o));
      if (m < M && l == 0) sh[m * nthr] = x;
    }
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = sh[m * nthr];
    }
    __syncthreads();
  } else {
    const int lane = tid & 31, wid = tid >> 5, nw = (nthr + 31) >> 5;
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = (ALLMAX || (LASTMAX && m == M - 1)) ? warp_max(v[m]) : warp_sum(v[m]);
    __syncthreads();
    if (lane == 0) {
#pragma unroll
      for (int m = 0; m < M; ++m) sh[wid * M + m] = v[m];
    }
    __syncthreads();
    if (wid == 0) {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        A x = (lane < nw) ? sh[lane * M + m] : ((ALLMAX || (LASTMAX && m == M - 1)) ? A(-1) : A(0));
        v[m] = (ALLMAX || (LASTMAX && m == M - 1)) ? warp_max(x) : warp_sum(x);
      }
    }
    __syncthreads();
  }
}

// Write this block's partials, then return true in every thread of the
// block that finished last (threadFenceReduction pattern).  The last block
// can then read all partials with __ldcg.
template <typename A>
__device__ __forceinline__ bool publish_and_check_last(const A* v, int M, A* partials, unsigned int* counter,
                                                       int* sh_flag) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const unsigned int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  const unsigned int nb = gridDim.x * gridDim.y * gridDim.z;
  if (tid == 0) {
    for (int m = 0; m < M; ++m) partials[(size_t)bid * M + m] = v[m];
    __threadfence();
    unsigned int prev = atomicAdd(counter, 1u);
    *sh_flag = (prev == nb - 1) ? 1 : 0;
  }
  __syncthreads();
  return *sh_flag != 0;
}

// In the last block: sum the partials of all blocks in a fixed order (each
// thread a strided subset, then the block tree), result in thread 0.
template <typename A, int M, bool LASTMAX, bool ALLMAX = false>
__device__ __forceinline__ void gather_partials(A (&out)[M], const A* partials, A* sh) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int nthr = blockDim.x * blockDim.y * blockDim.z;
  const unsigned int nb = gridDim.x * gridDim.y * gridDim.z;
#pragma unroll
  for (int m = 0; m < M; ++m) out[m] = (ALLMAX || (LASTMAX && m == M - 1)) ? A(-1) : A(0);
  if (tid < (int)nb) {
#pragma unroll
    for (int m = 0; m < M; ++m) out[m] = __ldcg(partials + (size_t)tid * M + m);
  }
  for (unsigned int b = tid + nthr; b < nb; b += nthr) {
#pragma unroll
    for (int m = 0; m < M; ++m) {
      A x = __ldcg(partials + (size_t)b * M + m);
      out[m] = (ALLMAX || (LASTMAX && m == M - 1)) ? fmax(out[m], x) : out[m] + x;
    }
  }
  block_reduce<A, M, LASTMAX, ALLMAX>(out, sh);
}

// Tile order of the one-wave column march (residual and line-search
// kernels).  The column-planes w = column * nz + z are split into G =
// gridDim.x equal contiguous shares; the shares of CTAs b and b + G / g
// (g = gcd(G, ncol)) start exactly ncol / g whole columns apart, so those
// CTAs march the same plane at the same time.  The columns that agree
// modulo m = ncol / g are therefore in lockstep, and they are given
// consecutive tiles (whole rows of tiles when ncol / m is a multiple of the
// row length): a tile's x-neighbours are then read in the same plane step,
// and the halo reads they share hit L2 instead of DRAM.
__device__ __forceinline__ int lockstep_classes(int G, int ncol) {
  int a = G, b = ncol;
  while (b != 0) {
    const int t = a % b;
    a = b;
    b = t;
  }
  return ncol / a;
}
__device__ __forceinline__ int lockstep_tile(int col, int m, int ncol) { return (col % m) * (ncol / m) + col / m; }

__device__ __forceinline__ int wrapi(int i, int n) {  // n a power of two
  return i & (n - 1);
}

// Asynchronous global -> shared copies (cp.async, 8 or 16 bytes, both
// addresses aligned to the size); a thread that reads back only its own
// copies needs cp_async_wait_all() and no barrier.
__device__ __forceinline__ void cp_async_8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// Close the current group of this thread's cp.async copies; wait until at
// most N of its groups are still in flight.
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// 1/x for finite x >= 1 (the FP32 preconditioner symbols): the hardware
// reciprocal estimate (rcp.approx) refined by one Newton-Raphson step
// r <- r + r (1 - x r), which squares the estimate's relative error, so the
// result is within an ulp or so of 1/x; x >= 1 keeps it clear of denormals.
__device__ __forceinline__ float recip_ge1(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
// 1/x for x >= 0 in FP64 (the symbols, the line search's slopes): the hardware estimate
// (rcp.approx.ftz.f64, about 20 bits) with one step of the third-order Newton-Householder
// iteration for the reciprocal, r (1 + e + e^2), e = 1 - x r, which leaves e^3: within an
// ulp of 1/x (tests/recip64_check.cu) in three FP64 operations.  The estimate flushes
// subnormal arguments and results: those, 0, infinity and NaN take the quotient.
__device__ __forceinline__ double recip_pos(double x) {
  if ((unsigned)__double2hiint(x) - 0x00100000u >= 0x7FC00000u) return 1.0 / x;  // outside [2^-1022, 2^1022)
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace psd
