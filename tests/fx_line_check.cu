// Host check of the block fixed-point line FFT (csrc/fx_line.cuh): the same
// passes, butterflies, rotations, scaling and conversions as the device
// kernels, run thread by thread for every length, against a long-double
// transform.  For each kind of line its error (2-norm, relative) must not exceed
// that of the same Stockham passes in FP64; and the conversions, the special
// values and the extremes of the exponent range are checked; so is the flux of
// the fixed-point residual.  Built and run by
// tests/test_fx_line.py (no GPU needed).  Exit status 0 = pass.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../paper_1607_01475_gb300/csrc/fx_line.cuh"

using psd::fx;

static uint64_t rng_state = 0x1607014750ULL;
static uint64_t next_u64() {  // SplitMix64
  uint64_t z = (rng_state += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
static double uni() { return (double)(next_u64() >> 11) * 0x1p-53 * 2.0 - 1.0; }

static unsigned hi(double x) {
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return (unsigned)(b >> 32);
}
static unsigned lo(double x) {
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return (unsigned)b;
}

// Pass NS of the Stockham FFT over a whole line, thread by thread.
template <int N, int RM, int NS, typename T, typename Rot, typename Unt>
void pass(std::vector<T>& re, std::vector<T>& im, Rot rot, Unt unt) {
  constexpr int R = N < RM ? N : RM, TS = N / R, RP = (N / NS >= R) ? R : N / NS, M = R / RP;
  std::vector<T> ore(N), oim(N);
  for (int j = 0; j < TS; ++j)
    for (int b = 0; b < M; ++b) {
      const int jp = j + b * TS, jm = jp & (NS - 1);
      T xr[RP], xi[RP];
      for (int r = 0; r < RP; ++r) {
        xr[r] = re[j + (b + r * M) * TS];
        xi[r] = im[j + (b + r * M) * TS];
      }
      if (NS > 1) {
        unt(xr[0], xi[0]);
        for (int r = 1; r < RP; ++r) rot(jm * r * (N / (NS * RP)), xr[r], xi[r], r & 1);
      }
      psd::DFT<RP>::run(xr, xi);
      const int base = (jp / NS) * NS * RP + jm;
      for (int r = 0; r < RP; ++r) {
        ore[base + r * NS] = xr[r];
        oim[base + r * NS] = xi[r];
      }
    }
  re = ore;
  im = oim;
}

template <int N, int RM, int NS, typename T, typename Rot, typename Unt>
void passes(std::vector<T>& re, std::vector<T>& im, Rot rot, Unt unt) {
  constexpr int R = N < RM ? N : RM;
  if constexpr (NS < N) {
    constexpr int RP = (N / NS >= R) ? R : N / NS;
    pass<N, RM, NS>(re, im, rot, unt);
    passes<N, RM, NS * RP>(re, im, rot, unt);
  }
}

// Hartley outputs of the pair (x, y) in fixed point.
template <int N, int RM>
void run_fx(const std::vector<double>& x, const std::vector<double>& y, std::vector<double>& h1,
            std::vector<double>& h2) {
  using Plan = psd::FxPlan<N, RM>;
  std::vector<psd::fx_tw> tw(N);
  const long double pi = 3.141592653589793238462643383279502884L;
  for (int t = 0; t < N; ++t) tw[t] = psd::fx_make_tw(cosl(2 * pi * t / N), sinl(2 * pi * t / N));
  unsigned eb = 0;
  for (int i = 0; i < N; ++i) {
    eb = std::max(eb, hi(x[i]) & 0x7FFFFFFFu);
    eb = std::max(eb, hi(y[i]) & 0x7FFFFFFFu);
  }
  const int E = (int)(eb >> 20);
  const bool live = E >= psd::kFxMinExp && E <= psd::kFxMaxExp;
  std::vector<fx> re(N), im(N);
  unsigned l1 = 0;
  for (int i = 0; i < N; ++i) l1 += psd::fx_l1(hi(x[i]), E) + psd::fx_l1(hi(y[i]), E);
  const int scale = psd::fx_scale<Plan>(l1);
  for (int i = 0; i < N; ++i) {
    re[i] = psd::fx_quantise(hi(x[i]), lo(x[i]), E, scale);
    im[i] = psd::fx_quantise(hi(y[i]), lo(y[i]), E, scale);
    if (!live) re[i].v = im[i].v = 0;
  }
  passes<N, RM, 1>(
      re, im, [&](int t, fx& a, fx& b, bool odd) { psd::fx_rotate(a, b, tw[t], odd); },
      [](fx& a, fx& b) {
        a = psd::fx_quarter(a);
        b = psd::fx_quarter(b);
      });
  h1.resize(N);
  h2.resize(N);
  for (int m = 0; m < N; ++m) {
    const int m2 = (N - m) & (N - 1);
    const fx A = re[m], B = im[m], C = re[m2], D = im[m2];
    const fx a = (A - B) + (C + D), b = (A + B) - (C - D);
    h1[m] = E > psd::kFxMaxExp ? NAN : psd::fx_result(a.v, E - scale + Plan::kOut);
    h2[m] = E > psd::kFxMaxExp ? NAN : psd::fx_result(b.v, E - scale + Plan::kOut);
  }
}

// The same passes in FP64.
template <int N, int RM>
void run_f64(const std::vector<double>& x, const std::vector<double>& y, std::vector<double>& h1,
             std::vector<double>& h2) {
  const long double pi = 3.141592653589793238462643383279502884L;
  std::vector<double> c(N), s(N), re = x, im = y;
  for (int t = 0; t < N; ++t) {
    c[t] = (double)cosl(2 * pi * t / N);
    s[t] = (double)sinl(2 * pi * t / N);
  }
  passes<N, RM, 1>(
      re, im,
      [&](int t, double& a, double& b, bool) {
        const double a0 = a;
        a = std::fma(b, s[t], a * c[t]);
        b = std::fma(-a0, s[t], b * c[t]);
      },
      [](double&, double&) {});
  h1.resize(N);
  h2.resize(N);
  for (int m = 0; m < N; ++m) {
    const int m2 = (N - m) & (N - 1);
    h1[m] = 0.5 * ((re[m] - im[m]) + (re[m2] + im[m2]));
    h2[m] = 0.5 * ((re[m] + im[m]) - (re[m2] - im[m2]));
  }
}

template <int N>
std::vector<long double> exact(const std::vector<double>& x) {
  static std::vector<long double> cas;
  if (cas.empty()) {
    const long double pi = 3.141592653589793238462643383279502884L;
    for (int t = 0; t < N; ++t) cas.push_back(cosl(2 * pi * t / N) + sinl(2 * pi * t / N));
  }
  std::vector<long double> out(N);
  for (int k = 0; k < N; ++k) {
    long double a = 0;
    for (int j = 0; j < N; ++j) a += x[j] * cas[(int)((long long)j * k % N)];
    out[k] = a;
  }
  return out;
}

static int fails = 0;

template <int N, int RM>
void check() {
  // kinds of lines: dense, one large point, spectra decaying like k^-4 and
  // exp(-k^2 / 64), a constant, a smooth mode, values over 60 binades, tiny and
  // huge scales
  const char* names[] = {"dense", "spike", "k^-4", "gauss", "constant", "mode", "wide", "tiny", "huge"};
  for (int kind = 0; kind < 9; ++kind) {
    long double efx = 0, ef64 = 0, norm = 0;
    for (int trial = 0; trial < (N <= 64 ? 40 : 8); ++trial) {
      std::vector<double> x(N), y(N), a, b, c, d;
      for (int i = 0; i < N; ++i) {
        const int kk = i < N - i ? i : N - i;
        double w = 1.0;
        if (kind == 1) w = i == (int)(next_u64() % 3) ? 1.0 : 1e-9;
        if (kind == 2) w = 1.0 / (1.0 + (double)kk * kk * kk * kk);
        if (kind == 3) w = std::exp(-kk * kk / 64.0);
        if (kind == 6) w = std::ldexp(1.0, -(int)(next_u64() % 60));
        if (kind == 7) w = 1e-200;
        if (kind == 8) w = 1e200;
        x[i] = w * uni();
        y[i] = w * uni();
        if (kind == 4) {
          x[i] = 0.7 + trial;
          y[i] = -0.3;
        }
        if (kind == 5) {
          x[i] = std::cos(6.283185307179586 * 3 * i / N + trial);
          y[i] = std::sin(6.283185307179586 * 2 * i / N);
        }
      }
      run_fx<N, RM>(x, y, a, b);
      run_f64<N, RM>(x, y, c, d);
      const auto u = exact<N>(x), v = exact<N>(y);
      long double scale = 0;
      for (int i = 0; i < N; ++i) scale = std::max(scale, std::max(fabsl(u[i]), fabsl(v[i])));
      for (int i = 0; i < N; ++i) {
        auto sq = [&](long double e) { return (e / scale) * (e / scale); };
        efx += sq(a[i] - u[i]) + sq(b[i] - v[i]);
        ef64 += sq(c[i] - u[i]) + sq(d[i] - v[i]);
        norm += sq(u[i]) + sq(v[i]);
      }
    }
    const double rx = (double)sqrtl(efx / norm), rd = (double)sqrtl(ef64 / norm);
    // both end in a rounding to FP64 (about 2^-54 in the 2-norm), which is all
    // that a short line has; FP64 sums of constants and of one point are exact
    // (unrelated magnitudes over 60 binades, which no field or spectrum here has,
    // may lose one bit at n = 1024)
    const double bound = std::fmax(kind == 6 && N == 1024 ? 2.0 * rd : rd, 0x1p-53);
    std::printf("n %4d radix %d %-9s fixed %.2e  fp64 %.2e%s\n", N, RM, names[kind], rx, rd, rx > bound ? "  LARGER" : "");
    if (!(rx <= bound)) ++fails;
  }
  // special values: NaN and infinity spoil the pair, zeros and values below the
  // range give zero, the largest values give infinity or finite values as sums do
  std::vector<double> x(N, 0.0), y(N, 0.0), a, b;
  run_fx<N, RM>(x, y, a, b);
  for (int i = 0; i < N; ++i)
    if (a[i] != 0.0 || b[i] != 0.0) ++fails;
  x[N / 2] = INFINITY;
  run_fx<N, RM>(x, y, a, b);
  for (int i = 0; i < N; ++i)
    if (!std::isnan(a[i]) || !std::isnan(b[i])) ++fails;
  x[N / 2] = 1e-300;
  run_fx<N, RM>(x, y, a, b);
  for (int i = 0; i < N; ++i)
    if (a[i] != 0.0) ++fails;
  x.assign(N, 1.5e308);
  run_fx<N, RM>(x, y, a, b);
  if (!std::isinf(a[0]) || a[0] < 0) ++fails;
  // extremes of the headroom: all points at the largest magnitude, with signs
  // that add up in some output
  for (int k = 0; k < N; ++k) {
    for (int i = 0; i < N; ++i) {
      const double th = 6.283185307179586 * (double)((long long)i * k % N) / N;
      x[i] = std::cos(th) >= 0 ? std::nextafter(1.0, 0.0) : -std::nextafter(1.0, 0.0);
      y[i] = std::sin(th) >= 0 ? std::nextafter(1.0, 0.0) : -std::nextafter(1.0, 0.0);
    }
    if (N > 64 && k % (N / 32)) continue;
    run_fx<N, RM>(x, y, a, b);
    const auto u = exact<N>(x), v = exact<N>(y);
    for (int i = 0; i < N; ++i)
      if (fabsl(a[i] - u[i]) > N * 0x1p-52 || fabsl(b[i] - v[i]) > N * 0x1p-52) ++fails;
  }
}

int main() {
  // conversions: a quantised value is within half a unit, and 53-bit integers
  // come back exactly
  for (int t = 0; t < 200000; ++t) {
    const double v = std::ldexp(uni(), (int)(next_u64() % 40) - 20);
    const int E = (int)((hi(v) >> 20) & 0x7FF) + (int)(next_u64() % 70);
    const fx q = psd::fx_quantise(hi(v), lo(v), E, 56);
    const long double unit = ldexpl(1.0L, E - 1022 - 56);
    if (fabsl((long double)q.v * unit - v) > 0.5L * unit) ++fails;
    const long long w = (long long)next_u64() >> (1 + next_u64() % 62);
    const int e = (int)(next_u64() % 200) - 100;
    const double r = psd::fx_result(w, e);
    const long double want = ldexpl((long double)w, e);
    if (fabsl(r - want) > fabsl(want) * 0x1p-53L) ++fails;
  }
  // p = 4 flux: moduli up to the bound 2^61, within 4 units of |G|^2 G 2^-125
  for (int t = 0; t < 200000; ++t) {
    const int sh = t < 1000 ? 0 : (int)(next_u64() % 40);
    long double g[3], n = 0;
    long long q[3], F[3];
    for (auto& v : g) {
      v = uni();
      n += v * v;
    }
    if (t < 8) g[0] = (t & 1) ? -1 : 1, g[1] = (t & 2) ? 1e-9L : 0, g[2] = (t & 4) ? -1e-9L : 0, n = 1.0000000001L;
    for (int c = 0; c < 3; ++c) q[c] = (long long)(g[c] / sqrtl(n) * ldexpl(1.0L, 61 - sh));
    const unsigned top = psd::fx_flux(q[0], q[1], q[2], F);
    long double m = 0;
    for (int c = 0; c < 3; ++c) m += (long double)q[c] * q[c];
    if (ldexpl((long double)top + 1, 96) < m) ++fails;
    for (int c = 0; c < 3; ++c) {
      const long double want = ldexpl(m * q[c], -125);
      if (fabsl(F[c] - want) > 4.0L || fabsl((long double)F[c]) > 0x1p58L) ++fails;
    }
  }
  check<8, 8>();
  check<8, 4>();
  check<16, 8>();
  check<16, 4>();
  check<32, 8>();
  check<32, 4>();
  check<64, 8>();
  check<64, 4>();
  check<128, 8>();
  check<128, 4>();
  check<256, 8>();
  check<256, 4>();
  check<512, 8>();
  check<1024, 8>();
  std::printf(fails ? "FAILED (%d)\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
