// Host check of the block fixed-point line FFT on lines whose points are neither
// all large nor few: one point over a dense background of 1/2 .. 1/512 of it, two
// such points, normal and slowly decaying lines.  On each, its error (2-norm,
// relative, against long double) must not exceed that of the same passes in FP64.
// The passes are those of fx_line_check.cu.  Built and run by
// tests/test_fx_peak.py (no GPU needed).  Exit status 0 = pass.
#define main fx_line_check_main
#include "fx_line_check.cu"
#undef main

template <int N, int RM>
void peaks() {
  for (int kind = 0; kind < 15; ++kind) {
    long double efx = 0, ef64 = 0, norm = 0;
    for (int trial = 0; trial < (N <= 64 ? 60 : 12); ++trial) {
      std::vector<double> x(N), y(N), a, b, c, d;
      const int at = (int)(next_u64() % N), at2 = (int)(next_u64() % N);
      for (int i = 0; i < N; ++i) {
        const int kk = i < N - i ? i : N - i;
        auto value = [&]() -> double {
          if (kind < 9) return (i == at ? 1.0 + 0.9 * std::fabs(uni()) : std::ldexp(uni(), -(kind + 1)));
          if (kind == 9) return i == at || i == at2 ? 1.5 : uni() / 16;
          if (kind == 10) return uni() + uni() + uni() + uni() + uni() + uni();  // nearly normal
          if (kind == 11) return uni() / (1.0 + kk);
          if (kind == 12) return uni() / std::sqrt(1.0 + kk);
          if (kind == 13) return i == at ? 1.0 : std::ldexp(uni(), -(int)(next_u64() % 12));
          return kk < 4 ? uni() : uni() / 32;
        };
        x[i] = value();
        y[i] = kind % 2 ? value() : value() / 8;
      }
      run_fx<N, RM>(x, y, a, b);
      run_f64<N, RM>(x, y, c, d);
      const auto u = exact<N>(x), v = exact<N>(y);
      for (int i = 0; i < N; ++i) {
        efx += (a[i] - u[i]) * (a[i] - u[i]) + (b[i] - v[i]) * (b[i] - v[i]);
        ef64 += (c[i] - u[i]) * (c[i] - u[i]) + (d[i] - v[i]) * (d[i] - v[i]);
        norm += u[i] * u[i] + v[i] * v[i];
      }
    }
    const double rx = (double)sqrtl(efx / norm), rd = (double)sqrtl(ef64 / norm);
    std::printf("n %4d radix %d kind %2d fixed %.2e  fp64 %.2e%s\n", N, RM, kind, rx, rd, rx > rd ? "  LARGER" : "");
    if (!(rx <= rd)) ++fails;
  }
}

// The bound behind the scale: it is not below the squared 2-norm, and with the
// chosen B every modulus stays within 2^61.
template <int N, int RM>
void headroom() {
  using Plan = psd::FxPlan<N, RM>;
  for (int trial = 0; trial < 2000; ++trial) {
    const double decay = std::ldexp(1.0, -(int)(next_u64() % 12));
    std::vector<double> v(2 * N);
    unsigned top = 0, l2 = 0;
    for (auto& x : v) x = next_u64() % 8 ? decay * uni() : (next_u64() % 2 ? -1.0 : 1.0) * (2.0 - 0x1p-20);
    for (double x : v) top = std::max(top, hi(x) & 0x7FFFFFFFu);
    const int E = (int)(top >> 20);
    long double s = 0;
    for (double x : v) {
      l2 += psd::fx_square(hi(x), E);
      s += (long double)x * x;
    }
    const long double unit = ldexpl(1.0L, 2 * (E - 1022));
    if (ldexpl((long double)l2, -20) * unit < s) ++fails;
    const int B = psd::fx_scale<Plan>(l2);
    if (B < Plan::B || B > 60) ++fails;
    if (B > Plan::B && Plan::R * (s / unit) * ldexpl(1.0L, 2 * B) > 0x1p122L) ++fails;
  }
}

template <int N, int RM>
void both() {
  peaks<N, RM>();
  headroom<N, RM>();
}

int main() {
  both<8, 8>();
  both<8, 4>();
  both<16, 8>();
  both<16, 4>();
  both<32, 8>();
  both<32, 4>();
  both<64, 8>();
  both<64, 4>();
  both<128, 8>();
  both<128, 4>();
  both<256, 8>();
  both<256, 4>();
  both<512, 8>();
  both<1024, 8>();
  std::printf(fails ? "FAILED (%d)\n" : "OK\n", fails);
  return fails ? 1 : 0;
}
