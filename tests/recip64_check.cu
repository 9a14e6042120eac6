// Device check of psd::recip_pos, the FP64 reciprocal of the symbol divisions and
// of the line search, against the IEEE quotient: every binade of the positive
// doubles (subnormals too) with random mantissas and the mantissas at its edges,
// and 0, infinity and NaN.  Built and run by tests/test_recip64.py on a GPU.
// Exit status 0 = every result within 1 ulp, special values equal.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../paper_1607_01475_gb300/csrc/psd_common.cuh"

__global__ void k_recip64(const double* x, double* out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = psd::recip_pos(x[i]);
}

static uint64_t rng_state = 0x5eed64ULL;
static uint64_t next_u64() {  // SplitMix64
  uint64_t z = (rng_state += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
static int64_t bits(double v) {
  int64_t b;
  std::memcpy(&b, &v, 8);
  return b;
}

int main() {
  std::vector<double> x;
  auto add = [&](uint64_t b) {
    double v;
    std::memcpy(&v, &b, 8);
    x.push_back(v);
  };
  const uint64_t M = (1ULL << 52) - 1;
  for (uint64_t e = 0; e < 2047; ++e) {
    for (uint64_t m : {uint64_t(0), uint64_t(1), M, M - 1, M / 2, M / 2 + 1}) add(e << 52 | m);
    for (int t = 0; t < 512; ++t) add(e << 52 | (next_u64() & M));
  }
  for (int k = 0; k < 52; ++k) add(1ULL << k);  // subnormal binades
  add(2047ULL << 52);                           // infinity
  add(2047ULL << 52 | 1ULL << 51);              // NaN
  const int n = (int)x.size();
  double *dx = nullptr, *da = nullptr;
  if (cudaMalloc(&dx, n * sizeof(double)) != cudaSuccess || cudaMalloc(&da, n * sizeof(double)) != cudaSuccess) {
    std::printf("cudaMalloc failed\n");
    return 2;
  }
  cudaMemcpy(dx, x.data(), n * sizeof(double), cudaMemcpyHostToDevice);
  k_recip64<<<152 * 4, 256>>>(dx, da, n);
  std::vector<double> a(n);
  const cudaError_t err = cudaMemcpy(a.data(), da, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (err != cudaSuccess) {
    std::printf("CUDA error: %s\n", cudaGetErrorString(err));
    return 2;
  }
  long long worst = 0, bad = 0, exact = 0;
  for (int i = 0; i < n; ++i) {
    const double want = 1.0 / x[i];
    if (std::isnan(want)) {
      bad += !std::isnan(a[i]);
      continue;
    }
    // of non-negative doubles: the distance of the bit patterns is that in ulps
    const long long d = std::llabs(bits(a[i]) - bits(want));
    if (d > 1 && bad++ < 5) std::printf("x %.17g got %.17g want %.17g\n", x[i], a[i], want);
    if (d > worst) worst = d;
    exact += d == 0;
  }
  std::printf("n %d worst %lld ulp, %.6f exactly rounded, %lld beyond 1 ulp\n", n, worst, (double)exact / n, bad);
  cudaFree(dx);
  cudaFree(da);
  if (bad == 0) std::printf("OK\n");
  return bad == 0 ? 0 : 1;
}
