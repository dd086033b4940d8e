// Compiled by tests/test_gpu_pairs.py: sbli::split_f64 over seeded values of
// every exponent from below the binary32 range to above it, ties, values
// whose high part carries into the next exponent, and the special values.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "fpconv.cuh"

__global__ void split(const double* v, long long n, float2* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) sbli::split_f64(v[i], out[i].x, out[i].y);
}

int main() {
  std::vector<double> h;
  uint64_t s = 88172645463325252ull;  // xorshift64
  auto rnd = [&]() {
    s ^= s << 13;
    s ^= s >> 7;
    s ^= s << 17;
    return s;
  };
  for (int e = -1080; e <= 1023; ++e)
    for (int k = 0; k < 200; ++k) {
      const double m = 1.0 + (double)(rnd() >> 12) / 4503599627370496.0;
      h.push_back(std::ldexp((rnd() & 1) ? m : -m, e));
    }
  for (int e = -60; e <= 60; ++e)
    for (uint64_t low : {0ull, 1ull, 0x0FFFFFFFull, 0x10000000ull, 0x10000001ull, 0x1FFFFFFFull})
      for (uint64_t top : {0ull, 1ull, 0x7FFFFFull}) {
        const uint64_t b = ((uint64_t)(1023 + e) << 52) | (top << 29) | low;
        double v;
        memcpy(&v, &b, 8);
        h.push_back(v);
        h.push_back(-v);
      }
  const double inf = INFINITY;
  for (double v : {0.0, -0.0, inf, -inf, (double)NAN, 1e300, -1e300}) h.push_back(v);
  const long long n = (long long)h.size();
  double* dv;
  float2* dr;
  if (cudaMalloc(&dv, n * 8) != cudaSuccess || cudaMalloc(&dr, n * 8) != cudaSuccess) return 2;
  cudaMemcpy(dv, h.data(), n * 8, cudaMemcpyHostToDevice);
  split<<<(unsigned)((n + 255) / 256), 256>>>(dv, n, dr);
  std::vector<float2> r(n);
  if (cudaMemcpy(r.data(), dr, n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  long long bad = 0;
  for (long long i = 0; i < n; ++i) {
    const double v = h[i], a = std::fabs(v), hi = r[i].x, lo = r[i].y;
    bool ok;
    if (std::isnan(v))
      ok = std::isnan(hi);
    else if (a >= std::ldexp(1.0, 128))
      ok = std::isinf(hi) && (hi > 0) == (v > 0);
    else if (a < std::ldexp(1.0, -126))
      ok = hi == 0 && lo == 0;
    else if (std::fabs(hi) > 3.4028235677973366e38)  // rounds up to 2^128
      ok = std::isinf(hi) && a > 3.40282346638528859e38;
    else  // hi: half a unit of 24 bits, hi + lo: half a unit of 24 more, or a lo below the binary32 normal range
      ok = std::fabs(v - hi) <= std::ldexp(a, -24) &&
           std::fabs(v - hi - lo) <= std::fmax(std::ldexp(a, -48), std::ldexp(1.0, -126));
    if (!ok && bad++ < 5) std::printf("split(%.17g) = %.9g + %.9g\n", v, hi, lo);
  }
  std::printf("%lld of %lld values wrong\n", bad, n);
  return bad ? 1 : 0;
}
