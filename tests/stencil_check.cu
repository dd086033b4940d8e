// Compiled by tests/test_stencil_int.py.  Seeded values -2, -1, 0, +1, +2 of
// narrow and wide ranges of exponents, zeros and special values; prints one
// line a case: the five values and the sums of stencil_int.cuh as bit
// patterns.  With the argument "gpu" also evaluates them on the GPU and compares
// bit for bit.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "stencil_int.cuh"

struct Case {
  double v[5], r[6];
};

__host__ __device__ void evaluate(Case& c) {
  const double* v = c.v;
  c.r[0] = sbli::stencil_first(v[0], v[1], v[3], v[4]);
  c.r[1] = sbli::stencil_second(v[0], v[1], v[2], v[3], v[4]);
  const uint32_t top = sbli::fixed::top_exponent(v[0], v[1], v[3], v[4]);
  double f;
  if (sbli::fixed::alignable(top))
    sbli::both_sums<true>(v[0], v[1], v[3], v[4], top, f, c.r[2]);
  else
    sbli::both_sums<false>(v[0], v[1], v[3], v[4], top, f, c.r[2]);
  c.r[3] = f;
  sbli::stencil_both(v[0], v[1], v[2], v[3], v[4], c.r[4], c.r[5]);
}
__global__ void run(Case* c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) evaluate(c[i]);
}

int main(int argc, char** argv) {
  uint64_t s = 88172645463325252ull;  // xorshift64
  auto rnd = [&]() {
    s ^= s << 13;
    s ^= s >> 7;
    s ^= s << 17;
    return s;
  };
  std::vector<Case> cases;
  const int spreads[6] = {1, 2, 8, 60, 130, 1900};
  for (int it = 0; it < 30000; ++it) {
    Case c;
    const int spread = spreads[it % 6], base = (it % 7) * 40 - 120;
    for (double& v : c.v) {
      const double m = 1.0 + (double)(rnd() >> 12) / 4503599627370496.0;
      v = std::ldexp((rnd() & 1) ? m : -m, base + (int)(rnd() % spread) - spread / 2);
      if (rnd() % 20 == 0) v = (rnd() & 1) ? 0.0 : -0.0;
    }
    if (it % 5 == 0) {  // a smooth field: neighbours that nearly cancel
      const double h = std::ldexp(1.0, -(int)(rnd() % 40));
      for (int k = 0; k < 5; ++k) c.v[k] = c.v[2] * (1.0 + h * (k - 2) + h * h * (k - 2) * (k - 2));
    }
    cases.push_back(c);
  }
  for (double x : {0.0, 1e308, -1e308, (double)INFINITY, (double)NAN, 5e-324, 1e-300})
    for (int k = 0; k < 5; ++k) {
      Case c{{1e-3, 2e-3, 3e-3, 4e-3, 5e-3}, {}};
      c.v[k] = x;
      cases.push_back(c);
      for (double& v : c.v) v = x;
      cases.push_back(c);
    }
  std::vector<Case> host = cases;
  for (Case& c : host) evaluate(c);
  for (const Case& c : host)  // both at once: the bits of each by itself
    for (int k = 0; k < 2; ++k)
      if (!(std::isnan(c.r[k]) && std::isnan(c.r[4 + k])) && memcmp(&c.r[k], &c.r[4 + k], 8)) return 3;
  if (argc > 1 && !strcmp(argv[1], "gpu")) {
    const int n = (int)cases.size();
    Case* d;
    if (cudaMalloc(&d, n * sizeof(Case)) != cudaSuccess) return 2;
    cudaMemcpy(d, cases.data(), n * sizeof(Case), cudaMemcpyHostToDevice);
    run<<<(n + 127) / 128, 128>>>(d, n);
    if (cudaMemcpy(cases.data(), d, n * sizeof(Case), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    int bad = 0;
    for (int i = 0; i < n; ++i)
      for (int k = 0; k < 6; ++k) {
        const double a = cases[i].r[k], b = host[i].r[k];
        if (!(std::isnan(a) && std::isnan(b)) && memcmp(&a, &b, 8)) ++bad;
      }
    std::printf("%d of %d sums differ\n", bad, 6 * n);
    return bad ? 1 : 0;
  }
  for (const Case& c : host) {
    uint64_t b[9];
    memcpy(b, c.v, 40);
    memcpy(b + 5, c.r, 32);
    for (int k = 0; k < 9; ++k) std::printf("%016llx%c", (unsigned long long)b[k], k < 8 ? ' ' : '\n');
  }
  return 0;
}
