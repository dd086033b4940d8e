// Compiled by tests/test_stencil_int.py.  Seeded values -2, -1, 0, +1, +2 of
// narrow and wide ranges of exponents, zeros and special values; prints one
// line a case: the five values and the sums of stencil_int.cuh as bit
// patterns; with the argument "eight" eight values and the first derivative of
// their sums in pairs.  With "gpu" evaluates both on the GPU too and compares bit
// for bit.
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
struct Eight {
  double x[4], y[4], r;
};
__host__ __device__ void evaluate(Eight& c) {
  uint32_t top = sbli::fixed::top_exponent(c.x[0], c.x[1], c.x[2], c.x[3]);
  const uint32_t ty = sbli::fixed::top_exponent(c.y[0], c.y[1], c.y[2], c.y[3]);
  top = ty > top ? ty : top;
  c.r = sbli::fixed::alignable(top) ? sbli::first_sum<true>(c.x, c.y, top) : sbli::first_sum<false>(c.x, c.y, top);
}
template <typename C>
__global__ void run(C* c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) evaluate(c[i]);
}
template <typename C>
bool on_gpu(std::vector<C>& cases) {
  const int n = (int)cases.size();
  C* d;
  if (cudaMalloc(&d, n * sizeof(C)) != cudaSuccess) return false;
  cudaMemcpy(d, cases.data(), n * sizeof(C), cudaMemcpyHostToDevice);
  run<<<(n + 127) / 128, 128>>>(d, n);
  const bool ok = cudaMemcpy(cases.data(), d, n * sizeof(C), cudaMemcpyDeviceToHost) == cudaSuccess;
  cudaFree(d);
  return ok;
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
  // the most that the sums hold: mantissas of ones at one exponent, every combination of signs
  const double ones = 2.0 - std::ldexp(1.0, -52);
  for (int e : {-900, 0, 900})
    for (int signs = 0; signs < 32; ++signs) {
      Case c;
      for (int k = 0; k < 5; ++k) c.v[k] = std::ldexp(signs >> k & 1 ? -ones : ones, e);
      cases.push_back(c);
    }
  // eight values: two neighbouring cases' four
  std::vector<Eight> eights;
  for (size_t i = 1; i < cases.size(); ++i) {
    const double *v = cases[i - 1].v, *w = cases[i].v;
    eights.push_back({{v[0], v[1], v[3], v[4]}, {w[0], w[1], w[3], w[4]}, 0});
  }
  for (int signs = 0; signs < 256; ++signs) {
    Eight c;
    for (int k = 0; k < 8; ++k) (k < 4 ? c.x : c.y)[k & 3] = signs >> k & 1 ? -ones : ones;
    eights.push_back(c);
  }
  std::vector<Eight> eights_host = eights;
  for (Eight& c : eights_host) evaluate(c);
  std::vector<Case> host = cases;
  for (Case& c : host) evaluate(c);
  for (const Case& c : host)  // both at once: the bits of each by itself
    for (int k = 0; k < 2; ++k)
      if (!(std::isnan(c.r[k]) && std::isnan(c.r[4 + k])) && memcmp(&c.r[k], &c.r[4 + k], 8)) return 3;
  if (argc > 1 && !strcmp(argv[1], "gpu")) {
    const int n = (int)cases.size();
    if (!on_gpu(cases) || !on_gpu(eights)) return 2;
    int bad = 0;
    for (int i = 0; i < n; ++i)
      for (int k = 0; k < 6; ++k) {
        const double a = cases[i].r[k], b = host[i].r[k];
        if (!(std::isnan(a) && std::isnan(b)) && memcmp(&a, &b, 8)) ++bad;
      }
    for (size_t i = 0; i < eights.size(); ++i) {
      const double a = eights[i].r, b = eights_host[i].r;
      if (!(std::isnan(a) && std::isnan(b)) && memcmp(&a, &b, 8)) ++bad;
    }
    std::printf("%d of %d sums differ\n", bad, 6 * n + (int)eights.size());
    return bad ? 1 : 0;
  }
  if (argc > 1 && !strcmp(argv[1], "eight")) {
    for (const Eight& c : eights_host) {
      uint64_t b[9];
      memcpy(b, &c, 72);
      for (int k = 0; k < 9; ++k) std::printf("%016llx%c", (unsigned long long)b[k], k < 8 ? ' ' : '\n');
    }
    return 0;
  }
  for (const Case& c : host) {
    uint64_t b[9];
    memcpy(b, c.v, 40);
    memcpy(b + 5, c.r, 32);
    for (int k = 0; k < 9; ++k) std::printf("%016llx%c", (unsigned long long)b[k], k < 8 ? ' ' : '\n');
  }
  return 0;
}
