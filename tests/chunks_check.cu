// Compiled by tests/test_chunks.py (host code): sbli::fewer_chunks visits, from 4
// up to n2, just the smallest planes per CTA of each number of CTAs.
#include <cstdio>

#include "sbli_internal.cuh"

int main() {
  int bad = 0;
  for (int n2 = 5; n2 <= 3000; ++n2) {
    auto chunks = [&](int zc) { return (n2 + zc - 1) / zc; };
    int next = 4;
    for (int zc = 4; zc <= n2; ++zc) {
      const bool first = zc == 4 || chunks(zc) < chunks(zc - 1);
      if (first != (zc == next)) ++bad;
      if (zc == next) next = sbli::fewer_chunks(n2, zc);
    }
    if (next <= n2) ++bad;
  }
  int steps = 0;
  for (int zc = 4; zc <= 1 << 24; zc = sbli::fewer_chunks(1 << 24, zc)) ++steps;
  std::printf("%d wrong, %d values for 2^24 planes\n", bad, steps);
  return bad || steps > 8192;
}
