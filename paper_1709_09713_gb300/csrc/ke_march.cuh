// ke_march.cuh -- volume sums of kinetic energy rho |u|^2 / 2 and enstrophy
// rho |curl u|^2 / 2 (Eq. 6 derivatives) of a binary64 state, shared by the
// workspace and the allocation-free entry points.
//
// Bound by the binary64 pipe, so every velocity is formed once where that is
// possible: a block marches along x2 over the columns of a 32 x 8 tile, each
// thread keeping its own column's velocities of five planes in registers (the
// x2 derivatives), the centre plane's going through shared memory (x0 and x1
// derivatives; the halo's, 0.625 a point, are formed anew), with the
// reciprocal of the density shared by the three components, and the stencils
// summed in integers.  About 26 binary64 instructions a point where dividing at
// every stencil point took about 260.  Blocks take contiguous runs of planes, two
// blocks per SM, so that all SMs end together and one block's binary64 work runs
// beside the other's integer sums and barriers (one block of 32 x 16: 160 x 200 x 120
// points 285 us instead of 232, 256^3 1113 instead of 926, 32^3 21 instead of 15; three or
// four blocks of fewer registers 238, 236).  160 x 200 x 120 points, both entry points
// with the state in and out, against dividing at every stencil point: 4.15 ->
// 0.54 ms.
#pragma once

#include <algorithm>

#include "fpconv.cuh"
#include "sbli_internal.cuh"
#include "stencil_int.cuh"

namespace sbli {

constexpr int KE_TX = 32, KE_TY = 8;
constexpr int KE_THREADS = KE_TX * KE_TY;
constexpr int KE_PER_SM = 2;  // blocks

inline long long ke_units(const Geom& g) {
  return (long long)((g.n0 + KE_TX - 1) / KE_TX) * ((g.n1 + KE_TY - 1) / KE_TY) * g.n2;
}
// blocks of a launch (and partial sums it writes): KE_PER_SM per SM, at most `most`
inline int ke_blocks(const Geom& g, int most) {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long units = ke_units(g);
  const int b = std::min(KE_PER_SM * sms, most);
  return (int)(units < b ? units : b);
}

// PLAIN: q holds the plain conserved variables, else deviations (rho - 1).
// Partial sums of block b in partials[2b], partials[2b + 1]: each thread's
// points in a fixed order, warps by shuffles, then the warps in order.
template <bool PLAIN>
__global__ void __launch_bounds__(KE_THREADS, KE_PER_SM)
    ke_march_kernel(Geom g, const __grid_constant__ Coef<double> c, const double* __restrict__ q,
                    double* __restrict__ partials) {
  __shared__ double su[2][3][KE_TY + 4][KE_TX + 4];
  __shared__ double red[2][KE_THREADS / 32];
  const long long P = g.P, plane = (long long)g.n0 * g.n1;
  const int n0 = g.n0, n1 = g.n1, n2 = g.n2;
  const int tid = threadIdx.x, tx = tid % KE_TX, ty = tid / KE_TX;
  const int tiles_x = (n0 + KE_TX - 1) / KE_TX, tiles_y = (n1 + KE_TY - 1) / KE_TY;
  const long long units = (long long)tiles_x * tiles_y * n2;
  // this thread's halo point of the centre plane: two columns on each side of
  // the tile's rows (u1, u2 read there), two rows above and below (u0, u2)
  int hx = 0, hy = 0, hc = -1;
  if (tid < 4 * KE_TY) {
    const int k = tid & 3;
    hx = k < 2 ? k : KE_TX + k;
    hy = (tid >> 2) + 2;
    hc = 1;
  } else if (tid < 4 * (KE_TX + KE_TY)) {
    const int h = tid - 4 * KE_TY, k = h / KE_TX;
    hx = h % KE_TX + 2;
    hy = k < 2 ? k : KE_TY + k;
    hc = 0;
  }
  auto recip_rho = [](double r) { return rcp_newton_f64(PLAIN ? r : 1.0 + r); };
  double ke = 0.0, en = 0.0;
  int buf = 0;
  long long u = units * blockIdx.x / gridDim.x;
  const long long end = units * (blockIdx.x + 1) / gridDim.x;
  while (u < end) {
    const int tile = (int)(u / n2), zbeg = (int)(u - (long long)tile * n2);
    const int zend = (int)min((long long)n2, zbeg + (end - u));
    u += zend - zbeg;
    const int x0 = (tile % tiles_x) * KE_TX, y0 = (tile / tiles_x) * KE_TY;
    const bool valid = x0 + tx < n0 && y0 + ty < n1;
    const double* own = q + wrapi(x0 + tx, n0) + (long long)n0 * wrapi(y0 + ty, n1);
    const double* halo = q + wrapi(x0 + hx - 2, n0) + (long long)n0 * wrapi(y0 + hy - 2, n1);
    // own column: u0, u1 of planes z-2 .. z+2, u2 and rho of z .. z+2
    double a0[5], a1[5], a2[3], rr[3];
    double pr, p0, p1, p2, hr = 1.0, hm = 0.0, h2 = 0.0;  // loads in flight
    auto load_own = [&](int z) {
      const double* s = own + plane * wrapi(z, n2);
      pr = s[0];
      p0 = s[P];
      p1 = s[2 * P];
      p2 = s[3 * P];
    };
    auto load_halo = [&](int z) {
      if (hc >= 0) {
        const double* s = halo + plane * z;
        hr = s[0];
        hm = s[(1 + hc) * P];
        h2 = s[3 * P];
      }
    };
    auto push = [&]() {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        a0[k] = a0[k + 1];
        a1[k] = a1[k + 1];
      }
      a2[0] = a2[1];
      a2[1] = a2[2];
      rr[0] = rr[1];
      rr[1] = rr[2];
      const double i = recip_rho(pr);
      a0[4] = p0 * i;
      a1[4] = p1 * i;
      a2[2] = p2 * i;
      rr[2] = PLAIN ? pr : 1.0 + pr;
    };
    load_own(zbeg - 2);
#pragma unroll
    for (int k = -1; k <= 2; ++k) {
      push();
      load_own(zbeg + k);
    }
    load_halo(zbeg);
    for (int z = zbeg; z < zend; ++z) {
      push();  // plane z + 2: the centre is a0[2], a1[2], a2[0], rr[0]
      su[buf][0][ty + 2][tx + 2] = a0[2];
      su[buf][1][ty + 2][tx + 2] = a1[2];
      su[buf][2][ty + 2][tx + 2] = a2[0];
      if (hc >= 0) {
        const double i = recip_rho(hr);
        su[buf][hc][hy][hx] = hm * i;
        su[buf][2][hy][hx] = h2 * i;
      }
      if (z + 1 < zend) {
        load_own(z + 3);
        load_halo(z + 1);
      }
      __syncthreads();  // the buffer of plane z is written again two planes on, after the next barrier
      const double(*s0)[KE_TX + 4] = su[buf][0] + ty + 2;
      const double(*s1)[KE_TX + 4] = su[buf][1] + ty + 2;
      const double(*s2)[KE_TX + 4] = su[buf][2] + ty + 2;
      const int i = tx + 2;
      // Eq. 6 derivatives, their sums in integers
      const double cx = c.c2[0], cy = c.c2[1], cz = c.c2[2];
      const double w0 = cy * stencil_first(s2[-2][i], s2[-1][i], s2[1][i], s2[2][i]) - cz * stencil_first(a1[0], a1[1], a1[3], a1[4]);
      const double w1 = cz * stencil_first(a0[0], a0[1], a0[3], a0[4]) -
                        cx * stencil_first(s2[0][i - 2], s2[0][i - 1], s2[0][i + 1], s2[0][i + 2]);
      const double w2 = cx * stencil_first(s1[0][i - 2], s1[0][i - 1], s1[0][i + 1], s1[0][i + 2]) -
                        cy * stencil_first(s0[-2][i], s0[-1][i], s0[1][i], s0[2][i]);
      if (valid) {
        const double hrho = 0.5 * rr[0];
        ke += hrho * (a0[2] * a0[2] + a1[2] * a1[2] + a2[0] * a2[0]);
        en += hrho * (w0 * w0 + w1 * w1 + w2 * w2);
      }
      buf ^= 1;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    ke += __shfl_down_sync(0xffffffffu, ke, o);
    en += __shfl_down_sync(0xffffffffu, en, o);
  }
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = ke;
    red[1][tid >> 5] = en;
  }
  __syncthreads();
  if (tid == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < KE_THREADS / 32; ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    partials[2 * blockIdx.x] = a;
    partials[2 * blockIdx.x + 1] = b;
  }
}

}  // namespace sbli
