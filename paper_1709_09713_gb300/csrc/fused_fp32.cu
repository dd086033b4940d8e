// fused_fp32.cu -- binary32 instantiations of the fused stage kernel.  Every
// stage reads binary32 fields (stage 0 the binary32 copy of the state that the
// previous step's last stage wrote); the accumulator is binary64 or, for the
// double-float mode, a hi/lo binary32 pair.  The residual alone (RHS only)
// may also read the binary64 state.  Tiles 32 x 8 (two CTAs per SM) and 32 x 16 (one
// CTA of 16 warps per SM); the TMEM-queue and two-column kernels are in
// their own files.
#include <algorithm>

#include "fused_stage.cuh"

namespace sbli {

template <int TY>
static cudaError_t dispatch32(const StageArgs& a, const Coef<float>& c, bool in_fp64, bool rhs_only,
                              cudaStream_t s) {
  if (rhs_only) {
    if (in_fp64) return launch_fused_t<float, double, float, TY, true, false>(a, c, s);
    return launch_fused_t<float, float, float, TY, true, false>(a, c, s);
  }
  if (in_fp64) return cudaErrorInvalidValue;  // stages read the binary32 copy of the state
  if (a.ke_partials) return launch_fused_t<float, float, float, TY, false, true>(a, c, s);
  return launch_fused_t<float, float, float, TY, false, false>(a, c, s);
}

cudaError_t launch_fused_fp32(const StageArgs& a, const Coef<float>& c, const FusedConfig& cfg, bool in_fp64,
                              bool rhs_only, cudaStream_t s) {
  if (cfg.px == 2) return launch_fused_fp32_pair(a, c, cfg, in_fp64, false, rhs_only, s);
  if (cfg.zq) return launch_fused_fp32_tmem(a, c, cfg, in_fp64, false, rhs_only, s);
  switch (cfg.ty) {
    case 8: return dispatch32<8>(a, c, in_fp64, rhs_only, s);
    case 16: return dispatch32<16>(a, c, in_fp64, rhs_only, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int TY>
static cudaError_t dispatch32df(const StageArgs& a, const Coef<float>& c, bool rhs_only, cudaStream_t s) {
  if (rhs_only) return launch_fused_t<float, float, float, TY, true, false, false>(a, c, s);
  if (a.ke_partials) return launch_fused_t<float, float, float, TY, false, true, true>(a, c, s);
  return launch_fused_t<float, float, float, TY, false, false, true>(a, c, s);
}

cudaError_t launch_fused_fp32df(const StageArgs& a, const Coef<float>& c, const FusedConfig& cfg, bool rhs_only,
                                cudaStream_t s) {
  if (cfg.px == 2) return launch_fused_fp32_pair(a, c, cfg, false, true, rhs_only, s);
  if (cfg.zq) return launch_fused_fp32_tmem(a, c, cfg, false, true, rhs_only, s);
  switch (cfg.ty) {
    case 8: return dispatch32df<8>(a, c, rhs_only, s);
    case 16: return dispatch32df<16>(a, c, rhs_only, s);
    default: return cudaErrorInvalidValue;
  }
}

int fused_num_ctas(const Geom& g, const FusedConfig& cfg) {
  const long long w = TX * (cfg.px == 2 ? 2 : 1);
  const long long gx = (g.n0 + w - 1) / w, gy = (g.n1 + cfg.ty - 1) / cfg.ty, gz = (g.n2 + cfg.zc - 1) / cfg.zc;
  return (int)(gx * gy * gz);
}

// Measured at 16^3 ... 160^3 (binary64 accumulator; the double-float one ranks
// alike): a plane of the shared ring takes 1.47 us with one CTA on an SM, 2.5 with
// two; one of the TMEM queue 1.69, 2.3 and with three 3.05, and 0.6 us for its
// allocation; the fill of a march 1.5 planes, a launch 1 us; CTAs go to SMs one each first.  Within 8 % of
// the measured time over both queues and 1 to 40 planes per CTA.
double binary32_stage_us(long long ctas, int zc, int zq, int sms) {
  const double plane[2][4] = {{0.0, 1.47, 2.5, 2.5}, {0.0, 1.69, 2.3, 3.05}};
  const int most = zq ? 3 : 2;
  const long long slots = (long long)sms * most;
  const long long full = ctas / slots, rest = ctas % slots;
  const int last = (int)((rest + sms - 1) / sms);
  return (zq ? 1.6 : 1.0) + (zc + 1.5) * ((double)full * plane[zq][most] + plane[zq][last]);
}

int binary32_launch_zc(const Geom& g, const FusedConfig& cfg, int sms) {
  if (cfg.zc != 4 || cfg.ty != 8 || cfg.px != 1) return cfg.zc;
  FusedConfig c = cfg;
  int best = 4;
  double cost = binary32_stage_us(fused_num_ctas(g, cfg), 4, cfg.zq, sms);
  for (c.zc = 3; c.zc >= 1; --c.zc) {
    const int ctas = fused_num_ctas(g, c);
    const double us = binary32_stage_us(ctas, c.zc, cfg.zq, sms);
    if (ctas <= MAX_SMALL_CTAS && us < cost) {
      cost = us;
      best = c.zc;
    }
  }
  return best;
}

// The longest CTA decides, in planes, each march's fill counting F64_FILL, and a
// plane of the even split 4 to 8 % more (its CTAs share no halos in L2; 8 % for
// double-float with the TMEM queue).  The even split against chunks, us a
// stage: double-float 32^3 10.0 against 16.9, shared ring 129x97x66 128 against 132, 128^3
// 259 against 264, but with the TMEM queue 128 against 126 and 255 against 249, and 96^3
// 117 against 114; binary64 32^3 27.9 against 46.2, 128^3 760 against 795, 256^3 5887 against 5959.
// Over 21 grids (shared ring) the rule loses 0.2 % on average to the better of the two.
//
// Two counts of even runs are ranked: as many as there are slots, and the most
// that cut every tile into equally many, so that no run crosses into a second
// tile and fills twice: on 304 slots 48^3 takes 288 runs of 3 planes (binary64 56.0 us
// a stage, double-float 19.7; 304 runs of up to 3 over two tiles 67.3 and 22.9), 40^3
// 300 of 2 (42.1 and 14.9; 49.7 and 17.9).
Split plan_split(const Geom& g, const FusedConfig& cfg, int slots, bool double_float) {
  const int zc = cfg.zc;
  const double plane = !double_float ? 1.04 : cfg.zq ? 1.08 : 1.05;
  const long long tiles = (long long)((g.n0 + F64_TILE_X - 1) / F64_TILE_X) * ((g.n1 + 7) / 8), units = tiles * g.n2;
  const long long chunks = tiles * ((g.n2 + zc - 1) / zc);
  const double waves = (double)((chunks + slots - 1) / slots);
  double best = waves * (std::min(zc, g.n2) + F64_FILL);
  Split split{(int)chunks, 0};
  const auto even = [&](long long ctas) {
    double longest = 0.0;
    for (long long c = 0; c < ctas; ++c) {
      const long long u = units * c / ctas, end = units * (c + 1) / ctas;
      const long long marches = (end - 1) / g.n2 - u / g.n2 + 1;
      longest = std::max(longest, plane * (double)(end - u) + F64_FILL * marches);
    }
    if (longest <= best) {
      best = longest;
      split = Split{(int)ctas, 1};
    }
  };
  even(std::min<long long>(units, slots));
  if (tiles <= slots) even(tiles * std::min<long long>(g.n2, slots / tiles));
  return split;
}

}  // namespace sbli
