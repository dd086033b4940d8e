// batch_kernel.cuh -- the multi-member stage launch shared by ensembles
// (batch.cu) and the serving loop (server.cu).
#pragma once

#include "sbli_internal.cuh"

namespace sbli {

constexpr int BATCH_MAX_MEMBERS = 64;  // members per launch (parameter space bound)

template <typename T>
struct BatchParams {
  int count;                                  // members in this launch
  // binary32 members: work items (z chunk x tile); binary64-register members:
  // planes of tiles, split evenly over the CTAs
  long long total_items;                      // sum of the members' items
  long long item_begin[BATCH_MAX_MEMBERS + 1];
  int tiles_x[BATCH_MAX_MEMBERS];
  int tiles_y[BATCH_MAX_MEMBERS];
  StageArgs a[BATCH_MAX_MEMBERS];             // geometry, zc, stage pointers, a_k dt, b_k dt
  Coef<T> c[BATCH_MAX_MEMBERS];
  double* ke_items;                           // (ke, ens) partials per item (even split: CTA + member), or nullptr
};

// One persistent launch of stage work for p.count members (grid = CTAs).
// in64: the members' stage inputs are binary64 (binary64-register kernels;
// binary32 stages always read binary32 fields, so it must be false for them);
// df: binary32 stages with the double-float accumulator (dacc pointers);
// zq: x2-neighbour records from a per-thread TMEM queue (1) or the
// shared-memory ring (0), as for single grids (bitwise the same results).
template <typename T>
cudaError_t launch_batch_t(const BatchParams<T>& p, bool in64, int grid, cudaStream_t s, bool df, int zq);

// The z-queue mode a batch of this precision starts with: binary32 members
// (either accumulator) the TMEM queue, the faster one on single grids; binary64 and
// double-float arithmetic the shared-memory ring, the faster one of marches below 24
// planes a CTA (single grids of longer ones take the TMEM queue, see default_config;
// the batch tuner times both).
inline int batch_default_zq(int precision) { return precision == SBLI_FP32 || precision == SBLI_FP32_DF ? 1 : 0; }

// Resident CTAs per SM of the multi-member launch: binary32 members run the
// TMEM-queue kernel (59 KiB shared, four warps of at most 168 registers: 3 per SM) or the shared
// ring (113 KiB: 2 per SM); binary64 and double-float-arithmetic members
// 16 x 8 tiles of the 107 KiB shared ring or the 69 KiB TMEM-queue kernel, whose
// registers fit twice.
inline int batch_ctas_per_sm(int precision, int zq) {
  if (precision == SBLI_FP32 || precision == SBLI_FP32_DF) return zq ? 3 : 2;
  return F64_CTAS_PER_SM;
}

// CTAs of a launch: persistent ones that fill the SMs.  The even split keeps
// a partial sum per CTA and member, which bounds them.
constexpr int BATCH_MAX_EVEN_CTAS = 512;
inline int batch_grid_ctas(int sms, int precision, int zq) {
  const int ctas = sms * batch_ctas_per_sm(precision, zq);
  const bool even = precision == SBLI_FP64 || precision == SBLI_DF64;
  return even && ctas > BATCH_MAX_EVEN_CTAS ? BATCH_MAX_EVEN_CTAS : ctas;
}

// Work items (z chunk of zc planes x 32 x 8 tile) of one member; batch_zc is
// the planes per item a member starts with.
inline int batch_zc(int n2) { return n2 < 32 ? n2 : 32; }
inline long long member_items(const int n[3], int zc) {
  return (long long)((n[0] + 31) / 32) * ((n[1] + 7) / 8) * ((n[2] + zc - 1) / zc);
}
// Planes of all 16 x 8 tiles of one member: the units of the even split.
inline long long member_planes(const int n[3]) {
  return (long long)((n[0] + F64_TILE_X - 1) / F64_TILE_X) * ((n[1] + 7) / 8) * n[2];
}

// Binary32 members under the default schedule: the cap on the planes per item
// (32, 16, 8 or 4; a member's own are batch_zc) that the model of a stage
// (binary32_stage_us) ranks best, so that a few small members fill the GPU too.
// edges(m) is member m's (n0, n1, n2).  Two 64^3 members are 64 items of 32
// planes, one for every other of 152 SMs with room for three each, but 256 of 8.
template <typename F>
int batch_zc_cap(int count, const F& edges, int zq, int sms) {
  int best = 32;
  double cost = 0.0;
  for (int cap = 32; cap >= 4; cap /= 2) {
    long long items = 0;
    for (int m = 0; m < count; ++m) {
      const int* n = edges(m);
      const int zc = batch_zc(n[2]);
      items += member_items(n, zc < cap ? zc : cap);
    }
    const double us = binary32_stage_us(items, cap, zq, sms);
    if (cap == 32 || us < cost) {
      cost = us;
      best = cap;
    }
  }
  return best;
}

// Per member m: fixed-order sum of partials [range[2m], range[2m+1]) times inv_p[m].
cudaError_t launch_batch_ke_finalize(const double* items, const long long* range, const double* inv_p, double* out,
                                     int count, cudaStream_t s);

}  // namespace sbli
