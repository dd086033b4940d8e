// fused_stage.cuh -- fused residual + low-storage RK stage kernel (sm_103a).
//
// One kernel evaluates R(Q) of Eqs. 1-3 (arXiv:1709.09713, §2) with every
// derivative of Eqs. 6-7 computed on the fly (no derivative arrays: the
// "store none" class of §2.5, ordered by velocity component as in SN2) and
// writes the Runge-Kutta stage of §2.2 / Fig. 1 in the same pass.
//
// Work decomposition (2.5D streaming):
//   * a CTA owns a tile of (x0, x1) columns and marches along x2 over a run of
//     planes: 32 x TY columns, a warp a row of them, in binary32 (one thread per
//     column, or two rows or two columns a thread, see below), 16 x 8, two rows a
//     warp, in binary64 and double-float (tile_x); every global access is a
//     coalesced row segment;
//   * a ring of 5 shared-memory slots holds the primitives of planes
//     z-2..z+2 on the tile plus a 2-point halo in x0 and x1 (corners
//     included), one 10-value record per point (array of structures, read
//     with 8- or 16-byte vector loads at bank-conflict-free strides).  A
//     plane's primitives are computed once, when it enters the ring, from the
//     conserved variables loaded from HBM (periodic wrap in the index
//     arithmetic replaces the boundary pass of Fig. 1);
//   * the loads of the next entering plane are issued as soon as the current
//     plane is stored, and the centre plane's accumulator values as its
//     derivative terms start, so HBM latency overlaps the arithmetic;
//   * x0/x1 derivatives read the centre slot, x2 derivatives read the ring;
//     each axis takes its four neighbour records (binary32 one at a time,
//     axis_terms_stream; binary64 sums its linear stencils in integers,
//     axis_terms_fixed; double-float takes differences first and two values at a
//     time, axis_terms_dw);
//   * ZT (the z queue): each thread keeps its own column's records of the
//     five ring planes, and their in-plane gradients, in tensor memory
//     (TMEM), so the x2 derivatives read TMEM and shared memory keeps full
//     records only for the entering, middle and centre planes: binary32 59 KiB
//     per 32 x 8 CTA, three CTAs per SM (binary64 and double-float records
//     take two TMEM columns per value and keep u_2 of the five planes for
//     D1_z u_2 on the halo: 69 KiB per 16 x 8 CTA, two CTAs).  32 x 16 binary32 tiles (one
//     CTA per SM) keep a fourth full-record plane (the one that was the
//     centre one plane earlier): the next entering plane then overwrites a
//     slot nobody reads any more, so the barrier that ends each plane is not
//     needed;
//   * the arithmetic type T is double, float, dfloat (double-float, binary64
//     storage) or f32x2: two points per thread in packed FP32x2 instructions,
//     two columns x and x + 32 with the shared ring, or with the TMEM queue (the
//     binary32 default) two neighbouring rows (row pairs, see FusedSmem);
//   * the mixed second derivatives of the stress divergence (the D1_a o D1_b
//     reading of the mixed term), for each i sum_{j != i} d2 u_j/dx_i dx_j:
//     - binary64 and double-float, by linearity of D1_i,
//         = D1_i( s_i ),  s_i = sum_{j != i} D1_j u_j,
//       so only the three diagonal gradients D1_j u_j are needed around a
//       point: D1_x u0 and D1_y u1 are kept per plane, D1_z u2 is formed on
//       the centre plane's tile and halo (a third barrier per plane);
//     - binary32, with every x2 derivative applied last (D1_a and D1_b
//       commute on the periodic grid):
//         i = 0:  D1_x(D1_y u1) + D1_z(D1_x u2)
//         i = 1:  D1_y(D1_x u0) + D1_z(D1_y u2)
//         i = 2:  D1_z(D1_x u0 + D1_y u1)
//       so the halo helpers D1_y u1 and D1_x u0 are in-plane, formed as a
//       plane enters (three planes of helper buffers), and the x2 parts come
//       from the thread's own column (D1_x u2, D1_y u2 kept per plane in a
//       second TMEM window): no u_2 on the halo and two barriers per plane.
//
// Variables are stored as deviations from the reference state
// (rho' = rho - 1, rho u_i, (rho E)' = rho E - p_ref/(gamma-1)), which keeps
// binary32 storage free of the low-Mach cancellation in rho E; the residual
// is the same algebraic expression (the constant parts of rho E and p enter
// only through the reference enthalpy term -H0 div u).
#pragma once

#include <atomic>
#include <type_traits>

#include "dfloat.cuh"
#include "f32x2.cuh"
#include "fpconv.cuh"
#include "sbli_internal.cuh"
#include "stencil_int.cuh"

namespace sbli {

constexpr int TX = 32;  // tile width along x0 (one warp)
constexpr int HALO = 2;
constexpr int NSLOT = 5;

// primitive values of one point record in a ring slot; V_H is E' + 2 p' (see
// StreamTerms), V_P holds 2 p' (the
// pressure enters Eqs. 2-3 only as 2 D_i p and 2 D_j(p u_j) in the combined
// skew form, so the factor 2 is applied once per point instead of once per
// stencil neighbour; scaling by 2 is exact)
enum { V_RHO, V_M0, V_M1, V_M2, V_H, V_U0, V_U1, V_U2, V_P, V_T, NV };
static_assert(V_U2 == V_U1 + 1 && V_U1 % 2 == 0, "u1, u2 form one 8-byte pair of a binary32 record");

// ZT (binary32 with the TMEM z queue): the x2 neighbours of a thread's own
// column come from tensor memory, so shared memory keeps full records only
// for the planes that are still to become the centre (entering, middle,
// centre: 3 slots), u_2 alone on the five ring planes (for D1_z u_2 on the
// halo), and no D1_x u0 / D1_y u1 ring.
template <typename T, int TY, bool ZT>
constexpr int full_slots() {
  return ZT ? (TY >= 16 && sizeof(T) == 4 ? 4 : 3) : NSLOT;
}
// Binary32 arithmetic types group the mixed second derivatives so that the
// x2 derivative is applied last (see fused_march): their helpers are
// in-plane and formed as each plane enters.
template <typename T>
constexpr bool mixz() {
  return std::is_same<T, float>::value || std::is_same<T, f32x2>::value;
}
// Tile width: 32 columns, a warp a row, for binary32; 16 for binary64 and
// double-float, two rows a warp.  A 16 x 8 tile of 80-byte records takes
// 107 KiB of the shared ring, so two CTAs of four warps share an SM and one's
// arithmetic runs through the other's barriers and latencies, and ragged edges
// waste half as much, for 1.88 instead of 1.69 records converted a point.  us a
// stage, one 32 x 8 CTA an SM -> two of 16 x 8: binary64 128^3 825 -> 781, 256^3
// 6380 -> 6035, 129x97x66 454 -> 386; double-float 279 -> 264, 2119 -> 1938, 154 -> 132.
template <typename T>
constexpr int tile_x() {
  return std::is_same<T, double>::value || std::is_same<T, dfloat>::value ? F64_TILE_X : TX;
}
// Row pairs (f32x2 with the TMEM queue): a thread owns two neighbouring rows
// of its column, and a record holds both rows' values side by side, so the
// rows of records are pairs: TY / 2 of them, with one pair of halo on each side.
// One point per thread was bound by shared-memory wavefronts (67 % of the L1
// pipe) and issue (62 %): a pair shares its x1 neighbours (four row loads for
// eight), its packed instructions do two points (466 instructions a point for
// 690), and 12 warps of 164 registers hold the points that 24 of 80 did.  Every
// operation rounds as in the one-point kernel, so results are bitwise the same.
// us a stage: 128^3 70.4 -> 63.7, 256^3 483 -> 450 (double-float accumulator 443 ->
// 416), 512^3 3640 -> 3443 (3328 -> 3163), 64-member ensemble 12 %.  Now bound by
// latency (issue 45 %; loads from memory, shared memory, barriers).
template <typename T, bool ZT>
constexpr bool row_pairs() {
  return std::is_same<T, f32x2>::value && ZT;
}
template <typename T, int TY, bool ZT = false>
struct FusedSmem {
  static constexpr int TX = tile_x<T>(), SX = TX + 2 * HALO;
  static constexpr bool RP = row_pairs<T, ZT>();
  static constexpr int HR = RP ? HALO / 2 : HALO;  // rows of halo records on each side
  static constexpr int NR = RP ? TY / 2 : TY;      // rows of records of the tile
  static constexpr int NTHREADS = TX * NR;
  static constexpr int SY = NR + 2 * HR;
  static constexpr int NFULL = full_slots<T, TY, ZT>();
  static constexpr bool MIXZ = mixz<T>();
  static constexpr bool U2 = ZT && !MIXZ;      // u_2 ring (binary64 / double-float TMEM queue)
  static constexpr int NDV = MIXZ ? 4 : 2;     // per-plane gradients in the shared ring
  static constexpr int NSB = MIXZ ? 3 : 1;     // planes of helper buffers
  T ring[NFULL][SY][SX][NV];  // rho', m_i, E', u_i, p', T' per haloed point
  T u2ring[U2 ? NSLOT : 1][U2 ? SY : 1][U2 ? SX : 1];  // u_2 per haloed point of the five ring planes
  // without the TMEM queue: D1_x u0, D1_y u1 (and, binary32, D1_x u2, D1_y u2)
  // per plane (tile only)
  T dring[ZT ? 1 : NSLOT][ZT ? 1 : NDV][ZT ? 1 : NR][ZT ? 1 : TX];
  // binary64 / double-float: s_0 = D1_y u1 + D1_z u2 and s_1 = D1_x u0 + D1_z u2
  // on the centre plane; binary32: D1_y u1 and D1_x u0 of the last three
  // planes to enter (x0-haloed rows, x1-haloed columns)
  T s0buf[NSB][NR][SX];
  T s1buf[NSB][SY][TX];
  double red[2][32];          // block reduction of (ke, enstrophy)
  uint32_t tmem_base[2];      // TMEM allocations (z queue variant)
};

// 1/rho for the primitives (Eqs. 4-5): a refined hardware approximation in
// binary64, a double-word reciprocal in double-float; binary32 takes the
// hardware approximation (rcp.approx, within one unit in the last place),
// far inside the binary32 tolerance and one instruction instead of the
// rounding-correction sequence.
__device__ __forceinline__ float rcp_approx_f32(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <typename T>
__device__ __forceinline__ T recip(T x);
template <>
__device__ __forceinline__ double recip<double>(double x) {
  return rcp_newton_f64(x);
}
template <>
__device__ __forceinline__ float recip<float>(float x) { return rcp_approx_f32(x); }
template <>
__device__ __forceinline__ dfloat recip<dfloat>(dfloat x) { return dw_reciprocal(x); }
template <>
__device__ __forceinline__ f32x2 recip<f32x2>(f32x2 x) { return f32x2(rcp_approx_f32(x.x), rcp_approx_f32(x.y)); }

// Record load/store with 8-byte (binary32: 40-byte records) or 16-byte
// (binary64: 80-byte records) vector accesses; both strides are bank-conflict
// free for the vector width used.
__device__ __forceinline__ void load_rec(const float* p, float (&r)[NV]) {
  const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) {
    const float2 t = q[i];
    r[2 * i] = t.x;
    r[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ void load_rec(const double* p, double (&r)[NV]) {
  const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) {
    const double2 t = q[i];
    r[2 * i] = t.x;
    r[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ void store_rec(float* p, const float (&r)[NV]) {
  float2* q = reinterpret_cast<float2*>(p);
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) q[i] = make_float2(r[2 * i], r[2 * i + 1]);
}
__device__ __forceinline__ void store_rec(double* p, const double (&r)[NV]) {
  double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) q[i] = make_double2(r[2 * i], r[2 * i + 1]);
}
// two-column binary32 records: 80 bytes, two values of both columns per 16-byte access
__device__ __forceinline__ void load_rec(const f32x2* p, f32x2 (&r)[NV]) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) {
    const float4 v = q[i];
    r[2 * i] = f32x2(v.x, v.y);
    r[2 * i + 1] = f32x2(v.z, v.w);
  }
}
__device__ __forceinline__ void store_rec(f32x2* p, const f32x2 (&r)[NV]) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) q[i] = make_float4(r[2 * i].x, r[2 * i].y, r[2 * i + 1].x, r[2 * i + 1].y);
}
// Double-float records: 80 bytes, five pairs of values of 16 bytes each, (hi,
// hi, lo, lo), so that a pair is one 16-byte access and comes as the operands
// of the packed instructions (dfloat2): (m0, m1), (m2, H), (u0, u1), (u2, T'),
// (rho', 2p').
enum { W_M01, W_M2H, W_U01, W_U2T, W_RHOP, NW };
constexpr int dw_slot(int v) {  // 2 * pair + lane of a value
  return v == V_RHO ? 8 : v == V_P ? 9 : v == V_T ? 7 : v <= V_H ? v - V_M0 : v - V_U0 + 4;
}
__device__ __forceinline__ void load_pairs(const dfloat* p, dfloat2 (&r)[NW]) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const float4 v = q[i];
    r[i] = dfloat2(make_float2(v.x, v.y), make_float2(v.z, v.w));
  }
}
__device__ __forceinline__ void store_rec(dfloat* p, const dfloat (&r)[NV]) {
  float4* q = reinterpret_cast<float4*>(p);
  dfloat s[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) s[dw_slot(v)] = r[v];
#pragma unroll
  for (int i = 0; i < NW; ++i) q[i] = make_float4(s[2 * i].hi, s[2 * i + 1].hi, s[2 * i].lo, s[2 * i + 1].lo);
}
// one value of a record
template <typename T>
__device__ __forceinline__ T rec_value(const T* r, int v) {
  return r[v];
}
// (the 16-byte load of its pair: 4-byte loads at this stride conflict 4-way)
__device__ __forceinline__ dfloat2 load_pair(const dfloat* r, int pair) {
  const float4 v = reinterpret_cast<const float4*>(r)[pair];
  return dfloat2(make_float2(v.x, v.y), make_float2(v.z, v.w));
}
__device__ __forceinline__ dfloat rec_value(const dfloat* r, int v) {
  const dfloat2 x = load_pair(r, dw_slot(v) / 2);
  return dw_slot(v) % 2 ? x.b() : x.a();
}

// ---- tensor memory (TMEM) as a per-thread queue of x2-neighbour records.
// Each warp of the CTA owns the 32 TMEM lanes of its quarter (warp % 4) and a
// column window (warp / 4); a thread keeps its own column's records of the
// five ring planes there.  A value takes W 32-bit columns (binary32: 1;
// binary64 and double-float: 2): fields 0-7 of slot s in columns 8W s ..
// 8W s + 8W - 1, fields 8-9 from column 40W + 2W s, and the pair
// (D1_x u0, D1_y u1) from column 50W + 2W s, so every access is aligned to
// its own width; windows are 64 W columns.  32x32b shapes: each thread of
// the warp reads or writes its own lane.
template <typename T>
struct TmLayout {
  static constexpr int W = sizeof(T) / 4;      // 32-bit columns per value
  static constexpr int HEAD = 8 * W;           // columns of fields 0-7 of one slot
  static constexpr int TAIL = HEAD * NSLOT;    // fields 8-9 of slot s: columns TAIL + 2W s ...
  static constexpr int DIAG = TAIL + 2 * W * NSLOT;  // D1_x u0, D1_y u1 of slot s: DIAG + 2W s ...
  static constexpr int COLS = 64 * W;          // window width
  static_assert(NV == 10 && DIAG + 2 * W * NSLOT <= COLS, "z queue must fit the warp's TMEM window");
};

// columns a CTA of NW warps allocates: a power of two, at least 32
template <int NW, typename T = float>
constexpr int tmem_columns() {
  constexpr int need = TmLayout<T>::COLS * ((NW + 3) / 4);
  int c = 32;
  while (c < need) c *= 2;
  return c;
}
// The binary32 queue's second window (a separate allocation): the pair
// (D1_x u2, D1_y u2) of slot s in columns 2s, 2s + 1 of a 16-column window.
template <typename T>
constexpr int tm_xcols() {
  return 16 * (int)(sizeof(T) / 4);
}
template <int NW, typename T = float>
constexpr int tmem_columns2() {
  if (!mixz<T>()) return 0;
  constexpr int need = tm_xcols<T>() * ((NW + 3) / 4);
  int c = 32;
  while (c < need) c *= 2;
  return c;
}

// The tensor-memory accesses below are warp-aligned (.sync.aligned): all lanes
// execute one together.  After code whose branches the lanes of a warp may take
// differently (halo points, the columns of a ragged tile, values that the integer
// sums cannot align) the march calls this first.
template <bool ZT>
__device__ __forceinline__ void tmem_converge() {
  if constexpr (ZT) __syncwarp();
}

// win: this thread's window address (lane and window column), slot: ring slot
__device__ __forceinline__ void tmem_store_rec(uint32_t win, int slot, const float (&r)[NV]) {
  using L = TmLayout<float>;
  const uint32_t taddr = win + (uint32_t)(L::HEAD * slot), ttail = win + (uint32_t)(L::TAIL + 2 * slot);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n\t"
      "tcgen05.st.sync.aligned.32x32b.x2.b32 [%9], {%10, %11};\n\t"
      "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
      "r"(__float_as_uint(r[0])), "r"(__float_as_uint(r[1])), "r"(__float_as_uint(r[2])), "r"(__float_as_uint(r[3])),
      "r"(__float_as_uint(r[4])), "r"(__float_as_uint(r[5])), "r"(__float_as_uint(r[6])), "r"(__float_as_uint(r[7])),
      "r"(ttail), "r"(__float_as_uint(r[8])), "r"(__float_as_uint(r[9]))
      : "memory");
}

__device__ __forceinline__ void tmem_load_rec(uint32_t win, int slot, float (&r)[NV]) {
  using L = TmLayout<float>;
  const uint32_t taddr = win + (uint32_t)(L::HEAD * slot), ttail = win + (uint32_t)(L::TAIL + 2 * slot);
  uint32_t v[NV];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%10];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8, %9}, [%11];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9])
      : "r"(taddr), "r"(ttail)
      : "memory");
#pragma unroll
  for (int i = 0; i < NV; ++i) r[i] = __uint_as_float(v[i]);
}
// the pair (D1_x u0, D1_y u1) of this thread's column in slot `slot`
__device__ __forceinline__ void tmem_store_diag(uint32_t win, int slot, float d00, float d11) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};\n\t"
      "tcgen05.wait::st.sync.aligned;" ::"r"(win + (uint32_t)(TmLayout<float>::DIAG + 2 * slot)),
      "r"(__float_as_uint(d00)), "r"(__float_as_uint(d11))
      : "memory");
}
__device__ __forceinline__ void tmem_load_diag(uint32_t win, int slot, float& d00, float& d11) {
  uint32_t a, b;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(a), "=r"(b)
      : "r"(win + (uint32_t)(TmLayout<float>::DIAG + 2 * slot))
      : "memory");
  d00 = __uint_as_float(a);
  d11 = __uint_as_float(b);
}

// 8-byte values as two 32-bit words: binary64 (low, high word), double-float (hi, lo)
__device__ __forceinline__ void to_words(double x, uint32_t& a, uint32_t& b) {
  a = (uint32_t)__double2loint(x);
  b = (uint32_t)__double2hiint(x);
}
__device__ __forceinline__ void from_words(uint32_t a, uint32_t b, double& x) {
  x = __hiloint2double((int)b, (int)a);
}
__device__ __forceinline__ void to_words(dfloat x, uint32_t& a, uint32_t& b) {
  a = __float_as_uint(x.hi);
  b = __float_as_uint(x.lo);
}
__device__ __forceinline__ void from_words(uint32_t a, uint32_t b, dfloat& x) {
  x.hi = __uint_as_float(a);
  x.lo = __uint_as_float(b);
}

template <typename T>
__device__ __forceinline__ void tmem_store_rec8(uint32_t win, int slot, const T (&r)[NV]) {
  using L = TmLayout<T>;
  const uint32_t taddr = win + (uint32_t)(L::HEAD * slot), ttail = win + (uint32_t)(L::TAIL + 4 * slot);
  uint32_t w[2 * NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) to_words(r[i], w[2 * i], w[2 * i + 1]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};\n\t"
      "tcgen05.st.sync.aligned.32x32b.x4.b32 [%17], {%18, %19, %20, %21};\n\t"
      "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(w[8]), "r"(w[9]),
      "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]), "r"(ttail), "r"(w[16]), "r"(w[17]),
      "r"(w[18]), "r"(w[19])
      : "memory");
}
template <typename T>
__device__ __forceinline__ void tmem_load_rec8(uint32_t win, int slot, T (&r)[NV]) {
  using L = TmLayout<T>;
  const uint32_t taddr = win + (uint32_t)(L::HEAD * slot), ttail = win + (uint32_t)(L::TAIL + 4 * slot);
  uint32_t w[2 * NV];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%20];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16, %17, %18, %19}, [%21];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]), "=r"(w[8]),
        "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15]), "=r"(w[16]),
        "=r"(w[17]), "=r"(w[18]), "=r"(w[19])
      : "r"(taddr), "r"(ttail)
      : "memory");
#pragma unroll
  for (int i = 0; i < NV; ++i) from_words(w[2 * i], w[2 * i + 1], r[i]);
}
template <typename T>
__device__ __forceinline__ void tmem_store_diag8(uint32_t win, int slot, T d00, T d11) {
  uint32_t w[4];
  to_words(d00, w[0], w[1]);
  to_words(d11, w[2], w[3]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n\t"
      "tcgen05.wait::st.sync.aligned;" ::"r"(win + (uint32_t)(TmLayout<T>::DIAG + 4 * slot)),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
      : "memory");
}
template <typename T>
__device__ __forceinline__ void tmem_load_diag8(uint32_t win, int slot, T& d00, T& d11) {
  uint32_t w[4];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
      : "r"(win + (uint32_t)(TmLayout<T>::DIAG + 4 * slot))
      : "memory");
  from_words(w[0], w[1], d00);
  from_words(w[2], w[3], d11);
}
__device__ __forceinline__ void tmem_store_rec(uint32_t win, int slot, const double (&r)[NV]) {
  tmem_store_rec8(win, slot, r);
}
__device__ __forceinline__ void tmem_load_rec(uint32_t win, int slot, double (&r)[NV]) { tmem_load_rec8(win, slot, r); }
// double-float records go through TMEM in the pair order of the shared-memory
// record, as ten 8-byte values (hi, hi), (lo, lo) a pair
__device__ __forceinline__ void tmem_store_rec(uint32_t win, int slot, const dfloat (&r)[NV]) {
  dfloat s[NV], w[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) s[dw_slot(v)] = r[v];
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    w[2 * i] = dfloat(s[2 * i].hi, s[2 * i + 1].hi);
    w[2 * i + 1] = dfloat(s[2 * i].lo, s[2 * i + 1].lo);
  }
  tmem_store_rec8(win, slot, w);
}
__device__ __forceinline__ void tmem_load_pairs(uint32_t win, int slot, dfloat2 (&r)[NW]) {
  dfloat w[NV];
  tmem_load_rec8(win, slot, w);
#pragma unroll
  for (int i = 0; i < NW; ++i)
    r[i] = dfloat2(make_float2(w[2 * i].hi, w[2 * i].lo), make_float2(w[2 * i + 1].hi, w[2 * i + 1].lo));
}
__device__ __forceinline__ void tmem_store_diag(uint32_t win, int slot, double d00, double d11) {
  tmem_store_diag8(win, slot, d00, d11);
}
__device__ __forceinline__ void tmem_load_diag(uint32_t win, int slot, double& d00, double& d11) {
  tmem_load_diag8(win, slot, d00, d11);
}
__device__ __forceinline__ void tmem_store_diag(uint32_t win, int slot, dfloat d00, dfloat d11) {
  tmem_store_diag8(win, slot, d00, d11);
}
__device__ __forceinline__ void tmem_load_diag(uint32_t win, int slot, dfloat& d00, dfloat& d11) {
  tmem_load_diag8(win, slot, d00, d11);
}
// row pairs: a value is two words, one a row
__device__ __forceinline__ void to_words(f32x2 x, uint32_t& a, uint32_t& b) {
  a = __float_as_uint(x.x);
  b = __float_as_uint(x.y);
}
__device__ __forceinline__ void from_words(uint32_t a, uint32_t b, f32x2& x) {
  x = f32x2(__uint_as_float(a), __uint_as_float(b));
}
__device__ __forceinline__ void tmem_store_rec(uint32_t win, int slot, const f32x2 (&r)[NV]) {
  tmem_store_rec8(win, slot, r);
}
__device__ __forceinline__ void tmem_load_rec(uint32_t win, int slot, f32x2 (&r)[NV]) { tmem_load_rec8(win, slot, r); }
__device__ __forceinline__ void tmem_store_diag(uint32_t win, int slot, f32x2 d00, f32x2 d11) {
  tmem_store_diag8(win, slot, d00, d11);
}
__device__ __forceinline__ void tmem_load_diag(uint32_t win, int slot, f32x2& d00, f32x2& d11) {
  tmem_load_diag8(win, slot, d00, d11);
}

// Allocate / release the CTA's TMEM columns (warp 0): NCOL for the queue
// and, binary32, NCOL2 for its second window, publishing the base addresses
// through shared memory.  The CTAs that shared memory lets share an SM never
// ask for more than the 512 columns available (binary32 32 x 8: 3 x (128 +
// 32); 32 x 16: 256 + 64; binary64 and double-float 16 x 8: 2 x 128),
// so the allocation never waits.
template <int NCOL, int NCOL2 = 0>
__device__ __forceinline__ void tmem_acquire(uint32_t (&smem_slot)[2], uint32_t& base, uint32_t& base2) {
  if ((threadIdx.x >> 5) == 0) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&smem_slot[0]);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(NCOL) : "memory");
    if (NCOL2 > 0) {
      const uint32_t dst2 = (uint32_t)__cvta_generic_to_shared(&smem_slot[1]);
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst2), "r"(NCOL2)
                   : "memory");
    }
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  base = *(volatile uint32_t*)&smem_slot[0];
  base2 = NCOL2 > 0 ? *(volatile uint32_t*)&smem_slot[1] : 0u;
}

template <int NCOL, int NCOL2 = 0>
__device__ __forceinline__ void tmem_release(uint32_t base, uint32_t base2) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(NCOL) : "memory");
    if (NCOL2 > 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base2), "r"(NCOL2) : "memory");
  }
}

// This thread's TMEM window: lane quarter of its warp, column window warp / 4.
template <typename T>
__device__ __forceinline__ uint32_t tmem_window(uint32_t base) {
  const uint32_t w = threadIdx.x >> 5;
  return base + (((w & 3u) * 32u) << 16) + (w >> 2) * (uint32_t)TmLayout<T>::COLS;
}
template <typename T>
__device__ __forceinline__ uint32_t tmem_window2(uint32_t base2) {
  const uint32_t w = threadIdx.x >> 5;
  return base2 + (((w & 3u) * 32u) << 16) + (w >> 2) * (uint32_t)tm_xcols<T>();
}
// the pair (D1_x u2, D1_y u2) of this thread's column in slot `slot` of the
// second window
__device__ __forceinline__ void tmem_store_xdiag(uint32_t win2, int slot, float d02, float d12) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};\n\t"
      "tcgen05.wait::st.sync.aligned;" ::"r"(win2 + (uint32_t)(2 * slot)),
      "r"(__float_as_uint(d02)), "r"(__float_as_uint(d12))
      : "memory");
}
__device__ __forceinline__ void tmem_load_xdiag(uint32_t win2, int slot, float& d02, float& d12) {
  uint32_t a, b;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(a), "=r"(b)
      : "r"(win2 + (uint32_t)(2 * slot))
      : "memory");
  d02 = __uint_as_float(a);
  d12 = __uint_as_float(b);
}

__device__ __forceinline__ void tmem_store_xdiag(uint32_t win2, int slot, f32x2 d02, f32x2 d12) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n\t"
      "tcgen05.wait::st.sync.aligned;" ::"r"(win2 + (uint32_t)(4 * slot)),
      "r"(__float_as_uint(d02.x)), "r"(__float_as_uint(d02.y)), "r"(__float_as_uint(d12.x)), "r"(__float_as_uint(d12.y))
      : "memory");
}
__device__ __forceinline__ void tmem_load_xdiag(uint32_t win2, int slot, f32x2& d02, f32x2& d12) {
  uint32_t w[4];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
      : "r"(win2 + (uint32_t)(4 * slot))
      : "memory");
  from_words(w[0], w[1], d02);
  from_words(w[2], w[3], d12);
}

// Stage input value in the arithmetic type (binary64 inputs to a binary32
// stage are narrowed with integer re-packing, see fpconv.cuh).
template <typename T, typename TIN>
__device__ __forceinline__ T to_compute(TIN v) {
  return T(v);
}
template <>
__device__ __forceinline__ float to_compute<float, double>(double v) {
  return narrow_f64_fast(v);
}
// binary64 -> double-float: hi = v rounded to nearest, ties away from zero, and the
// remainder (29 bits) rounded to 24, in integer and binary32 operations
template <>
__device__ __forceinline__ dfloat to_compute<dfloat, double>(double v) {
  float hi, lo;
  split_f64(v, hi, lo);
  return dfloat(hi, lo);
}

// A binary64 stage output in the stored type: itself, or (double-float
// stage fields) the same hi + lo split a binary64 input gets when it is
// loaded, so the consumer reads the pair it would have formed.
template <typename TOUT>
__device__ __forceinline__ TOUT to_output(double v) {
  return TOUT(v);
}
template <>
__device__ __forceinline__ dfloat to_output<dfloat>(double v) {
  return to_compute<dfloat, double>(v);
}

// a * b + c: left to the compiler's contraction for scalar types, an explicit
// packed FMA for f32x2 (whose operators are not contracted)
template <typename T>
__device__ __forceinline__ T mad(T a, T b, T c) {
  return a * b + c;
}
__device__ __forceinline__ f32x2 mad(f32x2 a, f32x2 b, f32x2 c) { return fma(a, b, c); }
__device__ __forceinline__ float mad(float a, float b, float c) { return ::fmaf(a, b, c); }
// rows y + 1, y + 2 from the pairs of rows (y, y + 1) and (y + 2, y + 3)
__device__ __forceinline__ f32x2 next_row(f32x2 a, f32x2 b) { return f32x2(a.y, b.x); }

// A stage value built from the stage input of each column a thread owns.
template <typename T, typename TIN>
__device__ __forceinline__ T from_lanes(const TIN (&v)[1]) {
  return to_compute<T, TIN>(v[0]);
}
template <typename T, typename TIN>
__device__ __forceinline__ T from_lanes(const TIN (&v)[2]) {
  return T(to_compute<float, TIN>(v[0]), to_compute<float, TIN>(v[1]));
}

// binary64-class arithmetic types (binary64 Runge-Kutta update in place)
template <typename T>
constexpr bool is_f64_class() {
  return std::is_same<T, double>::value || std::is_same<T, dfloat>::value;
}

// A stage value in binary64 for the Runge-Kutta update.
__device__ __forceinline__ double as_double(double x) { return x; }
__device__ __forceinline__ double as_double(float x) { return widen_f32_fast(x); }
__device__ __forceinline__ double as_double(dfloat x) { return widen_f32_fast(x.hi) + widen_f32_fast(x.lo); }

// a * b + c with one rounding in every scalar type (and lane): the streamed
// terms below never leave a contraction to the compiler, so that every
// instantiation of the kernel rounds alike.
__device__ __forceinline__ double fmadd(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ float fmadd(float a, float b, float c) { return ::fmaf(a, b, c); }
__device__ __forceinline__ f32x2 fmadd(f32x2 a, f32x2 b, f32x2 c) { return fma(a, b, c); }

// a + b, never contracted with the product that formed b
__device__ __forceinline__ double add_nc(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_nc(float a, float b) { return __fadd_rn(a, b); }
template <typename T>
__device__ __forceinline__ T add_nc(T a, T b) {
  return a + b;
}

// Accumulated terms of the residual at one point for the hardware FMA types.
// The centre values u_j^c, m_i^c are constant over a stencil, so the
// convective terms of Eqs. 2-3 share the weight w = c (u_j + u_j^c) and
//   E' (u_j + u_j^c) + 2 p' u_j = (E' + 2p')(u_j + u_j^c) - u_j^c 2p'
// makes those of Eq. 3 one multiply-add a neighbour with H = E' + 2p' (the
// record keeps H) and u_j^c times the pressure derivative that Eq. 2 needs
// anyway.  (The like for Eq. 1, m_j + u_j^c rho' = u_j + rho' (u_j + u_j^c), would
// take the rounding of u_j = m_j / rho into the mass balance: 1.45 times its
// error, so Eq. 1 keeps two.)  The viscous terms of Eq. 2 are accumulated as
// their sum (Laplacian + G/3), the symmetric off-diagonal gradients as their
// sum.  H carries one rounding that E' in its place would not (the centre's E' is
// H - 2p'), for one product fewer a neighbour.  Errors of the energy's residual
// against quadruple precision on 40 grids of 14 to 48 points an edge, with E' before
// and with H: binary64 6.70e-14, 6.66e-14, double-float 4.47e-12, 4.19e-12, binary32
// 5.05e-5 both (the rounding of its input).
// All that is 15 multiply-adds a neighbour in binary32 instead of the 17 of one
// accumulator per derivative (one point a thread, where the number of instructions
// counted most: 512^3, binary64 accumulator, 3.73 -> 3.63 ms a stage).  Binary64 takes the linear
// stencils in integers (axis_terms_sums) and the factors -1/2 (convective terms)
// and 1/3, 4/3 (viscous terms) in its weights; in binary32 the constants of that
// are too many for the uniform registers (256^3: 479 -> 504 us), and the factors
// are applied to the sums of an axis.
template <typename T>
constexpr bool scaled_weights() {
  return std::is_same<T, double>::value;
}
template <typename T>
struct StreamTerms {
  // with scaled_weights times -1/2:
  T rrho;     // sum_j D_j(m_j + u_j^c rho')                      (Eq. 1)
  T rM[3];    // sum_j D_j(m_i (u_j + u_j^c)) + 2 D_i p'          (Eq. 2)
  T rE;       // sum_j D_j(E' (u_j + u_j^c)) + 2 D_j(p' u_j)      (Eq. 3)
  T v[3];     // sum_j D2_j u_i + 1/3 sum_j d2 u_j / dx_i dx_j
  T lapT;     // sum_j D2_j T'
  T a[3];     // D1_j u_i + D1_i u_j for (i, j) = (0, 1), (0, 2), (1, 2)
  T lo[3];    // the first of the two alone, D1_j u_i (vorticity; diagnostics only)
  T gd[3];    // D1_j u_j
};

// No x2-regrouped mixed terms (every axis but the binary32 x2 axis).
struct NoXTerms {
  template <typename T>
  __device__ void operator()(int, T&, T&) const {}
};

// Binary32: all derivatives along axis A, the four neighbours streamed through
// registers one at a time, so only one record is live.  ldrec(k, r) loads the
// record of the neighbour k = 0..3 (offsets -2, -1, +1, +2 along A; Eq. 6
// weights +c2, -c1, +c1, -c2, Eq. 7 e2, e1, e1, e2); sfun(k) gives the
// mixed-term helper s_A there.  ZX (A = 2): the mixed derivatives
// that involve x2 are taken with the x2 derivative last, D1_z(D1_x u2) and
// D1_z(D1_y u2) from xfun(k, ...) (the neighbours' in-plane gradients of u2);
// the stream also forms D1_z u2 at the centre.  WITH_KE: also lo[].
template <int A, bool ZX, bool WITH_KE, bool HALVES = false, typename T = float, typename LD, typename SF, typename XF = NoXTerms>
__device__ __forceinline__ void axis_terms_stream(const LD& ldrec, const SF& sfun, const Coef<T>& c,
                                                  const T (&uc)[3], StreamTerms<T>& t, const XF& xfun = XF()) {
  static_assert(!ZX || A == 2, "x2-last mixed terms belong to the x2 axis");
  const T ua = uc[A];
  T dp = T(0);               // D1_A 2p'
  T lA = T(0), gA = T(0);    // D2_A u_A off-centre, D1_A s_A
  T gz0 = T(0), gz1 = T(0);  // ZX: the x2 parts of G_0, G_1
  auto sgn = [](int k, T inner, T outer) {  // the antisymmetric weight of neighbour k
    return k == 0 ? outer : k == 1 ? -inner : k == 2 ? inner : -outer;
  };
  // the per-axis products c u_A^c once, so that each neighbour's weight is one multiply-add
  const T cu1 = c.c1[A] * ua, cu2 = c.c2[A] * ua;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const T cd = sgn(k, c.c1[A], c.c2[A]);
    const T ed = (k == 0 || k == 3) ? c.e2[A] : c.e1[A];
    // rows that straddle two pairs: lane by lane, which spares putting the
    // values together in register pairs
    auto fm = [k](T x, T y, T z) {
      if constexpr (HALVES) {
        if (k == 1 || k == 2) return T(__fmaf_rn(x.x, y.x, z.x), __fmaf_rn(x.y, y.y, z.y));
      }
      return fmadd(x, y, z);
    };
    T r[NV];
    ldrec(k, r);
    const T w = fm(cd, r[V_U0 + A], sgn(k, cu1, cu2));
#pragma unroll
    for (int i = 0; i < 3; ++i) t.rM[i] = fm(w, r[V_M0 + i], t.rM[i]);
    t.rE = fm(w, r[V_H], t.rE);
    t.rrho = fm(cd, fm(ua, r[V_RHO], r[V_M0 + A]), t.rrho);
    dp = fm(cd, r[V_P], dp);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (i != A) {
        t.v[i] = fm(ed, r[V_U0 + i], t.v[i]);
        const int pair = i + A - 1;  // (0,1) -> 0, (0,2) -> 1, (1,2) -> 2
        t.a[pair] = fm(cd, r[V_U0 + i], t.a[pair]);
        if (WITH_KE && i < A) t.lo[pair] = fm(cd, r[V_U0 + i], t.lo[pair]);
      }
    }
    // the Laplacian and one third of Eq. 7 on j = A, one third of D1_A s_A
    lA = fm(ed, r[V_U0 + A], lA);
    gA = fm(cd, sfun(k), gA);
    t.lapT = fm(ed, r[V_T], t.lapT);
    if constexpr (ZX) {
      T x02, x12;
      xfun(k, x02, x12);
      gz0 = fm(cd, x02, gz0);
      gz1 = fm(cd, x12, gz1);
      t.gd[2] = fm(cd, r[V_U2], t.gd[2]);
    }
  }
  t.rM[A] = t.rM[A] + dp;
  t.rE = fmadd(-ua, dp, t.rE);
  t.v[A] = fmadd(T(4.0 / 3.0), lA, fmadd(T(1.0 / 3.0), gA, t.v[A]));
  if constexpr (ZX) {
    t.v[0] = fmadd(T(1.0 / 3.0), gz0, t.v[0]);
    t.v[1] = fmadd(T(1.0 / 3.0), gz1, t.v[1]);
  }
}

// Binary64: the linear stencils of an axis (Laplacians of u and T', cross
// gradients, D1_A of p', rho', m_A and s_A) in integers, the products with the
// velocities on the binary64 pipe: 33 binary64 instructions an axis instead of
// 62, beside some 800 integer ones that run while that pipe is busy.  32 x 8
// tiles: 256^3 8.86 -> 6.39 ms a stage, 64^3 168 -> 128 us; the pipe stays the
// bound: two CTAs of 16 x 8 keep it at 0.95 of its measured rate (512^3 0.97) with
// 175 instructions a point, the primitives of the halo included.
// The pressure sum folded into two multiply-adds and the reciprocal's third-order step
// (fpconv.cuh): 6.05 -> 5.89 ms, 64^3 122.9 -> 119.1 us.  Values too large to align,
// infinities and NaNs take the sums in binary64 (FIXED false).
template <int A, bool WITH_KE, bool FIXED>
__device__ __forceinline__ void axis_terms_sums(const double (&r)[4][NV], const double (&sx)[4], const double (&sy)[4],
                                                const uint32_t (&top)[NV], uint32_t stop, const Coef<double>& c,
                                                const double (&uc)[3], StreamTerms<double>& t) {
  const double ua = uc[A];
  const double hu1 = c.hc1[A] * ua, hu2 = c.hc2[A] * ua;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double hd = k == 0 ? c.hc2[A] : k == 1 ? -c.hc1[A] : k == 2 ? c.hc1[A] : -c.hc2[A];
    const double hu = k == 0 ? hu2 : k == 1 ? -hu1 : k == 2 ? hu1 : -hu2;
    const double w = fmadd(hd, r[k][V_U0 + A], hu);
#pragma unroll
    for (int i = 0; i < 3; ++i) t.rM[i] = fmadd(w, r[k][V_M0 + i], t.rM[i]);
    t.rE = fmadd(w, r[k][V_H], t.rE);
  }
  auto first = [&](int v) { return first_sum<FIXED>(r[0][v], r[1][v], r[2][v], r[3][v], top[v]); };
  auto second = [&](int v) { return second_sum<FIXED>(r[0][v], r[1][v], r[2][v], r[3][v], top[v]); };
  const double dp = first(V_P);
  t.rM[A] = fmadd(c.hc2[A], dp, t.rM[A]);
  t.rE = fmadd(-hu2, dp, t.rE);
  t.rrho = fmadd(c.hc2[A], fmadd(ua, first(V_RHO), first(V_M0 + A)), t.rrho);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int v = V_U0 + i;
    if (i == A) {  // the Laplacian and one third of Eq. 7 on j = A
      t.v[i] = fmadd(c.f2[A], second(v), t.v[i]);
    } else {
      double f, s;
      both_sums<FIXED>(r[0][v], r[1][v], r[2][v], r[3][v], top[v], f, s);
      t.v[i] = fmadd(c.e2[A], s, t.v[i]);
      const int pair = i + A - 1;  // (0,1) -> 0, (0,2) -> 1, (1,2) -> 2
      t.a[pair] = fmadd(c.c2[A], f, t.a[pair]);
      if (WITH_KE && i < A) t.lo[pair] = fmadd(c.c2[A], f, t.lo[pair]);
    }
  }
  t.lapT = fmadd(c.e2[A], second(V_T), t.lapT);
  const double ds = A == 2 ? first_sum<FIXED>(sx, sy, stop) : first_sum<FIXED>(sx[0], sx[1], sx[2], sx[3], stop);
  t.v[A] = fmadd(c.t2[A], ds, t.v[A]);
}
// ldrec(k, r) loads the record of neighbour k (offsets -2, -1, +1, +2); sfun(k, x,
// y) the mixed-term helper s_A there (x; x + y along x2).
template <int A, bool WITH_KE, typename LD, typename SF>
__device__ __forceinline__ void axis_terms_fixed(const LD& ldrec, const SF& sfun, const Coef<double>& c,
                                                 const double (&uc)[3], StreamTerms<double>& t) {
  double r[4][NV], sx[4], sy[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    ldrec(k, r[k]);
    sfun(k, sx[k], sy[k]);
  }
  uint32_t top[NV], worst = 0;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (v == V_H || (v >= V_M0 && v <= V_M2 && v != V_M0 + A)) continue;  // no linear stencil of these
    top[v] = fixed::top_exponent(r[0][v], r[1][v], r[2][v], r[3][v]);
    worst = max(worst, top[v]);
  }
  uint32_t stop = fixed::top_exponent(sx[0], sx[1], sx[2], sx[3]);
  if (A == 2) stop = max(stop, fixed::top_exponent(sy[0], sy[1], sy[2], sy[3]));
  worst = max(worst, stop);
  if (fixed::alignable(worst))
    axis_terms_sums<A, WITH_KE, true>(r, sx, sy, top, stop, c, uc, t);
  else
    axis_terms_sums<A, WITH_KE, false>(r, sx, sy, top, stop, c, uc, t);
}

// Eqs. 1-3 at one point from the streamed terms and the centre values.
template <typename T>
__device__ __forceinline__ void assemble_streamed(const StreamTerms<T>& t, T rho_p, const T (&mc)[3], T Ec,
                                                  const T (&uc)[3], const Coef<T>& c, T (&R)[5]) {
  constexpr bool SW = scaled_weights<T>();
  const T div = t.gd[0] + t.gd[1] + t.gd[2];
  const T hdiv = SW ? T(-0.5) * div : div;
  auto half = [](T x) { return SW ? x : T(-0.5) * x; };
  R[0] = half(fmadd(T(1) + rho_p, hdiv, t.rrho));
#pragma unroll
  for (int i = 0; i < 3; ++i) R[1 + i] = fmadd(c.inv_re, t.v[i], half(fmadd(mc[i], hdiv, t.rM[i])));
  // viscous dissipation du_i/dx_j (du_i/dx_j + du_j/dx_i - 2/3 div delta_ij) and the work of the viscous force
  T d = t.gd[0] * t.gd[0];
  d = fmadd(t.gd[2], t.gd[2], fmadd(t.gd[1], t.gd[1], d));
  T q = (T(-2.0 / 3.0) * div) * div;
  q = fmadd(t.a[2], t.a[2], fmadd(t.a[1], t.a[1], fmadd(t.a[0], t.a[0], q)));
  q = fmadd(T(2), d, q);
  q = fmadd(uc[2], t.v[2], fmadd(uc[1], t.v[1], fmadd(uc[0], t.v[0], q)));
  R[4] = fmadd(c.kappa, t.lapT, fmadd(c.inv_re, q, fmadd(-c.H0, div, half(fmadd(Ec, hdiv, t.rE)))));
}

// ---- double-float: the same terms in pairs.  A double-word sum costs 8
// instructions and a product 4, so differences and sums of neighbours come
// first, then one product with the common weight: with c1 = 8 c2 and
// e1 = -16 e2 (Eqs. 6-7) a first derivative is c2 (8 (f+1 - f-1) - (f+2 - f-2)) and
// the off-centre part of a second one e2 ((f+2 + f-2) - 16 (f+1 + f-1)), the scalings
// exact; the weights u_j + u_j^c take the 8 themselves.  Two values at a time
// go through packed two-lane instructions: the pairs of the record, and for
// the cross gradients and (m_A, s_A) pairs put together in registers.  256^3,
// 37 planes a CTA: 2.43 -> 2.20 ms a stage, 3727 -> about 2450 instructions a point;
// bound by the latency of dependent instructions and of shared memory at the
// two warps a sub-partition that the registers leave (16 x 8 tiles, two CTAs an SM:
// issue 50 %, 1.94 ms; three CTAs of the TMEM queue at 168 registers spill, 2.10).
struct DwTerms {
  dfloat2 m01, m2e;  // -1/2 the convective sums of Eq. 2 (i = 0, 1), (i = 2 and Eq. 3)
  dfloat2 v01, v2t;  // sum_j D2_j u_i + 1/3 sum_j d2 u_j / dx_i dx_j, and sum_j D2_j T'
  dfloat rho;        // -1/2 sum_j D_j(m_j + u_j^c rho')
  dfloat a01, a02, a12;  // D1_j u_i + D1_i u_j
  dfloat w01, w02, w12;  // their differences D1_j u_i - D1_i u_j, i < j (diagnostics only)
};
__device__ __forceinline__ dfloat2 dw_first(dfloat2 m2, dfloat2 m1, dfloat2 p1, dfloat2 p2, dfloat2 k) {
  return (dw_scale(p1 - m1, 8.0f) - (p2 - m2)) * k;
}
template <int A>
__device__ __forceinline__ dfloat pair_u(const dfloat2 (&r)[NW]) {  // u_A of a record
  return A == 0 ? r[W_U01].a() : A == 1 ? r[W_U01].b() : r[W_U2T].a();
}
template <int A>
__device__ __forceinline__ dfloat pair_m(const dfloat2 (&r)[NW]) {  // m_A
  return A == 0 ? r[W_M01].a() : A == 1 ? r[W_M01].b() : r[W_M2H].a();
}

// All terms along axis A; ldp(k, pairs) loads the record of neighbour k (offsets
// -2, -1, +1, +2), sfun(k) the mixed-term helper s_A there.
template <int A, bool WITH_KE, typename LD, typename SF>
__device__ __forceinline__ void axis_terms_dw(const LD& ldp, const SF& sfun, const Coef<dfloat>& c, dfloat ua,
                                              DwTerms& t) {
  const dfloat2 kh(c.hc2[A]);
  // the inner neighbours, then the outer ones: two records live at a time
  dfloat2 cm01, cm2e, rp, dms, l01, l2t, g;
  auto cross = [](const dfloat2(&r)[NW]) {  // (u_i, u_j), i, j != A
    return A == 2 ? r[W_U01] : dfloat2(A == 0 ? r[W_U01].b() : r[W_U01].a(), r[W_U2T].a());
  };
  {
    dfloat2 m[NW], p[NW];
    ldp(1, m);
    ldp(2, p);
    const dfloat2 wm(dw_scale(pair_u<A>(m) + ua, -8.0f)), wp(dw_scale(pair_u<A>(p) + ua, 8.0f));
    cm01 = wp * p[W_M01] + wm * m[W_M01];
    cm2e = wp * p[W_M2H] + wm * m[W_M2H];
    rp = dw_scale(p[W_RHOP] - m[W_RHOP], 8.0f);
    dms = dw_scale(dfloat2(pair_m<A>(p), sfun(2)) - dfloat2(pair_m<A>(m), sfun(1)), 8.0f);
    l01 = dw_scale(p[W_U01] + m[W_U01], 16.0f);
    l2t = dw_scale(p[W_U2T] + m[W_U2T], 16.0f);
    g = dw_scale(cross(p) - cross(m), 8.0f);
  }
  {
    dfloat2 m[NW], p[NW];
    ldp(0, m);
    ldp(3, p);
    const dfloat2 wm(pair_u<A>(m) + ua), wp(-(pair_u<A>(p) + ua));
    cm01 = (cm01 + (wp * p[W_M01] + wm * m[W_M01])) * kh;
    cm2e = (cm2e + (wp * p[W_M2H] + wm * m[W_M2H])) * kh;
    rp = (rp - (p[W_RHOP] - m[W_RHOP])) * kh;
    dms = (dms - (dfloat2(pair_m<A>(p), sfun(3)) - dfloat2(pair_m<A>(m), sfun(0)))) * dfloat2(c.hc2[A], c.t2[A]);
    // 4/3 e on u_A: Laplacian and one third of Eq. 7
    const dfloat e = c.e2[A], f = c.f2[A];
    l01 = ((p[W_U01] + m[W_U01]) - l01) * dfloat2(A == 0 ? f : e, A == 1 ? f : e);
    l2t = ((p[W_U2T] + m[W_U2T]) - l2t) * dfloat2(A == 2 ? f : e, e);
    g = (g - (cross(p) - cross(m))) * dfloat2(c.c2[A]);
  }
  t.m01 = t.m01 + cm01;
  t.m2e = t.m2e + cm2e;
  t.rho = t.rho + (dms.a() + ua * rp.a());
  const dfloat up = ua * rp.b();
  if (A == 0) t.m01 = dfloat2(t.m01.a() + rp.b(), t.m01.b());
  if (A == 1) t.m01 = dfloat2(t.m01.a(), t.m01.b() + rp.b());
  if (A == 2)
    t.m2e = t.m2e + dfloat2(rp.b(), -up);
  else
    t.m2e = dfloat2(t.m2e.a(), t.m2e.b() - up);
  t.v01 = t.v01 + l01;
  t.v2t = t.v2t + l2t;
  if (A == 0) t.v01 = dfloat2(t.v01.a() + dms.b(), t.v01.b());
  if (A == 1) t.v01 = dfloat2(t.v01.a(), t.v01.b() + dms.b());
  if (A == 2) t.v2t = dfloat2(t.v2t.a() + dms.b(), t.v2t.b());
  if (A == 0) {  // D_x u1, D_x u2
    t.a01 = g.a();
    t.a02 = g.b();
    if (WITH_KE) {
      t.w01 = -g.a();
      t.w02 = -g.b();
    }
  } else if (A == 1) {  // D_y u0, D_y u2
    t.a01 = t.a01 + g.a();
    t.a12 = g.b();
    if (WITH_KE) {
      t.w01 = t.w01 + g.a();
      t.w12 = -g.b();
    }
  } else {  // D_z u0, D_z u1
    t.a02 = t.a02 + g.a();
    t.a12 = t.a12 + g.b();
    if (WITH_KE) {
      t.w02 = t.w02 + g.a();
      t.w12 = t.w12 + g.b();
    }
  }
}

// Eqs. 1-3 from the terms, the centre record and the diagonal gradients
// (d00, d11), d22 and d00 + d11.
__device__ __forceinline__ void assemble_dw(const DwTerms& t, const dfloat2 (&cen)[NW], dfloat2 d01, dfloat d22,
                                            dfloat d0p1, const Coef<dfloat>& c, dfloat (&R)[5]) {
  const dfloat div = d0p1 + d22;
  const dfloat hdiv = dw_scale(div, -0.5f);
  R[0] = t.rho + (dfloat(1.0f, 0.0f) + cen[W_RHOP].a()) * hdiv;
  const dfloat Ec = cen[W_M2H].b() - cen[W_RHOP].b();
  const dfloat2 h2(hdiv);
  const dfloat2 r01 = (t.m01 + cen[W_M01] * h2) + t.v01 * dfloat2(c.inv_re);
  const dfloat2 r2e = (t.m2e + dfloat2(cen[W_M2H].a(), Ec) * h2) + t.v2t * dfloat2(c.inv_re, c.kappa);
  R[1] = r01.a();
  R[2] = r01.b();
  R[3] = r2e.a();
  // viscous dissipation and the work of the viscous force
  const dfloat2 a0(t.a01, t.a02), dd(d22, t.a12);
  const dfloat2 sq = (a0 * a0 + cen[W_U01] * t.v01) + dw_scale(d01 * d01, 2.0f);
  const dfloat2 s2 = dd * dd;
  dfloat q = (sq.a() + sq.b()) + (dw_scale(s2.a(), 2.0f) + s2.b());
  q = q + (cen[W_U2T].a() * t.v2t.a() - dfloat(2.0 / 3.0) * div * div);
  R[4] = r2e.b() + (c.inv_re * q - c.H0 * div);
}

// TIN: type of the stage input in HBM; TOUT: type of the stage output.
// CTAs per SM the launch bounds plan for: shared memory allows two 32 x 8
// binary32 CTAs per SM with the 5-slot ring (113 KiB each) and three with
// the TMEM queue and 3-slot ring (59 KiB each, row pairs: 168 registers); binary64 and
// double-float 16 x 8 tiles (107 KiB, 255 registers of four warps) two; 32 x 16
// tiles take one.
template <typename T, int TY, bool ZT = false>
constexpr int fused_min_blocks() {
  if (is_f64_class<T>()) return 2;
  return ((sizeof(T) == 4 && TY <= 8) || row_pairs<T, ZT>()) ? (ZT ? 3 : 2) : 1;
}
// tile width in points: the threads of a row, times the columns per thread
template <typename T, bool ZT>
constexpr int tile_width() {
  return row_pairs<T, ZT>() ? TX : tile_x<T>() * Lanes<T>::N;
}

// The z march of one CTA over the tile_width x TY column tile (bx, by), output
// planes [zbeg, min(zend, n2)), for the grid and stage described by `a`.
// Adds the stage input's kinetic energy and enstrophy of the tile's points
// to ke_acc / ens_acc when WITH_KE.  Ends with a barrier, so the shared
// memory can be reused by the caller.
template <typename T, typename TIN, typename TOUT, int TY, bool RHS_ONLY, bool WITH_KE, bool DF = false,
          bool ZT = false>
__device__ __forceinline__ void fused_march(const StageArgs& a, const Coef<T>& c, int bx, int by, int zbeg, int zend_req,
                                            FusedSmem<T, TY, ZT>& sm, double& ke_acc, double& ens_acc,
                                            uint32_t tmem_base = 0, uint32_t tmem_base2 = 0) {
  using S = FusedSmem<T, TY, ZT>;
  constexpr bool MIXZ = S::MIXZ;
  constexpr bool DW = std::is_same<T, dfloat>::value;     // double-float: terms in pairs
  constexpr bool FIXED = std::is_same<T, double>::value;  // binary64: linear stencils in integers
  constexpr int SY = S::SY;
  constexpr bool RP = S::RP;
  constexpr int TX = S::TX, SX = S::SX, HR = S::HR, NR = S::NR;
  constexpr int NT = TX * NR;
  constexpr int PTS = SX * SY;
  constexpr int NHALO = PTS - NT;                  // haloed points outside the tile
  constexpr int LPT = 1 + (NHALO + NT - 1) / NT;   // own point + halo points per thread

  constexpr int PP = Lanes<T>::N;  // points per thread: columns tx and tx + 32, or (RP) rows 2 ty and 2 ty + 1
  const int n0 = a.g.n0, n1 = a.g.n1, n2 = a.g.n2;
  const unsigned plane = (unsigned)n0 * (unsigned)n1;
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int x0 = bx * tile_width<T, ZT>(), y0 = by * TY;
  const int zend = min(zend_req, n2);
  bool valid[PP];
  unsigned own[PP];
#pragma unroll
  for (int j = 0; j < PP; ++j) {
    const int gx = x0 + tx + (RP ? 0 : TX * j);
    const int gy = y0 + (RP ? 2 * ty + j : ty);
    valid[j] = (gx < n0) && (gy < n1);
    own[j] = valid[j] ? (unsigned)gx + (unsigned)n0 * (unsigned)gy : 0u;
  }
  // per-field base pointers; offsets inside a field are 32-bit (P < 2^32)
  const TIN* qf[NF];
  const double* accf[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    qf[f] = static_cast<const TIN*>(a.q_in) + (long long)f * a.g.P;
    accf[f] = a.acc_in ? a.acc_in + (long long)f * a.g.P : nullptr;
  }

  // points this thread loads on every plane (periodic wrap): its own tile
  // point first, then at most LPT-1 points of the halo ring (the two rows
  // above and below the tile at full haloed width, then the two columns on
  // each side of the tile rows)
  int ld_off[LPT][PP], ld_s[LPT];
#pragma unroll
  for (int l = 0; l < LPT; ++l) {
    int sy = -1, sx = -1;
    if (l == 0) {
      sy = ty + HR;
      sx = tx + HALO;
    } else {
      const int h = tid + (l - 1) * NT;
      if (h < 2 * HR * SX) {
        const int r = h / SX;
        sy = (r < HR) ? r : NR + r;
        sx = h % SX;
      } else if (h < NHALO) {
        const int h2 = h - 2 * HR * SX;
        const int k = h2 & 3;
        sy = HR + (h2 >> 2);
        sx = (k < 2) ? k : TX + k;
      }
    }
    if (sy >= 0) {
#pragma unroll
      for (int j = 0; j < PP; ++j)
        ld_off[l][j] = wrapi(x0 - HALO + sx + (RP ? 0 : TX * j), n0) +
                       n0 * wrapi(y0 - HALO + (RP ? 2 * sy + j : sy), n1);
      ld_s[l] = sy * SX + sx;
    } else {
#pragma unroll
      for (int j = 0; j < PP; ++j) ld_off[l][j] = -1;
      ld_s[l] = 0;
    }
  }

  const int nplanes = zend - zbeg;
  const int nit = nplanes + 4;
  // the window address is warp-uniform; broadcasting lane 0's copy lets the
  // compiler keep it in a uniform register for the tcgen05 operands
  const uint32_t twin = ZT ? __shfl_sync(0xffffffffu, tmem_window<T>(tmem_base), 0) : 0u;
  const uint32_t twin2 = (ZT && MIXZ) ? __shfl_sync(0xffffffffu, tmem_window2<T>(tmem_base2), 0) : 0u;
  T d22 = T(0);
  T g00c = T(0), g11c = T(0);  // D1_x u0, D1_y u1 at the centre point

  // halo tasks of phase 2b, fixed for the whole z march: s_0 on the x0-halo
  // columns (4*TY points) and s_1 on the x1-halo rows (4*TX points)
  constexpr int NHT = 4 * NR + 2 * HR * TX;
  constexpr int HPT = (NHT + NT - 1) / NT;  // tasks per thread
  int hk[HPT], hxy[HPT], hdst[HPT];         // kind (0 none, 1 s_0, 2 s_1), packed (hy, hx), buffer index
#pragma unroll
  for (int j = 0; j < HPT; ++j) {
    const int h = tid + j * NT;
    if (h < 4 * NR) {
      const int r = h >> 2, k = h & 3;
      const int hx = (k < 2) ? k : TX + k;  // 0, 1, TX+2, TX+3
      hk[j] = 1;
      hxy[j] = ((r + HR) << 8) | hx;
      hdst[j] = r * SX + hx;
    } else if (h < NHT) {
      const int h2 = h - 4 * NR;
      const int col = h2 % TX, k = h2 / TX;
      const int hy = (k < HR) ? k : NR + k;
      hk[j] = 2;
      hxy[j] = (hy << 8) | (col + HALO);
      hdst[j] = hy * TX + col;
    } else {
      hk[j] = 0;
      hxy[j] = 0;
      hdst[j] = 0;
    }
  }
  // ring slots of planes e-4 .. e (e = entering plane), rotated each iteration
  int rs[NSLOT];
#pragma unroll
  for (int k = 0; k < NSLOT; ++k) rs[k] = (k + 1) % NSLOT;  // any permutation; warm-up fills all slots
  // full-record slots (ZT; otherwise the ring slots): planes e-2, e-1, e, and
  // e-3 in front of them when there are four
  constexpr int NFULL = S::NFULL;
  constexpr bool LAST_BARRIER = !ZT || NFULL < 4;  // the barrier that ends each plane
  int rf[ZT ? NFULL : 1];
#pragma unroll
  for (int k = 0; k < (ZT ? NFULL : 1); ++k) rf[k] = (k + 1) % (ZT ? NFULL : 1);
  // binary32 helper-buffer slots of planes e-2, e-1, e
  int rb[3] = {1, 2, 0};

  using Loads = TIN[LPT][NF][PP];
  Loads pf;
  int zl = wrapi(zbeg - HALO, n2);  // next plane to load (periodic), advanced one plane per load
  auto issue_loads = [&](Loads& pf) {
    const unsigned zoff = (unsigned)zl * plane;
    zl = (zl + 1 == n2) ? 0 : zl + 1;
#pragma unroll
    for (int l = 0; l < LPT; ++l) {
      if (l == 0 || ld_off[l][0] >= 0) {  // the own point always exists
#pragma unroll
        for (int j = 0; j < PP; ++j) {
          const unsigned o = zoff + (unsigned)ld_off[l][j];
#pragma unroll
          for (int f = 0; f < NF; ++f) pf[l][f][j] = qf[f][o];
        }
      }
    }
  };

  // A plane enters in three parts.  Its slots:
  auto rotate = [&]() {
    {
      const int t0 = rs[0];
#pragma unroll
      for (int k = 0; k < NSLOT - 1; ++k) rs[k] = rs[k + 1];
      rs[NSLOT - 1] = t0;
    }
    if constexpr (ZT) {
      const int t0 = rf[0];
#pragma unroll
      for (int k = 0; k < NFULL - 1; ++k) rf[k] = rf[k + 1];
      rf[NFULL - 1] = t0;
    }
    if constexpr (MIXZ) {
      const int t0 = rb[0];
      rb[0] = rb[1];
      rb[1] = rb[2];
      rb[2] = t0;
    }
  };
  // ---------------------------------------------------------------- phase 1
  // derive primitives (Eqs. 4-5 in deviation form) on the haloed tile from the
  // loaded Q' into ring slot se (full-record slot fe).
  auto convert = [&](const Loads& pf, int se, int fe) {
    {
      T* ring = &sm.ring[fe][0][0][0];
#pragma unroll
      for (int l = 0; l < LPT; ++l) {
        if (l == 0 || ld_off[l][0] >= 0) {  // the own point is always loaded
          T rec[NV];
          const T rho_p = from_lanes<T, TIN>(pf[l][0]);
          const T m0 = from_lanes<T, TIN>(pf[l][1]);
          const T m1 = from_lanes<T, TIN>(pf[l][2]);
          const T m2 = from_lanes<T, TIN>(pf[l][3]);
          const T E_p = from_lanes<T, TIN>(pf[l][4]);
          const T rinv = recip<T>(T(1) + rho_p);
          const T u0 = m0 * rinv, u1 = m1 * rinv, u2 = m2 * rinv;
          const T mu = mad(m2, u2, mad(m1, u1, m0 * u0));
          const T p2 = c.gm1x2 * mad(T(-0.5), mu, E_p);  // Eq. 4: 2 (p - p_ref)
          const T T_p = mad(c.hgM2, p2, -rho_p) * rinv;  // Eq. 5: T - 1
          rec[V_RHO] = rho_p;
          rec[V_M0] = m0;
          rec[V_M1] = m1;
          rec[V_M2] = m2;
          rec[V_H] = add_nc(E_p, p2);
          rec[V_U0] = u0;
          rec[V_U1] = u1;
          rec[V_U2] = u2;
          rec[V_P] = p2;
          rec[V_T] = T_p;
          store_rec(ring + ld_s[l] * NV, rec);
          if constexpr (S::U2) (&sm.u2ring[se][0][0])[ld_s[l]] = u2;
          if constexpr (ZT) {
            if (l == 0) {  // every thread
              tmem_converge<ZT>();
              tmem_store_rec(twin, se, rec);
            }
          }
        }
      }
    }
  };
  // --------------------------------------------------------------- phase 2a
  // in-plane diagonal gradients of the entering plane, kept for s_2 and
  // for the velocity gradient when the plane is the centre.
  auto gradients = [&](int se, int fe, int sbe) {
    if constexpr (DW) {
      const dfloat* r = &sm.ring[fe][ty + HALO][tx + HALO][0];
      dfloat2 g[4];  // u0 of the x0 neighbours beside u1 of the x1 neighbours
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int o = k < 2 ? k - 2 : k - 1;
        g[k] = dfloat2(rec_value(r + o * NV, V_U0), rec_value(r + o * SX * NV, V_U1));
      }
      const dfloat2 dg = dw_first(g[0], g[1], g[2], g[3], dfloat2(c.c2[0], c.c2[1]));
      if constexpr (ZT) {
        tmem_store_diag(twin, se, dg.a(), dg.b());  // this thread's column only
      } else {
        sm.dring[se][0][ty][tx] = dg.a();
        sm.dring[se][1][ty][tx] = dg.b();
      }
    } else if constexpr (FIXED) {
      const T(*R)[SX][NV] = sm.ring[fe];
      const int sy = ty + HALO, sx = tx + HALO;
      const T d00 = c.c2[0] * stencil_first(R[sy][sx - 2][V_U0], R[sy][sx - 1][V_U0], R[sy][sx + 1][V_U0],
                                            R[sy][sx + 2][V_U0]);
      const T d11 = c.c2[1] * stencil_first(R[sy - 2][sx][V_U1], R[sy - 1][sx][V_U1], R[sy + 1][sx][V_U1],
                                            R[sy + 2][sx][V_U1]);
      tmem_converge<ZT>();
      if constexpr (ZT) {
        tmem_store_diag(twin, se, d00, d11);  // this thread's column only
      } else {
        sm.dring[se][0][ty][tx] = d00;
        sm.dring[se][1][ty][tx] = d11;
      }
    } else {
      const T(*R)[SX][NV] = sm.ring[fe];
      const int sy = ty + HR, sx = tx + HALO;
      const T d00 = mad(c.c1[0], R[sy][sx + 1][V_U0] - R[sy][sx - 1][V_U0],
                        -c.c2[0] * (R[sy][sx + 2][V_U0] - R[sy][sx - 2][V_U0]));
      // u1 and u2 of the x1 neighbours (adjacent fields: one 8-byte load each
      // in binary32, whose records sit at 8-byte multiples)
      T y1[4], y2[4];
      if constexpr (RP) {
        f32x2 u1[3], u2[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float4 v = *reinterpret_cast<const float4*>(&R[sy + k - 1][sx][V_U1]);
          u1[k] = f32x2(v.x, v.y);
          u2[k] = f32x2(v.z, v.w);
        }
        y1[0] = u1[0], y1[1] = next_row(u1[0], u1[1]), y1[2] = next_row(u1[1], u1[2]), y1[3] = u1[2];
        y2[0] = u2[0], y2[1] = next_row(u2[0], u2[1]), y2[2] = next_row(u2[1], u2[2]), y2[3] = u2[2];
      } else {
        const int oy[4] = {-2, -1, 1, 2};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if constexpr (std::is_same<T, float>::value && MIXZ) {
            const float2 v = *reinterpret_cast<const float2*>(&R[sy + oy[k]][sx][V_U1]);
            y1[k] = v.x;
            y2[k] = v.y;
          } else {
            y1[k] = R[sy + oy[k]][sx][V_U1];
            y2[k] = R[sy + oy[k]][sx][V_U2];
          }
        }
      }
      const T d11 = mad(c.c1[1], y1[2] - y1[1], -c.c2[1] * (y1[3] - y1[0]));
      if constexpr (ZT) {
        tmem_store_diag(twin, se, d00, d11);  // this thread's column only
      } else {
        sm.dring[se][0][ty][tx] = d00;
        sm.dring[se][1][ty][tx] = d11;
      }
      if constexpr (MIXZ) {
        // binary32: the in-plane gradients of u2 (for D1_z of them at the
        // centre, from this thread's own column) and the helpers D1_y u1 on
        // the x0-haloed rows and D1_x u0 on the x1-haloed columns of the
        // entering plane, read when it becomes the centre
        const T d02 = mad(c.c1[0], R[sy][sx + 1][V_U2] - R[sy][sx - 1][V_U2],
                          -c.c2[0] * (R[sy][sx + 2][V_U2] - R[sy][sx - 2][V_U2]));
        const T d12 = mad(c.c1[1], y2[2] - y2[1], -c.c2[1] * (y2[3] - y2[0]));
        if constexpr (ZT) {
          tmem_store_xdiag(twin2, se, d02, d12);
        } else {
          sm.dring[se][2][ty][tx] = d02;
          sm.dring[se][3][ty][tx] = d12;
        }
        sm.s0buf[sbe][ty][sx] = d11;
        sm.s1buf[sbe][sy][tx] = d00;
#pragma unroll
        for (int j = 0; j < HPT; ++j) {
          const int hy = hxy[j] >> 8, hx = hxy[j] & 0xFF;
          if (hk[j] == 1) {
            T m2, m1, p1, p2;
            if constexpr (RP) {
              const T o = R[hy][hx][V_U1];
              m2 = R[hy - 1][hx][V_U1];
              p2 = R[hy + 1][hx][V_U1];
              m1 = next_row(m2, o);
              p1 = next_row(o, p2);
            } else {
              m2 = R[hy - 2][hx][V_U1];
              m1 = R[hy - 1][hx][V_U1];
              p1 = R[hy + 1][hx][V_U1];
              p2 = R[hy + 2][hx][V_U1];
            }
            (&sm.s0buf[sbe][0][0])[hdst[j]] = mad(c.c1[1], p1 - m1, -c.c2[1] * (p2 - m2));
          } else if (hk[j] == 2) {
            (&sm.s1buf[sbe][0][0])[hdst[j]] = mad(c.c1[0], R[hy][hx + 1][V_U0] - R[hy][hx - 1][V_U0],
                                                  -c.c2[0] * (R[hy][hx + 2][V_U0] - R[hy][hx - 2][V_U0]));
          }
        }
      }
    }
  };
  auto full_slot = [&]() { return ZT ? rf[ZT ? NFULL - 1 : 0] : rs[NSLOT - 1]; };  // of the entering plane

  // The first FILL planes enter together: their loads are in flight at the same
  // time and two barriers serve them all, where one plane after another paid
  // the latency of memory and of both phases for each.  Double-float 256^3 2.204
  // -> 2.091 ms a stage, 64^3 44.6 -> 42.3 us (the same code shape schedules
  // better in its full iterations too), binary64 and binary32 rings 1 to 4 % at
  // 16^3 ... 40^3.  Two columns per thread have no registers for it, nor has
  // the binary32 TMEM queue (the batch kernel spills, 1 % slower; 0.5 % faster alone).
  constexpr int FILL = PP == 2 || (sizeof(T) == 4 && ZT) ? 0 : (ZT ? 3 : 4);
  if constexpr (FILL > 0) {
    Loads pb[FILL > 0 ? FILL : 1];
    int se[FILL > 0 ? FILL : 1], fe[FILL > 0 ? FILL : 1], sbe[FILL > 0 ? FILL : 1];
#pragma unroll
    for (int p = 0; p < FILL; ++p) issue_loads(pb[p]);
#pragma unroll
    for (int p = 0; p < FILL; ++p) {
      rotate();
      se[p] = rs[NSLOT - 1];
      fe[p] = full_slot();
      sbe[p] = rb[2];
      convert(pb[p], se[p], fe[p]);
    }
    issue_loads(pf);
    __syncthreads();
#pragma unroll
    for (int p = 0; p < FILL; ++p) gradients(se[p], fe[p], sbe[p]);
    if constexpr (ZT) __syncthreads();  // the next plane's records replace the first one's
  } else {
    issue_loads(pf);
  }

  for (int it = FILL; it < nit; ++it) {
    // plane e = zbeg - 2 + it enters
    rotate();
    convert(pf, rs[NSLOT - 1], full_slot());
    if (it + 1 < nit) issue_loads(pf);
    __syncthreads();
    gradients(rs[NSLOT - 1], full_slot(), rb[2]);
    if (it < 4) continue;  // ring not yet full; slots written so far are not read again before the next sync

    const int zc = zbeg + it - 4;  // centre plane
    // slot of plane zc + o, o = -2..2
    const int sl[5] = {rs[0], rs[1], rs[2], rs[3], rs[4]};
    const int scen = sl[2];
    const int fc = ZT ? rf[ZT ? NFULL - 3 : 0] : scen;  // full-record slot of the centre plane
    unsigned oc[PP];  // offsets of the thread's centre points
#pragma unroll
    for (int j = 0; j < PP; ++j) oc[j] = (unsigned)zc * plane + own[j];

    // accumulator of the centre points (fetched as phase 3 starts, so that
    // its latency overlaps the derivative terms)
    double accv[NF][PP];
    float dhi[NF][PP], dlo[NF][PP];  // double-float accumulator (DF mode)
    auto fetch_acc = [&]() {
      if (!RHS_ONLY) {
#pragma unroll
        for (int j = 0; j < PP; ++j) {
          if (!valid[j]) continue;
          if (DF) {
#pragma unroll
            for (int f = 0; f < NF; ++f) {
              dhi[f][j] = a.dacc_in[(long long)f * a.g.P + oc[j]];
              dlo[f][j] = a.dacc_in[(long long)(NF + f) * a.g.P + oc[j]];
            }
          } else {
#pragma unroll
            for (int f = 0; f < NF; ++f) accv[f][j] = accf[f][oc[j]];
          }
        }
      }
    };

    // --------------------------------------------------------------- phase 2b
    // binary64 / double-float: s_0 and s_1 on the centre plane's tile and
    // halo; binary32 has its helpers already (phase 2a of the plane's entry)
    // and needs only the centre's in-plane gradients.
    if constexpr (MIXZ) {
      d22 = T(0);
      tmem_converge<ZT>();
      if constexpr (ZT) {
        tmem_load_diag(twin, scen, g00c, g11c);
      } else {
        g00c = sm.dring[scen][0][ty][tx];
        g11c = sm.dring[scen][1][ty][tx];
      }
    } else {
      auto u2at = [&](int slot, int yy, int xx) {
        if constexpr (ZT)
          return sm.u2ring[slot][yy][xx];
        else
          return rec_value(&sm.ring[slot][yy][xx][0], V_U2);
      };
      if constexpr (DW) {
        const int sy = ty + HALO, sx = tx + HALO;
        const int zs[4] = {sl[0], sl[1], sl[3], sl[4]};
        if constexpr (ZT) {
          tmem_load_diag(twin, scen, g00c, g11c);
        } else {
          g00c = sm.dring[scen][0][ty][tx];
          g11c = sm.dring[scen][1][ty][tx];
        }
        d22 = (dw_scale(u2at(zs[2], sy, sx) - u2at(zs[1], sy, sx), 8.0f) - (u2at(zs[3], sy, sx) - u2at(zs[0], sy, sx))) *
              c.c2[2];
        const dfloat2 s = dfloat2(g11c, g00c) + dfloat2(d22);
        sm.s0buf[0][ty][sx] = s.a();
        sm.s1buf[0][sy][tx] = s.b();
        const dfloat* R = &sm.ring[fc][0][0][0];
#pragma unroll
        for (int j = 0; j < HPT; ++j) {
          if (hk[j] == 0) continue;
          // kind 1: D1_y u1 (s_0), kind 2: D1_x u0 (s_1), beside D1_z u2
          const int hy = hxy[j] >> 8, hx = hxy[j] & 0xFF;
          const bool k1 = hk[j] == 1;
          const dfloat* q = R + (hy * SX + hx) * NV;
          const int st = NV * (k1 ? SX : 1);
          dfloat2 g[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const dfloat2 v = load_pair(q + (k < 2 ? k - 2 : k - 1) * st, W_U01);
            g[k] = dfloat2(k1 ? v.b() : v.a(), u2at(zs[k], hy, hx));
          }
          const dfloat2 dg = dw_first(g[0], g[1], g[2], g[3], dfloat2(k1 ? c.c2[1] : c.c2[0], c.c2[2]));
          (k1 ? &sm.s0buf[0][0][0] : &sm.s1buf[0][0][0])[hdst[j]] = dg.a() + dg.b();
        }
      } else {
        const int sy = ty + HALO, sx = tx + HALO;
        auto u2z = [&](int yy, int xx) {
          return c.c2[2] * stencil_first(u2at(sl[0], yy, xx), u2at(sl[1], yy, xx), u2at(sl[3], yy, xx), u2at(sl[4], yy, xx));
        };
        d22 = u2z(sy, sx);
        tmem_converge<ZT>();
        if constexpr (ZT) {
          tmem_load_diag(twin, scen, g00c, g11c);
        } else {
          g00c = sm.dring[scen][0][ty][tx];
          g11c = sm.dring[scen][1][ty][tx];
        }
        sm.s0buf[0][ty][sx] = add_nc(g11c, d22);
        sm.s1buf[0][sy][tx] = add_nc(g00c, d22);
#pragma unroll
        for (int j = 0; j < HPT; ++j) {
          if (hk[j] == 0) continue;
          // kind 1: D1_y u1 (s_0), kind 2: D1_x u0 (s_1)
          const int hy = hxy[j] >> 8, hx = hxy[j] & 0xFF;
          const bool k1 = hk[j] == 1;
          const T* q = &sm.ring[fc][hy][hx][k1 ? V_U1 : V_U0];
          const int st = k1 ? SX * NV : NV;
          const T dd = (k1 ? c.c2[1] : c.c2[0]) * stencil_first(q[-2 * st], q[-st], q[st], q[2 * st]);
          (k1 ? &sm.s0buf[0][0][0] : &sm.s1buf[0][0][0])[hdst[j]] = add_nc(dd, u2z(hy, hx));
        }
      }
      __syncthreads();
    }
    // ---------------------------------------------------------------- phase 3
    {
      fetch_acc();
      tmem_converge<ZT>();
      const int sy = ty + HR, sx = tx + HALO;
      const T(*C)[SX][NV] = sm.ring[fc];
      T rho_p, mc[3], uc[3];  // centre values

      // neighbours k = 0..3 (offsets -2, -1, +1, +2): records and mixed-term helpers
      const int sbc = MIXZ ? rb[0] : 0;  // helper buffers of the centre plane
      const int off[4] = {-2, -1, 1, 2};
      const int zs[4] = {sl[0], sl[1], sl[3], sl[4]};
      auto sf0 = [&](int k) { return sm.s0buf[sbc][ty][sx + off[k]]; };
      auto sf1 = [&](int k) {
        if constexpr (RP) {
          const int q = k < 2 ? sy - 1 : sy;
          if (k == 0) return sm.s1buf[sbc][sy - 1][tx];
          if (k == 3) return sm.s1buf[sbc][sy + 1][tx];
          return next_row(sm.s1buf[sbc][q][tx], sm.s1buf[sbc][q + 1][tx]);
        } else {
          return sm.s1buf[sbc][sy + off[k]][tx];
        }
      };
      auto sf2 = [&](int k) {
        if constexpr (ZT) {
          T a, b;
          tmem_load_diag(twin, zs[k], a, b);
          return a + b;
        } else {
          return sm.dring[zs[k]][0][ty][tx] + sm.dring[zs[k]][1][ty][tx];
        }
      };
      // binary32: D1_x u2 and D1_y u2 of the x2 neighbours
      auto xf = [&](int k, T& d02, T& d12) {
        if constexpr (MIXZ) {
          if constexpr (ZT) {
            tmem_load_xdiag(twin2, zs[k], d02, d12);
          } else {
            d02 = sm.dring[zs[k]][2][ty][tx];
            d12 = sm.dring[zs[k]][3][ty][tx];
          }
        }
      };

      T R[5];
      T w0 = T(0), w1 = T(0), w2 = T(0);  // vorticity (WITH_KE)
      // x0 group first (SN2 ordering), then x1, x2
      if constexpr (DW) {
        auto lp0 = [&](int k, dfloat2(&r)[NW]) { load_pairs(&C[sy][sx + off[k]][0], r); };
        auto lp1 = [&](int k, dfloat2(&r)[NW]) { load_pairs(&C[sy + off[k]][sx][0], r); };
        auto lp2 = [&](int k, dfloat2(&r)[NW]) {
          if constexpr (ZT)
            tmem_load_pairs(twin, zs[k], r);
          else
            load_pairs(&sm.ring[zs[k]][sy][sx][0], r);
        };
        dfloat2 cen[NW];
        if constexpr (ZT)
          tmem_load_pairs(twin, scen, cen);
        else
          load_pairs(&C[sy][sx][0], cen);
        const dfloat ua[3] = {cen[W_U01].a(), cen[W_U01].b(), cen[W_U2T].a()};
        DwTerms t;
        t.m01 = t.m2e = dfloat2(dfloat(0.0f, 0.0f));
        t.rho = dfloat(0.0f, 0.0f);
        t.v01 = dfloat2(c.v0[0], c.v0[1]) * cen[W_U01];
        t.v2t = dfloat2(c.v0[2], c.e0s) * cen[W_U2T];
        axis_terms_dw<0, WITH_KE>(lp0, sf0, c, ua[0], t);
        axis_terms_dw<1, WITH_KE>(lp1, sf1, c, ua[1], t);
        axis_terms_dw<2, WITH_KE>(lp2, sf2, c, ua[2], t);
        assemble_dw(t, cen, dfloat2(g00c, g11c), d22, g00c + g11c, c, R);
        if (WITH_KE) {
          rho_p = cen[W_RHOP].a();
          mc[0] = cen[W_M01].a();
          mc[1] = cen[W_M01].b();
          mc[2] = cen[W_M2H].a();
#pragma unroll
          for (int i = 0; i < 3; ++i) uc[i] = ua[i];
          w0 = t.w12;  // squared below: the sign does not matter
          w1 = t.w02;
          w2 = t.w01;
        }
      } else {
        auto ld0 = [&](int k, T(&r)[NV]) { load_rec(&C[sy][sx + off[k]][0], r); };
        T cen[NV];
        T yp[RP ? NV : 1];  // row pairs: the pair above, then the one below
        auto ld1 = [&](int k, T(&r)[NV]) {
          if constexpr (RP) {  // rows y + off, y + 1 + off: a pair, or halves of two
            if (k == 0) load_rec(&C[sy - 1][sx][0], yp);
            if (k == 2) load_rec(&C[sy + 1][sx][0], yp);
#pragma unroll
            for (int v = 0; v < NV; ++v)
              r[v] = k == 1 ? next_row(yp[v], cen[v]) : k == 2 ? next_row(cen[v], yp[v]) : yp[v];
          } else {
            load_rec(&C[sy + off[k]][sx][0], r);
          }
        };
        auto ld2 = [&](int k, T(&r)[NV]) {
          if constexpr (ZT)
            tmem_load_rec(twin, zs[k], r);
          else
            load_rec(&sm.ring[zs[k]][sy][sx][0], r);
        };
        if constexpr (ZT)
          tmem_load_rec(twin, scen, cen);
        else
          load_rec(&C[sy][sx][0], cen);
        rho_p = cen[V_RHO];
        const T Ec = cen[V_H] - cen[V_P];
        const T Tc = cen[V_T];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          mc[i] = cen[V_M0 + i];
          uc[i] = cen[V_U0 + i];
        }
        StreamTerms<T> t;
        t.rrho = t.rE = T(0);
        t.lapT = c.e0s * Tc;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          t.rM[i] = t.a[i] = t.lo[i] = T(0);
          t.v[i] = c.v0[i] * uc[i];
        }
        t.gd[0] = g00c;
        t.gd[1] = g11c;
        t.gd[2] = d22;
        // D1_i u_j, i < j, which axis i alone has put into the sum a when axis j starts (diagnostics)
        T hi[3];
        auto first_gradients = [&](int axis) {
          if (WITH_KE && axis == 0) hi[0] = t.a[0], hi[1] = t.a[1];
          if (WITH_KE && axis == 1) hi[2] = t.a[2];
        };
        if constexpr (FIXED) {
          auto at0 = [&](int k, T& x, T&) { x = sf0(k); };
          auto at1 = [&](int k, T& x, T&) { x = sf1(k); };
          auto at2 = [&](int k, T& x, T& y) {
            if constexpr (ZT) {
              tmem_load_diag(twin, zs[k], x, y);
            } else {
              x = sm.dring[zs[k]][0][ty][tx];
              y = sm.dring[zs[k]][1][ty][tx];
            }
          };
          axis_terms_fixed<0, WITH_KE>(ld0, at0, c, uc, t);
          first_gradients(0);
          axis_terms_fixed<1, WITH_KE>(ld1, at1, c, uc, t);
          first_gradients(1);
          tmem_converge<ZT>();
          axis_terms_fixed<2, WITH_KE>(ld2, at2, c, uc, t);
        } else {
          axis_terms_stream<0, false, WITH_KE>(ld0, sf0, c, uc, t);
          first_gradients(0);
          // shared-memory loads of one axis at a time: hoisted over the axes they spill at the binary32 ring
          // kernel's 128 registers (256^3: 674 us a stage without these two, 651 with)
          if constexpr (!ZT && sizeof(T) == 4) asm volatile("" ::: "memory");
          axis_terms_stream<1, false, WITH_KE, RP>(ld1, sf1, c, uc, t);
          first_gradients(1);
          if constexpr (!ZT && sizeof(T) == 4) asm volatile("" ::: "memory");
          axis_terms_stream<2, MIXZ, WITH_KE>(ld2, sf2, c, uc, t, xf);
        }
        assemble_streamed(t, rho_p, mc, Ec, uc, c, R);
        if (WITH_KE) {  // differences of two derivatives: D1_i u_j, i < j, and lo = D1_j u_i
          w2 = hi[0] - t.lo[0];
          w1 = t.lo[1] - hi[1];
          w0 = hi[2] - t.lo[2];
        }
      }

#pragma unroll
      for (int j = 0; j < PP; ++j) {
        if (!valid[j]) continue;
        const unsigned o = oc[j];
        TOUT qo[NF];
        if constexpr (RHS_ONLY) {
#pragma unroll
          for (int f = 0; f < NF; ++f) a.r_out[(long long)f * a.g.P + o] = double(lane(R[f], j));
        } else if constexpr (DF) {
          // binary32 stage, double-float accumulator (hi + lo, binary32
          // each): acc' = acc + (b dt R) by Dekker's Fast2Sum of hi and the
          // increment x = fl(b dt R), the error folded into lo; Q_{k+1} = hi'
          // + (lo' + (a - b) dt R).  Fast2Sum is exact when |hi| >= |x|;
          // otherwise (hi crossing zero) the pair misses hi + x by at most
          // about half an ulp of x, the size of the rounding x already
          // carries, so the accumulator keeps its precision where it
          // matters.  The pair (hi', lo') represents acc' whether or not it
          // is normalised; the last stage of a step renormalises it, so that
          // the state's hi fields are its binary32 rounding (the next step's
          // stage-0 input), the others leave it as it is.
          // Fields are updated two at a time with packed two-lane
          // instructions (the same correctly rounded binary32 operations as
          // one field at a time), the last field alone.
          const float bdt = a.b_dt32, ambdt = a.amb_dt32;
          float hi3[NF], lo3[NF], rr[NF];
#pragma unroll
          for (int f = 0; f < NF; ++f) rr[f] = float(lane(R[f], j));
          const float2 bdt2 = make_float2(bdt, bdt), ambdt2 = make_float2(ambdt, ambdt);
#pragma unroll
          for (int f = 0; f < NF; f += 2) {
            if (f + 1 < NF) {
              const float2 r2 = make_float2(rr[f], rr[f + 1]);
              const float2 h2 = make_float2(dhi[f][j], dhi[f + 1][j]);
              const float2 x2 = __fmul2_rn(bdt2, r2);
              const float2 s2 = __fadd2_rn(h2, x2);
              const float2 d2 = __fadd2_rn(s2, make_float2(-h2.x, -h2.y));
              const float2 e2 = __fadd2_rn(x2, make_float2(-d2.x, -d2.y));
              float2 l2 = __fadd2_rn(make_float2(dlo[f][j], dlo[f + 1][j]), e2);
              float2 hn = s2;
              if (a.df_normalize) {
                hn = __fadd2_rn(s2, l2);
                const float2 g2 = __fadd2_rn(hn, make_float2(-s2.x, -s2.y));
                l2 = __fadd2_rn(l2, make_float2(-g2.x, -g2.y));
              }
              const float2 q2 = __fadd2_rn(hn, __ffma2_rn(ambdt2, r2, l2));
              hi3[f] = hn.x;
              hi3[f + 1] = hn.y;
              lo3[f] = l2.x;
              lo3[f + 1] = l2.y;
              qo[f] = TOUT(q2.x);
              qo[f + 1] = TOUT(q2.y);
            } else {
              const float x = bdt * rr[f];
              const float s = __fadd_rn(dhi[f][j], x);
              const float err = __fsub_rn(x, __fsub_rn(s, dhi[f][j]));
              float h = s, l = __fadd_rn(dlo[f][j], err);
              if (a.df_normalize) {
                h = __fadd_rn(s, l);
                l = __fsub_rn(l, __fsub_rn(h, s));
              }
              hi3[f] = h;
              lo3[f] = l;
              qo[f] = TOUT(h + fmaf(ambdt, rr[f], l));
            }
          }
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            a.dacc_out[(long long)f * a.g.P + o] = hi3[f];
            a.dacc_out[(long long)(NF + f) * a.g.P + o] = lo3[f];
          }
        } else if constexpr (is_f64_class<T>()) {
          // binary64 (or double-float) stage: acc + b dt R and acc + a dt R,
          // binary64 fused multiply-adds
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            const double r = as_double(R[f]);
            a.acc_out[(long long)f * a.g.P + o] = fma(a.b_dt, r, accv[f][j]);
            qo[f] = to_output<TOUT>(fma(a.a_dt, r, accv[f][j]));
          }
        } else {
          // binary32 stage, binary64 accumulator: one DADD per field,
          //   acc' = acc + (b dt R),  Q_{k+1} = float(acc') + (a - b) dt R
          // (conversions by integer re-packing, fpconv.cuh; the narrowing
          // rounds to nearest, ties away from zero)
          const float bdt = a.b_dt32, ambdt = a.amb_dt32;
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            const float r = float(lane(R[f], j));
            const double accn = accv[f][j] + widen_f32_fast(bdt * r);
            a.acc_out[(long long)f * a.g.P + o] = accn;
            qo[f] = TOUT(narrow_f64_rna(accn) + ambdt * r);
          }
        }
        if constexpr (!RHS_ONLY) {
          if (a.q_out) {  // the stage field (absent on the last stage)
#pragma unroll
            for (int f = 0; f < NF; ++f) static_cast<TOUT*>(a.q_out)[(long long)f * a.g.P + o] = qo[f];
          }
        }
        if (WITH_KE) {
          const T ke_t = T(0.5) * mad(mc[2], uc[2], mad(mc[1], uc[1], mc[0] * uc[0]));
          const T ens_t = T(0.5) * (T(1) + rho_p) * mad(w2, w2, mad(w1, w1, w0 * w0));
          ke_acc += double(lane(ke_t, j));
          ens_acc += double(lane(ens_t, j));
        }
      }
    }
    // with four full-record slots the next plane writes the slot of plane
    // e-3, last read before this plane's first barrier
    if constexpr (LAST_BARRIER) __syncthreads();
  }
  if constexpr (!LAST_BARRIER) __syncthreads();  // the caller may reuse shared memory
}

// Fixed-order block reduction of (ke, ens) into out[0..1]: warp shuffles,
// then thread 0 over the warps.
template <int NT>
__device__ __forceinline__ void block_reduce_pair(double (&red)[2][32], double ke, double ens, double* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ke += __shfl_down_sync(0xffffffffu, ke, o);
    ens += __shfl_down_sync(0xffffffffu, ens, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = ke;
    red[1][threadIdx.x >> 5] = ens;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double k = 0.0, e = 0.0;
    for (int w = 0; w < NT / 32; ++w) {
      k += red[0][w];
      e += red[1][w];
    }
    out[0] = k;
    out[1] = e;
  }
  __syncthreads();
}

// How the work is split over CTAs.  Chunks: one CTA a (tile, z chunk).  Even
// split: every CTA takes a contiguous run of the planes of all tiles, numbered
// tile by tile (a run that crosses into the next tile starts a new march
// there), as many CTAs as fit the SMs at once, so that no SM idles in a last wave and a grid with
// fewer chunks than that still fills them.  The binary64-register kernels (two
// CTAs per SM, bound by arithmetic) choose by the longest CTA (plan_split); the
// binary32 kernels, bound by memory and its latency, keep the chunks:
// concurrent CTAs then march through the same planes and share their halos in
// L2.
template <typename T>
constexpr bool even_split() {
  return is_f64_class<T>();
}

// Single grid.  ZT: x2-neighbour records in TMEM.
template <typename T, typename TIN, typename TOUT, int TY, bool RHS_ONLY, bool WITH_KE, bool DF, bool ZT, bool EVEN>
__global__ void __launch_bounds__(FusedSmem<T, TY, ZT>::NTHREADS, fused_min_blocks<T, TY, ZT>())
    fused_stage_kernel(const StageArgs a, const Coef<T> c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FusedSmem<T, TY, ZT>& sm = *reinterpret_cast<FusedSmem<T, TY, ZT>*>(smem_raw);
  constexpr int NW = FusedSmem<T, TY, ZT>::NTHREADS / 32;  // warps
  constexpr int NCOL = tmem_columns<NW, T>();
  constexpr int NCOL2 = tmem_columns2<NW, T>();
  uint32_t tbase = 0, tbase2 = 0;
  if (ZT) tmem_acquire<NCOL, NCOL2>(sm.tmem_base, tbase, tbase2);
  double ke = 0.0, ens = 0.0;
  if constexpr (EVEN) {
    const int tiles_x = (a.g.n0 + tile_width<T, ZT>() - 1) / tile_width<T, ZT>(), tiles_y = (a.g.n1 + TY - 1) / TY;
    const long long units = (long long)tiles_x * tiles_y * a.g.n2;
    long long u = units * blockIdx.x / gridDim.x;
    const long long end = units * (blockIdx.x + 1) / gridDim.x;
    while (u < end) {
      const int tile = (int)(u / a.g.n2), z = (int)(u - (long long)tile * a.g.n2);
      const int len = (int)min((long long)(a.g.n2 - z), end - u);
      fused_march<T, TIN, TOUT, TY, RHS_ONLY, WITH_KE, DF, ZT>(a, c, tile % tiles_x, tile / tiles_x, z, z + len, sm,
                                                              ke, ens, tbase, tbase2);
      u += len;
    }
  } else {
    const int zbeg = blockIdx.z * a.zc;
    fused_march<T, TIN, TOUT, TY, RHS_ONLY, WITH_KE, DF, ZT>(a, c, blockIdx.x, blockIdx.y, zbeg, zbeg + a.zc, sm, ke,
                                                            ens, tbase, tbase2);
  }
  if (WITH_KE) {
    const long long b = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
    block_reduce_pair<32 * NW>(sm.red, ke, ens, a.ke_partials + 2 * b);
  }
  if (ZT) tmem_release<NCOL, NCOL2>(tbase, tbase2);
}

template <int TY, int W = TX>
inline dim3 fused_grid(const Geom& g, int zc) {
  return dim3((g.n0 + W - 1) / W, (g.n1 + TY - 1) / TY, (g.n2 + zc - 1) / zc);
}

// binary32 constants for two-lane arithmetic
inline Coef<f32x2> both_lanes(const Coef<float>& cf) {
  Coef<f32x2> c;
  for (int i = 0; i < 3; ++i) {
    c.c1[i] = f32x2(cf.c1[i], cf.c1[i]);
    c.c2[i] = f32x2(cf.c2[i], cf.c2[i]);
    c.e0[i] = f32x2(cf.e0[i], cf.e0[i]);
    c.e1[i] = f32x2(cf.e1[i], cf.e1[i]);
    c.e2[i] = f32x2(cf.e2[i], cf.e2[i]);
    c.hc1[i] = f32x2(cf.hc1[i], cf.hc1[i]);
    c.hc2[i] = f32x2(cf.hc2[i], cf.hc2[i]);
    c.t2[i] = f32x2(cf.t2[i], cf.t2[i]);
    c.f2[i] = f32x2(cf.f2[i], cf.f2[i]);
    c.v0[i] = f32x2(cf.v0[i], cf.v0[i]);
  }
  c.e0s = f32x2(cf.e0s, cf.e0s);
  c.gm1 = f32x2(cf.gm1, cf.gm1);
  c.gM2 = f32x2(cf.gM2, cf.gM2);
  c.gm1x2 = f32x2(cf.gm1x2, cf.gm1x2);
  c.hgM2 = f32x2(cf.hgM2, cf.hgM2);
  c.inv_re = f32x2(cf.inv_re, cf.inv_re);
  c.kappa = f32x2(cf.kappa, cf.kappa);
  c.H0 = f32x2(cf.H0, cf.H0);
  return c;
}

// The dynamic shared-memory limit is a per-device attribute of a kernel: set
// it on the current device the first time a kernel launches there (bit d of
// `done`).  Concurrent first launches may both set it, which is harmless.
template <typename K>
cudaError_t ensure_smem_limit(K kernel, size_t bytes, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

template <typename T, typename TIN, typename TOUT, int TY, bool RHS_ONLY, bool WITH_KE, bool DF, bool ZT, bool EVEN>
cudaError_t launch_fused_k(const StageArgs& a, const Coef<T>& c, cudaStream_t s) {
  auto k = fused_stage_kernel<T, TIN, TOUT, TY, RHS_ONLY, WITH_KE, DF, ZT, EVEN>;
  const size_t smem = sizeof(FusedSmem<T, TY, ZT>);
  static std::atomic<unsigned long long> done{0};  // devices this instantiation is configured on
  if (cudaError_t e = ensure_smem_limit(k, smem, done)) return e;
  const dim3 grid = EVEN ? dim3(a.ctas) : fused_grid<TY, tile_width<T, ZT>()>(a.g, a.zc);
  k<<<grid, FusedSmem<T, TY, ZT>::NTHREADS, smem, s>>>(a, c);
  return cudaGetLastError();
}

template <typename T, typename TIN, typename TOUT, int TY, bool RHS_ONLY, bool WITH_KE, bool DF = false,
          bool ZT = false>
cudaError_t launch_fused_t(const StageArgs& a, const Coef<T>& c, cudaStream_t s) {
  if constexpr (even_split<T>()) {
    if (a.even) return launch_fused_k<T, TIN, TOUT, TY, RHS_ONLY, WITH_KE, DF, ZT, true>(a, c, s);
  }
  return launch_fused_k<T, TIN, TOUT, TY, RHS_ONLY, WITH_KE, DF, ZT, false>(a, c, s);
}

}  // namespace sbli
