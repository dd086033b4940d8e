// storeall.cu -- the store-all ("BL") variant of §2.3.1 on the GPU, kept as
// the paper's memory-intensive comparison point.
//
// Exactly as the paper describes BL: (a) primitives and every product that
// is differentiated go to full-grid temporary arrays; (b) derivative
// kernels write each of the 60 distinct derivatives of Eqs. 1-3 to its own
// global array (Listing 1's derx; one launch for those of the fields, one for the
// mixed ones); (c) a residual kernel reads the arrays and assembles Eqs. 1-3;
// (d) the Runge-Kutta update of Fig. 1 runs as its own kernel.
//
// Variables are deviations from the reference state, as in the fused path.
#include <type_traits>

#include "primitives.cuh"
#include "sbli_internal.cuh"
#include "stencil_int.cuh"

namespace sbli {

namespace {

// scratch array indices (each P elements)
enum {
  A_U = 0,             // u_i                         3
  A_P = 3,             // p'                          1
  A_T = 4,             // T'                          1
  A_MU = 5,            // m_i u_j, symmetric pairs    6 (00,01,02,11,12,22)
  A_EU = 11,           // E' u_j                      3
  A_PU = 14,           // p' u_j                      3
  A_DRHOU = 17,        // D_j m_i        [i][j]       9
  A_DU = 26,           // D_j u_i        [i][j]       9
  A_DRHOUU = 35,       // D_j (m_i u_j)  [i][j]       9
  A_D2U = 44,          // D2_j u_i       [i][j]       9
  A_DDU = 53,          // D_i D_j u_j, i != j         6 (01,02,10,12,20,21)
  A_DRHO = 59,         // D_j rho'                    3
  A_DP = 62,           // D_j p'                      3
  A_DE = 65,           // D_j E'                      3
  A_DEU = 68,          // D_j (E' u_j)                3
  A_DPU = 71,          // D_j (p' u_j)                3
  A_D2T = 74,          // D2_j T'                     3
  A_R = 77,            // residual                    5
  A_COUNT = 82
};

__host__ __device__ inline int sym(int i, int j) {
  const int a = i < j ? i : j, b = i < j ? j : i;
  return a == 0 ? b : (a == 1 ? 2 + b : 5);  // (0,0)0 (0,1)1 (0,2)2 (1,1)3 (1,2)4 (2,2)5
}
__host__ __device__ inline int offd(int i, int j) { return 2 * i + (j > i ? j - 1 : j); }  // i != j -> 0..5

template <typename T, typename TIN>
__global__ void bl_primitives(Geom g, Coef<T> c, const TIN* __restrict__ q, T* __restrict__ s) {
  const long long P = g.P;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P; n += (long long)gridDim.x * blockDim.x) {
    const T rho_p = T(q[n]);
    const T m[3] = {T(q[P + n]), T(q[2 * P + n]), T(q[3 * P + n])};
    const T E_p = T(q[4 * P + n]);
    [[maybe_unused]] const T rho = T(1) + rho_p;
    T u[3], p_p, T_p;
    if constexpr (sizeof(T) == 8) {
      const Primitives r = primitives_f64(rho_p, m[0], m[1], m[2], E_p, c.gm1, c.gM2);
      for (int i = 0; i < 3; ++i) u[i] = r.u[i];
      p_p = r.p;
      T_p = r.t;
    } else {
      for (int i = 0; i < 3; ++i) u[i] = m[i] / rho;
      p_p = c.gm1 * (E_p - T(0.5) * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));  // Eq. 4
      T_p = (c.gM2 * p_p - rho_p) / rho;                                              // Eq. 5
    }
    for (int i = 0; i < 3; ++i) s[(A_U + i) * P + n] = u[i];
    s[A_P * P + n] = p_p;
    s[A_T * P + n] = T_p;
    for (int i = 0; i < 3; ++i)
      for (int j = i; j < 3; ++j) s[(A_MU + sym(i, j)) * P + n] = m[i] * u[j];
    for (int j = 0; j < 3; ++j) {
      s[(A_EU + j) * P + n] = E_p * u[j];
      s[(A_PU + j) * P + n] = p_p * u[j];
    }
  }
}

// Derivatives along one axis (Listing 1), each to its own array: Eq. 7 of one
// array into d2, with Eq. 6 into d1[0] (null: not wanted); or, without a d2, Eq. 6
// of up to BL_SET arrays (null: fewer).
constexpr int BL_SET = 3, BL_JOBS = 24;
template <typename T>
struct Derivative {
  const T* f[BL_SET];
  T* d1[BL_SET];
  T* d2;
  int axis;
};
template <typename T>
struct Derivatives {
  Derivative<T> job[BL_JOBS];  // those with a d2 first
  int with_second, count;
};

// A thread takes BL_Z derivatives of one column: BL_Z planes of one array, or
// BL_Z / BL_SET planes of a set.  Its wrapped offsets are formed once (by
// comparisons); the modulo of every wrapped index had bounded it as much as the
// binary64 pipe.  In binary64 the stencil is summed in integers, leaving one
// binary64 product a derivative, but the second array of a set in a binary64 sum
// beside the others, which balances the two pipes inside each thread.  (The array
// decides, not the plane, so that a shifted state has the shifted derivatives, bit
// for bit; every third plane in a binary64 sum took 1.036 ms a 128^3 stage, sets take
// 1.049, all in integers 1.123, all in binary64 1.312, and sums of one kind a block, the
// kinds in turn, 1.148.)  The binary64 sums take each its own weight, so that
// the large one rounds once less than times a common factor.
// All derivatives that do not read another's result are blocks of one
// launch: 128^3 points are little over a wave of blocks, so a launch per
// derivative left the SMs half idle in its last wave and between launches.
// With the bounds on registers here and of the residual kernel, the 128^3
// store-all stage takes 1.05 instead of 1.36 ms, the 64^3 one 151 instead of 298 us.
constexpr int BL_Z = 9;
template <bool INTEGER, typename T>
__device__ __forceinline__ T bl_first(T m2, T m1, T p1, T p2, T k1, T k2) {
  if constexpr (sizeof(T) == 8 && INTEGER) return k2 * stencil_first(m2, m1, p1, p2);  // k2 = 1/(12 h)
  return k1 * (p1 - m1) - k2 * (p2 - m2);
}
template <typename T>
__device__ __forceinline__ T bl_second(T m2, T m1, T c, T p1, T p2, T k0, T k1, T k2) {
  if constexpr (sizeof(T) == 8) {  // k2 = -1/(12 h^2)
    return -k2 * stencil_second(m2, m1, c, p1, p2);
  } else {
    return k0 * c + k1 * (p1 + m1) + k2 * (p2 + m2);
  }
}
__device__ __forceinline__ int bl_near(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }  // |offset| <= 2 < n
// in-plane offsets of the stencil's points, -2 .. +2 along AXIS
template <int AXIS>
__device__ __forceinline__ void bl_offsets(const Geom& g, int i, int j, int (&o)[5]) {
#pragma unroll
  for (int s = -2; s <= 2; ++s)
    o[s + 2] = (AXIS == 0 ? bl_near(i + s, g.n0) : i) + g.n0 * (AXIS == 1 ? bl_near(j + s, g.n1) : j);
}
// the second derivative of one array and (FIRST) its first; along x2 the
// values stay in registers
template <int AXIS, bool FIRST, typename T>
__device__ __forceinline__ void bl_column(const Geom& g, const Coef<T>& c, const T* __restrict__ f,
                                          T* __restrict__ d1, T* __restrict__ d2, int i, int j, int k0) {
  const long long pl = (long long)g.n0 * g.n1;
  int o[5];
  bl_offsets<AXIS>(g, i, j, o);
  const int own = o[2];
  T w[5];  // the stencil's values; AXIS 2 keeps planes k - 2 .. k + 1
  if constexpr (AXIS == 2) {
#pragma unroll
    for (int s = -2; s <= 1; ++s) w[s + 2] = f[own + pl * bl_near(k0 + s, g.n2)];
  }
#pragma unroll
  for (int q = 0; q < BL_Z; ++q) {
    const int k = k0 + q;
    if (k >= g.n2) break;
    if constexpr (AXIS == 2) {
      w[4] = f[own + pl * bl_near(k + 2, g.n2)];
    } else {
#pragma unroll
      for (int s = 0; s < 5; ++s) w[s] = f[o[s] + pl * k];
    }
    const long long at = own + pl * k;
    if constexpr (FIRST && sizeof(T) == 8) {
      double a, b;
      stencil_both(w[0], w[1], w[2], w[3], w[4], a, b);
      d1[at] = c.c2[AXIS] * a;
      d2[at] = -c.e2[AXIS] * b;
    } else {
      if constexpr (FIRST) d1[at] = bl_first<true>(w[0], w[1], w[3], w[4], c.c1[AXIS], c.c2[AXIS]);
      d2[at] = bl_second(w[0], w[1], w[2], w[3], w[4], c.e0[AXIS], c.e1[AXIS], c.e2[AXIS]);
    }
    if constexpr (AXIS == 2) {
#pragma unroll
      for (int s = 0; s < 4; ++s) w[s] = w[s + 1];
    }
  }
}
// first derivatives of a set of arrays
template <int AXIS, typename T>
__device__ __forceinline__ void bl_set(const Geom& g, const Coef<T>& c, const Derivative<T>& d, int i, int j, int k0) {
  const long long pl = (long long)g.n0 * g.n1;
  int o[5];
  bl_offsets<AXIS>(g, i, j, o);
#pragma unroll
  for (int q = 0; q < BL_Z / BL_SET; ++q) {
    const int k = k0 + q;
    if (k >= g.n2) break;
    auto at = [&](int s) { return o[s + 2] + pl * (AXIS == 2 ? bl_near(k + s, g.n2) : k); };
    const long long m2 = at(-2), m1 = at(-1), p1 = at(1), p2 = at(2), own = o[2] + pl * k;
    auto first = [&](auto integer, int m) {
      const T* __restrict__ f = d.f[m];
      d.d1[m][own] = bl_first<decltype(integer)::value>(f[m2], f[m1], f[p1], f[p2], c.c1[AXIS], c.c2[AXIS]);
    };
    first(std::true_type{}, 0);
    first(std::false_type{}, 1);
    if (d.f[2]) first(std::true_type{}, 2);
  }
}
// blocks of 32 x 8 columns, job by job
template <typename T>
__global__ void __launch_bounds__(256, 8) bl_derivatives(Geom g, const __grid_constant__ Coef<T> c,
                                                      const __grid_constant__ Derivatives<T> jobs) {
  const unsigned bx = (g.n0 + 31) / 32, by = (g.n1 + 7) / 8, bz = (g.n2 + BL_Z - 1) / BL_Z;
  constexpr int ZS = BL_Z / BL_SET;
  unsigned b = blockIdx.x;
  const int i = b % bx * 32 + threadIdx.x;
  b /= bx;
  const int j = b % by * 8 + threadIdx.y;
  b /= by;
  if (i >= g.n0 || j >= g.n1) return;
  if (b < jobs.with_second * bz) {
    const Derivative<T>& d = jobs.job[b / bz];
    const int k0 = b % bz * BL_Z;
    auto column = [&](auto axis) {
      constexpr int A = decltype(axis)::value;
      if (d.d1[0]) bl_column<A, true>(g, c, d.f[0], d.d1[0], d.d2, i, j, k0);
      else bl_column<A, false>(g, c, d.f[0], d.d1[0], d.d2, i, j, k0);
    };
    if (d.axis == 0) column(std::integral_constant<int, 0>{});
    else if (d.axis == 1) column(std::integral_constant<int, 1>{});
    else column(std::integral_constant<int, 2>{});
  } else {
    b -= jobs.with_second * bz;
    const unsigned bs = (g.n2 + ZS - 1) / ZS;
    const Derivative<T>& d = jobs.job[jobs.with_second + b / bs];
    const int k0 = b % bs * ZS;
    if (d.axis == 0) bl_set<0>(g, c, d, i, j, k0);
    else if (d.axis == 1) bl_set<1>(g, c, d, i, j, k0);
    else bl_set<2>(g, c, d, i, j, k0);
  }
}

// (The blocks of a launch stay below the grid's limit of 2^31 - 1: fewer than 2^32 points,
// 6.4 times as many with the padding of the narrowest tiles, 256 columns a block and
// at most 5.4 blocks a column and plane are 5.8e8.)
template <typename T>
cudaError_t launch_derivatives(const Geom& g, const Coef<T>& c, const Derivatives<T>& jobs, cudaStream_t s) {
  const long long tiles = (long long)((g.n0 + 31) / 32) * ((g.n1 + 7) / 8);
  const long long bz = (g.n2 + BL_Z - 1) / BL_Z, bs = (g.n2 + BL_Z / BL_SET - 1) / (BL_Z / BL_SET);
  const long long blocks = tiles * (jobs.with_second * bz + (jobs.count - jobs.with_second) * bs);
  bl_derivatives<T><<<(unsigned)blocks, dim3(32, 8), 0, s>>>(g, c, jobs);
  return cudaGetLastError();
}

// Bound by the binary64 pipe (at its measured rate): sums start from their first term, and three blocks on
// an SM instead of two (128^3 359 -> 314 us).
template <typename T>
__global__ void __launch_bounds__(256, 3) bl_residual(Geom g, Coef<T> c, const T* __restrict__ qrho, const T* __restrict__ qm,
                            const T* __restrict__ qE, long long qstride, T* __restrict__ s) {
  const long long P = g.P;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P; n += (long long)gridDim.x * blockDim.x) {
    auto A = [&](int a) { return s[(long long)a * P + n]; };
    const T rho = T(1) + qrho[n];
    T m[3], u[3];
    for (int i = 0; i < 3; ++i) {
      m[i] = qm[i * qstride + n];
      u[i] = A(A_U + i);
    }
    const T E = qE[n];
    T du[3][3];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) du[i][j] = A(A_DU + 3 * i + j);
    auto dd = [&](int i, int j) { return i == j ? A(A_D2U + 3 * i + i) : A(A_DDU + offd(i, j)); };
    const T div = du[0][0] + du[1][1] + du[2][2];
    // Eq. 1
    T conv = rho * div;
    for (int j = 0; j < 3; ++j) conv += A(A_DRHOU + 3 * j + j) + u[j] * A(A_DRHO + j);
    s[(A_R + 0) * P + n] = T(-0.5) * conv;
    // Eq. 2
    T vw = T(0);
    for (int i = 0; i < 3; ++i) {
      conv = m[i] * div;
      for (int j = 0; j < 3; ++j) conv += A(A_DRHOUU + 3 * i + j) + u[j] * A(A_DRHOU + 3 * i + j);
      const T lap = A(A_D2U + 3 * i) + A(A_D2U + 3 * i + 1) + A(A_D2U + 3 * i + 2);
      const T cross = dd(i, 0) + dd(i, 1) + dd(i, 2);
      const T sd = lap + T(1.0 / 3.0) * cross;  // Laplacian + G - 2/3 G
      vw = i == 0 ? u[0] * sd : vw + u[i] * sd;
      s[(A_R + 1 + i) * P + n] = (T(-0.5) * conv - A(A_DP + i)) + c.inv_re * sd;
    }
    // Eq. 3 (reference enthalpy carries the constant parts of rho E and p)
    conv = E * div;
    for (int j = 0; j < 3; ++j) conv += A(A_DEU + j) + u[j] * A(A_DE + j);
    const T pw = A(A_DPU) + A(A_DPU + 1) + A(A_DPU + 2);
    const T heat = A(A_D2T) + A(A_D2T + 1) + A(A_D2T + 2);
    // du_i/dx_j (du_i/dx_j + du_j/dx_i - 2/3 div delta_ij)
    T diag = du[0][0] * du[0][0], off = T(0);
    for (int i = 0; i < 3; ++i) {
      if (i > 0) diag += du[i][i] * du[i][i];
      const int j = (i + 1) % 3;
      const T a = du[i][j] + du[j][i];
      off = i == 0 ? a * a : off + a * a;
    }
    const T diss = T(2) * diag + (off - T(2.0 / 3.0) * div * div);
    s[(A_R + 4) * P + n] = ((T(-0.5) * conv - pw) - c.H0 * div) + (c.inv_re * (vw + diss) + c.kappa * heat);
  }
}

unsigned pgrid(long long n) {
  long long b = (n + 255) / 256;
  return (unsigned)(b < 4096 ? (b < 1 ? 1 : b) : 4096);
}

template <typename T, typename TIN>
cudaError_t storeall_rhs(const Geom& g, const Coef<T>& c, const TIN* q, T* s, cudaStream_t st) {
  const long long P = g.P;
  auto arr = [&](int a) { return s + (long long)a * P; };
  cudaError_t e;
#define SBLI_CK(x)                      \
  do {                                  \
    e = (x);                            \
    if (e != cudaSuccess) return e;     \
  } while (0)
  bl_primitives<T, TIN><<<pgrid(P), 256, 0, st>>>(g, c, q, s);
  SBLI_CK(cudaGetLastError());
  static_assert(std::is_same<TIN, T>::value, "storeall_rhs differentiates conserved fields in the arithmetic type");
  Derivatives<T> first{}, mixed{};
  // field by field, so that the three axes find it in L2
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      first.job[first.count++] = {{arr(A_U + i)}, {arr(A_DU + 3 * i + j)}, arr(A_D2U + 3 * i + j), j};
  for (int j = 0; j < 3; ++j) first.job[first.count++] = {{arr(A_T)}, {}, arr(A_D2T + j), j};
  first.with_second = first.count;
  for (int j = 0; j < 3; ++j)
    first.job[first.count++] = {{q + P, q + 2 * P, q + 3 * P},
                                {arr(A_DRHOU + j), arr(A_DRHOU + 3 + j), arr(A_DRHOU + 6 + j)}, nullptr, j};
  for (int j = 0; j < 3; ++j)
    first.job[first.count++] = {{arr(A_MU + sym(0, j)), arr(A_MU + sym(1, j)), arr(A_MU + sym(2, j))},
                                {arr(A_DRHOUU + j), arr(A_DRHOUU + 3 + j), arr(A_DRHOUU + 6 + j)}, nullptr, j};
  for (int j = 0; j < 3; ++j)
    first.job[first.count++] = {{q, arr(A_P), q + 4 * P}, {arr(A_DRHO + j), arr(A_DP + j), arr(A_DE + j)}, nullptr, j};
  for (int j = 0; j < 3; ++j)
    first.job[first.count++] = {{arr(A_EU + j), arr(A_PU + j)}, {arr(A_DEU + j), arr(A_DPU + j)}, nullptr, j};
  // mixed derivatives D_i (D_j u_j), i != j, from the stored diagonal gradients
  for (int i = 0; i < 3; ++i) {
    const int j = (i + 1) % 3, k = (i + 2) % 3;
    mixed.job[mixed.count++] = {{arr(A_DU + 4 * j), arr(A_DU + 4 * k)}, {arr(A_DDU + offd(i, j)), arr(A_DDU + offd(i, k))},
                                nullptr, i};
  }
  SBLI_CK(launch_derivatives(g, c, first, st));
  SBLI_CK(launch_derivatives(g, c, mixed, st));
  // conserved variables in the arithmetic type (callers pass T == TIN)
  const T* qrho = reinterpret_cast<const T*>(q);
  const T* qm = qrho + P;
  const T* qE = qrho + 4 * P;
  const long long qstride = P;
  bl_residual<T><<<pgrid(P), 256, 0, st>>>(g, c, qrho, qm, qE, qstride, s);
  SBLI_CK(cudaGetLastError());
#undef SBLI_CK
  return cudaSuccess;
}

template <typename TIN>
__global__ void to_float_kernel(long long n, const TIN* __restrict__ a, float* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = float(a[i]);
}

template <typename TR, typename TOUT>
__global__ void rk_update_kernel(long long n, const TR* __restrict__ r, const double* __restrict__ acc_in,
                                 double* __restrict__ acc_out, TOUT* __restrict__ q_out, double a_dt, double b_dt) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double rr = double(r[i]);
    const double a = acc_in[i];
    acc_out[i] = fma(b_dt, rr, a);
    if (q_out) q_out[i] = TOUT(fma(a_dt, rr, a));
  }
}

}  // namespace

cudaError_t launch_gradients_fp64(const Geom& g, const Coef<double>& c, const double* u, double* grad, cudaStream_t s) {
  Derivatives<double> d{};
  for (int j = 0; j < 3; ++j)
    d.job[d.count++] = {{u, u + g.P, u + 2 * g.P}, {grad + j * g.P, grad + (3 + j) * g.P, grad + (6 + j) * g.P}, nullptr, j};
  return launch_derivatives(g, c, d, s);
}

size_t storeall_scratch_doubles(const Geom& g, int elem_bytes) {
  // A_COUNT arrays of the arithmetic type, plus (binary32 only) a binary32
  // copy of the 5 conserved fields for a binary64 stage-0 input.
  const size_t elems = (size_t)A_COUNT * g.P + (elem_bytes == 4 ? 5 * (size_t)g.P : 0);
  return (elems * elem_bytes + 7) / 8;
}

long long storeall_r_offset(const Geom& g) { return (long long)A_R * g.P; }

cudaError_t launch_storeall_rhs_fp64(const Geom& g, const Coef<double>& c, const double* q_off, double* scratch,
                                     double* r_out, cudaStream_t s) {
  cudaError_t e = storeall_rhs<double, double>(g, c, q_off, scratch, s);
  if (e != cudaSuccess) return e;
  if (r_out) return cudaMemcpyAsync(r_out, scratch + (long long)A_R * g.P, 5 * g.P * sizeof(double),
                                    cudaMemcpyDeviceToDevice, s);
  return cudaSuccess;
}

cudaError_t launch_storeall_rhs_fp32(const Geom& g, const Coef<float>& c, const void* q_off, bool in_fp64,
                                     float* scratch, float* r_out, cudaStream_t s) {
  const float* q = static_cast<const float*>(q_off);
  if (in_fp64) {
    float* conv = scratch + (long long)A_COUNT * g.P;
    to_float_kernel<double><<<pgrid(5 * g.P), 256, 0, s>>>(5 * g.P, static_cast<const double*>(q_off), conv);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    q = conv;
  }
  cudaError_t e = storeall_rhs<float, float>(g, c, q, scratch, s);
  if (e != cudaSuccess) return e;
  if (r_out) return cudaMemcpyAsync(r_out, scratch + (long long)A_R * g.P, 5 * g.P * sizeof(float),
                                    cudaMemcpyDeviceToDevice, s);
  return cudaSuccess;
}

// R -> stage update of Fig. 1: acc_out = acc_in + b dt R; q_out = acc_in + a dt R.
cudaError_t launch_rk_update(const Geom& g, const void* r, bool r_fp64, const double* acc_in, double* acc_out,
                             void* q_out, bool out_fp64, double a_dt, double b_dt, cudaStream_t s) {
  const long long n = 5 * g.P;
  if (r_fp64) {
    if (out_fp64)
      rk_update_kernel<double, double><<<pgrid(n), 256, 0, s>>>(n, static_cast<const double*>(r), acc_in, acc_out,
                                                                static_cast<double*>(q_out), a_dt, b_dt);
    else
      rk_update_kernel<double, float><<<pgrid(n), 256, 0, s>>>(n, static_cast<const double*>(r), acc_in, acc_out,
                                                               static_cast<float*>(q_out), a_dt, b_dt);
  } else {
    if (out_fp64)
      rk_update_kernel<float, double><<<pgrid(n), 256, 0, s>>>(n, static_cast<const float*>(r), acc_in, acc_out,
                                                               static_cast<double*>(q_out), a_dt, b_dt);
    else
      rk_update_kernel<float, float><<<pgrid(n), 256, 0, s>>>(n, static_cast<const float*>(r), acc_in, acc_out,
                                                              static_cast<float*>(q_out), a_dt, b_dt);
  }
  return cudaGetLastError();
}

}  // namespace sbli
