// diag.cu -- Taylor-Green initial field, reference-state conversion and the
// binary64 kinetic-energy / enstrophy reduction.
#include <cuda.h>
#include <math.h>

#include "fpconv.cuh"
#include "ke_march.cuh"
#include "sbli_internal.cuh"

namespace sbli {

template <typename T>
Coef<T> make_coef(const int n[3], const sbli_params& p) {
  Coef<T> c;
  double e0s = 0.0;
  for (int a = 0; a < 3; ++a) {
    const double h = 2.0 * M_PI * p.L / (double)n[a];
    e0s += -5.0 / (2.0 * h * h);
  }
  c.e0s = T(e0s);
  for (int a = 0; a < 3; ++a) {
    const double h = 2.0 * M_PI * p.L / (double)n[a];
    c.c1[a] = T(2.0 / (3.0 * h));
    c.c2[a] = T(1.0 / (12.0 * h));
    c.e0[a] = T(-5.0 / (2.0 * h * h));
    c.e1[a] = T(4.0 / (3.0 * h * h));
    c.e2[a] = T(-1.0 / (12.0 * h * h));
    c.hc1[a] = T(-1.0 / (3.0 * h));
    c.hc2[a] = T(-1.0 / (24.0 * h));
    c.t2[a] = T(1.0 / (36.0 * h));
    c.f2[a] = T(-1.0 / (9.0 * h * h));
    c.v0[a] = T(e0s - 5.0 / (6.0 * h * h));
  }
  const double inv_re = isinf(p.Re) ? 0.0 : 1.0 / p.Re;
  c.gm1 = T(p.gamma - 1.0);
  c.gM2 = T(p.gamma * p.Mach * p.Mach);
  c.gm1x2 = T(2.0 * (p.gamma - 1.0));
  c.hgM2 = T(0.5 * p.gamma * p.Mach * p.Mach);
  c.inv_re = T(inv_re);
  c.kappa = T(inv_re / ((p.gamma - 1.0) * p.Mach * p.Mach * p.Pr));
  c.H0 = T(1.0 / ((p.gamma - 1.0) * p.Mach * p.Mach));
  return c;
}
template Coef<double> make_coef<double>(const int[3], const sbli_params&);
template Coef<float> make_coef<float>(const int[3], const sbli_params&);
template Coef<dfloat> make_coef<dfloat>(const int[3], const sbli_params&);

RefState make_ref(const sbli_params& p) {
  RefState r;
  r.rho0 = 1.0;
  r.E0 = 1.0 / (p.gamma * (p.gamma - 1.0) * p.Mach * p.Mach);  // p_ref/(gamma-1)
  return r;
}

// §4, Eqs. 9-12 with amplitude A; T = 1 so rho = gamma M^2 p (Eq. 5), rho E
// from Eq. 4.  Written as deviations from the reference state:
//   rho - 1 = gamma M^2 (p - p_ref),  rho E - E_ref = (p - p_ref)/(gamma-1) + rho |u|^2/2.
// The field is made of functions of one coordinate each, so a thread evaluates
// those of its column once for INIT_Z planes and a block those of x2 once for
// its planes: the binary64 pipe, which bounds this kernel, spends itself on
// the products and not on six trigonometric functions a point.  Block b takes part
// b % parts of the columns and planes INIT_Z (b / parts) ...: one grid dimension, as
// the others' limit of 65,535 is 2^21 planes.
constexpr int INIT_Z = 32;
__global__ void __launch_bounds__(256) init_tgv_kernel(Geom g, unsigned parts, double h0, double h1, double h2,
                                                       double L, double A, double gM2, double inv_gm1,
                                                       double* __restrict__ q) {
  __shared__ double cz[INIT_Z], c2z[INIT_Z];
  const int z0 = (int)(blockIdx.x / parts) * INIT_Z, nz = min(INIT_Z, g.n2 - z0);
  if ((int)threadIdx.x < nz) {
    const double z = (z0 + (int)threadIdx.x) * h2;
    cz[threadIdx.x] = cos(z / L);
    c2z[threadIdx.x] = cos(2.0 * z / L);
  }
  __syncthreads();
  const long long P = g.P, plane = (long long)g.n0 * g.n1;
  for (long long n = blockIdx.x % parts * 256LL + threadIdx.x; n < plane; n += parts * 256LL) {
    const double x = (int)(n % g.n0) * h0, y = (int)(n / g.n0) * h1;
    double sx, cx, sy, cy;
    sincos(x / L, &sx, &cx);
    sincos(y / L, &sy, &cy);
    const double cxy = cos(2.0 * x / L) + cos(2.0 * y / L);
    double* o = q + n + plane * z0;
    for (int k = 0; k < nz; ++k, o += plane) {
      const double u0 = A * sx * cy * cz[k];
      const double u1 = -A * cx * sy * cz[k];
      const double dp = A * A / 16.0 * cxy * (2.0 + c2z[k]);
      const double rho_p = gM2 * dp;
      const double rho = 1.0 + rho_p;
      o[0] = rho_p;
      o[P] = rho * u0;
      o[2 * P] = rho * u1;
      o[3 * P] = 0.0;
      o[4 * P] = dp * inv_gm1 + 0.5 * rho * (u0 * u0 + u1 * u1);
    }
  }
}

static unsigned grid_for(long long n, int block) {
  long long b = (n + block - 1) / block;
  return (unsigned)(b < 8192 ? (b < 1 ? 1 : b) : 8192);
}

cudaError_t launch_init_tgv(const Geom& g, const sbli_params& p, double amplitude, double* q, cudaStream_t s) {
  const double h0 = 2.0 * M_PI * p.L / g.n0, h1 = 2.0 * M_PI * p.L / g.n1, h2 = 2.0 * M_PI * p.L / g.n2;
  const long long plane = (long long)g.n0 * g.n1;
  const unsigned parts = grid_for(plane, 256);
  init_tgv_kernel<<<parts * ((g.n2 + INIT_Z - 1) / INIT_Z), 256, 0, s>>>(
      g, parts, h0, h1, h2, p.L, amplitude, p.gamma * p.Mach * p.Mach, 1.0 / (p.gamma - 1.0), q);
  return cudaGetLastError();
}

// Conversions between a caller's plain conserved variables and the library's
// own form of a state, one pass over memory each: a thread moves STATE_ITEMS
// values of one field (blockIdx.y), 256 apart, all loads issued before the
// stores, so every access is a coalesced row whatever the field's size and
// alignment.
constexpr int STATE_ITEMS = 4;
static dim3 state_grid(long long P) {
  const long long b = (P + 256 * STATE_ITEMS - 1) / (256 * STATE_ITEMS);
  return dim3((unsigned)(b < (1 << 20) ? b : (1 << 20)), 5);
}
template <typename L, typename F>
__device__ __forceinline__ void for_field(long long P, L&& load, F&& put) {
  const long long f = blockIdx.y;
  for (long long b = blockIdx.x; b * (256 * STATE_ITEMS) < P; b += gridDim.x) {
    const long long n0 = b * (256 * STATE_ITEMS) + threadIdx.x;
    double v[STATE_ITEMS];
#pragma unroll
    for (int k = 0; k < STATE_ITEMS; ++k)
      if (n0 + 256 * k < P) v[k] = load(f * P + n0 + 256 * k);
#pragma unroll
    for (int k = 0; k < STATE_ITEMS; ++k)
      if (n0 + 256 * k < P) put(f * P + n0 + 256 * k, v[k]);
  }
}
__device__ __forceinline__ double field_reference(double rho0, double E0) {
  return blockIdx.y == 0 ? rho0 : (blockIdx.y == 4 ? E0 : 0.0);
}

// plain -> own form: binary64 deviations with (copy32) the binary32 copy the
// binary32 stages read or (pairs) the (hi, lo) pairs the double-float stages
// read, or (dst64 null) the double-float register alone.
__global__ void __launch_bounds__(256) import_state_kernel(long long P, double rho0, double E0,
                                                           const double* __restrict__ src, double* __restrict__ dst64,
                                                           float* __restrict__ copy32, float2* __restrict__ pairs,
                                                           float* __restrict__ df) {
  const double ref = field_reference(rho0, E0);
  for_field(
      P, [&](long long i) { return src[i]; },
      [&](long long i, double x) {
        const double v = blockIdx.y % 4 == 0 ? x - ref : x;
        if (df) {
          const float hi = __double2float_rn(v);
          df[i] = hi;
          df[i + 5 * P] = __double2float_rn(v - (double)hi);
          return;
        }
        dst64[i] = v;
        if (copy32) copy32[i] = narrow_f64_rna(v);
        if (pairs) {
          float hi, lo;
          split_f64(v, hi, lo);
          pairs[i] = make_float2(hi, lo);
        }
      });
}

cudaError_t launch_import_state(long long P, const RefState& r, const double* src, const StateForm& to,
                                cudaStream_t s) {
  import_state_kernel<<<state_grid(P), 256, 0, s>>>(P, r.rho0, r.E0, src, to.f64, to.copy32,
                                                    reinterpret_cast<float2*>(to.pairs), to.df);
  return cudaGetLastError();
}

// deviation -> plain.  Fields 0 and 4 only differ; momenta are copied.
__global__ void __launch_bounds__(256) from_offset_kernel(long long P, double rho0, double E0, const double* src,
                                                          double* dst) {
  const double ref = field_reference(rho0, E0);
  for_field(
      P, [&](long long i) { return src[i]; },
      [&](long long i, double x) { dst[i] = blockIdx.y % 4 == 0 ? x + ref : x; });
}

cudaError_t launch_from_offset(const Geom& g, const RefState& r, const double* q_off, double* q_plain,
                               cudaStream_t s) {
  from_offset_kernel<<<state_grid(g.P), 256, 0, s>>>(g.P, r.rho0, r.E0, q_off, q_plain);
  return cudaGetLastError();
}

bool direct_device_access(const void* p, size_t bytes) {
  cudaPointerAttributes a;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type != cudaMemoryTypeDevice || a.device != dev || (uintptr_t)p % sizeof(double) != 0) return false;
  // the allocation that p lies in, from the driver (found once, for all threads)
  static const auto range_of = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return reinterpret_cast<decltype(&cuMemGetAddressRange)>(f);
  }();
  CUdeviceptr base = 0;
  size_t size = 0;
  if (!range_of || range_of(&base, &size, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS) return false;
  const size_t offset = (uintptr_t)p - (uintptr_t)base;
  return offset <= size && bytes <= size - offset;
}

__global__ void widen_kernel(long long n, const float* __restrict__ src, double* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = double(src[i]);
}

cudaError_t launch_widen(long long n, const float* src, double* dst, cudaStream_t s) {
  widen_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, src, dst);
  return cudaGetLastError();
}

// The binary32 copy of a binary64 state that stage 0 of the binary32 path
// reads: the same narrowing the stage kernels apply (narrow_f64_rna).
__global__ void narrow_kernel(long long n, const double* __restrict__ src, float* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = narrow_f64_rna(src[i]);
}

cudaError_t launch_narrow(long long n, const double* src, float* dst, cudaStream_t s) {
  narrow_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, src, dst);
  return cudaGetLastError();
}

__global__ void df_split_kernel(long long n5, long long P, double rho0, double E0, const double* __restrict__ src,
                                float* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n5; i += (long long)gridDim.x * blockDim.x) {
    const long long f = i / P;
    const double v = src[i] - (f == 0 ? rho0 : (f == 4 ? E0 : 0.0));
    const float hi = __double2float_rn(v);
    dst[i] = hi;
    dst[i + 5 * P] = __double2float_rn(v - (double)hi);
  }
}

__global__ void __launch_bounds__(256) df_join_kernel(long long P, double rho0, double E0,
                                                      const float* __restrict__ src, double* __restrict__ dst) {
  const double ref = field_reference(rho0, E0);
  for_field(
      P, [&](long long i) { return (double)src[i] + (double)src[i + 5 * P]; },
      [&](long long i, double x) { dst[i] = x + ref; });
}

cudaError_t launch_df_split(long long P, const RefState& r, const double* src, float* dst, cudaStream_t s) {
  df_split_kernel<<<grid_for(5 * P, 256), 256, 0, s>>>(5 * P, P, r.rho0, r.E0, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_df_join(long long P, const RefState& r, const float* src, double* dst, cudaStream_t s) {
  df_join_kernel<<<state_grid(P), 256, 0, s>>>(P, r.rho0, r.E0, src, dst);
  return cudaGetLastError();
}

// A binary64 field as interleaved double-float pairs, split as the stage
// kernels split a binary64 input (split_f64).
__global__ void pair_split_kernel(long long n, const double* __restrict__ src, float2* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    float hi, lo;
    split_f64(src[i], hi, lo);
    dst[i] = make_float2(hi, lo);
  }
}

cudaError_t launch_pair_split(long long n, const double* src, float* dst, cudaStream_t s) {
  pair_split_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, src, reinterpret_cast<float2*>(dst));
  return cudaGetLastError();
}

// A stage field of interleaved double-float pairs as binary64 (the sum of two
// binary32 values is exact in binary64).
__global__ void pair_join_kernel(long long n, const float2* __restrict__ src, double* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = src[i];
    dst[i] = (double)v.x + (double)v.y;
  }
}

cudaError_t launch_pair_join(long long n, const float* src, double* dst, cudaStream_t s) {
  pair_join_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, reinterpret_cast<const float2*>(src), dst);
  return cudaGetLastError();
}

// Plain conserved variables at listed points: out[f * count + i] for the
// point of linear index idx[i] (x0 fastest).  The binary64 state (q64) or the
// double-float state (qdf: hi fields, then lo fields) is in deviation form;
// the sums are those of the full-grid conversions, so a sample equals the
// corresponding entry of a full read-out bit for bit.  Indices outside
// [0, P) yield NaN in all five fields.
__global__ void sample_state_kernel(long long P, double rho0, double E0, const double* __restrict__ q64,
                                    const float* __restrict__ qdf, const long long* __restrict__ idx, int count,
                                    double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const long long n = idx[i];
    const bool inside = n >= 0 && n < P;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      double v = __longlong_as_double(0x7ff8000000000000LL);  // quiet NaN
      if (inside) {
        const long long m = (long long)f * P + n;
        if (q64) {  // as from_offset_kernel
          v = q64[m];
          if (f == 0) v += rho0;
          if (f == 4) v += E0;
        } else {  // as df_join_kernel
          v = ((double)qdf[m] + (double)qdf[m + 5 * P]) + (f == 0 ? rho0 : (f == 4 ? E0 : 0.0));
        }
      }
      out[(long long)f * count + i] = v;
    }
  }
}

cudaError_t launch_sample_state(long long P, const RefState& r, const double* q64, const float* qdf,
                                const long long* idx, int count, double* out, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  sample_state_kernel<<<grid_for(count, 256), 256, 0, s>>>(P, r.rho0, r.E0, q64, qdf, idx, count, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ KE
constexpr int KE_MAX_BLOCKS = 1024;  // partial sums the callers' scratch holds

int ke_num_partials(const Geom& g) { return ke_blocks(g, KE_MAX_BLOCKS); }

// One block: thread t sums pairs t, t+256, ... in order, then a fixed tree.
__global__ void __launch_bounds__(256) finalize_ke_kernel(const double* __restrict__ partials, int n, double inv_p,
                                                          double* __restrict__ out) {
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) {
    a += partials[2 * i];
    b += partials[2 * i + 1];
  }
  __shared__ double red[2][256];
  red[0][threadIdx.x] = a;
  red[1][threadIdx.x] = b;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      red[0][threadIdx.x] += red[0][threadIdx.x + s];
      red[1][threadIdx.x] += red[1][threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = red[0][0] * inv_p;
    out[1] = red[1][0] * inv_p;
  }
}

cudaError_t launch_finalize_ke(const double* partials, int n, double inv_p, double* out, cudaStream_t s) {
  finalize_ke_kernel<<<1, 256, 0, s>>>(partials, n, inv_p, out);
  return cudaGetLastError();
}

cudaError_t launch_ke(const Geom& g, const Coef<double>& c, const RefState& r, const double* q_off,
                      double* partials, double* out, cudaStream_t s) {
  (void)r;
  const int nb = ke_num_partials(g);
  ke_march_kernel<false><<<nb, KE_THREADS, 0, s>>>(g, c, q_off, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_finalize_ke(partials, nb, 1.0 / (double)g.P, out, s);
}

}  // namespace sbli
