// Shared device-side definitions of the SGS-PFP CUDA library (sm_103a).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sgs.h"

namespace sgs {

namespace cg = cooperative_groups;

constexpr int kMaxN = 32;          // velocity points per dimension supported
constexpr int kLanes = 32;         // cells per spectral group (one warp lane per cell)
constexpr double kPi = 3.14159265358979323846;

// ---------------------------------------------------------------------------------------
// Per-instance description in device memory.
// ---------------------------------------------------------------------------------------
struct InstDev {
  long long f_off;       // element offset of cell 0 in every field
  int J;                 // cells (nx ny in 2-D)
  int nx, ny;            // grid (ny = 1 in 1-D)
  int space_dim;
  int cell0;             // global index of cell 0 (collision-step cell list)
  int collision;         // sgs_collision
  int bc_kind[4];        // x_lo, x_hi, y_lo, y_hi
  double dx, dy, eps;    // dy = 1 in 1-D (cell measure dx dy)
  double b0;
  double bc_rho[4];      // inflow density (unused for diffuse walls)
  double wall_denom[4];  // sum over incoming v of w (v.n) Mhat_wall (diffuse walls)
  double inv_dx, inv_dy, inv_eps;
  double wall_scale[4];  // -w dv / wall_denom: diffuse-wall density per outgoing sum of (v.n / dv) f
  double tol2_w;         // inner_tol^2 / w: the inner tolerance as an unweighted sum of squares
  double total_mass;
  double inner_tol;
  int inner_max, inner_fixed, inner_method, newton_max;
  double newton_tol;
  // Unit wall Maxwellian of side s, separable: Mhat(v) = W[s][0][i1] W[s][1][i2] W[s][2][i3],
  // with the incoming half of the normal component kept and the outgoing half zeroed (in
  // W[s][0] for the x sides, W[s][1] for the y sides).
  double wall[4][3][kMaxN];
};

struct Counters {
  unsigned int status;
  unsigned int pad;
  unsigned long long visits, inner_iters, newton_iters, newton_solves, fallbacks;
};

// ---------------------------------------------------------------------------------------
// Velocity grid helpers: v_i = (i - N/2 + 1) dv.
// ---------------------------------------------------------------------------------------
__host__ __device__ inline double node(int i, int N, double dv) { return (double)(i - N / 2 + 1) * dv; }

// ---------------------------------------------------------------------------------------
// Double-float ("df64") arithmetic: a value is hi + lo with two FP32 numbers, |lo| <= ulp(hi)/2,
// carried through error-free transformations (Knuth's two-sum, Dekker's fast two-sum, and the
// FMA form of the exact product). Addition and multiplication keep about 48 significant bits
// relative to the operands, enough for the cancellations of the cell equation, and run on the
// FP32 pipes, which on this GPU have ~40x the FP64 throughput.
// ---------------------------------------------------------------------------------------
struct __align__(8) dfloat {
  float hi, lo;
};

__device__ __forceinline__ dfloat df_fast_two_sum(float a, float b) {  // |a| >= |b|
  float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ dfloat operator+(dfloat a, dfloat b) {
  float s = a.hi + b.hi;
  float bb = s - a.hi;
  float e = (a.hi - (s - bb)) + (b.hi - bb);
  e += a.lo + b.lo;
  return df_fast_two_sum(s, e);
}
__device__ __forceinline__ dfloat operator-(dfloat a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ dfloat operator-(dfloat a, dfloat b) { return a + (-b); }
__device__ __forceinline__ dfloat operator*(dfloat a, dfloat b) {
  float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return df_fast_two_sum(p, e);
}
__device__ __forceinline__ dfloat& operator+=(dfloat& a, dfloat b) { return a = a + b; }
__device__ __forceinline__ dfloat& operator-=(dfloat& a, dfloat b) { return a = a - b; }

// Exact split of a double into a double-float by bit manipulation (no FP64 instruction):
// hi keeps the leading 24 significand bits (truncated), lo the next bits rounded to 24.
// Magnitudes below 2^-100 (irrelevant next to the O(1) values they are summed with) map to 0.
__device__ __forceinline__ dfloat df_split(double x) {
  const unsigned int h = (unsigned int)__double2hiint(x), l = (unsigned int)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ffu) - 1023;
  if (e < -100) return {0.0f, 0.0f};
  const unsigned int sign = h & 0x80000000u;
  const float hi = __uint_as_float(sign | ((unsigned int)(e + 127) << 23) | ((h & 0xfffffu) << 3) | (l >> 29));
  // low 29 bits as a fraction of the last place of hi, 2^(e - 23), which is a normal number
  const float ulp = __uint_as_float(sign | ((unsigned int)(e + 104) << 23));
  const float lo = __uint2float_rn(l & 0x1fffffffu) * 1.862645149230957e-09f * ulp;
  return {hi, lo};
}

// exp in double-float arithmetic (no FP64 instruction): Cody and Waite's additive argument
// reduction x = k ln2 + r with ln2 split into three floats (the first with trailing zero bits,
// so k * c1 is exact for |k| < 512), then exp(r), |r| <= ln2/2, from its Taylor series to
// degree 13 by Horner's rule, and exp(x) = 2^k exp(r).
__device__ inline dfloat df_exp(dfloat x) {
  const float c1 = 0.693145751953125f, c2 = 1.428606765330187e-06f, c3 = 5.497923148104107e-14f;
  const float inv_ln2 = 1.4426950408889634f;
  if (x.hi < -87.0f) return {0.0f, 0.0f};
  float kf = rintf(x.hi * inv_ln2);
  // x.hi - kf c1 is exact (kf c1 is exact and, by Sterbenz's lemma, so is the difference)
  dfloat r = dfloat{x.hi - kf * c1, 0.0f} + dfloat{x.lo, 0.0f};
  float p = kf * c2;
  dfloat kc2 = {p, fmaf(kf, c2, -p)};
  r = r - kc2;
  r = r - dfloat{kf * c3, 0.0f};
  const float ch[14] = {1.0f, 1.0f, 0.5f, 0.1666666716337204f, 0.0416666679084301f, 0.008333333767950535f,
                        0.0013888889225199819f, 0.00019841270113829523f, 2.4801587642286904e-05f,
                        2.7557318844628753e-06f, 2.755731998149713e-07f, 2.5052107943679403e-08f,
                        2.0876755879584152e-09f, 1.6059044372074283e-10f};
  const float cl[14] = {0.0f, 0.0f, 0.0f, -4.967053879312289e-09f, -1.2417634698280722e-09f,
                        -4.34617203337595e-10f, -3.3631094437103215e-11f, -2.725596874933456e-12f,
                        -3.40699609366682e-13f, 3.793571224297229e-14f, -7.575112209051195e-15f,
                        4.4176230446483665e-16f, 1.1082839147459852e-16f, -5.352526511562726e-18f};
  // Estrin's scheme: the same degree-13 polynomial with a dependency chain of four
  // multiply-add levels instead of thirteen
  dfloat c[14];
#pragma unroll
  for (int n = 0; n < 14; n++) c[n] = dfloat{ch[n], cl[n]};
  dfloat r2 = r * r;
  dfloat r4 = r2 * r2;
  dfloat r8 = r4 * r4;
  dfloat pr[7];
#pragma unroll
  for (int n = 0; n < 7; n++) pr[n] = c[2 * n] + c[2 * n + 1] * r;
  dfloat q0 = pr[0] + pr[1] * r2, q1 = pr[2] + pr[3] * r2, q2 = pr[4] + pr[5] * r2;
  dfloat s0 = q0 + q1 * r4, s1 = q2 + pr[6] * r4;
  dfloat acc = s0 + s1 * r8;
  int k = (int)kf;
  return {ldexpf(acc.hi, k), ldexpf(acc.lo, k)};
}

// Conversions used by code templated on the arithmetic type E.
template <typename E>
__device__ __forceinline__ E cvt(double x);
template <>
__device__ __forceinline__ double cvt<double>(double x) { return x; }
template <>
__device__ __forceinline__ dfloat cvt<dfloat>(double x) {
  return df_split(x);
}
__device__ __forceinline__ double tod(double x) { return x; }
__device__ __forceinline__ double tod(dfloat x) { return (double)x.hi + (double)x.lo; }
__device__ __forceinline__ float tof(double x) { return (float)x; }
__device__ __forceinline__ float tof(float x) { return x; }
__device__ __forceinline__ float tof(dfloat x) { return x.hi; }

// The double of an FP32 number, and of a double-float, with the bits of the conversion: a normal
// number is widened by integer operations (a conversion holds the FP64 unit for 101 cycles).
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)x;  // subnormal, infinite, NaN
  const unsigned hi = (u & 0x80000000u) | (m == 0u ? 0u : (m >> 3) + 0x38000000u);
  return __hiloint2double((int)hi, (int)(u << 29));
}
__device__ __forceinline__ double widen(dfloat x) { return widen(x.hi) + widen(x.lo); }

__device__ __forceinline__ double shfl_x(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float shfl_x(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dfloat shfl_x(dfloat v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// ---------------------------------------------------------------------------------------
// Warp reductions (butterfly: every lane receives the total, in a fixed order).
// ---------------------------------------------------------------------------------------
template <int NV, typename T>
__device__ inline void warp_allsum(T (&x)[NV]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int q = 0; q < NV; q++) x[q] += shfl_x(x[q], o);
  }
}

// Solves A y = b (FP32) for the symmetric positive definite 5x5 matrix given by its upper
// triangle (row-major). Returns false if A is not numerically positive definite. The
// solution only serves as a Newton direction; the residual F stays in the caller's precision.
__device__ inline bool chol5_solve(const float* Au, const float* b, float* y) {
  float a[5][5];
  int t = 0;
#pragma unroll
  for (int i = 0; i < 5; i++)
#pragma unroll
    for (int j = i; j < 5; j++) {
      a[i][j] = Au[t];
      a[j][i] = Au[t];
      t++;
    }
  // symmetric diagonal scaling keeps the FP32 factorisation well conditioned
  float sc[5];
#pragma unroll
  for (int i = 0; i < 5; i++) {
    if (!(a[i][i] > 0.0f)) return false;
    sc[i] = rsqrtf(a[i][i]);
  }
  float l[5][5], dinv[5];
#pragma unroll
  for (int i = 0; i < 5; i++)
#pragma unroll
    for (int j = 0; j < 5; j++) l[i][j] = 0.0f;
#pragma unroll
  for (int j = 0; j < 5; j++) {
    float d = a[j][j] * sc[j] * sc[j];
#pragma unroll
    for (int k = 0; k < j; k++) d -= l[j][k] * l[j][k];
    if (!(d > 0.0f)) return false;
    // approximate reciprocal square root: the result is only a Newton direction
    float inv = rsqrtf(d);
    l[j][j] = d * inv;
    dinv[j] = inv;
#pragma unroll
    for (int i = j + 1; i < 5; i++) {
      float s = a[i][j] * sc[i] * sc[j];
#pragma unroll
      for (int k = 0; k < j; k++) s -= l[i][k] * l[j][k];
      l[i][j] = s * inv;
    }
  }
  float z[5];
#pragma unroll
  for (int i = 0; i < 5; i++) {
    float s = b[i] * sc[i];
#pragma unroll
    for (int k = 0; k < i; k++) s -= l[i][k] * z[k];
    z[i] = s * dinv[i];
  }
#pragma unroll
  for (int i = 4; i >= 0; i--) {
    float s = z[i];
#pragma unroll
    for (int k = i + 1; k < 5; k++) s -= l[k][i] * y[k];
    y[i] = s * dinv[i];
  }
#pragma unroll
  for (int i = 0; i < 5; i++) y[i] *= sc[i];
  return true;
}

// Continuum Maxwellian with the given moments (rho, rho U, sum |v|^2 f): initial guess.
template <typename E>
__device__ inline bool continuum_guess(const E* m, double* th) {
  double rho = tod(m[0]);
  if (!(rho > 0.0)) return false;
  double U0 = tod(m[1]) / rho, U1 = tod(m[2]) / rho, U2 = tod(m[3]) / rho;
  double uu = U0 * U0 + U1 * U1 + U2 * U2;
  double T = (tod(m[4]) / rho - uu) / 3.0;
  if (!(T > 0.0)) return false;
  th[4] = 0.5 / T;
  th[1] = U0 / T;
  th[2] = U1 / T;
  th[3] = U2 / T;
  th[0] = log(rho / (2.0 * kPi * T * sqrt(2.0 * kPi * T))) - 0.5 * uu / T;
  return true;
}

// ---------------------------------------------------------------------------------------
// PTX wrappers: mbarrier and bulk (TMA, non-tensor) global -> shared copies.
// ---------------------------------------------------------------------------------------
__device__ inline uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ inline void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ inline void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ inline void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

// Bounded wait on the phase with the given parity; returns false after max_spins polls.
__device__ inline bool mbar_wait(uint64_t* bar, uint32_t parity, long long max_spins) {
  uint32_t addr = smem_addr(bar);
  for (long long i = 0; i < max_spins; i++) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// 1-D bulk copy global -> shared, completion signalled on bar (bytes % 16 == 0, both
// addresses 16-byte aligned).
__device__ inline void bulk_g2s(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst_smem)),
      "l"(src_gmem), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

}  // namespace sgs
