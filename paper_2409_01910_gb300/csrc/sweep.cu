// Persistent symmetric Gauss-Seidel scan (eq. (29)) with the preconditioned fixed-point cell
// solve (eqs. (20), (24)-(26)).
//
// One thread-block cluster per instance walks that instance's cells in scan order inside a
// single launch. Each thread owns the same runs of four consecutive velocity nodes (one pencil,
// fixed i1, i2) in every cell, so a thread only ever reads and writes its own nodes: the
// upwind neighbour's new value is its own earlier write, and no two threads touch the same
// global element.
//
// The inner iteration runs on five numbers, not on the nodes. With c = |v1|/dx (+ |v2|/dy)
// and A = nu/eps, step 2 (eq. (25)) gives g = (A M+ - r) / (c + A), where r is fixed during the
// visit, 1 / (c + A) depends on v1 (and v2) only and M+ is separable. The moments of g are
//   sum phi g = A sum phi M+ / (c + A) - sum phi r / (c + A),
// products of 1-D sums (2-D: one sum over (v1, v2)) minus five constants of the visit, and the
// residual and the step-1 target of the new iterate follow from the same identity. So a visit
// is: one pass over the nodes that forms r and every sum the solve needs, one cluster
// reduction of those sums, the whole inner iteration on the evaluating warps of every CTA
// (each CTA computes the same numbers from the same totals: no further cluster traffic), and
// one pass that writes g. It is bound by the latency of the Newton evaluations. Measured on 64
// cells of 32^3 nodes in double-float (16 CTAs x 256 threads, 8.1 inner updates and 31 Newton
// iterations a visit): 40.6 us a visit, 32 of them in the inner iteration; with the moments of
// every update from a pass over the nodes and a cluster reduction, and a full evaluation for
// every Newton step, it was 167 us. FP64, 45 cells of 20^3: 113 instead of 380 us.
//
// Inside a Newton evaluation the chain is shortened as well: warps 0-2 evaluate the factors
// and 1-D sums of one velocity dimension each, warp 3 (2-D: and warp 1) the weighted sums; the sums of a
// warp are reduced together by halving exchanges (four values: 6 additions instead of 20);
// only the sums of the moments themselves are in E (three per warp), the others, which set a
// direction or a norm, are FP32; lane k holds component k of the exponents, the target and the
// moments; the exponential is table-driven; and, the weighted measure being a product, the
// Newton direction has a closed form in the basis that the measure makes orthogonal (no
// factorisation; the 2-D step-1 measure is a sum of two products and keeps the 5 x 5 solve).
//
// E is the arithmetic of the sums and the Newton residuals: double for the FP64 solver,
// double-float (two FP32 numbers, FP64-class accuracy, no FP64 instruction on the critical
// path) for the mixed solver.
#include <cfloat>

#include "common.cuh"
#include "kernels.h"

namespace sgs {

constexpr int kRed = 16;    // values of a visit's cluster reduction
constexpr int R = 4;        // nodes of a run: 32 bytes, one sector; divides every N
constexpr int kRows = 5;    // rows of 1-D sums of an evaluation (eval_row)
constexpr int kTeam = 4;    // evaluating warps: one per scheduler of the SM

template <typename E>
struct SweepSmem {
  E c1e[kMaxN];             // |v_i| / dx (step-1 weights, x part)
  E c2e[kMaxN];             // |v_i| / dy (step-1 weights, y part; 2-D)
  E cA[kMaxN];              // |v_i|/dx + nu/eps of the current cell (1-D)
  E den[kMaxN];             // its reciprocal (1-D)
  E ef[3][kMaxN];           // factors of the Maxwellian that the next pass over the nodes reads
  E W[4][3][kMaxN];         // unit wall Maxwellians
  E etab[64];               // 2^(j/64)
  double vm[2][kMaxN];      // 2-D FP64: node numbers m and m^2
  E rows[2][kRows][4];     // Newton evaluations, double-buffered: sums of powers 0-2, one row per warp
  E warp_part[kRed][8];
  E part[2][16][kRed];      // partial sums of every CTA of the cluster
  E tot[kRed];
  E rho[4];                 // wall densities of the sides
  E dpart[kTeam][4];       // 2-D: sums over (v1, v2) of M+ / (c + A)
  float rowsf[2][kRows][8];  // FP32: sums of powers 0-4, then (roles 0-2) those of the norm
  int ctl;                  // what the CTA does after the evaluating warps: bit 0 write, bit 1 second pass
};

// ---------------------------------------------------------------------------------------
// Small helpers in the arithmetic E.
// ---------------------------------------------------------------------------------------
// Velocities are measured in units of the node spacing inside a scan: node i is the integer
// m = i - N/2 + 1, which FP32 holds exactly, so a product with a node is a product with one
// FP32 number (Node<E>::M), and the exponents, targets and moments carry the powers of dv.
template <typename E>
struct Node;
template <>
struct Node<double> {  // FP64
  typedef double M;
};
template <>
struct Node<dfloat> {
  typedef float M;
};
// Node i and its square as M. An int -> FP64 conversion holds the FP64 unit of a scheduler for 101
// cycles (a multiply: 64), so the 2-D FP64 passes, two fifths of a visit there, read both from a
// table (40 x 40 cells, 20 velocities, BGK: 32.35 -> 31.59 ms). In 1-D FP64 the table costs the
// Newton loop more than the passes gain (16 cells, 16 velocities: 6.38 -> 6.62 ms), and in FP32 a
// conversion is as cheap as a load.
template <typename M, bool TWO_D>
__device__ __forceinline__ M node_m(const double (&vm)[2][kMaxN], int i, int N) {
  if constexpr (TWO_D && sizeof(M) == 8) return vm[0][i];
  return (M)(i + 1 - N / 2);
}
template <typename M, bool TWO_D>
__device__ __forceinline__ M node_q(const double (&vm)[2][kMaxN], int i, M m) {
  if constexpr (TWO_D && sizeof(M) == 8) return vm[1][i];
  return m * m;
}
// Double-float sums and products without the final renormalisation: (hi, lo) whose halves may
// overlap by a few bits. In a chain of additions the leading parts then depend on each other
// through one FP32 addition only, and an addition takes 8 operations instead of 11; norm()
// restores the form that a product needs.
__device__ __forceinline__ dfloat uadd(dfloat a, dfloat b) {
  const float s = a.hi + b.hi, bb = s - a.hi;
  return {s, (a.lo + b.lo) + ((a.hi - (s - bb)) + (b.hi - bb))};
}
__device__ __forceinline__ dfloat umul(dfloat a, dfloat b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  return {p, fmaf(a.lo, b.hi, e)};
}
__device__ __forceinline__ dfloat umul(dfloat a, float m) {
  const float p = a.hi * m;
  return {p, fmaf(a.lo, m, fmaf(a.hi, m, -p))};
}
__device__ __forceinline__ dfloat norm(dfloat a) { return df_fast_two_sum(a.hi, a.lo); }
__device__ __forceinline__ dfloat uadd_mul(dfloat acc, dfloat a, float m) { return uadd(acc, umul(a, m)); }
__device__ __forceinline__ dfloat addf(dfloat a, float b) { return norm(uadd(a, dfloat{b, 0.0f})); }
// FP32 difference of two nearby values
__device__ __forceinline__ float diff(dfloat a, dfloat b) { return (a.hi - b.hi) + (a.lo - b.lo); }
__device__ __forceinline__ double uadd(double a, double b) { return a + b; }
__device__ __forceinline__ double umul(double a, double b) { return a * b; }
__device__ __forceinline__ double norm(double a) { return a; }
__device__ __forceinline__ double uadd_mul(double acc, double a, double m) { return fma(a, m, acc); }
__device__ __forceinline__ double addf(double a, float b) { return a + (double)b; }
__device__ __forceinline__ float diff(double a, double b) { return (float)(a - b); }
// al + b m - g m^2 (exponent of a factor at node m)
__device__ __forceinline__ double exponent(double al, double b, double g, double m, double q) {
  return fma(-g, q, fma(b, m, al));
}
__device__ __forceinline__ dfloat exponent(dfloat al, dfloat b, dfloat g, float m, float q) {
  const dfloat t = umul(g, q);
  return uadd(uadd(umul(b, m), dfloat{-t.hi, -t.lo}), al);
}
__device__ __forceinline__ bool is_nan(double a) { return !(a == a); }
__device__ __forceinline__ bool is_nan(dfloat a) { return !(a.hi == a.hi); }
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
// 1/x: the FP32 reciprocal and a residual correction of second order (relative error about 2^-46)
__device__ __forceinline__ dfloat recip(dfloat x) {
  const float q = rcp_approx(x.hi);
  float r = fmaf(-q, x.hi, 1.0f);
  r = fmaf(-q, x.lo, r);
  return df_fast_two_sum(q, fmaf(q * r, r, q * r));
}
__device__ __forceinline__ float uadd(float a, float b) { return a + b; }
__device__ __forceinline__ double shfl_i(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ float shfl_i(float v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ dfloat shfl_i(dfloat v, int lane) {
  return {__shfl_sync(0xffffffffu, v.hi, lane), __shfl_sync(0xffffffffu, v.lo, lane)};
}
// FP64 value of a result that is stored: the float halves become doubles by bit operations, which
// leaves one FP64 instruction per value. An FP32 subnormal counts as zero (a double-float field
// ends at 2^-100): widen(), which branches for it, took 2617 -> 2687 us of the scan of 64 cells of
// 32^3 and 9567 -> 9960 us of an ordering of 64 x 64 cells.
__device__ __forceinline__ double f2d_bits(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  unsigned hi = (u & 0x80000000u) | ((m >> 3) + (m >= 0x7f800000u ? 0x70000000u : 0x38000000u));
  unsigned lo = u << 29;
  if (m < 0x00800000u) {
    hi = u & 0x80000000u;
    lo = 0u;
  }
  return __hiloint2double((int)hi, (int)lo);
}
__device__ __forceinline__ double to_store(double x) { return x; }
__device__ __forceinline__ double to_store(dfloat x) { return f2d_bits(x.hi) + f2d_bits(x.lo); }

// 2^(j/64), j = 0..63.
__device__ const double kExp2[64] = {
    1.0, 1.0108892860517005, 1.0218971486541166, 1.0330248790212284,
    1.0442737824274138, 1.0556451783605572, 1.0671404006768237, 1.0787607977571199,
    1.0905077326652577, 1.102382583307841, 1.1143867425958924, 1.1265216186082418,
    1.1387886347566916, 1.1511892299529827, 1.1637248587775775, 1.1763969916502812,
    1.189207115002721, 1.202156731452703, 1.215247359980469, 1.22848053610687,
    1.241857812073484, 1.255380757024691, 1.2690509571917332, 1.2828700160787783,
    1.2968395546510096, 1.3109612115247644, 1.3252366431597413, 1.339667524053303,
    1.3542555469368927, 1.3690024229745905, 1.383909881963832, 1.3989796725383112,
    1.4142135623730951, 1.42961333839197, 1.4451808069770467, 1.460917794180647,
    1.4768261459394993, 1.4929077282912648, 1.5091644275934228, 1.5255981507445384,
    1.5422108254079407, 1.559004400237837, 1.5759808451078865, 1.593142151342267,
    1.6104903319492543, 1.6280274218573478, 1.645755478153965, 1.6636765803267364,
    1.681792830507429, 1.7001063537185235, 1.718619298122478, 1.7373338352737062,
    1.7562521603732995, 1.7753764925265212, 1.7947090750031072, 1.8142521755003989,
    1.8340080864093424, 1.8539791250833855, 1.8741676341103, 1.8945759815869656,
    1.9152065613971474, 1.9360617934922943, 1.9571441241754002, 1.978456026387951};

// exp(x) by table lookup (P. T. P. Tang, Table-driven implementation of the exponential function,
// ACM TOMS 15, 1989): x = (64 j + i) ln2/64 + r, |r| <= ln2/128, exp(x) = 2^j 2^(i/64) exp(r), with
// a Taylor polynomial for exp(r) - 1. In double-float the reduction takes ln2/64 in three
// parts (the first of 11 bits, so that its product with the integer is exact) and only r and
// r^2/2 need both halves; the relative error is that of the argument, about 2^-48 |x|. One
// evaluation by a warp: 115 cycles instead of 485 (degree-13 polynomial in double-float).
__device__ __forceinline__ dfloat exp_tab(dfloat x, const dfloat* T) {
  const float magic = 12582912.0f;  // 1.5 2^23
  const float c1 = 0.01082611083984375f, c2 = 4.3138566e-06f, c3 = -2.0164599e-13f;
  const float t = fmaf(x.hi, 92.332482616893656f, magic);
  const int k = __float_as_int(t);
  const float kf = t - magic;
  const float r1 = fmaf(-kf, c1, x.hi);  // exact
  const float u = r1 + x.lo, ub = u - r1;
  const float ue = (r1 - (u - ub)) + (x.lo - ub);
  const float p = kf * c2, pe = fmaf(kf, c2, -p);
  const float s = u - p, sb = s - u;
  const float se = (u - (s - sb)) - (p + sb);
  const dfloat r = df_fast_two_sum(s, (ue + se) - (pe + kf * c3));
  // m = r + r^2/2 + r^3/6 + r^4/24 + r^5/120
  const float h = 0.5f * r.hi, q2 = h * r.hi, q2e = fmaf(h, r.hi, -q2);
  const float q = fmaf(r.hi, fmaf(r.hi, 0.0083333333f, 0.041666667f), 0.16666667f) * (r.hi * r.hi) * r.hi;
  const float m = r.hi + q2;
  const float me = (q2 - (m - r.hi)) + fmaf(r.hi, r.lo, q2e) + (r.lo + q);
  const dfloat tj = T[k & 63];
  const float ph = tj.hi * m;
  float pl = fmaf(tj.hi, m, -ph);
  pl = fmaf(tj.hi, me, pl);
  pl = fmaf(tj.lo, m, pl);
  const float w = tj.hi + ph;
  const dfloat o = df_fast_two_sum(w, (ph - (w - tj.hi)) + (tj.lo + pl));
  float sc = __int_as_float((int)(((unsigned)(k >> 6) + 127u) << 23));  // the magic number's own bits shift out
  if (!(x.hi >= -87.0f)) sc = x.hi < -87.0f ? 0.0f : x.hi;  // NaN stays
  if (x.hi > 88.0f) sc = __int_as_float(0x7f800000);
  return {o.hi * sc, o.lo * sc};
}
__device__ __forceinline__ double exp_tab(double x, const double* T) {
  const double magic = 6755399441055744.0;  // 1.5 2^52
  const double c1 = 0.010830424696249145, c2 = 3.623510646634843e-19;  // ln2/64 in two parts
  const double t = fma(x, 92.33248261689366, magic);
  const int k = __double2loint(t);
  const double kf = t - magic;
  const double r = fma(-kf, c2, fma(-kf, c1, x));
  double p = fma(r, 1.0 / 720.0, 1.0 / 120.0);
  p = fma(p, r, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  p = fma(p * r, r, r);
  const double tj = T[k & 63];
  const double o = fma(tj, p, tj);
  const int j = k >> 6;
  if (!(x >= -700.0)) return x < -700.0 ? 0.0 : x;
  if (x > 700.0) return __longlong_as_double(0x7ff0000000000000LL);
  return __hiloint2double(__double2hiint(o) + (j << 20), __double2loint(o));
}

// Sum over the warp of 2^m values per lane (NV = 16, 8 or 4): in each step a lane keeps half of
// its values and hands the other half to its partner, so the additions halve from step to step
// (16 values: 8 + 4 + 2 + 1, then one step per remaining lane bit). Lane l returns the total of
// value l * NV / 32 (not renormalised).
template <int NV, typename E>
__device__ __forceinline__ E warp_split_sum(E (&v)[NV], int lane) {
  int o = 16;
#pragma unroll
  for (int h = NV / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < h; q++) {
      const E send = up ? v[q] : v[q + h];
      const E keep = up ? v[q + h] : v[q];
      v[q] = uadd(keep, shfl_x(send, o));
    }
  }
#pragma unroll
  for (int s = 16 / NV; s >= 1; s >>= 1) v[0] = uadd(v[0], shfl_x(v[0], s));
  return v[0];
}

// ---------------------------------------------------------------------------------------
// Cluster-wide sums of kRed values per thread into sm.tot, identical in every CTA (fixed order:
// warp, CTA, cluster ranks). CTA partials are pushed into every CTA's shared memory, so one
// cluster barrier separates them from the final sum; the double buffer keeps a CTA that is
// already in the next reduction from overwriting values that another one still reads.
// ---------------------------------------------------------------------------------------
template <typename E>
__device__ __forceinline__ void cluster_sum(E (&v)[kRed], SweepSmem<E>& sm, int& buf, cg::cluster_group& cl, int CS,
                                            int rank) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  const E t = warp_split_sum<kRed, E>(v, lane);
  if ((lane & 1) == 0) sm.warp_part[lane >> 1][wid] = norm(t);
  __syncthreads();
  if (tid < 8 * kRed) {
    const int q = tid >> 3, k = tid & 7;
    E x = cvt<E>(0.0);
    if (k < nw) x = sm.warp_part[q][k];
    x = uadd(x, shfl_x(x, 1));
    x = uadd(x, shfl_x(x, 2));
    x = norm(uadd(x, shfl_x(x, 4)));
    if (CS == 1) {
      if (k == 0) sm.tot[q] = x;
    } else {
#pragma unroll 1
      for (int r = k; r < CS; r += 8) *cl.map_shared_rank(&sm.part[buf][rank][q], r) = x;
    }
  }
  if (CS > 1) {
    cl.sync();
#pragma unroll 1
    for (int s = tid; s < kRed * CS; s += blockDim.x) {
      const int q = s / CS, r = s % CS;
      E x = sm.part[buf][r][q];
#pragma unroll 1
      for (int o = CS >> 1; o > 0; o >>= 1) x = uadd(x, shfl_x(x, o));
      if (r == 0) sm.tot[q] = norm(x);
    }
    buf ^= 1;
  }
  __syncthreads();
}

// Binary exponents of the peaks exp(b_d^2 / 4 g) of the three factors of exponents th (the first one
// carries exp(th0)), and in sum their sum. The squares that form the norm of M+ - M[g] are taken
// of factors times 2^-k, k fixed for a visit: only the first factor carries exp(alpha), so at a
// tangential speed U the others peak at exp(U^2 / 2T), whose square leaves FP32 from 9.4 thermal
// speeds on, and the first one's differences sink below FP32 from about 7. A power of two changes
// no bit of a norm that was in range.
__device__ __forceinline__ float norm_scale(float th, int d, int& sum) {
  const float al = shfl_i(th, 0), q = 0.25f * rcp_approx(shfl_i(th, 4));
  int kd = 0;
  sum = 0;
#pragma unroll
  for (int t = 0; t < 3; t++) {
    const float b = shfl_i(th, 1 + t);
    const float x = 1.44269504f * ((t == 0 ? al : 0.0f) + b * b * q);
    const int k = (int)rintf(fminf(fmaxf(x, -120.0f), 120.0f));  // (a NaN becomes -120)
    sum += k;
    if (t == d) kd = k;
  }
  return __int_as_float((127 - kd) << 23);
}
// (out of line where E is FP64: in line it takes 0.6 % of an FP64 scan, out of line of a double-float one)
__device__ __noinline__ float norm_scale(double th, int d, int& sum) { return norm_scale((float)th, d, sum); }
__device__ __forceinline__ float norm_scale(dfloat th, int d, int& sum) { return norm_scale(th.hi, d, sum); }

// Barrier among the evaluating warps only (hardware barrier 1; __syncthreads uses 0).
__device__ __forceinline__ void eval_bar(int nwarps) {
  asm volatile("bar.sync 1, %0;" ::"r"(nwarps * 32) : "memory");
}

// ---------------------------------------------------------------------------------------
// One evaluation of the discrete Maxwellian exp(th0 + th1 v1 + th2 v2 + th3 v3 - th4 |v|^2) (lane k
// of th: component k) by evaluating warp `role`, lane = node. Rows of sums, y the factor e of the
// row's dimension times the row's weight:
//   rows 0-2: dimensions 1-3, unweighted; row 3: dimension 1, weight |v1|/dx (step 1);
//   row 4: in 1-D dimension 1, weight 1 / (|v1|/dx + nu/eps) (step 2); in 2-D dimension 2, weight
//   |v2|/dy (step 1).
// Warp r forms row r, and the warp that has the factors of row 4 (warp 3 in 1-D, 1 in 2-D) that
// one too: with four warps each has a scheduler to itself (a fifth shared one, which made every
// iteration 0.65 instead of 0.57 us).
// rows: sum y v^p, p = 0..2, in E; rowsf: the same and p = 3, 4 in FP32, and for rows 0-2 sum
// (e - p)^2 and sum p (e - p), p the factor of the Maxwellian that step 2 used (for the norm of
// M+ - M[g]; with p = 0 the first is sum e^2), of factors times sc (norm_scale); pf = p sc in
// FP32. Returns the lane's factor e.
// ---------------------------------------------------------------------------------------
template <bool TWO_D>
__device__ __forceinline__ int row_dim(int role) {  // dimension of a warp's rows
  return role < 3 ? role : 0;
}
template <bool TWO_D>
__device__ __forceinline__ bool two_rows(int role) {
  return role == (TWO_D ? 1 : 3);
}

template <typename E, bool TWO_D>
__device__ __forceinline__ E eval_row(SweepSmem<E>& sm, int N, E th, int role, int lane, int buf, E p, float sc) {
  typedef typename Node<E>::M M;
  const E zero = cvt<E>(0.0);
  const int d = row_dim<TWO_D>(role);
  const M m = (M)(lane + 1 - N / 2), q = m * m;
  const float mf = (float)m, qf = (float)q;
  const E b = shfl_i(th, 1 + d), g = shfl_i(th, 4), al = shfl_i(th, 0);
  E e = zero;
  if (lane < N) e = exp_tab(exponent(d == 0 ? al : zero, b, g, m, q), sm.etab);
  const float df = diff(e, p) * sc, pf = tof(p) * sc;
  const E y = role == 3 ? e * sm.c1e[lane] : e;
  const E y2 = umul(y, q);
  const float f3 = tof(y2) * mf, f4 = tof(y2) * qf;
  E t;
  float tf;
  int k = lane >> 3, row = role, kf = 3 + k;
  if (two_rows<TWO_D>(role)) {
    const E z = e * (TWO_D ? sm.c2e[lane] : sm.den[lane]);
    const E z2 = umul(z, q);
    E s[8] = {y, umul(y, m), y2, zero, z, umul(z, m), z2, zero};
    float f[8] = {f3, f4, df * df, pf * df, tof(z2) * mf, tof(z2) * qf, 0.0f, 0.0f};
    t = warp_split_sum<8, E>(s, lane);
    tf = warp_split_sum<8, float>(f, lane);
    k = (lane >> 2) & 3;
    row = lane < 16 ? role : 4;
    kf = 3 + k;
    if ((lane & 3) != 0) k = kf = -1;
  } else {
    E s[4] = {y, umul(y, m), y2, zero};
    float f[4] = {f3, f4, df * df, pf * df};
    t = warp_split_sum<4, E>(s, lane);
    tf = warp_split_sum<4, float>(f, lane);
    if ((lane & 7) != 0) k = kf = -1;
  }
  if (kf >= 0) {
    const E tn = norm(t);
    if (k < 3) {
      sm.rows[buf][row][k] = tn;
      sm.rowsf[buf][row][k] = tof(tn);
    }
    sm.rowsf[buf][row][kf] = tf;
  }
  return e;
}

// The last step of a Newton solve: a step whose exponent change is at most kLinear moves every
// factor by e -> e (1 + dx), dx = -(y0 + y_d v + y4 v^2) (second order: dx^2 / 2, below the rounding
// of E), so the sums
// of powers 0-2 follow from those of powers 0-4 and no exponential and no reduction is needed.
// What the step leaves of the residual is FP32 rounding of its direction: 1e-6 of the step for a
// gas at rest, up to 1e-6 (1 + U^2/T) for one that moves, as its cumulants come from raw moments. So
// does the residual itself, in E, which loses more than this step does: 72 cells each at 5 to 12
// thermal speeds differ from FP64 by 8e-13 to 3e-12 of max f with this step, with every step
// evaluated, and with a step that counts (1 + U^2/T) times (0.8 to 1.8 % slower). Reads buffer buf ^ 1 (every warp is past its
// barrier), writes buffer buf; y: the direction (the step is -y, +y4). Returns the new factor.
template <typename E>
constexpr float kLinear = sizeof(typename Node<E>::M) == 8 ? 1e-8f : 1e-7f;
template <typename E, bool TWO_D>
__device__ __forceinline__ E linear_row(SweepSmem<E>& sm, int N, const float (&y)[5], int role, int lane, int buf, E e,
                                        E p, float sc) {
  const int d = row_dim<TWO_D>(role);
  const float yd = d == 0 ? y[1] : (d == 1 ? y[2] : y[3]), ya = d == 0 ? y[0] : 0.0f;
  const float m = (float)(lane + 1 - N / 2);
  e = addf(e, -tof(e) * (ya + m * (yd + m * y[4])));
  const float df = diff(e, p) * sc;
  float f[2] = {df * df, tof(p) * sc * df};
  const float t = warp_split_sum<2, float>(f, lane);
  // lanes 0-4: the warp's own row, lanes 8-12: row 4
  const int k = lane & 7, row = lane < 8 ? role : 4;
  if (lane < (two_rows<TWO_D>(role) ? 16 : 8) && k < 5) {
    const float* s = sm.rowsf[buf ^ 1][row];
    float r = s[k];
    if (k < 3) {
      const E x = addf(sm.rows[buf ^ 1][row][k], -(ya * s[k] + yd * s[k + 1] + y[4] * s[k + 2]));
      sm.rows[buf][row][k] = x;
      r = tof(x);
    }
    sm.rowsf[buf][row][k] = r;
  }
  if ((lane & 15) == 15) sm.rowsf[buf][role][5 + (lane >> 4)] = t;
  return e;
}

// Lane k < 5 receives moment k (of 1, v1, v2, v3, |v|^2) of the product of three 1-D measures
// given by their sums; lanes 4-6 form the three parts of the last one. Other lanes return unused
// values.
template <typename E>
__device__ __forceinline__ E lane_moment(const E* r1, const E* r2, const E* r3, int lane) {
  const int k = lane & 7;
  const int i = k == 1 ? 1 : (k == 4 ? 2 : 0), j = k == 2 ? 1 : (k == 5 ? 2 : 0), l = k == 3 ? 1 : (k == 6 ? 2 : 0);
  const E x = umul(r1[i], norm(umul(r2[j], r3[l])));
  const E t5 = shfl_i(x, 5), t6 = shfl_i(x, 6);
  const E s = uadd(x, uadd(t5, t6));
  return norm(lane == 4 ? s : x);
}

// Newton direction y = A^{-1} F (FP32), A = sum m psi psi^T, psi = (1, v1, v2, v3, |v|^2), for a
// product measure m of 1-D sums r1, r2, r3 (powers 0..4). The functions 1, c_d = v_d - U_d and
// |c|^2 - sum V_d - sum (k3_d / V_d) c_d (U, V, k3: the 1-D means, variances and third central
// moments) are orthogonal under m, so A^{-1} needs no factorisation. prepare() is the part
// that does not need F: it overlaps the formation of the moments.
struct ProductMeasure {
  float U[3], iv[3], b[3];  // means, 1/variances, 2 U + k3/V
  float in0, wa, wb, a4s;   // 1/mass; weights of F0 in the last coefficient, of it in y0; its scale
  bool ok;                  // the measure is numerically positive
  __device__ __forceinline__ void prepare(const float* r1, const float* r2, const float* r3) {
    const float* r[3] = {r1, r2, r3};
    float q4[3];
    float n0 = r1[0] * r2[0] * r3[0];
    ok = r1[0] > 0.0f && r2[0] > 0.0f && r3[0] > 0.0f;
    wa = wb = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const float i0 = rcp_approx(r[d][0]);
      const float u = r[d][1] * i0, m2 = r[d][2] * i0, m3 = r[d][3] * i0, m4 = r[d][4] * i0;
      const float uu = u * u;
      const float var = m2 - uu;
      const float k3 = m3 - u * (3.0f * m2 - 2.0f * uu);
      const float k4 = m4 - u * (4.0f * m3 - u * (6.0f * m2 - 3.0f * uu));
      ok = ok && var > 0.0f;
      iv[d] = rcp_approx(var);
      const float kappa = k3 * iv[d];
      q4[d] = k4 - var * var - kappa * k3;
      U[d] = u;
      b[d] = 2.0f * u + kappa;
      wa += b[d] * u - (uu + var);
      wb += uu - var + kappa * u;
    }
    const float q = q4[0] + q4[1] + q4[2];
    ok = ok && q > 0.0f;
    in0 = rcp_approx(n0);
    a4s = in0 * rcp_approx(q);
  }
  __device__ __forceinline__ void direction(const float (&F)[5], float (&y)[5]) const {
    const float a4 = a4s * ((F[4] + wa * F[0]) - (b[0] * F[1] + b[1] * F[2] + b[2] * F[3]));
    float y0 = F[0] * in0 + a4 * wb;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const float ad = (F[1 + d] - U[d] * F[0]) * (in0 * iv[d]);
      y[1 + d] = ad - a4 * b[d];
      y0 -= ad * U[d];
    }
    y[0] = y0;
    y[4] = a4;
  }
};

// Upper triangle (row-major) of sum m psi psi^T for a product measure, added to A (FP32).
__device__ __forceinline__ void add_gram(const float* f1, const float* f2, const float* f3, float (&A)[15]) {
  const float q11 = f1[2] * f2[0] * f3[0], q22 = f1[0] * f2[2] * f3[0], q33 = f1[0] * f2[0] * f3[2];
  const float c1 = f1[3] * f2[0] * f3[0] + f1[1] * f2[2] * f3[0] + f1[1] * f2[0] * f3[2];
  const float c2 = f1[2] * f2[1] * f3[0] + f1[0] * f2[3] * f3[0] + f1[0] * f2[1] * f3[2];
  const float c3 = f1[2] * f2[0] * f3[1] + f1[0] * f2[2] * f3[1] + f1[0] * f2[0] * f3[3];
  const float e4 = f1[4] * f2[0] * f3[0] + f1[0] * f2[4] * f3[0] + f1[0] * f2[0] * f3[4] +
                   2.0f * (f1[2] * f2[2] * f3[0] + f1[2] * f2[0] * f3[2] + f1[0] * f2[2] * f3[2]);
  const float t[15] = {f1[0] * f2[0] * f3[0], f1[1] * f2[0] * f3[0], f1[0] * f2[1] * f3[0], f1[0] * f2[0] * f3[1],
                       q11 + q22 + q33, q11, f1[1] * f2[1] * f3[0], f1[1] * f2[0] * f3[1], c1, q22,
                       f1[0] * f2[1] * f3[1], c2, q33, c3, e4};
#pragma unroll
  for (int i = 0; i < 15; i++) A[i] += t[i];
}

// Continuum Maxwellian of five moments (sums over the nodes in units of dv): the guess that
// replaces a warm start from which Newton failed. Rare, kept out of line.
__device__ __noinline__ bool guess_theta(double dv, double m0, double m1, double m2, double m3, double m4, double* th) {
  const double w = dv * dv * dv;
  const double m[5] = {w * m0, w * dv * m1, w * dv * m2, w * dv * m3, w * dv * dv * m4};
  const bool ok = continuum_guess<double>(m, th);
  for (int k = 1; k < 4; k++) th[k] *= dv;
  th[4] *= dv * dv;
  return ok;
}

// Relaxed step 1 (the remark after eq. (26)) where eq. (26) fails for the target s: with a
// factor 1 + tau on the weighted moments of the new and the current Maxwellian the target
// becomes (tau m_w + s)/(1 + tau), m_w = sum phi c M[g]. 1 + tau = 2, 4, 8, ...: the first
// target that passes eq. (26) is left in s. Lane k holds component k; uniform over the warp.
template <typename E>
__device__ __noinline__ bool relax_target(E mw, E& s, int lane) {
  const double m = tod(mw), s0 = tod(s);
#pragma unroll 1
  for (double q = 2.0; q <= 1048576.0; q *= 2.0) {
    const double t = ((q - 1.0) * m + s0) / q;
    double b[5];
#pragma unroll
    for (int k = 0; k < 5; k++) b[k] = shfl_i(t, k);
    if (b[0] > 0.0 && b[0] * b[4] > b[1] * b[1] + b[2] * b[2] + b[3] * b[3]) {
      s = cvt<E>(t);
      return true;
    }
  }
  return false;
}

// One run of a field. WIDE: the fields start on 16 bytes. A field on 8 (a view into a larger array)
// is read and written by single values, in a kernel of its own: a test of the addresses in the
// kernel took 2 % of the scan of 64 cells of 32^3.
template <bool WIDE>
__device__ __forceinline__ void load_run(const double* p, double (&x)[R]) {
  if (WIDE) {
#pragma unroll
    for (int t = 0; t < R; t += 2) {
      const double2 v = *reinterpret_cast<const double2*>(p + t);
      x[t] = v.x;
      x[t + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int t = 0; t < R; t++) x[t] = p[t];
  }
}

// What a cell visit reads besides the tables: the cell's own value, its penalty and right-hand
// side, its neighbours (null at a wall), collision frequency and Maxwellian exponents.
struct CellIO {
  double* f;
  const double* P;
  const double* b;        // nullable
  const double* nb[4];    // x_lo, x_hi, y_lo, y_hi neighbours; null: wall ghost
  double nu;
  const double* theta;
};

struct Tally {
  unsigned long long inner = 0, newton = 0, solves = 0, fallback = 0;
  unsigned status = 0;
};

// Tables of a launch: nodes, transport weights, wall Maxwellians.
template <typename E, bool TWO_D>
__device__ __forceinline__ void scan_tables(SweepSmem<E>& sm, const InstDev& I, int N, double dv) {
  const int tid = threadIdx.x;
  if (tid < kMaxN) {
    const double v = tid < N ? node(tid, N, dv) : 0.0;
    sm.c1e[tid] = cvt<E>(fabs(v) * I.inv_dx);
    sm.c2e[tid] = TWO_D ? cvt<E>(fabs(v) * I.inv_dy) : cvt<E>(0.0);
    const double m = tid + 1 - N / 2;
    sm.vm[0][tid] = m;
    sm.vm[1][tid] = m * m;
  }
#pragma unroll 1
  for (int t = tid; t < (TWO_D ? 4 : 2) * 3 * kMaxN; t += blockDim.x)
    (&sm.W[0][0][0])[t] = cvt<E>((&I.wall[0][0][0])[t]);
  if (tid < 64) sm.etab[tid] = cvt<E>(kExp2[tid]);
}

// ---------------------------------------------------------------------------------------
// The visit of one cell by one cluster. rbuf: this CTA's r (its runs, thread-private slots);
// den2 (2-D): 1 / (|v1|/dx + |v2|/dy + nu/eps) at [i2][i1].
// ---------------------------------------------------------------------------------------
template <typename E, bool TWO_D, bool WIDE>
__device__ __forceinline__ void visit_cell(const SweepArgs& a, const InstDev& I, SweepSmem<E>& sm, E* rbuf, E* den2,
                                           const CellIO& io, cg::cluster_group& cl, int CS, int rank, int& buf,
                                           Tally& ty) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  typedef typename Node<E>::M M;
  const int N = a.N;
  constexpr int nev = kTeam;
  const E zero = cvt<E>(0.0);
  const E inv_eps = cvt<E>(I.inv_eps);
  const E A = cvt<E>(io.nu) * inv_eps;
  const bool team = wid < nev;

  // ---- the cell's coefficients, and the factors and sums of the collision step's Maxwellian
  if (TWO_D) {
#pragma unroll 1
    for (int t = tid; t < N * N; t += blockDim.x) {
      const int i2 = t / N, i1 = t - i2 * N;
      den2[t] = recip(sm.c1e[i1] + sm.c2e[i2] + A);
    }
  } else if (tid < kMaxN) {  // nodes beyond N have finite entries too: they meet zero factors
    const E c = sm.c1e[tid] + A;
    sm.cA[tid] = c;
    sm.den[tid] = recip(c);
  }
  const int kl = min(lane & 7, 4);  // this lane's component of exponents, targets and moments
  E th = zero;
  if (team) th = cvt<E>(io.theta[kl]) * cvt<E>(kl == 0 ? 1.0 : (kl < 4 ? a.dv : a.dv * a.dv));
  int cur = 0;  // buffer of the latest evaluation
  E e = zero;   // the lane's factor in it (roles 0-2)
  int ksum = 0;
  float sc = 1.0f;
  if (team) sc = norm_scale(th, row_dim<TWO_D>(wid), ksum);
  if (!TWO_D) __syncthreads();  // sm.den before role 4 reads it
  if (team) {
    e = eval_row<E, TWO_D>(sm, N, th, wid, lane, cur, zero, sc);
    if (wid < 3) sm.ef[wid][lane] = e;
  }
  __syncthreads();

  // ---- passes over the nodes, each followed by a cluster reduction: 0 the outgoing wall
  //      fluxes (wall cells; the ghosts need their density), 1 r and every sum of the solve, 2
  //      the same again for the residual, where Newton moved M[g] off the factors of pass 1
  bool any_flux = false;
#pragma unroll
  for (int s = 0; s < (TWO_D ? 4 : 2); s++) any_flux = any_flux || (!io.nb[s] && I.bc_kind[s] != SGS_INFLOW);
  if (tid < (TWO_D ? 4 : 2) && I.bc_kind[tid] == SGS_INFLOW) sm.rho[tid] = cvt<E>(I.bc_rho[tid]);
  if (!io.nb[0] || !io.nb[1] || (TWO_D && (!io.nb[2] || !io.nb[3]))) __syncthreads();

  const int runs = N * N * N / R, per = (runs + CS - 1) / CS;
  const int lo = rank * per, hi = min(runs, lo + per);
  const int prun = N / R;  // runs per pencil

  E thg = zero, eg = zero;
  float QQ[3];
  E momg = zero, tu = zero, Dl = zero, mw = zero, tgt = zero;  // lane k: component k
  E res2 = zero;
  int pass = any_flux ? 0 : 1;
#pragma unroll 1
  for (;;) {
    E v[kRed];
#pragma unroll
    for (int q = 0; q < kRed; q++) v[q] = zero;
    int slot = tid;
#pragma unroll 1
    for (int run = lo + tid; run < hi; run += blockDim.x, slot += R * blockDim.x) {
      const int pen = run / prun, i30 = (run - pen * prun) * R;
      const int i1 = pen / N, i2 = pen - i1 * N;
      const int e0 = run * R;
      const int sgn1 = i1 + 1 - N / 2, sgn2 = i2 + 1 - N / 2;  // v1, v2 in units of dv
      const M v1 = node_m<M, TWO_D>(sm.vm, i1, N), v2 = node_m<M, TWO_D>(sm.vm, i2, N);
      double x[R];
      load_run<WIDE>(io.f + e0, x);
      if (pass == 0) {
        E p0 = zero;
#pragma unroll
        for (int t = 0; t < R; t++) p0 = uadd(p0, cvt<E>(x[t]));
        p0 = norm(p0);
        if (!io.nb[0] && sgn1 < 0) v[0] = uadd_mul(v[0], p0, v1);
        if (!io.nb[1] && sgn1 > 0) v[1] = uadd_mul(v[1], p0, v1);
        if (TWO_D) {
          if (!io.nb[2] && sgn2 < 0) v[2] = uadd_mul(v[2], p0, v2);
          if (!io.nb[3] && sgn2 > 0) v[3] = uadd_mul(v[3], p0, v2);
        }
        continue;
      }
      const E e12 = sm.ef[0][i1] * sm.ef[1][i2];
      E cw, cAw, dn;
      if (TWO_D) {
        cw = sm.c1e[i1] + sm.c2e[i2];
        cAw = cw + A;
        dn = den2[i2 * N + i1];
      } else {
        cw = sm.c1e[i1];
        cAw = sm.cA[i1];
        dn = sm.den[i1];
      }
      {
        // r = -(|v1|/dx) f_up,x - (|v2|/dy) f_up,y - P/eps - b (upwind neighbours: latest values)
        double pv[R], u1[R], u2[R], bv[R];
        load_run<WIDE>(io.P + e0, pv);
        const int s1 = sgn1 > 0 ? 0 : 1, s2 = sgn2 > 0 ? 2 : 3;
        const double* up1 = sgn1 > 0 ? io.nb[0] : io.nb[1];
        const double* up2 = TWO_D ? (sgn2 > 0 ? io.nb[2] : io.nb[3]) : nullptr;
        const bool g1 = sgn1 != 0 && !up1, g2 = TWO_D && sgn2 != 0 && !up2;
        if (sgn1 != 0 && up1) load_run<WIDE>(up1 + e0, u1);
        if constexpr (TWO_D) {
          if (sgn2 != 0 && up2) load_run<WIDE>(up2 + e0, u2);
        }
        if (io.b) load_run<WIDE>(io.b + e0, bv);
        auto ghost = [&](int side, double(&u)[R]) {
          const E w12 = sm.rho[side] * (sm.W[side][0][i1] * sm.W[side][1][i2]);
#pragma unroll
          for (int t = 0; t < R; t++) u[t] = to_store(w12 * sm.W[side][2][i30 + t]);
        };
        if (g1) ghost(s1, u1);
        if constexpr (TWO_D) {
          if (g2) ghost(s2, u2);
        }
        const E c1 = sm.c1e[i1], c2 = sm.c2e[i2];
        E p0 = zero, p3 = zero, p4 = zero, q0 = zero, q3 = zero, q4 = zero;
#pragma unroll
        for (int t = 0; t < R; t++) {
          const int i3 = i30 + t;
          const M v3 = node_m<M, TWO_D>(sm.vm, i3, N), vq3 = node_q<M, TWO_D>(sm.vm, i3, v3);
          const E g = cvt<E>(x[t]);
          E r = -umul(cvt<E>(pv[t]), inv_eps);
          if (sgn1 != 0) r = uadd(r, -umul(c1, cvt<E>(u1[t])));
          if constexpr (TWO_D) {
            if (sgn2 != 0) r = uadd(r, -umul(c2, cvt<E>(u2[t])));
          }
          if (io.b) r = uadd(r, -cvt<E>(bv[t]));
          r = norm(r);
          rbuf[slot + t * blockDim.x] = r;
          p0 = uadd(p0, g);
          p3 = uadd_mul(p3, g, v3);
          p4 = uadd_mul(p4, g, vq3);
          q0 = uadd(q0, r);
          q3 = uadd_mul(q3, r, v3);
          q4 = uadd_mul(q4, r, vq3);
          // cell-equation residual at M of the collision step
          const E res = norm(uadd(uadd(umul(cAw, g), r), -umul(A, norm(umul(e12, sm.ef[2][i3])))));
          v[15] = uadd(v[15], umul(res, res));
        }
        const M vq12 = v1 * v1 + v2 * v2;
        p0 = norm(p0), p3 = norm(p3), p4 = norm(p4), q0 = norm(q0), q3 = norm(q3), q4 = norm(q4);
        // moments of g, of c g + r (step-1 target) and of r / (c + A) (step 2)
        const E z0[3] = {p0, norm(uadd(umul(cw, p0), q0)), norm(umul(dn, q0))},
                z3[3] = {p3, uadd(umul(cw, p3), q3), umul(dn, q3)},
                z4[3] = {p4, uadd(umul(cw, p4), q4), umul(dn, q4)};
#pragma unroll
        for (int k = 0; k < 3; k++) {
          v[5 * k] = uadd(v[5 * k], z0[k]);
          v[5 * k + 1] = uadd_mul(v[5 * k + 1], z0[k], v1);
          v[5 * k + 2] = uadd_mul(v[5 * k + 2], z0[k], v2);
          v[5 * k + 3] = uadd(v[5 * k + 3], z3[k]);
          v[5 * k + 4] = uadd(uadd_mul(v[5 * k + 4], z0[k], vq12), z4[k]);
        }
      }
    }
    cluster_sum<E>(v, sm, buf, cl, CS, rank);
    if (pass == 0) {
      if (tid < (TWO_D ? 4 : 2) && I.bc_kind[tid] != SGS_INFLOW) sm.rho[tid] = cvt<E>(I.wall_scale[tid]) * sm.tot[tid];
      __syncthreads();
      pass = 1;
      continue;
    }
    if (pass == 1 && !team) {
      __syncthreads();  // with the evaluating warps' barrier below
      if (sm.ctl & 2) {
        pass = 2;
        continue;
      }
      break;
    }
    if (pass == 2 && !team) break;

    // ---- evaluating warps
    const float Lf = (float)(N / 2);  // largest node
    const float ntol = (float)I.newton_tol, dvf = (float)a.dv;
    // converged as well once the scaled moment residual |F|/rho is at the arithmetic's
    // resolution (double-float and FP64 evaluate F to about 1e-14): with the residual already
    // there, a further step could only confirm it
    constexpr float ftol = 1e-13f;
    const bool pfp = I.inner_method != SGS_FP, relax = I.inner_method == SGS_PFP_RELAX;
    // inner_tol^2 / w in the units of the scaled norm; a positive tolerance stays positive
    const double tol2 = I.tol2_w;
    const float tol2f = tol2 > 0.0 ? fmaxf((float)(tol2 * __hiloint2double((1023 - 2 * ksum) << 20, 0)), FLT_MIN) : 0.0f;
    const int inner_fixed = I.inner_fixed, inner_max = I.inner_max, newton_max = I.newton_max;
    int it = 0;
    res2 = sm.tot[15];
    if (pass == 1) {
      momg = sm.tot[kl];
      tu = sm.tot[5 + kl];
      Dl = sm.tot[10 + kl];
    }

    enum { S_G0, S_P, S_PF, S_G };
    int state = S_G0, stage = 0;
    int have = 1, force = pass == 2, moved = 0;
    bool used = false, stop = false;
    E p = zero, momP = zero;
    float PP[3] = {0.0f, 0.0f, 0.0f};
    tgt = momg;
    if (pass == 2) {  // back from the residual pass: M[g] is solved already, its evaluation is the latest one
      th = thg;
      e = eg;
    }
    E keep = th;

#pragma unroll 1
    for (;;) {  // one Newton solve per round: target tgt, start th, weights by state
      // one copy of the solve for all states (the loop has to stay in the instruction caches)
      asm volatile("" : "+r"(state), "+r"(stage), "+r"(force));
      int ret;
      {
        const bool wtd = state == S_P;
        const E psub = state == S_G ? p : zero;
        const float it0 = rcp_approx(fabsf(shfl_i(tof(tgt), 0)));
        float fn_cur = 0.0f, lam = 1.0f, stepf = 0.0f, y[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        int itn = -1, hv = 0;  // itn < 0: at the start
        E tr = th;
        float yl = 0.0f;  // this lane's component of the step
#pragma unroll 1
        for (;;) {
          asm volatile("" : "+r"(have), "+r"(itn), "+r"(hv), "+r"(cur));
          if (!have) {
            cur ^= 1;
            e = eval_row<E, TWO_D>(sm, N, tr, wid, lane, cur, psub, sc);
            eval_bar(nev);
            moved = 1;
          }
          have = 0;
          const E(*rw)[4] = sm.rows[cur];
          const float(*rf)[8] = sm.rowsf[cur];
          ProductMeasure pm;
          if (!TWO_D || !wtd) pm.prepare(wtd ? rf[3] : rf[0], rf[1], rf[2]);
          E F = lane_moment<E>(wtd ? rw[3] : rw[0], rw[1], rw[2], lane);
          if (TWO_D && wtd) F = F + lane_moment<E>(rw[0], rw[4], rw[2], lane);
          const float Fl = diff(F, tgt);  // this lane's component of the residual
          float Ff[5];
#pragma unroll
          for (int k = 0; k < 5; k++) Ff[k] = shfl_i(Fl, k);
          // largest component, in units of the velocity; fmaxf drops a NaN, the sum keeps it
          float fn = fmaxf(fmaxf(fabsf(Ff[0]), dvf * fmaxf(fmaxf(fabsf(Ff[1]), fabsf(Ff[2])), fabsf(Ff[3]))),
                           dvf * dvf * fabsf(Ff[4]));
          fn = fmaf(0.0f, (Ff[0] + Ff[1]) + (Ff[2] + Ff[3]) + Ff[4], fn * it0);
          if (itn < 0) {
            fn_cur = fn;
            itn = 0;
            if (fn <= ftol || force) {
              ret = 0;
              break;
            }
          } else {
            const bool ok = fn == fn && (fn <= fn_cur || fn <= 1e-10f);
            if (!ok && ++hv < 40) {
              lam *= 0.5f;
              tr = addf(th, lam * yl);
              continue;
            }
            if (ok) fn_cur = fn;
            th = tr;
            itn++;
            const float step = lam * stepf;
            if (!(step == step)) {
              ret = -1;
              break;
            }
            if (step <= ntol || fn_cur <= ftol) {
              ret = itn;
              break;
            }
            if (itn >= newton_max) {
              ret = -1;
              break;
            }
          }
          bool pos;
          if (TWO_D && wtd) {
            float G[15];
#pragma unroll
            for (int k = 0; k < 15; k++) G[k] = 0.0f;
            add_gram(rf[3], rf[1], rf[2], G);
            add_gram(rf[0], rf[4], rf[2], G);
            pos = chol5_solve(G, Ff, y);
          } else {
            pm.direction(Ff, y);
            pos = pm.ok;
          }
          if (!pos) {
            ret = -1;
            break;
          }
          // exponent change of a full step, |d alpha| + L sum |d beta| + L^2 |d gamma|; the step is
          // -D A^{-1} F with D = diag(1, 1, 1, 1, -1)
          stepf = fabsf(y[0]) + Lf * (fabsf(y[1]) + fabsf(y[2]) + fabsf(y[3])) + Lf * Lf * fabsf(y[4]);
          yl = kl == 0 ? -y[0] : (kl == 1 ? -y[1] : (kl == 2 ? -y[2] : (kl == 3 ? -y[3] : y[4])));
          tr = addf(th, yl);
          if (stepf <= kLinear<E>) {
            cur ^= 1;
            e = linear_row<E, TWO_D>(sm, N, y, wid, lane, cur, e, psub, sc);
            eval_bar(nev);
            moved = 1;
            th = tr;
            ret = itn + 1;
            break;
          }
          lam = 1.0f;
          hv = 0;
        }
      }
      const bool forced = force != 0;
      force = 0;

      bool step2 = false;
      if (state == S_P) {
        ty.solves++;
        if (ret >= 0) {
          ty.newton += ret;
          used = true;
          p = e;
#pragma unroll
          for (int d = 0; d < 3; d++) PP[d] = moved ? sm.rowsf[cur][d][5] : QQ[d];
          step2 = true;
        } else {  // the latest evaluation is not M[g]'s: repeat that one, then the plain step
          th = thg;
          have = 0;
          force = 1;
          state = S_PF;
          continue;
        }
      } else if (state == S_PF) {
        step2 = true;
      } else {
        // M[g]: a failed warm start is followed by the continuum Maxwellian of the same moments,
        // a second failure keeps the start (reported)
        if (ret < 0) {
          bool again = false;
          if (stage == 0) {
            double m[5], tg[5];
#pragma unroll
            for (int k = 0; k < 5; k++) m[k] = tod(shfl_i(tgt, k));
            if (guess_theta(a.dv, m[0], m[1], m[2], m[3], m[4], tg)) {
              th = cvt<E>(kl == 0 ? tg[0] : (kl == 1 ? tg[1] : (kl == 2 ? tg[2] : (kl == 3 ? tg[3] : tg[4]))));
              stage = 1;
              again = true;
            } else {
              ty.status |= SGS_ST_NONPOSITIVE;
            }
          }
          if (!again) {
            ty.status |= SGS_ST_NEWTON_FAIL;
            th = keep;
            stage = 2;
            force = 1;
          }
          have = 0;
          continue;
        }
        if (!(forced && pass == 2 && state == S_G0)) ty.solves++;
        if (!forced) ty.newton += ret;
        thg = th;
        eg = e;
        const E(*rw)[4] = sm.rows[cur];
        const float(*rf)[8] = sm.rowsf[cur];
        mw = lane_moment<E>(rw[3], rw[1], rw[2], lane);
        if (TWO_D) mw += lane_moment<E>(rw[0], rw[4], rw[2], lane);
        E s;
        bool small, nan;
        if (state == S_G0) {
          if (pass == 1 && moved) {
            // pass 1 formed the residual with other factors: form it again where it decides
            if (wid < 3) sm.ef[wid][lane] = eg;
            if (inner_fixed == 0) {
              if (tid == 0) sm.ctl = 2;
              break;
            }
          }
#pragma unroll
          for (int d = 0; d < 3; d++) QQ[d] = rf[d][5];
          s = mw - tu;
          momg = tgt;
          small = to_store(res2) < tol2;  // in FP64: a double-float ends at 2^-100
          nan = is_nan(res2);
        } else {
          // norm of R = A (M+ - M[g]) and the next step-1 target from the step-2 identity
          // c g + r = A M+ - A g: with d = Q - P per dimension (P, Q the factors of M+ and M[g]),
          // Q1Q2Q3 - P1P2P3 = d1 P2 P3 + Q1 d2 P3 + Q1 Q2 d3, its square from sums per dimension
          // (PP, Pd, dd given; PQ = PP + Pd, dQ = Pd + dd, QQ = PQ + dQ). FP32: it only meets the
          // tolerance, and the differences were formed in E
          float dd[3], Pd[3], PQ[3], dQ[3];
#pragma unroll
          for (int d = 0; d < 3; d++) {
            dd[d] = moved ? rf[d][5] : 0.0f;
            Pd[d] = moved ? rf[d][6] : 0.0f;
            PQ[d] = PP[d] + Pd[d];
            dQ[d] = Pd[d] + dd[d];
            QQ[d] = PQ[d] + dQ[d];
          }
          const float cross = dQ[0] * Pd[1] * PP[2] + dQ[0] * PQ[1] * Pd[2] + QQ[0] * dQ[1] * Pd[2];
          const float nrm = tof(A) * tof(A) *
                            (dd[0] * PP[1] * PP[2] + QQ[0] * dd[1] * PP[2] + QQ[0] * QQ[1] * dd[2] + 2.0f * cross);
          s = mw - A * momP + A * tgt;
          momg = tgt;
          small = nrm < tol2f;
          nan = !(nrm == nrm);
        }
        if (inner_fixed > 0) {
          stop = it >= inner_fixed;
        } else {
          stop = small || it >= inner_max;
          if (stop && !small) ty.status |= SGS_ST_INNER_CAP;
        }
        if (nan) {
          ty.status |= SGS_ST_NONFINITE;
          stop = true;
        }
        if (stop) break;
        // existence test of step 1 (eq. (26)): s0 s4 > s1^2 + s2^2 + s3^2; where the FP32 values
        // leave it open (the ends of their range among it), in FP64
        const float sf = tof(s);
        const float f0 = shfl_i(sf, 0), f1 = shfl_i(sf, 1), f2 = shfl_i(sf, 2), f3 = shfl_i(sf, 3),
                    f4 = shfl_i(sf, 4);
        const float pl = f0 * f4, mi = f1 * f1 + f2 * f2 + f3 * f3, mag = fabsf(pl) + mi;
        bool exists = pfp && f0 > 0.0f && pl > mi;
        if (pfp && !(mag > 1e-25f && mag < 1e25f && fabsf(pl - mi) > 1e-5f * mag)) {
          const double sd = tod(s);
          const double x0 = shfl_i(sd, 0), x1 = shfl_i(sd, 1), x2 = shfl_i(sd, 2), x3 = shfl_i(sd, 3), x4 = shfl_i(sd, 4);
          exists = x0 > 0.0 && x0 * x4 > x1 * x1 + x2 * x2 + x3 * x3;
        }
        if (relax && !exists) exists = relax_target<E>(mw, s, lane);
        used = false;
        moved = 0;
        if (exists) {  // step 1 (eq. (24)); the latest evaluation is M[g]'s: reused as its first
          tgt = s;
          have = 1;
          state = S_P;
          continue;
        }
        step2 = true;
      }

      if (step2) {
        // ---- step 2 (eq. (25)) on the moments: from M+ (else M[g]: the fixed-point step, eq. (22))
        if (!used) {
          if (pfp) ty.fallback++;
          p = eg;
#pragma unroll
          for (int d = 0; d < 3; d++) PP[d] = QQ[d];
        }
        momP = used ? lane_moment<E>(sm.rows[cur][0], sm.rows[cur][1], sm.rows[cur][2], lane) : momg;
        E z;
        if (TWO_D) {
          // sum over (v1, v2) of E1 E2 / (c + A) times 1, v1, v2, v1^2 + v2^2: lane = v1, the v2 nodes
          // over the evaluating warps
          if (wid < 2) sm.ef[wid][lane] = p;
          eval_bar(nev);
          E w0 = zero, w1 = zero, w2 = zero;
          if (lane < N) {
#pragma unroll 1
            for (int i2 = wid; i2 < N; i2 += nev) {
              const E t = norm(umul(den2[i2 * N + lane], sm.ef[1][i2]));
              const M m2 = node_m<M, TWO_D>(sm.vm, i2, N);
              w0 = uadd(w0, t);
              w1 = uadd_mul(w1, t, m2);
              w2 = uadd_mul(w2, t, node_q<M, TWO_D>(sm.vm, i2, m2));
            }
          }
          const E e1 = lane < N ? sm.ef[0][lane] : zero;
          const M m1 = (M)(lane + 1 - N / 2);
          w0 = norm(umul(norm(w0), e1));
          E q4[4] = {w0, umul(w0, m1), umul(norm(w1), e1), uadd_mul(umul(norm(w2), e1), w0, m1 * m1)};
          const E t = warp_split_sum<4, E>(q4, lane);
          if ((lane & 7) == 0) sm.dpart[wid][lane >> 3] = norm(t);
          eval_bar(nev);
          // lane k: moment k; the slots of dimension 3 are powers of v3
          const int c = kl == 1 ? 1 : (kl == 2 ? 2 : (kl == 4 ? 3 : 0));
          E y0 = zero, y1 = zero;
#pragma unroll
          for (int k = 0; k < nev; k++) {
            y0 += sm.dpart[k][0];
            y1 += sm.dpart[k][c];
          }
          const E* r3 = sm.rows[cur][2];
          z = kl == 3 ? y0 * r3[1] : y1 * r3[0];
          if (kl == 4) z += y0 * r3[2];
        } else {
          z = lane_moment<E>(sm.rows[cur][4], sm.rows[cur][1], sm.rows[cur][2], lane);
        }
        tgt = A * z - Dl;
        it++;
        // M[g] of the new iterate; M+ approximates it
        if (!used) th = thg;
        keep = th;
        have = 1;
        moved = 0;
        stage = 0;
        state = S_G;
      }
    }

    if (pass == 1 && state == S_G0 && !stop) {  // to the second pass
      __syncthreads();
      pass = 2;
      continue;
    }
    ty.inner += it;
    if (wid < 3) sm.ef[wid][lane] = p;
    if (tid == 0) sm.ctl = it > 0 ? 1 : 0;
    if (pass == 1) __syncthreads();
    break;
  }
  __syncthreads();

  // ---- step 2 on the nodes: g = (A M+ - r) / (c + A) (without an update f stays as it is)
  if (sm.ctl & 1) {
    int slot = tid;
#pragma unroll 1
    for (int run = lo + tid; run < hi; run += blockDim.x, slot += R * blockDim.x) {
      const int pen = run / prun, i30 = (run - pen * prun) * R;
      const int i1 = pen / N, i2 = pen - i1 * N;
      const E e12 = sm.ef[0][i1] * sm.ef[1][i2];
      const E dn = TWO_D ? den2[i2 * N + i1] : sm.den[i1];
      double* o = io.f + run * R;
#pragma unroll
      for (int t = 0; t < R; t += 2) {
        const E x0 = (A * (e12 * sm.ef[2][i30 + t]) - rbuf[slot + t * blockDim.x]) * dn;
        const E x1 = (A * (e12 * sm.ef[2][i30 + t + 1]) - rbuf[slot + (t + 1) * blockDim.x]) * dn;
        const double d0 = to_store(x0), d1 = to_store(x1);
        if (WIDE) {
          *reinterpret_cast<double2*>(o + t) = make_double2(d0, d1);
        } else {
          o[t] = d0;
          o[t + 1] = d1;
        }
      }
    }
  }
  __syncthreads();  // the tables of this cell are no longer read
}

__device__ __forceinline__ void post_tally(const SweepArgs& a, int q, const Tally& ty, unsigned long long visits,
                                           bool first) {
  if (first) {
    Counters* c = a.cnt + q;
    atomicAdd(&c->visits, visits);
    atomicAdd(&c->inner_iters, ty.inner);
    atomicAdd(&c->newton_iters, ty.newton);
    atomicAdd(&c->newton_solves, ty.solves);
    atomicAdd(&c->fallbacks, ty.fallback);
  }
  if (threadIdx.x == 0 && ty.status) atomicOr(&a.cnt[q].status, ty.status);
}

template <typename E, bool WIDE>
__global__ void __launch_bounds__(256) k_sweep(SweepArgs a) {
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int q = blockIdx.x / CS;
  if (q >= a.n_inst) return;  // whole cluster, uniformly
  if (a.active && !a.active[q]) return;
  const InstDev& I = a.inst[q];
  __shared__ SweepSmem<E> sm;
  extern __shared__ __align__(16) unsigned char dyn[];
  E* rbuf = reinterpret_cast<E*>(dyn);
  const int N = a.N;
  const long long K = (long long)N * N * N;
  const int J = I.J;
  scan_tables<E, false>(sm, I, N, a.dv);
  cl.sync();  // every CTA runs before another one writes its shared memory
  Tally ty;
  int buf = 0;
  const int s_end = min(a.s1, J);
#pragma unroll 1
  for (int s = a.s0; s < s_end; s++) {
    const int j = a.dir > 0 ? s : J - 1 - s;
    const long long o = I.f_off + j * K;
    CellIO io;
    io.f = a.f + o;
    io.P = a.P + o;
    io.b = a.rhs ? a.rhs + o : nullptr;
    io.nb[0] = j > 0 ? io.f - K : nullptr;
    io.nb[1] = j < J - 1 ? io.f + K : nullptr;
    io.nb[2] = io.nb[3] = nullptr;
    io.nu = a.nu[I.cell0 + j];
    io.theta = a.theta + 5 * (long long)(I.cell0 + j);
    visit_cell<E, false, WIDE>(a, I, sm, rbuf, nullptr, io, cl, CS, rank, buf, ty);
  }
  // no CTA leaves while another may still write its shared memory
  cl.sync();
  post_tally(a, q, ty, (unsigned long long)max(0, s_end - a.s0), rank == 0 && threadIdx.x == 0);
}

// ---------------------------------------------------------------------------------------
// 2-D space: one sweep ordering is a sequence of anti-diagonal wavefronts. Cells on one
// wavefront depend only on the previous wavefront (their upwind x and y neighbours) and on
// not-yet-visited cells (downwind), so the cells of a wavefront are visited concurrently,
// one thread-block cluster per cell, one launch per wavefront (the launch boundary orders
// the wavefronts). The visit is the 1-D visit with the transport weight
// c = |v1|/dx + |v2|/dy, four neighbours (or wall ghosts) and step-1 weights w c, whose
// Newton sums are two separable terms.
// Ordering o: 0 SW->NE, 1 NE->SW, 2 NW->SE, 3 SE->NW; wavefront index wf counts from the
// ordering's starting corner.
// ---------------------------------------------------------------------------------------
template <typename E, bool WIDE>
__global__ void __launch_bounds__(256) k_sweep2d(SweepArgs a, int ordering, int wf) {
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const InstDev& I = a.inst[0];
  const int nx = I.nx, ny = I.ny;
  const int amin = max(0, wf - (ny - 1)), amax = min(nx - 1, wf);
  const int ak = amin + (int)(blockIdx.x / CS);
  if (ak > amax) return;  // whole cluster, uniformly
  if (a.active && !a.active[0]) return;
  const int dirx = (ordering == 0 || ordering == 2) ? 1 : -1;
  const int diry = (ordering == 0 || ordering == 3) ? 1 : -1;
  const int ci = dirx > 0 ? ak : nx - 1 - ak;
  const int bk = wf - ak;
  const int cj = diry > 0 ? bk : ny - 1 - bk;
  const int cell = cj * nx + ci;
  __shared__ SweepSmem<E> sm;
  extern __shared__ __align__(16) unsigned char dyn[];
  const int N = a.N;
  const long long K = (long long)N * N * N;
  E* den2 = reinterpret_cast<E*>(dyn);
  E* rbuf = den2 + N * N;
  scan_tables<E, true>(sm, I, N, a.dv);
  cl.sync();  // every CTA runs before another one writes its shared memory
  Tally ty;
  int buf = 0;
  const long long o = I.f_off + cell * K;
  CellIO io;
  io.f = a.f + o;
  io.P = a.P + o;
  io.b = a.rhs ? a.rhs + o : nullptr;
  io.nb[0] = ci > 0 ? io.f - K : nullptr;
  io.nb[1] = ci < nx - 1 ? io.f + K : nullptr;
  io.nb[2] = cj > 0 ? io.f - nx * K : nullptr;
  io.nb[3] = cj < ny - 1 ? io.f + nx * K : nullptr;
  io.nu = a.nu[I.cell0 + cell];
  io.theta = a.theta + 5 * (long long)(I.cell0 + cell);
  visit_cell<E, true, WIDE>(a, I, sm, rbuf, den2, io, cl, CS, rank, buf, ty);
  cl.sync();  // no CTA leaves while another may still write its shared memory
  post_tally(a, 0, ty, 1ULL, rank == 0 && threadIdx.x == 0);
}

// ---------------------------------------------------------------------------------------
// Latency probe of the scan's two serial building blocks in one cluster of a given launch
// shape: mode 0 runs `reps` cluster reductions (cluster_sum, as in every cell visit); mode 1
// runs `reps` dependent Newton iterations of the discrete Maxwellian by the evaluating warps
// (factors and 1-D sums of each velocity dimension, the barrier among those warps, the moments
// and the direction); mode 2 the hardware cluster barrier alone. The results feed a runtime test
// that never passes (the sentinel), so nothing is stored and nothing allocated.
// ---------------------------------------------------------------------------------------
__device__ double g_probe_sink;

template <typename E>
__global__ void __launch_bounds__(256) k_probe_scan(int N, double dv, int mode, int reps, double sentinel) {
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  __shared__ SweepSmem<E> sm;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const E zero = cvt<E>(0.0);
  if (tid < kMaxN) {
    const double v = tid < N ? node(tid, N, dv) : 0.0;
    sm.c1e[tid] = cvt<E>(fabs(v));
    sm.den[tid] = cvt<E>(1.0 / (1.0 + fabs(v)));
  }
  if (tid < 64) sm.etab[tid] = cvt<E>(kExp2[tid]);
  cl.sync();
  double acc = 0.0;
  if (mode == 0) {
    // inputs formed once (FP64 is scarce: forming them per repetition would time FP64
    // conversions, not the reduction); each repetition reduces a fresh copy
    int buf = 0;
    E v0[kRed];
#pragma unroll
    for (int q = 0; q < kRed; q++) v0[q] = cvt<E>(1e-3 * (double)(tid + q));
    E accE = zero;
#pragma unroll 1
    for (int r = 0; r < reps; r++) {
      E v[kRed];
#pragma unroll
      for (int q = 0; q < kRed; q++) v[q] = v0[q];
      cluster_sum<E>(v, sm, buf, cl, CS, rank);
      accE = accE + sm.tot[0];
    }
    acc = tod(accE);
  } else if (mode == 2) {
    // the hardware cluster barrier alone (one of the reduction's steps)
    for (int r = 0; r < reps; r++) {
      cl.sync();
      acc += (double)(tid + r);
    }
  } else if (wid < kTeam) {
    // unit Maxwellian exponents and its continuum moments (per node weight) as the target
    // (in units of dv)
    E th = cvt<E>(lane == 0 ? -1.5 * log(2.0 * kPi) : ((lane & 7) == 4 ? 0.5 * dv * dv : 0.0));
    const double iw = 1.0 / (dv * dv * dv);
    const E tgt = cvt<E>(lane == 0 ? iw : (lane == 4 ? 3.0 * iw / (dv * dv) : 0.0));
    int cur = 0;
    float accf = 0.0f;
#pragma unroll 1
    for (int r = 0; r < reps; r++) {
      cur ^= 1;
      eval_row<E, false>(sm, N, th, wid, lane, cur, zero, 1.0f);
      eval_bar(kTeam);
      ProductMeasure pm;
      pm.prepare(sm.rowsf[cur][0], sm.rowsf[cur][1], sm.rowsf[cur][2]);
      const float Fl = diff(lane_moment<E>(sm.rows[cur][0], sm.rows[cur][1], sm.rows[cur][2], lane), tgt);
      float Ff[5], y[5];
#pragma unroll
      for (int k = 0; k < 5; k++) Ff[k] = shfl_i(Fl, k);
      pm.direction(Ff, y);
      accf += y[0];
      if (lane == 0) th = addf(th, 1e-9f * y[0]);  // the next evaluation depends on this one
    }
    acc = (double)accf;
  }
  cl.sync();  // no CTA leaves while another may still write its shared memory
  if (acc == sentinel) g_probe_sink = acc;
}

namespace {

// Launch configuration of a kernel in clusters.
struct ClusterLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  ClusterLaunch(int blocks, int threads, int cluster, size_t smem, cudaStream_t st) {
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

constexpr int kMaxDyn = 160 * 1024;  // dynamic shared memory a scan kernel may be launched with

// The scan kernel of a launch, by arithmetic and by the alignment of its fields.
bool wide_fields(const SweepArgs& a) {
  return ((reinterpret_cast<uintptr_t>(a.f) | reinterpret_cast<uintptr_t>(a.P) | reinterpret_cast<uintptr_t>(a.rhs)) &
          15) == 0;
}
const void* sweep_kernel(int arith, bool wide) {
  if (arith == kSweepDF64) return wide ? (const void*)k_sweep<dfloat, true> : (const void*)k_sweep<dfloat, false>;
  return wide ? (const void*)k_sweep<double, true> : (const void*)k_sweep<double, false>;
}
const void* sweep2d_kernel(int arith, bool wide) {
  if (arith == kSweepDF64) return wide ? (const void*)k_sweep2d<dfloat, true> : (const void*)k_sweep2d<dfloat, false>;
  return wide ? (const void*)k_sweep2d<double, true> : (const void*)k_sweep2d<double, false>;
}

cudaError_t scan_attrs(const void* fn) {
  cudaError_t e = func_attr(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = func_attr(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn);
  return e;
}

// Dynamic shared memory of one CTA: r of its runs (8 bytes a node in either arithmetic), and in
// 2-D the table of 1 / (c + A).
size_t scan_smem(int N, int cluster, int tpb, bool two_d) {
  const int runs = N * N * N / R, per = (runs + cluster - 1) / cluster;
  return (size_t)((per + tpb - 1) / tpb) * R * tpb * 8 + (two_d ? (size_t)N * N * 8 : 0);
}

}  // namespace

// Default launch shape: cluster size (a power of two, at most 16) and threads per CTA (a multiple of 32
// in [160, 256]; warps 0-3 serve the Newton evaluations), and the nodes per thread (a divisor of N)
// that the scan inside sgs_dc_step holds.
SweepShape sweep_shape(int N) {
  SweepShape s;
  int K = N * N * N;
  s.ept = N <= 8 ? 2 : (N % 8 == 0 ? 8 : 4);
  int threads = K / s.ept;
  s.cluster = 1;
  while (s.cluster < 16 && s.cluster * 256 < threads) s.cluster *= 2;
  s.tpb = ((threads + s.cluster - 1) / s.cluster + 31) / 32 * 32;
  if (s.tpb < 160) s.tpb = 160;
  if (s.tpb > 256) {  // more nodes than 16 CTAs of 256 threads with this many each
    s.tpb = 256;
    s.ept = N;
  }
  return s;
}

cudaError_t probe_scan(int N, double dv, int arith, int cluster, int threads, int mode, int reps, cudaStream_t st) {
  if (cluster < 1 || cluster > 16 || (cluster & (cluster - 1)) || threads < 160 || threads > 256 || threads % 32 ||
      N < 8 || N > kMaxN || reps < 0)
    return cudaErrorInvalidConfiguration;
  const void* fn = arith == kSweepDF64 ? (const void*)k_probe_scan<dfloat> : (const void*)k_probe_scan<double>;
  cudaError_t e = func_attr(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  ClusterLaunch l(cluster, threads, cluster, 0, st);
  double sentinel = -1.0e300;
  void* args[] = {&N, &dv, &mode, &reps, &sentinel};
  return cudaLaunchKernelExC(&l.cfg, fn, args);
}

// One wavefront of a 2-D ordering: ncells clusters. The CTAs per cell are at most the shape's and
// as many as run at once, one CTA per SM (the registers allow no more): the inner iteration runs
// in every CTA of a cell, so a second wave of CTAs costs more than their share of the nodes
// saves; at least what holds r in shared memory. 64 x 64 cells of 24^3 nodes: 9.5 ms an ordering,
// 23 ms with two waves allowed, 53 ms with clusters of eight CTAs on every wavefront.
cudaError_t launch_sweep2d(const SweepArgs& a, const SweepShape& sh, int arith, int ordering, int wf, int ncells,
                           cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int cs = sh.cluster;
  while (cs > 1 && ncells * cs > sms) cs /= 2;
  while (cs < 16 && scan_smem(a.N, cs, sh.tpb, true) > 80 * 1024) cs *= 2;
  const void* fn = sweep2d_kernel(arith, wide_fields(a));
  e = scan_attrs(fn);
  if (e != cudaSuccess) return e;
  ClusterLaunch l(ncells * cs, sh.tpb, cs, scan_smem(a.N, cs, sh.tpb, true), st);
  SweepArgs args = a;
  void* p[] = {&args, &ordering, &wf};
  return cudaLaunchKernelExC(&l.cfg, fn, p);
}

bool sweep_ept_compiled(int ept) {
  return ept == 2 || ept == 4 || ept == 8 || ept == 12 || ept == 16 || ept == 20 || ept == 24 || ept == 28 ||
         ept == 32;
}

cudaError_t sweep_max_clusters(int N, const SweepShape& sh, int arith, int* n) {
  *n = 0;
  const void* fn = sweep_kernel(arith, true);
  cudaError_t e = scan_attrs(fn);
  if (e != cudaSuccess) return e;
  ClusterLaunch l(sh.cluster, sh.tpb, sh.cluster, scan_smem(N, sh.cluster, sh.tpb, false), nullptr);
  return cudaOccupancyMaxActiveClusters(n, fn, &l.cfg);
}

bool sweep_shape_valid(int N, const SweepShape& sh) {
  int K = N * N * N;
  if (sh.ept <= 0 || N % sh.ept != 0) return false;
  if (sh.cluster < 1 || sh.cluster > 16 || (sh.cluster & (sh.cluster - 1))) return false;
  if (sh.tpb < 160 || sh.tpb > 256 || sh.tpb % 32) return false;
  if ((long long)sh.cluster * sh.tpb * sh.ept < K) return false;
  return sweep_ept_compiled(sh.ept);
}

cudaError_t launch_sweep(const SweepArgs& a, const SweepShape& sh, int arith, cudaStream_t st) {
  if (!sweep_shape_valid(a.N, sh)) return cudaErrorInvalidConfiguration;
  const void* fn = sweep_kernel(arith, wide_fields(a));
  cudaError_t e = scan_attrs(fn);
  if (e != cudaSuccess) return e;
  ClusterLaunch l(a.n_inst * sh.cluster, sh.tpb, sh.cluster, scan_smem(a.N, sh.cluster, sh.tpb, false), st);
  SweepArgs args = a;
  void* p[] = {&args};
  return cudaLaunchKernelExC(&l.cfg, fn, p);
}

}  // namespace sgs
