#include <algorithm>
// Collision step (eqs. (13)-(16), (28)) for every cell of every instance.
//
// Q = Q^FSM[f,f] - Q^FSM[M,M] is evaluated as the single symmetric bilinear sum
//   Q_s(a, b)_k = sum_{l+m=k} beta_s(l, m) ahat_l bhat_m,   a = f - M, b = f + M,
//   beta_s(l, m) = G(|l+m|, |l-m|) - (G(2|l|, 0) + G(2|m|, 0)) / 2,
// which equals the two-evaluation form exactly (Q_s is symmetric and Q_s(f,f) = Q^FSM[f,f])
// and carries no cancellation between two large terms at small eps.
//
// Data flow per launch sequence:
//   k_moments        f -> moments, discrete Maxwellian theta, nu            (FP64)
//   k_dft_i3/i2/i1   f -+ M -> ahat, bhat in the spectral layout [group][k1][k2][k3][lane]
//   k_sum            ahat, bhat, weight blocks -> partial qhat per work unit
//   k_sum_reduce     partials -> qhat (fixed order, FP64 accumulation), Hermitian mirror
//   k_idft_k1/k2/k3  qhat -> Q(v), P = Q - nu (M - f)
// A spectral group packs 32 cells, one per warp lane, so every weight is warp-uniform.
#include <cstdio>

#include "common.cuh"
#include "kernels.h"

namespace sgs {

// Factor d of the Maxwellian with exponents th at node i (the first one carries exp(alpha)).
__device__ inline double maxwell_factor(const double* th, int d, int i, int N, double dv) {
  const double v = node(i, N, dv);
  double x = th[1 + d] * v - th[4] * v * v;
  if (d == 0) x += th[0];
  return exp(x);
}

// ---------------------------------------------------------------------------------------
// Discrete Maxwellian on the tensor grid (eqs. (13)-(14)).
//
// M_k = exp(alpha + beta.v_k - gamma |v_k|^2) factorises as
//   exp(alpha) * E_1(v_1) E_2(v_2) E_3(v_3),   E_d(v) = exp(beta_d v - gamma v^2),
// so every moment sum_k w phi_i phi_j M_k with phi = (1, v1, v2, v3, |v|^2) is a product of
// one-dimensional sums S_d^p = sum_i E_d(v_i) v_i^p, p = 0..4, and a Newton iteration costs O(N)
// instead of O(N^3). The iteration itself (undamped Newton with step halving while the scaled
// residual grows; stop one step after the exponent change |da| + L sum|db| + L^2 |dg| falls below
// tol) follows the discrete conservation equations directly.
//
// Called by four warps (wt = 0-3), each on its own scheduler: an FP64 instruction takes a scheduler
// 64 cycles, in a chain or not, so the solve is bound by the number of them in its longest chain.
// Warp d < 3 evaluates dimension d (lane i: node i), warp 3 the factor exp(alpha); after one
// barrier each warp combines the sums, lane k forming component k of the moments, residual and
// exponents (about 45 FP64 instructions an evaluation, 175 on one warp: 5.7 us), and takes the same
// decisions. FP64 expressions that the compiler may contract either way name their rounded product.
// ---------------------------------------------------------------------------------------
struct NewtonSmem {
  double S[2][3][5], ea[2];  // sums of an evaluation and its exp(alpha), double-buffered
  float Sf[2][3][5];
};

__device__ __forceinline__ void newton_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// Sums over the warp of five values per lane, lane l returning the total of value l / 4: in the first
// three steps a lane keeps half of its values and hands over the other half (the pairs of a
// butterfly over all of them with 9 additions instead of 25).
__device__ __forceinline__ double warp_sums5(const double (&x)[5], int lane) {
  double v[8] = {x[0], x[1], x[2], x[3], x[4], 0.0, 0.0, 0.0};
  int o = 16;
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < h; q++) {
      const double send = up ? v[q] : v[q + h], keep = up ? v[q + h] : v[q];
      v[q] = keep + shfl_x(send, o);
    }
  }
  v[0] += shfl_x(v[0], 2);
  return v[0] + shfl_x(v[0], 1);
}

// Moments of M at the exponents th (lane k: component k) minus the target (lane k: tl): Ff on every
// lane, the Jacobian A (upper triangle of sum w M phi phi^T, row-major, i <= j: it only sets the
// direction) and the largest |F|.
__device__ __forceinline__ void maxw_eval(NewtonSmem& sm, int N, double dv, double w, double tl, double th, int wt,
                                          int buf, float (&Ff)[5], float (&A)[15], double& amax) {
  const int lane = threadIdx.x & 31;
  if (wt < 3) {
    const double vd = node(lane < N ? lane : 0, N, dv), v2 = vd * vd;
    const double b = __shfl_sync(0xffffffffu, th, 1 + wt), g = __shfl_sync(0xffffffffu, th, 4);
    const double x = lane < N ? exp(b * vd - g * vd * vd) : 0.0;
    double v[5];
    v[0] = x;
    v[1] = x * vd;
    v[2] = v[1] * vd;
    v[3] = v[2] * vd;
    v[4] = v[2] * v2;
    const double t = warp_sums5(v, lane);
    const float tf = (float)t;
    if ((lane & 3) == 0 && lane < 20) {
      sm.S[buf][wt][lane >> 2] = t;
      sm.Sf[buf][wt][lane >> 2] = tf;
    }
  } else {
    const double ea = exp(__shfl_sync(0xffffffffu, th, 0));
    if (lane == 0) sm.ea[buf] = ea;
  }
  newton_bar();
  const double *S1 = sm.S[buf][0], *S2 = sm.S[buf][1], *S3 = sm.S[buf][2];
  const double c = w * sm.ea[buf];
  // lane k: sum of phi_k M over the grid, from the 1-D sums (lanes 5 and 6 form parts of the last one)
  const int i = lane == 1 ? 1 : (lane == 4 ? 2 : 0), j = lane == 2 ? 1 : (lane == 5 ? 2 : 0),
            l = lane == 3 ? 1 : (lane == 6 ? 2 : 0);
  double u = __dmul_rn(S2[j], S3[l]);
  const double u6 = __shfl_sync(0xffffffffu, u, 6);
  if (lane == 5) u = __fma_rn(S2[2], S3[0], u6);
  double m = __dmul_rn(S1[i], u);
  const double m5 = __shfl_sync(0xffffffffu, m, 5);
  if (lane == 4) m = __fma_rn(S1[2], u, m5);
  const double F = __fma_rn(c, m, -tl);
  const float Fl = (float)F;
#pragma unroll
  for (int k = 0; k < 5; k++) Ff[k] = __shfl_sync(0xffffffffu, Fl, k);
  // largest |F| of lanes 0-4 as an integer (non-negative doubles order like their bits); a NaN drops
  // out, as it does from fmax
  unsigned long long bits = (unsigned long long)__double_as_longlong(F) & 0x7fffffffffffffffull;
  if (lane > 4 || bits > 0x7ff0000000000000ull) bits = 0;
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, bits, o);
    bits = other > bits ? other : bits;
  }
  amax = __longlong_as_double((long long)__shfl_sync(0xffffffffu, bits, 0));
  // Jacobian entries in FP32
  const float *f1 = sm.Sf[buf][0], *f2 = sm.Sf[buf][1], *f3 = sm.Sf[buf][2];
  float q11 = f1[2] * f2[0] * f3[0], q22 = f1[0] * f2[2] * f3[0], q33 = f1[0] * f2[0] * f3[2];
  float q12 = f1[1] * f2[1] * f3[0], q13 = f1[1] * f2[0] * f3[1], q23 = f1[0] * f2[1] * f3[1];
  float c1 = f1[3] * f2[0] * f3[0] + f1[1] * f2[2] * f3[0] + f1[1] * f2[0] * f3[2];
  float c2 = f1[2] * f2[1] * f3[0] + f1[0] * f2[3] * f3[0] + f1[0] * f2[1] * f3[2];
  float c3 = f1[2] * f2[0] * f3[1] + f1[0] * f2[2] * f3[1] + f1[0] * f2[0] * f3[3];
  float e4 = f1[4] * f2[0] * f3[0] + f1[0] * f2[4] * f3[0] + f1[0] * f2[0] * f3[4] +
             2.0f * (f1[2] * f2[2] * f3[0] + f1[2] * f2[0] * f3[2] + f1[0] * f2[2] * f3[2]);
  const float cf = (float)c;
  const float B[15] = {f1[0] * f2[0] * f3[0], f1[1] * f2[0] * f3[0], f1[0] * f2[1] * f3[0], f1[0] * f2[0] * f3[1],
                       q11 + q22 + q33, q11, q12, q13, c1, q22, q23, c2, q33, c3, e4};
#pragma unroll
  for (int q = 0; q < 15; q++) A[q] = cf * B[q];
}

// Newton for the discrete Maxwellian from the guess in th (lane k: component k). The residual F is
// evaluated in FP64 and the direction from the FP32 factorisation (inexact Newton: the root is the
// one of F). The step is halved while the scaled residual max |F| / rho grows; the iteration stops
// right after a step whose exponent change |da| + L sum|db| + L^2 |dg| is below tol. Decisions are
// taken without FP64 where that leaves no doubt.
__device__ __forceinline__ int maxwellian_newton(NewtonSmem& sm, int N, double dv, double w, double tl, double& th,
                                                 double tol, int maxit, int wt) {
  const int kl = min((int)(threadIdx.x & 31), 4);
  const double L = node(N - 1, N, dv);
  const double rho = fabs(__shfl_sync(0xffffffffu, tl, 0));
  const float Lf = (float)L, tolf = (float)tol;
  float Ff[5], A[15];
  double amax;
  int buf = 0;
  maxw_eval(sm, N, dv, w, tl, th, wt, buf, Ff, A, amax);
  for (int it = 0; it < maxit; it++) {
    float y[5];
    if (!chol5_solve(A, Ff, y)) return -1;
    float yl = y[0];
#pragma unroll
    for (int k = 1; k < 5; k++)
      if (k == kl) yl = y[k];
    const double d = widen(kl == 4 ? yl : -yl);  // -D A^{-1} F
    const double before = amax;
    double lam = 1.0, tt;
    float lamf = 1.0f;
    for (int hv = 0; hv < 40; hv++) {
      tt = __fma_rn(lam, d, th);
      buf ^= 1;
      maxw_eval(sm, N, dv, w, tl, tt, wt, buf, Ff, A, amax);
      if (amax <= before || amax < 0.99e-10 * rho) break;  // (division by rho is monotone)
      const double fn = amax / rho, f0 = before / rho;
      if (fn == fn && (fn <= f0 || fn <= 1e-10)) break;
      lam *= 0.5;
      lamf *= 0.5f;
    }
    th = tt;
    const float sf = lamf * (fabsf(y[0]) + Lf * (fabsf(y[1]) + fabsf(y[2]) + fabsf(y[3])) + Lf * Lf * fabsf(y[4]));
    bool done = sf < tolf;
    if (!(tolf > 1e-30f && fabsf(sf - tolf) > 1e-4f * (sf + tolf))) {
      const double step =
          lam * (fabs((double)y[0]) + L * (fabs((double)y[1]) + fabs((double)y[2]) + fabs((double)y[3])) +
                 L * L * fabs((double)y[4]));
      if (!(step == step)) return -1;
      done = step <= tol;
    }
    if (done) return it + 1;
  }
  return -1;
}

// ---------------------------------------------------------------------------------------
// Moments and discrete Maxwellian of every cell, its collision frequency and the separable
// factors of the Maxwellian (E_d[i], E_1 with exp(alpha)) that the transforms read.
//
// The sums are bound by the FP64 pipe of one SM (8 instructions a node: 85 us for 32^3 nodes). For
// a call of few cells the eight warps of a cell are therefore two CTAs of a cluster (SPLIT), each
// warp on a scheduler of its own; every warp adds the same nodes in the same order in both forms,
// so the results are the same bits. What follows, the guess and Newton, runs on four warps of
// the first CTA. 8 cells of 8^3: 57 us in one CTA, 44 with Newton on one warp of a split cell, 25
// now; 64 cells of 32^3: 89 (32 cells) with one warp, 75 now. (Eight CTAs of four warps a
// cell don't fit side by side on the chip: 128 cells of 32^3 took 164 us instead of 98.)
// ---------------------------------------------------------------------------------------
template <bool SPLIT>
constexpr int kMomentsThreads = SPLIT ? 128 : 256;  // Newton's barrier needs four warps at least
template <bool SPLIT>
__global__ void __launch_bounds__(kMomentsThreads<SPLIT>) k_moments(const double* __restrict__ f, CellTables ct, int N,
                                                               double dv, double newton_tol, int newton_max,
                                                               double* __restrict__ theta, double* __restrict__ nu,
                                                               double* __restrict__ efac, Counters* cnt) {
  __shared__ double vv[kMaxN];
  __shared__ double part[8][5];
  __shared__ NewtonSmem sm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = SPLIT ? (int)(blockIdx.x & 1) : 0;  // in the cluster: a cluster is one cell
  const int wid = 4 * rank + warp;                     // part of the sums
  const int c = SPLIT ? blockIdx.x >> 1 : blockIdx.x;
  if (!cell_active(ct.active, ct.cell_inst, c)) return;  // whole cluster, uniformly
  int K = N * N * N;
  const double* fc = f + ct.cell_off[c];
  if (threadIdx.x < N) vv[threadIdx.x] = node(threadIdx.x, N, dv);
  if (SPLIT) cg::this_cluster().barrier_arrive();  // (every CTA runs before another writes into it)
  __syncthreads();
  double s[5] = {0, 0, 0, 0, 0};
#pragma unroll 4
  for (int e = wid * 32 + lane; e < K; e += 256) {
    int i3 = e % N, i2 = (e / N) % N, i1 = e / (N * N);
    double x = fc[e];
    double a = vv[i1], b = vv[i2], d = vv[i3];
    s[0] += x;
    s[1] += x * a;
    s[2] += x * b;
    s[3] += x * d;
    s[4] += x * (a * a + b * b + d * d);
  }
  const double sum = warp_sums5(s, lane);
  const bool holds = (lane & 3) == 0 && lane < 20;
  if (SPLIT) {
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_wait();
    if (holds) cl.map_shared_rank(&part[wid][0], 0)[lane >> 2] = sum;
    cl.sync();
    if (rank != 0) return;  // only its own writes were remote, and they have landed
  } else {
    if (holds) part[wid][lane >> 2] = sum;
    __syncthreads();
    if (warp >= 4) return;
  }
  const double w = dv * dv * dv;
  const int kl = min(lane, 4);
  double t = 0.0;
  for (int q = 0; q < 8; q++) t += part[q][kl];
  const double ml = w * t;  // lane k: moment k
  double m[5], th[5] = {0, 0, 0, 0, 0};
#pragma unroll
  for (int q = 0; q < 5; q++) m[q] = __shfl_sync(0xffffffffu, ml, q);
  const InstDev& I = ct.inst[ct.cell_inst[c]];
  int it = -1;
  double thl = 0.0;  // lane k: exponent k
  if (continuum_guess<double>(m, th)) {
    thl = th[0];
#pragma unroll
    for (int q = 1; q < 5; q++)
      if (q == kl) thl = th[q];
    it = maxwellian_newton(sm, N, dv, w, ml, thl, newton_tol, newton_max, warp);
#pragma unroll
    for (int q = 0; q < 5; q++) th[q] = __shfl_sync(0xffffffffu, thl, q);
  }
  if (warp < 3) {
    if (lane < N) efac[((long long)c * 3 + warp) * kMaxN + lane] = maxwell_factor(th, warp, lane, N, dv);
    return;
  }
  double rho = m[0];
  double T = (m[4] / rho - (m[1] * m[1] + m[2] * m[2] + m[3] * m[3]) / (rho * rho)) / 3.0;
  // penalty frequency of eq. (28): the loss frequency 4 pi b0 rho for Maxwell molecules;
  // for hard spheres its supremum over the truncated kernel |q| <= 2R, 4 pi b0 rho 2R with
  // R = 2L / (3 sqrt 2 + 1) and 2L = N dv, so that no stiff part of the loss term is left
  // in P (a mean loss frequency lets the explicit remainder grow at large |v|)
  double nuv = 4.0 * kPi * I.b0 * rho;
  if (I.collision == SGS_HARD_SPHERE) nuv *= 2.0 * (N * dv) / (3.0 * sqrt(2.0) + 1.0);
  if (lane < 5) theta[5 * c + lane] = thl;
  if (lane == 0) {
    nu[c] = nuv;
    unsigned bits = 0;
    if (it < 0) bits |= SGS_ST_NEWTON_FAIL;
    if (!(rho > 0.0) || !(T > 0.0)) bits |= SGS_ST_NONPOSITIVE;
    if (!(rho == rho) || !(T == T)) bits |= SGS_ST_NONFINITE;
    if (bits) atomicOr(&cnt[ct.cell_inst[c]].status, bits);
  }
}

// Separable factors of every cell's Maxwellian from theta (one block per cell): of a reference
// state, whose moments are not formed.
__global__ void k_factors(const double* theta, int N, double dv, double* efac) {
  if (threadIdx.x < 3 * N) {
    const int d = threadIdx.x / N, i = threadIdx.x % N;
    efac[((long long)blockIdx.x * 3 + d) * kMaxN + i] = maxwell_factor(theta + 5 * (long long)blockIdx.x, d, i, N, dv);
  }
}

// Outputs of the transforms that a thread forms together: four share the loads of their common
// operand and read the other one by one 16-byte load (the FP32 passes were bound by shared loads,
// four for every 12 FP32 instructions; 128 cells, 32 velocities, five passes: 567 -> 396 us). FP64
// is bound by its pipe and keeps single outputs. Every output is summed in the same order either
// way, and the additions below name the product that is rounded, so that it doesn't depend on the
// tile which one the compiler fuses: the increments of the defect-correction iteration amplify a
// changed last bit to 3e-7.
template <typename T>
constexpr int kDftTile = sizeof(T) == 4 ? 4 : 1;
template <typename T, int TR>
__device__ __forceinline__ void load_tile_row(const T* p, T (&x)[TR]) {
  if constexpr (TR == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
  } else {
    x[0] = p[0];
  }
}
__device__ __forceinline__ float mul_add(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mul_add(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_only(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_only(double a, double b) { return __dmul_rn(a, b); }
// (re, im) += (x, y) (c - i s)
template <typename T>
__device__ __forceinline__ void dft_add(T& re, T& im, T x, T y, T c, T s) {
  re += mul_add(x, c, mul_only(y, s));
  im += mul_add(y, c, -mul_only(x, s));
}
// (re, im) += (x, y) (c + i s)
template <typename T>
__device__ __forceinline__ void idft_add(T& re, T& im, T x, T y, T c, T s) {
  re += mul_add(x, c, -mul_only(y, s));
  im += mul_add(x, s, mul_only(y, c));
}

// ---------------------------------------------------------------------------------------
// Forward DFT, fhat_k = N^-3 sum_v f(v) exp(-i 2 pi k j / N), one index at a time.
// Pass 1 (index 3) forms a = f - M and b = f + M in FP64 and transforms them in T.
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_dft_i3(const double* __restrict__ f, CellTables ct, const double* efac,
                                                 const double* efac_ref, SpecBufs<T> sb, int N, double dv,
                                                 DftMode md) {
  extern __shared__ __align__(16) unsigned char smraw[];
  int n = N - 1;
  T* cs = (T*)smraw;             // [N][n] cos, transposed: k3 fastest, so that the threads of
  T* sn = cs + (n * N + 3) / 4 * 4;  // [N][n] sin  a warp (consecutive k3) read consecutive banks
  constexpr int TR = kDftTile<T>;
  const int NS = N + TR;         // row stride of the slabs: rows stay aligned, the stores spread over banks
  T* sa = sn + (n * N + 3) / 4 * 4;  // [i3][i2] a slab
  T* sbb = sa + N * NS;          // [i3][i2] b slab
  // M = E1[i1] E2[i2] E3[i3]: E12[i2] = E1[i1] E2[i2] for this block's i1, then one product
  __shared__ double E12[kMaxN], E3[kMaxN], E12r[kMaxN], E3r[kMaxN];
  int c = blockIdx.x, i1 = blockIdx.y;
  if (!cell_active(ct.active, ct.cell_inst, c)) return;
  if (threadIdx.x < N) {
    const double* e = efac + (long long)c * 3 * kMaxN;
    E12[threadIdx.x] = e[i1] * e[kMaxN + threadIdx.x];
    E3[threadIdx.x] = e[2 * kMaxN + threadIdx.x];
    if (md.mode != 0) {
      const double* er = efac_ref + (long long)c * 3 * kMaxN;
      E12r[threadIdx.x] = er[i1] * er[kMaxN + threadIdx.x];
      E3r[threadIdx.x] = er[2 * kMaxN + threadIdx.x];
    }
  }
  for (int t = threadIdx.x; t < n * N; t += blockDim.x) {
    int k3 = t / N, i3 = t % N;
    cs[i3 * n + k3] = sb.twc[t];
    sn[i3 * n + k3] = sb.tws[t];
  }
  __syncthreads();
  const long long off = ct.cell_off[c] + (long long)i1 * N * N;
  const double* fc = f + off;
  for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
    int i2 = t / N, i3 = t % N;
    double M = E12[i2] * E3[i3];
    double x = fc[t];
    if (md.mode == 0) {  // a = f - M, b = f + M
      sa[i3 * NS + i2] = (T)(x - M);
      sbb[i3 * NS + i2] = (T)(x + M);
    } else {  // increments against the reference state f_ref, M_ref (exact in FP64, then rounded)
      double Mr = E12r[i2] * E3r[i3];
      double xr = md.f_ref[off + t];
      if (md.mode == 1) {  // a = (f - M) - (f_ref - M_ref), b = f + M
        sa[i3 * NS + i2] = (T)((x - xr) - (M - Mr));
        sbb[i3 * NS + i2] = (T)(x + M);
      } else {  // a unused, b = (f + M) - (f_ref + M_ref)
        sa[i3 * NS + i2] = (T)0;
        sbb[i3 * NS + i2] = (T)((x - xr) + (M - Mr));
      }
    }
  }
  __syncthreads();
  typedef typename CplxOf<T>::type CT;
  CT* oa = sb.st1a + ((long long)c * N + i1) * N * n;
  CT* ob = sb.st1b + ((long long)c * N + i1) * N * n;
  for (int t = threadIdx.x; t < N / TR * n; t += blockDim.x) {
    const int i2 = t / n * TR, k3 = t % n;
    T ar[TR], ai[TR], br[TR], bi[TR];
#pragma unroll
    for (int q = 0; q < TR; q++) ar[q] = ai[q] = br[q] = bi[q] = 0;
    for (int i3 = 0; i3 < N; i3++) {
      const T co = cs[i3 * n + k3], si = sn[i3 * n + k3];
      T a[TR], b[TR];
      load_tile_row<T, TR>(sa + i3 * NS + i2, a);
      load_tile_row<T, TR>(sbb + i3 * NS + i2, b);
#pragma unroll
      for (int q = 0; q < TR; q++) {
        ar[q] += a[q] * co;
        ai[q] -= a[q] * si;
        br[q] += b[q] * co;
        bi[q] -= b[q] * si;
      }
    }
#pragma unroll
    for (int q = 0; q < TR; q++) {
      oa[(i2 + q) * n + k3] = make_cplx(ar[q], ai[q]);
      ob[(i2 + q) * n + k3] = make_cplx(br[q], bi[q]);
    }
  }
}

// Pass 2 (index 2): [c][i1][i2][k3] -> [c][i1][k2][k3].
template <typename T>
__global__ void __launch_bounds__(256) k_dft_i2(SpecBufs<T> sb, int N) {
  typedef typename CplxOf<T>::type CT;
  extern __shared__ __align__(16) unsigned char smraw[];
  int n = N - 1;
  constexpr int TR = kDftTile<T>;
  const int NS = (n + TR - 1) / TR * TR;  // outputs, padded to whole tiles
  T* cs = (T*)smraw;    // [i][k] cos
  T* sn = cs + NS * N;  // [i][k] sin
  CT* xa = (CT*)(sn + NS * N);  // [N][n]
  CT* xb = xa + N * n;
  int c = blockIdx.x, i1 = blockIdx.y;
  if (!cell_active(sb.active, sb.cell_inst, c)) return;
  for (int t = threadIdx.x; t < NS * N; t += blockDim.x) {
    const int i = t / NS, k = t % NS;
    cs[t] = k < n ? sb.twc[k * N + i] : (T)0;
    sn[t] = k < n ? sb.tws[k * N + i] : (T)0;
  }
  const CT* ia = sb.st1a + ((long long)c * N + i1) * N * n;
  const CT* ib = sb.st1b + ((long long)c * N + i1) * N * n;
  for (int t = threadIdx.x; t < N * n; t += blockDim.x) {
    xa[t] = ia[t];
    xb[t] = ib[t];
  }
  __syncthreads();
  CT* oa = sb.st2a + ((long long)c * N + i1) * n * n;
  CT* ob = sb.st2b + ((long long)c * N + i1) * n * n;
  for (int t = threadIdx.x; t < NS / TR * n; t += blockDim.x) {
    const int k2 = t / n * TR, k3 = t % n;
    T ar[TR], ai[TR], br[TR], bi[TR];
#pragma unroll
    for (int q = 0; q < TR; q++) ar[q] = ai[q] = br[q] = bi[q] = 0;
    for (int i2 = 0; i2 < N; i2++) {
      T co[TR], si[TR];
      load_tile_row<T, TR>(cs + i2 * NS + k2, co);
      load_tile_row<T, TR>(sn + i2 * NS + k2, si);
      const CT a = xa[i2 * n + k3], b = xb[i2 * n + k3];
#pragma unroll
      for (int q = 0; q < TR; q++) {
        dft_add(ar[q], ai[q], a.x, a.y, co[q], si[q]);
        dft_add(br[q], bi[q], b.x, b.y, co[q], si[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < TR; q++)
      if (k2 + q < n) {
        oa[(k2 + q) * n + k3] = make_cplx(ar[q], ai[q]);
        ob[(k2 + q) * n + k3] = make_cplx(br[q], bi[q]);
      }
  }
}

// Pass 3 (index 1): [c][i1][k2][k3] -> spectral layout [g][k1][k2][k3][lane], times N^-3.
template <typename T>
__global__ void __launch_bounds__(256) k_dft_i1(SpecBufs<T> sb, int N) {
  typedef typename CplxOf<T>::type CT;
  extern __shared__ __align__(16) unsigned char smraw[];
  int n = N - 1;
  constexpr int TR = kDftTile<T>;
  const int NS = (n + TR - 1) / TR * TR;  // outputs, padded to whole tiles
  T* cs = (T*)smraw;    // [i][k] cos
  T* sn = cs + NS * N;  // [i][k] sin
  CT* xa = (CT*)(sn + NS * N);  // [N][n] (i1, k3)
  CT* xb = xa + N * n;
  int c = blockIdx.x, k2 = blockIdx.y;
  if (!cell_active(sb.active, sb.cell_inst, c)) return;
  for (int t = threadIdx.x; t < NS * N; t += blockDim.x) {
    const int i = t / NS, k = t % NS;
    cs[t] = k < n ? sb.twc[k * N + i] : (T)0;
    sn[t] = k < n ? sb.tws[k * N + i] : (T)0;
  }
  for (int t = threadIdx.x; t < N * n; t += blockDim.x) {
    int i1 = t / n, k3 = t % n;
    long long src = (((long long)c * N + i1) * n + k2) * n + k3;
    xa[t] = sb.st2a[src];
    xb[t] = sb.st2b[src];
  }
  __syncthreads();
  T scale = (T)(1.0 / ((double)N * N * N));
  int g = c / kLanes, lane = c % kLanes;
  const int ls = g == sb.fold_group ? sb.fold_lanes : kLanes;  // lanes of the group's rows (SpecBufs)
  for (int t = threadIdx.x; t < NS / TR * n; t += blockDim.x) {
    const int k1 = t / n * TR, k3 = t % n;
    T ar[TR], ai[TR], br[TR], bi[TR];
#pragma unroll
    for (int q = 0; q < TR; q++) ar[q] = ai[q] = br[q] = bi[q] = 0;
    for (int i1 = 0; i1 < N; i1++) {
      T co[TR], si[TR];
      load_tile_row<T, TR>(cs + i1 * NS + k1, co);
      load_tile_row<T, TR>(sn + i1 * NS + k1, si);
      const CT a = xa[i1 * n + k3], b = xb[i1 * n + k3];
#pragma unroll
      for (int q = 0; q < TR; q++) {
        dft_add(ar[q], ai[q], a.x, a.y, co[q], si[q]);
        dft_add(br[q], bi[q], b.x, b.y, co[q], si[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < TR; q++)
      if (k1 + q < n) {
        const long long o = (long long)g * n * n * n * kLanes + (((long long)(k1 + q) * n + k2) * n + k3) * ls + lane;
        sb.ahat[o] = make_cplx(ar[q] * scale, ai[q] * scale);
        sb.bhat[o] = make_cplx(br[q] * scale, bi[q] * scale);
      }
  }
}

// ---------------------------------------------------------------------------------------
// Direct spectral sum. Work unit = one output row (k1, k2) of the Hermitian half and a range of
// m1; a step = one (m1, m2) with its weights, the rows ahat[(k1-m1, k2-m2, .)] and
// bhat[(m1, m2, .)], brought into shared memory by bulk copies while the previous step
// computes. Lane = cell (a lane group of 32 cells per four warps).
//
// With N = 4 BK the n = 4 BK - 1 outputs k3 and inputs m3 of a step fall into four blocks of BK
// (the last one short by one). Warp kb of a lane group accumulates the outputs of block kb in
// registers and walks the blocks c of m3: |kb - c| <= 1 is a full BK x BK square of valid pairs
// (|k3 - m3| <= H), |kb - c| = 2 a triangle, |kb - c| = 3 empty. Along m3 the BK values of ahat
// that meet the outputs slide by one, so a thread loads one value of each row per m3 and keeps
// the window in registers (its slots rotate; the loop is unrolled by BK). In FP32 this is the form for
// N >= 24 (k_sum_regs below that). It replaces a
// fully unrolled step of 721 pairs per warp with both rows in registers (FP32), which was bound
// by instruction fetch (69 KB of code) at 255 registers and two warps per scheduler, and a
// version with two shared loads per pair (FP64), whose 127 KB of rows for two warps left half
// of an SM's schedulers idle. Measured: FP32,
// 32 cells of 32^3, 1.62 -> 1.55 ms (42 TFLOP/s; 64 registers, 20 warps per SM; 0.73 of the issue
// slots, with 1.9 barrier and 0.8 operand-dispatch stalls per issue); FP64 is at 0.9 of the rate of one
// instruction per 64 cycles and scheduler, its cap. FP32 in packed pairs (fma.rn.f32x2 on outputs i, i + 1) took 1.94 ms: about
// one move per packed operand.
// Four warps do 3/14, 4/14, 4/14, 3/14 of the blocks; every other lane group (or block) takes
// them in the order 1, 0, 3, 2, so that the SM's schedulers get the same work.
// Each output is summed over m1, m2, m3 in ascending order in the arithmetic T, as before.
// ---------------------------------------------------------------------------------------
constexpr int kSumBlocksPerStep = 14;  // blocks of (k3, m3) pairs of a step

// Weights of a step: the valid blocks (kb, c), kb major, c ascending, each [m3][k3] of BK x BK
// (zero where the pair is not valid: 896 values at N = 32 for 721 pairs, 0.24 more of a table that is
// 1.9 GB of the 2.5 GB workspace of 64 cells in FP64 and 3.7 of 4.6 GB in the mixed solver).
__host__ __device__ constexpr int sum_first_block(int kb) { return kb == 0 ? 0 : (kb == 1 ? 3 : (kb == 2 ? 7 : 11)); }
__host__ __device__ constexpr int sum_weights(int BK) { return kSumBlocksPerStep * BK * BK; }

// Whether the FP32 sum of a grid keeps both rows in registers (k_sum_regs).
__host__ __device__ constexpr bool sum_in_registers(int BK) { return BK <= 5; }

// Weight row of one m3: BK consecutive values by the widest aligned loads.
template <typename T, int BK>
__device__ __forceinline__ void load_weights(const T* p, T (&w)[BK]) {
  constexpr int V = (BK % 4 == 0 && sizeof(T) == 4) ? 4 : (BK % 2 == 0 ? 2 : 1);
#pragma unroll
  for (int i = 0; i < BK; i += V) {
    if constexpr (V == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + i);
      w[i] = x.x, w[i + 1] = x.y, w[i + 2] = x.z, w[i + 3] = x.w;
    } else if constexpr (V == 2) {
      const typename CplxOf<T>::type x = *reinterpret_cast<const typename CplxOf<T>::type*>(p + i);
      w[i] = x.x, w[i + 1] = x.y;
    } else {
      w[i] = p[i];
    }
  }
}

// One block of a step for one warp. KIND 0: full; -1: the block below the band (kb - c = 2, pairs
// i < u); +1: above it (kb - c = -2, pairs i > u). win: the sliding window of ahat, slot
// (i - u) mod BK; ra: ahat of (k3 = first output, m3 = first input of the block), rb: bhat of
// that m3 (both already at this lane).
template <int KIND, typename T, int BK, int LS>
__device__ __forceinline__ void sum_block(const T* w, const typename CplxOf<T>::type* ra,
                                          const typename CplxOf<T>::type* rb, bool k_pad, bool m_pad,
                                          typename CplxOf<T>::type (&win)[BK], T (&accr)[BK], T (&acci)[BK]) {
  typedef typename CplxOf<T>::type CT;
  // FP64 skips the pairs of the padding output and input (k_pad, m_pad: this block has them); for
  // FP32 their zero weights cost less than the test
  constexpr bool kSkip = sizeof(T) == 8;
#pragma unroll
  for (int u = 0; u < BK; u++) {
    if (KIND == 0 || (KIND < 0 && u > 0)) win[(BK - u) % BK] = ra[-u * LS];
    if (kSkip && u == BK - 1 && m_pad) break;
    const CT bv = rb[u * LS];
    T wv[BK];
    load_weights<T, BK>(w + u * BK, wv);
#pragma unroll
    for (int i = 0; i < BK; i++) {
      if ((KIND < 0 && i >= u) || (KIND > 0 && i <= u)) continue;
      if (kSkip && i == BK - 1 && k_pad) break;
      const CT av = win[(i - u + BK) % BK];
      const T br = wv[i] * bv.x, bi = wv[i] * bv.y;
      accr[i] = fma(av.x, br, accr[i]);
      accr[i] = fma(-av.y, bi, accr[i]);
      acci[i] = fma(av.x, bi, acci[i]);
      acci[i] = fma(av.y, br, acci[i]);
    }
  }
}

// F > 1 (FP64, a last lane group of at most 32 / F cells): the group's rows hold 32 / F lanes, and
// the F parts of a warp take F consecutive steps at a time, summed at the end. The FP64 pipe
// works through all 32 lanes whether they hold a cell or not: 40 cells of 24^3 took as long as
// 64 (collision step 22.1 ms, folded 15.0).
template <typename T, int BK, int F>
__global__ void __launch_bounds__(512) k_sum(SumArgs<T> a) {
  typedef typename CplxOf<T>::type CT;
  constexpr int H = 2 * BK - 1, n = 4 * BK - 1;
  constexpr int VEC = 16 / (int)sizeof(T);
  constexpr int PW = (sum_weights(BK) + VEC - 1) / VEC * VEC;
  constexpr int PWS = PW + (F > 1 ? VEC : 0);      // the parts' weights start in different banks
  constexpr int LS = kLanes / F;                   // lanes of a row
  constexpr int kRow = n * LS;                     // ahat row; the bhat row has one more, of zeros
  constexpr int kRows = kRow + (n + 1) * LS;
  extern __shared__ __align__(128) unsigned char smraw[];
  T* Wb = (T*)smraw;                                   // [2][F][PWS]
  CT* rows = (CT*)(smraw + 2 * F * PWS * sizeof(T));   // [2][NG][F][kRows]
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int s_err;

  const int NG = blockDim.x >> 7;       // lane groups of a block, four warps each
  const int4 ud = a.units[blockIdx.x];  // k1, k2, m1_lo, m1_hi
  const long long step0 = a.unit_step0[blockIdx.x];
  const int k1 = ud.x, k2 = ud.y, m1lo = ud.z, m1hi = ud.w;
  const int m2lo = max(-H, k2 - H), m2hi = min(H, k2 + H);
  const int nm2 = m2hi - m2lo + 1;
  const int S = (m1hi - m1lo + 1) * nm2;
  const int B = (S + F - 1) / F;        // batches of F steps
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = warp >> 2;
  const int part = lane / LS, cell = lane % LS;
  const int kb = ((grp + blockIdx.x) & 1) ? ((warp & 3) ^ 1) : (warp & 3);
  const int g0 = a.g0 + blockIdx.y * NG;
  const int ng = min(NG, a.G - g0);
  const uint32_t row_bytes = kRow * sizeof(CT);

  if (a.active) {
    // a block whose lane groups hold no cell of an active instance has nothing to compute
    const int c = (g0 + grp) * kLanes + cell;
    if (!__syncthreads_or(grp < ng && c < a.C && a.active[a.cell_inst[c]])) return;
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    s_err = 0;
    fence_mbar_init();
  }
  for (int t = threadIdx.x; t < 2 * NG * F * LS; t += blockDim.x)
    rows[(t / LS + 1) * kRows - LS + t % LS] = make_cplx((T)0, (T)0);
  __syncthreads();

  auto issue = [&](int bt) {
    const int b = bt & 1, nf = min(F, S - bt * F);
    mbar_arrive_expect_tx(&bar[b], nf * (PW * sizeof(T) + ng * 2 * row_bytes));
    for (int h = 0; h < nf; h++) {
      const int s = bt * F + h, m1 = m1lo + s / nm2, m2 = m2lo + s % nm2;
      bulk_g2s(Wb + (b * F + h) * PWS, a.W + (step0 + s) * PW, PW * sizeof(T), &bar[b]);
      for (int w = 0; w < ng; w++) {
        const long long ga = (((long long)(k1 - m1 + H)) * n + (k2 - m2 + H)) * kRow;
        const long long gb = (((long long)(m1 + H)) * n + (m2 + H)) * kRow;
        const long long g = (long long)(g0 + w) * n * n * n * kLanes;
        CT* dst = rows + ((b * NG + w) * F + h) * kRows;
        bulk_g2s(dst, a.ahat + g + ga, row_bytes, &bar[b]);
        bulk_g2s(dst + kRow, a.bhat + g + gb, row_bytes, &bar[b]);
      }
    }
  };

  if (threadIdx.x == 0 && B > 0) issue(0);

  T accr[BK], acci[BK];
#pragma unroll
  for (int i = 0; i < BK; i++) accr[i] = acci[i] = (T)0;

  const bool active = grp < ng;
  int fail_b = 0, fail_par = 0;
  for (int s = 0; s < B; s++) {
    const int b = s & 1;
    if (!mbar_wait(&bar[b], (s >> 1) & 1, a.spin_max)) {
      s_err = 1;
      fail_b = b;
      fail_par = (s >> 1) & 1;
    }
    __syncthreads();
    if (s_err) break;
    // the other buffer was released by the barrier above: the next batch goes into it
    if (threadIdx.x == 0 && s + 1 < B) issue(s + 1);
    if (active && s * F + part < S) {
      // ahat of l = k3 - m3 is at l + H = BK (kb - c) + 2 BK - 1 + i - u
      const CT* ra = rows + ((b * NG + grp) * F + part) * kRows + (kb * BK + 2 * BK - 1) * LS + cell;
      const CT* rb = rows + ((b * NG + grp) * F + part) * kRows + kRow + cell;
      const T* w = Wb + (b * F + part) * PWS + sum_first_block(kb) * BK * BK;
      CT win[BK];
      int c = max(0, kb - 1);
      if (kb >= 2) {
        const int cl = kb - 2;
        sum_block<-1, T, BK, LS>(w, ra - cl * BK * LS, rb + cl * BK * LS, kb == 3, false, win, accr, acci);
        w += BK * BK;
      } else {
#pragma unroll
        for (int i = 1; i < BK; i++) win[i] = ra[i * LS];
      }
      const int c1 = min(3, kb + 1);
#pragma unroll 1
      for (; c <= c1; c++) {
        sum_block<0, T, BK, LS>(w, ra - c * BK * LS, rb + c * BK * LS, kb == 3, c == 3, win, accr, acci);
        w += BK * BK;
      }
      if (kb < 2) sum_block<1, T, BK, LS>(w, ra, rb + c * BK * LS, false, c == 3, win, accr, acci);
    }
  }
  if (s_err) {
    // A copy did not land within the spin limit: report, then wait (bounded) for that
    // phase so no copy is still writing this block's shared memory when it exits.
    if (threadIdx.x == 0) {
      atomicOr(&a.cnt[0].status, SGS_ST_TIMEOUT);
      mbar_wait(&bar[fail_b], fail_par, a.spin_max);
    }
    return;
  }
  if (F > 1) {
#pragma unroll
    for (int i = 0; i < BK; i++)
#pragma unroll
      for (int o = LS; o < kLanes; o <<= 1) {
        accr[i] += __shfl_xor_sync(0xffffffffu, accr[i], o);
        acci[i] += __shfl_xor_sync(0xffffffffu, acci[i], o);
      }
  }
  if (active) {
    CT* out = a.partial + ((long long)blockIdx.x * a.Gs + (g0 + grp)) * n * kLanes;
#pragma unroll
    for (int i = 0; i < BK; i++)
      if (kb * BK + i < n) out[(kb * BK + i) * kLanes + lane] = make_cplx(accr[i], acci[i]);
  }
}

// The FP32 sum of the smaller grids (sum_in_registers): a warp per lane group with both rows of a step in
// registers and the step fully unrolled. Same units, weights and order of additions as k_sum, so
// the same bits. A step has few pairs there (91 at N = 12, 271 at N = 20), and the four warps of a
// group in k_sum lose at its barrier, by the blocks they share unevenly and by the rows that each
// of them loads; this form loses where its code leaves the instruction cache (721 pairs at N = 32).
// k_sum -> here: 3000 cells of 8^3 61 -> 40 us, 1000 of 12^3 188 -> 142, 1000 of 16^3 830 -> 751, 64
// of 20^3 203 -> 181. At N = 24 k_sum is the better one for most cell counts (96: 0.87 against 1.08 ms, 200:
// 1.97 against 2.20, 64: 0.55 against 0.53).
template <int BK>
__global__ void __launch_bounds__(128) k_sum_regs(SumArgs<float> a) {
  constexpr int H = 2 * BK - 1, n = 4 * BK - 1;
  constexpr int PW = (sum_weights(BK) + 3) / 4 * 4;
  constexpr int kRow = n * kLanes;
  extern __shared__ __align__(128) unsigned char smraw[];
  float* Wb = (float*)smraw;                              // [2][PW]
  float2* rows = (float2*)(smraw + 2 * PW * sizeof(float));  // [NW][2][n][32]
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int s_err;

  const int NW = blockDim.x >> 5;
  const int4 ud = a.units[blockIdx.x];  // k1, k2, m1_lo, m1_hi
  const long long step0 = a.unit_step0[blockIdx.x];
  const int k1 = ud.x, k2 = ud.y, m1lo = ud.z, m1hi = ud.w;
  const int m2lo = max(-H, k2 - H), m2hi = min(H, k2 + H);
  const int nm2 = m2hi - m2lo + 1;
  const int S = (m1hi - m1lo + 1) * nm2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g0 = blockIdx.y * NW;
  const int ng = min(NW, a.G - g0);
  const uint32_t row_bytes = kRow * sizeof(float2);

  if (a.active) {
    // a block whose lane groups hold no cell of an active instance has nothing to compute
    const int c = (g0 + warp) * kLanes + lane;
    if (!__syncthreads_or(warp < ng && c < a.C && a.active[a.cell_inst[c]])) return;
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    s_err = 0;
    fence_mbar_init();
  }
  __syncthreads();

  auto issue = [&](int s) {
    const int m1 = m1lo + s / nm2, m2 = m2lo + s % nm2, b = s & 1;
    mbar_arrive_expect_tx(&bar[b], PW * sizeof(float) + ng * 2 * row_bytes);
    bulk_g2s(Wb + b * PW, a.W + (step0 + s) * PW, PW * sizeof(float), &bar[b]);
    for (int w = 0; w < ng; w++) {
      const long long ga = (((long long)(g0 + w) * n + (k1 - m1 + H)) * n + (k2 - m2 + H)) * kRow;
      const long long gb = (((long long)(g0 + w) * n + (m1 + H)) * n + (m2 + H)) * kRow;
      float2* dst = rows + w * 2 * kRow;
      bulk_g2s(dst, a.ahat + ga, row_bytes, &bar[b]);
      bulk_g2s(dst + kRow, a.bhat + gb, row_bytes, &bar[b]);
    }
  };

  if (threadIdx.x == 0 && S > 0) issue(0);

  float accr[n], acci[n];
#pragma unroll
  for (int i = 0; i < n; i++) accr[i] = acci[i] = 0.0f;

  const bool active = warp < ng;
  int fail_b = 0, fail_par = 0;
  for (int s = 0; s < S; s++) {
    const int b = s & 1;
    if (!mbar_wait(&bar[b], (s >> 1) & 1, a.spin_max)) {
      s_err = 1;
      fail_b = b;
      fail_par = (s >> 1) & 1;
    }
    float2 Ar[n], Br[n];
    if (active) {
      const float2* rw = rows + warp * 2 * kRow + lane;
#pragma unroll
      for (int i = 0; i < n; i++) {
        Ar[i] = rw[i * kLanes];
        Br[i] = rw[kRow + i * kLanes];
      }
    }
    __syncthreads();
    if (s_err) break;
    // every row is in registers: the next step's come into the same buffer
    if (threadIdx.x == 0 && s + 1 < S) issue(s + 1);
    if (active) {
      const float4* W4 = (const float4*)(Wb + b * PW);
      float4 wv;
      int have = -1;  // the quad of weights in wv
#pragma unroll
      for (int kb = 0; kb < 4; kb++)
#pragma unroll
        for (int c = (kb > 2 ? kb - 2 : 0); c <= (kb < 1 ? 2 : 3); c++)
#pragma unroll
          for (int t = 0; t < BK * BK; t++) {
            const int p = (sum_first_block(kb) + c - (kb > 2 ? kb - 2 : 0)) * BK * BK + t;
            const int m = c * BK + t / BK, k = kb * BK + t % BK, l = k - m + H;
            if (k >= n || m >= n || l < 0 || l >= n) continue;
            if (p / 4 != have) wv = W4[p / 4];
            have = p / 4;
            const float w = p % 4 == 0 ? wv.x : (p % 4 == 1 ? wv.y : (p % 4 == 2 ? wv.z : wv.w));
            const float br = w * Br[m].x, bi = w * Br[m].y;
            accr[k] = fmaf(Ar[l].x, br, accr[k]);
            accr[k] = fmaf(-Ar[l].y, bi, accr[k]);
            acci[k] = fmaf(Ar[l].x, bi, acci[k]);
            acci[k] = fmaf(Ar[l].y, br, acci[k]);
          }
    }
  }
  if (s_err) {
    // the failing thread waits (again bounded) for its copies in flight
    if (threadIdx.x == 0) {
      atomicOr(&a.cnt[0].status, SGS_ST_TIMEOUT);
      mbar_wait(&bar[fail_b], fail_par, a.spin_max);
    }
    return;
  }
  if (active) {
    float2* out = a.partial + ((long long)blockIdx.x * a.Gs + (g0 + warp)) * kRow;
#pragma unroll
    for (int i = 0; i < n; i++) out[i * kLanes + lane] = make_float2(accr[i], acci[i]);
  }
}

// ---------------------------------------------------------------------------------------
// Direct spectral sum in double-float arithmetic on the FP32 pipes (the high-precision
// evaluation of the defect correction). Same units, steps, blocks and weight order as k_sum; the
// transformed rows arrive split into (hi, lo) float pairs (k_split_spec) and the weights as
// the FP32 table (hi) plus its FP32 remainder table (lo). Products are formed exactly in
// their leading part (FMA two-product) with first-order cross terms, and accumulated by
// error-free two-sums into (hi, lo) accumulators, so each term carries about 2^-48 relative
// error instead of FP32's 2^-24. Bound by the FP32 pipes (56 operations per pair): 32 cells of
// 32^3 in 11.3 ms, 0.77 of the pipes' rate (13.1 ms with outputs strided over the warps, two
// shared loads and a range test per pair).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void df_mul_acc(float xh, float xl, float yh, float yl, float& ah, float& al) {
  // (ah, al) += (xh + xl)(yh + yl), to first order in the low parts
  float q = xh * yh;
  float e = fmaf(xh, yh, -q);
  e = fmaf(xh, yl, e);
  e = fmaf(xl, yh, e);
  float s = ah + q;
  float z = s - ah;
  float err = (ah - (s - z)) + (q - z);
  ah = s;
  al += err + e;
}

// Side of a square of the double-float sum: half a block where it divides (8 warps per lane
// group), which keeps the unrolled body (56 operations a pair) within the instruction cache:
// with whole blocks of N = 32 it is 121 KB of code and twice as slow.
__host__ __device__ constexpr int df_side(int BK) { return BK % 2 == 0 ? BK / 2 : BK; }

// Whether a square's rows m3 are a loop, the window moving by register copies, instead of an unrolled
// body with a rotating one: squares of 7 (N = 28) are 81 KB of code unrolled, 64 cells of 28^3 took
// 21.6 ms instead of 12.0; squares of 5 (N = 20) 1.63 ms instead of 1.42. Smaller ones lose by it
// (4, N = 32: 22.3 -> 25.0 ms; 3, N = 24: 3.94 -> 4.55).
__host__ __device__ constexpr bool df_loop(int BK) { return df_side(BK) >= 5; }

// One HB x HB square (KIND as in sum_block); rows of the weights are BK apart. LOOP: win[i] meets output
// i of the current m3, otherwise slot (i - u) mod HB.
template <int KIND, int BK, int HB>
__device__ __forceinline__ void sum_block_df(const float* wh, const float* wl, const float4* ra, const float4* rb,
                                             float4 (&win)[HB], float (&rh)[HB], float (&rl)[HB], float (&ih)[HB],
                                             float (&il)[HB]) {
  constexpr bool kLoop = df_loop(BK);
  auto row = [&](int u) {
    const float4 bv = rb[u * kLanes];
    float h[HB], l[HB];
    load_weights<float, HB>(wh + u * BK, h);
    load_weights<float, HB>(wl + u * BK, l);
#pragma unroll
    for (int i = 0; i < HB; i++) {
      if ((KIND < 0 && i >= u) || (KIND > 0 && i <= u)) continue;
      const float4 av = win[kLoop ? i : (i - u + HB) % HB];
      // w b = (w b_re, w b_im), leading parts exact
      float brh = h[i] * bv.x, brl = fmaf(h[i], bv.x, -brh);
      brl = fmaf(h[i], bv.y, brl);
      brl = fmaf(l[i], bv.x, brl);
      float bih = h[i] * bv.z, bil = fmaf(h[i], bv.z, -bih);
      bil = fmaf(h[i], bv.w, bil);
      bil = fmaf(l[i], bv.z, bil);
      // a (w b): re += a_re br - a_im bi, im += a_re bi + a_im br
      df_mul_acc(av.x, av.y, brh, brl, rh[i], rl[i]);
      df_mul_acc(-av.z, -av.w, bih, bil, rh[i], rl[i]);
      df_mul_acc(av.x, av.y, bih, bil, ih[i], il[i]);
      df_mul_acc(av.z, av.w, brh, brl, ih[i], il[i]);
    }
  };
  if constexpr (kLoop) {
#pragma unroll 1
    for (int u = KIND < 0 ? 1 : 0; u < HB; u++) {
#pragma unroll
      for (int i = HB - 1; i > 0; i--) win[i] = win[i - 1];
      if (KIND <= 0) win[0] = ra[-u * kLanes];
      row(u);
    }
  } else {
#pragma unroll
    for (int u = 0; u < HB; u++) {
      if (KIND == 0 || (KIND < 0 && u > 0)) win[(HB - u) % HB] = ra[-u * kLanes];
      row(u);
    }
  }
}

template <int BK>
__global__ void __launch_bounds__(128 * (BK / df_side(BK)), 2) k_sum_df(SumDfArgs a) {
  constexpr int H = 2 * BK - 1, n = 4 * BK - 1;
  constexpr int HB = df_side(BK), per = BK / HB;  // squares of HB; per block side
  constexpr int NB = 4 * per, D = 2 * per;         // squares along a row; |kb - c| = D is the triangle
  constexpr int PW = (sum_weights(BK) + 3) / 4 * 4;
  constexpr int kRow = n * kLanes;
  constexpr int kRows = kRow + (n + 1) * kLanes;
  extern __shared__ __align__(128) unsigned char smraw[];
  float* Wb = (float*)smraw;                                 // [2][2][PW]: buffer, (hi, lo)
  float4* rows = (float4*)(smraw + 4 * PW * sizeof(float));  // [2][kRows]: buffer, (a, b)
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int s_err;

  const int4 ud = a.units[blockIdx.x];
  const long long step0 = a.unit_step0[blockIdx.x];
  const int k1 = ud.x, k2 = ud.y, m1lo = ud.z, m1hi = ud.w;
  const int m2lo = max(-H, k2 - H), m2hi = min(H, k2 + H);
  const int nm2 = m2hi - m2lo + 1;
  const int S = (m1hi - m1lo + 1) * nm2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // warps kb and kb + 4 share a scheduler and have 11 full squares between them for every kb
  const int kb = warp;
  const int g = blockIdx.y;
  const uint32_t row_bytes = kRow * sizeof(float4);
  const uint32_t stage_bytes = 2 * PW * sizeof(float) + 2 * row_bytes;

  if (a.active) {
    // a group with no cell of an active instance has nothing to compute (every warp of the
    // block serves the same group: one warp's vote decides)
    const int c = g * kLanes + lane;
    const bool mine = c < a.C && a.active[a.cell_inst[c]];
    if (!__any_sync(0xffffffffu, mine)) return;
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    s_err = 0;
    fence_mbar_init();
  }
  if (warp < 2) rows[warp * kRows + kRows - kLanes + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  __syncthreads();

  auto issue = [&](int s) {
    int m1 = m1lo + s / nm2, m2 = m2lo + s % nm2;
    int b = s & 1;
    mbar_arrive_expect_tx(&bar[b], stage_bytes);
    bulk_g2s(Wb + (2 * b) * PW, a.Whi + (step0 + s) * PW, PW * sizeof(float), &bar[b]);
    bulk_g2s(Wb + (2 * b + 1) * PW, a.Wlo + (step0 + s) * PW, PW * sizeof(float), &bar[b]);
    long long ga = (((long long)g * n + (k1 - m1 + H)) * n + (k2 - m2 + H)) * kRow;
    long long gb = (((long long)g * n + (m1 + H)) * n + (m2 + H)) * kRow;
    float4* dst = rows + b * kRows;
    bulk_g2s(dst, a.ahat + ga, row_bytes, &bar[b]);
    bulk_g2s(dst + kRow, a.bhat + gb, row_bytes, &bar[b]);
  };

  if (threadIdx.x == 0 && S > 0) issue(0);

  float rh[HB], rl[HB], ih[HB], il[HB];
#pragma unroll
  for (int j = 0; j < HB; j++) rh[j] = rl[j] = ih[j] = il[j] = 0.0f;

  int fail_b = 0, fail_par = 0;
  for (int s = 0; s < S; s++) {
    const int b = s & 1;
    if (!mbar_wait(&bar[b], (s >> 1) & 1, a.spin_max)) {
      s_err = 1;
      fail_b = b;
      fail_par = (s >> 1) & 1;
    }
    __syncthreads();
    if (s_err) break;
    // the other buffer was released by the barrier above: prefetch the next step into it
    if (threadIdx.x == 0 && s + 1 < S) issue(s + 1);
    const float4* ra = rows + b * kRows + (kb * HB + 2 * BK - 1) * kLanes + lane;
    const float4* rb = rows + b * kRows + kRow + lane;
    // weights of square (kb, c): inside block (kb / per, c / per)
    const int kB = kb / per;
    const float* W0 = Wb + (2 * b) * PW + (sum_first_block(kB) - max(0, kB - 2)) * BK * BK + (kb % per) * HB;
    auto wat = [&](int c) { return W0 + (c / per) * BK * BK + (c % per) * HB * BK; };
    float4 win[HB];
    int c = max(0, kb - D + 1);
    if (kb >= D) {
      const int cl = kb - D;
      const float* w = wat(cl);
      sum_block_df<-1, BK, HB>(w, w + PW, ra - cl * HB * kLanes, rb + cl * HB * kLanes, win, rh, rl, ih, il);
    } else {
#pragma unroll
      for (int i = 1; i < HB; i++) win[df_loop(BK) ? i - 1 : i] = ra[i * kLanes];
    }
    const int c1 = min(NB - 1, kb + D - 1);
#pragma unroll 1
    for (; c <= c1; c++) {
      const float* w = wat(c);
      sum_block_df<0, BK, HB>(w, w + PW, ra - c * HB * kLanes, rb + c * HB * kLanes, win, rh, rl, ih, il);
    }
    if (kb < NB - D) {
      const float* w = wat(c);
      sum_block_df<1, BK, HB>(w, w + PW, ra, rb + c * HB * kLanes, win, rh, rl, ih, il);
    }
  }
  if (s_err) {
    if (threadIdx.x == 0) {
      atomicOr(&a.cnt[0].status, SGS_ST_TIMEOUT);
      mbar_wait(&bar[fail_b], fail_par, a.spin_max);
    }
    return;
  }
  double2* out = a.partial + ((long long)blockIdx.x * a.Gs + g) * kRow;
#pragma unroll
  for (int i = 0; i < HB; i++)
    if (kb * HB + i < n)
      out[(kb * HB + i) * kLanes + lane] =
          make_double2((double)rh[i] + (double)rl[i], (double)ih[i] + (double)il[i]);
}

// In place: every complex FP64 value of the transformed rows becomes its (hi, lo) float pairs
// (re_hi, re_lo, im_hi, im_lo), the layout k_sum_df reads.
__global__ void k_split_spec(double2* x, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    double2 v = x[i];
    dfloat r = df_split(v.x), m = df_split(v.y);
    reinterpret_cast<float4*>(x)[i] = make_float4(r.hi, r.lo, m.hi, m.lo);
  }
}

// Fixed-order sum of a row's unit partials (FP64 accumulation), written to qhat at (k1, k2,
// k3) and conjugated at (-k1, -k2, -k3); row (0, 0) is computed in full and not mirrored.
template <typename T>
__global__ void k_sum_reduce(RedArgs<T> a) {
  typedef typename CplxOf<T>::type CT;
  int row = blockIdx.x, g = blockIdx.y;
  int n = a.n, H = (n - 1) / 2;
  int k1 = a.row_k[row].x, k2 = a.row_k[row].y;
  int u0 = a.row_start[row], u1 = a.row_start[row + 1];
  for (int t = threadIdx.x; t < n * kLanes; t += blockDim.x) {
    double sr = 0.0, si = 0.0;
    for (int q = u0; q < u1; q++) {
      int u = a.row_units[q];
      CT v = a.partial[((long long)u * a.Gs + g) * n * kLanes + t];
      sr += (double)v.x;
      si += (double)v.y;
    }
    if (a.partial2)
      for (int q = u0; q < u1; q++) {
        int u = a.row_units[q];
        CT v = a.partial2[((long long)u * a.Gs + g) * n * kLanes + t];
        sr += (double)v.x;
        si += (double)v.y;
      }
    int k3i = t / kLanes, lane = t % kLanes;
    long long o = ((((long long)g * n + (k1 + H)) * n + (k2 + H)) * n + k3i) * kLanes + lane;
    a.qhat[o] = make_cplx((T)sr, (T)si);
    if (k1 != 0 || k2 != 0) {
      long long om = ((((long long)g * n + (H - k1)) * n + (H - k2)) * n + (n - 1 - k3i)) * kLanes + lane;
      a.qhat[om] = make_cplx((T)sr, (T)(-si));
    }
  }
}

// ---------------------------------------------------------------------------------------
// Inverse DFT, q(v) = Re sum_k qhat_k exp(+i 2 pi k j / N).
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_idft_k1(SpecBufs<T> sb, int N) {
  typedef typename CplxOf<T>::type CT;
  extern __shared__ __align__(16) unsigned char smraw[];
  int n = N - 1;
  T* cs = (T*)smraw;
  T* sn = cs + n * N;
  CT* x = (CT*)(sn + n * N);  // [k1][k3]
  int c = blockIdx.x, k2 = blockIdx.y;
  if (!cell_active(sb.active, sb.cell_inst, c)) return;
  int g = c / kLanes, lane = c % kLanes;
  for (int t = threadIdx.x; t < n * N; t += blockDim.x) {
    cs[t] = sb.twc[t];
    sn[t] = sb.tws[t];
  }
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    int k1 = t / n, k3 = t % n;
    x[t] = sb.qhat[((((long long)g * n + k1) * n + k2) * n + k3) * kLanes + lane];
  }
  __syncthreads();
  CT* o = sb.st2a + (long long)c * N * n * n;  // [i1][k2][k3]
  constexpr int TR = kDftTile<T>;
  for (int t = threadIdx.x; t < N / TR * n; t += blockDim.x) {
    const int i1 = t / n * TR, k3 = t % n;
    T re[TR], im[TR];
#pragma unroll
    for (int q = 0; q < TR; q++) re[q] = im[q] = 0;
    for (int k1 = 0; k1 < n; k1++) {
      T co[TR], si[TR];
      load_tile_row<T, TR>(cs + k1 * N + i1, co);
      load_tile_row<T, TR>(sn + k1 * N + i1, si);
      const CT v = x[k1 * n + k3];
#pragma unroll
      for (int q = 0; q < TR; q++) idft_add(re[q], im[q], v.x, v.y, co[q], si[q]);
    }
#pragma unroll
    for (int q = 0; q < TR; q++) o[((long long)(i1 + q) * n + k2) * n + k3] = make_cplx(re[q], im[q]);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_idft_k2(SpecBufs<T> sb, int N) {
  typedef typename CplxOf<T>::type CT;
  extern __shared__ __align__(16) unsigned char smraw[];
  int n = N - 1;
  T* cs = (T*)smraw;
  T* sn = cs + n * N;
  CT* x = (CT*)(sn + n * N);  // [k2][k3]
  int c = blockIdx.x, i1 = blockIdx.y;
  if (!cell_active(sb.active, sb.cell_inst, c)) return;
  for (int t = threadIdx.x; t < n * N; t += blockDim.x) {
    cs[t] = sb.twc[t];
    sn[t] = sb.tws[t];
  }
  const CT* src = sb.st2a + ((long long)c * N + i1) * n * n;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) x[t] = src[t];
  __syncthreads();
  CT* o = sb.st1a + ((long long)c * N + i1) * N * n;  // [i2][k3]
  constexpr int TR = kDftTile<T>;
  for (int t = threadIdx.x; t < N / TR * n; t += blockDim.x) {
    const int i2 = t / n * TR, k3 = t % n;
    T re[TR], im[TR];
#pragma unroll
    for (int q = 0; q < TR; q++) re[q] = im[q] = 0;
    for (int k2 = 0; k2 < n; k2++) {
      T co[TR], si[TR];
      load_tile_row<T, TR>(cs + k2 * N + i2, co);
      load_tile_row<T, TR>(sn + k2 * N + i2, si);
      const CT v = x[k2 * n + k3];
#pragma unroll
      for (int q = 0; q < TR; q++) idft_add(re[q], im[q], v.x, v.y, co[q], si[q]);
    }
#pragma unroll
    for (int q = 0; q < TR; q++) o[(i2 + q) * n + k3] = make_cplx(re[q], im[q]);
  }
}

// Last pass: real part along index 3, then Q and P = Q - nu (M - f) in FP64.
template <typename T>
__global__ void __launch_bounds__(256) k_idft_k3(SpecBufs<T> sb, const double* __restrict__ f, CellTables ct,
                                                  const double* efac, const double* nu, double* Q, double* P,
                                                  int N, double dv, const double* __restrict__ Qadd,
                                                  double* __restrict__ mom) {
  typedef typename CplxOf<T>::type CT;
  extern __shared__ __align__(16) unsigned char smraw[];
  int n = N - 1;
  T* cs = (T*)smraw;
  T* sn = cs + n * N;
  CT* x = (CT*)(sn + n * N);  // [i2][k3]
  __shared__ double E12[kMaxN], E3[kMaxN];
  int c = blockIdx.x, i1 = blockIdx.y;
  if (!cell_active(ct.active, ct.cell_inst, c)) return;
  if (threadIdx.x < N) {
    const double* e = efac + (long long)c * 3 * kMaxN;
    E12[threadIdx.x] = e[i1] * e[kMaxN + threadIdx.x];
    E3[threadIdx.x] = e[2 * kMaxN + threadIdx.x];
  }
  for (int t = threadIdx.x; t < n * N; t += blockDim.x) {
    cs[t] = sb.twc[t];
    sn[t] = sb.tws[t];
  }
  const CT* src = sb.st1a + ((long long)c * N + i1) * N * n;
  for (int t = threadIdx.x; t < N * n; t += blockDim.x) x[t] = src[t];
  __syncthreads();
  long long base = ct.cell_off[c] + (long long)i1 * N * N;
  double nuc = nu[c];
  // moments of this slab for the conservation projection: sum q, v2 q, v3 q, (v2^2 + v3^2) q
  double m0 = 0.0, m2 = 0.0, m3 = 0.0, m4 = 0.0;
  for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
    int i2 = t / N, i3 = t % N;
    T re = 0;
    for (int k3 = 0; k3 < n; k3++) {
      CT q = x[i2 * n + k3];
      re += q.x * cs[k3 * N + i3] - q.y * sn[k3 * N + i3];
    }
    double q = (double)re;
    if (Qadd) q += Qadd[base + t];
    if (Q) Q[base + t] = q;
    if (P) {
      double M = E12[i2] * E3[i3];
      P[base + t] = q - nuc * (M - f[base + t]);
    }
    if (mom) {
      double v2 = (i2 - N / 2 + 1) * dv, v3 = (i3 - N / 2 + 1) * dv;
      m0 += q;
      m2 += v2 * q;
      m3 += v3 * q;
      m4 += (v2 * v2 + v3 * v3) * q;
    }
  }
  if (mom) {  // fixed-order block reduction (warp butterflies, then warps in order)
    __shared__ double red[4][8];
    for (int o = 16; o > 0; o >>= 1) {
      m0 += __shfl_xor_sync(0xffffffffu, m0, o);
      m2 += __shfl_xor_sync(0xffffffffu, m2, o);
      m3 += __shfl_xor_sync(0xffffffffu, m3, o);
      m4 += __shfl_xor_sync(0xffffffffu, m4, o);
    }
    int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      red[0][w] = m0;
      red[1][w] = m2;
      red[2][w] = m3;
      red[3][w] = m4;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      for (int j = 0; j < 4; j++)
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) s[j] += red[j][k];
      double v1 = (i1 - N / 2 + 1) * dv;
      double* o = mom + ((long long)c * N + i1) * 5;
      o[0] = s[0];
      o[1] = v1 * s[0];
      o[2] = s[1];
      o[3] = s[2];
      o[4] = v1 * v1 * s[0] + s[3];
    }
  }
}

// Conservation projection (an option; not in the paper), applied to Q and to
// P = Q - nu (M - f) alike, with phi = (1, v1, v2, v3, |v|^2) and the moments sum_k phi Q from
// the slabs of k_idft_k3, summed here in i1 order (every block of a cell forms the same lambda):
//   mode 1: Q_c = Q - sum_i lambda_i phi_i,      (sum_k phi phi^T) lambda = sum_k phi Q,
//           with the inverse Gram matrix Ainv of the grid;
//   mode 2: Q_c = Q - M sum_i lambda_i phi_i,    (sum_k M phi phi^T) lambda = sum_k phi Q,
//           with the cell's Maxwellian M = E1(v1) E2(v2) E3(v3) (factors efac): its Gram
//           matrix is a sum of products of the 1-D sums S_d^p = sum_i E_d(v_i) v_i^p.
__device__ bool chol5_solve(double A[5][5], const double* b, double* x) {
  for (int i = 0; i < 5; i++)
    for (int j = 0; j <= i; j++) {
      double t = A[i][j];
      for (int k = 0; k < j; k++) t -= A[i][k] * A[j][k];
      if (i == j) {
        if (!(t > 0.0)) return false;
        A[i][i] = sqrt(t);
      } else {
        A[i][j] = t / A[j][j];
      }
    }
  double z[5];
  for (int i = 0; i < 5; i++) {
    double t = b[i];
    for (int k = 0; k < i; k++) t -= A[i][k] * z[k];
    z[i] = t / A[i][i];
  }
  for (int i = 4; i >= 0; i--) {
    double t = z[i];
    for (int k = i + 1; k < 5; k++) t -= A[k][i] * x[k];
    x[i] = t / A[i][i];
  }
  return true;
}

__global__ void __launch_bounds__(256) k_conserve_apply(const double* __restrict__ mom,
                                                        const double* __restrict__ Ainv,
                                                        const double* __restrict__ efac, int mode, CellTables ct,
                                                        double* Q, double* P, double* Qraw, int N, double dv) {
  __shared__ double sm[5], lam[5], S[3][5];
  int c = blockIdx.x, i1 = blockIdx.y;
  if (!cell_active(ct.active, ct.cell_inst, c)) return;
  const double* e = efac + (long long)c * 3 * kMaxN;
  if (threadIdx.x < 5) {
    double a = 0.0;
    const double* m = mom + (long long)c * N * 5 + threadIdx.x;
    for (int j = 0; j < N; j++) a += m[j * 5];
    sm[threadIdx.x] = a;
  } else if (mode == 2 && threadIdx.x < 20) {
    int d = (threadIdx.x - 5) / 5, p = (threadIdx.x - 5) % 5;
    double a = 0.0;
    for (int i = 0; i < N; i++) {
      double v = (i - N / 2 + 1) * dv, vp = 1.0;
      for (int k = 0; k < p; k++) vp *= v;
      a += e[d * kMaxN + i] * vp;
    }
    S[d][p] = a;
  }
  __syncthreads();
  if (mode == 1 && threadIdx.x < 5) {
    double a = 0.0;
    for (int k = 0; k < 5; k++) a += Ainv[threadIdx.x * 5 + k] * sm[k];
    lam[threadIdx.x] = a;
  } else if (mode == 2 && threadIdx.x == 0) {
    // phi as monomials v1^a v2^b v3^c: 1, v1, v2, v3 and |v|^2 = v1^2 + v2^2 + v3^2
    const int nm[5] = {1, 1, 1, 1, 3};
    const int mono[5][3][3] = {{{0, 0, 0}}, {{1, 0, 0}}, {{0, 1, 0}}, {{0, 0, 1}},
                               {{2, 0, 0}, {0, 2, 0}, {0, 0, 2}}};
    double A[5][5];
    for (int a = 0; a < 5; a++)
      for (int b = 0; b < 5; b++) {
        double t = 0.0;
        for (int x = 0; x < nm[a]; x++)
          for (int y = 0; y < nm[b]; y++)
            t += S[0][mono[a][x][0] + mono[b][y][0]] * S[1][mono[a][x][1] + mono[b][y][1]] *
                 S[2][mono[a][x][2] + mono[b][y][2]];
        A[a][b] = t;
      }
    double x[5];
    if (!chol5_solve(A, sm, x))
      for (int k = 0; k < 5; k++) x[k] = 0.0;
    for (int k = 0; k < 5; k++) lam[k] = x[k];
  }
  __syncthreads();
  double v1 = (i1 - N / 2 + 1) * dv;
  double c0 = lam[0] + lam[1] * v1 + lam[4] * v1 * v1;
  double e1 = mode == 2 ? e[i1] : 1.0;
  long long base = ct.cell_off[c] + (long long)i1 * N * N;
  for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
    int i2 = t / N, i3 = t % N;
    double v2 = (i2 - N / 2 + 1) * dv, v3 = (i3 - N / 2 + 1) * dv;
    double corr = c0 + lam[2] * v2 + lam[3] * v3 + lam[4] * (v2 * v2 + v3 * v3);
    if (mode == 2) corr *= e1 * e[kMaxN + i2] * e[2 * kMaxN + i3];
    if (Qraw) Qraw[base + t] = Q[base + t];  // the unprojected operator (increment-form reference)
    if (Q) Q[base + t] -= corr;
    if (P) P[base + t] -= corr;
  }
}

// BGK mode (eq. (12)): Q = nu (M - f), P = 0.
__global__ void __launch_bounds__(256) k_collide_bgk(const double* __restrict__ f, CellTables ct,
                                                      const double* theta, const double* nu, double* Q, double* P,
                                                      int N, double dv) {
  __shared__ double E[3 * kMaxN];
  int c = blockIdx.x, i1 = blockIdx.y;
  if (!cell_active(ct.active, ct.cell_inst, c)) return;
  if (threadIdx.x < 3 * N) {
    const int d = threadIdx.x / N, i = threadIdx.x % N;
    E[d * kMaxN + i] = maxwell_factor(theta + 5 * (long long)c, d, i, N, dv);
  }
  __syncthreads();
  long long base = ct.cell_off[c] + (long long)i1 * N * N;
  double nuc = nu[c];
  for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
    int i2 = t / N, i3 = t % N;
    double M = E[i1] * E[kMaxN + i2] * E[2 * kMaxN + i3];
    if (Q) Q[base + t] = nuc * (M - f[base + t]);
    if (P) P[base + t] = 0.0;
  }
}

// ---------------------------------------------------------------------------------------
// Setup: weights W[step][p] = beta_s of the (k3, m3) pairs of each (k1, k2, m1, m2) step, in the
// block order of k_sum, from the tables G[a2][b2] and Lo[m2] = G(2|m|, 0).
// ---------------------------------------------------------------------------------------
template <typename T, bool LO>
__global__ void k_build_weights(const int4* units, const long long* unit_step0, int n_units, int H, int PW,
                                const double* G, long long nb, const double* Lo, T* W) {
  int u = blockIdx.x;
  if (u >= n_units) return;
  int4 ud = units[u];
  int k1 = ud.x, k2 = ud.y;
  int m2lo = max(-H, k2 - H), m2hi = min(H, k2 + H);
  int nm2 = m2hi - m2lo + 1;
  int S = (ud.w - ud.z + 1) * nm2;
  const int BK = (H + 1) / 2, n = 2 * H + 1, np = sum_weights(BK);
  for (int s = blockIdx.y; s < S; s += gridDim.y) {
    int m1 = ud.z + s / nm2, m2 = m2lo + s % nm2;
    T* out = W + (unit_step0[u] + s) * PW;
    for (int p = threadIdx.x; p < PW; p += blockDim.x) {
      // p -> block (kb, c), m3, k3 in the k_sum order
      const int blk = p / (BK * BK), in = p % (BK * BK);
      const int kb = blk < 3 ? 0 : (blk < 7 ? 1 : (blk < 11 ? 2 : 3));
      const int c = max(0, kb - 2) + blk - sum_first_block(kb);
      const int ki = kb * BK + in % BK, mi = c * BK + in / BK;
      const int k3 = ki - H, m3 = mi - H;
      if (p >= np || ki >= n || mi >= n || abs(k3 - m3) > H) {
        out[p] = (T)0;
        continue;
      }
      long long a2 = (long long)k1 * k1 + (long long)k2 * k2 + (long long)k3 * k3;
      long long d1 = k1 - 2 * m1, d2 = k2 - 2 * m2, d3 = k3 - 2 * m3;
      long long b2 = d1 * d1 + d2 * d2 + d3 * d3;
      long long l1 = k1 - m1, l2 = k2 - m2, l3 = k3 - m3;
      long long ll = l1 * l1 + l2 * l2 + l3 * l3;
      long long mm = (long long)m1 * m1 + (long long)m2 * m2 + (long long)m3 * m3;
      double w = G[a2 * nb + b2] - 0.5 * (Lo[ll] + Lo[mm]);
      // LO: the FP32 remainder w - (float)w, the low half of a double-float weight whose high
      // half is the FP32 weight table
      out[p] = LO ? (T)(w - (double)(float)w) : (T)w;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Host-side launchers.
// ---------------------------------------------------------------------------------------
template <typename T>
static size_t dft_smem(int N, int extra_cplx, int extra_real) {
  typedef typename CplxOf<T>::type CT;
  // tables of at most N x N (padded tiles), then the slabs
  return 2 * N * N * sizeof(T) + extra_cplx * sizeof(CT) + extra_real * sizeof(T);
}

// Lane groups per block of a sum over `groups` of them that takes F steps at once: as many as asked
// for, within an SM's shared memory; one in FP64, where eight warps that wait for each other at a
// step's barrier leave the pipe idle more than four (two groups a block against one: 200 cells of 8^3 98
// against 87 us, 64 of 12^3 347 and 322, of 24^3 21.4 and 21.3 ms, of 32^3 128.4 and 126.8; the other way at
// 64 cells of 20^3, 6.81 and 6.88). The units don't follow it, so the bits don't either.
static size_t sum_group_bytes(int BK, int elem_bytes) {
  return (size_t)2 * (2 * (4 * BK - 1) + 1) * kLanes * 2 * elem_bytes;
}
static size_t sum_weight_bytes(int BK, int elem_bytes, int F) {
  return 2 * F * ((size_t)sum_pad(2 * BK - 1, elem_bytes) * elem_bytes + (F > 1 ? 16 : 0));
}
static int sum_groups(int BK, int elem_bytes, int F, int NW, int groups) {
  const int fit = (int)((220 * 1024 - sum_weight_bytes(BK, elem_bytes, F)) / sum_group_bytes(BK, elem_bytes));
  return std::max(1, std::min(std::min(elem_bytes == 8 ? 1 : NW, groups), fit));
}

template <typename T, int BK, int F>
static cudaError_t launch_sum_f(const SumArgs<T>& a, int NW, int n_units, cudaStream_t st) {
  const int groups = a.G - a.g0;
  const int NG = sum_groups(BK, sizeof(T), F, NW, groups);
  const size_t smem = sum_weight_bytes(BK, sizeof(T), F) + NG * sum_group_bytes(BK, sizeof(T));
  cudaError_t e = func_attr((const void*)k_sum<T, BK, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  dim3 grid(n_units, (groups + NG - 1) / NG);
  k_sum<T, BK, F><<<grid, NG * 128, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T, int BK>
static cudaError_t launch_sum_t(const SumArgs<T>& a, int NW, int n_units, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    if (a.fold > 1) {  // the last group's rows hold 32 / fold lanes; the others are as usual
      SumArgs<T> x = a;
      if (a.G > 1) {
        x.G = a.G - 1;
        cudaError_t e = launch_sum_f<T, BK, 1>(x, NW, n_units, st);
        if (e != cudaSuccess) return e;
        x.G = a.G;
      }
      x.g0 = a.G - 1;
      return a.fold == 4 ? launch_sum_f<T, BK, 4>(x, 1, n_units, st) : launch_sum_f<T, BK, 2>(x, 1, n_units, st);
    }
  }
  if constexpr (sizeof(T) == 4 && sum_in_registers(BK)) {
    constexpr size_t row_bytes = (size_t)2 * (4 * BK - 1) * kLanes * sizeof(float2);
    const int nw = std::min(NW, a.G);
    const size_t smem = 2 * sum_pad(2 * BK - 1, 4) * sizeof(float) + nw * row_bytes;
    cudaError_t e = func_attr((const void*)k_sum_regs<BK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_sum_regs<BK><<<dim3(n_units, (a.G + nw - 1) / nw), nw * 32, smem, st>>>(a);
    return cudaGetLastError();
  } else {
    return launch_sum_f<T, BK, 1>(a, NW, n_units, st);
  }
}

int sum_pad(int H, int elem_bytes) {
  int NP = sum_weights((H + 1) / 2), VEC = 16 / elem_bytes;
  return (NP + VEC - 1) / VEC * VEC;
}

template <typename T>
SumShape sum_shape(const SumArgs<T>& a, int H, int NW, int n_units) {
  const int BK = (H + 1) / 2, folded = a.fold > 1 ? 1 : 0, rest = a.G - folded;
  SumShape x;
  x.launches = (rest > 0 ? 1 : 0) + folded;
  x.warps = rest > 0 ? sum_groups(BK, sizeof(T), 1, NW, rest) : 1;
  x.blocks = n_units * ((rest + x.warps - 1) / x.warps + folded);
  return x;
}

template <typename T>
cudaError_t launch_sum(const SumArgs<T>& a, int H, int NW, int n_units, cudaStream_t st) {
  if (NW < 1 || NW > 4) return cudaErrorInvalidValue;
  switch (H) {
    case 3: return launch_sum_t<T, 2>(a, NW, n_units, st);
    case 5: return launch_sum_t<T, 3>(a, NW, n_units, st);
    case 7: return launch_sum_t<T, 4>(a, NW, n_units, st);
    case 9: return launch_sum_t<T, 5>(a, NW, n_units, st);
    case 11: return launch_sum_t<T, 6>(a, NW, n_units, st);
    case 13: return launch_sum_t<T, 7>(a, NW, n_units, st);
    case 15: return launch_sum_t<T, 8>(a, NW, n_units, st);
  }
  return cudaErrorInvalidValue;
}

template <int BK>
static cudaError_t launch_sum_df_t(const SumDfArgs& a, int n_units, cudaStream_t st) {
  constexpr int n = 4 * BK - 1;
  constexpr int PW = (sum_weights(BK) + 3) / 4 * 4;
  const size_t smem = 4 * PW * sizeof(float) + (size_t)2 * (2 * n + 1) * kLanes * sizeof(float4);
  cudaError_t e = func_attr((const void*)k_sum_df<BK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_sum_df<BK><<<dim3(n_units, a.G), 128 * (BK / df_side(BK)), smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sum_df(const SumDfArgs& a, int H, int n_units, cudaStream_t st) {
  switch (H) {
    case 3: return launch_sum_df_t<2>(a, n_units, st);
    case 5: return launch_sum_df_t<3>(a, n_units, st);
    case 7: return launch_sum_df_t<4>(a, n_units, st);
    case 9: return launch_sum_df_t<5>(a, n_units, st);
    case 11: return launch_sum_df_t<6>(a, n_units, st);
    case 13: return launch_sum_df_t<7>(a, n_units, st);
    case 15: return launch_sum_df_t<8>(a, n_units, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_split_spec(double2* x, long long count, cudaStream_t st) {
  k_split_spec<<<(int)std::min<long long>((count + 255) / 256, 152 * 16), 256, 0, st>>>(x, count);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_dft(const double* f, const CollideCtx<T>& x, const DftMode& md, cudaStream_t st) {
  int N = x.N, n = N - 1, C = x.C;
  cudaError_t e;
  // the factors of this step were written by launch_moments, those of the reference by the first
  // of the two transforms of an increment
  if (md.mode == 1) k_factors<<<C, 3 * N, 0, st>>>(md.theta_ref, N, x.dv, x.efac_ref);
  size_t sm1 = dft_smem<T>(N, 0, 2 * N * (N + kDftTile<T>));
  e = func_attr((const void*)k_dft_i3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm1);
  if (e != cudaSuccess) return e;
  k_dft_i3<T><<<dim3(C, N), 256, sm1, st>>>(f, x.ct, x.efac, x.efac_ref, x.sb, N, x.dv, md);
  size_t sm2 = dft_smem<T>(N, 2 * N * n, 0);
  e = func_attr((const void*)k_dft_i2<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2);
  if (e != cudaSuccess) return e;
  k_dft_i2<T><<<dim3(C, N), 256, sm2, st>>>(x.sb, N);
  e = func_attr((const void*)k_dft_i1<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2);
  if (e != cudaSuccess) return e;
  // lanes beyond the last cell hold anything and are never read back: no lane of a sum reads another
  // one's cell (a folded group's lanes are those of its cells)
  k_dft_i1<T><<<dim3(C, n), 256, sm2, st>>>(x.sb, N);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_spectral_sum(const CollideCtx<T>& x, typename CplxOf<T>::type* partial, cudaStream_t st) {
  SumArgs<T> a = x.sum;
  if (partial) a.partial = partial;
  return launch_sum<T>(a, x.H, x.NW, x.n_units, st);
}

template <typename T>
cudaError_t launch_reduce_idft(const double* f, double* Q, double* P, const CollideCtx<T>& x,
                               const typename CplxOf<T>::type* partial2, const double* Qadd, cudaStream_t st,
                               double* Qraw) {
  int N = x.N, n = N - 1, C = x.C;
  cudaError_t e;
  RedArgs<T> ra = x.red;
  ra.partial2 = partial2;
  // n_rows = 0: qhat is already complete (the fast operator writes it directly)
  if (x.red.n_rows > 0) k_sum_reduce<T><<<dim3(x.red.n_rows, x.red.G), 256, 0, st>>>(ra);
  size_t sm3 = dft_smem<T>(N, n * n, 0);
  e = func_attr((const void*)k_idft_k1<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm3);
  if (e != cudaSuccess) return e;
  k_idft_k1<T><<<dim3(C, n), 256, sm3, st>>>(x.sb, N);
  e = func_attr((const void*)k_idft_k2<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm3);
  if (e != cudaSuccess) return e;
  k_idft_k2<T><<<dim3(C, N), 256, sm3, st>>>(x.sb, N);
  size_t sm4 = dft_smem<T>(N, N * n, 0);
  e = func_attr((const void*)k_idft_k3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm4);
  if (e != cudaSuccess) return e;
  // the factors of this collision step were written by launch_moments
  k_idft_k3<T><<<dim3(C, N), 256, sm4, st>>>(x.sb, f, x.ct, x.efac, x.nu, Q, P, N, x.dv, Qadd, x.mom);
  e = cudaGetLastError();
  if (e != cudaSuccess || !x.mom) return e;
  if (Qraw && !Q) return cudaErrorInvalidValue;
  k_conserve_apply<<<dim3(C, N), 256, 0, st>>>(x.mom, x.cproj, x.efac, x.cproj_mode, x.ct, Q, P, Qraw, N, x.dv);
  return cudaGetLastError();
}

cudaError_t launch_factors(const double* theta, int C, int N, double dv, double* efac, cudaStream_t st) {
  k_factors<<<C, 3 * N, 0, st>>>(theta, N, dv, efac);
  return cudaGetLastError();
}

// Cells below which the warps of a cell go to different SMs: with more of them the chip's FP64
// pipes are busy either way, and a CTA per warp only adds launches (128 cells of 32^3: 132 us in
// one CTA a cell, 122 with a CTA per warp, 98 with two CTAs).
constexpr int kMomentsSplit = 304;

cudaError_t launch_moments(const double* f, const CellTables& ct, int C, int N, double dv, double tol, int maxit,
                           double* theta, double* nu, double* efac, Counters* cnt, cudaStream_t st) {
  if (C > kMomentsSplit) {
    k_moments<false><<<C, kMomentsThreads<false>, 0, st>>>(f, ct, N, dv, tol, maxit, theta, nu, efac, cnt);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * C);
  cfg.blockDim = dim3(kMomentsThreads<true>);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_moments<true>, f, ct, N, dv, tol, maxit, theta, nu, efac, cnt);
}

cudaError_t launch_collide_bgk(const double* f, const CellTables& ct, int C, int N, double dv, const double* theta,
                               const double* nu, double* Q, double* P, cudaStream_t st) {
  k_collide_bgk<<<dim3(C, N), 256, 0, st>>>(f, ct, theta, nu, Q, P, N, dv);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_build_weights(const int4* units, const long long* unit_step0, int n_units, int H, int PW,
                                 const double* G, long long nb, const double* Lo, T* W, cudaStream_t st) {
  k_build_weights<T, false><<<dim3(n_units, 8), 256, 0, st>>>(units, unit_step0, n_units, H, PW, G, nb, Lo, W);
  return cudaGetLastError();
}

cudaError_t launch_build_weights_lo(const int4* units, const long long* unit_step0, int n_units, int H, int PW,
                                    const double* G, long long nb, const double* Lo, float* W, cudaStream_t st) {
  k_build_weights<float, true><<<dim3(n_units, 8), 256, 0, st>>>(units, unit_step0, n_units, H, PW, G, nb, Lo, W);
  return cudaGetLastError();
}

template cudaError_t launch_dft<double>(const double*, const CollideCtx<double>&, const DftMode&, cudaStream_t);
template cudaError_t launch_dft<float>(const double*, const CollideCtx<float>&, const DftMode&, cudaStream_t);
template SumShape sum_shape<double>(const SumArgs<double>&, int, int, int);
template SumShape sum_shape<float>(const SumArgs<float>&, int, int, int);
template cudaError_t launch_spectral_sum<double>(const CollideCtx<double>&, double2*, cudaStream_t);
template cudaError_t launch_spectral_sum<float>(const CollideCtx<float>&, float2*, cudaStream_t);
template cudaError_t launch_reduce_idft<double>(const double*, double*, double*, const CollideCtx<double>&,
                                                const double2*, const double*, cudaStream_t, double*);
template cudaError_t launch_reduce_idft<float>(const double*, double*, double*, const CollideCtx<float>&,
                                               const float2*, const double*, cudaStream_t, double*);
template cudaError_t launch_build_weights<double>(const int4*, const long long*, int, int, int, const double*,
                                                  long long, const double*, double*, cudaStream_t);
template cudaError_t launch_build_weights<float>(const int4*, const long long*, int, int, int, const double*,
                                                 long long, const double*, float*, cudaStream_t);

}  // namespace sgs
