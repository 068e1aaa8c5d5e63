// The scan of sgs_dc_step (1-D, double-float): the same SGS scan as k_sweep (sweep.cu), with every
// inner update taken on the nodes: a pass over the cell and a cluster reduction per update.
//
// It is kept for its arithmetic. The increment-form FP32 collision that follows a scan turns a
// change in the last bits of f into its whole FP32 rounding noise: with k_sweep, whose f agrees
// to 4e-14, the Q of two defect-correction iterations differs by 3e-7 from the one with this
// kernel (the error of either against 64 bits is 8.5e-7). The iterates of sgs_dc_step, whose
// results callers compare between versions, therefore keep their scan; every other call runs
// k_sweep, which is faster still (from a cold start, 64 cells of 32^3: 2.4 instead of 10.7 ms with
// this kernel's first form).
//
// A visit is a serial chain: Newton evaluations (some 40) and cluster reductions (2 us each). It is
// bound by the latency of that chain, and an FP64 instruction, which holds its scheduler for 64
// cycles (a conversion: 101), is its dearest link. So a decision is taken in FP32 where that leaves
// no doubt, widening to FP64 is done by integer operations, components are spread over lanes, and a
// warp sum takes 9 double-float additions (warp_sums) instead of 25 to 35. All of it keeps the bits.
// A visit of the defect correction (64 cells, 32 velocities): 180 -> 116 us, 203 -> 125 us beside the
// sums; two iterations of sgs_dc_step 89.4 -> 74.0 ms.
//
// One thread-block cluster walks the instance's cells in scan order inside a single launch.
// Each thread owns EPT consecutive velocity nodes of one pencil (fixed i1, i2) in every cell.
//   - a velocity sum: per-thread partials -> warp butterfly -> block -> one thread per (value,
//     CTA rank) reads the partial through distributed shared memory and a shuffle tree forms the
//     total, identical in every CTA of the cluster (identical branches);
//   - a Newton iteration: warps 0-2 (and one for the step-1 weight) evaluate the factors and 1-D
//     sums of their velocity dimension; after one barrier each of them combines the sums,
//     factorises the Jacobian (FP32: inexact Newton) and takes the same decisions itself;
//   - after the first inner update, the residual and the step-1 target come from the step-2
//     identity (|v1|/dx + A) g + r = A M+ and separable sums.
#include "common.cuh"
#include "kernels.h"

namespace sgs {
namespace {

constexpr int kRedMax = 10;  // values per cluster reduction

typedef dfloat E;  // the arithmetic of the sums and the elementwise work

struct NodesSmem {
  E vv[kMaxN];         // nodes v_i
  E vq[kMaxN];         // v_i^2
  E c1e[kMaxN];        // |v_i| / dx (step-1 weights, x part)
  E den[kMaxN];        // 1 / (|v_i|/dx + nu/eps) of the current cell
  E c1A[kMaxN];        // |v_i|/dx + nu/eps of the current cell
  E ef[3][kMaxN];      // factors of the last Newton evaluation (ef[0] carries exp(alpha))
  E Eg[3][kMaxN];      // factors of M[g]
  E Ep[3][kMaxN];      // factors of the step-1 Maxwellian
  E S[3][5];           // 1-D sums of the last evaluation (unweighted)
  E S1w[5];            // dimension-1 sums with the step-1 weights |v1|/dx, same evaluation
  E Sb[2][4][5];       // Newton evaluations, double-buffered: row r = sums of evaluating warp r
  E Gs[3][6];          // per-dimension sums for the norm of M+ - M[g] (derived residual)
  E svE[5];            // step-1 target s
  E W3[2][kMaxN];      // third factor of each wall's unit Maxwellian
  E red_warp[32][kRedMax];
  E red_tote[kRedMax];
  E thE[5];            // trial theta in E
  E scal[3];           // per-visit scalars: wall densities of the sides, nu/eps
  double red_part[2][kRedMax];
  double red_tot[kRedMax];
  double thg[5], thp[5];
  int ctl;             // broadcast decisions of thread 0
  int nret;            // Newton result, for the warps that do not evaluate
};

__device__ __forceinline__ float shfl_i(float v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ dfloat shfl_i(dfloat v, int lane) { return {shfl_i(v.hi, lane), shfl_i(v.lo, lane)}; }

// Sums over the warp of NV <= 8 values per lane: lane l returns the total of value l / 4. The
// additions are those of a butterfly over all values (warp_allsum: the same pairs at every level,
// and an addition is commutative), but in each of the first three steps a lane keeps half of its
// values and hands over the other half, so there are 9 of them instead of 5 NV.
template <int NV>
__device__ __forceinline__ E warp_sums(const E (&x)[NV], int lane) {
  E v[8];
#pragma unroll
  for (int q = 0; q < 8; q++) v[q] = q < NV ? x[q] : cvt<E>(0.0);
  int o = 16;
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < h; q++) {
      const E send = up ? v[q] : v[q + h];
      const E keep = up ? v[q + h] : v[q];
      v[q] = keep + shfl_x(send, o);
    }
  }
  v[0] += shfl_x(v[0], 2);
  v[0] += shfl_x(v[0], 1);
  return v[0];
}

// Whether x < lim where FP32 leaves no doubt (x off by at most 1e-5 mag): 1 yes, 0 no, -1 open
// (also for NaN, infinities and the ends of the range).
__device__ __forceinline__ int clearly_less(float x, float mag, float lim) {
  if (!(lim > 1e-25f && lim < 1e25f)) return -1;
  if (!(fabsf(x - lim) > 1e-5f * (mag + lim))) return -1;
  return x < lim ? 1 : 0;
}
// Existence test of step 1 (eq. (26)), f0 > 0 and f0 f4 > f1^2 + f2^2 + f3^2, the same way.
__device__ __forceinline__ int clearly_exists(float f0, float f1, float f2, float f3, float f4) {
  const float pl = f0 * f4, mi = f1 * f1 + f2 * f2 + f3 * f3, mag = fabsf(pl) + mi;
  if (!(mag > 1e-25f && mag < 1e25f && fabsf(pl - mi) > 1e-5f * mag)) return -1;
  return f0 > 0.0f && pl > mi ? 1 : 0;
}

// ---------------------------------------------------------------------------------------
// Cluster-wide sum of NV values per thread; tot (double) and sm.red_tote (E) receive the
// totals, identical in every CTA.
// ---------------------------------------------------------------------------------------
template <int NV>
__device__ inline void cluster_reduce(E (&v)[NV], double (&tot)[NV], NodesSmem& sm, int& buf,
                                      cg::cluster_group& cl, int CS) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const E ws = warp_sums<NV>(v, lane);
  if ((lane & 3) == 0 && (lane >> 2) < NV) sm.red_warp[wid][lane >> 2] = ws;
  __syncthreads();
  if (threadIdx.x < NV) {
    E t = sm.red_warp[0][threadIdx.x];
    for (int k = 1; k < nw; k++) t += sm.red_warp[k][threadIdx.x];
    sm.red_part[buf][threadIdx.x] = widen(t);
  }
  cl.sync();
  // one thread per (value q, rank r): lanes of a warp hold segments of CS consecutive ranks
  if (CS == 1) {
    if (threadIdx.x < NV) sm.red_tot[threadIdx.x] = sm.red_part[buf][threadIdx.x];
  } else {
    const int per_warp = 32 / CS;  // values per warp
    const int nwarps = (NV + per_warp - 1) / per_warp;
    if (wid < nwarps) {
      int q = wid * per_warp + lane / CS, r = lane % CS;
      double x = 0.0;
      if (q < NV) x = cl.map_shared_rank(&sm.red_part[buf][0], r)[q];
      for (int o = CS >> 1; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (q < NV && r == 0) sm.red_tot[q] = x;
    }
  }
  __syncthreads();
  if (threadIdx.x < NV) sm.red_tote[threadIdx.x] = cvt<E>(sm.red_tot[threadIdx.x]);
#pragma unroll
  for (int q = 0; q < NV; q++) tot[q] = sm.red_tot[q];
  buf ^= 1;
  __syncthreads();
}

// ---------------------------------------------------------------------------------------
// Newton for the discrete Maxwellian, executed by the whole CTA with uniform control flow.
// ---------------------------------------------------------------------------------------
// Warps 0-2: factors and 1-D sums S_d^p of dimension d at the trial theta in sm.thE.
__device__ __noinline__ void eval_cta(NodesSmem& sm, int N) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid < 4) {
    // warps 0-2: dimension d; warp 3: dimension 1 again, weighted by |v1|/dx (step 1, eq. (24))
    const int d = wid == 3 ? 0 : wid;
    E e = cvt<E>(0.0);
    if (lane < N) {
      E x = sm.thE[1 + d] * sm.vv[lane] - sm.thE[4] * sm.vq[lane];
      if (d == 0) x += sm.thE[0];
      e = df_exp(x);
    }
    if (wid < 3) sm.ef[d][lane] = e;
    if (wid == 3) e = e * sm.c1e[lane];
    E s[5];
    s[0] = e;
    s[1] = e * sm.vv[lane];
    s[2] = e * sm.vq[lane];
    s[3] = s[2] * sm.vv[lane];
    s[4] = s[2] * sm.vq[lane];
    const E t = warp_sums<5>(s, lane);
    if ((lane & 3) == 0 && lane < 20) (wid < 3 ? sm.S[d] : sm.S1w)[lane >> 2] = t;
  }
  __syncthreads();
}

// Moments (E) and Jacobian (FP32) of the separable Maxwellian from its three 1-D sums.
__device__ inline void moments_from_sums(const E* S1, const E* S2, const E* S3, E (&mom)[5], float (&Aa)[15]) {
  E s23 = S2[0] * S3[0];
  mom[0] = S1[0] * s23;
  mom[1] = S1[1] * s23;
  mom[2] = S1[0] * (S2[1] * S3[0]);
  mom[3] = S1[0] * (S2[0] * S3[1]);
  mom[4] = S1[2] * s23 + S1[0] * (S2[2] * S3[0] + S2[0] * S3[2]);
  float f1[5], f2[5], f3[5];
#pragma unroll
  for (int p = 0; p < 5; p++) {
    f1[p] = tof(S1[p]);
    f2[p] = tof(S2[p]);
    f3[p] = tof(S3[p]);
  }
  float q11 = f1[2] * f2[0] * f3[0], q22 = f1[0] * f2[2] * f3[0], q33 = f1[0] * f2[0] * f3[2];
  float q12 = f1[1] * f2[1] * f3[0], q13 = f1[1] * f2[0] * f3[1], q23 = f1[0] * f2[1] * f3[1];
  float c1 = f1[3] * f2[0] * f3[0] + f1[1] * f2[2] * f3[0] + f1[1] * f2[0] * f3[2];
  float c2 = f1[2] * f2[1] * f3[0] + f1[0] * f2[3] * f3[0] + f1[0] * f2[1] * f3[2];
  float c3 = f1[2] * f2[0] * f3[1] + f1[0] * f2[2] * f3[1] + f1[0] * f2[0] * f3[3];
  float e4 = f1[4] * f2[0] * f3[0] + f1[0] * f2[4] * f3[0] + f1[0] * f2[0] * f3[4] +
             2.0f * (f1[2] * f2[2] * f3[0] + f1[2] * f2[0] * f3[2] + f1[0] * f2[2] * f3[2]);
  float t[15] = {f1[0] * f2[0] * f3[0], f1[1] * f2[0] * f3[0], f1[0] * f2[1] * f3[0], f1[0] * f2[0] * f3[1],
                 q11 + q22 + q33, q11, q12, q13, c1, q22, q23, c2, q33, c3, e4};
#pragma unroll
  for (int i = 0; i < 15; i++) Aa[i] = t[i];
}

// Component k of a five-element register array (static indices only).
template <typename T>
__device__ inline T pick5(const T (&v)[5], int k) {
  T r = v[0];
#pragma unroll
  for (int q = 1; q < 5; q++)
    if (k == q) r = v[q];
  return r;
}

// Lane k < 5 returns moment k, with the operations of moments_from_sums (lanes 5 and 6 form parts of
// the last one), so that a warp does a handful of double-float operations instead of forty.
__device__ __forceinline__ E lane_moment(const E* S1, const E* S2, const E* S3, int lane) {
  const int i = lane == 1 ? 1 : (lane == 4 ? 2 : 0), j = lane == 2 ? 1 : (lane == 5 ? 2 : 0),
            l = lane == 3 ? 1 : (lane == 6 ? 2 : 0);
  E u = S2[j] * S3[l];
  const E u6 = shfl_i(u, 6);
  if (lane == 5) u = u + u6;
  E x = S1[i] * u;
  const E x5 = shfl_i(x, 5);
  if (lane == 4) x = x + x5;
  return x;
}

// Residual of the moments against the target (lane k: component k of it, tl), in Ff on every
// lane, the Jacobian (FP32) and the scaled residual norm, from the 1-D sums. it0: |target_0|.
__device__ __forceinline__ void combine(const E* S1, const E* S2, const E* S3, E w, E tl, float it0, float (&Ff)[5],
                                        float (&A)[15], float& fn) {
  const float Fl = tof(w * lane_moment(S1, S2, S3, threadIdx.x & 31) - tl);
  float amax = 0.0f;
#pragma unroll
  for (int i = 0; i < 5; i++) {
    Ff[i] = shfl_i(Fl, i);
    amax = fmaxf(amax, fabsf(Ff[i]));
  }
  fn = amax / it0;
  E mom[5];
  float Aa[15];
  moments_from_sums(S1, S2, S3, mom, Aa);
  const float cf = tof(w);
#pragma unroll
  for (int i = 0; i < 15; i++) A[i] = cf * Aa[i];
}

// One evaluation by evaluating warp wid (warps 0-2: dimension wid, unweighted; warp 3:
// dimension 1 weighted by |v1|/dx) at the trial theta, of which lane k holds component k: factors
// of warps 0-2 to sm.ef, the five 1-D sums to row wid of sm.Sb[buf]. The same arithmetic as
// eval_cta.
__device__ __forceinline__ void eval_warp(NodesSmem& sm, int N, E thl, int wid, int buf) {
  const int lane = threadIdx.x & 31;
  const int d = wid == 3 ? 0 : wid;
  const E b = shfl_i(thl, 1 + d), g = shfl_i(thl, 4), al = shfl_i(thl, 0);
  E e = cvt<E>(0.0);
  if (lane < N) {
    E x = b * sm.vv[lane] - g * sm.vq[lane];
    if (d == 0) x += al;
    e = df_exp(x);
  }
  if (wid < 3) sm.ef[d][lane] = e;
  if (wid == 3) e = e * sm.c1e[lane];
  E s[5];
  s[0] = e;
  s[1] = e * sm.vv[lane];
  s[2] = e * sm.vq[lane];
  s[3] = s[2] * sm.vv[lane];
  s[4] = s[2] * sm.vq[lane];
  const E t = warp_sums<5>(s, lane);
  if ((lane & 3) == 0 && lane < 20) sm.Sb[buf][wid][lane >> 2] = t;
}

// Barrier among the evaluating warps only (hardware barrier 1; __syncthreads uses 0).
__device__ __forceinline__ void eval_bar(int nwarps) {
  asm volatile("bar.sync 1, %0;" ::"r"(nwarps * 32) : "memory");
}

// Newton from the theta in th (shared memory). With have_eval the last evaluation (sm.S,
// sm.S1w, sm.ef) is already at th and is reused. On success th holds the root, the
// last evaluation is at th, and the return value is the iteration count; -1 on failure.
// weighted: the step-1 weights |v1|/dx.
//
// Only the four evaluating warps take part, and each of them runs the whole iteration
// itself: it evaluates its dimension into a double-buffered row of sm.Sb, meets the others
// at one barrier, and then combines the rows, factorises the Jacobian (FP32: inexact Newton)
// and takes the line-search decisions in registers. All of them read the same rows and the
// same inputs through the same instructions, so their decisions agree and they pass every
// barrier the same number of times; one barrier per evaluation replaces the CTA barriers
// and thread-0 broadcasts of a split design. The FP64 theta is spread over the lanes (lane k:
// component k), the moments and sums too, so an iteration takes one FP64 instruction. With every
// component on lane 0 it took five of them and six conversions, about half of its 1.5 us.
__device__ __noinline__ int newton_cta(NodesSmem& sm, int N, E w, bool weighted, const E* target, double* th,
                                       double L, double tol, int maxit, bool have_eval) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int nev = 4;
  // Converged as well once the scaled moment residual |F|/rho is at the arithmetic's
  // resolution (double-float evaluates F to about 1e-14; 1e-13 bounds the relative
  // error of the Maxwellian near 1e-12 or below): with the residual already
  // there, a further step could only confirm it.
  constexpr float ftol = 1e-13f;
  if (wid < nev) {
    const int kl = min(lane, 4);  // this lane's component
    double thl = th[kl];
    const E tl = pick5(*reinterpret_cast<const E(*)[5]>(target), kl);
    const float it0 = fabsf(tof(target[0]));
    float Ff[5], A[15], fn = 0.0f;
    int buf = 0, last = -1;  // last: buffer of the latest evaluation (-1: the canonical sums)
    if (have_eval) {
      combine(weighted ? sm.S1w : sm.S[0], sm.S[1], sm.S[2], w, tl, it0, Ff, A, fn);
    } else {
      eval_warp(sm, N, cvt<E>(thl), wid, buf);
      eval_bar(nev);
      combine(sm.Sb[buf][weighted ? 3 : 0], sm.Sb[buf][1], sm.Sb[buf][2], w, tl, it0, Ff, A, fn);
      last = buf;
      buf ^= 1;
    }
    int ret = 0;
    if (!(fn <= ftol)) {
      ret = -1;
      float fn_cur = fn;
      for (int it = 0; it < maxit; it++) {
        float y[5];
        if (!chol5_solve(A, Ff, y)) break;
        // exponent change of a full step, |d alpha| + L sum |d beta| + L^2 |d gamma|
        const float Lf = (float)L;
        const float stepf = fabsf(y[0]) + Lf * (fabsf(y[1]) + fabsf(y[2]) + fabsf(y[3])) + Lf * Lf * fabsf(y[4]);
        // -D A^{-1} F, D = diag(1,1,1,1,-1)
        const float yl = pick5(y, kl);
        const double dirl = widen(kl == 4 ? yl : -yl);
        float lam = 1.0f;
        double lamd = 1.0, tt;
        for (int hv = 0; hv < 40; hv++) {
          tt = fma(lamd, dirl, thl);
          eval_warp(sm, N, cvt<E>(tt), wid, buf);
          eval_bar(nev);
          combine(sm.Sb[buf][weighted ? 3 : 0], sm.Sb[buf][1], sm.Sb[buf][2], w, tl, it0, Ff, A, fn);
          last = buf;
          buf ^= 1;
          if (fn == fn && (fn <= fn_cur || fn <= 1e-10f)) {
            fn_cur = fn;
            break;
          }
          lam *= 0.5f;
          lamd *= 0.5;
        }
        const float step = lam * stepf;
        thl = tt;
        if (!(step == step)) break;
        if (step <= (float)tol || fn_cur <= ftol) {
          ret = it + 1;
          break;
        }
      }
    }
    // publish the result: theta, and the latest evaluation's sums as the canonical ones (its
    // factors are in sm.ef already)
    if (wid == 0 && lane < 5) {
      th[lane] = thl;
      sm.thE[lane] = cvt<E>(thl);
    }
    if (last >= 0 && lane < 5) (wid < 3 ? sm.S[wid] : sm.S1w)[lane] = sm.Sb[last][wid][lane];
    if (wid == 0 && lane == 0) sm.nret = ret;
  }
  __syncthreads();
  return sm.nret;
}

__device__ inline void copy_factors(NodesSmem& sm, E (*dst)[kMaxN]) {
  if (threadIdx.x < 3 * kMaxN) {
    int d = threadIdx.x / kMaxN, i = threadIdx.x % kMaxN;
    dst[d][i] = sm.ef[d][i];
  }
  __syncthreads();
}

// M[g] of the moments in mom: warm start from th0 (have_eval: the last evaluation is at th0),
// then from the continuum Maxwellian; on failure keeps th0 (status reported).
// Result in sm.thg and sm.Eg; the last evaluation is at sm.thg afterwards.
__device__ __noinline__ int solve_mg(NodesSmem& sm, int N, E w, const E* mom, const double* th0, bool have_eval,
                                     double L, double tol, int maxit, unsigned& status) {
  const int tid = threadIdx.x;
  double keep[5];
#pragma unroll
  for (int k = 0; k < 5; k++) keep[k] = th0[k];
  __syncthreads();
  if (tid < 5) sm.thg[tid] = keep[tid];
  __syncthreads();
  int it = newton_cta(sm, N, w, false, mom, sm.thg, L, tol, maxit, have_eval);
  if (it < 0) {
    if (tid == 0) {
      double tg[5];
      bool ok = continuum_guess<E>(mom, tg);
      sm.ctl = ok;
      if (ok)
        for (int k = 0; k < 5; k++) sm.thg[k] = tg[k];
    }
    __syncthreads();
    if (sm.ctl) {
      it = newton_cta(sm, N, w, false, mom, sm.thg, L, tol, maxit, false);
    } else {
      status |= SGS_ST_NONPOSITIVE;
    }
  }
  if (it < 0) {
    status |= SGS_ST_NEWTON_FAIL;
    if (tid < 5) sm.thg[tid] = keep[tid];
    __syncthreads();
    if (tid < 5) sm.thE[tid] = cvt<E>(sm.thg[tid]);
    __syncthreads();
    eval_cta(sm, N);
  }
  copy_factors(sm, sm.Eg);
  return it;
}

// Relaxed step 1 (the remark after eq. (26)), for thread 0 when eq. (26) fails for the
// target sd: with a factor 1 + tau on the weighted moments of the new and the current
// Maxwellian the target becomes (tau m_w + s)/(1 + tau), m_w = sum w phi c M[g] (c the
// step-1 weight; its moments come from the separable sums of the last evaluation, which is
// M[g]'s). 1 + tau = 2, 4, 8, ...: the first target that passes eq. (26) replaces sd and
// sm.svE. Returns whether one was found.
__device__ inline bool relax_target(NodesSmem& sm, E w, double (&sd)[5]) {
  E m1[5];
  float Aa[15];
  moments_from_sums(sm.S1w, sm.S[1], sm.S[2], m1, Aa);
  double mw[5];
#pragma unroll
  for (int k = 0; k < 5; k++) mw[k] = tod(w * m1[k]);
  for (double q = 2.0; q <= 1048576.0; q *= 2.0) {
    double t[5];
#pragma unroll
    for (int k = 0; k < 5; k++) t[k] = ((q - 1.0) * mw[k] + sd[k]) / q;
    if (t[0] > 0.0 && t[0] * t[4] > t[1] * t[1] + t[2] * t[2] + t[3] * t[3]) {
#pragma unroll
      for (int k = 0; k < 5; k++) {
        sd[k] = t[k];
        sm.svE[k] = cvt<E>(t[k]);
      }
      return true;
    }
  }
  return false;
}

// After a step-2 update the cell equation holds up to the Maxwellians:
//   (|v1|/dx + A) g + r = A M+   =>   R(g) = A (M+ - M[g]),   A = nu/eps,
// where M+ is the Maxwellian step 2 used (step 1's, else M[g_old]). The norm of R then comes
// from per-dimension sums of the two factorisations P (M+, sm.Ep) and Q (M[g], sm.Eg): with
// d = Q - P per dimension, Q1Q2Q3 - P1P2P3 = d1 P2 P3 + Q1 d2 P3 + Q1 Q2 d3, whose squared
// norm is a sum of products of 1-D sums (no cancellation of large terms). Likewise the
// step-1 target s = sum w phi (c (M[g] - g) - r) (eq. (26)) with c g + r = A M+ - A g is
//   s = sum w phi c M[g] - A sum w phi M+ + A sum w phi g,
// from the separable sums of the last evaluation (M[g]'s), the moments of M+ and those of
// g. No pass over the nodes and no cluster reduction. Warps 0-2 form the sums; the caller's
// thread 0 takes the decisions. Returns the squared norm sum_k (M+ - M[g])^2 in thread 0.
__device__ inline void derived_sums(NodesSmem& sm) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid < 3) {
    const E p = sm.Ep[wid][lane], q = sm.Eg[wid][lane], dl = q - p;
    E x[6] = {p * p, p * dl, dl * dl, p * q, dl * q, q * q};
    const E t = warp_sums<6>(x, lane);
    if ((lane & 3) == 0 && lane < 24) sm.Gs[wid][lane >> 2] = t;
  }
  __syncthreads();
}

__device__ inline E derived_norm2(const NodesSmem& sm) {
  // columns of Gs: 0 PP, 1 Pd, 2 dd, 3 PQ, 4 dQ, 5 QQ
  const E* a = sm.Gs[0];
  const E* b = sm.Gs[1];
  const E* c = sm.Gs[2];
  E cross = a[4] * b[1] * c[0] + a[4] * b[3] * c[1] + a[5] * b[4] * c[1];
  return a[2] * b[0] * c[0] + a[5] * b[2] * c[0] + a[5] * b[5] * c[2] + cvt<E>(2.0) * cross;
}

// The same in FP32, mag the sum of its terms' magnitudes (clearly_less).
__device__ __forceinline__ float derived_norm2_f32(const NodesSmem& sm, float& mag) {
  float a[6], b[6], c[6];
#pragma unroll
  for (int k = 0; k < 6; k++) a[k] = tof(sm.Gs[0][k]), b[k] = tof(sm.Gs[1][k]), c[k] = tof(sm.Gs[2][k]);
  const float x0 = a[4] * b[1] * c[0], x1 = a[4] * b[3] * c[1], x2 = a[5] * b[4] * c[1];
  const float p = a[2] * b[0] * c[0] + a[5] * b[2] * c[0] + a[5] * b[5] * c[2];
  mag = p + 2.0f * (fabsf(x0) + fabsf(x1) + fabsf(x2));
  return p + 2.0f * (x0 + x1 + x2);
}

template <int EPT>
__global__ void __launch_bounds__(256) k_sweep_nodes(SweepArgs a) {
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int q = blockIdx.x / CS;
  if (q >= a.n_inst) return;  // whole cluster, uniformly
  if (a.active && !a.active[q]) return;
  const InstDev& I = a.inst[q];
  __shared__ NodesSmem sm;
  const int N = a.N, K = N * N * N;
  const double dv = a.dv, wd = a.dv * a.dv * a.dv;
  const E w = cvt<E>(wd);
  const int J = I.J;
  const double inv_dx = 1.0 / I.dx;
  const double L = node(N - 1, N, dv);
  const int tid = threadIdx.x;
  const bool pfp = I.inner_method == SGS_PFP || I.inner_method == SGS_PFP_RELAX;
  const bool relax = I.inner_method == SGS_PFP_RELAX;
  const double ntol = I.newton_tol;
  // inner_tol^2 / w; a tolerance that is not positive leaves every decision to FP64
  const float tol2f = I.inner_tol > 0.0 ? (float)I.tol2_w : -1.0f;
  const E inv_eps = cvt<E>(1.0 / I.eps);
  const E zero = cvt<E>(0.0);
  if (tid < kMaxN) {
    double v = tid < N ? node(tid, N, dv) : 0.0;
    sm.vv[tid] = cvt<E>(v);
    sm.vq[tid] = cvt<E>(v * v);
    sm.c1e[tid] = cvt<E>(fabs(v) * inv_dx);
    sm.W3[0][tid] = cvt<E>(tid < N ? I.wall[0][2][tid] : 0.0);
    sm.W3[1][tid] = cvt<E>(tid < N ? I.wall[1][2][tid] : 0.0);
  }
  __syncthreads();

  // this thread's nodes: pencil (i1, i2), i3 in [i30, i30 + EPT)
  const int tg = rank * blockDim.x + tid;
  const int e0 = tg * EPT;
  const bool own = e0 < K;
  const int pen = own ? e0 / N : 0, i30 = own ? e0 % N : 0;
  const int i1 = pen / N, i2 = pen % N;
  const double v1d = node(i1, N, dv);
  const E v1 = sm.vv[i1], v2 = sm.vv[i2];
  const E c1 = sm.c1e[i1];
  const E vpd = cvt<E>(fmax(v1d, 0.0) * inv_dx), vmd = cvt<E>(fmin(v1d, 0.0) * inv_dx);
  const E vq12 = sm.vq[i1] + sm.vq[i2];
  const E wl12 = cvt<E>(I.wall[0][0][i1] * I.wall[0][1][i2]);
  const E wr12 = cvt<E>(I.wall[1][0][i1] * I.wall[1][1][i2]);

  E g[EPT], r[EPT];
  int buf = 0;
  unsigned long long c_inner = 0, c_newton = 0, c_solves = 0, c_fallback = 0;
  unsigned int status = 0;

  const int s_end = min(a.s1, J);
  for (int s = a.s0; s < s_end; s++) {
    const int j = a.dir > 0 ? s : J - 1 - s;
    const long long cbase = I.f_off + (long long)j * K + e0;
    double* fj = a.f + cbase;
    const bool lw = j == 0, rw = j == J - 1;

    // ---- r = (-v1^+ f_{j-1} + v1^- f_{j+1}) / dx - P_j / eps - b_j (neighbours: latest values);
    //      a wall cell needs the wall density from reduction 1, every other cell forms r
    //      before it, so that its loads and conversions overlap the reduction
    auto form_r = [&](E rho_l, E rho_r) {
      const double* Pj = a.P + cbase;
      const double* bj = a.rhs ? a.rhs + cbase : nullptr;
#pragma unroll
      for (int t = 0; t < EPT; t++) {
        E left = lw ? rho_l * wl12 * sm.W3[0][i30 + t] : cvt<E>(fj[t - K]);
        E right = rw ? rho_r * wr12 * sm.W3[1][i30 + t] : cvt<E>(fj[t + K]);
        E rv = vmd * right - vpd * left - cvt<E>(Pj[t]) * inv_eps;
        if (bj) rv -= cvt<E>(bj[t]);
        r[t] = rv;
      }
    };
    const bool wall_cell = lw || rw;
    if (own && !wall_cell) form_r(zero, zero);
    // the cell's transport-plus-penalty coefficients (from its collision frequency), also
    // ahead of the reduction (read after its barriers)
    if (tid < N) {
      const double Ad = a.nu[I.cell0 + j] / I.eps;
      double c = fabs(node(tid, N, dv)) * inv_dx + Ad;
      sm.c1A[tid] = cvt<E>(c);
      sm.den[tid] = cvt<E>(1.0 / c);
      if (tid == 0) sm.scal[2] = cvt<E>(Ad);
    }

    // ---- reduction 1: moments of the stored value and the walls' outgoing fluxes
    E a0 = zero, a3 = zero, a4 = zero;
    if (own) {
#pragma unroll
      for (int t = 0; t < EPT; t++) {
        E x = cvt<E>(fj[t]);
        g[t] = x;
        a0 += x;
        a3 += x * sm.vv[i30 + t];
        a4 += x * sm.vq[i30 + t];
      }
    }
    E m7[7] = {a0, v1 * a0, v2 * a0, a3, vq12 * a0 + a4, (lw && v1d < 0.0) ? v1 * a0 : zero,
               (rw && v1d > 0.0) ? v1 * a0 : zero};
    double t7[7];
    cluster_reduce<7>(m7, t7, sm, buf, cl, CS);
    E mom[5];
#pragma unroll
    for (int k = 0; k < 5; k++) mom[k] = w * sm.red_tote[k];
    if (tid == 0 && lw)
      sm.scal[0] = cvt<E>(I.bc_kind[0] == SGS_INFLOW ? I.bc_rho[0] : -(wd * t7[5]) / I.wall_denom[0]);
    if (tid == 0 && rw)
      sm.scal[1] = cvt<E>(I.bc_kind[1] == SGS_INFLOW ? I.bc_rho[1] : -(wd * t7[6]) / I.wall_denom[1]);
    __syncthreads();
    const E rho_l = lw ? sm.scal[0] : zero, rho_r = rw ? sm.scal[1] : zero, Acoef = sm.scal[2];
    const float limf = tol2f / (tof(Acoef) * tof(Acoef));  // bound of sum (M+ - M[g])^2
    const E c1A = sm.c1A[i1], den = sm.den[i1];
    if (own && wall_cell) form_r(rho_l, rho_r);

    // ---- M[g] of the stored value, from the collision step's Maxwellian of the same f (the
    //      collision step that preceded this scan, or this group's, evaluated the stored
    //      value: the Newton solve only confirms it); a stale start costs iterations, not
    //      accuracy (the root is unique)
    {
      double th0[5];
#pragma unroll
      for (int k = 0; k < 5; k++) th0[k] = a.theta[5 * (long long)(I.cell0 + j) + k];
      int n0 = solve_mg(sm, N, w, mom, th0, false, L, ntol, I.newton_max, status);
      if (n0 > 0) c_newton += n0;
      c_solves++;
    }

    int it = 0;
    // decisions from the step-2 identity (double-float and FP64 scans) after the first update
    bool derived = false;
    E momg[5];  // moments of the current iterate g
#pragma unroll
    for (int k = 0; k < 5; k++) momg[k] = mom[k];
    // whether the inner iteration stops: small 1 / 0, or 2 for a NaN residual (thread 0)
    auto decide = [&](int small) {
      bool stop;
      if (I.inner_fixed > 0) {
        stop = it >= I.inner_fixed;
      } else {
        stop = small == 1 || it >= I.inner_max;
        if (stop && small != 1) status |= SGS_ST_INNER_CAP;
      }
      if (small == 2) {
        status |= SGS_ST_NONFINITE;
        stop = true;
      }
      return stop;
    };
    for (;;) {
      if (!derived) {
        // ---- pass B: cell-equation residual and the step-1 target s (eq. (26))
        E e12 = sm.Eg[0][i1] * sm.Eg[1][i2];
        E rs = zero, b0 = zero, b3 = zero, b4 = zero;
        if (own) {
#pragma unroll
          for (int t = 0; t < EPT; t++) {
            E M = e12 * sm.Eg[2][i30 + t];
            // (|v1|/dx) g + r - (nu/eps)(M - g) = (|v1|/dx + nu/eps) g + r - (nu/eps) M
            E res = c1A * g[t] + r[t] - Acoef * M;
            rs += res * res;
            E tt = c1 * (M - g[t]) - r[t];
            b0 += tt;
            b3 += tt * sm.vv[i30 + t];
            b4 += tt * sm.vq[i30 + t];
          }
        }
        E v6[6] = {rs, b0, v1 * b0, v2 * b0, b3, vq12 * b0 + b4};
        double t6[6];
        cluster_reduce<6>(v6, t6, sm, buf, cl, CS);
        // thread 0 decides: stop, and whether step 1 is attempted (existence test, eq. (26))
        if (tid == 0) {
          const float rf = tof(sm.red_tote[0]);
          int sml = clearly_less(rf, rf, tol2f);
          float f[5];
#pragma unroll
          for (int k = 0; k < 5; k++) {
            const E sk = w * sm.red_tote[1 + k];
            sm.svE[k] = sk;
            f[k] = tof(sk);
          }
          int ex = pfp ? clearly_exists(f[0], f[1], f[2], f[3], f[4]) : 0;
          if (sml < 0 || ex < 0 || (pfp && relax && ex == 0)) {  // in FP64
            const double res = sqrt(wd * t6[0]);
            sml = res < I.inner_tol;
            if (!(res == res)) sml = 2;
            double sd[5] = {wd * t6[1], wd * t6[2], wd * t6[3], wd * t6[4], wd * t6[5]};
            bool exists = pfp && sd[0] > 0.0 && sd[0] * sd[4] > sd[1] * sd[1] + sd[2] * sd[2] + sd[3] * sd[3];
            if (pfp && !exists && relax) exists = relax_target(sm, w, sd);
            ex = exists;
          }
          sm.ctl = (decide(sml) ? 1 : 0) | (ex ? 2 : 0);
        }
        __syncthreads();
      }
      const int ctl = sm.ctl;
      if (ctl & 1) break;

      // ---- step 1 (eq. (24)) from M[g]; else the plain fixed-point step (eq. (22))
      bool used = false;
      if (pfp) {
        if (ctl & 2) {
          E sv[5];
#pragma unroll
          for (int k = 0; k < 5; k++) sv[k] = sm.svE[k];
          if (tid < 5) sm.thp[tid] = sm.thg[tid];
          __syncthreads();
          // the last evaluation is M[g]'s: reused as the first one of step 1
          int n1 = newton_cta(sm, N, w, true, sv, sm.thp, L, ntol, I.newton_max, true);
          c_solves++;
          if (n1 >= 0) {
            c_newton += n1;
            used = true;
            copy_factors(sm, sm.Ep);
          }
        }
        if (!used) c_fallback++;
      }
      const bool eval_at_start = used || !(ctl & 2);  // last evaluation at the warm start below
      E (*Eu)[kMaxN] = used ? sm.Ep : sm.Eg;
      // moments of M+: step 1's last evaluation is at M+; M[g] has the moments of g
      E momP[5];
      if (used) {
        float Aa[15];
        moments_from_sums(sm.S[0], sm.S[1], sm.S[2], momP, Aa);
#pragma unroll
        for (int k = 0; k < 5; k++) momP[k] = w * momP[k];
      } else {
#pragma unroll
        for (int k = 0; k < 5; k++) momP[k] = momg[k];
      }

      // ---- step 2 (eq. (25)) and the moments of the new iterate
      E ep = Eu[0][i1] * Eu[1][i2];
      E c0 = zero, c3 = zero, c4 = zero;
      if (own) {
#pragma unroll
        for (int t = 0; t < EPT; t++) {
          E x = (Acoef * (ep * Eu[2][i30 + t]) - r[t]) * den;
          g[t] = x;
          c0 += x;
          c3 += x * sm.vv[i30 + t];
          c4 += x * sm.vq[i30 + t];
        }
      }
      // keep the factors of M+ in sm.Ep (the reduction below orders this before solve_mg)
      if (!used && tid < 3 * kMaxN) sm.Ep[tid / kMaxN][tid % kMaxN] = sm.Eg[tid / kMaxN][tid % kMaxN];
      E m5[5] = {c0, v1 * c0, v2 * c0, c3, vq12 * c0 + c4};
      double t5[5];
      cluster_reduce<5>(m5, t5, sm, buf, cl, CS);
      it++;
      E mm[5];
#pragma unroll
      for (int k = 0; k < 5; k++) mm[k] = w * sm.red_tote[k];
      // warm start: the step-1 Maxwellian approximates M of the updated iterate
      int n2 = solve_mg(sm, N, w, mm, used ? sm.thp : sm.thg, eval_at_start, L, ntol, I.newton_max, status);
      if (n2 > 0) c_newton += n2;
      c_solves++;
      // ---- residual and step-1 target of the new iterate from the step-2 identity
      derived_sums(sm);
      // warp 0 decides; its lanes form the five components of the step-1 target
      if (tid < 32) {
        const int lane = tid;
        const E mwk = lane_moment(sm.S1w, sm.S[1], sm.S[2], lane);  // sum phi (|v1|/dx) M[g]
        const E sk = w * mwk - Acoef * pick5(momP, lane) + Acoef * pick5(mm, lane);
        if (lane < 5) sm.svE[lane] = sk;
        float mag;
        const float nf = derived_norm2_f32(sm, mag);
        int sml = clearly_less(nf, mag, limf);
        float f[5];
#pragma unroll
        for (int k = 0; k < 5; k++) f[k] = shfl_i(tof(sk), k);
        int ex = pfp ? clearly_exists(f[0], f[1], f[2], f[3], f[4]) : 0;
        if (sml < 0 || ex < 0 || (pfp && relax && ex == 0)) {  // in FP64, from the full sums
          const double sdk = tod(sk);
          double nrm = lane == 5 ? tod(derived_norm2(sm)) : 0.0;
          double sd[5];
#pragma unroll
          for (int k = 0; k < 5; k++) sd[k] = __shfl_sync(0xffffffffu, sdk, k);
          nrm = __shfl_sync(0xffffffffu, nrm, 5);
          __syncwarp();  // the lanes' sm.svE before lane 0 may replace them (relaxed step 1)
          if (lane == 0) {
            const double res = fabs(tod(Acoef)) * sqrt(wd * nrm);
            sml = res < I.inner_tol;
            if (!(res == res)) sml = 2;
            bool exists = pfp && sd[0] > 0.0 && sd[0] * sd[4] > sd[1] * sd[1] + sd[2] * sd[2] + sd[3] * sd[3];
            if (pfp && !exists && relax) exists = relax_target(sm, w, sd);
            ex = exists;
          }
        }
        if (lane == 0) sm.ctl = (decide(sml) ? 1 : 0) | (ex ? 2 : 0);
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 5; k++) momg[k] = mm[k];
      derived = true;
    }

    if (own) {
#pragma unroll
      for (int t = 0; t < EPT; t++) fj[t] = widen(g[t]);
    }
    c_inner += it;
    // the next visit's first reduction is a cluster barrier: every CTA has finished this
    // cell before any reads of the next one's neighbours (each thread reads only its own
    // nodes, so no cross-thread ordering is needed beyond program order)
  }
  // no CTA leaves while another may still read its shared memory (the last reduction's
  // distributed-shared-memory loads)
  cl.sync();

  if (rank == 0 && tid == 0) {
    Counters* c = a.cnt + q;
    atomicAdd(&c->visits, (unsigned long long)max(0, s_end - a.s0));
    atomicAdd(&c->inner_iters, c_inner);
    atomicAdd(&c->newton_iters, c_newton);
    atomicAdd(&c->newton_solves, c_solves);
    atomicAdd(&c->fallbacks, c_fallback);
  }
  if (tid == 0 && status) atomicOr(&a.cnt[q].status, status);
}

// The kernel of a shape (null: not compiled) and its launch configuration.
const void* nodes_kernel(int ept) {
  switch (ept) {
    case 2: return (const void*)k_sweep_nodes<2>;
    case 4: return (const void*)k_sweep_nodes<4>;
    case 8: return (const void*)k_sweep_nodes<8>;
    case 12: return (const void*)k_sweep_nodes<12>;
    case 16: return (const void*)k_sweep_nodes<16>;
    case 20: return (const void*)k_sweep_nodes<20>;
    case 24: return (const void*)k_sweep_nodes<24>;
    case 28: return (const void*)k_sweep_nodes<28>;
    case 32: return (const void*)k_sweep_nodes<32>;
  }
  return nullptr;
}

struct NodesLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  NodesLaunch(const SweepShape& sh, int n_inst, cudaStream_t st) {
    cfg.gridDim = dim3(n_inst * sh.cluster);
    cfg.blockDim = dim3(sh.tpb);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = sh.cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

}  // namespace

cudaError_t launch_sweep_nodes(const SweepArgs& a, const SweepShape& sh, cudaStream_t st) {
  const void* fn = nodes_kernel(sh.ept);
  if (!fn || !sweep_shape_valid(a.N, sh)) return cudaErrorInvalidConfiguration;
  cudaError_t e = func_attr(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  NodesLaunch l(sh, a.n_inst, st);
  SweepArgs args = a;
  void* p[] = {&args};
  return cudaLaunchKernelExC(&l.cfg, fn, p);
}

cudaError_t sweep_nodes_max_clusters(const SweepShape& sh, int* n) {
  *n = 0;
  const void* fn = nodes_kernel(sh.ept);
  if (!fn) return cudaErrorInvalidConfiguration;
  cudaError_t e = func_attr(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  NodesLaunch l(sh, 1, nullptr);
  return cudaOccupancyMaxActiveClusters(n, fn, &l.cfg);
}

}  // namespace sgs
