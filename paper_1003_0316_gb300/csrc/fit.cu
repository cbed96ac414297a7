// a7: analytic continuation of Sigma^c(i w) by the multipole model of Eq. modelf,
// f(z) = sum_p a_p / (z - w_p), fitted in FP64 by Levenberg-Marquardt
// (Marquardt 1963, diagonal scaling), one warp per curve, or eight curves per warp where there
// are thousands.
//
// Cost C = 1/2 sum_j |f(i w_j) - y_j|^2 over the parameters
// theta = (Re a_p, Im a_p, Re w_p, Im w_p)_p. Each iteration accumulates
// A = J^T J and g = J^T r row by row from the analytic derivatives
// df/da_p = 1/(z - w_p), df/dw_p = a_p/(z - w_p)^2 (f is holomorphic in each
// parameter, so d/dRe = D and d/dIm = i D), solves (A + mu diag A) d = -g by
// Cholesky, and accepts the step when the cost drops (mu /= 10, floor 1e-15),
// otherwise mu *= 10 (give up above 1e15). Stops after an accepted step whose
// relative cost decrease is <= 1e-14, when C <= 1e-28 * (1/2 sum |y|^2), or after
// 200 iterations. Default start: w_p = s (0.5, 2, 5, 10, 20)_p - 0.1 i s (s the sign
// of the state energy) with residues from the linear least-squares problem.
#include <algorithm>

#include "gw_internal.cuh"
#include "fit_common.cuh"

namespace gw {

// One warp per curve: lanes take frequency points (j = lane, lane + 32) for the residual,
// the Jacobian rows and the cost; the normal matrix A = J^T J and g = J^T r are summed over
// points by lanes owning (a, b) entries; the damped system is factored column by column
// (lanes take the rows below the pivot) and solved by column sweeps. FP64 throughout; the
// iteration, damping and stopping rules are the ones stated at the top of this file.
constexpr int LM_WMAXNW = 64;
constexpr int LM_NPACK = LM_MAXP * (LM_MAXP + 1) / 2;

struct LmWarpSmem {
  double rowR[LM_WMAXNW][LM_MAXP];
  double rowI[LM_WMAXNW][LM_MAXP];
  double res[LM_WMAXNW][2];
  double A[LM_NPACK];
  double Ld[LM_NPACK];
  double g[LM_MAXP];
  double b[LM_MAXP];
  double dinv[LM_MAXP];     // reciprocals of the factor's diagonal
  double th[LM_MAXP];
  int flag;
};

// a b + c d and a b - c d with their roundings written out: both kernels use them, since a compiler may
// contract either product, and their results are equal bit for bit. (A single product added to a
// value can be contracted in one way only.)
__device__ __forceinline__ double lm_sum(double a, double b, double c, double d) {
  return fma(a, b, __dmul_rn(c, d));
}
__device__ __forceinline__ double lm_dif(double a, double b, double c, double d) {
  return fma(a, b, -__dmul_rn(c, d));
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// 1/2 sum_j |f(i w_j) - y_j|^2 for parameters t (all lanes hold t), warp-summed.
__device__ __forceinline__ double warp_cost(const double* om, const double2* yl, int nw, int npole,
                                            const double* t) {
  const int lane = threadIdx.x & 31;
  double c = 0.0;
  for (int h = 0; h < 2; ++h) {
    const int j = lane + 32 * h;
    if (j >= nw) break;
    double fx = 0.0, fy = 0.0;
    for (int p = 0; p < npole; ++p) {
      const double dx = -t[4 * p + 2], dy = om[j] - t[4 * p + 3];
      const double inv = 1.0 / lm_sum(dy, dy, dx, dx);
      const double px = dx * inv, py = -dy * inv;          // phi = 1 / (i w_j - w_p)
      fx += lm_dif(t[4 * p], px, t[4 * p + 1], py);
      fy += lm_sum(t[4 * p], py, t[4 * p + 1], px);
    }
    const double rx = fx - yl[h].x, ry = fy - yl[h].y;
    c += lm_sum(rx, rx, ry, ry);
  }
  return 0.5 * warp_sum(c);
}

// NPOLE: poles of the model (a template parameter, so that the parameter vectors and the
// loops over them stay in registers)
template <int NPOLE>
__global__ void __launch_bounds__(32) k_lm_warp(int ncurve, int nw, OmegaArr om,
                                                const double2* __restrict__ sigma,
                                                const double* __restrict__ sign,
                                                const double* __restrict__ theta_init,
                                                double* __restrict__ params,
                                                double* __restrict__ cost_out,
                                                int* __restrict__ iters_out,
                                                int* __restrict__ status_out, int keep_better) {
  __shared__ LmWarpSmem S;
  const int cidx = blockIdx.x;
  const int lane = threadIdx.x;
  if (cidx >= ncurve) return;
  const double2* y = sigma + size_t(cidx) * nw;
  constexpr int npole = NPOLE;
  constexpr int P = 4 * npole;
  constexpr int NP = P * (P + 1) / 2;
  double2 yl[2];
  for (int h = 0; h < 2; ++h) {
    const int j = lane + 32 * h;
    yl[h] = j < nw ? y[j] : make_double2(0.0, 0.0);
  }
  if (lane == 0) {
    if (theta_init) {
      for (int k = 0; k < P; ++k) S.th[k] = theta_init[size_t(cidx) * P + k];
    } else {
      const double s = sign ? (sign[cidx] >= 0.0 ? 1.0 : -1.0) : 1.0;
      lm_default_start(om.v, y, nw, npole, s, S.th);
    }
  }
  __syncwarp();
  double th[P], thn[P];
  for (int k = 0; k < P; ++k) th[k] = S.th[k];
  const double cscale = 0.5 * warp_sum(fma(yl[1].y, yl[1].y,
                                           fma(yl[1].x, yl[1].x, lm_sum(yl[0].x, yl[0].x, yl[0].y, yl[0].y))));
  double C = warp_cost(om.v, yl, nw, npole, th);
  // the packed entries e = lane + 32 h of A this lane sums: row ea[h], column eb[h]
  constexpr int EPL = (NP + 31) / 32;
  int ea[EPL], eb[EPL];
#pragma unroll
  for (int h = 0; h < EPL; ++h) {
    const int e = lane + 32 * h;
    int a = 0;
    while ((a + 1) * (a + 2) / 2 <= e) ++a;
    ea[h] = a;
    eb[h] = e - a * (a + 1) / 2;
  }
  double mu = -1.0;
  int it = 0, st = 1;
  for (; it < LM_MAXIT; ++it) {
    if (C <= LM_CTOL * cscale) {
      st = 0;
      break;
    }
    // Jacobian rows and residuals of this lane's points
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      if (j >= nw) break;
      double fx = 0.0, fy = 0.0;
      for (int p = 0; p < npole; ++p) {
        const double ax = th[4 * p], ay = th[4 * p + 1];
        const double dx = -th[4 * p + 2], dy = om.v[j] - th[4 * p + 3];
        const double inv = 1.0 / lm_sum(dy, dy, dx, dx);
        const double px = dx * inv, py = -dy * inv;        // phi
        const double tx = lm_dif(ax, px, ay, py), ty = lm_sum(ax, py, ay, px);   // a phi
        fx += tx;
        fy += ty;
        const double qx = lm_dif(tx, px, ty, py), qy = lm_sum(tx, py, ty, px);   // a phi^2
        // d f / d Re a = phi, d f / d Im a = i phi, d f / d Re w = a phi^2, d f / d Im w = i a phi^2
        S.rowR[j][4 * p] = px;
        S.rowI[j][4 * p] = py;
        S.rowR[j][4 * p + 1] = -py;
        S.rowI[j][4 * p + 1] = px;
        S.rowR[j][4 * p + 2] = qx;
        S.rowI[j][4 * p + 2] = qy;
        S.rowR[j][4 * p + 3] = -qy;
        S.rowI[j][4 * p + 3] = qx;
      }
      S.res[j][0] = fx - yl[h].x;
      S.res[j][1] = fy - yl[h].y;
    }
    __syncwarp();
    // A (packed lower) and g, summed over points
#pragma unroll
    for (int h = 0; h < EPL; ++h) {
      const int e = lane + 32 * h;
      if (e >= NP) break;
      const int a = ea[h], bcol = eb[h];
      double v = 0.0;
      for (int j = 0; j < nw; ++j) v += lm_sum(S.rowR[j][a], S.rowR[j][bcol], S.rowI[j][a], S.rowI[j][bcol]);
      S.A[e] = v;
    }
    if (lane < P) {
      double v = 0.0;
      for (int j = 0; j < nw; ++j) v += lm_sum(S.rowR[j][lane], S.res[j][0], S.rowI[j][lane], S.res[j][1]);
      S.g[lane] = v;
    }
    __syncwarp();
    double gm = 0.0, dm = 0.0;
    if (lane < P) {
      gm = fabs(S.g[lane]);
      dm = S.A[lane * (lane + 1) / 2 + lane];
    }
    gm = warp_max(gm);
    dm = warp_max(dm);
    if (gm <= LM_GTOL) {
      st = 0;
      break;
    }
    if (mu < 0.0) mu = 1e-3 * dm;
    double Cn = 0.0;
    bool give_up = false;
    while (true) {
      for (int e = lane; e < NP; e += 32) S.Ld[e] = S.A[e];
      __syncwarp();
      if (lane < P) {
        S.Ld[lane * (lane + 1) / 2 + lane] += mu * S.A[lane * (lane + 1) / 2 + lane];
        S.b[lane] = -S.g[lane];
      }
      if (lane == 0) S.flag = 1;
      __syncwarp();
      // Cholesky, column by column: the pivot by lane 0, the rows below it by lanes
      for (int jc = 0; jc < P; ++jc) {
        if (lane == 0) {
          double d = S.Ld[jc * (jc + 1) / 2 + jc];
          for (int k = 0; k < jc; ++k) d -= S.Ld[jc * (jc + 1) / 2 + k] * S.Ld[jc * (jc + 1) / 2 + k];
          if (!(d > 0.0)) S.flag = 0;
          const double r = d > 0.0 ? sqrt(d) : 1.0;
          S.Ld[jc * (jc + 1) / 2 + jc] = r;
          S.dinv[jc] = 1.0 / r;
        }
        __syncwarp();
        const int i = jc + 1 + lane;
        if (i < P) {
          double v = S.Ld[i * (i + 1) / 2 + jc];
          for (int k = 0; k < jc; ++k) v -= S.Ld[i * (i + 1) / 2 + k] * S.Ld[jc * (jc + 1) / 2 + k];
          S.Ld[i * (i + 1) / 2 + jc] = v * S.dinv[jc];
        }
        __syncwarp();
      }
      const bool ok = S.flag != 0;
      if (ok) {
        // L z = b by column sweeps, then L^T x = z
        for (int k = 0; k < P; ++k) {
          const double zk = S.b[k] * S.dinv[k];
          __syncwarp();
          const int i = k + 1 + lane;
          if (i < P) S.b[i] -= S.Ld[i * (i + 1) / 2 + k] * zk;
          if (lane == 0) S.b[k] = zk;
          __syncwarp();
        }
        for (int k = P - 1; k >= 0; --k) {
          const double xk = S.b[k] * S.dinv[k];
          __syncwarp();
          if (lane < k) S.b[lane] -= S.Ld[k * (k + 1) / 2 + lane] * xk;
          if (lane == 0) S.b[k] = xk;
          __syncwarp();
        }
        for (int k = 0; k < P; ++k) thn[k] = th[k] + S.b[k];
        Cn = warp_cost(om.v, yl, nw, npole, thn);
      }
      if (ok && Cn < C) {
        mu = fmax(mu / 10.0, LM_MU_MIN);
        break;
      }
      mu *= 10.0;
      if (mu > LM_MU_MAX) {
        give_up = true;
        break;
      }
    }
    if (give_up) {
      st = 2;
      break;
    }
    const double dec = C - Cn, Cold = C;
    for (int k = 0; k < P; ++k) th[k] = thn[k];
    C = Cn;
    if (dec <= LM_FTOL * Cold) {
      st = 0;
      ++it;
      break;
    }
  }
  if (lane != 0) return;
  if (keep_better) {
    // compare with the result already stored (the other start) and keep the lower cost
    if (!(C < cost_out[cidx])) return;
  }
  for (int k = 0; k < P; ++k) params[size_t(cidx) * P + k] = th[k];
  cost_out[cidx] = C;
  iters_out[cidx] = it;
  status_out[cidx] = st;
}

// ---- many curves: four lanes per curve, eight curves per warp -------------------------------------
// GB300's FP64 pipe takes as long for an instruction with one active lane as for a full one (16
// cycles per warp instruction and SM), and the warp-per-curve kernel issues most of its FP64
// instructions with few (the pivots with one, the sweeps with at most P = 4 N_p, the points with nw
// of 32). Here eight curves share a warp's instructions, with the same operations in the same
// order (sums over points as the warp's butterfly forms them, everything else through shared
// memory as there), so the results are bit-identical. A block draws its curves from a contiguous
// range through a counter, the lanes of a curve taking the next one when their fit ends; each trip
// of the loop is damped solve, cost, accept or reject for the curves that are not waiting for a
// Jacobian, and the Jacobian (two thirds of the instructions) for all that accepted, once these
// are more than half of the warp's curves: about every other step is rejected, so a Jacobian per
// trip would run with half its lanes. Still bound by the FP64 pipe. Not faster: one lane per curve
// (270 ms for 1e5 curves: its registers hold one curve's matrix, few warps run), eight lanes (216 ms
// against 182), two lanes (172 ms).
// The Jacobian takes phi and the residuals from the accepted trial's cost.
// One warp per curve -> this kernel, 24 points, two poles: 1e5 curves 440 -> 164 ms, 32,000 144 ->
// 63.6, 8,192 40.2 -> 23.8, 3,500 20.0 -> 17.6; three poles: 8,000 curves 116 -> 42.1 ms; one pole:
// 30,000 curves 20.4 -> 11.0 ms.
constexpr int LMG = 4;                // lanes per curve
// Curves from which this kernel is taken, by the number of poles:
// below them too few warps run (two poles, 3,000 curves: 17.3 -> 17.4 ms; one pole, 4,096: 4.7 ->
// 5.1; three poles, 1,500: 30.3 -> 29.6), the more so with the shared memory of more than 32 points
// (64 points: one pole, 6,500 curves 11.2 -> 11.8; two poles, 3,000 32 -> 34, 9,000 82 -> 70 ms).
constexpr int LM_GROUPS_MIN[2][3] = {{5000, 3500, 2000}, {8000, 5600, 3200}};   // [nw > 32]
// accepted curves of a warp's n that a Jacobian waits for
__host__ __device__ constexpr int LM_JAC(int n) { return n / 2 + 1; }

// Doubles of shared memory per curve: D (which the solve's L, right-hand side and reciprocal pivots
// share), residuals, A, g, theta and the trial. Lanes read consecutive entries, so curves that start
// LMG doubles apart (of the 16 that a row of the banks holds) do not collide (171 -> 164 ms).
__host__ __device__ constexpr int lm_group_d(int nw, int P) {
  return nw * P > P * (P + 1) / 2 + 2 * P ? nw * P : P * (P + 1) / 2 + 2 * P;
}
__host__ __device__ constexpr int lm_group_doubles(int nw, int P) {
  const int d = lm_group_d(nw, P) + 2 * nw + P * (P + 1) / 2 + 3 * P;
  return d + (LMG - d % 16 + 16) % 16;
}

// x with its sign flipped where bit 31 of m is set
__device__ __forceinline__ double lm_flip(double x, int m) {
  return __hiloint2double(__double2hiint(x) ^ m, __double2loint(x));
}

// the sum the butterfly of warp_sum forms of the lanes' values c(l), l = sub + G k held in c[k]
template <int G>
__device__ __forceinline__ double group_butterfly(double (&c)[32 / G]) {
#pragma unroll
  for (int n = 16 / G; n > 0; n /= 2)
#pragma unroll
    for (int k = 0; k < n; ++k) c[k] += c[k + n];
  double v = c[0];
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <int G>
__device__ __forceinline__ double group_max(double v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

template <int NPOLE>
__global__ void __launch_bounds__(64, 4) k_lm_groups(int ncurve, int nw, const __grid_constant__ OmegaArr om,
                                                   const double2* __restrict__ sigma,
                                                   const double* __restrict__ sign,
                                                   const double* theta_init, double* params,
                                                   double* __restrict__ cost_out,
                                                   int* __restrict__ iters_out,
                                                   int* __restrict__ status_out, int keep_better) {
  constexpr int npole = NPOLE;
  constexpr int P = 4 * npole;
  constexpr int NP = P * (P + 1) / 2;
  constexpr int EPL = (NP + LMG - 1) / LMG;     // packed entries per lane
  constexpr int GPL = (P + LMG - 1) / LMG;      // entries of g per lane
  constexpr int NL = 32 / LMG;                  // lanes of the warp kernel per lane
  extern __shared__ double lsm[];
  __shared__ int next;
  const int lane = threadIdx.x & 31, sub = lane & (LMG - 1);
  // D[j][a]: (Re phi, Im phi, Re a phi^2, Im a phi^2) of pole a / 4 at point j. The Jacobian's rows
  // are R[a] = +-D[a] (minus for odd a) and I[a] = D[a ^ 1].
  double* D = lsm + size_t(threadIdx.x / LMG) * lm_group_doubles(nw, P);
  // D is dead from the decision on a trial to the next trial's cost: the solve's arrays overlay it.
  double* Ld = D;
  double* sb = Ld + NP;
  double* dinv = sb + P;
  double* res = D + lm_group_d(nw, P);
  double* sA = res + 2 * nw;
  double* sg = sA + NP;
  double* sth = sg + P;
  double* sthn = sth + P;
  const int per = (ncurve + int(gridDim.x) - 1) / int(gridDim.x);
  const int c_end = min(ncurve, (int(blockIdx.x) + 1) * per);
  if (threadIdx.x == 0) next = int(blockIdx.x) * per;
  __syncthreads();
  // the packed entries e = sub + LMG h of A this lane sums: row (low half) and column
  int eab[EPL];
#pragma unroll
  for (int h = 0; h < EPL; ++h) {
    const int e = sub + LMG * h;
    int a = 0;
    while ((a + 1) * (a + 2) / 2 <= e) ++a;
    eab[h] = e < NP ? a | (e - a * (a + 1) / 2) << 16 : 0;
  }
  // per curve, the same in its lanes
  int cidx = 0, it = 0, st = 1;
  bool active = false, done = false, init = false, jac = false;
  double C = 0.0, cscale = 0.0, mu = -1.0;
  const double2* y = sigma;
  while (true) {
    const bool want = !active && !done;
    if (__any_sync(0xffffffffu, want)) {
      int c = 0;
      if (want && sub == 0) c = atomicAdd(&next, 1);
      c = __shfl_sync(0xffffffffu, c, 0, LMG);
      if (want) {
        if (c >= c_end) {
          done = true;
        } else {
          cidx = c;
          active = init = true;
          it = 0;
          st = 1;
          mu = -1.0;
          y = sigma + size_t(cidx) * nw;
          if (theta_init) {
            for (int k = sub; k < P; k += LMG) sthn[k] = theta_init[size_t(cidx) * P + k];
          } else if (sub == 0) {
            const double s = sign ? (sign[cidx] >= 0.0 ? 1.0 : -1.0) : 1.0;
            lm_default_start(om.v, y, nw, npole, s, sthn);
          }
        }
      }
      __syncwarp();
      double c4[NL];
#pragma unroll
      for (int k = 0; k < NL; ++k) {
        const int l = sub + LMG * k;
        const double2 a = init && l < nw ? y[l] : make_double2(0.0, 0.0);
        const double2 b = init && l + 32 < nw ? y[l + 32] : make_double2(0.0, 0.0);
        c4[k] = fma(b.y, b.y, fma(b.x, b.x, lm_sum(a.x, a.x, a.y, a.y)));
      }
      const double cs = 0.5 * group_butterfly<LMG>(c4);
      if (init) cscale = cs;
      if (!__any_sync(0xffffffffu, active)) break;
    }
    const bool trial = active && !jac;            // a new point: the start, or a damped step
    const bool solve = trial && !init;
    bool ok = true;
    if (__any_sync(0xffffffffu, solve)) {
      if (solve) {
        for (int e = sub; e < NP; e += LMG) Ld[e] = sA[e];
      }
      __syncwarp();
      if (solve) {
        for (int i = sub; i < P; i += LMG) {
          Ld[i * (i + 1) / 2 + i] += mu * sA[i * (i + 1) / 2 + i];
          sb[i] = -sg[i];
        }
      }
      __syncwarp();
      // Cholesky, column by column: the pivot by the curve's first lane, the rows below it by its lanes
      for (int jc = 0; jc < P; ++jc) {
        if (solve && sub == 0) {
          double d = Ld[jc * (jc + 1) / 2 + jc];
          for (int k = 0; k < jc; ++k) d -= Ld[jc * (jc + 1) / 2 + k] * Ld[jc * (jc + 1) / 2 + k];
          if (!(d > 0.0)) ok = false;
          const double r = d > 0.0 ? sqrt(d) : 1.0;
          Ld[jc * (jc + 1) / 2 + jc] = r;
          dinv[jc] = 1.0 / r;
        }
        __syncwarp();
        if (solve) {
          for (int i = jc + 1 + sub; i < P; i += LMG) {
            double v = Ld[i * (i + 1) / 2 + jc];
            for (int k = 0; k < jc; ++k) v -= Ld[i * (i + 1) / 2 + k] * Ld[jc * (jc + 1) / 2 + k];
            Ld[i * (i + 1) / 2 + jc] = v * dinv[jc];
          }
        }
        __syncwarp();
      }
      ok = __shfl_sync(0xffffffffu, int(ok), 0, LMG) != 0;
      // L z = b by column sweeps, then L^T x = z
      for (int k = 0; k < P; ++k) {
        const double zk = sb[k] * dinv[k];
        __syncwarp();
        if (solve) {
          for (int i = k + 1 + sub; i < P; i += LMG) sb[i] -= Ld[i * (i + 1) / 2 + k] * zk;
          if (sub == 0) sb[k] = zk;
        }
        __syncwarp();
      }
      for (int k = P - 1; k >= 0; --k) {
        const double xk = sb[k] * dinv[k];
        __syncwarp();
        if (solve) {
          for (int i = sub; i < k; i += LMG) sb[i] -= Ld[k * (k + 1) / 2 + i] * xk;
          if (sub == 0) sb[k] = xk;
        }
        __syncwarp();
      }
      if (solve)
        for (int k = sub; k < P; k += LMG) sthn[k] = sth[k] + sb[k];
      __syncwarp();
    }
    // the cost at the new point; phi and the residuals stay for its Jacobian
    double Cn = 0.0;
    if (__any_sync(0xffffffffu, trial)) {
      double c4[NL], thn[P];
#pragma unroll
      for (int k = 0; k < P; ++k) thn[k] = sthn[k];
#pragma unroll
      for (int k4 = 0; k4 < NL; ++k4) {
        double c = 0.0;
        for (int h = 0; h < 2; ++h) {
          const int j = sub + LMG * k4 + 32 * h;
          if (j >= nw || !trial) break;
          double fx = 0.0, fy = 0.0;
#pragma unroll
          for (int p = 0; p < npole; ++p) {
            const double dx = -thn[4 * p + 2], dy = om.v[j] - thn[4 * p + 3];
            const double inv = 1.0 / lm_sum(dy, dy, dx, dx);
            const double px = dx * inv, py = -dy * inv;          // phi = 1 / (i w_j - w_p)
            fx += lm_dif(thn[4 * p], px, thn[4 * p + 1], py);
            fy += lm_sum(thn[4 * p], py, thn[4 * p + 1], px);
            D[j * P + 4 * p] = px;
            D[j * P + 4 * p + 1] = py;
          }
          const double2 yj = y[j];
          const double rx = fx - yj.x, ry = fy - yj.y;
          res[2 * j] = rx;
          res[2 * j + 1] = ry;
          c += lm_sum(rx, rx, ry, ry);
        }
        c4[k4] = c;
      }
      Cn = 0.5 * group_butterfly<LMG>(c4);
    }
    bool end = false;
    if (trial) {
      bool accepted = init;
      double dec = 0.0, Cold = 0.0;
      if (!init) {
        accepted = ok && Cn < C;
        if (accepted) {
          mu = fmax(mu / 10.0, LM_MU_MIN);
          dec = C - Cn;
          Cold = C;
        } else {
          mu *= 10.0;
          if (mu > LM_MU_MAX) {
            st = 2;
            end = true;
          }
        }
      }
      if (accepted) {
        for (int k = sub; k < P; k += LMG) sth[k] = sthn[k];
        C = Cn;
        if (!init) {
          ++it;
          if (dec <= LM_FTOL * Cold) {
            st = 0;
            end = true;
          } else if (it >= LM_MAXIT) {
            end = true;
          }
        }
        init = false;
        if (!end) {
          if (C <= LM_CTOL * cscale) {
            st = 0;
            end = true;
          } else {
            jac = true;
          }
        }
      }
    }
    __syncwarp();
    // the Jacobian once enough curves wait for it, or when no other curve can go on
    const unsigned waits = __ballot_sync(0xffffffffu, jac);
    const unsigned goes = __ballot_sync(0xffffffffu, !jac && !done);
    if (waits != 0 && (__popc(waits) >= LMG * LM_JAC(32 / LMG) || goes == 0)) {
      double v[EPL], w[GPL];
#pragma unroll
      for (int h = 0; h < EPL; ++h) v[h] = 0.0;
#pragma unroll
      for (int h = 0; h < GPL; ++h) w[h] = 0.0;
      // a phi^2 at this lane's points (a phi as the cost's)
      if (jac) {
        for (int j = sub; j < nw; j += LMG) {
#pragma unroll
          for (int p = 0; p < npole; ++p) {
            double* d = D + j * P + 4 * p;
            const double ax = sth[4 * p], ay = sth[4 * p + 1], px = d[0], py = d[1];
            const double tx = lm_dif(ax, px, ay, py), ty = lm_sum(ax, py, ay, px);
            d[2] = lm_dif(tx, px, ty, py);
            d[3] = lm_sum(tx, py, ty, px);
          }
        }
      }
      __syncwarp();
      // A (packed lower) and g, summed over points
      if (jac) {
#pragma unroll 2
        for (int j = 0; j < nw; ++j) {
          const double* d = D + j * P;
#pragma unroll
          for (int h = 0; h < EPL; ++h) {
            const int ea = eab[h] & 0xffff, eb = eab[h] >> 16;
            v[h] += lm_sum(lm_flip(d[ea], (ea ^ eb) << 31), d[eb], d[ea ^ 1], d[eb ^ 1]);
          }
        }
#pragma unroll
        for (int h = 0; h < GPL; ++h) {
          const int a = sub + LMG * h;
          if (a < P)
            for (int j = 0; j < nw; ++j)
              w[h] += lm_sum(lm_flip(D[j * P + a], a << 31), res[2 * j], D[j * P + (a ^ 1)], res[2 * j + 1]);
        }
      }
      double gm = 0.0, dm = 0.0;
      if (jac) {
#pragma unroll
        for (int h = 0; h < EPL; ++h) {
          const int e = sub + LMG * h;
          if (e < NP) {
            sA[e] = v[h];
            if ((eab[h] & 0xffff) == eab[h] >> 16) dm = fmax(dm, v[h]);
          }
        }
#pragma unroll
        for (int h = 0; h < GPL; ++h) {
          const int a = sub + LMG * h;
          if (a < P) {
            sg[a] = w[h];
            gm = fmax(gm, fabs(w[h]));
          }
        }
      }
      __syncwarp();
      gm = group_max<LMG>(gm);
      dm = group_max<LMG>(dm);
      if (jac) {
        if (gm <= LM_GTOL) {
          st = 0;
          end = true;
        }
        if (mu < 0.0) mu = 1e-3 * dm;
        jac = false;
      }
    }
    if (end) {
      active = false;
      // the other start's result stays when it is not worse
      if (sub == 0 && (!keep_better || C < cost_out[cidx])) {
        for (int k = 0; k < P; ++k) params[size_t(cidx) * P + k] = sth[k];
        cost_out[cidx] = C;
        iters_out[cidx] = it;
        status_out[cidx] = st;
      }
    }
  }
}

template <int NPOLE>
static int launch_lm_groups(int ncurve, int nw, const OmegaArr& om, const double2* y, const double* sign,
                            const double* theta_init, double* params, double* cost, int* iters,
                            int* status, int keep_better, cudaStream_t s, const DeviceCtx& ctx) {
  const auto kern = k_lm_groups<NPOLE>;
  const size_t per_warp = size_t(32 / LMG) * lm_group_doubles(nw, 4 * NPOLE) * sizeof(double);
  // Two warps share a range of curves once every SM gets five such blocks; with fewer, blocks of
  // one warp spread over the SMs more evenly (8,192 curves 29.9 -> 25.9 ms; 1e5: 181 against 186).
  const int warps = ncurve >= 5 * 2 * (32 / LMG) * ctx.sm_count ? 2 : 1;
  const size_t smem = warps * per_warp;
  int rc = set_max_dyn_smem(reinterpret_cast<const void*>(kern), smem, ctx.device);
  if (rc) return rc;
  int fit = 0;                        // resident blocks per SM
  GW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, 32 * warps, smem));
  const int curves = warps * 32 / LMG;
  const int blocks = int(std::min<int64_t>((int64_t(ncurve) + curves - 1) / curves,
                                           int64_t(ctx.sm_count) * std::max(1, fit)));
  kern<<<blocks, 32 * warps, smem, s>>>(ncurve, nw, om, y, sign, theta_init, params, cost, iters, status,
                                       keep_better);
  GW_LAUNCH_CHECK("k_lm_groups");
  return GW_OK;
}

int launch_lm(int ncurve, int nw, const OmegaArr& om, const double* sigma, const double* sign,
              int npole, const double* theta_init, double* params, double* cost, int* iters,
              int* status, int keep_better, cudaStream_t s) {
  if (ncurve == 0) return GW_OK;
  if (nw > LM_WMAXNW) return set_error(GW_EINVAL, "the fit takes at most %d frequencies", LM_WMAXNW);
  const double2* y = reinterpret_cast<const double2*>(sigma);
  if (npole <= 3 && ncurve >= LM_GROUPS_MIN[nw > 32][npole - 1]) {
    DeviceCtx ctx;
    int rc = device_ctx(&ctx);
    if (rc) return rc;
    const auto run = npole == 1 ? launch_lm_groups<1> : npole == 2 ? launch_lm_groups<2> : launch_lm_groups<3>;
    return run(ncurve, nw, om, y, sign, theta_init, params, cost, iters, status, keep_better, s, ctx);
  }
  auto go = [&](auto kern) {
    kern<<<ncurve, 32, 0, s>>>(ncurve, nw, om, y, sign, theta_init, params, cost, iters, status,
                               keep_better);
  };
  switch (npole) {
    case 1: go(k_lm_warp<1>); break;
    case 2: go(k_lm_warp<2>); break;
    case 3: go(k_lm_warp<3>); break;
    case 4: go(k_lm_warp<4>); break;
    default: go(k_lm_warp<5>); break;
  }
  GW_LAUNCH_CHECK("k_lm_warp");
  return GW_OK;
}

}  // namespace gw
