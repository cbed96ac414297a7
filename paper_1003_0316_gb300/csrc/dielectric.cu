// a3: dielectric matrix and W^c in FP64 (Eqs. dielec_MB, screen_MB; W^c = W - v).
//
//   eps = 1 - v^1/2 P v^1/2      (Hermitian positive definite on the imaginary axis)
//   eps = L L^H                   blocked Cholesky
//   Z   = L^{-1}                  blocked triangular inversion
//   W^c = v^1/2 (Z^H Z - 1) v^1/2
//
// The caller-workspace entry points factorise a workspace copy of eps over many CTAs (per 32-wide
// panel: the diagonal block and its inverse, the panel below it, the trailing update of the lower
// 32x32 tiles), invert the factor by block columns and form W^c with one CTA per (system, 32-row
// block); each thread owns one row and four columns of a 32x32 tile staged in shared memory. About
// 4 N^3 real flops per system (N^3/6 complex multiply-adds per phase). Storage and arithmetic are
// float-float on the FP32 pipe, which GB300 executes 64 times faster than FP64 (see FF below): about
// 2^-48 relative per operation; P, v and W^c are FP64. For larger systems all products outside the
// diagonal 128-blocks and the current 128-column panel run on the tensor cores (DzChunk below). The
// no-allocation entry point keeps the factorisation and the inverse inside one CTA per system, in
// FP64.
#include <vector>
#include <algorithm>
#include <mutex>

#include "fp64_slices.cuh"
#include "gw_internal.cuh"

namespace gw {

constexpr int DB = 32;        // tile edge
constexpr int DLD = DB + 1;   // padded smem row
constexpr int DTHREADS = 256;

// One system. P and W^c are complex128 in global memory; the factor, the inverse and the
// panel (E, T) and the shared-memory tiles hold T: double2 for Hermitian systems, double for
// real symmetric ones (inversion-symmetric systems: the imaginary parts of P are zero and are
// not read, W^c is written with zero imaginary parts).
template <typename T>
struct DieSysT {
  const double2* P;
  double2* Wc;
  const double* v;
  T* E;      // N x N workspace (factor / inverse)
  T* Tp;     // N x DB workspace panel (inverse inside the CTA)
  T* Z;      // the inverse factor read by the W^c phase: E, or a buffer of its own
  T* D;      // inverted diagonal blocks [nt][DB][DB] (inverse by block columns), or NULL
  int n;
};

// scalar operations for the complex and the real systems
__device__ __forceinline__ double re_(double2 a) { return a.x; }
__device__ __forceinline__ double re_(double a) { return a; }
__device__ __forceinline__ double im_(double2 a) { return a.y; }
__device__ __forceinline__ double im_(double) { return 0.0; }
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double cconj(double a) { return a; }
__device__ __forceinline__ void cfma(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}
__device__ __forceinline__ void cfma(double& acc, double a, double b) { acc = fma(a, b, acc); }
__device__ __forceinline__ void csubmul(double2& x, double2 a, double2 b) {   // x -= a b
  x.x -= a.x * b.x - a.y * b.y;
  x.y -= a.x * b.y + a.y * b.x;
}
__device__ __forceinline__ void csubmul(double& x, double a, double b) { x -= a * b; }
__device__ __forceinline__ double2 scal(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double scal(double a, double s) { return a * s; }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double csub(double a, double b) { return a - b; }
__device__ __forceinline__ double2 add_re(double2 a, double d) { return make_double2(a.x + d, a.y); }
__device__ __forceinline__ double add_re(double a, double d) { return a + d; }
__device__ __forceinline__ bool fin(double2 a) { return isfinite(a.x) && isfinite(a.y); }
__device__ __forceinline__ bool fin(double a) { return isfinite(a); }
template <typename T> __device__ __forceinline__ T real_of(double d);
template <> __device__ __forceinline__ double2 real_of<double2>(double d) { return make_double2(d, 0.0); }
template <> __device__ __forceinline__ double real_of<double>(double d) { return d; }
template <typename T> __device__ __forceinline__ T from_c(double2 p);
template <> __device__ __forceinline__ double2 from_c<double2>(double2 p) { return p; }
template <> __device__ __forceinline__ double from_c<double>(double2 p) { return p.x; }
__device__ __forceinline__ double2 to_c(double2 a) { return a; }
__device__ __forceinline__ double2 to_c(double a) { return make_double2(a, 0.0); }

// Load a DB x DB tile of a row-major N x N (ld) matrix at (r0, c0) into smem.
// mode 0: plain; mode 1: keep only the lower triangle (col <= row), zeros elsewhere.
template <typename T>
__device__ __forceinline__ void load_tile(T* S, const T* A, int ld, int n_rows, int n_cols, int r0,
                                          int c0, int mode) {
  for (int e = threadIdx.x; e < DB * DB; e += DTHREADS) {
    int r = e / DB, c = e % DB;
    int R = r0 + r, C = c0 + c;
    T v = T{};
    if (R < n_rows && C < n_cols && (mode == 0 || C <= R)) v = A[size_t(R) * ld + C];
    S[r * DLD + c] = v;
  }
}

// acc[b] += sum_k opA(tr, k) * SB[k][tc + 8 b]; opA = SA[tr][k] or conj(SA[k][tr]).
template <bool A_CONJ_T, typename T>
__device__ __forceinline__ void tile_mac(T acc[4], const T* SA, const T* SB, int tr, int tc) {
#pragma unroll 8
  for (int k = 0; k < DB; ++k) {
    T a = A_CONJ_T ? cconj(SA[k * DLD + tr]) : SA[tr * DLD + k];
#pragma unroll
    for (int b = 0; b < 4; ++b) cfma(acc[b], a, SB[k * DLD + tc + 8 * b]);
  }
}

// ---- float-float tile products on the FP32 pipe ----------------------------------------------
// GB300 executes FP64 fused multiply-adds at 1/64 of its FP32 rate, so the tile products of the
// factorisation's trailing update, of the inverse by block columns and of Z^H Z run in
// float-float arithmetic: every FP64 operand becomes an unevaluated sum h + l of two FP32
// values (48 significant bits), each product h_x h_y is split exactly into its rounded value
// and error with one FMA (Dekker's product), the cross terms h_x l_y + l_x h_y are added in
// FP32 (l_x l_y and the rounding of the cross terms lie below 2^-48 of the product), and the
// running sum keeps its exact rounding errors by Knuth's two-sum in a compensation term; the
// result returns to FP64 as s + c. About 2^-48 relative per operation against 2^-53 for FP64.
// Intrinsics (__fmul_rn, __fadd_rn) keep the compiler from fusing the error-free steps.
struct FF {                // h + l, |l| <= ulp(h) / 2
  float h, l;
};
struct FFC {
  FF re, im;
};
struct FAcc {              // running sum s and compensation c: the value s + c
  float s, c;
};
struct FAccC {
  FAcc re, im;
};
template <typename T> struct FFOf;
template <> struct FFOf<double> { using tile = FF; using acc = FAcc; };
template <> struct FFOf<double2> { using tile = FFC; using acc = FAccC; };

__device__ __forceinline__ FF to_ff(double x) {
  const float h = __double2float_rn(x);
  return FF{h, __double2float_rn(x - double(h))};
}
// to_ff by integer arithmetic (each FP64 conversion occupies the FP64 pipe like a multiply-add): h
// from the magnitude rounded to 24 bits (to nearest, ties to even), l from the remaining bits, whose
// integer difference is exact. For small x the power of two of l leaves the FP32 range (from 2^-73 on) and
// is applied in two steps; |x| < 2^-126, where h is not normal, counts as zero.
__device__ __forceinline__ FF split_ff(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7fffffffffffffffull;
  const unsigned long long hb = (b + 0x0fffffffull + ((b >> 29) & 1ull)) & ~0x1fffffffull;
  const int ex = int(b >> 52);                                   // biased by 1023
  const uint32_t sign = static_cast<uint32_t>(__double2hiint(x)) & 0x80000000u;
  const long long hf = static_cast<long long>(hb >> 29) - (896ll << 23);
  const uint32_t hbits = hf < 0x00800000ll ? 0u : hf > 0x7f800000ll ? 0x7f800000u : uint32_t(hf);
  const float d = float(int(static_cast<long long>(b) - static_cast<long long>(hb)));
  const bool small = ex < 1023 - 32;
  const int se = min(ex - 1023 - 52 + 127 + (small ? 64 : 0), 254);              // 2^(e - 52), or 2^64 of it
  const float l = hbits == 0u ? 0.0f : d * __int_as_float(se << 23) * (small ? 5.42101086e-20f : 1.0f);
  return FF{__uint_as_float(hbits | sign), __uint_as_float(__float_as_uint(l) ^ sign)};
}
__device__ __forceinline__ FF split_ff_t(double x) { return split_ff(x); }
__device__ __forceinline__ FFC split_ff_t(double2 x) { return FFC{split_ff(x.x), split_ff(x.y)}; }
__device__ __forceinline__ FF to_ff_t(double x) { return to_ff(x); }
__device__ __forceinline__ FFC to_ff_t(double2 x) { return FFC{to_ff(x.x), to_ff(x.y)}; }
__device__ __forceinline__ FF ff_neg(FF x) { return FF{-x.h, -x.l}; }
__device__ __forceinline__ FFC ff_conj(FFC x) { return FFC{x.re, ff_neg(x.im)}; }
__device__ __forceinline__ FF ff_conj(FF x) { return x; }

// a += x y
__device__ __forceinline__ void ff_mac(FAcc& a, FF x, FF y) {
  const float p = __fmul_rn(x.h, y.h);
  const float e = __fmaf_rn(x.h, y.h, -p);                       // x.h y.h = p + e exactly
  const float t = __fmaf_rn(x.h, y.l, __fmul_rn(x.l, y.h));      // cross terms
  const float sum = __fadd_rn(a.s, p);                           // two-sum: a.s + p = sum + err
  const float bp = __fadd_rn(sum, -a.s);
  const float err = __fadd_rn(__fadd_rn(a.s, -__fadd_rn(sum, -bp)), __fadd_rn(p, -bp));
  a.s = sum;
  a.c = __fadd_rn(a.c, __fadd_rn(err, __fadd_rn(e, t)));
}
__device__ __forceinline__ void ff_cmac(FAcc& a, FF x, FF y) { ff_mac(a, x, y); }
__device__ __forceinline__ void ff_cmac(FAccC& a, FFC x, FFC y) {   // a += x y, complex
  ff_mac(a.re, x.re, y.re);
  ff_mac(a.re, ff_neg(x.im), y.im);
  ff_mac(a.im, x.re, y.im);
  ff_mac(a.im, x.im, y.re);
}
__device__ __forceinline__ double ff_value(FAcc a) { return double(a.s) + double(a.c); }
__device__ __forceinline__ double ff_value_t(FAcc a) { return ff_value(a); }
__device__ __forceinline__ double2 ff_value_t(FAccC a) { return make_double2(ff_value(a.re), ff_value(a.im)); }

// the float-float value h + l of an accumulator (two-sum of s and c)
__device__ __forceinline__ FF ff_renorm(FAcc a) {
  const float h = __fadd_rn(a.s, a.c);
  const float bp = __fadd_rn(h, -a.s);
  return FF{h, __fadd_rn(__fadd_rn(a.s, -__fadd_rn(h, -bp)), __fadd_rn(a.c, -bp))};
}
__device__ __forceinline__ FF ff_renorm_t(FAcc a) { return ff_renorm(a); }
__device__ __forceinline__ FFC ff_renorm_t(FAccC a) { return FFC{ff_renorm(a.re), ff_renorm(a.im)}; }
__device__ __forceinline__ FAcc ff_acc(FF x) { return FAcc{x.h, x.l}; }
__device__ __forceinline__ FAccC ff_acc(FFC x) { return FAccC{ff_acc(x.re), ff_acc(x.im)}; }
// x y rounded to float-float (the correction is below ulp(p), so a fast two-sum renormalises)
__device__ __forceinline__ FF ff_mul(FF x, FF y) {
  const float p = __fmul_rn(x.h, y.h);
  const float q = __fadd_rn(__fmaf_rn(x.h, y.h, -p), __fmaf_rn(x.h, y.l, __fmul_rn(x.l, y.h)));
  const float h = __fadd_rn(p, q);
  return FF{h, __fadd_rn(q, -__fadd_rn(h, -p))};
}
__device__ __forceinline__ FF ff_scale(FF x, FF r) { return ff_mul(x, r); }
__device__ __forceinline__ FFC ff_scale(FFC x, FF r) { return FFC{ff_mul(x.re, r), ff_mul(x.im, r)}; }
// acc -= x conj(l)
__device__ __forceinline__ void ff_csubmul_conj(FAcc& a, FF x, FF l) { ff_mac(a, ff_neg(x), l); }
__device__ __forceinline__ void ff_csubmul_conj(FAccC& a, FFC x, FFC l) {
  ff_mac(a.re, ff_neg(x.re), l.re);
  ff_mac(a.re, ff_neg(x.im), l.im);
  ff_mac(a.im, ff_neg(x.im), l.re);
  ff_mac(a.im, x.re, l.im);
}
// acc -= x y
__device__ __forceinline__ void ff_csubmul(FAcc& a, FF x, FF y) { ff_mac(a, ff_neg(x), y); }
__device__ __forceinline__ void ff_csubmul(FAccC& a, FFC x, FFC y) {
  ff_mac(a.re, ff_neg(x.re), y.re);
  ff_mac(a.re, x.im, y.im);
  ff_mac(a.im, ff_neg(x.re), y.im);
  ff_mac(a.im, ff_neg(x.im), y.re);
}
__device__ __forceinline__ FF ff_re(FF x) { return x; }
__device__ __forceinline__ FF ff_re(FFC x) { return x.re; }
template <typename FT> __device__ __forceinline__ FT ff_real(FF x);
template <> __device__ __forceinline__ FF ff_real<FF>(FF x) { return x; }
template <> __device__ __forceinline__ FFC ff_real<FFC>(FF x) { return FFC{x, FF{0.0f, 0.0f}}; }
// 1 / sqrt(d) for a positive d: the FP32 approximation y and one Newton step
// y + y (1 - d y^2) / 2 with the residual in float-float (relative error near 2^-46)
__device__ __forceinline__ FF ff_rsqrt(FF d) {
  const float y = rsqrtf(d.h);
  FAcc r = {1.0f, 0.0f};
  const float p = __fmul_rn(y, y);
  ff_mac(r, ff_neg(d), FF{p, __fmaf_rn(y, y, -p)});          // 1 - d y^2
  const FF e = ff_renorm(r);
  const float c = __fmul_rn(0.5f * y, e.h);
  // the second-order term 3/8 y e^2 keeps the result at the float-float level
  const float c2 = __fmaf_rn(__fmul_rn(0.375f * y, e.h), e.h, __fmul_rn(0.5f * y, e.l));
  return ff_renorm(FAcc{y, __fadd_rn(c, __fadd_rn(c2, __fmaf_rn(0.5f * y, e.h, -c)))});
}

// e - a rounded to float-float (e a float-float value, a an accumulator)
__device__ __forceinline__ FF ff_sub_acc(FF e, FAcc a) {
  const float sh = __fadd_rn(e.h, -a.s);                          // two-sum of e.h and -a.s
  const float bp = __fadd_rn(sh, -e.h);
  const float err = __fadd_rn(__fadd_rn(e.h, -__fadd_rn(sh, -bp)), __fadd_rn(-a.s, -bp));
  return ff_renorm(FAcc{sh, __fadd_rn(err, __fadd_rn(e.l, -a.c))});
}
__device__ __forceinline__ FF ff_sub_acc_t(FF e, FAcc a) { return ff_sub_acc(e, a); }
__device__ __forceinline__ FFC ff_sub_acc_t(FFC e, FAccC a) {
  return FFC{ff_sub_acc(e.re, a.re), ff_sub_acc(e.im, a.im)};
}
__device__ __forceinline__ FF ff_negate(FF x) { return ff_neg(x); }
__device__ __forceinline__ FFC ff_negate(FFC x) { return FFC{ff_neg(x.re), ff_neg(x.im)}; }

// The caller-workspace path keeps eps, its factor, the inverse factor and the inverted
// diagonal blocks in float-float form (the bytes of the FP64 element: complex FFC, real FF),
// so the tile products load them without FP64 conversions; the output W^c is FP64.
template <typename T>
using StorOf = typename FFOf<T>::tile;
template <typename T>
__device__ __forceinline__ StorOf<T>* stor(T* p) { return reinterpret_cast<StorOf<T>*>(p); }
template <typename T>
__device__ __forceinline__ const StorOf<T>* stor(const T* p) {
  return reinterpret_cast<const StorOf<T>*>(p);
}

// a DB x DB tile of float-float storage into shared memory (mode 1: lower triangle only)
template <typename FT>
__device__ __forceinline__ void load_tile_s(FT* S, const FT* A, int ld, int n_rows, int n_cols,
                                            int r0, int c0, int mode) {
  for (int e = threadIdx.x; e < DB * DB; e += DTHREADS) {
    int r = e / DB, c = e % DB;
    int R = r0 + r, C = c0 + c;
    FT v = FT{};
    if (R < n_rows && C < n_cols && (mode == 0 || C <= R)) v = A[size_t(R) * ld + C];
    S[r * DLD + c] = v;
  }
}
// load_tile into float-float shared memory
template <typename T>
__device__ __forceinline__ void load_tile_ff(typename FFOf<T>::tile* S, const T* A, int ld,
                                             int n_rows, int n_cols, int r0, int c0, int mode) {
  for (int e = threadIdx.x; e < DB * DB; e += DTHREADS) {
    int r = e / DB, c = e % DB;
    int R = r0 + r, C = c0 + c;
    T v = T{};
    if (R < n_rows && C < n_cols && (mode == 0 || C <= R)) v = A[size_t(R) * ld + C];
    S[r * DLD + c] = to_ff_t(v);
  }
}

// acc[b] += sum_k opA(tr, k) * SB[k][tc + 8 b] in float-float; opA = SA[tr][k] or conj(SA[k][tr])
template <bool A_CONJ_T, typename FT, typename FA>
__device__ __forceinline__ void tile_mac_ff(FA acc[4], const FT* SA, const FT* SB, int tr, int tc) {
#pragma unroll 4
  for (int k = 0; k < DB; ++k) {
    const FT a = A_CONJ_T ? ff_conj(SA[k * DLD + tr]) : SA[tr * DLD + k];
#pragma unroll
    for (int b = 0; b < 4; ++b) ff_cmac(acc[b], a, SB[k * DLD + tc + 8 * b]);
  }
}

constexpr int DMAXSYS = 256;   // systems per launch (descriptors passed by value)
template <typename T>
struct DieBatchT {
  DieSysT<T> s[DMAXSYS];
};

template <typename T>
__global__ void __launch_bounds__(DTHREADS) k_dielectric(const DieBatchT<T> batch, unsigned* status) {
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  T* smem = reinterpret_cast<T*>(dsm_raw);
  T* SA = smem;
  T* SB = smem + DB * DLD;
  T* SD = smem + 2 * DB * DLD;
  __shared__ int s_fail;

  const DieSysT<T> sys = batch.s[blockIdx.x];
  const int n = sys.n;
  T* E = sys.E;
  const int tid = threadIdx.x;
  const int tr = tid >> 3, tc = tid & 7;
  if (tid == 0) s_fail = 0;

  // ---- phase 0: eps = 1 - v^1/2 P v^1/2 (full matrix) ---------------------
  for (size_t e = tid; e < size_t(n) * n; e += DTHREADS) {
    int r = int(e / n), c = int(e % n);
    double s = sqrt(sys.v[r] * sys.v[c]);
    T x = scal(from_c<T>(sys.P[e]), -s);
    if (r == c) x = add_re(x, 1.0);
    if (!fin(x)) atomicOr(&s_fail, 2);
    E[e] = x;
  }
  __syncthreads();

  const int nt = (n + DB - 1) / DB;
  // ---- phase 1: Cholesky, lower, in place ---------------------------------
  for (int kt = 0; kt < nt; ++kt) {
    const int k0 = kt * DB;
    const int kb = min(DB, n - k0);
    load_tile(SD, E, n, n, n, k0, k0, 1);
    __syncthreads();
    for (int c = 0; c < kb; ++c) {
      if (tid == 0) {
        double d = re_(SD[c * DLD + c]);
        if (!(d > 0.0) || !isfinite(d)) {
          atomicOr(&s_fail, 1);
          d = 1.0;
        }
        SD[c * DLD + c] = real_of<T>(sqrt(d));
      }
      __syncthreads();
      double dinv = 1.0 / re_(SD[c * DLD + c]);
      for (int r = c + 1 + tid; r < kb; r += DTHREADS) SD[r * DLD + c] = scal(SD[r * DLD + c], dinv);
      __syncthreads();
      for (int e = tid; e < DB * DB; e += DTHREADS) {
        int r = e / DB, s = e % DB;
        if (r < kb && s > c && s <= r) {
          T x = SD[r * DLD + s];
          csubmul(x, SD[r * DLD + c], cconj(SD[s * DLD + c]));
          SD[r * DLD + s] = x;
        }
      }
      __syncthreads();
    }
    for (int e = tid; e < DB * DB; e += DTHREADS) {
      int r = e / DB, c = e % DB;
      if (r < kb && c <= r) E[size_t(k0 + r) * n + k0 + c] = SD[r * DLD + c];
    }
    __syncthreads();
    // panel: X L11^H = A21, one row per thread
    for (int r = k0 + kb + tid; r < n; r += DTHREADS) {
      T x[DB];
      T* row = E + size_t(r) * n + k0;
#pragma unroll
      for (int c = 0; c < DB; ++c) x[c] = c < kb ? row[c] : T{};
#pragma unroll
      for (int c = 0; c < DB; ++c) {
        if (c < kb) {
          T s = x[c];
#pragma unroll
          for (int k = 0; k < c; ++k) csubmul(s, x[k], cconj(SD[c * DLD + k]));
          x[c] = scal(s, 1.0 / re_(SD[c * DLD + c]));
        }
      }
#pragma unroll
      for (int c = 0; c < DB; ++c)
        if (c < kb) row[c] = x[c];
    }
    __syncthreads();
    // trailing update: A22 -= X X^H (lower tiles)
    for (int it = kt + 1; it < nt; ++it) {
      load_tile(SA, E, n, n, n, it * DB, k0, 0);   // X rows of tile it
      for (int jt = kt + 1; jt <= it; ++jt) {
        // SB[k][c] = conj(X[jt*DB + c][k0 + k])
        for (int e = tid; e < DB * DB; e += DTHREADS) {
          int k = e / DB, c = e % DB;
          int R = jt * DB + c;
          T v = T{};
          if (R < n && k < kb) v = cconj(E[size_t(R) * n + k0 + k]);
          SB[k * DLD + c] = v;
        }
        __syncthreads();
        T acc[4] = {T{}, T{}, T{}, T{}};
        tile_mac<false>(acc, SA, SB, tr, tc);
        int R = it * DB + tr;
        if (R < n) {
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int C = jt * DB + tc + 8 * b;
            if (C < n && C <= R) E[size_t(R) * n + C] = csub(E[size_t(R) * n + C], acc[b]);
          }
        }
        __syncthreads();
      }
    }
    __syncthreads();
  }
  if (s_fail) {
    if (tid == 0) raise_status(status, (s_fail & 1) ? ST_ENOTHPD : ST_ENONFINITE);
    return;
  }

  // ---- phase 2: Z = L^{-1}, lower, in place --------------------------------
  for (int kt = nt - 1; kt >= 0; --kt) {
    const int k0 = kt * DB;
    const int kb = min(DB, n - k0);
    load_tile(SD, E, n, n, n, k0, k0, 1);
    __syncthreads();
    // invert the diagonal block: column c handled by thread c
    if (tid < DB) {
      int c = tid;
      T z[DB];
#pragma unroll
      for (int i = 0; i < DB; ++i) z[i] = T{};
      if (c < kb) {
        z[c] = real_of<T>(1.0 / re_(SD[c * DLD + c]));
#pragma unroll
        for (int i = 0; i < DB; ++i) {
          if (i > c && i < kb) {
            T s = T{};
            for (int k = c; k < i; ++k) cfma(s, SD[i * DLD + k], z[k]);
            z[i] = scal(s, -1.0 / re_(SD[i * DLD + i]));
          }
        }
      }
      // stash the inverted column in SB (column c)
#pragma unroll
      for (int i = 0; i < DB; ++i) SB[i * DLD + c] = z[i];
    }
    __syncthreads();
    // SD <- inverse of the diagonal block
    for (int e = tid; e < DB * DB; e += DTHREADS) {
      int r = e / DB, c = e % DB;
      SD[r * DLD + c] = SB[r * DLD + c];
    }
    __syncthreads();
    if (k0 + kb < n) {
      // T[R] = Z22[R][:] * L21 over the trailing rows (Z22 already inverted)
      for (int it = kt + 1; it < nt; ++it) {
        T acc[4] = {T{}, T{}, T{}, T{}};
        for (int st = kt + 1; st <= it; ++st) {
          load_tile(SA, E, n, n, n, it * DB, st * DB, st == it ? 1 : 0);   // Z22 block
          load_tile(SB, E, n, n, n, st * DB, k0, 0);                        // L21 block
          __syncthreads();
          tile_mac<false>(acc, SA, SB, tr, tc);
          __syncthreads();
        }
        int R = it * DB + tr;
        if (R < n) {
#pragma unroll
          for (int b = 0; b < 4; ++b) sys.Tp[size_t(R) * DB + tc + 8 * b] = acc[b];
        }
      }
      __syncthreads();
      // Z21 = -T * Z11
      for (int it = kt + 1; it < nt; ++it) {
        load_tile(SA, sys.Tp, DB, n, DB, it * DB, 0, 0);
        __syncthreads();
        T acc[4] = {T{}, T{}, T{}, T{}};
        tile_mac<false>(acc, SA, SD, tr, tc);
        int R = it * DB + tr;
        if (R < n) {
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int C = tc + 8 * b;
            if (C < kb) E[size_t(R) * n + k0 + C] = scal(acc[b], -1.0);
          }
        }
        __syncthreads();
      }
    }
    for (int e = tid; e < DB * DB; e += DTHREADS) {
      int r = e / DB, c = e % DB;
      if (r < kb && c <= r) E[size_t(k0 + r) * n + k0 + c] = SD[r * DLD + c];
    }
    __syncthreads();
  }

  // phase 3 (W^c from Z) runs as its own launch over (system, block row): k_dielectric_w
}

// ---- phase 3: W^c = v^1/2 (Z^H Z - 1) v^1/2, one CTA per (system, 32-row block rt) ---------
// (the lower tiles ct <= rt of the block row and their Hermitian mirror)
template <typename T, bool FS>
__global__ void __launch_bounds__(DTHREADS) k_dielectric_w(const DieBatchT<T> batch) {
  using FT = typename FFOf<T>::tile;
  using FA = typename FFOf<T>::acc;
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  FT* SA = reinterpret_cast<FT*>(dsm_raw);      // float-float tiles (the size of T)
  FT* SB = SA + DB * DLD;
  const DieSysT<T> sys = batch.s[blockIdx.x];
  const int n = sys.n;
  const int nt = (n + DB - 1) / DB;
  const int rt = blockIdx.y;
  if (rt >= nt) return;                      // whole CTA, before any barrier
  const T* E = sys.Z;
  const int tid = threadIdx.x;
  const int tr = tid >> 3, tc = tid & 7;
  __shared__ double svr[DB], svc[DB];        // square roots of v of the tile's rows and columns
  if (tid < DB) svr[tid] = rt * DB + tid < n ? sqrt(sys.v[rt * DB + tid]) : 0.0;
  for (int ct = 0; ct <= rt; ++ct) {
    __syncthreads();                          // the previous tile's epilogue has read svc
    if (tid < DB) svc[tid] = ct * DB + tid < n ? sqrt(sys.v[ct * DB + tid]) : 0.0;
    FA acc[4] = {};
    for (int kt2 = rt; kt2 < nt; ++kt2) {
      if (FS) {                              // Z in float-float storage
        load_tile_s(SA, stor(E), n, n, n, kt2 * DB, rt * DB, 1);   // Z[K][R] (lower part)
        load_tile_s(SB, stor(E), n, n, n, kt2 * DB, ct * DB, 1);   // Z[K][S]
      } else {                               // Z in FP64 (the no-allocation entry)
        load_tile_ff<T>(SA, E, n, n, n, kt2 * DB, rt * DB, 1);
        load_tile_ff<T>(SB, E, n, n, n, kt2 * DB, ct * DB, 1);
      }
      __syncthreads();
      tile_mac_ff<true>(acc, SA, SB, tr, tc);
      __syncthreads();
    }
    int R = rt * DB + tr;
    if (R < n) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        int C = ct * DB + tc + 8 * b;
        if (C < n && C <= R) {
          T x = ff_value_t(acc[b]);
          if (C == R) x = real_of<T>(re_(x) - 1.0);
          x = scal(x, svr[tr] * svc[tc + 8 * b]);
          sys.Wc[size_t(R) * n + C] = to_c(x);
          if (C != R) sys.Wc[size_t(C) * n + R] = to_c(cconj(x));
        }
      }
    }
  }
}

// ---- the inverse Z = L^{-1} by block columns (the columns of Z are independent forward
// substitutions L Z_c = I_c); the diagonal blocks D_r were inverted by k_chol_diag.
// One CTA per (system, block column c): for r = c, c + 1, ...
//   Z[r][c] = D_r (delta_rc - sum_{k = c}^{r-1} L[r][k] Z[k][c])
// (with a group, only the rows of the column's group of blocks: the inverses of the diagonal groups)
// with the earlier blocks Z[k][c] of the same column read back from global memory.
template <typename T>
__global__ void __launch_bounds__(DTHREADS) k_dielectric_zcol(const DieBatchT<T> batch, int group) {
  using FT = typename FFOf<T>::tile;
  using FA = typename FFOf<T>::acc;
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  FT* SA = reinterpret_cast<FT*>(dsm_raw);      // float-float tiles (the size of T)
  FT* SB = SA + DB * DLD;
  const DieSysT<T> sys = batch.s[blockIdx.x];
  const int n = sys.n;
  const int nt = (n + DB - 1) / DB;
  const int c = blockIdx.y;
  if (c >= nt) return;                       // whole CTA, before any barrier
  const int tid = threadIdx.x;
  const int tr = tid >> 3, tc = tid & 7;
  StorOf<T>* Z = stor(sys.Z);
  const StorOf<T>* L = stor(sys.E);
  const int r_end = group ? min(nt, (c / group + 1) * group) : nt;
  for (int r = c; r < r_end; ++r) {
    FT out[4] = {FT{}, FT{}, FT{}, FT{}};
    if (r == c) {
      const FT* Dr = stor(sys.D) + size_t(r) * DB * DB;
#pragma unroll
      for (int b = 0; b < 4; ++b) out[b] = Dr[tr * DB + tc + 8 * b];
    } else {
      FA acc[4] = {};
      for (int k = c; k < r; ++k) {
        load_tile_s(SA, L, n, n, n, r * DB, k * DB, 0);              // L[r][k]
        load_tile_s(SB, Z, n, n, n, k * DB, c * DB, k == c ? 1 : 0); // Z[k][c]
        __syncthreads();
        tile_mac_ff<false>(acc, SA, SB, tr, tc);
        __syncthreads();
      }
      // out = -D_r acc: the product tile in SB, D_r in SA
#pragma unroll
      for (int b = 0; b < 4; ++b) SB[tr * DLD + tc + 8 * b] = ff_renorm_t(acc[b]);
      const FT* Dr = stor(sys.D) + size_t(r) * DB * DB;
      for (int e = tid; e < DB * DB; e += DTHREADS) SA[(e / DB) * DLD + e % DB] = Dr[e];
      __syncthreads();
      FA o[4] = {};
      tile_mac_ff<false>(o, SA, SB, tr, tc);
      __syncthreads();
#pragma unroll
      for (int b = 0; b < 4; ++b) out[b] = ff_negate(ff_renorm_t(o[b]));
    }
    const int R = r * DB + tr;
    if (R < n) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int C = c * DB + tc + 8 * b;
        if (C < n) Z[size_t(R) * n + C] = out[b];
      }
    }
    __syncthreads();                          // this block row is read by the next ones
  }
}

// ---- the factorisation over many CTAs (the caller-workspace entry points) -----------------
// One launch per step and 32-wide panel kt: the diagonal block with its inverse (one CTA per system),
// the panel below it (one CTA per system and 32 rows, a triangular solve in steps of 8 columns), the update of
// the lower tiles (one CTA per system and 32 x 32 tile): of all tiles behind the panel (right-looking)
// in small systems, of those inside the current 128 columns in large ones, whose panels of 128 first
// take one product with all columns before them (left-looking, DzChunk below). Every SM takes part
// however few systems there are (20 systems of N_b = 4096 would leave 132 of 152 SMs idle with
// one CTA per system).

// the lower triangle of eps = 1 - v^1/2 P v^1/2 (what the factorisation reads), with the whole of P
// checked for non-finite values: grid (32-row blocks, system). Three FP64 multiplications per
// complex entry; the square roots of v are taken once per row and column block and the split into
// float-float is integer work, since the FP64 pipe set the pace (128 systems of N_b = 600, the full
// matrix with FP64 conversions: 1.28 ms).
template <typename T>
__global__ void __launch_bounds__(DTHREADS) k_eps_fill(const DieBatchT<T> batch, unsigned* status) {
  __shared__ double svr[DB], svc[DTHREADS];
  const DieSysT<T>& sys = batch.s[blockIdx.y];
  const int n = sys.n;
  const int r0 = blockIdx.x * DB;
  if (r0 >= n) return;                       // whole CTA, before any barrier
  const int tid = threadIdx.x;
  if (tid < DB) svr[tid] = r0 + tid < n ? sqrt(sys.v[r0 + tid]) : 0.0;
  // exponent bits all ones: infinite or NaN
  auto bad_of = [](double x) { return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000; };
  bool bad = tid < DB && r0 + tid < n && bad_of(sys.v[r0 + tid]);
  for (int c0 = 0; c0 < n; c0 += DTHREADS) {
    __syncthreads();                          // the previous chunk's svc is read
    svc[tid] = c0 + tid < n ? sqrt(sys.v[c0 + tid]) : 0.0;
    __syncthreads();
    const int c = c0 + tid;
    if (c >= n) continue;
    const double sc = svc[tid];
#pragma unroll 4
    for (int rr = 0; rr < DB; ++rr) {
      if (r0 + rr >= n) break;
      const size_t e = size_t(r0 + rr) * n + c;
      const T p = from_c<T>(sys.P[e]);
      if (c > r0 + rr) {
        bad = bad || bad_of(re_(p)) || bad_of(im_(p));
        continue;
      }
      T x = scal(p, -(svr[rr] * sc));
      if (r0 + rr == c) x = add_re(x, 1.0);
      bad = bad || bad_of(re_(x)) || bad_of(im_(x));
      stor(sys.E)[e] = split_ff_t(x);
    }
  }
  if (bad) raise_status(status, ST_ENONFINITE);
}

// step 1 of panel kt: the diagonal block's factor and its inverse D_kt, one CTA per system, in
// float-float. Right-looking over the columns c: with y = 1 / sqrt(pivot), column c of L and row c of
// the inverse Z (which starts as the identity) are scaled by y, then every entry (r, s) below row c
// takes one product: x_rs -= L_rc conj(L_sc) for s > c, Z_rs -= L_rc Z_cs for s <= c. (In FP64, with
// one thread on each pivot and one on each column of the inverse, the two took 57 and about 50 us
// per panel of 128 systems; this takes 34, bound by its serial columns.)
template <typename T>
__global__ void __launch_bounds__(DTHREADS) k_chol_diag(const DieBatchT<T> batch, int kt,
                                                        unsigned* status) {
  using FT = typename FFOf<T>::tile;
  using FA = typename FFOf<T>::acc;
  __shared__ __align__(16) unsigned char raw[2 * DB * DLD * sizeof(FT)];
  FT* SD = reinterpret_cast<FT*>(raw);
  FT* SZ = SD + DB * DLD;
  const DieSysT<T>& sys = batch.s[blockIdx.x];
  const int n = sys.n, nt = (n + DB - 1) / DB;
  if (kt >= nt) return;                      // whole CTA, before any barrier
  const int k0 = kt * DB, kb = min(DB, n - k0), tid = threadIdx.x;
  load_tile_s(SD, stor(sys.E), n, n, n, k0, k0, 1);
  for (int e = tid; e < DB * DB; e += DTHREADS) SZ[(e / DB) * DLD + e % DB] = FT{};
  bool fail = false;
  for (int c = 0; c < kb; ++c) {
    __syncthreads();
    FF d = ff_re(SD[c * DLD + c]);
    if (!(d.h > 0.0f) || !isfinite(d.h)) {   // not positive definite: a pivot of 1
      fail = true;
      d = FF{1.0f, 0.0f};
    }
    const FF y = ff_rsqrt(d);
    __syncthreads();                          // the pivot is read
    if (tid < DB) {
      const int r = tid;
      if (r > c && r < kb) SD[r * DLD + c] = ff_scale(SD[r * DLD + c], y);
      if (r == c) SD[c * DLD + c] = ff_real<FT>(ff_mul(d, y));
    } else if (tid < 2 * DB) {
      const int q = tid - DB;
      if (q < c) SZ[c * DLD + q] = ff_scale(SZ[c * DLD + q], y);
      if (q == c) SZ[c * DLD + c] = ff_real<FT>(y);
    }
    __syncthreads();
    for (int e = tid; e < DB * DB; e += DTHREADS) {
      const int r = e / DB, q = e % DB;
      if (r <= c || r >= kb || q > r) continue;
      FT* x = (q > c ? SD : SZ) + r * DLD + q;
      FA acc = ff_acc(*x);
      const FT l = SD[r * DLD + c];
      if (q > c) ff_csubmul_conj(acc, l, SD[q * DLD + c]);
      else ff_csubmul(acc, l, SZ[c * DLD + q]);
      *x = ff_renorm_t(acc);
    }
  }
  __syncthreads();
  FT* E = stor(sys.E);
  FT* Dr = stor(sys.D) + size_t(kt) * DB * DB;
  for (int e = tid; e < DB * DB; e += DTHREADS) {
    const int r = e / DB, c = e % DB;
    if (r < kb && c <= r) E[size_t(k0 + r) * n + k0 + c] = SD[r * DLD + c];
    Dr[e] = SZ[r * DLD + c];
  }
  if (tid == 0 && fail) raise_status(status, ST_ENOTHPD);
}

// step 2: the panel X L_kk^H = A_ik below the diagonal block, in float-float; one CTA per (32-row
// block, system). A triangular solve in steps of PB = 8 columns, X_s = (A_s - sum_{t<s} X_t L_st^H)
// D_ss^H with the inverse of the 8 x 8 diagonal block of L (a block of D_kt: the inverse of a lower
// triangle has its blocks' inverses on the diagonal). One thread per row and column of a step, so a row
// stays in a quarter of a warp. Errors grow with the condition of the 8 x 8 blocks: with one product
// by the whole D_kt they grew with that of the 32 x 32 block (N_b = 64, condition of
// eps 1e6 / 1e9, mean over 24 matrices: W^c 1.5e-9 / 1.3e-6 off; 9.6e-10 / 7.2e-7 here, 1.0e-9 / 7.7e-7
// by substitution). 128 systems of N_b = 600, 18 panels: 0.91 ms (1.31 with the one product; a row
// per thread substituting one column after the other 4.1).
constexpr int PB = 8;
static_assert(DTHREADS == DB * PB && 32 % PB == 0, "a thread per row and column of a step");
template <typename T>
__global__ void __launch_bounds__(DTHREADS) k_chol_panel(const DieBatchT<T> batch, int kt) {
  using FT = typename FFOf<T>::tile;
  using FA = typename FFOf<T>::acc;
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  FT* SA = reinterpret_cast<FT*>(dsm_raw);   // A, then X
  FT* SL = SA + DB * DLD;                    // L_kk below the diagonal blocks, D_ss in them
  const DieSysT<T>& sys = batch.s[blockIdx.y];
  const int n = sys.n, nt = (n + DB - 1) / DB;
  const int it = kt + 1 + blockIdx.x;
  if (it >= nt) return;                      // whole CTA, before any barrier
  const int k0 = kt * DB;                    // a full block: kt < nt - 1
  FT* E = stor(sys.E);
  load_tile_s(SA, E, n, n, n, it * DB, k0, 0);
  const FT* Dr = stor(sys.D) + size_t(kt) * DB * DB;
  for (int e = threadIdx.x; e < DB * DB; e += DTHREADS) {
    const int r = e / DB, c = e % DB;
    SL[r * DLD + c] = r / PB == c / PB ? Dr[e] : c < r ? E[size_t(k0 + r) * n + k0 + c] : FT{};
  }
  __syncthreads();
  const int tr = threadIdx.x / PB, tc = threadIdx.x % PB;
  FT* row = SA + tr * DLD;
#pragma unroll 1
  for (int s = 0; s < DB; s += PB) {
    const FT* lc = SL + (s + tc) * DLD;
    FA acc = ff_acc(row[s + tc]);
#pragma unroll 4
    for (int k = 0; k < s; ++k) ff_csubmul_conj(acc, row[k], lc[k]);
    row[s + tc] = ff_renorm_t(acc);
    __syncwarp();
    acc = FA{};
#pragma unroll
    for (int k = 0; k < PB; ++k) ff_cmac(acc, row[s + k], ff_conj(lc[s + k]));    // D_ss is lower: zeros beyond
    __syncwarp();
    row[s + tc] = ff_renorm_t(acc);
    __syncwarp();
  }
  __syncthreads();
  for (int e = threadIdx.x; e < DB * DB; e += DTHREADS) {
    const int r = e / DB, c = e % DB;
    if (it * DB + r < n) E[size_t(it * DB + r) * n + k0 + c] = SA[r * DLD + c];
  }
}

// step 3: the trailing update A_ij -= L_ik L_jk^H for kt < j <= i (lower tiles; the diagonal
// tiles keep their lower triangle); grid (tiles of the largest system, system)
template <typename T>
__global__ void __launch_bounds__(DTHREADS) k_chol_update(const DieBatchT<T> batch, int kt, int jend) {
  using FT = typename FFOf<T>::tile;
  using FA = typename FFOf<T>::acc;
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  FT* SA = reinterpret_cast<FT*>(dsm_raw);      // float-float tiles (the size of T)
  FT* SB = SA + DB * DLD;
  const DieSysT<T>& sys = batch.s[blockIdx.y];
  const int n = sys.n, nt = (n + DB - 1) / DB;
  const int m = nt - kt - 1;                 // trailing block rows
  const int64_t t = blockIdx.x;
  int it, jt;
  if (jend < nt) {                           // tile columns kt + 1 .. jend - 1 only
    int u = int(t);
    for (jt = kt + 1; jt < jend && u >= nt - jt; ++jt) u -= nt - jt;
    if (jt >= jend) return;                  // whole CTA, before any barrier
    it = jt + u;
  } else {
    if (m <= 0 || t >= int64_t(m) * (m + 1) / 2) return;   // whole CTA, before any barrier
    // t -> (ii, jj), 0 <= jj <= ii < m, row by row
    int ii = int((sqrt(8.0 * double(t) + 1.0) - 1.0) * 0.5);
    while (int64_t(ii + 1) * (ii + 2) / 2 <= t) ++ii;
    while (int64_t(ii) * (ii + 1) / 2 > t) --ii;
    it = kt + 1 + ii;
    jt = kt + 1 + int(t - int64_t(ii) * (ii + 1) / 2);
  }
  const int k0 = kt * DB;
  const int tid = threadIdx.x, tr = tid >> 3, tc = tid & 7;
  FT* E = stor(sys.E);
  load_tile_s(SA, E, n, n, n, it * DB, k0, 0);                // L_ik
  for (int e = tid; e < DB * DB; e += DTHREADS) {             // SB[k][c] = conj(L_jk[c][k])
    const int k = e / DB, c = e % DB;
    const int R = jt * DB + c;
    SB[k * DLD + c] = R < n ? ff_conj(E[size_t(R) * n + k0 + k]) : FT{};
  }
  __syncthreads();
  FA acc[4] = {};
  tile_mac_ff<false>(acc, SA, SB, tr, tc);
  const int R = it * DB + tr;
  if (R < n) {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int C = jt * DB + tc + 8 * b;
      if (C < n && C <= R) E[size_t(R) * n + C] = ff_sub_acc_t(E[size_t(R) * n + C], acc[b]);
    }
  }
}

template <typename T>
static int launch_cholesky_grid(const DieBatchT<T>& batch, int nsys, int ntmax, cudaStream_t s,
                                const DeviceCtx& ctx) {
  const size_t smem_u = 2 * DB * DLD * sizeof(T);
  int rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_chol_update<T>), smem_u, ctx.device);
  if (!rc) rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_chol_panel<T>), smem_u, ctx.device);
  if (rc) return rc;
  int nmax = 0;
  for (int i = 0; i < nsys; ++i) nmax = std::max(nmax, batch.s[i].n);
  k_eps_fill<T><<<dim3(unsigned((nmax + DB - 1) / DB), unsigned(nsys)), DTHREADS, 0, s>>>(batch,
                                                                                        ctx.status);
  GW_LAUNCH_CHECK("k_eps_fill");
  for (int kt = 0; kt < ntmax; ++kt) {
    k_chol_diag<T><<<unsigned(nsys), DTHREADS, 0, s>>>(batch, kt, ctx.status);
    GW_LAUNCH_CHECK("k_chol_diag");
    const int64_t m = ntmax - kt - 1;
    if (m <= 0) continue;
    k_chol_panel<T><<<dim3(unsigned(m), unsigned(nsys)), DTHREADS, smem_u, s>>>(batch, kt);
    GW_LAUNCH_CHECK("k_chol_panel");
    k_chol_update<T><<<dim3(unsigned(m * (m + 1) / 2), unsigned(nsys)), DTHREADS, smem_u, s>>>(batch, kt, ntmax);
    GW_LAUNCH_CHECK("k_chol_update");
  }
  return GW_OK;
}

// ---- large systems: the products on the tensor cores ------------------------------------------
// The float-float tile products take 52 FP32 operations per complex multiply-add and keep the FP32
// pipe 80 % busy. For larger systems the products run as digit-slice products of 128 x 128 tiles on
// the tensor cores instead (fp64_slices.cuh, k_oz_gemm_cplx: 56 bits below the bound of a row or
// column, against the 48 of the float-float storage below the entry itself): the float-float operands are cut into slices, a launch forms the products
// C1, C2, S of all systems' tiles, and k_dz_combine turns them into W^c or float-float blocks.

// What to slice: blocks of 128 lines (columns of M, or rows with DZ_ROWS) and stages of 32 values
// along each line, of a float-float matrix M (row-major n x n); DZ_LOWER: entries above the
// diagonal count as zero, DZ_CONJ: the conjugate; DZ_FACTOR: rows of the Cholesky factor, whose
// magnitudes mx are bounds that hold for a positive definite eps only. DZ_KUP, DZ_KDOWN: the two
// operands of a product scaled along K by powers of two that cancel: a line's digits end 2^-55 below
// its largest entry, so entries that meet large partners must not be small on their line.
enum : int { DZ_ROWS = 1, DZ_LOWER = 2, DZ_CONJ = 4, DZ_FACTOR = 8, DZ_KUP = 16, DZ_KDOWN = 32 };
struct DzSlice {
  const void* M;            // FFC or FF entries
  char* out;                // (set, block, stage) = (0, 0, 0)
  float* mx;                // bound of |re| + |im| per line (block 0), zeroed before k_dz_max
  int64_t set, blk;         // strides in bytes
  int n, mode;
  int blk0, nblk, st0, nst;
  const float* kscale;      // DZ_KUP / DZ_KDOWN: value k times / over 2^(exponent of kscale[k])
};
constexpr int DZ_MAX = 256;
struct DzSliceBatch {
  DzSlice j[DZ_MAX];
};

__device__ __forceinline__ FFC ff_cplx(FFC x) { return x; }
__device__ __forceinline__ FFC ff_cplx(FF x) { return FFC{x, FF{0.0f, 0.0f}}; }

// entry k of line `line`, or zero outside the matrix (and the triangle)
template <typename FT>
__device__ __forceinline__ FFC dz_entry(const DzSlice& J, int line, int k) {
  const FT* M = static_cast<const FT*>(J.M);
  const bool in = line < J.n && k < J.n &&
                  (!(J.mode & DZ_LOWER) || ((J.mode & DZ_ROWS) ? k <= line : k >= line));
  if (!in) return FFC{};
  return ff_cplx((J.mode & DZ_ROWS) ? M[size_t(line) * J.n + k] : M[size_t(k) * J.n + line]);
}

// the exponent of value k's scale (0 without one)
__device__ __forceinline__ int dz_kexp(const DzSlice& J, int k) {
  if (!(J.mode & (DZ_KUP | DZ_KDOWN)) || k >= J.n) return 0;
  const int e = max(-60, min(60, (int(__float_as_uint(J.kscale[k]) >> 23) & 0xff) - 127));
  return (J.mode & DZ_KUP) ? e : -e;
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// whether values k0 .. k0 + 31 of a block's lines are all above the diagonal (never read)
__device__ __forceinline__ bool dz_empty(const DzSlice& J, int blk, int k0) {
  return (J.mode & DZ_LOWER) && ((J.mode & DZ_ROWS) ? k0 >= (blk + 1) * OT : k0 + OKS <= blk * OT);
}

// bound of |re|, |im| and |re +- im| (the third set of an entry or of its conjugate); NaN stays NaN
__device__ __forceinline__ float dz_mag(FFC x) { return 1.0000005f * (fabsf(x.re.h) + fabsf(x.im.h)); }

// largest magnitude per line, over 128 values: grid (blocks, value chunks, jobs)
template <typename FT>
__global__ void __launch_bounds__(OT) k_dz_max(const __grid_constant__ DzSliceBatch batch) {
  const DzSlice& J = batch.j[blockIdx.z];
  constexpr int SPB = OT / OKS;
  if (int(blockIdx.x) >= J.nblk || int(blockIdx.y) * SPB >= J.nst) return;
  const int line0 = (J.blk0 + blockIdx.x) * OT;
  const int k0 = (J.st0 + int(blockIdx.y) * SPB) * OKS;
  const int k1 = min(k0 + OT, (J.st0 + J.nst) * OKS);
  if (dz_empty(J, J.blk0 + blockIdx.x, (J.mode & DZ_ROWS) ? k0 : k1 - OKS)) return;
  if (J.mode & DZ_ROWS) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < OT; i += OT / 32) {
      float m = 0.0f;
      for (int k = k0 + lane; k < k1; k += 32) m = fmaxf(m, dz_mag(dz_entry<FT>(J, line0 + i, k)) * pow2f(dz_kexp(J, k)));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) atomicMax(reinterpret_cast<int*>(J.mx) + line0 + i, __float_as_int(m));
    }
  } else {
    const int line = line0 + threadIdx.x;
    float m = 0.0f;
    for (int k = k0; k < k1; ++k) m = fmaxf(m, dz_mag(dz_entry<FT>(J, line, k)) * pow2f(dz_kexp(J, k)));
    atomicMax(reinterpret_cast<int*>(J.mx) + line, __float_as_int(m));
  }
}

// The slices: grid (stages, blocks x 4, jobs), four lanes per line. The digits wrap beyond the
// line's exponent (an entry of 8 at a bound of 1 would read as zero), so every entry is compared with
// the bound: a row of the factor beyond sqrt(eps_ii) belongs to an eps that is not positive definite
// (its pivot would be negative), anything else beyond the largest magnitude is not finite.
template <typename FT>
__global__ void __launch_bounds__(OT) k_dz_slice(const __grid_constant__ DzSliceBatch batch,
                                                 unsigned* status) {
  const DzSlice& J = batch.j[blockIdx.z];
  const int b = blockIdx.y >> 2;
  if (int(blockIdx.x) >= J.nst || b >= J.nblk) return;
  const int st = J.st0 + blockIdx.x, kc = threadIdx.x & 3;
  if (dz_empty(J, J.blk0 + b, st * OKS)) return;
  const int n = int(blockIdx.y & 3) * 32 + (threadIdx.x >> 2);
  const int line = (J.blk0 + b) * OT + n, k0 = st * OKS + kc * 8;
  const float mx = J.mx[line], most = fminf(1.0001f * mx, 3.4e38f);
  const int E0 = exponent_of(mx);
  bool bad = false;
  char* out = J.out + (J.blk0 + b) * J.blk + int64_t(st) * OBLK;
  long long xr[8], xi[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const FFC x = dz_entry<FT>(J, line, k0 + k);
    const int e = dz_kexp(J, k0 + k), E = E0 - e;
    bad = bad || !(dz_mag(x) * pow2f(e) <= most);
    xr[k] = fixed_f32(x.re.h, E) + fixed_f32(x.re.l, E);
    if constexpr (sizeof(FT) == sizeof(FFC)) {
      const long long v = fixed_f32(x.im.h, E) + fixed_f32(x.im.l, E);
      xi[k] = (J.mode & DZ_CONJ) ? -v : v;
    }
  }
  if (bad) raise_status(status, (J.mode & DZ_FACTOR) ? ST_ENOTHPD : ST_ENONFINITE);
  uint32_t w[OSL][4];
  fixed_digits8(xr, w);
  store_digits(out, n, kc, w);
  if constexpr (sizeof(FT) == sizeof(FFC)) {
    fixed_digits8(xi, w);
    store_digits(out + J.set, n, kc, w);
#pragma unroll
    for (int k = 0; k < 8; ++k) xi[k] += xr[k];
    fixed_digits8(xi, w);
    store_digits(out + 2 * J.set, n, kc, w);
  }
}

// What becomes of the product tiles out_ab of one problem (rows I of a, columns J of b):
//   DZ_W:    W^c_IJ = sqrt(v_I v_J) (out_IJ - delta_IJ) for I <= J, and its Hermitian mirror
//   DZ_SUB:  M_IJ -= conj(out_IJ) for I >= J
//   DZ_PUT:  M_IJ = conj(out_IJ);  DZ_NEG: M_IJ = -out_IJ
struct DzCombine {
  const float2* G;
  void* M;                  // float-float matrix, row-major n x n
  double2* Wc;
  const double* v;
  int n, nprod, ntile;
  int a0, a1, b0, b1, flags;
};
constexpr int DZC_MAX = 256;
struct DzCombineBatch {
  DzCombine j[DZC_MAX];
};
enum : int { DZ_W, DZ_SUB, DZ_PUT, DZ_NEG };
template <typename FT> __device__ __forceinline__ FT ff_from(FFC x);
template <> __device__ __forceinline__ FFC ff_from<FFC>(FFC x) { return x; }
template <> __device__ __forceinline__ FF ff_from<FF>(FFC x) { return x.re; }

__device__ __forceinline__ FF ff_load(float2 x) { return FF{x.x, x.y}; }

template <typename FT, int WHAT>
__global__ void __launch_bounds__(256) k_dz_combine(const __grid_constant__ DzCombineBatch batch) {
  constexpr bool CPLX = sizeof(FT) == sizeof(FFC);
  const DzCombine& J = batch.j[blockIdx.y];
  const int t = blockIdx.x;
  if (t >= J.ntile) return;                  // whole CTA, before any barrier
  OzC L;
  L.a0 = J.a0;
  L.a1 = J.a1;
  L.b0 = J.b0;
  L.b1 = J.b1;
  L.flags = J.flags;
  int a, b;
  oz_tile(L, t, a, b);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = J.n;
  __shared__ double2 sW[32][33];             // a 32 x 32 block, transposed (FP64 W^c or float-float)
  __shared__ double sv[2][OT];               // square roots of v of the tile's rows and columns
  FFC (*sF)[33] = reinterpret_cast<FFC(*)[33]>(&sW[0][0]);
  if constexpr (WHAT == DZ_W) {
    const int g = (threadIdx.x < OT ? a : b) * OT + (threadIdx.x & (OT - 1));
    sv[threadIdx.x / OT][threadIdx.x & (OT - 1)] = g < n ? sqrt(J.v[g]) : 0.0;
    __syncthreads();
  }
  const size_t pstride = size_t(J.ntile) * OT * OT;
  const float2* G = J.G + size_t(t) * OT * OT;
  for (int s = 0; s < 16; ++s) {
    const int rl = (s & 3) * 32, cl = (s >> 2) * 32, r0 = a * OT + rl, c0 = b * OT + cl;
    if (r0 >= n || c0 >= n) continue;                        // whole CTA
    if (WHAT == DZ_W && r0 > c0 + 31) continue;
    if (WHAT == DZ_SUB && r0 + 31 < c0) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int cc = warp + 8 * i, I = r0 + lane, Jc = c0 + cc;
      const size_t e = size_t(cl + cc) * OT + rl + lane;
      FFC out;
      if constexpr (CPLX) {
        const FF c1 = ff_load(G[e]), c2 = ff_load(G[pstride + e]), ss = ff_load(G[2 * pstride + e]);
        out.re = ff_sub_acc(ff_sub_acc(ss, ff_acc(c1)), ff_acc(c2));
        out.im = ff_sub_acc(c1, ff_acc(c2));
      } else {
        out.re = ff_load(G[e]);
        out.im = FF{0.0f, 0.0f};
      }
      if constexpr (WHAT == DZ_W) {
        double2 x = make_double2(double(out.re.h) + double(out.re.l), 0.0);
        if (CPLX && I != Jc) x.y = double(out.im.h) + double(out.im.l);
        if (I == Jc) x.x -= 1.0;
        const double sc = sv[0][rl + lane] * sv[1][cl + cc];
        x = make_double2(x.x * sc, x.y * sc);
        if (I < n && Jc < n && I <= Jc)
          J.Wc[size_t(Jc) * n + I] = make_double2(x.x, -x.y);   // the mirror, lanes along I
        sW[cc][lane] = x;
      } else {
        sF[cc][lane] = out;
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {                            // lanes along J
      const int rr = warp + 8 * i, Ir = r0 + rr, Jc = c0 + lane;
      if (Ir >= n || Jc >= n) continue;
      if constexpr (WHAT == DZ_W) {
        if (Ir <= Jc) J.Wc[size_t(Ir) * n + Jc] = sW[lane][rr];
      } else {
        const FFC o = sF[lane][rr];
        FT* m = static_cast<FT*>(J.M) + size_t(Ir) * n + Jc;
        if (WHAT == DZ_SUB) {
          if (Ir >= Jc) *m = ff_sub_acc_t(*m, ff_acc(ff_from<FT>(ff_conj(o))));
        } else if (WHAT == DZ_PUT) {
          *m = ff_from<FT>(ff_conj(o));
        } else {
          *m = ff_from<FT>(ff_negate(o));
        }
      }
    }
    __syncthreads();
  }
}

// Systems that take this path, and the slice workspace of one of them. Chunks of systems share a
// launch while their slices stay within DZ_BUDGET. The lines lie where the slices win for many systems
// and lose little for few. Float-float tiles / slices, whole solve of 8, 32 and 128 systems in ms:
//   complex  257: 1.28 / 1.37, 1.69 / 1.94, 4.07 / 3.74    300: 1.54 / 1.53, 2.20 / 2.13, 5.32 / 4.18
//            449: 2.98 / 2.22, 5.33 / 3.47, 14.7 / 8.0     600: 4.62 / 3.11, 9.53 / 5.22, 29.1 / 13.1
//            2048 (2 systems): 40.1 / 10.6
//   real     400: 1.14 / 1.38, 1.54 / 1.80, 3.69 / 3.50    449: 1.41 / 1.53, 1.98 / 1.99, 4.95 / 3.89
//            600: 2.14 / 2.11, 3.34 / 2.91, 9.16 / 6.13    2048 (2 systems): 16.5 / 7.4
// (a real product is a third of a complex one, but its slicing costs half).
constexpr int DZ_MIN_N = 257, DZ_MIN_N_REAL = 449;
constexpr size_t DZ_BUDGET = size_t(6) << 30;
struct DzPlan {
  int nbb, nst, nset, levels, ntile;
  size_t b_x, b_mx, b_g;
  DzPlan(int n, bool cplx) {
    nbb = (n + OT - 1) / OT;
    nst = (n + OKS - 1) / OKS;
    nset = cplx ? 3 : 1;
    levels = 0;
    while ((1 << levels) < nbb) ++levels;
    ntile = oz_tiles(0, nbb, 0, nbb, OZC_UPPER);
    b_x = ws_round(size_t(nset) * nbb * nst * OBLK);            // one operand's slices
    b_mx = size_t(2 + 3 * levels) * nbb * OT * sizeof(float);   // magnitudes: L, Z, per level Z11, T, Z22
    b_g = ws_round(size_t(nset) * ntile * OT * OT * sizeof(float2));
  }
  size_t total() const { return 2 * b_x + b_mx + 256 + b_g; }
  int64_t set() const { return int64_t(nbb) * nst * OBLK; }
  int64_t blk() const { return int64_t(nst) * OBLK; }
};
static bool dz_takes(int n, bool cplx) { return n >= (cplx ? DZ_MIN_N : DZ_MIN_N_REAL); }

// slice workspace of a list of systems: every chunk stays within the budget or is one system
static size_t dz_workspace(const std::vector<int>& ns, bool cplx, int sm) {
  size_t all = 0, one = 0;
  for (int n : ns) {
    const size_t b = DzPlan(n, cplx).total();
    all += b;
    one = std::max(one, b);
  }
  return std::min(all, std::max(one, DZ_BUDGET)) + oz_sum_bytes(sm);
}

template <typename FT>
static int dz_launch_slices(const std::vector<DzSlice>& jobs, cudaStream_t s, const DeviceCtx& ctx,
                            bool find_max) {
  for (size_t j0 = 0; j0 < jobs.size(); j0 += DZ_MAX) {
    const int n = int(std::min<size_t>(DZ_MAX, jobs.size() - j0));
    DzSliceBatch b;
    int nblk = 0, nst = 0;
    for (int i = 0; i < n; ++i) {
      b.j[i] = jobs[j0 + i];
      nblk = std::max(nblk, b.j[i].nblk);
      nst = std::max(nst, b.j[i].nst);
    }
    if (nblk == 0 || nst == 0) continue;
    constexpr int SPB = OT / OKS;
    if (find_max) {
      k_dz_max<FT><<<dim3(unsigned(nblk), unsigned((nst + SPB - 1) / SPB), unsigned(n)), OT, 0, s>>>(b);
      GW_LAUNCH_CHECK("k_dz_max");
    }
    k_dz_slice<FT><<<dim3(unsigned(nst), unsigned(4 * nblk), unsigned(n)), OT, 0, s>>>(b, ctx.status);
    GW_LAUNCH_CHECK("k_dz_slice");
  }
  return GW_OK;
}

template <typename FT, int WHAT>
static int dz_launch_combine(const std::vector<DzCombine>& jobs, cudaStream_t s) {
  for (size_t j0 = 0; j0 < jobs.size(); j0 += DZC_MAX) {
    const int n = int(std::min<size_t>(DZC_MAX, jobs.size() - j0));
    DzCombineBatch b;
    int nt = 0;
    for (int i = 0; i < n; ++i) {
      b.j[i] = jobs[j0 + i];
      nt = std::max(nt, b.j[i].ntile);
    }
    k_dz_combine<FT, WHAT><<<dim3(unsigned(nt), unsigned(n)), 256, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_dz_combine");
  }
  return GW_OK;
}

// Bounds of the rows of L from the diagonal of eps: |L_ik| <= sqrt(eps_ii), and |re| + |im| of a
// complex entry at most sqrt 2 times that. (Close bounds matter: the error of a sum of K digit products is a
// multiple of the product of the two bounds. With 2.01 times the magnitude of the larger part instead,
// N_b = 600 and eigenvalues of eps over six decades, the error of W^c was 1.9e-9 instead of 6.2e-10;
// 5.7e-10 in float-float.)
template <typename FT>
__global__ void k_dz_diag(const __grid_constant__ DzSliceBatch batch) {
  const DzSlice& J = batch.j[blockIdx.y];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float up = sizeof(FT) == sizeof(FFC) ? 1.41422f : 1.00001f;
  if (i < J.n) J.mx[i] = up * sqrtf(fmaxf(ff_re(static_cast<const FT*>(J.M)[size_t(i) * J.n + i]).h, 0.0f));
}

// One chunk of large systems from eps to W^c:
//   Cholesky, left-looking over panels of 128 columns: the panel's rows take the products with all
//     columns before them (slices of L, cut once per panel; rows scaled by sqrt(eps_ii)), then the
//     panel is factorised with the 32-wide float-float steps;
//   Z = L^{-1}: the diagonal 128-blocks in float-float, then doubling: for neighbouring diagonal
//     groups with inverses Z11, Z22 the block below is Z21 = -Z22 (L21 Z11);
//   W^c from Z^H Z.
template <typename T>
struct DzChunk {
  using FT = StorOf<T>;
  static constexpr bool CPLX = sizeof(FT) == sizeof(FFC);
  struct Sys {
    DieSysT<T> S;
    DzPlan p;
    char *X1, *X2;          // slices of row operands (L, then Z22) and column operands (Z11, T, Z)
    float2* G;
    float* mx;              // [2 + 3 levels][128 nbb]
    float* mag(int i) const { return mx + size_t(i) * p.nbb * OT; }
  };
  std::vector<Sys> sys;
  float* ssum;
  cudaStream_t s;
  const DeviceCtx& ctx;

  DzChunk(float* ss, cudaStream_t st, const DeviceCtx& c) : ssum(ss), s(st), ctx(c) {}

  int place(const std::vector<DieSysT<T>>& list, WsCursor cur) {
    size_t mxb = 0;
    for (const DieSysT<T>& S : list) mxb += DzPlan(S.n, CPLX).b_mx;
    float* mx = static_cast<float*>(cur.take(mxb));
    if (!mx) return set_error(GW_EWORKSPACE, "internal: dielectric slice workspace too small");
    GW_CUDA_TRY(cudaMemsetAsync(mx, 0, mxb, s));
    for (const DieSysT<T>& S : list) {
      Sys y{S, DzPlan(S.n, CPLX), nullptr, nullptr, nullptr, mx};
      mx += y.p.b_mx / sizeof(float);
      y.X1 = static_cast<char*>(cur.take(y.p.b_x));
      y.X2 = static_cast<char*>(cur.take(y.p.b_x));
      y.G = static_cast<float2*>(cur.take(y.p.b_g));
      if (!y.X1 || !y.X2 || !y.G)
        return set_error(GW_EWORKSPACE, "internal: dielectric slice workspace too small");
      sys.push_back(y);
    }
    return GW_OK;
  }
  static DzSlice slice(const Sys& y, const T* M, char* out, float* mx, int mode, int blk0, int nblk,
                       int st0, int nst) {
    DzSlice j{};
    j.M = M;
    j.out = out;
    j.mx = mx;
    j.set = y.p.set();
    j.blk = y.p.blk();
    j.n = y.S.n;
    j.mode = mode;
    j.blk0 = blk0;
    j.nblk = nblk;
    j.st0 = st0;
    j.nst = nst;
    j.kscale = y.mag(0);                     // sqrt(eps_kk)
    return j;
  }
  static OzC product(const Sys& y, const char* X, const float* mx, const char* Y, const float* my, int a0,
                     int a1, int b0, int b1, int k0, int k1, int flags) {
    OzC q{};
    q.X = X;
    q.Y = Y;
    q.mx = mx;
    q.my = my;
    q.G = y.G;
    q.xset = q.yset = y.p.set();
    q.xblk = q.yblk = y.p.blk();
    q.a0 = a0;
    q.a1 = a1;
    q.b0 = b0;
    q.b1 = b1;
    q.k0 = k0;
    q.k1 = k1;
    q.flags = flags;
    q.nprod = y.p.nset;
    q.ntile = oz_tiles(a0, a1, b0, b1, flags);
    return q;
  }
  static DzCombine combine(const Sys& y, const OzC& q, T* M) {
    DzCombine c{};
    c.G = q.G;
    c.M = M;
    c.Wc = y.S.Wc;
    c.v = y.S.v;
    c.n = y.S.n;
    c.nprod = q.nprod;
    c.ntile = q.ntile;
    c.a0 = q.a0;
    c.a1 = q.a1;
    c.b0 = q.b0;
    c.b1 = q.b1;
    c.flags = q.flags;
    return c;
  }
  template <int WHAT>
  int run(const std::vector<OzC>& pr, const std::vector<DzCombine>& cb) {
    if (pr.empty()) return GW_OK;
    int rc = oz_cplx(pr.data(), int(pr.size()), ssum, s, ctx);
    return rc ? rc : dz_launch_combine<FT, WHAT>(cb, s);
  }

  static constexpr int SPB = OT / OKS;       // stages per 128-block
  static constexpr int TPB = OT / DB;        // 32-blocks per 128-block

  int cholesky(const DieBatchT<T>& batch, int ntmax) {
    const unsigned nsys = unsigned(sys.size());
    const size_t smem_u = 2 * DB * DLD * sizeof(T);
    int nmax = 0, nbbmax = 0;
    std::vector<DzSlice> dg;
    for (const Sys& y : sys) {
      nmax = std::max(nmax, y.S.n);
      nbbmax = std::max(nbbmax, y.p.nbb);
      dg.push_back(slice(y, y.S.E, nullptr, y.mag(0), 0, 0, 0, 0, 0));
    }
    k_eps_fill<T><<<dim3(unsigned((nmax + DB - 1) / DB), nsys), DTHREADS, 0, s>>>(batch, ctx.status);
    GW_LAUNCH_CHECK("k_eps_fill");
    for (size_t j0 = 0; j0 < dg.size(); j0 += DZ_MAX) {
      const unsigned n = unsigned(std::min<size_t>(DZ_MAX, dg.size() - j0));
      DzSliceBatch b;
      std::copy(dg.begin() + j0, dg.begin() + j0 + n, b.j);
      k_dz_diag<FT><<<dim3(unsigned((nmax + 127) / 128), n), 128, 0, s>>>(b);
      GW_LAUNCH_CHECK("k_dz_diag");
    }
    for (int kb = 0; kb < nbbmax; ++kb) {
      std::vector<OzC> pr;
      std::vector<DzCombine> cb;
      std::vector<DzSlice> sl;
      for (const Sys& y : sys) {
        if (kb > 0 && kb < y.p.nbb) {
          pr.push_back(product(y, y.X1, y.mag(0), y.X1, y.mag(0), kb, y.p.nbb, kb, kb + 1, 0, SPB * kb, 0));
          cb.push_back(combine(y, pr.back(), y.S.E));
        }
        if (kb + 1 < y.p.nbb)
          sl.push_back(slice(y, y.S.E, y.X1, y.mag(0), DZ_ROWS | DZ_FACTOR,
                             kb + 1, y.p.nbb - kb - 1, SPB * kb, SPB));
      }
      int rc = run<DZ_SUB>(pr, cb);
      if (rc) return rc;
      for (int kt = TPB * kb; kt < std::min(ntmax, TPB * (kb + 1)); ++kt) {
        k_chol_diag<T><<<nsys, DTHREADS, 0, s>>>(batch, kt, ctx.status);
        GW_LAUNCH_CHECK("k_chol_diag");
        const int m = ntmax - kt - 1;
        if (m <= 0) continue;
        k_chol_panel<T><<<dim3(unsigned(m), nsys), DTHREADS, smem_u, s>>>(batch, kt);
        GW_LAUNCH_CHECK("k_chol_panel");
        const int jend = TPB * (kb + 1);
        int64_t tiles = 0;
        for (int jt = kt + 1; jt < std::min(jend, ntmax); ++jt) tiles += ntmax - jt;
        if (tiles == 0) continue;
        k_chol_update<T><<<dim3(unsigned(tiles), nsys), DTHREADS, smem_u, s>>>(batch, kt, jend);
        GW_LAUNCH_CHECK("k_chol_update");
      }
      if ((rc = dz_launch_slices<FT>(sl, s, ctx, false))) return rc;
    }
    return GW_OK;
  }

  // Z from the inverses of its diagonal 128-blocks
  int inverse() {
    int lmax = 0;
    for (const Sys& y : sys) lmax = std::max(lmax, y.p.levels);
    for (int l = 0; l < lmax; ++l) {
      const int g = 1 << l;
      std::vector<DzSlice> s1, s2;
      std::vector<OzC> p1, p2;
      std::vector<DzCombine> c1, c2;
      for (const Sys& y : sys) {
        if (l >= y.p.levels) continue;
        float *m11 = y.mag(2 + 3 * l), *mt = y.mag(3 + 3 * l), *m22 = y.mag(4 + 3 * l);
        int tile0 = 0;
        for (int j = 0; j + g < y.p.nbb; j += 2 * g) {
          const int e = std::min(j + 2 * g, y.p.nbb), h = j + g;   // groups [j, h) and [h, e)
          const int ks1 = SPB * h, ks2 = std::min(SPB * e, y.p.nst);
          // conj(L21 Z11) from L and conj(Z11); T = L21 Z11 goes where Z21 will be
          s1.push_back(slice(y, y.S.Z, y.X2, m11, DZ_LOWER | DZ_CONJ, j, g, SPB * j, ks1 - SPB * j));
          OzC q = product(y, y.X1, y.mag(0), y.X2, m11, h, e, j, h, SPB * j, ks1, OZC_KB);
          q.G += size_t(tile0) * q.nprod * OT * OT;
          p1.push_back(q);
          c1.push_back(combine(y, q, y.S.Z));
          // -Z22 T from conj(Z22) and T, scaled along K to unit diagonal of eps: T has the size of
          // the rows of L, Z22 that of their reciprocals (with eps_ii over 6 decades, N = 600, the
          // error of W^c against 80 bits was 3e-10 without it, 1e-13 with it)
          s2.push_back(slice(y, y.S.Z, y.X2, mt, DZ_KDOWN, j, g, ks1, ks2 - ks1));
          s2.push_back(slice(y, y.S.Z, y.X1, m22, DZ_ROWS | DZ_LOWER | DZ_CONJ | DZ_KUP, h, e - h, ks1,
                             ks2 - ks1));
          q = product(y, y.X1, m22, y.X2, mt, h, e, j, h, ks1, ks2, OZC_KTOP);
          q.G += size_t(tile0) * q.nprod * OT * OT;
          p2.push_back(q);
          c2.push_back(combine(y, q, y.S.Z));
          tile0 += q.ntile;
        }
      }
      int rc = dz_launch_slices<FT>(s1, s, ctx, true);
      if (!rc) rc = run<DZ_PUT>(p1, c1);
      if (!rc) rc = dz_launch_slices<FT>(s2, s, ctx, true);
      if (!rc) rc = run<DZ_NEG>(p2, c2);
      if (rc) return rc;
    }
    return GW_OK;
  }

  int screened() {
    std::vector<DzSlice> sl;
    std::vector<OzC> pr;
    std::vector<DzCombine> cb;
    for (const Sys& y : sys) {
      sl.push_back(slice(y, y.S.Z, y.X2, y.mag(1), DZ_LOWER, 0, y.p.nbb, 0, y.p.nst));
      pr.push_back(product(y, y.X2, y.mag(1), y.X2, y.mag(1), 0, y.p.nbb, 0, y.p.nbb, 0, y.p.nst,
                           OZC_UPPER | OZC_KA | OZC_KB));
      cb.push_back(combine(y, pr.back(), nullptr));
    }
    int rc = dz_launch_slices<FT>(sl, s, ctx, true);
    return rc ? rc : run<DZ_W>(pr, cb);
  }
};

// dz: the slice workspace (caller-workspace entry points); ssum: the slice products' scratch
template <typename T>
static int launch_dielectric(std::vector<DieSysT<T>>& sys, WsCursor dz, float* ssum, cudaStream_t s,
                             const DeviceCtx& ctx) {
  const size_t smem = 3 * DB * DLD * sizeof(T);
  const size_t smem_w = 2 * DB * DLD * sizeof(T);
  {
    int rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_dielectric<T>), smem, ctx.device);
    if (!rc) rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_dielectric_w<T, true>), smem_w, ctx.device);
    if (!rc) rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_dielectric_w<T, false>), smem_w, ctx.device);
    if (!rc) rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_dielectric_zcol<T>), smem_w, ctx.device);
    if (!rc) rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_chol_update<T>), smem_w, ctx.device);
    if (!rc) rc = set_max_dyn_smem(reinterpret_cast<const void*>(k_chol_panel<T>), smem_w, ctx.device);
    if (rc) return rc;
  }
  constexpr bool CPLX = sizeof(T) == sizeof(double2);
  const bool by_columns = !sys.empty() && sys[0].D != nullptr;
  // a caller's workspace without room for the slices (of all, or of large systems): float-float
  const size_t room = ssum ? dz.size - std::min(dz.size, (dz.used + 255) & ~size_t(255)) : 0;
  auto sliced_path = [&](const DieSysT<T>& S) {
    return dz_takes(S.n, CPLX) && DzPlan(S.n, CPLX).total() <= room;
  };
  // The systems of the sliced path behind the others, whatever the order of the sizes in the call: a
  // batch is of one kind, and sizes that alternate around the limit would make a batch (a chain of
  // three launches per 32 columns) per q: 8 q of 250 and 260 in turn, 16 frequencies, 10.4 -> 4.6 ms.
  if (by_columns)
    std::stable_partition(sys.begin(), sys.end(),
                          [&](const DieSysT<T>& S) { return !sliced_path(S); });
  for (size_t b0 = 0; b0 < sys.size();) {
    // up to DMAXSYS systems; those of the sliced path apart from the others, within the slice budget
    const bool sliced = by_columns && sliced_path(sys[b0]);
    size_t nb_ = 0, bytes = 0;
    DieBatchT<T> batch;
    int ntmax = 1;
    while (b0 + nb_ < sys.size() && nb_ < DMAXSYS) {
      const DieSysT<T>& S = sys[b0 + nb_];
      if (by_columns && sliced_path(S) != sliced) break;
      if (sliced) {
        const size_t need = DzPlan(S.n, CPLX).total();
        if (nb_ > 0 && bytes + need > std::min(DZ_BUDGET, room)) break;
        bytes += need;
      }
      batch.s[nb_++] = S;
      ntmax = std::max(ntmax, (S.n + DB - 1) / DB);
    }
    const dim3 g2(static_cast<unsigned>(nb_), static_cast<unsigned>(ntmax));
    if (sliced) {
      DzChunk<T> c(ssum, s, ctx);
      int rc = c.place(std::vector<DieSysT<T>>(sys.begin() + b0, sys.begin() + b0 + nb_), dz);
      if (!rc) rc = c.cholesky(batch, ntmax);
      if (rc) return rc;
      k_dielectric_zcol<T><<<g2, DTHREADS, smem_w, s>>>(batch, DzChunk<T>::TPB);
      GW_LAUNCH_CHECK("k_dielectric_zcol");
      rc = c.inverse();
      if (!rc) rc = c.screened();
      if (rc) return rc;
    } else if (by_columns) {
      // caller workspace: the factorisation over many CTAs, then the inverse by block columns
      int rc = launch_cholesky_grid<T>(batch, int(nb_), ntmax, s, ctx);
      if (rc) return rc;
      k_dielectric_zcol<T><<<g2, DTHREADS, smem_w, s>>>(batch, 0);
      GW_LAUNCH_CHECK("k_dielectric_zcol");
      k_dielectric_w<T, true><<<g2, DTHREADS, smem_w, s>>>(batch);
    } else {
      // no-allocation entry: factorisation and inverse inside one CTA per system
      k_dielectric<T><<<unsigned(nb_), DTHREADS, smem, s>>>(batch, ctx.status);
      GW_LAUNCH_CHECK("k_dielectric");
      k_dielectric_w<T, false><<<g2, DTHREADS, smem_w, s>>>(batch);
    }
    GW_LAUNCH_CHECK("k_dielectric_w");
    b0 += nb_;
  }
  return GW_OK;
}

// E, Z, D of every system (what a call needs), and the slices of large ones
template <typename T>
static size_t dielectric_ws_t(int nq, const int* nb, int nw, bool slices) {
  size_t b = 0;
  std::vector<int> large;
  for (int q = 0; q < nq; ++q) {
    size_t n = size_t(nb[q]);
    const size_t nt = (n + DB - 1) / DB;
    b += size_t(nw) * ws_round((2 * n * n + nt * DB * DB) * sizeof(T));
    if (slices && dz_takes(nb[q], sizeof(T) == sizeof(double2))) large.insert(large.end(), nw, nb[q]);
  }
  if (large.empty()) return b;
  int sm = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
  cudaGetLastError();
  return b + dz_workspace(large, sizeof(T) == sizeof(double2), sm);
}

template <typename T>
static int dielectric_t(int nq, const int* nb, int nw, const double* const* v,
                        const double* const* P, double* const* Wc, void* ws, size_t ws_bytes,
                        cudaStream_t s, const DeviceCtx& ctx) {
  WsCursor cur{static_cast<char*>(ws), ws_bytes, 0};
  std::vector<DieSysT<T>> sys;
  for (int q = 0; q < nq; ++q) {
    size_t n = size_t(nb[q]);
    for (int j = 0; j < nw; ++j) {
      DieSysT<T> d;
      d.P = reinterpret_cast<const double2*>(P[q]) + size_t(j) * n * n;
      d.Wc = reinterpret_cast<double2*>(Wc[q]) + size_t(j) * n * n;
      d.v = v[q];
      const size_t nt = (n + DB - 1) / DB;
      char* blk = static_cast<char*>(cur.take((2 * n * n + nt * DB * DB) * sizeof(T)));
      if (!blk) return set_error(GW_EWORKSPACE, "internal: dielectric workspace too small");
      d.E = reinterpret_cast<T*>(blk);       // eps, then its Cholesky factor
      d.Tp = nullptr;                         // (the in-CTA inverse's panel: not used here)
      d.Z = d.E + n * n;                      // the inverse factor, by block columns
      d.D = d.Z + n * n;                      // the inverted diagonal blocks
      d.n = int(n);
      sys.push_back(d);
    }
  }
  float* ssum = nullptr;
  bool large = false;
  for (int q = 0; q < nq; ++q) large = large || dz_takes(nb[q], sizeof(T) == sizeof(double2));
  if (large) ssum = static_cast<float*>(cur.take(oz_sum_bytes(ctx.sm_count)));    // NULL: no room for slices
  return launch_dielectric<T>(sys, cur, ssum, s, ctx);
}

size_t dielectric_workspace(int nq, const int* nb, int nw, bool slices) {
  return dielectric_ws_t<double2>(nq, nb, nw, slices);
}
size_t dielectric_real_workspace(int nq, const int* nb, int nw, bool slices) {
  return dielectric_ws_t<double>(nq, nb, nw, slices);
}

int dielectric_wc(int nq, const int* nb, int nw, const double* const* v, const double* const* P,
                  double* const* Wc, void* ws, size_t ws_bytes, cudaStream_t s,
                  const DeviceCtx& ctx) {
  return dielectric_t<double2>(nq, nb, nw, v, P, Wc, ws, ws_bytes, s, ctx);
}

int dielectric_wc_real(int nq, const int* nb, int nw, const double* const* v,
                       const double* const* P, double* const* Wc, void* ws, size_t ws_bytes,
                       cudaStream_t s, const DeviceCtx& ctx) {
  return dielectric_t<double>(nq, nb, nw, v, P, Wc, ws, ws_bytes, s, ctx);
}

// ---------------------------------------------------------------- no-alloc variant
// Scratch for callers that cannot allocate: a static device array (one per device that
// loads the library). Host code only ever uses the device address looked up below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[GW_NOALLOC_SCRATCH_BYTES];
static std::mutex g_noalloc_mu;
static char* g_noalloc_ptr[64];

static int noalloc_scratch(const DeviceCtx& ctx, char** out) {
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[ctx.device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    g_noalloc_ptr[ctx.device] = static_cast<char*>(p);
  }
  *out = g_noalloc_ptr[ctx.device];
  return GW_OK;
}

int dielectric_wc_noalloc(int nb, int nw, const double* v, const double* P, double* Wc,
                          cudaStream_t s, const DeviceCtx& ctx) {
  const size_t n = size_t(nb);
  const size_t per = ws_round((n * n + n * DB) * sizeof(double2));
  if (per > GW_NOALLOC_SCRATCH_BYTES)
    return set_error(GW_EINVAL, "nb=%d needs %zu bytes of scratch per system, more than the "
                     "%u-byte static scratch of the no-alloc entry point", nb, per,
                     GW_NOALLOC_SCRATCH_BYTES);
  char* base = nullptr;
  int rc = noalloc_scratch(ctx, &base);
  if (rc) return rc;
  const size_t fit = std::min<size_t>(GW_NOALLOC_SCRATCH_BYTES / per, DMAXSYS);
  for (int j0 = 0; j0 < nw; j0 += int(fit)) {
    const int cnt = std::min<int>(int(fit), nw - j0);
    std::vector<DieSysT<double2>> sys(cnt);
    for (int i = 0; i < cnt; ++i) {
      DieSysT<double2>& d = sys[i];
      const int j = j0 + i;
      d.P = reinterpret_cast<const double2*>(P) + size_t(j) * n * n;
      d.Wc = reinterpret_cast<double2*>(Wc) + size_t(j) * n * n;
      d.v = v;
      d.E = reinterpret_cast<double2*>(base + size_t(i) * per);
      d.Tp = d.E + n * n;
      d.Z = d.E;                              // inverse in place, inside the CTA
      d.D = nullptr;
      d.n = nb;
    }
    rc = launch_dielectric<double2>(sys, WsCursor{nullptr, 0, 0}, nullptr, s, ctx);
    if (rc) return rc;
  }
  return GW_OK;
}

}  // namespace gw
