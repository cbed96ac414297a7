// Digit slices of FP64 and float-float operands (the layout that k_oz_gemm of fp64_tc.cu reads): per
// block of 128 rows (or columns) and stage of 32 K values, seven 8 KB tiles of BF16 digits.
#pragma once
#include "gw_internal.cuh"
#include "tc_ptx.cuh"

namespace gw {

constexpr int OT = 128;                     // tile edge
constexpr int OKS = 32;                     // K per stage
constexpr int OSL = 7;                      // digit slices
constexpr int SLB = OT * 64;                // one slice of one operand and stage: 8 KB
constexpr int NHI = 4;                      // slices 1-4: the stage's first part
constexpr int HIB = NHI * SLB, LOB = (OSL - NHI) * SLB;   // bytes of the parts, per operand
constexpr int OBLK = HIB + LOB;             // one operand's stage
constexpr int OSTAGE = 2 * OBLK;            // A 1-4, B 1-4, A 5-7, B 5-7

__device__ __forceinline__ uint32_t swz64(int n, int kc) {
  return uint32_t((n >> 3) * 512 + (n & 7) * 64 + ((kc ^ ((n & 7) >> 1)) << 4));
}

// Digits of 8 consecutive K values in fixed point, |X| < 0.996 2^55: for every slice 8 BF16 values
// d_i 256^(1-i), packed in K order. X plus the bias 128 sum 256^k has the digits (plus 128) as its
// bytes; a byte put into the low mantissa bits of a float of the slice's exponent, minus that
// float with the byte at 128, is the digit's value. Integer arithmetic throughout: the FP64
// pipe would take as long as the products.
__device__ __forceinline__ void fixed_digits8(const long long (&X)[8], uint32_t (&w)[OSL][4]) {
  constexpr unsigned long long BIAS = 128ull * (((1ull << 56) - 1) / 255);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    float f[2][OSL];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned long long y = BIAS + static_cast<unsigned long long>(X[2 * p + h]);
      const uint32_t lo = uint32_t(y), hi = uint32_t(y >> 32);
#pragma unroll
      for (int i = 0; i < OSL; ++i) {
        const uint32_t mg = 0x4B000000u - (uint32_t(8 * i) << 23);
        // byte 6 - i of y in place of mg's lowest byte
        const uint32_t bits = i < 3 ? __byte_perm(hi, mg, 0x7650u | uint32_t(2 - i))
                                    : __byte_perm(lo, mg, 0x7650u | uint32_t(6 - i));
        f[h][i] = __fsub_rn(__uint_as_float(bits), __uint_as_float(mg | 128u));
      }
    }
#pragma unroll
    for (int i = 0; i < OSL; ++i) w[i][p] = tc::cvt_bf16x2(f[0][i], f[1][i]);
  }
}

// round(v 2^(55-E)) of an FP64 value |v| < 2^E, and of an FP32 one
__device__ __forceinline__ long long fixed_f64(double v, int E) {
  const unsigned long long b = __double_as_longlong(v);
  const int ex = int(b >> 52) & 0x7ff;
  const int sh = min(E + 1022 - ex, 60);
  unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 2;
  // sh >= 0 by the choice of E; below the last digit (and for zero): zero
  m = ex == 0 ? 0ull : (m + ((1ull << sh) >> 1)) >> sh;
  return (b >> 63) ? -static_cast<long long>(m) : static_cast<long long>(m);
}
__device__ __forceinline__ long long fixed_f32(float v, int E) {
  const uint32_t b = __float_as_uint(v);
  const int ex = int(b >> 23) & 0xff;
  const int sh = ex - 95 - E;                 // 2^(ex - 150) in units of 2^(E - 55); at most 31
  const unsigned long long m = (b & 0x7fffffu) | 0x800000u;
  const int r = min(max(-sh, 0), 40);
  const unsigned long long f = ex == 0 ? 0ull : sh >= 0 ? m << min(sh, 38) : (m + ((1ull << r) >> 1)) >> r;
  return (b >> 31) ? -static_cast<long long>(f) : static_cast<long long>(f);
}

// digits of 8 FP64 values with exponent E (|v| < 0.996 2^E)
__device__ __forceinline__ void digits8(const double (&v)[8], int E, uint32_t (&w)[OSL][4]) {
  long long X[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) X[k] = fixed_f64(v[k], E);
  fixed_digits8(X, w);
}

// the same with an exponent per value (the line's E less the exponent of the value's own scale)
__device__ __forceinline__ void digits8(const double (&v)[8], const int (&E)[8], uint32_t (&w)[OSL][4]) {
  long long X[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) X[k] = fixed_f64(v[k], E[k]);
  fixed_digits8(X, w);
}

// 16 bytes of every slice of row n at K chunk kc of a stage's block
__device__ __forceinline__ void store_digits(char* blk, int n, int kc, const uint32_t (&w)[OSL][4]) {
  const uint32_t off = swz64(n, kc);
#pragma unroll
  for (int i = 0; i < OSL; ++i)
    *reinterpret_cast<uint4*>(blk + i * SLB + off) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// E with 1.005 m < 2^E for an FP32 magnitude m (zero, and what is below the normal range: -126)
__device__ __forceinline__ int exponent_of(float m) {
  return (int(__float_as_uint(1.005f * m) >> 23) & 0xff) - 126;
}

// ---- complex products of sliced operands (fp64_tc.cu, k_oz_gemm_cplx) ------------------------------
// out_ab = sum_k conj(X_ka) Y_kb for tiles (a, b) of 128 x 128, from the slices of the real parts (set
// 0), the imaginary parts (set 1) and their sums (set 2): the products C1 = Xr Yi, C2 = Xi Yr,
// S = Xs Ys give Re out = S - C1 - C2, Im out = C1 - C2. Real operands: set 0 only, one product.
// Every product tile goes to G as float-float pairs, [product][tile][column][row].
enum : int { OZC_UPPER = 1, OZC_KA = 2, OZC_KB = 4, OZC_KTOP = 8 };
struct OzC {
  const char* X;            // slices: set, block and stage (0, 0, 0); strides in bytes
  const char* Y;
  const float* mx;          // bound of the magnitudes of all sets per row of X, column of Y (block 0)
  const float* my;
  float2* G;
  int64_t xset, xblk, yset, yblk;
  int a0, a1, b0, b1;       // tiles: a0 <= a < a1 (OZC_UPPER: and a <= b), b0 <= b < b1
  int k0, k1;               // stages; with OZC_KA / _KB from 4 a / 4 b on, with OZC_KTOP up to 4 (a + 1)
  int flags;
  int nprod;                // 3, or 1 for real operands
  int ntile;                // oz_tiles of the above
};
constexpr int OZC_MAX = 192;   // problems per launch

__host__ __device__ inline int oz_tiles(int a0, int a1, int b0, int b1, int flags) {
  int n = 0;
  for (int b = b0; b < b1; ++b) {
    const int top = (flags & OZC_UPPER) && b + 1 < a1 ? b + 1 : a1;
    n += top > a0 ? top - a0 : 0;
  }
  return n;
}
// tile t -> (a, b)
__host__ __device__ inline void oz_tile(const OzC& L, int t, int& a, int& b) {
  for (b = L.b0; b < L.b1; ++b) {
    const int top = (L.flags & OZC_UPPER) && b + 1 < L.a1 ? b + 1 : L.a1;
    const int n = top > L.a0 ? top - L.a0 : 0;
    if (t < n) break;
    t -= n;
  }
  a = L.a0 + t;
}
size_t oz_sum_bytes(int sm);
// the products of `n` problems; s: oz_sum_bytes of scratch
int oz_cplx(const OzC* probs, int n, float* s, cudaStream_t st, const DeviceCtx& ctx);

}  // namespace gw
