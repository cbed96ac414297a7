// FP64 products on the tensor cores: the polarization (a2) and the pair coefficients (a5) of the
// FP64 precision, as error-free sliced products (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms
// 59, 2012).
//
// GB300 executes FP64 multiply-adds at 1/64 of its FP32 rate (1.17 TFLOP/s measured), so the
// plain FP64 kernels are bound by that pipe whatever their data movement. Here every FP64
// operand x of a column (of A or B) and K range (superblock) with |x| < 2^E becomes a 56-bit
// fixed-point integer cut into seven signed 8-bit digits, x = 2^(E-7) sum_i d_i 256^(1-i), each
// digit exact in BF16. A product x y is the sum of the 28 digit products with i + j <= 8 (what is
// left out is near 2^-56 of the largest product of the range); products of equal i + j = g form
// one group:
//   g = 2 .. 5 (g - 1 digit pairs): integer multiples of 256^(2-g), summed exactly by the FP32
//     accumulators of the tensor core while pairs x K x 2^14 <= 2^24: 32, 16, 8 and 8 stages of
//     K = 32 between drains (g = 5 is drained every 2, see below);
//   g = 6, 7, 8 (18 pairs, "low") together in one accumulator, 2^-32 below the leading group: their
//     truncating FP32 chain stays near 2^-50 of the product of the two bounds, where FP64 sums of evenly
//     distributed entries round as well. Uneven ones lie below their bounds and would lose: for them
//     the kernels ..6 sum g = 6 by itself (exactly) and take g = 9 as well (a quarter more time).
//     The complex products of the dielectric always do:
//     the entries of a Cholesky factor are far below the bound of their row, and both the truncation
//     and what is left out count against that bound, K^1/2 times. 4,096 basis functions, eigenvalues
//     of eps over six decades, error of eps^-1: 7.1e-9 without the exact g = 6, 3.7e-9 without g = 9,
//     3.1e-10 with both, 1.1e-9 in float-float; 128 systems of N_b = 600 12.34 -> 13.49 ms.
// The epilogue keeps three FP32 sums per element, s (groups 2-4), c (exact rounding errors of s,
// and group 5) and d (exact rounding errors of c, and the low groups), by two-sums, so nothing
// above 2^-24 of the low groups is lost; a superblock's result (s + c) + d goes to FP64 with the
// power of two of its row and column exponents.
//
// Measured: one q of K = 102,400, N_b = 600, 2 frequencies 314 ms (FP64 kernel, 0.94 TFLOP/s) ->
// 7.2 ms (41 TFLOP/s FP64-equivalent): k_oz_gemm 5.8 ms, slices 1.05, scales 0.25; relative error of
// P against 64-bit sums 1.1e-15 -> 5e-16. K = 896, N_b = 64, 8 frequencies 3.7 -> 0.14 ms. The MMAs
// take about 85 cycles instead of 64 (both operands from shared memory) and set the pace. Pair
// coefficients of 6,656 pairs, N_b = 600, 16 frequencies: 262 -> 5.8 ms (k_oz_gemm 5.5 ms).
//
// What an input may contain: the scale kernels see every operand first. A non-finite value, one
// outside [2^-100, 2^100], weights outside the FP32 range that count, a column of the polarization whose
// largest entry exceeds 1024 times its mean magnitude, or a pair whose digits would be off by more than
// FP64 sums (k_oz_pair_guard) set a bit of a device flag: the sliced kernels then return at once and
// the FP64 kernel, launched behind them and otherwise empty, does the work. A second bit sends uneven
// operands (k_oz_exps, k_oz_pair_guard) to the GEMM with the exact g = 6. The polarization's guards
// look at columns one by one: its errors are those of FP64 sums relative to sqrt(P_II P_JJ), not to
// an element that is small because its columns are large in different rows.
//
// Layout and roles of k_oz_gemm_* (384 threads, one persistent CTA per SM): 128 x 128 tiles; per stage
// (K = 32) 7 slices of A and of B, pre-split in global memory as 8 KB K-major, 64-byte-swizzled
// tiles, copied by bulk async copies into two shared-memory stages of 112 KB, each in two parts
// (slices 1-4 and 5-7). One warp issues the MMAs (both operands from shared memory). TMEM holds four
// accumulators (512 columns): C4, C3, C2 for the groups 4, 3, 2 and D, which alternates between
// the low groups and group 5 so that each is drained while C's MMAs run:
//   even stage: g4; low, drain; g3, g2; g5
//   odd stage:  g5 (continuing), drain; g4, g3, g2 (drains due every 8 stages); low, drain
// (with an exact g6, that follows low in D: five drains of D per two stages instead of three)
// (low starts afresh in every stage, its smallest products first: continuing it over a second
// stage adds 26 truncating MMAs to a large accumulator and cost 3x the error of P)
// Eight epilogue warps drain (two per lane quadrant, 64 columns each).
#include <algorithm>
#include <vector>

#include "gw_internal.cuh"
#include "fp64_slices.cuh"
#include "fp64_tc.cuh"
#include "tc_ptx.cuh"

namespace gw {
namespace {

constexpr int ONST = 2;                     // stages in shared memory
constexpr int SBMAX = 256;                  // stages per superblock at most (K = 8192)
constexpr int OTHREADS = 384;
constexpr int EPI_WARPS = 8;
constexpr int REG_E = 232, REG_P = 40;      // 256 x 232 + 128 x 40 = 384 x 168
static_assert(256 * REG_E + 128 * REG_P == OTHREADS * 168, "register split");
constexpr uint64_t OWAIT = 2000000000ull;   // ns per bounded wait
constexpr int CHROWS = 64;                  // rows per scale chunk (superblocks are multiples)
constexpr float RATIO_MAX = 1024.0f;        // largest entry against the mean magnitude of a column

// bits of a problem's flag: the FP64 kernel does it; the GEMM with an exact group 6 does it
enum : int { FLAG_FP64 = 1, FLAG_EXACT6 = 2 };

// One problem: a q point's polarization over a range of rows and frequencies, or (QF) the pair
// coefficients of a range of pairs and frequencies.
struct OzProb {
  // inputs
  const double2* M;         // polarization: the pass's first row
  const double* delta;      // ... of the whole q (Kall entries), with dbar and f or NULL
  const double* dbar;
  const double* f;
  double* w;                // s_tj [nw][Kall]; wp: of the pass's first row and frequency
  const double* wp;
  const double* x;          // QF: rows of the real operand [nrow][ncol]
  int* flag;                // FLAG_*: what else does this problem
  int* spread;              // polarization: largest spreads of the columns of A and of B (FP32 bits)
  // workspace
  float2* part;             // scale partials
  int* EA;                  // exponents [operand block][superblock][128]
  int* EB;
  int* eq;                  // QF: exponents of the basis functions' scales
  float2* cols;             // QF: largest magnitude and |diagonal| per column of the scaled U [f][128 nbj]
  char* A;                  // slices: [f (polarization)][block][stage][56 KB]
  char* B;                  // [f (QF)][block][stage][56 KB]
  double* G;                // polarization: [split][f][C, S][nbp][nbp], transposed tiles
  double* cpart;            // QF: [f][2 nbj][nrow]
  double2* P;               // polarization: the pass's first frequency
  int64_t Kall, K;          // rows of the q, rows of the pass
  int64_t nrow, ncol;       // QF
  int nb, nf;
  int nst, nsb, sbst;       // stages, superblocks, stages per superblock
  int sps, splits;          // superblocks per split, splits
  int nbi, nbj;             // QF: row and column blocks; polarization: nbj = ceil(N_b / 128)
  int ntile;
};
constexpr int OZQ = 16;     // problems per launch
struct OzBatch {
  OzProb q[OZQ];
  int64_t item0[OZQ + 1];
  float* s;                 // per CTA: the sums s of its tile, [column][row]
  int nq;
  int add;                  // G += instead of G =
};
struct OzCBatch {
  OzC q[OZC_MAX];
  int item0[OZC_MAX + 1];
  float* s;
  int nq;
};
static_assert(sizeof(OzCBatch) < 32000, "kernel parameter space");

// k_oz_gemm's modes: polarization, quadratic form, complex products
enum : int { OZ_POL, OZ_QUAD, OZ_CPLX };
template <int MODE> struct OzBatchOf { using B = OzBatch; using P = OzProb; };
template <> struct OzBatchOf<OZ_CPLX> { using B = OzCBatch; using P = OzC; };

// One work item: its problem, operand slices (stage 0), stage range, stages per superblock, and the
// indexes that its output needs.
template <int MODE>
struct OzItem {
  const typename OzBatchOf<MODE>::P* L;
  const char *a, *b;
  int st0, st1, sbst;
  int f, sp, bi, bj, kind;
};

// polarization: tiles of C = Mr^T D Mi (all) and S = (Mr+Mi)^T D (Mr+Mi) (upper), the layout of the
// split-precision polarization; quadratic form: every (row block, column block), whose column block
// bj needs K < 128 (bj + 1). False: another kernel does this problem.
template <int MODE, bool EXACT6>
__device__ __forceinline__ bool oz_item(const OzBatch& batch, int64_t item, OzItem<MODE>& it) {
  int q = 0;
  while (q + 1 < batch.nq && item >= batch.item0[q + 1]) ++q;
  const OzProb& L = batch.q[q];
  it.L = &L;
  item -= batch.item0[q];
  int u = int(item % L.ntile);
  item /= L.ntile;
  it.f = int(item % L.nf);
  it.sp = int(item / L.nf);
  it.st0 = it.sp * L.sps * L.sbst;
  it.st1 = min(L.nst, it.st0 + L.sps * L.sbst);
  it.sbst = L.sbst;
  if (MODE == OZ_QUAD) {
    it.bi = u % L.nbi;
    it.bj = L.nbj - 1 - u / L.nbi;      // the longest items first
    it.kind = 2;
    it.st1 = min(it.st1, (it.bj + 1) * (OT / OKS));
    it.a = L.A + size_t(it.bi) * L.nst * OBLK;
    it.b = L.B + size_t(it.f * L.nbj + it.bj) * L.nst * OBLK;
  } else {
    const int nbb = L.nbj;
    if (u < nbb * nbb) {
      it.bi = u % nbb;
      it.bj = u / nbb;
      it.kind = 0;
    } else {
      u -= nbb * nbb;
      int bj = 0;
      while (u > bj) {
        u -= bj + 1;
        ++bj;
      }
      it.bi = u + nbb;
      it.bj = bj + nbb;
      it.kind = 1;
    }
    it.a = L.A + size_t(it.f * 2 * nbb + it.bi) * L.nst * OBLK;
    it.b = L.B + size_t(it.bj) * L.nst * OBLK;
  }
  return __ldg(L.flag) == (EXACT6 ? FLAG_EXACT6 : 0);
}
// complex products: kind: the product, f: the tile's index, (bi, bj): the tile
template <int MODE, bool EXACT6>
__device__ __forceinline__ bool oz_item(const OzCBatch& batch, int64_t item, OzItem<MODE>& it) {
  int lo = 0, hi = batch.nq - 1;        // the last problem that starts at or before the item
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (item >= batch.item0[mid]) lo = mid;
    else hi = mid - 1;
  }
  const OzC& L = batch.q[lo];
  it.L = &L;
  const int u = int(item - batch.item0[lo]);
  it.f = u / L.nprod;
  it.kind = u - it.f * L.nprod;
  it.sp = 0;
  oz_tile(L, it.f, it.bi, it.bj);
  const int sx = L.nprod == 1 ? 0 : it.kind, sy = L.nprod == 1 ? 0 : it.kind == 2 ? 2 : 1 - it.kind;
  it.a = L.X + sx * L.xset + it.bi * L.xblk;
  it.b = L.Y + sy * L.yset + it.bj * L.yblk;
  constexpr int SPB = OT / OKS;         // stages per block
  it.st0 = max(L.k0, max((L.flags & OZC_KA) ? SPB * it.bi : 0, (L.flags & OZC_KB) ? SPB * it.bj : 0));
  it.st1 = (L.flags & OZC_KTOP) ? min(L.k1, SPB * (it.bi + 1)) : L.k1;
  it.sbst = SBMAX;
  return it.st1 > it.st0;
}

__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                        unsigned* status) {
  int ok = 0;
  if ((threadIdx.x & 31) == 0) {
    ok = (!*abort && tc::mbar_wait(bar, parity, abort, OWAIT)) ? 1 : 0;
    if (!ok && !*abort) {
      *abort = 1;
      raise_status(status, ST_ETIMEOUT);
    }
  }
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// FP64 of a register sum, and a global load, in volatile asm: they stay in program order, since
// 64 elements' conversions and loads moved up front would not fit beside the sums
__device__ __forceinline__ double to_f64(float v) {
  double r;
  asm volatile("cvt.f64.f32 %0, %1;" : "=d"(r) : "f"(v));
  return r;
}
// (s + c) + d of element i (c, d packed)
__device__ __forceinline__ double sum_f64(float s, const uint64_t (&c)[32], const uint64_t (&d)[32],
                                          int i) {
  auto part = [i](uint64_t x) {
    float l, h;
    tc::f2_unpack(x, l, h);
    return to_f64(i & 1 ? h : l);
  };
  return (to_f64(s) + part(c[i / 2])) + part(d[i / 2]);
}
__device__ __forceinline__ float ld_f32(const float* p) {
  float r;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(r) : "l"(p) : "memory");
  return r;
}
__device__ __forceinline__ double ld_f64(const double* p) {
  double r;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(r) : "l"(p) : "memory");
  return r;
}
__device__ __forceinline__ int4 ld_exp4(const int* p) {
  int4 r;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// EXACT6: group 6 summed by itself (exactly), and group 9 as well
template <int MODE, bool EXACT6>
__device__ __forceinline__ void oz_gemm(const typename OzBatchOf<MODE>::B& batch, unsigned* status) {
  constexpr uint32_t IDESC = tc::instr_desc(1u, OT, OT);
  if constexpr (MODE != OZ_CPLX) {            // nothing of the batch is this kernel's: whole grid
    bool any = false;
    for (int q = 0; q < batch.nq; ++q) any = any || __ldg(batch.q[q].flag) == (EXACT6 ? FLAG_EXACT6 : 0);
    if (!any) return;
  }
  extern __shared__ __align__(1024) char dsmem[];
  char* ring = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(dsmem) + 1023) & ~uintptr_t(1023));
  // full/empty per stage part (0: slices 1-4, 1: slices 5-7); D and C: the accumulators
  __shared__ __align__(8) uint64_t full[ONST][2], empty[ONST][2], fullD, emptyD, fullC, emptyC, done;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < ONST; ++i)
      for (int h = 0; h < 2; ++h) {
        tc::mbar_init(&full[i][h], 1);
        tc::mbar_init(&empty[i][h], 1);
      }
    tc::mbar_init(&fullD, 1);
    tc::mbar_init(&emptyD, EPI_WARPS);
    tc::mbar_init(&fullC, 1);
    tc::mbar_init(&emptyC, EPI_WARPS);
    tc::mbar_init(&done, 1);
    s_abort = 0;
    tc::mbar_fence_init();
  }
  if (warp == 0) {
    tc::tmem_alloc(&s_tmem, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = s_tmem;               // columns: D, C4, C3, C2 (128 each)
  const int64_t nitems = batch.item0[batch.nq];

  if (warp < EPI_WARPS) {
    tc::setmaxnreg_inc<REG_E>();
    const int qd = warp & 3, c0 = (warp >> 2) * 64;
    const int r = qd * 32 + lane;
    const uint32_t base = tmem + (uint32_t(qd * 32) << 16) + c0;
    uint64_t c[32], d[32];                    // packed FP32 pairs: columns 2 i, 2 i + 1
    // s is touched every 8 stages only: in L2 (64 KB per CTA, this thread's own entries), since
    // three sums of 64 columns leave too few registers for the two-sums (they spilled in
    // every drain)
    float* sp_s = batch.s + (size_t(blockIdx.x) * OT + c0) * OT + r;
    uint32_t gD = 0, gC = 0;                  // phases of fullD, fullC
    bool stop = false;
    // Paired FP32 adds in volatile asm, element by element: the compiler would otherwise move the
    // next chunks' work up and spill. add: x += v; two_sum: x + v = x' + e exactly (Knuth).
    auto add = [](uint64_t& x, uint64_t v) {
      asm volatile("add.rn.f32x2 %0, %0, %1;" : "+l"(x) : "l"(v));
    };
    auto two_sum = [](uint64_t& x, uint64_t v) {
      uint64_t e;
      asm volatile(
          "{\n.reg .b64 t, b, p, q;\nadd.rn.f32x2 t, %0, %2;\nsub.rn.f32x2 b, t, %0;\n"
          "sub.rn.f32x2 p, t, b;\nsub.rn.f32x2 p, %0, p;\nsub.rn.f32x2 q, %2, b;\n"
          "add.rn.f32x2 %1, p, q;\nmov.b64 %0, t;\n}\n"
          : "+l"(x), "=l"(e)
          : "l"(v));
      return e;
    };
    auto drain_c = [&](uint32_t col, bool fresh) {   // groups 2-4: s, then its error into c, then d
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float sv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) sv[i] = fresh ? 0.0f : ld_f32(sp_s + (h * 16 + i) * OT);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint64_t v[4];
          tc::tmem_ld8p(base + col + h * 16 + g * 8, v);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int e2 = g * 8 + 2 * i, k2 = h * 8 + g * 4 + i;
            uint64_t x = tc::f2_pack(__float_as_uint(sv[e2]), __float_as_uint(sv[e2 + 1]));
            const uint64_t e = two_sum(x, v[i]);
            tc::f2_unpack(x, sv[e2], sv[e2 + 1]);
            add(d[k2], two_sum(c[k2], e));
          }
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) sp_s[(h * 16 + i) * OT] = sv[i];
      }
    };
    // D: group 5 (and an exact group 6) into c, the low groups into d; false after an expired wait
    auto drain_d = [&](bool exact) {
      if (!oz_wait(&fullD, gD & 1, &s_abort, status)) return false;
      ++gD;
      tc::tc_fence_after();
      if constexpr (EXACT6) {
        // five drains per two stages: the accumulator is free as soon as it is in registers
        uint64_t v[32];
        tc::tmem_ld64p(base, v);
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&emptyD);
#pragma unroll
        for (int i = 0; i < 32; ++i) add(d[i], exact ? two_sum(c[i], v[i]) : v[i]);
        return true;
      }
      if (exact) {
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          uint64_t v[4];
          tc::tmem_ld8p(base + h * 8, v);
#pragma unroll
          for (int i = 0; i < 4; ++i) add(d[h * 4 + i], two_sum(c[h * 4 + i], v[i]));
        }
      } else {
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          uint64_t v[4];
          tc::tmem_ld8p(base + h * 8, v);
#pragma unroll
          for (int i = 0; i < 4; ++i) add(d[h * 4 + i], v[i]);
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&emptyD);
      return true;
    };
    for (int64_t item = blockIdx.x; item < nitems && !stop; item += gridDim.x) {
      OzItem<MODE> w;
      if (!oz_item<MODE, EXACT6>(batch, item, w)) continue;
      const auto& L = *w.L;
      const int f = w.f, sp = w.sp, bi = w.bi, bj = w.bj, kind = w.kind;
      double qsum = 0.0;
      bool first = true;
      for (int sb0 = w.st0; sb0 < w.st1 && !stop; sb0 += w.sbst) {
        const int n = min(w.sbst, w.st1 - sb0);
#pragma unroll
        for (int i = 0; i < 32; ++i) c[i] = d[i] = 0;
        bool fresh = true;                    // s is zero
        for (int k = 0; k < n; ++k) {
          const bool last = k == n - 1;
          // even: low, (6,) the accumulators due, group 5 unless the next odd stage continues it;
          // odd: group 5, the accumulators due, low(, 6)
          if (!drain_d(k & 1) || (EXACT6 && !(k & 1) && !drain_d(true))) {
            stop = true;
            break;
          }
          if ((k & 7) == 7 || last) {
            if (!oz_wait(&fullC, gC & 1, &s_abort, status)) {
              stop = true;
              break;
            }
            ++gC;
            tc::tc_fence_after();
            const int ng = last || (k & 31) == 31 ? 3 : (k & 15) == 15 ? 2 : 1;
#pragma unroll 1
            for (int gi = 1; gi <= ng; ++gi) {
              drain_c(gi * OT, fresh);
              fresh = false;
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&emptyC);
          }
          if ((((k & 1) || last) && !drain_d(!(k & 1))) || (EXACT6 && (k & 1) && !drain_d(true))) {
            stop = true;
            break;
          }
        }
        if (stop) break;
        if constexpr (MODE == OZ_CPLX) {
          // the product tile in float-float: s + c + d renormalised, times 2^(EX + EY - 14)
          const int ex = exponent_of(__ldg(L.mx + bi * OT + r)) - 14;
          const float* my = L.my + bj * OT + c0;
          float2* g = L.G + ((size_t(kind) * L.ntile + f) * OT + c0) * OT + r;
          float s16[16];
#pragma unroll
          for (int i = 0; i < 64; ++i) {
            if (i % 16 == 0) {                // 16 loads in flight (the volatile loads keep their order)
#pragma unroll
              for (int t = 0; t < 16; ++t) s16[t] = ld_f32(sp_s + (i + t) * OT);
            }
            const float sv = s16[i % 16];
            const int e = ex + exponent_of(__ldg(my + i)), e1 = max(-126, min(127, e >> 1)),
                      e2 = max(-126, min(127, e - e1));
            const float f1 = __int_as_float((e1 + 127) << 23), f2 = __int_as_float((e2 + 127) << 23);
            float cl, ch, dl, dh;
            tc::f2_unpack(c[i / 2], cl, ch);
            tc::f2_unpack(d[i / 2], dl, dh);
            const float cv = i & 1 ? ch : cl, dv = i & 1 ? dh : dl;
            const float h = __fadd_rn(sv, cv), b = __fsub_rn(h, sv);
            const float lo = __fadd_rn(__fadd_rn(__fsub_rn(sv, __fsub_rn(h, b)), __fsub_rn(cv, b)), dv);
            const float hh = __fadd_rn(h, lo);
            g[size_t(i) * OT] = make_float2(__fmul_rn(__fmul_rn(hh, f1), f2),
                                            __fmul_rn(__fmul_rn(__fsub_rn(lo, __fsub_rn(hh, h)), f1), f2));
          }
          continue;
        } else {
        // the superblock in FP64: ((s + c) + d) 2^(EA + EB - 14)
        const int sb = sb0 / w.sbst;
        const int* eb = L.EB + (size_t(MODE == OZ_QUAD ? f * L.nbj + bj : bj) * L.nsb + sb) * OT + c0;
        const int ea =
            L.EA[(size_t(MODE == OZ_QUAD ? bi : f * 2 * L.nbj + bi) * L.nsb + sb) * OT + r] - 14 + 1023;
        if constexpr (MODE == OZ_QUAD) {
          // this row's part of x . (x U) over the tile's columns: x 2^(EA + EB - 14) by integer
          // exponent arithmetic, s and c against it in FP64, d (2^-40 of s) in FP32
          const int64_t p = int64_t(bi) * OT + r;
          const int64_t col = int64_t(bj) * OT + c0;
          if (p < L.nrow) {
            const double* xr = L.x + p * L.ncol + col;
            float qd = 0.0f, s16[16];
            double x8[8];
#pragma unroll
            for (int g4 = 0; g4 < 16; ++g4) {
              const int4 e4 = ld_exp4(eb + 4 * g4);
              const int e[4] = {e4.x, e4.y, e4.z, e4.w};
              if (g4 % 4 == 0) {
#pragma unroll
                for (int t = 0; t < 16; ++t) s16[t] = ld_f32(sp_s + (4 * g4 + t) * OT);
              }
              if (g4 % 2 == 0) {
#pragma unroll
                for (int t = 0; t < 8; ++t) x8[t] = col + 4 * g4 + t < L.ncol ? ld_f64(xr + 4 * g4 + t) : 0.0;
              }
#pragma unroll
              for (int t = 0; t < 4; ++t) {
                const int i = 4 * g4 + t;
                const double xv = x8[4 * (g4 % 2) + t];
                const int hi = __double2hiint(xv), xe = (hi >> 20) & 0x7ff;
                const int ex = xe + ea - 1023 + e[t];
                const bool z = xe == 0 || ex < 1;                  // zero or underflow
                const double xs = z ? 0.0 : __hiloint2double(hi + ((ea - 1023 + e[t]) << 20),
                                                             __double2loint(xv));
                float cl, ch, dl, dh;
                tc::f2_unpack(c[i / 2], cl, ch);
                tc::f2_unpack(d[i / 2], dl, dh);
                qsum = fma(to_f64(s16[4 * (g4 % 4) + t]), xs, qsum);
                qsum = fma(to_f64(i & 1 ? ch : cl), xs, qsum);
                if (xe != 0 && ex >= 897 && ex <= 1120) {
                  const float xf = __int_as_float((hi & 0x80000000) | ((ex - 896) << 23) |
                                                  ((hi & 0xfffff) << 3) |
                                                  int(uint32_t(__double2loint(xv)) >> 29));
                  qd = fmaf(i & 1 ? dh : dl, xf, qd);
                } else {
                  qsum = fma(to_f64(i & 1 ? dh : dl), xs, qsum);   // outside the FP32 range
                }
              }
            }
            qsum += to_f64(qd);
          }
        } else {
          const size_t nbp = size_t(L.nbj) * OT;
          const int a = (kind ? bi - L.nbj : bi) * OT + r;
          const int b0 = (kind ? bj - L.nbj : bj) * OT + c0;
          double* g = L.G + ((size_t(sp) * L.nf + f) * 2 + kind) * nbp * nbp + size_t(b0) * nbp + a;
          const bool add = batch.add || !first;
          float s16[16];
#pragma unroll
          for (int g4 = 0; g4 < 16; ++g4) {
            if (g4 % 4 == 0) {
#pragma unroll
              for (int t = 0; t < 16; ++t) s16[t] = ld_f32(sp_s + (4 * g4 + t) * OT);
            }
            const int4 e4 = ld_exp4(eb + 4 * g4);
            const int e[4] = {e4.x, e4.y, e4.z, e4.w};
            double o[4] = {0.0, 0.0, 0.0, 0.0};
            if (add) {
#pragma unroll
              for (int t = 0; t < 4; ++t) o[t] = ld_f64(g + size_t(4 * g4 + t) * nbp);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const double v = sum_f64(s16[4 * (g4 % 4) + t], c, d, 4 * g4 + t);
              g[size_t(4 * g4 + t) * nbp] = fma(v, __hiloint2double((ea + e[t]) << 20, 0), o[t]);
            }
          }
        }
        }
        first = false;
      }
      if constexpr (MODE == OZ_QUAD) {
        const int64_t p = int64_t(bi) * OT + r;
        if (!stop && p < L.nrow)
          L.cpart[(size_t(f) * 2 * L.nbj + 2 * bj + (c0 ? 1 : 0)) * L.nrow + p] = qsum;
      }
    }
  } else {
    tc::setmaxnreg_dec<REG_P>();
    if (warp == EPI_WARPS && lane == 0) {
      // ---------------------------------------------- bulk copies of the slices
      uint32_t g = 0, half = 0;               // stages copied; 1: and slices 5-7 of the next one
      bool ok = true;
      for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
        OzItem<MODE> w;
        if (!oz_item<MODE, EXACT6>(batch, item, w)) continue;
        const char *a = w.a, *b = w.b;
        for (int st = w.st0; st < w.st1; ++st, ++g) {
          const int slot = g % ONST;
          const uint32_t par = ((g / ONST) & 1) ^ 1;
          char* dst = ring + slot * OSTAGE;
#pragma unroll
          for (int h = 1; h >= 0; --h) {              // slices 5-7 are free first
            if (!tc::mbar_wait(&empty[slot][h], par, &s_abort, OWAIT)) {
              ok = false;
              half = h ? 0 : 1;
              break;
            }
            const int nb = h ? LOB : HIB;
            char* to = dst + (h ? 2 * HIB : 0);
            const size_t off = size_t(st) * OBLK + (h ? HIB : 0);
            tc::mbar_arrive_expect_tx(&full[slot][h], 2 * nb);
            tc::bulk_g2s(to, a + off, nb, &full[slot][h]);
            tc::bulk_g2s(to + nb, b + off, nb, &full[slot][h]);
          }
          if (!ok) break;
        }
      }
      if (!ok && !s_abort) {
        s_abort = 1;
        raise_status(status, ST_ETIMEOUT);
      }
      // However the loop ended (its consumers may have given up): no copy into this CTA's shared
      // memory outlives the CTA. The last phase of every barrier that was armed.
      int never = 0;
      for (int h = 0; h < 2; ++h)
        for (uint32_t i = 0; i < ONST; ++i) {
          const uint32_t armed = (g + ONST - 1 - i) / ONST + (h && half && g % ONST == i ? 1 : 0);
          if (armed)
            tc::mbar_wait(&full[i][h], (armed - 1) & 1, reinterpret_cast<volatile int*>(&never), OWAIT);
        }
    } else if (warp == EPI_WARPS + 1) {
      // ---------------------------------------------- MMA issue (tc::elect_one)
      const uint32_t tm = tc::uniform(tmem);
      uint32_t g = 0, nD = 0, nC = 0;          // stages; drains of D and C so far
      bool ok = true;
      const uint64_t desc0 = tc::smem_desc(tc::uniform(tc::smem_u32(ring)), 512, 4);
      for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
        OzItem<MODE> w;
        if (!oz_item<MODE, EXACT6>(batch, item, w)) continue;
        for (int sb0 = w.st0; sb0 < w.st1 && ok; sb0 += w.sbst) {
          const int n = min(w.sbst, w.st1 - sb0);
          for (int k = 0; k < n; ++k, ++g) {
            const int slot = g % ONST;
            const uint32_t par = (g / ONST) & 1;
            const bool last = k == n - 1, odd = k & 1, due = (k & 7) == 7 || last;
            auto wait = [&](uint64_t* bar, uint32_t parity) {
              return ok = tc::mbar_wait_warp(bar, parity, &s_abort, OWAIT);
            };
            if (!wait(&full[slot][1], par) || !wait(&full[slot][0], par)) break;
            tc::tc_fence_after();
            const uint64_t sd = desc0 + uint64_t((slot * OSTAGE) >> 4);
            // slice i (1-based) of A and of B in the stage
            auto da = [&](int i) {
              return sd + uint64_t((i <= NHI ? (i - 1) * SLB : 2 * HIB + (i - 1 - NHI) * SLB) >> 4);
            };
            auto db = [&](int i) { return da(i) + uint64_t((i <= NHI ? HIB : LOB) >> 4); };
            auto group = [&](int gg, uint32_t dst, uint32_t acc) {
#pragma unroll
              for (int i = 1; i <= OSL; ++i) {
                const int j = gg - i;
                if (j < 1 || j > OSL) continue;
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                  tc::mma_f16(dst, da(i) + uint64_t((ks * 32) >> 4), db(j) + uint64_t((ks * 32) >> 4),
                              IDESC, acc);
                  acc = 1u;
                }
              }
            };
            auto low = [&]() {                          // a fresh D, the smallest products first
              if constexpr (EXACT6) group(9, tm, 0u);
              group(8, tm, EXACT6 ? 1u : 0u);
              group(7, tm, 1u);
              if constexpr (!EXACT6) {
                group(6, tm, 1u);
                tc::mma_commit(&empty[slot][1]);
              }
              tc::mma_commit(&fullD);
            };
            auto g6 = [&]() {                           // EXACT6: a D of its own
              group(6, tm, 0u);
              tc::mma_commit(&empty[slot][1]);
              tc::mma_commit(&fullD);
            };
            auto g4 = [&]() { group(4, tm + OT, (k & 7) ? 1u : 0u); };
            auto g32 = [&]() {
              group(3, tm + 2 * OT, (k & 15) ? 1u : 0u);
              group(2, tm + 3 * OT, (k & 31) ? 1u : 0u);
              if (due) tc::mma_commit(&fullC);
            };
            // the next D, once the epilogue has drained the last one
            auto next_d = [&]() {
              if (!wait(&emptyD, (nD & 1) ^ 1)) return false;
              tc::tc_fence_after();
              return true;
            };
            if (odd) {
              if (tc::elect_one()) {
                group(5, tm, 1u);
                tc::mma_commit(&fullD);
              }
              __syncwarp();
              ++nD;
              if (!wait(&emptyC, (nC & 1) ^ 1)) break;
              tc::tc_fence_after();
              // (with the drain of the accumulators due, before low, so that it runs beside it)
              if (tc::elect_one()) {
                g4();
                if (!EXACT6 || due) g32();
              }
              __syncwarp();
              if (!next_d()) break;
              if (tc::elect_one()) {
                low();
                if (EXACT6 && !due) g32();
                if (!EXACT6) tc::mma_commit(&empty[slot][0]);
              }
              __syncwarp();
              ++nD;
              if constexpr (EXACT6) {
                if (!next_d()) break;
                if (tc::elect_one()) {
                  g6();
                  tc::mma_commit(&empty[slot][0]);
                }
                __syncwarp();
                ++nD;
              }
            } else {
              if (!wait(&emptyC, (nC & 1) ^ 1)) break;
              tc::tc_fence_after();
              if (tc::elect_one()) g4();
              __syncwarp();
              if (!next_d()) break;
              if (tc::elect_one()) {
                low();
                if (!EXACT6) g32();
              }
              __syncwarp();
              ++nD;
              if constexpr (EXACT6) {
                if (!next_d()) break;
                if (tc::elect_one()) {
                  g6();
                  g32();
                }
                __syncwarp();
                ++nD;
              }
              if (!next_d()) break;
              if (tc::elect_one()) {
                group(5, tm, 0u);
                tc::mma_commit(&empty[slot][0]);
                if (last) tc::mma_commit(&fullD);
              }
              __syncwarp();
              if (last) ++nD;
            }
            if (due) ++nC;
          }
        }
      }
      if (lane == 0 && !ok && !s_abort) {
        s_abort = 1;
        raise_status(status, ST_ETIMEOUT);
      }
      if (tc::elect_one()) tc::mma_commit(&done);
      __syncwarp();
      int never = 0;
      tc::mbar_wait(&done, 0, reinterpret_cast<volatile int*>(&never), OWAIT);
    }
    __syncwarp();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz_gemm_pol(const __grid_constant__ OzBatch batch, unsigned* status) {
  oz_gemm<OZ_POL, false>(batch, status);
}
__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz_gemm_pol6(const __grid_constant__ OzBatch batch, unsigned* status) {
  oz_gemm<OZ_POL, true>(batch, status);
}
__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz_gemm_quad(const __grid_constant__ OzBatch batch, unsigned* status) {
  oz_gemm<OZ_QUAD, false>(batch, status);
}
__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz_gemm_quad6(const __grid_constant__ OzBatch batch, unsigned* status) {
  oz_gemm<OZ_QUAD, true>(batch, status);
}
__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz_gemm_cplx(const __grid_constant__ OzCBatch batch, unsigned* status) {
  oz_gemm<OZ_CPLX, true>(batch, status);
}

// ------------------------------------------------------------------ digits (fp64_slices.cuh)
// the exponent of a range: E with (largest magnitude) < 0.996 2^E, or a raised flag
__device__ __forceinline__ int range_exponent(float mx, float sum, float n, bool ratio, int* flag,
                                              float* spread = nullptr) {
  if (!(sum <= 3.0e38f) || !(mx < 1.2676506e30f)) {        // not finite, or from 2^100 on
    atomicOr(flag, FLAG_FP64);
    return 0;
  }
  if (mx == 0.0f) return 0;
  if (mx < 7.8886091e-31f || (ratio && mx * n > RATIO_MAX * sum)) {
    atomicOr(flag, FLAG_FP64);
    return 0;
  }
  if (spread) *spread = mx * n / sum;
  return ilogbf(mx * 1.005f) + 1;       // 1.005 mx < 2^E
}

// s_tj = prefactor f_t 2 Delta / (Delta^2 + w^2) (minus the same at Delta_bar with the extrapolar
// correction), FP64, [nw][K]
__global__ void k_oz_weights(const __grid_constant__ OzBatch batch, double pref, int nw, OmegaArr om,
                             unsigned* status) {
  const OzProb& L = batch.q[blockIdx.y];
  if (blockIdx.x == 0 && threadIdx.x == 0) *L.flag = L.spread[0] = L.spread[1] = 0;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < L.Kall;
       t += int64_t(gridDim.x) * blockDim.x) {
    const double d = L.delta[t];
    if (!(d > 0.0)) raise_status(status, ST_EINVAL);
    const double p2 = 2.0 * pref * (L.f ? L.f[t] : 1.0);
    const double db = L.dbar ? L.dbar[t] : 0.0;
    if (L.dbar && !(db > 0.0)) raise_status(status, ST_EINVAL);
    for (int j = 0; j < nw; ++j) {
      const double w2 = om.v[j] * om.v[j];
      double s = p2 * d / (d * d + w2);
      if (L.dbar) s -= p2 * db / (db * db + w2);
      L.w[size_t(j) * L.Kall + t] = s;
    }
  }
}

// |v| 2^e rounded up to FP32 by integer arithmetic (the FP64 pipe's conversions cost three times the
// reads of the scale kernel): the exponent re-biased, the top 23 mantissa bits plus one. Zero and
// magnitudes below 2^-126 become 2^-126, those above the FP32 range (and non-finite ones) infinite.
__device__ __forceinline__ float abs_up(double v, int e = 0) {
  const unsigned long long b = __double_as_longlong(v) & 0x7fffffffffffffffull;
  const long long f = (long long)(b >> 29) - ((896ll - e) << 23) + 1;  // FP32 bits of the next value up
  const int bits = f < 0x00800000ll ? 0x00800000 : f > 0x7f800000ll ? 0x7f800000 : int(f);
  return __int_as_float(b ? bits : 0);
}

// Bounds (within 2^-21) of the largest magnitude and of the magnitude sum of every column over
// chunks of 64 rows, in FP32: operand types 0 Mi, 1 Mr + Mi (B), 2 + 2 f and 3 + 2 f: s_f Mr,
// s_f (Mr + Mi) (A). Thread = column; grid (column blocks, chunks). Bound by the read of M. The products
// with the weights are rounded up, so that none becomes zero: a column whose largest product is below
// 2^-100 takes the FP64 kernel, and so do weights that abs_up raises to 2^-126 where an entry of M
// could lift them above that (and weights from 2^26 on, which lift raised entries of M).
__global__ void __launch_bounds__(OT) k_oz_scale(const __grid_constant__ OzBatch batch) {
  __shared__ float sw[4][CHROWS];
  __shared__ int odd;
  const OzProb& L = batch.q[blockIdx.z];
  const double2* __restrict__ M = L.M;
  const double* __restrict__ w = L.wp;
  const int64_t K = L.K, wld = L.Kall;
  const int nb = L.nb, nf = L.nf, ncolp = L.nbj * OT;
  if (int(blockIdx.x) >= L.nbj || int64_t(blockIdx.y) * CHROWS >= K) return;   // whole CTA
  const int col = blockIdx.x * OT + threadIdx.x;
  const int64_t t0 = int64_t(blockIdx.y) * CHROWS;
  const int n = int(K - t0 < CHROWS ? K - t0 : CHROWS);
  const int ntype = 2 + 2 * nf;
  float2* out = L.part + size_t(blockIdx.y) * ntype * ncolp + col;
  for (int f0 = 0; f0 < nf; f0 += 4) {
    const int nj = min(4, nf - f0);
    __syncthreads();
    if (threadIdx.x == 0) odd = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < 4 * CHROWS; e += OT) {
      const int j = e / CHROWS, t = e % CHROWS;
      const double v = j < nj && t < n ? w[size_t(f0 + j) * wld + t0 + t] : 0.0;
      sw[j][t] = abs_up(v);
      if (v != 0.0 && fabs(v) < 1.1754944e-38) atomicOr(&odd, 1);
      if (fabs(v) >= 6.7108864e7) atomicOr(&odd, 2);
    }
    __syncthreads();
    float mi = 0.f, ms = 0.f, si = 0.f, ss = 0.f, ma[4][2] = {}, sa[4][2] = {};
    if (col < nb) {
#pragma unroll 8
      for (int t = 0; t < n; ++t) {
        const double2 x = __ldg(M + (t0 + t) * nb + col);
        const float r = abs_up(x.x), i = abs_up(x.y);
        // |Mr + Mi| of the rounded parts, plus their rounding
        const bool same = (__double2hiint(x.x) ^ __double2hiint(x.y)) >= 0;
        const float s = (same ? r + i : fabsf(r - i)) + 4.7683716e-7f * (r + i);
        mi = fmaxf(mi, i);
        si += i;
        ms = fmaxf(ms, s);
        ss += s;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float pr = __fmul_ru(r, sw[j][t]), ps = __fmul_ru(s, sw[j][t]);
          ma[j][0] = fmaxf(ma[j][0], pr);
          sa[j][0] += pr;
          ma[j][1] = fmaxf(ma[j][1], ps);
          sa[j][1] += ps;
        }
      }
    }
    if ((odd & 2) || (odd && (mi >= 3.3e7f || ms >= 3.3e7f))) atomicOr(L.flag, FLAG_FP64);
    if (f0 == 0) {
      out[0] = make_float2(mi, si);
      out[ncolp] = make_float2(ms, ss);
    }
    for (int j = 0; j < nj; ++j) {
      out[size_t(2 + 2 * (f0 + j)) * ncolp] = make_float2(ma[j][0], sa[j][0]);
      out[size_t(3 + 2 * (f0 + j)) * ncolp] = make_float2(ma[j][1], sa[j][1]);
    }
  }
}

// Exponents of every (type, column, superblock) from the chunk partials, and the largest spreads: for a
// column of n rows with magnitudes of maximum m and mean a, m / (a n^1/4). The error of an element from
// digits is a multiple of 2^-53 n^1/2 m_A m_B, that of FP64 sums one of 2^-53 n (A^2 B^2 in the mean)^1/2,
// so the quotient of the two is at most the product of the spreads of A and B. Measured against sums
// in twice FP64's precision, rms relative to sqrt(P_II P_JJ) (FP64 kernel): Gaussian M and gaps from
// 0.05 Ha on, product 4 to 19: 1.0e-16 (1.1e-16) for K = 512, 2.7e-17 (2.6e-17) for 8,192; gaps of 0.003
// Ha, 100: 4.3e-16 (2.8e-16); entries of 30 to 300 times the others, 300 on: 5e-16 to 9e-16 (1e-16 to
// 2.4e-16). Above SPREAD_EXACT6 the GEMM with an exact group 6 takes over: 2.5e-17 to 7e-17 in all of
// these (5.85 -> 7.5 ms for K = 102,400, N_b = 600, 2 frequencies).
constexpr float SPREAD_EXACT6 = 32.0f;
__global__ void k_oz_exps(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.y];
  const float2* __restrict__ part = L.part;
  const int64_t K = L.K;
  const int nbb = L.nbj, nf = L.nf, nsb = L.nsb, sbst = L.sbst;
  int *EA = L.EA, *EB = L.EB;
  const int ncolp = nbb * OT, ntype = 2 + 2 * nf;
  const int64_t total = int64_t(ntype) * ncolp * nsb;
  const int cps = sbst * OKS / CHROWS;              // chunks per superblock
  const int nch = int((K + CHROWS - 1) / CHROWS);
  float top_a = 0.f, top_b = 0.f;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int col = int(e % ncolp), type = int(e / ncolp % ntype), sb = int(e / ncolp / ntype);
    float mx = 0.f, sum = 0.f;
    const int ch1 = min(nch, (sb + 1) * cps);
    for (int ch = sb * cps; ch < ch1; ++ch) {
      const float2 p = part[(size_t(ch) * ntype + type) * ncolp + col];
      mx = fmaxf(mx, p.x);
      sum += p.y;
    }
    const int64_t r0 = int64_t(sb) * sbst * OKS;
    const float rows = float(min(int64_t(sbst) * OKS, K - r0));
    float sp = 0.f;
    const int E = range_exponent(mx, sum, rows, true, L.flag, &sp);
    sp *= rsqrtf(sqrtf(rows));
    (type < 2 ? top_b : top_a) = fmaxf(type < 2 ? top_b : top_a, sp);
    const int cb = col / OT, n = col % OT;
    if (type < 2)
      EB[(size_t(type * nbb + cb) * nsb + sb) * OT + n] = E;
    else
      EA[(size_t((type - 2) / 2 * 2 * nbb + (type & 1) * nbb + cb) * nsb + sb) * OT + n] = E;
  }
  __syncwarp();
  const int a = __reduce_max_sync(0xffffffffu, __float_as_int(top_a));      // (positive: ordered as integers)
  const int b = __reduce_max_sync(0xffffffffu, __float_as_int(top_b));
  if ((threadIdx.x & 31) == 0) {
    atomicMax(L.spread, a);
    atomicMax(L.spread + 1, b);
  }
}

// The digit slices of one stage (32 rows) and 32 basis functions: B (Mi, Mr + Mi) and, per
// frequency, A (s Mr, s (Mr + Mi)). Four lanes per basis function, 8 rows each: a warp reads 128
// contiguous bytes per row and writes 512 per slice. (One lane per basis function wrote half
// sectors: 3.46 ms for one q of K = 102,400, N_b = 600, 2 frequencies.)
__global__ void __launch_bounds__(OT) k_oz_slice(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.z];
  const int nst = L.nst, nsb = L.nsb, sbst = L.sbst, nbb = L.nbj, nb = L.nb, nf = L.nf;
  if (int(blockIdx.x) >= nst || int(blockIdx.y) >= 4 * nbb || (__ldcg(L.flag) & FLAG_FP64)) return;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 &&
      __int_as_float(L.spread[0]) * __int_as_float(L.spread[1]) > SPREAD_EXACT6)
    atomicOr(L.flag, FLAG_EXACT6);            // read by the GEMMs
  const double2* __restrict__ M = L.M;
  const double* __restrict__ w = L.wp;
  const int64_t K = L.K, wld = L.Kall;
  const int* __restrict__ EA = L.EA;
  const int* __restrict__ EB = L.EB;
  char* __restrict__ A = L.A;
  char* __restrict__ B = L.B;
  const int cb = blockIdx.y >> 2, st = blockIdx.x, kc = threadIdx.x & 3;
  const int n = int(blockIdx.y & 3) * 32 + (threadIdx.x >> 2);
  const int col = cb * OT + n, sb = st / sbst;
  const size_t e0 = size_t(sb) * OT + n, eld = size_t(nsb) * OT;
  const int64_t t0 = int64_t(st) * OKS + kc * 8;
  double xr[8], xi[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const double2 x = t0 + k < K && col < nb ? __ldg(M + (t0 + k) * nb + col) : make_double2(0., 0.);
    xr[k] = x.x;
    xi[k] = x.y;
  }
  uint32_t dg[OSL][4];
  digits8(xi, EB[cb * eld + e0], dg);
  store_digits(B + (size_t(cb) * nst + st) * OBLK, n, kc, dg);
#pragma unroll
  for (int k = 0; k < 8; ++k) xi[k] = xr[k] + xi[k];
  digits8(xi, EB[(nbb + cb) * eld + e0], dg);
  store_digits(B + (size_t(nbb + cb) * nst + st) * OBLK, n, kc, dg);
  for (int f = 0; f < nf; ++f) {
    double y[8], wk[8];
    const size_t blk = size_t(f) * 2 * nbb + cb;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      wk[k] = t0 + k < K ? __ldg(w + size_t(f) * wld + t0 + k) : 0.0;
      y[k] = xr[k] * wk[k];
    }
    digits8(y, EA[blk * eld + e0], dg);
    store_digits(A + (blk * nst + st) * OBLK, n, kc, dg);
#pragma unroll
    for (int k = 0; k < 8; ++k) y[k] = xi[k] * wk[k];
    digits8(y, EA[(blk + nbb) * eld + e0], dg);
    store_digits(A + ((blk + nbb) * nst + st) * OBLK, n, kc, dg);
  }
}

// P (or P +=) from the tiles of C and S summed over the splits in order:
// P_ab = -S_ab + C_ab + C_ba + i (C_ab - C_ba), Hermitian exactly (S from its upper element)
__global__ void k_oz_combine(const __grid_constant__ OzBatch batch, int accumulate) {
  const OzProb& L = batch.q[blockIdx.y];
  if (__ldg(L.flag) & FLAG_FP64) return;
  double2* __restrict__ P = L.P;
  const double* __restrict__ G = L.G;
  const int nb = L.nb, nbp = L.nbj * OT, nf = L.nf, splits = L.splits;
  const int64_t n2 = int64_t(nb) * nb, total = n2 * nf;
  const size_t p2 = size_t(nbp) * nbp;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int f = int(e / n2);
    const int64_t rem = e % n2;
    const int a = int(rem / nb), b = int(rem % nb);
    const size_t ab = size_t(b) * nbp + a, ba = size_t(a) * nbp + b;
    double cab = 0.0, cba = 0.0, sab = 0.0;
    for (int sp = 0; sp < splits; ++sp) {
      const double* C = G + (size_t(sp) * nf + f) * 2 * p2;
      cab += C[ab];
      cba += C[ba];
      sab += C[p2 + (a <= b ? ab : ba)];
    }
    double re = (cab + cba) - sab, im = cab - cba;
    if (accumulate) {
      const double2 o = P[e];
      re += o.x;
      im += o.y;
    }
    P[e] = make_double2(re, im);
  }
}

// ------------------------------------------------------------------ quadratic form
// c_p = x_p R x_p^T of the pair projections' real rows x and the real form R of W^c (R[2I+a][2J+b] =
// Re W_IJ for a = b, -Im W_IJ for (0,1), Im W_IJ for (1,0)), as x U x^T with U the upper triangle
// U_kk = R_kk, U_kc = R_kc + R_ck (k < c), so that column block bj needs K < 128 (bj + 1) only.
__device__ __forceinline__ double u_entry(const double2* __restrict__ W, int nb, int k, int c) {
  if (k > c || c >= 2 * nb) return 0.0;
  const int I = k >> 1, a = k & 1, J = c >> 1, b = c & 1;
  const double2 w = __ldg(W + size_t(I) * nb + J);
  const double u = a == b ? w.x : a == 0 ? -w.y : w.y;
  if (k == c) return u;
  const double2 t = __ldg(W + size_t(J) * nb + I);
  return u + (a == b ? t.x : b == 0 ? -t.y : t.y);
}

// The basis is scaled by powers of two first: x'_I = x_I 2^e_I, W'_IJ = W_IJ 2^-(e_I + e_J) with
// 2^(2 e_I) near the largest |W_II| of the problem's frequencies. It changes no term and rounds
// nothing (the digits are cut with the shifted exponents), and a (semi)definite W, which W^c is, has
// |W'_IJ| <= 4 then, whatever units the basis functions have. Without it, scales of 10^+-2 at random left
// 1e-13 of the sum of the terms' magnitudes, 10^+-8 1e-6.
// 32 basis functions per CTA, eight threads each (the diagonals lie pages apart: latency).
constexpr int EQF = 8;
__global__ void __launch_bounds__(32 * EQF) k_oz_equilibrate(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.y];
  if (int(blockIdx.x) * 32 >= L.nb) return;   // whole CTA, before any barrier
  __shared__ double sm[EQF][32];
  const int lane = threadIdx.x & 31, f0 = threadIdx.x >> 5, I = blockIdx.x * 32 + lane;
  double d[GW_MAX_NW / EQF], m = 0.0;
#pragma unroll
  for (int k = 0; k < GW_MAX_NW / EQF; ++k) {
    const int f = f0 + EQF * k;
    d[k] = f < L.nf && I < L.nb ? __ldg(L.M + (size_t(f) * L.nb + I) * L.nb + I).x : 0.0;
    m = fmax(m, fabs(d[k]));
  }
  sm[f0][lane] = m;
  __syncthreads();
  if (I >= L.nb) return;
#pragma unroll
  for (int k = 0; k < EQF; ++k) m = fmax(m, sm[k][lane]);
  const int ex = (__double2hiint(m) >> 20) & 0x7ff;
  const int e = ex == 0 || ex == 0x7ff ? 0 : max(-64, min(64, (ex - 1023) >> 1));
  if (f0 == 0) L.eq[I] = e;
#pragma unroll
  for (int k = 0; k < GW_MAX_NW / EQF; ++k) {
    const int f = f0 + EQF * k;
    if (f >= L.nf) break;
    float2* c = L.cols + size_t(f) * L.nbj * OT + 2 * I;
    c[0].y = c[1].y = abs_up(d[k], -2 * e);
  }
}

// exponents of the rows of x, one warp per row and superblock (rows beyond nrow: zeros)
__global__ void __launch_bounds__(256) k_oz_rowexps(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int64_t rows = int64_t(L.nbi) * OT;
  for (int64_t e = blockIdx.x * 8 + (threadIdx.x >> 5); e < rows * L.nsb; e += int64_t(gridDim.x) * 8) {
    const int64_t row = e / L.nsb;
    const int sb = int(e % L.nsb);
    float mx = 0.f, sum = 0.f;
    if (row < L.nrow) {
      const int64_t c0 = int64_t(sb) * L.sbst * OKS, c1 = min(L.ncol, c0 + int64_t(L.sbst) * OKS);
      for (int64_t c = c0 + lane; c < c1; c += 32) {
        const float v = abs_up(__ldg(L.x + row * L.ncol + c), __ldg(L.eq + (c >> 1)));
        mx = fmaxf(mx, v);
        sum += v;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 0)
      L.EA[(size_t(row / OT) * L.nsb + sb) * OT + row % OT] = range_exponent(mx, sum, 1.0f, false, L.flag);
  }
}

// digit slices of x: grid (stages, row blocks x 4, problems), four lanes per row
__global__ void __launch_bounds__(OT) k_oz_slice_rows(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.z];
  if (int(blockIdx.x) >= L.nst || int(blockIdx.y) >= 4 * L.nbi || (__ldg(L.flag) & FLAG_FP64)) return;
  const int bi = blockIdx.y >> 2, st = blockIdx.x, kc = threadIdx.x & 3;
  const int n = int(blockIdx.y & 3) * 32 + (threadIdx.x >> 2);
  const int64_t row = int64_t(bi) * OT + n, c0 = int64_t(st) * OKS + kc * 8;
  double v[8];
#pragma unroll
  for (int k = 0; k < 8; k += 2) {            // ncol is even: whole pairs
    const double2 x = row < L.nrow && c0 + k < L.ncol
                          ? __ldg(reinterpret_cast<const double2*>(L.x + row * L.ncol + c0 + k))
                          : make_double2(0., 0.);
    v[k] = x.x;
    v[k + 1] = x.y;
  }
  uint32_t dg[OSL][4];
  const int E = L.EA[(size_t(bi) * L.nsb + st / L.sbst) * OT + n];
  int Ek[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) Ek[k] = E - (c0 + k < L.ncol ? __ldg(L.eq + ((c0 + k) >> 1)) : 0);
  digits8(v, Ek, dg);
  store_digits(L.A + (size_t(bi) * L.nst + st) * OBLK, n, kc, dg);
}

// largest magnitude of the columns of U over 128 of its rows: grid (column blocks, row chunks,
// problems x frequencies); thread = column and quarter of the rows. W: the problem's first
// frequency. The latency of the loads bounds it: N_b = 600, 16 frequencies 174 us with one thread per
// column and one row at a time, 90 us with quarters and eight rows in flight (N_b = 64: 46 -> 13 us).
constexpr int UROWS = 4;
__global__ void __launch_bounds__(OT * UROWS) k_oz_uscale(const __grid_constant__ OzBatch batch, int nfmax) {
  const OzProb& L = batch.q[blockIdx.z / nfmax];
  const int f = blockIdx.z % nfmax, cb = blockIdx.x, ch = blockIdx.y;
  if (f >= L.nf || cb >= L.nbj || ch > cb) return;
  const double2* W = L.M + size_t(f) * L.nb * L.nb;
  const int n = threadIdx.x % OT, g = threadIdx.x / OT, c = cb * OT + n;
  const int k0 = ch * OT + g * (OT / UROWS);
  const int ec = c < 2 * L.nb ? __ldg(L.eq + (c >> 1)) : 0;
  float mx = 0.f, sum = 0.f;
#pragma unroll 8
  for (int k = 0; k < OT / UROWS; ++k) {
    const int ek = k0 + k < 2 * L.nb ? __ldg(L.eq + ((k0 + k) >> 1)) : 0;
    const float v = abs_up(u_entry(W, L.nb, k0 + k, c), -(ek + ec));
    mx = fmaxf(mx, v);
    sum += v;
  }
  __shared__ float2 sh[UROWS][OT];
  sh[g][n] = make_float2(mx, sum);
  __syncthreads();
  if (g > 0) return;
#pragma unroll
  for (int h = 1; h < UROWS; ++h) {
    mx = fmaxf(mx, sh[h][n].x);
    sum += sh[h][n].y;
  }
  L.part[(size_t(f) * L.nbj + ch) * (size_t(L.nbj) * OT) + c] = make_float2(mx, sum);
}

// exponents of the scaled U's columns, plus that of the column's own scale (what the GEMM's epilogue
// multiplies with x, unscaled), and the columns' largest magnitudes
__global__ void k_oz_uexps(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.y];
  const int ncolp = L.nbj * OT, cps = L.sbst * OKS / OT;
  const int64_t total = int64_t(L.nf) * ncolp * L.nsb;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int c = int(e % ncolp), sb = int(e / ncolp % L.nsb), f = int(e / ncolp / L.nsb);
    const int cb = c / OT;
    float mx = 0.f, sum = 0.f;
    for (int ch = sb * cps; ch < (sb + 1) * cps && ch <= cb; ++ch) {
      const float2 p = L.part[(size_t(f) * L.nbj + ch) * ncolp + c];
      mx = fmaxf(mx, p.x);
      sum += p.y;
    }
    L.EB[(size_t(f * L.nbj + cb) * L.nsb + sb) * OT + c % OT] =
        range_exponent(mx, sum, 1.0f, false, L.flag) + (c < 2 * L.nb ? __ldg(L.eq + (c >> 1)) : 0);
    if (sb > 0) continue;
    for (int ch = cps; ch <= cb; ++ch)
      mx = fmaxf(mx, L.part[(size_t(f) * L.nbj + ch) * ncolp + c].x);
    L.cols[size_t(f) * ncolp + c].x = mx;
  }
}

// Whether the digits hold the pairs' coefficients. The error of a coefficient from digits is a
// multiple of 2^-53 max_k |x'_k| (sum_c (x'_c max_k |U'_kc|)^2)^1/2 (independent errors of the columns'
// sums), that of FP64 sums a multiple of 2^-53 of the sum of the terms' magnitudes, of which the diagonal
// sum_c |U'_cc| x'_c^2 is a part. R is the largest quotient of the two over pairs and frequencies: at
// most 1.0 for the W^c of the repository's workloads (N_b = 27 to 600), more where the diagonal of W falls
// off differently with the frequency for different basis functions, or where W is not definite.
// Measured errors relative to the sum of the terms' magnitudes, N_b = 16 to 600, rms (the FP64 kernel's:
// 3e-16 to 9e-16):
//   R       0.7 to 1         1.4 to 2          4 to 6            32 to 64          64 to 90
//   digits  3e-16 to 1.4e-15 3.4e-16 to 1.2e-15 7e-16 to 3.4e-15 5e-15 to 2e-14    8e-15 to 3e-14
//   exact6  3e-16 to 1e-15   2e-16 to 6e-16    3e-16 to 7e-16    4e-16 to 8e-16    6e-16 to 1.1e-15
// so above 2 a q takes the GEMM with an exact group 6 (6,656 pairs, N_b = 600, 16 frequencies: 5.5 ->
// 6.8 ms), above 64 the FP64 kernel (262 ms).
// 16 pairs per CTA, a pair in two lanes, which take different frequencies; 64 columns at a time.
constexpr float PAIR_EXACT6 = 2.0f, PAIR_FP64 = 64.0f;
constexpr int GP = 16, GC = 64, GT = 256, GF = GW_MAX_NW * GP / GT;
static_assert(GF * GT == GW_MAX_NW * GP, "a thread's frequencies");
__global__ void __launch_bounds__(GT) k_oz_pair_guard(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.y];
  const int64_t p0 = int64_t(blockIdx.x) * GP;
  if (p0 >= L.nrow) return;                   // whole CTA, before any barrier
  __shared__ float sx[GC][GP + 1];
  __shared__ float2 su[GW_MAX_NW][GC];
  __shared__ int se[GP];
  const int tid = threadIdx.x, pr = tid & (GP - 1), f0 = tid / GP, ncolp = L.nbj * OT;
  if (tid < GP) {                             // x' against the row's exponent: no overflow in FP32
    const int64_t p = p0 + tid;
    int e = -1000;
    for (int sb = 0; sb < L.nsb && p < L.nrow; ++sb)
      e = max(e, L.EA[(size_t(p / OT) * L.nsb + sb) * OT + p % OT]);
    se[tid] = e;
  }
  float top = 0.f, lhs[GF] = {}, rhs[GF] = {};
  for (int c0 = 0; c0 < int(L.ncol); c0 += GC) {
    __syncthreads();
#pragma unroll
    for (int j = 0; j < GP * GC / GT; ++j) {
      const int i = tid + j * GT, c = i % GC, r = i / GC;
      sx[c][r] = p0 + r < L.nrow && c0 + c < L.ncol
                     ? abs_up(__ldg(L.x + (p0 + r) * L.ncol + c0 + c), __ldg(L.eq + ((c0 + c) >> 1)) - se[r])
                     : 0.f;
    }
    for (int i = tid; i < L.nf * GC; i += GT) {
      const int c = i % GC, f = i / GC;
      float2 u = c0 + c < L.ncol ? L.cols[size_t(f) * ncolp + c0 + c] : make_float2(0.f, 0.f);
      if (u.x > 0.f) u.x = fmaxf(u.x, 8.7e-19f);                // (the squares stay above the FP32 range)
      su[f][c] = u;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < GF; ++i) {
      const int f = f0 + GT / GP * i;
      if (f >= L.nf) break;
      float a = 0.f, b = 0.f;
#pragma unroll 16
      for (int c = 0; c < GC; ++c) {
        const float x = sx[c][pr];
        const float2 u = su[f][c];
        const float t = x * u.x;
        top = fmaxf(top, x);
        a = fmaf(t, t, a);
        b = fmaf(x * x, u.y, b);
      }
      lhs[i] += a;
      rhs[i] += b;
    }
  }
  int bits = 0;
#pragma unroll
  for (int i = 0; i < GF; ++i) {
    const float err = top * sqrtf(lhs[i]);
    if (!(err <= PAIR_FP64 * rhs[i]) || (err == 0.f && rhs[i] > 0.f)) bits |= FLAG_FP64;
    else if (err > PAIR_EXACT6 * rhs[i]) bits |= FLAG_EXACT6;
  }
  bits = __reduce_or_sync(0xffffffffu, bits);
  if ((tid & 31) == 0 && bits) atomicOr(L.flag, bits);
}

// digit slices of U: grid (stages, column blocks x 4, problems x frequencies)
__global__ void __launch_bounds__(OT) k_oz_slice_u(const __grid_constant__ OzBatch batch, int nfmax) {
  const OzProb& L = batch.q[blockIdx.z / nfmax];
  const int f = blockIdx.z % nfmax, cb = blockIdx.y >> 2, st = blockIdx.x;
  if (f >= L.nf || cb >= L.nbj || st >= L.nst || st * OKS > cb * OT + OT - 1 || (__ldg(L.flag) & FLAG_FP64)) return;
  const double2* W = L.M + size_t(f) * L.nb * L.nb;
  const int kc = threadIdx.x & 3, n = int(blockIdx.y & 3) * 32 + (threadIdx.x >> 2);
  const int c = cb * OT + n, k0 = st * OKS + kc * 8;
  const size_t blk = size_t(f) * L.nbj + cb;
  const int E = L.EB[(blk * L.nsb + st / L.sbst) * OT + n];
  double v[8];
  int Ek[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    v[k] = u_entry(W, L.nb, k0 + k, c);
    Ek[k] = E + (k0 + k < 2 * L.nb ? __ldg(L.eq + ((k0 + k) >> 1)) : 0);
  }
  uint32_t dg[OSL][4];
  digits8(v, Ek, dg);
  store_digits(L.B + (blk * L.nst + st) * OBLK, n, kc, dg);
}

// c[f][p] from the column blocks' parts in order; ldc: pairs of the whole q
__global__ void k_oz_pair_reduce(const __grid_constant__ OzBatch batch) {
  const OzProb& L = batch.q[blockIdx.y];
  if (__ldg(L.flag) & FLAG_FP64) return;
  const int64_t total = L.nrow * L.nf;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < total;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t f = e / L.nrow, p = e % L.nrow;
    double v = 0.0;
    for (int b = 0; b < 2 * L.nbj; ++b) v += L.cpart[(f * 2 * L.nbj + b) * L.nrow + p];
    L.G[f * L.Kall + p] = v;
  }
}

size_t oz_smem() { return size_t(ONST) * OSTAGE + 1024; }

template <typename B>
int launch_oz(void (*kern)(B, unsigned*), const B& batch, cudaStream_t s, const DeviceCtx& ctx) {
  const int64_t items = batch.item0[batch.nq];
  if (items == 0) return GW_OK;
  int rc = set_max_dyn_smem(reinterpret_cast<const void*>(kern), oz_smem(), ctx.device);
  if (rc) return rc;
  const unsigned grid = unsigned(std::min<int64_t>(items, ctx.sm_count));
  kern<<<grid, OTHREADS, oz_smem(), s>>>(batch, ctx.status);
  GW_LAUNCH_CHECK("k_oz_gemm");
  return GW_OK;
}

// ------------------------------------------------------------------ polarization plan
// A q is done in passes over frequency chunks (nf) and K ranges (rows): the digit slices of a pass
// stay within DIGIT_BUDGET where a pass of one superblock and one frequency allows. q points
// of one pass share their launches, up to OZQ of them within the budget.
constexpr size_t DIGIT_BUDGET = size_t(6) << 30;

struct OzPlan {
  int nbb, ntile, nf, nst, sbst, nsb, sps, splits;
  int64_t rows;                     // per pass
  int npass, nchunk;                // K ranges and frequency chunks
  size_t digits;
  size_t b_w, b_part, b_ea, b_eb, b_A, b_B, b_G;
  size_t total() const {
    return b_w + b_part + size_t(npass) * nchunk * (b_ea + b_eb) + b_A + b_B + b_G;
  }
};

OzPlan oz_plan(int64_t K, int nb, int nw) {
  OzPlan p;
  p.nbb = (nb + OT - 1) / OT;
  p.ntile = p.nbb * p.nbb + p.nbb * (p.nbb + 1) / 2;
  const size_t blk_row = size_t(2) * p.nbb * OT * 2 * OSL;       // digit bytes per row and operand
  const int64_t unit = int64_t(SBMAX) * OKS;
  const int64_t one = std::min<int64_t>(K, unit);
  p.nf = int(std::max<int64_t>(1, std::min<int64_t>(nw, int64_t(DIGIT_BUDGET / (blk_row * one)) - 1)));
  const int64_t fit = int64_t(DIGIT_BUDGET / (blk_row * (p.nf + 1)));
  p.rows = std::min(K, std::max<int64_t>(1, fit / unit) * unit);
  p.nst = int((p.rows + OKS - 1) / OKS);
  p.npass = int((K + p.rows - 1) / p.rows);
  p.nchunk = (nw + p.nf - 1) / p.nf;
  p.digits = blk_row * size_t(p.nst) * OKS * (p.nf + 1);
  return p;
}

// Splits of the pass's K and the buffer sizes, for a share of `sm` SMs: every CTA takes about the
// same time per item, so whole waves of CTAs; at least 8 stages each, among the counts that give 3
// to 12 waves the best filled last one.
void oz_splits(OzPlan& p, int64_t K, int nw, int sm) {
  const int64_t items = int64_t(p.ntile) * p.nf;
  const int most = int(std::max<int64_t>(1, std::min<int64_t>((12 * int64_t(sm)) / items, (p.nst + 7) / 8)));
  const int least = int(std::min<int64_t>(most, (3 * int64_t(sm) + items - 1) / items));
  int pick = std::max(1, least);
  double best = 0.0;
  for (int sp = pick; sp <= most; ++sp) {
    const int sb = std::min(SBMAX, ((p.nst + sp - 1) / sp + 7) / 8 * 8);
    const int nsb = (p.nst + sb - 1) / sb, sps = (nsb + sp - 1) / sp;
    const int64_t it = items * ((nsb + sps - 1) / sps);
    const double fill = double(it) / double((it + sm - 1) / sm * sm);
    if (fill > best + 0.02) {
      best = fill;
      pick = sp;
    }
  }
  p.sbst = std::min(SBMAX, ((p.nst + pick - 1) / pick + 7) / 8 * 8);
  p.nsb = (p.nst + p.sbst - 1) / p.sbst;
  p.sps = (p.nsb + pick - 1) / pick;
  p.splits = (p.nsb + p.sps - 1) / p.sps;
  const int64_t nch = (p.rows + CHROWS - 1) / CHROWS;
  p.b_w = ws_round(size_t(nw) * size_t(K) * 8);
  p.b_part = ws_round(size_t(nch) * (2 + 2 * p.nf) * p.nbb * OT * sizeof(float2));
  p.b_ea = ws_round(size_t(p.nf) * 2 * p.nbb * p.nsb * OT * 4);
  p.b_eb = ws_round(size_t(2) * p.nbb * p.nsb * OT * 4);
  p.b_A = ws_round(size_t(p.nf) * 2 * p.nbb * p.nst * OBLK);
  p.b_B = ws_round(size_t(2) * p.nbb * p.nst * OBLK);
  p.b_G = ws_round(size_t(p.splits) * p.nf * 2 * p.nbb * OT * p.nbb * OT * 8);
}

// plans of one group of q points
std::vector<OzPlan> oz_plans(const std::vector<int>& qs, const int64_t* K, const int* nb, int nw, int sm) {
  std::vector<OzPlan> p;
  int64_t items = 0;
  for (int q : qs) {
    p.push_back(oz_plan(K[q], nb[q], nw));
    items += int64_t(p.back().ntile) * p.back().nf;
  }
  for (size_t i = 0; i < qs.size(); ++i) {
    const int64_t mine = int64_t(p[i].ntile) * p[i].nf;
    oz_splits(p[i], K[qs[i]], nw, int(std::max<int64_t>(1, (sm * mine + items / 2) / items)));
  }
  return p;
}

}  // namespace

size_t oz_sum_bytes(int sm) { return ws_round(size_t(sm) * OT * OT * sizeof(float)); }

int oz_cplx(const OzC* probs, int n, float* s, cudaStream_t st, const DeviceCtx& ctx) {
  for (int p0 = 0; p0 < n; p0 += OZC_MAX) {
    OzCBatch b;
    b.nq = std::min(OZC_MAX, n - p0);
    b.s = s;
    b.item0[0] = 0;
    for (int i = 0; i < b.nq; ++i) {
      b.q[i] = probs[p0 + i];
      b.item0[i + 1] = b.item0[i] + b.q[i].ntile * b.q[i].nprod;
    }
    int rc = launch_oz<OzCBatch>(k_oz_gemm_cplx, b, st, ctx);
    if (rc) return rc;
  }
  return GW_OK;
}

// From one stage of 32 rows on: K = 32, N_b = 8, 4 frequencies 0.08 ms against 0.14 with the FP64
// kernel, K = 128, N_b = 24 0.11 against 0.54 (16 such q in one call 0.18 against 0.55); fewer rows
// would be mostly padding.
bool oz_pol_eligible(int64_t K) { return K >= OKS; }

std::vector<std::vector<int>> oz_pol_groups(const std::vector<int>& qs, const int64_t* K, const int* nb,
                                            int nw) {
  std::vector<std::vector<int>> g;
  size_t bytes = 0;
  bool open = false;
  for (int q : qs) {
    const OzPlan p = oz_plan(K[q], nb[q], nw);
    const bool single = p.npass * p.nchunk == 1;
    if (!open || !single || int(g.back().size()) == OZQ || bytes + p.digits > DIGIT_BUDGET) {
      g.push_back({});
      bytes = 0;
    }
    g.back().push_back(q);
    bytes += p.digits;
    open = single;
  }
  return g;
}

size_t oz_pol_workspace(const std::vector<int>& group, const int64_t* K, const int* nb, int nw, int sm) {
  size_t b = 256 + oz_sum_bytes(sm);
  for (const OzPlan& p : oz_plans(group, K, nb, nw, sm)) b += p.total();
  return b;
}

int oz_pol(const std::vector<int>& group, const PolQ* qs, double pref, int nw, const OmegaArr& om,
           bool accumulate, void* ws, size_t ws_bytes, cudaStream_t s, const DeviceCtx& ctx,
           PolOpts& o) {
  const int n = int(group.size());
  std::vector<int64_t> K;
  std::vector<int> nb, idx;
  for (int i = 0; i < n; ++i) {
    K.push_back(qs[group[i]].K);
    nb.push_back(qs[group[i]].nb);
    idx.push_back(i);
  }
  const std::vector<OzPlan> plans = oz_plans(idx, K.data(), nb.data(), nw, ctx.sm_count);
  WsCursor cur{static_cast<char*>(ws), ws_bytes, 0};
  int* flags = static_cast<int*>(cur.take(256));
  static_assert(3 * OZQ * sizeof(int) <= 256, "flags and spreads");
  OzBatch b{};
  b.nq = n;
  b.s = static_cast<float*>(cur.take(oz_sum_bytes(ctx.sm_count)));
  std::vector<char*> exps(n);
  int64_t kmax = 0;
  for (int i = 0; i < n; ++i) {
    const OzPlan& p = plans[i];
    const PolQ& Q = qs[group[i]];
    OzProb& L = b.q[i];
    L.flag = flags + i;
    L.spread = flags + OZQ + 2 * i;
    L.w = static_cast<double*>(cur.take(p.b_w));
    L.part = static_cast<float2*>(cur.take(p.b_part));
    exps[i] = static_cast<char*>(cur.take(size_t(p.npass) * p.nchunk * (p.b_ea + p.b_eb)));
    L.A = static_cast<char*>(cur.take(p.b_A));
    L.B = static_cast<char*>(cur.take(p.b_B));
    L.G = static_cast<double*>(cur.take(p.b_G));
    if (!flags || !b.s || !L.w || !L.part || !exps[i] || !L.A || !L.B || !L.G)
      return set_error(GW_EWORKSPACE, "internal: FP64 slice workspace too small");
    L.delta = Q.delta;
    L.dbar = Q.dbar;
    L.f = Q.f;
    L.Kall = Q.K;
    L.nb = Q.nb;
    L.nbi = L.nbj = p.nbb;
    L.ntile = p.ntile;
    L.sbst = p.sbst;
    L.sps = p.sps;
    kmax = std::max(kmax, Q.K);
  }
  // the problems of a frequency chunk and K range (several only for a group of one q)
  const int npass = plans[0].npass, nchunk = plans[0].nchunk;
  auto set_pass = [&](int ch, int ps) {
    for (int i = 0; i < n; ++i) {
      const OzPlan& p = plans[i];
      const PolQ& Q = qs[group[i]];
      OzProb& L = b.q[i];
      const int f0 = ch * p.nf;
      const int64_t t0 = ps * p.rows;
      L.nf = std::min(p.nf, nw - f0);
      L.K = std::min(p.rows, Q.K - t0);
      L.nst = int((L.K + OKS - 1) / OKS);
      L.nsb = (L.nst + p.sbst - 1) / p.sbst;
      L.splits = (L.nsb + p.sps - 1) / p.sps;
      L.M = static_cast<const double2*>(Q.M) + t0 * Q.nb;
      L.wp = L.w + size_t(f0) * Q.K + t0;
      L.EA = reinterpret_cast<int*>(exps[i] + (size_t(ch) * npass + ps) * (p.b_ea + p.b_eb));
      L.EB = reinterpret_cast<int*>(reinterpret_cast<char*>(L.EA) + p.b_ea);
      L.P = reinterpret_cast<double2*>(Q.P) + size_t(f0) * Q.nb * Q.nb;
      b.item0[i + 1] = b.item0[i] + int64_t(p.ntile) * L.nf * L.splits;
    }
    b.add = ps > 0;                     // the first pass has the most splits: it writes every tile
  };
  auto over = [&](auto get) {           // the largest of a per-problem count
    int64_t m = 0;
    for (int i = 0; i < n; ++i) m = std::max<int64_t>(m, get(b.q[i]));
    return m;
  };
  const unsigned nq = unsigned(n);
  const int64_t cap = int64_t(ctx.sm_count) * 8;
  k_oz_weights<<<dim3(unsigned(std::min<int64_t>((kmax + 255) / 256, cap)), nq), 256, 0, s>>>(
      b, pref, nw, om, ctx.status);
  GW_LAUNCH_CHECK("k_oz_weights");
  // the exponents of the whole call first, so that the flags are final before P is touched
  for (int ch = 0; ch < nchunk; ++ch)
    for (int ps = 0; ps < npass; ++ps) {
      set_pass(ch, ps);
      const unsigned bl = unsigned(over([](const OzProb& L) { return int64_t(L.nbj); }));
      k_oz_scale<<<dim3(bl, unsigned(over([](const OzProb& L) { return (L.K + CHROWS - 1) / CHROWS; })), nq),
                   OT, 0, s>>>(b);
      GW_LAUNCH_CHECK("k_oz_scale");
      const int64_t ne = over([](const OzProb& L) { return int64_t(2 + 2 * L.nf) * L.nbj * OT * L.nsb; });
      k_oz_exps<<<dim3(unsigned((ne + 255) / 256), nq), 256, 0, s>>>(b);
      GW_LAUNCH_CHECK("k_oz_exps");
    }
  for (int ch = 0; ch < nchunk; ++ch) {
    for (int ps = 0; ps < npass; ++ps) {
      set_pass(ch, ps);
      k_oz_slice<<<dim3(unsigned(over([](const OzProb& L) { return int64_t(L.nst); })),
                        unsigned(over([](const OzProb& L) { return int64_t(4 * L.nbj); })), nq),
                   OT, 0, s>>>(b);
      GW_LAUNCH_CHECK("k_oz_slice");
      int rc = record_herk_event(o, o.launches, false, s);
      if (rc) return rc;
      if ((rc = launch_oz<OzBatch>(k_oz_gemm_pol, b, s, ctx))) return rc;
      if ((rc = launch_oz<OzBatch>(k_oz_gemm_pol6, b, s, ctx))) return rc;   // empty unless flagged
      if ((rc = record_herk_event(o, o.launches, true, s))) return rc;
      ++o.launches;
    }
    set_pass(ch, 0);                    // the splits of the first pass
    const int64_t tot = over([](const OzProb& L) { return int64_t(L.nf) * L.nb * L.nb; });
    k_oz_combine<<<dim3(unsigned(std::min<int64_t>((tot + 255) / 256, cap)), nq), 256, 0, s>>>(
        b, accumulate ? 1 : 0);
    GW_LAUNCH_CHECK("k_oz_combine");
  }
  return GW_OK;
}

// ------------------------------------------------------------------ pair coefficients
namespace {

// One problem per q, range of pairs and range of frequencies: the slices of x within half of the
// budget, those of U within the other half where one frequency allows; problems share launches.
struct PairPlan {
  int q, f0, nf;
  int64_t p0, np;
  int nst, nsb, nbi, nbj;
  size_t digits, b_part, b_ea, b_eb, b_eq, b_cols, b_A, b_B, b_c;
  size_t total() const { return b_part + b_ea + b_eb + b_eq + b_cols + b_A + b_B + b_c; }
};

std::vector<std::vector<PairPlan>> pair_batches(int nq, const int64_t* npair, const int* nb, int nw) {
  std::vector<std::vector<PairPlan>> out;
  size_t bytes = 0;
  for (int q = 0; q < nq; ++q) {
    if (npair[q] == 0) continue;
    const int nst = (2 * nb[q] + OKS - 1) / OKS, nbj = (2 * nb[q] + OT - 1) / OT;
    const size_t a1 = size_t(nst) * OBLK, u1 = size_t(nbj) * nst * OBLK;
    // (four grid rows per row block)
    const int64_t rmax = std::min<int64_t>(16000, std::max<int64_t>(1, int64_t(DIGIT_BUDGET / 2 / a1))) * OT;
    const int fmax = int(std::max<int64_t>(1, int64_t(DIGIT_BUDGET / 2 / u1)));
    for (int64_t p0 = 0; p0 < npair[q]; p0 += rmax)
      for (int f0 = 0; f0 < nw; f0 += fmax) {
        PairPlan p;
        p.q = q;
        p.f0 = f0;
        p.nf = std::min(fmax, nw - f0);
        p.p0 = p0;
        p.np = std::min(rmax, npair[q] - p0);
        p.nst = nst;
        p.nsb = (nst + SBMAX - 1) / SBMAX;
        p.nbi = int((p.np + OT - 1) / OT);
        p.nbj = nbj;
        p.b_A = ws_round(p.nbi * a1);
        p.b_B = ws_round(p.nf * u1);
        p.digits = p.b_A + p.b_B;
        p.b_part = ws_round(size_t(p.nf) * nbj * nbj * OT * sizeof(float2));
        p.b_ea = ws_round(size_t(p.nbi) * p.nsb * OT * 4);
        p.b_eb = ws_round(size_t(p.nf) * nbj * p.nsb * OT * 4);
        p.b_eq = ws_round(size_t(nb[q]) * sizeof(int));
        p.b_cols = ws_round(size_t(p.nf) * nbj * OT * sizeof(float2));
        p.b_c = ws_round(size_t(p.nf) * 2 * nbj * size_t(p.np) * 8);
        if (out.empty() || int(out.back().size()) == OZQ || bytes + p.digits > DIGIT_BUDGET) {
          out.push_back({});
          bytes = 0;
        }
        out.back().push_back(p);
        bytes += p.digits;
      }
  }
  return out;
}

}  // namespace

size_t oz_pair_workspace(int nq, const int64_t* npair, const int* nb, int nw, int sm) {
  size_t need = 0;
  for (const std::vector<PairPlan>& v : pair_batches(nq, npair, nb, nw)) {
    size_t b = 0;
    for (const PairPlan& p : v) b += p.total();
    need = std::max(need, b);
  }
  return need + ws_round(size_t(nq) * sizeof(int)) + oz_sum_bytes(sm);
}

int oz_pair(int nq, const int64_t* npair, const int* nb, const void* const* Msig, int nw,
            const double* const* Wc, double* const* c, void* ws, size_t ws_bytes, cudaStream_t s,
            const DeviceCtx& ctx) {
  WsCursor cur{static_cast<char*>(ws), ws_bytes, 0};
  int* flags = static_cast<int*>(cur.take(ws_round(size_t(nq) * sizeof(int))));
  float* ssum = static_cast<float*>(cur.take(oz_sum_bytes(ctx.sm_count)));
  if (!flags || !ssum) return set_error(GW_EWORKSPACE, "internal: FP64 pair workspace too small");
  GW_CUDA_TRY(cudaMemsetAsync(flags, 0, size_t(nq) * sizeof(int), s));
  const size_t base = cur.used;
  for (const std::vector<PairPlan>& v : pair_batches(nq, npair, nb, nw)) {
    cur.used = base;
    OzBatch b{};
    b.nq = int(v.size());
    b.s = ssum;
    int64_t nst = 0, nbi = 0, nbj = 0, nf = 0, nsb = 0, nred = 0, nrow = 0, nbmax = 0;
    for (int i = 0; i < b.nq; ++i) {
      const PairPlan& p = v[i];
      OzProb& L = b.q[i];
      L.flag = flags + p.q;
      L.part = static_cast<float2*>(cur.take(p.b_part));
      L.EA = static_cast<int*>(cur.take(p.b_ea));
      L.EB = static_cast<int*>(cur.take(p.b_eb));
      L.eq = static_cast<int*>(cur.take(p.b_eq));
      L.cols = static_cast<float2*>(cur.take(p.b_cols));
      L.A = static_cast<char*>(cur.take(p.b_A));
      L.B = static_cast<char*>(cur.take(p.b_B));
      L.cpart = static_cast<double*>(cur.take(p.b_c));
      if (!L.part || !L.EA || !L.EB || !L.eq || !L.cols || !L.A || !L.B || !L.cpart)
        return set_error(GW_EWORKSPACE, "internal: FP64 pair workspace too small");
      L.nb = nb[p.q];
      L.ncol = 2 * int64_t(nb[p.q]);
      L.nrow = p.np;
      L.x = static_cast<const double*>(Msig[p.q]) + p.p0 * L.ncol;
      L.M = reinterpret_cast<const double2*>(Wc[p.q]) + size_t(p.f0) * L.nb * L.nb;
      L.G = c[p.q] + size_t(p.f0) * npair[p.q] + p.p0;
      L.Kall = npair[p.q];
      L.nf = p.nf;
      L.nst = p.nst;
      L.nsb = p.nsb;
      L.sbst = SBMAX;
      L.sps = p.nsb;
      L.splits = 1;
      L.nbi = p.nbi;
      L.nbj = p.nbj;
      L.ntile = p.nbi * p.nbj;
      b.item0[i + 1] = b.item0[i] + int64_t(L.ntile) * L.nf;
      nst = std::max<int64_t>(nst, p.nst);
      nbi = std::max<int64_t>(nbi, p.nbi);
      nbj = std::max<int64_t>(nbj, p.nbj);
      nf = std::max<int64_t>(nf, p.nf);
      nsb = std::max<int64_t>(nsb, p.nsb);
      nred = std::max<int64_t>(nred, p.np * p.nf);
      nrow = std::max<int64_t>(nrow, p.np);
      nbmax = std::max<int64_t>(nbmax, L.nb);
    }
    const unsigned nq_ = unsigned(b.nq), nz = unsigned(b.nq * nf);
    const int64_t cap = int64_t(ctx.sm_count) * 16;
    k_oz_equilibrate<<<dim3(unsigned((nbmax + 31) / 32), nq_), 32 * EQF, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_oz_equilibrate");
    k_oz_rowexps<<<dim3(unsigned(std::min<int64_t>((nbi * OT * nsb + 7) / 8, cap)), nq_), 256, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_oz_rowexps");
    k_oz_uscale<<<dim3(unsigned(nbj), unsigned(nbj), nz), OT * UROWS, 0, s>>>(b, int(nf));
    GW_LAUNCH_CHECK("k_oz_uscale");
    k_oz_uexps<<<dim3(unsigned(std::min<int64_t>((nf * nbj * OT * nsb + 255) / 256, cap)), nq_), 256, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_oz_uexps");
    k_oz_pair_guard<<<dim3(unsigned((nrow + GP - 1) / GP), nq_), GT, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_oz_pair_guard");
    k_oz_slice_rows<<<dim3(unsigned(nst), unsigned(4 * nbi), nq_), OT, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_oz_slice_rows");
    k_oz_slice_u<<<dim3(unsigned(nst), unsigned(4 * nbj), nz), OT, 0, s>>>(b, int(nf));
    GW_LAUNCH_CHECK("k_oz_slice_u");
    int rc = launch_oz<OzBatch>(k_oz_gemm_quad, b, s, ctx);
    if (!rc) rc = launch_oz<OzBatch>(k_oz_gemm_quad6, b, s, ctx);    // empty unless a flag asks for it
    if (rc) return rc;
    k_oz_pair_reduce<<<dim3(unsigned(std::min<int64_t>((nred + 255) / 256, cap)), nq_), 256, 0, s>>>(b);
    GW_LAUNCH_CHECK("k_oz_pair_reduce");
  }
  return GW_OK;
}

}  // namespace gw
