// a7: learned initialiser of the multipole fit (Eq. modelf, N_p = 2): a multilayer
// perceptron 48 -> 128 -> 128 -> 8 with SiLU activations proposes (a_p, w_p) from the
// curve Sigma(i w_j) on 24 nodes; the FP64 Levenberg-Marquardt fit then starts there.
//
// Input: x = (Re y_j / s, Im y_j / s) interleaved per node, s = max_j |y_j| (1 if 0).
// Output o (8 values): a_p = s (o_{4p} + i o_{4p+1}), w_p = o_{4p+2} + i o_{4p+3}.
// Packed parameters (FP32): W1[128][48], b1[128], W2[128][128], b2[128], W3[8][128], b3[8].
//
// Inference (k_mlp_forward, k_mlp_start): BF16 storage arithmetic: the input, every weight
// and bias and both hidden activations are rounded to BF16 (round to nearest even), the
// dot products accumulate in FP32, SiLU is evaluated in FP32.
// Training (k_mlp_train): FP32 forward, the fit loss of the proposed parameters
//   L = (1/B) sum_b (1/24) sum_j |f_b(i w_j) - y_bj|^2 / s_b^2,
// its gradient by back-propagation (accumulated over the batch with FP32 atomics), and
// an optional Adam step (Kingma & Ba 2015; beta1 0.9, beta2 0.999, eps 1e-8).
//
// Inference: one CTA of 128 threads takes CPB curves; weights live in shared memory with padded
// row strides (49, 129) so that both row-wise and column-wise sweeps are free of bank
// conflicts; thread t owns hidden unit t for every curve of the CTA.
#include <cuda_bf16.h>

#include "gw_internal.cuh"

namespace gw {

namespace {

constexpr int NIN = MLP_NIN, NH = MLP_NH, NOUT = MLP_NOUT, NW = 24;
constexpr int S1 = NIN + 1;     // padded row stride of W1 in shared memory
constexpr int S2 = NH + 1;      // padded row stride of W2
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH,
              OFF_B2 = OFF_W2 + NH * NH, OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUT * NH;
static_assert(OFF_B3 + NOUT == MLP_NPARAM, "packed layout");
constexpr int CPB = 16;         // curves per CTA

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float dsilu_f(float z) {
  const float sg = 1.0f / (1.0f + expf(-z));
  return sg * (1.0f + z * (1.0f - sg));
}

struct MlpSmem {
  float W1[NH * S1];
  float W2[NH * S2];
  float W3[NOUT * NH];
  float b1[NH], b2[NH], b3[NOUT];
  float x[CPB][NIN];
  float h1[CPB][NH], h2[CPB][NH];
  float o[CPB][NOUT];
  double s[CPB];
};

// Weights into shared memory, rounded to BF16.
__device__ void load_weights(MlpSmem& S, const float* __restrict__ w) {
  for (int i = threadIdx.x; i < NH * NIN; i += blockDim.x) {
    const float v = w[OFF_W1 + i];
    S.W1[(i / NIN) * S1 + i % NIN] = bf16r(v);
  }
  for (int i = threadIdx.x; i < NH * NH; i += blockDim.x) {
    const float v = w[OFF_W2 + i];
    S.W2[(i / NH) * S2 + i % NH] = bf16r(v);
  }
  for (int i = threadIdx.x; i < NOUT * NH; i += blockDim.x) {
    const float v = w[OFF_W3 + i];
    S.W3[i] = bf16r(v);
  }
  for (int i = threadIdx.x; i < NH; i += blockDim.x) {
    S.b1[i] = bf16r(w[OFF_B1 + i]);
    S.b2[i] = bf16r(w[OFF_B2 + i]);
  }
  if (threadIdx.x < NOUT) S.b3[threadIdx.x] = bf16r(w[OFF_B3 + threadIdx.x]);
}

// Features of curves [c0, c0 + nc) into S.x and S.s (FP64 data, BF16 features).
__device__ void load_features(MlpSmem& S, const double2* __restrict__ sig, int c0, int nc) {
  if (threadIdx.x < CPB) {
    const int c = threadIdx.x;
    double m = 0.0;
    if (c < nc)
      for (int j = 0; j < NW; ++j) {
        const double2 y = sig[size_t(c0 + c) * NW + j];
        m = fmax(m, hypot(y.x, y.y));
      }
    S.s[c] = m > 0.0 ? m : 1.0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < CPB * NW; i += blockDim.x) {
    const int c = i / NW, j = i % NW;
    float re = 0.f, im = 0.f;
    if (c < nc) {
      const double2 y = sig[size_t(c0 + c) * NW + j];
      const double inv = 1.0 / S.s[c];
      re = float(y.x * inv);
      im = float(y.y * inv);
    }
    S.x[c][2 * j] = bf16r(re);
    S.x[c][2 * j + 1] = bf16r(im);
  }
  __syncthreads();
}

// Forward pass of the CTA's curves; outputs in S.o.
__device__ void forward(MlpSmem& S) {
  const int t = threadIdx.x;     // hidden unit
  float acc[CPB];
#pragma unroll
  for (int c = 0; c < CPB; ++c) acc[c] = S.b1[t];
  for (int k = 0; k < NIN; ++k) {
    const float w = S.W1[t * S1 + k];
#pragma unroll
    for (int c = 0; c < CPB; ++c) acc[c] = fmaf(w, S.x[c][k], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < CPB; ++c) {
    const float h = silu_f(acc[c]);
    S.h1[c][t] = bf16r(h);
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CPB; ++c) acc[c] = S.b2[t];
  for (int k = 0; k < NH; ++k) {
    const float w = S.W2[t * S2 + k];
#pragma unroll
    for (int c = 0; c < CPB; ++c) acc[c] = fmaf(w, S.h1[c][k], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < CPB; ++c) {
    const float h = silu_f(acc[c]);
    S.h2[c][t] = bf16r(h);
  }
  __syncthreads();
  {
    const int c = t / NOUT, o = t % NOUT;      // 128 threads = CPB x NOUT outputs
    float a = S.b3[o];
    for (int k = 0; k < NH; ++k) a = fmaf(S.W3[o * NH + k], S.h2[c][k], a);
    S.o[c][o] = a;
  }
  __syncthreads();
}
static_assert(CPB * NOUT == NH, "one output per thread in the last layer");

__global__ void __launch_bounds__(NH) k_mlp_forward(int n, const double2* __restrict__ sig,
                                                    const float* __restrict__ w,
                                                    float* __restrict__ out) {
  extern __shared__ __align__(16) char smraw[];
  MlpSmem& S = *reinterpret_cast<MlpSmem*>(smraw);
  load_weights(S, w);
  for (int c0 = blockIdx.x * CPB; c0 < n; c0 += gridDim.x * CPB) {
    const int nc = min(CPB, n - c0);
    load_features(S, sig, c0, nc);
    forward(S);
    const int c = threadIdx.x / NOUT, o = threadIdx.x % NOUT;
    if (c < nc) out[size_t(c0 + c) * NOUT + o] = S.o[c][o];
    __syncthreads();
  }
}

// Learned start of the fit: BF16 forward, decoded into theta = (Re a, Im a, Re w, Im w)_p.
__global__ void __launch_bounds__(NH) k_mlp_start(int n, const double2* __restrict__ sig,
                                                  const float* __restrict__ w,
                                                  double* __restrict__ theta) {
  extern __shared__ __align__(16) char smraw[];
  MlpSmem& S = *reinterpret_cast<MlpSmem*>(smraw);
  load_weights(S, w);
  for (int c0 = blockIdx.x * CPB; c0 < n; c0 += gridDim.x * CPB) {
    const int nc = min(CPB, n - c0);
    load_features(S, sig, c0, nc);
    forward(S);
    const int c = threadIdx.x / NOUT, o = threadIdx.x % NOUT;
    if (c < nc) {
      const double v = double(S.o[c][o]);
      theta[size_t(c0 + c) * NOUT + o] = (o % 4) < 2 ? v * S.s[c] : v;
    }
    __syncthreads();
  }
}

// One training pass over the batch: loss and gradient, added to grad and loss with FP32 atomics
// (both start at zero).
//
// A step's batch is small (512 curves by default) and latency bounds it, so it is spread over as
// many SMs as it fills: 512 threads take TC = 4 curves per pass, one (unit, curve) per thread. The
// forward sums run in the order of their inputs: a pole near a node amplifies their rounding a
// thousandfold, so a split would give another, equally rounded loss. The backward sum over the
// units is split over four groups of threads and folded through shared memory (one weight read
// feeds four curves), and every thread keeps its share of the gradient in registers over all
// passes of the CTA: four consecutive parameters, so that the batch sum takes one coalesced
// 16-byte atomic per four parameters at the end. 512 curves: 64.3 us with 16 curves per CTA of 128
// threads and one scattered atomic per parameter and pass; 14.9 us now.
constexpr int TTHREADS = 512, TC = 4, TG = TTHREADS / NH;
static_assert(TC == 4 && TG == 4, "float4 over the curves; one (unit, curve) per thread");
constexpr int S3 = NH + 4;                        // padded row stride of W3 and of h2
constexpr int TW = TTHREADS / 32, TROWS = NH / TW, TX = NH * NIN / 4 / TTHREADS;
static_assert(NH == 128 && TX * 4 * TTHREADS == NH * NIN, "gradient shares");

struct TrainSmem {
  float4 gz1T[NH], gz2T[NH];                     // [unit], one component per curve
  float4 part[TG][NH];                           // sums over a quarter of the inputs
  float x[TC][NIN], h1[TC][NH], h2[TC][S3], W3[NOUT * S3];
  float o[TC][NOUT], go[TC][NOUT], s[TC];
  float W1[NH * S1], W2[NH * S2];
  float b1[NH], b2[NH], b3[NOUT];
};

// a += w[0..3] . x[0..3], one after the other; x 16-byte aligned
__device__ __forceinline__ void dot4(float& a, const float* w, const float* x) {
  const float4 v = *reinterpret_cast<const float4*>(x);
  a = fmaf(w[0], v.x, a);
  a = fmaf(w[1], v.y, a);
  a = fmaf(w[2], v.z, a);
  a = fmaf(w[3], v.w, a);
}
__device__ __forceinline__ void fma4(float4& a, float w, const float4& x) {
  a.x = fmaf(w, x.x, a.x);
  a.y = fmaf(w, x.y, a.y);
  a.z = fmaf(w, x.z, a.z);
  a.w = fmaf(w, x.w, a.w);
}

// four consecutive floats at p (16-byte aligned when al)
__device__ __forceinline__ float4 load4(const float* __restrict__ p, bool al) {
  return al ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void add4(float* p, const float4& v, bool al) {
  if (al) {
    atomicAdd(reinterpret_cast<float4*>(p), v);
  } else {
    atomicAdd(p, v.x);
    atomicAdd(p + 1, v.y);
    atomicAdd(p + 2, v.z);
    atomicAdd(p + 3, v.w);
  }
}

// the total of unit t and curve c over the four input splits
__device__ __forceinline__ float part_sum(const TrainSmem& S, int t, int c) {
  float a = 0.f;
#pragma unroll
  for (int g = 0; g < TG; ++g) a += reinterpret_cast<const float*>(&S.part[g][t])[c];
  return a;
}

__global__ void __launch_bounds__(TTHREADS) k_mlp_train(int n, OmegaArr om,
                                                        const double2* __restrict__ sig,
                                                        const float* __restrict__ w,
                                                        float* __restrict__ grad,
                                                        float* __restrict__ loss, int al) {
  extern __shared__ __align__(16) char smraw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smraw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = tid & (NH - 1), g = tid / NH;      // unit; input split, or curve
  const float invB = 1.0f / float(n);
  // warp c < TC holds node `lane` of the pass's curve c
  auto node = [&](int c0) {
    return warp < TC && lane < NW && c0 + warp < n ? sig[size_t(c0 + warp) * NW + lane]
                                                   : make_double2(0.0, 0.0);
  };
  double2 y = node(int(blockIdx.x) * TC);
#pragma unroll
  for (int i = 0; i < NH * NH / 4 / TTHREADS; ++i) {
    const int e = 4 * (tid + i * TTHREADS);
    const float4 v = load4(w + OFF_W2 + e, al);
    float* d = S.W2 + (e / NH) * S2 + e % NH;
    d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
  }
#pragma unroll
  for (int i = 0; i < TX; ++i) {
    const int e = 4 * (tid + i * TTHREADS);
    const float4 v = load4(w + OFF_W1 + e, al);
    float* d = S.W1 + (e / NIN) * S1 + e % NIN;
    d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
  }
  for (int i = tid; i < NOUT * NH; i += TTHREADS) S.W3[(i / NH) * S3 + i % NH] = w[OFF_W3 + i];
  if (tid < NH) S.b1[tid] = w[OFF_B1 + tid];
  else if (tid < 2 * NH) S.b2[tid - NH] = w[OFF_B2 + tid - NH];
  else if (tid < 2 * NH + NOUT) S.b3[tid - 2 * NH] = w[OFF_B3 + tid - 2 * NH];

  float4 gw2[TROWS] = {}, gw1[TX] = {};            // this thread's share of the gradient
  float gw3[NOUT / TG] = {}, gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, gl = 0.f;
  for (int c0 = blockIdx.x * TC; c0 < n; c0 += gridDim.x * TC) {
    // features
    if (warp < TC) {
      double m = hypot(y.x, y.y);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) m = fmax(m, __shfl_xor_sync(~0u, m, d));
      if (!(m > 0.0)) m = 1.0;
      if (lane == 0) S.s[warp] = float(m);
      if (lane < NW) {
        const double inv = 1.0 / m;
        S.x[warp][2 * lane] = float(y.x * inv);
        S.x[warp][2 * lane + 1] = float(y.y * inv);
      }
    }
    __syncthreads();
    // forward: unit t of curve g, each sum in the order of its inputs
    float z1 = S.b1[t];
#pragma unroll
    for (int k = 0; k < NIN; k += 4) dot4(z1, S.W1 + t * S1 + k, &S.x[g][k]);
    S.h1[g][t] = silu_f(z1);
    __syncthreads();
    float z2 = S.b2[t];
#pragma unroll 8
    for (int k = 0; k < NH; k += 4) dot4(z2, S.W2 + t * S2 + k, &S.h1[g][k]);
    S.h2[g][t] = silu_f(z2);
    __syncthreads();
    if (tid < TC * NOUT) {
      const int c = tid / NOUT, o = tid % NOUT;
      float a = S.b3[o];
#pragma unroll 8
      for (int k = 0; k < NH; k += 4) dot4(a, S.W3 + o * S3 + k, &S.h2[c][k]);
      S.o[c][o] = a;
    }
    __syncthreads();
    // loss and dL/do (FP32 complex arithmetic), one node per lane
    if (warp < TC) {
      const int c = warp;
      const float s = S.s[c];
      float gr[NOUT] = {}, L = 0.f;
      if (lane < NW && c0 + c < n) {
        float ar[2], ai[2], pr[2], pi[2], fr = 0.f, fi = 0.f;
        const float oj = float(om.v[lane]);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          ar[p] = s * S.o[c][4 * p];
          ai[p] = s * S.o[c][4 * p + 1];
          // phi = 1 / (i w_j - w_p)
          const float dr = -S.o[c][4 * p + 2], di = oj - S.o[c][4 * p + 3];
          const float den = dr * dr + di * di;
          pr[p] = dr / den;
          pi[p] = -di / den;
          fr += ar[p] * pr[p] - ai[p] * pi[p];
          fi += ar[p] * pi[p] + ai[p] * pr[p];
        }
        const float coef = 2.0f * invB / (float(NW) * s * s);
        const float rr = fr - float(y.x), ri = fi - float(y.y);
        L = rr * rr + ri * ri;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          // d f / d(Re of output a) = s phi;  d f / d(Re w_p) = a_p phi^2
          const float qr = pr[p] * pr[p] - pi[p] * pi[p], qi = 2.f * pr[p] * pi[p];
          const float dwr = ar[p] * qr - ai[p] * qi, dwi = ar[p] * qi + ai[p] * qr;
          // Re(conj(r) D) and Re(conj(r) i D)
          gr[4 * p + 0] = coef * s * (rr * pr[p] + ri * pi[p]);
          gr[4 * p + 1] = coef * s * (rr * -pi[p] + ri * pr[p]);
          gr[4 * p + 2] = coef * (rr * dwr + ri * dwi);
          gr[4 * p + 3] = coef * (rr * -dwi + ri * dwr);
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        L += __shfl_xor_sync(~0u, L, d);
#pragma unroll
        for (int o = 0; o < NOUT; ++o) gr[o] += __shfl_xor_sync(~0u, gr[o], d);
      }
      gl += L * invB / (float(NW) * s * s);
      if (lane == 0) {
#pragma unroll
        for (int o = 0; o < NOUT; ++o) S.go[c][o] = gr[o];
      }
      y = node(c0 + int(gridDim.x) * TC);
    }
    __syncthreads();
    // back-propagation: gz2 = (go W3) * silu'(z2), gz1 = (gz2 W2) * silu'(z1)
    {
      float a = 0.f;
#pragma unroll
      for (int o = 0; o < NOUT; ++o) a = fmaf(S.go[g][o], S.W3[o * S3 + t], a);
      a *= dsilu_f(z2);
      gb2 += a;
      reinterpret_cast<float*>(&S.gz2T[t])[g] = a;
    }
    __syncthreads();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 16
    for (int u = 0; u < NH / TG; ++u)
      fma4(acc, S.W2[(g * (NH / TG) + u) * S2 + t], S.gz2T[g * (NH / TG) + u]);
    S.part[g][t] = acc;
    __syncthreads();
    {
      const float a = part_sum(S, t, g) * dsilu_f(z1);
      gb1 += a;
      reinterpret_cast<float*>(&S.gz1T[t])[g] = a;
    }
    // parameter gradients of the pass's curves: W2 rows warp * TROWS + i, columns 4 lane ..
    {
      float4 h[TC];
#pragma unroll
      for (int c = 0; c < TC; ++c) h[c] = *reinterpret_cast<const float4*>(&S.h1[c][4 * lane]);
#pragma unroll
      for (int i = 0; i < TROWS; ++i) {
        const float4 z = S.gz2T[warp * TROWS + i];
        fma4(gw2[i], z.x, h[0]);
        fma4(gw2[i], z.y, h[1]);
        fma4(gw2[i], z.z, h[2]);
        fma4(gw2[i], z.w, h[3]);
      }
#pragma unroll
      for (int i = 0; i < NOUT / TG; ++i)
#pragma unroll
        for (int c = 0; c < TC; ++c) gw3[i] = fmaf(S.go[c][g + i * TG], S.h2[c][t], gw3[i]);
      if (tid < NOUT) gb3 += S.go[0][tid] + S.go[1][tid] + S.go[2][tid] + S.go[3][tid];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TX; ++i) {
      const int e = tid + i * TTHREADS, r = e / (NIN / 4), k = 4 * (e % (NIN / 4));
      const float4 z = S.gz1T[r];
      fma4(gw1[i], z.x, *reinterpret_cast<const float4*>(&S.x[0][k]));
      fma4(gw1[i], z.y, *reinterpret_cast<const float4*>(&S.x[1][k]));
      fma4(gw1[i], z.z, *reinterpret_cast<const float4*>(&S.x[2][k]));
      fma4(gw1[i], z.w, *reinterpret_cast<const float4*>(&S.x[3][k]));
    }
    __syncthreads();
  }
  // this CTA's sums into the batch gradient
#pragma unroll
  for (int i = 0; i < TROWS; ++i)
    add4(grad + OFF_W2 + (warp * TROWS + i) * NH + 4 * lane, gw2[i], al);
#pragma unroll
  for (int i = 0; i < TX; ++i) add4(grad + OFF_W1 + 4 * (tid + i * TTHREADS), gw1[i], al);
#pragma unroll
  for (int i = 0; i < NOUT / TG; ++i) atomicAdd(grad + OFF_W3 + (g + i * TG) * NH + t, gw3[i]);
  S.part[g][t] = make_float4(gb1, gb2, 0.f, 0.f);
  __syncthreads();
  if (g < 2) atomicAdd(grad + (g == 0 ? OFF_B1 : OFF_B2) + t,
                       part_sum(S, t, g));
  if (tid < NOUT) atomicAdd(grad + OFF_B3 + tid, gb3);
  if (warp < TC && lane == 0) atomicAdd(loss, gl);
}

// gradient and loss to zero
__global__ void k_mlp_zero(float* __restrict__ grad, float* __restrict__ loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < MLP_NPARAM) grad[i] = 0.f;
  if (i == 0) *loss = 0.f;
}

__global__ void k_adam(int np, float* __restrict__ w, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, float lr, float bc1, float bc2) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

constexpr size_t SMEM_FWD = sizeof(MlpSmem);

int grid_for(int n, const DeviceCtx& ctx) {
  const int blocks = (n + CPB - 1) / CPB;
  return blocks < ctx.sm_count * 4 ? blocks : ctx.sm_count * 4;
}

template <typename K>
int set_smem(K kernel, size_t bytes) {
  GW_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
  return GW_OK;
}

}  // namespace

int mlp_forward(int n, const double* sigma, const float* w, float* out, cudaStream_t s) {
  DeviceCtx ctx;
  int rc = device_ctx(&ctx);
  if (rc) return rc;
  rc = set_smem(k_mlp_forward, SMEM_FWD);
  if (rc) return rc;
  k_mlp_forward<<<grid_for(n, ctx), NH, SMEM_FWD, s>>>(n, reinterpret_cast<const double2*>(sigma), w, out);
  GW_LAUNCH_CHECK("k_mlp_forward");
  return GW_OK;
}

int mlp_start(int n, const double* sigma, const float* w, double* theta, cudaStream_t s) {
  DeviceCtx ctx;
  int rc = device_ctx(&ctx);
  if (rc) return rc;
  rc = set_smem(k_mlp_start, SMEM_FWD);
  if (rc) return rc;
  k_mlp_start<<<grid_for(n, ctx), NH, SMEM_FWD, s>>>(n, reinterpret_cast<const double2*>(sigma), w, theta);
  GW_LAUNCH_CHECK("k_mlp_start");
  return GW_OK;
}

int mlp_train_step(int n, const OmegaArr& om, const double* sigma, float* w, float* grad, float* m,
                   float* v, float lr, int step, float* loss, cudaStream_t s) {
  DeviceCtx ctx;
  int rc = device_ctx(&ctx);
  if (rc) return rc;
  rc = set_smem(k_mlp_train, sizeof(TrainSmem));
  if (rc) return rc;
  k_mlp_zero<<<(MLP_NPARAM + 255) / 256, 256, 0, s>>>(grad, loss);
  GW_LAUNCH_CHECK("k_mlp_zero");
  const int al = (reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(grad)) % 16 == 0;
  const int grid = std::min((n + TC - 1) / TC, ctx.sm_count);
  k_mlp_train<<<grid, TTHREADS, sizeof(TrainSmem), s>>>(
      n, om, reinterpret_cast<const double2*>(sigma), w, grad, loss, al);
  GW_LAUNCH_CHECK("k_mlp_train");
  if (lr > 0.0f) {
    const float bc1 = 1.0f - powf(0.9f, float(step));
    const float bc2 = 1.0f - powf(0.999f, float(step));
    k_adam<<<(MLP_NPARAM + 255) / 256, 256, 0, s>>>(MLP_NPARAM, w, grad, m, v, lr, bc1, bc2);
    GW_LAUNCH_CHECK("k_adam");
  }
  return GW_OK;
}

}  // namespace gw
