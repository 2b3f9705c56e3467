// Learned initial guess for T2: a 3-layer MLP (width 128) mapping per-element
// features to a complex multiplier of the first-order amplitude,
//     x = (|t_MP2| / 0.05, -D / 10, |<ij||ab>| / max|<ij||ab>|),
//     h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), y = W3 h2 + b3,
//     t2 = (1 + y0 + i y1) t_MP2,
// trained on converged amplitudes of earlier solves (loss: mean |t2 - t2_conv|^2 /
// 0.05^2, Adam).  Hand-written forward, backward and update kernels.  bf16 mode
// (k_mlp_grad_bf, k_mlp_apply_bf): weights and activations rounded to BF16, and the
// three width-128 layer products (h1 W2^T forward, gz2 W2 and gz2^T h1 backward, the
// gradients rounded to BF16 as operands) on the tensor cores, mma m16n8k16 with FP32
// accumulation; check mode (k_mlp_grad, k_mlp_apply): plain FP32 on the SIMT pipes.
// The paper has no counterpart; the guess only changes the starting point of the
// amplitude iteration, never its fixed point.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <numeric>
#include <random>
#include <string>
#include <vector>

#include "ccsd.h"

namespace {
constexpr int NF = 3, W = 128, NO = 2;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + W * NF, OFF_W2 = OFF_B1 + W, OFF_B2 = OFF_W2 + W * W,
              OFF_W3 = OFF_B2 + W, OFF_B3 = OFF_W3 + NO * W, NPARAM = OFF_B3 + NO;
constexpr int TS = 32;  // samples per CTA tile
constexpr int MLP_SMEM = (2 * W * W + W * NF + 2 * W + NO * W + NO + 3 * TS * W + TS * NF + TS * NO) * 4 + 64;

struct Smem {
  float* W2;   // [u][k]
  float* W2T;  // [k][u]
  float* W1;   // [u][f]
  float* b1;
  float* b2;
  float* W3;   // [o][k]
  float* b3;
  float* h1;   // [s][u]
  float* h2;
  float* g;    // [s][u] gradient scratch
  float* x;    // [s][f]
  float* gy;   // [s][o]
};

__device__ Smem carve(float* base) {
  Smem m;
  m.W2 = base;
  m.W2T = m.W2 + W * W;
  m.W1 = m.W2T + W * W;
  m.b1 = m.W1 + W * NF;
  m.b2 = m.b1 + W;
  m.W3 = m.b2 + W;
  m.b3 = m.W3 + NO * W;
  m.h1 = m.b3 + NO;
  m.h2 = m.h1 + TS * W;
  m.g = m.h2 + TS * W;
  m.x = m.g + TS * W;
  m.gy = m.x + TS * NF;
  return m;
}

__device__ void load_params(const float* __restrict__ P, Smem& m) {
  for (int e = threadIdx.x; e < W * W; e += blockDim.x) {
    const int u = e / W, k = e % W;
    const float v = P[OFF_W2 + e];
    m.W2[e] = v;
    m.W2T[k * W + u] = v;
  }
  for (int e = threadIdx.x; e < W * NF; e += blockDim.x) m.W1[e] = P[OFF_W1 + e];
  for (int e = threadIdx.x; e < W; e += blockDim.x) { m.b1[e] = P[OFF_B1 + e]; m.b2[e] = P[OFF_B2 + e]; }
  for (int e = threadIdx.x; e < NO * W; e += blockDim.x) m.W3[e] = P[OFF_W3 + e];
  if (threadIdx.x < NO) m.b3[threadIdx.x] = P[OFF_B3 + threadIdx.x];
}

// forward for the TS samples whose features sit in m.x (ns valid); y into m.gy
__device__ void forward_tile(Smem& m, int ns) {
  for (int e = threadIdx.x; e < TS * W; e += blockDim.x) {
    const int s = e / W, u = e % W;
    float z = m.b1[u];
#pragma unroll
    for (int f = 0; f < NF; ++f) z += m.W1[u * NF + f] * m.x[s * NF + f];
    m.h1[e] = s < ns ? fmaxf(z, 0.f) : 0.f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < TS * W; e += blockDim.x) {
    const int s = e / W, u = e % W;
    float z = m.b2[u];
    for (int k = 0; k < W; ++k) z += m.W2T[k * W + u] * m.h1[s * W + k];
    m.h2[e] = s < ns ? fmaxf(z, 0.f) : 0.f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < TS * NO; e += blockDim.x) {
    const int s = e / NO, o = e % NO;
    float y = m.b3[o];
    for (int k = 0; k < W; ++k) y += m.W3[o * W + k] * m.h2[s * W + k];
    m.gy[e] = y;
  }
  __syncthreads();
}

// Gradient of the batch loss: idx[b0 .. b0+nb) index the sample arrays.  Each CTA
// walks tiles of TS samples (grid-stride) and keeps its gradient contributions in
// registers / shared memory owned by one thread each; one atomicAdd per entry per
// CTA at the end.
__global__ void __launch_bounds__(256) k_mlp_grad(const float* __restrict__ P, const float* __restrict__ X,
                                                  const float2* __restrict__ TM, const float2* __restrict__ TG,
                                                  const int* __restrict__ idx, int b0, int nb, float inv_n,
                                                  float* __restrict__ grad, double* __restrict__ loss) {
  extern __shared__ float sm[];
  Smem m = carve(sm);
  __shared__ float aW1[W * NF], ab1[W], ab2[W];
  __shared__ float lsum[TS];
  load_params(P, m);
  float gW2[W * W / 256];  // entries threadIdx.x + 256 j
  float gW3 = 0.f, gb3 = 0.f;
#pragma unroll
  for (int j = 0; j < W * W / 256; ++j) gW2[j] = 0.f;
  for (int e = threadIdx.x; e < W * NF; e += blockDim.x) aW1[e] = 0.f;
  for (int e = threadIdx.x; e < W; e += blockDim.x) { ab1[e] = 0.f; ab2[e] = 0.f; }
  double lacc = 0.0;
  const int ntile = (nb + TS - 1) / TS;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const int t0 = b0 + tile * TS;
    const int ns = max(0, min(TS, b0 + nb - t0));
    __syncthreads();
    for (int e = threadIdx.x; e < TS * NF; e += blockDim.x) {
      const int s = e / NF;
      m.x[e] = s < ns ? X[int64_t(idx[t0 + s]) * NF + e % NF] : 0.f;
    }
    __syncthreads();
    forward_tile(m, ns);
    if (threadIdx.x < TS) {
      const int s = threadIdx.x;
      float l = 0.f, g0 = 0.f, g1 = 0.f;
      if (s < ns) {
        const float2 tm = TM[idx[t0 + s]], tg = TG[idx[t0 + s]];
        const float mr = 1.f + m.gy[s * NO], mi = m.gy[s * NO + 1];
        const float rr = mr * tm.x - mi * tm.y - tg.x, ri = mr * tm.y + mi * tm.x - tg.y;
        const float c = 2.f * inv_n / (0.05f * 0.05f);
        l = (rr * rr + ri * ri) / (0.05f * 0.05f);
        g0 = c * (rr * tm.x + ri * tm.y);   // Re(conj(r) tmp2)
        g1 = c * (-rr * tm.y + ri * tm.x);  // Re(conj(r) i tmp2)
      }
      lsum[s] = l;
      m.gy[s * NO] = g0;
      m.gy[s * NO + 1] = g1;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int s = 0; s < TS; ++s) lacc += lsum[s];
    {  // output layer: entry threadIdx.x of W3 (NO * W == 256)
      const int o = threadIdx.x / W, k = threadIdx.x % W;
      for (int s = 0; s < ns; ++s) gW3 += m.gy[s * NO + o] * m.h2[s * W + k];
      if (threadIdx.x < NO)
        for (int s = 0; s < ns; ++s) gb3 += m.gy[s * NO + threadIdx.x];
    }
    for (int e = threadIdx.x; e < TS * W; e += blockDim.x) {  // gz2 = (gy W3) . relu'(z2)
      const int s = e / W, u = e % W;
      float a = 0.f;
#pragma unroll
      for (int o = 0; o < NO; ++o) a += m.gy[s * NO + o] * m.W3[o * W + u];
      m.g[e] = m.h2[e] > 0.f ? a : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < W * W / 256; ++j) {
      const int e = threadIdx.x + 256 * j, u = e / W, k = e % W;
      float a = 0.f;
      for (int s = 0; s < ns; ++s) a += m.g[s * W + u] * m.h1[s * W + k];
      gW2[j] += a;
    }
    if (threadIdx.x < W) {
      float a = 0.f;
      for (int s = 0; s < ns; ++s) a += m.g[s * W + threadIdx.x];
      ab2[threadIdx.x] += a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < TS * W; e += blockDim.x) {  // gz1 = (gz2 W2) . relu'(z1), over h2
      const int s = e / W, k = e % W;
      float a = 0.f;
      for (int u = 0; u < W; ++u) a += m.g[s * W + u] * m.W2[u * W + k];
      m.h2[e] = m.h1[e] > 0.f ? a : 0.f;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < W * NF; e += blockDim.x) {
      const int u = e / NF, f = e % NF;
      float a = 0.f;
      for (int s = 0; s < ns; ++s) a += m.h2[s * W + u] * m.x[s * NF + f];
      aW1[e] += a;
    }
    if (threadIdx.x < W) {
      float a = 0.f;
      for (int s = 0; s < ns; ++s) a += m.h2[s * W + threadIdx.x];
      ab1[threadIdx.x] += a;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < W * W / 256; ++j) atomicAdd(&grad[OFF_W2 + threadIdx.x + 256 * j], gW2[j]);
  atomicAdd(&grad[OFF_W3 + threadIdx.x], gW3);
  if (threadIdx.x < NO) atomicAdd(&grad[OFF_B3 + threadIdx.x], gb3);
  for (int e = threadIdx.x; e < W * NF; e += blockDim.x) atomicAdd(&grad[OFF_W1 + e], aW1[e]);
  for (int e = threadIdx.x; e < W; e += blockDim.x) {
    atomicAdd(&grad[OFF_B1 + e], ab1[e]);
    atomicAdd(&grad[OFF_B2 + e], ab2[e]);
  }
  if (threadIdx.x == 0) atomicAdd(loss, lacc * inv_n);
}

__global__ void k_adam(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ M1,
                       float* __restrict__ M2, int step, float lr) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NPARAM) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float g = G[k];
  const float m = b1 * M1[k] + (1.f - b1) * g, v = b2 * M2[k] + (1.f - b2) * g * g;
  M1[k] = m;
  M2[k] = v;
  const float mh = m / (1.f - powf(b1, float(step))), vh = v / (1.f - powf(b2, float(step)));
  P[k] -= lr * mh / (sqrtf(vh) + eps);
}

// First-order amplitude and features of one element from <ab||ij>, D and the instance's
// max |V|.  FP64 instructions are the cost (GB300 issues two a clock and SM): one square
// root serves |t| and |V| = |t| |D|.
__device__ __forceinline__ cplx elem_features(cplx v, double d, float vmax, float* x) {
  const cplx t = make_double2(v.x / d, v.y / d);
  const double ta = sqrt(t.x * t.x + t.y * t.y);  // (over- and underflow only beyond the FP32 range)
  x[0] = float(ta * 20.0);
  x[1] = float(d * -0.1);
  x[2] = vmax > 0.f ? float(ta * fabs(d)) / vmax : 0.f;
  return t;
}

__global__ void k_vmax(const cplx* __restrict__ V, int64_t vis, int64_t n2, float* __restrict__ vmax) {
  const int inst = blockIdx.y;
  unsigned long long q = 0;  // bits of the largest |V|^2: non-negative doubles order as their bits
  for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k < n2; k += int64_t(gridDim.x) * blockDim.x) {
    const cplx v = V[inst * vis + k];
    q = max(q, (unsigned long long)__double_as_longlong(fma(v.x, v.x, v.y * v.y)));
  }
  for (int o = 16; o; o >>= 1) q = max(q, __shfl_xor_sync(0xffffffffu, q, o));
  if ((threadIdx.x & 31) == 0)  // >= 0: int order = float order
    atomicMax((int*)&vmax[inst], __float_as_int(float(sqrt(__longlong_as_double((long long)q)))));
}

// training samples from the unique elements (a<b, i<j, no ghost) of converged instances
__global__ void k_extract(const cplx* __restrict__ V, int64_t vis, const double* __restrict__ D, const cplx* __restrict__ T,
                          int64_t namp, int64_t n1, const int64_t* __restrict__ elems, int ne,
                          const float* __restrict__ vmax, const int* __restrict__ inst_list, float* __restrict__ X,
                          float2* __restrict__ TM, float2* __restrict__ TG, int64_t base) {
  const int ii = blockIdx.y;
  const int inst = inst_list[ii];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < ne; k += gridDim.x * blockDim.x) {
    const int64_t p = elems[k];
    const int64_t o = base + int64_t(ii) * ne + k;
    float x[NF];
    const cplx tm = elem_features(V[inst * vis + p], D[inst * namp + n1 + p], vmax[inst], x);
    for (int f = 0; f < NF; ++f) X[o * NF + f] = x[f];
    TM[o] = make_float2(float(tm.x), float(tm.y));
    const cplx t = T[inst * namp + n1 + p];
    TG[o] = make_float2(float(t.x), float(t.y));
  }
}

// inference over every t2 element of every instance: t2 = (1 + y0 + i y1) <ab||ij> / D
__global__ void __launch_bounds__(256) k_mlp_apply(const float* __restrict__ P, const cplx* __restrict__ V, int64_t vis,
                                                   const double* __restrict__ D, cplx* __restrict__ T, int64_t namp,
                                                   int64_t n1, int64_t n2, const float* __restrict__ vmax) {
  extern __shared__ float sm[];
  Smem m = carve(sm);
  load_params(P, m);
  const int inst = blockIdx.y;
  __syncthreads();
  for (int64_t t0 = int64_t(blockIdx.x) * TS; t0 < n2; t0 += int64_t(gridDim.x) * TS) {
    const int ns = int(n2 - t0 < TS ? n2 - t0 : TS);
    for (int e = threadIdx.x; e < TS; e += blockDim.x) {
      if (e < ns) {
        elem_features(V[inst * vis + t0 + e], D[inst * namp + n1 + t0 + e], vmax[inst], &m.x[e * NF]);
      } else {
        for (int f = 0; f < NF; ++f) m.x[e * NF + f] = 0.f;
      }
    }
    __syncthreads();
    forward_tile(m, ns);
    for (int s = threadIdx.x; s < ns; s += blockDim.x) {
      const cplx v = V[inst * vis + t0 + s];
      const double d = D[inst * namp + n1 + t0 + s];
      const double mr = 1.0 + m.gy[s * NO], mi = m.gy[s * NO + 1];
      const double ar = v.x / d, ai = v.y / d;
      T[inst * namp + n1 + t0 + s] = make_double2(mr * ar - mi * ai, mr * ai + mi * ar);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// The bf16 mode.  Fragment layout of mma m16n8k16 .bf16 (PTX ISA; g = lane / 4, t = lane
// % 4): A registers {(g, 2t), (g + 8, 2t), (g, 2t + 8), (g + 8, 2t + 8)} with the next
// column in the high half; B registers {(2t, g), (2t + 8, g)} with the next row in the high
// half; D {(g, 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1)}.  So two neighbouring D
// column tiles, packed to BF16, are one A fragment of the next product, and a warp takes
// its samples through layers 1 and 2 in registers: layer 1 (three inputs) is computed
// straight into A fragments.  Layer 3 (two outputs) reads h2 back from shared memory, a
// whole row per lane, which sums y over the units in their order.
//
// What bounds it: instruction issue (the mma's with their operand loads and the FP32 layers
// about equally), then FP64 for the features.  The first
// form kept FP32 activations in shared memory, gathered every fragment element by element
// (12 loads and 6 conversions per mma) and gave the two-output layer to 64 of 256 threads:
// o=10 v=40, one guess of 64 instances (10.2 million elements): 28.6 -> 1.8 ms; one pass over
// 561,600 training samples in batches of 65,536: 2.52 -> 0.56 ms.
constexpr int LDB = W + 8;       // BF16 row stride in shared memory: 272 B, rows 16 B apart in the banks
constexpr int GT = 128;          // samples per group of the gradient: 16 per warp, four tiles of TS
constexpr int LDG = W + 4;       // FP32 row stride of gz1
constexpr int BF_THREADS = 256;
constexpr int BF_PART = (NPARAM + 31) / 32 * 32;  // row stride of the CTAs' shares of the gradient
// threads of the inference CTA: 3 of them an SM at up to 170 registers (168 used, 136 bytes spilled)
constexpr int BF_APPLY = 128;
constexpr int BF_PARAMS = W * 16 + W * 8 + W * 4;      // per unit: (W1 row, b1), W3 column, b2
constexpr int BF_FWD_SMEM = W * LDB * 2 + BF_PARAMS;   // + W2
constexpr int BF_APPLY_SMEM = BF_FWD_SMEM + BF_APPLY * LDB * 2;  // + h2
constexpr int BF_GRAD_SMEM = BF_FWD_SMEM + 3 * GT * LDB * 2 + GT * LDG * 4 + GT * 16 + GT * 8;

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }
__device__ __forceinline__ float bf_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// four 8 x 8 BF16 matrices; lane l gives the address of row l % 8 of matrix l / 8
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

struct BfParams {
  __nv_bfloat16* W2;  // [u][k], stride LDB
  float4* in;         // [u]: W1[u][0..2], b1[u]
  float2* W3;         // [u]: W3[0][u], W3[1][u]
  float* b2;          // [u]
};
__device__ BfParams bf_load(const float* __restrict__ P, uint8_t* base) {
  BfParams p;
  p.W2 = (__nv_bfloat16*)base;
  p.in = (float4*)(base + W * LDB * 2);
  p.W3 = (float2*)(p.in + W);
  p.b2 = (float*)(p.W3 + W);
  for (int e = threadIdx.x; e < W * W; e += blockDim.x)
    p.W2[(e / W) * LDB + e % W] = __float2bfloat16_rn(P[OFF_W2 + e]);
  for (int u = threadIdx.x; u < W; u += blockDim.x) {
    p.in[u] = make_float4(bf_round(P[OFF_W1 + u * NF]), bf_round(P[OFF_W1 + u * NF + 1]), bf_round(P[OFF_W1 + u * NF + 2]),
                          P[OFF_B1 + u]);
    p.W3[u] = make_float2(bf_round(P[OFF_W3 + u]), bf_round(P[OFF_W3 + W + u]));
    p.b2[u] = P[OFF_B2 + u];
  }
  return p;
}

// h1 = relu(W1 x + b1) of the warp's 16 samples as the A fragments of layer 2; x0, x1: the
// features of rows g and g + 8
__device__ __forceinline__ void bf_layer1(const BfParams& p, const float (&x0)[NF], const float (&x1)[NF],
                                          uint32_t (&a)[8][4]) {
  const int t = threadIdx.x & 3;
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const float4 u = p.in[16 * ks + 8 * half + 2 * t], w = p.in[16 * ks + 8 * half + 2 * t + 1];
      auto z = [](const float4& q, const float (&x)[NF]) {
        return fmaxf(q.w + q.x * x[0] + q.y * x[1] + q.z * x[2], 0.f);
      };
      a[ks][2 * half] = pack_bf16(z(u, x0), z(w, x0));
      a[ks][2 * half + 1] = pack_bf16(z(u, x1), z(w, x1));
    }
}

// Layer 2 of MT groups of 16 samples: h2 = relu(z2) rounded, to rows 16 mt + g (+ 8) of
// sh (row stride LDB).
template <int MT>
__device__ __forceinline__ void bf_layer2(const BfParams& p, const uint32_t (&a)[MT][8][4], __nv_bfloat16* sh) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // B[k][u] = W2[u][k]: matrices (u 0-7, k 0-7), (u 0-7, k 8-15), (u 8-15, k 0-7), (u 8-15, k 8-15)
  const __nv_bfloat16* wb = p.W2 + ((lane >> 4) * 8 + (lane & 7)) * LDB + ((lane >> 3) & 1) * 8;
#pragma unroll 2
  for (int n2 = 0; n2 < 8; ++n2) {  // 16 units at a time
    float d[MT][2][4] = {};
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      uint32_t b[4];
      ldsm4<false>(b, wb + 16 * n2 * LDB + 16 * ks);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        mma_16816(d[mt][0], a[mt][ks], b[0], b[1]);
        mma_16816(d[mt][1], a[mt][ks], b[2], b[3]);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float2 c = *reinterpret_cast<const float2*>(p.b2 + 16 * n2 + 8 * q + 2 * t);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int r = 0; r < 2; ++r)
          *reinterpret_cast<uint32_t*>(sh + (16 * mt + g + 8 * r) * LDB + 16 * n2 + 8 * q + 2 * t) =
              pack_bf16(fmaxf(d[mt][q][2 * r] + c.x, 0.f), fmaxf(d[mt][q][2 * r + 1] + c.y, 0.f));
    }
  }
}

// Gradient of the batch loss, bf16 mode.  A CTA walks tiles of TS samples (grid-stride),
// four at a time, a warp 16 samples: forward, loss, gz2 = (gy W3) . relu'(z2) and gz1 =
// (gz2 W2) . relu'(z1) in its own registers, then h1, h2, gz2 (BF16) and gz1 (FP32) of the
// group meet in shared memory for the sums over samples: gW2 = gz2^T h1 on the tensor
// cores (warp w the 16 rows u = 16w.., kept in registers over all tiles), the others in
// FP32, one chain per thread in sample order (a sum per tile for W1, b1 and b2, one running
// sum for W3 and b3).  Each CTA writes its share; k_mlp_fold adds them in a fixed order, so
// that equal samples give equal parameters in every run (summed by atomics, the shares'
// order differed from run to run, and with it the last bits of all that training led to).
__global__ void __launch_bounds__(BF_THREADS, 1)
    k_mlp_grad_bf(const float* __restrict__ P, const float* __restrict__ X, const float2* __restrict__ TM,
                  const float2* __restrict__ TG, const int* __restrict__ idx, int b0, int nb, float inv_n,
                  float* __restrict__ part, double* __restrict__ lpart) {
  extern __shared__ __align__(16) uint8_t bsm[];
  const BfParams p = bf_load(P, bsm);
  __syncthreads();
  __nv_bfloat16* sh1 = (__nv_bfloat16*)(bsm + BF_FWD_SMEM);  // [s][k]
  __nv_bfloat16* sh2 = sh1 + GT * LDB;                       // [s][u]
  __nv_bfloat16* sg2 = sh2 + GT * LDB;                       // [s][u]
  float* sg1 = (float*)(sg2 + GT * LDB);                     // [s][k]
  float4* sx = (float4*)(sg1 + GT * LDG);                    // [s] features
  float2* sgy = (float2*)(sx + GT);                          // [s] dL/dy
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float gW2[16][4] = {};
  const int cu = threadIdx.x & (W - 1), co = threadIdx.x / W;  // sums over samples: unit, output
  const float2 w3 = p.W3[cu];
  float cW3 = 0.f, cb3 = 0.f, cb2 = 0.f, cb1 = 0.f, cW1[NF] = {};
  double lacc = 0.0;
  const int ntile = (nb + TS - 1) / TS;
  for (int tile0 = blockIdx.x; tile0 < ntile; tile0 += 4 * gridDim.x) {
    // 16-sample piece w of the group: half w % 2 of tile tile0 + (w / 2) gridDim; the live
    // pieces are the first np
    auto first = [&](int w) { return (tile0 + (w >> 1) * int(gridDim.x)) * TS + 16 * (w & 1); };
    int np = 0;
    while (np < GT / 16 && first(np) < nb) ++np;
    const int t0 = first(warp);  // the warp's first sample in the batch
    if (warp < np) {
      // lane l < 16 reads sample l of the warp's
      float4 xs = make_float4(0.f, 0.f, 0.f, 0.f);
      float2 tm = make_float2(0.f, 0.f), tg = tm;
      if (lane < 16 && t0 + lane < nb) {
        const int64_t k = idx[b0 + t0 + lane];
        xs = make_float4(X[k * NF], X[k * NF + 1], X[k * NF + 2], 0.f);
        tm = TM[k];
        tg = TG[k];
      }
      if (lane < 16) sx[16 * warp + lane] = xs;
      float xr[2][NF];
      float2 tmr[2], tgr[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        xr[r][0] = __shfl_sync(0xffffffffu, xs.x, g + 8 * r);
        xr[r][1] = __shfl_sync(0xffffffffu, xs.y, g + 8 * r);
        xr[r][2] = __shfl_sync(0xffffffffu, xs.z, g + 8 * r);
        tmr[r] = make_float2(__shfl_sync(0xffffffffu, tm.x, g + 8 * r), __shfl_sync(0xffffffffu, tm.y, g + 8 * r));
        tgr[r] = make_float2(__shfl_sync(0xffffffffu, tg.x, g + 8 * r), __shfl_sync(0xffffffffu, tg.y, g + 8 * r));
      }
      uint32_t a[1][8][4];
      bf_layer1(p, xr[0], xr[1], a[0]);
      bf_layer2<1>(p, a, sh2 + 16 * warp * LDB);
      __syncwarp();
      // layer 3: lane = (sample, output)
      float y;
      {
        const int o = lane >> 4;
        const __nv_bfloat16* h = sh2 + (16 * warp + (lane & 15)) * LDB;
        const float* wo = reinterpret_cast<const float*>(p.W3) + o;
        y = P[OFF_B3 + o];
#pragma unroll 4
        for (int k = 0; k < W; k += 8) {
          const uint4 q = *reinterpret_cast<const uint4*>(h + k);
          const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            y += wo[2 * (k + 2 * j)] * bf_lo(v[j]);
            y += wo[2 * (k + 2 * j + 1)] * bf_hi(v[j]);
          }
        }
      }
      // loss and dL/dy of rows g and g + 8 (zero past the batch)
      float gy[2][NO];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float mr = 1.f + __shfl_sync(0xffffffffu, y, g + 8 * r), mi = __shfl_sync(0xffffffffu, y, 16 + g + 8 * r);
        const float rr = mr * tmr[r].x - mi * tmr[r].y - tgr[r].x, ri = mr * tmr[r].y + mi * tmr[r].x - tgr[r].y;
        const float c = 2.f * inv_n / (0.05f * 0.05f);
        const bool live = t0 + g + 8 * r < nb;
        gy[r][0] = live ? c * (rr * tmr[r].x + ri * tmr[r].y) : 0.f;   // Re(conj(r) tmp2)
        gy[r][1] = live ? c * (-rr * tmr[r].y + ri * tmr[r].x) : 0.f;  // Re(conj(r) i tmp2)
        if (t == 0) {
          if (live) lacc += double((rr * rr + ri * ri) / (0.05f * 0.05f));
          sgy[16 * warp + g + 8 * r] = make_float2(gy[r][0], gy[r][1]);
        }
      }
      // gz2, packed as the A fragments of gz2 W2, and h1, gz2 into shared memory
      uint32_t ga[8][4];
#pragma unroll
      for (int nt = 0; nt < 16; ++nt) {
        const float2 u = p.W3[8 * nt + 2 * t], w = p.W3[8 * nt + 2 * t + 1];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int at = (16 * warp + g + 8 * r) * LDB + 8 * nt + 2 * t;
          const uint32_t h = *reinterpret_cast<const uint32_t*>(sh2 + at);
          const float q0 = __fmaf_rn(gy[r][1], u.y, __fmul_rn(gy[r][0], u.x));
          const float q1 = __fmaf_rn(gy[r][1], w.y, __fmul_rn(gy[r][0], w.x));
          const uint32_t v = pack_bf16((h & 0xFFFFu) ? q0 : 0.f, (h >> 16) ? q1 : 0.f);
          ga[nt >> 1][(nt & 1) * 2 + r] = v;
          *reinterpret_cast<uint32_t*>(sh1 + at) = a[0][nt >> 1][(nt & 1) * 2 + r];
          *reinterpret_cast<uint32_t*>(sg2 + at) = v;
        }
      }
      // gz1: B[u][k] = W2[u][k] through transposed loads, 16 columns k at a time
      const __nv_bfloat16* wt = p.W2 + (((lane >> 3) & 1) * 8 + (lane & 7)) * LDB + (lane >> 4) * 8;
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) {
        float d[2][4] = {};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          uint32_t b[4];
          ldsm4<true>(b, wt + 16 * ks * LDB + 16 * n2);
          mma_16816(d[0], ga[ks], b[0], b[1]);
          mma_16816(d[1], ga[ks], b[2], b[3]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const uint32_t h = a[0][n2][2 * q + r];  // h1 at the same place: relu'(z1)
            *reinterpret_cast<float2*>(sg1 + (16 * warp + g + 8 * r) * LDG + 16 * n2 + 8 * q + 2 * t) =
                make_float2((h & 0xFFFFu) ? d[q][2 * r] : 0.f, (h >> 16) ? d[q][2 * r + 1] : 0.f);
          }
      }
    }
    __syncthreads();
    // gW2 += gz2^T h1 over the group's samples
    {
      const __nv_bfloat16* pa = sg2 + ((lane >> 4) * 8 + (lane & 7)) * LDB + 16 * warp + ((lane >> 3) & 1) * 8;
      const __nv_bfloat16* pb = sh1 + (((lane >> 3) & 1) * 8 + (lane & 7)) * LDB + (lane >> 4) * 8;
#pragma unroll 2
      for (int ks = 0; ks < np; ++ks) {
        uint32_t am[4];
        ldsm4<true>(am, pa + 16 * ks * LDB);
#pragma unroll
        for (int n2 = 0; n2 < 8; ++n2) {
          uint32_t b[4];
          ldsm4<true>(b, pb + 16 * ks * LDB + 16 * n2);
          mma_16816(gW2[2 * n2], am, b[0], b[1]);
          mma_16816(gW2[2 * n2 + 1], am, b[2], b[3]);
        }
      }
    }
    // sums over the samples, a tile at a time
    for (int s0 = 0; s0 < 16 * np; s0 += TS) {
      const int s1 = min(s0 + TS, 16 * np);
      if (co == 0) {  // W3[0], b2, b3[0]
        float a = 0.f;
#pragma unroll 8
        for (int s = s0; s < s1; ++s) {
          const float2 q = sgy[s];
          const float h = __bfloat162float(sh2[s * LDB + cu]);
          cW3 = __fmaf_rn(q.x, h, cW3);
          cb3 += q.x;
          a += h > 0.f ? __fmaf_rn(q.y, w3.y, __fmul_rn(q.x, w3.x)) : 0.f;
        }
        cb2 += a;
      } else {  // W3[1], b3[1], W1, b1
        float a = 0.f, a1[NF] = {};
#pragma unroll 8
        for (int s = s0; s < s1; ++s) {
          const float q = sgy[s].y;
          cW3 = __fmaf_rn(q, __bfloat162float(sh2[s * LDB + cu]), cW3);
          cb3 += q;
          const float z = sg1[s * LDG + cu];
          const float4 x = sx[s];
          a += z;
          a1[0] = __fmaf_rn(z, x.x, a1[0]);
          a1[1] = __fmaf_rn(z, x.y, a1[1]);
          a1[2] = __fmaf_rn(z, x.z, a1[2]);
        }
        cb1 += a;
#pragma unroll
        for (int f = 0; f < NF; ++f) cW1[f] += a1[f];
      }
    }
    __syncthreads();
  }
  float* out = part + int64_t(blockIdx.x) * BF_PART;
#pragma unroll
  for (int nt = 0; nt < 16; ++nt)
#pragma unroll
    for (int r = 0; r < 2; ++r)
      *reinterpret_cast<float2*>(&out[OFF_W2 + (16 * warp + g + 8 * r) * W + 8 * nt + 2 * t]) =
          make_float2(gW2[nt][2 * r], gW2[nt][2 * r + 1]);
  out[OFF_W3 + threadIdx.x] = cW3;
  if (cu == 0) out[OFF_B3 + co] = cb3;
  if (co == 0) {
    out[OFF_B2 + cu] = cb2;
  } else {
    out[OFF_B1 + cu] = cb1;
#pragma unroll
    for (int f = 0; f < NF; ++f) out[OFF_W1 + cu * NF + f] = cW1[f];
  }
  for (int o = 16; o; o >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
  if (lane == 0) lpart[int64_t(blockIdx.x) * (BF_THREADS / 32) + warp] = lacc * inv_n;
}

// The gradient and the loss from the shares of n CTAs, each entry summed in one order: 32
// entries a CTA, its warp w the shares w, w + 8, ..., then the warps in turn; the last CTA
// adds the loss.
__global__ void __launch_bounds__(BF_THREADS) k_mlp_fold(const float* __restrict__ part, const double* __restrict__ lpart,
                                                         int n, float* __restrict__ grad, double* __restrict__ loss) {
  constexpr int NW = BF_THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x == gridDim.x - 1) {
    if (warp) return;
    double s = 0.0;
    for (int k = lane; k < n * NW; k += 32) s += lpart[k];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) *loss += s;
    return;
  }
  __shared__ float sums[NW][32];
  const int k = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (k < NPARAM) {
#pragma unroll 8
    for (int c = warp; c < n; c += NW) s += part[int64_t(c) * BF_PART + k];
  }
  sums[warp][lane] = s;
  __syncthreads();
  if (warp || k >= NPARAM) return;
#pragma unroll
  for (int w = 1; w < NW; ++w) s += sums[w][lane];
  grad[k] = s;
}

// Inference, bf16 mode: 32 elements per warp step, one per lane for the features, layer 3
// and the result, two 16-row groups for layer 2 (each W2 fragment load serves both).
__global__ void __launch_bounds__(BF_APPLY, 3) k_mlp_apply_bf(const float* __restrict__ P, const cplx* __restrict__ V,
                                                              int64_t vis, const double* __restrict__ D,
                                                              cplx* __restrict__ T, int64_t namp, int64_t n1, int64_t n2,
                                                              const float* __restrict__ vmax) {
  extern __shared__ __align__(16) uint8_t bsm[];
  const BfParams p = bf_load(P, bsm);
  __syncthreads();
  const int inst = blockIdx.y, lane = threadIdx.x & 31, g = lane >> 2;
  __nv_bfloat16* sh = (__nv_bfloat16*)(bsm + BF_FWD_SMEM) + (threadIdx.x & ~31) * LDB;  // the warp's h2
  const float vm = vmax[inst];
  const cplx* v = V + inst * vis;
  const double* d = D + inst * namp + n1;
  cplx* out = T + inst * namp + n1;
  const int64_t step = int64_t(gridDim.x) * BF_APPLY;
  for (int64_t w0 = int64_t(blockIdx.x) * BF_APPLY + (threadIdx.x & ~31); w0 < n2; w0 += step) {
    const int64_t e = w0 + lane;
    float x[NF] = {0.f, 0.f, 0.f};
    cplx tm = make_double2(0.0, 0.0);
    if (e < n2) tm = elem_features(v[e], d[e], vm, x);
    uint32_t a[2][8][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      float x0[NF], x1[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        x0[f] = __shfl_sync(0xffffffffu, x[f], 16 * mt + g);
        x1[f] = __shfl_sync(0xffffffffu, x[f], 16 * mt + g + 8);
      }
      bf_layer1(p, x0, x1, a[mt]);
    }
    bf_layer2<2>(p, a, sh);
    __syncwarp();
    float y0 = P[OFF_B3], y1 = P[OFF_B3 + 1];
#pragma unroll 4
    for (int k = 0; k < W; k += 8) {
      const uint4 q = *reinterpret_cast<const uint4*>(sh + lane * LDB + k);
      const uint32_t h[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 w = *reinterpret_cast<const float4*>(p.W3 + k + 2 * j);
        y0 += w.x * bf_lo(h[j]);
        y1 += w.y * bf_lo(h[j]);
        y0 += w.z * bf_hi(h[j]);
        y1 += w.w * bf_hi(h[j]);
      }
    }
    __syncwarp();
    if (e < n2) {
      const double mr = 1.0 + y0, mi = y1;
      out[e] = make_double2(mr * tm.x - mi * tm.y, mr * tm.y + mi * tm.x);
    }
  }
}

__global__ void k_zero_t1(cplx* __restrict__ T, int64_t namp, int64_t n1) {
  const int inst = blockIdx.y;
  for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k < n1; k += int64_t(gridDim.x) * blockDim.x)
    T[inst * namp + k] = make_double2(0.0, 0.0);
}

__global__ void k_init_params(float* __restrict__ P, uint64_t seed) {
  // He-style initialisation of W1, W2 from a hashed counter; zero biases and output layer
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NPARAM) return;
  float v = 0.f;
  if (k < OFF_B1 || (k >= OFF_W2 && k < OFF_B2)) {
    uint64_t z = seed * 0x9E3779B97F4A7C15ull + uint64_t(k) * 0xBF58476D1CE4E5B9ull;
    z ^= z >> 31; z *= 0x94D049BB133111EBull; z ^= z >> 29;
    const float u1 = ((z >> 11) + 0.5f) * 0x1p-53f, u2 = (((z * 0x2545F4914F6CDD1Dull) >> 11) + 0.5f) * 0x1p-53f;
    const float g = sqrtf(-2.f * logf(u1)) * cosf(6.2831853f * u2);
    v = g * (k < OFF_B1 ? sqrtf(2.f / NF) : sqrtf(2.f / W));
  }
  P[k] = v;
}
}  // namespace

// ---------------------------------------------------------------------------
struct exp_mlp {
  exp_allocator alloc{};
  cudaStream_t stream = nullptr;
  int bf = 1;
  int sms = 1;
  int step = 0;
  float* P = nullptr;
  float* G = nullptr;
  float* M1 = nullptr;
  float* M2 = nullptr;
  double* d_loss = nullptr;
  float* part = nullptr;    // bf16 mode: the CTAs' shares of the gradient and the loss
  double* lpart = nullptr;
  float* X = nullptr;
  float2* TM = nullptr;
  float2* TG = nullptr;
  int* idx = nullptr;
  int64_t n = 0, cap = 0;
  std::vector<void*> owned;
  std::string err;
  void* al(size_t b) {
    void* p = alloc.alloc(std::max<size_t>(b, 256), alloc.user);
    if (!p) throw ExpError{EXP_ENOMEM, "allocator returned NULL"};
    owned.push_back(p);
    return p;
  }
};

static thread_local std::string g_mlp_err;

#define MLP_TRY try {
#define MLP_CATCH(m)                                                                     \
  }                                                                                      \
  catch (const ExpError& e) {                                                            \
    g_mlp_err = e.msg;                                                                   \
    if (m) (m)->err = e.msg;                                                             \
    return e.s;                                                                          \
  }                                                                                      \
  catch (const CudaError& e) {                                                           \
    g_mlp_err = std::string(e.where) + ": " + cudaGetErrorString(e.e);                   \
    if (m) (m)->err = g_mlp_err;                                                         \
    return EXP_ECUDA;                                                                    \
  }

extern "C" int exp_mlp_num_params(void) { return NPARAM; }

extern "C" exp_status exp_mlp_create(const exp_allocator* alloc, void* stream, uint64_t seed, int bf16,
                                     exp_mlp** out) {
  exp_mlp* m = nullptr;
  MLP_TRY
  if (!alloc || !alloc->alloc || !alloc->free || !out) throw ExpError{EXP_EINVAL, "null argument"};
  m = new exp_mlp();
  m->alloc = *alloc;
  m->stream = (cudaStream_t)stream;
  m->bf = bf16 ? 1 : 0;
  int dev = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, dev));
  m->P = (float*)m->al(sizeof(float) * NPARAM);
  m->G = (float*)m->al(sizeof(float) * NPARAM);
  m->M1 = (float*)m->al(sizeof(float) * NPARAM);
  m->M2 = (float*)m->al(sizeof(float) * NPARAM);
  m->d_loss = (double*)m->al(sizeof(double));
  CK(cudaMemsetAsync(m->M1, 0, sizeof(float) * NPARAM, m->stream));
  CK(cudaMemsetAsync(m->M2, 0, sizeof(float) * NPARAM, m->stream));
  k_init_params<<<(NPARAM + 255) / 256, 256, 0, m->stream>>>(m->P, seed);
  CK(cudaGetLastError());
  CK(cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM));
  CK(cudaFuncSetAttribute(k_mlp_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM));
  CK(cudaFuncSetAttribute(k_mlp_grad_bf, cudaFuncAttributeMaxDynamicSharedMemorySize, BF_GRAD_SMEM));
  CK(cudaFuncSetAttribute(k_mlp_apply_bf, cudaFuncAttributeMaxDynamicSharedMemorySize, BF_APPLY_SMEM));
  CK(cudaStreamSynchronize(m->stream));
  *out = m;
  return EXP_OK;
  }
  catch (const ExpError& e) {
    g_mlp_err = e.msg;
    if (m) { for (void* p : m->owned) m->alloc.free(p, m->alloc.user); delete m; }
    return e.s;
  }
  catch (const CudaError& e) {
    g_mlp_err = std::string(e.where) + ": " + cudaGetErrorString(e.e);
    if (m) { for (void* p : m->owned) m->alloc.free(p, m->alloc.user); delete m; }
    return EXP_ECUDA;
  }
}

extern "C" void exp_mlp_destroy(exp_mlp* m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  for (void* p : m->owned) m->alloc.free(p, m->alloc.user);
  delete m;
}

extern "C" const char* exp_mlp_last_error(const exp_mlp* m) {
  return m && !m->err.empty() ? m->err.c_str() : g_mlp_err.c_str();
}

extern "C" exp_status exp_mlp_params(exp_mlp* m, float* get, const float* set) {
  MLP_TRY
  if (!m) throw ExpError{EXP_EINVAL, "null model"};
  if (set) {
    CK(cudaMemcpyAsync(m->P, set, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, m->stream));
    CK(cudaMemsetAsync(m->M1, 0, sizeof(float) * NPARAM, m->stream));
    CK(cudaMemsetAsync(m->M2, 0, sizeof(float) * NPARAM, m->stream));
    m->step = 0;
  }
  if (get) CK(cudaMemcpyAsync(get, m->P, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream));
  CK(cudaStreamSynchronize(m->stream));
  return EXP_OK;
  MLP_CATCH(m)
}

static void ensure_capacity(exp_mlp* m, int64_t need) {
  if (need <= m->cap) return;
  const int64_t cap = std::max<int64_t>(need, 2 * m->cap);
  float* X = (float*)m->al(sizeof(float) * NF * cap);
  float2* TM = (float2*)m->al(sizeof(float2) * cap);
  float2* TG = (float2*)m->al(sizeof(float2) * cap);
  int* idx = (int*)m->al(sizeof(int) * cap);
  if (m->n) {
    CK(cudaMemcpyAsync(X, m->X, sizeof(float) * NF * m->n, cudaMemcpyDeviceToDevice, m->stream));
    CK(cudaMemcpyAsync(TM, m->TM, sizeof(float2) * m->n, cudaMemcpyDeviceToDevice, m->stream));
    CK(cudaMemcpyAsync(TG, m->TG, sizeof(float2) * m->n, cudaMemcpyDeviceToDevice, m->stream));
  }
  m->X = X;
  m->TM = TM;
  m->TG = TG;
  m->idx = idx;
  m->cap = cap;
}

// vmax per instance of a context, on the context stream
static float* ctx_vmax(exp_mlp* m, Ctx& c) {
  const Tensor* Vd = ccsd_driver_integral(c);
  float* vm = (float*)m->al(sizeof(float) * c.ninst);
  CK(cudaMemsetAsync(vm, 0, sizeof(float) * c.ninst, c.stream));
  k_vmax<<<dim3(std::max<int64_t>(1, std::min<int64_t>((c.n2 + 255) / 256, 304)), c.ninst), 256, 0, c.stream>>>(
      Vd->d, Vd->is, c.n2, vm);
  CK(cudaGetLastError());
  return vm;
}

extern "C" exp_status exp_mlp_add_training_data(exp_mlp* m, exp_ctx* x) {
  MLP_TRY
  if (!m || !x) throw ExpError{EXP_EINVAL, "null argument"};
  Ctx& c = x->c;
  if (!c.guessed) throw ExpError{EXP_ESTATE, "context has no amplitudes"};
  CK(cudaStreamSynchronize(m->stream));
  // converged instances only
  std::vector<int> st(4 * c.ninst), list;
  CK(cudaMemcpy(st.data(), c.d_diis_state, sizeof(int) * 4 * c.ninst, cudaMemcpyDeviceToHost));
  for (int k = 0; k < c.ninst; ++k)
    if (st[k * 4 + 2] == 1) list.push_back(k);  // converged (2 = failed)
  if (list.empty()) return EXP_OK;
  // unique real elements a<b, i<j of the t2 layout
  std::vector<SubBlock> sb;
  enumerate_blocks(c.t2.L, c.spaces, sb);
  std::vector<int64_t> el;
  const Space& SO = c.spaces[SP_OCC];
  const Space& SV = c.spaces[SP_VIRT];
  for (auto& b : sb)
    for (int la = 0; la < b.n[0]; ++la)
      for (int lb = 0; lb < b.n[1]; ++lb) {
        const int ga = SV.off[b.irr[0]] + la, gb = SV.off[b.irr[1]] + lb;
        if (ga >= gb) continue;
        for (int li = 0; li < b.n[2]; ++li)
          for (int lj = 0; lj < b.n[3]; ++lj) {
            const int gi = SO.off[b.irr[2]] + li, gj = SO.off[b.irr[3]] + lj;
            if (gi >= gj || c.occ_real[gi] < 0 || c.occ_real[gj] < 0) continue;
            el.push_back(b.base + la * b.st[0] + lb * b.st[1] + li * b.st[2] + lj * b.st[3]);
          }
      }
  const int ne = int(el.size());
  const int64_t add = int64_t(ne) * list.size();
  ensure_capacity(m, m->n + add);
  CK(cudaStreamSynchronize(m->stream));
  int64_t* d_el = (int64_t*)c.dalloc(sizeof(int64_t) * std::max(ne, 1));
  int* d_list = (int*)c.dalloc(sizeof(int) * list.size());
  upload(c, d_el, el.data(), sizeof(int64_t) * ne);
  upload(c, d_list, list.data(), sizeof(int) * list.size());
  float* vm = ctx_vmax(m, c);
  const Tensor* Vd = ccsd_driver_integral(c);
  k_extract<<<dim3(std::max(1, std::min((ne + 255) / 256, 1024)), int(list.size())), 256, 0, c.stream>>>(
      Vd->d, Vd->is, c.d_D, c.d_T, c.namp, c.n1, d_el, ne, vm, d_list, m->X, m->TM, m->TG, m->n);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(c.stream));
  m->n += add;
  return EXP_OK;
  MLP_CATCH(m)
}

static void grad_batch(exp_mlp* m, const float* X, const float2* TM, const float2* TG, const int* idx, int64_t b0,
                       int64_t nb) {
  const int most = 2 * m->sms, blocks = int(std::min<int64_t>((nb + TS - 1) / TS, most));
  if (m->bf) {
    if (!m->lpart) {
      m->part = (float*)m->al(sizeof(float) * BF_PART * most);
      m->lpart = (double*)m->al(sizeof(double) * (BF_THREADS / 32) * most);
    }
    k_mlp_grad_bf<<<blocks, BF_THREADS, BF_GRAD_SMEM, m->stream>>>(m->P, X, TM, TG, idx, int(b0), int(nb), 1.f / float(nb),
                                                                   m->part, m->lpart);
    CK(cudaGetLastError());
    k_mlp_fold<<<BF_PART / 32 + 1, BF_THREADS, 0, m->stream>>>(m->part, m->lpart, blocks, m->G, m->d_loss);
  } else {
    CK(cudaMemsetAsync(m->G, 0, sizeof(float) * NPARAM, m->stream));
    k_mlp_grad<<<blocks, 256, MLP_SMEM, m->stream>>>(m->P, X, TM, TG, idx, int(b0), int(nb), 1.f / float(nb), m->G,
                                                     m->d_loss);
  }
  CK(cudaGetLastError());
}

extern "C" exp_status exp_mlp_train(exp_mlp* m, int epochs, int batch, double lr, uint64_t seed, double* loss_out) {
  MLP_TRY
  if (!m || epochs < 0 || batch < 1 || !(lr > 0)) throw ExpError{EXP_EINVAL, "bad argument"};
  if (m->n == 0) throw ExpError{EXP_ESTATE, "no training data"};
  std::vector<int> perm(m->n);
  std::mt19937_64 rng(seed);
  for (int ep = 0; ep < epochs; ++ep) {
    std::iota(perm.begin(), perm.end(), 0);
    std::shuffle(perm.begin(), perm.end(), rng);
    CK(cudaMemcpyAsync(m->idx, perm.data(), sizeof(int) * m->n, cudaMemcpyHostToDevice, m->stream));
    CK(cudaMemsetAsync(m->d_loss, 0, sizeof(double), m->stream));
    int nbat = 0;
    for (int64_t b0 = 0; b0 < m->n; b0 += batch) {
      const int64_t nb = std::min<int64_t>(batch, m->n - b0);
      grad_batch(m, m->X, m->TM, m->TG, m->idx, b0, nb);
      ++m->step;
      k_adam<<<(NPARAM + 255) / 256, 256, 0, m->stream>>>(m->P, m->G, m->M1, m->M2, m->step, float(lr));
      CK(cudaGetLastError());
      ++nbat;
    }
    double l = 0.0;
    CK(cudaMemcpyAsync(&l, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    CK(cudaStreamSynchronize(m->stream));  // the permutation buffer is reused next epoch
    if (loss_out) loss_out[ep] = l / nbat;
  }
  return EXP_OK;
  MLP_CATCH(m)
}

extern "C" int64_t exp_mlp_num_samples(const exp_mlp* m) { return m ? m->n : 0; }

extern "C" exp_status exp_mlp_samples(exp_mlp* m, int64_t first, int64_t count, float* x, float* tmp2, float* target) {
  MLP_TRY
  if (!m || first < 0 || count < 0 || first + count > m->n) throw ExpError{EXP_EINVAL, "bad range"};
  if (x) CK(cudaMemcpyAsync(x, m->X + first * NF, sizeof(float) * NF * count, cudaMemcpyDeviceToHost, m->stream));
  if (tmp2) CK(cudaMemcpyAsync(tmp2, m->TM + first, sizeof(float2) * count, cudaMemcpyDeviceToHost, m->stream));
  if (target) CK(cudaMemcpyAsync(target, m->TG + first, sizeof(float2) * count, cudaMemcpyDeviceToHost, m->stream));
  CK(cudaStreamSynchronize(m->stream));
  return EXP_OK;
  MLP_CATCH(m)
}

extern "C" exp_status exp_mlp_eval(exp_mlp* m, double* loss) {
  MLP_TRY
  if (!m || !loss) throw ExpError{EXP_EINVAL, "null argument"};
  if (m->n == 0) throw ExpError{EXP_ESTATE, "no training data"};
  std::vector<int> id(m->n);
  std::iota(id.begin(), id.end(), 0);
  CK(cudaMemcpyAsync(m->idx, id.data(), sizeof(int) * m->n, cudaMemcpyHostToDevice, m->stream));
  CK(cudaMemsetAsync(m->d_loss, 0, sizeof(double), m->stream));
  grad_batch(m, m->X, m->TM, m->TG, m->idx, 0, m->n);
  CK(cudaMemcpyAsync(loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  CK(cudaStreamSynchronize(m->stream));
  return EXP_OK;
  MLP_CATCH(m)
}

extern "C" exp_status exp_mlp_loss_grad(exp_mlp* m, int n, const float* x, const double* tmp2, const double* target,
                                        double* loss, float* grad) {
  MLP_TRY
  if (!m || n < 1 || !x || !tmp2 || !target) throw ExpError{EXP_EINVAL, "bad argument"};
  std::vector<float2> tm(n), tg(n);
  for (int k = 0; k < n; ++k) {
    tm[k] = make_float2(float(tmp2[2 * k]), float(tmp2[2 * k + 1]));
    tg[k] = make_float2(float(target[2 * k]), float(target[2 * k + 1]));
  }
  std::vector<int> id(n);
  std::iota(id.begin(), id.end(), 0);
  float* dX = (float*)m->al(sizeof(float) * NF * n);
  float2* dTM = (float2*)m->al(sizeof(float2) * n);
  float2* dTG = (float2*)m->al(sizeof(float2) * n);
  int* dI = (int*)m->al(sizeof(int) * n);
  CK(cudaMemcpyAsync(dX, x, sizeof(float) * NF * n, cudaMemcpyHostToDevice, m->stream));
  CK(cudaMemcpyAsync(dTM, tm.data(), sizeof(float2) * n, cudaMemcpyHostToDevice, m->stream));
  CK(cudaMemcpyAsync(dTG, tg.data(), sizeof(float2) * n, cudaMemcpyHostToDevice, m->stream));
  CK(cudaMemcpyAsync(dI, id.data(), sizeof(int) * n, cudaMemcpyHostToDevice, m->stream));
  CK(cudaMemsetAsync(m->d_loss, 0, sizeof(double), m->stream));
  grad_batch(m, dX, dTM, dTG, dI, 0, n);
  if (loss) CK(cudaMemcpyAsync(loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  if (grad) CK(cudaMemcpyAsync(grad, m->G, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream));
  CK(cudaStreamSynchronize(m->stream));
  return EXP_OK;
  MLP_CATCH(m)
}

extern "C" exp_status exp_mlp_apply(exp_mlp* m, exp_ctx* x) {
  MLP_TRY
  if (!m || !x) throw ExpError{EXP_EINVAL, "null argument"};
  Ctx& c = x->c;
  if (!c.have_integrals) throw ExpError{EXP_ESTATE, "exp_init_integrals must come first"};
  CK(cudaStreamSynchronize(m->stream));
  float* vm = ctx_vmax(m, c);
  const Tensor* Vd = ccsd_driver_integral(c);
  if (m->bf) {
    // three CTAs an SM are resident; eight waves' worth over all instances, each keeping its
    // parameters for many elements
    const int64_t most = std::max<int64_t>(1, (8 * 3 * m->sms + c.ninst - 1) / c.ninst);
    const int blocks = int(std::max<int64_t>(1, std::min<int64_t>((c.n2 + BF_APPLY - 1) / BF_APPLY, most)));
    k_mlp_apply_bf<<<dim3(blocks, c.ninst), BF_APPLY, BF_APPLY_SMEM, c.stream>>>(m->P, Vd->d, Vd->is, c.d_D, c.d_T, c.namp,
                                                                                 c.n1, c.n2, vm);
  } else {
    const int blocks = int(std::max<int64_t>(1, std::min<int64_t>((c.n2 + TS - 1) / TS, 2 * 304)));
    k_mlp_apply<<<dim3(blocks, c.ninst), 256, MLP_SMEM, c.stream>>>(m->P, Vd->d, Vd->is, c.d_D, c.d_T, c.namp, c.n1, c.n2,
                                                                    vm);
  }
  CK(cudaGetLastError());
  k_zero_t1<<<dim3(std::max<int64_t>(1, std::min<int64_t>((c.n1 + 255) / 256, 64)), c.ninst), 256, 0, c.stream>>>(
      c.d_T, c.namp, c.n1);
  CK(cudaGetLastError());
  ccsd_mark_guessed(c);
  CK(cudaStreamSynchronize(c.stream));
  return EXP_OK;
  MLP_CATCH(m)
}
