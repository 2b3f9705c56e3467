// Plain complex-FP64 grouped GEMM: step 3 of the TTGT list (Sec. II.B), all
// symmetry blocks and instances of one contraction in one launch (the block
// loop of Fig. "mult" flattened into a list of outputs).  Row-major operands,
// C[MxN] = alpha A[MxK] B[KxN] (+ C).  SIMT FP64 FMA: GB300's FP64 rate is the
// roofline for this path.
#include <algorithm>
#include <cmath>

#include "engine.h"
#include "fpbits.h"

constexpr int GEMM_LEAF = 64;  // terms to a leaf of a thread's sum
constexpr int GEMM_PAIRWISE_K = 512;  // longest K, and terms a thread, of pairwise sums
constexpr int GEMM_PAIRWISE_TERMS = 64;

// sum of the next N terms (a power of two), leaves of LEAF terms added pairwise
template <int N, int LEAF>
__device__ __forceinline__ cplx pairwise(const cplx*& a, const cplx*& b, int64_t astep, int64_t bstep) {
  if constexpr (N <= LEAF) {
    double r = 0.0, i = 0.0;
#pragma unroll
    for (int q = 0; q < N; ++q, a += astep, b += bstep) {
      const cplx x = *a, y = *b;
      r = fma(x.x, y.x, r);
      r = fma(-x.y, y.y, r);
      i = fma(x.x, y.y, i);
      i = fma(x.y, y.x, i);
    }
    return make_double2(r, i);
  } else {
    const cplx u = pairwise<N / 2, LEAF>(a, b, astep, bstep), v = pairwise<N / 2, LEAF>(a, b, astep, bstep);
    return make_double2(u.x + v.x, u.y + v.y);
  }
}

// One output element per thread (lanes = 1), or per group of `lanes` threads that
// share its K (lanes a power of two, then a fixed butterfly; above a warp a fixed
// sum over the group's warps in shared memory).
//
// What bounds it: the FP64 pipe, two FMAs per clock per SM -- one warp-wide FMA holds
// its SM partition's pipe for 64 clocks, so the four FMAs of one k take 256 clocks a
// warp while its two 16-byte loads a lane take a few.  Operand reuse is therefore not
// what matters (64 consecutive outputs re-reading B from L2 ask for 8 B a clock of
// the SM); what matters is that every lane holds an output and that the four
// partitions of all SMs get the same share.  So: outputs numbered along the rows of
// all blocks (no padded rows or columns at any shape), CTAs of two warps (the last
// wave is then a small part of the launch), and K shared among lanes only where the
// outputs alone do not fill the chip.
//
// The K terms of a thread are summed in leaves of 64, the leaves in sequence, so that
// the rounding error grows with 64 + K / 64 rather than with K, for two FP64 additions
// in 256 FMAs.  rms error of an output (in 2^-53, normal terms) in one sequence per
// thread -> so: 300 x 300 x 4000 2374 -> 377, 700 x 700 x 8000 4487 -> 563, 109 x 109 x
// 12000 (8 lanes) 2454 -> 595 (in ranges of 256 terms: 605, 1456, 1087); 1024^3 6.91 ->
// 6.98 ms.  Leaves of 32 in branches of 16 have two thirds of that error and take 7.05 ms.
// (Loads of 8 terms ahead serve the few CTAs of 256 threads, 16 x 16 x 500000 1.30 -> 1.01
// ms; where CTAs fill the chip 4 are better, 400 x 400 x 5000 5.74 -> 5.53 ms.)
//
// Measured against 64 x 64 shared-memory tiles (with a warp per output for small
// products), TFLOP/s of complex work, exp_zgemm calls: 1024^3 1.17 -> 1.22, 300^3 0.16 ->
// 0.81, 6000 x 24 x 400 0.27 -> 0.98, 64 x 64 x 5000 0.14 -> 0.70 (the kernel alone: 1.23,
// 1.09, 1.18, 1.10 of the pipe's 1.26); one CCSD iteration at o=10 v=40 8.2 -> 2.2 ms, at
// o=40 v=200 Z8 278 -> 204 ms (1.21 TFLOP/s), (T) at o=24 v=120 Z8 1940 -> 95 ms.
template <int THREADS, int LEAF>
__global__ void __launch_bounds__(THREADS) k_gemm_fp64(const GemmProb* __restrict__ probs, int n_probs,
                                                       const cplx* __restrict__ A, const cplx* __restrict__ B,
                                                       cplx* __restrict__ C, int64_t ais, int64_t bis, int64_t cis,
                                                       cplx alpha, int beta, int64_t n_out, int lanes) {
  const int group = threadIdx.x / lanes, lane = threadIdx.x - group * lanes;
  const int64_t it = int64_t(blockIdx.x) * (THREADS / lanes) + group;
  const bool live = it < n_out;
  int lo = 0, hi = n_probs - 1;
  while (lo < hi) {  // the block that holds output `it`
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].out0 <= it) lo = mid;
    else hi = mid - 1;
  }
  const GemmProb& P = probs[lo];
  const int64_t e = it - P.out0;
  double sr = 0.0, si = 0.0;
  if (live) {
    const int64_t m = e / P.N, n = e - m * P.N;
    const cplx* a = A + blockIdx.y * ais + P.a + m * P.K + lane;
    const cplx* b = B + blockIdx.y * bis + P.b + int64_t(lane) * P.N + n;
    const int64_t bstep = int64_t(lanes) * P.N;
    if constexpr (LEAF > 0) {  // pairwise
      int left = P.K > lane ? (P.K - lane - 1) / lanes + 1 : 0;
      auto add = [&](cplx t) {
        sr += t.x;
        si += t.y;
      };
      for (; left >= 16; left -= 16) add(pairwise<16, LEAF>(a, b, lanes, bstep));
      if (left & 8) add(pairwise<8, LEAF>(a, b, lanes, bstep));
      if (left & 4) add(pairwise<4, LEAF>(a, b, lanes, bstep));
      if (left & 2) add(pairwise<2, LEAF>(a, b, lanes, bstep));
      if (left & 1) add(pairwise<1, LEAF>(a, b, lanes, bstep));
    } else {
      double lr = 0.0, li = 0.0;
      auto term = [&] {
        const cplx x = *a, y = *b;
        lr = fma(x.x, y.x, lr);
        lr = fma(-x.y, y.y, lr);
        li = fma(x.x, y.y, li);
        li = fma(x.y, y.x, li);
        a += lanes;
        b += bstep;
      };
      // (the same number of whole leaves for all lanes: one that has a term more would
      // send the warp through both loops)
      const int full = P.K / (lanes * GEMM_LEAF);
      for (int f = 0; f < full; ++f) {
#pragma unroll(THREADS > 64 ? 8 : 4)
        for (int q = 0; q < GEMM_LEAF; ++q) term();
        sr += lr;
        si += li;
        lr = li = 0.0;
      }
#pragma unroll 4
      for (int k = full * GEMM_LEAF * lanes + lane; k < P.K; k += lanes) term();
      sr += lr;
      si += li;
    }
  }
  for (int o = min(lanes, 32) >> 1; o; o >>= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, o);
    si += __shfl_xor_sync(0xffffffffu, si, o);
  }
  if (THREADS > 64 && lanes > 32) {  // lanes is uniform over the launch
    __shared__ cplx part[THREADS / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_double2(sr, si);
    __syncthreads();
    if (lane == 0)
      for (int w = 1; w < lanes / 32; ++w) {
        const cplx p = part[(threadIdx.x >> 5) + w];
        sr += p.x;
        si += p.y;
      }
  }
  if (live && lane == 0) {
    double vr = alpha.x * sr - alpha.y * si, vi = alpha.x * si + alpha.y * sr;
    cplx* dp = C + blockIdx.y * cis + P.c + e;
    if (beta) { const cplx o = *dp; vr += o.x; vi += o.y; }
    *dp = make_double2(vr, vi);
  }
}

// Threads per output: 1 when the outputs of all instances give every SM partition
// four warps, else the smallest power of two that does, while each lane keeps at
// least four k (a shorter share costs more butterfly additions than it saves: each
// halving of a lane's k adds two additions to four FMAs a k).
//
// Matrix-vector products and small ones (GemmPlan::matvec) keep the accuracy of the
// kernel they ran on before, a warp per output with a term or a few per lane: one
// sequence per thread had up to five times its error.  K above GEMM_PAIRWISE_K is shared
// by a warp at least (a lane's sequence is then as short as there); below, a thread adds
// its terms pairwise, in leaves of two (K < 128, where the pairs decide) or four.  rms
// error of an output in 2^-53 and time, a warp per output / one sequence per thread /
// now: 360 x 360 x 32 9.0, 157 us / 20.3, 32 us / 9.1, 42 us; 100 x 100 x 400 53, 42 us
// / 89, 35 us / 44, 40 us; 100000 x 1 x 5000 549, 3395 us / 3035, 3988 us / 339, 3371
// us.  The lanes also read a row of A side by side: with one thread to a row, the last
// product was slower than a warp per output.
void gemm_lanes(const Ctx& c, GemmPlan& g, int kmax) {
  const int64_t want = int64_t(std::max(c.sm_count, 1)) * 4 * 4 * 32, outputs = g.n_out * c.ninst;
  g.lanes = 1;
  while (g.lanes < GEMM_MAX_LANES && outputs * g.lanes < want && kmax >= 8 * g.lanes) g.lanes *= 2;
  if (!g.matvec) return;
  if (kmax > GEMM_PAIRWISE_K) {
    g.lanes = std::max(g.lanes, 32);
  } else if (g.lanes <= 32) {
    while (kmax > GEMM_PAIRWISE_TERMS * g.lanes) g.lanes *= 2;
    g.leaf = kmax < 128 ? 2 : 4;
  }
}

void launch_gemm_fp64(Ctx& c, const GemmPlan& g, const cplx* A, const cplx* B, cplx* C, int64_t ais,
                      int64_t bis, int64_t cis, cplx alpha, bool beta) {
  if (g.n_out == 0) return;
  const int threads = g.lanes > 32 ? GEMM_MAX_LANES : 64;
  const int64_t per = threads / g.lanes;
  const int64_t blocks = (g.n_out + per - 1) / per;
  if (blocks > INT32_MAX) throw ExpError{EXP_EINVAL, "FP64 product: too many outputs in one launch"};
  const auto kernel = threads > 64 ? k_gemm_fp64<GEMM_MAX_LANES, 0>
                      : g.leaf == 2 ? k_gemm_fp64<64, 2>
                      : g.leaf == 4 ? k_gemm_fp64<64, 4>
                                    : k_gemm_fp64<64, 0>;
  kernel<<<dim3(unsigned(blocks), c.ninst), threads, 0, c.stream>>>(g.d_probs, g.n_probs, A, B, C, ais, bis, cis, alpha,
                                                                    beta, g.n_out, g.lanes);
  KCHECK(c);
}

// ---------------------------------------------------------------------------
// Short contractions (K <= DS_KMAX) under the emulated precision: complex
// products in double-single arithmetic on the FP32 pipe (about 64x GB300's FP64
// rate), every operand split into h + l (48 bits), products and sums carried with
// error-free transformations and the result rounded once to FP64 -- a relative
// error near K 2^-47 of sum |a||b|, below that of the BF16-sliced emulation.  For
// short K that emulation pays for slicing and padding each K half to 16 and for a
// tile pipeline with one k-block per tile; here a product is one pass over A.
// CTA = DS_ROWS rows x DS_NC columns of one problem (the column chunks of a row
// block are adjacent CTAs, so its A block is read from HBM about once): the A
// block (rows contiguous, K each) is read coalesced and split into shared memory,
// the chunk of alpha B staged as double-single pairs; every thread (one row)
// forms its DS_NC outputs.
#define DS_KMAX 16
#define DS_NC 16
#define DS_NG 4  // columns per accumulator group
#define DS_ROWS 128
#define DS_AST (DS_KMAX + 1)  // A row stride in float4: odd, so the row reads of a warp spread over the banks

__global__ void __launch_bounds__(DS_ROWS) k_gemm_ds(const GemmProb* __restrict__ probs, int n_probs,
                                                     const cplx* __restrict__ A, const cplx* __restrict__ B,
                                                     cplx* __restrict__ C, int64_t ais, int64_t bis, int64_t cis,
                                                     cplx alpha, float ascale, int general, int beta) {
  __shared__ float4 As[DS_ROWS * DS_AST];  // (Re h, Re l, Im h, Im l) of A[r0 + r][k]
  __shared__ float4 Bs[DS_KMAX * DS_NC];   // the same for alpha B[k][j0 + jj]
  const int tile = blockIdx.x;
  int pi = 0;
  while (pi + 1 < n_probs && probs[pi + 1].tile0 <= tile) ++pi;
  const GemmProb P = probs[pi];
  const int lt = tile - P.tile0;
  const int rb = lt / P.tiles_n;
  const int r0 = rb * DS_ROWS, j0 = (lt - rb * P.tiles_n) * DS_NC;
  const int nr = min(DS_ROWS, P.M - r0), nc = min(DS_NC, P.N - j0);
  A += blockIdx.y * ais + P.a + int64_t(r0) * P.K;
  B += blockIdx.y * bis + P.b;
  C += blockIdx.y * cis + P.c + int64_t(r0) * P.N;
  for (int e = threadIdx.x; e < nr * P.K; e += blockDim.x) {
    const cplx x = A[e];
    const int r = e / P.K, k = e - r * P.K;
    const float2 xr = ds_split(x.x), xi = ds_split(x.y);
    As[r * DS_AST + k] = make_float4(xr.x, xr.y, xi.x, xi.y);
  }
  const int row = threadIdx.x;
  for (int t = threadIdx.x; t < P.K * DS_NC; t += blockDim.x) {
    const int k = t / DS_NC, jj = t - k * DS_NC;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (jj < nc) {
      cplx b = B[int64_t(k) * P.N + j0 + jj];
      if (general) b = make_double2(alpha.x * b.x - alpha.y * b.y, alpha.x * b.y + alpha.y * b.x);
      const float2 br = ds_split(b.x), bq = ds_split(b.y);
      // ascale = +-2^k (exact in FP32) or 1
      v = make_float4(br.x * ascale, br.y * ascale, bq.x * ascale, bq.y * ascale);
    }
    Bs[t] = v;
  }
  __syncthreads();
  if (row >= nr) return;
  // columns in groups of DS_NG (accumulators of a group in registers; a small loop
  // body, 2 DS_NG independent accumulation chains)
  cplx* crow = C + int64_t(row) * P.N + j0;
  for (int g0 = 0; g0 < nc; g0 += DS_NG) {
    float sr[DS_NG], cr[DS_NG], si[DS_NG], ci[DS_NG];
#pragma unroll
    for (int u = 0; u < DS_NG; ++u) sr[u] = cr[u] = si[u] = ci[u] = 0.f;
    for (int k = 0; k < P.K; ++k) {
      const float4 a = As[row * DS_AST + k];
#pragma unroll
      for (int u = 0; u < DS_NG; ++u) {
        const float4 b = Bs[k * DS_NC + g0 + u];  // zero past nc
        ds_mac(sr[u], cr[u], a.x, a.y, b.x, b.y);    // Re += Re a Re b
        ds_mac(sr[u], cr[u], -a.z, -a.w, b.z, b.w);  //     - Im a Im b
        ds_mac(si[u], ci[u], a.x, a.y, b.z, b.w);    // Im += Re a Im b
        ds_mac(si[u], ci[u], a.z, a.w, b.x, b.y);    //     + Im a Re b
      }
    }
#pragma unroll
    for (int u = 0; u < DS_NG; ++u) {
      if (g0 + u < nc) {
        double vr = ds_to_double(sr[u], cr[u]), vi = ds_to_double(si[u], ci[u]);
        if (beta) {
          const cplx o = crow[g0 + u];
          vr += o.x;
          vi += o.y;
        }
        crow[g0 + u] = make_double2(vr, vi);
      }
    }
  }
}

bool ds_wanted(Ctx& c, const GemmPlan& g) {
  if (c.cfg.precision != EXP_EMU_BF16 || g.matvec || g.h_probs.empty()) return false;
  int kmax = 0;
  for (const GemmProb& p : g.h_probs) kmax = std::max(kmax, p.K);
  return kmax >= 1 && kmax <= DS_KMAX;
}

void ds_prepare(Ctx& c, GemmPlan& g) {
  if (g.d_ds) return;
  for (const GemmProb& p : g.h_probs)
    if (p.K > DS_KMAX) throw ExpError{EXP_EINVAL, "double-single GEMM: K above 16"};
  std::vector<GemmProb> v = g.h_probs;
  int tiles = 0;
  for (GemmProb& p : v) {  // CTAs: DS_ROWS rows x DS_NC columns, column chunks adjacent
    p.tiles_m = (p.M + DS_ROWS - 1) / DS_ROWS;
    p.tiles_n = (p.N + DS_NC - 1) / DS_NC;
    p.tile0 = tiles;
    tiles += p.tiles_m * p.tiles_n;
  }
  g.ds_tiles = tiles;
  g.d_ds = (GemmProb*)c.dalloc(sizeof(GemmProb) * std::max<size_t>(v.size(), 1));
  upload(c, g.d_ds, v.data(), sizeof(GemmProb) * v.size());
}

void launch_gemm_ds(Ctx& c, const GemmPlan& g, const cplx* A, const cplx* B, cplx* C, int64_t ais, int64_t bis,
                    int64_t cis, cplx alpha, bool beta) {
  if (!g.d_ds) throw ExpError{EXP_ESTATE, "double-single GEMM not prepared"};
  if (g.ds_tiles == 0) return;
  // alpha = +-2^k folds into the FP32 parts exactly; any other alpha multiplies B in FP64
  int ex = 0;
  const double fr = std::frexp(std::fabs(alpha.x), &ex);
  const bool pow2 = alpha.y == 0.0 && fr == 0.5 && ex > -100 && ex < 100;
  k_gemm_ds<<<dim3(g.ds_tiles, c.ninst), DS_ROWS, 0, c.stream>>>(g.d_ds, g.n_probs, A, B, C, ais, bis, cis, alpha,
                                                                 pow2 ? float(alpha.x) : 1.0f, pow2 ? 0 : 1,
                                                                 beta ? 1 : 0);
  KCHECK(c);
}
