// One training step of the CROM manifold (paper §3, Eq. loss; App. D): strided
// 1D-convolution encoder + MLP decoder, MSE over sampled points, hand-written
// reverse pass and Adam with FP32 master weights.
//
// Encoder (App. D): convolutions of kernel 6, stride 4, one channel, no padding,
// ELU after each, repeated while the output length stays >= 32; then a dense
// layer to 32 (ELU) and a linear layer to r.  Decoder: g(x, q) with the layer
// sizes of the crom_decoder_desc.  Loss: mean over the B x S sampled points of
// (g(x_j, e(f_b)) - f_b(x_j))^2.  Adam with beta1 = 0.9, beta2 = 0.999, eps = 1e-8.
//
// Parameter vector (FP32, also the layout of crom_trainer_get/set_params):
// decoder layers as in crom_set_weights (W row-major, then b), then for each
// convolution w[6], b, then the dense layers (W [32][L_last], b[32]),
// (W [r][32], b[r]).
//
// The decoder pass runs either here in FP32 (one tiled FP32 GEMM with strided
// operands and fused epilogues, bias + ELU and multiply by s'(z); weight gradients
// reduce over the B*S points with a fixed split along K and a second pass that adds
// the splits in order, so a step is deterministic) or, with CROM_PREC_BF16_MIXED, on
// the tensor cores (train_tc.cu).  The encoder, the latent gradient and Adam are
// shared.
#include <math.h>

#include <algorithm>
#include <vector>

#include "crom_internal.h"
#include "tc_common.cuh"

namespace crom {
namespace {

constexpr int kSplitK = 32;       // K ranges of the weight gradients

// Both without a divergent branch (a NaN stays a NaN).
__device__ __forceinline__ float elu_f(float z) {
  const float e = expm1f(z > 0.f ? 0.f : z);
  return z > 0.f ? z : e;
}
__device__ __forceinline__ float elu_d(float z) {
  const float e = expf(z > 0.f ? 0.f : z);
  return z > 0.f ? 1.f : e;
}

// Compensated (Kahan) FP32 accumulation: the running sum s - c stays within a few
// ulps of the exact sum whatever the number of terms, in FP32 instructions (FP64 is
// a slow pipe on this GPU: per-element FP64 adds made these reductions FP64-bound).
struct CompSum {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float y = __fsub_rn(v, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

enum Epi { kEpiStore = 0, kEpiBiasElu = 1, kEpiTimesEluD = 2 };

// C[i][j] = sum_k A(i, k) B(k, j): A(i, k) = A[i * lda + k] (kAK) or A[k * lda + i],
// B(k, j) = B[j * ldb + k] (kBK) or B[k * ldb + j].  Every output is one FMA chain in
// ascending k.  Epilogues: kEpiStore (C row-major, ldc); kEpiBiasElu (Z = C + bias[j]
// stored in C, ELU(Z) stored in H); kEpiTimesEluD (C *= s'(Zp[i][j])).  blockIdx.z splits
// K into gridDim.z contiguous ranges writing to C + z * split_stride (kEpiStore only).
//
// BM x BN outputs per CTA, 8 x CN per thread (two quads of rows by one or two of columns):
// with CN = 8 shared memory delivers operands as fast as the FP32 pipe takes them (a 4 x 4
// tile needs twice the loads).  The next 16 values of K (32 with four columns) are on their
// way in registers while the current ones are multiplied; the row pairs feed the packed FMA.  The former 64 x 64 x 16
// tiles of 4 x 4 took 81 us for 32768 x 128 x 128 (13 TFLOP/s), these 33 us (the 152 SMs
// hold 256 tiles two to an SM, unevenly: 17 us of FMAs, then the ELU).  Weight gradients of 128
// x 128 over 32768 rows: 196 us before, 35 us (50 with 16 values on their way); their K ranges are fixed (the sums' order is
// part of the result), which leaves four warps per SM.
struct GemmArgs {
  int M, N, K;
  const float *A, *B;
  long lda, ldb;
  float* C;
  long ldc, split_stride;
  int epi;
  const float* bias;
  float* H;
  const float* Zp;
  bool va, vb, vc;  // 16-byte accesses to A, B and the outputs
};
constexpr int kTK = 16;

template <int BM, int BN, int CN, bool kAK, bool kBK>
__global__ void __launch_bounds__(BM * BN / 8 / CN, CN == 8 ? 512 / (BM * BN / 8 / CN) : 2) gemm_kernel(GemmArgs g) {
  constexpr int TK = CN == 8 ? kTK : 2 * kTK, NT = BM * BN / 8 / CN, TX = BN / CN, LA = BM + 4, LB = BN + 4;
  __shared__ __align__(16) float As[2][TK][LA];
  __shared__ __align__(16) float Bs[2][TK][LB];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
  const int splits = gridDim.z;
  const int kchunk = ((g.K + splits - 1) / splits + kTK - 1) / kTK * kTK;
  const int kbeg = blockIdx.z * kchunk, kend = min(g.K, kbeg + kchunk);
  // operand X (rows r < R of the tile at row0 of `rows`): float4 e of the 16 x BX tile
  constexpr int QA = BM * TK / 4 / NT, QB = BN * TK / 4 / NT;
  float4 ra[QA], rb[QB];
  auto fetch = [&](const float* X, long ld, int row0, int rows, int k0, int e, bool kmajor, int BX, bool wide) -> float4 {
    float v[4];
    if (kmajor) {  // four values of k of one row
      const int r = e / (TK / 4), k = k0 + 4 * (e % (TK / 4));
      const float* x = X + (long)(row0 + r) * ld + k;
      const bool in = row0 + r < rows;
      if (wide && in && k + 4 <= kend) return *reinterpret_cast<const float4*>(x);
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = in && k + q < kend ? x[q] : 0.f;
    } else {  // four rows at one k
      const int k = k0 + e / (BX / 4), r = 4 * (e % (BX / 4));
      const float* x = X + (long)k * ld + row0 + r;
      const bool in = k < kend;
      if (wide && in && row0 + r + 4 <= rows) return *reinterpret_cast<const float4*>(x);
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = in && row0 + r + q < rows ? x[q] : 0.f;
    }
    return make_float4(v[0], v[1], v[2], v[3]);
  };
  auto place = [&](float* S, int LD, int e, float4 v, bool kmajor, int BX) {
    if (kmajor) {
      const int r = e / (TK / 4), k = 4 * (e % (TK / 4));
      S[k * LD + r] = v.x;
      S[(k + 1) * LD + r] = v.y;
      S[(k + 2) * LD + r] = v.z;
      S[(k + 3) * LD + r] = v.w;
    } else {
      *reinterpret_cast<float4*>(S + e / (BX / 4) * LD + 4 * (e % (BX / 4))) = v;
    }
  };
  auto fetch_all = [&](int k0) {
#pragma unroll
    for (int q = 0; q < QA; ++q) ra[q] = fetch(g.A, g.lda, i0, g.M, k0, tid + q * NT, kAK, BM, g.va);
#pragma unroll
    for (int q = 0; q < QB; ++q) rb[q] = fetch(g.B, g.ldb, j0, g.N, k0, tid + q * NT, kBK, BN, g.vb);
  };
  auto place_all = [&](int buf) {
#pragma unroll
    for (int q = 0; q < QA; ++q) place(&As[buf][0][0], LA, tid + q * NT, ra[q], kAK, BM);
#pragma unroll
    for (int q = 0; q < QB; ++q) place(&Bs[buf][0][0], LB, tid + q * NT, rb[q], kBK, BN);
  };
  // row pairs 4 ty + {0, 1}, {2, 3}, BM / 2 + .. by columns 4 tx + 0..3, BN / 2 + ..
  tc::f32x2 acc[4][CN];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < CN; ++q) acc[p][q] = 0ull;
  if (kbeg < kend) {
    fetch_all(kbeg);
    place_all(0);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += TK) {
    const bool more = k0 + TK < kend;
    if (more) fetch_all(k0 + TK);
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(&As[buf][kk][4 * ty]);
      const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(&As[buf][kk][BM / 2 + 4 * ty]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][4 * tx]);
      const float4 b1 = CN == 8 ? *reinterpret_cast<const float4*>(&Bs[buf][kk][BN / 2 + 4 * tx]) : b0;
      const tc::f32x2 a[4] = {a0.x, a0.y, a1.x, a1.y};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int q = 0; q < CN; ++q) {
        const tc::f32x2 bb = tc::pk2(b[q], b[q]);
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p][q] = tc::fma2(a[p], bb, acc[p][q]);
      }
    }
    if (more) place_all(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  float* Cz = g.C + (long)blockIdx.z * g.split_stride;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int i = i0 + (p < 4 ? 0 : BM / 2) + 4 * ty + (p & 3);
    if (i >= g.M) continue;
#pragma unroll
    for (int h = 0; h < CN / 4; ++h) {
      const int j = j0 + h * (BN / 2) + 4 * tx;
      float v[4], z[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float lo, hi;
        tc::unpk2(acc[p >> 1][4 * h + q], lo, hi);
        v[q] = (p & 1) ? hi : lo;
      }
      const long o = (long)i * g.ldc + j;
      const bool whole = g.vc && j + 4 <= g.N;
      if (g.epi == kEpiBiasElu) {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] += j + q < g.N ? g.bias[j + q] : 0.f;
      } else if (g.epi == kEpiTimesEluD) {
        if (whole) {
          const float4 x = *reinterpret_cast<const float4*>(g.Zp + o);
          z[0] = x.x; z[1] = x.y; z[2] = x.z; z[3] = x.w;
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) z[q] = j + q < g.N ? g.Zp[o + q] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] *= elu_d(z[q]);
      }
      if (whole) *reinterpret_cast<float4*>(Cz + o) = make_float4(v[0], v[1], v[2], v[3]);
      else
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j + q < g.N) Cz[o + q] = v[q];
      if (g.epi == kEpiBiasElu) {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = elu_f(v[q]);
        if (whole) *reinterpret_cast<float4*>(g.H + o) = make_float4(v[0], v[1], v[2], v[3]);
        else
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (j + q < g.N) g.H[o + q] = v[q];
      }
    }
  }
}

// part[c][u] = sum over row range c of dg[n] H[n][u] (the output layer's weight gradient,
// the K ranges and chains of the GEMM form): 32 columns per CTA, one warp holds the chains
// and eight bring the next kWoutRows rows in meanwhile: 12 us for 32768 rows of 128.
constexpr int kWoutRows = 128;
__global__ void __launch_bounds__(256) wout_part_kernel(const float* __restrict__ dg, const float* __restrict__ H, int rows,
                                                        int w, int per, float* part) {
  __shared__ float hs[2][kWoutRows][32], ds[2][kWoutRows];
  constexpr int kQ = kWoutRows / 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, u = blockIdx.x * 32 + lane;
  const int r0 = min(rows, (int)blockIdx.y * per), r1 = min(rows, r0 + per);
  float v[kQ], d = 0.f;
  auto fetch = [&](int n0) {
#pragma unroll
    for (int k = 0; k < kQ; ++k) {
      const int n = n0 + warp + 8 * k;
      v[k] = n < r1 && u < w ? __ldg(H + (long)n * w + u) : 0.f;
    }
    d = threadIdx.x < kWoutRows && n0 + (int)threadIdx.x < r1 ? __ldg(dg + n0 + threadIdx.x) : 0.f;
  };
  float s = 0.f;
  int buf = 0;
  if (r0 < r1) fetch(r0);
  for (int n0 = r0; n0 < r1; n0 += kWoutRows, buf ^= 1) {
#pragma unroll
    for (int k = 0; k < kQ; ++k) hs[buf][warp + 8 * k][lane] = v[k];
    if (threadIdx.x < kWoutRows) ds[buf][threadIdx.x] = d;
    __syncthreads();
    if (n0 + kWoutRows < r1) fetch(n0 + kWoutRows);
    if (warp == 0) {
      const int nr = min(kWoutRows, r1 - n0);
      if (nr == kWoutRows) {
#pragma unroll 16
        for (int k = 0; k < kWoutRows; ++k) s = fmaf(ds[buf][k], hs[buf][k][lane], s);
      } else {
        for (int k = 0; k < nr; ++k) s = fmaf(ds[buf][k], hs[buf][k][lane], s);
      }
    }
  }
  if (warp == 0 && u < w) part[(long)blockIdx.y * w + u] = s;
}

// out[e] = sum_s parts[s * n + e], in order of s, the loads ahead of the additions.
__global__ void __launch_bounds__(128) sum_splits_kernel(const float* __restrict__ parts, long n, float* out) {
  const long e = blockIdx.x * 128L + threadIdx.x;
  if (e >= n) return;
  float v[kSplitK], s = 0.f;
#pragma unroll
  for (int k = 0; k < kSplitK; ++k) v[k] = __ldg(parts + k * n + e);
#pragma unroll
  for (int k = 0; k < kSplitK; ++k) s += v[k];
  out[e] = s;
}

// Column sums of X [rows][cols] in fixed order: out[c] = sum_r X[r][c] (one block per column).
// Column sums of X [rows][cols] in two fixed-order passes (deterministic):

// colsum_part_kernel: block (32 columns x 8 row lanes) per (column group, row chunk),
// coalesced across columns; colsum_final_kernel adds the chunk partials in order.
constexpr int kColChunks = 128;
__global__ void colsum_part_kernel(const float* X, long rows, int cols, double* part) {
  const int c = blockIdx.x * 32 + threadIdx.x;
  const long per = (rows + gridDim.y - 1) / gridDim.y;
  const long r0 = (long)blockIdx.y * per, r1 = min(rows, r0 + per);
  CompSum s;
  if (c < cols)
    for (long r = r0 + threadIdx.y; r < r1; r += 8) s.add(X[r * cols + c]);
  __shared__ double red[8][33];
  red[threadIdx.y][threadIdx.x] = s.value();
  __syncthreads();
  if (threadIdx.y == 0 && c < cols) {
    double t = 0.0;
    for (int y = 0; y < 8; ++y) t += red[y][threadIdx.x];
    part[(long)blockIdx.y * cols + c] = t;
  }
}
// Column sums four columns at a time (cols % 4 == 0): block (kColQuads column quads x 4
// row lanes) per (column-quad group, row chunk).
constexpr int kColQuads = 16;
__global__ void colsum_part4_kernel(const float* X, long rows, int cols, double* part) {
  const int q = blockIdx.x * kColQuads + threadIdx.x, cols4 = cols / 4;
  const long per = (rows + gridDim.y - 1) / gridDim.y;
  const long r0 = (long)blockIdx.y * per, r1 = min(rows, r0 + per);
  CompSum s0, s1, s2, s3;
  if (q < cols4) {
    long r = r0 + threadIdx.y;
    for (; r + 60 < r1; r += 64) {  // sixteen rows' loads ahead of the additions
      float4 v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __ldg(reinterpret_cast<const float4*>(X + (r + 4 * k) * cols) + q);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        s0.add(v[k].x);
        s1.add(v[k].y);
        s2.add(v[k].z);
        s3.add(v[k].w);
      }
    }
    for (; r < r1; r += 4) {
      const float4 v = reinterpret_cast<const float4*>(X + r * cols)[q];
      s0.add(v.x);
      s1.add(v.y);
      s2.add(v.z);
      s3.add(v.w);
    }
  }
  __shared__ double red[4][kColQuads][4];
  red[threadIdx.y][threadIdx.x][0] = s0.value();
  red[threadIdx.y][threadIdx.x][1] = s1.value();
  red[threadIdx.y][threadIdx.x][2] = s2.value();
  red[threadIdx.y][threadIdx.x][3] = s3.value();
  __syncthreads();
  if (threadIdx.y == 0 && q < cols4)
    for (int e = 0; e < 4; ++e)
      part[(long)blockIdx.y * cols + 4 * q + e] =
          (red[0][threadIdx.x][e] + red[1][threadIdx.x][e]) + (red[2][threadIdx.x][e] + red[3][threadIdx.x][e]);
}
// Sum over the 32 lanes by a fixed butterfly (every lane ends with the same value).
__device__ __forceinline__ double warp_sum_fixed(double t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double u = __shfl_xor_sync(0xffffffffu, t, o);
    t = (threadIdx.x & o) ? u + t : t + u;  // the lower lane's value first on both lanes
  }
  return t;
}
// out[c] = sum of the chunks' partials of column c: one warp per column, lanes take
// every 32nd chunk, then a fixed butterfly.
__global__ void colsum_final_kernel(const double* part, int chunks, int cols, float* out) {
  const int c = (int)((blockIdx.x * (long)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= cols) return;  // whole warps leave together
  double t = 0.0;
  for (int k = lane; k < chunks; k += 32) t += part[(long)k * cols + c];
  t = warp_sum_fixed(t);
  if (lane == 0) out[c] = (float)t;
}

__global__ void conv_fwd_kernel(const float* x, int Lin, int Lout, int B, const float* w, float* z, float* h) {
  const long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (e >= (long)B * Lout) return;
  const int b = (int)(e / Lout), i = (int)(e % Lout);
  const float* xb = x + (long)b * Lin + 4 * i;
  float s = w[6];
  for (int k = 0; k < 6; ++k) s = fmaf(w[k], xb[k], s);
  z[e] = s;
  h[e] = elu_f(s);
}

// Input gradient of one convolution, dx[b][j] = sum over i with 0 <= j - 4i < 6 of
// w[j - 4i] dz[b][i].
__device__ __forceinline__ float conv_dx(const float* w, const float* dz, int Lout, int j) {
  float s = 0.f;
  for (int i = min(j / 4, Lout - 1); i >= 0 && j - 4 * i < 6; --i) s = fmaf(w[j - 4 * i], dz[i], s);
  return s;
}
// z of the previous convolution becomes its dz = dx s'(z).
__global__ void conv_dz_kernel(const float* dz, int Lin, int Lout, int B, const float* w, float* z) {
  const long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (e >= (long)B * Lin) return;
  z[e] = conv_dx(w, dz + e / Lin * Lout, Lout, (int)(e % Lin)) * elu_d(z[e]);
}

// Parameter gradients of every convolution, gw[k] = sum_{b,i} dz[b][i] x[b][4i+k] and gb =
// sum dz: a block per chunk of a convolution's B * Lout terms, 256 lanes through them (every
// 256th) by four groups with two of the seven sums each.  Products are split exactly into
// p + err (one FMA), the p summed with compensation.  The lanes' sums are added as
// unevaluated triples (two-sum): as close as FP64, which is a slow pipe here (a block
// per sum, with an FP64 tree, took 31 us for the 2^20 terms of the longest one alone).
struct ConvGrads {
  int n, B;
  int lin[16], lout[16], chunks[16];
  const float *dz[16], *x[16];
  double* part[16];  // [chunk][7]
};
struct Triple {
  float a, b, c;
};
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
__device__ __forceinline__ Triple add3(Triple x, Triple y) {
  const float2 s = two_sum(x.a, y.a), t = two_sum(x.b, y.b), u = two_sum(t.x, s.y);
  return {s.x, u.x, __fadd_rn(__fadd_rn(x.c, y.c), __fadd_rn(t.y, u.y))};
}
__global__ void __launch_bounds__(1024) conv_grads_kernel(const __grid_constant__ ConvGrads g) {
  int l = 0, chunk = blockIdx.x;
  while (chunk >= g.chunks[l]) chunk -= g.chunks[l++];
  const int Lin = g.lin[l], Lout = g.lout[l], k0 = (threadIdx.x >> 8) * 2, lane = threadIdx.x & 255;
  const long n = (long)g.B * Lout, per = (n + g.chunks[l] - 1) / g.chunks[l];
  const long e0 = chunk * per, e1 = min(n, e0 + per);
  const float* dz = g.dz[l];
  CompSum s[2];
  float err[2] = {0.f, 0.f};
  long e = e0 + lane;
  const float* xb = g.x[l] + e / Lout * Lin;  // the term's snapshot and place in it
  int i = (int)(e % Lout);
  constexpr int kAhead = 8;
  while (e < e1) {
    float a[kAhead], x[kAhead][2];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      const bool in = e + 256L * q < e1;
      a[q] = in ? __ldg(dz + e + 256L * q) : 0.f;
#pragma unroll
      for (int k = 0; k < 2; ++k) x[q][k] = in && k0 + k < 6 ? __ldg(xb + 4 * i + k0 + k) : 1.f;
      for (i += 256; i >= Lout; i -= Lout) xb += Lin;
    }
#pragma unroll
    for (int q = 0; q < kAhead; ++q)
      if (e + 256L * q < e1) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float p = __fmul_rn(a[q], x[q][k]);
          err[k] += fmaf(a[q], x[q][k], -p);
          s[k].add(p);
        }
      }
    e += 256L * kAhead;
  }
  __shared__ Triple red[8][8];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    Triple v = {s[k].s, -s[k].c, err[k]};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      v = add3(v, Triple{__shfl_xor_sync(0xffffffffu, v.a, o), __shfl_xor_sync(0xffffffffu, v.b, o),
                         __shfl_xor_sync(0xffffffffu, v.c, o)});
    if ((lane & 31) == 0) red[k0 + k][lane >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 7) {
    Triple v = red[threadIdx.x][0];
#pragma unroll
    for (int q = 1; q < 8; ++q) v = add3(v, red[threadIdx.x][q]);
    g.part[l][7L * chunk + threadIdx.x] = (double)v.a + ((double)v.b + (double)v.c);
  }
}

// The encoder below its long convolutions: a CTA per snapshot takes the convolutions of at
// most kEncLin inputs and both dense layers, layer by layer through shared memory.  A
// launch per layer and direction spent 3 to 8 us on each of them for well under a
// microsecond of work: with the reverse pass's products and sums 235 us of the step at 64
// snapshots of 65536 points, now 67 us.  Longer convolutions (one snapshot's no longer a
// CTA's few passes) keep launches over all snapshots.  Every output is the same FMA chain
// as in the layer-wise form.
// (kEncLout: the outputs of kEncLin inputs; kEncDense: the longest row not convolved again.)
constexpr int kEncLin = 16384, kEncLout = 4096, kEncDense = 129, kEncConvs = 4, kEncThreads = 1024;
struct EncConv {
  int lin, lout;
  const float *w, *x;  // x [b][lin]: the layer's input
  float *z, *h;        // the reverse pass leaves dz in z
};
struct EncArgs {
  int n;               // convolutions
  EncConv conv[kEncConvs];
  int Ll, r;
  const float* hl;     // [b][Ll]: the dense part's input
  const float *w1, *b1, *w2, *b2;
  float *d1z, *d1h, *q;
  // reverse pass
  const float* dq;
  float* ed1;
  float* zx;           // z of the convolution before conv[0], or null
};

__global__ void __launch_bounds__(kEncThreads) enc_fwd_kernel(EncArgs a) {
  __shared__ float buf0[kEncLout], buf1[kEncLout / 4], w1s[32 * (kEncDense | 1)], hid[32];
  const int b = blockIdx.x, tid = threadIdx.x, ldw = a.Ll | 1;
  for (int e = tid; e < 32 * a.Ll; e += kEncThreads) w1s[e / a.Ll * ldw + e % a.Ll] = a.w1[e];
  const float* x = nullptr;
  for (int c = 0; c < a.n; ++c) {
    const EncConv& v = a.conv[c];
    if (c == 0) x = v.x + (long)b * v.lin;
    float* y = (c & 1) ? buf1 : buf0;
    for (int i = tid; i < v.lout; i += kEncThreads) {
      float s = v.w[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) s = fmaf(v.w[k], x[4 * i + k], s);
      const float h = elu_f(s);
      v.z[(long)b * v.lout + i] = s;
      v.h[(long)b * v.lout + i] = h;
      y[i] = h;
    }
    __syncthreads();
    x = y;
  }
  if (a.n == 0) {
    for (int i = tid; i < a.Ll; i += kEncThreads) buf0[i] = a.hl[(long)b * a.Ll + i];
    __syncthreads();
    x = buf0;
  }
  if (tid < 32) {
    float s = 0.f;
#pragma unroll 8
    for (int k = 0; k < a.Ll; ++k) s = fmaf(x[k], w1s[tid * ldw + k], s);
    s += a.b1[tid];
    const float h = elu_f(s);
    a.d1z[b * 32L + tid] = s;
    a.d1h[b * 32L + tid] = h;
    hid[tid] = h;
    __syncwarp();
    if (tid < a.r) {
      float q = 0.f;
#pragma unroll
      for (int k = 0; k < 32; ++k) q = fmaf(hid[k], a.w2[tid * 32 + k], q);
      a.q[(long)b * a.r + tid] = q + a.b2[tid];
    }
  }
}

// dz1 = (dq W2) s'(z1), dh = dz1 W1, then the convolutions last to first: dz = dh s'(z)
// and the input gradient for the one before.
__global__ void __launch_bounds__(kEncThreads) enc_bwd_kernel(EncArgs a) {
  __shared__ float buf[2][kEncLout], dz1[32];
  const int b = blockIdx.x, tid = threadIdx.x;
  if (tid < 32) {
    float s = 0.f;
    for (int k = 0; k < a.r; ++k) s = fmaf(a.dq[(long)b * a.r + k], a.w2[k * 32 + tid], s);
    s *= elu_d(a.d1z[b * 32L + tid]);
    a.ed1[b * 32L + tid] = s;
    dz1[tid] = s;
  }
  if (a.n == 0) return;
  __syncthreads();
  for (int l = tid; l < a.Ll; l += kEncThreads) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 32; ++k) s = fmaf(dz1[k], a.w1[k * a.Ll + l], s);
    float* z = a.conv[a.n - 1].z + (long)b * a.Ll + l;
    *z = buf[0][l] = s * elu_d(*z);
  }
  for (int c = a.n - 1; c >= 0; --c) {
    const float* d = buf[(a.n - 1 - c) & 1];
    float* dn = buf[(a.n - c) & 1];
    float* z = c > 0 ? a.conv[c - 1].z : a.zx;
    if (!z) return;
    const int lin = a.conv[c].lin, lout = a.conv[c].lout;
    const float* w = a.conv[c].w;
    z += (long)b * lin;
    __syncthreads();
#pragma unroll 4
    for (int j = tid; j < lin; j += kEncThreads) {
      const float s = conv_dx(w, d, lout, j) * elu_d(z[j]);
      z[j] = s;
      if (c > 0) dn[j] = s;
    }
  }
}

// The encoder's parameter gradients, sums over the snapshots.  A thread forms one weight
// of the dense layers, an FMA chain in snapshot order with the loads ahead of it; the next
// blocks one bias each per warp (up to kColChunks snapshots; n_bias = 0 leaves them to
// the column sums), the last n_conv blocks a convolution's seven: lanes every 32nd term in
// FP64, then a fixed butterfly.
struct EncGrads {
  int B, Ll, r, n_conv, n_bias;
  const float *ed1, *hl, *dq, *d1h;
  float *gw1, *gb1, *gw2, *gb2;
  const double* part[16];
  int chunks[16];
  float* gconv[16];
};
constexpr int kGradThreads = 224;  // seven warps
__host__ __device__ inline int enc_weight_blocks(int Ll, int r) { return (32 * (Ll + r) + kGradThreads - 1) / kGradThreads; }
__global__ void __launch_bounds__(kGradThreads) enc_grads_kernel(EncGrads g) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = enc_weight_blocks(g.Ll, g.r), nb = (g.n_bias + 6) / 7;
  if ((int)blockIdx.x < nw) {
    const int o = blockIdx.x * kGradThreads + threadIdx.x, n1 = 32 * g.Ll;
    if (o >= n1 + 32 * g.r) return;
    const bool w1 = o < n1;
    const int i = w1 ? o / g.Ll : (o - n1) / 32, j = w1 ? o % g.Ll : (o - n1) % 32;
    const float* p = w1 ? g.ed1 + i : g.dq + i;
    const float* q = w1 ? g.hl + j : g.d1h + j;
    const int sp = w1 ? 32 : g.r, sq = w1 ? g.Ll : 32;
    float s = 0.f;
    int b = 0;
    for (; b + 16 <= g.B; b += 16) {
      float x[16], y[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        x[k] = __ldg(p + (long)(b + k) * sp);
        y[k] = __ldg(q + (long)(b + k) * sq);
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) s = fmaf(x[k], y[k], s);
    }
    for (; b < g.B; ++b) s = fmaf(p[(long)b * sp], q[(long)b * sq], s);
    (w1 ? g.gw1 : g.gw2 - n1)[o] = s;
    return;
  }
  double t = 0.0;
  float* out;
  if ((int)blockIdx.x < nw + nb) {
    const int o = ((int)blockIdx.x - nw) * 7 + warp;
    if (o >= g.n_bias) return;
    const float* p = o < 32 ? g.ed1 + o : g.dq + (o - 32);
    const int sp = o < 32 ? 32 : g.r;
    for (int b = lane; b < g.B; b += 32) t += (double)p[(long)b * sp];
    out = o < 32 ? g.gb1 + o : g.gb2 + (o - 32);
  } else {
    const int c = (int)blockIdx.x - nw - nb;
    for (int k = lane; k < g.chunks[c]; k += 32) t += g.part[c][7L * k + warp];
    out = g.gconv[c] + warp;
  }
  t = warp_sum_fixed(t);
  if (lane == 0) *out = (float)t;
}

__global__ void gather_kernel(const float* snaps, const int* pt_idx, const float* coords, const float* q, int B,
                              int S, int P, int m, int r, float* in, float* target) {
  const long n = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (n >= (long)B * S) return;
  const int b = (int)(n / S);
  const int node = pt_idx[n];
  const int ld = m + r;
  for (int k = 0; k < m; ++k) in[n * ld + k] = coords[(long)node * m + k];
  for (int j = 0; j < r; ++j) in[n * ld + m + j] = q[(long)b * r + j];
  target[n] = snaps[(long)b * P + node];
}
// The tensor-core pass's inputs: the points' coordinates x [B*S][m] (the latent part
// of the input layer is formed per snapshot) and the targets.
__global__ void gather_x_kernel(const float* snaps, const int* pt_idx, const float* coords, int B, int S, int P,
                                int m, float* x, float* target) {
  const long n = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (n >= (long)B * S) return;
  const int b = (int)(n / S);
  const int node = pt_idx[n];
  for (int k = 0; k < m; ++k) x[n * m + k] = coords[(long)node * m + k];
  target[n] = snaps[(long)b * P + node];
}

// Output layer g = w_out . h + b_out, residual and dL/dg = 2 (g - t) / N; per-block
// partial sums of the squared residual (FP64).
__global__ void output_loss_kernel(const float* H, int w, long N, const float* wout, const float* bout,
                                   const float* target, float* dg, double* partial) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const long n = blockIdx.x * 8L + warp;
  double sq = 0.0;
  if (n < N) {
    float s = 0.f;
    for (int u = lane; u < w; u += 32) s = fmaf(wout[u], H[n * w + u], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float res = s + bout[0] - target[n];
    if (lane == 0) {
      dg[n] = 2.f * res / (float)N;
      sq = (double)res * (double)res;
    }
  }
  __shared__ double red[8];
  if (lane == 0) red[warp] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < 8; ++i) s += red[i];
    partial[blockIdx.x] = s;
  }
}
// loss = sum(partial) / N: 1024 threads, strided partial sums, fixed tree.
__global__ void loss_final_kernel(const double* partial, int n, long N, double* loss) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += partial[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = red[0] / (double)N;
}
// delta_L[n][u] = dL/dg_n w_out[u] s'(z_L[n][u]).
__global__ void out_delta_kernel(const float* dg, const float* wout, const float* Z, int w, long N, float* delta) {
  const long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (e >= N * w) return;
  const long n = e / w;
  const int u = (int)(e % w);
  delta[e] = dg[n] * wout[u] * elu_d(Z[e]);
}
// The same, four units per thread (w % 4 == 0, N * w / 4 < 2^31, 16-byte aligned):
// quad e covers row e / (w / 4), units 4 (e % (w / 4)) ..
__global__ void out_delta4_kernel(const float* dg, const float* wout, const float* Z, int w, unsigned n_quads,
                                  float* delta) {
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_quads) return;
  const unsigned q = (unsigned)w / 4;
  const long n = e / q;
  const int u = 4 * (int)(e % q);
  const float d = dg[n];
  const float4 z = *reinterpret_cast<const float4*>(Z + n * w + u);
  const float4 wo = *reinterpret_cast<const float4*>(wout + u);
  *reinterpret_cast<float4*>(delta + n * w + u) =
      make_float4(d * wo.x * elu_d(z.x), d * wo.y * elu_d(z.y), d * wo.z * elu_d(z.z), d * wo.w * elu_d(z.w));
}

// dq[b][j] = sum_s din[b S + s][m + j] (din rows ld floats apart): one block per
// (snapshot, latent component), 256 row lanes with compensated sums, fixed-order tree.
__global__ void dq_kernel(const float* din, int ld, int B, int S, int m, int r, float* dq) {
  const int b = blockIdx.x, j = blockIdx.y;
  __shared__ double red[256];
  CompSum s;
  for (int i = threadIdx.x; i < S; i += blockDim.x) s.add(din[((long)b * S + i) * ld + m + j]);
  red[threadIdx.x] = s.value();
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) dq[(long)b * r + j] = (float)red[0];
}
__global__ void adam_kernel(float* p, const float* g, float* m, float* v, long n, float lr, float c1, float c2) {
  const long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const float gi = g[e];
  const float mi = 0.9f * m[e] + 0.1f * gi;
  const float vi = 0.999f * v[e] + 0.001f * gi * gi;
  m[e] = mi;
  v[e] = vi;
  p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

inline unsigned blocks(long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

size_t trainer_param_count(const crom_trainer* t) { return (size_t)t->lay.total; }

cudaError_t trainer_alloc(crom_trainer* t) {
  auto A = [&](size_t bytes) -> void* {
    void* p = nullptr;
    if (cudaMalloc(&p, bytes > 0 ? bytes : 16) != cudaSuccess) p = nullptr;
    t->owned.push_back(p);  // a failed allocation leaves a nullptr here for the check below
    return p;
  };
  const int m = t->dec.m, r = t->dec.r, w = t->dec.width, L = t->dec.hidden;
  const long N = (long)t->B * t->S;
  // parameter layout
  TrainerLayout& lay = t->lay;
  long o = 0;
  std::vector<int> dims = {m + r};
  for (int l = 0; l < L; ++l) dims.push_back(w);
  dims.push_back(1);
  for (int l = 0; l + 1 < (int)dims.size(); ++l) {
    lay.dec_w.push_back(o);
    o += (long)dims[l + 1] * dims[l];
    lay.dec_b.push_back(o);
    o += dims[l + 1];
  }
  for (size_t c = 1; c < t->lens.size(); ++c) {
    lay.conv.push_back(o);
    o += 7;
  }
  const int Llast = t->lens.back();
  lay.d1w = o; o += 32L * Llast;
  lay.d1b = o; o += 32;
  lay.d2w = o; o += (long)r * 32;
  lay.d2b = o; o += r;
  lay.total = o;
  t->params = (float*)A(o * 4);
  t->grads = (float*)A(o * 4);
  t->am = (float*)A(o * 4);
  t->av = (float*)A(o * 4);
  for (size_t c = 1; c < t->lens.size(); ++c) {
    t->conv_z.push_back((float*)A((size_t)t->B * t->lens[c] * 4));
    t->conv_h.push_back((float*)A((size_t)t->B * t->lens[c] * 4));
  }
  t->d1z = (float*)A((size_t)t->B * 32 * 4);
  t->d1h = (float*)A((size_t)t->B * 32 * 4);
  t->q = (float*)A((size_t)t->B * r * 4);
  t->in0 = (float*)A((size_t)N * (m + r) * 4);
  t->target = (float*)A((size_t)N * 4);
  t->g = (float*)A((size_t)N * 4);
  t->dg = (float*)A((size_t)N * 4);
  for (int l = 0; l < L; ++l) {
    t->Z.push_back((float*)A((size_t)N * w * 4));
    t->H.push_back((float*)A((size_t)N * w * 4));
  }
  t->delta = (float*)A((size_t)N * w * 4);
  t->delta2 = (float*)A((size_t)N * w * 4);
  t->din = (float*)A((size_t)N * (m + r) * 4);
  t->dq = (float*)A((size_t)t->B * r * 4);
  t->split = (float*)A((size_t)kSplitK * w * std::max(w, m + r) * 4);
  t->ed1 = (float*)A((size_t)t->B * 32 * 4);
  t->partial = (double*)A((size_t)blocks(N, 8) * 8);
  t->loss_dev = (double*)A(8);
  t->red = (double*)A((size_t)kColChunks * std::max(std::max(w, 32), r) * 8);
  t->conv_part = (double*)A((t->lens.size() - 1) * kColChunks * 7 * 8);
  for (void* p : t->owned)
    if (!p) return cudaErrorMemoryAllocation;
  cudaError_t e = clear_device(t->am, o * 4);
  if (e == cudaSuccess) e = clear_device(t->av, o * 4);
  return e;
}

void trainer_free(crom_trainer* t) {
  for (void* p : t->owned) cudaFree(p);
  t->owned.clear();
  t->tc = TrainerTc{};
}

template <int BM, int BN, int CN, bool kAK, bool kBK>
static void launch_tiles(const GemmArgs& g, int splits, cudaStream_t s) {
  dim3 grid(blocks(g.N, BN), blocks(g.M, BM), splits);
  constexpr int kNT = BM * BN / 8 / CN;
  gemm_kernel<BM, BN, CN, kAK, kBK><<<grid, kNT, 0, s>>>(g);
}

template <bool kAK, bool kBK>
static void launch_gemm(const crom_trainer* t, const GemmArgs& g, int splits, cudaStream_t s) {
  // the largest tiles that still give the GPU a CTA per SM; where even the smallest do not
  // (the weight gradients of narrow layers, their K ranges fixed), half the columns per
  // thread for a warp on each of the SM's schedulers
  const long big = (long)blocks(g.M, 128) * blocks(g.N, 128) * splits;
  const long small = (long)blocks(g.M, 64) * blocks(g.N, 64) * splits;
  if (g.N > 64 && big >= t->num_sms) launch_tiles<128, 128, 8, kAK, kBK>(g, splits, s);
  else if (g.M > 64 && (long)blocks(g.M, 128) * blocks(g.N, 64) * splits >= t->num_sms) launch_tiles<128, 64, 8, kAK, kBK>(g, splits, s);
  else if (small >= 2 * t->num_sms) launch_tiles<64, 64, 8, kAK, kBK>(g, splits, s);
  else launch_tiles<64, 64, 4, kAK, kBK>(g, splits, s);
}

// C = A * B with an epilogue; K split over partials (then added in order) when `split` is
// given.  A[i][k] = A[i * sai + k * sak], B[k][j] = B[k * sbk + j * sbj]; one of each pair
// of strides is 1 (row-major or transposed storage).
static cudaError_t gemm(crom_trainer* t, cudaStream_t s, int M, int N, int K, const float* A, long sai, long sak,
                        const float* B, long sbk, long sbj, float* C, long ldc, int epi, const float* bias,
                        float* H, const float* Zp, float* split = nullptr) {
  GemmArgs g{M, N, K, A, B, sak == 1 ? sai : sak, sbk == 1 ? sbj : sbk, split ? split : C, ldc, split ? (long)M * ldc : 0,
             split ? (int)kEpiStore : epi, bias, H, Zp, false, false, false};
  auto quads = [](const void* p, long ld) { return ((uintptr_t)p & 15) == 0 && (ld & 3) == 0; };
  g.va = quads(A, g.lda);
  g.vb = quads(B, g.ldb);
  g.vc = quads(g.C, ldc) && (!H || quads(H, ldc)) && (!Zp || quads(Zp, ldc)) && (g.split_stride & 3) == 0;
  const int splits = split ? kSplitK : 1;
  if (sak == 1) {
    if (sbk == 1) launch_gemm<true, true>(t, g, splits, s);
    else launch_gemm<true, false>(t, g, splits, s);
  } else {
    if (sbk == 1) launch_gemm<false, true>(t, g, splits, s);
    else launch_gemm<false, false>(t, g, splits, s);
  }
  if (split) sum_splits_kernel<<<blocks((long)M * ldc, 128), 128, 0, s>>>(split, (long)M * ldc, C);
  return cudaGetLastError();
}

// Deterministic column sums (two passes through t->red).
static void colsum(crom_trainer* t, cudaStream_t s, const float* X, long rows, int cols, float* out) {
  const int chunks = (int)std::min<long>(kColChunks, std::max<long>(rows, 1));
  if (cols % 4 == 0 && ((uintptr_t)X & 15) == 0)
    colsum_part4_kernel<<<dim3(blocks(cols / 4, kColQuads), chunks), dim3(kColQuads, 4), 0, s>>>(X, rows, cols, t->red);
  else
    colsum_part_kernel<<<dim3(blocks(cols, 32), chunks), dim3(32, 8), 0, s>>>(X, rows, cols, t->red);
  colsum_final_kernel<<<blocks(32L * cols, 128), 128, 0, s>>>(t->red, chunks, cols, out);
}

int trainer_set_precision(crom_trainer* t, int precision) {
  if (precision == CROM_PREC_BF16_MIXED && trainer_tc_alloc(t) != cudaSuccess) return CROM_ERR_CUDA;
  t->precision = precision;
  return CROM_OK;
}

// The convolutions and dense layers of the per-snapshot kernels; *first is the first of
// those convolutions (1-based), the ones before it are long.
static EncArgs enc_args(const crom_trainer* t, const float* snaps, int* first) {
  EncArgs a{};
  const TrainerLayout& lay = t->lay;
  int c = 1;
  for (; c < (int)t->lens.size() && t->lens[c - 1] > kEncLin; ++c) {}
  *first = c;
  const float* x = c > 1 ? t->conv_h[c - 2] : snaps;
  for (; c < (int)t->lens.size(); ++c) {
    a.conv[a.n++] = {t->lens[c - 1], t->lens[c], t->params + lay.conv[c - 1], x, t->conv_z[c - 1], t->conv_h[c - 1]};
    x = t->conv_h[c - 1];
  }
  a.Ll = t->lens.back();
  a.r = t->dec.r;
  a.hl = x;
  a.w1 = t->params + lay.d1w;
  a.b1 = t->params + lay.d1b;
  a.w2 = t->params + lay.d2w;
  a.b2 = t->params + lay.d2b;
  a.d1z = t->d1z;
  a.d1h = t->d1h;
  return a;
}

cudaError_t trainer_encode(crom_trainer* t, int nb, const float* snaps, float* q_out, cudaStream_t s) {
  // nb <= B; forward through the encoder only
  int first;
  EncArgs a = enc_args(t, snaps, &first);
  const float* x = snaps;
  for (int c = 1; c < first; ++c) {
    const int Lin = t->lens[c - 1], Lout = t->lens[c];
    conv_fwd_kernel<<<blocks((long)nb * Lout, 256), 256, 0, s>>>(x, Lin, Lout, nb, t->params + t->lay.conv[c - 1],
                                                                t->conv_z[c - 1], t->conv_h[c - 1]);
    x = t->conv_h[c - 1];
  }
  a.q = q_out;
  enc_fwd_kernel<<<nb, kEncThreads, 0, s>>>(a);
  return cudaGetLastError();
}

// Reverse pass from dL/dq (t->dq) to the encoder's gradients.
static cudaError_t trainer_encoder_bwd(crom_trainer* t, const float* snaps, cudaStream_t s) {
  const TrainerLayout& lay = t->lay;
  const int B = t->B;
  float* gr = t->grads;
  int first;
  EncArgs a = enc_args(t, snaps, &first);
  a.dq = t->dq;
  a.ed1 = t->ed1;
  a.zx = first > 1 ? t->conv_z[first - 2] : nullptr;
  enc_bwd_kernel<<<B, kEncThreads, 0, s>>>(a);
  for (int c = first - 1; c > 1; --c)  // through the long convolutions
    conv_dz_kernel<<<blocks((long)B * t->lens[c - 1], 256), 256, 0, s>>>(t->conv_z[c - 1], t->lens[c - 1], t->lens[c], B,
                                                                        t->params + lay.conv[c - 1], t->conv_z[c - 2]);
  const int n_conv = (int)t->lens.size() - 1;
  const bool few = B <= kColChunks;
  ConvGrads cg{};
  cg.n = n_conv;
  cg.B = B;
  EncGrads g{B, a.Ll, a.r, n_conv, few ? 32 + a.r : 0, t->ed1, a.hl, t->dq, t->d1h, gr + lay.d1w, gr + lay.d1b,
             gr + lay.d2w, gr + lay.d2b, {}, {}, {}};
  int chunks = 0;
  for (int c = 0; c < n_conv; ++c) {
    cg.lin[c] = t->lens[c];
    cg.lout[c] = t->lens[c + 1];
    cg.dz[c] = t->conv_z[c];
    cg.x[c] = c == 0 ? snaps : t->conv_h[c - 1];
    g.part[c] = cg.part[c] = t->conv_part + (size_t)c * kColChunks * 7;
    g.chunks[c] = cg.chunks[c] = (int)std::min<long>(kColChunks, std::max<long>((long)B * t->lens[c + 1] / 1024, 1));
    g.gconv[c] = gr + lay.conv[c];
    chunks += cg.chunks[c];
  }
  if (n_conv > 0) conv_grads_kernel<<<chunks, 1024, 0, s>>>(cg);
  enc_grads_kernel<<<enc_weight_blocks(a.Ll, a.r) + (g.n_bias + 6) / 7 + n_conv, kGradThreads, 0, s>>>(g);
  if (!few) {
    colsum(t, s, t->ed1, B, 32, gr + lay.d1b);
    colsum(t, s, t->dq, B, a.r, gr + lay.d2b);
  }
  return cudaGetLastError();
}

cudaError_t trainer_step(crom_trainer* t, const float* snaps, const int* pt_idx, const float* coords, float lr,
                         double* loss_out, cudaStream_t s) {
  const int m = t->dec.m, r = t->dec.r, w = t->dec.width, L = t->dec.hidden;
  const int B = t->B, S = t->S, P = t->P;
  const long N = (long)B * S;
  const TrainerLayout& lay = t->lay;
  float* p = t->params;
  float* gr = t->grads;
  cudaError_t e;
  // ---- encoder forward: q_b
  if ((e = trainer_encode(t, B, snaps, t->q, s)) != cudaSuccess) return e;
  // ---- decoder forward and reverse pass on the sampled points
  const bool tc = t->precision == CROM_PREC_BF16_MIXED;
  if (tc) {
    gather_x_kernel<<<blocks(N, 256), 256, 0, s>>>(snaps, pt_idx, coords, B, S, P, m, t->tc.xin, t->target);
    // the decoder pass also leaves dL/dq_b in t->dq
    if ((e = trainer_decoder_tc(t, loss_out, t->num_sms, s)) != cudaSuccess) return e;
  } else {
    gather_kernel<<<blocks(N, 256), 256, 0, s>>>(snaps, pt_idx, coords, t->q, B, S, P, m, r, t->in0, t->target);
    const float* hin = t->in0;
    int kin = m + r;
    for (int l = 0; l < L; ++l) {
      e = gemm(t, s, (int)N, w, kin, hin, kin, 1, p + lay.dec_w[l], 1, kin, t->Z[l], w, kEpiBiasElu, p + lay.dec_b[l],
               t->H[l], nullptr);
      if (e != cudaSuccess) return e;
      hin = t->H[l];
      kin = w;
    }
    output_loss_kernel<<<blocks(N, 8), 256, 0, s>>>(t->H[L - 1], w, N, p + lay.dec_w[L], p + lay.dec_b[L], t->target,
                                                     t->dg, t->partial);
    loss_final_kernel<<<1, 1024, 0, s>>>(t->partial, (int)blocks(N, 8), N, loss_out ? loss_out : t->loss_dev);
    // output layer: gW_out[u] = sum_n dg[n] H_L[n][u], gb_out = sum dg
    {
      const int per = (int)blocks(blocks(N, kSplitK), kTK) * kTK;
      wout_part_kernel<<<dim3(blocks(w, 32), kSplitK), 256, 0, s>>>(t->dg, t->H[L - 1], (int)N, w, per, t->split);
      sum_splits_kernel<<<blocks(w, 128), 128, 0, s>>>(t->split, w, gr + lay.dec_w[L]);
    }
    colsum(t, s, t->dg, N, 1, gr + lay.dec_b[L]);
    const float* wout = p + lay.dec_w[L];
    const float* zl = t->Z[L - 1];
    if (w % 4 == 0 && ((uintptr_t)wout & 15) == 0 && ((uintptr_t)zl & 15) == 0 && ((uintptr_t)t->delta & 15) == 0 &&
        N * (w / 4) < (1L << 31)) {
      const unsigned nq = (unsigned)(N * (w / 4));
      out_delta4_kernel<<<blocks(N * (w / 4), 256), 256, 0, s>>>(t->dg, wout, zl, w, nq, t->delta);
    } else {
      out_delta_kernel<<<blocks(N * w, 256), 256, 0, s>>>(t->dg, wout, zl, w, N, t->delta);
    }
    float* dcur = t->delta;
    float* dnext = t->delta2;
    for (int l = L - 1; l >= 0; --l) {
      const float* hprev = (l == 0) ? t->in0 : t->H[l - 1];
      const int kprev = (l == 0) ? m + r : w;
      // gW_l [w][kprev] = delta^T hprev (K = N, split), gb_l = column sums of delta
      e = gemm(t, s, w, kprev, (int)N, dcur, 1, w, hprev, kprev, 1, gr + lay.dec_w[l], kprev, kEpiStore, nullptr,
               nullptr, nullptr, t->split);
      if (e != cudaSuccess) return e;
      colsum(t, s, dcur, N, w, gr + lay.dec_b[l]);
      if (l > 0) {
        // delta_{l-1} = (delta_l W_l) * s'(Z_{l-1})
        e = gemm(t, s, (int)N, w, w, dcur, w, 1, p + lay.dec_w[l], w, 1, dnext, w, kEpiTimesEluD, nullptr, nullptr,
                 t->Z[l - 1]);
      } else {
        // input gradient din = delta_1 W_1  [N][m + r]
        e = gemm(t, s, (int)N, m + r, w, dcur, w, 1, p + lay.dec_w[0], m + r, 1, t->din, m + r, kEpiStore, nullptr,
                 nullptr, nullptr);
      }
      if (e != cudaSuccess) return e;
      float* tmp = dcur;
      dcur = dnext;
      dnext = tmp;
    }
  }
  if (!tc) dq_kernel<<<dim3(B, r), 256, 0, s>>>(t->din, m + r, B, S, m, r, t->dq);
  if ((e = trainer_encoder_bwd(t, snaps, s)) != cudaSuccess) return e;
  // ---- Adam
  t->step += 1;
  const float c1 = (float)(1.0 - pow(0.9, (double)t->step));
  const float c2 = (float)(1.0 - pow(0.999, (double)t->step));
  adam_kernel<<<blocks(lay.total, 256), 256, 0, s>>>(p, gr, t->am, t->av, lay.total, lr, c1, c2);
  return cudaGetLastError();
}

}  // namespace crom
