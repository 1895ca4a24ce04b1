// FP32 CUDA-core path: forward-mode decoder evaluation with derivative channels
// (paper Algorithm 2, App. E.1.1, extended to second order), used by
// crom_decode, FP32 crom_reconstruct and the plain FP32 crom_step.
//
// Three kernels form the same sums in the same order (bit-identical results):
// fwd_tile_kernel and fwd_small_kernel (simt_tile.cuh) for many and for few samples, and
// fwd_fp32_kernel for the shapes neither holds (many channels at the largest widths).
//
// fwd_fp32_kernel: one CTA = KS threads per hidden unit (blockDim = KS * width) and a
// tile of S samples.  All channels of a (unit, sample) pair live in one thread, so the
// ELU chain rule needs no communication:
//   z = W h + b;  dz = W dh;  d2z = W d2h
//   h = s(z);     dh = s'(z) dz;  d2h = s''(z) dz^2 + s'(z) d2z
// The activations of the whole tile (width x S*C floats) sit in shared memory;
// the transposed hidden matrices are read through L1 (coalesced in the unit index).
// Each contraction over the width is split in KS slices (one per thread of a unit)
// whose partial sums are added through shared memory, which shortens the serial
// dependency chain.
//
// The FP32 step spreads one instance over ceil(|M_i| / S) CTAs.  Each CTA forms
// its partial normal equations sum_j J_j J_j^T and sum_j J_j rho_j in FP64 from
// the FP32 Jacobian rows (exact products), writes them to scratch and takes a
// ticket; the CTA holding the last ticket adds the partials in a fixed order
// (finish_cta), solves by FP64 Cholesky and updates q (paper §4.3, App. C).
// Nothing ever waits on another CTA.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "crom_internal.h"
#include "linalg.cuh"
#include "tc_common.cuh"

namespace crom {
namespace {

constexpr int kMaxM = 3;
constexpr int kMaxR = 32;
constexpr int kSumGroups = 16;  // groups of partial-row chains (finish_cta)
constexpr int kKSplit = 4;  // threads per hidden unit (width <= 256 -> <= 1024 threads)

enum Mode { kModeDecode = 0, kModeRecon = 1, kModeStep = 2 };

struct FwdParams {
  int mode;
  // decoder
  int m, r, width, hidden;
  const float* w1;
  const float* w1t;  // W_1 transposed, [m + r][width]
  const double* w1q;  // its latent rows in FP64, [r][width]
  const float* b1;
  const float* wt;
  const float* bh;
  const float* wout;
  float bout;
  // channels carried: [value, (difference), dg/dx_k..., second order..., dg/dq_j...]
  int diff, nx, second, nq, C;
  int S;   // samples per CTA
  int LD;  // row stride (floats) of the activation buffers
  // inputs
  const double* q;  // [n][r]
  const int* off;   // decode: pt_off, step: s_off
  const float* x;   // [n][m]
  int n_pts;
  int n_inst;
  int act;        // CROM_ACT_ELU or CROM_ACT_SIREN
  float omega0;   // SIREN frequency
  // decode / recon
  float* out;
  unsigned want;
  // decode of a directional derivative (nq == 1): the one latent channel is seeded
  // with jvp_seed[instance][unit] = (W_1q u_i)[unit] instead of a W_1q column
  const float* jvp_seed;
  // step
  int iter;
  int pde;
  int coef_per_sample;  // alpha indexed by sample (1) or by instance (0)
  double dt;
  const float* alpha;
  const float* vel;
  int max_samples;
  double* qio;
  int* status;
  int n_samples;  // length of the sample arrays: every instance's range must lie inside
  double* partials;
  int max_tiles;  // partial rows per instance
  int n_entries;
  int PS;         // samples per partial row (divides S)
  int groups;     // groups the chains of partial rows are dealt to (1: the last CTA adds all)
  int* counters;        // [n_inst], zero between launches
  int* group_counters;  // [n_inst][groups], zero between launches
  double* targets;  // Delta f_j per sample (FP64), written at GN iteration 0
  double* qbase;    // q_n per instance, written at GN iteration 0
};

__device__ __forceinline__ void elu3(float z, float& s0, float& s1, float& s2) {
  // without a divergent branch (a NaN stays a NaN)
  const float zm = z > 0.f ? 0.f : z, e = expf(zm), em = expm1f(zm);
  s0 = z > 0.f ? z : em;
  s1 = z > 0.f ? 1.f : e;
  s2 = z > 0.f ? 0.f : e;
}

// s(a) - s(a - d) without cancellation: the difference channel carries
// h(q^(k)) - h(q_n) through the network, so that the Gauss-Newton residual
// g(y, q^(k)) - g(y, q_n) - Delta f keeps its relative accuracy when the two
// evaluations agree to many digits.
__device__ __forceinline__ float elu_diff(float a, float d) {
  const float b = a - d;
  if (a > 0.f && b > 0.f) return d;
  if (a <= 0.f && b <= 0.f) return -expf(a) * expm1f(-d);
  const float sa = a > 0.f ? a : expm1f(a);
  const float sb = b > 0.f ? b : expm1f(b);
  return sa - sb;
}

// SIREN, s(z) = sin(w z): s' = w cos(w z), s'' = -w^2 sin(w z).
__device__ __forceinline__ void siren3(float z, float w, float& s0, float& s1, float& s2) {
  float sn, cs;
  sincosf(w * z, &sn, &cs);
  s0 = sn;
  s1 = w * cs;
  s2 = -w * w * sn;
}

// sin(w a) - sin(w (a - d)) = 2 cos(w (a - d/2)) sin(w d / 2), without the
// cancellation of the direct difference.
__device__ __forceinline__ float siren_diff(float a, float d, float w) {
  return 2.f * cosf(w * (a - 0.5f * d)) * sinf(0.5f * w * d);
}

// Apply the activation chain in place to row `row` (pre-activation channels of
// one hidden unit) for the samples s0, s0 + ds, ... < S.
__device__ __forceinline__ void activate_row(float* row, const FwdParams& p, int sbeg, int ds) {
  const int C = p.C;
  for (int s = sbeg; s < p.S; s += ds) {
    float* c = row + s * C;
    float s0, s1, s2;
    const float za = c[0];
    if (p.act == CROM_ACT_SIREN) {
      siren3(za, p.omega0, s0, s1, s2);
      if (p.diff) c[1] = siren_diff(za, c[1], p.omega0);
    } else {
      elu3(za, s0, s1, s2);
      if (p.diff) c[1] = elu_diff(za, c[1]);
    }
    c[0] = s0;
    const int ox = 1 + p.diff;
    float zx[kMaxM];
    float sq = 0.f;
    for (int k = 0; k < p.nx; ++k) {
      zx[k] = c[ox + k];
      c[ox + k] = s1 * zx[k];
      sq += zx[k] * zx[k];
    }
    int o = ox + p.nx;
    if (p.second == kSecondPerK) {
      for (int k = 0; k < p.m; ++k) c[o + k] = s2 * zx[k] * zx[k] + s1 * c[o + k];
      o += p.m;
    } else if (p.second == kSecondLap) {
      c[o] = s2 * sq + s1 * c[o];
      o += 1;
    }
    for (int j = 0; j < p.nq; ++j) c[o + j] *= s1;
  }
}

__device__ int find_instance(const int* off, int n_inst, int point) {
  int lo = 0, hi = n_inst - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (__ldg(&off[mid]) <= point) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// ---- shared by the forward kernels: the linear output layer and what a CTA does with it

// outv[t] = w_out . (column t of the last activations), one thread per column, one FMA
// chain in k; the value channel's columns (t < S with the [channel][sample] order, S > 0;
// else every C-th) get b_out.
__device__ __forceinline__ void output_layer(const FwdParams& p, const float* wout, const float* H, int LD, int NP,
                                             float* outv, int S) {
  const int W = p.width;
  for (int t = threadIdx.x; t < NP; t += blockDim.x) {
    float acc = 0.f;
#pragma unroll 16
    for (int k = 0; k < W; ++k) acc = fmaf(wout[k], H[k * LD + t], acc);
    if (S > 0 ? t < S : t % p.C == 0) acc += p.bout;
    outv[t] = acc;
  }
}

// Entry e of the packed normal equations: (a, b), a <= b, of J^T J in row order, or
// (a, -1) of J^T rho.
__device__ __forceinline__ void entry_of(int e, int r, int ntri, int& a, int& b) {
  if (e < ntri) {
    // row a starts at a r - a (a - 1) / 2
    const float t = r + 0.5f;
    a = (int)(t - sqrtf(t * t - 2.f * e));
    if (a * r - a * (a - 1) / 2 > e) --a;
    if ((a + 1) * r - (a + 1) * a / 2 <= e) ++a;
    b = a + e - (a * r - a * (a - 1) / 2);
  } else {
    a = e - ntri;
    b = -1;
  }
}
// x[0] + x[stride] + .. (n terms, in order), kAhead loads issued ahead of the additions.
template <int kAhead>
__device__ __forceinline__ double chain_sum(const double* x, int n, size_t stride) {
  double acc = 0.0;
  for (int k0 = 0; k0 < n; k0 += kAhead) {
    double v[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k)
      if (k0 + k < n) v[k] = __ldcg(x + (size_t)(k0 + k) * stride);
#pragma unroll
    for (int k = 0; k < kAhead; ++k)
      if (k0 + k < n) acc += v[k];
  }
  return acc;
}

// A ticket that publishes the CTA's writes before it (ordered by a barrier) and, to
// whoever draws the last one, those before the others (a full fence on each side of a
// relaxed atomic cost 2 us more per launch with the groups' second ticket).
__device__ __forceinline__ int ticket(int* counter, int n) {
  int old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(counter), "r"(n) : "memory");
  return old;
}

// Output channels c of sample s at outv[s * ss + c * cs]: written out (decode,
// reconstruction), or (step) the residuals, this CTA's partial normal equations and, in
// the instance's last CTA, their sum and the solve.  rho [S], Amat [r][r + 1], jd [S][r]
// and red2 ([max(4 width, entries)]) are shared memory.
//
// The FP64 sums are formed in one fixed order whatever the tiling: a partial row per
// p.PS samples (in order of the samples; `total` = the instance's); row t belongs to chain t mod `per` (per =
// 4 width / entries, at least 1); a chain adds its rows in order, and the chains are
// added in order.  A call's result therefore does not depend on which kernel ran.
// FP64 is slow here (64 clocks per warp instruction), so with p.groups > 1 the chains
// are dealt to that many groups, and the CTA that completes a group's last row adds its
// chains (into their first rows); the CTA that completes the last group adds the chains.
//
// kAhead: partial rows read ahead of their addition (20 hide the memory latency of a chain
// of a few hundred samples; the general kernel's 64 registers hold 4).
template <int kAhead, bool kPoints = false>
__device__ __forceinline__ void finish_cta(const FwdParams& p, const float* outv, int ss, int cs, int inst, int first,
                                           int ns, int ntiles, int total, double* rho, double* Amat, double* jd,
                                           double* red2) {
  __shared__ int s_flag;
  __shared__ unsigned s_groups;
  const int tid = threadIdx.x, NT = blockDim.x, m = p.m, r = p.r;
  if (p.mode == kModeRecon) {
    for (int s = tid; s < ns; s += NT) p.out[(size_t)blockIdx.y * p.n_pts + first + s] = outv[s * ss];
    return;
  }
  const int n2 = (p.second == kSecondPerK) ? m : (p.second == kSecondLap ? 1 : 0);
  const int ox = 1 + p.diff, o2 = ox + p.nx, oq = o2 + n2;
  if (p.mode == kModeDecode) {
    for (int s = tid; s < ns; s += NT) {
      const float* c = outv + s * ss;
      const size_t N = (size_t)p.n_pts, pt = (size_t)(first + s);
      int row = 0;
      if (p.want & CROM_WANT_VAL) p.out[(row++) * N + pt] = c[0];
      if (p.want & CROM_WANT_DX)
        for (int k = 0; k < m; ++k) p.out[(row++) * N + pt] = c[(ox + k) * cs];
      if (p.want & CROM_WANT_DXX)
        for (int k = 0; k < m; ++k) p.out[(row++) * N + pt] = c[(o2 + k) * cs];
      if (p.want & CROM_WANT_LAP) {
        float lap = 0.f;
        for (int k = 0; k < n2; ++k) lap += c[(o2 + k) * cs];
        p.out[(row++) * N + pt] = lap;
      }
      if (p.want & CROM_WANT_DQ)  // r rows, or the one directional row of a tangent decode
        for (int j = 0; j < p.nq; ++j) p.out[(row++) * N + pt] = c[(oq + j) * cs];
    }
    return;
  }
  if constexpr (kPoints) return;  // decode and reconstruction alone

  // ---- step: residual per sample (Step 2 at iteration 0), partial normal equations
  for (int i = tid; i < ns * r; i += NT) jd[i] = (double)outv[i / r * ss + (oq + i % r) * cs];
  for (int s = NT - 1 - tid; s < ns; s += NT) {
    double res;
    const float* c = outv + s * ss;
    const size_t j = (size_t)(first + s);
    if (p.iter == 0) {
      double df;
      const double a = (double)p.alpha[p.coef_per_sample ? j : (size_t)inst];
      if (p.pde == CROM_PDE_HEAT) {
        df = p.dt * a * (double)c[o2 * cs];
      } else {
        double adv = 0.0;
        for (int k = 0; k < m; ++k) adv += (double)p.vel[j * m + k] * (double)c[(ox + k) * cs];
        df = p.dt * (-adv + a * (double)c[o2 * cs]);
      }
      p.targets[j] = df;
      res = -df;  // g(y_j, q^(0)) - f_{n+1}(y_j) with f_{n+1} = g(y_j, q_n) + Delta f_j
    } else {
      // g(y_j, q^(k)) - f_{n+1}(y_j) = [g(y_j, q^(k)) - g(y_j, q_n)] - Delta f_j,
      // the bracket being the difference channel.
      res = (double)c[cs] - p.targets[j];
    }
    rho[s] = res;
  }
  __syncthreads();
  const int ne = p.n_entries, ntri = r * (r + 1) / 2;
  const int row0 = blockIdx.y * (p.S / p.PS), rows = (ns + p.PS - 1) / p.PS;  // this CTA's partial rows
  double* base = p.partials + (size_t)inst * p.max_tiles * ne;
  for (int e = tid; e < ne; e += NT) {
    int a, b;
    entry_of(e, r, ntri, a, b);  // (a, b) of J^T J, or (a, -1) of J^T rho
    for (int t = 0; t < rows; ++t) {
      double acc = 0.0;
      const int s1 = min(ns, (t + 1) * p.PS);
      for (int s = t * p.PS; s < s1; ++s) acc += jd[s * r + a] * (b >= 0 ? jd[s * r + b] : rho[s]);
      base[(size_t)(row0 + t) * ne + e] = acc;
    }
  }
  const int nrows = (total + p.PS - 1) / p.PS;
  const int per = max(1, 4 * p.width / ne), chains = min(per, nrows);
  const int groups = min(p.groups, chains);
  int* counters = p.counters + inst;  // CTAs, or completed groups
  // the barrier makes every thread's rows visible to thread 0, whose ticket publishes them
  // (release is cumulative)
  __syncthreads();
  if (groups > 1) {
    int* gcount = p.group_counters + (size_t)inst * p.groups;
    if (tid < 32) {
      // lane g: this CTA's rows of group g (chains g, g + groups, ..) and the group's rows in all
      int mine = 0, all = 0;
      if (tid < groups) {
        for (int t = row0; t < row0 + rows; ++t) mine += t % per % groups == tid;
        for (int j = tid; j < chains; j += groups) all += (nrows - j + per - 1) / per;
      }
      const bool last = mine > 0 && ticket(&gcount[tid], mine) == all - mine;
      const unsigned d = __ballot_sync(0xffffffffu, last);
      if (tid == 0) s_groups = d;
    }
    __syncthreads();
    const unsigned done = s_groups;
    if (!done) return;
    for (int g = 0; g < groups; ++g) {
      if (!(done >> g & 1)) continue;
      const int nc = (chains - g + groups - 1) / groups;
      for (int i = tid; i < nc * ne; i += NT) {
        const int j = g + i / ne * groups;
        double* row = base + (size_t)j * ne + i % ne;
        *row = chain_sum<kAhead>(row, (nrows - j + per - 1) / per, (size_t)per * ne);
      }
      if (tid == 0) gcount[g] = 0;
    }
    __syncthreads();
    if (tid == 0) {
      const int n = __popc(done);
      s_flag = ticket(counters, n) == groups - n;
    }
  } else if (tid == 0) {
    s_flag = ticket(counters, 1) == ntiles - 1;
  }
  __syncthreads();
  if (!s_flag) return;

  // ---- last CTA of the instance: add the chains in order, solve, update q
  if (groups <= 1) {
    for (int i = tid; i < chains * ne; i += NT) {
      const int e = i % ne, j = i / ne;
      red2[i] = chain_sum<kAhead>(base + (size_t)j * ne + e, (nrows - j + per - 1) / per, (size_t)per * ne);
    }
    __syncthreads();
  }
  for (int e = tid; e < ne; e += NT) {
    double acc;
    if (groups > 1) {
      acc = chain_sum<kAhead>(base + e, chains, (size_t)ne);
    } else {
      acc = 0.0;
      for (int j = 0; j < chains; ++j) acc += red2[j * ne + e];
    }
    int a, b;
    entry_of(e, r, ntri, a, b);
    if (b >= 0) {
      Amat[a * (r + 1) + b] = acc;
      Amat[b * (r + 1) + a] = acc;
    } else {
      Amat[a * (r + 1) + r] = -acc;  // right-hand side -J^T rho
    }
  }
  __syncthreads();
  if (tid < 32) {
    // Cholesky A = L L^T and the two triangular solves, spread over one warp
    const int st = chol_solve_warp(Amat, r, tid);
    if (st == CROM_OK && tid < r) {
      if (p.iter == 0) p.qbase[(size_t)inst * r + tid] = p.qio[(size_t)inst * r + tid];
      p.qio[(size_t)inst * r + tid] += Amat[tid * (r + 1) + r];
    }
    if (tid == 0) {
      p.status[inst] = st;
      counters[0] = 0;
    }
  }
}

#include "simt_tile.cuh"

// What an instantiation serves: the step, decode and reconstruction, or the
// tangent-velocity decode, whose directional channel is seeded per instance.  Apart, since
// each has 64 registers (1024 threads): a decode's products leave out the step's reduction
// and solve.
enum Serves { kServesStep, kServesPoints, kServesTangent };
template <Serves kServes>
__device__ __forceinline__ void fwd_fp32_body(const FwdParams& p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = p.width, S = p.S, C = p.C, LD = p.LD, m = p.m, r = p.r;
  // KS threads per hidden unit: thread (u, ks) owns unit u and the ks-th slice of
  // the K range of every contraction (and the samples s = ks mod KS elsewhere).
  const int tid = threadIdx.x, NT = blockDim.x;
  const int u = tid % W, ks = tid / W, KS = NT / W;
  const int NP = S * C;
  const int NPP = (NP + 15) & ~15;

  float* Hin = reinterpret_cast<float*>(smem_raw);
  float* Hout = Hin + W * LD;
  double* qs = reinterpret_cast<double*>(Hout + W * LD);  // [S][r]
  double* rho = qs + S * r;                               // [S]
  double* Amat = rho + S;                                 // [r][r + 1]
  double* dqs = Amat + r * (r + 1);                       // [r]: q^(k) - q_n
  float* xs = reinterpret_cast<float*>(dqs + r);          // [S][m]
  float* outv = xs + S * m;                               // [NPP]
  // [KS][W][16] split-K partial sums (16-byte aligned: also reused as doubles)
  float* red = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(outv + NPP) + 15) & ~uintptr_t(15));

  // ---- which samples does this CTA own?
  int inst = 0, first = 0, ns = 0, ntiles = 0, msz = 0;
  if constexpr (kServes == kServesStep) {
    inst = blockIdx.x;
    const int t = blockIdx.y;
    const int o0 = __ldg(&p.off[inst]);
    msz = __ldg(&p.off[inst + 1]) - o0;
    if (p.iter == 0) {
      if (msz < r || msz > p.max_samples || o0 < 0 || o0 + msz > p.n_samples) {
        if (t == 0 && tid == 0) p.status[inst] = CROM_ERR_INVALID_ARG;
        return;
      }
    } else if (p.status[inst] != CROM_OK) {
      return;
    }
    ntiles = (msz + S - 1) / S;
    if (t >= ntiles) return;
    first = o0 + t * S;
    ns = min(S, msz - t * S);
  } else {
    first = blockIdx.x * S;
    ns = min(S, p.n_pts - first);
    if (ns <= 0) return;
  }

  // ---- stage coordinates and latent codes (padding samples repeat the first one)
  for (int i = tid; i < S * m; i += NT) {
    const int s = i / m, k = i % m;
    xs[i] = p.x[(size_t)(first + (s < ns ? s : 0)) * m + k];
  }
  for (int i = tid; i < S * r; i += NT) {
    const int s = i / r, j = i % r;
    int code;
    if (p.mode == kModeStep) code = inst;
    else if (p.mode == kModeRecon) code = blockIdx.y;
    else code = find_instance(p.off, p.n_inst, first + (s < ns ? s : 0));
    qs[i] = (p.mode == kModeStep) ? p.qio[(size_t)code * r + j] : p.q[(size_t)code * r + j];
  }
  if (p.diff)
    for (int j = tid; j < r; j += NT) dqs[j] = p.qio[(size_t)inst * r + j] - p.qbase[(size_t)inst * r + j];
  for (int i = tid; i < 2 * W * LD; i += NT) Hin[i] = 0.f;  // zero both buffers incl. padding
  __syncthreads();

  // ---- layer 1: pre-activation channels of unit u, then the activation chain
  {
    float* row = Hin + u * LD;
    const float* w1 = p.w1t + u;  // entry k at w1[k * W]
    const double* w1q = p.w1q + u;
    const double b1 = (double)p.b1[u];
    double cshared = b1;
    const bool shared_q = (p.mode != kModeDecode);
    if (shared_q) {
      for (int j = 0; j < r; ++j) cshared += w1q[j * W] * qs[j];
    }
    double zd = 0.0;
    if (p.diff) {
      for (int j = 0; j < r; ++j) zd += w1q[j * W] * dqs[j];
    }
    for (int s = ks; s < S; s += KS) {
      double c = cshared;
      if (!shared_q) {
        c = b1;
        for (int j = 0; j < r; ++j) c += w1q[j * W] * qs[s * r + j];
      }
      float z = (float)c;
      for (int k = 0; k < m; ++k) z = fmaf(w1[k * W], xs[s * m + k], z);
      float* ch = row + s * C;
      ch[0] = z;
      if (p.diff) ch[1] = (float)zd;
      const int ox = 1 + p.diff;
      for (int k = 0; k < p.nx; ++k) ch[ox + k] = w1[k * W];
      int o = ox + p.nx;
      const int n2 = (p.second == kSecondPerK) ? m : (p.second == kSecondLap ? 1 : 0);
      for (int k = 0; k < n2; ++k) ch[o + k] = 0.f;
      o += n2;
      if (kServes == kServesTangent) {
        const int code = find_instance(p.off, p.n_inst, first + (s < ns ? s : 0));
        ch[o] = __ldg(&p.jvp_seed[(size_t)code * W + u]);
      } else {
        for (int j = 0; j < p.nq; ++j) ch[o + j] = w1[(m + j) * W];
      }
    }
    activate_row(row, p, ks, KS);
  }
  __syncthreads();

  // ---- hidden layers 2..hidden
  for (int l = 0; l < p.hidden - 1; ++l) {
    const float* Wt = p.wt + (size_t)l * W * W;
    float* orow = Hout + u * LD;
    const int kper = W / KS;
    for (int j0 = 0; j0 < NPP; j0 += 16) {
      float acc[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[i] = 0.f;
      const float* hcol = Hin + j0;
      // The next kWAhead weights are on their way while the current ones are used (kper is a
      // multiple of 8; the step's registers hold four).  Left to the compiler's unrolling, the
      // loads in flight, and the time, changed with the code around this loop: 16137 points
      // of 36 channels, width 96, 7.9 ms, 7.2 so; a step of 204 x 32 samples, r = 32, width
      // 160, 7.7 and 7.0 ms.
      constexpr int kWAhead = kServes == kServesStep ? 4 : 8;
      const int kbeg = ks * kper, kend = kbeg + kper;
      float next[kWAhead];
#pragma unroll
      for (int i = 0; i < kWAhead; ++i) next[i] = __ldg(&Wt[(size_t)(kbeg + i) * W + u]);
#pragma unroll 1
      for (int k0 = kbeg; k0 < kend; k0 += kWAhead) {
        float wv[kWAhead];
#pragma unroll
        for (int i = 0; i < kWAhead; ++i) wv[i] = next[i];
        if (k0 + kWAhead < kend) {
#pragma unroll
          for (int i = 0; i < kWAhead; ++i) next[i] = __ldg(&Wt[(size_t)(k0 + kWAhead + i) * W + u]);
        }
#pragma unroll
        for (int i = 0; i < kWAhead; ++i) {
          const float wk = wv[i];
          const float4* h4 = reinterpret_cast<const float4*>(hcol + (k0 + i) * LD);
          const float4 a = h4[0], b = h4[1], c = h4[2], d = h4[3];
          acc[0] = fmaf(wk, a.x, acc[0]);  acc[1] = fmaf(wk, a.y, acc[1]);
          acc[2] = fmaf(wk, a.z, acc[2]);  acc[3] = fmaf(wk, a.w, acc[3]);
          acc[4] = fmaf(wk, b.x, acc[4]);  acc[5] = fmaf(wk, b.y, acc[5]);
          acc[6] = fmaf(wk, b.z, acc[6]);  acc[7] = fmaf(wk, b.w, acc[7]);
          acc[8] = fmaf(wk, c.x, acc[8]);  acc[9] = fmaf(wk, c.y, acc[9]);
          acc[10] = fmaf(wk, c.z, acc[10]); acc[11] = fmaf(wk, c.w, acc[11]);
          acc[12] = fmaf(wk, d.x, acc[12]); acc[13] = fmaf(wk, d.y, acc[13]);
          acc[14] = fmaf(wk, d.z, acc[14]); acc[15] = fmaf(wk, d.w, acc[15]);
        }
      }
      // add the KS partial sums of unit u: thread (u, ks) finishes 16 / KS of the columns
      float* mine = red + ((size_t)ks * W + u) * 16;
#pragma unroll
      for (int i = 0; i < 16; ++i) mine[i] = acc[i];
      __syncthreads();
      for (int i = ks * (16 / KS); i < (ks + 1) * (16 / KS); ++i) {
        float v = 0.f;
        for (int kk = 0; kk < KS; ++kk) v += red[((size_t)kk * W + u) * 16 + i];
        orow[j0 + i] = v;
      }
      __syncthreads();
    }
    const float bias = p.bh[(size_t)l * W + u];
    for (int s = ks; s < S; s += KS) orow[s * C] += bias;
    activate_row(orow, p, ks, KS);
    __syncthreads();
    float* tmp = Hin; Hin = Hout; Hout = tmp;
  }

  output_layer(p, p.wout, Hin, LD, NP, outv, 0);
  __syncthreads();
  finish_cta<4, kServes != kServesStep>(p, outv, C, 1, inst, first, ns, ntiles, msz, rho, Amat, qs, reinterpret_cast<double*>(red));
}

// (up to 1024 threads per CTA: the bound keeps it within 64 registers)
template <Serves kServes>
__global__ void __launch_bounds__(1024) fwd_fp32_kernel(FwdParams p) { fwd_fp32_body<kServes>(p); }

size_t fwd_smem_bytes(int W, int S, int C, int m, int r, int* LD_out) {
  const int NP = S * C;
  const int NPP = (NP + 15) & ~15;
  int LD = NPP + 4;
  *LD_out = LD;
  size_t b = (size_t)2 * W * LD * sizeof(float);
  b += (size_t)S * r * sizeof(double) + (size_t)S * sizeof(double) + (size_t)r * (r + 1) * sizeof(double) +
       (size_t)r * sizeof(double);
  b += (size_t)S * m * sizeof(float) + (size_t)NPP * sizeof(float);
  b += (size_t)kKSplit * W * 16 * sizeof(float);  // split-K partial sums
  return b + 64;
}

// Which of the forward kernels runs a launch.
enum FwdKernel { kFwdGeneral = 0, kFwdTile2, kFwdTile3, kFwdSmall };
constexpr size_t kMaxSmem = kMaxDynSmem;

cudaError_t launch_fwd(FwdParams& p, FwdKernel kind, dim3 grid, cudaStream_t s) {
  const int W = p.width;
  auto go = [&](auto kernel, int threads, size_t smem) -> cudaError_t {
    const cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, threads, smem, s>>>(p);
    return cudaGetLastError();
  };
  const bool siren = p.act == CROM_ACT_SIREN;
  if (kind == kFwdTile2 || kind == kFwdTile3) {
    p.LD = tile_ld(p.C, p.S);
    const size_t smem = tile_smem_bytes(W, p.S, p.C, p.m, p.r);
    const int tq = kind == kFwdTile2 ? 2 : 3, threads = tile_threads(W, p.S, p.C, tq);
    auto tile = [&](auto k68, auto k132) { return p.LD == 68 ? go(k68, threads, smem) : go(k132, threads, smem); };
    if (tq == 2)
      return siren ? tile(fwd_tile_kernel<2, true, 68>, fwd_tile_kernel<2, true, 132>)
                   : tile(fwd_tile_kernel<2, false, 68>, fwd_tile_kernel<2, false, 132>);
    return siren ? tile(fwd_tile_kernel<3, true, 68>, fwd_tile_kernel<3, true, 132>)
                 : tile(fwd_tile_kernel<3, false, 68>, fwd_tile_kernel<3, false, 132>);
  }
  if (kind != kFwdGeneral) {
    // more threads than the products need fetch the weights and share the activation passes
    const size_t smem = small_smem_bytes(W, p.S, p.C, p.m, p.r, p.hidden);
    // The two widths of the decoders in use are compile-time: eight rows of K unrolled against
    // two (a step of 200 samples 66.8 against 69.2 us at width 128, 52.1 against 55.2 at 64,
    // values alone 16.6 against 17.7).
    const auto kernel = W == 64 ? fwd_small_kernel<64> : W == 128 ? fwd_small_kernel<128> : fwd_small_kernel<0>;
    if (p.mode != kModeStep) return go(kernel, kSmallThreads, smem);
    // a chain of launches that each wait for one CTA's solve: the next one's CTAs start and
    // load the decoder meanwhile (200 samples, width 128: 71.5 us a step of two without, 66.8 with;
    // width 64: 53.5 and 52.1)
    const cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
  }
  const size_t smem = fwd_smem_bytes(W, p.S, p.C, p.m, p.r, &p.LD);
  const auto kernel = p.mode == kModeStep ? fwd_fp32_kernel<kServesStep>
                      : p.jvp_seed        ? fwd_fp32_kernel<kServesTangent>
                                          : fwd_fp32_kernel<kServesPoints>;
  return go(kernel, W * kKSplit, smem);
}

// The tile kernel's variant for S samples of C channels, or kFwdGeneral if none fits.
FwdKernel tile_variant(int W, int S, int C, int m, int r) {
  if (tile_ld(C, S) == 0 || tile_smem_bytes(W, S, C, m, r) > kMaxSmem) return kFwdGeneral;
  // three quads per thread where they give whole 128-thread CTAs of 8 samples
  if (S == 8 && tile_threads(W, S, C, 3) <= 128) return kFwdTile3;
  if (tile_threads(W, S, C, 2) <= 256) return kFwdTile2;
  if (tile_threads(W, S, C, 3) <= 256) return kFwdTile3;
  return kFwdGeneral;
}
// Samples per CTA of the tile kernel for `sets` groups of n samples: 8 with three quads
// per thread if that fills 128 threads, else the largest multiple of 4 with at most 128
// threads (256 for a lone value channel), in any case two CTAs per SM.
FwdKernel tile_plan(const crom_ctx* ctx, long long sets, long long n, int C, int* S) {
  const int W = ctx->desc.width, m = ctx->desc.m, r = ctx->desc.r;
  auto many = [&](int t) { return t == 4 || sets * ((n + t - 1) / t) >= 2LL * ctx->num_sms; };
  const int t3 = tile_threads(W, 8, C, 3);
  if (t3 > 96 && t3 <= 128 && many(8) && tile_variant(W, 8, C, m, r) != kFwdGeneral) {
    *S = 8;
    return kFwdTile3;
  }
  for (int t = 64; t >= 4; t -= 4) {
    if (t > 4 && (tile_threads(W, t, C, 2) > (C == 1 ? 256 : 128) || !many(t))) continue;
    const FwdKernel k = tile_variant(W, t, C, m, r);
    if (k != kFwdGeneral) {
      *S = t;
      return k;
    }
  }
  return kFwdGeneral;
}
// Whether the latency kernel holds S samples of C channels.
bool small_fits(int W, int S, int C, int m, int r, int hidden) {
  return S * C <= kSmallLD - 4 && small_smem_bytes(W, S, C, m, r, hidden) <= kMaxSmem &&
         small_gemm_threads(W, S, C) <= kSmallThreads;
}

int pick_samples(int W, int C, int m, int r, int want);

// Which kernel N samples of C channels get (decode, reconstruction and step); all three
// measured on 1450 shapes (widths 32 to 256, 1 to 36 channels, 1 to 10^5 samples), 900 of
// them around the lines: with these the choice is 5 % from the best on average there, and
// nowhere more than 2 % slower than the general kernel was alone.
//  * The tile kernel from 3.25 warps per SM on (a warp: 8 units x 8 columns a lane): 0.3 to
//    0.9 of the general kernel's time above the line, 1.2 to 3.5 times it below (one warp
//    per CTA walks all of K: 1362 values of width 256, 471 us against 181 us).  With two to
//    four channels from 4.25, and in proportion to the width above 160, as a CTA's chain over K
//    grows while the general kernel splits it (3364 points of two channels, width 224: 236
//    against 164 us).  A lone channel needs four at width 128 and so on in proportion; at
//    width 32 with SIREN 12 (its sines outweigh the products: 50 x 1158 values 131 against
//    101 us).  One layer has no products at all: seven (3483 points of nine channels, width
//    64, 17 against 13 us).  The step's bound on N counts every instance at its largest: six,
//    in 1D (few channels, short uneven instances) ten, of the channels that its iterations
//    carry on average (seven instances of 415 samples, r = 1, three iterations: 657 against
//    591 us).  A bound far above the samples that there are gives CTAs without work: of
//    these four (one instance of 1768 samples bounded by 6284, width 32: 364 against 251 us),
//    20 for more than ten channels of width 32 (95 instances, r = 6, four layers: 435
//    against 397).  One layer has only the channels' activations to gain from: ten (in 1D
//    15), and a width of seven times the channels (two instances of 2181 samples, r = 8,
//    width 64: 185 against 131 us).  Both take at least 64 and four instances: the small
//    CTAs' threads are alone with a long instance's sums (two of 20000 samples, 13 channels,
//    width 32: 1961 against 1666 us).  By 1300 steps, half of them of one layer: two above
//    1.015 of the general kernel's time (1.042, 1.017), 0.66 on average where tiles are used.
//  * Else the latency kernel, two samples per CTA where one would not fit the GPU at once
//    (200 samples of a 2D step: 67 us with two, 91 us with one per CTA), if its CTAs take
//    no more rounds of the GPU than (C + 1) / 2 (step: C / 2): its time grows with the rounds, the
//    general kernel's with the channels (1000 values of width 64: 1.7 times, 45 x 5
//    channels of 600: 0.9 times).  Width 32 and two layers leave too little to gain in a
//    second round, three layers in a third.  Steps of one layer with up to six codes, and
//    of two up to width 96 with up to three, take it for instances of at most 16 samples:
//    longer ones spend more on its rows' tickets and sums than the products gain (one
//    instance of 213, r = 1, width 128, one layer: 33 against 23 us; 320 steps of one and
//    two layers: none above 1.02 of the general kernel's time, 0.87 and, as rollouts, 0.91
//    on average).
//  * Else the general kernel.
// (columns: N C; held: a step's, of the samples that there are)
bool tile_pays(const crom_ctx* ctx, long long columns, int C, bool step, long long held = 0, int n_inst = 0) {
  const int W = ctx->desc.width;
  const long long warps = columns * W / 2048, sms = ctx->num_sms;
  long long quarters;  // of a warp per SM
  if (step) {
    const bool one = ctx->desc.hidden == 1;
    const bool narrow = W == 32 && C > 10;
    const int least = one ? (ctx->desc.m == 1 ? 15 : 10) : narrow ? 20 : 4;
    if ((one && (7 * C > W || n_inst < 4)) || (!one && narrow && n_inst < 64) || held * W / 2048 < least * sms) return false;
    quarters = ctx->desc.m == 1 ? 40 : 24;
  } else if (ctx->desc.hidden == 1) quarters = 28;
  else if (C == 1) quarters = W == 32 && ctx->desc.activation == CROM_ACT_SIREN ? 48 : std::max(12, W / 8);
  else quarters = C > 4 ? 13 : std::max(17, W / 8 - 4);
  return 4 * warps >= quarters * sms;
}
bool small_pays(const crom_ctx* ctx, long long N, int S, int C, bool step) {
  const long long ctas = (N + S - 1) / S, rounds = (ctas + ctx->num_sms - 1) / ctx->num_sms;
  const int hidden = ctx->desc.hidden;
  return rounds <= 1 || (ctx->desc.width > 32 && hidden > 2 && (hidden > 3 || rounds <= 2) && 2 * rounds <= C + !step);
}

FwdKernel plan_points(const crom_ctx* ctx, long long sets, long long n, int C, int general_want, int* S) {
  const int W = ctx->desc.width, m = ctx->desc.m, r = ctx->desc.r;
  const long long N = sets * n;
  if (tile_pays(ctx, N * C, C, false)) {
    const FwdKernel k = tile_plan(ctx, sets, n, C, S);
    if (k != kFwdGeneral) return k;
  }
  for (*S = N > ctx->num_sms ? 2 : 1; *S >= 1; --*S)
    if (small_fits(W, *S, C, m, r, ctx->desc.hidden) && small_pays(ctx, N, *S, C, false)) return kFwdSmall;
  *S = pick_samples(W, C, m, r, general_want);
  return kFwdGeneral;
}

void fill_decoder(FwdParams& p, const crom_ctx* ctx) {
  p.m = ctx->desc.m;
  p.r = ctx->desc.r;
  p.width = ctx->desc.width;
  p.hidden = ctx->desc.hidden;
  p.w1 = ctx->w.w1;
  p.w1t = ctx->w.w1t;
  p.w1q = ctx->w.w1q;
  p.b1 = ctx->w.b1;
  p.wt = ctx->w.wt;
  p.bh = ctx->w.bh;
  p.wout = ctx->w.wout;
  p.bout = ctx->w.bout;
  p.act = ctx->desc.activation;
  p.omega0 = ctx->desc.omega0;
}

// Largest tile that keeps the two activation buffers within 200 KB.
int pick_samples(int W, int C, int m, int r, int want) {
  int S = want;
  int LD;
  while (S > 1 && fwd_smem_bytes(W, S, C, m, r, &LD) > 200 * 1024) S >>= 1;
  return S;
}

}  // namespace

namespace {
// Layer-1 seed of the directional derivative along qdot_i = (q_i - q_prev_i) / dt:
// seed[i][u] = sum_j W_1[u][m + j] qdot_i[j], an FP64 sum rounded once.
__global__ void jvp_seed_kernel(const float* __restrict__ w1, int m, int r, int W, const double* __restrict__ q,
                                const double* __restrict__ q_prev, double inv_dt, int n_inst, float* seed) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_inst * W) return;
  const int i = e / W, u = e % W;
  double v = 0.0;
  for (int j = 0; j < r; ++j)
    v += (double)w1[(size_t)u * (m + r) + m + j] * ((q[(size_t)i * r + j] - q_prev[(size_t)i * r + j]) * inv_dt);
  seed[e] = (float)v;
}
}  // namespace

// Tangent velocity v = dg/dq . qdot as one forward-mode directional channel (the
// DQ channel machinery with the seed W_1q qdot instead of r columns of W_1q).
cudaError_t launch_tangent_fp32(const crom_ctx* ctx, int n_inst, const double* q, const double* q_prev, double dt,
                                const int* pt_off, const float* x, int n_pts, float* seed, float* out,
                                cudaStream_t s) {
  FwdParams p{};
  p.mode = kModeDecode;
  fill_decoder(p, ctx);
  const int W = p.width;
  jvp_seed_kernel<<<(n_inst * W + 255) / 256, 256, 0, s>>>(p.w1, p.m, p.r, W, q, q_prev, 1.0 / dt, n_inst, seed);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  p.nx = 0;
  p.second = kSecondNone;
  p.nq = 1;
  p.C = ChannelSet{p.nx, p.second, p.nq}.count(p.m);
  const FwdKernel kind = plan_points(ctx, 1, n_pts, p.C, 8, &p.S);
  p.q = q;
  p.off = pt_off;
  p.x = x;
  p.n_pts = n_pts;
  p.n_inst = n_inst;
  p.out = out;
  p.want = CROM_WANT_DQ;
  p.jvp_seed = seed;
  dim3 grid((n_pts + p.S - 1) / p.S, 1);
  return launch_fwd(p, kind, grid, s);
}

cudaError_t launch_decode_fp32(const crom_ctx* ctx, int n_inst, const double* q, const int* pt_off,
                               const float* x, int n_pts, unsigned want, float* out, cudaStream_t s) {
  FwdParams p{};
  p.mode = kModeDecode;
  fill_decoder(p, ctx);
  const int m = p.m;
  p.nx = (want & (CROM_WANT_DX | CROM_WANT_DXX | CROM_WANT_LAP)) ? m : 0;
  p.second = (want & CROM_WANT_DXX) ? kSecondPerK : ((want & CROM_WANT_LAP) ? kSecondLap : kSecondNone);
  p.nq = (want & CROM_WANT_DQ) ? p.r : 0;
  p.C = ChannelSet{p.nx, p.second, p.nq}.count(m);
  const FwdKernel kind = plan_points(ctx, 1, n_pts, p.C, 8, &p.S);
  p.q = q;
  p.off = pt_off;
  p.x = x;
  p.n_pts = n_pts;
  p.n_inst = n_inst;
  p.out = out;
  p.want = want;
  dim3 grid((n_pts + p.S - 1) / p.S, 1);
  return launch_fwd(p, kind, grid, s);
}

cudaError_t launch_recon_fp32(const crom_ctx* ctx, int n_codes, const double* q, int n_pts,
                              const float* x, float* out, cudaStream_t s) {
  FwdParams p{};
  p.mode = kModeRecon;
  fill_decoder(p, ctx);
  p.nx = 0;
  p.second = kSecondNone;
  p.nq = 0;
  p.C = 1;
  const FwdKernel kind = plan_points(ctx, n_codes, n_pts, 1, 32, &p.S);
  p.q = q;
  p.x = x;
  p.n_pts = n_pts;
  p.n_inst = n_codes;
  p.out = out;
  dim3 grid((n_pts + p.S - 1) / p.S, n_codes);
  return launch_fwd(p, kind, grid, s);
}

// Samples per CTA of the FP32 step: enough CTAs to cover the GPU at least twice
// when possible, within the shared-memory budget of the first iteration's channels.
int step_samples_per_cta(const crom_ctx* ctx, int n_inst, int max_samples) {
  const int m = ctx->desc.m, r = ctx->desc.r;
  const int C0 = ChannelSet{m, kSecondLap, r}.count(m);
  int S = 4;
  while (S > 1 && (long long)n_inst * ((max_samples + S - 1) / S) < 2LL * ctx->num_sms) S >>= 1;
  return pick_samples(ctx->desc.width, C0, m, r, S);
}

// Kernel, samples per CTA (S) and per partial row (PS, which bounds the grid and the
// scratch, and fixes the order of the FP64 sums) of the FP32 step.
FwdKernel plan_step(const crom_ctx* ctx, int n_inst, int n_samples, int max_samples, int gn_iters, int* S, int* PS) {
  const int W = ctx->desc.width, m = ctx->desc.m, r = ctx->desc.r;
  const int C0 = ChannelSet{m, kSecondLap, r}.count(m);
  *PS = step_samples_per_cta(ctx, n_inst, max_samples);
  const long long N = (long long)n_inst * max_samples;
  const int gn = gn_iters, C = C0 + (gn - 1) * (r + 2);  // later iterations carry r + 2 channels
  if (tile_pays(ctx, N * C / gn, C0, true, std::min<long long>(N, n_samples) * C / gn, n_inst)) {
    const FwdKernel k = tile_plan(ctx, n_inst, max_samples, C0, S);
    if (k != kFwdGeneral) return k;
  }
  const int hidden = ctx->desc.hidden;
  const bool shallow = (hidden == 1 && r <= 6) || (hidden == 2 && r <= 3 && W <= 96);
  for (*S = N > ctx->num_sms ? 2 : 1; *S >= 1 && (!shallow || max_samples <= 16); --*S)
    if (*S % *PS == 0 && small_fits(W, *S, C0, m, r, ctx->desc.hidden) && small_pays(ctx, N, *S, C0, true)) return kFwdSmall;
  *S = *PS;
  return kFwdGeneral;
}

int step_fp32_max_tiles(const crom_ctx* ctx, int n_inst, int max_samples) {
  const int S = step_samples_per_cta(ctx, n_inst, max_samples);
  const long long t = ((long long)max_samples + S - 1) / S;
  return t > (1LL << 30) ? (1 << 30) : (int)t;
}

cudaError_t launch_step_fp32(crom_ctx* ctx, const crom_step_desc* step, int n_inst, double* q,
                             const float* alpha, const float* vel, const int* s_off,
                             const float* samples, int n_samples, int max_samples, int* status,
                             cudaStream_t s) {
  FwdParams p{};
  p.mode = kModeStep;
  fill_decoder(p, ctx);
  const int m = p.m, r = p.r;
  int S, PS;
  const FwdKernel kind = plan_step(ctx, n_inst, n_samples, max_samples, step->gn_iters, &S, &PS);
  const int max_tiles = (max_samples + PS - 1) / PS;  // partial rows per instance
  const int n_entries = r * (r + 1) / 2 + r;

  // Scratch: partial normal equations, per-instance tickets, per-sample targets.
  // The chains of partial rows go in groups (finish_cta) for few instances of many rows,
  // whose last CTA would be alone with the sums.
  int groups = kind == kFwdSmall && max_tiles > 16 ? kSumGroups : 1;
  cudaError_t e = grow(ctx, &ctx->partials, &ctx->partials_cap, (size_t)n_inst * max_tiles * n_entries);
  if (e == cudaSuccess) e = grow(ctx, &ctx->counters, &ctx->counters_cap, (size_t)n_inst, true);
  if (e == cudaSuccess && groups > 1) {  // the same sums without them
    bool have;
    e = try_grow_kept(ctx, s, &ctx->group_counters, &ctx->group_counters_cap, (size_t)n_inst * groups, true, &have);
    if (!have) groups = 1;
  }
  if (e == cudaSuccess) e = grow(ctx, &ctx->targets, &ctx->targets_cap, (size_t)n_samples);
  if (e == cudaSuccess) e = grow(ctx, &ctx->qbase, &ctx->qbase_cap, (size_t)n_inst * r);
  if (e != cudaSuccess) return e;

  p.S = S;
  p.off = s_off;
  p.x = samples;
  p.n_inst = n_inst;
  p.pde = step->pde;
  p.coef_per_sample = step->coef_per_sample;
  p.dt = step->dt;
  p.alpha = alpha;
  p.vel = vel;
  p.max_samples = max_samples;
  p.qio = q;
  p.status = status;
  p.n_samples = n_samples;
  p.partials = ctx->partials;
  p.max_tiles = max_tiles;
  p.n_entries = n_entries;
  p.counters = ctx->counters;
  p.PS = PS;
  p.groups = groups;
  p.group_counters = ctx->group_counters;
  p.targets = ctx->targets;
  p.qbase = ctx->qbase;
  if (max_tiles > 65535) return cudaErrorInvalidValue;
  dim3 grid(n_inst, (max_samples + S - 1) / S);
  for (int it = 0; it < step->gn_iters; ++it) {
    // Iteration 0: value, dg/dx_k, Laplacian, dg/dq at q_n.  Later iterations:
    // value and dg/dq at q^(k) plus the difference channel h(q^(k)) - h(q_n).
    p.iter = it;
    p.diff = (it == 0) ? 0 : 1;
    p.nx = (it == 0) ? m : 0;
    p.second = (it == 0) ? kSecondLap : kSecondNone;
    p.nq = r;
    p.C = 1 + p.diff + ChannelSet{p.nx, p.second, p.nq}.count(m) - 1;
    e = launch_fwd(p, kind, grid, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace crom

// ---------------------------------------------------------------------------
// FP32 step without any device allocation (crom_step_noalloc).
//
// Some callers cannot allocate device memory at the time they step: a host
// application or framework that owns the device's memory through its own pool
// and forbids direct cudaMalloc/cudaFree by libraries it loads, and
// latency-critical loops where an allocation may synchronise the device.  For them this variant of the FP32 step
// takes its scratch (per-CTA partial normal equations, per-instance tickets,
// per-sample Delta f and per-instance q_n) from one file-scope device array of
// fixed size instead of the context's growable buffers.
//
// The array exists once per device for the life of the process (every GPU that
// loads the library holds its 8 MiB).  All calls on a device share it and it
// keeps the last call's contents: the tickets are cleared with a memset at every
// call; two calls whose kernels overlap on the GPU (different streams, no
// ordering between them) race on it and must not be issued.
namespace crom {
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(8) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kMaxDevices = 64;
void* g_noalloc_ptr[kMaxDevices] = {};
int g_noalloc_ready[kMaxDevices] = {};

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

size_t noalloc_scratch_capacity() { return kNoAllocScratchBytes; }

// Set-up, once per device and with that device current: the host-side name of
// the array is only a stand-in, the kernel needs its device address.
cudaError_t noalloc_scratch_address(int device, void** out) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  if (!g_noalloc_ready[device]) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[device] = ptr;
    g_noalloc_ready[device] = 1;
  }
  *out = g_noalloc_ptr[device];
  return cudaSuccess;
}

cudaError_t launch_step_fp32_noalloc(const crom_ctx* ctx, const crom_step_desc* step, int n_inst, double* q,
                                     const float* alpha, const float* vel, const int* s_off,
                                     const float* samples, int n_samples, int max_samples, int* status,
                                     cudaStream_t s, size_t* need_bytes) {
  FwdParams p{};
  p.mode = kModeStep;
  fill_decoder(p, ctx);
  const int m = p.m, r = p.r;
  int S, PS;
  const FwdKernel kind = plan_step(ctx, n_inst, n_samples, max_samples, step->gn_iters, &S, &PS);
  const int max_tiles = (max_samples + PS - 1) / PS;  // partial rows per instance
  const int n_entries = r * (r + 1) / 2 + r;
  // layout inside the static array
  const size_t off_cnt = 0;
  const size_t off_part = off_cnt + align256((size_t)n_inst * sizeof(int));
  const size_t off_tgt = off_part + align256((size_t)n_inst * max_tiles * n_entries * sizeof(double));
  const size_t off_qb = off_tgt + align256((size_t)n_samples * sizeof(double));
  const size_t total = off_qb + align256((size_t)n_inst * r * sizeof(double));
  *need_bytes = total;
  if (total > kNoAllocScratchBytes || max_tiles > 65535) return cudaErrorInvalidValue;
  void* base = nullptr;
  cudaError_t e = noalloc_scratch_address(ctx->device, &base);
  if (e != cudaSuccess) return e;
  unsigned char* b = static_cast<unsigned char*>(base);
  e = cudaMemsetAsync(b + off_cnt, 0, (size_t)n_inst * sizeof(int), s);
  if (e != cudaSuccess) return e;
  p.S = S;
  p.off = s_off;
  p.x = samples;
  p.n_inst = n_inst;
  p.pde = step->pde;
  p.coef_per_sample = step->coef_per_sample;
  p.dt = step->dt;
  p.alpha = alpha;
  p.vel = vel;
  p.max_samples = max_samples;
  p.qio = q;
  p.status = status;
  p.n_samples = n_samples;
  p.partials = reinterpret_cast<double*>(b + off_part);
  p.max_tiles = max_tiles;
  p.n_entries = n_entries;
  p.counters = reinterpret_cast<int*>(b + off_cnt);
  p.PS = PS;
  p.groups = 1;
  p.targets = reinterpret_cast<double*>(b + off_tgt);
  p.qbase = reinterpret_cast<double*>(b + off_qb);
  dim3 grid(n_inst, (max_samples + S - 1) / S);
  for (int it = 0; it < step->gn_iters; ++it) {
    p.iter = it;
    p.diff = (it == 0) ? 0 : 1;
    p.nx = (it == 0) ? m : 0;
    p.second = (it == 0) ? kSecondLap : kSecondNone;
    p.nq = r;
    p.C = 1 + p.diff + ChannelSet{p.nx, p.second, p.nq}.count(m) - 1;
    e = launch_fwd(p, kind, grid, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace crom
