// Tiled forward-mode evaluation of the FP32 CUDA-core path (included by simt_fp32.cu
// after FwdParams and the activation helpers).  Both kernels form every output of a
// hidden layer exactly as fwd_fp32_kernel does: four partial sums over the quarters of
// K, each one FMA chain in ascending k, added in order; so the three kernels agree bit
// for bit and only their speed differs.
//
//  * fwd_tile_kernel: throughput.  A CTA holds S (a multiple of 4) samples with all
//    their channels; a thread owns 8 units x 4 samples of TQ channels in registers and
//    walks K.  The weights stream through a two-stage cp.async ring, the activations
//    stay in shared memory.  Bound by the FP32 pipe and the issue slots that the
//    activation chain takes from it (FMA pipe 55-66 % busy; the bare product loop
//    reaches 62 of 80 TFLOP/s).  fwd_fp32_kernel, one unit x 16 columns per thread,
//    waits for every weight and reads four activations per FMA group: 16384 points x 13
//    channels, width 128: 2.56 -> 0.83 ms; 8 x 256^2 values, width 256: 18.4 -> 6.8 ms;
//    a SIREN step of 64 instances: 4.7 -> 1.8 ms.
//  * fwd_small_kernel: latency, for problems of too few samples to fill the GPU that
//    way (one instance of a few hundred samples).  One or two samples per CTA, the
//    quarters of K go to different threads, a whole layer of weights is in flight while
//    the one before is used.  A step of 200 samples, width 128: 150 -> 67 us, of which
//    one CTA's reduction and solve take a third.
#pragma once

// ------------------------------------------------------------------ cp.async
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kLeft) : "memory");
}

// Two FP32 values in a register pair (one FMA instruction for both).
typedef unsigned long long f2;
__device__ __forceinline__ f2 dup2(float a) {
  f2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ f2 fma2p(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 add2p(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float lo2(f2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(f2 v) { return __uint_as_float((uint32_t)(v >> 32)); }

// s(z), s'(z), s''(z).
template <bool kSiren>
__device__ __forceinline__ void act3(const FwdParams& p, float z, float& s0, float& s1, float& s2) {
  if (kSiren) siren3(z, p.omega0, s0, s1, s2);
  else elu3(z, s0, s1, s2);
}
template <bool kSiren>
__device__ __forceinline__ float act_value(const FwdParams& p, float z) {
  if (kSiren) return sinf(p.omega0 * z);
  const float em = expm1f(z > 0.f ? 0.f : z);
  return z > 0.f ? z : em;
}
// elu_diff / siren_diff with e = exp(min(a, 0)) at hand; only mixed signs branch.
template <bool kSiren>
__device__ __forceinline__ float act_diff(const FwdParams& p, float a, float d, float e) {
  if (kSiren) return siren_diff(a, d, p.omega0);
  const float b = a - d;
  const bool ap = a > 0.f, an = a <= 0.f, bp = b > 0.f, bn = b <= 0.f;
  float v = -e * expm1f(-d);
  if (ap && bp) v = d;
  if (!(ap && bp) && !(an && bn)) v = elu_diff(a, d);
  return v;
}

// Coordinates, codes and the FP64 layer-1 constants c_u = b_u + W_1q q (rounded once)
// of a CTA whose samples share one code; with several codes (decode) csf is not formed
// and the codes of all samples are in qs.  Ends with a barrier.
struct TileShared {
  double* qs;   // [r], or [S][r] with several codes
  double* dqs;  // [r]: q^(k) - q_n
  float* xs;    // [S][m]
  float* csf;   // [W]
  float* zdf;   // [W]: W_1q (q^(k) - q_n)
  int* code;    // [S]
};
__device__ __forceinline__ bool stage_inputs(const FwdParams& p, const TileShared& t, const double* w1q,
                                             const float* b1, int inst, int first, int ns, bool have_q = false) {
  const int tid = threadIdx.x, NT = blockDim.x, S = p.S, m = p.m, r = p.r, W = p.width;
  for (int i = tid; i < S * m; i += NT) {
    const int s = i / m, k = i % m;
    t.xs[i] = p.x[(size_t)(first + (s < ns ? s : 0)) * m + k];
  }
  bool one = true;
  if (p.mode == kModeDecode) {
    for (int s = tid; s < S; s += NT) t.code[s] = find_instance(p.off, p.n_inst, first + (s < ns ? s : 0));
    __syncthreads();
    one = t.code[0] == t.code[ns - 1];
    const int n = one ? r : S * r;
    for (int i = tid; i < n; i += NT) t.qs[i] = p.q[(size_t)t.code[i / r] * r + i % r];
  } else if (!have_q) {
    const double* q = p.mode == kModeStep ? p.qio + (size_t)inst * r : p.q + (size_t)blockIdx.y * r;
    for (int j = tid; j < r; j += NT) t.qs[j] = q[j];
  }
  if (p.diff && !have_q)
    for (int j = tid; j < r; j += NT) t.dqs[j] = p.qio[(size_t)inst * r + j] - p.qbase[(size_t)inst * r + j];
  __syncthreads();
  // FP64 is a slow pipe on this GPU (2 FMA per clock and SM): one thread per unit, not
  // one per (unit, sample)
  if (one || p.diff) {
    for (int u = tid; u < W; u += NT) {
      double c = (double)b1[u], zd = 0.0;
#pragma unroll 8
      for (int j = 0; j < r; ++j) {
        const double w = w1q[j * W + u];
        c += w * t.qs[j];
        if (p.diff) zd += w * t.dqs[j];
      }
      t.csf[u] = (float)c;
      t.zdf[u] = (float)zd;
    }
    __syncthreads();
  }
  return one;
}
__device__ __forceinline__ float layer1_const(const FwdParams& p, const TileShared& t, bool one, int u, int s) {
  if (one) return t.csf[u];
  double c = (double)p.b1[u];
#pragma unroll 4
  for (int j = 0; j < p.r; ++j) c += p.w1q[j * p.width + u] * t.qs[s * p.r + j];
  return (float)c;
}

// Which samples a CTA owns; false: nothing to do.
__device__ __forceinline__ bool tile_range(const FwdParams& p, int& inst, int& first, int& ns, int& ntiles, int& total) {
  const int S = p.S;
  inst = ntiles = total = 0;
  if (p.mode == kModeStep) {
    inst = blockIdx.x;
    const int t = blockIdx.y;
    const int o0 = __ldg(&p.off[inst]);
    const int msz = __ldg(&p.off[inst + 1]) - o0;
    const int st = p.iter == 0 ? CROM_OK : p.status[inst];
    if (p.iter == 0) {
      if (msz < p.r || msz > p.max_samples || o0 < 0 || o0 + msz > p.n_samples) {
        if (t == 0 && threadIdx.x == 0) p.status[inst] = CROM_ERR_INVALID_ARG;
        return false;
      }
    } else if (st != CROM_OK) {
      return false;
    }
    total = msz;
    ntiles = (msz + S - 1) / S;
    if (t >= ntiles) return false;
    first = o0 + t * S;
    ns = min(S, msz - t * S);
    return true;
  }
  first = blockIdx.x * S;
  ns = min(S, p.n_pts - first);
  return ns > 0;
}

// ------------------------------------------------------------------ the products
// acc += W^T h over kRows values of k for 8 units (4 at w, 4 at w2) x TQ column quads:
// unit pair a, column e of quad t in acc[t][a][e].  kPrefetch loads the next row's
// operands before this row's products (for kernels of one or two warps per scheduler).
template <int TQ, int kRows, bool kPrefetch>
__device__ __forceinline__ void gemm_rows(f2 (&acc)[TQ][4][4], const float* w, const float* w2, int ws,
                                          const float* const (&h)[TQ], int ld) {
  struct Row {
    ulonglong2 a, b;
    float4 h[TQ];
  };
  auto load = [&](int k) {
    Row r;
    r.a = *reinterpret_cast<const ulonglong2*>(w + k * ws);
    r.b = *reinterpret_cast<const ulonglong2*>(w2 + k * ws);
#pragma unroll
    for (int t = 0; t < TQ; ++t) r.h[t] = *reinterpret_cast<const float4*>(h[t] + k * ld);
    return r;
  };
  Row cur = load(0);
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    Row next = cur;
    if (kPrefetch && k + 1 < kRows) next = load(k + 1);
    const f2 wp[4] = {cur.a.x, cur.a.y, cur.b.x, cur.b.y};
#pragma unroll
    for (int t = 0; t < TQ; ++t) {
      const float4 c = cur.h[t];
      const f2 hd[4] = {dup2(c.x), dup2(c.y), dup2(c.z), dup2(c.w)};
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[t][a][e] = fma2p(wp[a], hd[e], acc[t][a][e]);
    }
    if (!kPrefetch && k + 1 < kRows) next = load(k + 1);
    cur = next;
  }
}
// The four columns of unit i (0..7) of a quad's accumulators.
__device__ __forceinline__ float4 unit_row(const f2 (&x)[4][4], int i) {
  const f2(&p)[4] = x[i >> 1];
  return (i & 1) ? make_float4(hi2(p[0]), hi2(p[1]), hi2(p[2]), hi2(p[3]))
                 : make_float4(lo2(p[0]), lo2(p[1]), lo2(p[2]), lo2(p[3]));
}

// ------------------------------------------------------------------ throughput kernel
// Activation chain of 4 samples of one unit, in place: the pre-activations of the value
// channel in z (bias included), of the difference, gradient and second-order channels
// (the "special" ones, before the dg/dq channels) in row[c * S + 0..3].  s1 = s'(z).
template <bool kSiren>
__device__ __forceinline__ void act_quad(const FwdParams& p, const float (&z)[4], float* row, float (&s1)[4]) {
  const int S = p.S;
  float s0[4], s2[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) act3<kSiren>(p, z[i], s0[i], s1[i], s2[i]);
  *reinterpret_cast<float4*>(row) = make_float4(s0[0], s0[1], s0[2], s0[3]);
  float* c = row + S;
  if (p.diff) {
    float4 d = *reinterpret_cast<float4*>(c);
    d.x = act_diff<kSiren>(p, z[0], d.x, s1[0]); d.y = act_diff<kSiren>(p, z[1], d.y, s1[1]);
    d.z = act_diff<kSiren>(p, z[2], d.z, s1[2]); d.w = act_diff<kSiren>(p, z[3], d.w, s1[3]);
    *reinterpret_cast<float4*>(c) = d;
    c += S;
  }
  float4 zx[kMaxM];
  float4 sq = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < kMaxM; ++k) {
    if (k < p.nx) {
      zx[k] = *reinterpret_cast<float4*>(c);
      *reinterpret_cast<float4*>(c) = make_float4(s1[0] * zx[k].x, s1[1] * zx[k].y, s1[2] * zx[k].z, s1[3] * zx[k].w);
      sq.x += zx[k].x * zx[k].x; sq.y += zx[k].y * zx[k].y;
      sq.z += zx[k].z * zx[k].z; sq.w += zx[k].w * zx[k].w;
      c += S;
    }
  }
  if (p.second == kSecondPerK) {
#pragma unroll
    for (int k = 0; k < kMaxM; ++k) {
      if (k < p.m) {
        float4 v = *reinterpret_cast<float4*>(c);
        v.x = s2[0] * zx[k].x * zx[k].x + s1[0] * v.x; v.y = s2[1] * zx[k].y * zx[k].y + s1[1] * v.y;
        v.z = s2[2] * zx[k].z * zx[k].z + s1[2] * v.z; v.w = s2[3] * zx[k].w * zx[k].w + s1[3] * v.w;
        *reinterpret_cast<float4*>(c) = v;
        c += S;
      }
    }
  } else if (p.second == kSecondLap) {
    float4 v = *reinterpret_cast<float4*>(c);
    v.x = s2[0] * sq.x + s1[0] * v.x; v.y = s2[1] * sq.y + s1[1] * v.y;
    v.z = s2[2] * sq.z + s1[2] * v.z; v.w = s2[3] * sq.w + s1[3] * v.w;
    *reinterpret_cast<float4*>(c) = v;
  }
}

constexpr int kTileRows = 8;      // rows of K per ring stage (a quarter of K is a multiple of 8)
constexpr int kRingStride = 256;  // floats per ring row, whatever the width
// Row stride of the activations: an odd number of 16-byte groups, 0 if none holds the columns.
inline int tile_ld(int C, int S) {
  const int n = C * S;
  return n <= 64 ? 68 : n <= 128 ? 132 : 0;
}

// A thread's register tile is 8 units x TQ column quads (4 samples of one channel each):
// shared memory delivers 32 words per clock, so a tile of 8 x 4 TQ costs 8 + 4 TQ clocks
// of loads per 8 TQ clocks of FMA and warp; at TQ = 1 the loads would bind.
template <int TQ, bool kSiren, int LD>
__global__ void __launch_bounds__(256, 4 - TQ) fwd_tile_kernel(FwdParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = p.width, S = p.S, C = p.C, m = p.m, r = p.r, NQ = S >> 2;
  const int tid = threadIdx.x, NT = blockDim.x;
  const int sub = W / 4 / kTileRows;
  const int NP = S * C;

  float* H = reinterpret_cast<float*>(smem_raw);  // [W][LD]: column c * S + s
  float* Ws = H + W * LD;                         // [2][kTileRows][kRingStride]
  float* s1b = Ws + 2 * kTileRows * kRingStride;  // [W][S]
  TileShared ts;
  ts.qs = reinterpret_cast<double*>(s1b + (C > 1 ? W * S : 0));  // [S][r]
  double* rho = ts.qs + S * r;                     // [S]
  double* Amat = rho + S;                          // [r][r + 1]
  ts.dqs = Amat + r * (r + 1);                     // [r]
  ts.xs = reinterpret_cast<float*>(ts.dqs + r);    // [S][m]
  float* outv = ts.xs + S * m;                     // [NP]
  ts.csf = outv + NP;
  ts.zdf = ts.csf + W;
  ts.code = reinterpret_cast<int*>(ts.zdf + W);    // [S]

  int inst, first, ns, ntiles, total;
  if (!tile_range(p, inst, first, ns, ntiles, total)) return;
  // the running sums of the quarters of K wait in tensor memory (lane = thread of the
  // warp's quadrant, 32 TQ columns per thread), which nothing else here uses: a second
  // set of 32 TQ registers would halve the warps per SM
  __shared__ uint32_t s_tmem;
  constexpr uint32_t kCols = TQ == 3 ? 256 : 64 * TQ;  // two warpgroups
  if (tid < 32) {
    tc::tmem_alloc(&s_tmem, kCols);
    tc::tmem_relinquish();
  }

  // weight ring: chunk g = rows g * kTileRows .. of the stacked hidden matrices
  const int per_layer = 4 * sub, chunks = (p.hidden - 1) * per_layer, W4 = W >> 2;
  auto fetch = [&](int g) {
    const float* src = p.wt + (size_t)g * kTileRows * W;
    float* dst = Ws + (g & 1) * (kTileRows * kRingStride);
    int row = tid / W4, c = tid - row * W4;
    while (row < kTileRows) {
      cp_async16(dst + row * kRingStride + 4 * c, src + row * W + 4 * c);
      for (c += NT; c >= W4; c -= W4) ++row;
    }
  };
  if (chunks > 0) fetch(0);
  cp_async_commit();

  const bool one = stage_inputs(p, ts, p.w1q, p.b1, inst, first, ns);
  const int ox = 1 + p.diff, n2 = (p.second == kSecondPerK) ? m : (p.second == kSecondLap ? 1 : 0);
  const int o2 = ox + p.nx, oq = o2 + n2;
  const bool value_only = C == 1;

  // ---- layer 1: a thread forms one unit for every (NT / W)-th sample quad
  const int qstep = max(1, NT / W);
  for (int u = tid; u < W * qstep; u += NT) {
    const int uu = u % W;
    float wx[kMaxM];
#pragma unroll
    for (int k = 0; k < kMaxM; ++k) wx[k] = k < m ? p.w1t[k * W + uu] : 0.f;
    for (int sq = u / W; sq < NQ; sq += qstep) {
      float* row = H + uu * LD + 4 * sq;
      float z[4], s1[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int s = 4 * sq + e;
        z[e] = layer1_const(p, ts, one, uu, s);
#pragma unroll
        for (int k = 0; k < kMaxM; ++k)
          if (k < m) z[e] = fmaf(wx[k], ts.xs[s * m + k], z[e]);
      }
      if (value_only) {
        *reinterpret_cast<float4*>(row) = make_float4(act_value<kSiren>(p, z[0]), act_value<kSiren>(p, z[1]),
                                                      act_value<kSiren>(p, z[2]), act_value<kSiren>(p, z[3]));
        continue;
      }
      auto fill = [&](int c, float v) { *reinterpret_cast<float4*>(row + c * S) = make_float4(v, v, v, v); };
      if (p.diff) fill(1, ts.zdf[uu]);
#pragma unroll
      for (int k = 0; k < kMaxM; ++k)
        if (k < p.nx) fill(ox + k, wx[k]);
      for (int k = 0; k < n2; ++k) fill(o2 + k, 0.f);
      act_quad<kSiren>(p, z, row, s1);
      if (p.jvp_seed) {
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = __ldg(&p.jvp_seed[(size_t)ts.code[4 * sq + e] * W + uu]) * s1[e];
        *reinterpret_cast<float4*>(row + oq * S) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll 8
        for (int j = 0; j < p.nq; ++j) {
          const float w = p.w1t[(m + j) * W + uu];
          *reinterpret_cast<float4*>(row + (oq + j) * S) = make_float4(w * s1[0], w * s1[1], w * s1[2], w * s1[3]);
        }
      }
    }
  }

  // ---- hidden layers 2..hidden: this thread's units 4 ug + 0..3 and W/2 + 4 ug + 0..3,
  // column quads ng, ng + GN, .. (quad c * NQ + sq = samples 4 sq.. of channel c)
  const int quads = C * NQ, GN = (quads + TQ - 1) / TQ;
  const int ng = (tid >> 2) % GN, ug = (tid >> 2) / GN * 4 + (tid & 3);
  const bool active = ug < W / 8;
  const int u0 = active ? 4 * ug : 0;
  auto unit = [&](int i) { return u0 + (i & 3) + (i < 4 ? 0 : W / 2); };
  int col[TQ], chan[TQ];  // first column; channel, or C where the quad is past the end
#pragma unroll
  for (int t = 0; t < TQ; ++t) {
    const int qd = ng + t * GN;
    chan[t] = active && qd < quads ? qd / NQ : C;
    col[t] = 4 * min(qd, quads - 1);
  }

  // (stage_inputs' barriers published the allocation)
  const uint32_t tm = s_tmem + ((uint32_t)(tid >> 5 & 3) << 21) + (uint32_t)(tid >> 7) * (32 * TQ);
  f2 acc[TQ][4][4];  // [quad][unit pair][sample]
  // chunk ch (16 values) of the accumulators: quad ch / 2, unit pairs 2 (ch & 1) ..
  auto save = [&](int ch) {
    float x[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[2 * i] = lo2(acc[ch >> 1][2 * (ch & 1) + (i >> 2)][i & 3]);
      x[2 * i + 1] = hi2(acc[ch >> 1][2 * (ch & 1) + (i >> 2)][i & 3]);
    }
    tc::tmem_st16(tm + 16 * ch, x);
  };
  auto add_saved = [&](int ch) {
    float x[16];
    tc::tmem_ld16(tm + 16 * ch, x);
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]), "+f"(x[4]), "+f"(x[5]), "+f"(x[6]), "+f"(x[7]),
                   "+f"(x[8]), "+f"(x[9]), "+f"(x[10]), "+f"(x[11]), "+f"(x[12]), "+f"(x[13]), "+f"(x[14]),
                   "+f"(x[15])
                 :
                 : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      f2& a = acc[ch >> 1][2 * (ch & 1) + (i >> 2)][i & 3];
      a = add2p(tc::pk2(x[2 * i], x[2 * i + 1]), a);
    }
  };
  for (int l = 0; l < p.hidden - 1; ++l) {
    for (int quarter = 0; quarter < 4; ++quarter) {
#pragma unroll
      for (int t = 0; t < TQ; ++t)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[t][a][e] = 0ull;
      for (int part = 0; part < sub; ++part) {
        const int g = l * per_layer + quarter * sub + part;
        cp_async_wait<0>();
        __syncthreads();  // chunk g has landed; chunk g - 1's stage and the activations' writers are done
        if (g + 1 < chunks) fetch(g + 1);
        cp_async_commit();
        const float* hrow = H + (quarter * sub + part) * kTileRows * LD;
        const float* hq[TQ];
#pragma unroll
        for (int t = 0; t < TQ; ++t) hq[t] = hrow + col[t];
        const float* w = Ws + (g & 1) * (kTileRows * kRingStride) + u0;
        gemm_rows<TQ, kTileRows, false>(acc, w, w + W / 2, kRingStride, hq, LD);
      }
      // v = ((p_0 + p_1) + p_2) + p_3: v in tensor memory, after the last quarter in acc
      if (quarter > 0) {
        tc::tmem_st_wait();
#pragma unroll
        for (int ch = 0; ch < 2 * TQ; ++ch) add_saved(ch);
      }
      if (quarter < 3) {
#pragma unroll
        for (int ch = 0; ch < 2 * TQ; ++ch) save(ch);
      }
    }
    __syncthreads();  // every read of H is done
    const float* bias = p.bh + (size_t)l * W;
    auto pre = [&](int t, int i) { return unit_row(acc[t], i); };
    if (value_only) {
#pragma unroll
      for (int t = 0; t < TQ; ++t) {
        if (chan[t] < C) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float b = __ldg(bias + unit(i));
            const float4 z = pre(t, i);
            *reinterpret_cast<float4*>(H + unit(i) * LD + col[t]) =
                make_float4(act_value<kSiren>(p, z.x + b), act_value<kSiren>(p, z.y + b),
                            act_value<kSiren>(p, z.z + b), act_value<kSiren>(p, z.w + b));
          }
        }
      }
      continue;  // the next barrier (next chunk or the output layer's) orders these writes
    }
    // the special channels' pre-activations through shared memory: their chain couples them
#pragma unroll
    for (int t = 0; t < TQ; ++t)
      if (chan[t] < oq) {
#pragma unroll
        for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(H + unit(i) * LD + col[t]) = pre(t, i);
      }
    __syncthreads();
    for (int i = tid; i < W * NQ; i += NT) {
      const int u = i % W, q4 = i / W;
      float* row = H + u * LD + 4 * q4;
      const float b = __ldg(bias + u);
      const float4 zv = *reinterpret_cast<const float4*>(row);
      const float z[4] = {zv.x + b, zv.y + b, zv.z + b, zv.w + b};
      float s1[4];
      act_quad<kSiren>(p, z, row, s1);
      *reinterpret_cast<float4*>(s1b + u * S + 4 * q4) = make_float4(s1[0], s1[1], s1[2], s1[3]);
    }
    if (p.nq == 0) continue;
    __syncthreads();
    // dg/dq channels: times s'(z), from registers
#pragma unroll
    for (int t = 0; t < TQ; ++t)
      if (chan[t] >= oq && chan[t] < C) {
        const int s = col[t] - chan[t] * S;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 s1 = *reinterpret_cast<const float4*>(s1b + unit(i) * S + s);
          const float4 a = pre(t, i);
          *reinterpret_cast<float4*>(H + unit(i) * LD + col[t]) =
              make_float4(a.x * s1.x, a.y * s1.y, a.z * s1.z, a.w * s1.w);
        }
      }
  }
  __syncthreads();
  if (tid < 32) tc::tmem_dealloc(s_tmem, kCols);
  output_layer(p, p.wout, H, LD, NP, outv, S);
  __syncthreads();
  finish_cta<20>(p, outv, 1, S, inst, first, ns, ntiles, total, rho, Amat, ts.qs, reinterpret_cast<double*>(H));
}

inline size_t tile_smem_bytes(int W, int S, int C, int m, int r) {
  size_t b = (size_t)W * tile_ld(C, S) * 4 + 2u * kTileRows * kRingStride * 4 + (C > 1 ? (size_t)W * S * 4 : 0);
  b += ((size_t)S * r + S + (size_t)r * (r + 1) + r) * 8;
  b += ((size_t)S * m + (size_t)S * C + 2u * W + S) * 4;
  return b + 16;
}
inline int tile_threads(int W, int S, int C, int tq) {
  return (W / 8 * ((C * S / 4 + tq - 1) / tq) + 31) / 32 * 32;
}

// ------------------------------------------------------------------ latency kernel
constexpr int kSmallLD = 36;  // row stride of the activations (at most 32 columns)
// Rows of every quarter of K per ring stage (two stages within 128 KB): the whole
// quarter up to width 128.
__host__ __device__ constexpr int small_rows(int W) { return W <= 128 ? W / 4 : W / 16; }
constexpr int kSmallThreads = 512;

// Everything the CTA will need from global memory is requested up front (first layer,
// biases, output row, the first two weight stages), so that one memory latency is paid, not
// one per layer.  kW: the width, 0 = any (p.width).
template <int kW>
__global__ void __launch_bounds__(kSmallThreads, 1) fwd_small_kernel(FwdParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = kW ? kW : p.width, quarter = W / 4, kRS = kW ? small_rows(kW) : small_rows(W);
  constexpr int LD = kSmallLD, TQ = 1;
  const int S = p.S, C = p.C, m = p.m, r = p.r, kin = m + r;
  const int tid = threadIdx.x, NT = blockDim.x;
  const int NP = S * C, quads = (NP + 3) / 4, NPP = 4 * quads;

  float* H = reinterpret_cast<float*>(smem_raw);             // [W][LD]: column s * C + c
  float* Ws = H + W * LD;                                    // [2][4][kRS][W]
  float* red = Ws + 2 * 4 * kRS * W;                         // [4][NPP][W]: the quarters' partial sums
  double* wqs = reinterpret_cast<double*>(red + (size_t)4 * NPP * W);  // [r][W]
  float* w1s = reinterpret_cast<float*>(wqs + r * W);        // [kin][W]
  float* b1s = w1s + W * kin;                                // [W]
  float* bhs = b1s + W;                                      // [hidden - 1][W]
  float* wos = bhs + (p.hidden - 1) * W;                     // [W]
  TileShared ts;
  ts.qs = reinterpret_cast<double*>(wos + W);
  double* rho = ts.qs + S * r;
  double* Amat = rho + S;
  ts.dqs = Amat + r * (r + 1);
  ts.xs = reinterpret_cast<float*>(ts.dqs + r);
  float* outv = ts.xs + S * m;
  ts.csf = outv + NPP;
  ts.zdf = ts.csf + W;
  ts.code = reinterpret_cast<int*>(ts.zdf + W);

  auto copy = [&](float* dst, const float* src, int n) {
    for (int i = tid * 4; i < n; i += NT * 4) cp_async16(dst + i, src + i);
  };
  copy(reinterpret_cast<float*>(wqs), reinterpret_cast<const float*>(p.w1q), 2 * r * W);
  copy(w1s, p.w1t, W * kin);
  copy(b1s, p.b1, W);
  copy(bhs, p.bh, (p.hidden - 1) * W);
  copy(wos, p.wout, W);
  cp_async_commit();
  // threads that take part in the products come first; the others fetch the weights
  const int GN = (quads + TQ - 1) / TQ, gemm_threads = (W / 8 * GN * 4 + 31) / 32 * 32;
  const int f0 = gemm_threads < NT ? gemm_threads : 0, fn = NT - f0;
  const int per_layer = quarter / kRS, qfloats = kRS * W, stage_floats = 4 * qfloats;
  const int stages = (p.hidden - 1) * per_layer;
  auto fetch = [&](int g, int t0, int n) {  // rows j0.. of every quarter of K, by threads t0 .. t0 + n - 1
    if (tid < t0) return;
    const int l = g / per_layer, j0 = (g % per_layer) * kRS;
    float* dst = Ws + (g & 1) * stage_floats;
    const float* src = p.wt + (size_t)l * W * W + (size_t)j0 * W;
    for (int i = (tid - t0) * 4; i < qfloats; i += n * 4)
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) cp_async16(dst + ks * qfloats + i, src + (size_t)ks * quarter * W + i);
  };
  if (stages > 0) fetch(0, 0, NT);
  cp_async_commit();
  if (stages > 1) fetch(1, 0, NT);
  cp_async_commit();
  // A step's launches overlap: up to here a CTA reads the decoder alone, while the last
  // CTA of the launch before may still add and solve (a third of its time, on one SM).
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const bool step = p.mode == kModeStep && tid < r;  // its codes come along with its range
  const double qk = step ? p.qio[(size_t)blockIdx.x * r + tid] : 0.0;
  const double qn = step && p.diff ? p.qbase[(size_t)blockIdx.x * r + tid] : 0.0;
  int inst, first, ns, ntiles, total;
  if (!tile_range(p, inst, first, ns, ntiles, total)) {
    cp_async_wait<0>();
    return;
  }
  if (step) {
    ts.qs[tid] = qk;
    ts.dqs[tid] = qk - qn;
  }
  if (NP < NPP)
    for (int u = tid; u < W; u += NT)
      for (int c = NP; c < NPP; ++c) H[u * LD + c] = 0.f;  // padding columns
  cp_async_wait<2>();  // the first-layer group; stage_inputs has a barrier before its first use
  const bool one = stage_inputs(p, ts, wqs, b1s, inst, first, ns, p.mode == kModeStep);
  const int ox = 1 + p.diff, n2 = (p.second == kSecondPerK) ? m : (p.second == kSecondLap ? 1 : 0);
  const int o2 = ox + p.nx, oq = o2 + n2;
  // activation items (unit, sample, part): part 0 the special channels, the others a
  // share of the dg/dq channels each (every part forms s'(z) itself)
  const int parts = p.nq > 0 ? max(1, min(4, NT / (W * S))) : 1;
  auto chain = [&](int u, int s, int part, float z, auto pre) {
    float* c = H + u * LD + s * C;
    float s0, s1, s2;
    const bool siren = p.act == CROM_ACT_SIREN;
    if (siren) act3<true>(p, z, s0, s1, s2);
    else act3<false>(p, z, s0, s1, s2);
    if (part == 0) {
      c[0] = s0;
      if (p.diff) c[1] = siren ? act_diff<true>(p, z, pre(1), s1) : act_diff<false>(p, z, pre(1), s1);
      float zx[kMaxM], sq = 0.f;
#pragma unroll
      for (int k = 0; k < kMaxM; ++k)
        if (k < p.nx) {
          zx[k] = pre(ox + k);
          c[ox + k] = s1 * zx[k];
          sq += zx[k] * zx[k];
        }
      if (p.second == kSecondPerK) {
#pragma unroll
        for (int k = 0; k < kMaxM; ++k)
          if (k < m) c[o2 + k] = s2 * zx[k] * zx[k] + s1 * pre(o2 + k);
      } else if (p.second == kSecondLap) {
        c[o2] = s2 * sq + s1 * pre(o2);
      }
    }
    const int step = parts > 1 ? parts - 1 : 1;
    if (parts == 1 || part > 0) {
#pragma unroll 4
      for (int j = parts > 1 ? part - 1 : 0; j < p.nq; j += step) c[oq + j] = pre(oq + j) * s1;
    }
  };
  // ---- layer 1
  for (int i = tid; i < W * S * parts; i += NT) {
    const int u = i % W, s = (i / W) % S, part = i / (W * S);
    const float* w1 = w1s + u;  // entry k at w1[k * W]
    float z = layer1_const(p, ts, one, u, s);
    for (int k = 0; k < m; ++k) z = fmaf(w1[k * W], ts.xs[s * m + k], z);
    chain(u, s, part, z, [&](int c) {
      if (c >= oq) return p.jvp_seed ? __ldg(&p.jvp_seed[(size_t)ts.code[s] * W + u]) : w1[(m + c - oq) * W];
      if (c >= o2) return 0.f;
      return c >= ox ? w1[(c - ox) * W] : ts.zdf[u];
    });
  }

  // ---- hidden layers: thread (unit group, column group, quarter of K)
  const int ng = (tid >> 2) % GN, hi = (tid >> 2) / GN;
  const int ug = hi % (W / 32) * 4 + (tid & 3), ks = hi / (W / 32);
  const bool active = ks < 4;
  const int u0 = 4 * ug;
  int col[TQ];
#pragma unroll
  for (int t = 0; t < TQ; ++t) col[t] = 4 * min(ng + t * GN, quads - 1);
  for (int l = 0; l < p.hidden - 1; ++l) {
    f2 acc[TQ][4][4];
#pragma unroll
    for (int t = 0; t < TQ; ++t)
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][a][e] = 0ull;
    for (int st = 0; st < per_layer; ++st) {
      const int g = l * per_layer + st;
      if (g == 0) cp_async_wait<1>();
      else cp_async_wait<0>();
      __syncthreads();
      if (g > 0 && g + 1 < stages) fetch(g + 1, f0, fn);
      cp_async_commit();
      if (active) {
        const float* w = Ws + (g & 1) * stage_floats + ks * qfloats + u0;
        const float* hq[TQ];
#pragma unroll
        for (int t = 0; t < TQ; ++t) hq[t] = H + (ks * quarter + st * kRS) * LD + col[t];
        constexpr int kStep = kW ? 8 : 2;  // kRS is a multiple
#pragma unroll 1
        for (int k = 0; k < kRS; k += kStep) {
          gemm_rows<TQ, kStep, true>(acc, w, w + W / 2, W, hq, LD);
          w += kStep * W;
#pragma unroll
          for (int t = 0; t < TQ; ++t) hq[t] += kStep * LD;
        }
      }
    }
    if (active) {
#pragma unroll
      for (int t = 0; t < TQ; ++t)
        if (ng + t * GN < quads) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float* o = red + ((size_t)ks * NPP + col[t] + e) * W + u0;
            *reinterpret_cast<ulonglong2*>(o) = make_ulonglong2(acc[t][0][e], acc[t][1][e]);
            *reinterpret_cast<ulonglong2*>(o + W / 2) = make_ulonglong2(acc[t][2][e], acc[t][3][e]);
          }
        }
    }
    __syncthreads();
    const float* bias = bhs + l * W;
    const int kst = NPP * W;
    for (int i = tid; i < W * S * parts; i += NT) {
      const int u = i % W, s = (i / W) % S, part = i / (W * S);
      const float* base = red + s * C * W + u;
      auto pre = [&](int c) {
        const float* x = base + c * W;
        return ((0.f + x[0]) + x[kst]) + x[2 * kst] + x[3 * kst];
      };
      chain(u, s, part, pre(0) + bias[u], pre);
    }
  }
  __syncthreads();
  output_layer(p, wos, H, LD, NP, outv, 0);
  __syncthreads();
  finish_cta<20>(p, outv, C, 1, inst, first, ns, ntiles, total, rho, Amat, ts.qs, reinterpret_cast<double*>(red));
}

inline size_t small_smem_bytes(int W, int S, int C, int m, int r, int hidden) {
  const size_t npp = (S * C + 3) / 4 * 4;
  size_t b = (size_t)W * kSmallLD * 4 + 2u * 4 * small_rows(W) * W * 4 + 4 * npp * W * 4;
  b += (size_t)W * (m + 3 * r + hidden + 1) * 4;
  b += ((size_t)S * r + S + (size_t)r * (r + 1) + r) * 8;
  b += ((size_t)S * m + npp + 2u * W + S) * 4;
  return b + 16;
}
inline int small_gemm_threads(int W, int S, int C) {
  return (W / 8 * ((S * C + 3) / 4) * 4 + 31) / 32 * 32;
}
