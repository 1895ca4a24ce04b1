// Full-order models, all time steps of a call in one launch (see fom.cu for the
// schemes): a field stays on the chip from its load to its store, so that a call moves
// each field once, not once per step, and pays one launch.
//
//  * fom_tile_kernel (2D, sides that are multiples of 4, up to 256): a cluster of NC
//    CTAs per field, each a band of rows; a thread owns RT rows x 4 columns in registers
//    together with its face velocities or coefficients.  Per step the threads publish
//    the rims of their tiles in shared memory (the rows at a band's border in the
//    neighbouring CTA's shared memory), meet once at the cluster barrier, and update.
//    Bound by the FP32 pipe for many fields (17 operations a node for advection,
//    6 for heat, where the step-by-step kernels move 16 and 8 bytes a node through HBM
//    or L2), by the barrier's latency for few.
//    8 fields of 128^2, heat, 100 steps: 410 -> 53 us; 400 of 200^2, 20 steps: 1230 -> 408.
//  * fom_wide_kernel: the same for many fields of sides 128 and 256.  64 fields of 256^2,
//    advection-diffusion, 10 steps: 84 -> 48 us with the velocities in L2 from the call
//    before (96 -> 54 without; 512 fields: 784 -> 379; 1024 fields of 128^2, heat: 203 -> 60).
//  * fom_line_kernel (1D) and fom_field_kernel (2D, other sides up to kFieldMaxHeat and
//    kFieldMaxAdv): one CTA per field, the field twice in shared memory, one barrier per
//    step (100 steps of 256 nodes: 409 -> 14 us; 10 steps of 97^2, heat: 41 -> 24 us).
#include <algorithm>
#include <atomic>

#include "crom_internal.h"

namespace crom {
namespace {

enum Scheme { kHeat = 0, kHeatField = 1, kUpwind = 2, kCentral = 3 };

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16-byte store into the shared memory of cluster CTA `rank`, at this CTA's address p.
__device__ __forceinline__ void store_peer(float4* p, uint32_t rank, float4 v) {
  asm volatile(
      "{\n\t.reg .b32 a;\n\t"
      "mapa.shared::cluster.u32 a, %0, %1;\n\t"
      "st.shared::cluster.v4.f32 [a], {%2, %3, %4, %5};\n\t}" ::"r"(smem_addr(p)),
      "r"(rank), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
      : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// What crosses the face between the cells c (left, upper) and cn (right, lower) in one
// step, counted into c: heat: the difference cn - c (the coefficient follows at the
// node); advection-diffusion: K (cn - c) - A f with K = dt nu / h^2, A = dt a / h (half
// of it for the central mean) and f the upwind cell or the sum of the two.
template <int kScheme>
__device__ __forceinline__ float through(float A, float K, float c, float cn) {
  const float d = cn - c;
  if (kScheme <= kHeatField) return d;
  return fmaf(-A, kScheme == kCentral ? c + cn : (A > 0.f ? c : cn), K * d);
}

template <bool kCen>
__device__ __forceinline__ float flux(float a, float left, float right) {
  return kCen ? a * (0.5f * (left + right)) : a * (a > 0.f ? left : right);
}

struct FomParams {
  float* u;
  const float *ax, *ay, *coef;
  int n, steps, NC;
  float dt, inv_h, inv_h2;  // heat: dt = dt / h^2
};

constexpr int kTileThreads = 512;

template <int kScheme, int RT>
__global__ void __launch_bounds__(kTileThreads, 1) fom_tile_kernel(FomParams p) {
  constexpr bool kAdv = kScheme >= kUpwind, kPeriodic = kAdv;
  extern __shared__ float4 smem4[];
  const int n = p.n, NX = n >> 2, TR = n / RT, NC = p.NC;
  const int rank = blockIdx.x, tid = threadIdx.x;
  const int t0 = rank * TR / NC, t1 = (rank + 1) * TR / NC, rows = t1 - t0;  // this CTA's tile rows
  const int cap = (TR + NC - 1) / NC;
  // rims, by step parity: top and bottom rows, left and right columns of the tiles, and
  // the neighbouring bands' border rows
  float4* top = smem4;                   // [2][cap][NX]
  float4* bot = top + 2 * cap * NX;      // [2][cap][NX]
  float4* above = bot + 2 * cap * NX;    // [2][NX]: last row of the band above
  float4* below = above + 2 * NX;        // [2][NX]: first row of the band below
  float* lef = reinterpret_cast<float*>(below + 2 * NX);  // [2][cap][RT][NX]
  float* rig = lef + 2 * cap * RT * NX;                   // [2][cap][RT][NX]
  const int tx = tid % NX, ty = tid / NX;
  const bool active = ty < rows;
  const size_t base = (size_t)blockIdx.y * n * n;
  const int i0 = (t0 + ty) * RT, j0 = 4 * tx;
  const uint32_t up_rank = rank > 0 ? rank - 1 : NC - 1, dn_rank = rank + 1 < NC ? rank + 1 : 0;
  const bool first = t0 + ty == 0, last = t0 + ty == TR - 1;  // tile rows at the field's border
  const int txl = tx > 0 ? tx - 1 : NX - 1, txr = tx + 1 < NX ? tx + 1 : 0;

  float c[RT][4], a[RT + 1][4], b[RT][5], nu[RT][4];
  const float nu0 = kScheme == kHeatField ? 0.f : p.coef[blockIdx.y];
  // per node: heat r = dt / h^2 nu; advection K = dt nu / h^2, face coefficients dt a / h
  const float K = kAdv ? (float)((double)p.dt * (double)nu0 * (double)p.inv_h2) : p.dt * nu0;
  const float fa = (kScheme == kCentral ? 0.5f : 1.f) * (p.dt * p.inv_h);
  auto load4 = [&](const float* f, int i, float* v, float scale) {
    const float4 x = *reinterpret_cast<const float4*>(f + base + (size_t)i * n + j0);
    v[0] = scale * x.x; v[1] = scale * x.y; v[2] = scale * x.z; v[3] = scale * x.w;
  };
  if (active) {
#pragma unroll
    for (int k = 0; k < RT; ++k) {
      load4(p.u, i0 + k, c[k], 1.f);
      if (kAdv) {
        load4(p.ax, i0 + k, a[k + 1], fa);  // faces (i + 1/2, j)
        load4(p.ay, i0 + k, b[k] + 1, fa);  // faces (i, j + 1/2)
        b[k][0] = fa * p.ay[base + (size_t)(i0 + k) * n + (j0 > 0 ? j0 - 1 : n - 1)];
      }
      if (kScheme == kHeatField) load4(p.coef, i0 + k, nu[k], p.dt);
    }
    if (kAdv) load4(p.ax, i0 > 0 ? i0 - 1 : n - 1, a[0], fa);
  }
  if (NC > 1) {  // every CTA of the cluster runs before its memory is written
    cluster_arrive();
    cluster_wait();
  }

  for (int s = 0; s < p.steps; ++s) {
    const int par = s & 1;
    float4* tp = top + par * cap * NX;
    float4* bp = bot + par * cap * NX;
    float* lp = lef + par * cap * RT * NX;
    float* rp = rig + par * cap * RT * NX;
    if (active) {
      const float4 ct = make_float4(c[0][0], c[0][1], c[0][2], c[0][3]);
      const float4 cb = make_float4(c[RT - 1][0], c[RT - 1][1], c[RT - 1][2], c[RT - 1][3]);
      tp[ty * NX + tx] = ct;
      bp[ty * NX + tx] = cb;
#pragma unroll
      for (int k = 0; k < RT; ++k) {
        lp[(ty * RT + k) * NX + tx] = c[k][0];
        rp[(ty * RT + k) * NX + tx] = c[k][3];
      }
      if (ty == 0 && (kPeriodic || !first)) {
        if (NC > 1) store_peer(below + par * NX + tx, up_rank, ct);
        else below[par * NX + tx] = ct;
      }
      if (ty == rows - 1 && (kPeriodic || !last)) {
        if (NC > 1) store_peer(above + par * NX + tx, dn_rank, cb);
        else above[par * NX + tx] = cb;
      }
    }
    if (NC > 1) cluster_arrive();
    // while the rims travel: the faces inside the tile
    float o[RT][4];
#pragma unroll
    for (int k = 0; k < RT; ++k) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float t = through<kScheme>(b[k][q + 1], K, c[k][q], c[k][q + 1]);
        o[k][q] = q == 0 ? t : o[k][q] + t;
        o[k][q + 1] = -t;
      }
    }
#pragma unroll
    for (int k = 0; k + 1 < RT; ++k) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float t = through<kScheme>(a[k + 1][q], K, c[k][q], c[k + 1 < RT ? k + 1 : k][q]);
        o[k][q] += t;
        o[k + 1 < RT ? k + 1 : k][q] -= t;
      }
    }
    if (NC > 1) cluster_wait();
    else __syncthreads();
    if (active) {
      float up[4], dn[4];
      {
        const float4 x = ty > 0 ? bp[(ty - 1) * NX + tx] : above[par * NX + tx];
        const float4 y = ty + 1 < rows ? tp[(ty + 1) * NX + tx] : below[par * NX + tx];
        up[0] = x.x; up[1] = x.y; up[2] = x.z; up[3] = x.w;
        dn[0] = y.x; dn[1] = y.y; dn[2] = y.z; dn[3] = y.w;
      }
      if (!kPeriodic) {  // mirror ghosts: u_{-1} = u_1, u_n = u_{n-2}
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float second = RT > 1 ? c[RT > 1 ? 1 : 0][q] : dn[q], before = RT > 1 ? c[RT > 1 ? RT - 2 : 0][q] : up[q];
          if (first) up[q] = second;
          if (last) dn[q] = before;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        o[0][q] -= through<kScheme>(a[0][q], K, up[q], c[0][q]);
        o[RT - 1][q] += through<kScheme>(a[RT][q], K, c[RT - 1][q], dn[q]);
      }
#pragma unroll
      for (int k = 0; k < RT; ++k) {
        float l = rp[(ty * RT + k) * NX + txl], r = lp[(ty * RT + k) * NX + txr];
        if (!kPeriodic) {
          if (tx == 0) l = c[k][1];
          if (tx == NX - 1) r = c[k][2];
        }
        o[k][0] -= through<kScheme>(b[k][0], K, l, c[k][0]);
        o[k][3] += through<kScheme>(b[k][4], K, c[k][3], r);
      }
#pragma unroll
      for (int k = 0; k < RT; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          c[k][q] = kAdv ? c[k][q] + o[k][q] : fmaf(kScheme == kHeatField ? nu[k][q] : K, o[k][q], c[k][q]);
    }
  }
  if (active) {
#pragma unroll
    for (int k = 0; k < RT; ++k)
      *reinterpret_cast<float4*>(p.u + base + (size_t)(i0 + k) * n + j0) =
          make_float4(c[k][0], c[k][1], c[k][2], c[k][3]);
  }
}

inline size_t tile_bytes(int n, int RT, int NC) {
  const size_t nx = n / 4, cap = (n / RT + NC - 1) / NC;
  return (4 * cap * nx + 4 * nx) * 16 + 4 * cap * RT * nx * 4;
}
inline int tile_thr(int n, int RT, int NC) { return (n / 4 * ((n / RT + NC - 1) / NC) + 31) / 32 * 32; }

// The same for many fields of sides 128 and 256: 1024 threads per CTA (64 registers), so
// that a field takes a quarter of the CTAs and clusters of four pack onto the GPU (of the
// eight-CTA clusters about twelve run at a time: 64 fields of 256^2 took 70 us).  Those two
// sides alone: a row is then one or two whole warps, which the lane exchange needs, and
// the CTA's 1024 threads divide into rows.  Other sides stay with fom_tile_kernel, 0.32 to
// 0.59 of a launch per step's time where the GPU is full (400 fields of 200^2, five steps:
// heat 138 against 329 us, advection 192 against 388; 300 of 252^2, ten: 213 against 676
// and 292 against 800; 800 of 180^2, upwind, ten: 663 against 1127).  The
// face velocities (or the coefficient field) lie in shared memory; column neighbours and
// the fluxes through the tiles' sides come from the adjacent lanes, what crosses the two
// warps of a 256-node row and the rows at the tiles' borders through shared memory.
constexpr int kWideThreads = 1024, kWideRT = 4;

template <int kScheme, int NX>
__global__ void __launch_bounds__(kWideThreads, 1) fom_wide_kernel(FomParams p) {
  constexpr bool kAdv = kScheme >= kUpwind, kPeriodic = kAdv;
  constexpr int n = 4 * NX, RT = kWideRT, rows = kWideThreads / NX, NC = n / RT / rows;
  extern __shared__ float4 smem4[];
  float4* top = smem4;                 // [2][rows][NX]
  float4* bot = top + 2 * rows * NX;   // [2][rows][NX]
  float4* above = bot + 2 * rows * NX;  // [2][NX]
  float4* below = above + 2 * NX;       // [2][NX]
  float4* av = below + 2 * NX;          // advection: [RT rows + 1][NX] x-face coefficients; field: nu
  float4* bv = av + (kAdv ? RT * rows + 1 : kScheme == kHeatField ? RT * rows : 0) * NX;  // [RT rows][NX]
  float2* rim = reinterpret_cast<float2*>(bv + (kAdv ? RT * rows * NX : 0));  // [2][RT rows][2]: a warp's end columns
  const int rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int tx = tid % NX, ty = tid / NX, wx = tx >> 5;
  const size_t base = (size_t)blockIdx.y * n * n;
  const int band = rank * rows * RT, i0 = band + ty * RT, j0 = 4 * tx;
  const uint32_t up_rank = rank > 0 ? rank - 1 : NC - 1, dn_rank = rank + 1 < NC ? rank + 1 : 0;
  const bool first = rank == 0 && ty == 0, last = rank == NC - 1 && ty == rows - 1;
  const float nu0 = kScheme == kHeatField ? 0.f : p.coef[blockIdx.y];
  const float K = kAdv ? (float)((double)p.dt * (double)nu0 * (double)p.inv_h2) : p.dt * nu0;
  const float fa = (kScheme == kCentral ? 0.5f : 1.f) * (p.dt * p.inv_h);
  auto scaled = [](float4 x, float f) { return make_float4(f * x.x, f * x.y, f * x.z, f * x.w); };
  auto at4 = [&](const float* f, int i, int t) { return *reinterpret_cast<const float4*>(f + base + (size_t)i * n + 4 * t); };
  float c[RT][4];
#pragma unroll
  for (int k = 0; k < RT; ++k) {
    const float4 x = at4(p.u, i0 + k, tx);
    c[k][0] = x.x; c[k][1] = x.y; c[k][2] = x.z; c[k][3] = x.w;
  }
  if (kAdv) {
#pragma unroll
    for (int k = 0; k < RT; ++k) {  // row r of av: the faces between rows band + r - 1 and band + r
      av[(ty * RT + k + 1) * NX + tx] = scaled(at4(p.ax, i0 + k, tx), fa);
      bv[(ty * RT + k) * NX + tx] = scaled(at4(p.ay, i0 + k, tx), fa);
    }
    if (ty == 0) av[tx] = scaled(at4(p.ax, band > 0 ? band - 1 : n - 1, tx), fa);
  }
  if (kScheme == kHeatField) {
#pragma unroll
    for (int k = 0; k < RT; ++k) av[(ty * RT + k) * NX + tx] = scaled(at4(p.coef, i0 + k, tx), p.dt);
  }
  if (NC > 1) cluster_arrive();
  if (NC > 1) cluster_wait();
  else __syncthreads();

  for (int s = 0; s < p.steps; ++s) {
    const int par = s & 1;
    float4* tp = top + par * rows * NX;
    float4* bp = bot + par * rows * NX;
    float2* rp = rim + par * RT * rows * 2;
    const float4 ct = make_float4(c[0][0], c[0][1], c[0][2], c[0][3]);
    const float4 cb = make_float4(c[RT - 1][0], c[RT - 1][1], c[RT - 1][2], c[RT - 1][3]);
    tp[ty * NX + tx] = ct;
    bp[ty * NX + tx] = cb;
    if (NX > 32 && lane == 0) {
#pragma unroll
      for (int k = 0; k < RT; ++k) rp[(ty * RT + k) * 2 + wx].x = c[k][0];
    }
    if (NX > 32 && lane == 31) {
#pragma unroll
      for (int k = 0; k < RT; ++k) rp[(ty * RT + k) * 2 + wx].y = c[k][3];
    }
    if (NC > 1) {
      if (ty == 0 && (kPeriodic || !first)) store_peer(below + par * NX + tx, up_rank, ct);
      if (ty == rows - 1 && (kPeriodic || !last)) store_peer(above + par * NX + tx, dn_rank, cb);
      cluster_arrive();
    }
    // while the rims travel: the faces inside the tile, and to the adjacent lanes' tiles
    float o[RT][4];
#pragma unroll
    for (int k = 0; k < RT; ++k) {
      float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kAdv) b = bv[(ty * RT + k) * NX + tx];
      const float bq[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float t = through<kScheme>(bq[q], K, c[k][q], c[k][q + 1]);
        o[k][q] = q == 0 ? t : o[k][q] + t;
        o[k][q + 1] = -t;
      }
      float r = __shfl_sync(0xffffffffu, c[k][0], (lane + 1) & 31);
      if (!kPeriodic && tx == NX - 1) r = c[k][2];
      const float t = through<kScheme>(bq[3], K, c[k][3], r);
      if (NX == 32 || lane < 31) o[k][3] += t;
      // the left face's flux from the left lane
      float l = __shfl_sync(0xffffffffu, t, (lane + 31) & 31);
      if (!kPeriodic && tx == 0) l = c[k][0] - c[k][1];  // heat: c - u_{-1}, u_{-1} = u_1
      if (NX == 32 || lane > 0 || (!kPeriodic && tx == 0)) o[k][0] -= l;
      if (NX > 32 && !kPeriodic && tx == NX - 1) o[k][3] += t;
    }
#pragma unroll
    for (int k = 0; k + 1 < RT; ++k) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kAdv) a = av[(ty * RT + k + 1) * NX + tx];
      const float aq[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float t = through<kScheme>(aq[q], K, c[k][q], c[k + 1][q]);
        o[k][q] += t;
        o[k + 1][q] -= t;
      }
    }
    if (NC > 1) cluster_wait();
    else __syncthreads();
    {  // the rows above and below
      float4 x = ty > 0 ? bp[(ty - 1) * NX + tx] : NC > 1 ? above[par * NX + tx] : bp[(rows - 1) * NX + tx];
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kAdv) a = av[ty * RT * NX + tx];
      if (!kPeriodic && first) x = make_float4(c[1][0], c[1][1], c[1][2], c[1][3]);
      o[0][0] -= through<kScheme>(a.x, K, x.x, c[0][0]);
      o[0][1] -= through<kScheme>(a.y, K, x.y, c[0][1]);
      o[0][2] -= through<kScheme>(a.z, K, x.z, c[0][2]);
      o[0][3] -= through<kScheme>(a.w, K, x.w, c[0][3]);
      float4 y = ty + 1 < rows ? tp[(ty + 1) * NX + tx] : NC > 1 ? below[par * NX + tx] : tp[tx];
      if (kAdv) a = av[(ty * RT + RT) * NX + tx];
      if (!kPeriodic && last) y = make_float4(c[RT - 2][0], c[RT - 2][1], c[RT - 2][2], c[RT - 2][3]);
      o[RT - 1][0] += through<kScheme>(a.x, K, c[RT - 1][0], y.x);
      o[RT - 1][1] += through<kScheme>(a.y, K, c[RT - 1][1], y.y);
      o[RT - 1][2] += through<kScheme>(a.z, K, c[RT - 1][2], y.z);
      o[RT - 1][3] += through<kScheme>(a.w, K, c[RT - 1][3], y.w);
    }
    if (NX > 32) {  // the faces between a row's two warps, and (periodic) between its ends
      if (lane == 31 && (kPeriodic || tx < NX - 1)) {
#pragma unroll
        for (int k = 0; k < RT; ++k) {
          const float b = kAdv ? bv[(ty * RT + k) * NX + tx].w : 0.f;
          o[k][3] += through<kScheme>(b, K, c[k][3], rp[(ty * RT + k) * 2 + (wx ^ 1)].x);
        }
      }
      if (lane == 0 && (kPeriodic || tx > 0)) {
        const int tl = tx > 0 ? tx - 1 : NX - 1;
#pragma unroll
        for (int k = 0; k < RT; ++k) {
          const float b = kAdv ? bv[(ty * RT + k) * NX + tl].w : 0.f;
          o[k][0] -= through<kScheme>(b, K, rp[(ty * RT + k) * 2 + (wx ^ 1)].y, c[k][0]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < RT; ++k) {
      float4 nu = make_float4(K, K, K, K);
      if (kScheme == kHeatField) nu = av[(ty * RT + k) * NX + tx];
      const float nq[4] = {nu.x, nu.y, nu.z, nu.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) c[k][q] = kAdv ? c[k][q] + o[k][q] : fmaf(nq[q], o[k][q], c[k][q]);
    }
  }
#pragma unroll
  for (int k = 0; k < RT; ++k)
    *reinterpret_cast<float4*>(p.u + base + (size_t)(i0 + k) * n + j0) = make_float4(c[k][0], c[k][1], c[k][2], c[k][3]);
}

template <int kScheme, int NX>
constexpr size_t wide_bytes() {
  constexpr int rows = kWideThreads / NX;
  constexpr size_t coef = kScheme >= kUpwind ? 2 * kWideRT * rows + 1 : kScheme == kHeatField ? kWideRT * rows : 0;
  return (4 * rows * NX + 4 * NX + coef * NX) * 16 + (NX > 32 ? 2 * kWideRT * rows * 2 * 8 : 0);
}

// 1D heat, one CTA per field.
constexpr int kLineMax = 8192;
template <bool kField>
__global__ void __launch_bounds__(1024) fom_line_kernel(float* u, const float* coef, int P, int steps, float r_over) {
  extern __shared__ float4 smem4[];
  float* src = reinterpret_cast<float*>(smem4);
  float* dst = src + P;
  const size_t base = (size_t)blockIdx.x * P;
  for (int i = threadIdx.x; i < P; i += blockDim.x) src[i] = u[base + i];
  const float nu0 = kField ? 0.f : coef[blockIdx.x];
  __syncthreads();
  for (int s = 0; s < steps; ++s) {
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
      float v = 0.f;
      if (i > 0 && i < P - 1) {
        const float c = src[i], nu = kField ? __ldg(coef + base + i) : nu0;
        v = fmaf(r_over * nu, src[i - 1] + src[i + 1] - 2.f * c, c);
      }
      dst[i] = v;
    }
    __syncthreads();
    float* t = src;
    src = dst;
    dst = t;
  }
  for (int i = threadIdx.x; i < P; i += blockDim.x) u[base + i] = src[i];
}

// 2D, other sides, one CTA per field, nodes dealt to the threads; the face velocities
// are in shared memory too.  A step takes 1.8 us (heat) and 3.2 us (advection) at side
// 97, growing with the area, against 4.1 us for a launch per step: the largest sides.
constexpr int kFieldMaxHeat = 128, kFieldMaxAdv = 100;
template <int kScheme>
__device__ __forceinline__ void fom_field_body(const FomParams& p) {
  constexpr bool kAdv = kScheme >= kUpwind, kCen = kScheme == kCentral;
  extern __shared__ float4 smem4[];
  const int n = p.n, N = n * n, NT = blockDim.x;
  const int di = NT / n, dj = NT - di * n;  // the next node of a thread is NT further on
  float* src = reinterpret_cast<float*>(smem4);
  float* dst = src + N;
  const size_t base = (size_t)blockIdx.x * N;
  const float *ax = p.ax + base, *ay = p.ay + base;
  for (int e = threadIdx.x; e < N; e += blockDim.x) src[e] = p.u[base + e];
  if (kAdv) {
    float *as = dst + N, *bs = as + N;
    for (int e = threadIdx.x; e < N; e += blockDim.x) {
      as[e] = ax[e];
      bs[e] = ay[e];
    }
    ax = as;
    ay = bs;
  }
  const float nu0 = kScheme == kHeatField ? 0.f : p.coef[blockIdx.x];
  __syncthreads();
  for (int s = 0; s < p.steps; ++s) {
    int i = threadIdx.x / n, j = threadIdx.x - i * n;
    for (int e = threadIdx.x; e < N; e += NT) {
      const int row = i * n;
      const int up = i > 0 ? row - n : kAdv ? N - n : n, dn = i < n - 1 ? row + n : kAdv ? 0 : row - n;
      const int jl = j > 0 ? j - 1 : kAdv ? n - 1 : 1, jr = j < n - 1 ? j + 1 : kAdv ? 0 : n - 2;
      const float c = src[row + j], uim = src[up + j], uip = src[dn + j], ujm = src[row + jl], ujp = src[row + jr];
      if (kAdv) {
        const float fr = flux<kCen>(ax[row + j], c, uip), fl = flux<kCen>(ax[up + j], uim, c);
        const float gr = flux<kCen>(ay[row + j], c, ujp), gl = flux<kCen>(ay[row + jl], ujm, c);
        const float div = (fr - fl + gr - gl) * p.inv_h;
        const float lap = (uim + uip + ujm + ujp - 4.f * c) * p.inv_h2;
        dst[row + j] = fmaf(p.dt, fmaf(nu0, lap, -div), c);
      } else {
        const float lap = (uim + uip - 2.f * c) + (ujm + ujp - 2.f * c);
        dst[row + j] = fmaf(p.dt * (kScheme == kHeatField ? __ldg(p.coef + base + row + j) : nu0), lap, c);
      }
      i += di;
      j += dj;
      if (j >= n) {
        j -= n;
        ++i;
      }
    }
    __syncthreads();
    float* t = src;
    src = dst;
    dst = t;
  }
  for (int e = threadIdx.x; e < N; e += blockDim.x) p.u[base + e] = src[e];
}
// Two CTAs on an SM for many fields: 3000 fields of 57^2, heat, one step, 67 us with one,
// 48 with two.  The heat form spills 28 bytes for it (one field of 49^2, 20 steps: 15
// against 19 us), so few fields take the one without the bound.
template <int kScheme>
__global__ void __launch_bounds__(1024, 2) fom_field_kernel(FomParams p) { fom_field_body<kScheme>(p); }
__global__ void __launch_bounds__(1024) fom_field_few_kernel(FomParams p) { fom_field_body<kHeat>(p); }

// Whether one launch of fom_field_kernel pays against a launch per step, in microseconds
// as measured over sides 49 to 127, 1 to 3000 fields and 1 to 50 steps (with these lines
// no shape is more than 4 % slower than a launch per step).
//  * Fewer fields than SMs: the launch takes 9 and, per step, 3.0 (heat), 3.75 (with a
//    coefficient field) or 4.7 (advection) at side 127 in proportion to the area; a launch
//    per step 4.2 (more where the fields' bytes take longer; an odd count copies back as
//    long as a step), a call at least 13.  Ten fields of 127^2 with a coefficient field,
//    four steps: 26 against 18 us; 20 steps: 85 against 84; of 97^2, eight: 26 against 35.
//  * Heat from side 120 on (one field an SM), one or two steps of many fields: the loads
//    are not overlapped.  1000 with a coefficient field, 127^2, one step: 115 against 87
//    us, two 141 against 121; 3000 of heat 266 against 225.
bool field_pays(int scheme, int n, int n_batch, int steps, int sms) {
  const double nodes = (double)n * n;
  if (n_batch < sms) {
    const double per_step = (scheme == kHeat ? 3.0 : scheme == kHeatField ? 3.75 : 4.7) * nodes / (127 * 127);
    const double launch = std::max(4.2, 3.3 + (scheme >= kUpwind ? 8e-6 : 3.5e-6) * n_batch * nodes);
    return 9.0 + steps * per_step <= std::max(13.0, (steps + (steps & 1)) * launch);
  }
  return scheme >= kUpwind || n < 120 || steps > 2 || n_batch <= (scheme == kHeatField ? 4 : 12) * sms;
}

// SMs of the current device.  Asked for once per device: the attribute query took 0.7 us
// of each call, 5 % of one with a launch or two.
cudaError_t sm_count(int* sms) {
  static std::atomic<int> known[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  *sms = dev < 64 ? known[dev].load(std::memory_order_relaxed) : 0;
  if (*sms > 0) return cudaSuccess;
  e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && dev < 64) known[dev].store(*sms, std::memory_order_relaxed);
  return e;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

template <typename Kernel>
cudaError_t launch_cluster(Kernel kernel, const FomParams& p, int nc, int n_batch, int threads, size_t smem, cudaStream_t s) {
  const cudaError_t e = allow_smem(kernel, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nc, n_batch);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = nc;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <int kScheme>
cudaError_t launch_2d(const FomParams& p, int n_batch, cudaStream_t s, bool* done) {
  const int n = p.n;
  const bool field = kScheme == kHeatField, adv = kScheme >= kUpwind;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  // One or two steps of a batch that streams through HBM gain nothing from staying on
  // the chip, and the velocities' load is not overlapped there: 512 fields of 256^2, one
  // step 142 against 122 us, two 167 against 156 us (three: 194 against 234 us).
  if (adv && n_batch > 2 * sms && p.steps <= (n > 128 ? 2 : 1) && n != 128) return cudaSuccess;
  if (n % 4 == 0 && n <= 256 && aligned16(p.u) && (!adv || (aligned16(p.ax) && aligned16(p.ay))) &&
      (!field || aligned16(p.coef))) {
    // Many fields: tiles of four rows (the fewest rim values per node), the fewest CTAs
    // per field.  Few fields: as many CTAs of a cluster as the GPU has room for (sides
    // above 64: one CTA needs no cluster barrier) and tiles of fewer rows, for at most
    // 256 threads.
    int RT = 4, NC = 1;
    while (NC < 8 && tile_thr(n, RT, NC) > kTileThreads) NC *= 2;
    if ((n == 128 || n == 256) && (long long)n_batch * NC > sms / 2) {
      // (37 to 300 fields of 256^2, two steps of either model: 1.05 to 1.4 times a launch per step's time)
      if (n == 256 && p.steps <= 2) return cudaSuccess;
      *done = true;
      if (n == 128) return launch_cluster(fom_wide_kernel<kScheme, 32>, p, 1, n_batch, kWideThreads, wide_bytes<kScheme, 32>(), s);
      return launch_cluster(fom_wide_kernel<kScheme, 64>, p, 4, n_batch, kWideThreads, wide_bytes<kScheme, 64>(), s);
    }
    // One step by clusters of eight CTAs, the GPU full: the loads and stores of such a call
    // are not overlapped.  Sides 180 to 192 leave 288 threads a CTA: 600 fields of 180^2,
    // heat with a coefficient field, 115 against 107 us.  Advection: 300 fields of 212^2 88
    // against 84 us, of 180^2 74 (two steps 95) against 63 (92); up to 200 fields no slower.
    const int thr = tile_thr(n, RT, NC);
    if (NC == 8 && ((adv && 2 * n_batch > 3 * sms && p.steps <= (thr <= 288 ? 2 : 1)) ||
                    (field && thr <= 288 && n_batch >= sms && p.steps == 1)))
      return cudaSuccess;
    if ((long long)n_batch * NC < sms) {
      while (n > 64 && NC < 8 && (long long)n_batch * NC * 2 <= sms) NC *= 2;
      while (RT > 1 && tile_thr(n, RT / 2, NC) <= (NC > 1 ? 256 : kTileThreads)) RT /= 2;
    }
    if (tile_thr(n, RT, NC) <= kTileThreads) {
      FomParams q = p;
      q.NC = NC;
      *done = true;
      return launch_cluster(RT == 4 ? fom_tile_kernel<kScheme, 4> : RT == 2 ? fom_tile_kernel<kScheme, 2> : fom_tile_kernel<kScheme, 1>,
                            q, NC, n_batch, tile_thr(n, RT, NC), tile_bytes(n, RT, NC), s);
    }
  }
  // (two steps of advection at side 97: 14.5 us against 13.8 us for two launches)
  if (n <= (adv ? kFieldMaxAdv : kFieldMaxHeat) && (!adv || p.steps > 2) && field_pays(kScheme, n, n_batch, p.steps, sms)) {
    const size_t smem = (size_t)(adv ? 4 : 2) * n * n * sizeof(float);
    const auto kernel = kScheme == kHeat && n_batch <= sms ? fom_field_few_kernel : fom_field_kernel<kScheme>;
    e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    *done = true;
    kernel<<<n_batch, std::min(1024, (n * n + 31) / 32 * 32), smem, s>>>(p);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_fom_fused(int kind, int n_batch, int nx, const float* coef, const float* ax, const float* ay,
                             double dt, int n_steps, float* u, cudaStream_t s, bool* done) {
  *done = false;
  if (kind == CROM_FOM_HEAT1D_DIRICHLET || kind == CROM_FOM_HEAT1D_DIRICHLET_FIELD) {
    if (nx > kLineMax) return cudaSuccess;
    // One or two steps of many short lines: a CTA per line does not overlap its load, step
    // and store.  16000 lines of 1500 with a coefficient field, one step: 155 against 117
    // us; 8000 of 700, two: 38 against 34; without, 8000 of 1024, one: 33 against 31 (16000,
    // which no longer stay in L2 with their copies: 61 against 77).
    const long long nodes = (long long)n_batch * nx;
    const bool short_lines = kind == CROM_FOM_HEAT1D_DIRICHLET_FIELD
                                 ? (n_steps == 1 && nx <= 4096) || (n_steps == 2 && nx < 2048)
                                 : n_steps == 1 && nx <= 1024 && nodes < 12000000;
    if (nodes > 5000000 && short_lines) return cudaSuccess;
    const double dx = 1.0 / (nx - 1);
    const float r_over = (float)(dt / (dx * dx));
    const size_t smem = (size_t)2 * nx * sizeof(float);
    auto kernel = kind == CROM_FOM_HEAT1D_DIRICHLET ? fom_line_kernel<false> : fom_line_kernel<true>;
    const cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    *done = true;
    kernel<<<n_batch, std::min(1024, (nx + 31) / 32 * 32), smem, s>>>(u, coef, nx, n_steps, r_over);
    return cudaGetLastError();
  }
  FomParams p{};
  p.u = u;
  p.ax = ax;
  p.ay = ay;
  p.coef = coef;
  p.n = nx;
  p.steps = n_steps;
  if (kind == CROM_FOM_HEAT2D_NEUMANN || kind == CROM_FOM_HEAT2D_NEUMANN_FIELD) {
    const double h = 1.0 / (nx - 1);
    p.dt = (float)(dt / (h * h));
    return kind == CROM_FOM_HEAT2D_NEUMANN ? launch_2d<kHeat>(p, n_batch, s, done)
                                           : launch_2d<kHeatField>(p, n_batch, s, done);
  }
  const double h = 1.0 / nx;
  p.dt = (float)dt;
  p.inv_h = (float)(1.0 / h);
  p.inv_h2 = (float)(1.0 / (h * h));
  return kind == CROM_FOM_ADVDIFF2D_PERIODIC_CENTRAL ? launch_2d<kCentral>(p, n_batch, s, done)
                                                     : launch_2d<kUpwind>(p, n_batch, s, done);
}

}  // namespace crom
