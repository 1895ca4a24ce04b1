// Small dense linear algebra shared by the step kernels: the r x r normal
// equations (J^T J) delta = -J^T rho of one Gauss-Newton iteration (paper App. C),
// solved in FP64.
#pragma once

#include <math.h>

#include "../../include/crom.h"

namespace crom {

// Warp-parallel FP64 Cholesky solve of A x = b, r <= 32, with A = a[i*(r+1)+j] in
// shared memory (both triangles) and b in column r.  Status: NONFINITE when A or b holds
// a NaN/Inf, SINGULAR when a pivot is <= 1e-14 * max diag(A); on success x_k is left in
// a[k*(r+1)+r].  All 32 lanes of the warp must call it.
//
// A single warp's FP64 instruction takes 64 clocks here whatever its active lanes, and a
// reciprocal square root about 380, so the chain is kept short: right-looking, the
// forward substitution carried along as one more column, the trailing entries
// (i, k), j < k <= i, and the right-hand sides dealt over the lanes (two instructions at
// r = 8, not the longest row's length), the back substitution in registers.  Every entry
// sees the same operations in the same order as the row-per-lane form (17k clocks at
// r = 8, this form 9.7k).
__device__ __forceinline__ int chol_solve_warp(double* A, int r, int lane) {
  const int R = r + 1;
  // FP64 comparisons and conversions cost as much as additions: the checks compare bit
  // patterns (non-negative doubles order like integers)
  const long long kInf = 0x7ff0000000000000ll;
  bool bad = false;
  for (int e = lane; e < r * R; e += 32) bad |= (__double_as_longlong(A[e]) & kInf) == kInf;
  if (__any_sync(0xffffffffu, bad)) return CROM_ERR_NONFINITE;
  long long dmax = lane < r ? max(0ll, __double_as_longlong(A[lane * R + lane])) : 0ll;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  const long long tol = __double_as_longlong(1e-14 * __longlong_as_double(dmax));
  // this lane's first two trailing entries: row a (a + 2 entries: columns 0..a, then b)
  auto entry = [](int e, int& a, int& c) {
    a = (int)((sqrtf(9.f + 8.f * e) - 3.f) * 0.5f);
    if (a * (a + 3) / 2 > e) --a;
    if ((a + 1) * (a + 4) / 2 <= e) ++a;
    c = e - a * (a + 3) / 2;
  };
  int a0, c0, a1, c1;
  entry(lane, a0, c0);
  entry(lane + 32, a1, c1);
  double inv_mine = 0.0;  // lane j: 1 / l_jj
  for (int j = 0; j < r; ++j) {
    const double d = A[j * R + j];
    const int i0 = j + 1 + lane, at0 = i0 < r ? i0 * R + j : j * R + r;
    const double col = i0 <= r ? A[at0] : 0.0;
    const long long dl = __double_as_longlong(d);
    if (!(dl > tol && dl <= kInf)) return CROM_ERR_SINGULAR;  // !(d > tol), NaN included
    // one reciprocal square root instead of a square root and a division
    const double inv = rsqrt(d);
    if (lane == j) inv_mine = inv;
    // column j of L, and y_j = b_j / l_jj (r - j <= 32 of them)
    if (i0 <= r) A[at0] = col * inv;
    __syncwarp();
    // trailing entries of the n rows below j
    const int n = r - 1 - j, cnt = n * (n + 3) / 2;
    for (int e = lane; e < cnt; e += 32) {
      int a = a0, c = c0;
      if (e >= 32) { a = a1; c = c1; }
      if (e >= 64) entry(e, a, c);
      const int i = j + 1 + a;
      const int at = i * R + (c <= a ? j + 1 + c : r);
      const double w = c <= a ? A[(j + 1 + c) * R + j] : A[j * R + r];
      A[at] -= A[i * R + j] * w;
    }
    __syncwarp();
  }
  // L^T x = y: lane i carries y_i
  double y = lane < r ? A[lane * R + r] : 0.0;
  for (int k = r - 1; k >= 0; --k) {
    const double lk = lane < k ? A[k * R + lane] : 0.0;
    const double xk = __shfl_sync(0xffffffffu, y * inv_mine, k);
    if (lane == k) A[k * R + r] = xk;
    if (lane < k) y -= lk * xk;
  }
  __syncwarp();
  return CROM_OK;
}

}  // namespace crom
