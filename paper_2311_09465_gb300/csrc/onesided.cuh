// Eigenpairs of the symmetric positive definite (2N-1) x (2N-1) matrices of
// eq. (3D-tau) in FP32, one matrix per group of N lanes, entirely in registers:
// M = L L^T (Cholesky), then one-sided Jacobi (Hestenes 1958; on a Cholesky
// factor: Veselic & Hari 1989) on the columns of L.  Plane rotations from the
// right, L J = F, make the columns of F orthogonal; then M = F F^T gives the
// eigenvectors f_a / |f_a| and the eigenvalues |f_a|^2, so only one matrix is
// rotated (the two-sided form rotates rows and columns of M and accumulates V).
//
// Layout: NM = 2N-1 columns in a line of slots 0..2N-2; lane p of a group
// holds slot 2p-1 in x and slot 2p in y (lane 0: only y, its x stays zero).
// Odd-even ordering (every pair of columns meets once in NM rounds): a round
// rotates neighbouring slots and exchanges them.  The pairs (2p-1, 2p) are in
// one lane; for the pairs (2p, 2p+1) the right lane's x moves over and one
// column moves back, so a round costs one column of shuffles on average.
// Lanes without a partner do a rotation by a right angle with a zero column,
// which leaves their column in its slot without any select.
//
// What bounds it: 128 FP32 lanes and 32 shuffle lanes a clock and SM; a round
// is about 90 FP32 instructions and 14 shuffles a lane at N = 7, with no
// shared memory in the loop.
#pragma once
#include "common.cuh"

namespace ts {

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// 1/sqrt(x) with one Newton step on the hardware approximation
__device__ __forceinline__ float rsqrt_newton(float x) {
  const float r = rsqrt_ftz(x);
  return fmaf(0.5f * r, fmaf(-x * r, r, 1.f), r);
}

// rotation that makes X and Y orthogonal: X' = X - s (Y + ta X), Y' = Y + s (X - ta Y);
// ax, ay: their squared norms, g: their product; t = s/c is returned for the norms
__device__ __forceinline__ void rotation_of(float ax, float ay, float g, float& s, float& ta, float& t) {
  const float d = ay - ax;
  const float h2 = fmaf(2.f * g, 2.f * g, d * d);
  const float h = h2 * rsqrt_ftz(h2);
  t = 2.f * g * rcp_ftz(d + copysignf(h, d));
  if (!(h2 > 1e-36f)) t = 0.f;
  const float c = rsqrt_ftz(fmaf(t, t, 1.f));
  s = t * c;
  ta = s * rcp_ftz(1.f + c);
}

// Cholesky factor of the group's matrix: on entry x, y hold the full columns 2p-1
// and 2p, on return the columns of L (zeros above the diagonal).  rows: scratch
// of NM rows of LD floats (16-byte aligned, LD a multiple of 4 and >= NM), of
// which a lane uses its own two.  base: the group's first lane; own: whether the
// lane belongs to a group.  floor: a lower bound of the eigenvalues, hence of the
// exact pivots; rounding may take a computed pivot below it.  Returns the smallest
// pivot as computed, the same in the whole group (lanes outside: of the first group).
// ROLLED: a loop over pivots in which the registers move up one row a step, so
// that the pivot is always at index 0, and finished columns go through shared
// memory.  Unrolled it needs no memory and half the shuffles, but is up to a
// quarter of a kernel's code: rolled where that no longer fits the instruction
// cache (fixed-point tau, N = 10: 34.5 ms unrolled, 8.0 rolled; N = 7: 10.8 and
// 10.7; N = 5: 3.6 and 3.7; FP32 tau, N = 10: 2.42 and 2.16, N = 7: 2.60 and 2.99).
template <int N, int LD, bool ROLLED>
__device__ __forceinline__ float cholesky_columns(float (&x)[2 * N - 1], float (&y)[2 * N - 1], int p, bool own, int base,
                                                  float floor, float* rows) {
  constexpr int NM = 2 * N - 1;
  float least = 3e38f;
  if constexpr (!ROLLED) {
    // a lane outside a group must stay zero: no column of it is a pivot
    const int jx = own ? 2 * p - 1 : 4 * N, jy = own ? 2 * p : 4 * N;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      const int src = base + (k + 1) / 2;
      float l[NM];
#pragma unroll
      for (int i = k; i < NM; ++i) l[i] = __shfl_sync(0xffffffffu, (k & 1) ? x[i] : y[i], src);
      const float piv = fmaxf(l[k], floor), rd = rsqrt_newton(piv);
      least = fminf(least, l[k]);
      const float mx = jx > k ? x[k] * rd * rd : 0.f, my = jy > k ? y[k] * rd * rd : 0.f;
#pragma unroll
      for (int i = k + 1; i < NM; ++i) {
        const float sx = fmaf(-l[i], mx, x[i]), sy = fmaf(-l[i], my, y[i]);
        x[i] = jx == k ? l[i] * rd : sx;
        y[i] = jy == k ? l[i] * rd : sy;
      }
      if (jx >= k) x[k] = jx == k ? piv * rd : 0.f;
      if (jy >= k) y[k] = jy == k ? piv * rd : 0.f;
    }
    return least;
  }
  float* rx = rows + (own && p > 0 ? 2 * p - 1 : 0) * LD;
  float* ry = rows + 2 * p * LD;
  if (own) {
#pragma unroll
    for (int i = 0; i < (NM + 3) / 4; ++i) {
      if (p > 0) reinterpret_cast<float4*>(rx)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      reinterpret_cast<float4*>(ry)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
#pragma unroll 1
  for (int k = 0; k < NM; ++k) {
    const int src = base + (k + 1) / 2;
    const bool odd = k & 1;
    float l[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) l[i] = __shfl_sync(0xffffffffu, odd ? x[i] : y[i], src);
    const float rd = rsqrt_newton(fmaxf(l[0], floor));
    least = fminf(least, l[0]);
    l[0] = fmaxf(l[0], floor);
    if (own && p == (k + 1) / 2) {
      float* dst = (odd ? rx : ry) + k;
#pragma unroll
      for (int i = 0; i < NM; ++i)
        if (i < NM - k) dst[i] = l[i] * rd;
    }
    // a column j > k loses l l_j, l_j = rd A_jk
    const float mx = 2 * p - 1 > k ? x[0] * rd * rd : 0.f;
    const float my = 2 * p > k ? y[0] * rd * rd : 0.f;
#pragma unroll
    for (int i = 0; i + 1 < NM; ++i) {
      x[i] = fmaf(-l[i + 1], mx, x[i + 1]);
      y[i] = fmaf(-l[i + 1], my, y[i + 1]);
    }
    x[NM - 1] = y[NM - 1] = 0.f;
  }
#pragma unroll
  for (int j = 0; j < (NM + 3) / 4; ++j) {
    const float4 a = reinterpret_cast<const float4*>(rx)[j], b = reinterpret_cast<const float4*>(ry)[j];
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (4 * j + t < NM) {
        x[4 * j + t] = own && p > 0 ? av[t] : 0.f;
        y[4 * j + t] = own ? bv[t] : 0.f;
      }
  }
  return least;
}

// One-sided Jacobi on the group's columns.  Sweeps until every pair of the warp
// had a squared cosine of at most ortho2 before its rotation; that last sweep
// leaves cosines of the order of ortho2.  Returns whether this lane's pairs had.
constexpr int ONESIDED_SWEEPS = 15;

template <int N>
__device__ __forceinline__ bool onesided_jacobi(float (&x)[2 * N - 1], float (&y)[2 * N - 1], int p, int lane,
                                                float ortho2) {
  constexpr int NM = 2 * N - 1;
  if constexpr (N == 1) return true;
  const int up = (lane + 31) & 31, down = (lane + 1) & 31;
  const bool first = p == 0, last = p == N - 1;
  bool rotated = true;
#pragma unroll 1
  for (int sweep = 0; sweep < ONESIDED_SWEEPS; ++sweep) {
    float ax = 0.f, ay = 0.f;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      ax = fmaf(x[i], x[i], ax);
      ay = fmaf(y[i], y[i], ay);
    }
    rotated = false;
#pragma unroll 1
    for (int rr = 0; rr < N; ++rr) {
      float g = 0.f, s, ta, t;
      // pairs (2p-1, 2p)
      {
        float g0 = 0.f, g1 = 0.f;
#pragma unroll
        for (int i = 0; i < NM; i += 2) g0 = fmaf(x[i], y[i], g0);
#pragma unroll
        for (int i = 1; i < NM; i += 2) g1 = fmaf(x[i], y[i], g1);
        g = g0 + g1;
      }
      rotation_of(ax, ay, g, s, ta, t);
      rotated |= g * g > ortho2 * ax * ay;
      if (first) s = -1.f, ta = -1.f;
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const float nx = fmaf(-s, fmaf(ta, x[i], y[i]), x[i]);
        const float ny = fmaf(s, fmaf(-ta, y[i], x[i]), y[i]);
        x[i] = ny;
        y[i] = nx;
      }
      {
        const float na = fmaf(-t, g, ax), nb = fmaf(t, g, ay);
        ax = first ? 0.f : nb;
        ay = first ? ay : na;
      }
      // pairs (2p, 2p+1)
      float z[NM];
#pragma unroll
      for (int i = 0; i < NM; ++i) z[i] = __shfl_sync(0xffffffffu, x[i], down);
      float az = __shfl_sync(0xffffffffu, ax, down);
      {
        float g0 = 0.f, g1 = 0.f;
#pragma unroll
        for (int i = 0; i < NM; i += 2) g0 = fmaf(y[i], z[i], g0);
#pragma unroll
        for (int i = 1; i < NM; i += 2) g1 = fmaf(y[i], z[i], g1);
        g = g0 + g1;
      }
      rotation_of(ay, az, g, s, ta, t);
      rotated |= g * g > ortho2 * ay * az;
      if (last) s = 1.f, ta = 1.f;
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const float nx = fmaf(-s, fmaf(ta, y[i], z[i]), y[i]);
        const float ny = fmaf(s, fmaf(-ta, z[i], y[i]), z[i]);
        y[i] = ny;
        x[i] = __shfl_sync(0xffffffffu, nx, up);
      }
      {
        const float na = last ? 0.f : fmaf(-t, g, ay), nb = last ? ay : fmaf(t, g, az);
        ay = nb;
        ax = __shfl_sync(0xffffffffu, na, up);
      }
    }
    if (!__any_sync(0xffffffffu, rotated)) break;
  }
  return !rotated;
}

}  // namespace ts
