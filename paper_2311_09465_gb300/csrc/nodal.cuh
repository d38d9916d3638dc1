// Shared by the kernels that form nodal blocks of the tangent (precond.cu,
// assembled.cu): small dense matrices of a quadrature point, n = 2N - 1, in the
// orthonormal basis (x_0, sqrt2 Re, sqrt2 Im), with a group of N lanes a matrix
// and two columns a lane (2p-1 and 2p, lane 0 only 0), as in tau.cu.
//
// In this basis tau and Conv(beta) are symmetric and Omega is antisymmetric, so
// W_qa = -lambda_qa Omega + Conv(beta_qa) is the transpose of
// S_qa = lambda_qa Omega + Conv(beta_qa), W tau is the transpose of X = tau S, and
// W tau S = S^T X: one full product and a second one where the storage
// coordinates of the fields need three.  A left matrix is read row by row from
// shared memory (16-byte loads that the group shares) against the lane's two
// columns in registers, eight multiply-adds a load; with one output a lane and
// both operands in shared memory it was two loads a multiply-add.
//
// Needs four groups a warp (N <= 7).
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace ts {

template <int N>
struct Nodal {
  static constexpr int NM = 2 * N - 1, C = 2 * N, L = N - 1, NT = NM * (NM + 1) / 2, NTP = Dims<N>::NT_PAD;
  static constexpr int LD = (2 * N + 3) & ~3;          // floats a row, 16-byte multiple
  static constexpr int MAT0 = NM * LD;
  // matrices of the four groups start 4 words apart mod 32: their 16-byte reads do not collide
  static constexpr int MAT = MAT0 + ((4 - MAT0) % 32 + 32) % 32;
  static constexpr int TW = 3 * N;                     // modes -(N-1) .. 2(N-1)
};

// a double to FP32 (ties away from zero) with integer instructions: the
// conversion instruction runs on the FP64 pipe
__device__ __forceinline__ float nodal_float(float x) { return x; }
__device__ __forceinline__ float nodal_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)(b >> 52) & 0x7ff;
  if (e < 897) return 0.f;
  if (e > 1149) return e == 0x7ff && (b << 12) ? __int_as_float(0x7fffffff) : __int_as_float((int)(sign | 0x7f800000u));
  return __int_as_float((int)(((unsigned)((b + 0x10000000ull) >> 29) - 0xc0000000u) | sign));
}
// the FP32 value of a state entry: FP32, or the leading part of a double-float pair
__device__ __forceinline__ float nodal_value(float x) { return x; }
__device__ __forceinline__ float nodal_value(float2 x) { return x.x; }

// 16-byte asynchronous global -> shared copies (LDGSTS), grouped per stage
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

// What a warp reads of an element, copied to shared memory one element ahead
// (the loads of a row's elements depend on its lists, and the register tiles
// leave 8 warps an SM: waiting for them took 60% of the time): tau of the four
// points as stored, the state's rows of the four nodes, the geometry record.  One
// buffer is enough: it is read at the start of an element and refilled behind the
// element's products.
// Every part starts and ends on 16 bytes (NT_PAD and 4 C are multiples of 4).
template <typename T, typename U, int N>
struct NodalStage {
  static constexpr int TAU_B = 4 * Nodal<N>::NTP * (int)sizeof(T), ROW_B = 8 * N * (int)sizeof(U),
                       GEO_B = GEO_STRIDE * (int)sizeof(T), BYTES = TAU_B + 4 * ROW_B + GEO_B;
  static_assert(TAU_B % 16 == 0 && ROW_B % 16 == 0 && GEO_B % 16 == 0, "16-byte parts");
  static __device__ __forceinline__ void issue(char* dst, int64_t e, int4 nd, const T* tau, const U* u0, const T* geo,
                                               int lane) {
    const char* ts = reinterpret_cast<const char*>(tau) + e * TAU_B;
    for (int t = lane * 16; t < TAU_B; t += 512) cp_async16(dst + t, ts + t);
    for (int t = lane * 16; t < 4 * ROW_B; t += 512) {
      const int b = t / ROW_B;
      const int node = b == 0 ? nd.x : b == 1 ? nd.y : b == 2 ? nd.z : nd.w;
      cp_async16(dst + TAU_B + t, reinterpret_cast<const char*>(u0) + (int64_t)node * ROW_B + (t - b * ROW_B));
    }
    const char* gs = reinterpret_cast<const char*>(geo) + e * GEO_B;
    for (int t = lane * 16; t < GEO_B; t += 512) cp_async16(dst + TAU_B + 4 * ROW_B + t, gs + t);
    cp_async_commit();
  }
  static __device__ __forceinline__ const T* tau_of(const char* s) { return reinterpret_cast<const T*>(s); }
  static __device__ __forceinline__ const U* rows_of(const char* s) { return reinterpret_cast<const U*>(s + TAU_B); }
  static __device__ __forceinline__ const T* geo_of(const char* s) {
    return reinterpret_cast<const T*>(s + TAU_B + 4 * ROW_B);
  }
};

// packed upper-triangle index -> word offsets of (r, s) and (s, r) in a matrix
template <int N>
__device__ __forceinline__ void nodal_offsets(int* table, int tid, int nthreads) {
  using D = Nodal<N>;
  for (int t = tid; t < D::NT; t += nthreads) {
    int r = 0, rem = t;
    while (rem >= D::NM - r) {
      rem -= D::NM - r;
      ++r;
    }
    const int s = r + rem;
    table[t] = (r * D::LD + s) | (s * D::LD + r) << 16;
  }
}

// tau of a point, packed, to a full matrix (lane p of the group)
template <int N, typename T>
__device__ __forceinline__ void nodal_tau(const T* packed, const int* table, float* dst, int p) {
  for (int t = p; t < Nodal<N>::NT; t += N) {
    const float v = nodal_float(packed[t]);
    const int o = table[t];
    dst[o & 0xffff] = v;
    dst[o >> 16] = v;
  }
}

// mode p of a convolution's argument into its zero-padded table [2][TW] (re, im)
template <int N>
__device__ __forceinline__ void nodal_modes(float* table, int p, float re, float im) {
  constexpr int L = N - 1, TW = Nodal<N>::TW;
  float* tr = table + L;
  tr[p] = re;
  tr[TW + p] = im;
  if (p > 0) {
    tr[-p] = re;
    tr[TW - p] = -im;
    tr[L + p] = 0.f;
    tr[TW + L + p] = 0.f;
  }
}

// columns 2p-1 (x) and 2p (y) of om Omega + Conv (om = lambda times omega)
template <int N>
__device__ __forceinline__ void nodal_columns(const float* table, int p, float om, float (&x)[2 * N - 1],
                                              float (&y)[2 * N - 1]) {
  constexpr int L = N - 1, TW = Nodal<N>::TW;
  constexpr float S2 = Real<float>::SQRT2;
  const float* tr = table + L;
  const float* ti = tr + TW;
  const float w = p * om;
  x[0] = p == 0 ? 0.f : S2 * tr[p];
  y[0] = p == 0 ? tr[0] : S2 * ti[p];
#pragma unroll
  for (int k = 1; k < N; ++k) {
    const float pl = tr[k - p], ph = tr[k + p], ql = ti[k - p], qh = ti[k + p];
    const float d = k == p ? w : 0.f;
    x[2 * k - 1] = p == 0 ? 0.f : pl + ph;
    x[2 * k] = p == 0 ? 0.f : ql + qh + d;
    y[2 * k - 1] = p == 0 ? S2 * pl : qh - ql - d;
    y[2 * k] = p == 0 ? S2 * ql : pl - ph;
  }
}

template <int W>
__device__ __forceinline__ void nodal_row(const float* src, float (&dst)[W]) {
#pragma unroll
  for (int j = 0; j < W / 4; ++j) {
    const float4 v = reinterpret_cast<const float4*>(src)[j];
    dst[4 * j] = v.x;
    dst[4 * j + 1] = v.y;
    dst[4 * j + 2] = v.z;
    dst[4 * j + 3] = v.w;
  }
}
// the lane's two columns as rows 2p-1, 2p of a matrix (its transpose, row-major)
template <int N>
__device__ __forceinline__ void nodal_store_rows(float* m, int p, const float (&x)[2 * N - 1], const float (&y)[2 * N - 1]) {
  using D = Nodal<N>;
  float* dx = m + (2 * p - 1) * D::LD;
  float* dy = m + 2 * p * D::LD;
#pragma unroll
  for (int j = 0; j < D::LD / 4; ++j) {
    float a[4], b[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int i = 4 * j + t < D::NM ? 4 * j + t : D::NM - 1;
      a[t] = 4 * j + t < D::NM ? x[i] : 0.f;
      b[t] = 4 * j + t < D::NM ? y[i] : 0.f;
    }
    if (p > 0) reinterpret_cast<float4*>(dx)[j] = make_float4(a[0], a[1], a[2], a[3]);
    reinterpret_cast<float4*>(dy)[j] = make_float4(b[0], b[1], b[2], b[3]);
  }
}
// entries (i, 2p-1) and (i, 2p) of a row-major matrix
template <int N>
__device__ __forceinline__ void nodal_store_columns(float* m, int p, const float (&x)[2 * N - 1],
                                                    const float (&y)[2 * N - 1]) {
  using D = Nodal<N>;
#pragma unroll
  for (int i = 0; i < D::NM; ++i) {
    if (p > 0) m[i * D::LD + 2 * p - 1] = x[i];
    m[i * D::LD + 2 * p] = y[i];
  }
}
// the lane's columns of a row-major matrix's transpose (its rows 2p-1 and 2p)
template <int N>
__device__ __forceinline__ void nodal_load_rows(const float* m, int p, float (&x)[2 * N - 1], float (&y)[2 * N - 1]) {
  using D = Nodal<N>;
  float a[D::LD], b[D::LD];
  nodal_row<D::LD>(m + (p > 0 ? 2 * p - 1 : 0) * D::LD, a);
  nodal_row<D::LD>(m + 2 * p * D::LD, b);
#pragma unroll
  for (int i = 0; i < D::NM; ++i) {
    x[i] = p > 0 ? a[i] : 0.f;
    y[i] = b[i];
  }
}
// (ox, oy) += M (x, y), M row-major in shared memory
template <int N>
__device__ __forceinline__ void nodal_product(const float* m, const float (&x)[2 * N - 1], const float (&y)[2 * N - 1],
                                              float (&ox)[2 * N - 1], float (&oy)[2 * N - 1]) {
  using D = Nodal<N>;
#pragma unroll
  for (int i = 0; i < D::NM; ++i) {
    float row[D::LD];
    nodal_row<D::LD>(m + i * D::LD, row);
#pragma unroll
    for (int j = 0; j < D::NM; ++j) {
      ox[i] = fmaf(row[j], x[j], ox[i]);
      oy[i] = fmaf(row[j], y[j], oy[i]);
    }
  }
}

}  // namespace ts
