// tau at every quadrature point, eq. (3D-tau):
//   tau = [A_i G_ij A_j + C_I nu^2 G_ij G_ij I]^{-1/2}
// computed, as the paper prescribes after eq. (3D-tau), from the eigenpairs
// of the matrix under the root (section 2.2), at every quadrature point
// (section 4).
//
// GB300 mapping: a group of N lanes owns one quadrature point; a warp holds
// floor(32/N) points.  With G = L L^T (3x3 Cholesky) the argument becomes
// M = sum_m C_m C_m + C_I nu^2 (G:G) I, C_m = A(w_m), w_m = sum_i L_im u_i,
// because the convolution matrix is linear in the velocity modes.  In FP32
// (tau32_kernel) the eigenpairs of the real (2N-1)x(2N-1) form of M come from a
// one-sided Jacobi iteration in registers (onesided.cuh); in FP64 by default from
// tau_fx.cu.  tau_kernel is the FP64 form on request: parallel cyclic Jacobi on M in
// shared memory (round-robin ordering, N disjoint rotations per round, one per
// lane), padded with a decoupled dummy row to size 2N.
// tau = V diag(lambda^{-1/2}) V^T is written as a packed upper triangle.
#include <algorithm>

#include "common.cuh"
#include "jacobi.cuh"
#include "kernels.h"
#include "onesided.cuh"

namespace ts {

template <int N>
struct TauLayout {
  using D = Dims<N>;
  static constexpr int NP = D::NP, NM = D::NM, C = D::C;
  static constexpr int LD = NP + 1;
  static constexpr int GPW = 32 / N;
  static constexpr int CM = 0;                       // [3][NM][NM]
  static constexpr int M = CM + 3 * NM * NM;         // [NP][LD]
  static constexpr int V = M + NP * LD;              // [NP][LD]
  static constexpr int W = V + NP * LD;              // [3][C]
  static constexpr int GROUP = ((W + 3 * C) + 1) & ~1;
  static constexpr int WARP = GPW * GROUP + 64;      // + reduction scratch
};

template <typename T, int N>
__global__ void __launch_bounds__(128) tau_kernel(const int4* __restrict__ tets,
                                                  const T* __restrict__ geo,
                                                  const T* __restrict__ y, int64_t n_qp,
                                                  T* __restrict__ tau_out, T nu, T C_I,
                                                  int max_sweeps, T tol2,
                                                  unsigned* __restrict__ n_unconverged,
                                                  float* __restrict__ eig_out) {
  using D = Dims<N>;
  using L = TauLayout<N>;
  constexpr int NP = D::NP, NM = D::NM, C = D::C, LD = L::LD, GPW = L::GPW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / N, k = lane - (lane / N) * N;
  const bool in_group = g < GPW;
  T* wbase = smem + warp * L::WARP;
  T* base = wbase + (in_group ? g : 0) * L::GROUP;
  T* Cm = base + L::CM;
  T* M = base + L::M;
  T* Vv = base + L::V;
  T* w = base + L::W;
  T* red = wbase + GPW * L::GROUP;       // [32] partial sums, [32..] flags

  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t qb = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * GPW; qb < n_qp;
       qb += warps_total * GPW) {
    const int64_t gq = qb + g;
    const bool live = in_group && gq < n_qp;
    const int64_t e = live ? gq >> 2 : 0;
    const int q = (int)(gq & 3);
    T l00 = 0, l10 = 0, l20 = 0, l11 = 0, l21 = 0, l22 = 0, diff = 0;
    if (live) {
      const T* gg = geo + e * GEO_STRIDE + GEO_G;
      T gxx = gg[0], gxy = gg[1], gxz = gg[2], gyy = gg[3], gyz = gg[4], gzz = gg[5];
      l00 = Real<T>::sqrt(gxx);
      l10 = gxy / l00;
      l20 = gxz / l00;
      l11 = Real<T>::sqrt(gyy - l10 * l10);
      l21 = (gyz - l20 * l10) / l11;
      l22 = Real<T>::sqrt(gzz - l20 * l20 - l21 * l21);
      T GG = gxx * gxx + gyy * gyy + gzz * gzz + T(2) * (gxy * gxy + gxz * gxz + gyz * gyz);
      diff = C_I * nu * nu * GG;
      const int4 nd = tets[e];
      const int node[4] = {nd.x, nd.y, nd.z, nd.w};
      // velocity modes at the point, then w_m = sum_i L_im u_i
      for (int c = k; c < C; c += N) {
        T u[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const T lam = (T)qp_bary(q, a);
          const T* ya = y + (int64_t)node[a] * 4 * C;
#pragma unroll
          for (int i = 0; i < 3; ++i) u[i] += lam * ya[i * C + c];
        }
        if (c == 1) u[0] = u[1] = u[2] = 0;
        w[0 * C + c] = l00 * u[0] + l10 * u[1] + l20 * u[2];
        w[1 * C + c] = l11 * u[1] + l21 * u[2];
        w[2 * C + c] = l22 * u[2];
      }
    }
    __syncwarp();
    if (live) {
      for (int t = k; t < 3 * NM * NM; t += N) {
        int m = t / (NM * NM), rs = t - m * NM * NM;
        int r = rs / NM, s = rs - r * NM;
        Cm[t] = conv_entry<T, N>(w + m * C, r, s);
      }
    }
    __syncwarp();
    if (live) {
      for (int t = k; t < NP * NP; t += N) {
        int r = t / NP, s = t - r * NP;
        if (r > s) continue;
        T acc = 0;
        if (r < NM && s < NM) {
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            const T* cr = Cm + m * NM * NM + r * NM;
            const T* cs = Cm + m * NM * NM + s * NM;
            for (int j = 0; j < NM; ++j) acc += cr[j] * cs[j];
          }
          if (r == s) acc += diff;
        } else if (r == s) {
          acc = T(1);                      // decoupled dummy
        }
        M[r * LD + s] = acc;
        M[s * LD + r] = acc;
        Vv[r * LD + s] = (r == s) ? T(1) : T(0);
        Vv[s * LD + r] = (r == s) ? T(1) : T(0);
      }
    }
    __syncwarp();
    // parallel cyclic Jacobi
    const bool converged = jacobi_group<T, N>(M, Vv, k, g, lane, live, red, max_sweeps, tol2);
    if (live && k == 0 && !converged) atomicAdd(n_unconverged, 1u);
    // eigenpairs for the derivative of tau (exact tangent), when asked
    if (live && eig_out) {
      float* eo = eig_out + gq * D::EIG;
      for (int t = k; t < NM * NM; t += N) eo[t] = (float)Vv[(t / NM) * LD + t % NM];
      for (int j = k; j < NM; j += N) eo[NM * NM + j] = (float)M[j * LD + j];
    }
    // tau = V diag(lambda^{-1/2}) V^T, packed upper triangle
    if (live) {
      T* out = tau_out + gq * Dims<N>::NT_PAD;
      for (int t = k; t < NM * NM; t += N) {
        int r = t / NM, s = t - r * NM;
        if (r > s) continue;
        T acc = 0;
        for (int j = 0; j < NM; ++j) {
          T lam = M[j * LD + j];
          acc += Vv[r * LD + j] * Vv[s * LD + j] * Real<T>::rsqrt(lam);
        }
        out[packed_index(r, s, NM)] = acc;
      }
      if (k == 0)
        for (int t = Dims<N>::NT; t < Dims<N>::NT_PAD; ++t) out[t] = T(0);
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// FP32 tau.  A group of N lanes owns a point (GPW points a warp); lane p holds
// two columns of every matrix in registers: 2p-1 and 2p, i.e. Re and Im of
// mode p (lane 0: the mean).  Steps: w_m at the point, the columns of C_m
// (gathered from a zero-padded table of the modes of w_m), M = sum C_m C_m +
// c I with C_m read back row by row from shared memory (a 16-byte broadcast
// feeds eight multiply-adds), Cholesky and one-sided Jacobi (onesided.cuh),
// tau = sum_a f_a f_a^T / |f_a|^3, and 16-byte stores through shared memory.
// The point is scaled by a power of two (sum_m beta_m + sqrt(c) <= 1, beta_m a
// bound of |C_m|), undone exactly at the end.
//
// Bound by FP32 issue: at N = 7 about 10 k instructions a lane and group of
// four points.
template <int N>
struct Tau32Layout {
  static constexpr int NM = 2 * N - 1, C = 2 * N, L = N - 1, GPW = 32 / N;
  static constexpr int LDC = (2 * N + 3) & ~3;        // matrix row, 16-byte multiple
  static constexpr int TW = 3 * N;                    // modes -(N-1) .. 2(N-1), zero beyond N-1 (+ pad)
  static constexpr int T = 0;                         // [3][2][TW] re, im of the modes of w_m
  static constexpr int CM = (3 * 2 * TW + 3) & ~3;    // [3][NM][LDC]; then the scaled f_a [NM][LDC]
  static constexpr int OUTP = CM + NM * LDC;          // packed tau, over the later C_m (N > 1)
  static constexpr int RAW = CM + 3 * NM * LDC + (N == 1 ? 4 : 0);
  // 16-byte reads of the warp's groups fall into different banks: stride 4 mod 32 words
  static constexpr int GROUP = RAW + ((4 - RAW) % 32 + 32) % 32;
  static constexpr int WARP = GPW * GROUP;
  static_assert(OUTP + Dims<N>::NT_PAD <= GROUP, "packed tau fits over the matrices");
};

// a 16-byte aligned row of W floats (W a multiple of 4) to registers
template <int W>
__device__ __forceinline__ void load_row(const float* src, float (&dst)[W]) {
#pragma unroll
  for (int j = 0; j < W / 4; ++j) {
    const float4 v = reinterpret_cast<const float4*>(src)[j];
    dst[4 * j] = v.x;
    dst[4 * j + 1] = v.y;
    dst[4 * j + 2] = v.z;
    dst[4 * j + 3] = v.w;
  }
}

// Blocks an SM asked of the compiler: at N = 5 it takes 111 registers by itself, and 96
// with 5 blocks are faster (187,266 tetrahedra: 0.89 ms against 0.98), at N = 7 128, and 96 with
// 12 words spilled are faster (52,650: 744 us against 767); its own choice (0) is the fastest
// elsewhere.
constexpr int tau32_blocks(int N) { return N == 5 || N == 7 ? 5 : 0; }

template <int N>
__global__ void __launch_bounds__(128, tau32_blocks(N)) tau32_kernel(const int4* __restrict__ tets, const float* __restrict__ geo,
                                                    const float* __restrict__ y, int64_t n_qp,
                                                    float* __restrict__ tau_out, float nu, float C_I,
                                                    unsigned* __restrict__ n_unconverged,
                                                    float* __restrict__ eig_out) {
  using D = Dims<N>;
  using Lt = Tau32Layout<N>;
  constexpr int NM = D::NM, C = D::C, LDC = Lt::LDC, GPW = Lt::GPW, TW = Lt::TW, L = N - 1;
  extern __shared__ __align__(16) float tau32_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / N, p = lane - (lane / N) * N;
  const bool in_group = g < GPW;
  float* base = tau32_smem + warp * Lt::WARP + (in_group ? g : 0) * Lt::GROUP;
  float* tw = base + Lt::T;
  float* cm = base + Lt::CM;
  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t qb = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * GPW; qb < n_qp; qb += warps_total * GPW) {
    const bool live = in_group && qb + g < n_qp;
    const int64_t gq = live ? qb + g : qb;     // idle lanes redo the warp's first point, unstored
    const int64_t e = gq >> 2;
    const int q = (int)(gq & 3);
    // w_m = sum_i L_im u_i for mode p
    float w[3][2];
    float diff;
    {
      const float* gg = geo + e * GEO_STRIDE + GEO_G;
      const float gxx = gg[0], gxy = gg[1], gxz = gg[2], gyy = gg[3], gyz = gg[4], gzz = gg[5];
      const float l00 = sqrtf(gxx), l10 = gxy / l00, l20 = gxz / l00;
      const float l11 = sqrtf(gyy - l10 * l10), l21 = (gyz - l20 * l10) / l11;
      const float l22 = sqrtf(gzz - l20 * l20 - l21 * l21);
      const float GG = gxx * gxx + gyy * gyy + gzz * gzz + 2.f * (gxy * gxy + gxz * gxz + gyz * gyz);
      diff = C_I * nu * nu * GG;
      const int4 nd = tets[e];
      const int node[4] = {nd.x, nd.y, nd.z, nd.w};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float u[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float lam = (float)qp_bary(q, a);
          const float* ya = y + (int64_t)node[a] * 4 * C + 2 * p + h;
#pragma unroll
          for (int i = 0; i < 3; ++i) u[i] += lam * ya[i * C];
        }
        if (p == 0 && h == 1) u[0] = u[1] = u[2] = 0.f;
        w[0][h] = l00 * u[0] + l10 * u[1] + l20 * u[2];
        w[1][h] = l11 * u[1] + l21 * u[2];
        w[2][h] = l22 * u[2];
      }
    }
    // |C_m| <= beta_m = |w_0| + 2 sum |w_n|; 2^-ex scales the point
    float bound = 0.f;
#pragma unroll
    for (int m = 0; m < 3; ++m) bound += (fabsf(w[m][0]) + fabsf(w[m][1])) * (p == 0 ? 1.f : 2.f);
    if constexpr (N > 1) {
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) sum += __shfl_sync(0xffffffffu, bound, (in_group ? g * N : 0) + j);
      bound = sum;
    }
    bound = 1.0001f * (bound + sqrtf(diff));
    const bool finite = bound < 1e37f && bound > 1e-37f;
    int ex = 0;
    if (finite) frexpf(bound, &ex);
    const float sc = ldexpf(1.f, -ex);
    // a point that is not finite takes a harmless matrix here and NaN at the end: the
    // rotations mix in neighbouring lanes' values times zero
    const float cd = finite ? diff * sc * sc : 0.5f;
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      float* tr = tw + m * 2 * TW + L;        // mode k at tr[k], im at tr[TW + k]
      const float re = finite ? w[m][0] * sc : 0.f, im = finite ? w[m][1] * sc : 0.f;
      if (in_group) {
        tr[p] = re;
        tr[TW + p] = im;
        if (p > 0) {
          tr[-p] = re;
          tr[TW - p] = -im;
          tr[L + p] = 0.f;
          tr[TW + L + p] = 0.f;
        }
      }
    }
    __syncwarp();
    float x[NM], yy[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) x[i] = yy[i] = 0.f;
    // the lane's columns of C_m (Re p, Im p; lane 0: the mean) to shared memory
    float* colx = cm + (2 * p - 1) * LDC;
    float* coly = cm + (2 * p) * LDC;
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {
      const float* tr = tw + m * 2 * TW + L;
      const float* ti = tr + TW;
      float cx[NM], cy[NM];
      constexpr float S2 = Real<float>::SQRT2;
      cx[0] = S2 * tr[p];
      cy[0] = p == 0 ? tr[0] : S2 * ti[p];
#pragma unroll
      for (int k = 1; k < N; ++k) {
        const float pl = tr[k - p], ph = tr[k + p], ql = ti[k - p], qh = ti[k + p];
        cx[2 * k - 1] = pl + ph;
        cx[2 * k] = ql + qh;
        cy[2 * k - 1] = p == 0 ? S2 * pl : qh - ql;
        cy[2 * k] = p == 0 ? S2 * ql : pl - ph;
      }
      if (in_group) {
        float* dx = colx + m * NM * LDC;
        float* dy = coly + m * NM * LDC;
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          if (p > 0) dx[i] = cx[i];
          dy[i] = cy[i];
        }
      }
      __syncwarp();
      // M's columns: row i of the symmetric C_m is a 16-byte broadcast stream
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        float row[LDC], sx = x[i], sy = yy[i];
        load_row<LDC>(cm + (m * NM + i) * LDC, row);
#pragma unroll
        for (int j = 0; j < NM; ++j) {
          sx = fmaf(row[j], cx[j], sx);
          sy = fmaf(row[j], cy[j], sy);
        }
        x[i] = sx;
        yy[i] = sy;
      }
    }
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      x[i] += i == 2 * p - 1 ? cd : 0.f;
      yy[i] += i == 2 * p ? cd : 0.f;
      if (p == 0 || !in_group) x[i] = 0.f;
      if (!in_group) yy[i] = 0.f;
    }
    __syncwarp();                       // all lanes have read C_m
    const float least =
        cholesky_columns<N, LDC, (N > 7)>(x, yy, p, in_group, in_group ? g * N : 0, fmaxf(cd, 1e-30f), cm);
    // a pivot that rounding took to zero or below: FP32 does not resolve the smallest
    // eigenvalue, the factor means nothing (its columns may overflow) and the point is NaN
    const bool resolved = least > 0.f;
    if (__any_sync(0xffffffffu, !resolved)) {
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        x[i] = resolved ? x[i] : in_group && i == 2 * p - 1 ? 1.f : 0.f;
        yy[i] = resolved ? yy[i] : in_group && i == 2 * p ? 1.f : 0.f;
      }
    }
    __syncwarp();
    const bool conv = onesided_jacobi<N>(x, yy, p, lane, 1e-8f);
    {
      const unsigned bad = __ballot_sync(0xffffffffu, live && !conv);
      const unsigned mine = N == 32 ? ~0u : ((1u << N) - 1u) << (in_group ? g * N : 0);
      if (live && p == 0 && (bad & mine)) atomicAdd(n_unconverged, 1u);
    }
    float ax = 0.f, ay = 0.f;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      ax = fmaf(x[i], x[i], ax);
      ay = fmaf(yy[i], yy[i], ay);
    }
    // eigenpairs for the derivative of tau (exact tangent), when asked: the
    // lane's two vectors are columns 2p-1 and 2p of the cache
    if (live && eig_out) {
      float* eo = eig_out + gq * D::EIG;
      const float back = finite && resolved ? ldexpf(1.f, 2 * ex) : __int_as_float(0x7fc00000);
      const float ix = rsqrt_newton(ax), iy = rsqrt_newton(ay);
      if (p > 0) {
#pragma unroll
        for (int i = 0; i < NM; ++i) eo[i * NM + 2 * p - 1] = x[i] * ix;
        eo[NM * NM + 2 * p - 1] = ax * back;
      }
#pragma unroll
      for (int i = 0; i < NM; ++i) eo[i * NM + 2 * p] = yy[i] * iy;
      eo[NM * NM + 2 * p] = ay * back;
    }
    // h_a = f_a / |f_a|^{3/2} (so that tau = sum_a h_a h_a^T), stored one float
    // off so that a lane's two entries are an aligned pair
    __syncwarp();
    {
      const float rx = rsqrt_newton(ax), ry = rsqrt_newton(ay);
      const float hx = rx * sqrtf(rx), hy = ry * sqrtf(ry);
      if (in_group) {
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          if (p > 0) colx[i + 1] = x[i] * hx;
          coly[i + 1] = yy[i] * hy;
        }
        if (p == 0)
          for (int a = 0; a < NM; ++a) cm[a * LDC] = 0.f;
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NM; ++i) x[i] = yy[i] = 0.f;
#pragma unroll 1
    for (int a = 0; a < NM; ++a) {
      const float* ha = cm + a * LDC;
      const float2 own = *reinterpret_cast<const float2*>(ha + 2 * p);   // entries 2p-1 and 2p
      float row[LDC];
      load_row<LDC>(ha, row);
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        x[i] = fmaf(row[i + 1], own.x, x[i]);
        yy[i] = fmaf(row[i + 1], own.y, yy[i]);
      }
    }
    // packed upper triangle through shared memory
    float* op = base + Lt::OUTP;
    const float un = finite && resolved ? sc : __int_as_float(0x7fc00000);
    __syncwarp();
    if (in_group) {
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        if (p > 0 && i <= 2 * p - 1) op[packed_index(i, 2 * p - 1, NM)] = x[i] * un;
        if (i <= 2 * p) op[packed_index(i, 2 * p, NM)] = yy[i] * un;
      }
      if (p == 0)
        for (int t = D::NT; t < D::NT_PAD; ++t) op[t] = 0.f;
    }
    __syncwarp();
    if (live) {
      float4* out = reinterpret_cast<float4*>(tau_out + gq * D::NT_PAD);
      for (int t = p; t < D::NT_PAD / 4; t += N) out[t] = *reinterpret_cast<const float4*>(op + 4 * t);
    }
    __syncwarp();
  }
}

template <int N>
size_t tau32_smem(int* warps) {
  using L = Tau32Layout<N>;
  *warps = 4;
  while (*warps > 1 && (size_t)*warps * L::WARP * sizeof(float) > 100 * 1024) *warps >>= 1;
  return (size_t)*warps * L::WARP * sizeof(float);
}

template <typename T, int N>
int launch_tau(const int4* tets, const T* geo, const T* y, int64_t n_elem, T* tau_out, T nu,
               T C_I, unsigned* n_unconverged, cudaStream_t st, float* eig_out) {
  const int64_t n_qp = n_elem * 4, groups = (n_qp + 32 / N - 1) / (32 / N);
  if constexpr (sizeof(T) == 4) {
    int warps;
    const size_t smem = tau32_smem<N>(&warps);
    if (cudaFuncSetAttribute(tau32_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return -2;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((groups + warps - 1) / warps, 152 * 64));
    count_launches(1);
    tau32_kernel<N><<<(int)blocks, warps * 32, smem, st>>>(tets, geo, y, n_qp, tau_out, nu, C_I, n_unconverged, eig_out);
  } else {
    using L = TauLayout<N>;
    const int warps = 4;
    const size_t smem = (size_t)warps * L::WARP * sizeof(T);
    cudaFuncSetAttribute(tau_kernel<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((groups + warps - 1) / warps, 152 * 64));
    count_launches(1);
    tau_kernel<T, N><<<(int)blocks, warps * 32, smem, st>>>(tets, geo, y, n_qp, tau_out, nu, C_I,
                                                            20, T(1e-28), n_unconverged, eig_out);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

// Loads the FP32 tau kernel into the current device's context without launching
// it (with lazy module loading a kernel is otherwise loaded at its first launch).
template <typename T, int N>
int preload_tau() {
  static_assert(sizeof(T) == 4, "FP32 only");
  int warps;
  const size_t smem = tau32_smem<N>(&warps);
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, tau32_kernel<N>) != cudaSuccess) return -2;
  return cudaFuncSetAttribute(tau32_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) ==
                 cudaSuccess ? 0 : -2;
}

// ---------------------------------------------------------------------------
// FP64 tau from FP32 eigenvectors.  The FP32 Jacobi gives V32 with
// V32^T M V32 diagonal to about 1e-7 ||M||.  In FP64: one Newton-Schulz step
// (two) make V orthonormal to FP64 rounding, B = V^T M V, and f(B) = B^{-1/2} is
// expanded to second order around diag(B) with the Daleckii-Krein formulas
// (Frechet derivatives of a matrix function at a diagonal matrix are
// Hadamard-type sums with the divided differences of f).  For f = l^{-1/2}
// with s = sqrt(l) the divided differences have cancellation-free forms
//   f[a,b]   = -1 / (s_a s_b (s_a + s_b))
//   f[a,b,c] = (s_a + s_b + s_c) / (s_a s_b s_c (s_a+s_b)(s_b+s_c)(s_a+s_c)),
// which gives, with X_ik = E_ik / (s_i s_k (s_i + s_k)) and E = offdiag(B),
//   Z = diag(1/s) - X + X D_s X + (X D_{s^2} X) ./ (s_i + s_j),
// tau = V Z V^T, error third order in E / (s_i s_j).
//
// LISTED: the points that the fixed-point form leaves out (tau_fx.cu), mostly with large
// condition numbers.  E, 1e-7 of the largest eigenvalue, is not small there against the
// smallest ones, so Jacobi sweeps in FP64 on B (two or three: it starts nearly diagonal)
// reduce it first; M is scaled to FP32's range by a power of four, and eigenvalues are at
// least c = C_I nu^2 G:G, their lower bound.  The sweeps stop early or late with equal
// eigenvalues, where the expansion needs no more.  Bound by the FP64 pipe.
template <int N>
struct PolishLayout {
  static constexpr int NP = 2 * N, NM = 2 * N - 1, C = 2 * N, LD = NP + 1;
  static constexpr int GPW = 32 / N;
  // in doubles
  static constexpr int CM = 0;                       // [3][NM][NM] scratch
  static constexpr int M64 = CM + 3 * NM * NM;       // [NP][LD]
  static constexpr int V64 = M64 + NP * LD;          // [NP][LD]
  static constexpr int W = V64 + NP * LD;            // [3][C]
  static constexpr int F32 = W + 3 * C;              // start of the float part
  static constexpr int GROUP = F32 + NP * LD;        // 2 [NP][LD] float matrices = NP*LD doubles
  static constexpr int WARP = GPW * GROUP + 64 + 32; // + double and float reduction scratch
};

template <int N, bool LISTED>
__global__ void __launch_bounds__(LISTED ? 256 : 128) tau_polish_kernel(const int4* __restrict__ tets,
                                                         const double* __restrict__ geo,
                                                         const double* __restrict__ y,
                                                         int64_t n_qp, double* __restrict__ tau_out,
                                                         double nu, double C_I,
                                                         unsigned* __restrict__ n_unconverged,
                                                         float* __restrict__ eig_out,
                                                         const unsigned* __restrict__ hard) {
  using L = PolishLayout<N>;
  constexpr int NP = L::NP, NM = L::NM, C = L::C, LD = L::LD, GPW = L::GPW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* smem = reinterpret_cast<double*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / N, k = lane - (lane / N) * N;
  const bool in_group = g < GPW;
  double* wbase = smem + warp * L::WARP;
  double* base = wbase + (in_group ? g : 0) * L::GROUP;
  double* Cm = base + L::CM;
  double* M = base + L::M64;
  double* Vd = base + L::V64;
  double* w = base + L::W;
  float* Mf = reinterpret_cast<float*>(base + L::F32);
  float* Vf = Mf + NP * LD;
  double* red_d = wbase + GPW * L::GROUP;
  float* red_f = reinterpret_cast<float*>(red_d + 64);

  if (LISTED) n_qp = hard[0];
  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t qb = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * GPW; qb < n_qp;
       qb += warps_total * GPW) {
    const bool live = in_group && qb + g < n_qp;
    const int64_t gq = LISTED ? (live ? hard[HARD_LIST + qb + g] : 0) : qb + g;
    const int64_t e = live ? gq >> 2 : 0;
    const int q = (int)(gq & 3);
    double diff = 0;
    if (live) {
      const double* gg = geo + e * GEO_STRIDE + GEO_G;
      const double gxx = gg[0], gxy = gg[1], gxz = gg[2], gyy = gg[3], gyz = gg[4], gzz = gg[5];
      const double l00 = sqrt(gxx), l10 = gxy / l00, l20 = gxz / l00;
      const double l11 = sqrt(gyy - l10 * l10), l21 = (gyz - l20 * l10) / l11;
      const double l22 = sqrt(gzz - l20 * l20 - l21 * l21);
      const double GG = gxx * gxx + gyy * gyy + gzz * gzz + 2.0 * (gxy * gxy + gxz * gxz + gyz * gyz);
      diff = C_I * nu * nu * GG;
      const int4 nd = tets[e];
      const int node[4] = {nd.x, nd.y, nd.z, nd.w};
      for (int c = k; c < C; c += N) {
        double u[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const double lam = qp_bary(q, a);
          const double* ya = y + (int64_t)node[a] * 4 * C;
#pragma unroll
          for (int i = 0; i < 3; ++i) u[i] += lam * ya[i * C + c];
        }
        if (c == 1) u[0] = u[1] = u[2] = 0;
        w[0 * C + c] = l00 * u[0] + l10 * u[1] + l20 * u[2];
        w[1 * C + c] = l11 * u[1] + l21 * u[2];
        w[2 * C + c] = l22 * u[2];
      }
    }
    __syncwarp();
    if (live)
      for (int t = k; t < 3 * NM * NM; t += N) {
        const int m = t / (NM * NM), rs = t - m * NM * NM;
        const int r = rs / NM, s = rs - r * NM;
        Cm[t] = conv_entry<double, N>(w + m * C, r, s);
      }
    __syncwarp();
    if (live)
      for (int t = k; t < NP * NP; t += N) {
        const int r = t / NP, s = t - r * NP;
        if (r > s) continue;
        double acc = 0;
        if (r < NM && s < NM) {
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            const double* cr = Cm + m * NM * NM + r * NM;
            const double* cs = Cm + m * NM * NM + s * NM;
            for (int j = 0; j < NM; ++j) acc += cr[j] * cs[j];
          }
          if (r == s) acc += diff;
        } else if (r == s) {
          acc = 1.0;   // decoupled dummy
        }
        M[r * LD + s] = acc;
        M[s * LD + r] = acc;
        if (!LISTED) {
          Mf[r * LD + s] = (float)acc;
          Mf[s * LD + r] = (float)acc;
        }
        Vf[r * LD + s] = (r == s) ? 1.f : 0.f;
        Vf[s * LD + r] = (r == s) ? 1.f : 0.f;
      }
    __syncwarp();
    if (LISTED) {
      if (live) {
        double top = 0;
        for (int i = 0; i < NM; ++i) top = fmax(top, M[i * LD + i]);
        int ex;
        frexp(top, &ex);
        const double sc = ldexp(1.0, -ex);
        for (int t = k; t < NP * NP; t += N) {
          const int r = t / NP, s = t - r * NP;
          Mf[r * LD + s] = r < NM && s < NM ? (float)(M[r * LD + s] * sc) : r == s ? 1.f : 0.f;
        }
      }
      __syncwarp();
    }
    const bool conv32 = jacobi_group<float, N>(Mf, Vf, k, g, lane, live, red_f, 12, 1e-12f);
    if (!LISTED && live && k == 0 && !conv32) atomicAdd(n_unconverged, 1u);
    // V in FP64, re-orthonormalised by two Newton-Schulz steps V <- V (3I - V^T V) / 2
    // (the FP32 eigenvectors are orthonormal only to FP32 rounding)
    if (live)
      for (int t = k; t < NP * NP; t += N) Vd[(t / NP) * LD + t % NP] = (double)Vf[(t / NP) * LD + t % NP];
    __syncwarp();
    for (int it = 0; it < 2; ++it) {
      if (live)
        for (int t = k; t < NM * NM; t += N) {
          const int r = t / NM, s = t - r * NM;
          double acc = 0;
          for (int i = 0; i < NM; ++i) acc += Vd[i * LD + r] * Vd[i * LD + s];
          Cm[t] = ((r == s) ? 3.0 : 0.0) - acc;      // 3I - V^T V
        }
      __syncwarp();
      if (live)
        for (int t = k; t < NM * NM; t += N) {
          const int r = t / NM, s = t - r * NM;
          double acc = 0;
          for (int j = 0; j < NM; ++j) acc += Vd[r * LD + j] * Cm[j * NM + s];
          Cm[NM * NM + t] = 0.5 * acc;
        }
      __syncwarp();
      if (live)
        for (int t = k; t < NM * NM; t += N) Vd[(t / NM) * LD + t % NM] = Cm[NM * NM + t];
      __syncwarp();
    }
    // P = M V, then B = V^T M V over the NM x NM block of M (dummy row/column unchanged)
    if (live)
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s = t - r * NM;
        double acc = 0;
        for (int j = 0; j < NM; ++j) acc += M[r * LD + j] * Vd[j * LD + s];
        Cm[t] = acc;
      }
    __syncwarp();
    if (live)
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s = t - r * NM;
        if (r > s) continue;
        double acc = 0;
        for (int i = 0; i < NM; ++i) acc += Vd[i * LD + r] * Cm[i * NM + s];
        M[r * LD + s] = acc;
        M[s * LD + r] = acc;
      }
    __syncwarp();
    if (LISTED) {
      jacobi_group<double, N>(M, Vd, k, g, lane, live, red_d, 8, 1e-36);
      if (live)
        for (int i = k; i < NM; i += N) {
          // below half of its bound: FP64 does not resolve it
          if (!(M[i * LD + i] > 0.5 * diff)) atomicAdd(n_unconverged, 1u);
          M[i * LD + i] = fmax(M[i * LD + i], diff);
        }
      __syncwarp();
    }
    if (live && eig_out) {
      float* eo = eig_out + gq * Dims<N>::EIG;
      for (int t = k; t < NM * NM; t += N) eo[t] = (float)Vd[(t / NM) * LD + t % NM];
      for (int j = k; j < NM; j += N) eo[NM * NM + j] = (float)M[j * LD + j];
    }
    // s = sqrt(diag B) once per point (reusing the w rows: 3C >= 2 NM)
    double* sq = w;          // [NM] sqrt(b_ii)
    double* sq2 = w + NM;    // [NM] b_ii
    if (live)
      for (int i = k; i < NM; i += N) {
        sq[i] = sqrt(M[i * LD + i]);
        sq2[i] = M[i * LD + i];
      }
    __syncwarp();
    // X_ik = E_ik / (s_i s_k (s_i + s_k)), E = offdiag B
    if (live)
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s = t - r * NM;
        const double sr = sq[r], ss = sq[s];
        Cm[t] = (r == s) ? 0.0 : M[r * LD + s] / (sr * ss * (sr + ss));
      }
    __syncwarp();
    // Z = diag(1/s) - X + sum_k X_ik X_kj (s_k + s_k^2 / (s_i + s_j))   (second order)
    if (live)
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s = t - r * NM;
        const double sr = sq[r], ss = sq[s];
        const double inv_rs = 1.0 / (sr + ss);
        double acc = 0;
        for (int j = 0; j < NM; ++j) acc += Cm[r * NM + j] * Cm[j * NM + s] * (sq[j] + sq2[j] * inv_rs);
        Cm[NM * NM + t] = ((r == s) ? 1.0 / sr : 0.0) - Cm[t] + acc;
      }
    __syncwarp();
    // Q = Z V^T in the third scratch slot
    if (live)
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s = t - r * NM;
        double acc = 0;
        for (int j = 0; j < NM; ++j) acc += Cm[NM * NM + r * NM + j] * Vd[s * LD + j];
        Cm[2 * NM * NM + t] = acc;
      }
    __syncwarp();
    if (live) {
      double* out = tau_out + gq * Dims<N>::NT_PAD;
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s = t - r * NM;
        if (r > s) continue;
        double acc = 0;
        for (int j = 0; j < NM; ++j) acc += Vd[r * LD + j] * Cm[2 * NM * NM + j * NM + s];
        out[packed_index(r, s, NM)] = acc;
      }
      if (k == 0)
        for (int t = Dims<N>::NT; t < Dims<N>::NT_PAD; ++t) out[t] = 0.0;
    }
    __syncwarp();
  }
}

template <int N>
int launch_tau_polish(const int4* tets, const double* geo, const double* y, int64_t n_elem,
                      double* tau_out, double nu, double C_I, unsigned* n_unconverged,
                      cudaStream_t st, float* eig_out) {
  using L = PolishLayout<N>;
  int warps = 4;
  while (warps > 1 && (size_t)warps * L::WARP * sizeof(double) > 200 * 1024) --warps;
  const size_t smem = (size_t)warps * L::WARP * sizeof(double);
  if (smem > 227 * 1024) return -6;
  cudaFuncSetAttribute(tau_polish_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int64_t n_qp = n_elem * 4;
  const int64_t groups = (n_qp + L::GPW - 1) / L::GPW;
  int64_t blocks = (groups + warps - 1) / warps;
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (blocks < 1) blocks = 1;
  count_launches(1);
  tau_polish_kernel<N, false><<<(int)blocks, warps * 32, smem, st>>>(tets, geo, y, n_qp, tau_out, nu, C_I,
                                                                     n_unconverged, eig_out, nullptr);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

// One block an SM: the list is empty for most flows, and a full one keeps the FP64 pipe
// busy with the 5 warps (N = 7) that fit.
template <int N>
int launch_tau_hard(const int4* tets, const double* geo, const double* y, const unsigned* hard, double* tau_out,
                    double nu, double C_I, unsigned* n_unconverged, cudaStream_t st, float* eig_out) {
  using L = PolishLayout<N>;
  int warps = 8;
  while (warps > 1 && (size_t)warps * L::WARP * sizeof(double) > 200 * 1024) --warps;
  const size_t smem = (size_t)warps * L::WARP * sizeof(double);
  static_assert(L::WARP * sizeof(double) <= 227 * 1024, "a warp's shared memory");
  if (cudaFuncSetAttribute(tau_polish_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return -2;
  count_launches(1);
  tau_polish_kernel<N, true><<<152, warps * 32, smem, st>>>(tets, geo, y, 0, tau_out, nu, C_I, n_unconverged, eig_out,
                                                            hard);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

#define TS_INST_POLISH(T, N)                                                                  \
  template int launch_tau_polish<N>(const int4*, const double*, const double*, int64_t,      \
                                    double*, double, double, unsigned*, cudaStream_t, float*);
TS_FOR_EACH_N(TS_INST_POLISH, double)
#define TS_INST_HARD(T, N)                                                                     \
  template int launch_tau_hard<N>(const int4*, const double*, const double*, const unsigned*, double*, double, double, \
                                  unsigned*, cudaStream_t, float*);
TS_FOR_EACH_N(TS_INST_HARD, double)


// ---------------------------------------------------------------------------
// Backflow stabilisation (section 2.6): at every point of a Neumann face,
// |A_n|_- = (A_n - |A_n|)/2 with A_n = A_i n_i = A(u . n), taken through the
// eigenpairs of A_n (remark 1 of section 2.6), stored like tau as a packed
// upper triangle in the orthonormal real basis.  Face points: the 3-point
// degree-2 rule (barycentric 2/3, 1/6, 1/6), weights area/3.
__host__ __device__ constexpr double face_bary(int g, int b) { return g == b ? 2.0 / 3.0 : 1.0 / 6.0; }

template <int N>
struct BackflowLayout {
  static constexpr int NP = 2 * N, C = 2 * N, LD = NP + 1, GPW = 32 / N;
  static constexpr int M = 0, V = M + NP * LD, W = V + NP * LD;
  static constexpr int GROUP = (W + C + 1) & ~1;
  static constexpr int WARP = GPW * GROUP + 64;
};

template <typename T, int N>
__global__ void __launch_bounds__(128) backflow_neg_kernel(const int32_t* __restrict__ faces,
                                                           const T* __restrict__ normals,
                                                           const T* __restrict__ y, int64_t n_pts,
                                                           T* __restrict__ bneg) {
  using L = BackflowLayout<N>;
  constexpr int NP = L::NP, NM = 2 * N - 1, C = L::C, LD = L::LD, GPW = L::GPW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / N, k = lane - (lane / N) * N;
  const bool in_group = g < GPW;
  T* wbase = smem + warp * L::WARP;
  T* base = wbase + (in_group ? g : 0) * L::GROUP;
  T* M = base + L::M;
  T* Vv = base + L::V;
  T* w = base + L::W;
  T* red = wbase + GPW * L::GROUP;
  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t pb = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * GPW; pb < n_pts;
       pb += warps_total * GPW) {
    const int64_t gp = pb + g;
    const bool live = in_group && gp < n_pts;
    const int64_t f = live ? gp / 3 : 0;
    const int gq = (int)(gp - (gp / 3) * 3);
    if (live) {
      const T nx = normals[f * 3], ny = normals[f * 3 + 1], nz = normals[f * 3 + 2];
      for (int c = k; c < C; c += N) {
        T un = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const T* yb = y + (int64_t)faces[f * 3 + b] * 4 * C;
          un += (T)face_bary(gq, b) * (nx * yb[c] + ny * yb[C + c] + nz * yb[2 * C + c]);
        }
        w[c] = (c == 1) ? T(0) : un;
      }
    }
    __syncwarp();
    if (live)
      for (int t = k; t < NP * NP; t += N) {
        const int r = t / NP, s2 = t - r * NP;
        T val;
        if (r < NM && s2 < NM) val = conv_entry<T, N>(w, r, s2);
        else val = (r == s2) ? T(1) : T(0);   // decoupled dummy
        M[r * LD + s2] = val;
        Vv[r * LD + s2] = (r == s2) ? T(1) : T(0);
      }
    __syncwarp();
    jacobi_group<T, N>(M, Vv, k, g, lane, live, red, sizeof(T) == 4 ? 12 : 20,
                       sizeof(T) == 4 ? T(1e-12) : T(1e-28));
    if (live) {
      T* out = bneg + gp * Dims<N>::NT_PAD;
      for (int t = k; t < NM * NM; t += N) {
        const int r = t / NM, s2 = t - r * NM;
        if (r > s2) continue;
        T acc = 0;
        for (int j = 0; j < NM; ++j) {
          const T lam = M[j * LD + j];
          if (lam < T(0)) acc += Vv[r * LD + j] * Vv[s2 * LD + j] * lam;
        }
        out[packed_index(r, s2, NM)] = acc;
      }
      if (k == 0)
        for (int t = Dims<N>::NT; t < Dims<N>::NT_PAD; ++t) out[t] = T(0);
    }
    __syncwarp();
  }
}

// out[A][i] += coef * sum_g (area/3) N_A(g) |A_n|_- u_i(g), one thread per (face, point, i)
template <typename T, int N>
__global__ void backflow_apply_kernel(const int32_t* __restrict__ faces, const T* __restrict__ area,
                                      const T* __restrict__ bneg, const T* __restrict__ v,
                                      const uint8_t* __restrict__ dmask, int mask_input, T coef,
                                      T* __restrict__ out, int64_t n_faces) {
  constexpr int C = 2 * N, NM = 2 * N - 1, NTP = Dims<N>::NT_PAD;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_faces * 9;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = t / 9;
    const int gi = (int)(t - f * 9), g = gi / 3, i = gi - (gi / 3) * 3;
    int nb[3];
    T u[C];
#pragma unroll
    for (int c = 0; c < C; ++c) u[c] = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      nb[b] = faces[f * 3 + b];
      if (mask_input && dmask[nb[b]]) continue;
      const T* vb = v + (int64_t)nb[b] * 4 * C + i * C;
#pragma unroll
      for (int c = 0; c < C; ++c) u[c] += (T)face_bary(g, b) * vb[c];
    }
    u[1] = 0;
    const T* B = bneg + (f * 3 + g) * NTP;
    T z[C];
#pragma unroll
    for (int r = 0; r < NM; ++r) {
      T acc = 0;
#pragma unroll
      for (int kk = 0; kk < NM; ++kk) {
        const int a = r < kk ? r : kk, b = r < kk ? kk : r;
        T bv = B[packed_index(a, b, NM)];
        if (r == 0 && kk > 0) bv *= Real<T>::SQRT2;
        if (r > 0 && kk == 0) bv *= Real<T>::INV_SQRT2;
        acc += bv * u[stor_of(kk)];
      }
      z[stor_of(r)] = acc;
    }
    const T wq = coef * area[f] / T(3);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (dmask[nb[b]]) continue;
      T* dst = out + (int64_t)nb[b] * 4 * C + i * C;
      const T s = wq * (T)face_bary(g, b);
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (c != 1) atomicAdd(dst + c, s * z[c]);
    }
  }
}

template <typename T, int N>
int launch_backflow(const int32_t* faces, const T* normals, const T* area, int64_t n_faces,
                    const T* y_for_matrix, T* bneg, const T* v, const uint8_t* dmask, int mask_input,
                    T coef, T* out, cudaStream_t st) {
  if (n_faces <= 0) return 0;
  if (y_for_matrix) {
    using L = BackflowLayout<N>;
    const int warps = 4;
    const size_t smem = (size_t)warps * L::WARP * sizeof(T);
    cudaFuncSetAttribute(backflow_neg_kernel<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t n_pts = n_faces * 3;
    int64_t blocks = ((n_pts + L::GPW - 1) / L::GPW + warps - 1) / warps;
    if (blocks > 152 * 32) blocks = 152 * 32;
    count_launches(1);
    backflow_neg_kernel<T, N><<<(int)blocks, warps * 32, smem, st>>>(faces, normals, y_for_matrix, n_pts, bneg);
  }
  int64_t blocks = (n_faces * 9 + 127) / 128;
  if (blocks > 152 * 16) blocks = 152 * 16;
  count_launches(1);
  backflow_apply_kernel<T, N><<<(int)blocks, 128, 0, st>>>(faces, area, bneg, v, dmask, mask_input, coef, out, n_faces);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

#define TS_INST_BACKFLOW(T, N)                                                                 \
  template int launch_backflow<T, N>(const int32_t*, const T*, const T*, int64_t, const T*, T*, \
                                     const T*, const uint8_t*, int, T, T*, cudaStream_t);
TS_FOR_EACH_N(TS_INST_BACKFLOW, float)
TS_FOR_EACH_N(TS_INST_BACKFLOW, double)

#define TS_INST_TAU(T, N)                                                                 \
  template int launch_tau<T, N>(const int4*, const T*, const T*, int64_t, T*, T, T,       \
                                unsigned*, cudaStream_t, float*);
#define TS_INST_PRELOAD_TAU(T, N) template int preload_tau<T, N>();
TS_FOR_EACH_N(TS_INST_PRELOAD_TAU, float)
TS_FOR_EACH_N(TS_INST_TAU, float)
TS_FOR_EACH_N(TS_INST_TAU, double)

}  // namespace ts
