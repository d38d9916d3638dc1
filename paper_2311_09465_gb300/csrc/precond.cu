// Nodal block-Jacobi preconditioner of the tangent H (eq. tangent, eq. K_mat,
// section 2.4): for every node A the 8N x 8N block H_AA that couples the node's
// own unknowns (3 velocity fields and pressure, modes 0..N-1, re/im), summed
// over the elements around the node, then inverted.
//
// With A and tau frozen (eq. K_mat), per element, quadrature point q (weight
// w = V/4) and local node a, in the real storage coordinates of a mode vector:
//   S_qa = lambda_qa Omega + Conv(beta_qa),  W_qa = -lambda_qa Omega + Conv(beta_qa),
//   beta_qa = sum_j dN_a/dx_j u0_j(q)   (so Conv(beta_qa) = A_j dN_a/dx_j)
//   K_aa += w rho (lambda_qa S_qa + W_qa tau_q S_qa) + mu V |grad N_a|^2 I + m_aa I
//   G_i  += -V/4 dN_a/dx_i I + w dN_a/dx_i W_qa tau_q        (LS part: FROZEN)
//   D_j  +=  w dN_a/dx_j I   + w dN_a/dx_j tau_q S_qa         (LS part: FROZEN)
//   L    += (w / rho) |grad N_a|^2 tau_q
// with m_aa = c1 rho/dt V/10 (the consistent mass, section 2.5.3) and, on a
// resistance outlet, R (int N_A n_i)(int N_A n_j) per mode.  K is the same
// for the three velocity fields; the paper's variant drops the LS parts of G
// and D (section 2.5.2).  The derivative of A_j (LIN_A) is not part of the
// block: the blocks of a LIN_A problem are those of the frozen tangent.
//
// Conv(beta) is the truncated convolution of eq. (phi-def) written on the
// storage coordinates (x_0, Re x_n, Im x_n): with y_m = sum_n beta_{m-n} x_n
// and x_{-n} = conj(x_n), the column of Re x_n (n >= 1) is beta_{m-n} +
// beta_{m+n} and the column of Im x_n is i (beta_{m-n} - beta_{m+n}).
//
// GB300 mapping: one warp per node gathers its (element, local node) pairs
// from a node-to-element list, so each block is summed in shared memory and
// written once (no atomics, deterministic), and inverted before it leaves the
// chip: for N <= 7 register tiles and the Schur complement of the velocity
// fields (nodal_block_kernel), above that in place by Gauss-Jordan with partial
// pivoting (block_diag_kernel).  Stored column-major;
// the apply kernel (one warp per node, coalesced column reads) multiplies it
// with the node's slice of a Krylov vector.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "nodal.cuh"

namespace ts {

template <int N>
struct BlockLayout {
  static constexpr int C = 2 * N;
  static constexpr int NB = 4 * C;              // block size (unknowns per node)
  static constexpr int CC = C * C;
  // per-warp workspace (floats): the final block F [NB][NB] (its first 5 CC
  // also serve as per-point temporaries while summing), the accumulators
  // K, G_0..2, D_0..2, L [8][C][C], and small per-element arrays
  static constexpr int F = 0;
  static constexpr int TAU = 0, SM = CC, WM = 2 * CC, XM = 3 * CC, YM = 4 * CC;
  static constexpr int ACC = NB * NB;           // K at ACC, G_i at ACC+(1+i)CC, D_j at ACC+(4+j)CC, L at ACC+7CC
  static constexpr int GEO = ACC + 8 * CC;      // 20 (+4)
  static constexpr int UN = GEO + 24;           // u0 velocity at the 4 nodes [4][3][C]
  static constexpr int GAM = UN + 12 * C;       // gamma_b = sum_j dN_a/dx_j u0_bj [4][C]
  static constexpr int BET = GAM + 4 * C;       // beta_q [C]
  static constexpr int PIV = BET + C;           // pivot rows [NB]
  static constexpr int WARP = (PIV + NB + 3) & ~3;
};

// (re, im) of mode k of a conjugate-symmetric vector stored as (x_0, re/im of 1..N-1)
template <int N>
__device__ __forceinline__ float2 mode_of(const float* b, int k) {
  if (k <= -N || k >= N) return make_float2(0.f, 0.f);
  if (k >= 0) return make_float2(b[2 * k], k == 0 ? 0.f : b[2 * k + 1]);
  return make_float2(b[-2 * k], -b[-2 * k + 1]);
}

// entry (row r, column s) of Conv(beta) on storage coordinates
template <int N>
__device__ __forceinline__ float conv_entry(const float* beta, int r, int s) {
  if (s == 1) return 0.f;
  const int m = r >> 1, n = s >> 1;
  const bool im_row = r & 1;
  if (n == 0) {
    const float2 b = mode_of<N>(beta, m);
    return im_row ? b.y : b.x;
  }
  const float2 lo = mode_of<N>(beta, m - n), hi = mode_of<N>(beta, m + n);
  if (!(s & 1)) return im_row ? lo.y + hi.y : lo.x + hi.x;
  return im_row ? lo.x - hi.x : hi.y - lo.y;
}

// Omega on storage coordinates: (Omega x)_{2n} = -n w x_{2n+1}, (Omega x)_{2n+1} = n w x_{2n}
__device__ __forceinline__ float omega_entry(int r, int s, float omega) {
  const int n = r >> 1;
  if (n == 0 || (r ^ 1) != s) return 0.f;
  return (r & 1) ? n * omega : -n * omega;
}

// C = A B for C x C matrices in shared memory (row-major), lanes over outputs
template <int C>
__device__ __forceinline__ void warp_mm(const float* A, const float* B, float* out, int lane) {
  for (int t = lane; t < C * C; t += 32) {
    const int r = t / C, s = t - r * C;
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < C; ++k) acc = fmaf(A[r * C + k], B[k * C + s], acc);
    out[t] = acc;
  }
}

// Inverts the NB x NB block F (shared memory, row-major) in place, Gauss-Jordan
// with partial pivoting, one warp, and stores it column-major; a block without
// an inverse is counted and stored as the identity.
template <int NB>
__device__ void invert_block(float* F, int* piv, float* __restrict__ dst, int lane, unsigned* n_singular) {
  bool singular = false;
  for (int k = 0; k < NB; ++k) {
    float best = -1.f;
    int bi = k;
    for (int i = k + lane; i < NB; i += 32) {
      const float v = fabsf(F[i * NB + k]);
      if (v > best) {
        best = v;
        bi = i;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) {
        best = ov;
        bi = oi;
      }
    }
    if (!(best > 0.f) || !isfinite(best)) {
      singular = true;
      break;
    }
    if (lane == 0) piv[k] = bi;
    if (bi != k)
      for (int j = lane; j < NB; j += 32) {
        const float tmp = F[k * NB + j];
        F[k * NB + j] = F[bi * NB + j];
        F[bi * NB + j] = tmp;
      }
    __syncwarp();
    const float inv = 1.f / F[k * NB + k];
    __syncwarp();
    for (int j = lane; j < NB; j += 32) F[k * NB + j] = j == k ? inv : F[k * NB + j] * inv;
    __syncwarp();
    for (int t = lane; t < NB * NB; t += 32) {
      const int i = t / NB, j = t - i * NB;
      if (i == k) continue;
      const float fik = F[i * NB + k];
      if (j == k) continue;
      F[t] = fmaf(-fik, F[k * NB + j], F[t]);
    }
    __syncwarp();
    for (int i = lane; i < NB; i += 32)
      if (i != k) F[i * NB + k] = -F[i * NB + k] * inv;
    __syncwarp();
  }
  if (singular) {
    if (lane == 0) atomicAdd(n_singular, 1u);
    for (int t = lane; t < NB * NB; t += 32) dst[t] = (t / NB == t % NB) ? 1.f : 0.f;
    __syncwarp();
    return;
  }
  // undo the row exchanges as column exchanges, in reverse order
  for (int k = NB - 1; k >= 0; --k) {
    const int pk = piv[k];
    if (pk != k)
      for (int i = lane; i < NB; i += 32) {
        const float tmp = F[i * NB + k];
        F[i * NB + k] = F[i * NB + pk];
        F[i * NB + pk] = tmp;
      }
    __syncwarp();
  }
  // column-major store for the apply kernel
  for (int t = lane; t < NB * NB; t += 32) {
    const int col = t / NB, row = t - col * NB;
    dst[t] = F[row * NB + col];
  }
  __syncwarp();
}

template <typename T, int N, bool PAPER, bool INVERT>
__global__ void __launch_bounds__(128)
    block_diag_kernel(const int32_t* __restrict__ node_off, const int32_t* __restrict__ node_elem,
                      const int4* __restrict__ tets, const T* __restrict__ geo, const T* __restrict__ u0,
                      const T* __restrict__ tau, const uint8_t* __restrict__ dmask,
                      const float* __restrict__ outdiag, Phys<float> ph, float* __restrict__ out,
                      int64_t n_nodes, unsigned* __restrict__ n_singular) {
  using L = BlockLayout<N>;
  using D = Dims<N>;
  constexpr int C = L::C, NB = L::NB, CC = L::CC, NM = D::NM, NT = D::NT, NTP = D::NT_PAD;
  extern __shared__ __align__(16) float smem_f[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  float* ws = smem_f + warp * L::WARP;
  float* F = ws + L::F;
  float* tq = ws + L::TAU;
  float* Sm = ws + L::SM;
  float* Wm = ws + L::WM;
  float* Xm = ws + L::XM;
  float* Ym = ws + L::YM;
  float* Kacc = ws + L::ACC;
  float* Gacc = Kacc + CC;
  float* Dacc = Kacc + 4 * CC;
  float* Lacc = Kacc + 7 * CC;
  float* sg = ws + L::GEO;
  float* un = ws + L::UN;
  float* gam = ws + L::GAM;
  float* bet = ws + L::BET;
  int* piv = reinterpret_cast<int*>(ws + L::PIV);
  const float rho = ph.rho, omega = ph.omega;

  for (int64_t A = (int64_t)blockIdx.x * wpb + warp; A < n_nodes; A += (int64_t)gridDim.x * wpb) {
    for (int t = lane; t < 8 * CC; t += 32) Kacc[t] = 0.f;
    __syncwarp();
    const int p0 = node_off[A], p1 = node_off[A + 1];
    for (int p = p0; p < p1; ++p) {
      const int packed = node_elem[p];
      const int64_t e = packed >> 2;
      const int a = packed & 3;
      const int4 nd = tets[e];
      const int node[4] = {nd.x, nd.y, nd.z, nd.w};
      if (lane < GEO_STRIDE) sg[lane] = (float)geo[e * GEO_STRIDE + lane];
      for (int t = lane; t < 12 * C; t += 32) {
        const int b = t / (3 * C), r = t - b * 3 * C;
        const int c = r % C;
        un[t] = c == 1 ? 0.f : (float)u0[(int64_t)node[b] * 4 * C + r];
      }
      __syncwarp();
      const float vol = sg[GEO_VOL], w4 = 0.25f * vol;
      const float da0 = sg[a * 3 + 0], da1 = sg[a * 3 + 1], da2 = sg[a * 3 + 2];
      for (int t = lane; t < 4 * C; t += 32) {
        const int b = t / C, c = t - b * C;
        gam[t] = da0 * un[(b * 3 + 0) * C + c] + da1 * un[(b * 3 + 1) * C + c] + da2 * un[(b * 3 + 2) * C + c];
      }
      for (int q = 0; q < 4; ++q) {
        const float laq = (float)qp_bary(q, a);
        __syncwarp();
        for (int c = lane; c < C; c += 32) {
          float acc = 0.f;
#pragma unroll
          for (int b = 0; b < 4; ++b) acc += (float)qp_bary(q, b) * gam[b * C + c];
          bet[c] = acc;
        }
        // tau_q: packed upper triangle in the orthonormal basis -> storage coordinates
        for (int t = lane; t < CC; t += 32) tq[t] = 0.f;
        __syncwarp();
        const T* tp = tau + (e * 4 + q) * NTP;
        for (int t = lane; t < NT; t += 32) {
          int r = 0, rem = t;
          while (rem >= NM - r) {
            rem -= NM - r;
            ++r;
          }
          const int s = r + rem;
          const float val = (float)tp[t];
          const float drs = (r == 0 && s > 0) ? Real<float>::SQRT2 : 1.f;
          const float dsr = (r == 0 && s > 0) ? Real<float>::INV_SQRT2 : 1.f;
          tq[stor_of(r) * C + stor_of(s)] = val * drs;
          tq[stor_of(s) * C + stor_of(r)] = val * dsr;
        }
        for (int t = lane; t < CC; t += 32) {
          const int r = t / C, s = t - r * C;
          const float cv = conv_entry<N>(bet, r, s), om = omega_entry(r, s, omega);
          Sm[t] = laq * om + cv;
          Wm[t] = -laq * om + cv;
        }
        __syncwarp();
        warp_mm<C>(tq, Sm, Xm, lane);   // X = tau S
        warp_mm<C>(Wm, tq, Ym, lane);   // Y = W tau
        __syncwarp();
        for (int t = lane; t < CC; t += 32) {
          const int r = t / C, s = t - r * C;
          float wx = 0.f;
#pragma unroll
          for (int k = 0; k < C; ++k) wx = fmaf(Wm[r * C + k], Xm[k * C + s], wx);
          Kacc[t] += w4 * rho * (laq * Sm[t] + wx);
          Lacc[t] += (w4 / rho) * (da0 * da0 + da1 * da1 + da2 * da2) * tq[t];
          if (!PAPER) {
            Gacc[t] += w4 * da0 * Ym[t];
            Gacc[CC + t] += w4 * da1 * Ym[t];
            Gacc[2 * CC + t] += w4 * da2 * Ym[t];
            Dacc[t] += w4 * da0 * Xm[t];
            Dacc[CC + t] += w4 * da1 * Xm[t];
            Dacc[2 * CC + t] += w4 * da2 * Xm[t];
          }
        }
      }
      __syncwarp();
      // identity parts: viscous, consistent mass, Galerkin pressure and divergence
      const float g2 = da0 * da0 + da1 * da1 + da2 * da2;
      for (int c = lane; c < C; c += 32) {
        Kacc[c * C + c] += ph.mu * vol * g2 + ph.mass_coef * vol * 0.1f;
        Gacc[c * C + c] += -0.25f * vol * da0;
        Gacc[CC + c * C + c] += -0.25f * vol * da1;
        Gacc[2 * CC + c * C + c] += -0.25f * vol * da2;
        Dacc[c * C + c] += w4 * da0;
        Dacc[CC + c * C + c] += w4 * da1;
        Dacc[2 * CC + c * C + c] += w4 * da2;
      }
      __syncwarp();
    }
    // ---- the full block F [NB][NB], rows/columns (field, storage coordinate)
    const bool dir = dmask[A] != 0;
    const float* od = outdiag + A * 6;   // R w_i w_j (xx, xy, xz, yy, yz, zz)
    for (int t = lane; t < NB * NB; t += 32) {
      const int row = t / NB, col = t - row * NB;
      const int f = row / C, c = row - f * C, g = col / C, d = col - g * C;
      float val;
      if (f < 3 && g < 3) {
        val = f == g ? Kacc[c * C + d] : 0.f;
        if (c == d) {
          const int lo = f < g ? f : g, hi = f < g ? g : f;
          const int k = lo == 0 ? hi : (lo == 1 ? 2 + hi : 5);
          val += od[k];
        }
      } else if (f < 3) {
        val = Gacc[f * CC + c * C + d];
      } else if (g < 3) {
        val = Dacc[g * CC + c * C + d];
      } else {
        val = Lacc[c * C + d];
      }
      // fixed unknowns: Im(mode 0) of every field, velocity of a Dirichlet node
      const bool fr = c == 1 || (dir && f < 3), fc = d == 1 || (dir && g < 3);
      if (fr || fc) val = (INVERT && row == col) ? 1.f : 0.f;
      F[t] = val;
    }
    __syncwarp();
    float* dst = out + A * NB * NB;
    if (!INVERT) {
      for (int t = lane; t < NB * NB; t += 32) dst[t] = F[t];
      __syncwarp();
      continue;
    }
    invert_block<NB>(F, piv, dst, lane, n_singular);
  }
}

// ---------------------------------------------------------------------------
// N <= 7: the same blocks with register tiles (nodal.cuh).  A warp owns a node;
// its four groups of N lanes take the four quadrature points of an element and
// sum over the node's elements in registers: K += w rho (lambda S + S^T X),
// X = tau S, GX_i += w dN/dx_i X (the least-squares part of D_i; of G_i,
// transposed), L += (w / rho) |grad N|^2 tau.
//
// Inverse: with the velocity block K (the same for three fields) and no outlet
// coupling,
//   E_i = K^-1 G_i, S = L - sum_i D_i E_i, H_j = S^-1 D_j K^-1, H_p = -S^-1,
//   inverse_ij = delta_ij K^-1 + E_i H_j (j = 1..3, p), row p = -H_j,
// two n x n inversions and about 20 products instead of one (8N)^3 elimination.
// The n x n inversions do not exchange rows; a node where a pivot is less than
// PIVOT_OK of the largest candidate, and the outlet nodes, take the full
// elimination.
//
// N = 7, 52,650 tetrahedra, with inverse: 1.16 ms (8.4 ms before: the sums were two
// shared-memory loads a multiply-add and the elimination one warp's passes over
// 3136 entries); the inverse is 0.04 ms of it.  Bound by issue and shared memory
// at 8 warps an SM (255 registers hold the five n x n sums of a group; the inverting form
// spills 17 words at N = 7).
constexpr float PIVOT_OK = 0.1f;

template <int N>
struct NodalBlock {
  using D = Nodal<N>;
  static constexpr int C = 2 * N, NB = 8 * N;
  // while summing: tau [4], S [4], tables [4][2][TW]
  static constexpr int TAU = 0, S = TAU + 4 * D::MAT, TAB = S + 4 * D::MAT, SUM_END = TAB + 4 * 2 * D::TW;
  // then: K (columns as rows), GX_0..2 (row-major), L; and over the rest K^-1, S^-1, E_0..2 or the full block
  static constexpr int K = 0, GX = D::MAT, LM = 4 * D::MAT, REST = 5 * D::MAT;
  static constexpr int KI = REST, SI = KI + D::MAT, E = SI + D::MAT, SCHUR_END = E + 3 * D::MAT;
  static constexpr int F = REST, PIV = F + NB * NB, FULL_END = PIV + NB;
  static constexpr int MAX1 = SUM_END > SCHUR_END ? SUM_END : SCHUR_END;
  static constexpr int WARP = ((MAX1 > FULL_END ? MAX1 : FULL_END) + 3) & ~3;
};

// In-place Gauss-Jordan inverse of the group's matrix (columns in lanes), without
// row exchanges; false where a pivot is small.  The rows move up one a step, so
// that the pivot is at index 0 and the loop can stay rolled.
template <int N>
__device__ __forceinline__ bool nodal_invert(float (&x)[2 * N - 1], float (&y)[2 * N - 1], int p, int base) {
  constexpr int NM = 2 * N - 1;
  bool ok = true;
#pragma unroll 1
  for (int k = 0; k < NM; ++k) {
    const int src = base + (k + 1) / 2;
    const bool odd = k & 1;
    float c[NM], big = 0.f;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      c[i] = __shfl_sync(0xffffffffu, odd ? x[i] : y[i], src);
      if (i < NM - k) big = fmaxf(big, fabsf(c[i]));
    }
    ok = ok && fabsf(c[0]) > PIVOT_OK * big && isfinite(big);
    const float rd = 1.f / c[0];
    const bool px = 2 * p - 1 == k, py = 2 * p == k;
    const float tx = px ? rd : x[0] * rd, ty = py ? rd : y[0] * rd;
#pragma unroll
    for (int i = 1; i < NM; ++i) {
      x[i - 1] = fmaf(-c[i], tx, px ? 0.f : x[i]);
      y[i - 1] = fmaf(-c[i], ty, py ? 0.f : y[i]);
    }
    x[NM - 1] = tx;
    y[NM - 1] = ty;
  }
  return ok;
}

template <typename T, typename U, int N, bool PAPER, bool INVERT>
__global__ void __launch_bounds__(128, 2)
    nodal_block_kernel(const int32_t* __restrict__ node_off, const int32_t* __restrict__ node_elem,
                       const int4* __restrict__ tets, const T* __restrict__ geo, const U* __restrict__ u0,
                       const T* __restrict__ tau, const uint8_t* __restrict__ dmask,
                       const float* __restrict__ outdiag, Phys<float> ph, float* __restrict__ out, int64_t n_nodes,
                       unsigned* __restrict__ n_singular) {
  using D = Nodal<N>;
  using W = NodalBlock<N>;
  constexpr int NM = D::NM, C = D::C, NB = W::NB, LD = D::LD, MAT = D::MAT, NTP = D::NTP;
  extern __shared__ __align__(16) float nodal_smem[];
  __shared__ int offs[D::NT];
  nodal_offsets<N>(offs, threadIdx.x, blockDim.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const int g0 = lane / N, p = lane - g0 * N;
  const bool in_group = g0 < 4;
  const int g = in_group ? g0 : 0, base = g * N;
  using Stage = NodalStage<T, U, N>;
  float* ws = nodal_smem + warp * (W::WARP + Stage::BYTES / 4);
  char* stage = reinterpret_cast<char*>(ws + W::WARP);
  float* tq = ws + W::TAU + g * MAT;
  float* Sq = ws + W::S + g * MAT;
  float* tab = ws + W::TAB + g * 2 * D::TW;
  const float rho = ph.rho, bq = (float)qp_bary(0, 1), dq = (float)(qp_bary(0, 0) - qp_bary(0, 1));

  for (int64_t A = (int64_t)blockIdx.x * wpb + warp; A < n_nodes; A += (int64_t)gridDim.x * wpb) {
    float Kx[NM], Ky[NM], Gx[3][NM], Gy[3][NM], Lx[NM], Ly[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      Kx[i] = Ky[i] = Lx[i] = Ly[i] = 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j) Gx[j][i] = Gy[j][i] = 0.f;
    }
    float kd = 0.f, gd[3] = {0.f, 0.f, 0.f};
    const int p0 = node_off[A], p1 = node_off[A + 1];
    // list entries three elements ahead, nodes two, the copies one: no load waits for
    // another's result
    int pk0 = p0 < p1 ? node_elem[p0] : 0, pk1 = p0 + 1 < p1 ? node_elem[p0 + 1] : 0,
        pk2 = p0 + 2 < p1 ? node_elem[p0 + 2] : 0;
    int4 nd0 = p0 < p1 ? tets[pk0 >> 2] : make_int4(0, 0, 0, 0), nd1 = p0 + 1 < p1 ? tets[pk1 >> 2] : nd0;
    __syncwarp();
    if (p0 < p1) Stage::issue(stage, pk0 >> 2, nd0, tau, u0, geo, lane);
#pragma unroll 1
    for (int pi = p0; pi < p1; ++pi) {
      const int a = pk0 & 3;
      const char* in = stage;
      cp_async_wait<0>();
      __syncwarp();                       // the copies; the previous element's matrices are read
      const T* ge = Stage::geo_of(in);
      const float w4 = 0.25f * nodal_float(ge[GEO_VOL]);
      const float d[3] = {nodal_float(ge[a * 3]), nodal_float(ge[a * 3 + 1]), nodal_float(ge[a * 3 + 2])};
      const float lam = a == g ? bq + dq : bq, g2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
      // beta_q = sum_j dN_a/dx_j u0_j(q), mode p
      float be[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float sum = 0.f, own = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const U* ub = Stage::rows_of(in) + b * 4 * C + 2 * p + h;
          const float v = d[0] * nodal_value(ub[0]) + d[1] * nodal_value(ub[C]) + d[2] * nodal_value(ub[2 * C]);
          sum += v;
          own = b == g ? v : own;
        }
        be[h] = p == 0 && h == 1 ? 0.f : fmaf(bq, sum, dq * own);
      }
      if (in_group) {
        nodal_modes<N>(tab, p, be[0], be[1]);
        nodal_tau<N>(Stage::tau_of(in) + g * NTP, offs, tq, p);
      }
      __syncwarp();
      // the stage is consumed: the next element's copies run behind the products
      if (pi + 1 < p1) {
        Stage::issue(stage, pk1 >> 2, nd1, tau, u0, geo, lane);
        pk0 = pk1;
        pk1 = pk2;
        nd0 = nd1;
        if (pi + 2 < p1) nd1 = tets[pk1 >> 2];
        if (pi + 3 < p1) pk2 = node_elem[pi + 3];
      }
      float sx[NM], sy[NM], X[NM], Y[NM];
      nodal_columns<N>(tab, p, lam * ph.omega, sx, sy);
      if (in_group) nodal_store_rows<N>(Sq, p, sx, sy);
#pragma unroll
      for (int i = 0; i < NM; ++i) X[i] = Y[i] = 0.f;
      nodal_product<N>(tq, sx, sy, X, Y);
      const float wr = w4 * rho;
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        Kx[i] = fmaf(wr * lam, sx[i], Kx[i]);
        Ky[i] = fmaf(wr * lam, sy[i], Ky[i]);
        if (!PAPER) {
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            Gx[j][i] = fmaf(w4 * d[j], X[i], Gx[j][i]);
            Gy[j][i] = fmaf(w4 * d[j], Y[i], Gy[j][i]);
          }
        }
        X[i] *= wr;
        Y[i] *= wr;
      }
      nodal_load_rows<N>(tq, p, sx, sy);  // tau's columns
      const float wl = w4 / rho * g2;
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        Lx[i] = fmaf(wl, sx[i], Lx[i]);
        Ly[i] = fmaf(wl, sy[i], Ly[i]);
      }
      __syncwarp();
      nodal_product<N>(Sq, X, Y, Kx, Ky); // rows of Sq are S's columns: S^T X
      // identity parts: viscous, consistent mass; Galerkin divergence (and, negated, pressure)
      kd += 4.f * w4 * (ph.mu * g2 + 0.1f * ph.mass_coef);
#pragma unroll
      for (int j = 0; j < 3; ++j) gd[j] = fmaf(w4, d[j], gd[j]);
    }
    // sums over the four points into group 0, then to shared memory
    auto fold = [&](float v) {
      v += __shfl_down_sync(0xffffffffu, v, 2 * N);
      return v + __shfl_down_sync(0xffffffffu, v, N);
    };
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      Kx[i] = fold(Kx[i]) + (i == 2 * p - 1 ? kd : 0.f);
      Ky[i] = fold(Ky[i]) + (i == 2 * p ? kd : 0.f);
      Lx[i] = fold(Lx[i]);
      Ly[i] = fold(Ly[i]);
      if (!PAPER) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          Gx[j][i] = fold(Gx[j][i]);
          Gy[j][i] = fold(Gy[j][i]);
        }
      }
    }
    __syncwarp();
    if (lane < N) {
      nodal_store_rows<N>(ws + W::K, p, Kx, Ky);
      nodal_store_rows<N>(ws + W::LM, p, Lx, Ly);
#pragma unroll
      for (int j = 0; j < 3; ++j) nodal_store_columns<N>(ws + W::GX + j * MAT, p, Gx[j], Gy[j]);
    }
    __syncwarp();
    const bool dir = dmask[A] != 0;
    const float* od = outdiag + A * 6;   // R w_i w_j (xx, xy, xz, yy, yz, zz)
    float* dst = out + A * NB * NB;
    // an entry of the full block in storage coordinates (x_0, Re x_n, Im x_n): row and
    // column scaled by D = diag(1, 1/sqrt2, ...) and its inverse
    auto entry = [&](int row, int col) {
      const int f = row / C, c = row - f * C, h = col / C, k = col - h * C;
      const bool fr = c == 1 || (dir && f < 3), fc = k == 1 || (dir && h < 3);
      if (fr || fc) return INVERT && row == col ? 1.f : 0.f;
      const int r = c == 0 ? 0 : c - 1, s = k == 0 ? 0 : k - 1;
      float v;
      if (f < 3 && h < 3) {
        v = f == h ? ws[W::K + s * LD + r] : 0.f;
        if (r == s) {
          const int lo = f < h ? f : h, hi = f < h ? h : f;
          v += od[lo == 0 ? hi : (lo == 1 ? 2 + hi : 5)];
        }
      } else if (f < 3) {
        v = ws[W::GX + f * MAT + s * LD + r] - (r == s ? (f == 0 ? gd[0] : f == 1 ? gd[1] : gd[2]) : 0.f);
      } else if (h < 3) {
        v = ws[W::GX + h * MAT + r * LD + s] + (r == s ? (h == 0 ? gd[0] : h == 1 ? gd[1] : gd[2]) : 0.f);
      } else {
        v = ws[W::LM + s * LD + r];
      }
      return r == 0 && s > 0 ? v * Real<float>::SQRT2 : r > 0 && s == 0 ? v * Real<float>::INV_SQRT2 : v;
    };
    if (!INVERT) {
      for (int t = lane; t < NB * NB; t += 32) dst[t] = entry(t / NB, t % NB);
      __syncwarp();
      continue;
    }
    bool ok = od[0] == 0.f && od[3] == 0.f && od[5] == 0.f;   // no outlet coupling (the same for the warp)
    float Hx[NM], Hy[NM];                                    // group j: H_j, group 3: H_p
    if (ok) {
      float* KI = ws + W::KI;
      float* SI = ws + W::SI;
      float kx[NM], ky[NM], ex[NM], ey[NM], tx[NM], ty[NM];
      nodal_load_rows<N>(ws + W::LM, p, tx, ty);
      const int j3 = g < 3 ? g : 0;
      const float gg = g == 0 ? gd[0] : g == 1 ? gd[1] : gd[2];
      const float* GXg = ws + W::GX + j3 * MAT;
      if (!dir) {
        nodal_load_rows<N>(ws + W::K, p, kx, ky);
        ok = nodal_invert<N>(kx, ky, p, base);
        if (lane < N) nodal_store_columns<N>(KI, p, kx, ky);
        __syncwarp();
        // E_i = K^-1 G_i, G_i = GX_i^T - gd_i I (group i)
        nodal_load_rows<N>(GXg, p, Hx, Hy);
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          Hx[i] -= i == 2 * p - 1 ? gg : 0.f;
          Hy[i] -= i == 2 * p ? gg : 0.f;
          ex[i] = ey[i] = 0.f;
        }
        nodal_product<N>(KI, Hx, Hy, ex, ey);
        if (in_group && g < 3) nodal_store_columns<N>(ws + W::E + g * MAT, p, ex, ey);
        // S = L - sum_i D_i E_i, D_i = GX_i + gd_i I
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          Hx[i] = gg * ex[i];
          Hy[i] = gg * ey[i];
        }
        nodal_product<N>(GXg, ex, ey, Hx, Hy);
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          tx[i] -= __shfl_sync(0xffffffffu, Hx[i], p) + __shfl_sync(0xffffffffu, Hx[i], N + p) +
                   __shfl_sync(0xffffffffu, Hx[i], 2 * N + p);
          ty[i] -= __shfl_sync(0xffffffffu, Hy[i], p) + __shfl_sync(0xffffffffu, Hy[i], N + p) +
                   __shfl_sync(0xffffffffu, Hy[i], 2 * N + p);
        }
      }
      const bool ok2 = nodal_invert<N>(tx, ty, p, base);
      ok = __all_sync(0xffffffffu, (ok && ok2) || !in_group);
      if (lane < N) nodal_store_columns<N>(SI, p, tx, ty);
      __syncwarp();
      // H_j = S^-1 D_j K^-1 (groups 0..2), H_p = -S^-1 (group 3)
      if (!dir) {
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          ex[i] = gg * kx[i];
          ey[i] = gg * ky[i];
          Hx[i] = Hy[i] = 0.f;
        }
        nodal_product<N>(GXg, kx, ky, ex, ey);
        nodal_product<N>(SI, ex, ey, Hx, Hy);
      }
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        if (g == 3) {
          Hx[i] = -tx[i];
          Hy[i] = -ty[i];
        } else if (dir) {
          Hx[i] = Hy[i] = 0.f;
        }
      }
      if (ok) {
        // the lane's columns, storage coordinates: 2p and 2p+1 of field g (lane 0: 0; its 1 is Im(mode 0))
        constexpr float S2 = Real<float>::SQRT2, IS2 = Real<float>::INV_SQRT2;
        float* cx = dst + (int64_t)(g * C + 2 * p) * NB;
        float* cy = cx + NB;
#pragma unroll 1
        for (int f = 0; f < 4; ++f) {
          float ox[NM], oy[NM];
          if (f < 3 && !dir) {
#pragma unroll
            for (int i = 0; i < NM; ++i) {
              ox[i] = f == g ? kx[i] : 0.f;
              oy[i] = f == g ? ky[i] : 0.f;
            }
            nodal_product<N>(ws + W::E + f * MAT, Hx, Hy, ox, oy);
          } else {
#pragma unroll
            for (int i = 0; i < NM; ++i) {
              ox[i] = f == 3 ? -Hx[i] : (f == g && i == 2 * p - 1 ? 1.f : 0.f);
              oy[i] = f == 3 ? -Hy[i] : (f == g && i == 2 * p ? 1.f : 0.f);
            }
          }
          if (in_group) {
            // lane p > 0: x is stored column 2p, y is 2p + 1; lane 0: y is column 0
            float2* sx = reinterpret_cast<float2*>(cx + f * C);
            float2* sy = reinterpret_cast<float2*>(cy + f * C);
            if (p == 0) {
              sx[0] = make_float2(oy[0], 0.f);
              sy[0] = make_float2(0.f, f == g ? 1.f : 0.f);
            } else {
              sx[0] = make_float2(ox[0] * S2, 0.f);
              sy[0] = make_float2(oy[0] * S2, 0.f);
            }
#pragma unroll
            for (int n = 1; n < N; ++n) {
              if (p == 0) {
                sx[n] = make_float2(oy[2 * n - 1] * IS2, oy[2 * n] * IS2);
                sy[n] = make_float2(0.f, 0.f);
              } else {
                sx[n] = make_float2(ox[2 * n - 1], ox[2 * n]);
                sy[n] = make_float2(oy[2 * n - 1], oy[2 * n]);
              }
            }
          }
        }
      }
    }
    if (!ok) {
      __syncwarp();
      float* F = ws + W::F;
      for (int t = lane; t < NB * NB; t += 32) F[t] = entry(t / NB, t % NB);
      __syncwarp();
      invert_block<NB>(F, reinterpret_cast<int*>(ws + W::PIV), dst, lane, n_singular);
    }
    __syncwarp();
  }
}

// z[A] = Binv[A] x[A] per node (column-major FP32 blocks, FP64 vectors)
template <int N>
__global__ void __launch_bounds__(256)
    block_apply_kernel(const float* __restrict__ binv, const double* __restrict__ x, double* __restrict__ z,
                       int64_t n_nodes) {
  constexpr int NB = 8 * N;
  constexpr int R = (NB + 31) / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  for (int64_t A = (int64_t)blockIdx.x * wpb + warp; A < n_nodes; A += (int64_t)gridDim.x * wpb) {
    const double* xa = x + A * NB;
    float xr[R];
#pragma unroll
    for (int s = 0; s < R; ++s) xr[s] = lane + 32 * s < NB ? (float)xa[lane + 32 * s] : 0.f;
    float acc[R];
#pragma unroll
    for (int s = 0; s < R; ++s) acc[s] = 0.f;
    const float* B = binv + A * NB * NB;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const float xj = __shfl_sync(0xffffffffu, xr[j >> 5], j & 31);
#pragma unroll
      for (int s = 0; s < R; ++s)
        if (lane + 32 * s < NB) acc[s] = fmaf(B[j * NB + lane + 32 * s], xj, acc[s]);
    }
    double* za = z + A * NB;
#pragma unroll
    for (int s = 0; s < R; ++s)
      if (lane + 32 * s < NB) za[lane + 32 * s] = (double)acc[s];
  }
}

template <typename T, int N>
int launch_block_diag(int variant_paper, int invert, const int32_t* node_off, const int32_t* node_elem,
                      const int4* tets, const T* geo, const T* u0, const T* uc, const T* tau, const uint8_t* dmask,
                      const float* outdiag, Phys<float> ph, float* out, int64_t n_nodes,
                      unsigned* n_singular, cudaStream_t st) {
  if (n_nodes <= 0) return 0;
  auto go = [&](auto kern, size_t smem, int warps, auto u) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -2;
    const int64_t blocks = std::min<int64_t>((n_nodes + warps - 1) / warps, 152 * 16);
    count_launches(1);
    kern<<<(int)blocks, warps * 32, smem, st>>>(node_off, node_elem, tets, geo, u, tau, dmask, outdiag, ph, out,
                                               n_nodes, n_singular);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
  };
  if constexpr (N <= NODAL_MAX_N) {
    using U = typename PairOfStore<T>::V;
    const size_t smem = (size_t)4 * (NodalBlock<N>::WARP * sizeof(float) + NodalStage<T, U, N>::BYTES);
    static_assert(4 * (NodalBlock<N>::WARP * 4 + NodalStage<T, U, N>::BYTES) <= 113 * 1024, "two blocks an SM");
    const U* u = reinterpret_cast<const U*>(uc);
    if (variant_paper)
      return invert ? go(nodal_block_kernel<T, U, N, true, true>, smem, 4, u)
                    : go(nodal_block_kernel<T, U, N, true, false>, smem, 4, u);
    return invert ? go(nodal_block_kernel<T, U, N, false, true>, smem, 4, u)
                  : go(nodal_block_kernel<T, U, N, false, false>, smem, 4, u);
  } else {
    // the register tiles of N > 7 do not fit: five n x n sums a group
    using L = BlockLayout<N>;
    int warps = 4;
    while (warps > 1 && (size_t)warps * L::WARP * sizeof(float) > 200 * 1024) --warps;
    const size_t smem = (size_t)warps * L::WARP * sizeof(float);
    if (smem > 227 * 1024) return -6;
    if (variant_paper)
      return invert ? go(block_diag_kernel<T, N, true, true>, smem, warps, u0)
                    : go(block_diag_kernel<T, N, true, false>, smem, warps, u0);
    return invert ? go(block_diag_kernel<T, N, false, true>, smem, warps, u0)
                  : go(block_diag_kernel<T, N, false, false>, smem, warps, u0);
  }
}

template <int N>
int launch_block_apply(const float* binv, const double* x, double* z, int64_t n_nodes, cudaStream_t st) {
  if (n_nodes <= 0) return 0;
  const int threads = 256;
  int64_t blocks = (n_nodes + 7) / 8;
  if (blocks > 152 * 8) blocks = 152 * 8;
  count_launches(1);
  block_apply_kernel<N><<<(int)blocks, threads, 0, st>>>(binv, x, z, n_nodes);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

#define TS_INST_BLOCK(T, N)                                                                          \
  template int launch_block_diag<T, N>(int, int, const int32_t*, const int32_t*, const int4*, const T*, \
                                       const T*, const T*, const T*, const uint8_t*, const float*, Phys<float>,  \
                                       float*, int64_t, unsigned*, cudaStream_t);
TS_FOR_EACH_N(TS_INST_BLOCK, float)
TS_FOR_EACH_N(TS_INST_BLOCK, double)
#define TS_INST_BAPPLY(T, N) template int launch_block_apply<N>(const float*, const double*, double*, int64_t, cudaStream_t);
TS_FOR_EACH_N(TS_INST_BAPPLY, float)

}  // namespace ts
