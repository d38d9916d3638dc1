// Assembled block-structured tangent of the paper's variant (section 2.5.2) and
// its sparse matrix-vector product.
//
// With A and tau frozen (eq. K_mat) and the least-squares parts dropped from
// G_i and D_j, the tangent of eq. (tangent) between nodes A and B is
//   [[K, 0, 0, G_1], [0, K, 0, G_2], [0, 0, K, G_3], [D_1, D_2, D_3, L]]
// where K_AB and L_AB are full mode matrices, but G_i = -int dN_A/dx_i N_B I
// and D_j = int N_A dN_B/dx_j I are scalars times the identity: per mesh
// connection the paper stores K once (reused for the three velocity fields),
// L, and six scalars (section 2.5.2), instead of the 16 full blocks.  Per
// element and quadrature point (weight w = V/4), in storage coordinates:
//   K_AB += w rho (lambda_qa S_qb + W_qa tau_q S_qb) + (mu V grad N_a . grad N_b
//           + c1 rho/dt V (1 + delta_ab)/20) I
//   L_AB += (w / rho) grad N_a . grad N_b tau_q
//   G_AB,i += -(V/4) dN_a/dx_i,   D_AB,j += (V/4) dN_b/dx_j
// with S_qb = lambda_qb Omega + Conv(beta_qb), W_qa = -lambda_qa Omega +
// Conv(beta_qa), beta_qb = sum_j dN_b/dx_j u0_j(q) (see precond.cu).
//
// Storage: the node graph in CSR (row A, sorted columns B, A itself
// included); per connection one record of HB = 2 C^2 + 8 floats:
// K [C][C], L [C][C], G_1..3, D_1..3, two pad floats (16-byte records).
//
// GB300 mapping.  Assembly: one warp per row gathers the row's (element,
// local node) pairs from the node-to-element list and adds every element
// contribution to the row's records (the warp owns the row: no atomics,
// deterministic).  Product: a warp streams the records of a few rows
// (1.6 KB each at N = 7); the records are the only large HBM stream, so the
// product is bound by HBM bandwidth.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "nodal.cuh"

namespace ts {

namespace {

template <int N>
struct AsmLayout {
  static constexpr int C = 2 * N, CC = C * C;
  static constexpr int HB = 2 * CC + 8;
  // assembly workspace per warp (floats)
  static constexpr int TAU = 0, WM = CC, YM = 2 * CC, SM = 3 * CC, TSUM = 4 * CC;
  static constexpr int ZACC = 5 * CC;            // [4][C][C] LS + Galerkin parts of K_ab
  static constexpr int GEO = ZACC + 4 * CC;      // 20 (+4)
  static constexpr int UN = GEO + 24;            // u0 velocity at the 4 nodes [4][3][C]
  static constexpr int BET = UN + 12 * C;        // beta_qb [4][C] for the current q
  static constexpr int WARP = (BET + 4 * C + 3) & ~3;
  // product workspace per warp: the record and x_B
  static constexpr int PWARP = HB + 4 * C;
};

template <int N>
__device__ __forceinline__ float2 amode(const float* b, int k) {
  if (k <= -N || k >= N) return make_float2(0.f, 0.f);
  if (k >= 0) return make_float2(b[2 * k], k == 0 ? 0.f : b[2 * k + 1]);
  return make_float2(b[-2 * k], -b[-2 * k + 1]);
}

// Conv(beta) on storage coordinates (the truncated convolution of eq. phi-def)
template <int N>
__device__ __forceinline__ float aconv(const float* beta, int r, int s) {
  if (s == 1) return 0.f;
  const int m = r >> 1, n = s >> 1;
  const bool im_row = r & 1;
  if (n == 0) {
    const float2 b = amode<N>(beta, m);
    return im_row ? b.y : b.x;
  }
  const float2 lo = amode<N>(beta, m - n), hi = amode<N>(beta, m + n);
  if (!(s & 1)) return im_row ? lo.y + hi.y : lo.x + hi.x;
  return im_row ? lo.x - hi.x : hi.y - lo.y;
}

__device__ __forceinline__ float aomega(int r, int s, float omega) {
  const int n = r >> 1;
  if (n == 0 || (r ^ 1) != s) return 0.f;
  return (r & 1) ? n * omega : -n * omega;
}

}  // namespace

template <typename T, int N>
__global__ void __launch_bounds__(128)
    assemble_paper_kernel(const int32_t* __restrict__ node_off, const int32_t* __restrict__ node_elem,
                          const int32_t* __restrict__ row_off, const int32_t* __restrict__ cols,
                          const int4* __restrict__ tets, const T* __restrict__ geo, const T* __restrict__ u0,
                          const T* __restrict__ tau, Phys<float> ph, float* __restrict__ H, int64_t n_nodes) {
  using L = AsmLayout<N>;
  using D = Dims<N>;
  constexpr int C = L::C, CC = L::CC, HB = L::HB, NM = D::NM, NT = D::NT, NTP = D::NT_PAD;
  extern __shared__ __align__(16) float smem_f[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  float* ws = smem_f + warp * L::WARP;
  float* tq = ws + L::TAU;
  float* Wm = ws + L::WM;
  float* Ym = ws + L::YM;
  float* Sm = ws + L::SM;
  float* Ts = ws + L::TSUM;
  float* Z = ws + L::ZACC;
  float* sg = ws + L::GEO;
  float* un = ws + L::UN;
  float* bet = ws + L::BET;
  const float rho = ph.rho, omega = ph.omega;

  for (int64_t A = (int64_t)blockIdx.x * wpb + warp; A < n_nodes; A += (int64_t)gridDim.x * wpb) {
    const int r0 = row_off[A], r1 = row_off[A + 1];
    for (int64_t t = (int64_t)r0 * HB + lane; t < (int64_t)r1 * HB; t += 32) H[t] = 0.f;
    __syncwarp();
    for (int p = node_off[A]; p < node_off[A + 1]; ++p) {
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
      for (int t = lane; t < 4 * CC; t += 32) Z[t] = 0.f;
      for (int t = lane; t < CC; t += 32) Ts[t] = 0.f;
      // slot of each column node[b] in row A (lane b searches)
      int slot = -1;
      if (lane < 4) {
        const int Bn = node[lane];
        for (int s = r0; s < r1; ++s)
          if (cols[s] == Bn) {
            slot = s;
            break;
          }
      }
      __syncwarp();
      const float vol = sg[GEO_VOL], w4 = 0.25f * vol;
      for (int q = 0; q < 4; ++q) {
        const float laq = (float)qp_bary(q, a);
        // beta_qb for b = 0..3
        for (int t = lane; t < 4 * C; t += 32) {
          const int b = t / C, c = t - b * C;
          float acc = 0.f;
#pragma unroll
          for (int bb = 0; bb < 4; ++bb) {
            const float lam = (float)qp_bary(q, bb);
            acc += lam * (sg[b * 3 + 0] * un[(bb * 3 + 0) * C + c] + sg[b * 3 + 1] * un[(bb * 3 + 1) * C + c] +
                          sg[b * 3 + 2] * un[(bb * 3 + 2) * C + c]);
          }
          bet[t] = acc;
        }
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
          Wm[t] = -laq * aomega(r, s, omega) + aconv<N>(bet + a * C, r, s);
        }
        __syncwarp();
        // Y = W_qa tau_q; Tsum += tau_q
        for (int t = lane; t < CC; t += 32) {
          const int r = t / C, s = t - r * C;
          float acc = 0.f;
#pragma unroll
          for (int k = 0; k < C; ++k) acc = fmaf(Wm[r * C + k], tq[k * C + s], acc);
          Ym[t] = acc;
          Ts[t] += tq[t];
        }
        for (int b = 0; b < 4; ++b) {
          const float lbq = (float)qp_bary(q, b);
          __syncwarp();
          for (int t = lane; t < CC; t += 32) {
            const int r = t / C, s = t - r * C;
            Sm[t] = lbq * aomega(r, s, omega) + aconv<N>(bet + b * C, r, s);
          }
          __syncwarp();
          // Z_b += laq S_qb + Y S_qb  (times w rho at the end)
          for (int t = lane; t < CC; t += 32) {
            const int r = t / C, s = t - r * C;
            float acc = laq * Sm[t];
#pragma unroll
            for (int k = 0; k < C; ++k) acc = fmaf(Ym[r * C + k], Sm[k * C + s], acc);
            Z[b * CC + t] += acc;
          }
        }
        __syncwarp();
      }
      // add the element's contributions to the four records of row A
      const float da0 = sg[a * 3 + 0], da1 = sg[a * 3 + 1], da2 = sg[a * 3 + 2];
      for (int b = 0; b < 4; ++b) {
        const int sb = __shfl_sync(0xffffffffu, slot, b);
        if (sb < 0) continue;   // cannot happen for a consistent graph
        float* rec = H + (int64_t)sb * HB;
        const float gab = da0 * sg[b * 3 + 0] + da1 * sg[b * 3 + 1] + da2 * sg[b * 3 + 2];
        const float diag = ph.mu * vol * gab + ph.mass_coef * vol * (a == b ? 0.1f : 0.05f);
        for (int t = lane; t < CC; t += 32) {
          const int r = t / C, s = t - r * C;
          rec[t] += w4 * rho * Z[b * CC + t] + (r == s ? diag : 0.f);
          rec[CC + t] += (w4 / rho) * gab * Ts[t];
        }
        if (lane < 3) rec[2 * CC + lane] += -w4 * sg[a * 3 + lane];
        else if (lane < 6) rec[2 * CC + lane] += w4 * sg[b * 3 + lane - 3];
        __syncwarp();
      }
    }
  }
}

// ---------------------------------------------------------------------------
// N <= 7: the assembly with register tiles (nodal.cuh).  A warp owns a row and
// takes one (element, local node) at a time: its four groups of N lanes first
// form X_a = tau_q S_qa at the four points (W_qa tau_q is its transpose), then
// each takes one column node b and sums K_ab = sum_q (lambda_qa + W_qa tau_q) S_qb
// in registers; the records are updated in place by the warp that owns the row.
// 52,650 tetrahedra, N = 3 / 5 / 7: 0.47 / 0.83 / 1.81 ms (1.47 / 3.09 / 6.53 ms with one
// output a lane and both operands in shared memory); bound by shared-memory reads
// (81% at N = 5); 128 registers, at N = 7 with 4 to 6 words spilled.
template <int N>
struct NodalAssembly {
  using D = Nodal<N>;
  static constexpr int TAU = 0, Y = 4 * D::MAT, TAB = Y + 4 * D::MAT;      // tables [q][b][2][TW]
  static constexpr int WARP = (TAB + 16 * 2 * D::TW + 3) & ~3;             // then one NodalStage
};

template <typename T, typename U, int N>
__global__ void __launch_bounds__(128, 4)
    nodal_assemble_kernel(const int32_t* __restrict__ node_off, const int32_t* __restrict__ node_elem,
                          const int32_t* __restrict__ row_off, const int32_t* __restrict__ cols,
                          const int4* __restrict__ tets, const T* __restrict__ geo, const U* __restrict__ u0,
                          const T* __restrict__ tau, Phys<float> ph, float* __restrict__ H, int64_t n_nodes) {
  using D = Nodal<N>;
  using W = NodalAssembly<N>;
  constexpr int NM = D::NM, C = D::C, CC = C * C, HB = AsmLayout<N>::HB, MAT = D::MAT, NTP = D::NTP, TW = D::TW;
  extern __shared__ __align__(16) float nodal_smem[];
  __shared__ int offs[D::NT];
  nodal_offsets<N>(offs, threadIdx.x, blockDim.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const int g0 = lane / N, p = lane - g0 * N;
  const bool in_group = g0 < 4;
  const int g = in_group ? g0 : 0;
  using Stage = NodalStage<T, U, N>;
  float* ws = nodal_smem + warp * (W::WARP + Stage::BYTES / 4);
  char* stage = reinterpret_cast<char*>(ws + W::WARP);
  float* tq = ws + W::TAU + g * MAT;
  float* yq = ws + W::Y + g * MAT;
  float* tabs = ws + W::TAB;
  const float bq = (float)qp_bary(0, 1), dq = (float)(qp_bary(0, 0) - qp_bary(0, 1));

  for (int64_t A = (int64_t)blockIdx.x * wpb + warp; A < n_nodes; A += (int64_t)gridDim.x * wpb) {
    const int r0 = row_off[A], r1 = row_off[A + 1];
    {
      float4* h = reinterpret_cast<float4*>(H + (int64_t)r0 * HB);
      const int64_t n4 = (int64_t)(r1 - r0) * HB / 4;
      for (int64_t t = lane; t < n4; t += 32) h[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
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
      const int node[4] = {nd0.x, nd0.y, nd0.z, nd0.w};
      const char* in = stage;
      cp_async_wait<0>();
      __syncwarp();                       // the copies; the previous element's matrices are read
      const T* ge = Stage::geo_of(in);
      const float w4 = 0.25f * nodal_float(ge[GEO_VOL]);
      float d[4][3];
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int j = 0; j < 3; ++j) d[b][j] = nodal_float(ge[b * 3 + j]);
      // slot of the group's column node in row A
      int slot = -1;
#pragma unroll 1
      for (int s = r0; s < r1; s += 32) {
        const int col = s + lane < r1 ? cols[s + lane] : -1;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const unsigned hit = __ballot_sync(0xffffffffu, col == node[b]);
          if (hit && b == g) slot = s + __ffs(hit) - 1;
        }
      }
      // velocity at the group's point, then beta_qb for the four column nodes
      float be[4][2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float u[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          float sum = 0.f, own = 0.f;
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float v = nodal_value(Stage::rows_of(in)[b * 4 * C + j * C + 2 * p + h]);
            sum += v;
            own = b == g ? v : own;
          }
          u[j] = p == 0 && h == 1 ? 0.f : fmaf(bq, sum, dq * own);
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) be[b][h] = d[b][0] * u[0] + d[b][1] * u[1] + d[b][2] * u[2];
      }
      if (in_group) {
#pragma unroll
        for (int b = 0; b < 4; ++b) nodal_modes<N>(tabs + (g * 4 + b) * 2 * TW, p, be[b][0], be[b][1]);
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
      nodal_columns<N>(tabs + (g * 4 + a) * 2 * TW, p, (g == a ? bq + dq : bq) * ph.omega, sx, sy);
#pragma unroll
      for (int i = 0; i < NM; ++i) X[i] = Y[i] = 0.f;
      nodal_product<N>(tq, sx, sy, X, Y);
      if (in_group) nodal_store_rows<N>(yq, p, X, Y);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < NM; ++i) X[i] = Y[i] = 0.f;   // K_ab of the group's column node b = g
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const float la = q == a ? bq + dq : bq;
        nodal_columns<N>(tabs + (q * 4 + g) * 2 * TW, p, (q == g ? bq + dq : bq) * ph.omega, sx, sy);
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          X[i] = fmaf(la, sx[i], X[i]);
          Y[i] = fmaf(la, sy[i], Y[i]);
        }
        nodal_product<N>(ws + W::Y + q * MAT, sx, sy, X, Y);
      }
      // sum of tau over the points: the lane's columns
      float tx[NM], ty[NM];
      nodal_load_rows<N>(ws + W::TAU, p, tx, ty);
#pragma unroll 1
      for (int q = 1; q < 4; ++q) {
        nodal_load_rows<N>(ws + W::TAU + q * MAT, p, sx, sy);
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          tx[i] += sx[i];
          ty[i] += sy[i];
        }
      }
      if (in_group && slot >= 0) {
        float* rec = H + (int64_t)slot * HB;
        float dA[3], dB[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          dA[j] = a == 0 ? d[0][j] : a == 1 ? d[1][j] : a == 2 ? d[2][j] : d[3][j];
          dB[j] = g == 0 ? d[0][j] : g == 1 ? d[1][j] : g == 2 ? d[2][j] : d[3][j];
        }
        const float gab = dA[0] * dB[0] + dA[1] * dB[1] + dA[2] * dB[2];
        const float diag = 4.f * w4 * (ph.mu * gab + ph.mass_coef * (a == g ? 0.1f : 0.05f));
        const float wk = w4 * ph.rho, wl = w4 / ph.rho * gab;
        constexpr float S2 = Real<float>::SQRT2, IS2 = Real<float>::INV_SQRT2;
        // storage coordinates: lane p > 0 has the stored columns 2p, 2p + 1, lane 0 column
        // 0.  All loads of a matrix are issued before its stores: they come from L2
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          float* at = rec + part * CC + 2 * p;
          float2 v[NM];
#pragma unroll
          for (int i = 0; i < NM; ++i) v[i] = *reinterpret_cast<const float2*>(at + stor_of(i) * C);
#pragma unroll
          for (int i = 0; i < NM; ++i) {
            float x = part == 0 ? wk * X[i] + (i == 2 * p - 1 ? diag : 0.f) : wl * tx[i];
            float y = part == 0 ? wk * Y[i] + (i == 2 * p ? diag : 0.f) : wl * ty[i];
            if (p == 0) {
              x = y * (i == 0 ? 1.f : IS2);
              y = 0.f;
            } else if (i == 0) {
              x *= S2;
              y *= S2;
            }
            *reinterpret_cast<float2*>(at + stor_of(i) * C) = make_float2(v[i].x + x, v[i].y + y);
          }
        }
        if (p == 0) {
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            rec[2 * CC + j] -= w4 * dA[j];
            rec[2 * CC + 3 + j] += w4 * dB[j];
          }
        }
        // the coefficient of Im(mode 0): the Galerkin identity parts alone
        if (p == 0) {
          rec[C + 1] += diag;
        }
      }
      __syncwarp();                       // record writes before the next element's reads by other lanes
    }
  }
}

// y = H x on the assembled records; Dirichlet velocity and Im(mode 0) inputs
// are ignored and the same rows of y are zero.
//
// Bound by the record stream once enough of it is in flight.  A warp takes a few
// consecutive rows, whose records lie one behind the other, and copies them with
// their x_B through a ring of shared-memory slots that runs on across the ends
// of rows; columns and Dirichlet marks come 32 at a time, a window ahead.  A lane
// owns fixed pairs of adjacent columns of K and L (position t = row t / N, pair
// t % N) and keeps its partial sums in registers over the whole row: each
// coefficient of K is read once and feeds the three velocity components, and
// the N partial sums of an output meet once per row.  K of a Dirichlet row is not
// copied (its products are not used).
// 9,996 rows, 138 k records: N = 5 (118 MB) 35 us, N = 7 (227 MB) 52 us, N = 15
// (1.0 GB) 176 us, 5.8 TB/s; with one lane per output and one record in flight a
// warp, each coefficient of K read three times from shared memory, 48, 65 and
// 237 us.
constexpr int SPMV_WARPS = 4;   // warps (groups of rows in flight) per block
constexpr int SPMV_ROWS = 31;   // most rows a warp takes at a time (row_off in one warp load)

template <int N>
struct SpmvShape {
  // slots a warp and blocks an SM: enough records in flight at 4 to 16 warps and more an SM
  static constexpr int S = N <= 10 ? 4 : 3;
  static constexpr int SLOT = AsmLayout<N>::PWARP;
  static constexpr int BYTES = SPMV_WARPS * S * SLOT * (int)sizeof(float);
  static constexpr int FIT = (220 * 1024) / (BYTES + 1024);
  static constexpr int BLOCKS = FIT > 9 ? 9 : FIT;
};

template <int N>
__global__ void __launch_bounds__(32 * SPMV_WARPS, SpmvShape<N>::BLOCKS)
    spmv_paper_kernel(const int32_t* __restrict__ row_off, const int32_t* __restrict__ cols,
                      const float* __restrict__ H, const uint8_t* __restrict__ dmask,
                      const float* __restrict__ x, float* __restrict__ y, int64_t n_nodes, int rows) {
  using L = AsmLayout<N>;
  using K = SpmvShape<N>;
  constexpr int C = L::C, CC = L::CC, HB = L::HB, NB = 4 * C, NPOS = CC / 2, S = K::S;
  constexpr int P = (NPOS + 31) / 32;
  static_assert(C <= 32 && NB / 4 <= 32, "lane r adds the identity parts of row r");
  extern __shared__ __align__(16) float smem_f[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* ring = smem_f + warp * S * K::SLOT;
  const int64_t n_groups = (n_nodes + rows - 1) / rows;
  for (int64_t grp = (int64_t)blockIdx.x * SPMV_WARPS + warp; grp < n_groups;
       grp += (int64_t)gridDim.x * SPMV_WARPS) {
    const int64_t A0 = grp * rows;
    const int nr = n_nodes - A0 < rows ? (int)(n_nodes - A0) : rows;
    const int off = lane <= nr ? row_off[A0 + lane] : 0;
    const unsigned dir_rows = __ballot_sync(0xffffffffu, lane < nr && dmask[A0 + lane] != 0);
    const int p0 = __shfl_sync(0xffffffffu, off, 0), p1 = __shfl_sync(0xffffffffu, off, nr);
    // windows of 32 columns: [base, base + 32) and the one behind it
    auto window = [&](int base) { return base + lane < p1 ? cols[base + lane] : 0; };
    int base = p0, c_cur = window(p0), c_next = window(p0 + 32);
    int row_s = 0, end_s = __shfl_sync(0xffffffffu, off, 1);   // row of the record staged next
    float* at_s = ring;
    float* const last = ring + (S - 1) * K::SLOT;
    auto stage = [&](int p) {
      if (p < p1) {
        while (p >= end_s) end_s = __shfl_sync(0xffffffffu, off, ++row_s + 1);
        if (p - base == 32) {
          base += 32;
          c_cur = c_next;
          c_next = window(base + 32);
        }
        const float4* src = reinterpret_cast<const float4*>(H + (int64_t)p * HB) + lane;
        const int first = (dir_rows >> row_s) & 1 ? CC / 4 : 0;
#pragma unroll
        for (int j = 0; j < (HB / 4 + 31) / 32; ++j)
          if (lane + 32 * j >= first && lane + 32 * j < HB / 4) cp_async16(at_s + 4 * (lane + 32 * j), src + 32 * j);
        const float4* xb =
            reinterpret_cast<const float4*>(x + (int64_t)__shfl_sync(0xffffffffu, c_cur, p - base) * NB);
        if (lane < NB / 4) cp_async16(at_s + HB + 4 * lane, xb + lane);
      }
      cp_async_commit();
      at_s = at_s == last ? ring : at_s + K::SLOT;
    };
#pragma unroll
    for (int i = 0; i < S - 1; ++i) stage(p0 + i);
    unsigned dir_cols = 0;                       // Dirichlet marks of 32 columns from p on
    int p = p0;
    float* rec = ring;
    for (int a = 0; a < nr; ++a) {
      const int64_t A = A0 + a;
      const bool dirA = (dir_rows >> a) & 1;
      const int r1 = __shfl_sync(0xffffffffu, off, a + 1);
      float k0[P], k1[P], k2[P], kl[P], g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < P; ++j) k0[j] = k1[j] = k2[j] = kl[j] = 0.f;
      for (; p < r1; ++p) {
        stage(p + S - 1);
        if (((p - p0) & 31) == 0)
          dir_cols = __ballot_sync(0xffffffffu, p + lane < p1 && dmask[cols[p + lane]] != 0);
        const bool dirB = (dir_cols >> ((p - p0) & 31)) & 1;
        cp_async_wait<S - 1>();
        __syncwarp();
        const float* xs = rec + HB;
#pragma unroll
        for (int j = 0; j < P; ++j) {
          const int t = lane + 32 * j;
          if (t < NPOS) {
            const int c = 2 * (t % N);
            const float2 l = *reinterpret_cast<const float2*>(rec + CC + 2 * t);
            float2 v = *reinterpret_cast<const float2*>(xs + 3 * C + c);
            if (c == 0) v.y = 0.f;
            kl[j] = fmaf(l.x, v.x, fmaf(l.y, v.y, kl[j]));
            if (!dirA && !dirB) {
              const float2 k = *reinterpret_cast<const float2*>(rec + 2 * t);
              float2 v0 = *reinterpret_cast<const float2*>(xs + c);
              float2 v1 = *reinterpret_cast<const float2*>(xs + C + c);
              float2 v2 = *reinterpret_cast<const float2*>(xs + 2 * C + c);
              if (c == 0) v0.y = v1.y = v2.y = 0.f;
              k0[j] = fmaf(k.x, v0.x, fmaf(k.y, v0.y, k0[j]));
              k1[j] = fmaf(k.x, v1.x, fmaf(k.y, v1.y, k1[j]));
              k2[j] = fmaf(k.x, v2.x, fmaf(k.y, v2.y, k2[j]));
            }
          }
        }
        if (lane < C) {
          const float4 q0 = *reinterpret_cast<const float4*>(rec + 2 * CC);
          const float2 q1 = *reinterpret_cast<const float2*>(rec + 2 * CC + 4);
          const float xp = xs[3 * C + lane];
          g[0] = fmaf(q0.x, xp, g[0]);
          g[1] = fmaf(q0.y, xp, g[1]);
          g[2] = fmaf(q0.z, xp, g[2]);
          if (!dirB)
            g[3] = fmaf(q0.w, xs[lane], fmaf(q1.x, xs[C + lane], fmaf(q1.y, xs[2 * C + lane], g[3])));
        }
        rec = rec == last ? ring : rec + K::SLOT;
        __syncwarp();
      }
      // the slot before the next record's is free: the partial sums of the row meet there
      float* part = rec == ring ? last : rec - K::SLOT;
#pragma unroll
      for (int j = 0; j < P; ++j) {
        const int t = lane + 32 * j;
        if (t < NPOS) {
          part[t] = k0[j];
          part[NPOS + t] = k1[j];
          part[2 * NPOS + t] = k2[j];
          part[3 * NPOS + t] = kl[j];
        }
      }
      __syncwarp();
      if (lane < C) {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          float s = g[f];
#pragma unroll
          for (int k = 0; k < N; ++k) s += part[f * NPOS + lane * N + k];
          y[A * NB + f * C + lane] = (lane == 1 || (dirA && f < 3)) ? 0.f : s;
        }
      }
      __syncwarp();
    }
    cp_async_wait<0>();                  // the groups still open are empty
    __syncwarp();
  }
}

// The same product for records of a few rows (N <= 3), where a record is less
// work than its staging: a lane owns one output (field, row) and reads the row
// of K or L and x_B directly; 32 / 8N records (N = 1, 2) share a warp.  9,996
// rows: N = 2 15.6 us, N = 3 22.5 us (22.5 and 26.3 with one record at a time staged
// in shared memory).
template <int N>
__global__ void __launch_bounds__(128)
    spmv_small_kernel(const int32_t* __restrict__ row_off, const int32_t* __restrict__ cols,
                      const float* __restrict__ H, const uint8_t* __restrict__ dmask,
                      const float* __restrict__ x, float* __restrict__ y, int64_t n_nodes) {
  using L = AsmLayout<N>;
  constexpr int C = L::C, CC = L::CC, HB = L::HB, NB = 4 * C, SUB = 32 / NB;
  static_assert(SUB >= 1, "one lane an output");
  const int lane = threadIdx.x & 31;
  const int sub = lane / NB, o = lane - sub * NB, f = o / C, r = o - f * C;
  const int64_t A = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (A >= n_nodes) return;
  float s = 0.f, g = 0.f;
  if (sub < SUB) {
    const int r1 = row_off[A + 1];
    const int mat = (f < 3 ? 0 : CC) + r * C;
#pragma unroll 4
    for (int p = row_off[A] + sub; p < r1; p += SUB) {
      const float* rec = H + (int64_t)p * HB;
      const int B = cols[p];
      const float* xb = x + (int64_t)B * NB;
      const bool dirB = dmask[B] != 0;
      const bool drop = dirB && f < 3;
      float t = 0.f;
#pragma unroll
      for (int c = 0; c < N; ++c) {
        const float2 a = *reinterpret_cast<const float2*>(rec + mat + 2 * c);
        float2 v = *reinterpret_cast<const float2*>(xb + f * C + 2 * c);
        if (drop) v.x = 0.f;
        if (drop || c == 0) v.y = 0.f;
        t = fmaf(a.x, v.x, fmaf(a.y, v.y, t));
      }
      s += t;
      if (f < 3) {
        g = fmaf(rec[2 * CC + f], xb[3 * C + r], g);
      } else if (!dirB) {
        g = fmaf(rec[2 * CC + 3], xb[r], g);
        g = fmaf(rec[2 * CC + 4], xb[C + r], g);
        g = fmaf(rec[2 * CC + 5], xb[2 * C + r], g);
      }
    }
  }
  s += g;
#pragma unroll
  for (int d = NB; SUB > 1 && d < 32; d *= 2) s += __shfl_down_sync(0xffffffffu, s, d);
  if (lane < NB) y[A * NB + lane] = (r == 1 || (dmask[A] != 0 && f < 3)) ? 0.f : s;
}

// One colour of a symmetric block Gauss-Seidel sweep with the assembled
// records: for each node A of the colour (rows[0..n_rows)),
//   z_A = Binv_A (r_A - sum_{B != A} H_AB z_B)
// with z read as it stands (earlier colours of this sweep already updated).
// Binv: inverted nodal diagonal blocks, column-major (precond.cu).  One warp
// per row.  A colour holds only a few thousand rows (a few warps per SM), so
// each warp keeps SGS_STAGES - 1 copies in flight through a ring of
// SGS_STAGES shared-memory slots: first the row's connections (one record
// plus z_B per slot), then its inverted block in chunks of whole columns, so
// that the block is already on its way while the last connections are
// multiplied.  The terms of every output are added in the same order as a
// plain loop over the connections and then over the block's columns.
constexpr int SGS_STAGES = 2;
constexpr int SGS_WARPS = 2;   // warps (rows in flight) per block

template <int N>
struct SgsChunks {
  static constexpr int NB = 8 * N;
  static constexpr int CPC = AsmLayout<N>::PWARP / NB;     // block columns per slot
  static constexpr int NCH = (NB + CPC - 1) / CPC;         // chunks per block
};

template <int N>
__global__ void __launch_bounds__(256)
    sgs_colour_kernel(const int32_t* __restrict__ rows, int64_t n_rows, const int32_t* __restrict__ row_off,
                      const int32_t* __restrict__ cols, const float* __restrict__ H,
                      const float* __restrict__ binv, const uint8_t* __restrict__ dmask,
                      const float* __restrict__ r, float* __restrict__ z, int diag_only) {
  using L = AsmLayout<N>;
  using K = SgsChunks<N>;
  constexpr int C = L::C, CC = L::CC, HB = L::HB, NB = 4 * C, S = SGS_STAGES;
  constexpr int CPC = K::CPC, NCH = K::NCH;
  constexpr int R = (NB + 31) / 32;
  static_assert(CPC >= 1 && (CPC * NB) % 4 == 0, "block chunk must be whole 16-byte copies");
  extern __shared__ __align__(16) float smem_f[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  float* buf0 = smem_f + warp * S * L::PWARP;   // [S][PWARP]
  for (int64_t k = (int64_t)blockIdx.x * wpb + warp; k < n_rows; k += (int64_t)gridDim.x * wpb) {
    const int A = rows[k];
    const bool dirA = dmask[A] != 0;
    float acc[R], rv[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int o = lane + 32 * j;
      acc[j] = 0.f;
      rv[j] = o < NB ? r[(int64_t)A * NB + o] : 0.f;
    }
    const int r0 = row_off[A], r1 = row_off[A + 1];
    // position of the diagonal connection in the row (rows hold at most a
    // few dozen connections): the i-th off-diagonal one is r0 + i, or
    // r0 + i + 1 from the diagonal on
    int pd = r1;
    for (int b = r0; b < r1; b += 32) {
      const unsigned hit = __ballot_sync(0xffffffffu, b + lane < r1 && cols[b + lane] == A);
      if (hit) {
        pd = b + __ffs(hit) - 1;
        break;
      }
    }
    // diag_only: every z_B is zero (the sweep's first colour), so is the sum
    const int n_off = diag_only ? 0 : (r1 - r0) - (pd < r1 ? 1 : 0);
    const int n_items = n_off + NCH;
    auto conn = [&](int i) { return r0 + i + (r0 + i >= pd ? 1 : 0); };
    const float* Bi = binv + (int64_t)A * NB * NB;
    // one commit group per ring position, empty past the row's end, so that
    // waiting for all but the newest S - 1 groups always means "slot i landed"
    auto stage = [&](int i) {
      float* dst = buf0 + (i % S) * L::PWARP;
      if (i < n_off) {
        const int p = conn(i);
        const float4* src = reinterpret_cast<const float4*>(H + (int64_t)p * HB);
        for (int t = lane; t < HB / 4; t += 32) cp_async16(dst + 4 * t, src + t);
        const float4* zb = reinterpret_cast<const float4*>(z + (int64_t)cols[p] * NB);
        for (int t = lane; t < NB / 4; t += 32) cp_async16(dst + HB + 4 * t, zb + t);
      } else if (i < n_items) {
        const int c0 = (i - n_off) * CPC;
        const int ncol = NB - c0 < CPC ? NB - c0 : CPC;
        const float4* src = reinterpret_cast<const float4*>(Bi + (int64_t)c0 * NB);
        for (int t = lane; t < ncol * NB / 4; t += 32) cp_async16(dst + 4 * t, src + t);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < S - 1; ++i) stage(i);
    float tv[R], out[R];
#pragma unroll
    for (int j = 0; j < R; ++j) tv[j] = out[j] = 0.f;
    for (int i = 0; i < n_items; ++i) {
      // slot (i + S - 1) % S was used in iteration i - 1 (synced below)
      stage(i + S - 1);
      cp_async_wait<S - 1>();
      __syncwarp();
      float* rec = buf0 + (i % S) * L::PWARP;
      if (i < n_off) {
        float* xs = rec + HB;
        const bool dirB = dmask[cols[conn(i)]] != 0;
        for (int t = lane; t < NB; t += 32) {
          const int f = t / C, c = t - f * C;
          if (c == 1 || (dirB && f < 3)) xs[t] = 0.f;
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int o = lane + 32 * j;
          if (o < NB) {
            const int f = o / C, rr = o - f * C;
            float s = acc[j];
            if (f < 3) {
              const float2* Kr = reinterpret_cast<const float2*>(rec + rr * C);
              const float2* xi = reinterpret_cast<const float2*>(xs + f * C);
#pragma unroll
              for (int c = 0; c < C / 2; ++c) {
                const float2 a = Kr[c], b = xi[c];
                s = fmaf(a.x, b.x, fmaf(a.y, b.y, s));
              }
              s = fmaf(rec[2 * CC + f], xs[3 * C + rr], s);
            } else {
              const float2* Lr = reinterpret_cast<const float2*>(rec + CC + rr * C);
              const float2* xp = reinterpret_cast<const float2*>(xs + 3 * C);
#pragma unroll
              for (int c = 0; c < C / 2; ++c) {
                const float2 a = Lr[c], b = xp[c];
                s = fmaf(a.x, b.x, fmaf(a.y, b.y, s));
              }
              s = fmaf(rec[2 * CC + 3], xs[rr], s);
              s = fmaf(rec[2 * CC + 4], xs[C + rr], s);
              s = fmaf(rec[2 * CC + 5], xs[2 * C + rr], s);
            }
            acc[j] = s;
          }
        }
      } else {
        // t = r_A - (off-diagonal sum), kept in registers; each block column
        // takes its entry of t from the lane that holds it
        if (i == n_off) {
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const int o = lane + 32 * j;
            const int f = o / C, c = o - f * C;
            tv[j] = (o >= NB || c == 1 || (dirA && f < 3)) ? 0.f : rv[j] - acc[j];
          }
        }
        const int c0 = (i - n_off) * CPC;
        const int ncol = NB - c0 < CPC ? NB - c0 : CPC;
        for (int u = 0; u < ncol; ++u) {
          const int col = c0 + u;
          float xc = 0.f;
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const float v = __shfl_sync(0xffffffffu, tv[j], col & 31);
            if ((col >> 5) == j) xc = v;
          }
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const int o = lane + 32 * j;
            if (o < NB) out[j] = fmaf(rec[u * NB + o], xc, out[j]);
          }
        }
      }
      __syncwarp();
    }
    // the groups still open are empty (positions past the row's end)
    cp_async_wait<0>();
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int o = lane + 32 * j;
      if (o < NB) z[(int64_t)A * NB + o] = out[j];
    }
    __syncwarp();
  }
}

template <int N>
int launch_sgs_colour(const int32_t* rows, int64_t n_rows, const int32_t* row_off, const int32_t* cols,
                      const float* H, const float* binv, const uint8_t* dmask, const float* r, float* z,
                      int diag_only, cudaStream_t st) {
  using L = AsmLayout<N>;
  if (n_rows <= 0) return 0;
  int warps = SGS_WARPS;
  while (warps > 1 && (size_t)warps * SGS_STAGES * L::PWARP * sizeof(float) > 200 * 1024) --warps;
  const size_t smem = (size_t)warps * SGS_STAGES * L::PWARP * sizeof(float);
  if (smem > 227 * 1024) return -6;
  cudaFuncSetAttribute(sgs_colour_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int64_t blocks = (n_rows + warps - 1) / warps;
  if (blocks > 152 * 64) blocks = 152 * 64;
  count_launches(1);
  sgs_colour_kernel<N><<<(int)blocks, warps * 32, smem, st>>>(rows, n_rows, row_off, cols, H, binv, dmask, r, z,
                                                               diag_only);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

template <typename T, int N>
int launch_assemble_paper(const int32_t* node_off, const int32_t* node_elem, const int32_t* row_off,
                          const int32_t* cols, const int4* tets, const T* geo, const T* u0, const T* uc, const T* tau,
                          Phys<float> ph, float* H, int64_t n_nodes, cudaStream_t st) {
  if (n_nodes <= 0) return 0;
  if constexpr (N <= NODAL_MAX_N) {
    using U = typename PairOfStore<T>::V;
    const size_t smem = (size_t)4 * (NodalAssembly<N>::WARP * sizeof(float) + NodalStage<T, U, N>::BYTES);
    if (cudaFuncSetAttribute(nodal_assemble_kernel<T, U, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
      return -2;
    const int64_t blocks = std::min<int64_t>((n_nodes + 3) / 4, 152 * 32);
    count_launches(1);
    nodal_assemble_kernel<T, U, N><<<(int)blocks, 128, smem, st>>>(node_off, node_elem, row_off, cols, tets, geo,
                                                                   reinterpret_cast<const U*>(uc), tau, ph, H, n_nodes);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
  } else {
    using L = AsmLayout<N>;
    int warps = 4;
    while (warps > 1 && (size_t)warps * L::WARP * sizeof(float) > 200 * 1024) --warps;
    const size_t smem = (size_t)warps * L::WARP * sizeof(float);
    if (smem > 227 * 1024) return -6;
    cudaFuncSetAttribute(assemble_paper_kernel<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int64_t blocks = (n_nodes + warps - 1) / warps;
    if (blocks > 152 * 32) blocks = 152 * 32;
    count_launches(1);
    assemble_paper_kernel<T, N><<<(int)blocks, warps * 32, smem, st>>>(node_off, node_elem, row_off, cols, tets,
                                                                      geo, u0, tau, ph, H, n_nodes);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
  }
}

template <int N>
int launch_spmv_paper(const int32_t* row_off, const int32_t* cols, const float* H, const uint8_t* dmask,
                      const float* x, float* y, int64_t n_nodes, cudaStream_t st) {
  if (n_nodes <= 0) return 0;
  // 9,996 rows: N = 3 22.5 us (25.8 with the ring), N = 4 32.5 (27.1)
  if constexpr (N <= 3) {
    count_launches(1);
    spmv_small_kernel<N><<<(unsigned)((n_nodes + 3) / 4), 128, 0, st>>>(row_off, cols, H, dmask, x, y, n_nodes);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
  } else {
    using K = SpmvShape<N>;
    if (cudaFuncSetAttribute(spmv_paper_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::BYTES) != cudaSuccess)
      return -2;
    const int64_t warps = (int64_t)152 * K::BLOCKS * SPMV_WARPS;   // one wave
    const int rows = (int)std::min<int64_t>((n_nodes + warps - 1) / warps, SPMV_ROWS);
    const int64_t groups = (n_nodes + rows - 1) / rows;
    const int64_t blocks = std::min<int64_t>((groups + SPMV_WARPS - 1) / SPMV_WARPS, 152 * 64);
    count_launches(1);
    spmv_paper_kernel<N><<<(int)blocks, 32 * SPMV_WARPS, K::BYTES, st>>>(row_off, cols, H, dmask, x, y, n_nodes, rows);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
  }
}

int assembled_record_floats(int N) { return 2 * (2 * N) * (2 * N) + 8; }

#define TS_INST_ASM(T, N)                                                                                   \
  template int launch_assemble_paper<T, N>(const int32_t*, const int32_t*, const int32_t*, const int32_t*,  \
                                           const int4*, const T*, const T*, const T*, const T*, Phys<float>, float*, \
                                           int64_t, cudaStream_t);
TS_FOR_EACH_N(TS_INST_ASM, float)
TS_FOR_EACH_N(TS_INST_ASM, double)
#define TS_INST_SGS(T, N)                                                                                  \
  template int launch_sgs_colour<N>(const int32_t*, int64_t, const int32_t*, const int32_t*, const float*, \
                                    const float*, const uint8_t*, const float*, float*, int, cudaStream_t);
TS_FOR_EACH_N(TS_INST_SGS, float)
#define TS_INST_SPMV(T, N)                                                                          \
  template int launch_spmv_paper<N>(const int32_t*, const int32_t*, const float*, const uint8_t*, \
                                    const float*, float*, int64_t, cudaStream_t);
TS_FOR_EACH_N(TS_INST_SPMV, float)

}  // namespace ts
