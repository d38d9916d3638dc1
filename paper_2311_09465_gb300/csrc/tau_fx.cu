// tau of eq. (3D-tau) to FP64 accuracy without FP64 arithmetic: FP32 eigenpairs
// (onesided.cuh) and Newton corrections whose residuals are formed in 58-bit
// fixed point on the integer multiply-add pipe.
//
// With the point scaled so that the eigenvalues of M lie in (0, 1] and X near
// M^{-1/2}, one correction is
//   R = I - X M X,   S E + E S = R with S = M^{1/2},   X <- X + E.
// Only R needs more than FP32 (it is the small difference of large terms); the
// Sylvester equation is solved in the FP32 eigenbasis, E_ab = R_ab / (s_a + s_b).
// The start X0 = U diag(1/s) U^T rounded to 29 bits leaves |R| near 1e-6; the
// first correction leaves |R| near 1e-11 and the second is below the output's
// rounding.  With the eigenbasis held fixed the corrections converge only from FP32
// eigenpairs that resolve the smallest eigenvalue, and the integers hold R only while
// |M X| stays near 1; a point whose smallest eigenvalue is below FX_LAMBDA of its
// scale, or whose last R is not small, is therefore put on a list, and
// tau_polish_kernel redoes it in FP64 (tau.cu; the point's result here is overwritten).
// Without the list such points came out wrong by up to a factor of 1000 (one harmonic
// without a mean, u h / nu = 3e4 and above).
//
// Fixed point: a value v, |v| <= 1, is the integer V = v 2^58, split into two
// signed limbs V = 2^29 h + l, |h| <= 2^29, |l| <= 2^28, l kept as FP32 (24 bits:
// v is then good to 2^-54).  A dot product of length n <= 29 sums h h' exactly in
// a 64-bit integer (29 * 2^58 < 2^63) and the mixed products h l' + l h', 2^29
// smaller, in FP32; l l' is left out.  A term is one 32 x 32 -> 64 bit multiply-add
// (4.8 issue cycles of an SM sub-partition, measured with all operands in vector
// registers) and two FP32 ones, about 7 cycles against 12 to 15 for a double-float
// term, with an absolute error near 2^-53 instead of 2^-47.  With the mixed
// products in a second 64-bit accumulator it was 14 cycles.  In R the scale of X
// enters twice, so R is known to about cond(M) 2^-53.
//
// Mapping: as tau32_kernel (tau.cu), a group of N lanes owns a point and lane p
// the columns 2p-1 and 2p of every matrix.  A product reads the left matrix
// row by row from shared memory (16-byte loads, the same address in the whole
// group where a full product is needed) against the lane's columns in registers.
// Symmetric results (M, R, E) are formed for half of their entries: rows
// 2p-1 .. 2p+N-1 (cyclic) of the lane's two columns cover every pair (r, s), and
// both triangles are written.  The loops over rows stay rolled: a correction is
// one instruction stream of a few hundred instructions, not of several thousand.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "ddfloat.cuh"
#include "kernels.h"
#include "onesided.cuh"

namespace ts {

namespace {

constexpr int FX_MAX_IT = 10;
constexpr float FX_ORTHO2 = 1e-6f;   // leaves cosines near 1e-6: the corrections absorb them
// Smallest eigenvalue, of a point's scale of 1, that this form takes.  tau's error there
// is a few 2^-54 / lambda, up to 6e-11 at 2^-20, below the double-float refinement's and within
// ten times the FP64 Jacobi form's (five kinds of flow, N = 2 to 15).  FP64 costs 15 times
// as much a point: with 2^-14 as the line, one harmonic without a mean at u h / nu = 1e3, N = 7,
// 187,266 tetrahedra, took 128 ms instead of 12, a reversing flow at N = 15 177 instead of 8.5.
constexpr float FX_LAMBDA = 9.5367431640625e-7f;
// Pivots of the FP32 factor below this mean a point for the list: a pivot is no smaller
// than the smallest eigenvalue, and FP32 rounding, n 2^-24, is about as large
constexpr float FX_PIVOT = 0.25f * FX_LAMBDA;
// Bound of |R| (2-norm, as n times the largest entry) in a correction.  With a smallest
// eigenvalue of k times its FP32 value y = X M^{1/2} starts at k^{1/2} in its direction and goes
// to y + k^{1/2} (1 - y^2) / 2: unbounded, k = 4 would end at -1, a negative root of M^{-1}
constexpr float FX_STEP = 0.5f;
// Smallest diagonal entry that this form takes.  Where a mode hardly couples to the
// others (a cosine without a mean, N = 2: its sine) the entry is an eigenvalue, which
// floating point has to a relative 2^-53 and fixed point to 2^-54 of the scale: 1e-14
// of it at 2^-8.  Tests and bench: above 2^-6.
constexpr float FX_DIAGONAL = 3.90625e-3f;

using i64 = long long;

// acc += a b; written out because a reassociated sum of products costs 64-bit adds
__device__ __forceinline__ void fx_mad(i64& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

struct __align__(8) Limbs {
  int h;
  float l;
};

__device__ __forceinline__ Limbs fx_split(i64 v) {
  const int l = (int)((unsigned)v << 3) >> 3;   // the low 29 bits, signed
  return {(int)((v - l) >> 29), (float)l};
}
__device__ __forceinline__ i64 fx_join(int h, float l) { return ((i64)h << 29) + (int)l; }

// Conversions between FP32 and 64-bit integers by way of 32 bits: the direct
// instructions run on the FP64 pipe, at 1/64 of the FP32 rate.
// |x| < 2^58, rounded to the nearest integer
__device__ __forceinline__ i64 fx_int(float x) {
  const int hi = __float2int_rn(x * 3.7252902984619140625e-9f);           // 2^-28
  return ((i64)hi << 28) + __float2int_rn(fmaf((float)hi, -268435456.f, x));
}
__device__ __forceinline__ float fx_float(i64 v) {
  return fmaf((float)(int)(v >> 32), 4294967296.f, (float)(unsigned)v);
}

// v sqrt(2) for |v| <= 2^58 (rounded to the last place)
__device__ __forceinline__ i64 fx_sqrt2(i64 v) {
  constexpr i64 S = 6521908912666391106;        // sqrt(2) 2^62
  return (__mul64hi(v << 4, S) + 2) >> 2;
}

__device__ __forceinline__ i64 fx_from_dd(dd a) {   // |a| <= 1
  constexpr float B = 288230376151711744.f;         // 2^58
  return fx_int(a.hi * B) + fx_int(a.lo * B);
}

// V 2^e as a double, rounded to nearest (ties away from zero)
__device__ __forceinline__ double fx_to_double(i64 v, int e) {
  if (v == 0) return 0.0;
  const unsigned long long u = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int lz = __clzll((i64)u);
  const unsigned long long m = u << lz;
  unsigned long long b = (m >> 11) + ((m >> 10) & 1);
  b += (unsigned long long)(1022 + 63 - lz + e) << 52;
  return __longlong_as_double((i64)(b | (v < 0 ? 1ull << 63 : 0ull)));
}

// Sums over j of row[j] a[j] and row[j] b[j], as integers times 2^-58; row: limb
// pairs stored one place off (entry j at j + 1), so that a lane's columns 2p-1
// and 2p are one 16-byte unit.
template <int NM>
__device__ __forceinline__ void fx_dot2(const int4* __restrict__ row, const Limbs (&a)[NM], const Limbs (&b)[NM],
                                        const float (&ah)[NM], const float (&bh)[NM], i64& va, i64& vb) {
  i64 h0 = 0, h1 = 0;
  float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
#pragma unroll
  for (int j = 0; j < NM; ++j) {
    const int4 r = row[(j + 1) / 2];
    const int rh = (j & 1) ? r.x : r.z;
    const float rl = __int_as_float((j & 1) ? r.y : r.w), rf = (float)rh;
    fx_mad(h0, rh, a[j].h);
    fx_mad(h1, rh, b[j].h);
    x0 = fmaf(rf, a[j].l, x0);
    x1 = fmaf(rf, b[j].l, x1);
    y0 = fmaf(rl, ah[j], y0);
    y1 = fmaf(rl, bh[j], y1);
  }
  // mixed products times 2^-29: below 2^31.4 (rows and columns have 2-norms of at
  // most 1), converted as half of it
  constexpr float U = 1.f / 1073741824.f;   // 2^-30
  va = h0 + ((i64)__float2int_rn((x0 + y0) * U) << 1);
  vb = h1 + ((i64)__float2int_rn((x1 + y1) * U) << 1);
}

template <int W>
__device__ __forceinline__ void load_floats(const float* src, float (&dst)[W]) {
#pragma unroll
  for (int j = 0; j < W / 4; ++j) {
    const float4 v = reinterpret_cast<const float4*>(src)[j];
    dst[4 * j] = v.x;
    dst[4 * j + 1] = v.y;
    dst[4 * j + 2] = v.z;
    dst[4 * j + 3] = v.w;
  }
}

// a row from registers (times f), one place off
template <int NM, int W>
__device__ __forceinline__ void store_floats(float* dst, const float (&v)[NM], float f) {
#pragma unroll
  for (int j = 0; j < W / 4; ++j) {
    if (4 * j > NM) break;
    float t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = 4 * j + k - 1;
      t[k] = i >= 0 && i < NM ? v[i < 0 ? 0 : i >= NM ? NM - 1 : i] * f : 0.f;
    }
    reinterpret_cast<float4*>(dst)[j] = make_float4(t[0], t[1], t[2], t[3]);
  }
}
}  // namespace

template <int N>
struct FxLayout {
  static constexpr int NM = 2 * N - 1, C = 2 * N, L = N - 1, GPW = 32 / N;
  // entry i of a row is stored at i + 1; a row of limbs is an odd number of 16-byte
  // units, so that 16-byte reads of different rows by the lanes of a group spread over
  // the banks (rows of floats are mostly read by the whole group at once: kept short,
  // which makes it 12 warps an SM at N = 7 instead of 10)
  static constexpr int LDQ = (N & 1) ? 2 * N : 2 * N + 2;            // limb pairs a row
  static constexpr int LDF = (2 * N + 3) & ~3;                       // floats a row
  // in 4-byte words
  static constexpr int M = 0;                           // [NM][LDQ] limbs
  static constexpr int X = M + 2 * NM * LDQ;            // [NM][LDQ] limbs
  static constexpr int F = X + 2 * NM * LDQ;            // [NM][LDF]: h_a, R, U^T R, E
  static constexpr int U = F + NM * LDF;                // [NM][LDF]: row a = sqrt(eigenvalue a), eigenvector a
  static constexpr int END = U + NM * LDF;
  static constexpr int TW = 2 * N - 1;                  // modes -(N-1) .. N-1
  static constexpr int T = F;                           // [3][2][TW] limbs of the modes of w_m: over F, U
  static constexpr int HD = T + 2 * 3 * 2 * TW;         // [NH] complex 64-bit diagonals of sum_m C_m C_m
  static constexpr int NH = N * (N + 1) / 2 + N - 1;
  static constexpr int TEND = HD + 4 * NH;
  static constexpr int OUTP = M;                        // packed tau (doubles) over M
  static constexpr int RAW0 = END > TEND ? END : TEND;
  static constexpr int RAW1 = (RAW0 > 2 * Dims<N>::NT_PAD ? RAW0 : 2 * Dims<N>::NT_PAD);
  static constexpr int RAW = (RAW1 + 3) & ~3;
  static constexpr int GROUP = RAW + ((4 - RAW) % 32 + 32) % 32;   // groups in different banks
  static constexpr int WARP = GPW * GROUP;
};

// y: the velocity field as double-float pairs [V][4][C]; nu2 2^nu2_exp = C_I nu^2; hard: the list
// (HARD_LIST in kernels.h).  Blocks of 128 threads an SM:
// N <= 3 6 (85 registers; N = 3, 187,266 tetrahedra: 735 us, 751 with 4), N = 4, 5 4 (2.63 ms at N = 5,
// 2.74 with 2, 2.81 with 5), N = 7 3, above that the compiler's choice (N = 10 with 3: 6.1 ms, 5.6 so).
template <int N>
__global__ void __launch_bounds__(128, N <= 3 ? 6 : N <= 5 ? 4 : N == 7 ? 3 : 1) tau_fx_kernel(const int4* __restrict__ tets, const double* __restrict__ geo,
                                                     const float2* __restrict__ y, int64_t n_qp,
                                                     double* __restrict__ tau_out, dd nu2, int nu2_exp,
                                                     unsigned* __restrict__ hard,
                                                     float* __restrict__ eig_out) {
  using Lt = FxLayout<N>;
  constexpr int NM = Lt::NM, C = Lt::C, L = Lt::L, LDQ = Lt::LDQ, LDF = Lt::LDF, GPW = Lt::GPW, TW = Lt::TW;
  constexpr int NT = Dims<N>::NT, NTP = Dims<N>::NT_PAD;
  extern __shared__ __align__(16) int fx_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / N, p = lane - (lane / N) * N;
  const bool in_group = g < GPW;
  const int first = in_group ? g * N : 0;               // first lane of the group
  int* base = fx_smem + warp * Lt::WARP + (in_group ? g : 0) * Lt::GROUP;
  Limbs* Ms = reinterpret_cast<Limbs*>(base + Lt::M);
  Limbs* Xs = reinterpret_cast<Limbs*>(base + Lt::X);
  float* F = reinterpret_cast<float*>(base + Lt::F);
  float* U = reinterpret_cast<float*>(base + Lt::U);
  Limbs* T = reinterpret_cast<Limbs*>(base + Lt::T);
  longlong2* Hd = reinterpret_cast<longlong2*>(base + Lt::HD);
  // the lane's columns, and whether it has a first one
  const int cx = 2 * p - 1, cy = 2 * p;
  const bool hx = in_group && p > 0, hy = in_group;
  // row o of the lane's half: (2p - 1 + o) mod NM
  auto half_row = [&](int o) {
    int r = 2 * p - 1 + o;
    if (r < 0) r += NM;
    return r >= NM ? r - NM : r;
  };

  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t qb = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * GPW; qb < n_qp; qb += warps_total * GPW) {
    const bool live = in_group && qb + g < n_qp;
    const int64_t gq = live ? qb + g : qb;              // idle lanes redo the warp's first point, unstored
    const int64_t e = gq >> 2;
    const int q = (int)(gq & 3);
    // ---- w_m = sum_i L_im u_i for mode p, G = L L^T (double-float)
    dd diff;
    int ed;
    float n2 = 0.f;
    __syncwarp();
    {
      const double* gg = geo + e * GEO_STRIDE + GEO_G;
      const dd gxx = dd_split(gg[0]), gxy = dd_split(gg[1]), gxz = dd_split(gg[2]), gyy = dd_split(gg[3]),
               gyz = dd_split(gg[4]), gzz = dd_split(gg[5]);
      // C_I nu^2 G:G = diff 2^ed, from G 2^-eg: squares of 1 / h^2 leave FP32's range (and
      // from h = 1e8 on their low parts) long before anything else does
      const int eg = min((int)((__float_as_uint(gxx.hi) >> 23) & 0xff) - 127, 126);
      const float f = __uint_as_float((unsigned)(127 - eg) << 23);
      const dd sxx = dd_scale(gxx, f), sxy = dd_scale(gxy, f), sxz = dd_scale(gxz, f), syy = dd_scale(gyy, f),
               syz = dd_scale(gyz, f), szz = dd_scale(gzz, f);
      const dd off = dd_fma(sxy, sxy, dd_fma(sxz, sxz, dd_mul(syz, syz)));
      const dd dia = dd_fma(sxx, sxx, dd_fma(syy, syy, dd_mul(szz, szz)));
      diff = dd_mul(nu2, dd_add(dia, dd_scale(off, 2.f)));
      ed = nu2_exp + 2 * eg;
      const dd l00 = dd_sqrt(gxx), r00 = dd_rcp(l00);
      const dd l10 = dd_mul(gxy, r00), l20 = dd_mul(gxz, r00);
      const dd l11 = dd_sqrt(dd_fma(dd_neg(l10), l10, gyy)), r11 = dd_rcp(l11);
      const dd l21 = dd_mul(dd_fma(dd_neg(l20), l10, gyz), r11);
      const dd l22 = dd_sqrt(dd_fma(dd_neg(l21), l21, dd_fma(dd_neg(l20), l20, gzz)));
      const int4 nd = tets[e];
      const int node[4] = {nd.x, nd.y, nd.z, nd.w};
      // lambda_a(q) = b + (a - b) delta_aq: u = b sum_a y_a + (a - b) y_q
      constexpr double BQ = qp_bary(0, 1), DQ = qp_bary(0, 0) - qp_bary(0, 1);
      constexpr float BH = (float)BQ, BL = (float)(BQ - (double)BH), DH = (float)DQ, DL = (float)(DQ - (double)DH);
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        dd u[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          dd v[4];
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const float2 f = y[(int64_t)node[a] * 4 * C + i * C + 2 * p + h];
            v[a] = dd{f.x, f.y};
          }
          const dd vq = q == 0 ? v[0] : q == 1 ? v[1] : q == 2 ? v[2] : v[3];
          const dd sum = dd_add(dd_add(v[0], v[1]), dd_add(v[2], v[3]));
          u[i] = dd_fma(dd{DH, DL}, vq, dd_mul(dd{BH, BL}, sum));
          if (p == 0 && h == 1) u[i] = dd{0.f, 0.f};
        }
        const dd w0 = dd_fma(l00, u[0], dd_fma(l10, u[1], dd_mul(l20, u[2])));
        const dd w1 = dd_fma(l11, u[1], dd_mul(l21, u[2]));
        const dd w2 = dd_mul(l22, u[2]);
        // parked as pairs in the table's places until the scale is known
        float2* park = reinterpret_cast<float2*>(T + h * TW + L + p);
        if (in_group) {
          park[0] = make_float2(w0.hi, w0.lo);
          park[2 * TW] = make_float2(w1.hi, w1.lo);
          park[4 * TW] = make_float2(w2.hi, w2.lo);
        }
        n2 = fmaf(w0.hi, w0.hi, fmaf(w1.hi, w1.hi, fmaf(w2.hi, w2.hi, n2)));
      }
    }
    // |C_m| <= beta_m = |w_m0| + 2 sum_n |w_mn|, so |sum_m C_m^2| <= sum_m beta_m^2 <=
    // (|w_0| + 2 sum_n |w_n|)^2, |w_n| over the three m: with that plus c at most 1 after
    // the scale 2^-ex, M's eigenvalues (and so its entries) are at most 1
    float bound;
    {
      const float mag = sqrtf(n2) * (p == 0 ? 1.f : 2.f);
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) sum += __shfl_sync(0xffffffffu, mag, first + j);
      bound = 1.0001f * sqrtf(fmaf(sum, sum, ldexpf(diff.hi, ed)));
    }
    const bool finite = bound < 4e18f && bound > 2e-19f;   // 2^-ex squared stays in range
    int ex = 0;
    if (finite) frexpf(bound, &ex);
    const float sc = ldexpf(1.f, -ex);
    const i64 cfix = finite ? fx_from_dd(dd_scale(diff, ldexpf(1.f, ed - 2 * ex))) : (1ll << 57);
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {
      Limbs* tr = T + m * 2 * TW + L;                   // mode k at tr[k], its imaginary part at tr[TW + k]
      const float2 wr = *reinterpret_cast<const float2*>(tr + p), wi = *reinterpret_cast<const float2*>(tr + TW + p);
      const Limbs re = fx_split(finite ? fx_from_dd(dd{wr.x * sc, wr.y * sc}) : 0);
      const Limbs im = fx_split(finite ? fx_from_dd(dd{wi.x * sc, wi.y * sc}) : 0);
      __syncwarp();
      if (in_group) {
        tr[p] = re;
        tr[TW + p] = im;
        if (p > 0) {
          tr[-p] = re;
          tr[TW - p] = Limbs{-im.h, -im.l};
        }
      }
    }
    __syncwarp();
    // ---- H = sum_m T_m T_m, T_m the complex Hermitian Toeplitz matrix t_{i-j} of w_m
    // (|i - j| < N), by diagonals: with rows and columns numbered 0..2L, L = N - 1,
    //   H_0j = sum_k t_{-k} t_{k-j},   H_ij = H_{i-1,j-1} + t_i t_{-j} for i, j <= L,
    // constant along a diagonal where i <= L <= j, and H_{2L-i,2L-j} = conj H_ij: an
    // entry costs one product instead of a row of them.  Lane p takes diagonal p
    // (L + 1 products for its first entry, one for each of the L - p others) and the
    // first entry of diagonal 2L + 1 - p (p products): 2L + 1 products a lane and m
    // (N = 7, 187,266 tetrahedra: 7.3 ms for the whole kernel, 8.7 with half of the
    // dense products).
    {
      i64 hr = 0, hi = 0;
      auto add = [&](int ka, int kb) {                  // += sum_m t_ka t_kb
        i64 r = 0, i = 0;
        float xr = 0.f, xi = 0.f;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const Limbs* tr = T + m * 2 * TW + L;
          const Limbs ar = tr[ka], ai = tr[TW + ka], br = tr[kb], bi = tr[TW + kb];
          const float arf = (float)ar.h, aif = (float)ai.h, brf = (float)br.h, bif = (float)bi.h;
          fx_mad(r, ar.h, br.h);
          fx_mad(i, ar.h, bi.h);
          fx_mad(r, -ai.h, bi.h);
          fx_mad(i, ai.h, br.h);
          xr = fmaf(arf, br.l, fmaf(ar.l, brf, xr));
          xi = fmaf(arf, bi.l, fmaf(ar.l, bif, xi));
          xr = fmaf(-aif, bi.l, fmaf(-ai.l, bif, xr));
          xi = fmaf(aif, br.l, fmaf(ai.l, brf, xi));
        }
        constexpr float U = 1.f / 1073741824.f;         // 2^-30
        hr += r + ((i64)__float2int_rn(xr * U) << 1);
        hi += i + ((i64)__float2int_rn(xi * U) << 1);
      };
      longlong2* diag = Hd + (p * N - p * (p - 1) / 2);  // entries (i, i + p), i = 0..L - p
#pragma unroll 1
      for (int k = 0; k <= L; ++k) add(-k, k - p);
      if (in_group) diag[0] = make_longlong2(hr, hi);
#pragma unroll 1
      for (int i = 1; i <= L; ++i) {
        const bool own = i <= L - p;
        if (i == L - p + 1) hr = hi = 0;
        add(own ? i : -i, own ? -(i + p) : i - 1 + p - 2 * L);
        if (in_group && own) diag[i] = make_longlong2(hr, hi);
      }
      if (in_group && p > 0) Hd[N * (N + 1) / 2 + L - p] = make_longlong2(hr, hi);   // diagonal 2L + 1 - p
    }
    __syncwarp();
    // ---- M = H + c I in the orthonormal real basis; lane a takes the mode pairs (a, b), b <= a:
    // P = M_{a,b} = conj H_{L-a,L-b}, Q = M_{a,-b} = conj of diagonal a + b where it is constant
#pragma unroll 1
    for (int b = 0; b <= L; ++b) {
      if (!in_group || b > p) continue;
      const int d = p - b, s = p + b;
      const longlong2 Pc = Hd[d * N - d * (d - 1) / 2 + L - p];
      const longlong2 Qc = Hd[s <= L ? s * N - s * (s - 1) / 2 + L - s : N * (N + 1) / 2 + s - L - 1];
      auto put = [&](int r, int c, i64 v) {
        const Limbs l = fx_split(v);
        Ms[r * LDQ + c + 1] = l;
        Ms[c * LDQ + r + 1] = l;
      };
      if (p == 0) {
        put(0, 0, Pc.x + cfix);
      } else if (b == 0) {                              // M_{0,a} = conj P
        put(0, cx, fx_sqrt2(Pc.x));
        put(0, cy, -fx_sqrt2(Pc.y));
      } else {
        const i64 c = d == 0 ? cfix : 0;
        put(cx, 2 * b - 1, Pc.x + Qc.x + c);            // Re, Re: Re P + Re Q
        put(cy, 2 * b, Pc.x - Qc.x + c);                // Im, Im: Re P - Re Q
        put(cy, 2 * b - 1, -Pc.y - Qc.y);               // Im a, Re b: Im P + Im Q (conjugates stored)
        if (d != 0) put(cx, 2 * b, Pc.y - Qc.y);        // Re a, Im b: -Im P + Im Q
      }
    }
    __syncwarp();
    // ---- FP32 eigenpairs: f_a with M = sum f_a f_a^T
    int xe;                                             // |X| <= 2^xe
    bool on_list;
    {
      float x[NM], yv[NM];
      constexpr float H = 1.f / 536870912.f, HL = H * H;   // 2^-29, 2^-58
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const int4 mm = *reinterpret_cast<const int4*>(Ms + i * LDQ + 2 * p);   // (i, 2p-1) and (i, 2p)
        x[i] = hx ? fmaf(__int_as_float(mm.y), HL, (float)mm.x * H) : 0.f;
        yv[i] = hy ? fmaf(__int_as_float(mm.w), HL, (float)mm.z * H) : 0.f;
      }
      const float least = cholesky_columns<N, LDF, (N > 5)>(x, yv, p, in_group, first, FX_PIVOT, F);
      {
        const float dx = hx ? (float)Ms[cx * LDQ + cx + 1].h : 1e9f, dy = hy ? (float)Ms[cy * LDQ + cy + 1].h : 1e9f;
        const unsigned small = __ballot_sync(0xffffffffu, fminf(dx, dy) < FX_DIAGONAL * 536870912.f);   // 2^29
        on_list = !(least > FX_PIVOT) || (small & (((1u << N) - 1u) << first));
      }
      if (__any_sync(0xffffffffu, on_list)) {
        // the factor of such a point means nothing: I takes its place
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          x[i] = !on_list ? x[i] : hx && i == cx ? 1.f : 0.f;
          yv[i] = !on_list ? yv[i] : hy && i == cy ? 1.f : 0.f;
        }
      }
      __syncwarp();
      onesided_jacobi<N>(x, yv, p, lane, FX_ORTHO2);
      float ax = 0.f, ay = 0.f;
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        ax = fmaf(x[i], x[i], ax);
        ay = fmaf(yv[i], yv[i], ay);
      }
      const float ix = hx ? rsqrt_newton(ax) : 0.f, iy = hy ? rsqrt_newton(ay) : 0.f;
      const float jx = ix * sqrtf(ix), jy = iy * sqrtf(iy);
      float big = fmaxf(ix, iy), all = 0.f;
#pragma unroll
      for (int j = 0; j < N; ++j) all = fmaxf(all, __shfl_sync(0xffffffffu, big, first + j));
      on_list = on_list || !(all * all * FX_LAMBDA <= 1.f);
      frexpf(1.01f * all, &xe);
      xe = min(max(xe, 0), 28);
      // FP32 eigenpairs for the derivative of tau (exact tangent), when asked; launch_tau_pairs refines them
      if (live && eig_out) {
        float* eo = eig_out + gq * Dims<N>::EIG;
        const float back = finite ? ldexpf(1.f, 2 * ex) : __int_as_float(0x7fc00000);
        if (hx) {
#pragma unroll
          for (int i = 0; i < NM; ++i) eo[i * NM + cx] = x[i] * ix;
          eo[NM * NM + cx] = ax * back;
        }
#pragma unroll
        for (int i = 0; i < NM; ++i) eo[i * NM + cy] = yv[i] * iy;
        eo[NM * NM + cy] = ay * back;
      }
      // U, s, and h_a = f_a / |f_a|^{3/2}
      if (hx) {
        store_floats<NM, LDF>(U + cx * LDF, x, ix);
        U[cx * LDF] = ax * ix;
        store_floats<NM, LDF>(F + cx * LDF, x, jx);
      }
      if (hy) {
        store_floats<NM, LDF>(U + cy * LDF, yv, iy);
        U[cy * LDF] = ay * iy;
        store_floats<NM, LDF>(F + cy * LDF, yv, jy);
      }
    }
    __syncwarp();
    // ---- X0 = sum_a h_a h_a^T rounded to one limb
    {
      float x[NM], yv[NM];
#pragma unroll
      for (int i = 0; i < NM; ++i) x[i] = yv[i] = 0.f;
#pragma unroll 1
      for (int a = 0; a < NM; ++a) {
        const float2 own = *reinterpret_cast<const float2*>(F + a * LDF + 2 * p);
        float row[LDF];
        load_floats<LDF>(F + a * LDF, row);
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          x[i] = fmaf(row[i + 1], own.x, x[i]);
          yv[i] = fmaf(row[i + 1], own.y, yv[i]);
        }
      }
      const float to = ldexpf(1.f, 29 - xe);
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const int4 v = make_int4(hx ? __float2int_rn(x[i] * to) : 0, 0, __float2int_rn(yv[i] * to), 0);
        if (hy) *reinterpret_cast<int4*>(Xs + i * LDQ + 2 * p) = v;
      }
    }
    const float rscale = ldexpf(1.f, xe - 58), escale = ldexpf(1.f, 58 - xe);
    // what is left to correct; never reached (negative) at a point for the list, always
    // (infinite) at one that is not finite
    constexpr float NEVER = -1.f, ALWAYS = 3e38f;
    const float small = !finite ? ALWAYS : on_list ? NEVER : fmaxf(1e-10f, ldexpf(64.f, 2 * xe - 58));
    // ---- corrections
#pragma unroll 1
    for (int it = 0;; ++it) {
      __syncwarp();
      // R = I - X (M X), half of the entries
      float rmax = 0.f;
      {
        Limbs pa[NM], pb[NM];
        float pah[NM], pbh[NM];
        {
          // M X: M is symmetric, so row j of M times X_j,col adds to all rows of the column
          i64 ha[NM], hb[NM];
          float xa[NM], xb[NM];
#pragma unroll
          for (int r = 0; r < NM; ++r) {
            ha[r] = hb[r] = 0;
            xa[r] = xb[r] = 0.f;
          }
#pragma unroll 1
          for (int j = 0; j < NM; ++j) {
            const int4* row = reinterpret_cast<const int4*>(Ms + j * LDQ);
            const int4 v = *reinterpret_cast<const int4*>(Xs + j * LDQ + 2 * p);
            const float v0l = __int_as_float(v.y), v1l = __int_as_float(v.w), v0h = (float)v.x, v1h = (float)v.z;
#pragma unroll
            for (int r = 0; r < NM; ++r) {
              const int4 w4 = row[(r + 1) / 2];
              const int mh = (r & 1) ? w4.x : w4.z;
              const float ml = __int_as_float((r & 1) ? w4.y : w4.w), mf = (float)mh;
              fx_mad(ha[r], mh, v.x);
              fx_mad(hb[r], mh, v.z);
              xa[r] = fmaf(ml, v0h, fmaf(mf, v0l, xa[r]));
              xb[r] = fmaf(ml, v1h, fmaf(mf, v1l, xb[r]));
            }
          }
          // to 2^-58 (|M X| <= 1)
          const float to = ldexpf(1.f, xe - 29);
#pragma unroll
          for (int r = 0; r < NM; ++r) {
            pa[r] = fx_split((ha[r] << xe) + fx_int(xa[r] * to));
            pb[r] = fx_split((hb[r] << xe) + fx_int(xb[r] * to));
            pah[r] = (float)pa[r].h;
            pbh[r] = (float)pb[r].h;
          }
        }
        const i64 one = (1ll << 58) >> xe;
#pragma unroll 1
        for (int o = 0; o <= N; ++o) {
          const int r = half_row(o);
          i64 v0, v1;
          fx_dot2<NM>(reinterpret_cast<const int4*>(Xs + r * LDQ), pa, pb, pah, pbh, v0, v1);
          constexpr float LIM = FX_STEP / NM;
          const float r0 = fminf(fmaxf(fx_float((r == cx ? one : 0) - v0) * rscale, -LIM), LIM);
          const float r1 = fminf(fmaxf(fx_float((r == cy ? one : 0) - v1) * rscale, -LIM), LIM);
          if (hx && o < N) {
            rmax = fmaxf(rmax, fabsf(r0));
            F[r * LDF + cx + 1] = r0;
            F[cx * LDF + r + 1] = r0;
          }
          if (hy && o > 0) {
            rmax = fmaxf(rmax, fabsf(r1));
            F[r * LDF + cy + 1] = r1;
            F[cy * LDF + r + 1] = r1;
          }
        }
      }
      const unsigned left = __ballot_sync(0xffffffffu, live && rmax > small);
      const bool more = __any_sync(0xffffffffu, live && rmax > small && small > 0.f) && it + 1 < FX_MAX_IT;
      if (left && !more) {
        const unsigned mine = ((1u << N) - 1u) << first;
        if (live && p == 0 && (left & mine)) hard[HARD_LIST + atomicAdd(hard, 1u)] = (unsigned)gq;
      }
      __syncwarp();
      // E = U [(U^T R U)_ab / (s_a + s_b)] U^T, row by row; R is symmetric (column = row)
      float rx[LDF], ry[LDF];
      load_floats<LDF>(F + (hx ? cx : 0) * LDF, rx);
      load_floats<LDF>(F + cy * LDF, ry);
      __syncwarp();
#pragma unroll 1
      for (int a = 0; a < NM; ++a) {                    // U^T R over R
        float row[LDF], sx = 0.f, sy = 0.f;
        load_floats<LDF>(U + a * LDF, row);
#pragma unroll
        for (int i = 1; i <= NM; ++i) {
          sx = fmaf(row[i], rx[i], sx);
          sy = fmaf(row[i], ry[i], sy);
        }
        if (hy) *reinterpret_cast<float2*>(F + a * LDF + 2 * p) = make_float2(sx, sy);
      }
      __syncwarp();
      load_floats<LDF>(U + (hx ? cx : 0) * LDF, rx);
      load_floats<LDF>(U + cy * LDF, ry);
      {
        const float s0 = rx[0], s1 = ry[0];
#pragma unroll 1
        for (int a = 0; a < NM; ++a) {                  // times U, divided, in place
          float row[LDF], sx = 0.f, sy = 0.f;
          load_floats<LDF>(F + a * LDF, row);
#pragma unroll
          for (int i = 1; i <= NM; ++i) {
            sx = fmaf(row[i], rx[i], sx);
            sy = fmaf(row[i], ry[i], sy);
          }
          const float sa = U[a * LDF];
          __syncwarp();
          if (hy)
            *reinterpret_cast<float2*>(F + a * LDF + 2 * p) = make_float2(sx * rcp_ftz(sa + s0), sy * rcp_ftz(sa + s1));
        }
      }
      __syncwarp();
      {
        float ea[NM], eb[NM];
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          const float2 v = *reinterpret_cast<const float2*>(U + i * LDF + 2 * p);
          rx[i + 1] = v.x;
          ry[i + 1] = v.y;
          ea[i] = eb[i] = 0.f;
        }
#pragma unroll 1
        for (int a = 0; a < NM; ++a) {
          float row[LDF], sx = 0.f, sy = 0.f;
          load_floats<LDF>(F + a * LDF, row);
#pragma unroll
          for (int i = 1; i <= NM; ++i) {
            sx = fmaf(row[i], rx[i], sx);
            sy = fmaf(row[i], ry[i], sy);
          }
          load_floats<LDF>(U + a * LDF, row);
#pragma unroll
          for (int i = 0; i < NM; ++i) {
            ea[i] = fmaf(row[i + 1], sx, ea[i]);
            eb[i] = fmaf(row[i + 1], sy, eb[i]);
          }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NM; ++i)
          if (hy) *reinterpret_cast<float2*>(F + i * LDF + 2 * p) = make_float2(ea[i], eb[i]);
      }
      __syncwarp();
      // X <- X + E on half of the entries, both triangles written (a pair (r, c) is one lane's)
      const int e2 = xe - 58 - ex;
      double* op = reinterpret_cast<double*>(base + Lt::OUTP);
#pragma unroll 1
      for (int o = 0; o <= N; ++o) {
        const int r = half_row(o);
        const int4 v = *reinterpret_cast<const int4*>(Xs + r * LDQ + 2 * p);
        const float2 ev = *reinterpret_cast<const float2*>(F + r * LDF + 2 * p);
        const i64 n0 = fx_join(v.x, __int_as_float(v.y)) + fx_int(ev.x * escale);
        const i64 n1 = fx_join(v.z, __int_as_float(v.w)) + fx_int(ev.y * escale);
        if (more) {
          if (hx && o < N) Xs[r * LDQ + cx + 1] = Xs[cx * LDQ + r + 1] = fx_split(n0);
          if (hy && o > 0) Xs[r * LDQ + cy + 1] = Xs[cy * LDQ + r + 1] = fx_split(n1);
        } else {
          // packed upper triangle through shared memory (over M)
          const double bad = __longlong_as_double(0x7ff8000000000000ll);
          if (hx && o < N) op[packed_index(min(r, cx), max(r, cx), NM)] = small != ALWAYS ? fx_to_double(n0, e2) : bad;
          if (hy && o > 0) op[packed_index(min(r, cy), max(r, cy), NM)] = small != ALWAYS ? fx_to_double(n1, e2) : bad;
        }
      }
      if (!more) break;
    }
    if (in_group && p == 0) {
#pragma unroll
      for (int t = NT; t < NTP; ++t) reinterpret_cast<double*>(base + Lt::OUTP)[t] = 0.0;
    }
    __syncwarp();
    if (live) {
      const double2* op = reinterpret_cast<const double2*>(base + Lt::OUTP);
      double2* out = reinterpret_cast<double2*>(tau_out + gq * NTP);
      for (int t = p; t < NTP / 2; t += N) out[t] = op[t];
    }
    __syncwarp();
  }
}

template <int N>
int launch_tau_fx(const int4* tets, const double* geo, const float2* y, int64_t n_elem, double* tau_out, double nu,
                  double C_I, unsigned* hard, cudaStream_t st, float* eig_out) {
  using Lt = FxLayout<N>;
  // warps a block (1..4) that keep the most warps resident in 227 KB of shared memory
  int warps = 1, best = 0;
  for (int wb = 1; wb <= 4; ++wb) {
    const size_t per_block = (size_t)wb * Lt::WARP * 4;
    if (per_block > 227 * 1024) break;
    const int resident = wb * (int)((228 * 1024) / (per_block + 1024));
    if (resident > best) {
      best = resident;
      warps = wb;
    }
  }
  const size_t smem = (size_t)warps * Lt::WARP * 4;
  if (cudaFuncSetAttribute(tau_fx_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return -2;
  const int64_t n_qp = n_elem * 4, groups = (n_qp + Lt::GPW - 1) / Lt::GPW;
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((groups + warps - 1) / warps, 152 * 128));
  int ke;
  const double k = std::frexp(C_I * nu * nu, &ke);
  const float kh = (float)k;
  count_launches(1);
  tau_fx_kernel<N><<<(int)blocks, warps * 32, smem, st>>>(tets, geo, y, n_qp, tau_out, dd{kh, (float)(k - (double)kh)}, ke,
                                                          hard, eig_out);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

#define TS_INST_TAU_FX(T, N)                                                                             \
  template int launch_tau_fx<N>(const int4*, const double*, const float2*, int64_t, double*, double, double, \
                                unsigned*, cudaStream_t, float*);
TS_FOR_EACH_N(TS_INST_TAU_FX, double)

// double -> (hi, lo) pairs of FP32 numbers; empties tau's list
__global__ void split_dd_kernel(const double* __restrict__ in, float2* __restrict__ out, int64_t n,
                                unsigned* __restrict__ hard) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *hard = 0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const dd v = dd_from_double(in[t]);
    out[t] = make_float2(v.hi, v.lo);
  }
}

int launch_split_dd(const double* in, float2* out, int64_t n, unsigned* hard, cudaStream_t st) {
  if (n <= 0) return 0;
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 152 * 16);
  count_launches(1);
  split_dd_kernel<<<(int)blocks, 256, 0, st>>>(in, out, n, hard);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

}  // namespace ts
