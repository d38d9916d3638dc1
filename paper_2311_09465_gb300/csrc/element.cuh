// Element operator of the time-spectral GLS method in one launch: the residual
// of eq. (Rmc) and the tangent products of eq. (K_mat), with the formulas of
// apply.cu, in double-float (FP64 data) or FP32.
//
// Three launches make one evaluation:
//  1. node_prepass_kernel: per node, the field without fixed entries (clean
//     copy) and its velocity on the K = 3N-2 time samples;
//  2. element_kernel: a block owns EB elements at a time and writes their
//     4 x 4 x C rows to a scratch array;
//  3. gather_kernel: per node, the sum of its elements' rows in the order of the
//     node-to-element list.
// No atomics and no colouring (the coloured form is one launch a colour, 24 to
// 31 of them): the sums have one fixed order, and the row scratch costs
// 2 x 16 C values an element of HBM traffic, a few per cent of the arithmetic.
//
// The velocity at a quadrature point is lambda_a(q) u_a = b sum_a u_a + d u_q
// (b, d the two weights of the symmetric rule), so products and inverse
// transforms are formed at the nodes, c_i(a, t) = u_j(a, t) dv_i/dx_j(t), and
// interpolated as modes.  An element takes 12 inverse transforms of c, 12
// forward ones of T = tau L (24 for LIN_A), 9 forward ones of grad v (18) and 9
// inverse ones of the SUPG sums.
//
// A transform is one lane's work (or SPLIT lanes', each with a share of the
// outputs): inputs in registers, samples k and K-k folded (they share cosines
// and negate sines), coefficients broadcast from shared memory.  Loops over
// outputs stay rolled, so that the whole pass stays in the instruction cache.
//
// Double-float sums are compensated: the products' leading parts are added with
// TwoSum, all errors in a second FP32 accumulator (12 FP32 instructions a term,
// one dependent addition); values are (hi, lo) pairs in 8 bytes.  What bounds
// the double-float form is FP32 issue, about 9 k multiply-adds of 12
// instructions an element at N = 7 (residual); EB and SPLIT keep shared memory a
// warp small enough for 15 to 18 warps an SM.
#pragma once
#include <algorithm>

#include "common.cuh"
#include "ddfloat.cuh"
#include "kernels.h"

namespace ts {

namespace {

template <typename V>
struct Ar;

template <>
struct Ar<float> {
  struct Acc {
    float s;
    __device__ __forceinline__ Acc(float v) : s(v) {}
    __device__ __forceinline__ void add(float a, float b) { s = fmaf(a, b, s); }
    __device__ __forceinline__ float get() const { return s; }
  };
  static __device__ __forceinline__ float zero() { return 0.f; }
  static __device__ __forceinline__ float of(double x) { return (float)x; }
  static __device__ __forceinline__ float add(float a, float b) { return a + b; }
  static __device__ __forceinline__ float sub(float a, float b) { return a - b; }
  static __device__ __forceinline__ float mul(float a, float b) { return a * b; }
  static __device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }
  static __device__ __forceinline__ float neg(float a) { return -a; }
  static __device__ __forceinline__ float twice(float a) { return 2.f * a; }
  static __device__ __forceinline__ float load(const float* p) { return *p; }
  static __device__ __forceinline__ float from(float x) { return x; }
  static __device__ __forceinline__ float to(float x) { return x; }
};

// FP64 as it is (the tracer: its residual has always been native FP64)
template <>
struct Ar<double> {
  struct Acc {
    double s;
    __device__ __forceinline__ Acc(double v) : s(v) {}
    __device__ __forceinline__ void add(double a, double b) { s = ::fma(a, b, s); }
    __device__ __forceinline__ double get() const { return s; }
  };
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double of(double x) { return x; }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double sub(double a, double b) { return a - b; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
  static __device__ __forceinline__ double neg(double a) { return -a; }
  static __device__ __forceinline__ double twice(double a) { return a + a; }
  static __device__ __forceinline__ double from(double x) { return x; }
  static __device__ __forceinline__ double to(double x) { return x; }
};

template <>
struct Ar<float2> {
  static __device__ __forceinline__ dd d(float2 a) { return dd{a.x, a.y}; }
  static __device__ __forceinline__ float2 v(dd a) { return make_float2(a.hi, a.lo); }
  struct Acc {
    float s, c;
    __device__ __forceinline__ Acc(float2 a) : s(a.x), c(a.y) {}
    __device__ __forceinline__ void add(float2 a, float2 b) {
      const float p = a.x * b.x;
      float e = fmaf(a.x, b.x, -p);
      e = fmaf(a.x, b.y, e);
      e = fmaf(a.y, b.x, e);
      float t;
      two_sum(s, p, s, t);
      c += t + e;
    }
    __device__ __forceinline__ float2 get() const {
      float2 r;
      fast_two_sum(s, c, r.x, r.y);
      return r;
    }
  };
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ float2 of(double x) { return v(dd_split(x)); }
  static __device__ __forceinline__ float2 add(float2 a, float2 b) { return v(dd_add(d(a), d(b))); }
  static __device__ __forceinline__ float2 sub(float2 a, float2 b) { return v(dd_add(d(a), dd_neg(d(b)))); }
  static __device__ __forceinline__ float2 mul(float2 a, float2 b) { return v(dd_mul(d(a), d(b))); }
  static __device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return v(dd_fma(d(a), d(b), d(c))); }
  static __device__ __forceinline__ float2 twice(float2 a) { return make_float2(2.f * a.x, 2.f * a.y); }
  static __device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ float2 from(double x) { return v(dd_split(x)); }
  static __device__ __forceinline__ double to(float2 a) { return (double)a.x + (double)a.y; }
};

}  // namespace

constexpr int EL_THREADS = 96;

template <typename V, int N, int MODE>
struct ElementLayout {
  static constexpr int C = 2 * N, K = 3 * N - 2, NM = 2 * N - 1, NT = NM * (NM + 1) / 2;
  static constexpr int KH = K / 2, H = (K - 1) / 2;     // table rows 0..KH; pairs (k, K-k), k = 1..H
  static constexpr int KS = K | 1, CS = C | 1;          // odd row strides
  // elements a block; where transforms are short, 8 with a lane each instead of 4 with
  // two (187,266 tetrahedra, residual in double-float: N = 2 405 us against 436, N = 3 702
  // against 694; in FP32 N = 2 158 against 185, N = 3 250 against 277, N = 4 371 against 367)
  static constexpr int EB = N <= 2 || (N == 3 && sizeof(V) == 4) ? 8 : N <= 7 ? 4 : 2;
  static constexpr int SPLIT = EL_THREADS / (12 * EB);  // lanes a transform
  static constexpr bool PAPER = MODE == MODE_JVP_PAPER;
  // per element, in values
  static constexpr int GEO = 0;                         // dN (12), w = V/4
  static constexpr int A = 13;                          // samples of c, then of T [12][KS]
  static constexpr int B = A + 12 * KS;                 // samples of grad v, later of W [9][KS]
  static constexpr int GM = B + 9 * KS;                 // modes of grad v (f * 3 + j, f < 3) and grad p [12][CS]
  static constexpr int M1 = GM + 12 * CS;               // (LIN_A: grad u0,) c at the nodes, then T [12][CS]
  static constexpr int M2 = M1 + 12 * CS;               // L, then W [9][CS]
  static constexpr int M3 = M2 + 12 * CS;               // rho (Omega v + c), then minus Omega T
  static constexpr int M4 = M3 + 12 * CS;               // PAPER: tau grad p
  static constexpr int END = M4 + (PAPER ? 12 * CS : 0);
  static constexpr int ELEM = END | 1;
  // tau of the four points, converted once, over the samples while they are dead
  static constexpr bool STAGED = 4 * NT <= 21 * KS;
  static constexpr int TABLE = 2 * N * (KH + 1) + N;    // cos, sin [N][KH + 1]; n omega [N]
  static constexpr size_t BYTES = sizeof(V) * (TABLE + (size_t)EB * ELEM) + EB * 4 * sizeof(int);
};

// modes of one row of samples: out[2n], out[2n+1] for n = part, part + SPLIT, ...
// (times K: the factor 1/K is in the operands)
template <typename V, int N, int SPLIT>
__device__ __forceinline__ void inverse_row(const V* s, V* out, const V* cosv, const V* sinv, int part) {
  using R = Ar<V>;
  constexpr int K = 3 * N - 2, KH = K / 2, H = (K - 1) / 2;
  V p[H > 0 ? H : 1], m[H > 0 ? H : 1];
  const V s0 = s[0];
#pragma unroll
  for (int k = 1; k <= H; ++k) {
    const V a = s[k], b = s[K - k];
    p[k - 1] = R::add(a, b);
    m[k - 1] = R::sub(a, b);
  }
#pragma unroll 1
  for (int n = part; n < N; n += SPLIT) {
    const V* cr = cosv + n * (KH + 1);
    const V* sr = sinv + n * (KH + 1);
    V init = s0;
    if constexpr ((K & 1) == 0) init = (n & 1) ? R::sub(s0, s[KH]) : R::add(s0, s[KH]);
    typename R::Acc re(init), im(R::zero());
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      re.add(p[k - 1], cr[k]);
      im.add(m[k - 1], sr[k]);
    }
    out[2 * n] = re.get();
    out[2 * n + 1] = R::neg(im.get());
  }
}

// samples of one mode row x (harmonics doubled, x[1] unused): k and K-k for k = part, part + SPLIT, ...
template <typename V, int N, int SPLIT>
__device__ __forceinline__ void forward_row(const V (&x)[2 * N], V* out, const V* cosv, const V* sinv, int part) {
  using R = Ar<V>;
  constexpr int K = 3 * N - 2, KH = K / 2;
#pragma unroll 1
  for (int k = part; k <= KH; k += SPLIT) {
    typename R::Acc e(x[0]), o(R::zero());
#pragma unroll
    for (int n = 1; n < N; ++n) {
      e.add(x[2 * n], cosv[n * (KH + 1) + k]);
      o.add(x[2 * n + 1], sinv[n * (KH + 1) + k]);
    }
    const V ev = e.get(), ov = o.get();
    out[k] = R::sub(ev, ov);
    if (k > 0 && 2 * k != K) out[K - k] = R::add(ev, ov);
  }
}

// out[j * CS] = d/dx_j of entry fc of the field x (`stride` entries a node)
template <typename V, int C, int CS>
__device__ __forceinline__ void gradient_of(const V* __restrict__ x, const int* nd, int fc, int stride, const V* dN,
                                            V* out) {
  using R = Ar<V>;
  const V x0 = x[(int64_t)nd[0] * stride + fc];
  V d[3];
#pragma unroll
  for (int a = 1; a < 4; ++a) d[a - 1] = R::sub(x[(int64_t)nd[a] * stride + fc], x0);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    typename R::Acc s(R::zero());
#pragma unroll
    for (int a = 1; a < 4; ++a) s.add(dN[a * 3 + j], d[a - 1]);
    out[j * CS] = s.get();
  }
}

template <typename V, int N, int MODE>
__global__ void __launch_bounds__(EL_THREADS) element_kernel(ElementArgs<V> P) {
  using R = Ar<V>;
  using S = typename StoreOf<V>::S;
  using L = ElementLayout<V, N, MODE>;
  constexpr int C = L::C, K = L::K, NM = L::NM, NT = L::NT, NTP = Dims<N>::NT_PAD, KH = L::KH, KS = L::KS, CS = L::CS;
  constexpr int EB = L::EB, SPLIT = L::SPLIT, PARTS = 3 * SPLIT;
  constexpr bool RES = MODE == MODE_RESIDUAL, PAPER = L::PAPER, LINA = MODE == MODE_JVP_LIN_A;
  extern __shared__ __align__(16) unsigned char el_smem[];
  V* cosv = reinterpret_cast<V*>(el_smem);
  V* sinv = cosv + N * (KH + 1);
  V* om = sinv + N * (KH + 1);
  V* es = om + N;
  int* nodes = reinterpret_cast<int*>(es + EB * L::ELEM);
  const int tid = threadIdx.x;
  for (int t = tid; t < 2 * N * (KH + 1); t += EL_THREADS) cosv[t] = P.trig[t];
  for (int t = tid; t < N; t += EL_THREADS) om[t] = R::mul(P.omega, R::of((double)t));
  const V bq = R::of(qp_bary(0, 1)), dq = R::of(qp_bary(0, 0) - qp_bary(0, 1));
  const V bqK = R::of(qp_bary(0, 1) / K), dqK = R::of((qp_bary(0, 0) - qp_bary(0, 1)) / K);
  const V rho = P.rho;

  for (int64_t e0 = (int64_t)blockIdx.x * EB; e0 < P.n_elem; e0 += (int64_t)gridDim.x * EB) {
    const int nel = (int)(P.n_elem - e0 < EB ? P.n_elem - e0 : EB);
    __syncthreads();                                    // tables; the previous elements' last reads
    for (int t = tid; t < nel * 16; t += EL_THREADS) {
      const int el = t / 16, x = t & 15;
      V* g = es + el * L::ELEM + L::GEO;
      if (x < 13) {
        const V val = R::from(P.geo[(e0 + el) * GEO_STRIDE + (x < 12 ? x : GEO_VOL)]);
        g[x] = x < 12 ? val : R::mul(val, R::of(0.25));
      }
    }
    for (int t = tid; t < nel * 4; t += EL_THREADS) nodes[t] = reinterpret_cast<const int*>(P.tets + e0)[t];
    __syncthreads();
    // ---- gradients as modes, then on samples; products at the nodes on samples,
    // c_i(a) = u_j(a) dv_i/dx_j (+ v_j(a) du_i/dx_j), times K.  Gradients are formed
    // from differences to node 0: their error is then relative to the differences,
    // not to the velocity itself
    for (int t = tid; t < nel * 4 * C; t += EL_THREADS) {
      const int el = t / (4 * C), fc = t - el * 4 * C, f = fc / C, c = fc - f * C;
      V* E = es + el * L::ELEM;
      gradient_of<V, C, CS>(P.vd, nodes + 4 * el, fc, 4 * C, E + L::GEO, E + L::GM + f * 3 * CS + c);
    }
    if constexpr (LINA) {
      for (int t = tid; t < nel * 3 * C; t += EL_THREADS) {
        const int el = t / (3 * C), fc = t - el * 3 * C, f = fc / C, c = fc - f * C;
        V* E = es + el * L::ELEM;
        gradient_of<V, C, CS>(P.ud, nodes + 4 * el, fc, 4 * C, E + L::GEO, E + L::M1 + f * 3 * CS + c);
      }
    }
#pragma unroll 1
    for (int pass = 0; pass < (LINA ? 2 : 1); ++pass) {
      __syncthreads();
      for (int t = tid; t < nel * 9 * SPLIT; t += EL_THREADS) {
        const int part = t % SPLIT, row = (t / SPLIT) % 9, el = t / (9 * SPLIT);
        V* E = es + el * L::ELEM;
        const V* src = E + (pass == 0 ? L::GM : L::M1) + row * CS;
        V x[C];
#pragma unroll
        for (int c = 0; c < C; ++c) x[c] = c > 1 ? R::twice(src[c]) : src[c];
        forward_row<V, N, SPLIT>(x, E + L::B + row * KS, cosv, sinv, part);
      }
      __syncthreads();
      const V* ut = pass == 0 ? P.u0t : P.vt;
      for (int t = tid; t < nel * 3 * K; t += EL_THREADS) {
        const int el = t / (3 * K), ik = t - el * 3 * K, i = ik / K, k = ik - i * K;
        V* E = es + el * L::ELEM;
        const int* nd = nodes + 4 * el;
        V g[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) g[j] = E[L::B + (i * 3 + j) * KS + k];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          V* o = E + L::A + (a * 3 + i) * KS + k;
          typename R::Acc s(pass == 0 ? R::zero() : *o);
#pragma unroll
          for (int j = 0; j < 3; ++j) s.add(ut[((int64_t)nd[a] * 3 + j) * K + k], g[j]);
          *o = s.get();
        }
      }
    }
    __syncthreads();
    // ---- to modes
    for (int t = tid; t < nel * 12 * SPLIT; t += EL_THREADS) {
      const int part = t % SPLIT, row = (t / SPLIT) % 12, el = t / (12 * SPLIT);
      V* E = es + el * L::ELEM;
      inverse_row<V, N, SPLIT>(E + L::A + row * KS, E + L::M1 + row * CS, cosv, sinv, part);
    }
    __syncthreads();
    // ---- at the points: rho (Omega v + c) and L = that + grad p; tau to the arithmetic's form
    for (int t = tid; t < nel * 12 * SPLIT; t += EL_THREADS) {
      const int part = t % SPLIT, qi = (t / SPLIT) % 12, el = t / (12 * SPLIT), q = qi / 3, i = qi - q * 3;
      V* E = es + el * L::ELEM;
      const int* nd = nodes + 4 * el;
#pragma unroll 1
      for (int n = part; n < N; n += SPLIT) {
        V vq[2], cq[2], gp[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = 2 * n + h;
          V v[4], m[4];
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            v[a] = P.vd[(int64_t)nd[a] * 4 * C + i * C + c];
            m[a] = E[L::M1 + (a * 3 + i) * CS + c];
          }
          gp[h] = E[L::GM + (9 + i) * CS + c];
          const V va = q == 0 ? v[0] : q == 1 ? v[1] : q == 2 ? v[2] : v[3];
          const V ma = q == 0 ? m[0] : q == 1 ? m[1] : q == 2 ? m[2] : m[3];
          vq[h] = R::fma(bq, R::add(R::add(v[0], v[1]), R::add(v[2], v[3])), R::mul(dq, va));
          cq[h] = R::fma(bqK, R::add(R::add(m[0], m[1]), R::add(m[2], m[3])), R::mul(dqK, ma));
        }
        const V w = om[n];
        const V re = R::mul(rho, R::fma(R::neg(w), vq[1], cq[0]));
        const V im = n == 0 ? R::zero() : R::mul(rho, R::fma(w, vq[0], cq[1]));
        V* x3 = E + L::M3 + qi * CS + 2 * n;
        x3[0] = re;
        x3[1] = im;
        if constexpr (!PAPER) {
          E[L::M2 + qi * CS + 2 * n] = R::add(re, gp[0]);
          E[L::M2 + qi * CS + 2 * n + 1] = R::add(im, gp[1]);
        }
      }
    }
    if constexpr (L::STAGED) {
      for (int t = tid; t < nel * 4 * NT; t += EL_THREADS) {
        const int el = t / (4 * NT), r = t - el * 4 * NT, q = r / NT;
        es[el * L::ELEM + L::A + r] = R::from(P.tau[((e0 + el) * 4 + q) * NTP + r - q * NT]);
      }
    }
    __syncthreads();
    // ---- T = tau L.  tau acts in the orthonormal basis, T_r = (1/d_r) sum_s tau_rs d_s L_s,
    // d_0 = 1, d_s = sqrt2: with L_0 / sqrt2 in place of L_0 only row 0 keeps a factor sqrt2
    for (int t = tid; t < nel * 4 * PARTS; t += EL_THREADS) {
      const int part = t % PARTS, q = (t / PARTS) & 3, el = t / (4 * PARTS);
      V* E = es + el * L::ELEM;
      const S* tg = P.tau + ((e0 + el) * 4 + q) * NTP;
      const V* tq = E + L::A + q * NT;
      const V isq2 = R::of(0.70710678118654752440), sq2 = R::of(1.41421356237309504880);
      const V* l = E + (PAPER ? L::M3 : L::M2) + q * 3 * CS;
      const V* gp = E + L::GM + 9 * CS;
      V l0[3], g0[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        l0[i] = R::mul(l[i * CS], isq2);
        if constexpr (PAPER) g0[i] = R::mul(gp[i * CS], isq2);
      }
#pragma unroll 1
      for (int r = part; r < NM; r += PARTS) {
        auto tau_at = [&](int s) {
          const int k = r <= s ? packed_index(r, s, NM) : packed_index(s, r, NM);
          if constexpr (L::STAGED) return tq[k];
          else return R::from(tg[k]);
        };
        const V t0v = tau_at(0);
        typename R::Acc a0(R::mul(t0v, l0[0])), a1(R::mul(t0v, l0[1])), a2(R::mul(t0v, l0[2]));
        typename R::Acc b0(R::zero()), b1(R::zero()), b2(R::zero());
        if constexpr (PAPER) {
          b0.add(t0v, g0[0]);
          b1.add(t0v, g0[1]);
          b2.add(t0v, g0[2]);
        }
#pragma unroll 2
        for (int s = 1; s < NM; ++s) {
          const V ts = tau_at(s);
          a0.add(ts, l[s + 1]);
          a1.add(ts, l[CS + s + 1]);
          a2.add(ts, l[2 * CS + s + 1]);
          if constexpr (PAPER) {
            b0.add(ts, gp[s + 1]);
            b1.add(ts, gp[CS + s + 1]);
            b2.add(ts, gp[2 * CS + s + 1]);
          }
        }
        V x0 = a0.get(), x1 = a1.get(), x2 = a2.get();
        if (r == 0) {
          x0 = R::mul(x0, sq2);
          x1 = R::mul(x1, sq2);
          x2 = R::mul(x2, sq2);
        }
        V* o = E + L::M1 + q * 3 * CS + stor_of(r);
        o[0] = x0;
        o[CS] = x1;
        o[2 * CS] = x2;
        if constexpr (PAPER) {
          x0 = b0.get(), x1 = b1.get(), x2 = b2.get();
          if (r == 0) {
            x0 = R::mul(x0, sq2);
            x1 = R::mul(x1, sq2);
            x2 = R::mul(x2, sq2);
          }
          V* o4 = E + L::M4 + q * 3 * CS + stor_of(r);
          o4[0] = x0;
          o4[CS] = x1;
          o4[2 * CS] = x2;
        }
      }
      if (part == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          E[L::M1 + (q * 3 + i) * CS + 1] = R::zero();
          if constexpr (PAPER) E[L::M4 + (q * 3 + i) * CS + 1] = R::zero();
        }
      }
    }
    __syncthreads();
    // ---- T (and L) to their caches; rho (Omega v + c) - Omega T; T to samples
    if constexpr (RES) {
      for (int t = tid; t < nel * 12 * C; t += EL_THREADS) {
        const int row = t / C, c = t - row * C, el = row / 12;
        P.t0[e0 * 12 * C + t] = R::to(es[el * L::ELEM + L::M1 + (row - el * 12) * CS + c]);
        if (P.l0) P.l0[e0 * 12 * C + t] = R::to(es[el * L::ELEM + L::M2 + (row - el * 12) * CS + c]);
      }
    }
    for (int t = tid; t < nel * 12 * N; t += EL_THREADS) {
      const int n = t % N, row = t / N, el = row / 12, qi = row - el * 12;
      V* E = es + el * L::ELEM;
      V* g = E + L::M3 + qi * CS + 2 * n;
      const V* tm = E + L::M1 + qi * CS + 2 * n;
      const V w = om[n], tr = tm[0], ti = tm[1];
      g[0] = R::fma(w, ti, g[0]);
      g[1] = R::fma(R::neg(w), tr, g[1]);
    }
    for (int pass = 0; pass < (LINA ? 2 : 1); ++pass) {
      if (pass == 1) __syncthreads();
      for (int t = tid; t < nel * 12 * SPLIT; t += EL_THREADS) {
        const int part = t % SPLIT, qi = (t / SPLIT) % 12, el = t / (12 * SPLIT);
        V* E = es + el * L::ELEM;
        V x[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          x[c] = pass == 0 ? E[L::M1 + qi * CS + c] : R::from(P.t0[((e0 + el) * 12 + qi) * C + c]);
          if (c > 1) x[c] = R::twice(x[c]);
        }
        forward_row<V, N, SPLIT>(x, E + L::A + qi * KS, cosv, sinv, part);
      }
      __syncthreads();
      // ---- SUPG sums on samples: W_ji = sum_q u_j(q) T_i(q) (pass 1: + v_j(q) T0_i(q))
      const V* ut = pass == 0 ? P.u0t : P.vt;
      for (int t = tid; t < nel * 3 * K; t += EL_THREADS) {
        const int el = t / (3 * K), ik = t - el * 3 * K, i = ik / K, k = ik - i * K;
        V* E = es + el * L::ELEM;
        const int* nd = nodes + 4 * el;
        V tq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) tq[q] = E[L::A + (q * 3 + i) * KS + k];
        const V ts = R::mul(bq, R::add(R::add(tq[0], tq[1]), R::add(tq[2], tq[3])));
        // sum_q (b sum_a u_a + d u_q) T_q = sum_a u_a (b sum_q T_q + d T_a)
#pragma unroll
        for (int q = 0; q < 4; ++q) tq[q] = R::fma(dq, tq[q], ts);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          V* o = E + L::B + (j * 3 + i) * KS + k;
          typename R::Acc s(pass == 0 ? R::zero() : *o);
#pragma unroll
          for (int a = 0; a < 4; ++a) s.add(ut[((int64_t)nd[a] * 3 + j) * K + k], tq[a]);
          *o = s.get();
        }
      }
    }
    __syncthreads();
    // ---- to modes (times K)
    for (int t = tid; t < nel * 9 * SPLIT; t += EL_THREADS) {
      const int part = t % SPLIT, row = (t / SPLIT) % 9, el = t / (9 * SPLIT);
      V* E = es + el * L::ELEM;
      inverse_row<V, N, SPLIT>(E + L::B + row * KS, E + L::M2 + row * CS, cosv, sinv, part);
    }
    __syncthreads();
    // ---- the element's rows
    for (int t = tid; t < nel * 4 * C; t += EL_THREADS) {
      const int el = t / (4 * C), fc = t - el * 4 * C, f = fc / C, c = fc - f * C;
      const V* E = es + el * L::ELEM;
      const V* dN = E + L::GEO;
      const V w = dN[12];
      const int* nd = nodes + 4 * el;
      V* out = P.rows + ((e0 + el) * 4) * 4 * C + fc;
      if (c == 1) {
#pragma unroll
        for (int a = 0; a < 4; ++a) out[a * 4 * C] = R::zero();
        continue;
      }
      if (f < 3) {
        V v[4], G[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          v[a] = P.vd[(int64_t)nd[a] * 4 * C + fc];
          G[a] = E[L::M3 + (a * 3 + f) * CS + c];
        }
        const V ps = R::add(R::add(P.vd[(int64_t)nd[0] * 4 * C + 3 * C + c], P.vd[(int64_t)nd[1] * 4 * C + 3 * C + c]),
                            R::add(P.vd[(int64_t)nd[2] * 4 * C + 3 * C + c], P.vd[(int64_t)nd[3] * 4 * C + 3 * C + c]));
        V X[3];
        const V mu4 = P.mu4, iK = R::of(1.0 / K);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          X[j] = R::fma(mu4, E[L::GM + (f * 3 + j) * CS + c], R::mul(E[L::M2 + (j * 3 + f) * CS + c], iK));
          if (j == f) X[j] = R::sub(X[j], ps);          // the pressure acts like a normal stress
        }
        V base = R::mul(bq, R::add(R::add(G[0], G[1]), R::add(G[2], G[3])));
        const V m5 = P.mass5;
        if (!RES) base = R::fma(m5, R::add(R::add(v[0], v[1]), R::add(v[2], v[3])), base);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          typename R::Acc s(base);
          s.add(dq, G[a]);
          if (!RES) s.add(m5, v[a]);
#pragma unroll
          for (int j = 0; j < 3; ++j) s.add(dN[a * 3 + j], X[j]);
          out[a * 4 * C] = R::mul(w, s.get());
        }
      } else {
        const V* gm = E + L::GM + c;
        const V dv = R::add(R::add(gm[0], gm[4 * CS]), gm[8 * CS]);
        V ts[3];
        const V irho = P.irho;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const V* tm = E + (PAPER ? L::M4 : L::M1) + i * CS + c;
          ts[i] = R::mul(irho, R::add(R::add(tm[0], tm[3 * CS]), R::add(tm[6 * CS], tm[9 * CS])));
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          typename R::Acc s(dv);
#pragma unroll
          for (int i = 0; i < 3; ++i) s.add(dN[a * 3 + i], ts[i]);
          out[a * 4 * C] = R::mul(w, s.get());
        }
      }
    }
  }
}

// one thread a (node, field): the field without fixed entries and, for the
// velocity, its samples.  S: the caller's type
template <typename V, int N>
__global__ void __launch_bounds__(128) node_prepass_kernel(const typename StoreOf<V>::S* __restrict__ y,
                                                           const uint8_t* __restrict__ dmask, V* __restrict__ clean,
                                                           V* __restrict__ samples, const V* __restrict__ trig,
                                                           int64_t n_nodes, unsigned* __restrict__ zero,
                                                           typename StoreOf<V>::S* __restrict__ copy) {
  using R = Ar<V>;
  constexpr int C = 2 * N, K = 3 * N - 2, KH = K / 2;
  __shared__ V table[2 * N * (KH + 1)];
  if (zero && blockIdx.x == 0 && threadIdx.x == 0) *zero = 0;
  for (int t = threadIdx.x; t < 2 * N * (KH + 1); t += blockDim.x) table[t] = trig[t];
  __syncthreads();
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_nodes * 4; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t node = t >> 2;
    const int f = (int)(t & 3);
    const bool fixed = dmask && f < 3 && dmask[node];
    V x[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const typename StoreOf<V>::S value = y[t * C + c];
      if (copy) copy[t * C + c] = value;
      x[c] = c == 1 || fixed ? R::zero() : R::from(value);
      if (clean) clean[t * C + c] = x[c];
      if (c > 1) x[c] = R::twice(x[c]);
    }
    if (f < 3) forward_row<V, N, 1>(x, samples + (node * 3 + f) * K, table, table + N * (KH + 1), 0);
  }
}

// Sum of a node's element rows.  The rows of a nearly converged state are large against
// their sum, so pairs are added to more than FP64: s, c, d take the rounding errors of the
// one before.  (As double-float additions the sum was good to 2^-46 of the largest row.)
template <typename V>
struct RowSum {
  V s = V(0);
  __device__ __forceinline__ void add(V a) { s += a; }
  __device__ __forceinline__ V get() const { return s; }
};
template <>
struct RowSum<float2> {
  float s = 0.f, c = 0.f, d = 0.f;
  __device__ __forceinline__ void add(float2 a) {
    float e, f, g;
    two_sum(s, a.x, s, e);
    two_sum(c, e, c, f);
    two_sum(c, a.y, c, g);
    d += f + g;
  }
  __device__ __forceinline__ double get() const { return (double)s + ((double)c + (double)d); }
};

// out[node][f][c] = sum of the node's element rows; Im(mode 0) and, on Dirichlet
// nodes, the first `masked` of the fields are zero
template <typename V>
__global__ void __launch_bounds__(256) gather_kernel(const int32_t* __restrict__ node_off,
                                                     const int32_t* __restrict__ node_elem,
                                                     const V* __restrict__ rows, const uint8_t* __restrict__ dmask,
                                                     typename StoreOf<V>::S* __restrict__ out, int64_t n_nodes, int C,
                                                     int fields, int masked) {
  const int FC = fields * C;
  const int64_t total = n_nodes * FC;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t node = t / FC;
    const int fc = (int)(t - node * FC), f = fc / C, c = fc - f * C;
    RowSum<V> sum;
    if (c != 1 && !(f < masked && dmask[node])) {
      const int p1 = node_off[node + 1];
      for (int p = node_off[node]; p < p1; p += 4) {     // four loads in flight
        V v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (p + u < p1) v[u] = rows[(int64_t)node_elem[p + u] * FC + fc];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (p + u < p1) sum.add(v[u]);
      }
    }
    out[t] = sum.get();
  }
}

template <typename V, int N, int MODE>
int launch_element_mode(const ElementArgs<V>& P, cudaStream_t st) {
  using L = ElementLayout<V, N, MODE>;
  static_assert(L::BYTES <= 227 * 1024, "shared memory of a block");
  if (cudaFuncSetAttribute(element_kernel<V, N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::BYTES) !=
      cudaSuccess)
    return -2;
  const int64_t blocks = std::min<int64_t>((P.n_elem + L::EB - 1) / L::EB, 152 * 256);
  count_launches(1);
  element_kernel<V, N, MODE><<<(int)blocks, EL_THREADS, L::BYTES, st>>>(P);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

template <typename V, int N>
int launch_element(int mode, const ElementArgs<V>& P, cudaStream_t st) {
  if (P.n_elem <= 0) return 0;
  switch (mode) {
    case MODE_RESIDUAL: return launch_element_mode<V, N, MODE_RESIDUAL>(P, st);
    case MODE_JVP_PAPER: return launch_element_mode<V, N, MODE_JVP_PAPER>(P, st);
    case MODE_JVP_FROZEN: return launch_element_mode<V, N, MODE_JVP_FROZEN>(P, st);
    case MODE_JVP_LIN_A: return launch_element_mode<V, N, MODE_JVP_LIN_A>(P, st);
  }
  return -1;
}

template <typename V, int N>
int launch_node_prepass(const typename StoreOf<V>::S* y, const uint8_t* dmask, V* clean, V* samples, const V* trig,
                        int64_t n_nodes, cudaStream_t st, unsigned* zero,
                        typename StoreOf<V>::S* copy) {
  if (n_nodes <= 0) return 0;
  const int64_t blocks = std::min<int64_t>((n_nodes * 4 + 127) / 128, 152 * 32);
  count_launches(1);
  node_prepass_kernel<V, N><<<(int)blocks, 128, 0, st>>>(y, dmask, clean, samples, trig, n_nodes, zero, copy);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

template <typename V>
int launch_gather(const int32_t* node_off, const int32_t* node_elem, const V* rows, const uint8_t* dmask,
                  typename StoreOf<V>::S* out, int64_t n_nodes, int C, int fields, int masked, cudaStream_t st) {
  if (n_nodes <= 0) return 0;
  const int64_t blocks = std::min<int64_t>((n_nodes * fields * C + 255) / 256, 152 * 64);
  count_launches(1);
  gather_kernel<V><<<(int)blocks, 256, 0, st>>>(node_off, node_elem, rows, dmask, out, n_nodes, C, fields, masked);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

// ---------------------------------------------------------------- tracer
// Time-spectral GLS convection-diffusion of a scalar phi (eq. 3D-weak with
// eq. 3D-weak-def, section 2.2) advected by a given velocity a: per element and
// quadrature point (weights V/4)
//   res  = Omega phi + A_j dphi/dx_j          (A_j = A(a_j), eq. phi-def)
//   T    = tau res                            (tau of eq. 3D-tau with kappa)
//   r_a += w [N_a res - N_a Omega T + dN_a/dx_j A_j T] + kappa V dN_a/dx_j dphi/dx_j
// The flow operator's structure with one field: an element takes 3 forward
// transforms of grad phi, 4 inverse ones of the products at the nodes, 4 forward
// ones of T and 3 inverse ones of the SUPG sums.  N = 7, 26,784 tetrahedra, FP64:
// 1.33 ms with one warp an element in 30 coloured launches; bound by the FP64
// pipe, about 3 k multiply-adds an element.
template <typename V, int N>
struct TracerLayout {
  static constexpr int C = 2 * N, K = 3 * N - 2, KH = K / 2, KS = K | 1, CS = C | 1;
  static constexpr int EB = N <= 7 ? 8 : 4, PARTS = EL_THREADS / (4 * EB);   // lanes a row
  static constexpr int GEO = 0, A = 13, B = A + 4 * KS, GM = B + 3 * KS, M1 = GM + 3 * CS, M2 = M1 + 4 * CS,
                       M3 = M2 + 4 * CS, ELEM = (M3 + 4 * CS) | 1;
  static constexpr int TABLE = 2 * N * (KH + 1) + N;
  static constexpr size_t BYTES = sizeof(V) * (TABLE + (size_t)EB * ELEM) + EB * 4 * sizeof(int);
};

template <typename V, int N>
__global__ void __launch_bounds__(EL_THREADS) tracer_kernel(TracerArgs<V> P) {
  using R = Ar<V>;
  using L = TracerLayout<V, N>;
  constexpr int C = L::C, K = L::K, NM = 2 * N - 1, NTP = Dims<N>::NT_PAD, KH = L::KH, KS = L::KS, CS = L::CS;
  constexpr int EB = L::EB, PARTS = L::PARTS;
  extern __shared__ __align__(16) unsigned char el_smem[];
  V* cosv = reinterpret_cast<V*>(el_smem);
  V* sinv = cosv + N * (KH + 1);
  V* om = sinv + N * (KH + 1);
  V* es = om + N;
  int* nodes = reinterpret_cast<int*>(es + EB * L::ELEM);
  const int tid = threadIdx.x;
  for (int t = tid; t < 2 * N * (KH + 1); t += EL_THREADS) cosv[t] = P.trig[t];
  for (int t = tid; t < N; t += EL_THREADS) om[t] = R::mul(P.omega, R::of((double)t));
  const V bq = R::of(qp_bary(0, 1)), dq = R::of(qp_bary(0, 0) - qp_bary(0, 1));
  const V bqK = R::of(qp_bary(0, 1) / K), dqK = R::of((qp_bary(0, 0) - qp_bary(0, 1)) / K), iK = R::of(1.0 / K);

  for (int64_t e0 = (int64_t)blockIdx.x * EB; e0 < P.n_elem; e0 += (int64_t)gridDim.x * EB) {
    const int nel = (int)(P.n_elem - e0 < EB ? P.n_elem - e0 : EB);
    __syncthreads();
    for (int t = tid; t < nel * 16; t += EL_THREADS) {
      const int el = t / 16, x = t & 15;
      if (x < 13) {
        const V val = R::from(P.geo[(e0 + el) * GEO_STRIDE + (x < 12 ? x : GEO_VOL)]);
        es[el * L::ELEM + L::GEO + x] = x < 12 ? val : R::mul(val, R::of(0.25));
      }
    }
    for (int t = tid; t < nel * 4; t += EL_THREADS) nodes[t] = reinterpret_cast<const int*>(P.tets + e0)[t];
    __syncthreads();
    // ---- gradient: modes, samples; products at the nodes c(a) = a_j(a) dphi/dx_j, times K
    for (int t = tid; t < nel * C; t += EL_THREADS) {
      const int el = t / C, c = t - el * C;
      V* E = es + el * L::ELEM;
      gradient_of<V, C, CS>(P.phi, nodes + 4 * el, c, C, E + L::GEO, E + L::GM + c);
    }
    __syncthreads();
    for (int t = tid; t < nel * 3 * PARTS; t += EL_THREADS) {
      const int part = t % PARTS, row = (t / PARTS) % 3, el = t / (3 * PARTS);
      V* E = es + el * L::ELEM;
      V x[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const V v = E[L::GM + row * CS + c];
        x[c] = c > 1 ? R::twice(v) : v;
      }
      forward_row<V, N, PARTS>(x, E + L::B + row * KS, cosv, sinv, part);
    }
    __syncthreads();
    for (int t = tid; t < nel * 4 * K; t += EL_THREADS) {
      const int el = t / (4 * K), ak = t - el * 4 * K, a = ak / K, k = ak - a * K;
      V* E = es + el * L::ELEM;
      typename R::Acc s(R::zero());
#pragma unroll
      for (int j = 0; j < 3; ++j) s.add(P.at[((int64_t)nodes[4 * el + a] * 3 + j) * K + k], E[L::B + j * KS + k]);
      E[L::A + a * KS + k] = s.get();
    }
    __syncthreads();
    for (int t = tid; t < nel * 4 * PARTS; t += EL_THREADS) {
      const int part = t % PARTS, row = (t / PARTS) & 3, el = t / (4 * PARTS);
      V* E = es + el * L::ELEM;
      inverse_row<V, N, PARTS>(E + L::A + row * KS, E + L::M1 + row * CS, cosv, sinv, part);
    }
    __syncthreads();
    // ---- res at the points (M2 for tau, M3 for the rows)
    for (int t = tid; t < nel * 4 * N; t += EL_THREADS) {
      const int n = t % N, q = (t / N) & 3, el = t / (4 * N);
      V* E = es + el * L::ELEM;
      V pq[2], cq[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = 2 * n + h;
        V v[4], m[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          v[a] = P.phi[(int64_t)nodes[4 * el + a] * C + c];
          m[a] = E[L::M1 + a * CS + c];
        }
        const V va = q == 0 ? v[0] : q == 1 ? v[1] : q == 2 ? v[2] : v[3];
        const V ma = q == 0 ? m[0] : q == 1 ? m[1] : q == 2 ? m[2] : m[3];
        pq[h] = R::fma(bq, R::add(R::add(v[0], v[1]), R::add(v[2], v[3])), R::mul(dq, va));
        cq[h] = R::fma(bqK, R::add(R::add(m[0], m[1]), R::add(m[2], m[3])), R::mul(dqK, ma));
      }
      const V w = om[n];
      V* x2 = E + L::M2 + q * CS + 2 * n;
      V* x3 = E + L::M3 + q * CS + 2 * n;
      x2[0] = x3[0] = R::fma(R::neg(w), pq[1], cq[0]);
      x2[1] = x3[1] = n == 0 ? R::zero() : R::fma(w, pq[0], cq[1]);
    }
    __syncthreads();
    // ---- T = tau res (orthonormal basis: see element_kernel), zero without the least-squares terms
    for (int t = tid; t < nel * 4 * PARTS; t += EL_THREADS) {
      const int part = t % PARTS, q = (t / PARTS) & 3, el = t / (4 * PARTS);
      V* E = es + el * L::ELEM;
      const typename TracerArgs<V>::S* tg = P.tau + ((e0 + el) * 4 + q) * NTP;
      const V* l = E + L::M2 + q * CS;
      V* o = E + L::M1 + q * CS;
      const V l0 = R::mul(l[0], R::of(0.70710678118654752440));
#pragma unroll 1
      for (int r = part; r < NM; r += PARTS) {
        typename R::Acc a(R::mul(R::from(tg[r]), l0));                 // packed (0, r)
#pragma unroll 4
        for (int s = 1; s < NM; ++s)
          a.add(R::from(tg[r <= s ? packed_index(r, s, NM) : packed_index(s, r, NM)]), l[s + 1]);
        const V v = r == 0 ? R::mul(a.get(), R::of(1.41421356237309504880)) : a.get();
        o[stor_of(r)] = P.gls ? v : R::zero();
      }
      if (part == 0) o[1] = R::zero();
    }
    __syncthreads();
    for (int t = tid; t < nel * 4 * N; t += EL_THREADS) {
      const int n = t % N, q = (t / N) & 3, el = t / (4 * N);
      V* E = es + el * L::ELEM;
      V* g = E + L::M3 + q * CS + 2 * n;
      const V* tm = E + L::M1 + q * CS + 2 * n;
      const V w = om[n], tr = tm[0], ti = tm[1];
      g[0] = R::fma(w, ti, g[0]);
      g[1] = R::fma(R::neg(w), tr, g[1]);
    }
    for (int t = tid; t < nel * 4 * PARTS; t += EL_THREADS) {
      const int part = t % PARTS, q = (t / PARTS) & 3, el = t / (4 * PARTS);
      V* E = es + el * L::ELEM;
      V x[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const V v = E[L::M1 + q * CS + c];
        x[c] = c > 1 ? R::twice(v) : v;
      }
      forward_row<V, N, PARTS>(x, E + L::A + q * KS, cosv, sinv, part);
    }
    __syncthreads();
    // ---- SUPG sums W_j = sum_a a_j(a) (b sum_q T_q + d T_a)
    for (int t = tid; t < nel * 3 * K; t += EL_THREADS) {
      const int el = t / (3 * K), jk = t - el * 3 * K, j = jk / K, k = jk - j * K;
      V* E = es + el * L::ELEM;
      V tq[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) tq[q] = E[L::A + q * KS + k];
      const V ts = R::mul(bq, R::add(R::add(tq[0], tq[1]), R::add(tq[2], tq[3])));
      typename R::Acc s(R::zero());
#pragma unroll
      for (int a = 0; a < 4; ++a)
        s.add(P.at[((int64_t)nodes[4 * el + a] * 3 + j) * K + k], R::fma(dq, tq[a], ts));
      E[L::B + j * KS + k] = s.get();
    }
    __syncthreads();
    for (int t = tid; t < nel * 3 * PARTS; t += EL_THREADS) {
      const int part = t % PARTS, row = (t / PARTS) % 3, el = t / (3 * PARTS);
      V* E = es + el * L::ELEM;
      inverse_row<V, N, PARTS>(E + L::B + row * KS, E + L::M2 + row * CS, cosv, sinv, part);
    }
    __syncthreads();
    // ---- the element's rows
    for (int t = tid; t < nel * C; t += EL_THREADS) {
      const int el = t / C, c = t - el * C;
      const V* E = es + el * L::ELEM;
      const V* dN = E + L::GEO;
      V* out = P.rows + (e0 + el) * 4 * C + c;
      V G[4], X[3];
#pragma unroll
      for (int q = 0; q < 4; ++q) G[q] = E[L::M3 + q * CS + c];
#pragma unroll
      for (int j = 0; j < 3; ++j) X[j] = R::fma(P.kappa4, E[L::GM + j * CS + c], R::mul(E[L::M2 + j * CS + c], iK));
      const V base = R::mul(bq, R::add(R::add(G[0], G[1]), R::add(G[2], G[3])));
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        typename R::Acc s(base);
        s.add(dq, G[a]);
#pragma unroll
        for (int j = 0; j < 3; ++j) s.add(dN[a * 3 + j], X[j]);
        out[a * C] = c == 1 ? R::zero() : R::mul(dN[12], s.get());
      }
    }
  }
}

template <typename V, int N>
int launch_tracer(const TracerArgs<V>& P, cudaStream_t st) {
  using L = TracerLayout<V, N>;
  static_assert(L::BYTES <= 227 * 1024, "shared memory of a block");
  if (P.n_elem <= 0) return 0;
  if (cudaFuncSetAttribute(tracer_kernel<V, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::BYTES) != cudaSuccess)
    return -2;
  const int64_t blocks = std::min<int64_t>((P.n_elem + L::EB - 1) / L::EB, 152 * 256);
  count_launches(1);
  tracer_kernel<V, N><<<(int)blocks, EL_THREADS, L::BYTES, st>>>(P);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

// out = in without Im(mode 0), [V][C]
template <typename V>
__global__ void clean_kernel(const V* __restrict__ in, V* __restrict__ out, int64_t n, int C) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    out[t] = t % C == 1 ? V(0) : in[t];
}
template <typename V>
int launch_clean(const V* in, V* out, int64_t n, int C, cudaStream_t st) {
  if (n <= 0) return 0;
  count_launches(1);
  clean_kernel<V><<<(int)std::min<int64_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(in, out, n, C);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

}  // namespace ts
