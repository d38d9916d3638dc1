// Kernel launchers of the GB300 time-spectral GLS library (internal).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

// Mode counts with compiled kernels.  Each entry instantiates the tau,
// operator and boundary kernels in FP32 and FP64.
#define TS_FOR_EACH_N(X, T) X(T, 1) X(T, 2) X(T, 3) X(T, 4) X(T, 5) X(T, 7) X(T, 10) X(T, 15)
#define TS_N_LIST 1, 2, 3, 4, 5, 7, 10, 15

namespace ts {

// process-wide count of kernel launches issued by this library
void count_launches(int n);
unsigned long long launches_total();

template <typename T, int N>
int launch_tau(const int4* tets, const T* geo, const T* y, int64_t n_elem, T* tau_out, T nu,
               T C_I, unsigned* n_unconverged, cudaStream_t st, float* eig_out = nullptr);

// load a kernel into the current device's context without launching it
// (instantiated for T = float only)
template <typename T, int N>
int preload_tau();
template <typename T, int N>
int preload_apply_residual();

// FP64 tau from FP32 Jacobi eigenvectors plus an FP64 polish (tau.cu)
template <int N>
int launch_tau_polish(const int4* tets, const double* geo, const double* y, int64_t n_elem,
                      double* tau_out, double nu, double C_I, unsigned* n_unconverged,
                      cudaStream_t st, float* eig_out = nullptr);

// FP64 tau from FP32 eigenpairs and Newton corrections with residuals in 58-bit
// fixed point (tau_fx.cu); y: the state as double-float pairs [V][4][C].  Points it
// does not take (tau_fx.cu) are listed in hard, to be redone by launch_tau_hard:
// hard[0] their number (zero before the launch), hard[HARD_LIST..] element * 4 + point
constexpr int HARD_LIST = 4;
template <int N>
int launch_tau_fx(const int4* tets, const double* geo, const float2* y, int64_t n_elem, double* tau_out, double nu,
                  double C_I, unsigned* hard, cudaStream_t st, float* eig_out = nullptr);
// FP64 tau of the listed points, for any condition number: the FP64 refinement with
// Jacobi sweeps in FP64 on its nearly diagonal matrix (tau.cu); y: [V][4][C].
// n_unconverged counts points whose smallest eigenvalues FP64 does not resolve.  eig_out
// (may be null): their eigenpairs
template <int N>
int launch_tau_hard(const int4* tets, const double* geo, const double* y, const unsigned* hard, double* tau_out,
                    double nu, double C_I, unsigned* n_unconverged, cudaStream_t st, float* eig_out = nullptr);
// n doubles as (hi, lo) FP32 pairs; hard[0] = 0
int launch_split_dd(const double* in, float2* out, int64_t n, unsigned* hard, cudaStream_t st);

// Backflow stabilisation on one Neumann face set (tau.cu): when y_for_matrix
// is given, first |A_n|_- at the 3 points of every face into bneg; then
// out[A][i] += coef * int N_A |A_n|_- v_i over the faces (atomics).
template <typename T, int N>
int launch_backflow(const int32_t* faces, const T* normals, const T* area, int64_t n_faces,
                    const T* y_for_matrix, T* bneg, const T* v, const uint8_t* dmask, int mask_input,
                    T coef, T* out, cudaStream_t st);

// One colour range [e0, e1) of the element operator (see apply.cu).
template <typename T, int N>
int launch_apply(int mode, const int4* tets, const T* geo, const T* v, const T* u0,
                 const T* tau, T* t0cache, const uint8_t* dmask, T* out, const T* dft,
                 Phys<T> ph, int64_t e0, int64_t e1, cudaStream_t st, T* l0cache = nullptr);

// y[node][i][c] = vals[k][i][c] for the k-th listed node, velocity fields i < 3
// (the inlet Dirichlet data of the initial guess)
template <typename T>
int launch_inlet_fill(const int32_t* nodes, const double* vals, int64_t n, int C, T* y, cudaStream_t st);

// The same element operator in one launch (element.cuh).  V: the arithmetic's
// value type, float or float2 = double-float pair; S: the caller's type
template <typename V>
struct StoreOf;
template <>
struct StoreOf<float> {
  using S = float;
};
template <>
struct StoreOf<float2> {
  using S = double;
};
template <>
struct StoreOf<double> {
  using S = double;
};
template <typename S>
struct PairOfStore;
template <>
struct PairOfStore<float> {
  using V = float;
};
template <>
struct PairOfStore<double> {
  using V = float2;
};

template <typename V>
struct ElementArgs {
  using S = typename StoreOf<V>::S;
  const int4* tets;
  const S* geo;
  const V* u0t;      // [V][3][K] linearisation velocity on samples
  const V* vt;       // [V][3][K] the operand's
  const V* ud;       // [V][4][C] linearisation state
  const V* vd;       // [V][4][C] the operand without fixed entries
  const S* tau;
  S* t0;             // [E][4][3][C] tau L (written by the residual, read by LIN_A)
  S* l0;             // [E][4][3][C] L (residual, exact tangent only) or null
  const V* trig;     // cos, sin of 2 pi n k / K: [2][N][KH + 1]
  V* rows;           // [E][4][4][C]
  V rho, irho, mu4, mass5, omega;   // rho, 1/rho, 4 mu, mass coefficient / 5, omega
  int64_t n_elem;
};

template <typename V, int N>
int launch_element(int mode, const ElementArgs<V>& P, cudaStream_t st);
// clean (may be null) = y without fixed entries (dmask null: all velocities kept),
// samples of its velocity; *zero = 0, copy = y as it is (both may be null)
template <typename V, int N>
int launch_node_prepass(const typename StoreOf<V>::S* y, const uint8_t* dmask, V* clean, V* samples, const V* trig,
                        int64_t n_nodes, cudaStream_t st, unsigned* zero = nullptr,
                        typename StoreOf<V>::S* copy = nullptr);
// out = per node the sum of its element rows [4][fields][C]; on Dirichlet nodes the
// first `masked` fields are zero
template <typename V>
int launch_gather(const int32_t* node_off, const int32_t* node_elem, const V* rows, const uint8_t* dmask,
                  typename StoreOf<V>::S* out, int64_t n_nodes, int C, int fields, int masked, cudaStream_t st);

// Tracer residual of eq. (3D-weak) in one launch (element.cuh), V = float or double
template <typename V>
struct TracerArgs {
  using S = V;
  const int4* tets;
  const V* geo;
  const V* at;       // [V][3][K] advecting velocity on samples
  const V* phi;      // [V][C] without Im(mode 0)
  const V* tau;
  const V* trig;
  V* rows;           // [E][4][C]
  V omega, kappa4;   // kappa4: 4 kappa
  int64_t n_elem;
  int gls;
};
template <typename V, int N>
int launch_tracer(const TracerArgs<V>& P, cudaStream_t st);
// out = in [V][C] without Im(mode 0)
template <typename V>
int launch_clean(const V* in, V* out, int64_t n, int C, cudaStream_t st);
template <typename T>
int launch_repack_velocity(const T* a, T* a4, int64_t V, int C, cudaStream_t st);

// Resistance outlets: out[A][i][c] += R w_Ai Q_c with Q_c = sum_B w_Bi v[B][i][c]
template <typename T>
int launch_outlet(const int32_t* nodes, const T* w, int n_nodes, T R, const T* v,
                  const uint8_t* dmask, int mask_input, T* out, int C, cudaStream_t st);

// One instance's operands of an FP32 tangent product (jvp32.cuh); also the
// per-instance entry of the batched launch.
struct J32Inst {
  const int4* tets;
  const float* geo;
  const float* v;
  const float* u0t;      // [V][K] float4: u0 velocity sampled in time (x, y, z, 0)
  float* vt;             // [V][K] float4 scratch: masked v sampled in time (node pre-pass)
  const float* tau;
  const float* t0cache;
  const uint8_t* dmask;
  float* out;
  Phys<float> ph;
  int64_t n_elem;
  int64_t n_nodes;
  int N;
  const float* dT = nullptr;   // [E][4][3][C] d tau[v] L(u0) (exact tangent only)
};

// Batched LIN_A tangent products of instances with N <= J32_MAX_N in one
// element launch after one node pre-pass (jvp32_batch.cu); every out must be
// zero on entry.  d_counts holds {n_inst, n_tiles, n_nodes} on the device,
// tile_off n_inst + 1 prefix sums of ceil(n_elem / 2), node_off n_inst + 1
// prefix sums of the node counts.  Shared memory per warp: j32_batch_warp_bytes().
int launch_jvp32_batch(const J32Inst* d_insts, const int64_t* d_tile_off, const int64_t* d_node_off,
                       const int64_t* d_counts, int warps_per_block, int blocks, cudaStream_t st);
size_t j32_batch_warp_bytes();
int j32_batch_configure();
int j32_upload_batch(const float* host_all);

// FP32 tangent product (jvp32.cuh): a node pre-pass (v sampled into I.vt,
// I.out cleared) and one element launch
// (with e_before / e_after: events recorded around the element launch)
template <int N>
int launch_jvp32(int mode, const J32Inst& I, cudaStream_t st, cudaEvent_t e_before = nullptr,
                 cudaEvent_t e_after = nullptr);
// FP32 eigenpairs of M by launch_tau_fx, refined in place on its tau (dtau.cu; N <=
// J32_MAX_N, above which nothing reads them).  Listed points: meaningless until
// launch_tau_hard writes them
template <int N>
int launch_tau_pairs(const double* tau, int64_t n_elem, float* eig, cudaStream_t st);
// d tau[v] L_i(u0) at every quadrature point (dtau.cu): the Frechet derivative of
// tau = M^{-1/2} (eq. 3D-tau) in the direction of v, from the cached eigenpairs
// of M (eig [E*4][EIG]) and strong residual L(u0) (l0 [E][4][3][C]);
// dT [E][4][3][C], storage coordinates
template <int N>
int launch_dtau(const int4* tets, const float* geo, const float* u0, const float* v, const uint8_t* dmask,
                const float* eig, const float* l0, float* dT, int64_t n_elem, cudaStream_t st);

// u0 velocity at the nodes as time samples [V][K] float4 (x, y, z, 0)
template <int N>
int launch_node_samples(const float* u0, float* u0t, int64_t V, cudaStream_t st);
// the table of all compiled N (forward [K][C] then inverse [C][K] each)
int dft_constant_total();
int dft_constant_offset(int N);
// each fast-path translation unit copies its slice into its constant bank
int j32_upload_n123(const float* host_all);
int j32_upload_n45(const float* host_all);
int j32_upload_n7(const float* host_all);
constexpr int J32_MAX_N = 7;   // largest N with the single-launch FP32 kernel
constexpr int NODAL_MAX_N = 7;   // largest N with the register-tiled nodal kernels (nodal.cuh)

// Nodal diagonal blocks H_AA of the tangent (precond.cu): one 8N x 8N block per
// node from the node-to-element list (packed element * 4 + local node; uc: the
// state u0 as in node_prepass, N <= 7 only); with
// invert the inverse, column-major, else H_AA row-major.  Fixed unknowns
// (Im(mode 0), Dirichlet velocity) have zero rows and columns (identity when
// inverted); n_singular counts blocks that could not be inverted (stored as I).
template <typename T, int N>
int launch_block_diag(int variant_paper, int invert, const int32_t* node_off, const int32_t* node_elem,
                      const int4* tets, const T* geo, const T* u0, const T* uc, const T* tau, const uint8_t* dmask,
                      const float* outdiag, Phys<float> ph, float* out, int64_t n_nodes,
                      unsigned* n_singular, cudaStream_t st);
// z[A] = Binv[A] x[A] for every node (FP32 blocks, FP64 vectors)
template <int N>
int launch_block_apply(const float* binv, const double* x, double* z, int64_t n_nodes, cudaStream_t st);

// Assembled tangent of the paper's variant (assembled.cu): per node-graph
// connection a record of assembled_record_floats(N) floats (K, L, G_1..3, D_1..3)
template <typename T, int N>
int launch_assemble_paper(const int32_t* node_off, const int32_t* node_elem, const int32_t* row_off,
                          const int32_t* cols, const int4* tets, const T* geo, const T* u0, const T* uc, const T* tau,
                          Phys<float> ph, float* H, int64_t n_nodes, cudaStream_t st);
template <int N>
int launch_spmv_paper(const int32_t* row_off, const int32_t* cols, const float* H, const uint8_t* dmask,
                      const float* x, float* y, int64_t n_nodes, cudaStream_t st);
int assembled_record_floats(int N);
// one colour of a block Gauss-Seidel sweep: z_A = Binv_A (r_A - sum_{B != A} H_AB z_B)
template <int N>
int launch_sgs_colour(const int32_t* rows, int64_t n_rows, const int32_t* row_off, const int32_t* cols,
                      const float* H, const float* binv, const uint8_t* dmask, const float* r, float* z,
                      int diag_only, cudaStream_t st);

// FP64 Krylov helpers (krylov.cu)
// h_out[j] = basis_j . w (j < nvec), with self also h_out[nvec] = w . w;
// with *skip != 0 (device flag) every h_out is 0 and nothing is read
int krylov_dots(const double* basis, int64_t ld, int nvec, const double* w, int64_t n,
                double* partial, double* h_out, cudaStream_t st, int self = 0,
                const double* skip = nullptr);
// w -= sum_j h_j basis_j, nothing when *skip != 0
int krylov_sub(double* w, const double* basis, int64_t ld, int nvec, const double* h, int64_t n,
               cudaStream_t st, const double* skip = nullptr);
// flag = 1 when the second Gram-Schmidt pass can be skipped (see krylov.cu)
int krylov_reorth_test(const double* h, int nvec, double* flag, cudaStream_t st);
int krylov_combine(double* x, const double* basis, int64_t ld, int nvec, const double* coef,
                   int64_t n, cudaStream_t st);
int vec_scale(double* out, const double* in, double a, int64_t n, cudaStream_t st);
int vec_axpy(double* y, const double* x, double a, int64_t n, cudaStream_t st);
int vec_cast_d2f(float* out, const double* in, int64_t n, cudaStream_t st);
int vec_cast_f2d(double* out, const float* in, int64_t n, cudaStream_t st);
int krylov_partial_blocks();
int vec_mul(double* out, const double* a, const double* b, int64_t n, cudaStream_t st);
// out = in / sqrt(*n2) with the squared norm read on the device
int vec_normalise(double* out, const double* in, const double* n2, int64_t n, cudaStream_t st);
// out = (float)(a b)
int vec_mul_d2f(float* out, const double* a, const double* b, int64_t n, cudaStream_t st);
// D = approximate inverse diagonal of the tangent for right preconditioning, 1 on
// fixed unknowns; part: scratch of 12 values an element
int launch_diag(const int4* tets, const double* geo, const double* y, int N, Phys<double> ph, const int32_t* node_off,
                const int32_t* node_elem, const uint8_t* dmask, double* part, double* D, int64_t n_elem,
                int64_t n_nodes, cudaStream_t st);

}  // namespace ts
