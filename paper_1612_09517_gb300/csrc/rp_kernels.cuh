// Device-side data structures and kernel launchers of the radical-pair
// propagation (stochastic trace, Eqs. 13-23 of Lewis, Fay and Manolopoulos).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rp {

constexpr int kMaxNucDev = 24;

// Field-independent Hamiltonian constants in the layout order (rad/us).
// Per nucleus at position p: electron rad[p] (0 or 1), dimension d[p],
// configuration stride stride[p], the 2x2 electron matrix
//   U_p = sum_a u_a S_a,  u_a = (A_ax - i A_ay)/2,
// that multiplies I_+ in S.A.I = sum_a S_a (u_a I_+ + conj(u_a) I_- + A_az I_z),
// stored row-major as (re, im) pairs, and the column (A_xz, A_yz, A_zz).
template <typename T>
struct alignas(16) HamDev {
  long long Z;
  int n_nuc, n_half, n_one, aniso;
  T Je;     // 2J S1.S2 coupling J in rad/us
  T kappa;  // (k_S - k_T)/4: H' = H - i kappa (P_S - P_T)
  int rad[kMaxNucDev];
  int d[kMaxNucDev];
  long long stride[kMaxNucDev];
  T U[kMaxNucDev][8];
  T v[kMaxNucDev][3];
};

// Per-field scalars: Zeeman omega, 1/dE and the shift sh with
// z = (1/dE) H' a - sh a  (sh = E_c/dE for propagation).
template <typename T>
struct FieldDev {
  T omega, s, sh_re, sh_im;
};

enum StepMode { MODE_APPLY = 0, MODE_FIRST = 1, MODE_MID = 2, MODE_LAST = 3 };

// Terms that the accumulator takes with term n in the per-term kernels: three at a time
// in FP32 (phi_n, phi_{n-1} and phi_{n-2} are at hand), which cuts a term from 5.25 to 3.9
// vector passes on average; FP64 is bound by arithmetic and adds each.
inline int term_nacc(bool fp64, int n, int mode) {
  return mode == MODE_FIRST  ? 2
         : fp64              ? 1
         : mode == MODE_LAST ? (n - 2) % 3 + 1
                             : ((n - 1) % 3 == 0 ? 3 : 0);
}

// Vector passes (multiples of one state vector of every active row) of the
// Chebyshev term n of a macro-step in the per-term kernels: reads of
// phi_{n-1} (and phi_{n-2}), write of phi_n (not at the last term), the
// accumulator write (first term) or read-modify-write, the singlet slices (a
// quarter each).
inline double term_vector_passes(bool fp64, int n, int n_c) {
  if (n == 1) return 3.5;
  const bool last = n == n_c - 1;
  const double acc = term_nacc(fp64, n, last ? MODE_LAST : MODE_MID) ? 2.0 : 0.0;
  return (last ? 2.25 : 3.25) + acc;
}

// Per-row (one propagation) metadata, device arrays of length rows.  A row is
// active in the macro-steps start <= k < end of its window; rows are refilled
// with new work items as their windows end.
struct RowsDev {
  int* field;        // field index (into the per-field tables)
  int2* win;         // {start, end} macro-step window
  long long* sample; // sample index (coherent) or basis index (deterministic)
  long long* out;    // output slot in the per-sample array
  int* flag;         // rows selected for init / norm / finalize
  double* integral;  // int |P_S psi|^2 dt accumulated (FP64)
  double* survival;  // |psi(T)|^2
};

// Layout description for the state-initialisation kernels.
struct LayoutDev {
  long long Z;
  int n_nuc, n_half, n_one;
  int d[kMaxNucDev];
  int input_index[kMaxNucDev];  // Philox counter word 0 of the nucleus at position p
  long long stride[kMaxNucDev];
};

// Systems of one launch: device arrays of per-system constants, the system of
// each row (NULL: every row is system 0), the slot stride in configurations
// of the row buffers (>= every system's Z), and the Philox pair word of each
// system (pair_of[s], or pair_base + s when pair_of is NULL).
template <typename T>
struct SysTab {
  const HamDev<T>* ham;
  const LayoutDev* lay;
  const double* k_S;
  const int* row_sys;
  long long Zslot;
  uint32_t pair_base;
  const uint32_t* pair_of;
  int* err = nullptr;  // device error word (bit 0: a bounded wait gave up), may be NULL
  // J_z-sector superposition (deterministic = 3): rank of every configuration
  // within its nuclear-M class, and 1/sqrt(n_i) of propagation i (n_i states)
  const int* sec_rank = nullptr;
  const double* sec_scale = nullptr;
  long long plane = 0;  // > 0: state vectors in planes [row][e][plane], else [row][m][e]
  // rotated nuclear frames (anisotropic systems, or NULL): per system and layout
  // position the 10 x 10 complex matrix that takes laboratory amplitudes to it
  const double* frame = nullptr;
};

// ---- launchers (return cudaGetLastError after the launch) ----
// row_flag may be NULL (all rows).  coef holds 4 n_c values per field: the
// Chebyshev coefficients c_n (re, im) in T, then in FP32 the remainders
// c_n - fl(c_n), which the FP32 kernels add so that the coefficients act with
// FP64 accuracy (zero and unused in FP64).

template <typename T>
cudaError_t launch_coherent_amps(const SysTab<T>& S, const long long* row_sample,
                                 const int* row_flag, int rows, uint64_t seed, double* amps,
                                 double* uv, cudaStream_t st, int deterministic = 0);

template <typename T>
cudaError_t launch_init_state(const SysTab<T>& S, const double* amps, const long long* row_sample,
                              const int* row_flag, const int2* row_win, int rows,
                              int deterministic, T* S0, T* S1, double* integral, double* survival,
                              cudaStream_t st);

// One Chebyshev term over every row (see k_cheb_step), every row being the system `one`
// (its constants travel as kernel parameters).  aniso selects the anisotropic hyperfine
// path; singlet slices go to X[row][n][m] complex.  The allocation-free entry runs it; the
// others take launch_term.
template <typename T>
cudaError_t launch_step(const SysTab<T>& S, const HamDev<T>& one, int aniso,
                        const FieldDev<T>* fields, const int* row_field, const int2* row_win,
                        int macro, int rows, const T* cur, const T* prev, T* next, T* acc, T* X,
                        const T* coef, int n_c, int n, int mode, cudaStream_t st);

// y = (H - i K) x for `rows` state vectors (rp_apply_h).  FP32 systems with >= 8 spin-1/2
// nuclei whose partner tiles fit in shared memory stage them by bulk copies
// (k_cheb_step_bulk), the others run k_cheb_step.
template <typename T>
cudaError_t launch_apply(const HamDev<T>& one, int aniso, const FieldDev<T>& field, int rows,
                         const T* x, T* y, cudaStream_t st);

// Largest Z (configurations) that launch_macro_small can hold.
template <typename T>
int small_max_configs();

// A whole macro-step (terms 1 .. n_c - 1) of every active row in one launch,
// one CTA per row with the row's vectors in shared memory (S.Zslot must be
// <= small_max_configs<T>()): reads psi from P, writes the propagated psi to Q
// and the singlet slices to X.
template <typename T>
cudaError_t launch_macro_small(const SysTab<T>& S, const HamDev<T>* one, int aniso,
                               const FieldDev<T>* fields, const int* row_field,
                               const int2* row_win, int macro, const int* macro_dev, int rows,
                               const T* P, T* Q, T* X, const T* coef, int n_c, cudaStream_t st);

// A work item of the persistent launch: field index, system index, macro-steps,
// Philox sample (or basis index) and the slot in the per-sample output.
struct PItem {
  int field, sys, n_macro, pad;
  long long sample, out;
};

// One launch over all n_items work items of small systems (S.Zslot <=
// small_max_configs<T>()): each CTA takes items from *counter (zero before the
// launch) and propagates each item's whole horizon on chip, writing phi_S,
// phi_T and survival to per_sample[3 out ..] (see k_persistent_small).
// Xscratch holds n_c x Zslot complex per CTA; persistent_ctas gives the grid
// (CTAs resident at once; it also sets the kernel's shared-memory attribute,
// so it runs before the launch), persistent_smem the shared memory of a CTA.
template <typename T>
size_t persistent_smem(long long Zs, int n_c);
template <typename T>
int persistent_ctas(long long Zs, int n_c, int aniso);
template <typename T>
cudaError_t launch_persistent_small(const SysTab<T>& S, int aniso, const FieldDev<T>* fields,
                                    const T* coef, const T* L, const int2* meta,
                                    const PItem* items, int n_items, int* counter, int n_c, int deterministic,
                                    uint64_t seed, T* Xscratch, int ctas, double* per_sample,
                                    cudaStream_t st);

// ---- whole propagations of isotropic systems that fit one SM (rp_chip.cu) ----

struct ElecOp;

// Tables of a launch: per-system and per-field constants in FP64 (folded and
// rounded to T in the kernel), real sum coefficients per field r_n then
// r_n - fl(r_n) (2 n_c values), the time-integral factor.
template <typename T>
struct ChipArgs {
  const HamDev<double>* ham;
  const LayoutDev* lay;
  const double* k_S;
  const FieldDev<double>* fields;
  const T* coef;
  const T* L;
  int ldk;
  const int2* meta;
  uint32_t pair_base;
  const uint32_t* pair_of;
  int n_c, max_nuc, deterministic;
  uint64_t seed;
  const int* sec_rank;
  const double* sec_scale;
  const double* frame;  // as SysTab::frame
};

struct ChipPlan {
  bool split = false;  // one thread per configuration and electron state
  bool aniso = false;  // the same for anisotropic systems (ham and frame: rotated frames)
  int lk = 0;        // log2 of the configurations per thread
  int cb = 0;        // log2 of the CTAs per row (a cluster)
  int rpc = 1;       // rows per CTA (items launch)
  int threads = 0, slots = 0;
  size_t smem = 0;
};

// SMs of GB300: the rules of the launch plans are for this chip (grids ask the device).
constexpr int kChipSms = 152;

// Launch shape for systems of at most Zmax configurations, at least min_half
// spin-1/2 and at most max_nuc nuclei each, `load` configurations in all over
// n_items propagations; false if they do not fit one CTA.
template <typename T>
bool chip_plan(long long Zmax, int min_half, int max_nuc, long long load, int n_items, int n_c,
               bool trace, ChipPlan* out);
// The same for systems of spin-1/2 and spin-1 nuclei beyond one CTA, in FP32.
bool chip_cluster_plan(long long Zmax, int min_half, int max_nuc, int n_items, int n_c, bool spin1_only,
                       ChipPlan* out);
// The same for anisotropic systems (Z up to 2048 FP32, 1024 FP64, where they have the
// spin-1/2 nuclei to split by).
template <typename T>
bool aniso_plan(long long Zmax, int min_half, int max_nuc, int n_items, int n_c, bool trace,
                ChipPlan* out);
template <typename T>
int chip_ctas(const ChipPlan& P);  // CTAs resident at once; before the first launch

// One launch over all groups (groups[i] = first item and count, items of one
// field); scratch: n_c x slots x 2^lk complex per CTA.  trace != NULL: time-trace sums
// (as launch_trace) instead of the time integral.
template <typename T>
cudaError_t launch_chip_items(const ChipArgs<T>& A, const ChipPlan& P, const PItem* items,
                              const int2* groups, int n_groups, int* counter, T* Xscratch, int ctas,
                              double* per_sample, double* trace, const ElecOp& op,
                              cudaStream_t st);
// One macro-step of every active row: psi -> out, singlet slices to X (row
// stride n_c Zslot, any order within a slice).
template <typename T>
cudaError_t launch_chip_macro(const ChipArgs<T>& A, const ChipPlan& P, const int* row_sys,
                              const int* row_field, const int2* row_win, int macro,
                              const int* macro_dev, int rows, const T* psi, T* out, T* X,
                              long long Zslot, cudaStream_t st);

// ---- one Chebyshev term per launch (rp_term.cu) ----

// Constants of one field, 2/dE folded in: g_p = a_p/2 (isotropic) or the real
// entry of U_p, (ur, ui) its complex entry (rotated nuclear frame), both x sqrt 2
// for spin 1; D = the uniform part of the diagonal less the shift; s2 = 2/dE.
template <typename T>
struct alignas(16) TermField {
  T g[kMaxNucDev], ur[kMaxNucDev], ui[kMaxNucDev];
  T D[3], s2, J, kappa, pad[2];
};

// One system: p_in = spin-1/2 nuclei whose partner lies in the tile; the table of
// nuclear fields covers m mod tm (nuclei p < p_out) from entry tab.
template <typename T>
struct alignas(16) TermSys {
  long long Z, tab, tm, otab;  // otab: per tile, the nuclei p >= p_out (ring kernels)
  int n_half, n_nuc, p_in, p_out;
  unsigned rad;
  int pad2[3];
  int d[kMaxNucDev];
  long long stride[kMaxNucDev];
  T v[kMaxNucDev][3];
};

template <typename T>
struct TermArgs {
  const TermSys<T>* sys;
  const TermField<T>* field;
  const T* btab;
  const T* coef;  // r_n with the sign of (-i)^n, then r_n - fl(r_n)
  const int* row_sys;
  const int* row_field;
  const int2* row_win;
  long long Zslot, plane;  // row slot and plane stride in configurations
  int n_c;
  int xblk;  // slices in the tensor-core Gram layout
  int ring;  // k_term_ring (FP32, every n_half >= 9)
};

template <typename T>
int term_lk(bool aniso, int min_half);
int term_tile(int lk);  // configurations per block
template <typename T>
cudaError_t launch_term_table(const HamDev<double>* ham, const TermSys<T>* sys, int n_sys,
                              long long tm_max, long long tiles_max, bool aniso, T* btab,
                              cudaStream_t st);
// One term over every active row: vectors in planes [row][e][plane], slices to X
// (may be NULL); modes as k_cheb_step.
template <typename T>
cudaError_t launch_term(const TermArgs<T>& A, int lk, bool aniso, const T* cur, const T* prev,
                        T* next, T* acc, T* X, int macro, const int* macro_dev, int rows, int n,
                        int mode, cudaStream_t st);

// A whole macro-step of every active row of one isotropic FP32 system on a
// thread-block cluster per row, the row's Chebyshev vectors in distributed
// shared memory (see k_macro_cluster): reads psi from P, writes the propagated
// psi to Q and the singlet slices to X (tensor-core layout if xblk).
// macro_cluster_plan: whether the system fits (isotropic spin-1/2 and spin-1
// nuclei, Z / 2^c <= 2688 with c <= min(3, n_half)), and the launch shape;
// macro_cluster_max_active:
// clusters of that shape that fit the device at once (0 if none or on error).
struct ClusterPlan {
  int cbits = 0;    // log2 of the CTAs per cluster (per row)
  int local = 0;    // configurations per CTA
  int kpt = 1;      // configurations per thread
  int threads = 0;  // threads per CTA
  size_t smem = 0;  // dynamic shared memory per CTA
};
bool macro_cluster_plan(const HamDev<float>& H, ClusterPlan* out);
// Whether kernel = 0 takes the cluster path: the shapes with a compiled
// instance (measured faster than the per-term kernels).
bool macro_cluster_default(const HamDev<float>& H);
int macro_cluster_max_active(const HamDev<float>& H);
cudaError_t launch_macro_cluster(const HamDev<float>& H, const FieldDev<float>* fields,
                                 const int* row_field, const int2* row_win, int macro,
                                 const int* macro_dev, int rows, const float* P, float* Q,
                                 float* X, const float* coef, int n_c, long long Zslot, int xblk,
                                 cudaStream_t st);

// One field's time integral: Chebyshev half-width and macro-step length, and
// the decay rate (k_S + k_T)/2 factored out of the propagator.
struct IntegralIn {
  double dE, h, kbar;
};

// Low-rank factor of the time-integral weights of every field (see
// k_plan_integral): L[f][n][k], n < n_c, k < integral_ldk(n_c) (zero past the
// rank), meta[f] = (rank, leading terms that count), and, if W is not NULL, the
// complex weights W[f][n][m] themselves (L may be NULL then).  host_in: the
// same records on the host (they size the launch).
int integral_ldk(int n_c);
template <typename T>
cudaError_t launch_plan_integral(const IntegralIn* in, const IntegralIn* host_in, int n_fields,
                                 int n_c, T* L, int2* meta, double* W, cudaStream_t st);

// integral[r] += sum_z sum_k |sum_n L_nk (-i)^n x_n(z)|^2 for the macro-step
// just finished (x_n = singlet slices X[r][n]); one FP64 atomic per CTA.
template <typename T>
cudaError_t launch_project(const SysTab<T>& S, const T* X, const T* L, const int2* meta,
                           const int* row_field, const int2* row_win, int macro,
                           const int* macro_dev, int rows, int n_c, double* integral,
                           cudaStream_t st);

// The same time integral on the tensor cores (FP32 singlet slices that
// launch_term and launch_macro_cluster write with xblk = 1; tcgen05.mma kind::tf32 with a hi/lo split of
// every value, FP64 contraction with W).  Row r covers the configurations of
// its system ham[row_sys[r]] (row_sys NULL: system 0); Zs is the slot stride.
// n_sm sizes the grid; err receives
// bit 0 if a bounded wait gave up.  gram_tc_supported: the accumulator blocks
// of 2 n_c rows fit one 256-column buffer (n_c <= 96).  gram_tc_smem_bytes:
// dynamic shared memory of one CTA.
bool gram_tc_supported(int n_c);
size_t gram_tc_smem_bytes(int n_c);
cudaError_t launch_gram_tc(const float* X, const double* W, const int* row_field,
                           const int2* row_win, int macro, const int* macro_dev, int rows, int n_c,
                           long long Zs, const HamDev<float>* ham, const int* row_sys, int n_sm,
                           double* integral, int* err, cudaStream_t st);

// Floats per row of the singlet slices in the tensor-core Gram layout.
size_t xblk_floats_per_row(long long Zs, int n_c);

// *macro_dev += 1 (one thread): ends a graph-replayed macro-step.
cudaError_t launch_tick(int* macro_dev, cudaStream_t st);

// A 4 x 4 complex operator on the electron states e = 2 e1 + e2 (row-major),
// applied as A x 1 on the nuclei; on = 0 switches it off.
struct ElecOp {
  double re[16], im[16];
  int on;
};

// After macro-step `macro`, for every row active in it (psi = psi(t_i) in Q,
// i = macro + 1 - start): trace[4 i] += |<S|psi>|^2, trace[4 i + 1] += |psi|^2,
// and if A.on trace[4 i + 2] + i trace[4 i + 3] += <psi| A x 1 |psi>.
template <typename T>
cudaError_t launch_trace(const SysTab<T>& S, const T* Q, const int2* row_win, int macro, int rows,
                         const ElecOp& A, double* trace, cudaStream_t st);

template <typename T>
cudaError_t launch_norm(const SysTab<T>& S, const T* S0, const T* S1, const int2* row_win,
                        const int* row_flag, int rows, double* survival, cudaStream_t st);

template <typename T>
cudaError_t launch_finalize(const SysTab<T>& S, const RowsDev& R, int rows, double* per_sample,
                            cudaStream_t st);

// out[f] = (mean phi_S, mean phi_T, SE_S, SE_T, mean survival) over
// per_sample[off[f] .. off[f] + cnt[f]).
cudaError_t launch_stats(const double* per_sample, const long long* off, const long long* cnt,
                         int n_fields, double* out, cudaStream_t st);

// out[f] = (sum_i w_i phi_S, sum_i w_i phi_T, 0, 0, sum_i w_i survival) over
// entry i of per_sample[off[f] .. off[f] + cnt[f]) (w has cnt[f] entries):
// a deterministic trace assembled from weighted propagations.
cudaError_t launch_stats_weighted(const double* per_sample, const long long* off,
                                  const long long* cnt, const double* w, int n_fields,
                                  double* out, cudaStream_t st);

cudaError_t launch_zero(double* p, size_t n, cudaStream_t st);

}  // namespace rp
