// Internal interface between the C-ABI layer (api.cu) and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/bopgb.h"
#include "common.cuh"

// Allows fn every size of dynamic shared memory that a launch here asks for.
// The 48 KB that need no permission cover the static arrays too, so a size a
// little below them is refused like a larger one; and the permission does not
// follow the size of one call, which would take it from another thread's
// launch of the same kernel.
constexpr size_t SMEM_MAX = 225 * 1024;
template <class F>
bool allow_smem(F fn) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX) == cudaSuccess;
}

// Cell, its inverse and the linked-cell grid of one structure.
struct Geometry {
  double cell[9];  // rows = lattice vectors
  double inv[9];   // inverse matrix: frac = pos * inv
  int nc[3];       // linked cells per axis (cell width >= rc)
  int nimg[3];     // image search range for axes with fewer than 3 cells
  int pbc[3];
  double rc;
};

// Per-CTA scratch of the cluster builder (global memory).
struct ClusterScratch {
  unsigned long long* hkeys;  // [slots][hcap]
  int* hvals;                 // [slots][hcap]
  unsigned long long* skeys;  // [slots][maxs] site keys in cluster order
  int* sslot;                 // [slots][maxs] hash slot of every site
  int* scount;                // [slots][maxs] adjacency count / offset per site
  int hcap, maxs, newcap;
};

// Outputs of the cluster builder.
struct ClusterOut {
  int* level_end;        // [n][K+1]
  int* atom_nsite;       // [n]  (pass 1)
  int* atom_nadj;        // [n]  (pass 1)
  int* max_level;        // [K+2] largest |C_k| over atoms, then the largest adjacency (pass 1)
  const long long* site_off;  // [n+1] (pass 2 input)
  const long long* adj_base;  // [n+1] (pass 2 input)
  int* site_atom;        // [S]
  signed char* site_img; // [S][3]
  long long* adj_off;    // [S+1]
  int2* adj;             // [A]
  unsigned long long* n_products;  // block products of one moments pass (pass 2)
  unsigned long long* lvcnt;       // [S] per-level entry counts (pass 2)
  unsigned* order;                 // [S] ClusterView, may be null (pass 2)
  unsigned* top;                   // [S], [n], [S]: the pair form of the last level, may be null (pass 2)
  int* ntop;
  unsigned* topmask;
};

namespace bopk {
// nbr.cu
__global__ void k_bin_atoms(int n, const double* pos, Geometry g, int* cell_of, int* cell_count);
__global__ void k_fill_cells(int n, const int* cell_of, const int* cell_start, int* cell_fill, int* cell_atoms,
                             int* cell_slot);
__global__ void k_edge_flags(int n, const long long* row_ptr, const int* col, const signed char* img, int* flag);
__global__ void k_bonds(int n, const long long* row_ptr, const int* col, const signed char* img, const int* flag,
                        const int* bond_scan, int* bond_of_edge, int* bond_atoms, signed char* bond_img,
                        unsigned* status);
__global__ void k_bond_blocks(int nb, const double* pos, Geometry g, BondModel m, const int* bond_atoms,
                              const signed char* bond_img, double* bond_d, double* H64, float* H32, int HS);
__global__ void k_frac_range(int n, const double* pos, Geometry g, double* out);
}  // namespace bopk

// Host launchers (defined in the .cu files that hold the templates).
void launch_neighbors(int mode, int n, const double* pos, Geometry g, const int* cell_of, const int* cell_start,
                      const int* cell_atoms, int* deg, const long long* row_ptr, int* col, signed char* img,
                      unsigned* status, cudaStream_t s);
// Path-radius cut: with r2 > 0 only sites closer than sqrt(r2) to the
// cluster's atom (bond_vector arithmetic) join its cluster.
struct PathCut {
  const double* pos;  // [n][3] device
  double cell[9];
  double r2;
};
int launch_cluster(int pass, int n, int K, const long long* row_ptr, const int* col, const signed char* img,
                   const int* bond_of_edge, PathCut pc, ClusterScratch sc, ClusterOut out, int grid,
                   unsigned* status, cudaStream_t s);

void launch_level_sums(int n, int K, const int* level_end, long long* out, cudaStream_t s);
// Grid builder (cluster.cu): the same outputs as launch_cluster through a
// table of linked cells in shared memory, for rows of at most 32 neighbours.
constexpr int GRID_UNIT = 1 << 20;
struct GridPlan {
  int py, pz;   // periods of the second and third axis, in cells
  int slots;    // atoms per linked cell
  int origin;   // address of slot 0 of the cluster's own cell
  int tsize;    // addresses
  int mx, my, mz;  // images of sites: [-m, m] along each axis
};
// Plan of a structure from its maxima (launch_grid_maxima); false: the table
// has more than 65,535 addresses.
bool grid_plan(const Geometry& g, int K, const int* maxima, GridPlan* p);
void launch_grid_maxima(int n, const long long* row_ptr, int ncell, const int* cell_start, long long nb,
                        const double* bond_d, const Geometry& g, int* out, cudaStream_t s);
// {col, image}, {address offset, bond} of every directed edge, {first edge, degree} of every atom
int launch_pack_edges(int n, const GridPlan& p, const Geometry& g, const long long* row_ptr, const int* col,
                      const signed char* img, const int* bond_of_edge, const int* cell_of, const int* slot,
                      int2* epack, int2* eoff, int2* rows, cudaStream_t s);
struct GridArgs {
  int n, K;                  // clusters of the first n atoms
  int origin, tsize;         // GridPlan
  unsigned mx, my, mz;       // likewise
  unsigned ncode, qbits;     // cluster_key_codes, log2(newcap): sort keys (atom, image) << qbits | entry
  int lpr_shift;             // lanes per neighbour row: 4 (16 lanes) or 5 (32)
  int maxs, newcap;          // sites of one cluster, new sites of one level (a power of two)
  int sites;                 // pass 1: largest cluster (pass 0 found it)
  const int2* rows;          // [atoms] {first edge, degree}
  const int2* epack;         // [E] {col, image bytes + 128}
  const int2* eoff;          // [E] {address offset, bond}
  const int* slot;           // [atoms] place of an atom in its linked cell
  unsigned long long* recs;  // [n][maxs] site records kept from pass 0 to pass 1
  unsigned char* counts;     // [n][maxs] adjacency counts, likewise
  int* fail;                 // != 0 after pass 0: a cluster exceeds maxs, newcap or the table
  unsigned* status;
};
int launch_pair_mirror(int n, int K, const long long* site_off, const int* level_end, const int* site_atom,
                       const signed char* site_img, unsigned* mirror, unsigned* status, cudaStream_t s);
extern "C" int cluster_key_codes(int n, int ncode, int newcap);
int launch_cluster_grid(int pass, const GridArgs& a, const PathCut& pc, const ClusterOut& out, cudaStream_t s);

struct MomentsArgs {
  ClusterView cv;
  const void* H;       // float or double [nb][HS]
  int HS;
  const void* onsite;  // float or double [S][n_on][norb]
  int n, n_spin, norb, n_mom;  // n: atoms with clusters (centers), the first n of the structure
  int n_on;            // atoms of the structure (stride of the onsite levels)
  int cap_even;        // largest stored even level |C_k| (k < K) over atoms
  int cap_odd;         // largest stored odd level |C_k| (k < K) over atoms
  int max_sites;       // largest cluster |C_K|
  int max_adj;         // largest adjacency of one cluster
  double* mu;          // [S][n][norb][n_mom]
  // optional store of every Psi_k (NULL = none): rows of the item
  // (spin, atom) at spin psi_tot + psi_off[atom] rows, level k at row offset
  // sum_{j<k} |C_j|; row = norb x norb values padded
  void* pstore;
  const long long* psi_off;  // [n+1] prefix sums of sum_k |C_k| over atoms
  long long psi_tot;
  // pair form (needs cv.top; every atom a centre): FP64 computes, and both
  // precisions store, the selected rows of Psi_K only
  bool pair;
  // FP64 pair form: launch_pair_mirror's, and scratch of {row sum with Psi_K-1,
  // row sum of squares} per spin, site of every cluster and orbital
  const unsigned* mirror;
  double2* rowsum;
  long long nsite;     // sites of all clusters
  // Psi of two levels in global memory (moments_in_gmem): in the store, or in
  // scratch, one slot (moments_slot_bytes) per CTA
  bool gmem;
  void* scratch;
  size_t scratch_bytes;
};
size_t moments_slot_bytes(int norb, int cap_sum, int fp64);
bool moments_in_gmem(int norb, int cap_sum, int fp64);
int launch_moments(const MomentsArgs& a, int fp64, cudaStream_t s);

struct AdjointArgs {
  ClusterView cv;
  const void* H;
  int HS;
  const void* onsite;  // [S][n_on][norb]
  int n, n_spin, norb, n_mom;  // n: centers, as MomentsArgs
  int n_on;            // atoms of the structure (stride of onsite and Ebar)
  const double* w;     // [S][n][norb][n_mom]
  void* scratch;       // per-CTA Psi / Psi-bar storage
  size_t slot_elems;   // elements of T per CTA
  int slots;
  void* Hbar;          // [nb][HSh] (+=), the product type T (bond_cotangent_stride)
  int HSh;
  double* Ebar;        // [S][n_on][norb] (+=), may be null
  // reverse sweep over stored Psi (pstore != NULL; layout of MomentsArgs.pstore)
  const void* pstore;
  const long long* psi_off;
  long long psi_tot;
  bool gmem;           // stored-Psi sweep: Psi-bar of two levels in scratch (MomentsArgs::gmem)
  size_t scratch_bytes;
  int cap_even, cap_odd;  // largest even / odd level |C_k|, k = 1..K
  int max_sites, max_adj, cap_eb;  // cap_eb: largest |C_K-1|; max_adj: entries of its rows
  // stored-Psi sweep only: per cluster site t of work item (spin, atom i),
  // sum over the orbitals of dL/dE_t (+=), at siteval[spin * sv_stride +
  // site_off[i] + t] (t < |C_K-1|); may be null
  double* siteval;
  long long sv_stride;
  bool pair;           // stored-Psi sweep, no siteval: last level in the pair form (MomentsArgs::pair)
};
int launch_moments_adjoint(const AdjointArgs& a, int fp64, cudaStream_t s);
// Elements per bond of the cotangent array Hbar: the unique block elements
// (1, 15, 21), padded to a multiple of four in FP32 (float4 reductions).
int bond_cotangent_stride(int norb, int fp64);

// Non-collinear spin moments (moments.cu): work item (atom, orbital), the
// two local spin states of the atom as starting spinors.
struct NcArgs {
  ClusterView cv;
  const void* H;       // float or double [nb][HS]
  int HS;
  const void* onsite;  // float or double [2][n][norb]: E_up, E_dn
  const double* sdir;  // [n][3] unit moment directions
  int n, norb, n_mom;
  int cap_even, cap_odd;  // largest even / odd level |C_k| (k < K) over atoms (forward in shared memory)
  int rev_even, rev_odd;  // the same for k = 1..K (Psi-bar), |C_K-1| and the entries of its rows
  int cap_eb, rev_adj;
  int max_sites, max_adj; // largest cluster, largest adjacency
  // store of every Psi_k for the reverse sweep (NULL: none; k_nc recomputes):
  // rows of norb x 8 reals of item (atom, alpha) at alpha psi_tot + psi_off[atom]
  void* pstore;
  const long long* psi_off;
  long long psi_tot;
  void* scratch;       // per-CTA Psi / Psi-bar storage
  size_t slot_elems;   // elements of T per CTA: 2 sum_k max |C_k| norb 8
  int slots;
  // forward (w == NULL): local channel moments and Tr(sigma M_n)
  double* mu;          // [2][n][norb][n_mom]
  double* vmom;        // [n][norb][n_mom][3]
  // reverse (w != NULL): cotangents of sum w mu
  const double* w;     // [2][n][norb][n_mom]
  void* Hbar;          // [nb][HSh] (+=), the product type T (bond_cotangent_stride)
  int HSh;
  // FP32, over stored Psi: elements from Hbar to a second such array (else 0),
  // which the forces kernel adds to the first.  The sweep adds the cotangents
  // of a bond level by level and item by item, thousands of additions whose
  // rounding is a good part of the forces' error; centres take the arrays in
  // turn, for half the additions to each.  Forces of 432 bcc atoms at 9
  // moments, rms against FP64: d 2.77e-6 -> 2.46e-6, sd 3.82e-6 -> 3.12e-6,
  // with Psi recomputed and one addition per item and bond 2.69e-6 and 3.56e-6
  // eV/A.  (Rows in turn: no gain for d, the terms of one centre cancel.)
  size_t second;
  double* obar;        // [n][norb][4] (+=): d/d(Ebar, h_x, h_y, h_z)
};
// Two levels of the forward sweep, and of the reverse sweep with its onsite
// cotangents, fit shared memory.  The reverse one needs up to three times as
// much: it has a route of its own.
bool nc_fwd_in_shared(const NcArgs& a, int fp64);
bool nc_rev_in_shared(const NcArgs& a, int fp64);
int launch_nc(const NcArgs& a, int fp64, cudaStream_t s);
int launch_torques(int n, int norb, int n_mom, const double* onsite, const double* sdir, const double* w,
                   const double* vmom, const double* obar, double* t, cudaStream_t s);

// Band centre / width estimate of the constant terminator (BOP_BW_* of
// bopgb.h): mode, beta of the weighted average, (A, B) of the global mode.
struct BandSel {
  int mode;
  double beta, ga, gb;
};

// scalar.cu
struct ScalarArgs {
  int M;               // orbitals (all spins)
  int n_mom, n_exp;
  const double* mu;    // [M][n_mom]
  double* a;           // [M][Kp]
  double* b;           // [M][Kp+1]
  int* nlev;           // [M]
  double* a_inf;       // [M]
  double* b_inf;       // [M]
  double* gsig;        // [n_exp+1][M]   (coefficient-major)
  const double* g;     // [n_exp+1] damping
  unsigned* status;
  BandSel bw;
  unsigned* n_unbounded;  // may be null: orbitals with some |sigma_m| > m + 1
  int sig32 = 0;          // 1: the sigma_m recurrence in FP32 (FP32-products mode)
};
int launch_expand(const ScalarArgs& a, cudaStream_t s);
void launch_jackson(double* g, int n_exp, cudaStream_t s);

struct FermiState {
  double lo, hi, mid, ef;
  int done, iters, pad0, pad1;
};
int launch_fermi(int M, const double* D, const double* gsig, const double* a_inf, const double* b_inf, int n_exp,
                 double spin_factor, double target, FermiState* st, double* partials, unsigned* counter,
                 int max_rounds, double tol, cudaStream_t s);

// One piece of a Fermi-level solve spread over several processes (chain.cu):
// mode 0: out = {-min(a_inf - 2 b_inf), max(a_inf + 2 b_inf)}; mode 1: out =
// {sum N_o(E), sum n_o(E)} over this process's M orbitals (out device [2]).
int launch_fermi_eval(int mode, int M, const double* gsig, const double* inv, const double* a_inf,
                      const double* b_inf, int n_exp, double E, double* partials, unsigned* counter, double* out,
                      cudaStream_t s);
int launch_orbital_NU(int M, int n_exp, const double* gsig, const double* inv, const double* a_inf,
                      const double* b_inf, const double* onsite, const FermiState* st, double* N, double* U,
                      double* dos, cudaStream_t s);
int launch_orbital_N(int M, int n_exp, const double* gsig, const double* inv, const double* a_inf,
                     const double* b_inf, const FermiState* st, double* N, double* dos, cudaStream_t s);
// Newton steps inside the bisection bracket (chain.cu); warm: start from st->ef
int launch_fermi_newton(int M, const double* gsig, const double* inv, const double* a_inf, const double* b_inf,
                        int n_exp, double spin_factor, double target, FermiState* st, double* partials,
                        unsigned* counter, int warm, int rounds, int max_rounds, double tol, cudaStream_t s);
int launch_fermi_more(int M, const double* gsig, const double* inv, const double* a_inf, const double* b_inf,
                      int n_exp, double spin_factor, double target, FermiState* st, double* partials,
                      unsigned* counter, int rounds, int max_rounds, double tol, cudaStream_t s);
void launch_inverse_table(double* inv, int n, cudaStream_t s);
// The whole Fermi solve (bracket, Newton rounds, N and DOS at E_F) in one
// cooperative launch; partials: >= 4 x (grid) doubles.  -2: cooperative
// launch unavailable.
int launch_fermi_coop(int M, const double* gsig, const double* inv, const double* a_inf, const double* b_inf,
                      int n_exp, double spin_factor, double target, FermiState* st, double* partials, int warm,
                      int max_rounds, double tol, double* N, double* dos, cudaStream_t s,
                      const float* gs32 = nullptr);
// FP32 copy of gsig [n_exp+1][M] (the starting point of a cold Fermi search).
int launch_gsig_f32(int M, int n_exp, const double* gsig, float* gs32, cudaStream_t s);

struct ScfArgs {
  int n, norb, n_spin, mode;  // mode 1 = LCN, 2 = Stoner
  double spin_factor, n0, eta, tol, dos_floor, stoner_I, m_mix, onsite0;
  const double* N;     // [S][n][norb]
  const double* dos;   // [S][n][norb]
  double* delta;       // [n]
  double* m;           // [n]
  double* delta_new;   // [n]
  double* m_new;       // [n]
  double* onsite;      // [S][n][norb] (rebuilt)
  float* onsite32;
  double* red;         // partials [grid][64]
  unsigned* counter;
  double* result;      // [4]: max|res|, max|dm|, converged, mean
  int mixer;           // 0 linear, 1 Anderson
  int hist;            // Anderson history depth (<= 8)
  int it;              // iteration index of this update (0-based)
  double* hx;          // [(hist+1)][ncomp*n] iterates
  double* hf;          // [(hist+1)][ncomp*n] preconditioned residuals
  double* gamma;       // [hist] least-squares coefficients
  const double* grad;  // mode 3 (variational): dU_B/d delta_i [n]
  double J;            // mode 3: onsite charging J_ii
};
int launch_scf_residual(const ScfArgs& a, cudaStream_t s);
int launch_scf_apply(const ScfArgs& a, cudaStream_t s);
void launch_to_float(const double* in, float* out, size_t n, cudaStream_t s);
void launch_build_onsite(int n, int norb, int n_spin, double onsite0, double onsite_s, double stoner_I,
                         const double* delta,
                         const double* m, double* onsite, float* onsite32, cudaStream_t s);

// e_i = s sum U (- I m_i^2 / 4 with m) (+ J q_i^2 / 2, q_i = s sum N - n0, with N)
//       (+ erep_i with erep)
int launch_energy(int n, int norb, int n_spin, double spin_factor, double stoner_I, const double* U,
                  const double* m, double J, const double* N, double n0, const double* erep, double* e_atom,
                  double* red, unsigned* counter, double* e_total, cudaStream_t s);

struct WeightArgs {
  int M, n_mom, n_exp, norb;
  const double* mu;
  const double* onsite;  // [M]
  const FermiState* st;
  const double* g;
  const float* g32;      // the same in FP32 (a conversion costs a double-precision instruction)
  const double* inv;     // [n_exp+16] 1/k
  double cU;             // L = cU*U + cN*N
  const double* lam;     // device scalar: cN = -cU * (*lam)  (E_F response); NULL: cN = cN0
  double cN0;
  double* w;             // [M][n_mom]
  double* dU_dE;         // [M] direct derivative of L w.r.t. the onsite level, may be null
  double* zscratch;      // [2][n_exp+1][M]: sigma_m and its cotangent
  unsigned* status;
  BandSel bw;
  // n_spin 1 only: per-atom cN = cU (var_J var_q[i] - var_lam[0]) when var_q
  // is set (the variational SCF's binding energy U_B); else lam / cN0 above
  const double* var_q;
  const double* var_lam;
  double var_J;
  int sig32 = 0;  // 1: the sigma_m recurrences (forward and reverse) in FP32 (FP32-products mode)
};
int launch_weights(const WeightArgs& a, cudaStream_t s);
// Weights of L1 = cU1 U + cN1 N into a.w and of L2 = cU2 U + cN2 N into w2 at
// fixed E_F (a.lam unused), one lane per seed; a.zscratch: [4][n_exp+1][M].
int launch_weights_pair(const WeightArgs& a, double cU1, double cN1, double cU2, double cN2, double* w2,
                        cudaStream_t s);
int launch_ef_response(int M, const double* onsite, const double* dos, const FermiState* st, double* red,
                       unsigned* counter, double* lam, cudaStream_t s);

// learned.cu: the learned terminator (n_mom = 9, continued to 8 levels)
struct LearnedArgs {
  int M, n_exp, fp64;
  int sig32;             // 1: the sigma_m recurrences in FP32
  const double* mu;      // [M][9]
  double* base;          // [M][10]: a_0..a_3, b_1..b_4, a_inf, b_inf of the 9-moment chain
  int* nlev;             // [M] levels of the 9-moment chain
  unsigned char* flag;   // [M]: 1 = inputs inside the training range, 2 = continued chain used
  void* xs;              // T [M][18] standardised inputs (T = double if fp64 else float)
  const void* ys;        // T [M][10] standardised outputs
  const float* norm;     // [BOP_MLP_NNORM] standardisation and training range
  double* a_inf;         // [M] terminator of the chain used
  double* b_inf;
  double* gsig;          // [n_exp+1][M]
  const double* g;       // [n_exp+1] damping
  unsigned* n_learned;   // += orbitals on the continued chain
  unsigned* status;
  void* ybar;            // T [M][10] cotangent of the standardised outputs
  double* cot;           // [M][10] cotangent of the base record
  const void* xbar;      // T [M][18] cotangent of the standardised inputs
  WeightArgs W;          // E_F, onsite, damping, 1/k table, cU, lam, w, zscratch
};
// stage 0: features, 1: continued chain + expansion, 2: reverse of the chain
// part, 3: reverse of features / Gershgorin / recursion -> W.w
int launch_learned(int stage, const LearnedArgs& a, cudaStream_t s);
int launch_mlp_dataset(long long M, const double* mu17, float* x, float* t, float* mask, cudaStream_t s);

// mlp.cu: network on M rows with the bfloat16 inference weights
int mlp_infer_forward(int fp64, int M, const void* xs, const float* params, const void* wbf, void* Z1, void* H1,
                      void* Z2, void* H2, void* ys, cudaStream_t s);
int mlp_infer_backward(int fp64, int M, const void* ybar, const void* wbf, void* Z1, void* Z2, void* dZ1, void* dZ2,
                       void* xbar, cudaStream_t s);
const float* mlp_params_dev(const bop_mlp* net);
const void* mlp_wbf_dev(const bop_mlp* net);
const float* mlp_norm_dev(const bop_mlp* net);

// scf_adjoint.cu: vector kernels of the SCF-response solve (nu = n or 2n unknowns)
// w_out = (wU or 0) + sign * c_{atom,spin} * wN, c = s v[atom] + sigma_spin v[n + atom] (Stoner)
// Variational SCF: q_i = s sum_alpha N - n0 into q, and the E_F multiplier
// of U_B = U_bond + J sum q^2 / 2 into lam[0]:
// Lambda = sum_i D_i (E_F - E_i + J q_i) / sum_i D_i, D_i = s sum_alpha dos.
int launch_var_lambda(int n, int norb, double s, double J, double n0, const double* N, const double* dos,
                      const double* onsite, const FermiState* st, double* q, double* lam, double* red,
                      unsigned* counter, cudaStream_t stream);
int launch_scale_by_inv_norm(int nu, double* u, const double* nsq, cudaStream_t stream);
// The GMRES solve J^T y = rhs over the rows of J as per-site values
// (launch_jt_build, AdjointArgs.siteval): right preconditioner diag(P),
// cycles of GM_KRYLOV steps, relative residual rtol or max_it steps.
// V [GM_KRYLOV + 1][nu], x, xy [nu] scratch; part GMRES_PART doubles;
// out: iterations, relative residual, converged.  -2: cooperative launch not
// possible.
constexpr int GM_KRYLOV = 40;      // basis size per cycle
constexpr int GM_CYCLES = 3;       // cycles (restarts + 1)
constexpr int GMRES_BLOCKS = 512;  // most blocks of the launch
constexpr int GMRES_PART = GMRES_BLOCKS * (2 * (GM_KRYLOV + 1) + 1);
struct GmresArgs {
  int n, nu, max_it;           // nu = n, or 2n with the Stoner moments
  long long stride;            // val: spin s at val + s stride
  const long long *ptr, *idx;
  const int* row;
  const double *val, *rhs, *P;
  double s, I, rtol;
  double *V, *x, *xy, *y, *part, *out;
};
int launch_gmres(const GmresArgs& g, cudaStream_t stream);
// J^T v of the SCF response from the per-site values of one sweep with the
// dN/dmu weights (AdjointArgs.siteval).  The transpose of the rows: for
// every atom j the global sites of other atoms' clusters (first |C_K-1|
// sites) whose atom is j, with the owning atom (stage 0: counts into cnt;
// stage 1 after the scan of cnt into ptr: fill, cnt zeroed first).  Then
// Eb[spin][j] = sum over the entries of c_{i,spin} val[spin][site], c =
// s v[i] (+ sigma_spin v[n + i] for Stoner).  Eb: [S][n].
int launch_jt_build(int n, int K, const long long* site_off, const int* level_end, const int* site_atom,
                    int* cnt, int stage, const long long* ptr, long long* idx, int* row, cudaStream_t stream);
int launch_jt_gather(int n, int S, const long long* ptr, const long long* idx, const int* row, const double* val,
                     long long stride, const double* v, double s, int stoner, double* Eb, cudaStream_t stream);
int launch_scale_weights(int n, int norb, int S, int n_mom, double s, int stoner, const double* v, double sign,
                         const double* wN, const double* wU, double* w_out, cudaStream_t st);
// out_u = derivative w.r.t. u of a function whose onsite-level derivative is Eb (+ dUE):
//   delta part sum_{alpha,nu}; Stoner moment part sum_alpha (-I/2 up + I/2 down),
//   plus mcoef * m[i] (energy: -I/2 m) and minus v_m[i] if v_m (the -m_i of Q_i)
int launch_project(int n, int norb, int S, double I, const double* Eb, const double* dUE, const double* m,
                   double mcoef, const double* v_m, double* out, cudaStream_t st);
// P = diagonal preconditioner: -1/max(s sum n_i, floor) for delta, -1 for m
int launch_precond_diag(int n, int norb, int S, double s, double floor_, const double* dos, double* P,
                        cudaStream_t st);
int launch_dots(int nu, int nvec, const double* V, const double* w, double* out, cudaStream_t st);
// w -= sum_k coef[k] V[k]  (coef device)
int launch_axpy_multi(int nu, int nvec, const double* V, const double* coef, double* w, cudaStream_t st);
// out = scale * (sum_k coef[k] V[k]) * (P if P else 1)
int launch_lincomb(int nu, int nvec, const double* V, const double* coef, const double* P, double scale,
                   double* out, cudaStream_t st);
// out = a * x * (P if P else 1)
int launch_scale_vec(int nu, const double* x, const double* P, double a, double* out, cudaStream_t st);

// forces.cu
// Pair repulsion per atom (half of each of its bonds) into erep [n].
int launch_rep_energy(int n, BondModel m, const long long* row_ptr, const int* bond_of_edge, const double* bond_d,
                      double* erep, cudaStream_t s);
int launch_forces(int nb, BondModel m, const double* bond_d, const int* bond_atoms, const void* Hbar, int HSh,
                  size_t second, int fp64, double* forces, double* virial, cudaStream_t s);

// batch.cu
// Up to ZERO_MAX arrays of 4-byte words set to zero in one launch (blocks is
// filled in by the launcher).
constexpr int ZERO_MAX = 10, ZERO_WORDS = 4096;
struct ZeroArgs {
  int n;
  unsigned* p[ZERO_MAX];
  long long words[ZERO_MAX];
  int blocks[ZERO_MAX];
};
int launch_zero(ZeroArgs z, cudaStream_t s);
// Up to COLLECT_MAX pieces of 4-byte words copied to dst + at[q] (pinned host
// memory).
constexpr int COLLECT_MAX = 16;
struct CollectArgs {
  int n;
  const unsigned* src[COLLECT_MAX];
  int at[COLLECT_MAX], words[COLLECT_MAX];
  unsigned* dst;
};
int launch_collect(const CollectArgs& a, cudaStream_t s);
// Exclusive prefix sums of n <= SCAN_SMALL elements, of a second array too
// where in1 is not NULL.
constexpr int SCAN_SMALL = 8192;
template <class Tin, class Tout>
int launch_scan_small(const Tin* in0, Tout* out0, const Tin* in1, Tout* out1, int n, cudaStream_t s);
