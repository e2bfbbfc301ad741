// Device-side declarations shared by the kernels and the C-ABI layer.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace geo {

template <int P> struct Dim;
template <> struct Dim<2> {
  static constexpr int N = 8, M = 2, NC1 = 3, NC1P = 4, QTRI = 12, NC = 4, NB = 7, NQR = 4, NQS = 4, NQT = 24,
                       NS = 1, SMAX = 6, NBIN = 3 * NC + NQT + 6, NNZ = 16, NFN = 4, NEN = 2, RL = 2;
};
template <> struct Dim<3> {
  static constexpr int N = 20, M = 3, NC1 = 9, NC1P = 12, QTRI = 60, NC = 10, NB = 16, NQR = 4, NQS = 4, NQT = 24,
                       NS = 2, SMAX = 26, NBIN = 3 * NC + NQT + 6, NNZ = 96, NFN = 8, NEN = 3, RL = 8;
};
template <> struct Dim<4> {
  static constexpr int N = 32, M = 4, NC1 = 19, NC1P = 20, QTRI = 220, NC = 20, NB = 30, NQR = 9, NQS = 6, NQT = 42,
                       NS = 3, SMAX = 32, NBIN = 3 * NC + NQT + 6, NNZ = 192, NFN = 12, NEN = 4, RL = 8;
};

// Reference-element constants of one order in the bulk arithmetic type R, kept
// in constant memory (every thread of a warp reads the same entry, so the
// constant cache broadcasts).
template <int P, typename R> struct RefConst {
  R Dval[3 * Dim<P>::NNZ];                      // CSC values of D^xi, D^eta, D^zeta
  unsigned char Drow[3 * Dim<P>::NNZ];          // row (node i) of each value
  unsigned short Dptr[3 * (Dim<P>::N + 1)];     // column (node j) pointers
  R Eval[3 * Dim<P>::RL * Dim<P>::N];           // the same matrices by rows, padded to RL
  unsigned char Ecol[3 * Dim<P>::RL * Dim<P>::N];  // entries per row: [alpha][slot][row i]
  R psiFc[Dim<P>::NQT * Dim<P>::NFN];           // face-node basis at the face points
  unsigned char fnode[6 * Dim<P>::NFN];
  R psiEc[12 * Dim<P>::NS * Dim<P>::NEN];       // edge-node basis at the edge points
  unsigned char enode[12 * Dim<P>::NEN];
  R R_[Dim<P>::M * Dim<P>::M];
  R Dpat[3 * Dim<P>::NNZ];                      // D^alpha at the compiled pattern (refpattern.h)
  // ring order of the predictor's contraction and point values (ader_ring.cuh):
  // place 4 k + q of each node around each axis; point weights of a side face, of
  // the distinct points of a radial face (corner, middle of a side, centre) and of an
  // edge on their nodes in ring order; sums over m > 1 of the rows of R
  unsigned char rpos[3 * Dim<P>::N], tnode[Dim<P>::N];
  R wS[Dim<P>::NQS * Dim<P>::NFN], wR[3 * Dim<P>::NFN], wEd[Dim<P>::NS * P], Rs[Dim<P>::M - 1];
};

// Per-column matrices used by the bulk arithmetic, in its type R.  The FP64
// form points at the FP64 tables; the FP32-bulk form at FP32 copies made once
// at mesh creation (the FP64 masters stay on the device).  GB (the KKT rows of the
// nodal values), GM (those of the zone mean) and TN are stored
// [ncol][NBIN][3N], [ncol][3][NBIN] and [ncol][NC1][N], so that the
// threads of a node team read consecutive entries.
template <typename R> struct BulkTables {
  // pinvH: [ncol][SMAX][NC1P] (coefficients of one stencil zone adjacent, padded to
  // 16-byte vectors); Qs (FP32 only): upper triangle of Q by rows, off-diagonals doubled, each row
  // padded to a multiple of 4 entries
  const R *pinvH, *oct_inv, *Q, *Qs, *TF, *nF, *wF, *GB, *GM, *TN, *J0, *iJ0, *Sm, *gcl, *JF, *JE;
  // edge geometry: unit tangents and face normals at the edge points (around a radial
  // edge in ring order, svr_fn [nsv][4][NS][3])
  const R *se_t, *se_nang, *se_nradL, *se_nradR, *svr_fn, *sv_t;
  // Gauss weight times point weight: [ncol][M-1][NQT] of the face points, [nse][M-1][NS]
  // and [nsv][M-1][NS] of the edge points (times |dl|), at shell 0
  const R *WFt, *se_w, *sv_w;
  // [ncol] (l_0 / |x_0|)^2 of the column's zones (the same along a self-similar
  // column): the mesh scale of the WENO-AO eps, eps = 1e-12 + weta u_0^2
  const R* weta;
  // [ncol][NQT], [ncol][12 NS]: 1 / (interpolated J) at the face and edge points
  const R *iJF, *iJE;
};

// Read-only tables in device memory (see host_tables.h for the layouts).
struct DevTables {
  int n, nr, ncol, nsv, nse;
  long long Z, F, E, F_rad, E_rad;
  double gamma;
  int positivity;      // 1: scale nodal and point states toward the zone mean (rho, p > 0)
  int predictor;       // GEO_PRED_*: the predictor's execution schedule
  int riemann;         // GEO_RIEMANN_*: the face solver
  int* status;         // [1] bit 0 set by the U update when a zone leaves rho > 0, p > 0 (or is not finite)
  const double* qpow;  // [nr + 2]: q^k
  const double* iA0;   // [ncol][6]: 1 / A0 (reciprocal face areas at shell 0)
  const double* iq2;   // [nr + 2]: q^-2k
  const double* iq3;   // [nr + 2]: q^-3k
  const double* iV0;   // [ncol]: 1 / V0
  const double* dz0;   // [ncol]: in-sphere diameter 6 V0 / S0 of the zone at shell 0
  const double *D, *R, *wt, *psiF, *psiE, *wE;
  const int* st_n;
  const int* st_nb;
  const double* pinvH;
  const int* oct_nb;
  const double *oct_inv, *Q, *V0, *l0, *S0, *A0, *TF, *nF, *wF, *WF, *GB, *GM, *TN, *J0, *iJ0, *Sm, *gcl, *JF, *JE;
  const int *col_side_se, *col_side_sgn;
  const int *se_v, *se_col, *se_lf, *se_perm, *se_le, *se_rev;
  const double *se_t, *se_nang, *se_nradL, *se_nradR;
  const int *sv_nc, *sv_fse;
  const double* sv_t;
  // zones around a radial edge in ring order (face j between zones j and j + 1; three
  // zones: the fourth entry repeats the first): column, local edge [nsv][4]
  const int *svr_col, *svr_le;
  BulkTables<double> b64;
  BulkTables<float> b32;
};

// Mutable device state and work arrays of one mesh.
// Work arrays marked (R) hold the bulk arithmetic type (double or float).
struct DevState {
  double* U;     // [8][Z]
  double* phi;   // [F]
  void* Wc;      // (R) [8*NC1][Z] WENO-AO Taylor coefficients
  void* Bp;      // (R) [NQmax][F]  nodal normal B per face (canonical orientation)
  void* trF;     // (R) [(M-1)*NQT][Z][8] predictor states at the zone's face points
  void* trE;     // (R) [(M-1)*12*NS][Z][8] predictor states at the zone's edge points
  double* Ff;    // [8][F] time-integrated face fluxes (FP64 accumulation)
  double* Ee;    // [E]   time-integrated edge EMFs (FP64 accumulation)
  double* red;   // reduction scratch
  unsigned* ticket;   // [1] zero between reductions: blocks that have finished
  double* host_out;   // [1] pinned host word that takes a reduction's result
  int* status_out;    // [1] pinned host word that takes the physical-state flag after each step
  bool hl_fresh;      // Uhl is the split of U (a predictor run alone changes U's field)
  float* Uhl;    // FP32-bulk only: [16][Z] U split as hi = fl(U), lo = fl(U - hi), for the WENO differences
};

// Work arrays of the adjoint step (FP64): cotangents of every forward quantity.
struct AdjState {
  const double* gUp;    // [8][Z] cotangent of U at t+dt (input)
  const double* gphip;  // [F]    cotangent of phi at t+dt (input)
  double* gU;           // [8][Z] cotangent of U at t (output; accumulated)
  double* gphi;         // [F]    cotangent of phi at t (output)
  double* gFf;          // [8][F]
  double* gEe;          // [E]
  double* gtrF;         // like trF
  double* gtrE;         // like trE
  double* gW;           // [8*NC1][Z]
  double* gBpz;         // [NQT][Z] cotangent of the zone's KKT inputs from the face fields
  double* gphiz;        // [6][Z]   cotangent of the zone's face-mean inputs
  const double* U0;     // [8][Z] checkpoint state (read only, pristine)
  // Picard iterates of the checkpoint's predictor stored by its forward recompute
  // ([P-1][M-1][8][N][Z]), or null: the reverse predictor then recomputes them
  const double* It = nullptr;
};

enum Stage { ST_WENO = 0, ST_BPERP, ST_ADER, ST_FACE, ST_EDGE, ST_UPD_U, ST_UPD_PHI, N_STAGES };

struct Tables;
// copy the order-P reference constants into constant memory in type R (kernels.cu)
template <int P, typename R>
cudaError_t upload_reference_constants(const Tables& T);

// D^axis as the ring kernels apply it (kernels.cu), [N][N] at the order p; returns N
int ring_matrix_any(int p, int axis, bool transposed, double* D);

// launchers (kernels.cu); return cudaGetLastError() of the launch
template <int P, typename R>
cudaError_t launch_stage(int stage, const DevTables& T, const DevState& S, double dt, cudaStream_t st);
// stages ST_FACE .. ST_UPD_PHI of a small mesh in two launches; false (nothing launched)
// where the mesh is not small
template <int P, typename R>
bool launch_corrector_small(const DevTables& T, const DevState& S, double dt, cudaStream_t st, cudaError_t& e);
// the FP64 predictor (no positivity) that also stores its Picard
// iterates for the reverse sweep (It: [P-1][M-1][8][N][Z] doubles)
template <int P>
cudaError_t launch_ader_store_iterates(const DevTables& T, const DevState& S, double* It, double dt, cudaStream_t st);
cudaError_t launch_cfl(const DevTables& T, const DevState& S, double cfl, double* out_host,
                       cudaStream_t st);
cudaError_t launch_divb(const DevTables& T, const DevState& S, double* out2_host, cudaStream_t st);
// refresh S.Uhl from S.U (FP32-bulk meshes, after an upload)
cudaError_t launch_split_u(const DevTables& T, const DevState& S, cudaStream_t st);
cudaError_t probe_fma(int prec, cudaStream_t st, double* flops_per_s);
// reverse sweep of one step (FP64); the forward intermediates of the checkpoint
// state are in S (Wc, Bp, trF, trE), the pristine checkpoint in A.U0
template <int P>
cudaError_t launch_adjoint(const DevTables& T, const DevState& S, const AdjState& A, double dt, cudaStream_t st);
// the reverse kernel of one forward stage alone (ST_WENO, ST_ADER, ST_FACE, ST_EDGE)
template <int P>
cudaError_t launch_adjoint_stage(int stage, const DevTables& T, const DevState& S, const AdjState& A, double dt,
                                 cudaStream_t st);
int reduction_blocks(long long n);
cudaError_t launch_outer_br2(const DevTables& T, const double* phi, double* out_dev, double* gphi, cudaStream_t st);

}  // namespace geo
