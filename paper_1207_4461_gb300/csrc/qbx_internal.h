// qbx_internal.h -- launch descriptors shared by the library's translation
// units (host side of the kernels).  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <vector>
#include "../../include/qbx.h"

namespace qbx {

struct cplx;

constexpr int kApplyThreads = 128;   // threads per CTA of the fused apply (and of the far and grad D kernels)
constexpr int kApplyCentres = 32;    // centres per CTA of the fused apply (one per lane, four warps)
// centre blocks of a fused apply: 32 consecutive centres of one side
inline int apply_units(int n_ctr, int n_tgt) {
  return (n_tgt + kApplyCentres - 1) / kApplyCentres * (n_ctr / n_tgt);
}
constexpr int kSrcTile = 128;        // sources staged in shared memory per step (far, form and grad D kernels)
constexpr int kFormThreads = 64;     // threads per CTA of form_locals (two warps for 32 centres)
constexpr int kMaxSplit = 64;        // source splits of the split reductions

struct SrcView {
  const double *x, *y, *nx, *ny;
  int n;
};

// Fused storage-free apply (a2-a6 fused) of an operator subset, one launch
// per chunk of `nr` rhs.
struct ApplyArgs {
  int ops;                // bit (1 << QBX_OP_S) | (1 << QBX_OP_D) | (1 << QBX_OP_GRAD_S)
  int p;
  double kre, kim;
  int n_ctr;              // centres in this launch
  const double *cx, *cy;  // [n_ctr]
  int n_tgt;              // target of centre c is c mod n_tgt
  const double *tx, *ty;  // [n_tgt]
  SrcView src;
  const void* wd[3];      // per operator (S, D, grad S): [n_src][nrhs] complex
  int nrhs, rhs0, nr;     // total rhs, first rhs of this chunk, chunk width
  int nsplit, src_per_split;
  void* part;             // [nsplit][n_ctr][ncomp][nrhs] complex, comps S, D, grad S (x, y)
  double eta2;            // near-only QBX: if > 0, sources with |x_s - c|^2 >= eta2 r^2 by the
                          // smooth rule at the target; otherwise (default) all through the expansion
  int near_q_tgt, near_q_src;   // > 0: near-field items first (node counts per panel); 0: plain order
  int one_w;              // 1: wd[] of every requested operator is one array and nr = 1 (weighted
                          // seeds: the density multiplies H0, H1); 0: per-pair kernel values
  const double* hk_tab;   // complex k: the amplitude table of this k's ray (launch_hk_table), or null
  const int *near, *near_cnt;   // near leaves of every 32-target block (near_q_src sources each; [blocks][near_stride], counts
                                // at [blocks][3]); the launch then covers their sources only.  null: all sources
  int near_stride;
};
// Amplitudes B_n = H_n(z) e^{-i(z - pi/4)}, n = 0, 1, along the ray z = k rho
// (|z| >= 2) as piecewise polynomials in s = |z|^{-1/2}, in the layout of the
// real-axis table (hk_table_doubles() doubles), for Im k > 0.
int hk_table_doubles();
cudaError_t launch_hk_table(double kre, double kim, double* tab, cudaStream_t st);
cudaError_t launch_debug_hankel_ray(double kre, double kim, const double* tab, const double* rho, int n, void* h0,
                                    void* h1, cudaStream_t st);
cudaError_t launch_apply_fused(const ApplyArgs& a, cudaStream_t st);
cudaError_t launch_apply_fused_real(const ApplyArgs& a, cudaStream_t st);
cudaError_t launch_apply_fused_cplx(const ApplyArgs& a, cudaStream_t st);
cudaError_t launch_apply_fused_local_real(const ApplyArgs& a, cudaStream_t st);
cudaError_t launch_apply_fused_local_cplx(const ApplyArgs& a, cudaStream_t st);
int apply_occupancy_local(int ops, bool ck, int p, int nr, bool one_w = false);   // near-only instances
// Storage-free grad D (one rhs per launch, a.rhs0; a.wd[0] the weighted
// density): partial sums [nsplit][n_ctr][2][nrhs] of the expansion gradient
// without the factor i/4.
cudaError_t launch_grad_d_fused(const ApplyArgs& a, cudaStream_t st);
size_t grad_d_fused_smem(bool ck, int p);
int grad_d_fused_occupancy(bool ck, int p);
size_t apply_smem_bytes(int ops, bool ck, int p, int nr);
size_t apply_smem_bytes_real(int ops, int p, int nr);
size_t apply_smem_bytes_cplx(int ops, int p, int nr);
int apply_chunk(int ops);   // rhs per launch for an operator subset
int apply_occupancy_real(int ops, int p, int nr, bool one_w = false);   // resident CTAs per SM
int apply_occupancy_cplx(int ops, int p, int nr, bool one_w = false);

// Far targets: plain quadrature partial sums.
struct FarArgs {
  int op;
  double kre, kim;
  int n_far;
  const double* xy;       // [n_far][2]
  SrcView src;
  const void* wd;
  int nrhs, rhs0, nr;
  int nsplit, src_per_split;
  void* part;             // [nsplit][n_far][ncomp][nrhs]
  const double* hk_tab;   // complex k: the amplitude table of this k's ray, or null
};
cudaError_t launch_far(const FarArgs& a, cudaStream_t st);

// Unfused coefficients (a4).
struct FormArgs {
  int kind, p;
  double kre, kim;
  int n_ctr, n_tgt;
  const double *cx, *cy;
  const int *near, *near_cnt;   // near leaves per 32-target block, as ApplyArgs::near (near_q sources each); null: all
  int near_stride, near_q;
  SrcView src;
  const void* wd;
  int nrhs, rhs0, nr;
  int nsplit, src_per_split;
  void* part;             // [nsplit][n_ctr][2p+1][nrhs]
  const double* hk_tab;   // complex k: the amplitude table of this k's ray, or null
};
cudaError_t launch_form(const FormArgs& a, cudaStream_t st);
size_t form_smem_bytes(int p, int nr);

// Evaluation of stored coefficients (a5 + a6).
struct EvalArgs {
  int what, p;
  double kre, kim;
  int n_eval;
  const double *ex, *ey;  // targets (may be null: default on-surface)
  const int* ectr;        // centre per target (null: identity)
  const double *cx, *cy;
  int n_tgt;
  const double *tx, *ty;
  const void* alpha;      // [n_ctr][2p+1][nrhs]
  int nrhs;
  void* out;
  int n_ctr;              // centres of the side (bound for ectr)
  int* status;
};
cudaError_t launch_eval(const EvalArgs& a, cudaStream_t st);

// Reductions over splits and epilogues.
// comp0: first component of operator `op` among the ncomp_total components
// of each partial-sum row.
cudaError_t launch_apply_finish(int op, int side, int limit, int n_tgt, int nsplit, int n_ctr,
                                int nrhs, int comp0, int ncomp_total, const void* part,
                                const void* dens_tgt, const double* tgt_nx, const double* tgt_ny,
                                void* out, int* status, cudaStream_t st);
cudaError_t launch_far_finish(int op, double kre, double kim, int n_far, int nsplit, int nrhs,
                              const void* part, void* out, int* status, cudaStream_t st);
cudaError_t launch_form_finish(int n_ctr, int ncoef, int nsplit, int nrhs, const void* part,
                               void* alpha, int* status, cudaStream_t st);

// Geometry, oversampling, centre assignment.
cudaError_t launch_geometry(int M, int q_tgt, int q_src, const double* t_edges,
                            const double* gam_tgt, const double* dgam_tgt,
                            const double* gam_src, const double* dgam_src,
                            const double* wgl_tgt, const double* wgl_src, double r_factor, int rule,
                            const qbx_geom& g, cudaStream_t st);
cudaError_t launch_upsample(int M, int q_tgt, int q_src, int nrhs, const double* interp,
                            const double* src_w, const void* dens_tgt, void* wdens,
                            cudaStream_t st);
cudaError_t launch_grad_d_finish(int n_tgt, int q_tgt, int nsides, int side0, int limit, int nrhs, const void* ev,
                                 const void* dens, const double* tnx, const double* tny, const double* tw,
                                 const double* wgl, const double* Dx, void* out, int* status, cudaStream_t st);
cudaError_t launch_tangents(int n, const double* nx, const double* ny, double* tx, double* ty, cudaStream_t st);
cudaError_t launch_assign(int n, const double* xy, int n_ctr, const double* cx,
                          const double* cy, const double* cr, int* out, cudaStream_t st);
cudaError_t launch_debug_hankel(const void* z, int n, void* h0, void* h1, cudaStream_t st);
cudaError_t launch_debug_besselj(const void* z, int n, int nmax, void* j, cudaStream_t st);

// Host helpers shared by the C-ABI translation units (qbx_capi.cu).
void host_interp_matrix(int q_tgt, int q_src, std::vector<double>& M);
size_t host_align256(size_t b);
int host_choose_split(int num_sms, int n_units, int n_src, size_t bytes_per_split, size_t avail);
int host_choose_split_waves(int num_sms, int occ, int n_units, int n_src, size_t bytes_per_split,
                            size_t avail, int min_waves = 1);
int host_split_len(int n_src, int ns);
int host_fail(int code, const char* msg);   // sets qbx_last_error(), returns code
void host_plan_info(const qbx_plan* plan, int* device, int* q_tgt, int* q_src, const double** interp);
// V_{j+1} = A V_j for a column-major n x n matrix (qbx_matmul_cm) and a basis V
// [.][n][nrhs], j = *step; nothing while *gate is 0 (both on the device).
int matmul_cm_step(int n, int nrhs, const qbx_c64* A, qbx_c64* V, void* work, size_t work_bytes, const int* gate,
                   const int* step, void* stream);

}  // namespace qbx

namespace qbx {

// ---- many right-hand sides and batches: the group kernel ------------------
constexpr int kGrpCentres = 32;   // centres per CTA (one per lane)
constexpr int kGrpWarps = 4;      // warps per CTA: rhs groups in phase 2
constexpr int kGrpRhsWide = 64;   // the rg code of the eight-warp instances (64 rhs per pass)
// the group kernel's operator set of the combined field D - i eta S (OPB_C)
constexpr int kOpsCombined = 16;
constexpr int kGrpTile = 32;      // sources per shared-memory tile

// One curve of a batch (or the single curve of a many-rhs apply).
struct GroupInst {
  double kre, kim;
  int n_src, n_tgt, n_ctr;        // n_ctr: centres of the side set
  int n_row;                      // rows of the partial sums: n_ctr, or n_tgt with both sides merged
  int side, nsplit, M;            // nsplit: partial sums of all kernels
  int nsplit_near;                // of the pair kernel
  const int *near, *near_cnt;     // near leaves per 32-target block, as ApplyArgs::near; null: all sources
  int near_stride, near_q;        // list stride, sources per leaf
  const double *sx, *sy, *snx, *sny, *sw;
  const double *cx, *cy;          // centres of the side set
  const double *tx, *ty, *tnx, *tny;
  const void* wd;                 // [n_src][nrhs] oversampled weighted density
  const void* dens;               // [n_tgt][nrhs] density on the target grid (jump terms)
  void* part;                     // [nsplit][n_row][ncomp][nrhs] raw sums
  void* out[3];                   // per operator (S, D, grad S) outputs, for the finish
  const double* hk_tab;           // complex k: the amplitude table of this curve's k, or null
};
// A work item: the rows [row0, row1) of the partial sums of instance inst, 32
// at most (centres: of one side, as a near list's block, or across the sides;
// merged: targets), sources [src0, src1) or the split's share of the near
// leaves, partial-sum slot `split`.
struct GroupItem {
  int inst, row0, row1, split, src0, src1;
};
struct GroupArgs {
  int ops, p, nrhs;
  int nsd;                        // 2: both sides of a target averaged per pair (S, D, S + D, D - i eta S), else 1
  const GroupInst* inst;          // dynamic mode: instance table
  GroupInst inst0;                // static mode: the one instance
  int n_items;
  const GroupItem* items;         // dynamic mode: item list (longest first)
  int* counter;                   // dynamic mode: next item (zeroed before launch)
  int st_units, st_nsplit, st_split_len;   // static mode (items == nullptr): one instance
  double eta2;                    // near-only QBX (> 0): sources with |x_s - c|^2 >= eta2 r^2 by the
                                  // smooth rule at the target; 0: all through the expansion
  double cf_re, cf_im;            // ops == OPB_C: eta of the combined field D - i eta S
};
cudaError_t launch_group_real(const GroupArgs& a, int rg, int grid, cudaStream_t st);
cudaError_t launch_group_cplx(const GroupArgs& a, int rg, int grid, cudaStream_t st);
size_t group_smem_real(int ops, int p, int rg, int nsd);
size_t group_smem_cplx(int ops, int p, int rg, int nsd);
int group_occupancy_real(int ops, int p, int rg, int nsd);
int group_occupancy_cplx(int ops, int p, int rg, int nsd);
// near-only instances of the group kernel (GroupArgs::eta2 > 0)
cudaError_t launch_group_local(const GroupArgs& a, bool ck, int rg, int grid, cudaStream_t st);
int group_occupancy_local(int ops, bool ck, int p, int rg, int nsd);

}  // namespace qbx

namespace qbx {

struct TreeArgs;
// ---- adjoint (transposed sweep) -------------------------------------------
struct AdjArgs {
  int ops, p, nrhs;
  double kre, kim;
  int n_ctr, n_tgt, n_src;
  const double *cx, *cy, *tx, *ty;
  const double *sx, *sy, *snx, *sny;
  const void* gc;        // [n_ctr][nrhs] gradient carried to each centre
  void* coef;            // [n_ctr][nslots][p+2] coefficient columns (workspace)
  double* cgeo;          // [n_ctr][3] target direction and 1/r (workspace)
  int nsplit, ctr_per_split;
  const int *near, *near_cnt;   // near leaves of every 32-source block (near_q targets each, all their centres);
  int near_stride, near_q;      // null: every centre
  void* part;            // [nsplit][n_src][ncomp][nrhs]
  const double* hk_tab;  // complex k: the amplitude table of this k's ray, or null
};
cudaError_t launch_adjoint_real(const AdjArgs& a, cudaStream_t st);
cudaError_t launch_adjoint_cplx(const AdjArgs& a, cudaStream_t st);
// the plan's side stream and the events that fork it from and join it to a call's stream
void host_plan_side(const qbx_plan* plan, cudaStream_t* side, cudaEvent_t* fork, cudaEvent_t* join);
// what qbx_debug_route reports of the call (t: its clusters, or null)
void host_plan_route(qbx_plan* plan, const TreeArgs* t);
void host_plan_workspace(const qbx_plan* plan, void** ws, size_t* bytes, int* num_sms, int** status);
cudaError_t adjoint_sums(AdjArgs& a, TreeArgs* tr, qbx_plan* plan, const qbx_geom* g, int c0, int nc, qbx_c64 k,
                         int fops, int nd, int mode, int num_sms, char* tree_base, cudaStream_t st);
// The plan's amplitude table for complex k (made on st when k changes, or in
// every captured call), or null for real k.
const double* host_plan_hk_table(qbx_plan* plan, qbx_c64 k, cudaStream_t st, cudaError_t* err);

}  // namespace qbx

namespace qbx {

// ---- cluster moments (qbx_tree.cu) -----------------------------------------
// Order of a cluster's outgoing expansion: admits clusters at 4.2 radii.  24
// would leave 8.0 near panels per block instead of 6.1 (starfish, 256 panels;
// 266k instead of 204k FP64 instructions of pairs per target), 36 6.0; a warp
// holds one order per lane.
constexpr int kTreeP = 30;
constexpr int kTreeLocal = 32;    // near-only QBX: orders of a centre's expansion that stands for the smooth rule
constexpr int kTreeMinPanels = 16;   // fewer panels: every source pair by pair (no cluster of 8 is far from any block)
constexpr int kTreeLevels = 16;
constexpr int kTreeUpCols = 8192;   // leaf columns up to which every level sums the sources again (TreeArgs::up = 0)
constexpr int kTreeSets = 4;
constexpr int kSupLevels = 7;
// what a moment set is made of: the density itself, or dipoles along n_s, x, y
enum { kSetMono = 0, kSetNormal = 1, kSetX = 2, kSetY = 3, kSetCombined = 4,
       kSetQuadX = 5, kSetQuadY = 6 };   // (the dipoles' derivatives along x, y)

struct TreeArgs {
  const TreeArgs* inst;       // a batch: one entry per curve (device memory), blockIdx.z the curve; else null
  double kre, kim;
  int p;                      // order of the centres' expansions
  int pl;                     // orders of the list entries (p, or kTreeLocal for near-only QBX)
  int nd;                     // derivatives taken on one side of a kernel (D, grad S: 1)
  double eta;                 // near-only QBX (> 0)
  int only_loc;               // lists: leaves that do not go through the block's local expansion are near
  int all_l;                  // stored coefficients: far nodes are evaluated for every order l <= p
  int M, q_src, n_src;        // leaves (halves of panels, or panels), sources per leaf, sources
  const double *sx, *sy, *snx, *sny;
  // adjoint sweeps: the nodes hold the discs of n_ctr_n centres (dcx, dcy) of
  // the targets (sx, sy), and the blocks evaluation points (tx = cx)
  int discs, n_ctr_n;
  const double *dcx, *dcy;
  int n_tgt, n_ctr;           // n_ctr = n_tgt or 2 n_tgt centres
  const double *cx, *cy, *tx, *ty;
  const double* hk_tab;
  int lev;                    // levels; node (l, j) is off[l] + j
  int off[kTreeLevels + 1];   // off[lev]: node count
  int n_blk;                  // 32-target blocks
  double* node;               // [nodes + n_blk + n_sup][4]: centre x, y, radius; then the blocks, super-blocks
  int* near;                  // [n_blk][M] near leaves
  int* far;                   // [n_blk][M + 1][2] far nodes: index, orders (cluster | centre << 8);
                              // last the block's local expansion (index nodes + block, bit 16 set)
  int* loc;                   // [n_blk][M][2] nodes of the local expansion: index, orders (cluster | block << 8)
  int* cnt;                   // [n_blk][3] counts: near, far, loc
  // super-blocks: 2^B consecutive blocks, B = 1..sup_lev, index
  // sup_off[B] + j; their entries follow the blocks' in node and coef
  int n_sup, sup_lev, sup_c, sup_off[kSupLevels + 2], sup_stride;
  int* sloc;                  // [n_sup][sup_stride][2] as loc
  int* scnt;                  // [n_sup][2] entries, largest centre order
  unsigned char* scov;        // [n_sup][M] leaves in the list of the super-block or of one above it
  int nset, nrhs;
  int kind[kTreeSets];
  int slot[kTreeSets];        // which of the call's densities
  const void* wd[kTreeSets];  // [n_src][nrhs] weighted densities
  int up;                     // many columns: the leaves' coefficients, carried upward node by node;
                              // few: leaf contributions to every level
  double eta_re, eta_im;      // kSetCombined: dipoles - i eta density
  void* mom;                  // few columns: [lev][M][nset nrhs][kTreeP + 2][2] leaf contributions
  int ncset;                  // coefficient column sets: a moment set, or its x, y derivative
  int base[2 * kTreeSets], shift[2 * kTreeSets], plain[kTreeSets];
  void* coef;                 // [nodes + n_blk + n_sup][kTreeP + 2][ncset nrhs][2] coefficients
  // evaluation (launch_far_clusters)
  int ops;                    // OPB_* bits
  int set_s, set_d, set_g, set_gx, set_x;   // column sets (grad S: the density's, its x derivative; y after x)
  int rhs0, nr;
  int nparts;                 // warps that share a far entry (1..4)
  int nsplit, split0;         // partial-sum rows split0 .. split0 + nsplit - 1
  void* part;                 // as ApplyArgs::part
};
// leaves, levels and node offsets of a run of panels; returns the node count
int tree_levels(int panels, int q_src, TreeArgs* a);
// device bytes of the arrays of `a` (lev, off, n_blk, nset, nrhs set); with
// base != null also their addresses
size_t tree_layout(TreeArgs* a, char* base);
// (several curves: a.inst and n_inst; a then holds the largest M, n_blk, node
// count and levels over the curves)
cudaError_t launch_tree_lists(const TreeArgs& a, cudaStream_t st, int n_inst = 1);    // nodes, block lists
// moments, coefficients, local expansions; ck: complex k
cudaError_t launch_tree_moments(const TreeArgs& a, bool ck, cudaStream_t st, int n_inst = 1);
cudaError_t launch_far_clusters(TreeArgs a, cudaStream_t st);         // partial sums of the far nodes
bool far_clusters_fit(const TreeArgs& a);                             // whether their kernel can hold the orders
// the same for many columns of S, D or the combined field (both sides of a
// target averaged when n_ctr = 2 n_tgt)
cudaError_t launch_far_group(const TreeArgs& a, bool ck, cudaStream_t st, int n_inst = 1);
bool far_group_fit(const TreeArgs& a, bool ck, int nsd);
// Coefficients alpha_l of every centre from its block's far nodes (column set
// set_s): partial sums [split][n_ctr][2p+1][nrhs] at split0 as FormArgs::part
cudaError_t launch_form_far(const TreeArgs& a, cudaStream_t st);
bool form_far_fit(const TreeArgs& a);
// Plain quadrature at points that share no blocks: every point walks the nodes
// on its own (columns set_s, or set_gx and the next for the gradient)
struct FarPointArgs {
  TreeArgs t;          // nodes and coefficients (no lists)
  int grad, dip;       // gradient; the pairs of near leaves: D kernel
  int n_far, nsplit, rhs0, nr;
  const double* xy;
  const void* wd;
  void* part;          // as FarArgs::part
};
cudaError_t launch_far_points(FarPointArgs a, cudaStream_t st);
// Far entries of the assembled matrix (t: leaves are whole panels, columns the interpolation's)
struct MatrixFarArgs {
  TreeArgs t;
  const double* tw;
  void* out;           // [n_tgt][n_tgt] column-major
};
size_t matrix_tree_setup(MatrixFarArgs* q, const qbx_geom* g, qbx_c64 k, qbx_c64 eta, int p, const double* hk_tab,
                         char* base);
cudaError_t launch_matrix_far(const MatrixFarArgs& q, const double* sw, const double* P, int num_sms, cudaStream_t st);
// nodes and coefficients only
cudaError_t launch_tree_nodes(const TreeArgs& a, cudaStream_t st);
// adjoint sweeps: the tree over the discs of the centres, evaluated at the
// source nodes (columns by ops: value, gradient, second derivatives), its
// arrays and far sums at `base`; returns their bytes (base null: only those),
// 0 where no clusters are formed
size_t adj_tree_setup(TreeArgs* t, const qbx_geom* g, int c0, int nc, qbx_c64 k, int p, int ops, int nd, int nrhs,
                      const double* hk_tab, const void* gc, int num_sms, char* base);
cudaError_t launch_adj_far(const TreeArgs& a, int mode, const double* snx, const double* sny, void* row,
                           cudaStream_t st);
// moment and column sets of a->ops, the densities of S, D, grad S (and X) in slots `slot`
void tree_columns(TreeArgs* a, const int slot[3]);
void tree_columns_grad_d(TreeArgs* a, bool sources);   // grad D (OPB_G); with sources also the dipoles' derivatives (OPB_X)
void tree_columns_discs(TreeArgs* a);                  // adjoint: value (S), gradient (G), d_xx and d_xy (X)

}  // namespace qbx
