// Kernel declarations shared by the engine and the kernel translation units.
#pragma once
#include <vector>

#include "common.cuh"

namespace ptk {

constexpr int QR_THREADS_ = 512;

struct Super4;

__global__ void k_site_contract(Tables T, const SiteWork* work, int n_work);
__global__ void k_site_swap(Tables T, const SiteWork* work, int n_work);
__global__ void k_build_blocks(Tables T, const BondWork* work, int n_work);
__global__ void k_householder(Tables T, const BondWork* work, int n_work);
__global__ void k_theta_gate(Tables T, const BondWork* work, int n_work);
__global__ void k_nan_guard(Tables T, const BondWork* work, int n_work);
constexpr int BOND_LOG_INTS = 10;
__global__ void k_bond_log(Tables T, const BondWork* work, int n_work, int layer, int* log, int cap_steps, int nb);
// the autotuner's synthetic full-capacity state: every Gamma at capacity filled with seeded values
// in (-1, 1), every lambda with a decaying unit-norm profile (dims set by the host beforehand)
__global__ void k_tune_fill(Tables T, int n_sites, int n_lams, unsigned seed);
// rsvd: the singular values are the range finder's l = info[9] values, plus the part of D outside
// its subspace as one lumped value ||D - Q Q^H D||_F (info[12..13]) when l < min(m, n)
__global__ void k_truncate(Tables T, const BondWork* work, int n_work, int chi_max, double eps,
                           double mtol, int rsvd = 0);
__global__ void k_recover(Tables T, const BondWork* work, int n_work);
__global__ void k_caps(Tables T, int n_mpos);
__global__ void k_step_inc(int* step);
__global__ void k_svd_load(const double2* A, int m, int n, int batch, double2* work_A,
                           size_t strideA);
__global__ void k_svd_store(const double2* work_A, const double2* work_V, const double* sig,
                            const int* perm, int m, int n, int batch, size_t strideA,
                            size_t strideV, double* sigma_out, double2* U, double2* V);

// whole-GPU Householder QR/LQ of the outer blocks of every bond of a layer (hqr_grid.cu), and the
// same factorisation over a list of matrices: A (m x n, m >= n, column-major, ld m) is replaced by
// the explicit Q, R (n x n, ld n) receives the triangular factor, H (m x n) and tau (n) are scratch
struct QRItem {
  double2* A;
  double2* H;
  double2* R;
  double* tau;
  int m, n;
};
void launch_hqr_items(const QRItem* items, int n_items, int blocks, unsigned* sync3, int* status, cudaStream_t st);
int hqr_items_ok();
int hqr_grid_ok();
int hqr_grid_fits(int total_cols_cap, int n_items, int blocks);
void launch_hqr_grid(const Tables& T, const BondWork* work, int n_work, int blocks, unsigned* sync3,
                     cudaStream_t st);

// blocked QR with the explicit Q (qr_block.cu): panels by clusters, the rest as nine-slice tensor-core products.
// One QRBlk per matrix: its workspace at capacity m_cap x n_cap (qr_block_bytes lays it out from base; base NULL:
// the size only); q is written by the call from the live dims
struct ZGemmItem;
struct QRBlk {
  QRItem q;
  double2 *Wp, *X, *S;
  unsigned char *TA, *TB, *TA2, *TB2;
  int m_cap, n_cap;
};
struct QRBlkList {
  QRBlk* blk = nullptr;    // device, n_items
  ZGemmItem* ops = nullptr;    // device, qr_block_ops(n_items, n_cap)
  int n_items = 0, m_cap = 1, n_cap = 1;
  int cluster = 0;         // qr_block_cluster(n_items, m_cap)
};
int qr_block_cluster(int n_items, int m_cap);
constexpr int QR_BLOCK_MAX_ROWS = 6400;      // the longest panel that the largest cluster holds
size_t qr_block_bytes(int m, int n, QRBlk* B, char* base);
size_t qr_block_ops(int n_items, int n_cap);
// the whole factorisation of small matrices, one CTA each (items' live shapes at most m_cap x n_cap)
int qr_small_fits(int m_cap, int n_cap);
void launch_qr_small(const QRItem* items, int n_items, int m_cap, int n_cap, int* status, cudaStream_t st);
// list: the matrices (n_items of them), or NULL: the outer blocks of the layer's bonds (matrix 2 w: B_L of bond w,
// 2 w + 1: B_R^H)
void launch_qr_block(const Tables& T, const BondWork* work, const QRItem* list, const QRBlkList& L, int* status,
                     cudaStream_t st);

// cluster-parallel FP64 bond SVD (jacobi_cluster.cu)
int jacobi_cluster_size(int want);
void launch_jacobi_cluster(const BondWork* work, int n_work, int cluster, int max_sweeps, int* status,
                           cudaStream_t st);

// whole-GPU FP64 bond SVD (jacobi_grid.cu): blocks = the SM count (0 if not co-schedulable); rows_cap: the
// largest column length at capacity (rows of the matrix, plus those of V with with_v); sync3: 3 words of device
// memory (arrival count, unused, abort flag). Sweeps go to info[3], rotation counters in info[4..5].
int jacobi_grid_blocks();
constexpr double JACOBI_FLOOR2 = 1.232595164407831e-32;      // squared noise floor: u^2 = 2^-106
// on_b: 0 = the matrix in A, 1 = B = R^H of the pivoted QR (Na x info[8]), 2 = R^H of the range finder's l x l
// factor R in G64 (l = info[9]), formed and overwritten by its left vectors in V; with_v: accumulate V; tol_scale: rotation
// threshold in units of the unit roundoff (0: the row count); floor2: columns at floor2 ||A||_F^2 or below (squared norms)
// are left as they are; wait_cycles: the part of the waits' limit that does not grow with a sweep (0: the usual one)
cudaError_t launch_jacobi_grid(const BondWork* work, int n_work, int blocks, int rows_cap, int max_sweeps,
                               unsigned* sync3, int* status, cudaStream_t st, int on_b, int with_v, double tol_scale,
                        double floor2 = JACOBI_FLOOR2, long long wait_cycles = 0);

// the standalone batched SVD's Jacobi (k_svd_load before it, k_svd_store after it) on Ma x Na matrices: the whole
// GPU where it can be co-scheduled and a launch takes the batch, else one cluster per matrix; sync3 as above; tune: the
// CTAs and the wait limit of a diagnostic call (0: the usual ones)
struct JacobiTune {
  int ctas = 0;
  long long wait_cycles = 0;
};
void launch_svd_jacobi(const BondWork* items, int batch, int Ma, int Na, int max_sweeps, int* status, unsigned* sync3,
                       cudaStream_t st, const JacobiTune& tune = JacobiTune{});

// the standalone SVD after two QRs (svd_qr.cu): its workspaces (of size svd_qr_layout), the host copies of its lists
// (kept until the stream is synchronised); items: n x n matrices in SvdQr::T with V in wV
struct SvdQr {
  double2 *Y, *T, *M, *Vp;
  double *tau, *nrm;
  int *pcol, *prow;
  QRItem* qr;
  QRBlk* blk;
  struct ZGemmItem *mul, *ops;
  char* blk_ws;
  unsigned char* pack;
  size_t per_blk, per_a, per_b;
};
struct SvdQrHost;
// by shape alone (the workspace's size follows it); and whether the current device takes the panels' clusters
bool svd_qr_shape(int Ma, int Na, int batch);
bool svd_qr_fits(int Ma, int Na, int batch);
size_t svd_qr_layout(int Ma, int Na, int batch, SvdQr* out, char* base);
void launch_svd_qr(const double2* A, int m, int n, int batch, const BondWork* items, double2* wA, double2* wV,
                   double* sig, int* perm, const SvdQr& s, SvdQrHost* h, int max_sweeps, int* status,
                   unsigned* sync3, double* sigma, double2* U, double2* V, cudaStream_t st);

// QR preconditioning of the bond SVD (qrcp.cu): pivoted QR of D into Y64, B = R^H into G64;
// after the Jacobi on B: V_D = P U', U_D = D V_D / sigma
// cluster size for which matrices up to m_cap x n_cap stay in shared memory (0: none)
int qrcp_smem_cluster(int m_cap, int n_cap);
// tau2: squared relative noise level of D at which the pivoted QR stops (rank-revealing);
// kmax: stop after at most kmax reflectors (the autotuner times a prefix; otherwise INT_MAX)
// cluster: CTAs per matrix (0: by the number of matrices; columns that do not fit shared memory stay in L2)
void launch_qrcp_precondition(const BondWork* work, int n_work, int cluster, int k_cap, int m_cap, double tau2,
                              int kmax, int* status, cudaStream_t st);
// after the truncation: V_D and U_D on the kept columns (lam_chi: the tables' bond dims)
void launch_qrcp_finish(const BondWork* work, int n_work, int k_cap, int m_cap, const int* lam_chi,
                        cudaStream_t st);
void launch_mix_gemm_av(const BondWork* work, int n_work, int k_cap, int m_cap, const int* lam_chi, cudaStream_t st);

// tensor-core theta + gate of the fast path (tc_theta.cu); precision: 1 TF32x3, 2 BF16x3, 3 TF32x1,
// 4 BF16 fixed-point slices. Packed operand bytes of a bond (which: 0 = A, 1 = B'), its output tile
// capacity, and the launch (pack kernels + the persistent GEMM) over one layer.
size_t tc_pack_bytes(const BondWork& W, int which, int precision);
int tc_tile_cap(const BondWork& W, int precision);
void launch_tc_theta(const Tables& T, const BondWork* work, int n_work, int tile_cap, int precision,
                     cudaStream_t st);

// batched complex GEMM on the tensor cores with an FP64-class result (tc_zgemm.cu):
// C = opA(A) opB(B), M x N, inner dimension K, per item; live dims in device memory (M, N or K = 0:
// the item is skipped and C left untouched). TA / TB: the item's packed operands, sized by
// zgemm_pack_bytes for its capacities (cap_m x cap_k for A, cap_n x cap_k for B).
enum : int { ZOP_N = 0, ZOP_T = 1, ZOP_C = 2 };
struct ZGemmItem {
  const double2* A;
  const double2* B;
  double2* C;
  int lda, ldb, ldc;
  int M, N, K;
  int opA, opB;            // ZOP_N as stored (column-major), ZOP_T transposed, ZOP_C conjugate transpose
  const int* bcol;         // column n of opB(B) is its stored column bcol[n] (NULL: n)
  unsigned char* TA;
  unsigned char* TB;
  int cap_m, cap_n, cap_k;
  int* flag;               // set to 1 when a product entry is not finite (NULL: not reported)
  int acc;                 // 0: C = opA(A) opB(B); -1: C = C - opA(A) opB(B)
  int skip_a;              // 1: A's slice planes and row exponents are already in TA (packed earlier)
  const double2* A2;       // rows a_split .. M - 1 of opA(A) come from A2 (same op and leading dimension); NULL: all from A
  int a_split;
  long long split;         // > 0: each K chunk's product goes to C + chunk * split (zgemm9_chunks of them)
  int split_ks;            // the chunks' length in steps of 16 of K (0: the longest)
};
struct SvdQrHost {
  std::vector<QRItem> qr;
  std::vector<QRBlk> blk;
  std::vector<ZGemmItem> mul;
};
size_t zgemm_pack_bytes(int rows_cap, int k_cap, int which);
// the A operands' slice planes and row exponents alone (for items whose later products skip them)
void launch_zgemm_pack_a(const ZGemmItem* items, int n_items, int m_cap_max, int* status, cudaStream_t st);
int zgemm_tile_cap(int m_cap, int n_cap);
// tile_cap: total output tiles of the item list at capacity (the persistent grid's upper bound);
// m_cap_max / n_cap_max: the largest M and N capacities (pack grid sizes); k_cap_max: the largest K capacity where it
// is at most 64 (the preparation then takes more rows per block)
void launch_zgemm(const ZGemmItem* items, int n_items, int tile_cap, int m_cap_max, int n_cap_max, int* status,
                  cudaStream_t st, int k_cap_max = 1 << 30);
// the same product from nine slices, for uses that need an FP64 product's accuracy (2^-60 of max|row| max|column| per
// term, one FP64 rounding per 256-long chunk of K, the chunks added in FP64). Its operands' packed sizes, the
// number of K chunks; unit_cap: output tiles (128 x 32), times the chunks where items are split
size_t zgemm9_pack_bytes(int rows_cap, int k_cap, int which);
constexpr int Z9_KSTEPS = 16;   // the longest chunk, in steps of 16 of K
inline int zgemm9_chunks(int k) { return ((k < 1 ? 1 : k) + 16 * Z9_KSTEPS - 1) / (16 * Z9_KSTEPS); }
void launch_zgemm9(const ZGemmItem* items, int n_items, long long unit_cap, int m_cap_max, int n_cap_max, int k_cap_max,
                   int* status, cudaStream_t st);
// the most items one launch_zgemm takes
int zgemm_max_items();

// the fast path's PT site contraction on the tensor cores (tc_contract.cu): items[w] is site w's GEMM
// (output scratch C, packed planes TA / TB and their capacities set at init; a plan kernel writes the
// operands and live dims every step, so the launch sequence is graph-safe); writes Gamma' into the
// sites' second buffers, to be swapped in by k_site_swap
void launch_site_tc(const Tables& T, const SiteWork* work, int n_work, ZGemmItem* items, int gx, int tile_cap,
                    int m_cap_max, int n_cap_max, cudaStream_t st);
// the fast path's Gamma recovery on the tensor cores (tc_contract.cu): items[2w], items[2w + 1] are
// bond w's left and right products (C in the bond's Householder scratch HH and HH + mL_cap nL_cap,
// packed planes and caps set at init), bcols[w] its column maps (nL_cap + mR_cap ints)
void launch_recover_tc(const Tables& T, const BondWork* work, int n_work, ZGemmItem* items, int* const* bcols,
                       int gx, int tile_cap, int m_cap_max, int n_cap_max, cudaStream_t st);

// the fast path's randomized truncated SVD of every bond of a layer (rsvd.cu): device item lists
// (one entry per bond each) and their launch capacities
struct RsvdLists {
  ZGemmItem *gy1, *gz1, *gy2, *gz2, *gres, *gu, *gv;
  QRItem *q1, *qz, *q2, *qb;
  double* fro_part;        // RSVD_FRO_PARTS doubles per bond: partial sums of the tail norm
  int tile_cap;            // output tiles of one product over the layer at capacity
  int m_cap, l_cap;        // largest row count and range-finder width of the layer's bonds
};
constexpr int RSVD_OVERSAMPLE = 32;
// power iterations: the subspace error at the cut chi falls like (s_{l+1} / s_chi)^(2q+1)
constexpr int RSVD_POWER = 2;
void launch_rsvd_omega(double2* Om, int rows, int cols, unsigned seed, cudaStream_t st);
// the order of a layer: plan (item lists, l into info[9]); gy1 -> QR q1; RSVD_POWER times
// (gz1 -> QR qz, gy2 -> QR q2); gz2; gres (D - Q Z^H); tail norm; QR qb (l x l factor into G64);
// Jacobi on its R^H (launch_jacobi_grid, on_b = 2); truncation (k_truncate, rsvd = 1); vectors
void launch_rsvd_plan(const Tables& T, const BondWork* work, int n_work, const RsvdLists& L, int chi_max, int p,
                      const double2* Om, int ld_om, cudaStream_t st);
// part: RSVD_FRO_PARTS doubles per bond (scratch of the two-pass, fixed-order sum)
constexpr int RSVD_FRO_PARTS = 64;
void launch_rsvd_tail_norm(const BondWork* work, int n_work, double* part, cudaStream_t st);
// R Wr / S of the kept columns (R in G64, Wr in V, columns by perm) into RH, l x chi: Ur of R = Ur S Wr^H
void launch_rsvd_left(const BondWork* work, int n_work, int l_cap, const int* lam_chi, cudaStream_t st);
void launch_rsvd_vectors(const Tables& T, const BondWork* work, int n_work, const RsvdLists& L, cudaStream_t st);

// set the message returned by pt_tebd_last_error(NULL) (engine.cu)
void set_global_error(const char* msg);

// readout (readout.cu): Tr(O_j rho) of every site and operator and the trace of every chain at the current
// step; Mbuf holds 5 planes [chi_l][chi_r] per site at moff, Lbuf / Rbuf n_max + 1 vectors of ld per chain
void launch_observe(const Tables& T, int n_chains, int n_max, int gx_m, const double2* ops, int n_ops, double2* obs,
                    double2* trace, double2* Lbuf, double2* Rbuf, int ld, int use_history, double2* Mbuf,
                    const size_t* moff, cudaStream_t st);

// local super-operator launch (struct passed by value lives in the kernel TU)
void launch_apply_local(const Tables& T, int site, int lam, const double2* s16, cudaStream_t st);

}  // namespace ptk
