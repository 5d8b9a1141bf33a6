// Kernel launchers shared between the .cu translation units of libfsi.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "fsi_internal.h"

namespace fsi {

// Lets launches of a kernel take dynamic shared memory up to what an SM has for
// one thread block (227 KB less the kernel's static arrays).  The limit belongs to the
// kernel, not to the launch: were it set to each launch's own amount, another host
// thread's smaller launch could lower it between this one's setting and its launch.
template <typename K>
inline bool allow_dynamic_smem(K kern) {
  cudaFuncAttributes a;
  return cudaFuncGetAttributes(&a, kern) == cudaSuccess &&
         cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              227 * 1024 - (int)a.sharedSizeBytes) == cudaSuccess;
}

struct PhysParams {
  double rho_f, mu_f, rho_s, mu_s;
  int ale_op;
  double mr_c2;         // Mooney-Rivlin C2 (0: Neo-Hookean); 2 C1 = mu_s - 2 C2
  // transient (BDF) terms: q_t = (a0 q + yold) * idt with yold = a1 q_n + a2 q_{n-1}
  int transient;
  double a0, idt;
  const double* yold;   // internal layout, finest level (nullptr when steady)
};

// bounds-check build (-DFSI_BOUNDS_CHECK): the first failed index check of
// each translation unit's kernels since the last call (FSI_SITE code: unit *
// 100000 + line; 0: none), cleared by the read; always 0 in the normal build
int bounds_site_schwarz();
int bounds_site_linalg();
int bounds_site_coarse();
int bounds_site_slab();

// k_assemble.cu
// scratch: 3D only, assemble_3d_scratch_doubles(scratch_ne) doubles (2D: unused); false (nothing
// launched) when one pass of ne elements needs more scratch than that
bool launch_assemble_2d(bool solid, const int32_t* elems, int ne, const double* y, const int32_t* elem_nodes,
                        const uint8_t* node_class, const double* elem_geo, int64_t n_nodes, PhysParams pp,
                        double* Ke, double* Re, int32_t* status, double* scratch, int scratch_ne, cudaStream_t st);
bool launch_assemble_3d(bool solid, const int32_t* elems, int ne, const double* y, const int32_t* elem_nodes,
                        const uint8_t* node_class, const double* elem_geo, int64_t n_nodes, PhysParams pp,
                        double* Ke, double* Re, int32_t* status, double* scratch, int scratch_ne, cudaStream_t st);
size_t assemble_3d_scratch_doubles(int max_ne);
int assemble_launches(int dim, int ne);   // kernel launches of one launch_assemble_* call
double assemble_flops_per_element(int dim, bool solid, int mode);   // executed FP64 flops (ncu count)
double galerkin_flops_per_coarse_element(int dim);
void launch_galerkin_3d(int ncx, int ncy, int ncz, const double* Kf, const int32_t* f_nodes, const uint8_t* f_class,
                        const uint8_t* f_dir, const int32_t* c_nodes, const uint8_t* c_class, const uint8_t* c_dir,
                        double* Kc, cudaStream_t st);
// element matrices -> block values (every entry written) and, with res set,
// element residuals -> residual, summed in the order of the gather lists
void launch_gather_elements(int dim, int64_t nnzb, const int32_t* blk_ptr, const int32_t* blk_src, const double* Ke,
                            double* val, int64_t nb, const int32_t* res_ptr, const int32_t* res_src,
                            const double* Re, double* res, cudaStream_t st);
void launch_dirichlet(const int32_t* dir_list, int64_t n_dir, const int32_t* rowptr, const int32_t* col, double* val,
                      int B, const double* y, const double* g, double alpha, double* res, cudaStream_t st);
void launch_galerkin_2d(int ncx, int ncy, const double* Kf, const int32_t* f_nodes, const uint8_t* f_class,
                        const uint8_t* f_dir, const int32_t* c_nodes, const uint8_t* c_class, const uint8_t* c_dir,
                        double* Kc, cudaStream_t st);

// k_linalg.cu
void launch_bsr_residual(int B, int64_t nb, const int32_t* rowptr, const int32_t* col, const double* val,
                         const double* x, const double* b, double* y, cudaStream_t st);
void launch_bsr_residual_f32(int B, int64_t nb, const int32_t* rowptr, const int32_t* col, const float* val,
                             const float* x, const float* b, float* y, int sub, cudaStream_t st);
void launch_csr_spmv(int64_t nrows, const int32_t* ptr, const int32_t* col, const double* val, const double* x,
                     double* y, bool add, cudaStream_t st);
void launch_gather(int64_t n, const int32_t* map, const double* in, double* out, cudaStream_t st);
void launch_axpby(int64_t n, double a, const double* x, double b, double* y, cudaStream_t st);
void launch_scale_by(int64_t n, const double* src, const double* dev_scalar, double* dst, cudaStream_t st);
void launch_reduce(const double* partial, int nvec, int nblk, double* out, bool sqrt_out, cudaStream_t st);
// fused Arnoldi passes (nvec <= 72; partial holds (nvec + 1) * nblk doubles)
void launch_arnoldi_dots(int64_t n, const double* V, int64_t ldv, int nvec, const double* w, bool with_norm,
                         double* partial, int nblk, cudaStream_t st);
void launch_arnoldi_update_norm(int64_t n, const double* V, int64_t ldv, int nvec, const double* h, double* w,
                                double* partial, int nblk, cudaStream_t st);
// one Arnoldi step in one cooperative launch (nvec <= 32; false: not launched); partial holds
// 3 (nvec + 1) max_blocks doubles
bool launch_arnoldi_step(int64_t n, const double* V, int64_t ldv, int nvec, int passes, double* w, double* vnext,
                         double* partial, int max_blocks, double* out, cudaStream_t st);
void launch_cgs_update(int64_t n, const double* V, int64_t ldv, int nvec, const double* h, double* w, cudaStream_t st);
void launch_combo(int64_t n, const double* Z, int64_t ldz, int nvec, const double* coef, double* x, cudaStream_t st);
void launch_norm_partial(int64_t n, const double* w, double* partial, int nblk, cudaStream_t st);
void launch_nonfinite_check(int64_t n, const double* v, int32_t* status, cudaStream_t st);

// k_schwarz.cu (T = double: FP64 path, T = float: mixed path)
// Schwarz blocks of one level for the tensor-core factorisation; several
// levels can share one launch (blocks first .. first + n_patches - 1)
constexpr int kGjMaxLevels = 24;   // levels of one launch (several instances may share it)
template <typename T>
struct GjLevelT {
  const int32_t* p_n;
  const int32_t* p_nown;
  const int64_t* dense_off;
  const int64_t* own_off;
  const int32_t* own;
  const int64_t* inv_off;
  T* dense;
  T* invT;
  int32_t* status;   // status flags of the instance the level belongs to
  const int32_t* sel; // blocks of the level to factor (nullptr: all of them)
  int first;
};
template <typename T>
struct GjLevelsT {
  int nlev;
  // iteration limit of the first bounded wait of each block on its tensor-core
  // work (the drain waits before tensor memory is released keep their full limit)
  long long first_wait;
  GjLevelT<T> l[kGjMaxLevels];
};
using GjLevel = GjLevelT<float>;
using GjLevels = GjLevelsT<float>;
constexpr long long kTcWaitIters = 1LL << 22;
// Gauss-Jordan variant code: 16-column panels on 64-column tiles with 256
// tensor-memory columns, so that two blocks share an SM (blocks <= 512 unknowns)
constexpr int kGjPanelPair = 216;
// false when the blocks do not fit the tensor-core kernel (the caller then
// factors level by level)
// panel: preferred panel width (16 or 32; 0 = 32 when the blocks fit, else 16)
bool launch_patch_gj_tc_levels(const GjLevels& lv, int nblocks, int max_n, int32_t* status, cudaStream_t st,
                               int panel = 0);
// panel width of the tensor-core variant that launch_patch_gj_tc_levels picks
// for blocks up to max_n with preference `panel` (0: none fits)
int gj_tc_variant(int max_n, int panel);
// the gathers of the Schwarz levels of one instance in one launch
template <typename T>
struct GatherLevelT {
  const int32_t* p_n;
  const int64_t* dense_off;
  const int64_t* gmap_off;
  const int32_t* gmap;
  const int64_t* boff_off;
  const int32_t* boff;   // per local block its dense offset * 8 + width
  const int64_t* pad_off;
  const int32_t* padpos;
  const double* bsr_val;
  T* dense;
  const int64_t* idx_off;
  T* dr;
  T* dc;
  int first;   // first thread block of the level
};
template <typename T>
struct GatherLevelsT {
  int nlev, B;
  GatherLevelT<T> l[kGjMaxLevels];
};
template <typename T>
void launch_patch_gather_levels(const GatherLevelsT<T>& lv, int nblocks, cudaStream_t st);
// FP64 blocks of the levels in one launch; false when they fit no shared-memory
// variant (the caller then factors level by level)
bool launch_patch_gj_levels_f64(const GjLevelsT<double>& lv, int nblocks, int max_n, cudaStream_t st);
template <typename T>
void launch_patch_gj_t(int np, int max_n, const int32_t* p_n, const int32_t* p_nown, const int64_t* dense_off,
                       const int64_t* own_off, const int32_t* own, const int64_t* inv_off, T* dense, T* invT,
                       int32_t* status, bool n_mult4, cudaStream_t st);
// sel: the np blocks to apply (nullptr: blocks 0 .. np - 1); nv: length of r and x
template <typename T>
void launch_patch_apply_t(int np, int64_t nv, int max_n, int max_nown, const int32_t* p_n, const int32_t* p_nown,
                          const int64_t* idx_off, const int32_t* idx, const int64_t* own_off, const int32_t* own,
                          const int64_t* inv_off, const T* invT, const T* r, T* x, double omega, const T* dr,
                          const T* dc, int sm_count, int want_slices, int want_groups, cudaStream_t st,
                          const int32_t* sel = nullptr);
// ILU(0) of the fluid Schwarz blocks listed in sel (Sec. 3.3, 4.1), in place
// on their gathered, equilibrated dense blocks; blocks of at most
// kIluMaxRows unknowns
constexpr int kIluMaxRows = 1024;
void launch_patch_ilu0(int nsel, const int32_t* sel, const int32_t* p_n, const int64_t* dense_off,
                       const int64_t* gmap_off, const int32_t* gmap, const int64_t* boff_off, const int32_t* boff,
                       int B, float* dense, int32_t* status, cudaStream_t st);
// x[own] += omega (R^0)^T U^{-1} L^{-1} R^delta r for the ILU(0) blocks in sel (at most max_n
// unknowns and max_nb node / element blocks each)
void launch_patch_apply_ilu(int nsel, int max_n, int max_nb, const int32_t* sel, const int32_t* p_n,
                            const int32_t* p_nown,
                            const int64_t* idx_off, const int32_t* idx, const int64_t* own_off, const int32_t* own,
                            const int64_t* dense_off, const int64_t* gmap_off, const int32_t* gmap,
                            const int64_t* boff_off, const int32_t* boff, const int32_t* gptr, int B,
                            const float* dense, const float* r, float* x, double omega, const float* dr,
                            const float* dc, cudaStream_t st);
// Launch shape of one level's Schwarz apply: kind 0 = one block per patch
// (k_patch_apply_t), kind 1 = `slices` row slices per patch of `vps` owned-row
// vectors, `groups` column groups per block (k_patch_apply_rows).
// want_slices 0 / want_groups 0 = the built-in rule; want_slices 1 = kind 0.
struct ApplyShape { int kind, slices, vps, groups; };
ApplyShape apply_shape(int np, int max_nown, int vec_width, int sm_count, int want_slices, int want_groups);

void launch_dense_gather(int B, int64_t nb, const int32_t* rowptr, const int32_t* col, const double* val,
                         const int32_t* pad_list, int npad, const int32_t* perm, int64_t n, double* dr, double* A,
                         cudaStream_t st);
int launch_coarse_lu_inverse(int64_t n, int kl, int ku, double* M, double* rdiag, double* Ainv, int32_t* piv,
                             const int32_t* perm, const int32_t* pinv, int32_t* status, int sm_count,
                             cudaStream_t st);
// k_coarse.cu: explicit inverse of the block-tridiagonal 2D coarse operator by
// merging the inverses of its slab ranges.  off: leaves; merge i joins [a, m)
// and [m, b), s = size of the first leaf right of m; level[l] .. level[l + 1]
// are the merges of one level
constexpr int kMaxLeaves = FSI_MAX_BREAKS + 1;
struct CoarseMerge { int a, m, b, s; };
struct CoarseTree {
  int nleaf, nlev;
  int off[kMaxLeaves + 1];
  CoarseMerge merge[kMaxLeaves];
  int level[9];
};
bool coarse_merge_fits(int max_leaf, int p, int max_s);
// A: the dense operator in the banded ordering (overwritten); Lbuf, Bbuf: n p
// doubles each; gh: 2 p p doubles per merge of the widest level.  0 or an
// error; a breakdown raises ST_COARSE_RETRY
int launch_coarse_merge(const CoarseTree& tr, int64_t n, int p, int max_leaf, int max_s, double* A, double* Lbuf,
                        double* Bbuf, double* gh, double* Ainv, int32_t* status, int sm_count, cudaStream_t st);
// test vector on the unknowns with pos >= 0, zero elsewhere
void launch_coarse_probe(int64_t ni, const int32_t* pos, double* v, cudaStream_t st);
void launch_coarse_check(int B, int64_t nb, const int32_t* rowptr, const int32_t* col, const double* val,
                         const double* v, const double* x, double tol, const int32_t* pos, int32_t* status,
                         cudaStream_t st);

// k_slab.cu: 3D coarse factorisation and solve from both ends of the slab chain
struct SlabJob {
  const double* S;   // m x m, column-major
  double* T;         // slab_gj_scratch(m) doubles
  double* X;         // its inverse
  int m;
  int32_t* piv;      // m
  double* rd;        // m
  int* flag;         // slab_gj_panels(m); never equal to a coming epoch
};
struct SlabJobs { int n; SlabJob j[2]; };
struct SlabGemm {
  int m, n, k;
  double alpha, beta;
  const double* A;
  int64_t lda;
  const double* B;
  int64_t ldb;
  double* C;
  int64_t ldc;
};
struct SlabGemms { int tiles0; SlabGemm g[2]; };
struct SlabChain {
  int K, mid, p, mmax;
  int off[FSI_MAX_BREAKS];        // slab k = positions off[k] .. off[k + 1] - 1
  int64_t inv[FSI_MAX_BREAKS];    // its inverse's offset
};
size_t slab_gj_scratch(int m);
int slab_gj_panels(int m);
bool slab_gj_fits(int m, int sm_count);
// inverses of up to two slab complements at once; epoch: another one on every call with the same flags.
// wait: iteration limit of a wait for a panel.  A zero pivot raises ST_COARSE_RETRY, a wait that ran out
// ST_SLAB_TIMEOUT
constexpr long long kSlabWaitIters = 1LL << 21;
int launch_slab_gj(const SlabJobs& jobs, int epoch, long long wait, int32_t* status, int sm_count, cudaStream_t st);
void launch_slab_gemm(const SlabGemm* g, int n, cudaStream_t st);   // n <= 2 products
// x = A^{-1} w (w is overwritten); u: 2 mmax doubles
int launch_slab_solve(const SlabChain& ch, const double* A, int64_t n, const double* sinv, double* w, double* x,
                      double* u, int sm_count, cudaStream_t st);

// coarse apply over an ordering of n of the ni unknowns (the others are
// identity rows), dr its row scales: part holds ceil(n / 32) * n doubles of scratch
template <typename TX, typename TY>
void launch_gemv(int64_t ni, int64_t n, const double* A, const int32_t* pos, const int32_t* map, const double* dr,
                 const TX* x, TY* y, double* part, cudaStream_t st);
// b less the columns of the unknowns that the ordering leaves out
template <typename TX>
void launch_coarse_rhs(int B, int64_t nb, const int32_t* rowptr, const int32_t* col, const double* val,
                       const int32_t* pos, const TX* b, double* out, cudaStream_t st);
template <typename TB>
void launch_coarse_pick(int64_t ni, int64_t n, const int32_t* map, const double* dr, const TB* b, double* out,
                        cudaStream_t st);
template <typename TB, typename TY>
void launch_coarse_scatter(int64_t ni, const int32_t* pos, const double* x, const TB* b, TY* y, cudaStream_t st);
// slab-blocked coarse solve: column-major FP64 sub-matrices with leading dimensions
void launch_dgemm_nn(int m, int n, int k, double alpha, const double* A, int64_t lda, const double* Bm, int64_t ldb,
                     double beta, double* C, int64_t ldc, cudaStream_t st);
void launch_copy2d(int m, int n, const double* src, int64_t lds, double* dst, int64_t ldd, cudaStream_t st);
// y = beta y + alpha A x; part holds ceil(nc / 32) * m doubles of scratch
void launch_gemv_sub(int m, int nc, double alpha, const double* A, int64_t lda, const double* x, double beta,
                     double* y, double* part, cudaStream_t st);
void launch_csr_spmv_f32(int64_t nrows, const int32_t* ptr, const int32_t* col, const float* val, const float* x,
                         float* y, bool add, cudaStream_t st);
void launch_to_f32(int64_t n, const double* in, float* out, cudaStream_t st);
void launch_to_f64(int64_t n, const float* in, double* out, cudaStream_t st);
void launch_combo_mixed(int64_t n, const float* Z, int64_t ldz, int nvec, const double* coef, double* x,
                        cudaStream_t st);

}  // namespace fsi
