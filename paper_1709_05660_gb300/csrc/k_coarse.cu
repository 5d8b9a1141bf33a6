// Coarse level in 2D: the explicit inverse of the block-tridiagonal coarse
// operator by merging halves (Sec. 3, 4.1: direct solve of the coarsest grid).
//
// In the banded (x-slab) ordering the operator couples neighbouring slabs
// through one node plane only: with P the last plane of the left part and S
// the first slab of the right part, a range of slabs reads
//     A = [ A1        E_P B ]      B: P x S,  C: S x P.
//         [ C E_P^T   A2    ]
// With X1 = A1^{-1}, X2 = A2^{-1}, the block elimination of A2 changes A1 by
// the rank-p term E_P G E_P^T, G = B X2[S,S] C, and the Woodbury formula gives
// the inverse as a rank-p correction of diag(X1, X2):
//     T     = (I - G X1[P,P])^{-1}
//     U_top = T [ G X1[P,:] | -B X2[S,:] ]
//     U_bot = -[ X1[P,:] | 0 ] - X1[P,P] U_top
//     A^{-1} = diag(X1, X2) + [ X1[:,P] U_top ; X2[:,S] C U_bot ].
// The leaves (one slab each) are inverted by Gauss-Jordan with
// partial pivoting, one thread block per leaf, and the parts are merged in
// log2(slabs) levels, all merges of a level together.
//
// Over the free unknowns of the 16 x 4 grid (1,074; slabs of 68, planes of 28)
// it takes 0.70 ms on GB300 where the banded LU and its triangular solves over
// all 1,444 (2 n dependent column steps) took 6.2.  Its dependent chain is
// n / 16 + 4 p pivot steps and four grid barriers a level; the rank-p updates
// alone need 0.1 ms of the FP64 pipe (two fused multiply-adds per SM and cycle).
#include <cooperative_groups.h>

#include <algorithm>

#include "bounds.cuh"
#include "fp64_util.cuh"
#include "gj_smem.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace fsi {

namespace {
constexpr int kMergeThreads = 512;
}  // namespace

// One cooperative launch: the leaves, then the merge levels.  Per level
//  1. Y = X2[:,S] C and copies of X1[:,P] and B (the update below overwrites
//     them) over all thread blocks;   2. G = B Y[S,:];
//  3. H = I - G X1[P,P];
//  4. tasks of at most kMergeCols columns of a merge: H inverted in shared
//     memory (by every task: cheaper than one block inverting for all and a
//     further barrier), the task's columns of U, and the rank-p update of its
//     columns of the merged range, one row per lane and one accumulator per
//     column.  The last level writes the inverse.
// X lives in the diagonal blocks of the dense operator itself; the coupling
// blocks B, C are outside them until their merge.
template <int kMergeCols>
__global__ void __launch_bounds__(kMergeThreads) k_coarse_merge(CoarseTree tr, int64_t n, int p,
                                                                double* __restrict__ A, double* __restrict__ Lbuf,
                                                                double* __restrict__ Bbuf, double* __restrict__ gh,
                                                                double* __restrict__ Ainv,
                                                                int32_t* __restrict__ status) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ GjStep step;
  const int lane = threadIdx.x % kWarp, wid = threadIdx.x / kWarp, nw = blockDim.x / kWarp;
  double* M = reinterpret_cast<double*>(smem_raw);
  for (int leaf = blockIdx.x; leaf < tr.nleaf; leaf += gridDim.x) {
    const int64_t o = tr.off[leaf];
    const int m = (int)(tr.off[leaf + 1] - o);
    double* f = M + (size_t)m * m;
    double* rd = f + 2 * m;
    int* piv = reinterpret_cast<int*>(rd + m);
    int* qinv = piv + m;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) M[e] = A[(o + e / m) * n + o + e % m];
    if (!gj_inverse_smem(M, m, m, f, rd, piv, qinv, step, nullptr) && threadIdx.x == 0)
      atomicExch(&status[ST_COARSE_RETRY], 1);
    double* out = tr.nlev > 0 ? A : Ainv;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int c = e / m, r = e % m;
      if (FSI_IN(piv[r], m, FSI_SITE(3)) && FSI_IN(qinv[c], m, FSI_SITE(3)))
        out[(o + c) * n + o + r] = rd[piv[r]] * M[piv[r] + qinv[c] * m];
    }
    __syncthreads();
  }
  for (int lv = 0; lv < tr.nlev; ++lv) {
    const int i0 = tr.level[lv], i1 = tr.level[lv + 1];
    const bool last = lv + 1 == tr.nlev;
    grid.sync();
    // left factors.  Copies: row r (column c) of the level's merge that holds it
    auto merge_of = [&](int r) {
      int i = i0;
      while (i < i1 && r >= tr.merge[i].b) ++i;
      return i < i1 && r >= tr.merge[i].a ? i : -1;
    };
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * p; e += (int64_t)gridDim.x * blockDim.x) {
      const int r = (int)(e % n), q = (int)(e / n), i = merge_of(r);
      if (i >= 0 && r < tr.merge[i].m) Lbuf[e] = A[(int64_t)(tr.merge[i].m - p + q) * n + r];
      const int c = (int)(e / p), k = (int)(e % p), ic = merge_of(c);
      if (ic >= 0 && c >= tr.merge[ic].m && c < tr.merge[ic].m + tr.merge[ic].s)
        Bbuf[e] = A[(int64_t)c * n + tr.merge[ic].m - p + k];
    }
    // Y: tasks of 8 rows (so that the last level's half occupies most SMs), operands staged in shared memory
    int first = 0;
    for (int i = i0; i < i1; ++i) {
      const CoarseMerge g = tr.merge[i];
      const int ntask = (g.b - g.m + 7) / 8;
      int t = (int)blockIdx.x - first % (int)gridDim.x;
      if (t < 0) t += gridDim.x;
      first += ntask;
      for (; t < ntask; t += gridDim.x) {
        double* Cs = M;                         // s x p by column
        double* Xs = Cs + (size_t)g.s * p;      // 8 x s by column
        const int r0 = g.m + t * 8, nr = min(8, g.b - r0);
        for (int e = threadIdx.x; e < g.s * p; e += blockDim.x)
          Cs[e] = A[(int64_t)(g.m - p + e / g.s) * n + g.m + e % g.s];
        for (int e = threadIdx.x; e < g.s * 8; e += blockDim.x)
          Xs[e] = e % 8 < nr ? A[(int64_t)(g.m + e / 8) * n + r0 + e % 8] : 0.0;
        __syncthreads();
        for (int e = threadIdx.x; e < 8 * p; e += blockDim.x) {
          const int r = e % 8, q = e / 8;
          double a0 = 0.0, a1 = 0.0;
          int k = 0;
          for (; k + 1 < g.s; k += 2) {
            a0 = fma(Xs[k * 8 + r], Cs[q * g.s + k], a0);
            a1 = fma(Xs[k * 8 + 8 + r], Cs[q * g.s + k + 1], a1);
          }
          if (k < g.s) a0 = fma(Xs[k * 8 + r], Cs[q * g.s + k], a0);
          if (r < nr) Lbuf[(int64_t)q * n + r0 + r] = a0 + a1;
        }
        __syncthreads();
      }
    }
    grid.sync();
    // G = B Y[S,:] (first p x p matrix of a merge's scratch), one entry per thread
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < (i1 - i0) * p * p; t += gridDim.x * blockDim.x) {
      const CoarseMerge g = tr.merge[i0 + t / (p * p)];
      const int q = t % p, c = (t / p) % p;
      double acc = 0.0;
#pragma unroll 8
      for (int k = 0; k < g.s; ++k)
        acc = fma(Bbuf[(int64_t)(g.m + k) * p + q], Lbuf[(int64_t)c * n + g.m + k], acc);
      gh[(int64_t)(t / (p * p)) * 2 * p * p + c * p + q] = acc;
    }
    grid.sync();
    // H = I - G X1[P,P] (second matrix)
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < (i1 - i0) * p * p; t += gridDim.x * blockDim.x) {
      const CoarseMerge g = tr.merge[i0 + t / (p * p)];
      const double* G = gh + (int64_t)(t / (p * p)) * 2 * p * p;
      const int q = t % p, c = (t / p) % p;
      double acc = q == c ? 1.0 : 0.0;
#pragma unroll 4
      for (int k = 0; k < p; ++k) acc = fma(-G[k * p + q], Lbuf[(int64_t)c * n + g.m - p + k], acc);
      gh[(int64_t)(t / (p * p)) * 2 * p * p + p * p + c * p + q] = acc;
    }
    grid.sync();
    first = 0;
    for (int i = i0; i < i1; ++i) {
      const CoarseMerge g = tr.merge[i];
      const int ntask = (g.b - g.a + kMergeCols - 1) / kMergeCols;
      const double* G = gh + (int64_t)(i - i0) * 2 * p * p;
      int t = (int)blockIdx.x - first % (int)gridDim.x;   // this level's tasks in turn over the thread blocks
      if (t < 0) t += gridDim.x;
      first += ntask;
      for (; t < ntask; t += gridDim.x) {
        const int c0 = g.a + t * kMergeCols, nc = min(kMergeCols, g.b - c0), w = max(p, g.s);
        double* H = M;                          // p x p, inverted in place
        double* f = H + (size_t)p * p;          // 2 p, and the p reciprocal pivots
        double* rd = f + 2 * p;
        double* V = rd + p;                     // w x nc: X1[P, cols] or X2[S, cols] (by column)
        double* R = V + (size_t)w * kMergeCols; // p x nc: [G X1[P,:] | -B X2[S,:]]
        double* Ut = R + (size_t)p * kMergeCols;   // by row: kMergeCols entries
        double* Ub = Ut + (size_t)p * kMergeCols;
        int* piv = reinterpret_cast<int*>(Ub + (size_t)p * kMergeCols);
        int* qinv = piv + p;
        for (int e = threadIdx.x; e < p * p; e += blockDim.x) H[e] = G[p * p + e];
        for (int e = threadIdx.x; e < w * nc; e += blockDim.x) {
          const int j = e / w, k = e % w, c = c0 + j;
          const int r = c < g.m ? g.m - p + k : g.m + k;
          if (k < (c < g.m ? p : g.s)) V[j * w + k] = A[(int64_t)c * n + r];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < p * nc; e += blockDim.x) {
          const int j = e / p, q = e % p;
          const bool left = c0 + j < g.m;
          const double* K = left ? G + q : Bbuf + (int64_t)g.m * p + q;   // row q of G or B
          const int len = left ? p : g.s;
          double acc = 0.0;
#pragma unroll 8
          for (int k = 0; k < len; ++k) acc = fma(K[k * p], V[j * w + k], acc);
          R[j * p + q] = left ? acc : -acc;
        }
        if (!gj_inverse_smem(H, p, p, f, rd, piv, qinv, step, nullptr) && threadIdx.x == 0)
          atomicExch(&status[ST_COARSE_RETRY], 1);
        for (int e = threadIdx.x; e < p * kMergeCols; e += blockDim.x) {
          const int j = e / p, q = e % p;
          double acc = 0.0;
          if (j < nc)
            for (int k = 0; k < p; ++k)
              if (FSI_IN(piv[q], p, FSI_SITE(3)) && FSI_IN(qinv[k], p, FSI_SITE(3)))
                acc = fma(H[piv[q] + qinv[k] * p], R[j * p + k], acc);
          Ut[q * kMergeCols + j] = acc * rd[piv[q]];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < p * kMergeCols; e += blockDim.x) {
          const int j = e / p, q = e % p;
          double acc = 0.0;
          if (j < nc) {
            if (c0 + j < g.m) acc = -V[j * w + q];
            for (int k = 0; k < p; ++k)
              acc = fma(-Lbuf[(int64_t)k * n + g.m - p + q], Ut[k * kMergeCols + j], acc);
          }
          Ub[q * kMergeCols + j] = acc;
        }
        __syncthreads();
        // rank-p update of the task's columns: lane = row
        for (int r0 = g.a + wid * kWarp; r0 < g.b; r0 += nw * kWarp) {
          const int r = r0 + lane;
          const bool ok = r < g.b;
          // a warp whose rows lie on both sides of m takes the factor per lane
          const bool top = r < g.m;
          const bool mixed = r0 < g.m && r0 + kWarp > g.m;
          double acc[kMergeCols];
#pragma unroll
          for (int j = 0; j < kMergeCols; ++j) {
            const int c = c0 + j;
            acc[j] = (ok && j < nc && (c < g.m) == top) ? A[(int64_t)c * n + r] : 0.0;
          }
          const double* Lr = Lbuf + (ok ? r : g.a);
          const double* U = (mixed ? top : r0 < g.m) ? Ut : Ub;
#pragma unroll 4
          for (int q = 0; q < p; ++q) {
            const double l = Lr[(int64_t)q * n];
            const double2* u2 = reinterpret_cast<const double2*>(U + q * kMergeCols);
#pragma unroll
            for (int j = 0; j < kMergeCols / 2; ++j) {
              const double2 u = u2[j];
              acc[2 * j] = fma(l, u.x, acc[2 * j]);
              acc[2 * j + 1] = fma(l, u.y, acc[2 * j + 1]);
            }
          }
          if (ok) {
            double* out = last ? Ainv : A;
#pragma unroll
            for (int j = 0; j < kMergeCols; ++j)
              if (j < nc) out[(int64_t)(c0 + j) * n + r] = acc[j];
          }
        }
        __syncthreads();
      }
    }
  }
}

namespace {
constexpr int kMaxMergeCols = 16;

size_t merge_smem(int max_leaf, int p, int max_s, int cols) {
  const size_t leaf = ((size_t)max_leaf * max_leaf + 3 * max_leaf) * sizeof(double) + 2 * (size_t)max_leaf * sizeof(int);
  const size_t task = ((size_t)p * p + 3 * p + (size_t)std::max(p, max_s) * cols + 3 * (size_t)p * cols) *
                          sizeof(double) + 2 * (size_t)p * sizeof(int);
  const size_t left = ((size_t)max_s * p + 8 * (size_t)max_s) * sizeof(double);
  return std::max(std::max(leaf, left), task);
}

template <int COLS>
int run_merge(const CoarseTree& tr, int64_t n, int p, size_t smem, double* A, double* Lbuf, double* Bbuf, double* gh,
              double* Ainv, int32_t* status, int sm_count, cudaStream_t st) {
  const auto kern = k_coarse_merge<COLS>;
  if (!allow_dynamic_smem(kern)) return -1;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMergeThreads, smem);
  if (per_sm < 1) return -1;
  CoarseTree t = tr;
  void* args[] = {(void*)&t, (void*)&n, (void*)&p, (void*)&A, (void*)&Lbuf, (void*)&Bbuf, (void*)&gh,
                  (void*)&Ainv, (void*)&status};
  const int grid = (int)std::min<int64_t>(sm_count, std::max<int64_t>(tr.nleaf, (n + COLS - 1) / COLS));
  return cudaLaunchCooperativeKernel((const void*)kern, grid, kMergeThreads, args, smem, st) == cudaSuccess ? 0 : -2;
}
}  // namespace

bool coarse_merge_fits(int max_leaf, int p, int max_s) {
  // leaves and planes as gj_inverse_smem takes them (16 x 8 cells, slabs of 144: coarse factor 3.2 ms; 16 x 9, slabs
  // of 163, by the banded LU: 27.8); 2 KB of the 227 KB are left to the static shared memory
  return max_leaf <= kGjSmemMax && p <= kGjSmemMax && p % 2 == 0 &&
         merge_smem(max_leaf, p, max_s, kMaxMergeCols) <= 225 * 1024;
}

// Columns per task: the last level's n columns as one task per SM where the
// accumulators allow it (the 16 x 4 grid's 1,074: 8).  An unused accumulator costs as
// much as a used one: over all 1,444 unknowns of that grid, before the Dirichlet ones
// were left out, the last level took 215 us with 10 columns a task and 250 with 12.
int launch_coarse_merge(const CoarseTree& tr, int64_t n, int p, int max_leaf, int max_s, double* A, double* Lbuf,
                        double* Bbuf, double* gh, double* Ainv, int32_t* status, int sm_count,
                        cudaStream_t st) {
  const int64_t want = (n + sm_count - 1) / sm_count;
  auto go = [&](auto f, int cols) {
    return f(tr, n, p, merge_smem(max_leaf, p, max_s, cols), A, Lbuf, Bbuf, gh, Ainv, status, sm_count, st);
  };
  if (want <= 4) return go(run_merge<4>, 4);
  if (want <= 6) return go(run_merge<6>, 6);
  if (want <= 8) return go(run_merge<8>, 8);
  if (want <= 10) return go(run_merge<10>, 10);
  if (want <= 12) return go(run_merge<12>, 12);
  if (want > 2 * 12 && want <= 2 * 14) return go(run_merge<14>, 14);
  return go(run_merge<16>, 16);
}

// Check of an explicit coarse inverse on one vector: x = Ainv v is compared
// row by row with v, |v - A x| <= tol (|v| + |A| |x|); a row that fails (or
// is not finite) raises ST_COARSE_RETRY.  Rows that the ordering leaves out (pos < 0) are skipped.
__global__ void k_coarse_check(int B, int64_t nb, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                               const double* __restrict__ val, const double* __restrict__ v,
                               const double* __restrict__ x, double tol, const int32_t* __restrict__ pos,
                               int32_t* __restrict__ status) {
  // eight lanes per row
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 8;
  const int sub = threadIdx.x % 8;
  const bool on = i < nb * B && pos[i] >= 0;
  double s = 0.0, a = 0.0;
  if (on) {
    const int64_t br = i / B;
    const int ci = (int)(i % B);
    for (int32_t k = rowptr[br] + sub; k < rowptr[br + 1]; k += 8)
      for (int c = 0; c < B; ++c) {
        if (!FSI_IN(col[k], nb, FSI_SITE(3))) continue;
        const double t = val[((int64_t)k * B + ci) * B + c] * x[(int64_t)col[k] * B + c];
        s += t;
        a += fabs(t);
      }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    a += __shfl_xor_sync(0xffffffffu, a, o);
  }
  if (on && sub == 0 && !(fabs(v[i] - s) <= tol * (a + fabs(v[i])))) atomicExch(&status[ST_COARSE_RETRY], 1);
}

// entries in (-1, 1), none of them zero, at the unknowns of the ordering
__global__ void k_coarse_probe(int64_t ni, const int32_t* __restrict__ pos, double* __restrict__ v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ni) return;
  const uint32_t h = (uint32_t)i * 2654435761u;
  v[i] = pos[i] >= 0 ? (double)(int32_t)(h | 1u) * (1.0 / 2147483648.0) : 0.0;
}

void launch_coarse_probe(int64_t ni, const int32_t* pos, double* v, cudaStream_t st) {
  k_coarse_probe<<<(unsigned)((ni + 255) / 256), 256, 0, st>>>(ni, pos, v);
}

void launch_coarse_check(int B, int64_t nb, const int32_t* rowptr, const int32_t* col, const double* val,
                         const double* v, const double* x, double tol, const int32_t* pos, int32_t* status,
                         cudaStream_t st) {
  const int64_t n = nb * B;
  k_coarse_check<<<(unsigned)((n * 8 + 255) / 256), 256, 0, st>>>(B, nb, rowptr, col, val, v, x, tol, pos, status);
}

FSI_BOUNDS_READER(bounds_site_coarse)

}  // namespace fsi
