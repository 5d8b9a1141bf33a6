// Slab-blocked coarse solve in 3D from both ends (Sec. 3, 4.1): the coarse
// operator is block tridiagonal over x-slabs, and slabs k - 1 and k couple
// through the last node plane P of slab k - 1 only.  Block elimination runs from
// the first slab to the middle one and from the last slab to the middle one at
// the same time,
//     left   S_k = A_kk - A_{k,k-1}[:,P] (S_{k-1}^{-1}[P,P] A_{k-1,k}[P,:]),
//     right  S_k = A_kk - E_P (A_{k,k+1}[P,:] S_{k+1}^{-1} A_{k+1,k}[:,P]) E_P^T,
// which halves the chain of dependent slab inverses; the middle slab takes both
// corrections.  The slab complements are inverted by Gauss-Jordan with
// partial pivoting, spread over half of the SMs per side (k_slab_gj), and the
// solve (k_slab_solve) is one launch.
#include <cooperative_groups.h>

#include <algorithm>

#include "bounds.cuh"
#include "fp64_util.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace fsi {

namespace {
constexpr int kSlabThreads = 512;
constexpr int kSlabRows = 2;                 // rows per thread: slabs of at most 1,024 unknowns
constexpr int kSlabW = 4;                    // panel width
constexpr int kSlabWarps = kSlabThreads / kWarp;

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
}  // namespace

// In-place Gauss-Jordan inverses of up to two m x m matrices (S, column-major),
// `ng` thread blocks each.  Panels of kSlabW columns are dealt to the blocks in
// turn and stay in shared memory.  The owner of panel k factors it and
// publishes the composite transform T_k = G - E_P of its steps (m x kSlabW) and
// its pivot rows; every block applies T_0, T_1, ... to its panels as they are
// published, the next owner to its own next panel first, so that it factors
// panel k + 1 while the others still apply T_k.  Rows stay unscaled (as in
// gj_inverse_smem).
//
// The chain of one block's panel work bounds it: per panel kSlabW pivot steps
// over m rows and the transform of the previous panel, both on one SM's FP64 pipe
// (two fused multiply-adds per cycle), and the hand-over.  Their cost per column
// is m (kSlabW + kSlabW) / 2 cycles plus (hand-over) / kSlabW, hence narrow
// panels: 4 columns.  Nine rounds of two slabs of 652
// unknowns with their products: 25.2 ms against 88 one after the other by the
// banded LU kernels.
//
// The launch is cooperative (all blocks resident), the waits are bounded: a
// block whose wait runs out raises ST_SLAB_TIMEOUT and returns, and so do those
// that wait for it.
__global__ void __launch_bounds__(kSlabThreads, 1) k_slab_gj(SlabJobs jobs, int ng, int epoch, long long wait,
                                                             int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SlabJob& J = jobs.j[blockIdx.x / ng];
  const int m = J.m, g = blockIdx.x % ng;
  const int np = (m + kSlabW - 1) / kSlabW;
  const int slots = g < np ? (np - g + ng - 1) / ng : 0;      // panels g, g + ng, ...
  const int ms = (m + 1) & ~1;
  double* T = reinterpret_cast<double*>(smem_raw);            // [2][kSlabW][ms]
  double* X = T + 2 * kSlabW * (size_t)ms;                    // [slots * kSlabW][ms]
  __shared__ double s_R[64 * kSlabW], s_prow[2][kSlabW], s_rp;
  __shared__ unsigned long long s_key[2][kSlabWarps];
  __shared__ int s_row[2][kSlabWarps], s_piv[2][kSlabW], s_abort, s_sing;
  __shared__ uint8_t s_used[kSlabThreads * kSlabRows];
  const int tid = threadIdx.x, lane = tid % kWarp, wid = tid / kWarp;
  for (int i = tid; i < m; i += kSlabThreads) s_used[i] = 0;
  if (tid == 0) { s_abort = 0; s_sing = 0; }
  for (int c = wid; c < slots * kSlabW; c += kSlabWarps) {
    const int col = ((c / kSlabW) * ng + g) * kSlabW + c % kSlabW;
    for (int i = lane; i < m; i += kWarp) X[(size_t)c * ms + i] = col < m ? J.S[(size_t)col * m + i] : 0.0;
  }
  __syncthreads();

  // T of buffer b (pivot rows s_piv[b]) on the columns [c0, c1) of the block
  auto apply = [&](int b, int c0, int c1) {
    const double* Tb = T + (size_t)b * kSlabW * ms;
    __syncthreads();
    for (int t = tid; t < (c1 - c0) * kSlabW; t += kSlabThreads)
      s_R[t] = X[(size_t)(c0 + t / kSlabW) * ms + s_piv[b][t % kSlabW]];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSlabRows; ++r) {
      const int i = tid + r * kSlabThreads;
      if (r * kSlabThreads + wid * kWarp >= m) break;
      if (i >= m) continue;
      double t[kSlabW];
#pragma unroll
      for (int w = 0; w < kSlabW; ++w) t[w] = Tb[w * ms + i];
      for (int c = c0; c < c1; ++c) {
        const double* R = s_R + (c - c0) * kSlabW;
        double x = X[(size_t)c * ms + i];
#pragma unroll
        for (int w = 0; w < kSlabW; ++w) x = fma(t[w], R[w], x);
        X[(size_t)c * ms + i] = x;
      }
    }
  };

  // Factors the panel in the columns c0 .. c0 + kSlabW of the block (wp of them
  // real): buffer b gets T and its pivot rows, the columns their final values.
  auto factor = [&](int k, int b, int c0, int wp) {
    double a[kSlabRows][kSlabW];
    bool used[kSlabRows];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSlabRows; ++r) {
      const int i = tid + r * kSlabThreads;
      used[r] = i >= m || s_used[i] != 0;
#pragma unroll
      for (int w = 0; w < kSlabW; ++w) a[r][w] = i < m ? X[(size_t)(c0 + w) * ms + i] : 0.0;
    }
    // the block's candidate of panel column w: key and row of each warp's best unused row
    auto offer = [&](int w) {
      unsigned long long best = 0ull;
      uint32_t row = 0xffffffffu;
#pragma unroll
      for (int r = 0; r < kSlabRows; ++r)
        if (!used[r]) {
          unsigned long long key = 0ull;
#pragma unroll
          for (int v = 0; v < kSlabW; ++v)
            if (v == w) key = abs_key(a[r][v]);
          if (row == 0xffffffffu || key > best) { best = key; row = tid + r * kSlabThreads; }
        }
      const bool has = row != 0xffffffffu;
      const uint32_t hi = __reduce_max_sync(0xffffffffu, has ? (uint32_t)(best >> 32) : 0u);
      const bool in = has && (uint32_t)(best >> 32) == hi;
      const uint32_t lo = __reduce_max_sync(0xffffffffu, in ? (uint32_t)best : 0u);
      const uint32_t win = __reduce_min_sync(0xffffffffu, in && (uint32_t)best == lo ? row : 0xffffffffu);
      if (lane == 0) {
        s_key[w & 1][wid] = ((unsigned long long)hi << 32) | lo;
        s_row[w & 1][wid] = (int)win;   // -1: no unused row
      }
    };
    // the best of the warps' candidates (every warp finds the same one)
    auto choose = [&](int w, unsigned long long& key) {
      const bool has = lane < kSlabWarps && s_row[w & 1][lane % kSlabWarps] >= 0;
      const unsigned long long k0 = has ? s_key[w & 1][lane % kSlabWarps] : 0ull;
      const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(k0 >> 32));
      const bool in = has && (uint32_t)(k0 >> 32) == hi;
      const uint32_t lo = __reduce_max_sync(0xffffffffu, in ? (uint32_t)k0 : 0u);
      key = ((unsigned long long)hi << 32) | lo;
      return (int)__reduce_min_sync(0xffffffffu,
                                    in && (uint32_t)k0 == lo ? (uint32_t)s_row[w & 1][lane % kSlabWarps] : 0xffffffffu);
    };
    // reciprocal pivot (thread 0) and the pivot row's values (its owner)
    auto publish = [&](int w, int pr, unsigned long long key) {
#pragma unroll
      for (int r = 0; r < kSlabRows; ++r)
        if (tid + r * kSlabThreads == pr) {
#pragma unroll
          for (int v = 0; v < kSlabW; ++v) s_prow[w & 1][v] = a[r][v];
          double pv = 1.0;
#pragma unroll
          for (int v = 0; v < kSlabW; ++v)
            if (v == w) pv = a[r][v];
          if (key == 0ull || key >= 0x7FF0000000000000ull) {
            s_sing = 1;
            pv = 1.0;
          }
          const double rp = 1.0 / pv;
          s_rp = rp;
          J.rd[pr] = rp;
          J.piv[k * kSlabW + w] = pr;
          s_piv[b][w] = pr;
          s_used[pr] = 1;
        }
    };
    offer(0);
    __syncthreads();
    unsigned long long key;
    int pr = choose(0, key);
    publish(0, pr, key);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kSlabW; ++w) {
      if (w >= wp) break;
      double f[kSlabRows];
      const double rp = s_rp;
      double row[kSlabW];
#pragma unroll
      for (int v = 0; v < kSlabW; ++v) row[v] = s_prow[w & 1][v];
      bool mine[kSlabRows];
#pragma unroll
      for (int r = 0; r < kSlabRows; ++r) {
        if (r * kSlabThreads + wid * kWarp >= m) break;
        mine[r] = tid + r * kSlabThreads == pr;
        if (mine[r]) used[r] = true;
        f[r] = mine[r] ? 0.0 : a[r][w] * rp;
        if (w + 1 < kSlabW) a[r][(w + 1) % kSlabW] = fma(-f[r], row[(w + 1) % kSlabW], a[r][(w + 1) % kSlabW]);
      }
      const bool more = w + 1 < wp;
      if (more) offer(w + 1);
      __syncthreads();
      int next = -1;
      if (more) next = choose(w + 1, key);
#pragma unroll
      for (int r = 0; r < kSlabRows; ++r) {
        if (r * kSlabThreads + wid * kWarp >= m) break;
#pragma unroll
        for (int v = 0; v < kSlabW; ++v)
          if (v != w && v != w + 1) a[r][v] = fma(-f[r], row[v], a[r][v]);
        a[r][w] = mine[r] ? 1.0 : -f[r];
      }
      if (more) publish(w + 1, next, key);
      pr = next;
      __syncthreads();
    }
    double* Tb = T + (size_t)b * kSlabW * ms;
    double* Tg = J.T + (size_t)k * kSlabW * ms;
#pragma unroll
    for (int r = 0; r < kSlabRows; ++r) {
      const int i = tid + r * kSlabThreads;
      if (i >= m) continue;
#pragma unroll
      for (int w = 0; w < kSlabW; ++w) {
        X[(size_t)(c0 + w) * ms + i] = a[r][w];
        const double t = w < wp ? (i == s_piv[b][w] ? a[r][w] - 1.0 : a[r][w]) : 0.0;
        Tb[w * ms + i] = t;
        Tg[w * ms + i] = t;
      }
    }
    if (tid < kSlabW && tid >= wp) s_piv[b][tid] = 0;   // its T column is zero
    __threadfence();
    __syncthreads();
    if (tid == 0) st_release(J.flag + k, epoch);
  };

  int ahead = -1;   // panel of this block that was factored ahead of its turn
  for (int k = 0; k < np; ++k) {
    const int b = k & 1;
    if (k % ng == g) {
      if (ahead != k) factor(k, b, (k / ng) * kSlabW, min(kSlabW, m - k * kSlabW));   // only k = 0, or one block
    } else {
      __syncthreads();
      if (tid == 0) {
        long long it = 0;
        while (it < wait && ld_acquire(J.flag + k) != epoch) ++it;
        if (it >= wait) s_abort = 1;
      }
      __syncthreads();
      if (s_abort) {
        if (tid == 0) atomicExch(&status[ST_SLAB_TIMEOUT], 1);
        return;
      }
      const double2* src = reinterpret_cast<const double2*>(J.T + (size_t)k * kSlabW * ms);
      double2* dst = reinterpret_cast<double2*>(T + (size_t)b * kSlabW * ms);
      for (int t = tid; t < kSlabW * ms / 2; t += kSlabThreads) dst[t] = __ldcg(src + t);
      if (tid < kSlabW) {
        const int pr = k * kSlabW + tid < m ? __ldcg(J.piv + k * kSlabW + tid) : 0;
        s_piv[b][tid] = FSI_IN(pr, m, FSI_SITE(4)) ? pr : 0;
        if (k * kSlabW + tid < m && FSI_IN(pr, m, FSI_SITE(4))) s_used[pr] = 1;
      }
    }
    // the next panel first, if it is this block's
    const int nx = k + 1;
    const int skip = k % ng == g ? k / ng : -1;
    const bool next = nx < np && nx % ng == g && ng > 1;
    if (next) {
      apply(b, (nx / ng) * kSlabW, (nx / ng + 1) * kSlabW);
      factor(nx, b ^ 1, (nx / ng) * kSlabW, min(kSlabW, m - nx * kSlabW));
      ahead = nx;
    }
    // the block's other panels (the transform leaves its own panel's columns alone)
    const int done = next ? nx / ng : -1;
    for (int s = 0; s < slots; ) {
      if (s == skip || s == done) { ++s; continue; }
      int s1 = s;
      while (s1 < slots && s1 != skip && s1 != done && s1 - s < 64 / kSlabW) ++s1;
      apply(b, s * kSlabW, s1 * kSlabW);
      s = s1;
    }
  }
  __syncthreads();
  // inverse[r][c] = rd[piv[r]] M[piv[r]][j], c the pivot row of column j: needs
  // every panel's pivots, which this block has waited for
  for (int c = wid; c < slots * kSlabW; c += kSlabWarps) {
    const int col = ((c / kSlabW) * ng + g) * kSlabW + c % kSlabW;
    if (col >= m) continue;
    const int oc = __ldcg(J.piv + col);
    if (!FSI_IN(oc, m, FSI_SITE(4))) continue;
    double* out = J.X + (size_t)oc * m;
    for (int r = lane; r < m; r += kWarp) {
      const int pr = __ldcg(J.piv + r);
      if (FSI_IN(pr, m, FSI_SITE(4))) out[r] = __ldcg(J.rd + pr) * X[(size_t)c * ms + pr];
    }
  }
  if (tid == 0 && s_sing) atomicExch(&status[ST_COARSE_RETRY], 1);
}

namespace {
size_t slab_gj_smem(int m, int ng) {
  const size_t ms = (m + 1) & ~1, np = (m + kSlabW - 1) / kSlabW;
  return (2 * kSlabW + (np + ng - 1) / ng * kSlabW) * ms * sizeof(double);
}
}  // namespace

size_t slab_gj_scratch(int m) { return (size_t)((m + kSlabW - 1) / kSlabW) * kSlabW * ((m + 1) & ~1); }
int slab_gj_panels(int m) { return (m + kSlabW - 1) / kSlabW; }

// Two rows per thread, and the block's panels in shared memory.  16 x 5 x 4 cells (slabs of
// 836): coarse factor 36 ms; 16 x 5 x 5 (1,072, from one end by the banded LU kernels): 188.
bool slab_gj_fits(int m, int sm_count) {
  return m <= kSlabThreads * kSlabRows && sm_count >= 4 && slab_gj_smem(m, sm_count / 2) <= 200 * 1024;
}

int launch_slab_gj(const SlabJobs& jobs, int epoch, long long wait, int32_t* status, int sm_count, cudaStream_t st) {
  int ng = jobs.n == 1 ? sm_count : sm_count / 2, mmax = 0;
  for (int i = 0; i < jobs.n; ++i) mmax = std::max(mmax, jobs.j[i].m);
  ng = std::min(ng, slab_gj_panels(mmax));
  const size_t smem = slab_gj_smem(mmax, ng);
  if (!allow_dynamic_smem(k_slab_gj)) return -1;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_slab_gj, kSlabThreads, smem);
  if (per_sm < 1) return -1;
  SlabJobs jb = jobs;
  void* args[] = {(void*)&jb, (void*)&ng, (void*)&epoch, (void*)&wait, (void*)&status};
  return cudaLaunchCooperativeKernel((const void*)k_slab_gj, ng * jobs.n, kSlabThreads, args, smem, st) == cudaSuccess
             ? 0 : -2;
}

// ---------------------------------------------------------------------------
// products of the elimination: C = beta C + alpha A B of up to two jobs in one
// launch (column-major).  32 x 32 output tiles, so that the two sides' products
// of 294 to 652 unknowns give every SM several tiles; the FP64 pipe bounds them,
// so terms in which a whole column of the A tile or row of the B tile is zero
// are left out: one factor of every product is a coupling block of the coarse
// operator, whose nodes meet their neighbours only.  16 slabs of 652 unknowns: the
// 17 launches take 3.8 ms, 6.7 with all terms.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_slab_gemm(SlabGemms jobs) {
  __shared__ double As[16][32 + 1], Bs[16][32 + 1];
  __shared__ uint8_t anz[16];      // column kk of the A tile has a nonzero
  __shared__ uint32_t bnz[16];     // rows of the B tile with a nonzero, per loading warp
  int t = blockIdx.x, j = 0;
  if (t >= jobs.tiles0) { t -= jobs.tiles0; j = 1; }
  const SlabGemm& g = jobs.g[j];
  const int tr = (g.m + 31) / 32, r0 = (t % tr) * 32, c0 = (t / tr) * 32;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[2][2] = {};
  for (int k0 = 0; k0 < g.k; k0 += 16) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = threadIdx.x + 256 * q;
      const int r = e % 32, kk = e / 32;            // A tile: rows fastest (coalesced columns)
      const double a = (r0 + r < g.m && k0 + kk < g.k) ? g.A[(int64_t)(k0 + kk) * g.lda + r0 + r] : 0.0;
      As[kk][r] = a;
      const int kb = e % 16, cb = e / 16;           // B tile: k fastest (coalesced columns)
      const double b = (k0 + kb < g.k && c0 + cb < g.n) ? g.B[(int64_t)(c0 + cb) * g.ldb + k0 + kb] : 0.0;
      Bs[kb][cb] = b;
      const bool na = __any_sync(0xffffffffu, nonzero(a));
      const uint32_t nb = __ballot_sync(0xffffffffu, nonzero(b));
      if (e % 32 == 0) {
        anz[kk] = na;
        bnz[e / 32] = nb | nb >> 16;
      }
    }
    __syncthreads();
    uint32_t live = 0u;
#pragma unroll
    for (int q = 0; q < 16; ++q) live |= bnz[q];
#pragma unroll
    for (int q = 0; q < 16; ++q)
      if (!anz[q]) live &= ~(1u << q);
#pragma unroll 4
    for (int kk = 0; kk < 16; ++kk) {
      if (!((live >> kk) & 1u)) continue;
      const double a0 = As[kk][tx], a1 = As[kk][tx + 16], b0 = Bs[kk][ty], b1 = Bs[kk][ty + 16];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int r = r0 + tx + 16 * i, c = c0 + ty + 16 * k;
      if (r < g.m && c < g.n) {
        double* p = g.C + (int64_t)c * g.ldc + r;
        *p = (g.beta == 0.0 ? 0.0 : g.beta * *p) + g.alpha * acc[i][k];
      }
    }
}

void launch_slab_gemm(const SlabGemm* g, int n, cudaStream_t st) {
  SlabGemms jobs{};
  int total = 0;
  for (int i = 0; i < n; ++i) {
    jobs.g[i] = g[i];
    total += ((g[i].m + 31) / 32) * ((g[i].n + 31) / 32);
    if (i == 0) jobs.tiles0 = total;
  }
  if (total > 0) k_slab_gemm<<<total, 256, 0, st>>>(jobs);
}

// ---------------------------------------------------------------------------
// solve
// ---------------------------------------------------------------------------
namespace {
constexpr int kSvThreads = 512;
constexpr int kSvMinRows = 4;                          // rows of a thread block's part of a product (a sector)
constexpr int kSvAhead = 16;                           // matrix entries per thread loaded ahead of the barrier

// out = beta y + alpha A x, rows [0, nr) over `nb` thread blocks
struct SvGemv {
  const double* A;
  int64_t lda;
  int nr, nc, b, nb;
  const double* x;
  double alpha, beta;
  const double* y;
  double* out;
};

// A thread block's part of a product: rows [r0, r0 + rb), rb = ceil(nr / nb).
// Threads over rows, then column groups; their sums are added in a fixed order.
struct SvPart {
  int rb, r0, cnt, ng, r, g;
  const double* col;   // entry (r0 + r, g)
  __device__ explicit SvPart(const SvGemv& j) {
    rb = max(kSvMinRows, (j.nr + j.nb - 1) / j.nb);
    r0 = j.b * rb;
    cnt = min(rb, j.nr - r0);
    ng = kSvThreads / rb;
    r = threadIdx.x % rb;
    g = threadIdx.x / rb;
    if (r >= cnt) g = j.nc;   // no columns
    col = j.A + (r0 + r) + (int64_t)g * j.lda;
  }
};
}  // namespace

// x = A^{-1} b over the slab ordering (b in w, overwritten; x in x): elimination
// from both ends, the middle slab, back substitution to both ends; each stage is
// a product over the thread blocks followed by a grid barrier, the left
// side's on the even blocks and the right side's on the odd ones, two products
// per slab and direction, in one launch.  A stage is a chain (barrier, x from
// L2, products, sums), so the matrix, which no stage changes, is loaded a stage
// ahead, the rows are spread over all blocks, and the column sums are added by 16
// lanes a row.  16 slabs of 652 unknowns (33 stages): 0.25 ms a solve; 0.41 with 16
// rows to a block (half of the SMs), 0.27 with the loads just before the
// barrier, 1.5 as 134 launches.
__global__ void __launch_bounds__(kSvThreads) k_slab_solve(SlabChain ch, const double* __restrict__ A, int64_t n,
                                                           const double* __restrict__ sinv, double* w, double* x,
                                                           double* u) {
  cg::grid_group grid = cg::this_grid();
  __shared__ double red[kSvThreads];
  const int side = blockIdx.x & 1, b0 = blockIdx.x >> 1, nbk = gridDim.x >> 1;
  const int K = ch.K, mid = ch.mid, p = ch.p;
  double* us = u + (size_t)side * ch.mmax;
  auto off = [&](int k) { return (int64_t)ch.off[k]; };
  auto len = [&](int k) { return ch.off[k + 1] - ch.off[k]; };
  auto inv = [&](int k) { return sinv + ch.inv[k]; };
  const int steps = max(mid, K - 1 - mid);
  // both sides correct the middle slab in the last step: the right one in a stage of its own
  const int clash = mid > 0 && mid == K - 1 - mid ? 1 : 0;
  const int fwd = 2 * steps + clash, total = fwd + 1 + 2 * steps;
  // this block's side's product of stage i (nr = 0: none)
  auto stage = [&](int i) {
    SvGemv j{A, n, 0, 0, b0, nbk, w, 1.0, 0.0, w, w};
    if (i < fwd) {
      const int s = min(i / 2, steps - 1), ph = i - 2 * s;
      const int kl = s + 1, kr = K - 2 - s;   // slabs that take a correction
      const bool apart = clash && s == steps - 1;
      if (side == 0 && kl <= mid) {
        if (ph == 0) {                        // u = S_{kl-1}^{-1}[P,:] w_{kl-1}
          const int m = len(kl - 1);
          j = SvGemv{inv(kl - 1) + (m - p), m, p, m, b0, nbk, w + off(kl - 1), 1.0, 0.0, us, us};
        } else if (ph == 1) {                 // w_kl -= A_{kl,kl-1}[:,P] u
          j = SvGemv{A + (off(kl) - p) * n + off(kl), n, len(kl), p, b0, nbk, us, -1.0, 1.0, w + off(kl), w + off(kl)};
        }
      }
      if (side == 1 && kr >= mid) {
        const int m = len(kr + 1);
        if (ph == 0) {                        // u = S_{kr+1}^{-1} w_{kr+1}
          j = SvGemv{inv(kr + 1), m, m, m, b0, nbk, w + off(kr + 1), 1.0, 0.0, us, us};
        } else if (ph == (apart ? 2 : 1)) {   // w_kr[P] -= A_{kr,kr+1}[P,:] u
          const int64_t o = off(kr + 1) - p;
          j = SvGemv{A + off(kr + 1) * n + o, n, p, m, b0, nbk, us, -1.0, 1.0, w + o, w + o};
        }
      }
    } else if (i == fwd) {                    // the middle slab, over the blocks of both sides
      const int m = len(mid);
      j = SvGemv{inv(mid), m, m, m, (int)blockIdx.x, (int)gridDim.x, w + off(mid), 1.0, 0.0, x + off(mid), x + off(mid)};
    } else if (i < total) {
      const int s = (i - fwd - 1) / 2, ph = (i - fwd - 1) % 2;
      const int k = side == 0 ? mid - 1 - s : mid + 1 + s;
      if (k >= 0 && k < K) {
        const int m = len(k);
        if (ph == 1) {
          j = SvGemv{inv(k), m, m, m, b0, nbk, w + off(k), 1.0, 0.0, x + off(k), x + off(k)};
        } else if (side == 0) {               // w_k[P] -= A_{k,k+1}[P,:] x_{k+1}
          const int64_t o = off(k + 1) - p;
          j = SvGemv{A + off(k + 1) * n + o, n, p, len(k + 1), b0, nbk, x + off(k + 1), -1.0, 1.0, w + o, w + o};
        } else {                              // w_k -= A_{k,k-1}[:,P] x_{k-1}[P]
          j = SvGemv{A + (off(k) - p) * n + off(k), n, m, p, b0, nbk, x + off(k) - p, -1.0, 1.0, w + off(k), w + off(k)};
        }
      }
    }
    return j;
  };
  auto ahead = [&](const SvGemv& j, double (&v)[kSvAhead]) {
    const SvPart t(j);
#pragma unroll
    for (int q = 0; q < kSvAhead; ++q)
      v[q] = t.g < t.ng && t.g + q * t.ng < j.nc ? __ldg(t.col + (int64_t)q * t.ng * j.lda) : 0.0;
  };
  double a[kSvAhead], an[kSvAhead];
  SvGemv j = stage(0);
  ahead(j, a);
  for (int i = 0; i < total; ++i) {
    const SvGemv jn = stage(i + 1);
    ahead(jn, an);
    const SvPart t(j);
    if (t.cnt > 0) {
      double s = 0.0;
      if (t.g < t.ng) {
        double xv[kSvAhead];
#pragma unroll
        for (int q = 0; q < kSvAhead; ++q) {
          const int c = t.g + q * t.ng;
          xv[q] = c < j.nc ? __ldcg(j.x + c) : 0.0;
        }
        double s1 = 0.0;
#pragma unroll
        for (int q = 0; q < kSvAhead; q += 2) {
          if (t.g + q * t.ng < j.nc) s = fma(a[q], xv[q], s);
          if (t.g + (q + 1) * t.ng < j.nc) s1 = fma(a[q + 1], xv[q + 1], s1);
        }
        for (int c = t.g + kSvAhead * t.ng; c < j.nc; c += t.ng)
          s = fma(__ldg(t.col + (int64_t)(c - t.g) * j.lda), __ldcg(j.x + c), s);
        s += s1;
      }
      red[threadIdx.x] = s;
      __syncthreads();
      for (int e0 = threadIdx.x / 32 * 32; e0 < t.rb * 16; e0 += kSvThreads) {   // 16 lanes a row
        const int e = e0 + threadIdx.x % 32, r = e / 16;
        double v = 0.0;
        if (r < t.cnt)
          for (int g = e % 16; g < t.ng; g += 16) v += red[g * t.rb + r];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (e % 16 == 0 && r < t.cnt) {
          const double b = j.beta == 0.0 ? 0.0 : j.beta * __ldcg(j.y + t.r0 + r);
          __stcg(j.out + t.r0 + r, fma(j.alpha, v, b));
        }
      }
    }
    if (i + 1 == total) break;
    grid.sync();
    j = jn;
#pragma unroll
    for (int q = 0; q < kSvAhead; ++q) a[q] = an[q];
  }
}

int launch_slab_solve(const SlabChain& ch, const double* A, int64_t n, const double* sinv, double* w, double* x,
                      double* u, int sm_count, cudaStream_t st) {
  const int grid = std::max(2, std::min(sm_count & ~1, 2 * ((ch.mmax + kSvMinRows - 1) / kSvMinRows)));
  SlabChain c = ch;
  void* args[] = {(void*)&c, (void*)&A, (void*)&n, (void*)&sinv, (void*)&w, (void*)&x, (void*)&u};
  return cudaLaunchCooperativeKernel((const void*)k_slab_solve, grid, kSvThreads, args, 0, st) == cudaSuccess ? 0 : -2;
}

FSI_BOUNDS_READER(bounds_site_slab)

}  // namespace fsi
