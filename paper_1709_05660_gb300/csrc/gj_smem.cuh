// Dense FP64 Gauss-Jordan inverse of a small matrix in shared memory by one
// thread block: the leaves and interface systems of the coarse inverse and the
// small Schwarz blocks.
#pragma once

#include <cstdint>

#include "bounds.cuh"
#include "fp64_util.cuh"

namespace fsi {
namespace {
constexpr int kGjU = 5;                      // rows per lane
constexpr int kGjSmemMax = kGjU * kWarp;     // largest matrix

struct GjStep {        // step state handed from warp 0 to the others (double-buffered)
  int row[2];          // pivot row
  uint32_t live[2];    // bit u: rows 32 u .. 32 u + 31 hold a nonzero multiplier
  int sing;
};

// In-place Gauss-Jordan inverse of the n x n matrix M (shared memory, column
// c at M + c ld) by the whole thread block, with partial pivoting by unused
// rows: piv[k] is the row that step k used and rd[piv[k]] the reciprocal of its
// pivot; rows stay unscaled, so on return
// inverse[r][c] = rd[piv[r]] M[piv[r] + qinv[c] ld] with qinv[piv[k]] = k.
// Warp 0 runs one step ahead: it updates the next pivot column, searches it
// and forms the multipliers while other warps update the remaining columns,
// so a step costs one block barrier.  A warp-wide FP64 operation occupies its
// sub-partition's pipe for 64 cycles however many lanes it has, so a column
// costs ceil(n / 32) of them and nothing else (hence the unscaled rows), the
// pivot search runs on integer keys, and for small n, where warp 0's chain
// bounds the step, the warps of its sub-partition stay idle.  Columns whose
// pivot-row entry is zero and groups of 32 rows without a multiplier are
// skipped.  A dense 88 x 88 block: 300 us, 400
// with scaled rows and a 64-bit shuffle search (the FP64 pipe alone: 190).
// own (may be null): rows of the inverse that the caller reads; a row that
// becomes another one (the pivot row of a column k with own[k] = 0) is not
// updated any more.  f: 2 n doubles, rd: n doubles.  Returns false (whole
// block) when a pivot was zero or not finite.
__device__ bool gj_inverse_smem(double* M, int n, int ld, double* f, double* rd, int* piv, int* qinv, GjStep& st,
                                const uint8_t* own) {
  const int lane = threadIdx.x % kWarp, wid = threadIdx.x / kWarp, nw = blockDim.x / kWarp;
  const int nu = (n + kWarp - 1) / kWarp;
  // warp 0: bit u of row lane + 32 u: has been a pivot row; is not needed any more
  uint32_t used = 0u, dead = 0u;
  if (threadIdx.x == 0) st.sing = 0;
  // search column k (largest |a| of the unused rows, ties to the lowest row)
  // and form the multipliers of step k (warp 0)
  auto prepare = [&](int k) {
    const double* Mk = M + (size_t)k * ld;
    double* fk = f + (k & 1) * n;
    double v[kGjU];
    uint32_t hi = 0u;
#pragma unroll
    for (int u = 0; u < kGjU; ++u) {
      const int r = lane + u * kWarp;
      v[u] = u < nu && r < n ? Mk[r] : 0.0;
      if (!((used >> u) & 1u)) hi = max(hi, (uint32_t)(abs_key(v[u]) >> 32));
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    uint32_t lo = 0u;
#pragma unroll
    for (int u = 0; u < kGjU; ++u) {
      const unsigned long long key = abs_key(v[u]);
      if (!((used >> u) & 1u) && (uint32_t)(key >> 32) == hi) lo = max(lo, (uint32_t)key);
    }
    lo = __reduce_max_sync(0xffffffffu, lo);
    const unsigned long long best = ((unsigned long long)hi << 32) | lo;
    uint32_t row = 0xffffffffu;
#pragma unroll
    for (int u = kGjU - 1; u >= 0; --u)
      if (u < nu && !((used >> u) & 1u) && lane + u * kWarp < n && abs_key(v[u]) == best) row = lane + u * kWarp;
    const int bi = (int)__reduce_min_sync(0xffffffffu, row);
    double rp = 0.0;
    if (lane == 0 && FSI_IN(bi, n, FSI_SITE(5))) {
      double pv = Mk[bi];
      if (best == 0ull || best >= 0x7FF0000000000000ull) {
        st.sing = 1;
        pv = 1.0;
      }
      rp = 1.0 / pv;
      rd[bi] = rp;
      st.row[k & 1] = bi;
      piv[k] = bi;
    }
    rp = __shfl_sync(0xffffffffu, rp, 0);
    uint32_t live = 0u;
#pragma unroll
    for (int u = 0; u < kGjU; ++u) {
      if (u >= nu) break;
      const int r = lane + u * kWarp;
      // the pivot row itself and rows that nobody needs stay as they are
      const double m = r == bi || ((dead >> u) & 1u) ? 0.0 : v[u] * rp;
      if (r < n) fk[r] = m;
      if (__any_sync(0xffffffffu, nonzero(m))) live |= 1u << u;
      if (r == bi) {
        used |= 1u << u;
        if (own && !own[k]) dead |= 1u << u;
      }
    }
    if (lane == 0) st.live[k & 1] = live;
  };
  // column j of step k: M[r][j] -= f[r] M[pr][j]
  auto update = [&](int j, int pr, uint32_t live, const double (&fr)[kGjU]) {
    double* Mj = M + (size_t)j * ld;
    const double t = Mj[pr];
    if (!nonzero(t)) return;
    double x[kGjU];
#pragma unroll
    for (int u = 0; u < kGjU; ++u) {
      if (!((live >> u) & 1u)) continue;
      const int r = lane + u * kWarp;
      x[u] = r < n ? Mj[r] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kGjU; ++u) {
      if (!((live >> u) & 1u)) continue;
      const int r = lane + u * kWarp;
      x[u] = fma(-fr[u], t, x[u]);
      if (r < n) Mj[r] = x[u];
    }
  };
  __syncthreads();
  if (wid == 0) prepare(0);
  // workers: every warp but warp 0, or only those of the other sub-partitions
  const bool spread = n > 2 * kWarp;
  const int nwork = spread ? nw - 1 : nw - nw / 4;
  const int mine = wid == 0 || (!spread && wid % 4 == 0) ? n : spread ? wid - 1 : wid - 1 - wid / 4;
  for (int k = 0; k < n; ++k) {
    __syncthreads();
    const int pr = st.row[k & 1];
    if (!FSI_IN(pr, n, FSI_SITE(5))) break;   // the whole block
    const uint32_t live = st.live[k & 1];
    double fr[kGjU];
#pragma unroll
    for (int u = 0; u < kGjU; ++u) {
      const int r = lane + u * kWarp;
      fr[u] = u < nu && r < n ? f[(k & 1) * n + r] : 0.0;
    }
    if (wid == 0) {
      if (k + 1 < n) {
        update(k + 1, pr, live, fr);
        __syncwarp();
        prepare(k + 1);
      }
      double* Mk = M + (size_t)k * ld;
#pragma unroll
      for (int u = 0; u < kGjU; ++u) {
        const int r = lane + u * kWarp;
        if (u < nu && r < n) Mk[r] = r == pr ? 1.0 : -fr[u];
      }
    } else {
      for (int j = mine; j < n; j += nwork)
        if (j != k && j != k + 1) update(j, pr, live, fr);
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) qinv[k] = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) qinv[piv[k]] = k;
  __syncthreads();
  return st.sing == 0;
}
}  // namespace
}  // namespace fsi
