// Element-batched residual + exact Jacobian assembly and Galerkin coarsening.
//
// Assembly (Sec. 2.3, 2.5, 3): the fluxes at a quadrature point depend on the
// element unknowns only through a few fields (gradients and values of u and d,
// p), so they are evaluated in forward-mode dual arithmetic along those fields
// (the derivative of the discrete residual, as the paper obtains with automatic
// differentiation) and contracted with the bases of trial and test functions one
// direction after the other.  Element matrices are written to an element-matrix
// buffer; a gather adds them into the block-sparse Jacobian, each entry over its
// elements in a fixed order.
//
// Galerkin (Sec. 3.2): J_{l-1} = R J_l P is formed element by element.  A
// coarse element matrix is sum_children R_c A_c P_c, where P_c interpolates
// the coarse element's Q2 / P1disc unknowns to the child's and R_c is its
// transpose restricted to equations of the same kind (momentum, solid
// kinematic, ALE) with Dirichlet rows and columns dropped.
#include <cooperative_groups.h>

#include "kernels.h"

namespace fsi {

namespace {

struct Dual {
  double v, d;
};
__device__ __forceinline__ Dual mk(double v, double d) { return Dual{v, d}; }
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return {a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return {a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ Dual operator-(Dual a) { return {-a.v, -a.d}; }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return {a.v * b.v, a.d * b.v + a.v * b.d}; }
__device__ __forceinline__ Dual operator*(Dual a, double s) { return {a.v * s, a.d * s}; }
__device__ __forceinline__ Dual operator+(Dual a, double s) { return {a.v + s, a.d}; }
// a / b given inv = 1 / b.v (one reciprocal shared by several quotients of the
// same divisor)
__device__ __forceinline__ Dual div_inv(Dual a, Dual b, double inv) {
  const double q = a.v * inv;
  return {q, (a.d - b.d * q) * inv};
}

// 1D quadratic Lagrange basis (nodes -1, 0, 1) and derivative at the three
// Gauss points -sqrt(3/5), 0, sqrt(3/5).
__device__ __forceinline__ double gp(int q) { return q == 0 ? -0.7745966692414834 : (q == 1 ? 0.0 : 0.7745966692414834); }
__device__ __forceinline__ double gw(int q) { return q == 1 ? 8.0 / 9.0 : 5.0 / 9.0; }
__device__ __forceinline__ double L1(int m, double x) {
  return m == 0 ? 0.5 * x * (x - 1.0) : (m == 1 ? 1.0 - x * x : 0.5 * x * (x + 1.0));
}
__device__ __forceinline__ double dL1(int m, double x) { return m == 0 ? x - 0.5 : (m == 1 ? -2.0 * x : x + 0.5); }

constexpr int kDim = 2;
constexpr int kB = 4;           // unknowns per node block
constexpr int kNloc = 9;        // Q2 nodes per element
constexpr int kNN = kB * kNloc; // node unknowns per element
constexpr int kNdofe = kNN + kDim + 1;   // 39
constexpr int kEPB = 4;         // elements per thread block

}  // namespace

// ---------------------------------------------------------------------------
// element residual + Jacobian (2D)
//
// At a quadrature point the weak-form fluxes (stresses, convection, inertia,
// kinematic, ALE and mass terms) depend on the element unknowns only through
// 13 field quantities: d, grad d, u, grad u and p.  Column j of the element
// Jacobian is therefore sum_f (d flux / d field_f) (d field_f / d y_j), where
// d field_f / d y_j is a basis value or gradient of unknown j (nonzero for at
// most three fields).  The kernel differentiates the fluxes along the 13
// field directions with dual numbers (9 points x 13 directions = 117 dual
// evaluations per element, three per thread) and contracts them with the trial
// and test basis; the result is the exact Jacobian of the discrete residual, as
// with one dual evaluation per unknown, at about a third of the FP64 work.
//
// The contraction is sum-factorised (the Q2 basis is a product of 1D ones):
// first over the points of a column (7 coefficient combinations), then along x
// (4), 1.5 thousand fused multiply-adds per pair of components instead of 3.6
// thousand; the mesh and kinematic rows, whose coefficients are constant, are
// products of 1D integrals.  The FP64 pipe bounds the kernel.  6-level channel
// (65,536 elements): 11.7 -> 5.9 ms on GB300.
// ---------------------------------------------------------------------------
namespace {
constexpr int kQ = 9;            // Gauss points (3 x 3)
constexpr int kNF = 13;          // differentiated fields
constexpr int kNFV = 17;         // + BDF history values (u_old, d_old)
constexpr int kNFVcn = 26;       // Crank-Nicolson: + the t_n fields (u_n, d_n, grad d_n, grad u_n, p_n)
constexpr int kNO = 11;          // flux outputs per point
// fields: 0,1 d_i | 2..5 dd_i/dx_k (2 + 2 i + k) | 6,7 u_i | 8..11 du_i/dx_k (8 + 2 i + k) | 12 p
//         13,14 u-history | 15,16 d-history
// outputs, fluid: 0..3 T_ck (2 c + k) | 4,5 convection_c | 6..9 ALE A_ck (6 + 2 c + k) | 10 mass
//          solid: 0..3 T_ck | 4,5 inertia_c | 6,7 kinematic_c | 10 mass
// (every output carries its quadrature weight; T and A multiply a test gradient
// in reference coordinates scaled by 2 / h, the others a test value)
//         CN: 13,14 u_n | 15,16 d_n | 17..20 d d_n,i/dx_k (17 + 2 i + k) | 21..24 d u_n,i/dx_k | 25 p_n
constexpr int kND = 7;            // differentiated outputs kept: T 0..3, body 4,5, mass 6 (the others are constant)
constexpr int kNH = 2 * kB * 4 * 3 * 9;   // column sums: [c][s][2 tx + rx][qx][3 ja + jb]
constexpr size_t asm_elem_doubles(int nfv) {
  return (size_t)kQ * nfv + (size_t)kQ * kNF * kND + (size_t)kQ * kNO + kNH;
}

// First Piola stress of the incompressible solid (Sec. 2.2):
// P = -p J F^{-T} + 2 C1 J F - 2 C2 J F^{-T} F^{-1} F^{-T}, 2 C1 = mu_s - 2 C2
__device__ __forceinline__ void piola_2d(const Dual (&F)[2][2], const Dual (&Fi)[2][2], Dual J, Dual p,
                                         const PhysParams& pp, Dual (&P)[2][2]) {
  const Dual pJ = p * J;
  const Dual muJ = J * (pp.mu_s - 2.0 * pp.mr_c2);
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int k = 0; k < 2; ++k) P[c][k] = muJ * F[c][k] - pJ * Fi[k][c];
  if (pp.mr_c2 != 0.0) {
    Dual Q[2][2];   // F^{-1} F^{-T}
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) Q[a][b] = Fi[a][0] * Fi[b][0] + Fi[a][1] * Fi[b][1];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int k = 0; k < 2; ++k) P[c][k] = P[c][k] - (Fi[0][c] * Q[0][k] + Fi[1][c] * Q[1][k]) * J * (2.0 * pp.mr_c2);
  }
}
}  // namespace

// MODE: 0 steady, 1 BDF (yold = a1 y_n + a2 y_{n-1}), 2 Crank-Nicolson (yold = y_n)
template <bool SOLID, int MODE>
__global__ void __launch_bounds__(kEPB * kNdofe, MODE == 2 ? 2 : 3)
k_assemble_2d(const int32_t* __restrict__ elems, int ne, const double* __restrict__ y,
              const int32_t* __restrict__ elem_nodes, const uint8_t* __restrict__ node_class,
              const double* __restrict__ elem_geo, int64_t n_nodes, PhysParams pp,
              double* __restrict__ Ke, double* __restrict__ Re, int32_t* __restrict__ status) {
  constexpr bool TRANS = MODE != 0;
  constexpr bool CN = MODE == 2;
  constexpr int NFV = CN ? kNFVcn : kNFV;
  __shared__ double s_y[kEPB][kNdofe];
  __shared__ double s_yo[kEPB][kNdofe];
  __shared__ double s_geo[kEPB][2 * kDim];
  __shared__ unsigned s_iface[kEPB];
  __shared__ double s_scl[kEPB][3];   // 2 / hx, 2 / hy, 1 / (hx hy): divided once per element
  __shared__ double s_wq[kEPB][kQ];    // quadrature weights times the Jacobian of the element map
  __shared__ double s_N[kQ][kNloc], s_Dx[kQ][kNloc], s_Dy[kQ][kNloc];   // reference basis at the points
  // products of the 1D reference basis at the three points, [kind][point][3 a + b], and their integrals;
  // kind: bit 1 the test (a) side is a derivative, bit 0 the trial (b) side
  __shared__ double s_PP[4][3][9], s_I1[4][9];
  __shared__ int s_e[kEPB];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int le = threadIdx.x / kNdofe;
  const int j = threadIdx.x % kNdofe;
  const int el = blockIdx.x * kEPB + le;
  const bool active = le < kEPB && el < ne;
  const int e = active ? elems[el] : 0;
  for (int t = threadIdx.x; t < kQ * kNloc; t += blockDim.x) {
    const int q = t / kNloc, a = t % kNloc;
    const double xi = gp(q % 3), eta = gp(q / 3);
    const int ia = a % 3, ja = a / 3;
    s_N[q][a] = L1(ia, xi) * L1(ja, eta);
    s_Dx[q][a] = dL1(ia, xi) * L1(ja, eta);
    s_Dy[q][a] = L1(ia, xi) * dL1(ja, eta);
  }
  if (threadIdx.x < 108) {
    const int ab = threadIdx.x % 9, q = (threadIdx.x / 9) % 3, kind = threadIdx.x / 27;
    const double x = gp(q);
    s_PP[kind][q][ab] = (kind & 2 ? dL1(ab / 3, x) : L1(ab / 3, x)) * (kind & 1 ? dL1(ab % 3, x) : L1(ab % 3, x));
  }
  if (j == 0 && le < kEPB) s_e[le] = active ? e : -1;
  if (active) {
    if (j < kNN) {
      const int a = j / kB, s = j % kB;
      const int64_t gi = (int64_t)elem_nodes[(int64_t)e * kNloc + a] * kB + s;
      s_y[le][j] = y[gi];
      if (TRANS) s_yo[le][j] = pp.yold[gi];
    } else {
      s_y[le][j] = y[(n_nodes + e) * kB + (j - kNN)];
      if (CN) s_yo[le][j] = pp.yold[(n_nodes + e) * kB + (j - kNN)];
    }
    if (j < 2 * kDim) s_geo[le][j] = elem_geo[(int64_t)e * 2 * kDim + j];
    if (j == 0) {
      unsigned m = 0;
      for (int a = 0; a < kNloc; ++a)
        if (node_class[elem_nodes[(int64_t)e * kNloc + a]] == kIface) m |= 1u << a;
      s_iface[le] = m;
      const double ghx = elem_geo[(int64_t)e * 2 * kDim + 2], ghy = elem_geo[(int64_t)e * 2 * kDim + 3];
      s_scl[le][0] = 2.0 / ghx;
      s_scl[le][1] = 2.0 / ghy;
      s_scl[le][2] = 1.0 / (ghx * ghy);
    }
    if (j < kQ) {
      const double vol_e = elem_geo[(int64_t)e * 2 * kDim + 2] * elem_geo[(int64_t)e * 2 * kDim + 3];
      s_wq[le][j] = gw(j % 3) * gw(j / 3) * vol_e * 0.25;
    }
  }
  __syncthreads();
  const int le_c = le < kEPB ? le : 0;
  double* Fv = reinterpret_cast<double*>(smem_raw) + (size_t)le_c * asm_elem_doubles(NFV);   // [kQ][NFV]
  double* Dd = Fv + kQ * NFV;                                                               // [kQ][kNF][kND]
  double* Vo = Dd + kQ * kNF * kND;                                                     // [kQ][kNO]
  const double* ye = s_y[le_c];
  const double* yo = s_yo[le_c];
  const double sx = s_scl[le_c][0], sy = s_scl[le_c][1];
  const double kale = s_scl[le_c][2];

  // 1. field values at the points
  if (active) {
    for (int it = j; it < kQ * NFV; it += kNdofe) {
      const int q = it / NFV, f = it % NFV;
      double v = 0.0;
      if (f == 12) {
        v = ye[kNN] + ye[kNN + 1] * gp(q % 3) + ye[kNN + 2] * gp(q / 3);
      } else if (CN && f == 25) {
        v = yo[kNN] + yo[kNN + 1] * gp(q % 3) + yo[kNN + 2] * gp(q / 3);
      } else if (f < 13 || TRANS) {
        // source component, basis kind (0 value, 1 d/dx, 2 d/dy), history flag
        int comp, kind;
        const double* src = ye;
        if (f < 2) { comp = f; kind = 0; }
        else if (f < 6) { comp = (f - 2) / 2; kind = 1 + (f - 2) % 2; }
        else if (f < 8) { comp = 2 + (f - 6); kind = 0; }
        else if (f < 12) { comp = 2 + (f - 8) / 2; kind = 1 + (f - 8) % 2; }
        else if (f < 15) { comp = 2 + (f - 13); kind = 0; src = yo; }
        else if (f < 17) { comp = f - 15; kind = 0; src = yo; }
        else if (f < 21) { comp = (f - 17) / 2; kind = 1 + (f - 17) % 2; src = yo; }
        else { comp = 2 + (f - 21) / 2; kind = 1 + (f - 21) % 2; src = yo; }
        const double* tb = kind == 0 ? s_N[q] : (kind == 1 ? s_Dx[q] : s_Dy[q]);
#pragma unroll
        for (int a = 0; a < kNloc; ++a) v += src[a * kB + comp] * tb[a];
        if (kind == 1) v *= sx;
        if (kind == 2) v *= sy;
      }
      Fv[q * NFV + f] = v;
    }
  }
  __syncthreads();

  // 2. flux values and their derivatives along each field direction
  bool tangled = false;
  if (active) {
#pragma unroll 1
    for (int it = j; it < kQ * kNF; it += kNdofe) {
      const int q = it / kNF, f = it % kNF;
      const double* fv = Fv + q * NFV;
      double* dout = Dd + (q * kNF + f) * kND;
      if (!TRANS && f < 2) {   // d itself enters only the BDF terms
#pragma unroll
        for (int o = 0; o < kND; ++o) dout[o] = 0.0;
        continue;
      }
      const double wq = s_wq[le_c][q];
      Dual gd[2][2], gu[2][2], u[2], ut[2], dt_[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          gd[i][k] = mk(fv[2 + 2 * i + k], f == 2 + 2 * i + k ? 1.0 : 0.0);
          gu[i][k] = mk(fv[8 + 2 * i + k], f == 8 + 2 * i + k ? 1.0 : 0.0);
        }
        u[i] = mk(fv[6 + i], f == 6 + i ? 1.0 : 0.0);
        if (TRANS) {
          const Dual di = mk(fv[i], f == i ? 1.0 : 0.0);
          ut[i] = (u[i] * pp.a0 + fv[13 + i]) * pp.idt;
          dt_[i] = (di * pp.a0 + fv[15 + i]) * pp.idt;
        }
      }
      const Dual p = mk(fv[12], f == 12 ? 1.0 : 0.0);
      Dual F[2][2];
      F[0][0] = gd[0][0] + 1.0; F[0][1] = gd[0][1];
      F[1][0] = gd[1][0];       F[1][1] = gd[1][1] + 1.0;
      const Dual J = F[0][0] * F[1][1] - F[0][1] * F[1][0];
      if (!(J.v > 0.0)) tangled = true;
      Dual Fi[2][2];
      const double iJ = 1.0 / J.v;
      Fi[0][0] = div_inv(F[1][1], J, iJ); Fi[0][1] = div_inv(-F[0][1], J, iJ);
      Fi[1][0] = div_inv(-F[1][0], J, iJ); Fi[1][1] = div_inv(F[0][0], J, iJ);
      Dual out[kNO];
      if (CN) {
        // Crank-Nicolson (Sec. 2.5): stresses and convection averaged over
        // t_{n+1} and t_n, the conservative ALE inertia (rho J u)_{n+1} -
        // (rho J u)_n over dt with -(div w) u averaged, w = (d - d_n) / dt;
        // the t_n state enters as constants (zero derivative)
        const double un[2] = {fv[13], fv[14]};
        Dual Fn[2][2], Fin[2][2], gw[2][2], w[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          w[i] = (mk(fv[i], f == i ? 1.0 : 0.0) + (-fv[15 + i])) * pp.idt;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            Fn[i][k] = mk(fv[17 + 2 * i + k] + (i == k ? 1.0 : 0.0), 0.0);
            gw[i][k] = (gd[i][k] + (-fv[17 + 2 * i + k])) * pp.idt;
          }
        }
        const Dual Jn = Fn[0][0] * Fn[1][1] - Fn[0][1] * Fn[1][0];
        if (!(Jn.v > 0.0)) tangled = true;
        const double iJn = 1.0 / Jn.v;
        Fin[0][0] = div_inv(Fn[1][1], Jn, iJn); Fin[0][1] = div_inv(-Fn[0][1], Jn, iJn);
        Fin[1][0] = div_inv(-Fn[1][0], Jn, iJn); Fin[1][1] = div_inv(Fn[0][0], Jn, iJn);
        const Dual pn = mk(fv[25], 0.0);
        if (SOLID) {
          Dual P1[2][2], Pn[2][2];
          piola_2d(F, Fi, J, p, pp, P1);
          piola_2d(Fn, Fin, Jn, pn, pp, Pn);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
#pragma unroll
            for (int k = 0; k < 2; ++k) out[2 * c + k] = (P1[c][k] + Pn[c][k]) * (0.5 * wq);
            out[4 + c] = (u[c] * J - Jn * un[c]) * (pp.rho_s * pp.idt * wq);
            out[6 + c] = ((u[c] + un[c]) * 0.5 - w[c]) * wq;
          }
          out[8] = mk(0.0, 0.0);
          out[9] = mk(0.0, 0.0);
          out[10] = (J + (-1.0)) * wq;
        } else {
          Dual gx[2][2], gxn[2][2];
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              gx[i][k] = gu[i][0] * Fi[0][k] + gu[i][1] * Fi[1][k];
              gxn[i][k] = Fin[0][k] * fv[21 + 2 * i] + Fin[1][k] * fv[21 + 2 * i + 1];
            }
          Dual sig[2][2], sgn[2][2];
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              sig[i][k] = (gx[i][k] + gx[k][i]) * pp.mu_f;
              sgn[i][k] = (gxn[i][k] + gxn[k][i]) * pp.mu_f;
            }
          sig[0][0] = sig[0][0] - p;
          sig[1][1] = sig[1][1] - p;
          sgn[0][0] = sgn[0][0] - pn;
          sgn[1][1] = sgn[1][1] - pn;
          const Dual divw1 = gw[0][0] * Fi[0][0] + gw[0][1] * Fi[1][0] + gw[1][0] * Fi[0][1] + gw[1][1] * Fi[1][1];
          const Dual divwn =
              gw[0][0] * Fin[0][0] + gw[0][1] * Fin[1][0] + gw[1][0] * Fin[0][1] + gw[1][1] * Fin[1][1];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
              out[2 * c + k] = ((sig[c][0] * Fi[k][0] + sig[c][1] * Fi[k][1]) * J +
                                (sgn[c][0] * Fin[k][0] + sgn[c][1] * Fin[k][1]) * Jn) * (0.5 * wq);
            const Dual conv1 = gx[c][0] * (u[0] - w[0]) + gx[c][1] * (u[1] - w[1]);
            const Dual convn = gxn[c][0] * (-w[0] + un[0]) + gxn[c][1] * (-w[1] + un[1]);
            const Dual val = (u[c] * J - Jn * un[c]) * pp.idt - divw1 * J * u[c] * 0.5 - divwn * Jn * (0.5 * un[c]) +
                             conv1 * J * 0.5 + convn * Jn * 0.5;
            out[4 + c] = val * (pp.rho_f * wq);
#pragma unroll
            for (int k = 0; k < 2; ++k)
              out[6 + 2 * c + k] = (pp.ale_op == 0 ? gd[c][k] + gd[k][c] : gd[c][k]) * (kale * wq);
          }
          out[10] = J * (gx[0][0] + gx[1][1]) * wq;
        }
      } else if (SOLID) {
        // P = J sigma F^{-T} = -p J F^{-T} + 2 C1 J F - 2 C2 J F^{-T} F^{-1} F^{-T}
        // (sigma = -p I + 2 C1 B - 2 C2 B^{-1}, 2 C1 = mu_s - 2 C2; C2 = 0: Neo-Hookean)
        Dual P[2][2];
        piola_2d(F, Fi, J, p, pp, P);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
#pragma unroll
          for (int k = 0; k < 2; ++k) out[2 * c + k] = P[c][k] * wq;
          out[4 + c] = TRANS ? ut[c] * J * (pp.rho_s * wq) : mk(0.0, 0.0);
          out[6 + c] = (TRANS ? u[c] - dt_[c] : u[c]) * wq;
        }
        out[8] = mk(0.0, 0.0);
        out[9] = mk(0.0, 0.0);
        out[10] = (J + (-1.0)) * wq;
      } else {
        Dual gx[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int k = 0; k < 2; ++k) gx[i][k] = gu[i][0] * Fi[0][k] + gu[i][1] * Fi[1][k];
        Dual sig[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int k = 0; k < 2; ++k) sig[i][k] = (gx[i][k] + gx[k][i]) * pp.mu_f;
        sig[0][0] = sig[0][0] - p;
        sig[1][1] = sig[1][1] - p;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
#pragma unroll
          for (int k = 0; k < 2; ++k) out[2 * c + k] = (sig[c][0] * Fi[k][0] + sig[c][1] * Fi[k][1]) * J * wq;
          const Dual cv = TRANS ? gx[c][0] * (u[0] - dt_[0]) + gx[c][1] * (u[1] - dt_[1]) + ut[c]
                                : gx[c][0] * u[0] + gx[c][1] * u[1];
          out[4 + c] = cv * J * (pp.rho_f * wq);
#pragma unroll
          for (int k = 0; k < 2; ++k)
            out[6 + 2 * c + k] = (pp.ale_op == 0 ? gd[c][k] + gd[k][c] : gd[c][k]) * (kale * wq);
        }
        out[10] = J * (gx[0][0] + gx[1][1]) * wq;
      }
      // gradient outputs and gradient fields in reference coordinates: fold the 2 / h scales
      const double sf = f >= 2 && f < 12 && f != 6 && f != 7 ? (f & 1 ? sy : sx) : 1.0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        dout[2 * c] = out[2 * c].d * (sx * sf);
        dout[2 * c + 1] = out[2 * c + 1].d * (sy * sf);
        dout[4 + c] = out[4 + c].d * sf;
      }
      dout[6] = out[10].d * sf;
      if (f == 12) {   // any direction carries the values
#pragma unroll
        for (int o = 0; o < kNO; ++o) Vo[q * kNO + o] = out[o].v;
      }
    }
  }
  if (tangled) atomicExch(&status[ST_TANGLED], 1);
  __syncthreads();

  // 3. y: item = (element, test component c, trial component s, qx, pair (ja, jb) of 1D nodes in y).  Component s
  //    moves the fields value / d/dx / d/dy of its unknown.
  const size_t estride = asm_elem_doubles(NFV), oD = (size_t)kQ * NFV, oV = oD + (size_t)kQ * kNF * kND,
               oH = oV + (size_t)kQ * kNO;
  double* base = reinterpret_cast<double*>(smem_raw);
  auto f_val = [](int s) { return s < 2 ? s : 4 + s; };
  auto f_grad = [](int s) { return s < 2 ? 2 + 2 * s : 4 + 2 * s; };
  for (int t = threadIdx.x; t < kEPB * 216; t += blockDim.x) {
    const int l = t / 216, yp = t % 9, qx = (t / 9) % 3, s = (t / 27) % 4, c = (t / 108) % 2;
    const double* D = base + l * estride + oD;
    double h0 = 0.0, h1 = 0.0, h2 = 0.0, h3 = 0.0;
#pragma unroll
    for (int qy = 0; qy < 3; ++qy) {
      const double vv = s_PP[0][qy][yp], vd = s_PP[1][qy][yp], dv = s_PP[2][qy][yp], dd = s_PP[3][qy][yp];
      const double* dq = D + (qx + 3 * qy) * (kNF * kND);
      const double *gx = dq + f_grad(s) * kND, *gy = gx + kND, *g0 = dq + f_val(s) * kND;
      h0 = fma(gx[2 * c], vv, h0);
      h1 = fma(gy[2 * c], vd, h1);
      h2 = fma(gx[2 * c + 1], dv, fma(gx[4 + c], vv, h2));
      h3 = fma(gy[2 * c + 1], dd, fma(gy[4 + c], vd, fma(g0[4 + c], vv, h3)));
    }
    double* H = base + l * estride + oH + ((c * kB + s) * 12 + qx) * 9 + yp;   // + 27 k: combination k
    H[0] = h0;
    H[27] = h1;
    H[54] = h2;
    H[81] = h3;
  }
  // 1D integrals of the constant-coefficient rows; pressure rows and columns
  if (threadIdx.x < 36) {
    const int ab = threadIdx.x % 9, kind = threadIdx.x / 9;
    s_I1[kind][ab] = s_PP[kind][0][ab] * gw(0) + s_PP[kind][1][ab] * gw(1) + s_PP[kind][2][ab] * gw(2);
  }
  for (int t = threadIdx.x; t < kEPB * (kNN + 18); t += blockDim.x) {
    const int l = t / (kNN + 18), u = t % (kNN + 18);
    if (s_e[l] < 0) continue;
    const double* D = base + l * estride + oD;
    double* K = Ke + (int64_t)s_e[l] * kNdofe * kNdofe;
    const bool row = u < kNN;   // pressure rows of unknown u, or the pressure columns of momentum row (a, c)
    const int a = row ? u / kB : (u - kNN) / 2, s = row ? u % kB : (u - kNN) % 2;
    double v0 = 0.0, v1 = 0.0, v2 = 0.0;
    for (int q = 0; q < kQ; ++q) {
      const double* d = D + (q * kNF + (row ? f_grad(s) : 12)) * kND + (row ? 6 : 2 * s);
      const double v = d[0] * s_Dx[q][a] + d[row ? kND : 1] * s_Dy[q][a];
      v0 += v;
      v1 = fma(v, gp(q % 3), v1);
      v2 = fma(v, gp(q / 3), v2);
    }
    if (row) {
      K[kNN * kNdofe + u] = v0;
      K[(kNN + 1) * kNdofe + u] = v1;
      K[(kNN + 2) * kNdofe + u] = v2;
    } else {
      const int m = SOLID || ((s_iface[l] >> a) & 1u) ? 0 : 2;
      double* k = K + (a * kB + m + s) * kNdofe + kNN;
      k[0] = v0;
      k[1] = v1;
      k[2] = v2;
      k = K + (a * kB + 2 - m + s) * kNdofe + kNN;
      k[0] = k[1] = k[2] = 0.0;
    }
  }
  if (active && j < 9) Ke[(int64_t)e * kNdofe * kNdofe + (kNN + j / 3) * kNdofe + kNN + j % 3] = 0.0;
  // residual row j from the flux values and the test functions
  if (active) {
    const int a = j < kNN ? j / kB : 0, s = j % kB, c = s % 2;
    const bool ifc = (s_iface[le] >> a) & 1u;
    const bool mom = SOLID || ifc ? s < 2 : s >= 2;
    const int og = mom ? 2 * c : (!SOLID && !ifc ? 6 + 2 * c : -1);
    const int ov = mom ? 4 + c : (SOLID ? 6 + c : -1);
    double v = 0.0;
    for (int q = 0; q < kQ; ++q) {
      const double* vq = Vo + q * kNO;
      if (j >= kNN) {
        v += vq[10] * (j == kNN ? 1.0 : (j == kNN + 1 ? gp(q % 3) : gp(q / 3)));
      } else {
        if (og >= 0) v += vq[og] * (s_Dx[q][a] * sx) + vq[og + 1] * (s_Dy[q][a] * sy);
        if (ov >= 0) v = fma(vq[ov], s_N[q][a], v);
      }
    }
    Re[(int64_t)e * kNdofe + j] = v;
  }
  __syncthreads();

  // 4. x: item = (element, c, y pair, x pair, s): entry (node a, c) x (node b, s) of the momentum row and of the
  //    node's other row (kinematic: solid, mesh: fluid, none: interface)
  const double cu = CN ? 0.5 : 1.0, cd = CN ? -pp.idt : (TRANS ? -pp.a0 * pp.idt : 0.0);
  for (int t = threadIdx.x; t < kEPB * 648; t += blockDim.x) {
    const int l = t / 648, s = t % 4, xp = (t / 4) % 9, yp = (t / 36) % 9, c = (t / 324) % 2;
    if (s_e[l] < 0) continue;
    const double* H = base + l * estride + oH + (c * kB + s) * 108 + yp;
    double k = 0.0;
#pragma unroll
    for (int qx = 0; qx < 3; ++qx)
      k = fma(H[qx * 9], s_PP[3][qx][xp],
              fma(H[27 + qx * 9], s_PP[2][qx][xp], fma(H[54 + qx * 9], s_PP[1][qx][xp], fma(H[81 + qx * 9], s_PP[0][qx][xp], k))));
    const int a = xp / 3 + 3 * (yp / 3), b = xp % 3 + 3 * (yp % 3);
    const bool ifc = (s_iface[l] >> a) & 1u;
    double r = 0.0;
    if (SOLID) {
      if (s % 2 == c) r = s_I1[0][xp] * s_I1[0][yp] * (0.25 * s_geo[l][2] * s_geo[l][3]) * (s < 2 ? cd : cu);
    } else if (!ifc && s < 2) {
      // k = 1 / V_el cancels the element area: the reference integrals with the 2 / h scales; the transposed term
      // has its test derivative along s, its trial derivative along c
      const double gx = s_scl[l][0], gy = s_scl[l][1];
      const double xx = gx * gx * s_I1[3][xp] * s_I1[0][yp], yy = gy * gy * s_I1[0][xp] * s_I1[3][yp];
      if (s == c) r = xx + yy;
      if (pp.ale_op == 0)
        r += s == c ? (c == 0 ? xx : yy) : gx * gy * (s == 0 ? s_I1[2][xp] * s_I1[1][yp] : s_I1[1][xp] * s_I1[2][yp]);
      r *= 0.25;
    }
    double* K = Ke + (int64_t)s_e[l] * kNdofe * kNdofe + b * kB + s;
    const int m = SOLID || ifc ? 0 : 2;
    K[(a * kB + m + c) * kNdofe] = k;
    K[(a * kB + 2 - m + c) * kNdofe] = r;
  }
}

// Dirichlet rows -> identity rows; residual r_i = y_i - g_i
__global__ void k_dirichlet(const int32_t* __restrict__ dir_list, int64_t n_dir, const int32_t* __restrict__ rowptr,
                            const int32_t* __restrict__ col, double* __restrict__ val, int B,
                            const double* __restrict__ y, const double* __restrict__ g, double alpha,
                            double* __restrict__ res) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_dir) return;
  const int32_t i = dir_list[t];
  const int32_t br = i / B, ci = i % B;
  for (int32_t k = rowptr[br]; k < rowptr[br + 1]; ++k) {
    double* v = val + (int64_t)k * B * B + ci * B;
    for (int cj = 0; cj < B; ++cj) v[cj] = (col[k] == br && cj == ci) ? 1.0 : 0.0;
  }
  if (res != nullptr) res[i] = y[i] - alpha * g[i];
}

// ---------------------------------------------------------------------------
// element-wise Galerkin coarsening (2D)
// ---------------------------------------------------------------------------
namespace {
// Interpolation from the parent's three 1D nodes to the child's and its
// transpose: the weight of parent node m at the child's local node i, child side
// s, is the 1D quadratic Lagrange basis m at the parent reference coordinate
// -1 + (2 s + i) / 2, i.e. at -1, -1/2, 0 (s = 0) or 0, 1/2, 1 (s = 1):
//     s = 0:  (1, 0, 0)  (3/8, 3/4, -1/8)  (0, 1, 0)
// and s = 1 is its mirror image.  x_m = sum_i w_im x_i in place: three FP64
// operations, the weights are exact.
__device__ __forceinline__ void quarter_1d(double& x0, double& x1, double& x2, bool side) {
  const double l = fma(0.375, x1, side ? x2 : x0), m = fma(0.75, x1, side ? x0 : x2), r = -0.125 * x1;
  x0 = side ? r : l;
  x1 = m;
  x2 = side ? l : r;
}
__device__ __forceinline__ void quarter_2d(double (&v)[kNloc], int sx, int sy) {
#pragma unroll
  for (int q = 0; q < 3; ++q) quarter_1d(v[3 * q], v[3 * q + 1], v[3 * q + 2], sx != 0);
#pragma unroll
  for (int q = 0; q < 3; ++q) quarter_1d(v[q], v[q + 3], v[q + 6], sy != 0);
}
// a child's pressure (value and slopes) from the parent's, direction k's half
__device__ __forceinline__ double quarter_p(double p0, double pk, int side) {
  return fma(0.5, pk, p0 * (side ? 0.5 : -0.5));
}
__device__ __forceinline__ int row_kind(int cls, int slot) {
  if (cls == kFluid) return slot < kDim ? 2 : 0;
  return slot < kDim ? 0 : 1;
}
constexpr int kGaLd = 44;   // row stride of T: the (row, slot) lanes' 8-byte stores hit each bank once
}  // namespace

// Per child: T = A_c P_c in shared memory (straight from the child's matrix),
// then C += R_c T with C in registers.  P_c and R_c interpolate each field by the
// tensor product of the 1D weights, so a thread takes the 9 nodal values of one
// field of one row (column): 18 FP64 operations, every lane the same number
// (the 25 nonzero products of the weights took lists of 1 to 4).  T is double-
// buffered: one barrier per child.  The FP64 pipe bounds it.  The five levels
// below 65,536 elements: 1.38 ms, 3.17 with the lists.
__global__ void __launch_bounds__(256, 4)
k_galerkin_2d(int ncx, int ncy, const double* __restrict__ Kf, const int32_t* __restrict__ f_nodes,
              const uint8_t* __restrict__ f_class, const uint8_t* __restrict__ f_dir,
              const int32_t* __restrict__ c_nodes, const uint8_t* __restrict__ c_class,
              const uint8_t* __restrict__ c_dir, double* __restrict__ Kc) {
  __shared__ double sT[2][kNdofe * kGaLd];
  // index 0 .. 3: the children, 4: the coarse element
  __shared__ uint8_t msk[5][kNN], cls[5][kNloc];
  __shared__ uint8_t row[5][3][kDim][kNloc];   // row (a, slot) of a kind and component, 255: none (or Dirichlet)
  __shared__ int s_kinds;
  const int E = blockIdx.x, tid = threadIdx.x;
  const int cx = E % ncx, cy = E / ncx;
  const int fcx = 2 * ncx;
  auto child = [&](int ch) { return (2 * cx + (ch & 1)) + (int64_t)fcx * (2 * cy + (ch >> 1)); };
  if (tid == 0) s_kinds = 0;
  for (int t = tid; t < 5 * kNN; t += blockDim.x) {
    const int w = t / kNN, a = t % kNN / kB, s = t % kB;
    const int32_t nd = w == 4 ? c_nodes[(int64_t)E * kNloc + a] : f_nodes[child(w) * kNloc + a];
    msk[w][t % kNN] = (w == 4 ? c_dir : f_dir)[(int64_t)nd * kB + s] ? 0 : 1;
    if (s == 0) cls[w][a] = (w == 4 ? c_class : f_class)[nd];
  }
  __syncthreads();
  for (int t = tid; t < 5 * 3 * kDim * kNloc; t += blockDim.x) {
    const int a = t % kNloc, c = t / kNloc % kDim, kind = t / (kNloc * kDim) % 3, w = t / (kNloc * kDim * 3);
    const int sl = row_kind(cls[w][a], c) == kind ? c : (row_kind(cls[w][a], kDim + c) == kind ? kDim + c : -1);
    const bool ok = sl >= 0 && msk[w][a * kB + sl];
    row[w][kind][c][a] = (uint8_t)(ok ? a * kB + sl : 255);
    if (w == 4 && ok) atomicOr(&s_kinds, 1 << kind);
  }
  __syncthreads();
  // C += R T: thread (kind, component, J) for the unknowns, (k, J) from the other
  // end for the pressures
  const int kinds = s_kinds;
  const int J = tid % kNdofe, c = tid / kNdofe % kDim, w = tid / (kNdofe * kDim);
  int kind = 0;
  for (int n = 0; kind < 3; ++kind)
    if ((kinds >> kind) & 1 && n++ == w) break;
  const bool unk = w < 3 && kind < 3;
  const int pt = (int)blockDim.x - 1 - tid, pi = pt / 3, pk = pt % 3;   // T's pressure columns: row pi
  const int pJ = pt % kNdofe, pc = pt / kNdofe;                         // C's pressure rows: row pc
  const bool press = pt < 3 * kNdofe;
  double acc[kNloc], pacc = 0.0;
#pragma unroll
  for (int b = 0; b < kNloc; ++b) acc[b] = 0.0;
  for (int ch = 0; ch < 4; ++ch) {
    const int sx = ch & 1, sy = ch >> 1;
    const double* A = Kf + child(ch) * kNdofe * kNdofe;
    double* T = sT[ch & 1];
    if (tid < kNdofe * kB) {   // T = A P: thread (i, slot)
      const int i = tid / kB, sl = tid % kB;
      double v[kNloc];
#pragma unroll
      for (int a = 0; a < kNloc; ++a) v[a] = msk[ch][a * kB + sl] ? __ldg(A + i * kNdofe + a * kB + sl) : 0.0;
      quarter_2d(v, sx, sy);
#pragma unroll
      for (int b = 0; b < kNloc; ++b) T[i * kGaLd + b * kB + sl] = msk[4][b * kB + sl] ? v[b] : 0.0;
    }
    if (press) {
      const double* p = A + pi * kNdofe + kNN;
      T[pi * kGaLd + kNN + pk] = pk == 0 ? p[0] : quarter_p(p[0], p[pk], pk == 1 ? sx : sy);
    }
    __syncthreads();
    if (unk) {
      double v[kNloc];
#pragma unroll
      for (int a = 0; a < kNloc; ++a) {
        const int r = row[ch][kind][c][a];
        v[a] = r != 255 ? T[r * kGaLd + J] : 0.0;
      }
      quarter_2d(v, sx, sy);
#pragma unroll
      for (int b = 0; b < kNloc; ++b) acc[b] += v[b];
    }
    if (press) {
      const double p0 = T[kNN * kGaLd + pJ];
      pacc += pc == 0 ? p0 : quarter_p(p0, T[(kNN + pc) * kGaLd + pJ], pc == 1 ? sx : sy);
    }
  }
  double* C = Kc + (int64_t)E * kNdofe * kNdofe;
  if (unk)
#pragma unroll
    for (int b = 0; b < kNloc; ++b) {
      const int r = row[4][kind][c][b];
      if (r != 255) C[r * kNdofe + J] = acc[b];
    }
  if (press) C[(kNN + pc) * kNdofe + pJ] = pacc;
  for (int t = tid; t < kNN * kNdofe; t += blockDim.x)   // Dirichlet rows
    if (!msk[4][t / kNdofe]) C[t] = 0.0;
}

// ---------------------------------------------------------------------------
// 3D: element residual + Jacobian (27-node hexahedra, 166 unknowns)
// ---------------------------------------------------------------------------
namespace {
constexpr int k3Dim = 3;
constexpr int k3B = 6;
constexpr int k3Nloc = 27;
constexpr int k3NN = k3B * k3Nloc;        // 162
constexpr int k3Ndofe = k3NN + k3Dim + 1; // 166
constexpr int k3Fields = 31;              // gd 9, gu 9, u 3, d 3, p 1, u_old 3, d_old 3
constexpr int k3FieldsCN = 50;            // + (Crank-Nicolson) gd_n 31..39, gu_n 40..48, p_n 49
__device__ __forceinline__ int row_kind3(int cls, int slot) {
  if (cls == kFluid) return slot < k3Dim ? 2 : 0;
  return slot < k3Dim ? 0 : 1;
}
}  // namespace

// As in 2D, the fluxes at a quadrature point depend on the element unknowns
// only through the fields (grad d 9, grad u 9, u 3, d 3, p 1: 25 directions
// against 166 unknowns).  k_flux_3d evaluates them along the 25 directions in
// dual arithmetic (27 x 25 = 675 evaluations per element) and stores the
// derivatives and values of the 22 flux outputs; k_assemble_3d contracts them
// with the trial and test basis to the exact element Jacobian.  The flux
// derivatives (119 KB per element) pass through a global scratch, one chunk of
// elements at a time.
namespace {
constexpr int k3Q = 27;
constexpr int k3NF = 25;   // differentiated fields (fv indices 0..24)
constexpr int k3NO = 22;   // outputs: 0..8 T_ck (3 c + k) | 9..11 convection / inertia_c |
                           // solid 12..14 kinematic_c, fluid 12..20 ALE A_ck (12 + 3 c + k) | 21 mass
constexpr size_t k3FluxDoubles = (size_t)k3Q * k3NF * k3NO + (size_t)k3Q * k3NO;   // per element
constexpr int k3Chunk = 1024;                                                      // elements per pass
}  // namespace

size_t assemble_3d_scratch_doubles(int max_ne) {
  return (size_t)std::min(max_ne, k3Chunk) * k3FluxDoubles;
}

// First Piola stress of the incompressible solid (Sec. 2.2), 3D:
// P = -p J F^{-T} + 2 C1 J F - 2 C2 J F^{-T} F^{-1} F^{-T}, 2 C1 = mu_s - 2 C2
__device__ __forceinline__ void piola_3d(const Dual (&F)[3][3], const Dual (&Fi)[3][3], Dual J, Dual p,
                                         const PhysParams& pp, Dual (&P)[3][3]) {
  const Dual pJ = p * J;
  const Dual muJ = J * (pp.mu_s - 2.0 * pp.mr_c2);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < 3; ++k) P[c][k] = muJ * F[c][k] - pJ * Fi[k][c];
  if (pp.mr_c2 != 0.0) {
    Dual Q[3][3];   // F^{-1} F^{-T}
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) Q[a][b] = Fi[a][0] * Fi[b][0] + Fi[a][1] * Fi[b][1] + Fi[a][2] * Fi[b][2];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < 3; ++k)
        P[c][k] = P[c][k] - (Fi[0][c] * Q[0][k] + Fi[1][c] * Q[1][k] + Fi[2][c] * Q[2][k]) * J * (2.0 * pp.mr_c2);
  }
}

// F^{-1} and det F of a 3 x 3 Dual matrix (cofactors)
__device__ __forceinline__ Dual inv3(const Dual (&F)[3][3], Dual (&Fi)[3][3]) {
  Dual C[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, k1 = (k + 1) % 3, k2 = (k + 2) % 3;
      C[i][k] = F[i1][k1] * F[i2][k2] - F[i1][k2] * F[i2][k1];
    }
  const Dual J = F[0][0] * C[0][0] + F[0][1] * C[0][1] + F[0][2] * C[0][2];
  const double iJ = 1.0 / J.v;
  const Dual rJ = mk(iJ, -J.d * iJ * iJ);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) Fi[i][k] = C[k][i] * rJ;
  return J;
}

// fields at the 27 points, then flux values and derivatives along each field
// MODE: 0 steady, 1 BDF (yold = a1 y_n + a2 y_{n-1}), 2 Crank-Nicolson (yold = y_n)
template <bool SOLID, int MODE>
__global__ void __launch_bounds__(256)
k_flux_3d(const int32_t* __restrict__ elems, const double* __restrict__ y, const int32_t* __restrict__ elem_nodes,
          const double* __restrict__ elem_geo, int64_t n_nodes, PhysParams pp, double* __restrict__ Dg,
          int32_t* __restrict__ status) {
  constexpr bool TRANS = MODE != 0;
  constexpr bool CN = MODE == 2;
  constexpr int NFLD = CN ? k3FieldsCN : k3Fields;
  __shared__ double ye[k3Ndofe], yo[k3Ndofe];
  __shared__ double bt[k3Q][k3Nloc][4];   // physical basis: N, d/dx, d/dy, d/dz
  __shared__ double fvs[k3Q][NFLD];
  __shared__ double geo[2 * k3Dim];
  const int e = elems[blockIdx.x];
  for (int t = threadIdx.x; t < k3Ndofe; t += blockDim.x) {
    if (t < k3NN) {
      const int64_t gi = (int64_t)elem_nodes[(int64_t)e * k3Nloc + t / k3B] * k3B + t % k3B;
      ye[t] = y[gi];
      yo[t] = TRANS ? pp.yold[gi] : 0.0;
    } else {
      ye[t] = y[(n_nodes + e) * k3B + (t - k3NN)];
      yo[t] = CN ? pp.yold[(n_nodes + e) * k3B + (t - k3NN)] : 0.0;
    }
  }
  if (threadIdx.x < 2 * k3Dim) geo[threadIdx.x] = elem_geo[(int64_t)e * 2 * k3Dim + threadIdx.x];
  __syncthreads();
  const double hx = geo[3], hy = geo[4], hz = geo[5];
  const double vol = hx * hy * hz;
  const double kale = 1.0 / vol;
  for (int t = threadIdx.x; t < k3Q * k3Nloc; t += blockDim.x) {
    const int q = t / k3Nloc, a = t % k3Nloc;
    const double xi = gp(q % 3), eta = gp((q / 3) % 3), zeta = gp(q / 9);
    const int ia = a % 3, ja = (a / 3) % 3, ka = a / 9;
    const double lx = L1(ia, xi), ly = L1(ja, eta), lz = L1(ka, zeta);
    bt[q][a][0] = lx * ly * lz;
    bt[q][a][1] = dL1(ia, xi) * ly * lz * (2.0 / hx);
    bt[q][a][2] = lx * dL1(ja, eta) * lz * (2.0 / hy);
    bt[q][a][3] = lx * ly * dL1(ka, zeta) * (2.0 / hz);
  }
  __syncthreads();
  for (int it = threadIdx.x; it < k3Q * NFLD; it += blockDim.x) {
    const int q = it / NFLD, t = it % NFLD;
    double acc = 0.0;
    if (t < 18) {           // gd (t < 9) and gu: d_i / dx_k of d or u
      const int i = (t % 9) / 3, k = t % 3, off = t < 9 ? 0 : 3;
      for (int a = 0; a < k3Nloc; ++a) acc += ye[a * k3B + off + i] * bt[q][a][1 + k];
    } else if (t < 24) {    // u (18..20), d (21..23)
      const int i = (t - 18) % 3, off = t < 21 ? 3 : 0;
      for (int a = 0; a < k3Nloc; ++a) acc += ye[a * k3B + off + i] * bt[q][a][0];
    } else if (t == 24) {   // pressure
      acc = ye[k3NN] + ye[k3NN + 1] * gp(q % 3) + ye[k3NN + 2] * gp((q / 3) % 3) + ye[k3NN + 3] * gp(q / 9);
    } else if (TRANS && t < 31) {     // u_old (25..27), d_old (28..30)
      const int i = (t - 25) % 3, off = t < 28 ? 3 : 0;
      for (int a = 0; a < k3Nloc; ++a) acc += yo[a * k3B + off + i] * bt[q][a][0];
    } else if (CN && t < 49) {        // t_n gradients: d (31..39), u (40..48)
      const int tt = t - 31, i = (tt % 9) / 3, k = tt % 3, off = tt < 9 ? 0 : 3;
      for (int a = 0; a < k3Nloc; ++a) acc += yo[a * k3B + off + i] * bt[q][a][1 + k];
    } else if (CN) {                  // p_n
      acc = yo[k3NN] + yo[k3NN + 1] * gp(q % 3) + yo[k3NN + 2] * gp((q / 3) % 3) + yo[k3NN + 3] * gp(q / 9);
    }
    fvs[q][t] = acc;
  }
  __syncthreads();
  double* De = Dg + (size_t)blockIdx.x * k3FluxDoubles;   // [q][f][o], then values [q][o]
  double* Ve = De + (size_t)k3Q * k3NF * k3NO;
  bool tangled = false;
#pragma unroll 1
  for (int it = threadIdx.x; it < k3Q * k3NF; it += blockDim.x) {
    const int q = it / k3NF, f = it % k3NF;
    double* dout = De + (size_t)(q * k3NF + f) * k3NO;
    if (!TRANS && f >= 21 && f < 24) {   // d itself enters only the BDF terms
      for (int o = 0; o < k3NO; ++o) dout[o] = 0.0;
      continue;
    }
    const double* fv = fvs[q];
    const double wq = gw(q % 3) * gw((q / 3) % 3) * gw(q / 9) * vol * 0.125;
    Dual gd[3][3], u[3], ut[3], dt_[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
      for (int k = 0; k < 3; ++k) gd[i][k] = mk(fv[i * 3 + k], f == i * 3 + k ? 1.0 : 0.0);
      u[i] = mk(fv[18 + i], f == 18 + i ? 1.0 : 0.0);
      if (TRANS) {
        const Dual di = mk(fv[21 + i], f == 21 + i ? 1.0 : 0.0);
        ut[i] = (u[i] * pp.a0 + fv[25 + i]) * pp.idt;
        dt_[i] = (di * pp.a0 + fv[28 + i]) * pp.idt;
      }
    }
    const Dual p = mk(fv[24], f == 24 ? 1.0 : 0.0);
    Dual F[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) F[i][k] = i == k ? gd[i][k] + 1.0 : gd[i][k];
    Dual C[3][3];   // cofactors
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, k1 = (k + 1) % 3, k2 = (k + 2) % 3;
        C[i][k] = F[i1][k1] * F[i2][k2] - F[i1][k2] * F[i2][k1];
      }
    const Dual J = F[0][0] * C[0][0] + F[0][1] * C[0][1] + F[0][2] * C[0][2];
    if (!(J.v > 0.0)) tangled = true;
    const double iJ = 1.0 / J.v;
    const Dual rJ = mk(iJ, -J.d * iJ * iJ);   // 1 / J
    Dual Fi[3][3];   // F^{-1} = C^T / J
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) Fi[i][k] = C[k][i] * rJ;
    Dual out[k3NO];
#pragma unroll
    for (int o = 0; o < k3NO; ++o) out[o] = mk(0.0, 0.0);
    if (CN) {
      // Crank-Nicolson (Sec. 2.5), as in the 2D kernel: stresses and convection
      // averaged over t_{n+1} and t_n, conservative ALE inertia, w = (d - d_n) / dt
      Dual Fn[3][3], Fin[3][3], gw[3][3], w[3];
      double un[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        un[i] = fv[25 + i];
        w[i] = (mk(fv[21 + i], f == 21 + i ? 1.0 : 0.0) + (-fv[28 + i])) * pp.idt;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          Fn[i][k] = mk(fv[31 + 3 * i + k] + (i == k ? 1.0 : 0.0), 0.0);
          gw[i][k] = (gd[i][k] + (-fv[31 + 3 * i + k])) * pp.idt;
        }
      }
      const Dual Jn = inv3(Fn, Fin);
      if (!(Jn.v > 0.0)) tangled = true;
      const Dual pn = mk(fv[49], 0.0);
      if (SOLID) {
        Dual P1[3][3], Pn[3][3];
        piola_3d(F, Fi, J, p, pp, P1);
        piola_3d(Fn, Fin, Jn, pn, pp, Pn);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
          for (int k = 0; k < 3; ++k) out[3 * c + k] = (P1[c][k] + Pn[c][k]) * (0.5 * wq);
          out[9 + c] = (u[c] * J - Jn * un[c]) * (pp.rho_s * pp.idt * wq);
          out[12 + c] = ((u[c] + un[c]) * 0.5 - w[c]) * wq;
        }
        out[21] = (J + (-1.0)) * wq;
      } else {
        Dual gx[3][3], gxn[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const Dual gu0 = mk(fv[9 + i * 3 + 0], f == 9 + i * 3 + 0 ? 1.0 : 0.0);
            const Dual gu1 = mk(fv[9 + i * 3 + 1], f == 9 + i * 3 + 1 ? 1.0 : 0.0);
            const Dual gu2 = mk(fv[9 + i * 3 + 2], f == 9 + i * 3 + 2 ? 1.0 : 0.0);
            gx[i][k] = gu0 * Fi[0][k] + gu1 * Fi[1][k] + gu2 * Fi[2][k];
            gxn[i][k] = Fin[0][k] * fv[40 + 3 * i] + Fin[1][k] * fv[40 + 3 * i + 1] + Fin[2][k] * fv[40 + 3 * i + 2];
          }
        Dual divw1 = mk(0.0, 0.0), divwn = mk(0.0, 0.0);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            divw1 = divw1 + gw[i][k] * Fi[k][i];
            divwn = divwn + gw[i][k] * Fin[k][i];
          }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          Dual sig[3], sgn[3];
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            sig[m] = (gx[c][m] + gx[m][c]) * pp.mu_f;
            sgn[m] = (gxn[c][m] + gxn[m][c]) * pp.mu_f;
            if (m == c) {
              sig[m] = sig[m] - p;
              sgn[m] = sgn[m] - pn;
            }
          }
#pragma unroll
          for (int k = 0; k < 3; ++k)
            out[3 * c + k] = ((sig[0] * Fi[k][0] + sig[1] * Fi[k][1] + sig[2] * Fi[k][2]) * J +
                              (sgn[0] * Fin[k][0] + sgn[1] * Fin[k][1] + sgn[2] * Fin[k][2]) * Jn) * (0.5 * wq);
          const Dual conv1 = gx[c][0] * (u[0] - w[0]) + gx[c][1] * (u[1] - w[1]) + gx[c][2] * (u[2] - w[2]);
          const Dual convn = gxn[c][0] * (-w[0] + un[0]) + gxn[c][1] * (-w[1] + un[1]) + gxn[c][2] * (-w[2] + un[2]);
          const Dual val = (u[c] * J - Jn * un[c]) * pp.idt - divw1 * J * u[c] * 0.5 - divwn * Jn * (0.5 * un[c]) +
                           conv1 * J * 0.5 + convn * Jn * 0.5;
          out[9 + c] = val * (pp.rho_f * wq);
#pragma unroll
          for (int k = 0; k < 3; ++k)
            out[12 + 3 * c + k] = (pp.ale_op == 0 ? gd[c][k] + gd[k][c] : gd[c][k]) * (kale * wq);
        }
        out[21] = J * (gx[0][0] + gx[1][1] + gx[2][2]) * wq;
      }
    } else if (SOLID) {
      // P = -p J F^{-T} + 2 C1 J F - 2 C2 J F^{-T} F^{-1} F^{-T}, 2 C1 = mu_s - 2 C2
      const Dual pJ = p * J;
      const Dual muJ = J * (pp.mu_s - 2.0 * pp.mr_c2);
      Dual G[3][3];
      if (pp.mr_c2 != 0.0) {
        Dual Q[3][3];   // F^{-1} F^{-T}
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) Q[a][b] = Fi[a][0] * Fi[b][0] + Fi[a][1] * Fi[b][1] + Fi[a][2] * Fi[b][2];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int k = 0; k < 3; ++k)
            G[c][k] = (Fi[0][c] * Q[0][k] + Fi[1][c] * Q[1][k] + Fi[2][c] * Q[2][k]) * J * (2.0 * pp.mr_c2);
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int k = 0; k < 3; ++k) G[c][k] = mk(0.0, 0.0);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int k = 0; k < 3; ++k) out[3 * c + k] = (muJ * F[c][k] - pJ * Fi[k][c] - G[c][k]) * wq;
        if (TRANS) out[9 + c] = ut[c] * J * (pp.rho_s * wq);
        out[12 + c] = (TRANS ? u[c] - dt_[c] : u[c]) * wq;
      }
      out[21] = (J + (-1.0)) * wq;
    } else {
      Dual gx[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const Dual gu0 = mk(fv[9 + i * 3 + 0], f == 9 + i * 3 + 0 ? 1.0 : 0.0);
          const Dual gu1 = mk(fv[9 + i * 3 + 1], f == 9 + i * 3 + 1 ? 1.0 : 0.0);
          const Dual gu2 = mk(fv[9 + i * 3 + 2], f == 9 + i * 3 + 2 ? 1.0 : 0.0);
          gx[i][k] = gu0 * Fi[0][k] + gu1 * Fi[1][k] + gu2 * Fi[2][k];
        }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        Dual sig[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          sig[m] = (gx[c][m] + gx[m][c]) * pp.mu_f;
          if (m == c) sig[m] = sig[m] - p;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) out[3 * c + k] = (sig[0] * Fi[k][0] + sig[1] * Fi[k][1] + sig[2] * Fi[k][2]) * J * wq;
        const Dual cv = TRANS
                            ? gx[c][0] * (u[0] - dt_[0]) + gx[c][1] * (u[1] - dt_[1]) + gx[c][2] * (u[2] - dt_[2]) + ut[c]
                            : gx[c][0] * u[0] + gx[c][1] * u[1] + gx[c][2] * u[2];
        out[9 + c] = cv * J * (pp.rho_f * wq);
#pragma unroll
        for (int k = 0; k < 3; ++k)
          out[12 + 3 * c + k] = (pp.ale_op == 0 ? gd[c][k] + gd[k][c] : gd[c][k]) * (kale * wq);
      }
      out[21] = J * (gx[0][0] + gx[1][1] + gx[2][2]) * wq;
    }
#pragma unroll
    for (int o = 0; o < k3NO; ++o) dout[o] = out[o].d;
    if (f == 24) {   // any direction carries the values
#pragma unroll
      for (int o = 0; o < k3NO; ++o) Ve[q * k3NO + o] = out[o].v;
    }
  }
  if (tangled) atomicExch(&status[ST_TANGLED], 1);
}

// Element matrix from the flux derivatives, one thread block per element, by
// sum factorisation.  Every momentum entry is a sum over the 27 points of
// (test kind: value or a gradient component) x coefficient x (trial kind), and
// the Q2 basis is a product of 1D ones, so the points are contracted one
// axis at a time (z, y, x), carrying 13, 9 and 4 coefficient combinations: 18.5
// thousand fused multiply-adds per pair of components instead of the 98
// thousand of a sum over points for every entry - which is what bounds the
// kernel, as the FP64 pipe of GB300 retires two per SM and cycle.  One test
// component at a time with all six trial ones, so that a thread of the last stage
// holds the six trial components of a node pair and writes them together.
// The mesh (ALE) rows and the solid kinematic rows have constant coefficients:
// products of 1D integrals.  908,422-unknown box (16,384 elements), this kernel
// and the flux derivatives: 155.6 -> 28.6 ms on GB300.
namespace {
constexpr int kSfThreads = 256;
constexpr int kSfPP = 3 * 4 * 3 * 9;              // [axis][kind][point][3 a + b]: products of 1D bases
constexpr int kSfI = 3 * 4 * 9;                   // their integrals
constexpr int kSfC = k3Q * 24 * 4;                // [point][field][T_c0..2, body_c]
constexpr int kSfG = 6 * 9 * 9 * 9;               // [s][3 tx + rx][qx + 3 qy][zp]
constexpr int kSfH = 6 * 4 * 3 * 81;              // [s][2 tx + rx][qx][9 zp + yp]
}  // namespace

size_t assemble_3d_smem() { return (size_t)(kSfPP + kSfI + kSfC + kSfG + kSfH) * sizeof(double); }

// cu, cd: coefficients of u and d in the solid kinematic equation
template <bool SOLID>
__global__ void __launch_bounds__(kSfThreads, 2)
k_assemble_3d(const int32_t* __restrict__ elems, const int32_t* __restrict__ elem_nodes,
              const uint8_t* __restrict__ node_class, const double* __restrict__ elem_geo,
              const double* __restrict__ Dg, int ale_op, double cu, double cd, double* __restrict__ Ke,
              double* __restrict__ Re) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* PP = reinterpret_cast<double*>(smem_raw);
  double* I1 = PP + kSfPP;
  double* C = I1 + kSfI;
  double* G = C + kSfC;
  double* H = G + kSfG;
  __shared__ double V1[3][3][3][2];   // [axis][point][node]: 1D basis, derivative times 2 / h
  __shared__ unsigned s_iface;
  const int e = elems[blockIdx.x];
  const int tid = threadIdx.x;
  const double* geo = elem_geo + (int64_t)e * 2 * k3Dim + k3Dim;
  if (tid < 27) {
    const int ax = tid / 9, q = (tid / 3) % 3, a = tid % 3;
    V1[ax][q][a][0] = L1(a, gp(q));
    V1[ax][q][a][1] = dL1(a, gp(q)) * (2.0 / geo[ax]);
  }
  if (tid == 32) {
    unsigned m = 0;
    for (int a = 0; a < k3Nloc; ++a)
      if (node_class[elem_nodes[(int64_t)e * k3Nloc + a]] == kIface) m |= 1u << a;
    s_iface = m;
  }
  __syncthreads();
  // kinds: bit 1 the test (a) side is a derivative, bit 0 the trial (b) side
  for (int t = tid; t < kSfPP; t += kSfThreads) {
    const int ab = t % 9, q = (t / 9) % 3, kind = (t / 27) % 4, ax = t / 108;
    PP[t] = V1[ax][q][ab / 3][kind >> 1] * V1[ax][q][ab % 3][kind & 1];
  }
  __syncthreads();
  for (int t = tid; t < kSfI; t += kSfThreads) {
    const int ab = t % 9, kind = (t / 9) % 4, ax = t / 36;
    const double* p = PP + (ax * 4 + kind) * 27 + ab;
    const double hh = 0.5 * geo[ax];
    I1[t] = p[0] * (gw(0) * hh) + p[9] * (gw(1) * hh) + p[18] * (gw(2) * hh);
  }
  const unsigned iface = s_iface;
  const double* De = Dg + (size_t)blockIdx.x * k3FluxDoubles;
  const double* Ve = De + (size_t)k3Q * k3NF * k3NO;
  double* Kg = Ke + (int64_t)e * k3Ndofe * k3Ndofe;
  const double *PX = PP, *PY = PP + 108, *PZ = PP + 216;

  for (int c = 0; c < 3; ++c) {
    for (int t = tid; t < kSfC; t += kSfThreads) {
      const int o = t % 4, f = (t / 4) % 24, q = t / 96;
      C[t] = De[((size_t)q * k3NF + f) * k3NO + (o < 3 ? 3 * c + o : 9 + c)];
    }
    __syncthreads();
    // z: item = (trial component s, point (qx, qy), z pair)
    for (int t = tid; t < 6 * 81; t += kSfThreads) {
      const int zp = t % 9, qxy = (t / 9) % 9, s = t / 81;
      const int fv = s < 3 ? 21 + s : 15 + s, fg = 3 * s;   // value and first gradient field of s
      double g[9] = {};
#pragma unroll
      for (int qz = 0; qz < 3; ++qz) {
        const double vv = PZ[qz * 9 + zp], vd = PZ[27 + qz * 9 + zp], dv = PZ[54 + qz * 9 + zp],
                     dd = PZ[81 + qz * 9 + zp];
        const double* cq = C + (size_t)(qxy + 9 * qz) * 96;
        const double *cx = cq + fg * 4, *cy = cx + 4, *cz = cx + 8, *c0 = cq + fv * 4;
        g[0] = fma(cx[0], vv, g[0]);
        g[1] = fma(cy[0], vv, g[1]);
        g[2] = fma(cz[0], vd, g[2]);
        g[3] = fma(cx[1], vv, g[3]);
        g[4] = fma(cy[1], vv, g[4]);
        g[5] = fma(cz[1], vd, g[5]);
        g[6] = fma(cx[2], dv, fma(cx[3], vv, g[6]));
        g[7] = fma(cy[2], dv, fma(cy[3], vv, g[7]));
        g[8] = fma(cz[2], dd, fma(cz[3], vd, fma(c0[3], vv, g[8])));
      }
#pragma unroll
      for (int k = 0; k < 9; ++k) G[((s * 9 + k) * 9 + qxy) * 9 + zp] = g[k];
    }
    __syncthreads();
    // y: item = (s, qx, z pair, y pair)
    for (int t = tid; t < 6 * 3 * 81; t += kSfThreads) {
      const int zy = t % 81, yp = zy % 9, zp = zy / 9, qx = (t / 81) % 3, s = t / 243;
      double h[4] = {};
#pragma unroll
      for (int qy = 0; qy < 3; ++qy) {
        const double vv = PY[qy * 9 + yp], vd = PY[27 + qy * 9 + yp], dv = PY[54 + qy * 9 + yp],
                     dd = PY[81 + qy * 9 + yp];
        const double* gq = G + ((size_t)s * 81 + qx + 3 * qy) * 9 + zp;   // + 81 k: combination k
        h[0] = fma(gq[0], vv, h[0]);
        h[1] = fma(gq[81], vd, fma(gq[162], vv, h[1]));
        h[2] = fma(gq[243], dv, fma(gq[486], vv, h[2]));
        h[3] = fma(gq[324], dd, fma(gq[405], dv, fma(gq[567], vd, fma(gq[648], vv, h[3]))));
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) H[((s * 4 + k) * 3 + qx) * 81 + zy] = h[k];
    }
    __syncthreads();
    // x: item = (z pair, y pair, x pair) = node pair (a, b)
    for (int t = tid; t < 729; t += kSfThreads) {
      const int xp = t % 9, zy = t / 9, yp = zy % 9, zp = zy / 9;
      const int a = xp / 3 + 3 * (yp / 3) + 9 * (zp / 3), b = xp % 3 + 3 * (yp % 3) + 9 * (zp % 3);
      double k[6] = {};
#pragma unroll
      for (int qx = 0; qx < 3; ++qx) {
        const double vv = PX[qx * 9 + xp], vd = PX[27 + qx * 9 + xp], dv = PX[54 + qx * 9 + xp],
                     dd = PX[81 + qx * 9 + xp];
#pragma unroll
        for (int s = 0; s < 6; ++s) {
          const double* hq = H + (s * 12 + qx) * 81 + zy;   // + 243 k: combination k
          k[s] = fma(hq[0], dd, fma(hq[243], dv, fma(hq[486], vd, fma(hq[729], vv, k[s]))));
        }
      }
      const bool ifc = (iface >> a) & 1u;
      // momentum sits in the d-row of solid and interface nodes, in the u-row of fluid ones
      double2* mrow = reinterpret_cast<double2*>(Kg + (a * k3B + (SOLID || ifc ? 0 : 3) + c) * k3Ndofe + b * k3B);
      mrow[0] = make_double2(k[0], k[1]);
      mrow[1] = make_double2(k[2], k[3]);
      mrow[2] = make_double2(k[4], k[5]);
      // the node's other row: kinematic (solid), nothing (interface), ALE (fluid)
      const double *ix = I1 + xp, *iy = I1 + 36 + yp, *iz = I1 + 72 + zp;   // + 9 kind
      double r[6] = {};
      if (SOLID) {
        const double m = ix[0] * iy[0] * iz[0];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          r[s] = s == c ? m * cd : 0.0;
          r[3 + s] = s == c ? m * cu : 0.0;
        }
      } else if (!ifc) {
        const double kale = 1.0 / (geo[0] * geo[1] * geo[2]);
        const double lap = ix[27] * iy[0] * iz[0] + ix[0] * iy[27] * iz[0] + ix[0] * iy[0] * iz[27];
        // the transposed term: test derivative along s, trial derivative along c
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          double v = s == c ? lap : 0.0;
          if (ale_op == 0) {
            const int k0 = (s == 0 ? 2 : 0) + (c == 0 ? 1 : 0), k1 = (s == 1 ? 2 : 0) + (c == 1 ? 1 : 0),
                      k2 = (s == 2 ? 2 : 0) + (c == 2 ? 1 : 0);
            v += ix[9 * k0] * iy[9 * k1] * iz[9 * k2];
          }
          r[s] = v * kale;
        }
      }
      double2* orow = reinterpret_cast<double2*>(Kg + (a * k3B + (SOLID || ifc ? 3 : 0) + c) * k3Ndofe + b * k3B);
      orow[0] = make_double2(r[0], r[1]);
      orow[1] = make_double2(r[2], r[3]);
      orow[2] = make_double2(r[4], r[5]);
    }
    __syncthreads();
  }
  // pressure rows and columns and the residual, point by point with the nine
  // points of a z layer per item; partial sums of the layers added afterwards
  double* bt = G;   // [point][node]: N, d/dx, d/dy, d/dz
  for (int t = tid; t < k3Q * k3Nloc; t += kSfThreads) {
    const int q = t / k3Nloc, a = t % k3Nloc;
    const double *x = V1[0][q % 3][a % 3], *y = V1[1][(q / 3) % 3][(a / 3) % 3], *z = V1[2][q / 9][a / 9];
    const double yz = y[0] * z[0];
    bt[t * 4] = x[0] * yz;
    bt[t * 4 + 1] = x[1] * yz;
    bt[t * 4 + 2] = x[0] * y[1] * z[0];
    bt[t * 4 + 3] = x[0] * y[0] * z[1];
  }
  __syncthreads();
  double *pc = H, *pr = pc + 243 * 4, *rs = pr + 486 * 4;   // partial sums: pressure columns, rows, residual
  for (int t = tid; t < 243 + 486 + 486 + 12; t += kSfThreads) {
    if (t < 243) {
      const int ac = t % 81, a = ac / 3, c = ac % 3, qz = t / 81;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0;
      for (int q = 9 * qz; q < 9 * qz + 9; ++q) {
        const double* d = De + ((size_t)q * k3NF + 24) * k3NO + 3 * c;
        const double* w = bt + (q * k3Nloc + a) * 4;
        const double v = d[0] * w[1] + d[1] * w[2] + d[2] * w[3];
        s0 += v;
        s1 = fma(v, gp(q % 3), s1);
        s2 = fma(v, gp((q / 3) % 3), s2);
      }
      pc[t * 4] = s0;
      pc[t * 4 + 1] = s1;
      pc[t * 4 + 2] = s2;
      pc[t * 4 + 3] = s0 * gp(qz);
    } else if (t < 729) {
      const int u = t - 243, bs = u % 162, b = bs / 6, s = bs % 6, qz = u / 162;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0;
      for (int q = 9 * qz; q < 9 * qz + 9; ++q) {
        const double* d = De + ((size_t)q * k3NF + 3 * s) * k3NO + 21;
        const double* w = bt + (q * k3Nloc + b) * 4;
        const double v = d[0] * w[1] + d[k3NO] * w[2] + d[2 * k3NO] * w[3];
        s0 += v;
        s1 = fma(v, gp(q % 3), s1);
        s2 = fma(v, gp((q / 3) % 3), s2);
      }
      pr[u * 4] = s0;
      pr[u * 4 + 1] = s1;
      pr[u * 4 + 2] = s2;
      pr[u * 4 + 3] = s0 * gp(qz);
    } else if (t < 1215) {
      const int u = t - 729, j = u % 162, a = j / 6, s = j % 6, c = s % 3, qz = u / 162;
      const bool ifc = (iface >> a) & 1u;
      // momentum (outputs 3 c .. with body 9 + c), ALE (12 + 3 c ..), kinematic (12 + c) or no row
      const bool mom = SOLID || ifc ? s < 3 : s >= 3;
      const int og = mom ? 3 * c : (!SOLID && !ifc ? 12 + 3 * c : -1);
      const int ov = mom ? 9 + c : (SOLID ? 12 + c : -1);
      double v = 0.0;
      for (int q = 9 * qz; q < 9 * qz + 9; ++q) {
        const double* d = Ve + (size_t)q * k3NO;
        const double* w = bt + (q * k3Nloc + a) * 4;
        if (og >= 0) v += d[og] * w[1] + d[og + 1] * w[2] + d[og + 2] * w[3];
        if (ov >= 0) v = fma(d[ov], w[0], v);
      }
      rs[u] = v;
    } else {
      const int u = t - 1215, pk = u % 4, qz = u / 4;
      double v = 0.0;
      for (int q = 9 * qz; q < 9 * qz + 9; ++q)
        v += Ve[(size_t)q * k3NO + 21] * (pk == 0 ? 1.0 : (pk == 1 ? gp(q % 3) : (pk == 2 ? gp((q / 3) % 3) : gp(qz))));
      rs[486 + u] = v;
    }
  }
  __syncthreads();
  for (int t = tid; t < 324 + 648 + 166 + 16; t += kSfThreads) {
    if (t < 324) {
      const int pk = t % 4, ac = t / 4, a = ac / 3, c = ac % 3;
      const double v = pc[ac * 4 + pk] + pc[(81 + ac) * 4 + pk] + pc[(162 + ac) * 4 + pk];
      const int m = SOLID || ((iface >> a) & 1u) ? 0 : 3;
      Kg[(a * k3B + m + c) * k3Ndofe + k3NN + pk] = v;
      Kg[(a * k3B + 3 - m + c) * k3Ndofe + k3NN + pk] = 0.0;
    } else if (t < 972) {
      const int u = t - 324, bs = u % 162, pk = u / 162;
      Kg[(k3NN + pk) * k3Ndofe + bs] = pr[bs * 4 + pk] + pr[(162 + bs) * 4 + pk] + pr[(324 + bs) * 4 + pk];
    } else if (t < 1138) {
      const int j = t - 972;
      Re[(int64_t)e * k3Ndofe + j] = j < k3NN ? rs[j] + rs[162 + j] + rs[324 + j]
                                              : rs[486 + j - k3NN] + rs[490 + j - k3NN] + rs[494 + j - k3NN];
    } else {
      const int u = t - 1138;
      Kg[(k3NN + u / 4) * k3Ndofe + k3NN + u % 4] = 0.0;
    }
  }
}

// Element-wise Galerkin coarsening in 3D.  Per child: T = A_c P_c is formed in
// shared memory from the child's matrix (global, row-major), then the coarse
// element matrix (global, accumulated over the 8 children) gets R_c T.  P_c and
// R_c interpolate each of the fields by the tensor product of the 1D table, so a
// thread takes the 27 nodal values of one field of one row (column) in registers
// and applies the three 1D interpolations in turn: 81 FP64 operations, against
// 125 for the nonzero products of the three tables, and every lane the same
// number of them.  FP64 and the loads ahead of it bound it (one block of 512
// threads per SM: T takes the shared memory).  The two coarse
// levels below 900,000 unknowns: 9.2 ms, 21.1 with lists of the nonzero products.
size_t galerkin_3d_smem() { return (size_t)k3Ndofe * k3Ndofe * sizeof(double); }

namespace {
__device__ __forceinline__ void quarter_3d(double (&v)[k3Nloc], int sx, int sy, int sz) {
#pragma unroll
  for (int q = 0; q < 9; ++q) quarter_1d(v[3 * q], v[3 * q + 1], v[3 * q + 2], sx != 0);
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const int o = q / 3 * 9 + q % 3;
    quarter_1d(v[o], v[o + 3], v[o + 6], sy != 0);
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) quarter_1d(v[q], v[q + 9], v[q + 18], sz != 0);
}
}  // namespace

__global__ void __launch_bounds__(512)
k_galerkin_3d(int ncx, int ncy, int ncz, const double* __restrict__ Kf, const int32_t* __restrict__ f_nodes,
              const uint8_t* __restrict__ f_class, const uint8_t* __restrict__ f_dir,
              const int32_t* __restrict__ c_nodes, const uint8_t* __restrict__ c_class,
              const uint8_t* __restrict__ c_dir, double* __restrict__ Kc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* T = reinterpret_cast<double*>(smem_raw);   // [i][J]
  // row (a, slot) of a row kind and component at a node, 255: none (another
  // kind, or a Dirichlet row)
  __shared__ uint8_t f_row[3][k3Dim][k3Nloc], c_row[3][k3Dim][k3Nloc];
  __shared__ uint8_t c_msk[k3NN], f_msk[k3NN];
  __shared__ int s_kinds;
  const int E = blockIdx.x;
  const int cx = E % ncx, cy = (E / ncx) % ncy, cz = E / (ncx * ncy);
  const int fcx = 2 * ncx, fcy = 2 * ncy;
  (void)ncz;
  double* C = Kc + (int64_t)E * k3Ndofe * k3Ndofe;
  for (int t = threadIdx.x; t < k3Ndofe * k3Ndofe; t += blockDim.x) C[t] = 0.0;
  if (threadIdx.x == 0) s_kinds = 0;
  __syncthreads();
  // per node, kind and component: each kind has at most one slot there
  auto row_of = [](const uint8_t* msk, int cls, int kind, int c, int a) {
    const int sl = row_kind3(cls, c) == kind ? c : (row_kind3(cls, k3Dim + c) == kind ? k3Dim + c : -1);
    return (uint8_t)(sl >= 0 && msk[a * k3B + sl] ? a * k3B + sl : 255);
  };
  auto tables = [&](const int32_t* nodes, const uint8_t* cls, const uint8_t* dir, uint8_t* msk,
                    uint8_t (&row)[3][k3Dim][k3Nloc], bool coarse) {
    if (threadIdx.x < k3NN)
      msk[threadIdx.x] = dir[(int64_t)nodes[threadIdx.x / k3B] * k3B + threadIdx.x % k3B] ? 0 : 1;
    __syncthreads();
    if (threadIdx.x < 3 * k3NN / 2) {
      const int a = threadIdx.x % k3Nloc, c = threadIdx.x / k3Nloc % k3Dim, kind = threadIdx.x / (k3Nloc * k3Dim);
      row[kind][c][a] = row_of(msk, cls[nodes[a]], kind, c, a);
      if (coarse && row[kind][c][a] != 255) atomicOr(&s_kinds, 1 << kind);
    }
    __syncthreads();
  };
  tables(c_nodes + (int64_t)E * k3Nloc, c_class, c_dir, c_msk, c_row, true);
  const int kinds = s_kinds, nk = __popc(kinds);
  for (int ch = 0; ch < 8; ++ch) {
    const int sx = ch & 1, sy = (ch >> 1) & 1, sz = ch >> 2;
    const int64_t ef = (2 * cx + sx) + (int64_t)fcx * ((2 * cy + sy) + (int64_t)fcy * (2 * cz + sz));
    const double* A = Kf + ef * k3Ndofe * k3Ndofe;
    tables(f_nodes + ef * k3Nloc, f_class, f_dir, f_msk, f_row, false);
    // T = A P: thread (i, slot)
    for (int t = threadIdx.x; t < k3Ndofe * k3B; t += blockDim.x) {
      const int i = t / k3B, sl = t % k3B;
      const double* Ai = A + (int64_t)i * k3Ndofe + sl;
      double v[k3Nloc];
#pragma unroll
      for (int a = 0; a < k3Nloc; ++a) v[a] = f_msk[a * k3B + sl] ? __ldg(Ai + a * k3B) : 0.0;
      quarter_3d(v, sx, sy, sz);
      double* Ti = T + i * k3Ndofe + sl;
#pragma unroll
      for (int b = 0; b < k3Nloc; ++b) Ti[b * k3B] = c_msk[b * k3B + sl] ? v[b] : 0.0;
    }
    for (int t = threadIdx.x; t < k3Ndofe * 4; t += blockDim.x) {
      const int i = t / 4, k = t % 4;
      const double* Ai = A + (int64_t)i * k3Ndofe + k3NN;
      T[i * k3Ndofe + k3NN + k] = k == 0 ? Ai[0] : quarter_p(Ai[0], Ai[k], k == 1 ? sx : (k == 2 ? sy : sz));
    }
    __syncthreads();
    // C += R T: thread (kind, component, J); each row of C has one kind
    for (int t = threadIdx.x; t < nk * k3Dim * k3Ndofe; t += blockDim.x) {
      const int J = t % k3Ndofe, c = t / k3Ndofe % k3Dim, w = t / (k3Ndofe * k3Dim);
      int kind = 0;
      for (int n = 0; kind < 3; ++kind)
        if ((kinds >> kind) & 1 && n++ == w) break;
      double v[k3Nloc];
#pragma unroll
      for (int a = 0; a < k3Nloc; ++a) {
        const int r = f_row[kind][c][a];
        v[a] = r != 255 ? T[r * k3Ndofe + J] : 0.0;
      }
      quarter_3d(v, sx, sy, sz);
#pragma unroll
      for (int b = 0; b < k3Nloc; ++b) {
        const int r = c_row[kind][c][b];
        if (r != 255) C[r * k3Ndofe + J] += v[b];
      }
    }
    for (int t = threadIdx.x; t < 4 * k3Ndofe; t += blockDim.x) {
      const int k = t / k3Ndofe, J = t % k3Ndofe;
      const double p0 = T[k3NN * k3Ndofe + J];
      C[(k3NN + k) * k3Ndofe + J] +=
          k == 0 ? p0 : quarter_p(p0, T[(k3NN + k) * k3Ndofe + J], k == 1 ? sx : (k == 2 ? sy : sz));
    }
    __syncthreads();   // T is free again
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
bool launch_assemble_2d(bool solid, const int32_t* elems, int ne, const double* y, const int32_t* elem_nodes,
                        const uint8_t* node_class, const double* elem_geo, int64_t n_nodes, PhysParams pp,
                        double* Ke, double* Re, int32_t* status, double* scratch, int scratch_ne, cudaStream_t st) {
  (void)scratch;
  (void)scratch_ne;
  if (ne <= 0) return true;
  const int grid = (ne + kEPB - 1) / kEPB;
  const size_t smem = (size_t)kEPB * asm_elem_doubles(pp.transient == 2 ? kNFVcn : kNFV) * sizeof(double);
  auto go = [&](auto kern) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<grid, kEPB * kNdofe, smem, st>>>(elems, ne, y, elem_nodes, node_class, elem_geo, n_nodes, pp, Ke, Re,
                                           status);
  };
  if (solid) {
    if (pp.transient == 2) go(k_assemble_2d<true, 2>);
    else if (pp.transient) go(k_assemble_2d<true, 1>);
    else go(k_assemble_2d<true, 0>);
  } else {
    if (pp.transient == 2) go(k_assemble_2d<false, 2>);
    else if (pp.transient) go(k_assemble_2d<false, 1>);
    else go(k_assemble_2d<false, 0>);
  }
  return true;
}

// Deterministic gather of the element matrices into the block-sparse values
// and of the element residuals into the residual: one thread per matrix
// entry (or residual entry) sums its element contributions in list order
// (colour-group order, the order of a coloured scatter into zeroed arrays)
// and writes the entry once; padding entries of the pressure blocks get 0.
template <int NLOC, int B, int NDOFE>
__global__ void __launch_bounds__(256) k_gather_blocks(int64_t nnzb, const int32_t* __restrict__ ptr,
                                                       const int32_t* __restrict__ src,
                                                       const double* __restrict__ Ke, double* __restrict__ val) {
  constexpr int NN = NLOC * B, NP = NDOFE - NN, NL1 = NLOC + 1;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nnzb * B * B) return;
  const int64_t blk = t / (B * B);
  const int ij = (int)(t % (B * B)), ci = ij / B, cj = ij % B;
  double v = 0.0;
  const int32_t q1 = ptr[blk + 1];
  for (int32_t q = ptr[blk]; q < q1; ++q) {
    const int32_t sq = src[q];
    const int e = sq / (NL1 * NL1), ab = sq % (NL1 * NL1), a = ab / NL1, b = ab % NL1;
    const int i = a < NLOC ? a * B + ci : (ci < NP ? NN + ci : -1);
    const int j = b < NLOC ? b * B + cj : (cj < NP ? NN + cj : -1);
    if (i >= 0 && j >= 0) v += Ke[(int64_t)e * NDOFE * NDOFE + i * NDOFE + j];
  }
  val[t] = v;
}

template <int NLOC, int B, int NDOFE>
__global__ void __launch_bounds__(256) k_gather_res(int64_t nb, const int32_t* __restrict__ ptr,
                                                    const int32_t* __restrict__ src, const double* __restrict__ Re,
                                                    double* __restrict__ res) {
  constexpr int NN = NLOC * B, NP = NDOFE - NN, NL1 = NLOC + 1;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nb * B) return;
  const int64_t r = t / B;
  const int ci = (int)(t % B);
  double v = 0.0;
  const int32_t q1 = ptr[r + 1];
  for (int32_t q = ptr[r]; q < q1; ++q) {
    const int32_t sq = src[q];
    const int e = sq / NL1, a = sq % NL1;
    const int i = a < NLOC ? a * B + ci : (ci < NP ? NN + ci : -1);
    if (i >= 0) v += Re[(int64_t)e * NDOFE + i];
  }
  res[t] = v;
}

void launch_gather_elements(int dim, int64_t nnzb, const int32_t* blk_ptr, const int32_t* blk_src, const double* Ke,
                            double* val, int64_t nb, const int32_t* res_ptr, const int32_t* res_src,
                            const double* Re, double* res, cudaStream_t st) {
  if (dim == 2) {
    k_gather_blocks<kNloc, kB, kNdofe><<<(unsigned)((nnzb * kB * kB + 255) / 256), 256, 0, st>>>(nnzb, blk_ptr,
                                                                                              blk_src, Ke, val);
    if (res)
      k_gather_res<kNloc, kB, kNdofe><<<(unsigned)((nb * kB + 255) / 256), 256, 0, st>>>(nb, res_ptr, res_src, Re,
                                                                                        res);
  } else {
    k_gather_blocks<k3Nloc, k3B, k3Ndofe><<<(unsigned)((nnzb * k3B * k3B + 255) / 256), 256, 0, st>>>(
        nnzb, blk_ptr, blk_src, Ke, val);
    if (res)
      k_gather_res<k3Nloc, k3B, k3Ndofe><<<(unsigned)((nb * k3B + 255) / 256), 256, 0, st>>>(nb, res_ptr, res_src,
                                                                                            Re, res);
  }
}

void launch_dirichlet(const int32_t* dir_list, int64_t n_dir, const int32_t* rowptr, const int32_t* col, double* val,
                      int B, const double* y, const double* g, double alpha, double* res, cudaStream_t st) {
  if (n_dir <= 0) return;
  k_dirichlet<<<(unsigned)((n_dir + 255) / 256), 256, 0, st>>>(dir_list, n_dir, rowptr, col, val, B, y, g, alpha,
                                                               res);
}

void launch_galerkin_2d(int ncx, int ncy, const double* Kf, const int32_t* f_nodes, const uint8_t* f_class,
                        const uint8_t* f_dir, const int32_t* c_nodes, const uint8_t* c_class, const uint8_t* c_dir,
                        double* Kc, cudaStream_t st) {
  k_galerkin_2d<<<ncx * ncy, 256, 0, st>>>(ncx, ncy, Kf, f_nodes, f_class, f_dir, c_nodes, c_class, c_dir, Kc);
}

}  // namespace fsi

namespace fsi {

bool launch_assemble_3d(bool solid, const int32_t* elems, int ne, const double* y, const int32_t* elem_nodes,
                        const uint8_t* node_class, const double* elem_geo, int64_t n_nodes, PhysParams pp,
                        double* Ke, double* Re, int32_t* status, double* scratch, int scratch_ne, cudaStream_t st) {
  if (ne <= 0) return true;
  if (std::min(ne, k3Chunk) > scratch_ne) return false;   // the flux scratch holds scratch_ne elements
  const size_t smem = assemble_3d_smem();
  // solid kinematic equation: u, u - (a0 d + history) / dt, (u + u_n) / 2 - (d - d_n) / dt
  const double cu = pp.transient == 2 ? 0.5 : 1.0;
  const double cd = pp.transient == 2 ? -pp.idt : (pp.transient ? -pp.a0 * pp.idt : 0.0);
  auto go = [&](auto flux, auto cols) {
    cudaFuncSetAttribute(cols, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    for (int e0 = 0; e0 < ne; e0 += k3Chunk) {
      const int nc = std::min(k3Chunk, ne - e0);
      flux<<<nc, 256, 0, st>>>(elems + e0, y, elem_nodes, elem_geo, n_nodes, pp, scratch, status);
      cols<<<nc, kSfThreads, smem, st>>>(elems + e0, elem_nodes, node_class, elem_geo, scratch, pp.ale_op, cu, cd, Ke,
                                         Re);
    }
  };
  if (solid) {
    if (pp.transient == 2) go(k_flux_3d<true, 2>, k_assemble_3d<true>);
    else if (pp.transient) go(k_flux_3d<true, 1>, k_assemble_3d<true>);
    else go(k_flux_3d<true, 0>, k_assemble_3d<true>);
  } else {
    if (pp.transient == 2) go(k_flux_3d<false, 2>, k_assemble_3d<false>);
    else if (pp.transient) go(k_flux_3d<false, 1>, k_assemble_3d<false>);
    else go(k_flux_3d<false, 0>, k_assemble_3d<false>);
  }
  return true;
}

// FP64 operations executed per element (2 per DFMA, 1 per DMUL / DADD) by the
// element-matrix kernels, counted with ncu on GB300 (sm_103a build of these
// kernels) for each dimension, material and time discretisation (0 steady,
// 1 BDF, 2 Crank-Nicolson; Mooney-Rivlin adds a few percent in the solid);
// used for the FP64-ALU fraction of the assembly in the per-class timings.
double assemble_flops_per_element(int dim, bool solid, int mode) {
  static const double f2[2][3] = {{58243.0, 66127.0, 100480.0}, {44932.0, 51325.0, 63655.0}};
  // 3D: flux derivatives + sums over the quadrature points
  static const double f3[2][3] = {{437386.0 + 839713.0, 531264.0 + 839713.0, 1057143.0 + 839713.0},
                                  {242395.0 + 770633.0, 313568.0 + 770633.0, 502742.0 + 770633.0}};
  mode = mode < 0 ? 0 : (mode > 2 ? 2 : mode);
  return dim == 2 ? f2[solid][mode] : f3[solid][mode];
}
// the same count for the Galerkin kernels, per coarse element away from the
// fluid-solid interface, from their loops: 1D interpolations of 5 operations, the
// sums over the children and the pressures
double galerkin_flops_per_coarse_element(int dim) {
  const double rows = dim == 2 ? kNdofe : k3Ndofe, fields = dim == 2 ? kB : k3B, nodes = dim == 2 ? kNloc : k3Nloc;
  const double line = dim == 2 ? 6 * 5 : 27 * 5;   // of one field's values
  const double child = rows * fields * (2 * line + nodes) + rows * (dim * 3 + 1 + dim * 4);
  return (dim == 2 ? 4 : 8) * child;
}

int assemble_launches(int dim, int ne) { return dim == 2 || ne <= 0 ? (ne > 0) : 2 * ((ne + k3Chunk - 1) / k3Chunk); }

void launch_galerkin_3d(int ncx, int ncy, int ncz, const double* Kf, const int32_t* f_nodes, const uint8_t* f_class,
                        const uint8_t* f_dir, const int32_t* c_nodes, const uint8_t* c_class, const uint8_t* c_dir,
                        double* Kc, cudaStream_t st) {
  const size_t smem = galerkin_3d_smem();
  cudaFuncSetAttribute(k_galerkin_3d, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_galerkin_3d<<<ncx * ncy * ncz, 512, smem, st>>>(ncx, ncy, ncz, Kf, f_nodes, f_class, f_dir, c_nodes, c_class,
                                                     c_dir, Kc);
}

}  // namespace fsi
