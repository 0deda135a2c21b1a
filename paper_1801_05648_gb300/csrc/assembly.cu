// Residual and Jacobian of the monolithic ALE fluid-structure system on the GPU
// (the Newton step of Alg. 1, Sec. 3.3; variational form Eq. (fsi:all) with the
// strong form of Sec. 2), on the structured Q2/Q2/Q1 box meshes the solver is
// benchmarked on.  Declarations and the data contract are in include/fsi.h
// (fsi_asm_*).
//
// Per cell and quadrature point, with F = I + grad u, J = det F, A = grad(v) F^-1,
// X = J (mu (A + A^T) dtt - p I), mu = rho_f nu_f, dtt = dt theta, dto = dt (1 - theta),
// J^theta = theta J + (1 - theta) J_old:
//   fluid cells   f0 = rho_f [J^theta (v - v_old) - J A (u - u_old) + dtt J A v + dto J_old A_old v_old]
//                 f1 = X F^-T + dto J_old sigma_v,old F_old^-T     f0 tested with phi, f1 with grad phi
//                 g0 = J tr(A)                                     tested with psi (pressure)
//                 hm = grad(u) / J                                 tested with grad phi on mesh rows
//   solid cells   f0 = rho_s (v - v_old),  f1 = dtt F Sigma (+ dto F_old Sigma_old),
//                 Sigma = 2 mu_s E + lambda_s tr(E) I,  E = (F^T F - I) / 2
//                 k0 = (u - u_old) - dtt v (- dto v_old)           tested with phi on u rows
//   outflow face  c = -dtt mu J A^T n', n' = F^-T e_0 (theta < 1 adds the previous level's
//   (fluid cells on x_0 = L_0)  term weighted dto)                 tested with phi on v rows
// The Jacobian is the exact derivative of this discrete residual, in closed form.  With
// the deformed gradient G_b = F^-T grad phi_b of the trial function b, s_b = G_b . c,
// c = dtt v - (u - u_old), the variations along component k of v or u at node b are
//   dv:  dA_ij = delta_ik G_bj
//        df0_i = delta_ik rho_f (J^theta phi_b + J s_b) + rho_f dtt J A_ik phi_b
//        df1_ij = J dtt mu (delta_ik (F^-1 G_b)_j + G_bi F^-1_jk),          dg0 = J G_bk
//   du:  dJ = J G_bk,  dA_ij = -A_ik G_bj,  dF^-1_jl = -F^-1_jk G_bl
//        df0_i = G_bk rho_f J [theta (v - v_old) + A c]_i - A_ik rho_f J (s_b + phi_b)
//        df1_ij = G_bk (X F^-T)_ij - (X G_b)_i F^-1_jk - J dtt mu (A_ik (F^-1 G_b)_j + G_bi (F^-1 A)_jk)
//        dg0 = J (G_bk tr A - (A^T G_b)_k),  dhm_ij = (delta_ik d_j phi_b - (grad u)_ij G_bk) / J
//   solid du: df1_ij = dtt [delta_ik (Sigma grad phi_b)_j + mu_s ((F F^T)_ik d_j phi_b + (F grad phi_b)_i F_kj)
//                           + lambda_s (F grad phi_b)_k F_ij];  the mass terms are the same for every cell
//
// The GB300 retires 1.7 FP64 FMAs per clock and SM, so FP64 instructions are what an
// assembly costs and the work is split to need few of them (see k_jacobian).  Cells are
// launched colour by colour (the parities of their lattice coordinates): two cells of one
// colour share no node, so the in-place additions never race, and the order in
// which contributions reach an entry is fixed (deterministic, no atomics on values).
#include "../../include/fsi.h"
#include "common.cuh"

#include <cmath>
#include <cstring>
#include <vector>

namespace fsi {
namespace {

// Element shape: PD = 0 continuous Q1 pressure (2^D vertex functions), PD = 1 the
// discontinuous P1 pressure of the paper's Q2-Q2-P1disc pair (D + 1 functions per cell).
template <int D, int PD> struct Sh;
template <int PD> struct Sh<2, PD> {
  static constexpr int NQ2 = 9, NQ1 = PD ? 3 : 4, NL = 36 + NQ1, NQP = 9, NFP = 3;
  static constexpr int JCELLS = 8;    // most cells per CTA of the Jacobian: 36 units of a kind per cell,
  static constexpr int JTHREADS = 288;   // 288 in all, one per thread
  static constexpr int RCELLS = 28;   // ... of the residual: 252 of 256 threads hold a point
};
template <int PD> struct Sh<3, PD> {
  static constexpr int NQ2 = 27, NQ1 = PD ? 4 : 8, NL = 162 + NQ1, NQP = 27, NFP = 9;
  static constexpr int JCELLS = 1, JTHREADS = 256;   // 243 units of a kind per cell
  static constexpr int RCELLS = 4;
};
constexpr int kAsmThreads = 256;

// Quadrature tables of one mesh (reference cell scaled by the cell size h).
struct Tables {
  const double* N;    // [NQP][NQ2]
  const double* dN;   // [NQP][NQ2][D]
  const double* Np;   // [NQP][NQ1]
  const double* w;    // [NQP]
  const double* Nf;   // [NFP][NQ2]   outflow face x_0 = 1 of the reference cell
  const double* dNf;  // [NFP][NQ2][D]
  const double* wf;   // [NFP]
  const double* M;    // [NQ2][NQ2]   sum_q w N_a N_b
};
// 1D factors of the Q2 basis at the three Gauss points: the basis function with lattice
// index (a_0, a_1, a_2) is the product of N[q_d][a_d], its derivative along direction d
// takes dN[d][q_d][a_d] there.  Kernel parameters, so FMAs read them as constants.
struct Basis1 {
  double N[3][3];
  double dN[3][3][3];
};

struct Phys {
  double rho_f, nu_f, mu_s, lambda_s, rho_s, dt, theta;
};

struct CellGeom {
  int n[3];           // cells per direction
  int color;          // parity pattern of the launched cells
  int m[3];           // cells of this colour per direction
};

template <int D>
__device__ __forceinline__ int64_t colour_cell(const CellGeom& g, int64_t k, int* c) {
  int64_t r = k;
  for (int d = 0; d < D; ++d) {
    const int i = (int)(r % g.m[d]);
    r /= g.m[d];
    c[d] = 2 * i + ((g.color >> d) & 1);
  }
  int64_t idx = c[D - 1];
  for (int d = D - 2; d >= 0; --d) idx = idx * g.n[d] + c[d];
  return idx;
}

template <int D>
__device__ __forceinline__ double det(const double (&F)[D][D]) {
  if constexpr (D == 2) return F[0][0] * F[1][1] - F[0][1] * F[1][0];
  else
    return F[0][0] * (F[1][1] * F[2][2] - F[1][2] * F[2][1]) - F[0][1] * (F[1][0] * F[2][2] - F[1][2] * F[2][0]) +
           F[0][2] * (F[1][0] * F[2][1] - F[1][1] * F[2][0]);
}
// F^-1 = cof(F)^T / J
template <int D>
__device__ __forceinline__ void invert(const double (&F)[D][D], double iJ, double (&R)[D][D]) {
  if constexpr (D == 2) {
    R[0][0] = F[1][1] * iJ; R[0][1] = -F[0][1] * iJ;
    R[1][0] = -F[1][0] * iJ; R[1][1] = F[0][0] * iJ;
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int j1 = (j + 1) % 3, j2 = (j + 2) % 3, i1 = (i + 1) % 3, i2 = (i + 2) % 3;
        R[i][j] = (F[j1][i1] * F[j2][i2] - F[j1][i2] * F[j2][i1]) * iJ;   // cofactor_ji / J
      }
  }
}
// C = A B
template <int D>
__device__ __forceinline__ void matmul(const double (&A)[D][D], const double (&B)[D][D], double (&C)[D][D]) {
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) {
      double s = A[i][0] * B[0][j];
#pragma unroll
      for (int k = 1; k < D; ++k) s += A[i][k] * B[k][j];
      C[i][j] = s;
    }
}
// C = A B^T
template <int D>
__device__ __forceinline__ void matmul_t(const double (&A)[D][D], const double (&B)[D][D], double (&C)[D][D]) {
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) {
      double s = A[i][0] * B[j][0];
#pragma unroll
      for (int k = 1; k < D; ++k) s += A[i][k] * B[j][k];
      C[i][j] = s;
    }
}

// Doubles that order as unsigned 64-bit integers (for atomicMin on min det F).
__host__ __device__ inline unsigned long long order_key(double x) {
#ifdef __CUDA_ARCH__
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long b;
  std::memcpy(&b, &x, 8);
#endif
  return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}
inline double order_value(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? k & 0x7FFFFFFFFFFFFFFFull : ~k;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}

// Scalars at a point, in the order they are interpolated: v (D), u (D), grad v (D x D),
// grad u (D x D), then of the previous level v (D), u (D) and, for theta < 1, grad u, grad v.
template <int D>
struct Raw {
  static constexpr int v = 0, u = D, Gv = 2 * D, Gu = 2 * D + D * D, vo = 2 * D + 2 * D * D, uo = vo + D,
                       Guo = uo + D, Gvo = Guo + D * D, kNow = Guo, kAll = Gvo + D * D;
};

// Quantity r of point pt (of the face when face) of an element with values U and Uold.
template <int D, int PD>
__device__ __forceinline__ double interpolate(const Tables& T, bool face, int pt, int r, const double* U,
                                              const double* Uo) {
  constexpr int NQ2 = Sh<D, PD>::NQ2;
  const double* N = face ? T.Nf + pt * NQ2 : T.N + pt * NQ2;
  const double* dN = face ? T.dNf + pt * NQ2 * D : T.dN + pt * NQ2 * D;
  using R = Raw<D>;
  const double* w;
  const double* x;
  int ws = 1;
  if (r < R::Gv) {
    w = N; x = U + (r < R::u ? r : NQ2 * D + r - R::u);
  } else if (r < R::vo) {
    const bool gu = r >= R::Gu;
    const int e = r - (gu ? R::Gu : R::Gv);
    w = dN + e % D; ws = D; x = U + (gu ? NQ2 * D : 0) + e / D;
  } else if (r < R::Guo) {
    w = N; x = Uo + (r < R::uo ? r - R::vo : NQ2 * D + r - R::uo);
  } else {
    const bool gv = r >= R::Gvo;
    const int e = r - (gv ? R::Gvo : R::Guo);
    w = dN + e % D; ws = D; x = Uo + (gv ? 0 : NQ2 * D) + e / D;
  }
  double s = 0.0;
#pragma unroll 9
  for (int k = 0; k < NQ2; ++k) s += w[k * ws] * x[k * D];
  return s;
}

template <int D>
__device__ __forceinline__ void read_mat(const double* p, double (&M)[D][D]) {
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) M[i][j] = p[i * D + j];
}
template <int D>
__device__ __forceinline__ void write_mat(double* p, double s, const double (&M)[D][D]) {
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) p[i * D + j] = s * M[i][j];
}
// F = I + grad u
template <int D>
__device__ __forceinline__ void read_F(const double* gu, double (&F)[D][D]) {
  read_mat<D>(gu, F);
#pragma unroll
  for (int i = 0; i < D; ++i) F[i][i] += 1.0;
}

// ====================================================================== residual
// One CTA takes up to RCELLS cells of a colour (cells_per_cta).  All threads interpolate (one scalar of one
// point per step), then one thread per point forms the point fluxes, then one thread per
// element row sums its test function over the points.  2D 256x128: about 3,000 FP64
// instructions per cell.  256x128 P1disc: 0.37 ms.  An earlier form gave each cell a CTA of
// its own, whose phase of point fluxes kept 12 of 256 threads busy: 3.35 ms.
template <int D> constexpr int kFlux = 2 * D + 2 * D * D + 1;   // f0, f1, hm, k0 (D), g0
template <int D, int PD>
struct ResSmem {
  using E = Sh<D, PD>;
  double U[E::RCELLS][E::NL];
  double Uo[E::RCELLS][2 * E::NQ2 * D];
  double raw[E::RCELLS][E::NQP + E::NFP][Raw<D>::kAll];   // the point's fluxes replace its raw values
  int gdof[E::RCELLS][E::NL];
  unsigned flags[E::RCELLS];
  unsigned long long minkey;
};

template <int D, int PD>
__global__ void __launch_bounds__(kAsmThreads) k_residual(CellGeom geom, int64_t ncol, int per, Tables T, Phys P,
                                                          const int* __restrict__ cell_dof,
                                                          const unsigned* __restrict__ cell_flags,
                                                          const unsigned char* __restrict__ row_fixed,
                                                          const double* __restrict__ Ug,
                                                          const double* __restrict__ Uold, double* __restrict__ out,
                                                          unsigned long long* __restrict__ minkey) {
  using E = Sh<D, PD>;
  using R = Raw<D>;
  constexpr int NQ2 = E::NQ2, NQ1 = E::NQ1, NL = E::NL, NQP = E::NQP, NFP = E::NFP, NV = NQ2 * D;
  constexpr int F0 = 0, F1 = D, HM = D + D * D, K0 = HM + D * D, G0 = K0 + D;
  static_assert(G0 + 1 == kFlux<D> && kFlux<D> <= R::kAll, "fluxes fit the raw slots");
  extern __shared__ __align__(16) unsigned char asm_smem[];
  ResSmem<D, PD>& S = *reinterpret_cast<ResSmem<D, PD>*>(asm_smem);
  const int64_t k0 = (int64_t)blockIdx.x * per;
  const int nc = (int)(ncol - k0 < per ? ncol - k0 : per);
  const bool prev = P.theta != 1.0;
  const double dtt = P.dt * P.theta, dto = P.dt * (1.0 - P.theta), mu = P.rho_f * P.nu_f;
  for (int t = threadIdx.x; t < nc * NL; t += blockDim.x) {
    const int ce = t / NL, l = t % NL;
    int cc[3];
    const int64_t cell = colour_cell<D>(geom, k0 + ce, cc);
    const int g = cell_dof[cell * NL + l];
    S.gdof[ce][l] = g;
    S.U[ce][l] = Ug[g];
    if (l < 2 * NV) S.Uo[ce][l] = Uold ? Uold[g] : 0.0;
    if (l == 0) S.flags[ce] = cell_flags[cell];
  }
  if (threadIdx.x == 0) S.minkey = ~0ull;
  __syncthreads();
  const int nr = prev ? R::kAll : R::kNow;
  for (int t = threadIdx.x; t < nc * NQP * nr; t += blockDim.x) {
    const int ce = t / (NQP * nr), e = t % (NQP * nr);
    S.raw[ce][e / nr][e % nr] = interpolate<D, PD>(T, false, e / nr, e % nr, S.U[ce], S.Uo[ce]);
  }
  for (int ce = 0; ce < nc; ++ce)
    if ((S.flags[ce] & 3u) == 2u)
      for (int e = threadIdx.x; e < NFP * nr; e += blockDim.x)
        S.raw[ce][NQP + e / nr][e % nr] = interpolate<D, PD>(T, true, e / nr, e % nr, S.U[ce], S.Uo[ce]);
  __syncthreads();

  double my_min = 1e300;
  for (int t = threadIdx.x; t < nc * (NQP + NFP); t += blockDim.x) {
    // volume points first, so that the cells' points fill whole warps
    const bool face = t >= nc * NQP;
    const int ce = face ? (t - nc * NQP) / NFP : t / NQP;
    const int pt = face ? NQP + (t - nc * NQP) % NFP : t % NQP;
    const bool solid = S.flags[ce] & 1u;
    if (face && (S.flags[ce] & 3u) != 2u) continue;
    double* q = S.raw[ce][pt];
    double F[D][D], Gv[D][D], Fo[D][D], Gvo[D][D], v[D], dv[D], du[D], vo[D];
    read_F<D>(q + R::Gu, F);
    read_mat<D>(q + R::Gv, Gv);
    if (prev) { read_F<D>(q + R::Guo, Fo); read_mat<D>(q + R::Gvo, Gvo); }
#pragma unroll
    for (int i = 0; i < D; ++i) {
      v[i] = q[R::v + i];
      vo[i] = q[R::vo + i];
      dv[i] = v[i] - vo[i];
      du[i] = q[R::u + i] - q[R::uo + i];
    }
    const double J = det<D>(F);
    if (!face && J < my_min) my_min = J;
    if (solid) {
      // E = (F^T F - I) / 2, f1 = w F Sigma
      auto stress = [&](const double (&X)[D][D], double w, double (&O)[D][D]) {
        double C[D][D], tr = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
          for (int j = 0; j < D; ++j) {
            double s = X[0][i] * X[0][j];
#pragma unroll
            for (int m = 1; m < D; ++m) s += X[m][i] * X[m][j];
            C[i][j] = 0.5 * (s - (i == j ? 1.0 : 0.0));
          }
#pragma unroll
        for (int i = 0; i < D; ++i) tr += C[i][i];
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
          for (int j = 0; j < D; ++j) C[i][j] = w * (2.0 * P.mu_s * C[i][j] + (i == j ? P.lambda_s * tr : 0.0));
        matmul<D>(X, C, O);
      };
      double f1[D][D], fo[D][D];
      stress(F, dtt, f1);
      if (prev) stress(Fo, dto, fo);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        q[F0 + i] = P.rho_s * dv[i];
        q[K0 + i] = du[i] - dtt * v[i] - (prev ? dto * vo[i] : 0.0);
#pragma unroll
        for (int j = 0; j < D; ++j) q[F1 + i * D + j] = f1[i][j] + (prev ? fo[i][j] : 0.0);
      }
      continue;
    }
    double Fi[D][D], A[D][D], Fio[D][D], Ao[D][D], Jo = 1.0;
    const double iJ = 1.0 / J;
    invert<D>(F, iJ, Fi);
    matmul<D>(Gv, Fi, A);
    if (prev) {
      Jo = det<D>(Fo);
      invert<D>(Fo, 1.0 / Jo, Fio);
      matmul<D>(Gvo, Fio, Ao);
    }
    if (face) {
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double s = 0.0, so = 0.0;
#pragma unroll
        for (int m = 0; m < D; ++m) s += A[m][i] * Fi[0][m];
        if (prev)
#pragma unroll
          for (int m = 0; m < D; ++m) so += Ao[m][i] * Fio[0][m];
        q[F0 + i] = -dtt * mu * J * s - (prev ? dto * mu * Jo * so : 0.0);
      }
      continue;
    }
    double p = 0.0;
#pragma unroll
    for (int a = 0; a < NQ1; ++a) p += T.Np[pt * NQ1 + a] * S.U[ce][2 * NV + a];
    double X[D][D], f1[D][D], hm[D][D], trA = 0.0;
    const double m = dtt * mu * J;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      trA += A[i][i];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        X[i][j] = m * (A[i][j] + A[j][i]) - (i == j ? J * p : 0.0);
        hm[i][j] = q[R::Gu + i * D + j] * iJ;
      }
    }
    matmul_t<D>(X, Fi, f1);
    if (prev) {
      const double mo = dto * mu * Jo;
      double Xo[D][D], fo[D][D];
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) Xo[i][j] = mo * (Ao[i][j] + Ao[j][i]);
      matmul_t<D>(Xo, Fio, fo);
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) f1[i][j] += fo[i][j];
    }
    const double Jt = prev ? P.theta * J + (1.0 - P.theta) * Jo : J;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      double ac = 0.0, co = 0.0;
#pragma unroll
      for (int j = 0; j < D; ++j) ac += A[i][j] * (dtt * v[j] - du[j]);
      if (prev)
#pragma unroll
        for (int j = 0; j < D; ++j) co += Ao[i][j] * vo[j];
      q[F0 + i] = P.rho_f * (Jt * dv[i] + J * ac + (prev ? dto * Jo * co : 0.0));
    }
    write_mat<D>(q + F1, 1.0, f1);
    write_mat<D>(q + HM, 1.0, hm);
    q[G0] = J * trA;
  }
  if (my_min < 1e300) atomicMin(&S.minkey, order_key(my_min));
  __syncthreads();
  if (threadIdx.x == 0 && S.minkey != ~0ull) atomicMin(minkey, S.minkey);

  for (int t = threadIdx.x; t < nc * NL; t += blockDim.x) {
    const int ce = t / NL, r = t % NL;
    const int gr = S.gdof[ce][r];
    const unsigned flags = S.flags[ce];
    const bool solid = flags & 1u, prow = r >= 2 * NV, urow = !prow && r >= NV;
    if (row_fixed[gr] || (solid && prow)) continue;              // solid cells own no pressure rows
    const int l = urow ? r - NV : r, a = l / D, i = l % D;
    if (!solid && urow && !((flags >> (2 + a)) & 1u)) continue;  // fluid cell: mesh rows only
    double acc = 0.0;
    for (int pt = 0; pt < NQP; ++pt) {
      const double* q = S.raw[ce][pt];
      const double* dN = T.dN + (pt * NQ2 + a) * D;
      double s;
      if (prow) {
        s = T.Np[pt * NQ1 + (r - 2 * NV)] * q[G0];
      } else if (!urow || solid) {
        s = T.N[pt * NQ2 + a] * q[(urow ? K0 : F0) + i];
        if (!urow)
#pragma unroll
          for (int j = 0; j < D; ++j) s += dN[j] * q[F1 + i * D + j];
      } else {
        s = dN[0] * q[HM + i * D];
#pragma unroll
        for (int j = 1; j < D; ++j) s += dN[j] * q[HM + i * D + j];
      }
      acc += T.w[pt] * s;
    }
    if ((flags & 3u) == 2u && !urow && !prow)
      for (int f = 0; f < NFP; ++f) acc += T.wf[f] * T.Nf[f * NQ2 + a] * S.raw[ce][NQP + f][F0 + i];
    out[gr] += acc;
  }
}

// ====================================================================== Jacobian
// One CTA takes up to JCELLS cells of a colour (cells_per_cta).  What the variations above need is tabulated
// in shared memory once per point (PT slots) and once per (point, trial node) (TR slots,
// quadrature weight folded in).  A unit of work is one trial component (b, k) against
// one test component i: a thread forms the unit's f0 and reference flux f1 at a line of
// three points at a time and contracts them with the 3^D test functions by sum
// factorisation (direction 0, then 1, then 2; the functions are products of 1D factors):
// 729 FMAs per 3D unit instead of 2,916 for point x test function, 135 instead of 243
// in 2D, and 4 to 14 more per point for the fields.  Neighbouring lanes take neighbouring
// (b, k), so their additions into a CSR row are contiguous along a lattice line.
// Positions in the CSR rows are searched once per (row, trial node), not per entry.
// Measured, against one dual-number evaluation per point and column with a search per
// entry: 256x128 16.17 -> 2.52 ms, 32x16x16 at theta = 1/2 197.0 -> 14.0 ms (0.77e6 FP64
// FMAs per fluid cell; all cells take 9.9 ms at the FP64 pipe's measured 0.529e12 per second).
template <int D>
struct Pt {   // per point
  static constexpr int Fi = 0, A = D * D, Fim = 2 * D * D, FA = 3 * D * D, PX = 4 * D * D, GuJ = 5 * D * D,
                       e = 6 * D * D, wJ = e + D, trA = wJ + 1, wJi = trA + 1, kN = wJi + 1;
  // solid cells: F, w dtt mu F, w dtt lambda F, w dtt mu F F^T, w dtt Sigma
  static constexpr int sF = 0, smF = D * D, slF = 2 * D * D, sB = 3 * D * D, sS = 4 * D * D;
  // face points: F^-1, A, A^T n', -w m J
  static constexpr int fFi = 0, fA = D * D, fq = 2 * D * D, fm = fq + D;
};
template <int D>
struct Tr {   // per (point, trial node)
  static constexpr int G = 0, FG = D, XG = 2 * D, al = 3 * D, nb = al + 1, r = nb + 1, kN = r + 1;
  // solid cells: F grad phi, w dtt Sigma grad phi, grad phi; mesh rows: w grad phi / J in FG
  static constexpr int sf = 0, sS = D, sd = 2 * D;
};
constexpr unsigned short kNoPos = 0xFFFFu;

template <int D, int PD>
struct JacCell {
  using E = Sh<D, PD>;
  static constexpr int NC = 2 * E::NQ2 + E::NQ1;    // trial nodes: v, u, pressure functions
  double U[E::NL];
  double Uo[2 * E::NQ2 * D];
  double pt[E::NQP][Pt<D>::kN];
  double face[E::NFP][2 * D * D + D + 1];
  double tr[E::NQP][E::NQ2][Tr<D>::kN];              // the raw point values first
  long long row[E::NL];                              // first CSR entry of each local row, -1: not assembled
  int gdof[E::NL];
  unsigned flags;
  unsigned short pos[E::NL][NC];                     // of the node's first component within the row
  unsigned char cfix[E::NL];
};
template <int D, int PD>
struct JacSmem {
  JacCell<D, PD> c[Sh<D, PD>::JCELLS];
  unsigned long long minkey;
};

// acc += the contraction of one unit's point fields with the test functions:
// field(q, f0, f1) gives the fields of point q.  HAS0: f0 is not identically zero.
template <int D, bool HAS0, class Field>
__device__ __forceinline__ void contract(const Basis1& B, const Field& field, double (&acc)[D == 2 ? 9 : 27]) {
#pragma unroll
  for (int t = 0; t < (D == 2 ? 9 : 27); ++t) acc[t] = 0.0;
#pragma unroll 1
  for (int qz = 0; qz < (D == 2 ? 1 : 3); ++qz) {
    double h[9], hz[9];   // sums over directions 0 and 1, for the value and the derivative in direction 2
    if constexpr (D == 3)
#pragma unroll
      for (int t = 0; t < 9; ++t) h[t] = hz[t] = 0.0;
#pragma unroll
    for (int qy = 0; qy < 3; ++qy) {
      double t0[3] = {0.0, 0.0, 0.0}, ty[3] = {0.0, 0.0, 0.0}, tz[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int qx = 0; qx < 3; ++qx) {
        double f0 = 0.0, f1[D];
        field(qx + 3 * qy + 9 * qz, f0, f1);
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          if (HAS0) t0[ax] = fma(B.N[qx][ax], f0, t0[ax]);
          t0[ax] = fma(B.dN[0][qx][ax], f1[0], t0[ax]);
          ty[ax] = fma(B.N[qx][ax], f1[1], ty[ax]);
          if constexpr (D == 3) tz[ax] = fma(B.N[qx][ax], f1[2], tz[ax]);
        }
      }
#pragma unroll
      for (int ay = 0; ay < 3; ++ay)
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          double& o = D == 2 ? acc[3 * ay + ax] : h[3 * ay + ax];
          o = fma(B.N[qy][ay], t0[ax], o);
          o = fma(B.dN[1][qy][ay], ty[ax], o);
          if constexpr (D == 3) hz[3 * ay + ax] = fma(B.N[qy][ay], tz[ax], hz[3 * ay + ax]);
        }
    }
    if constexpr (D == 3) {
#pragma unroll
      for (int az = 0; az < 3; ++az)
#pragma unroll
        for (int t = 0; t < 9; ++t)
          acc[9 * az + t] = fma(B.dN[2][qz][az], hz[t], fma(B.N[qz][az], h[t], acc[9 * az + t]));
    }
  }
}

// Position of column col in a CSR row of len sorted columns, or -1.
__device__ __forceinline__ int find_col(const int* __restrict__ ci, int len, int col) {
  int lo = 0, hi = len;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(ci + mid) < col) lo = mid + 1; else hi = mid;
  }
  return lo < len && __ldg(ci + lo) == col ? lo : -1;
}

template <int D, int PD>
__global__ void __launch_bounds__(Sh<D, PD>::JTHREADS, 2) k_jacobian(CellGeom geom, int64_t ncol, int per, Tables T,
                                                             const __grid_constant__ Basis1 B, Phys P,
                                                             const int* __restrict__ cell_dof,
                                                             const unsigned* __restrict__ cell_flags,
                                                             const int64_t* __restrict__ rowptr,
                                                             const int* __restrict__ colind,
                                                             const unsigned char* __restrict__ row_fixed,
                                                             const double* __restrict__ Ug,
                                                             const double* __restrict__ Uold,
                                                             double* __restrict__ out,
                                                             unsigned long long* __restrict__ minkey,
                                                             int* __restrict__ err) {
  using E = Sh<D, PD>;
  using R = Raw<D>;
  using C = JacCell<D, PD>;
  constexpr int NQ2 = E::NQ2, NQ1 = E::NQ1, NL = E::NL, NQP = E::NQP, NFP = E::NFP, NV = NQ2 * D, NC = C::NC;
  constexpr int UNITS = NQ2 * D * D;
  static_assert(R::kAll <= NQ2 * Tr<D>::kN, "raw values fit a point's trial slots");
  extern __shared__ __align__(16) unsigned char asm_smem[];
  JacSmem<D, PD>& S = *reinterpret_cast<JacSmem<D, PD>*>(asm_smem);
  // the last cells first: the solid ones, a third of a fluid cell's work, lie at the low end of
  // the last direction in the meshes of Sec. 6 and fill the SMs' last slots better
  const int64_t k0 = (int64_t)(gridDim.x - 1 - blockIdx.x) * per;
  const int nc = (int)(ncol - k0 < per ? ncol - k0 : per);
  const bool prev = P.theta != 1.0;
  const double dtt = P.dt * P.theta, mu = P.rho_f * P.nu_f;
  for (int t = threadIdx.x; t < nc * NL; t += blockDim.x) {
    C& c = S.c[t / NL];
    const int l = t % NL;
    int cc[3];
    const int64_t cell = colour_cell<D>(geom, k0 + t / NL, cc);
    const unsigned flags = cell_flags[cell];
    const bool solid = flags & 1u, prow = l >= 2 * NV, urow = !prow && l >= NV;
    const int g = cell_dof[cell * NL + l];
    const bool fixed = row_fixed[g];
    c.gdof[l] = g;
    c.U[l] = Ug[g];
    if (l < 2 * NV) c.Uo[l] = Uold ? Uold[g] : 0.0;
    if (l == 0) c.flags = flags;
    c.cfix[l] = fixed || (solid && prow);
    const bool skip = fixed || (solid && prow) ||                            // solid cells own no pressure rows
                      (!solid && urow && !((flags >> (2 + (l - NV) / D)) & 1u));   // fluid cells: mesh rows only
    c.row[l] = skip ? -1 : rowptr[g];
  }
  if (threadIdx.x == 0) S.minkey = ~0ull;
  __syncthreads();
  // raw point values, in the trial slots of the point
  const int nr = prev ? R::Gvo : R::kNow;
  for (int t = threadIdx.x; t < nc * NQP * nr; t += blockDim.x) {
    C& c = S.c[t / (NQP * nr)];
    const int e = t % (NQP * nr);
    c.tr[e / nr][0][e % nr] = interpolate<D, PD>(T, false, e / nr, e % nr, c.U, c.Uo);
  }
  __syncthreads();

  // ---- point tables, in the first warps
  constexpr int kPointThreads = (E::JCELLS * NQP + 31) / 32 * 32;
  static_assert(kPointThreads < E::JTHREADS, "warps left for the positions");
  double my_min = 1e300;
  if ((int)threadIdx.x < nc * NQP) {
    const int t = threadIdx.x;
    C& c = S.c[t / NQP];
    const int q = t % NQP;
    const double* raw = c.tr[q][0];
    double* o = c.pt[q];
    const double w = T.w[q];
    double F[D][D];
    read_F<D>(raw + R::Gu, F);
    const double J = det<D>(F);
    if (J < my_min) my_min = J;
    using K = Pt<D>;
    const bool solid = c.flags & 1u;
    if (solid) {
      double Bm[D][D], Sg[D][D], tr = 0.0;
      matmul_t<D>(F, F, Bm);
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) {
          double s = F[0][i] * F[0][j];
#pragma unroll
          for (int m = 1; m < D; ++m) s += F[m][i] * F[m][j];
          Sg[i][j] = 0.5 * (s - (i == j ? 1.0 : 0.0));
        }
#pragma unroll
      for (int i = 0; i < D; ++i) tr += Sg[i][i];
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) Sg[i][j] = 2.0 * P.mu_s * Sg[i][j] + (i == j ? P.lambda_s * tr : 0.0);
      write_mat<D>(o + K::sF, 1.0, F);
      write_mat<D>(o + K::smF, w * dtt * P.mu_s, F);
      write_mat<D>(o + K::slF, w * dtt * P.lambda_s, F);
      write_mat<D>(o + K::sB, w * dtt * P.mu_s, Bm);
      write_mat<D>(o + K::sS, w * dtt, Sg);
    }
    if (!solid) {
      double Fi[D][D], A[D][D], Gv[D][D], X[D][D], Y[D][D], p = 0.0, trA = 0.0, Jo = 1.0;
      read_mat<D>(raw + R::Gv, Gv);
      const double iJ = 1.0 / J;
      invert<D>(F, iJ, Fi);
      matmul<D>(Gv, Fi, A);
      if (prev) {
        double Fo[D][D];
        read_F<D>(raw + R::Guo, Fo);
        Jo = det<D>(Fo);
      }
#pragma unroll
      for (int a = 0; a < NQ1; ++a) p += T.Np[q * NQ1 + a] * c.U[2 * NV + a];
      const double m = dtt * mu, wJ = w * J;
      write_mat<D>(o + K::Fi, 1.0, Fi);
      write_mat<D>(o + K::A, 1.0, A);
      write_mat<D>(o + K::Fim, wJ * m, Fi);
      matmul<D>(Fi, A, Y);
      write_mat<D>(o + K::FA, wJ * m, Y);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        trA += A[i][i];
#pragma unroll
        for (int j = 0; j < D; ++j) X[i][j] = wJ * (m * (A[i][j] + A[j][i]) - (i == j ? p : 0.0));
      }
      matmul_t<D>(X, Fi, Y);
      write_mat<D>(o + K::PX, 1.0, Y);
      const double wi = w * iJ;
#pragma unroll
      for (int i = 0; i < D * D; ++i) o[K::GuJ + i] = wi * raw[R::Gu + i];
      double cv[D];
#pragma unroll
      for (int j = 0; j < D; ++j) cv[j] = dtt * raw[R::v + j] - (raw[R::u + j] - raw[R::uo + j]);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double s = (prev ? P.theta : 1.0) * (raw[R::v + i] - raw[R::vo + i]);
#pragma unroll
        for (int j = 0; j < D; ++j) s += A[i][j] * cv[j];
        o[K::e + i] = wJ * P.rho_f * s;
      }
      o[K::wJ] = wJ;
      o[K::trA] = trA;
      o[K::wJi] = wi;
      // for the trial tables: c, and J^theta w rho_f; kept in raw slots that no other point reads
      double* z = c.tr[q][0] + R::Gv;
#pragma unroll
      for (int j = 0; j < D; ++j) z[j] = cv[j];
      z[D] = w * P.rho_f * (prev ? P.theta * J + (1.0 - P.theta) * Jo : J);
      z[D + 1] = p;
    }
  }
  // meanwhile, in the other warps: positions of the trial nodes in the rows (the components' rows of a
  // node have equal patterns as a rule, so the first component's position is tried first)
  for (int t = (int)threadIdx.x - kPointThreads; t >= 0 && t < nc * NC * (2 * NQ2 + NQ1);
       t += (int)blockDim.x - kPointThreads) {
    C& c = S.c[t / (NC * (2 * NQ2 + NQ1))];
    const int e = t % (NC * (2 * NQ2 + NQ1)), rn = e / NC, cn = e % NC;
    const int nrows = rn < 2 * NQ2 ? D : 1, r0 = rn < 2 * NQ2 ? rn * D : 2 * NV + rn - 2 * NQ2;
    const int ncols = cn < 2 * NQ2 ? D : 1, col0 = c.gdof[cn < 2 * NQ2 ? cn * D : 2 * NV + cn - 2 * NQ2];
    const bool solid = c.flags & 1u;
    const bool urow = rn >= NQ2 && rn < 2 * NQ2;
    if (!solid && urow && (cn < NQ2 || cn >= 2 * NQ2)) continue;             // mesh rows: u columns only
    if (cn >= 2 * NQ2 && rn >= 2 * NQ2) continue;                            // no pressure-pressure coupling
    int hint = -1;
    for (int i = 0; i < nrows; ++i) {
      const long long base = c.row[r0 + i];
      unsigned short found = kNoPos;
      if (base >= 0) {
        const int len = (int)(rowptr[c.gdof[r0 + i] + 1] - base);
        const int* ci = colind + base;
        int p = hint >= 0 && hint < len && __ldg(ci + hint) == col0 ? hint : find_col(ci, len, col0);
        if (p >= 0) {
          hint = p;
          bool all = p + ncols <= len && p < kNoPos;
          for (int k = 1; k < ncols && all; ++k) all = __ldg(ci + p + k) == col0 + k;
          if (all) found = (unsigned short)p;
        }
      }
      c.pos[r0 + i][cn] = found;
    }
  }
  if (my_min < 1e300) atomicMin(&S.minkey, order_key(my_min));
  __syncthreads();
  if (threadIdx.x == 0 && S.minkey != ~0ull) atomicMin(minkey, S.minkey);
  // outflow faces of these cells
  for (int ce = 0; ce < nc; ++ce) {
    C& c = S.c[ce];
    if ((c.flags & 3u) != 2u) continue;
    for (int f = threadIdx.x; f < NFP; f += blockDim.x) {
      double F[D][D], Gv[D][D], Fi[D][D], A[D][D];
      for (int e = 0; e < D * D; ++e) {
        Gv[e / D][e % D] = interpolate<D, PD>(T, true, f, R::Gv + e, c.U, c.Uo);
        F[e / D][e % D] = interpolate<D, PD>(T, true, f, R::Gu + e, c.U, c.Uo) + (e / D == e % D ? 1.0 : 0.0);
      }
      const double J = det<D>(F);
      invert<D>(F, 1.0 / J, Fi);
      matmul<D>(Gv, Fi, A);
      double* o = c.face[f];
      write_mat<D>(o + Pt<D>::fFi, 1.0, Fi);
      write_mat<D>(o + Pt<D>::fA, 1.0, A);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double s = 0.0;
#pragma unroll
        for (int m = 0; m < D; ++m) s += A[m][i] * Fi[0][m];
        o[Pt<D>::fq + i] = s;
      }
      o[Pt<D>::fm] = -T.wf[f] * dtt * mu * J;
    }
  }
  // ---- trial tables: a warp takes whole points (3 in 2D, 1 in 3D), so that a point's c and J^theta
  // (in the slots that the tables overwrite) are read by all of its lanes before any lane writes
  {
    constexpr int PW = 32 / NQ2;
    static_assert(NQP % PW == 0, "whole points of one cell per warp");
    const int lane = threadIdx.x & 31;
    for (int u = threadIdx.x >> 5; u < nc * (NQP / PW); u += blockDim.x >> 5) {
      C& c = S.c[u / (NQP / PW)];
      const bool on = lane < PW * NQ2;
      const int q = u % (NQP / PW) * PW + (on ? lane / NQ2 : 0), b = lane % NQ2;
      const double* o = c.pt[q];
      double cv[D], jt = 0.0, p = 0.0;
      const bool solid = c.flags & 1u;
      if (!solid) {
        const double* z = c.tr[q][0] + R::Gv;
#pragma unroll
        for (int j = 0; j < D; ++j) cv[j] = z[j];
        jt = z[D];
        p = z[D + 1];
      }
      __syncwarp();
      if (on) {
        double* tr = c.tr[q][b];
        const double* dN = T.dN + (q * NQ2 + b) * D;
        const double N = T.N[q * NQ2 + b];
        if (solid) {
#pragma unroll
          for (int i = 0; i < D; ++i) {
            double f = 0.0, s = 0.0;
#pragma unroll
            for (int j = 0; j < D; ++j) {
              f += o[Pt<D>::sF + i * D + j] * dN[j];
              s += o[Pt<D>::sS + i * D + j] * dN[j];
            }
            tr[Tr<D>::sf + i] = f;
            tr[Tr<D>::sS + i] = s;
            tr[Tr<D>::sd + i] = dN[i];
          }
        } else {
          double G[D], sb = 0.0;
#pragma unroll
          for (int k = 0; k < D; ++k) {
            double g = 0.0;
#pragma unroll
            for (int l = 0; l < D; ++l) g += dN[l] * o[Pt<D>::Fi + l * D + k];
            G[k] = g;
            sb += g * cv[k];
          }
          const double wJ = o[Pt<D>::wJ], m = dtt * mu;
#pragma unroll
          for (int i = 0; i < D; ++i) {
            double fg = 0.0, xg = 0.0;
#pragma unroll
            for (int j = 0; j < D; ++j) {
              fg += o[Pt<D>::Fim + i * D + j] * G[j];
              xg += (o[Pt<D>::A + i * D + j] + o[Pt<D>::A + j * D + i]) * G[j];
            }
            tr[Tr<D>::G + i] = G[i];
            tr[Tr<D>::FG + i] = fg;
            tr[Tr<D>::XG + i] = wJ * (m * xg - p * G[i]);
          }
          const double wr = wJ * P.rho_f;
          tr[Tr<D>::al] = jt * N + wr * sb;
          tr[Tr<D>::nb] = wr * dtt * N;
          tr[Tr<D>::r] = wr * (sb + N);
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();

  // ---- units
  // adds acc (one value per test node) at column (node cn, component k of ncol) to the rows rbase + a * rstride
  auto scatter = [&](C& c, int rbase, int cn, int col, int k, const double (&acc)[NQ2]) {
    const int gc = c.gdof[col];
#pragma unroll
    for (int a0 = 0; a0 < NQ2; a0 += 9) {
      double* at[9];
      double old[9];
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        const int r = rbase + (a0 + t) * D;
        const long long base = c.row[r];
        at[t] = nullptr;
        if (base < 0) continue;
        int p = c.pos[r][cn];
        if (p != kNoPos) p += k;
        else p = find_col(colind + base, (int)(rowptr[c.gdof[r] + 1] - base), gc);
        if (p >= 0) at[t] = out + base + p;
        else if (acc[a0 + t] != 0.0) atomicExch(err, 1);      // an entry outside the pattern
      }
#pragma unroll
      for (int t = 0; t < 9; ++t) old[t] = at[t] ? *at[t] : 0.0;
#pragma unroll
      for (int t = 0; t < 9; ++t)
        if (at[t]) *at[t] = old[t] + acc[a0 + t];
    }
  };
  // the outflow term of unit (i, b, k): added to the test nodes on the face (lattice index 2 in direction 0)
  auto add_face = [&](const C& c, bool along_u, int i, int b, int k, double (&acc)[NQ2]) {
    for (int f = 0; f < NFP; ++f) {
      const double* o = c.face[f];
      const double* dN = T.dNf + (f * NQ2 + b) * D;
      double G[D];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        double g = 0.0;
#pragma unroll
        for (int l = 0; l < D; ++l) g += dN[l] * o[Pt<D>::fFi + l * D + j];
        G[j] = g;
      }
      double gi = 0.0, gk = 0.0, ag = 0.0;
#pragma unroll
      for (int l = 0; l < D; ++l) {
        gi = l == i ? G[l] : gi;
        gk = l == k ? G[l] : gk;
        ag += o[Pt<D>::fA + l * D + i] * G[l];
      }
      double d = gi * o[Pt<D>::fFi + k];                        // A^T n' along v
      if (along_u) d = gk * o[Pt<D>::fq + i] - gi * o[Pt<D>::fq + k] - o[Pt<D>::fFi + k] * ag;
      d *= o[Pt<D>::fm];
#pragma unroll
      for (int a = 2; a < NQ2; a += 3) acc[a] += T.Nf[f * NQ2 + a] * d;
    }
  };
  // rows of v, columns of v (fluid); solid cells: the mass terms of all three pairs of v and u
  for (int t = threadIdx.x; t < nc * UNITS; t += blockDim.x) {
    C& c = S.c[t / UNITS];
    const int u = t % UNITS, i = u / NV, b = (u % NV) / D, k = u % D;
    if (c.flags & 1u) {
      if (i != k) continue;
      double m[NQ2], x[NQ2];
#pragma unroll
      for (int a = 0; a < NQ2; ++a) m[a] = T.M[a * NQ2 + b];
      if (!c.cfix[b * D + k]) {
#pragma unroll
        for (int a = 0; a < NQ2; ++a) x[a] = P.rho_s * m[a];
        scatter(c, i, b, b * D + k, k, x);
#pragma unroll
        for (int a = 0; a < NQ2; ++a) x[a] = -dtt * m[a];
        scatter(c, NV + i, b, b * D + k, k, x);
      }
      if (!c.cfix[NV + b * D + k]) scatter(c, NV + i, NQ2 + b, NV + b * D + k, k, m);
      continue;
    }
    if (c.cfix[b * D + k]) continue;
    double acc[NQ2];
    contract<D, true>(B, [&](int q, double& f0, double (&f1)[D]) {
      const double* o = c.pt[q];
      const double* tr = c.tr[q][b];
      const double g = tr[Tr<D>::G + i];
      f0 = fma(o[Pt<D>::A + i * D + k], tr[Tr<D>::nb], i == k ? tr[Tr<D>::al] : 0.0);
#pragma unroll
      for (int j = 0; j < D; ++j) f1[j] = fma(g, o[Pt<D>::Fim + j * D + k], i == k ? tr[Tr<D>::FG + j] : 0.0);
    }, acc);
    if (c.flags & 2u) add_face(c, false, i, b, k, acc);
    scatter(c, i, b, b * D + k, k, acc);
  }
  // rows of v, columns of u
  for (int t = threadIdx.x; t < nc * UNITS; t += blockDim.x) {
    C& c = S.c[t / UNITS];
    const int u = t % UNITS, i = u / NV, b = (u % NV) / D, k = u % D;
    if (c.cfix[NV + b * D + k]) continue;
    double acc[NQ2];
    if (c.flags & 1u) {
      contract<D, false>(B, [&](int q, double&, double (&f1)[D]) {
        const double* o = c.pt[q];
        const double* tr = c.tr[q][b];
        const double bik = o[Pt<D>::sB + i * D + k], fi = tr[Tr<D>::sf + i], fk = tr[Tr<D>::sf + k];
#pragma unroll
        for (int j = 0; j < D; ++j) {
          double s = fma(bik, tr[Tr<D>::sd + j], i == k ? tr[Tr<D>::sS + j] : 0.0);
          s = fma(fi, o[Pt<D>::smF + k * D + j], s);
          f1[j] = fma(fk, o[Pt<D>::slF + i * D + j], s);
        }
      }, acc);
    } else {
      contract<D, true>(B, [&](int q, double& f0, double (&f1)[D]) {
        const double* o = c.pt[q];
        const double* tr = c.tr[q][b];
        const double gk = tr[Tr<D>::G + k], gi = tr[Tr<D>::G + i], xg = tr[Tr<D>::XG + i];
        const double aik = o[Pt<D>::A + i * D + k];
        f0 = fma(gk, o[Pt<D>::e + i], -aik * tr[Tr<D>::r]);
#pragma unroll
        for (int j = 0; j < D; ++j) {
          double s = gk * o[Pt<D>::PX + i * D + j];
          s = fma(-xg, o[Pt<D>::Fi + j * D + k], s);
          s = fma(-aik, tr[Tr<D>::FG + j], s);
          f1[j] = fma(-gi, o[Pt<D>::FA + j * D + k], s);
        }
      }, acc);
      if (c.flags & 2u) add_face(c, true, i, b, k, acc);
    }
    scatter(c, i, NQ2 + b, NV + b * D + k, k, acc);
  }
  // rows of v, columns of the pressure: df1_ij = -J psi F^-1_ji
  for (int t = threadIdx.x; t < nc * NQ1 * D; t += blockDim.x) {
    C& c = S.c[t / (NQ1 * D)];
    const int u = t % (NQ1 * D), i = u / NQ1, b = u % NQ1;
    if (c.cfix[2 * NV + b]) continue;                     // solid cells: no pressure columns
    double acc[NQ2];
    contract<D, false>(B, [&](int q, double&, double (&f1)[D]) {
      const double* o = c.pt[q];
      const double s = -o[Pt<D>::wJ] * T.Np[q * NQ1 + b];
#pragma unroll
      for (int j = 0; j < D; ++j) f1[j] = s * o[Pt<D>::Fi + j * D + i];
    }, acc);
    scatter(c, i, 2 * NQ2 + b, 2 * NV + b, 0, acc);
  }
  // rows of the pressure, columns (b, k) of v and of u
  for (int t = threadIdx.x; t < nc * NV; t += blockDim.x) {
    C& c = S.c[t / NV];
    const int b = (t % NV) / D, k = t % D;
    if (c.flags & 1u) continue;
    double av[NQ1], au[NQ1];
#pragma unroll
    for (int a = 0; a < NQ1; ++a) av[a] = au[a] = 0.0;
#pragma unroll 3
    for (int q = 0; q < NQP; ++q) {
      const double* o = c.pt[q];
      const double* tr = c.tr[q][b];
      double ag = 0.0;
#pragma unroll
      for (int l = 0; l < D; ++l) ag += o[Pt<D>::A + l * D + k] * tr[Tr<D>::G + l];
      const double gv = o[Pt<D>::wJ] * tr[Tr<D>::G + k];
      const double gu = fma(gv, o[Pt<D>::trA], -o[Pt<D>::wJ] * ag);
#pragma unroll
      for (int a = 0; a < NQ1; ++a) {
        av[a] = fma(T.Np[q * NQ1 + a], gv, av[a]);
        au[a] = fma(T.Np[q * NQ1 + a], gu, au[a]);
      }
    }
#pragma unroll
    for (int a = 0; a < NQ1; ++a) {
      const int r = 2 * NV + a;
      const long long base = c.row[r];
      if (base < 0) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (c.cfix[h * NV + b * D + k]) continue;
        const double x = h ? au[a] : av[a];
        int p = c.pos[r][h * NQ2 + b];
        if (p != kNoPos) p += k;
        else p = find_col(colind + base, (int)(rowptr[c.gdof[r] + 1] - base), c.gdof[h * NV + b * D + k]);
        if (p >= 0) out[base + p] += x;
        else if (x != 0.0) atomicExch(err, 1);
      }
    }
  }
  __syncthreads();
  // mesh rows, columns of u: w grad phi_b / J takes the place of FG
  for (int t = threadIdx.x; t < nc * NQP * NQ2; t += blockDim.x) {
    C& c = S.c[t / (NQP * NQ2)];
    const int q = t % (NQP * NQ2) / NQ2, b = t % NQ2;
    if (c.flags & 1u) continue;
#pragma unroll
    for (int j = 0; j < D; ++j)
      c.tr[q][b][Tr<D>::FG + j] = c.pt[q][Pt<D>::wJi] * T.dN[(q * NQ2 + b) * D + j];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nc * UNITS; t += blockDim.x) {
    C& c = S.c[t / UNITS];
    const int u = t % UNITS, i = u / NV, b = (u % NV) / D, k = u % D;
    if ((c.flags & 1u) || (c.flags >> 2) == 0u || c.cfix[NV + b * D + k]) continue;
    double acc[NQ2];
    contract<D, false>(B, [&](int q, double&, double (&f1)[D]) {
      const double* o = c.pt[q];
      const double* tr = c.tr[q][b];
      const double gk = tr[Tr<D>::G + k];
#pragma unroll
      for (int j = 0; j < D; ++j) f1[j] = fma(-gk, o[Pt<D>::GuJ + i * D + j], i == k ? tr[Tr<D>::FG + j] : 0.0);
    }, acc);
    scatter(c, NV + i, NQ2 + b, NV + b * D + k, k, acc);
  }
}

// fixed rows: the identity entry
__global__ void k_fixed_rows(int64_t n, const int64_t* __restrict__ rowptr, const unsigned char* __restrict__ fixed,
                             double* __restrict__ vals) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n && fixed[r]) vals[rowptr[r]] = 1.0;
}

// max |R_i| over the rows into *key (the bits of a non-negative double order as integers; NaN
// entries are passed over)
__global__ void k_absmax(int64_t n, const double* __restrict__ x, unsigned long long* __restrict__ key) {
  double m = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs(x[i]));
  for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(key, (unsigned long long)__double_as_longlong(m));
}

__global__ void k_axpy_inplace(int64_t n, double alpha, const double* __restrict__ x, double* __restrict__ y) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] += alpha * x[i];
}

// ------------------------------------------------------------------ host tables
double q2b(int a, double x) { return a == 0 ? 2.0 * (x - 0.5) * (x - 1.0) : a == 1 ? -4.0 * x * (x - 1.0) : 2.0 * x * (x - 0.5); }
double q2d(int a, double x) { return a == 0 ? 4.0 * x - 3.0 : a == 1 ? 4.0 - 8.0 * x : 4.0 * x - 1.0; }
double q1b(int a, double x) { return a == 0 ? 1.0 - x : x; }

}  // namespace

struct Assembler {
  int dim = 2;
  int pdisc = 0;                  // pressure: 0 continuous Q1, 1 discontinuous P1
  int64_t n = 0, ncell = 0;
  int ncd[3] = {1, 1, 1};
  Phys phys{};
  cudaStream_t s = nullptr;
  bool own_stream = false;
  DBuf<double> tab;               // N, dN, Np, w, Nf, dNf, wf
  Tables T{};
  DBuf<int> cell_dof;
  DBuf<unsigned> cell_flags;
  DBuf<int64_t> rowptr;
  DBuf<int> colind;
  DBuf<unsigned char> fixed;
  Basis1 B1{};
  // results of a call: [0] order key of min det F, [1] bits of max |R_i|, [2] entries outside the
  // pattern (low 32 bits); the host reads them through `host`
  DBuf<unsigned long long> res;
  unsigned long long* host = nullptr;   // pinned
  int64_t nnz = 0;
  std::string msg;
  ~Assembler() {
    if (host) cudaFreeHost(host);
    if (own_stream && s) cudaStreamDestroy(s);
  }
};

namespace {

void build_tables(Assembler& A, const double* h) {
  const int D = A.dim;
  const int NQ2 = D == 2 ? 9 : 27, NQ1 = A.pdisc ? D + 1 : (D == 2 ? 4 : 8), NQP = NQ2, NFP = D == 2 ? 3 : 9;
  // 3-point Gauss-Legendre rule on [0, 1]: nodes 1/2 -+ sqrt(3/5)/2, weights 5/18, 8/18, 5/18
  const double r = std::sqrt(0.6);
  const double gx[3] = {0.5 - 0.5 * r, 0.5, 0.5 + 0.5 * r};
  const double gw[3] = {5.0 / 18.0, 8.0 / 18.0, 5.0 / 18.0};
  std::vector<double> N(NQP * NQ2), dN(NQP * NQ2 * D), Np(NQP * NQ1), w(NQP);
  std::vector<double> Nf(NFP * NQ2), dNf(NFP * NQ2 * D), wf(NFP);
  double vol = 1.0;
  for (int d = 0; d < D; ++d) vol *= h[d];
  auto basis = [&](const double* xi, double* Nrow, double* dNrow, double* Nprow) {
    for (int a = 0; a < NQ2; ++a) {
      const int ai[3] = {a % 3, (a / 3) % 3, a / 9};
      double val = 1.0;
      for (int d = 0; d < D; ++d) val *= q2b(ai[d], xi[d]);
      Nrow[a] = val;
      for (int j = 0; j < D; ++j) {
        double g = 1.0;
        for (int d = 0; d < D; ++d) g *= (d == j) ? q2d(ai[d], xi[d]) / h[d] : q2b(ai[d], xi[d]);
        dNrow[a * D + j] = g;
      }
    }
    if (Nprow)
      for (int a = 0; a < NQ1; ++a) {
        double val = 1.0;
        if (A.pdisc) {
          val = a == 0 ? 1.0 : 2.0 * xi[a - 1] - 1.0;   // P1disc: 1 and the centred linears of the cell
        } else {
          const int ai[3] = {a % 2, (a / 2) % 2, a / 4};
          for (int d = 0; d < D; ++d) val *= q1b(ai[d], xi[d]);
        }
        Nprow[a] = val;
      }
  };
  for (int q = 0; q < NQP; ++q) {
    const int qi[3] = {q % 3, (q / 3) % 3, q / 9};
    double xi[3] = {0, 0, 0}, ww = vol;
    for (int d = 0; d < D; ++d) { xi[d] = gx[qi[d]]; ww *= gw[qi[d]]; }
    w[q] = ww;
    basis(xi, &N[q * NQ2], &dN[(size_t)q * NQ2 * D], &Np[q * NQ1]);
  }
  double area = 1.0;
  for (int d = 1; d < D; ++d) area *= h[d];
  for (int f = 0; f < NFP; ++f) {
    const int fi[2] = {f % 3, f / 3};
    double xi[3] = {1.0, 0.0, 0.0}, ww = area;
    for (int d = 1; d < D; ++d) { xi[d] = gx[fi[d - 1]]; ww *= gw[fi[d - 1]]; }
    wf[f] = ww;
    basis(xi, &Nf[f * NQ2], &dNf[(size_t)f * NQ2 * D], nullptr);
  }
  std::vector<double> M((size_t)NQ2 * NQ2, 0.0);
  for (int a = 0; a < NQ2; ++a)
    for (int b = 0; b < NQ2; ++b)
      for (int q = 0; q < NQP; ++q) M[a * NQ2 + b] += w[q] * N[q * NQ2 + a] * N[q * NQ2 + b];
  for (int q = 0; q < 3; ++q)
    for (int a = 0; a < 3; ++a) {
      A.B1.N[q][a] = q2b(a, gx[q]);
      for (int d = 0; d < D; ++d) A.B1.dN[d][q][a] = q2d(a, gx[q]) / h[d];
    }
  std::vector<double> all;
  size_t off[8];
  const std::vector<double>* parts[8] = {&N, &dN, &Np, &w, &Nf, &dNf, &wf, &M};
  for (int t = 0; t < 8; ++t) {
    off[t] = all.size();
    all.insert(all.end(), parts[t]->begin(), parts[t]->end());
  }
  A.tab.alloc(all.size());
  FSI_CUDA(cudaMemcpyAsync(A.tab.p, all.data(), sizeof(double) * all.size(), cudaMemcpyHostToDevice, A.s));
  FSI_CUDA(cudaStreamSynchronize(A.s));
  A.T = Tables{A.tab.p + off[0], A.tab.p + off[1], A.tab.p + off[2], A.tab.p + off[3],
               A.tab.p + off[4], A.tab.p + off[5], A.tab.p + off[6], A.tab.p + off[7]};
}

// f(geometry, cells) for each colour that has cells
template <int D, class F>
void for_colours(const Assembler& A, F&& f) {
  for (int col = 0; col < (1 << D); ++col) {
    CellGeom g{};
    int64_t cnt = 1;
    for (int d = 0; d < 3; ++d) {
      g.n[d] = A.ncd[d];
      if (d < D) {
        const int b = (col >> d) & 1;
        g.m[d] = (A.ncd[d] - b + 1) / 2;
        cnt *= g.m[d];
      } else {
        g.m[d] = 1;
      }
    }
    g.color = col;
    if (cnt == 0) continue;
    require(cnt < ((int64_t)1 << 31), "fsi_asm: too many cells for one launch");
    f(g, cnt);
    FSI_CHECK_LAUNCH();
  }
}

// Cells per CTA for a colour of cnt cells: as many as the tables take, but no more than leave every SM two
// CTAs.  What a CTA's cells cost is the FP64 pipe of its SM: with full groups on a mesh of a few
// hundred cells, a handful of SMs did all the work (14x7: Jacobian 517 us, now 257, residual 262, now 94; one
// CTA per cell and column chunk, before the groups, took 390 and 170).
inline int cells_per_cta(int64_t cnt, int most) {
  const int64_t spread = (cnt + 2 * device_sms() - 1) / (2 * device_sms());
  return (int)(spread < most ? spread : most);
}

template <int D, int PD>
void run_residual(Assembler& A, const double* U, const double* Uold, double* out) {
  constexpr size_t sm = sizeof(ResSmem<D, PD>);
  static OncePerDevice attr;
  once_per_device(attr, [](int) {
    FSI_CUDA(cudaFuncSetAttribute(k_residual<D, PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  });
  for_colours<D>(A, [&](const CellGeom& g, int64_t cnt) {
    const int per = cells_per_cta(cnt, Sh<D, PD>::RCELLS);
    k_residual<D, PD><<<div_up(cnt, per), kAsmThreads, sm, A.s>>>(
        g, cnt, per, A.T, A.phys, A.cell_dof.p, A.cell_flags.p, A.fixed.p, U, Uold, out, A.res.p);
  });
}

template <int D, int PD>
void run_jacobian(Assembler& A, const double* U, const double* Uold, double* vals) {
  constexpr size_t sm = sizeof(JacSmem<D, PD>);
  static_assert(sm <= 227 * 1024, "Jacobian tables exceed the shared memory of a CTA");
  static OncePerDevice attr;
  once_per_device(attr, [](int) {
    FSI_CUDA(cudaFuncSetAttribute(k_jacobian<D, PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  });
  for_colours<D>(A, [&](const CellGeom& g, int64_t cnt) {
    const int per = cells_per_cta(cnt, Sh<D, PD>::JCELLS);
    k_jacobian<D, PD><<<div_up(cnt, per), Sh<D, PD>::JTHREADS, sm, A.s>>>(
        g, cnt, per, A.T, A.B1, A.phys, A.cell_dof.p, A.cell_flags.p, A.rowptr.p, A.colind.p, A.fixed.p, U, Uold, vals,
        A.res.p, reinterpret_cast<int*>(A.res.p + 2));
  });
}

void begin(Assembler& A) {
  FSI_CUDA(cudaMemsetAsync(A.res.p, 0xFF, sizeof(unsigned long long), A.s));
  FSI_CUDA(cudaMemsetAsync(A.res.p + 1, 0, 2 * sizeof(unsigned long long), A.s));
}

void finish(Assembler& A, double* minJ, double* rmax) {
  FSI_CUDA(cudaMemcpyAsync(A.host, A.res.p, 3 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, A.s));
  FSI_CUDA(cudaStreamSynchronize(A.s));
  if (minJ) *minJ = A.host[0] == ~0ull ? 1e300 : order_value(A.host[0]);   // 1e300: no point with a finite det F
  if (rmax) std::memcpy(rmax, A.host + 1, sizeof(double));
  require((int)(A.host[2] & 0xFFFFFFFFull) == 0, "fsi_asm: a Jacobian entry falls outside the CSR pattern");
}

}  // namespace

void asm_residual(Assembler& A, const double* U, const double* Uold, double* R, double* minJ, double* rmax) {
  begin(A);
  FSI_CUDA(cudaMemsetAsync(R, 0, sizeof(double) * A.n, A.s));   // fixed rows stay 0
  if (A.dim == 2) {
    if (A.pdisc) run_residual<2, 1>(A, U, Uold, R); else run_residual<2, 0>(A, U, Uold, R);
  } else {
    if (A.pdisc) run_residual<3, 1>(A, U, Uold, R); else run_residual<3, 0>(A, U, Uold, R);
  }
  if (rmax) {
    const int cap = device_sms() * 8, g = div_up(A.n, 256);
    k_absmax<<<g < cap ? g : cap, 256, 0, A.s>>>(A.n, R, A.res.p + 1);
    FSI_CHECK_LAUNCH();
  }
  finish(A, minJ, rmax);
}

void asm_jacobian(Assembler& A, const double* U, const double* Uold, double* vals, double* minJ) {
  begin(A);
  FSI_CUDA(cudaMemsetAsync(vals, 0, sizeof(double) * A.nnz, A.s));
  if (A.dim == 2) {
    if (A.pdisc) run_jacobian<2, 1>(A, U, Uold, vals); else run_jacobian<2, 0>(A, U, Uold, vals);
  } else {
    if (A.pdisc) run_jacobian<3, 1>(A, U, Uold, vals); else run_jacobian<3, 0>(A, U, Uold, vals);
  }
  k_fixed_rows<<<div_up(A.n, 256), 256, 0, A.s>>>(A.n, A.rowptr.p, A.fixed.p, vals);
  FSI_CHECK_LAUNCH();
  finish(A, minJ, nullptr);
}

void asm_axpy(Assembler& A, double alpha, const double* x, double* y) {
  const int cap = device_sms() * 16;
  k_axpy_inplace<<<div_up(A.n, 256) < cap ? div_up(A.n, 256) : cap, 256, 0, A.s>>>(A.n, alpha, x, y);
  FSI_CHECK_LAUNCH();
  FSI_CUDA(cudaStreamSynchronize(A.s));
}

void asm_create(Assembler& A, const fsi_asm_mesh& m, const fsi_asm_physics& p, void* stream) {
  require(m.dim == 2 || m.dim == 3, "fsi_asm: dim must be 2 or 3");
  require(m.n > 0 && m.n < ((int64_t)1 << 31), "fsi_asm: n out of range");
  require(m.cell_dof && m.cell_flags && m.rowptr && m.colind && m.row_fixed, "fsi_asm: null mesh array");
  require(m.pressure == 0 || m.pressure == 1, "fsi_asm: pressure must be 0 (continuous Q1) or 1 (P1disc)");
  note_device_context();
  A.dim = m.dim;
  A.pdisc = m.pressure;
  A.n = m.n;
  A.ncell = 1;
  for (int d = 0; d < m.dim; ++d) {
    require(m.cells[d] >= 1 && m.h[d] > 0.0, "fsi_asm: cells and h must be positive");
    A.ncd[d] = m.cells[d];
    A.ncell *= m.cells[d];
  }
  require(p.theta > 0.0 && p.theta <= 1.0 && p.dt > 0.0, "fsi_asm: need 0 < theta <= 1 and dt > 0");
  A.phys = Phys{p.rho_f, p.nu_f, p.mu_s, p.lambda_s, p.rho_s, p.dt, p.theta};
  if (stream) {
    A.s = static_cast<cudaStream_t>(stream);
  } else {
    FSI_CUDA(cudaStreamCreateWithFlags(&A.s, cudaStreamNonBlocking));
    A.own_stream = true;
  }
  const int NL = 2 * (m.dim == 2 ? 9 : 27) * m.dim + (m.pressure ? m.dim + 1 : (m.dim == 2 ? 4 : 8));
  A.nnz = m.rowptr[m.n];
  for (int64_t c = 0; c < A.ncell * NL; ++c)
    require(m.cell_dof[c] >= 0 && m.cell_dof[c] < m.n, "fsi_asm: cell DOF out of range");
  build_tables(A, m.h);
  A.cell_dof.alloc((size_t)A.ncell * NL);
  A.cell_flags.alloc(A.ncell);
  A.rowptr.alloc(A.n + 1);
  A.colind.alloc(A.nnz > 0 ? A.nnz : 1);
  A.fixed.alloc(A.n);
  A.res.alloc(3);
  FSI_CUDA(cudaMallocHost(&A.host, 3 * sizeof(unsigned long long)));
  FSI_CUDA(cudaMemcpyAsync(A.cell_dof.p, m.cell_dof, sizeof(int) * A.ncell * NL, cudaMemcpyHostToDevice, A.s));
  FSI_CUDA(cudaMemcpyAsync(A.cell_flags.p, m.cell_flags, sizeof(unsigned) * A.ncell, cudaMemcpyHostToDevice, A.s));
  FSI_CUDA(cudaMemcpyAsync(A.rowptr.p, m.rowptr, sizeof(int64_t) * (A.n + 1), cudaMemcpyHostToDevice, A.s));
  if (A.nnz) FSI_CUDA(cudaMemcpyAsync(A.colind.p, m.colind, sizeof(int) * A.nnz, cudaMemcpyHostToDevice, A.s));
  FSI_CUDA(cudaMemcpyAsync(A.fixed.p, m.row_fixed, A.n, cudaMemcpyHostToDevice, A.s));
  FSI_CUDA(cudaStreamSynchronize(A.s));
}

}  // namespace fsi

// ====================================================================== C ABI
struct fsi_asm {
  fsi::Assembler A;
};

namespace {
thread_local std::string g_asm_create_error;

template <class F>
int asm_guarded(fsi_asm* a, F&& f) {
  std::string& err = a ? a->A.msg : g_asm_create_error;
  try {
    f();
    err.clear();
    return FSI_OK;
  } catch (const fsi::Error& e) {
    err = e.what();
    return e.code;
  } catch (const std::exception& e) {
    err = e.what();
    return FSI_ECUDA;
  }
}
}  // namespace

extern "C" {

int fsi_asm_create(fsi_asm** out, const fsi_asm_mesh* mesh, const fsi_asm_physics* phys, void* cuda_stream) {
  if (!out) return FSI_EINVAL;
  *out = nullptr;
  if (!mesh || !phys) return FSI_EINVAL;
  fsi_asm* a = nullptr;
  try {
    a = new fsi_asm();
  } catch (...) {
    return FSI_ENOMEM;
  }
  const int rc = asm_guarded(nullptr, [&] { fsi::asm_create(a->A, *mesh, *phys, cuda_stream); });
  if (rc != FSI_OK) {
    delete a;
    return rc;
  }
  *out = a;
  return FSI_OK;
}

int fsi_asm_residual(fsi_asm* a, const double* U_dev, const double* Uold_dev, double* R_dev, double* min_J,
                     double* r_absmax) {
  if (!a) return FSI_EINVAL;
  return asm_guarded(a, [&] {
    fsi::require(U_dev && R_dev, "fsi_asm_residual: null vector");
    fsi::asm_residual(a->A, U_dev, Uold_dev, R_dev, min_J, r_absmax);
  });
}

int fsi_asm_jacobian(fsi_asm* a, const double* U_dev, const double* Uold_dev, double* vals_dev, double* min_J) {
  if (!a) return FSI_EINVAL;
  return asm_guarded(a, [&] {
    fsi::require(U_dev && vals_dev, "fsi_asm_jacobian: null vector");
    fsi::asm_jacobian(a->A, U_dev, Uold_dev, vals_dev, min_J);
  });
}

int fsi_asm_axpy(fsi_asm* a, double alpha, const double* x_dev, double* y_dev) {
  if (!a) return FSI_EINVAL;
  return asm_guarded(a, [&] {
    fsi::require(x_dev && y_dev, "fsi_asm_axpy: null vector");
    fsi::asm_axpy(a->A, alpha, x_dev, y_dev);
  });
}

const char* fsi_asm_last_error(const fsi_asm* a) { return a ? a->A.msg.c_str() : g_asm_create_error.c_str(); }

void fsi_asm_free(fsi_asm* a) { delete a; }

}  // extern "C"
