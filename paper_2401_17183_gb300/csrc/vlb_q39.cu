// vlb_q39.cu -- the time step, initialisation, moments and state access for the
// 6th-order isotropic D3Q39 velocity set (vlb_q39.cuh) on periodic meshes, in
// FP64. Streaming is in place with the A-A pattern of the other kernels (even
// steps: slot a of q in, slot abar of q out; odd steps: slot abar of q - c_a
// in, slot a of q + c_a out), with neighbours wrapped periodically on every
// axis (each axis at least 3 cells long, speeds at most 3).
//
// The collision (section 2.2) takes directions in pairs (p, pbar = p + 19) with
// c_pbar = -c_p and writes the force map of Eq. 27 as a polynomial in U~ with
// coefficients of the cell's geometry and tau alone (Rec39, build_record39), as the
// D3Q19 kernel does: one chord step costs about 75 FP64 operations instead of a
// pass over the 39 directions, and N' is formed once, at the converged force.
// With Phi = J F, m = sum N, s_p = N_p + N_pbar, t_p = N_p - N_pbar, M_p = K_p +
// K_pbar, D_p = K_p - K_pbar, f^eq = rho w (1 + xe +- xo) (Eq. 33) and
// P = J deltaPi (Eq. 30), linear in the xo_p,
//   Phi_new = m G + sum_p (am M_p s_p + ad D_p t_p) - m/(2 tau) sum_p w_p M_p
//             - m/2 sum_p {w_p M_p xe_p / tau + Ao_p xo_p} - 1/2 TT Phi,
//   am = -(2 - 1/tau)/4, ad = 1/(4 tau),
//   Ao^i_p = w_p [D^i_p / tau - (1 - 1/(2 tau)) c_p.R^i.M_p],
//   R^i_kl = sum_p w_p M^i_p (c^k c^l / T0 - delta_kl) / T0,  TT^i_j = sum_p w_p D^i_p c^j_p / T0,
// and xe is linear in B = (g - delta) T0 + U~U~, xo in U and the symmetric C^jkl of Eq. 33.
// Where the records do not fit into device memory, every relation is evaluated
// direction pair by pair instead, with 12 values per cell (collide39).
// The link coefficients K^i_a = sum_j c^j_a Theta^i_j(q + c_a, q) (Eq. 11)
// come from the mesh's FP64 geometry, so the relations of Eqs. 27 and 30 read
//   sum_j c^j_a Theta^i_j(q - c_a, q) = -K^i_abar.
#include "vlb_addr.cuh"
#include "vlb_collide.cuh"
#include "vlb_q39.cuh"

namespace vlb {
namespace {

constexpr int kQ39 = 39, kH39 = 19;
constexpr int kQ39Threads = 128;

// the velocity set and weights as a table in constant memory: the direction
// loops below are not unrolled, and a warp reads one entry at a time
struct Q39Table {
  double c[kQ39][3];
  double w[kQ39];
};
constexpr Q39Table make_q39_table() {
  Q39Table t{};
  for (int a = 0; a < kQ39; a++) {
    for (int d = 0; d < 3; d++) t.c[a][d] = Lat<39>::c(a, d);
    t.w[a] = q39_w(a);
  }
  return t;
}
__constant__ Q39Table kT39 = make_q39_table();

struct Q39Args {
  double *f;  // populations [39][ncell]
  int64_t ncell;
  int64_t n[3];
  const double *J, *gl, *gu, *ginv, *K;
  // records of the polynomial force map (Rec39), or NULL
  const double *rec;
  // without them, per cell: the chord matrix H = (I - dG/dF)^-1 of the force map at the
  // rest state (row-major) and the rest state's force at rho = 1, 12 values;
  // NULL before q39_prepare has filled them
  const double *chord;
  double body[3];
  double tau, itau, tol;
  int32_t max_iter;
  int *err;
};

__device__ __forceinline__ int opp39(int a) { return a == 0 ? 0 : (a <= kH39 ? a + kH39 : a - kH39); }

__device__ __forceinline__ int64_t wrap(int64_t i, int64_t n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// cell index of q + s c_a (periodic on every axis; |c| <= 3 <= n)
__device__ __forceinline__ int64_t nb39(const Q39Args &A, const int64_t ic[3], int a, int s) {
  const int64_t i0 = wrap(ic[0] + s * Lat<39>::c(a, 0), A.n[0]);
  const int64_t i1 = wrap(ic[1] + s * Lat<39>::c(a, 1), A.n[1]);
  const int64_t i2 = wrap(ic[2] + s * Lat<39>::c(a, 2), A.n[2]);
  return (i0 * A.n[1] + i1) * A.n[2] + i2;
}

__device__ __forceinline__ void coords(const Q39Args &A, int64_t c, int64_t ic[3]) {
  ic[2] = c % A.n[2];
  const int64_t r = c / A.n[2];
  ic[1] = r % A.n[1];
  ic[0] = r / A.n[1];
}

// storage location of the arrived population N_a(q) (A-A)
template <bool ODD>
__device__ __forceinline__ int64_t src39(const Q39Args &A, int64_t c, const int64_t ic[3], int a) {
  if (!ODD || a == 0) return (int64_t)a * A.ncell + c;
  return (int64_t)opp39(a) * A.ncell + nb39(A, ic, a, -1);
}
// storage location that receives N'_a(q)
template <bool ODD>
__device__ __forceinline__ int64_t dst39(const Q39Args &A, int64_t c, const int64_t ic[3], int a) {
  if (!ODD) return (int64_t)opp39(a) * A.ncell + c;
  if (a == 0) return c;
  return (int64_t)a * A.ncell + nb39(A, ic, a, +1);
}

// g^ij - delta^ij of a cell (full 3 x 3) and G^i = G . g^i
__device__ void cell_metric(const Q39Args &A, int64_t c, double gd[3][3], double G[3]) {
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++) gd[i][j] = A.ginv[c * 6 + sym<3>(i, j)] - (i == j ? 1.0 : 0.0);
  for (int i = 0; i < 3; i++) {
    double s = 0.0;
    for (int d = 0; d < 3; d++) s += A.body[d] * A.gu[(c * 3 + i) * 3 + d];
    G[i] = s;
  }
}

// The two Hermite tensors of Eq. 33, with B^ij = (g^ij - delta^ij) T0 +
// U~^i U~^j and C^ijk = T0 [(g^ij U~^k - delta^ij U^k) + cyclic] + U~^i U~^j U~^k,
// V^i = C^ijj and tr B, formed once per evaluation
struct Herm39 {
  double B[3][3], C[3][3][3], V[3], trB;
};
__device__ void herm39(const double U[3], const double Ut[3], const double gd[3][3], Herm39 &h) {
  const double T0 = kT0_39;
  h.trB = 0.0;
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++) h.B[i][j] = gd[i][j] * T0 + Ut[i] * Ut[j];
  for (int i = 0; i < 3; i++) h.trB += h.B[i][i];
  // g^ij U~^k - delta^ij U^k = gd^ij U~^k + delta^ij (U~^k - U^k)
  auto term = [&](int i, int j, int k) { return gd[i][j] * Ut[k] + (i == j ? Ut[k] - U[k] : 0.0); };
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++)
      for (int k = 0; k < 3; k++)
        h.C[i][j][k] = T0 * (term(i, j, k) + term(j, k, i) + term(k, i, j)) + Ut[i] * Ut[j] * Ut[k];
  for (int i = 0; i < 3; i++) h.V[i] = h.C[i][0][0] + h.C[i][1][1] + h.C[i][2][2];
}

// The bracket of Eq. 33 for direction c split into its even part (the same
// for c and -c) and its odd part (opposite signs):
//   f^eq_{+-c} = rho w {ev +- od},  ev = 1 + (c.B.c / T0 - tr B) / (2 T0),
//   od = c.U / T0 + (C:ccc - 3 T0 c.V) / (6 T0^3),
// with the symmetric contractions over their distinct components (c.B.c from
// 6 terms, C:ccc from 10)
__device__ __forceinline__ void feq39_pair(const Herm39 &h, const double U[3], double x, double y, double z,
                                           double &ev, double &od) {
  const double T0 = kT0_39;
  const double cu = x * U[0] + y * U[1] + z * U[2];
  const double cV = x * h.V[0] + y * h.V[1] + z * h.V[2];
  const double cBc = x * x * h.B[0][0] + y * y * h.B[1][1] + z * z * h.B[2][2] +
                     2.0 * (x * y * h.B[0][1] + x * z * h.B[0][2] + y * z * h.B[1][2]);
  const double cCc = x * x * x * h.C[0][0][0] + y * y * y * h.C[1][1][1] + z * z * z * h.C[2][2][2] +
                     3.0 * (x * x * y * h.C[0][0][1] + x * x * z * h.C[0][0][2] + y * y * x * h.C[1][1][0] +
                            y * y * z * h.C[1][1][2] + z * z * x * h.C[2][2][0] + z * z * y * h.C[2][2][1]) +
                     6.0 * x * y * z * h.C[0][1][2];
  ev = 1.0 + (cBc / T0 - h.trB) / (2.0 * T0);
  od = cu / T0 + (cCc - 3.0 * T0 * cV) / (6.0 * T0 * T0 * T0);
}

// Eq. 33 for every direction (used at set-up and for initialisation)
__device__ void feq39(double rho, const double U[3], const double Ut[3], const double gd[3][3],
                      double f[kQ39]) {
  Herm39 h;
  herm39(U, Ut, gd, h);
  f[0] = rho * kT39.w[0] * (1.0 - h.trB / (2.0 * kT0_39));
#pragma unroll 1
  for (int p = 1; p <= kH39; p++) {
    double ev, od;
    feq39_pair(h, U, kT39.c[p][0], kT39.c[p][1], kT39.c[p][2], ev, od);
    f[p] = rho * kT39.w[p] * (ev + od);
    f[p + kH39] = rho * kT39.w[p] * (ev - od);
  }
}

// One evaluation of the collision at force F (Eqs. 20, 27, 30, 31, 33):
// post-collision N' and the updated F. Directions are taken in pairs
// (p, pbar = p + 19) with c_pbar = -c_p, so each pair's contractions are
// formed once and split into even and odd parts.
__device__ void eval39(const double N[kQ39], double J, double rho, const double U[3], const double F[3],
                       const double gd[3][3], const double G[3], const double *K, double tau,
                       double Np[kQ39], double Fn[3]) {
  const double T0 = kT0_39;
  double Ut[3];
  for (int i = 0; i < 3; i++) Ut[i] = U[i] + 0.5 * (F[i] / rho);
  Herm39 h;
  herm39(U, Ut, gd, h);
  // rho w_p times the even and odd parts of each pair's bracket
  double fe[kH39 + 1], fo[kH39 + 1];
  fe[0] = rho * kT39.w[0] * (1.0 - h.trB / (2.0 * T0));
  fo[0] = 0.0;
  // deltaPi^ij = -1/2 (1 - 1/(2 tau)) sum_a c^i_a (K^j_a + K^j_abar) f^eq_a   (Eq. 30);
  // over a pair, c_p (K_p + K_pbar) (f^eq_p - f^eq_pbar) = c_p (K_p + K_pbar) 2 rho w_p od_p
  double dP[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll 1
  for (int p = 1; p <= kH39; p++) {
    const double x = kT39.c[p][0], y = kT39.c[p][1], z = kT39.c[p][2];
    double ev, od;
    feq39_pair(h, U, x, y, z, ev, od);
    const double rw = rho * kT39.w[p];
    fe[p] = rw * ev;
    fo[p] = rw * od;
    const double cv[3] = {x, y, z};
    const double d2 = 2.0 * fo[p];
    for (int j = 0; j < 3; j++) {
      const double m = (K[p * 3 + j] + K[(p + kH39) * 3 + j]) * d2;
      for (int i = 0; i < 3; i++) dP[i][j] += cv[i] * m;
    }
  }
  const double cp = -0.5 * (1.0 - 1.0 / (2.0 * tau));
  double tr = 0.0;
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++) dP[i][j] *= cp;
  for (int i = 0; i < 3; i++) tr += dP[i][i];
  // c.dP.c over the diagonal and the symmetrised off-diagonal components
  const double s01 = dP[0][1] + dP[1][0], s02 = dP[0][2] + dP[2][0], s12 = dP[1][2] + dP[2][1];
  // deltaN_a = w_a J [c.F / T0 + (c.deltaPi.c / T0 - tr deltaPi) / T0]   (Eq. 31)
  // N'_a = N_a - (N_a - J f^eq_a) / tau + deltaN_a   (Eqs. 12, 20)
  Np[0] = N[0] - (N[0] - J * fe[0]) / tau + kT39.w[0] * J * (-tr / T0);
#pragma unroll 1
  for (int p = 1; p <= kH39; p++) {
    const double x = kT39.c[p][0], y = kT39.c[p][1], z = kT39.c[p][2];
    const double cF = x * F[0] + y * F[1] + z * F[2];
    const double cPc = x * x * dP[0][0] + y * y * dP[1][1] + z * z * dP[2][2] + x * y * s01 + x * z * s02 + y * z * s12;
    const double wJ = kT39.w[p] * J;
    const double dNe = wJ * ((cPc / T0 - tr) / T0), dNo = wJ * (cF / T0);
    const int pb = p + kH39;
    Np[p] = N[p] - (N[p] - J * (fe[p] + fo[p])) / tau + (dNe + dNo);
    Np[pb] = N[pb] - (N[pb] - J * (fe[p] - fo[p])) / tau + (dNe - dNo);
  }
  // J F^i = -1/2 sum_a (K^i_a N'_a + K^i_abar N_a) + J rho G^i   (Eq. 27 and the body force)
  for (int i = 0; i < 3; i++) {
    double s = 0.0;
    for (int a = 1; a < kQ39; a++) s += K[a * 3 + i] * Np[a] + K[opp39(a) * 3 + i] * N[a];
    Fn[i] = -0.5 * s / J + rho * G[i];
  }
}

// The local fixed point on F (Eq. 27 with the body force). With the cell's
// chord data ch: the chord iteration F <- F + H (G(F) - F) from rho F_rest
// (the map is homogeneous of degree one in (N, F) at rest, so rho F_rest is
// the rest state's fixed point at density rho); H inverts the linear part of
// G at rest, so a few evaluations suffice. Without it (ch NULL): the plain
// iteration F <- G(F) from F = 0. Converged when the change is at most
// tol max(rho, |F|); N' at the converged F (to within that change). False if
// max_iter is reached.
__device__ bool collide39(const double N[kQ39], double J, const double gd[3][3], const double G[3],
                          const double *K, const double *chord, int64_t c, double tau, double tol, int max_iter,
                          double Np[kQ39], double &rho, double U[3], double F[3]) {
  const double *ch = chord ? chord + c * 12 : nullptr;
  rho = 0.0;
  for (int a = 0; a < kQ39; a++) rho += N[a] / J;
  for (int i = 0; i < 3; i++) {
    double s = 0.0;
    for (int a = 0; a < kQ39; a++) s += kT39.c[a][i] * (N[a] / J);
    U[i] = s / rho;
    F[i] = ch ? rho * ch[9 + i] : 0.0;
  }
  bool conv = false;
  double Fn[3];
  for (int it = 0; it < max_iter; it++) {
    eval39(N, J, rho, U, F, gd, G, K, tau, Np, Fn);
    double diff = 0.0, fmax = 0.0;
    if (ch) {
      double r[3];
      for (int i = 0; i < 3; i++) r[i] = Fn[i] - F[i];
      for (int i = 0; i < 3; i++) {
        const double d = ch[3 * i] * r[0] + ch[3 * i + 1] * r[1] + ch[3 * i + 2] * r[2];
        F[i] += d;
        diff = maxnan(diff, fabs(d));
        fmax = maxnan(fmax, fabs(F[i]));
      }
    } else {
      for (int i = 0; i < 3; i++) {
        diff = maxnan(diff, fabs(Fn[i] - F[i]));
        fmax = maxnan(fmax, fabs(Fn[i]));
        F[i] = Fn[i];
      }
    }
    if (diff <= tol * (rho > fmax ? rho : fmax)) {
      conv = true;
      break;
    }
  }
  // N' at the converged F: with the chord iteration the last evaluation was
  // at the F that the final correction, below tol max(rho, |F|), moved off,
  // so its N' is kept; the plain iteration evaluates once more
  if (!(ch && conv)) eval39(N, J, rho, U, F, gd, G, K, tau, Np, Fn);
  return conv;
}

// Chord data of every cell: the rest state N = J f^eq(1, 0) of Eq. 33, its
// force F_rest by the plain iteration (to 1e-15), and the Jacobian of the map
// F -> G(F) there by central differences (G is a cubic polynomial in F, so
// the difference error is of the order of the step squared); H = (I - Jac)^-1.
__global__ void __launch_bounds__(kQ39Threads) k_prep39(const Q39Args A, double *out) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    double gd[3][3], G[3], U0[3] = {0.0, 0.0, 0.0}, N[kQ39], Np[kQ39], F[3] = {0.0, 0.0, 0.0}, Fn[3];
    cell_metric(A, c, gd, G);
    const double J = A.J[c];
    feq39(1.0, U0, U0, gd, N);
    for (int a = 0; a < kQ39; a++) N[a] *= J;
    const double *K = A.K + c * kQ39 * 3;
    for (int it = 0; it < 400; it++) {
      eval39(N, J, 1.0, U0, F, gd, G, K, A.tau, Np, Fn);
      double diff = 0.0, fm = 0.0;
      for (int i = 0; i < 3; i++) {
        diff = maxnan(diff, fabs(Fn[i] - F[i]));
        fm = maxnan(fm, fabs(Fn[i]));
        F[i] = Fn[i];
      }
      if (diff <= 1e-15 * (fm > 1.0 ? fm : 1.0)) break;
    }
    double Jac[3][3];
    const double h = 1e-6;
    for (int j = 0; j < 3; j++) {
      double Fp[3] = {F[0], F[1], F[2]}, Fm[3] = {F[0], F[1], F[2]}, Gp[3], Gm[3];
      Fp[j] += h;
      Fm[j] -= h;
      eval39(N, J, 1.0, U0, Fp, gd, G, K, A.tau, Np, Gp);
      eval39(N, J, 1.0, U0, Fm, gd, G, K, A.tau, Np, Gm);
      for (int i = 0; i < 3; i++) Jac[i][j] = (Gp[i] - Gm[i]) / (2.0 * h);
    }
    double M[3][3], C[3][3];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) M[i][j] = (i == j ? 1.0 : 0.0) - Jac[i][j];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) {
        const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
        C[i][j] = M[i1][j1] * M[i2][j2] - M[i1][j2] * M[i2][j1];
      }
    const double det = M[0][0] * C[0][0] + M[0][1] * C[0][1] + M[0][2] * C[0][2];
    double *o = out + c * 12;
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) o[3 * i + j] = C[j][i] / det;
    for (int i = 0; i < 3; i++) o[9 + i] = F[i];
  }
}

// ------------------------------------------------- the polynomial force map
// Record of one cell: value k of cell c at ((c / 32) NR + k) 32 + c % 32, so that a
// warp reads 256 consecutive bytes per value.
struct Rec39 {
  static constexpr int GD = 0;              // g^ij - delta^ij, packed (6)
  static constexpr int BC = GD + 6;         // terms of the map proportional to m (3)
  static constexpr int PO1 = BC + 3;        // coefficient of U, row-major (9)
  static constexpr int HM = PO1 + 9;        // chord matrix (9)
  static constexpr int QM = HM + 9;         // H times the coefficients of the 6 + 10 monomials (3 x 16)
  static constexpr int FR = QM + 48;        // F of the rest state at rho = 1 (3)
  static constexpr int IJ = FR + 3;         // 1 / J
  static constexpr int LK = IJ + 1;         // per pair: am M_p (3), ad D_p (3)
  static constexpr int NR = LK + 6 * kH39;
};
static_assert(Rec39::NR == kRec39, "record size");
__device__ __forceinline__ int64_t rec39(int64_t c) { return (c >> 5) * (Rec39::NR * 32) + (c & 31); }

// the distinct components of a symmetric third-rank tensor
__host__ __device__ constexpr int sym3(int i, int j, int k) {
  const int a = i < j ? (i < k ? i : k) : (j < k ? j : k), c = i > j ? (i > k ? i : k) : (j > k ? j : k);
  const int b = i + j + k - a - c;
  // 000 001 002 011 012 022 111 112 122 222
  return a == 0 ? (b == 0 ? c : b == 1 ? 2 + c : 5) : a == 1 ? (b == 1 ? 5 + c : 8) : 9;
}
__host__ __device__ constexpr int q39_len(int p) {   // largest |c| component of pair p
  const int x = Lat<39>::c(p, 0), y = Lat<39>::c(p, 1), z = Lat<39>::c(p, 2);
  const int ax = x < 0 ? -x : x, ay = y < 0 ? -y : y, az = z < 0 ? -z : z;
  return ax > ay ? (ax > az ? ax : az) : (ay > az ? ay : az);
}
__host__ __device__ constexpr int q39_nnz(int p) {
  return (Lat<39>::c(p, 0) != 0) + (Lat<39>::c(p, 1) != 0) + (Lat<39>::c(p, 2) != 0);
}

// polynomial part of a chord step: a^i = sum_k QM[i][k] monomial_k(U~)
template <typename LD>
__device__ __forceinline__ void map39(const double Ut[3], LD ld, double a[3]) {
  const double x = Ut[0], y = Ut[1], z = Ut[2];
  const double xx = x * x, yy = y * y, zz = z * z;
  const double mono[16] = {xx, x * y, x * z, yy, y * z, zz,
                           xx * x, xx * y, xx * z, x * yy, (x * y) * z, x * zz, yy * y, yy * z, y * zz, zz * z};
#pragma unroll
  for (int i = 0; i < 3; i++) {
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 16; k++) v = fma(ld(Rec39::QM + 16 * i + k), mono[k], v);
    a[i] = v;
  }
}

// Fills the record of every cell from its geometry (see the top of the file):
//   PE = R / (2 tau),  S^i_jkl = 1/(6 T0^3) sum_p Ao^i_p h^jkl_p,
//   h = ccc - T0 (c delta + cyclic),  PO1 = sum_p Ao_p c / T0,
//   LO^i_l = 3 T0 sum_jk (g - delta)_jk S^i_jkl,  LD^i_l = 3 T0 sum_j S^i_jjl,
// so that Phi_new = Pb - m/2 {PE : U~U~ + S : U~U~U~ + LO U~} - (TT + LD/2) Phi / 2 and, with
// U~ = U + Phi / (2m), A = LO/4 + (TT + LD/2)/2 and H = (I + A)^-1, the chord step is
// Phi <- H (Pc - m/2 Q(U~)), Pc = m BC + sum_p (am M s + ad D t) - m/2 (PO1 + LO) U.
__global__ void __launch_bounds__(kQ39Threads) k_prep39_rec(const Q39Args A, double *out) {
  const double T0 = kT0_39, itau = 1.0 / A.tau, am = -0.25 * (2.0 - itau), ad = 0.25 * itau;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    double *o = out + rec39(c);
    const double *K = A.K + c * kQ39 * 3;
    double gd[3][3], G[3];
    cell_metric(A, c, gd, G);
    const double J = A.J[c];
    double R[3][6], TT[3][3], KW[3];
    for (int i = 0; i < 3; i++) {
      KW[i] = 0.0;
      for (int k = 0; k < 6; k++) R[i][k] = 0.0;
      for (int j = 0; j < 3; j++) TT[i][j] = 0.0;
    }
#pragma unroll 1
    for (int p = 1; p <= kH39; p++) {
      const double cv[3] = {kT39.c[p][0], kT39.c[p][1], kT39.c[p][2]}, w = kT39.w[p];
#pragma unroll
      for (int i = 0; i < 3; i++) {
        const double M = K[p * 3 + i] + K[(p + kH39) * 3 + i], D = K[p * 3 + i] - K[(p + kH39) * 3 + i];
        o[(Rec39::LK + 6 * (p - 1) + i) * 32] = am * M;
        o[(Rec39::LK + 6 * (p - 1) + 3 + i) * 32] = ad * D;
        KW[i] += w * M;
#pragma unroll
        for (int k = 0; k < 3; k++) {
          TT[i][k] += w * D * cv[k] / T0;
#pragma unroll
          for (int l = k; l < 3; l++) R[i][sym<3>(k, l)] += w * M * (cv[k] * cv[l] / T0 - (k == l ? 1.0 : 0.0)) / T0;
        }
      }
    }
    double S[3][10], PO1[3][3];
    for (int i = 0; i < 3; i++) {
      for (int k = 0; k < 10; k++) S[i][k] = 0.0;
      for (int k = 0; k < 3; k++) PO1[i][k] = 0.0;
    }
#pragma unroll 1
    for (int p = 1; p <= kH39; p++) {
      const double cv[3] = {kT39.c[p][0], kT39.c[p][1], kT39.c[p][2]}, w = kT39.w[p];
      double M[3];
#pragma unroll
      for (int i = 0; i < 3; i++) M[i] = K[p * 3 + i] + K[(p + kH39) * 3 + i];
#pragma unroll
      for (int i = 0; i < 3; i++) {
        double cRM = 0.0;
#pragma unroll
        for (int k = 0; k < 3; k++)
#pragma unroll
          for (int l = 0; l < 3; l++) cRM += cv[k] * R[i][sym<3>(k, l)] * M[l];
        const double D = K[p * 3 + i] - K[(p + kH39) * 3 + i];
        const double Ao = w * (itau * D - (1.0 - 0.5 * itau) * cRM);
#pragma unroll
        for (int l = 0; l < 3; l++) PO1[i][l] += Ao * cv[l] / T0;
#pragma unroll
        for (int j = 0; j < 3; j++)
#pragma unroll
          for (int k = j; k < 3; k++)
#pragma unroll
            for (int l = k; l < 3; l++) {
              const double h = cv[j] * cv[k] * cv[l] - T0 * ((k == l ? cv[j] : 0.0) + (j == l ? cv[k] : 0.0) +
                                                             (j == k ? cv[l] : 0.0));
              S[i][sym3(j, k, l)] += Ao * h / (6.0 * T0 * T0 * T0);
            }
      }
    }
    double Am[3][3], LO[3][3], BC[3];
    for (int i = 0; i < 3; i++) {
      double ce = 0.0;
#pragma unroll
      for (int k = 0; k < 3; k++)
#pragma unroll
        for (int l = 0; l < 3; l++) ce += T0 * 0.5 * itau * R[i][sym<3>(k, l)] * gd[k][l];
      BC[i] = G[i] - 0.5 * itau * KW[i] - 0.5 * ce;
#pragma unroll
      for (int l = 0; l < 3; l++) {
        double lo = 0.0, ld = 0.0;
#pragma unroll
        for (int j = 0; j < 3; j++) {
          ld += 3.0 * T0 * S[i][sym3(j, j, l)];
#pragma unroll
          for (int k = 0; k < 3; k++) lo += 3.0 * T0 * gd[j][k] * S[i][sym3(j, k, l)];
        }
        LO[i][l] = lo;
        Am[i][l] = (i == l ? 1.0 : 0.0) + 0.25 * lo + 0.5 * (TT[i][l] + 0.5 * ld);
      }
    }
    double Hm[3][3];
    {
      double C[3][3];
#pragma unroll
      for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
          const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
          C[i][j] = Am[i1][j1] * Am[i2][j2] - Am[i1][j2] * Am[i2][j1];
        }
      const double det = Am[0][0] * C[0][0] + Am[0][1] * C[0][1] + Am[0][2] * C[0][2];
#pragma unroll
      for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) Hm[i][j] = C[j][i] / det;
    }
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int j = i; j < 3; j++) o[(Rec39::GD + sym<3>(i, j)) * 32] = gd[i][j];
    double QM[3][16];
#pragma unroll
    for (int i = 0; i < 3; i++) {
      o[(Rec39::BC + i) * 32] = BC[i];
#pragma unroll
      for (int l = 0; l < 3; l++) {
        o[(Rec39::PO1 + 3 * i + l) * 32] = PO1[i][l] + LO[i][l];
        o[(Rec39::HM + 3 * i + l) * 32] = Hm[i][l];
      }
#pragma unroll
      for (int k = 0; k < 3; k++)
#pragma unroll
        for (int l = k; l < 3; l++) {
          double v = 0.0;
#pragma unroll
          for (int j = 0; j < 3; j++) v += Hm[i][j] * R[j][sym<3>(k, l)];
          QM[i][sym<3>(k, l)] = (k == l ? 0.5 : 1.0) * itau * v;
        }
#pragma unroll
      for (int j = 0; j < 3; j++)
#pragma unroll
        for (int k = j; k < 3; k++)
#pragma unroll
          for (int l = k; l < 3; l++) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < 3; q++) v += Hm[i][q] * S[q][sym3(j, k, l)];
            QM[i][6 + sym3(j, k, l)] = (j == l ? 1.0 : j == k || k == l ? 3.0 : 6.0) * v;
          }
#pragma unroll
      for (int k = 0; k < 16; k++) o[(Rec39::QM + 16 * i + k) * 32] = QM[i][k];
    }
    o[Rec39::IJ * 32] = 1.0 / J;
    // the rest state (rho = 1, U = 0): N = J w (1 + xe) with B = (g - delta) T0, m = J
    double Pc[3], Pt[3], Phi[3] = {0.0, 0.0, 0.0}, trg = gd[0][0] + gd[1][1] + gd[2][2];
    for (int i = 0; i < 3; i++) Pc[i] = J * BC[i];
#pragma unroll 1
    for (int p = 1; p <= kH39; p++) {
      const double x = kT39.c[p][0], y = kT39.c[p][1], z = kT39.c[p][2];
      const double cgc = x * x * gd[0][0] + y * y * gd[1][1] + z * z * gd[2][2] +
                         2.0 * (x * y * gd[0][1] + x * z * gd[0][2] + y * z * gd[1][2]);
      const double sp = 2.0 * J * kT39.w[p] * (1.0 + 0.5 * (cgc / T0 - trg));
#pragma unroll
      for (int i = 0; i < 3; i++) Pc[i] += am * (K[p * 3 + i] + K[(p + kH39) * 3 + i]) * sp;
    }
    for (int i = 0; i < 3; i++) Pt[i] = Hm[i][0] * Pc[0] + Hm[i][1] * Pc[1] + Hm[i][2] * Pc[2];
    for (int it = 0; it < 100; it++) {
      double Ut[3], a[3], diff = 0.0, fm = 0.0;
      for (int i = 0; i < 3; i++) Ut[i] = 0.5 * Phi[i] / J;
      map39(Ut, [&](int k) { return QM[(k - Rec39::QM) / 16][(k - Rec39::QM) % 16]; }, a);
      for (int i = 0; i < 3; i++) {
        const double pn = Pt[i] - 0.5 * J * a[i];
        diff = maxnan(diff, fabs(pn - Phi[i]));
        fm = maxnan(fm, fabs(pn));
        Phi[i] = pn;
      }
      if (diff <= 1e-15 * (fm > J ? fm : J)) break;
    }
    for (int i = 0; i < 3; i++) o[(Rec39::FR + i) * 32] = Phi[i] / J;
  }
}

// One cell's arrived populations as pair sums and differences (s[0] = N_0)
// and what the collision makes of them. ld(k): record value k.
struct Cell39 {
  double s[kH39 + 1], t[kH39 + 1];
  double m, h2m, U[3], Phi[3];   // h2m = 1 / (2 m)
};
constexpr double kIT0_39 = 1.5;   // 1 / T0, exactly (a division takes some 15 FP64 operations)

// m, U and the force: the chord iteration Phi <- H (Pc - m/2 Q(U~)), started, tested
// and accepted as in FP64 D3Q19 cells (collide_f64): three evaluations in FP32 from
// Pt = H Pc, then FP64 ones until the change, or a bound on the next one, is at most
// tol max(m, |Phi|); below four iterations allowed from m F_rest
template <typename LD>
__device__ __forceinline__ bool force39(Cell39 &q, LD ld, double tol, int max_iter) {
  double m = q.s[0], mu[3] = {0.0, 0.0, 0.0}, Pc[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int p = 1; p <= kH39; p++) {
    m += q.s[p];
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const int ci = Lat<39>::c(p, i);
      if (ci == 1) mu[i] += q.t[p];
      else if (ci == -1) mu[i] -= q.t[p];
      else if (ci != 0) mu[i] = fma((double)ci, q.t[p], mu[i]);
      Pc[i] = fma(ld(Rec39::LK + 6 * (p - 1) + i), q.s[p], Pc[i]);
      Pc[i] = fma(ld(Rec39::LK + 6 * (p - 1) + 3 + i), q.t[p], Pc[i]);
    }
  }
  q.m = m;
  const double im = 1.0 / m, h2m = 0.5 * im, hm = 0.5 * m;
  q.h2m = h2m;
#pragma unroll
  for (int i = 0; i < 3; i++) q.U[i] = mu[i] * im;
#pragma unroll
  for (int i = 0; i < 3; i++) {
    Pc[i] = fma(m, ld(Rec39::BC + i), Pc[i]);
    // m/2 (PO1 + LO) U = 1/2 (PO1 + LO) (m U)
    double v = 0.0;
#pragma unroll
    for (int l = 0; l < 3; l++) v = fma(ld(Rec39::PO1 + 3 * i + l), mu[l], v);
    Pc[i] = fma(-0.5, v, Pc[i]);
  }
  double Pt[3];
#pragma unroll
  for (int i = 0; i < 3; i++)
    Pt[i] = fma(ld(Rec39::HM + 3 * i), Pc[0],
                fma(ld(Rec39::HM + 3 * i + 1), Pc[1], ld(Rec39::HM + 3 * i + 2) * Pc[2]));
  const Unit64 un(m);
  const float mf = trunc_f32(m, un.m), tolf = (float)tol;
  float lip = 1.0e30f;
  int it = 0;
  if (max_iter >= 4) {
    float Uf[3], Pf[3], df[3] = {0.f, 0.f, 0.f}, l2 = 0.f, l3 = 0.f, um = 0.f;
    const float hf = trunc_f32(h2m, un.inv), hmf = 0.5f * mf;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      Uf[i] = trunc_f32(q.U[i]);
      Pf[i] = trunc_f32(Pt[i], un.m);
    }
#pragma unroll 1
    for (int r = 0; r < 3; r++) {
      float x[3];
#pragma unroll
      for (int i = 0; i < 3; i++) {
        x[i] = fmaf(Pf[i] + df[i], hf, Uf[i]);
        um = fmaxf(um, fabsf(x[i]));
      }
      const float xx = x[0] * x[0], yy = x[1] * x[1], zz = x[2] * x[2];
      const float mono[16] = {xx, x[0] * x[1], x[0] * x[2], yy, x[1] * x[2], zz,
                              xx * x[0], xx * x[1], xx * x[2], x[0] * yy, (x[0] * x[1]) * x[2], x[0] * zz,
                              yy * x[1], yy * x[2], x[1] * zz, zz * x[2]};
      l2 = l3 = 0.f;
#pragma unroll
      for (int i = 0; i < 3; i++) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < 16; k++) {
          const float c = trunc_f32(ld(Rec39::QM + 16 * i + k));
          v = fmaf(c, mono[k], v);
          if (k < 6)
            l2 += fabsf(c);
          else
            l3 += fabsf(c);
        }
        df[i] = -hmf * v;
      }
    }
    it = 3;
    um *= 1.01f;
    lip = fmaf(0.5f * l2, um, 0.75f * l3 * um * um);
#pragma unroll
    for (int i = 0; i < 3; i++) q.Phi[i] = fma((double)df[i], un.one, Pt[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 3; i++) q.Phi[i] = m * ld(Rec39::FR + i);
  }
#pragma unroll 1
  while (it < max_iter) {
    double Ut[3], a[3];
    float diff = 0.f, pm = 0.f;
#pragma unroll
    for (int i = 0; i < 3; i++) Ut[i] = fma(q.Phi[i], h2m, q.U[i]);
    map39(Ut, ld, a);
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const double pn = fma(-hm, a[i], Pt[i]);
      diff = maxnan(diff, fabsf(trunc_f32(pn - q.Phi[i], un.m)));
      pm = maxnan(pm, fabsf(trunc_f32(pn, un.m)));
      q.Phi[i] = pn;
    }
    it++;
    const float scale = tolf * maxnan(mf, pm);
    if (diff <= scale || 64.f * lip * diff <= scale) return true;
  }
  return false;
}

// Even and odd parts of the equilibrium bracket over the pairs, folded by the kind
// of pair, with the sums that several pairs share formed once. Even: y0 + c.Y.c for a
// symmetric Y. Odd: c.u + k C:ccc for symmetric C; with b^i = k C^iii, q^ji = 3 k C^jji,
// d = 6 k C^012,
//   axis of length L:  L u_i + L^3 b_i,
//   corner (1 s1 s2):  a_0 + s1 a_1 + s2 a_2 + s1 s2 d,  a_i = u_i + b_i + sum_{j != i} q_ji,
//   (2 s_i, 2 s_j):    s_i e_ij + s_j e_ji,  e_ij = 2 u_i + 8 (b_i + q_ji).
// (Every axis vector of the positive half points along +i, every corner has c^0 = 1.)
__host__ __device__ constexpr int q39_axis(int p, int k) {   // k-th non-zero axis of pair p
  int n = 0;
  for (int i = 0; i < 3; i++)
    if (Lat<39>::c(p, i) != 0) {
      if (n == k) return i;
      n++;
    }
  return -1;
}
struct Odd39 {
  double u2[3], u[3], b[3], ap, am, a2, e[3][3], d;
  __device__ __forceinline__ Odd39(const double (&uu)[3], const double (&kC)[10]) {
    double a[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
      u[i] = uu[i];
      u2[i] = uu[i] + uu[i];
      b[i] = kC[sym3(i, i, i)];
      a[i] = u[i] + b[i];
#pragma unroll
      for (int j = 0; j < 3; j++) {
        if (j == i) continue;
        const double q = kC[sym3(j, j, i)];
        a[i] = fma(3.0, q, a[i]);
        e[i][j] = fma(8.0, fma(3.0, q, b[i]), u2[i]);
      }
    }
    ap = a[0] + a[1];
    am = a[0] - a[1];
    a2 = a[2];
    d = 6.0 * kC[sym3(0, 1, 2)];
  }
  __device__ __forceinline__ double operator()(int p) const {
    const int L = q39_len(p), nz = q39_nnz(p), i = q39_axis(p, 0), j = q39_axis(p, 1);
    if (nz == 1) return L == 1 ? u[i] + b[i] : L == 2 ? fma(8.0, b[i], u2[i]) : fma(27.0, b[i], u2[i] + u[i]);
    if (nz == 3) {
      const int s1 = Lat<39>::c(p, 1), s2 = Lat<39>::c(p, 2);
      const double t = s1 > 0 ? ap : am, v = s2 > 0 ? t + a2 : t - a2;
      return s1 * s2 > 0 ? v + d : v - d;
    }
    const double v = Lat<39>::c(p, i) > 0 ? e[i][j] : -e[i][j];
    return Lat<39>::c(p, j) > 0 ? v + e[j][i] : v - e[j][i];
  }
};
struct Even39 {
  double y0, Y[6], corner, plane[3];   // plane[k]: the two axes other than k
  __device__ __forceinline__ Even39(double y, const double (&Yv)[6]) {
    y0 = y;
#pragma unroll
    for (int k = 0; k < 6; k++) Y[k] = Yv[k];
    const double s01 = Y[sym<3>(0, 0)] + Y[sym<3>(1, 1)];
    corner = y0 + (s01 + Y[sym<3>(2, 2)]);
    plane[2] = fma(4.0, s01, y0);
    plane[1] = fma(4.0, Y[sym<3>(0, 0)] + Y[sym<3>(2, 2)], y0);
    plane[0] = fma(4.0, Y[sym<3>(1, 1)] + Y[sym<3>(2, 2)], y0);
  }
  __device__ __forceinline__ double operator()(int p) const {
    const int L = q39_len(p), nz = q39_nnz(p), i = q39_axis(p, 0), j = q39_axis(p, 1);
    if (nz == 1) return L == 1 ? y0 + Y[sym<3>(i, i)] : fma((double)(L * L), Y[sym<3>(i, i)], y0);
    if (nz == 2) return fma(2.0 * Lat<39>::c(p, i) * Lat<39>::c(p, j), Y[sym<3>(i, j)], plane[3 - i - j]);
    const double s1 = Lat<39>::c(p, 1), s2 = Lat<39>::c(p, 2);
    return fma(2.0 * s1, Y[sym<3>(0, 1)], fma(2.0 * s2, Y[sym<3>(0, 2)], fma(2.0 * s1 * s2, Y[sym<3>(1, 2)], corner)));
  }
};

// B (packed) and C / (6 T0^3), u = U / T0 - V / (2 T0^2) of Eq. 33 (V^i = C^ijj)
__device__ __forceinline__ void herm39_packed(const double (&gd)[6], const double U[3], const double Ut[3],
                                              double (&B)[6], double (&kC)[10], double (&u)[3]) {
  const double T0 = kT0_39;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = i; j < 3; j++) B[sym<3>(i, j)] = fma(gd[sym<3>(i, j)], T0, Ut[i] * Ut[j]);
  const double k = 1.0 / (6.0 * T0 * T0 * T0), kt = k * T0;
  double du[3];
#pragma unroll
  for (int i = 0; i < 3; i++) du[i] = Ut[i] - U[i];
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = i; j < 3; j++)
#pragma unroll
      for (int l = j; l < 3; l++) {
        double v = gd[sym<3>(i, j)] * Ut[l];
        v = fma(gd[sym<3>(j, l)], Ut[i], v);
        v = fma(gd[sym<3>(i, l)], Ut[j], v);
        if (i == j) v += du[l];
        if (j == l) v += du[i];
        if (i == l) v += du[j];
        kC[sym3(i, j, l)] = fma(k, (Ut[i] * Ut[j]) * Ut[l], kt * v);
      }
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const double v = kC[sym3(i, 0, 0)] + kC[sym3(i, 1, 1)] + kC[sym3(i, 2, 2)];
    u[i] = fma(-3.0 * T0, v, U[i] * kIT0_39);
  }
}

template <bool ODD>
__device__ __forceinline__ void pull39(const Q39Args &A, int64_t c, const int64_t ic[3], Cell39 &q) {
  q.s[0] = A.f[c];
  q.t[0] = 0.0;
#pragma unroll
  for (int p = 1; p <= kH39; p++) {
    const double a = A.f[src39<ODD>(A, c, ic, p)], b = A.f[src39<ODD>(A, c, ic, p + kH39)];
    q.s[p] = a + b;
    q.t[p] = a - b;
  }
}

// One time step with the polynomial force map. Bounded by the FP64 pipe (two
// lanes per clock and SM): about 900 FP64 operations per cell update, against 3,000 per
// evaluation of the map direction by direction. 64^3 cells: 0.42 ms a step (620
// MLUPS), 168 registers, three blocks per SM; 5.9 ms direction by direction, 0.80 ms with
// all evaluations of the map in FP64 and divisions by T0, 0.66 ms with the first three
// in FP32 (see force39), 0.42 ms with the shared sums of Odd39 and Even39.
template <bool ODD>
__global__ void __launch_bounds__(kQ39Threads, 3) k_step39_rec(const Q39Args A) {
  const int64_t c = (int64_t)blockIdx.x * kQ39Threads + threadIdx.x;
  if (c >= A.ncell) return;
  int64_t ic[3];
  coords(A, c, ic);
  const double *rec = A.rec + rec39(c);
  auto ld = [&](int k) { return __ldg(rec + k * 32); };
  Cell39 q;
  pull39<ODD>(A, c, ic, q);
  if (!force39(q, ld, A.tol, A.max_iter)) atomicOr(A.err, ERR_NOCONV);
  const double itau = A.itau;
  double Ut[3], gd[6], B[6], kC[10], u[3];
#pragma unroll
  for (int i = 0; i < 3; i++) Ut[i] = fma(q.Phi[i], q.h2m, q.U[i]);
#pragma unroll
  for (int i = 0; i < 6; i++) gd[i] = ld(Rec39::GD + i);
  herm39_packed(gd, q.U, Ut, B, kC, u);
  const Odd39 xo(u, kC);
  // P^kl = J deltaPi^kl = 2 m sum_p w_p c^k am M^l_p xo_p  (Eq. 30), its symmetric part
  double P[3][3];
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int l = 0; l < 3; l++) P[k][l] = 0.0;
#pragma unroll
  for (int p = 1; p <= kH39; p++) {
    const double x = q39_w(p) * q39_len(p) * xo(p);
#pragma unroll
    for (int l = 0; l < 3; l++) {
      const double M = ld(Rec39::LK + 6 * (p - 1) + l);
#pragma unroll
      for (int k = 0; k < 3; k++) {
        // (pair k + 1 is the first with a component along k)
        if (p == k + 1) P[k][l] = M * x;
        else if (Lat<39>::c(p, k) > 0) P[k][l] = fma(M, x, P[k][l]);
        else if (Lat<39>::c(p, k) < 0) P[k][l] = fma(-M, x, P[k][l]);
      }
    }
  }
  // N'_p = (1 - 1/tau) N_p + w [y0 + c.Y.c] +- w [(m/tau) xo + c.Phi / T0], the even part
  // (m/tau)(1 + xe) + (c.P.c / T0 - tr P) / T0 with xe = (c.B.c / T0 - tr B) / (2 T0)
  const double mt = q.m * itau, m2 = 2.0 * q.m;
  double Y[6], kZ[10], uz[3];
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = i; j < 3; j++)
      Y[sym<3>(i, j)] = (0.5 * mt * B[sym<3>(i, j)] + m2 * (i == j ? P[i][i] : 0.5 * (P[i][j] + P[j][i]))) * (kIT0_39 * kIT0_39);
  const double y0 = mt * (1.0 - (0.5 * kIT0_39) * (B[0] + B[3] + B[5])) - (kIT0_39 * m2) * (P[0][0] + P[1][1] + P[2][2]);
#pragma unroll
  for (int k = 0; k < 10; k++) kZ[k] = mt * kC[k];
#pragma unroll
  for (int i = 0; i < 3; i++) uz[i] = fma(mt, u[i], q.Phi[i] * kIT0_39);
  const Odd39 zo(uz, kZ);
  const Even39 ze(y0, Y);
  const double omt = 1.0 - itau, h = 0.5 * omt;
  A.f[c] = fma(omt, q.s[0], q39_w(0) * y0);
#pragma unroll
  for (int p = 1; p <= kH39; p++) {
    const double ev = fma(h, q.s[p], q39_w(p) * ze(p));
    const double od = fma(h, q.t[p], q39_w(p) * zo(p));
    A.f[dst39<ODD>(A, c, ic, p)] = ev + od;
    A.f[dst39<ODD>(A, c, ic, p + kH39)] = ev - od;
  }
}

template <bool ODD>
__global__ void __launch_bounds__(kQ39Threads) k_step39(const Q39Args A) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    int64_t ic[3];
    coords(A, c, ic);
    double N[kQ39], Np[kQ39];
#pragma unroll 1
    for (int a = 0; a < kQ39; a++) N[a] = A.f[src39<ODD>(A, c, ic, a)];
    double gd[3][3], G[3], rho, U[3], F[3];
    cell_metric(A, c, gd, G);
    if (!collide39(N, A.J[c], gd, G, A.K + c * kQ39 * 3, A.chord, c, A.tau, A.tol, A.max_iter, Np, rho, U, F))
      atomicOr(A.err, ERR_NOCONV);
#pragma unroll 1
    for (int a = 0; a < kQ39; a++) A.f[dst39<ODD>(A, c, ic, a)] = Np[a];
  }
}

__global__ void __launch_bounds__(kQ39Threads) k_init39(const Q39Args A, const double *rho, const double *u) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    double gd[6], U[3], B[6], kC[10], uu[3];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int j = i; j < 3; j++) gd[sym<3>(i, j)] = A.ginv[c * 6 + sym<3>(i, j)] - (i == j ? 1.0 : 0.0);
#pragma unroll
    for (int i = 0; i < 3; i++) {
      double s = 0.0;
#pragma unroll
      for (int d = 0; d < 3; d++) s += u[c * 3 + d] * A.gu[(c * 3 + i) * 3 + d];  // U^i = u . g^i
      U[i] = s;
    }
    herm39_packed(gd, U, U, B, kC, uu);
    const Odd39 xo(uu, kC);
    // N = J rho w (1 + xe +- xo)
    const double m = A.J[c] * rho[c];
    double Y[6];
#pragma unroll
    for (int i = 0; i < 6; i++) Y[i] = B[i] * (0.5 * kIT0_39 * kIT0_39);
    const double y0 = 1.0 - (0.5 * kIT0_39) * (B[0] + B[3] + B[5]);
    const Even39 xe(y0, Y);
    A.f[c] = m * (q39_w(0) * y0);
#pragma unroll
    for (int p = 1; p <= kH39; p++) {
      const double ev = xe(p), od = xo(p), mw = m * q39_w(p);
      A.f[(int64_t)p * A.ncell + c] = mw * (ev + od);
      A.f[(int64_t)(p + kH39) * A.ncell + c] = mw * (ev - od);
    }
  }
}

__device__ __forceinline__ double warp_sum39(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// rho [ncell], u [ncell][3], u~ [ncell][3] into out; per-block conservation
// sums (mass, P = sum e_a N_a, M = sum 1/2 [e_a(q) + e_a(q - c_a)] N_a) into
// partial[block][7]. M is regrouped so that a cell needs only its own tangents:
// with p = q - c_a in its second half, M = 1/2 sum_p g_i(p) sum_a c^i_a [N_a(p) +
// N_a(p + c_a)], and N_a(p + c_a) sits at slot a of p + c_a (even parity) or at slot
// abar of p (odd). REC: the polynomial force map, else collide39.
template <bool ODD, bool REC>
__global__ void __launch_bounds__(kMomThreads) k_moments39(const Q39Args A, double *out, double *partial) {
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    int64_t ic[3];
    coords(A, c, ic);
    double mass, rho, U[3], aF[3], bP[3] = {0.0, 0.0, 0.0}, bN[3] = {0.0, 0.0, 0.0};   // aF = F / (2 rho)
    if constexpr (REC) {
      Cell39 q;
      pull39<ODD>(A, c, ic, q);
      const double *rec = A.rec + rec39(c);
      auto ld = [&](int k) { return __ldg(rec + k * 32); };
      if (!force39(q, ld, A.tol, A.max_iter)) atomicOr(A.err, ERR_NOCONV);
      mass = q.m;
      rho = q.m * ld(Rec39::IJ);
#pragma unroll
      for (int i = 0; i < 3; i++) {
        U[i] = q.U[i];
        aF[i] = q.Phi[i] * q.h2m;
        bP[i] = q.U[i] * q.m;
      }
    } else {
      double N[kQ39], Np[kQ39], gd[3][3], G[3], F[3];
#pragma unroll 1
      for (int a = 0; a < kQ39; a++) N[a] = A.f[src39<ODD>(A, c, ic, a)];
      cell_metric(A, c, gd, G);
      if (!collide39(N, A.J[c], gd, G, A.K + c * kQ39 * 3, A.chord, c, A.tau, A.tol, A.max_iter, Np, rho, U, F))
        atomicOr(A.err, ERR_NOCONV);
      mass = 0.0;
      for (int a = 0; a < kQ39; a++) mass += N[a];
      for (int i = 0; i < 3; i++) {
        aF[i] = 0.5 * (F[i] / rho);
        for (int a = 0; a < kQ39; a++) bP[i] += kT39.c[a][i] * N[a];
      }
    }
    double gl[9];
#pragma unroll
    for (int k = 0; k < 9; k++) gl[k] = A.gl[c * 9 + k];
    out[c] = rho;
    bool finite = isfinite(rho);
#pragma unroll
    for (int d = 0; d < 3; d++) {
      double uu = 0.0, ut = 0.0;
#pragma unroll
      for (int i = 0; i < 3; i++) {
        uu += U[i] * gl[i * 3 + d];             // u = U^i g_i (Eq. 34)
        ut += (U[i] + aF[i]) * gl[i * 3 + d];   // u~ = U~^i g_i
      }
      out[A.ncell + c * 3 + d] = uu;
      out[A.ncell * 4 + c * 3 + d] = ut;
      finite = finite && isfinite(uu) && isfinite(ut);
    }
    if (!finite) atomicOr(A.err, ERR_NONFINITE);
    // sum_a c_a N_a(p + c_a), the pair (p, pbar) at a time
#pragma unroll
    for (int p = 1; p <= kH39; p++) {
      const double a = ODD ? A.f[(int64_t)(p + kH39) * A.ncell + c] : A.f[(int64_t)p * A.ncell + nb39(A, ic, p, +1)];
      const double b = ODD ? A.f[(int64_t)p * A.ncell + c] : A.f[(int64_t)(p + kH39) * A.ncell + nb39(A, ic, p, -1)];
      const double t = a - b;
#pragma unroll
      for (int i = 0; i < 3; i++) {
        const int ci = Lat<39>::c(p, i);
        if (ci != 0) bN[i] = fma((double)ci, t, bN[i]);
      }
    }
    acc[0] += mass;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      double pp = 0.0, nn = 0.0;
#pragma unroll
      for (int i = 0; i < 3; i++) {
        pp += gl[i * 3 + d] * bP[i];
        nn += gl[i * 3 + d] * bN[i];
      }
      acc[1 + d] += pp;
      acc[4 + d] += 0.5 * (pp + nn);
    }
  }
  __shared__ double sh[7][kMomThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < 7; k++) {
    const double s = warp_sum39(acc[k]);
    if (lane == 0) sh[k][warp] = s;
  }
  __syncthreads();
  if (warp == 0) {
    for (int k = 0; k < 7; k++) {
      double s = lane < (int)(blockDim.x >> 5) ? sh[k][lane] : 0.0;
      s = warp_sum39(s);
      if (lane == 0) partial[(int64_t)blockIdx.x * 7 + k] = s;
    }
  }
}

template <bool ODD>
__global__ void k_get39(const Q39Args A, double *N_out) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    int64_t ic[3];
    coords(A, c, ic);
    for (int a = 0; a < kQ39; a++) N_out[(int64_t)a * A.ncell + c] = A.f[src39<ODD>(A, c, ic, a)];
  }
}

template <bool ODD>
__global__ void k_set39(const Q39Args A, const double *N_in) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < A.ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    int64_t ic[3];
    coords(A, c, ic);
    for (int a = 0; a < kQ39; a++) A.f[src39<ODD>(A, c, ic, a)] = N_in[(int64_t)a * A.ncell + c];
  }
}

// per block: [min J, -max J, min f^eq_rest / w, min g^ii, -max g^ii]
__global__ void __launch_bounds__(kStatThreads) k_stats39(const double *J, const double *ginv, int64_t ncell,
                                                         double *partial) {
  double v[5] = {1e300, 1e300, 1e300, 1e300, 1e300};
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    double gd[3][3], U0[3] = {0, 0, 0}, f[kQ39];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) gd[i][j] = ginv[c * 6 + sym<3>(i, j)] - (i == j ? 1.0 : 0.0);
    feq39(1.0, U0, U0, gd, f);
    v[0] = fmin(v[0], J[c]);
    v[1] = fmin(v[1], -J[c]);
    for (int a = 0; a < kQ39; a++) v[2] = fmin(v[2], f[a] / q39_w(a));
    for (int i = 0; i < 3; i++) {
      const double g = ginv[c * 6 + sym<3>(i, i)];
      v[3] = fmin(v[3], g);
      v[4] = fmin(v[4], -g);
    }
  }
  __shared__ double sh[5][kStatThreads];
  for (int k = 0; k < 5; k++) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 5; k++) {
      double m = sh[k][0];
      for (int t = 1; t < (int)blockDim.x; t++) m = fmin(m, sh[k][t]);
      partial[(int64_t)blockIdx.x * 5 + k] = m;
    }
  }
}

Q39Args make_args(const vlb_sim *sim) {
  const vlb_mesh *m = sim->mesh;
  Q39Args A;
  A.f = static_cast<double *>(sim->d_f);
  A.ncell = m->ncell;
  for (int d = 0; d < 3; d++) {
    A.n[d] = m->md.n[d];
    A.body[d] = sim->p.body_force[d];
  }
  A.J = m->d_J;
  A.gl = m->d_gl;
  A.gu = m->d_gu;
  A.ginv = m->d_ginv;
  A.K = m->d_K;
  A.rec = sim->nc == kRec39 ? static_cast<const double *>(sim->d_coef) : nullptr;
  A.chord = sim->nc == kRec39 ? nullptr : static_cast<const double *>(sim->d_coef);
  A.tau = sim->p.tau;
  A.itau = 1.0 / A.tau;
  A.tol = sim->p.tol;
  A.max_iter = sim->p.max_iter;
  A.err = sim->d_err;
  return A;
}

unsigned grid_for(int64_t ncell, int threads) {
  int dev = 0, nsm = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (ncell + threads - 1) / threads;
  const int64_t cap = (int64_t)nsm * 16;
  return (unsigned)(want < cap ? (want > 0 ? want : 1) : cap);
}

}  // namespace

cudaError_t q39_mesh_stats(const vlb_mesh *m, double *d_partial, int64_t nblk, cudaStream_t s) {
  k_stats39<<<(unsigned)nblk, kStatThreads, 0, s>>>(m->d_J, m->d_ginv, m->ncell, d_partial);
  return cudaGetLastError();
}

cudaError_t q39_prepare(const vlb_sim *sim, cudaStream_t s) {
  Q39Args A = make_args(sim);
  A.chord = nullptr;
  double *out = static_cast<double *>(sim->d_coef);
  if (A.rec)
    k_prep39_rec<<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A, out);
  else
    k_prep39<<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A, out);
  return cudaGetLastError();
}

cudaError_t q39_init(const vlb_sim *sim, const double *d_rho, const double *d_u, cudaStream_t s) {
  const Q39Args A = make_args(sim);
  k_init39<<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A, d_rho, d_u);
  return cudaGetLastError();
}

cudaError_t q39_step(const vlb_sim *sim, int odd, cudaStream_t s) {
  const Q39Args A = make_args(sim);
  if (A.rec) {
    const unsigned blocks = (unsigned)((A.ncell + kQ39Threads - 1) / kQ39Threads);
    if (odd)
      k_step39_rec<true><<<blocks, kQ39Threads, 0, s>>>(A);
    else
      k_step39_rec<false><<<blocks, kQ39Threads, 0, s>>>(A);
    return cudaGetLastError();
  }
  if (odd)
    k_step39<true><<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A);
  else
    k_step39<false><<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A);
  return cudaGetLastError();
}

cudaError_t q39_moments(const vlb_sim *sim, double *d_out, double *d_partial, int64_t nblk, cudaStream_t s) {
  const Q39Args A = make_args(sim);
  const unsigned n = (unsigned)nblk;
  if (sim->t & 1) {
    if (A.rec)
      k_moments39<true, true><<<n, kMomThreads, 0, s>>>(A, d_out, d_partial);
    else
      k_moments39<true, false><<<n, kMomThreads, 0, s>>>(A, d_out, d_partial);
  } else {
    if (A.rec)
      k_moments39<false, true><<<n, kMomThreads, 0, s>>>(A, d_out, d_partial);
    else
      k_moments39<false, false><<<n, kMomThreads, 0, s>>>(A, d_out, d_partial);
  }
  return cudaGetLastError();
}

cudaError_t q39_get_state(const vlb_sim *sim, double *d_N, cudaStream_t s) {
  const Q39Args A = make_args(sim);
  if (sim->t & 1)
    k_get39<true><<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A, d_N);
  else
    k_get39<false><<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A, d_N);
  return cudaGetLastError();
}

// written in the layout of time 0 (even), which the caller then sets
cudaError_t q39_set_state(const vlb_sim *sim, const double *d_N, cudaStream_t s) {
  const Q39Args A = make_args(sim);
  k_set39<false><<<grid_for(A.ncell, kQ39Threads), kQ39Threads, 0, s>>>(A, d_N);
  return cudaGetLastError();
}

}  // namespace vlb
