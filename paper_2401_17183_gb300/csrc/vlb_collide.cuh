// vlb_collide.cuh -- the local part of one time step for one cell (section 2.2):
// moments (Eqs. 14, 15, 17), the implicit inertial force F (Eq. 27, with
// deltaPi of Eq. 30 and deltaN of Eq. 31), the curvilinear equilibrium
// (Eq. 33) with U~ = U + F/(2 rho), and the BGK post-collision populations
// N' = N + Omega + deltaN (Eqs. 12, 20). Shared by the step, moments and
// coefficient-packing kernels.
//
// Populations enter and leave as deviations d_a = N_a - w_a n_ref from a
// uniform reference n_ref = rho_0 J_ref (n_ref = 0 gives plain populations).
// The reference is the same in every cell, so advection and bounce-back move
// deviations exactly as they move populations, while every product below
// works on small numbers: that keeps FP32 rounding relative to the deviation,
// not to N. The force is carried as Phi = J F.
//
// Directions come in pairs (p, pbar = p + H) with c_pbar = -c_p; every sum over
// directions is a sum over pairs of an even part (same for p and pbar) and an
// odd part (opposite signs), with the link coefficients stored as
// M_p = K_p + K_pbar and D_p = K_p - K_pbar (stored with the weights they
// carry in the constant part of the map).
//
// The map Phi -> Phi_new of Eq. 27 is evaluated in a reduced form. Writing
//   N'_a - w_a n_ref = (1 - 1/tau) d_a + w_a (mdev + m x_a)/tau + deltaN_a,
// with J f^eq_a = w_a m (1 + x_a) and x_p = xe_p + xo_p, x_pbar = xe_p - xo_p,
// deltaN_p = E_p + O_p, deltaN_pbar = E_p - O_p (Eq. 31, 1/T0 = 3),
//   E_p = 3 w_p J (3 c_p.S.c_p - tr S),  O_p = 3 w_p c_p.Phi,
// S the symmetric part of deltaPi (Eq. 30), linear in the xo_q, gives
//   Phi_new = Pb - 1/2 { m [sum_p Ae_p xe_p + sum_p Ao_p xo_p] + T Phi },
// where Pb holds everything fixed during the iteration. Because xe_p is
// linear in B = gd T0 + U~ U~ and xo_p linear in U and in C^kkl (k != l),
// the pair sums collapse into a polynomial in U~ with per-cell constant
// coefficients (build_record):
//   Phi_new = Pb' - 1/2 { m [PE : U~U~ + PO2 : (U~^k)^2 U~^l + LO U~] + TL Phi },
//   Pb' = Pb - 1/2 m (CE + PO1 U).
// The post-collision populations themselves are formed once, at the converged
// Phi, direction by direction.
//
// In FP32, pairs of identical operations run in the two lanes of packed FP32
// instructions (sm_100 and later): a direction pair (p, pbar) of the final
// pass, rows 0 and 1 of the map and of the chord correction, and components 0
// and 1 of the constant part, each pair with the same roundings in the same
// order as two scalar operations.
#pragma once

#include "vlb_internal.cuh"

namespace vlb {

template <int Q, typename R>
struct CollideState {
  static constexpr int D = Lat<Q>::D;
  R rho;
  R U[D];
  R F[D];
  int iters;
  bool conv;
};

// Extruded meshes (EXT; D3Q19, plane records): the first two coordinates of a cell's
// position do not depend on the fastest axis and the third on nothing else (vlb_mesh::
// extruded). Then K^2_a = 0, g^02 = g^12 = 0, and K_a depends on (c^0_a, c^1_a) alone, so that
//  - the nine pairs have four sets of link coefficients: pairs 1, 6 and 7 share those of
//    pair 1, pairs 2, 8 and 9 those of pair 2, pair 3 has none;
//  - component 2 of Phi is m G^2, outside the iteration (row and column 2 of H - I and
//    of PO1, row 2 of the map and CE^2, KW^2 are zero);
//  - of the map's twelve monomials, those odd in U~^2 have coefficient zero.
// The steps are bound by issue (FP32, 16 bits) and by the FP64 pipe: 100 steps with reset and
// moments of D3Q19 channels, FP64 64^3 22.2 -> 17.0 ms, FP32 75 x 67 x 101 2.9 -> 2.6 ms.
// 16-bit storage (FR0) keeps the order of every sum and with it the rounding of every
// population: where all of these entries are zero in the FP32 records (vlb_sim::zero_ext,
// k_zero_entries) it leaves out the terms that they multiply, pair 3 and row and column 2
// of the map among them, and a product with zero changes no sum. FP16 128^3: 69.9 -> 60.6 us
// a step over both parities (55.4 with the sums regrouped as above, and other roundings).
template <bool EXT, int D>
__device__ constexpr bool map_mono(int s) {   // has monomial s of a chord step a coefficient?
  return !EXT || !(s == sym<D>(0, 2) || s == sym<D>(1, 2) || s == D * (D + 1) / 2 + offd<D>(0, 2) ||
                   s == D * (D + 1) / 2 + offd<D>(1, 2));
}

// D x D inverse (D = 2 or 3) by cofactors, FP64
template <int D>
__device__ void inverse_small(const double (&A)[D][D], double (&X)[D][D]) {
  if (D == 2) {
    const double det = A[0][0] * A[1][1] - A[0][1] * A[1][0];
    X[0][0] = A[1][1] / det;
    X[0][1] = -A[0][1] / det;
    X[1][0] = -A[1][0] / det;
    X[1][1] = A[0][0] / det;
  } else {
    double C[D][D];
    for (int i = 0; i < D; i++)
      for (int j = 0; j < D; j++) {
        const int i1 = (i + 1) % D, i2 = (i + 2) % D, j1 = (j + 1) % D, j2 = (j + 2) % D;
        C[i][j] = A[i1][j1] * A[i2][j2] - A[i1][j2] * A[i2][j1];
      }
    double det = 0.0;
    for (int j = 0; j < D; j++) det += A[0][j] * C[0][j];
    for (int i = 0; i < D; i++)
      for (int j = 0; j < D; j++) X[i][j] = C[j][i] / det;
  }
}

// Coefficient record of one cell in FP64 from its geometry: J, g^ij (packed),
// G^i = G . g^i and the link coefficients K^i_a (Eq. 25). Every entry is
// filled except FR, the rest state and UW, which are left zero. With itau = 1/tau,
// cpi = -(1 - itau/2) and the pair sums over p = 1..H:
//   R^i_kl  = sum_p w_p M^i_p (3 c^k_p c^l_p - delta_kl)
//   Ao^i_p  = w_p [itau D^i_p + 3 cpi c_p.R^i.M_p]    (xo_p: BGK part and, via S, E_p)
//   PE^i_kl = (3/2) itau R^i_kl                        (xe_p: BGK part)
//   PO1^i_l = 3 sum_p Ao^i_p c^l_p
//   PO2^i_kl = (9/2) sum_p Ao^i_p c^l_p (3 (c^k_p)^2 - 1),  k != l
//   TT^i_j  = 3 sum_p w_p D^i_p c^j_p                  (O_p)
//   LO^i_j  = T0 [sum_{k != j} PO2^i_kj gd_kk + 2 sum_{l != j} PO2^i_jl gd_jl]
//   LD^i_j  = T0 sum_{k != j} PO2^i_kj,   TL = TT + LD / 2
//   CE^i    = T0 sum_kl PE^i_kl gd_kl
// so that the map of Eq. 27 reads
//   Phi_new = Pb' - 1/2 { m [PE : U~U~ + PO2 : (U~^k)^2 U~^l + LO U~] + TL Phi },
//   Pb' = Pb - 1/2 m (CE + PO1 U).
// With U~ = U + Phi / (2m) the LO term splits into 1/2 m LO U and LO Phi / 4,
// so Phi_new = Pc - 1/2 m Q(U~) - A Phi with Pc = Pb - 1/2 m (CE + (PO1 + LO) U),
// Q = PE : U~U~ + PO2 : (U~^k)^2 U~^l and A = LO/4 + TL/2, the part of the
// map's Jacobian that stays as U -> 0. The chord step with H = (I + A)^-1,
//   Phi <- Phi + H (Phi_new - Phi) = H (Pc - 1/2 m Q(U~)),
// therefore needs only H, H PE and H PO2; the record stores PO1 + LO in
// place of PO1, H - I, and H PE, H PO2 side by side (QM). PE is taken over k <= l
// with the off-diagonal entries doubled (U~U~ is symmetric).
template <int Q>
__device__ void build_record(double J, const double *ginv, const double *G,
                             const double (&K)[Q][Lat<Q>::D], double tau, double *rec) {
  using L = CoefLayout<Q>;
  constexpr int D = Lat<Q>::D, H = Lat<Q>::H, NS = L::NS;
  const double T0 = kT0, itau = 1.0 / tau, cpi = -(1.0 - 0.5 * itau);
  for (int k = 0; k < L::NC; k++) rec[k] = 0.0;
  rec[L::J] = J;
  rec[L::IJ] = 1.0 / J;
  double gd[D][D];
  for (int i = 0; i < D; i++)
    for (int j = 0; j < D; j++) gd[i][j] = ginv[sym<D>(i, j)] - (i == j ? 1.0 : 0.0);
  for (int i = 0; i < D; i++)
    for (int j = i; j < D; j++) rec[L::GH + sym<D>(i, j)] = 0.5 * gd[i][j];
  for (int i = 0; i < D; i++) {
    rec[L::BODY + i] = G[i];
    double s = 0.0;
    for (int a = 1; a < Q; a++) s += lat_w<Q, double>(a) * K[a][i];
    rec[L::KW + i] = s;
  }
  double M[H + 1][D], Dk[H + 1][D], c[H + 1][D], w[H + 1];
  for (int p = 1; p <= H; p++) {
    w[p] = lat_w<Q, double>(p);
    for (int i = 0; i < D; i++) {
      M[p][i] = K[p][i] + K[p + H][i];
      Dk[p][i] = K[p][i] - K[p + H][i];
      c[p][i] = Lat<Q>::c(p, i);
      // stored with the weights they carry in the constant part of the map
      rec[L::mp(p, i)] = -0.25 * (2.0 - itau) * M[p][i];
      rec[L::dk(p, i)] = 0.25 * itau * Dk[p][i];
    }
  }
  double Rt[D][D][D];
  for (int i = 0; i < D; i++)
    for (int k = 0; k < D; k++)
      for (int l = 0; l < D; l++) {
        double s = 0.0;
        for (int p = 1; p <= H; p++)
          s += w[p] * M[p][i] * (3.0 * c[p][k] * c[p][l] - (k == l ? 1.0 : 0.0));
        Rt[i][k][l] = s;
      }
  double Ao[H + 1][D];
  for (int p = 1; p <= H; p++)
    for (int i = 0; i < D; i++) {
      double cRM = 0.0;
      for (int k = 0; k < D; k++)
        for (int l = 0; l < D; l++) cRM += c[p][k] * Rt[i][k][l] * M[p][l];
      Ao[p][i] = w[p] * (itau * Dk[p][i] + 3.0 * cpi * cRM);
    }
  double PE[D][NS], PO2[D][D][D], PO1[D][D], LO[D][D], TL[D][D];
  for (int i = 0; i < D; i++) {
    double ce = 0.0;
    for (int k = 0; k < D; k++)
      for (int l = 0; l < D; l++) {
        const double pe = 1.5 * itau * Rt[i][k][l];
        ce += T0 * pe * gd[k][l];
        if (k <= l) PE[i][sym<D>(k, l)] = (k == l ? 1.0 : 2.0) * pe;
      }
    rec[L::CE + i] = ce;
    for (int l = 0; l < D; l++) {
      double s = 0.0;
      for (int p = 1; p <= H; p++) s += Ao[p][i] * c[p][l];
      PO1[i][l] = 3.0 * s;
    }
    for (int k = 0; k < D; k++)
      for (int l = 0; l < D; l++) {
        PO2[i][k][l] = 0.0;
        if (k == l) continue;
        double s = 0.0;
        for (int p = 1; p <= H; p++) s += Ao[p][i] * c[p][l] * (3.0 * c[p][k] * c[p][k] - 1.0);
        PO2[i][k][l] = 4.5 * s;
      }
  }
  for (int i = 0; i < D; i++)
    for (int j = 0; j < D; j++) {
      double tt = 0.0;
      for (int p = 1; p <= H; p++) tt += 3.0 * w[p] * Dk[p][i] * c[p][j];
      double lo = 0.0, ld = 0.0;
      for (int k = 0; k < D; k++) {
        if (k == j) continue;
        lo += T0 * (PO2[i][k][j] * gd[k][k] + 2.0 * PO2[i][j][k] * gd[j][k]);
        ld += T0 * PO2[i][k][j];
      }
      LO[i][j] = lo;
      TL[i][j] = tt + 0.5 * ld;
      rec[L::PO1 + i * D + j] = PO1[i][j] + lo;
    }
  double A[D][D], Hm[D][D];
  for (int i = 0; i < D; i++)
    for (int j = 0; j < D; j++) A[i][j] = (i == j ? 1.0 : 0.0) + 0.25 * LO[i][j] + 0.5 * TL[i][j];
  inverse_small<D>(A, Hm);
  // H - I: its entries are of the size of A, so rounding them leaves the
  // product (H - I) Pc, and with it the fixed point, far more accurate than
  // rounding H itself would
  for (int i = 0; i < D; i++)
    for (int j = 0; j < D; j++) rec[L::row(L::HM, D, i, j)] = Hm[i][j] - (i == j ? 1.0 : 0.0);
  for (int i = 0; i < D; i++) {
    for (int s = 0; s < NS; s++) {
      double v = 0.0;
      for (int j = 0; j < D; j++) v += Hm[i][j] * PE[j][s];
      rec[L::row(L::QM, L::NQ, i, s)] = v;
    }
    for (int k = 0; k < D; k++)
      for (int l = 0; l < D; l++) {
        if (k == l) continue;
        double v = 0.0;
        for (int j = 0; j < D; j++) v += Hm[i][j] * PO2[j][k][l];
        rec[L::row(L::QM, L::NQ, i, NS + offd<D>(k, l))] = v;
      }
  }
}

// x y = p + e exactly (FMA two-product)
__device__ __forceinline__ float two_prod_err(float x, float y, float p) { return fmaf(x, y, -p); }
__device__ __forceinline__ double two_prod_err(double x, double y, double p) { return fma(x, y, -p); }

// packed FP32 helpers: both lanes the same value
__device__ __forceinline__ float2 bcast2(float v) { return make_float2(v, v); }

// A record as the collision reads it: values by their CoefLayout index, pairs and
// quads where they are aligned. In memory (shared, global or local):
template <typename R>
struct PtrRecord {
  const R *__restrict__ p;
  __device__ __forceinline__ R operator[](int k) const { return p[k]; }
  __device__ __forceinline__ float4 v4(int k) const { return *reinterpret_cast<const float4 *>(p + k); }
  __device__ __forceinline__ float2 v2(int k) const { return *reinterpret_cast<const float2 *>(p + k); }
};

// A CellLayout record in registers with the entries it leaves out, formed in FP32
// from the link coefficients a_p = am M_p, d_p = ad D_p (see build_record):
//   R = sum_p w a (3 c c - I) / am,  Ao = w [4 d + (6 / am) c.R'.a]  with R' = am R,
//   PE = (3/2) (itau / am) R',  PO1, PO2, LO, LD from Ao,  TT = 12 tau sum_p w d c,
//   A = LO/4 + (TT + LD/2)/2,  H - I = -(I + A)^-1 A,  QM = (PE, PO2) + (H - I)(PE, PO2).
// About 450 FP32 operations per cell against the 57 values (D3Q19) they replace; PO1,
// H - I and QM multiply U, Pc and U U, so their rounding is far below that of the
// terms stored: against an 80-bit run the populations' error after 1 and 20 steps is 0.96 to
// 1.02 times that with records formed in FP64 (twelve meshes, D2Q9 and D3Q19;
// u 0.98 to 1.04, geometric mean 1.00). Every index is a constant after unrolling: v lives in registers.
template <int Q>
struct CellRecord {
  using L = CoefLayout<Q>;
  using CL = CellLayout<Q>;
  static constexpr int D = L::D, H = L::H, NS = L::NS, NQ = L::NQ;
  float v[L::RR];
  __device__ __forceinline__ float operator[](int k) const { return v[k]; }
  __device__ __forceinline__ float4 v4(int k) const { return make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]); }
  __device__ __forceinline__ float2 v2(int k) const { return make_float2(v[k], v[k + 1]); }
  // cell: index within [0, ncell); k6am = 6 / am, kpe = (3/2) itau / am, ktt = 12 tau
  __device__ __forceinline__ void load(const float4 *__restrict__ rec, int64_t cell) {
    const float4 *p = rec + (cell >> 5) * (CL::NG * 32) + (cell & 31);
#pragma unroll
    for (int g = 0; g < CL::NG; g++) {
      const float4 q = __ldcs(p + g * 32);
      const float e[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (CL::entry(4 * g + u) >= 0) v[CL::entry(4 * g + u)] = e[u];
    }
  }
  // the values as if just read: a loop that keeps the record may not move
  // arithmetic on it out of its body, where products and sums would be contracted
  // differently from the step kernel's
  __device__ __forceinline__ void opaque() {
#pragma unroll
    for (int k = 0; k < L::RR; k++)
      if (k <= L::IJ || (k >= L::MPD && k < L::MPD + 2 * H * D) || (k >= L::HM && k < L::HM + D * D) ||
          (k >= L::QM && k < L::QM + D * NQ))
        asm volatile("" : "+f"(v[k]));
  }
  __device__ __forceinline__ float2 a01(int p) const { return make_float2(v[L::mp(p, 0)], v[L::mp(p, 1)]); }
  __device__ __forceinline__ float2 d01(int p) const { return make_float2(v[L::dk(p, 0)], v[L::dk(p, 1)]); }
  __device__ __forceinline__ void form(float k6am, float kpe, float ktt) {
    // components 0 and 1 in the two lanes, component 2 (D = 3) apart
    float2 R0[NS], S1[D], TT[D], C2[D][D], A0[D];   // R', 3-sum of Ao c, TT, PO2, A
    float R2[NS], S1z[D], TTz[D], C2z[D][D], A2[D];
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = k; l < D; l++) {
        float2 r = make_float2(0.f, 0.f);
        float rz = 0.f;
#pragma unroll
        for (int p = 1; p <= H; p++) {
          const float c = lat_w<Q, float>(p) * (float)(3 * Lat<Q>::c(p, k) * Lat<Q>::c(p, l) - (k == l ? 1 : 0));
          if (3 * Lat<Q>::c(p, k) * Lat<Q>::c(p, l) - (k == l ? 1 : 0) == 0) continue;
          r = __ffma2_rn(bcast2(c), a01(p), r);
          if constexpr (D == 3) rz = fmaf(c, v[L::mp(p, 2)], rz);
        }
        R0[sym<D>(k, l)] = r;
        R2[sym<D>(k, l)] = rz;
      }
#pragma unroll
    for (int k = 0; k < D; k++) {
      S1[k] = TT[k] = make_float2(0.f, 0.f);
      S1z[k] = TTz[k] = 0.f;
#pragma unroll
      for (int l = 0; l < D; l++) {
        C2[k][l] = make_float2(0.f, 0.f);
        C2z[k][l] = 0.f;
      }
    }
#pragma unroll
    for (int p = 1; p <= H; p++) {
      // c.R'.a, component by component of a
      float2 x = make_float2(0.f, 0.f);
      float xz = 0.f;
#pragma unroll
      for (int l = 0; l < D; l++) {
        float2 cr = make_float2(0.f, 0.f);
        float crz = 0.f;
#pragma unroll
        for (int k = 0; k < D; k++) {
          const int ck = Lat<Q>::c(p, k);
          if (ck == 0) continue;
          cr = __ffma2_rn(bcast2((float)ck), R0[sym<D>(k, l)], cr);
          if constexpr (D == 3) crz = fmaf((float)ck, R2[sym<D>(k, l)], crz);
        }
        const float al = v[L::mp(p, l)];
        x = __ffma2_rn(cr, bcast2(al), x);
        if constexpr (D == 3) xz = fmaf(crz, al, xz);
      }
      const float w = lat_w<Q, float>(p), wk = w * k6am;
      const float2 Ao = __ffma2_rn(bcast2(wk), x, __fmul2_rn(bcast2(4.f * w), d01(p)));
      const float Aoz = D == 3 ? fmaf(wk, xz, (4.f * w) * v[L::dk(p, 2)]) : 0.f;
#pragma unroll
      for (int l = 0; l < D; l++) {
        const int cl = Lat<Q>::c(p, l);
        if (cl == 0) continue;
        S1[l] = __ffma2_rn(bcast2(3.f * cl), Ao, S1[l]);
        TT[l] = __ffma2_rn(bcast2(w * cl), d01(p), TT[l]);
        if constexpr (D == 3) {
          S1z[l] = fmaf(3.f * cl, Aoz, S1z[l]);
          TTz[l] = fmaf(w * cl, v[L::dk(p, 2)], TTz[l]);
        }
#pragma unroll
        for (int k = 0; k < D; k++) {
          if (k == l) continue;
          const float c = 4.5f * cl * (float)(3 * Lat<Q>::c(p, k) * Lat<Q>::c(p, k) - 1);
          C2[k][l] = __ffma2_rn(bcast2(c), Ao, C2[k][l]);
          if constexpr (D == 3) C2z[k][l] = fmaf(c, Aoz, C2z[k][l]);
        }
      }
    }
    // LO^i_j = (2/3) [sum_{k != j} PO2^i_kj GH_kk + 2 sum_{l != j} PO2^i_jl GH_jl], PO1 + LO, A
#pragma unroll
    for (int j = 0; j < D; j++) {
      float2 lo = make_float2(0.f, 0.f), ld = make_float2(0.f, 0.f);
      float loz = 0.f, ldz = 0.f;
#pragma unroll
      for (int k = 0; k < D; k++) {
        if (k == j) continue;
        const float gkk = (2.f / 3.f) * v[L::GH + sym<D>(k, k)], gjk = (4.f / 3.f) * v[L::GH + sym<D>(j, k)];
        lo = __ffma2_rn(C2[k][j], bcast2(gkk), __ffma2_rn(C2[j][k], bcast2(gjk), lo));
        ld = __fadd2_rn(ld, C2[k][j]);
        if constexpr (D == 3) {
          loz = fmaf(C2z[k][j], gkk, fmaf(C2z[j][k], gjk, loz));
          ldz += C2z[k][j];
        }
      }
      const float2 po = __fadd2_rn(S1[j], lo);
      v[L::PO1 + j] = po.x;
      v[L::PO1 + D + j] = po.y;
      if constexpr (D == 3) v[L::PO1 + 2 * D + j] = S1z[j] + loz;
      // A = LO/4 + TT/2 + LD/4, LD = T0 sum PO2
      A0[j] = __ffma2_rn(bcast2(0.25f), lo, __ffma2_rn(bcast2(0.5f * ktt), TT[j], __fmul2_rn(bcast2(1.f / 12.f), ld)));
      A2[j] = fmaf(0.25f, loz, fmaf(0.5f * ktt, TTz[j], (1.f / 12.f) * ldz));
    }
    // H - I = -(I + A)^-1 A
    float B[D][D], Am[D][D], Hi[D][D];
#pragma unroll
    for (int j = 0; j < D; j++) {
      Am[0][j] = A0[j].x;
      Am[1][j] = A0[j].y;
      if constexpr (D == 3) Am[2][j] = A2[j];
#pragma unroll
      for (int i = 0; i < D; i++) B[i][j] = Am[i][j] + (i == j ? 1.f : 0.f);
    }
    if constexpr (D == 2) {
      const float id = -1.f / (B[0][0] * B[1][1] - B[0][1] * B[1][0]);
      Hi[0][0] = B[1][1] * id;
      Hi[0][1] = -B[0][1] * id;
      Hi[1][0] = -B[1][0] * id;
      Hi[1][1] = B[0][0] * id;
    } else {
      float C[D][D], det = 0.f;
#pragma unroll
      for (int i = 0; i < D; i++)
#pragma unroll
        for (int j = 0; j < D; j++) {
          const int i1 = (i + 1) % D, i2 = (i + 2) % D, j1 = (j + 1) % D, j2 = (j + 2) % D;
          C[i][j] = fmaf(B[i1][j1], B[i2][j2], -(B[i1][j2] * B[i2][j1]));
        }
#pragma unroll
      for (int j = 0; j < D; j++) det = fmaf(B[0][j], C[0][j], det);
      const float id = -1.f / det;
#pragma unroll
      for (int i = 0; i < D; i++)
#pragma unroll
        for (int j = 0; j < D; j++) Hi[i][j] = C[j][i] * id;
    }
    float2 H0[D];
    float Hz[D];
#pragma unroll
    for (int j = 0; j < D; j++) {
      float h[D];
#pragma unroll
      for (int i = 0; i < D; i++) {
        h[i] = 0.f;
#pragma unroll
        for (int k = 0; k < D; k++) h[i] = fmaf(Hi[i][k], Am[k][j], h[i]);
        v[L::row(L::HM, D, i, j)] = h[i];
      }
      H0[j] = make_float2(h[0], h[1]);
      Hz[j] = D == 3 ? h[D - 1] : 0.f;
    }
    // QM = X + (H - I) X for the columns X of (PE, PO2)
    auto column = [&](int s, float2 x, float xz) {
      float2 y = __ffma2_rn(H0[0], bcast2(x.x), __ffma2_rn(H0[1], bcast2(x.y), x));
      if constexpr (D == 3) {
        y = __ffma2_rn(H0[D - 1], bcast2(xz), y);
        v[L::row(L::QM, NQ, 2, s)] = fmaf(Hz[0], x.x, fmaf(Hz[1], x.y, fmaf(Hz[D - 1], xz, xz)));
      }
      v[L::row(L::QM, NQ, 0, s)] = y.x;
      v[L::row(L::QM, NQ, 1, s)] = y.y;
    };
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = k; l < D; l++) {
        const float c = k == l ? kpe : 2.f * kpe;
        column(sym<D>(k, l), __fmul2_rn(bcast2(c), R0[sym<D>(k, l)]), c * R2[sym<D>(k, l)]);
      }
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = 0; l < D; l++)
        if (k != l) column(NS + offd<D>(k, l), C2[k][l], C2z[k][l]);
  }
};
// the factors of CellRecord::form
struct CellFactors {
  float k6am, kpe, ktt;
};
inline CellFactors cell_factors(double tau) {
  const double itau = 1.0 / tau, am = -0.25 * (2.0 - itau);
  return CellFactors{(float)(6.0 / am), (float)(1.5 * itau / am), (float)(12.0 * tau)};
}

// The weights times 1/T0 = 3 of the axis (a1) and diagonal (a2) directions,
// chosen so that the identities of Eq. 10 that the momentum balance of a
// collision rests on hold exactly in R, not merely to rounding:
//   first moment of the U term of f^eq and of deltaN (Eqs. 28, 32),
//     3 sum_a w_a c_a c_a = I:        2 a1 + 4 a2 = 1 (D2Q9), 2 a1 + 8 a2 = 1 (D3Q19);
//   no momentum in the third-order Hermite part of Eq. 33, whose axis terms
//   carry b1 = 4 a2 (D2Q9) or 2 a2 (D3Q19) in place of a1.
// With 1/18 and 1/36 (or 1/9 and 1/36) rounded to FP32 each identity is off
// by about 3e-8, and every collision then changes the momentum by that
// fraction of U (or of the third-order part) -- an error that grows linearly
// with the number of steps. One constant is rounded; the others follow from
// the identities, and every operation in between is exact (scaling by powers
// of two, Sterbenz).
template <int Q, typename R>
struct MomentWeights;
template <typename R>
struct MomentWeights<19, R> {
  static constexpr R a2 = R(1) / R(12);
  static constexpr R a1 = (R(1) - R(8) * a2) / R(2);
  static constexpr R b1 = R(2) * a2;
  static_assert(R(2) * a1 + R(8) * a2 == R(1), "3 sum w c c = I must hold exactly");
  static_assert(R(4) * a2 - R(2) * b1 == R(0), "the cubic Hermite part must carry no momentum");
};
template <typename R>
struct MomentWeights<9, R> {
  static constexpr R a1 = R(1) / R(3);
  static constexpr R a2 = (R(1) - R(2) * a1) / R(4);
  static constexpr R b1 = R(4) * a2;
  static_assert(R(2) * a1 + R(4) * a2 == R(1), "3 sum w c c = I must hold exactly");
  static_assert(R(8) * a2 - R(2) * b1 == R(0), "the cubic Hermite part must carry no momentum");
};

// Post-collision deviations dp_a = N'_a - w_a n_ref at a given Phi:
//   N'_a = N_a + Omega_a + deltaN_a, Omega_a = -(N_a - J f^eq_a)/tau (Eqs. 12, 20).
// The non-equilibrium part is formed first, from the arrived populations
// relative to the cell's own rest state (rho = 1, U = 0 in Eq. 33),
// N_a = J w_a (1 + x^0_a) + n_a:
//   N_a - J f^eq_a = n_a - w_a (1 + x^0_a) (m - J) - w_a m (x_a - x^0_a),
// so that every term is of the size of the flow. Formed from d_a instead, the
// metric part of the rest state (w_a x^0_a, a sizeable fraction of w_a on a
// curved mesh) would enter every product, and its FP32 rounding shows up as a
// systematic error of the relaxed stress -- a viscosity error of about 1e-5.
//
// The bracket x_a of Eq. 33 divided by 3, split over a pair into an even and
// an odd part, from B and C^kkl scaled by 3/2 (T0 = 1/3); the rest state's
// part (g^ij - delta^ij) T0 of B stays out of xe (it is in x^0):
//   xe_p / 3 = c_p.Bh.c_p - tr Bh / 3,                  Bh = (3/2) U~U~,
//   xo_p / 3 = c_p.U + sum_{k != l} C2h^kl c^l_p (3 (c^k_p)^2 - 1),   C2h = (3/2) C^kkl.
// On velocity sets with components in {-1, 0, 1} the odd part only needs,
// per axis l, T0_l = U^l - sum_{k != l} C2h^kl (an axis direction) and
// T_lk = T0_l + 3 C2h^kl (a direction with components on l and k):
//   axis e_l: xo / 3 = c^l T0_l;   diagonal: xo / 3 = c^l T_lk + c^k T_kl,
// and the even part of a diagonal is Bh_ll + Bh_kk - tr Bh / 3 + 2 c^l c^k Bh_lk.
// mn = m - J is the mass of the flow. With REST the populations come in, and
// go out, relative to the cell's own rest state already (d_a = n_a, and
// dp_a = N'_a - o_a), so the subtraction of the rest deviation drops out.
// With RREC the rest state comes from the record (RR, RW); otherwise it is
// formed here from J and Gh = (g - I)/2, x^0_p / 3 = c_p.Gh.c_p - tr Gh / 3:
//   RW_p = w_p + 3 w_p (x^0_p / 3),  RR_p = w_p (J - n_ref) + 3 w_p J (x^0_p / 3),
// and then mn = mdev - sum_a RR_a. Every term is formed relative to its own
// size, and the identity behind the final pass holds for whatever J it uses,
// as long as RR, their sum and mn use the same one.
template <int Q, typename R, bool REST, bool RREC, bool EXT, bool FR0, typename RC>
__device__ __forceinline__ void form_np(const R (&d)[Q], const RC &rc, R m, R mdev, R mn,
                                        R nref, R h2m, R rho, R itau, const R (&U)[Lat<Q>::D],
                                        const R (&Phi)[Lat<Q>::D], R (&dp)[Q]) {
  using L = CoefLayout<Q>;
  constexpr int D = Lat<Q>::D, H = Lat<Q>::H, NS = L::NS;
  constexpr bool ZERO = EXT && FR0, GRP = EXT && !FR0;   // see map_mono
  static_assert(RREC || !REST, "rest-relative storage keeps the rest state in the record");
  R gh[NS];
#pragma unroll
  for (int i = 0; i < NS; i++) gh[i] = rc[L::GH + i];
  R rwc[RREC ? 1 : H + 1], rrc[RREC ? 1 : H + 1];
  if constexpr (!RREC) {
    const R Jc = rc[L::J], Jd = Jc - nref;
    R trg = gh[sym<D>(0, 0)];
#pragma unroll
    for (int i = 1; i < D; i++) trg += gh[sym<D>(i, i)];
    const R tr3 = trg * R(1.0 / 3.0);
    R rsum = R(0);
#pragma unroll
    for (int p = 0; p <= H; p++) {
      R t;
      if (p == 0) {
        t = -tr3;
      } else {
        const int l = nz_axis<Q>(p, 0), k = nz_axis<Q>(p, 1);
        if (k < 0) {
          t = gh[sym<D>(l, l)] - tr3;
        } else {
          const int sg = Lat<Q>::c(p, l) * Lat<Q>::c(p, k);
          t = fmar(R(2 * sg), gh[sym<D>(l, k)], gh[sym<D>(l, l)] + gh[sym<D>(k, k)]) - tr3;
        }
      }
      const R w = lat_w<Q, R>(p), w3 = R(3) * w;
      rwc[p] = fmar(w3, t, w);
      rrc[p] = fmar(w3 * Jc, t, w * Jd);
      rsum += p == 0 ? rrc[p] : R(2) * rrc[p];
    }
    mn = mdev - rsum;
  }
  auto rw_at = [&](int p) -> R {
    if constexpr (RREC)
      return rc[L::RW + p];
    else
      return rwc[p];
  };
  auto rr_at = [&](int p) -> R {
    if constexpr (RREC)
      return rc[L::RR + p];
    else
      return rrc[p];
  };
  const R hh = R(0.5) * h2m;
  R Ut[D], Uh[D], U2[D], Ut2x[D], v[D];
#pragma unroll
  for (int i = 0; i < D; i++) {
    Ut[i] = fmar(Phi[i], h2m, U[i]);
    Uh[i] = R(1.5) * Ut[i];
    U2[i] = Uh[i] * Ut[i];
    Ut2x[i] = Ut[i] + Ut[i];
    v[i] = Phi[i] * hh;   // (U~ - U) / 2
  }
  // Bh = (3/2) U~ U~ (T0 = 1/3), packed symmetric
  R Bh[NS];
#pragma unroll
  for (int i = 0; i < D; i++)
#pragma unroll
    for (int j = i; j < D; j++) Bh[sym<D>(i, j)] = Uh[i] * Ut[j];
  R tB3 = Bh[sym<D>(0, 0)];
#pragma unroll
  for (int i = 1; i < D; i++) tB3 += Bh[sym<D>(i, i)];
  tB3 *= R(1.0 / 3.0);
  // C2h^kl = (1/2) [(gd_kk U~^l + (U~^l - U^l)) + 2 gd_kl U~^k] + (3/2) (U~^k)^2 U~^l
  R C2h[D][D], Sc[D], T0[D], T[D][D];
#pragma unroll
  for (int k = 0; k < D; k++)
#pragma unroll
    for (int l = 0; l < D; l++) {
      if (k == l) continue;
      R t = fmar(U2[k], Ut[l], v[l]);
      if (!EXT || (k < 2 && l < 2)) t = fmar(gh[sym<D>(k, l)], Ut2x[k], t);
      C2h[k][l] = fmar(gh[sym<D>(k, k)], Ut[l], t);
    }
  using MW = MomentWeights<Q, R>;
  R Oax[D];   // axis pairs: a1 U^l - b1 sum_{k != l} C2h^kl
#pragma unroll
  for (int l = 0; l < D; l++) {
    Sc[l] = R(0);
#pragma unroll
    for (int k = 0; k < D; k++)
      if (k != l) Sc[l] += C2h[k][l];
    T0[l] = U[l] - Sc[l];
    Oax[l] = fmar(MW::a1, U[l], -(MW::b1 * Sc[l]));
  }
#pragma unroll
  for (int l = 0; l < D; l++)
#pragma unroll
    for (int k = 0; k < D; k++)
      if (k != l) T[l][k] = fmar(R(3), C2h[k][l], T0[l]);
  // even and odd parts per pair
  R xe[H + 1], xo[H + 1];
  xe[0] = -tB3;
#pragma unroll
  for (int p = 1; p <= H; p++) {
    const int l = nz_axis<Q>(p, 0), k = nz_axis<Q>(p, 1);
    const int sl = Lat<Q>::c(p, l);
    if (k < 0) {
      xe[p] = Bh[sym<D>(l, l)] - tB3;
      xo[p] = sl > 0 ? T0[l] : -T0[l];
    } else {
      const int sk = Lat<Q>::c(p, k);
      const R sd = (Bh[sym<D>(l, l)] + Bh[sym<D>(k, k)]) - tB3;
      xe[p] = fmar(R(2 * sl * sk), Bh[sym<D>(l, k)], sd);
      const R a = sl > 0 ? T[l][k] : -T[l][k];
      xo[p] = sk > 0 ? a + T[k][l] : a - T[k][l];
    }
  }
  // deltaPi^ij = -1/2 (1 - 1/(2 tau)) sum_a c^i_a (K^j_a - L^j_a) f^eq_a   (Eq. 30):
  // K_a - L_a = K_a + K_abar = M_p, and a pair contributes c_p (f_p - f_pbar)
  // with f_p - f_pbar = 2 rho w_p xo_p = 6 rho w_p (xo_p / 3). The record holds
  // am M_p with am = -(2 - 1/tau)/4, and -1/2 (1 - 1/(2 tau)) 2 rho = 2 rho am.
  const R r6 = R(6) * rho;
  const R r6w1 = r6 * lat_w<Q, R>(1), r6w2 = r6 * lat_w<Q, R>(Lat<Q>::H);
  R dP[D][D];
#pragma unroll
  for (int i = 0; i < D; i++)
#pragma unroll
    for (int j = 0; j < D; j++) dP[i][j] = R(0);
  if constexpr (GRP) {
    // pairs with the same coefficients together: xo of pairs 6 and 7 is T_02 +- T_20, of
    // pairs 8 and 9 T_12 +- T_21, and the axis weight twice the diagonal one. In units of
    // 2 r6w2 (taken into a9 below); column 2 is zero.
    const float2 m4 = rc.v2(L::mp(4, 0)), m5 = rc.v2(L::mp(5, 0)), mx = rc.v2(L::mp(1, 0)), my = rc.v2(L::mp(2, 0));
    const float2 t4 = __fmul2_rn(m4, bcast2(0.5f * xo[4]));
    const float x5 = 0.5f * xo[5];
    const float2 P0 = __ffma2_rn(mx, bcast2(T0[0] + T[0][2]), __ffma2_rn(m5, bcast2(x5), t4));
    const float2 P1 = __ffma2_rn(my, bcast2(T0[1] + T[1][2]), __ffma2_rn(m5, bcast2(-x5), t4));
    const float2 P2 = __ffma2_rn(my, bcast2(T[2][1]), __fmul2_rn(mx, bcast2(T[2][0])));
    dP[0][0] = P0.x;
    dP[0][1] = P0.y;
    dP[1][0] = P1.x;
    dP[1][1] = P1.y;
    dP[2][0] = P2.x;
    dP[2][1] = P2.y;
  } else {
    // columns 0 and 1 in the two lanes of packed FP32 instructions
    float2 P01[D];
#pragma unroll
    for (int i = 0; i < D; i++) P01[i] = make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 1; p <= H; p++) {
      if (ZERO && p == 3) continue;
      const R df = (lat_nnz<Q>(p) == 1 ? r6w1 : r6w2) * xo[p];
      const float2 am01 = rc.v2(L::mp(p, 0));
#pragma unroll
      for (int i = 0; i < D; i++) {
        const int ci = Lat<Q>::c(p, i);
        if (ci == 0) continue;
        const R sdf = ci > 0 ? df : -df;
        P01[i] = __ffma2_rn(am01, bcast2(sdf), P01[i]);
        if constexpr (D == 3 && !EXT) dP[i][2] = fmar(rc[L::mp(p, 2)], sdf, dP[i][2]);
      }
    }
#pragma unroll
    for (int i = 0; i < D; i++) {
      dP[i][0] = P01[i].x;
      dP[i][1] = P01[i].y;
    }
  }
  R tr = dP[0][0];
#pragma unroll
  for (int i = 1; i < (EXT ? 2 : D); i++) tr += dP[i][i];
  const R J = GRP ? rc[L::J] * (R(2) * r6w2) : rc[L::J];   // J times the unit of dP
  // E_p = 9 w J c.dP.c - 3 w J tr dP; O_p = 3 w c.Phi (Eq. 31, 1/T0 = 3)
  const R a9_1 = (R(9) * lat_w<Q, R>(1)) * J, a9_2 = (R(9) * lat_w<Q, R>(Lat<Q>::H)) * J;
  const R tr3 = tr * R(1.0 / 3.0);
  const R b3_1 = a9_1 * tr3, b3_2 = a9_2 * tr3;
  {
    const R w = lat_w<Q, R>(0);
    const R n0 = REST ? d[0] : d[0] - rr_at(0);
    const R neq = (n0 - rw_at(0) * mn) - (R(3) * w * m) * xe[0];
    dp[0] = d[0] - itau * neq - (R(3) * w * J) * tr;
  }
  const R wm1 = MW::a1 * m, wm2 = MW::a2 * m;
#pragma unroll
  for (int p = 1; p <= H; p++) {
    const int l = nz_axis<Q>(p, 0), k = nz_axis<Q>(p, 1);
    const int sl = Lat<Q>::c(p, l);
    const bool axis = k < 0;
    R cPc, cF;
    if (axis) {
      cPc = EXT && l == 2 ? R(0) : dP[l][l];
      cF = sl > 0 ? Phi[l] : -Phi[l];
    } else {
      const int sk = Lat<Q>::c(p, k);
      const bool flat = EXT && k == 2;
      const R so = flat ? dP[k][l] : dP[l][k] + dP[k][l];
      const R sd = flat ? dP[l][l] : dP[l][l] + dP[k][k];
      cPc = sl * sk > 0 ? sd + so : sd - so;
      const R f = sl > 0 ? Phi[l] : -Phi[l];
      cF = sk > 0 ? f + Phi[k] : f - Phi[k];
    }
    const R Ep = EXT && axis && l == 2 ? -b3_1 : fmar(axis ? a9_1 : a9_2, cPc, -(axis ? b3_1 : b3_2));
    const R Op = (axis ? MW::a1 : MW::a2) * cF;
    const R wm = axis ? wm1 : wm2;
    const R rw = rw_at(p);
    // odd part of J f^eq over 3 w: m xo on diagonals, m O on axis pairs
    {
      // the pair in the two lanes of packed FP32 instructions (same roundings)
      const float2 dd = make_float2(d[p], d[p + H]);
      const float2 bs = __ffma2_rn(bcast2(-rw), bcast2(mn), REST ? dd : __fadd2_rn(dd, bcast2(-rr_at(p))));
      float2 nq;
      if (axis) {
        const R o = sl > 0 ? Oax[l] : -Oax[l];
        nq = __ffma2_rn(bcast2(-wm), bcast2(xe[p]), bs);
        nq = __ffma2_rn(make_float2(-m, m), bcast2(o), nq);
      } else {
        const float2 xs = __fadd2_rn(bcast2(xe[p]), make_float2(xo[p], -xo[p]));
        nq = __ffma2_rn(bcast2(-wm), xs, bs);
      }
      const float2 r = __fadd2_rn(__ffma2_rn(bcast2(-itau), nq, dd),
                                  __fadd2_rn(bcast2(Ep), make_float2(Op, -Op)));
      dp[p] = r.x;
      dp[p + H] = r.y;
    }
  }
}

// x 2^-e as FP32 by integer operations, truncated (a conversion instruction would take a turn of
// the FP64 pipe); below the FP32 range 0, above it NaN. unit: kUnit1 + e 2^20.
constexpr int32_t kUnit1 = 0x38000000;
__device__ __forceinline__ float trunc_f32(double x, int32_t unit = kUnit1) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int32_t t = (int32_t)(hi & 0x7fffffffu) - unit;
  const uint32_t b = ((uint32_t)t << 3) | (lo >> 29);
  return __uint_as_float((t < 0x00100000 ? 0u : t >= 0x0ff00000 ? 0x7fc00000u : b) | (hi & 0x80000000u));
}
// The FP32 part of an FP64 force solve measures m and Phi in units of the power of two below
// |m|, so that it does what it does at m = 1 for every density (in FP32's own range a density
// of 1e39 was NaN). An exact scaling, by integer operations alone.
struct Unit64 {
  int32_t m, inv;   // units for trunc_f32: of m and Phi, and of 1 / m
  double one;       // the power of two
  __device__ __forceinline__ explicit Unit64(double v) {
    int32_t e = __double2hiint(v) & 0x7ff00000;
    e = min(max(e, 0x08000000), 0x77000000);   // (2^-895 to 2^881)
    m = kUnit1 + (e - 0x3ff00000);
    inv = kUnit1 - (e - 0x3ff00000);
    one = __hiloint2double(e, 0);
  }
};

// RR, RW and the sum of the RR (see CoefLayout) of a record that ends before them, in FP64. (Written
// so that no product can be contracted into a sum: the multi-step kernel forms them once a
// launch, the step kernel once a cell, with the same last bits.)
template <int Q, typename RC>
__device__ __forceinline__ void rest_state(const RC &rc, double nref, double (&rr)[Lat<Q>::H + 1],
                                           double (&rw)[Lat<Q>::H + 1], double &rsum) {
  using L = CoefLayout<Q>;
  constexpr int D = Lat<Q>::D, H = Lat<Q>::H;
  const double Jc = rc[L::J], Jd = Jc - nref;
  double tr = rc[L::GH + sym<D>(0, 0)];
#pragma unroll
  for (int i = 1; i < D; i++) tr += rc[L::GH + sym<D>(i, i)];
  const double tr3 = __dmul_rn(tr, 1.0 / 3.0);
  rsum = 0.0;
#pragma unroll
  for (int q = 0; q <= H; q++) {
    double x = -tr3;
    if (q > 0) {
      const int l = nz_axis<Q>(q, 0), k = nz_axis<Q>(q, 1);
      x = rc[L::GH + sym<D>(l, l)];
      if (k >= 0)
        x = fma((double)(2 * Lat<Q>::c(q, l) * Lat<Q>::c(q, k)), rc[L::GH + sym<D>(l, k)],
                x + rc[L::GH + sym<D>(k, k)]);
      x -= tr3;
    }
    const double w = lat_w<Q, double>(q);
    rw[q] = fma(3.0 * w, x, w);
    rr[q] = fma(__dmul_rn(3.0 * w, Jc), x, __dmul_rn(w, Jd));
    rsum += q == 0 ? rr[q] : 2.0 * rr[q];
  }
}

// The whole local collision in FP64 (see collide_cell). GB300 runs an FP64
// instruction of a warp in 64 cycles of its quarter SM, so only the FP64 operations
// count, about 540 per D3Q19 cell here (920 when the FP32 form was used in FP64):
//  - the chord iteration starts from Pt = H Pc with three evaluations of the
//    polynomial in FP32: its value is of the order of curvature times U^2, so FP32 leaves
//    an error of about 1e-13 m, which one evaluation in FP64 reduces by the map's
//    contraction. It is accepted when its change is at most tol max(m, |Phi|), or when a
//    bound on the contraction times the change is below that by a factor 64; that next
//    change is then added to first order, in FP32. Below four iterations
//    allowed: the plain iteration from the rest state's force.
//  - the test reads the sizes by integer operations on the high words;
//  - N' is formed once per pair and part from what differs from the cell's own rest state, n_a =
//    J w (1 + x0) - w n_ref (RR, RW; see form_np), so that no term of the metric's size is rounded
//    at every step:
//      even: s/2 - (1/tau) [s/2 - RR - RW (m - J)] + w [y0 + c.Y.c],  odd: t/2 - t/(2 tau) + w [(m/tau) xo + 3 c.Phi],
//    Y = (9/2)(m/tau) U~U~ + 9 P, P = J deltaPi (Eq. 30) symmetrised,
//    y0 = -(3/2)(m/tau) U~.U~ - 3 tr P.
//    (From mdev and the whole of B instead, 60 operations fewer, errors against an 80-bit run were
//    0.9 to 1.5 times as large in N after 20 steps and up to 7 times in u; 0.99 to 1.02 so.)
// D3Q19 channel, 64^3: 383 -> 181 us a step, the FP64 pipe 85% busy.
template <int Q, bool FINAL, bool EXT, bool RREC, typename RC>
__device__ __forceinline__ void collide_f64(const double (&d)[Q], const RC &rc, double nref, double itau, double tol,
                                            int max_iter, double (&dp)[Q], CollideState<Q, double> &st) {
  using L = CoefLayout<Q>;
  constexpr int D = Lat<Q>::D, H = Lat<Q>::H, NS = L::NS, NQ = L::NQ;
  static_assert(!EXT || Q == 19, "extruded meshes are D3Q19's");
  constexpr int DI = EXT ? 2 : D;   // components of Phi that are iterated
  double s[H + 1], t[H + 1], mu[D], Pc[D], Pt[D], mdev = d[0];
#pragma unroll
  for (int i = 0; i < D; i++) mu[i] = Pc[i] = 0.0;
#pragma unroll
  for (int p = 1; p <= H; p++) {
    s[p] = d[p] + d[p + H];
    t[p] = d[p] - d[p + H];
    if constexpr (EXT) continue;
    mdev += s[p];
#pragma unroll
    for (int i = 0; i < D; i++) {
      const int ci = Lat<Q>::c(p, i);
      if (ci > 0) mu[i] += t[p];
      if (ci < 0) mu[i] -= t[p];
      Pc[i] = fma(rc[L::mp(p, i)], s[p], Pc[i]);
      Pc[i] = fma(rc[L::dk(p, i)], t[p], Pc[i]);
    }
  }
  if constexpr (EXT) {
    const double sg[4] = {s[1] + (s[6] + s[7]), s[2] + (s[8] + s[9]), s[4], s[5]};
    const double tg[4] = {t[1] + (t[6] + t[7]), t[2] + (t[8] + t[9]), t[4], t[5]};
    mdev += s[3] + ((sg[0] + sg[1]) + (sg[2] + sg[3]));
    mu[0] = tg[0] + (tg[2] + tg[3]);
    mu[1] = tg[1] + (tg[2] - tg[3]);
    mu[2] = t[3] + ((t[6] - t[7]) + (t[8] - t[9]));
#pragma unroll
    for (int g = 0; g < 4; g++) {
      const int p = g < 2 ? g + 1 : g + 2;
#pragma unroll
      for (int i = 0; i < 2; i++) {
        Pc[i] = fma(rc[L::mp(p, i)], sg[g], Pc[i]);
        Pc[i] = fma(rc[L::dk(p, i)], tg[g], Pc[i]);
      }
    }
  }
  const double m = nref + mdev, im = 1.0 / m, h2m = 0.5 * im, hm = 0.5 * m;
  const double kf = (0.5 * itau) * mdev;
  st.rho = m * rc[L::IJ];
  double hmu[D];
#pragma unroll
  for (int i = 0; i < D; i++) {
    st.U[i] = mu[i] * im;
    hmu[i] = -0.5 * mu[i];
  }
  // Pc = sum_p (am M s + ad D t) + m G - (mdev itau/2) KW - m/2 (CE + (PO1 + LO) U) - n_ref KW,
  // the last and largest product exact
#pragma unroll
  for (int i = 0; i < DI; i++) {
    double v = fma(m, rc[L::BODY + i], Pc[i]);
    v = fma(-hm, rc[L::CE + i], v);
#pragma unroll
    for (int l = 0; l < DI; l++) v = fma(rc[L::PO1 + i * D + l], hmu[l], v);
    Pc[i] = fma(-nref, rc[L::KW + i], fma(-kf, rc[L::KW + i], v));
  }
#pragma unroll
  for (int i = 0; i < DI; i++) {
    Pt[i] = Pc[i];
#pragma unroll
    for (int j = 0; j < DI; j++) Pt[i] = fma(rc[L::row(L::HM, D, i, j)], Pc[j], Pt[i]);
  }
  if constexpr (EXT) Pt[2] = m * rc[L::BODY + 2];
  double Phi[D];
  float lip = 1.0e30f;   // bound on the contraction of one evaluation
  int it = 0;
  const Unit64 un(m);
  const float mf = trunc_f32(m, un.m);
  if (max_iter >= 4) {
    float qf[D][NQ], Uf[D], Pf[D], df[D], l2 = 0.f, l3 = 0.f, um = 0.f;
    const float hf = trunc_f32(h2m, un.inv), hmf = 0.5f * mf;
#pragma unroll
    for (int i = 0; i < D; i++) {
      Uf[i] = trunc_f32(st.U[i]);
      Pf[i] = trunc_f32(Pt[i], un.m);
      df[i] = 0.f;
#pragma unroll
      for (int k = 0; k < NQ; k++) {
        if (i >= DI || !map_mono<EXT, D>(k)) continue;
        qf[i][k] = trunc_f32(rc[L::row(L::QM, NQ, i, k)]);
        if (k < NS)
          l2 += fabsf(qf[i][k]);
        else
          l3 += fabsf(qf[i][k]);
      }
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
      float x[D], mono[NQ];
#pragma unroll
      for (int i = 0; i < D; i++) {
        x[i] = fmaf(Pf[i] + df[i], hf, Uf[i]);
        um = fmaxf(um, fabsf(x[i]));
      }
#pragma unroll
      for (int k = 0; k < D; k++)
#pragma unroll
        for (int l = 0; l < D; l++) {
          if (k <= l) mono[sym<D>(k, l)] = x[k] * x[l];
          if (k != l) mono[NS + offd<D>(k, l)] = (x[k] * x[k]) * x[l];
        }
#pragma unroll
      for (int i = 0; i < DI; i++) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < NQ; k++)
          if (map_mono<EXT, D>(k)) v = fmaf(qf[i][k], mono[k], v);
        df[i] = -hmf * v;
      }
    }
    it = 3;
    // |d Phi_new| <= m/2 |dQ/dU~| |d Phi| / (2 m) <= (l2 2 um + l3 3 um^2) / 4, with room for
    // U~ to lie outside the FP32 iterates
    um *= 1.01f;
    lip = fmaf(0.5f * l2, um, 0.75f * l3 * um * um);
#pragma unroll
    for (int i = 0; i < DI; i++) Phi[i] = fma((double)df[i], un.one, Pt[i]);
  } else {
#pragma unroll
    for (int i = 0; i < DI; i++) Phi[i] = m * rc[L::FR + i];
  }
  if constexpr (EXT) Phi[2] = Pt[2];
  st.conv = false;
  const float tolf = (float)tol, epsf = (float)(64.0 / 9007199254740992.0);
  float dl[D];
#pragma unroll
  for (int i = 0; i < D; i++) dl[i] = 0.f;
#pragma unroll 1
  while (it < max_iter) {
    double Ut[D], mono[NQ];
    float diff = 0.f, pmax = EXT ? fabsf(trunc_f32(Phi[D - 1], un.m)) : 0.f;
#pragma unroll
    for (int i = 0; i < D; i++) Ut[i] = fma(Phi[i], h2m, st.U[i]);
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = k; l < D; l++) mono[sym<D>(k, l)] = Ut[k] * Ut[l];
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = 0; l < D; l++)
        if (k != l) mono[NS + offd<D>(k, l)] = mono[sym<D>(k, k)] * Ut[l];
#pragma unroll
    for (int i = 0; i < DI; i++) {
      // two partial sums: the chain of a small mesh is bound by latency
      double a = rc[L::row(L::QM, NQ, i, 0)] * mono[0], b = rc[L::row(L::QM, NQ, i, 1)] * mono[1];
#pragma unroll
      for (int k = 2; k < NQ; k++) {
        if (!map_mono<EXT, D>(k)) continue;
        if (k & 1)
          b = fma(rc[L::row(L::QM, NQ, i, k)], mono[k], b);
        else
          a = fma(rc[L::row(L::QM, NQ, i, k)], mono[k], a);
      }
      const double pn = fma(-hm, a + b, Pt[i]);
      dl[i] = trunc_f32(pn - Phi[i], un.m);
      diff = maxnan(diff, fabsf(dl[i]));
      pmax = maxnan(pmax, fabsf(trunc_f32(pn, un.m)));
      Phi[i] = pn;
    }
    it++;
    const float scale = fmaxf(tolf * maxnan(mf, pmax), epsf * pmax);
    if (diff <= scale || 64.f * lip * diff <= scale) {
      st.conv = true;
      break;
    }
  }
  st.iters = it;
  // What the accepted step leaves, the next change, to first order: -m/2 Q'(U~) dU~ of the last
  // change, in FP32 (its error is 2^-22 of a change below tol / 64). Without it 6 to 15% of the
  // populations of a step were a last bit off those of a solve to the end, now 0.2 to 1%.
  if (st.conv) {
    float x[D], dm[NQ];
    const float hf = trunc_f32(h2m, un.inv), hmf = 0.5f * mf;
#pragma unroll
    for (int i = 0; i < D; i++) {
      x[i] = fmaf(trunc_f32(Phi[i], un.m), hf, trunc_f32(st.U[i]));
      dl[i] *= hf;
    }
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = 0; l < D; l++) {
        if (k <= l) dm[sym<D>(k, l)] = fmaf(x[k], dl[l], dl[k] * x[l]);
        if (k != l) dm[NS + offd<D>(k, l)] = x[k] * fmaf(x[k], dl[l], 2.f * dl[k] * x[l]);
      }
#pragma unroll
    for (int i = 0; i < DI; i++) {
      float v = 0.f;
#pragma unroll
      for (int k = 0; k < NQ; k++)
        if (map_mono<EXT, D>(k)) v = fmaf(trunc_f32(rc[L::row(L::QM, NQ, i, k)]), dm[k], v);
      Phi[i] = fma((double)(-hmf * v), un.one, Phi[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < D; i++) st.F[i] = Phi[i] * rc[L::IJ];
  if constexpr (FINAL) {
    double Ut[D], B[NS], Bd[D], C2[D][D], Sc[D], T0[D], T[D][D], tb = 0.0;
#pragma unroll
    for (int i = 0; i < D; i++) Ut[i] = fma(Phi[i], h2m, st.U[i]);
    // 3 B = (g - I) + 3 U~U~ (T0 = 1/3); (3/2) C^kkl = (1/2)[gd_kk U~^l + (U~^l - U^l) + 2 gd_kl U~^k]
    // + (3/2)(U~^k)^2 U~^l, with GH = gd / 2
    double U3[D], du[D];
#pragma unroll
    for (int i = 0; i < D; i++) {
      U3[i] = 3.0 * Ut[i];
      du[i] = Phi[i] * (0.5 * h2m);   // (U~ - U) / 2
    }
#pragma unroll
    for (int i = 0; i < D; i++)
#pragma unroll
      for (int j = i; j < D; j++)
        B[sym<D>(i, j)] = U3[i] * Ut[j];
#pragma unroll
    for (int i = 0; i < D; i++) {
      tb += B[sym<D>(i, i)];
      Bd[i] = fma(U3[i], Ut[i], 2.0 * rc[L::GH + sym<D>(i, i)]);
    }
    // per axis l: xo/3 of an axis direction is T0_l = U^l - sum_k C2^kl, of a diagonal
    // c^l T_lk + c^k T_kl with T_lk = T0_l + 3 C2^kl
#pragma unroll
    for (int l = 0; l < D; l++) {
      Sc[l] = 0.0;
#pragma unroll
      for (int k = 0; k < D; k++) {
        if (k == l) continue;
        // gd_kk/2 + (3/2) U~k^2 = B_kk / 2
        const double x = EXT && (k == 2 || l == 2) ? du[l] : fma(rc[L::GH + sym<D>(k, l)], Ut[k] + Ut[k], du[l]);
        C2[k][l] = fma(0.5 * Bd[k], Ut[l], x);
        Sc[l] += C2[k][l];
      }
      T0[l] = st.U[l] - Sc[l];
    }
#pragma unroll
    for (int l = 0; l < D; l++)
#pragma unroll
      for (int k = 0; k < D; k++)
        if (k != l) T[l][k] = fma(3.0, C2[k][l], T0[l]);
    // P^kl = J deltaPi^kl = 2 m sum_p w c^k am M^l xo = sum_p (6 m w) c^k am M^l (xo / 3)
    double P[D][D];
#pragma unroll
    for (int i = 0; i < D; i++)
#pragma unroll
      for (int j = 0; j < D; j++) P[i][j] = 0.0;
    auto xo3 = [&](int p) {
      const int l = nz_axis<Q>(p, 0), k = nz_axis<Q>(p, 1);
      const int sl = Lat<Q>::c(p, l);
      if (k < 0) return sl > 0 ? T0[l] : -T0[l];
      const double a = sl > 0 ? T[l][k] : -T[l][k];
      return Lat<Q>::c(p, k) > 0 ? a + T[k][l] : a - T[k][l];
    };
    // the axis weight is 2 (D3Q19) or 4 (D2Q9) times the diagonal one
    constexpr double wr = D == 3 ? 2.0 : 4.0;
    const double w2 = lat_w<Q, double>(H);
    if constexpr (EXT) {
      // pairs with the same coefficients together (see form_np), in units of 2
      const double x4 = 0.5 * xo3(4), x5 = 0.5 * xo3(5);
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const double t4 = rc[L::mp(4, j)] * x4;
        P[0][j] = fma(rc[L::mp(1, j)], T0[0] + T[0][2], fma(rc[L::mp(5, j)], x5, t4));
        P[1][j] = fma(rc[L::mp(2, j)], T0[1] + T[1][2], fma(rc[L::mp(5, j)], -x5, t4));
        P[2][j] = fma(rc[L::mp(2, j)], T[2][1], rc[L::mp(1, j)] * T[2][0]);
      }
    }
#pragma unroll
    for (int p = 1; p <= (EXT ? 0 : H); p++) {
      const double x = lat_nnz<Q>(p) == 1 ? wr * xo3(p) : xo3(p);
#pragma unroll
      for (int j = 0; j < D; j++) {
        const double M = rc[L::mp(p, j)];
#pragma unroll
        for (int i = 0; i < D; i++) {
          const int ci = Lat<Q>::c(p, i);
          if (ci > 0) P[i][j] = fma(M, x, P[i][j]);
          if (ci < 0) P[i][j] = fma(-M, x, P[i][j]);
        }
      }
    }
    // everything times w2: Y = w2 [(9/2)(m/tau) B + 9 P], B = (3 B) / 3
    constexpr double pu = EXT ? 2.0 : 1.0;   // the unit of P
    const double mt = m * itau, yb = (1.5 * w2) * mt, yp = (54.0 * w2 * w2 * pu) * m;
    double Y[NS], trP = 0.0;
#pragma unroll
    for (int i = 0; i < D; i++) {
      if (i < DI) trP = i == 0 ? P[0][0] : trP + P[i][i];
#pragma unroll
      for (int j = i; j < D; j++) {
        if (EXT && j == 2)
          Y[sym<D>(i, j)] = i == 2 ? yb * B[sym<D>(i, j)] : fma(0.5 * yp, P[j][i], yb * B[sym<D>(i, j)]);
        else
          Y[sym<D>(i, j)] = fma(yb, B[sym<D>(i, j)], i == j ? yp * P[i][i] : (0.5 * yp) * (P[i][j] + P[j][i]));
      }
    }
    // y0 = w2 [(mdev - m (3 tr B) / 2) / tau - 3 tr P]
    const double y0 = fma(-((18.0 * w2 * w2 * pu) * m), trP, -(w2 * itau) * (hm * tb));
    // (the weights of the odd part are MomentWeights': no momentum is made by rounding them)
    using MW = MomentWeights<Q, double>;
    const double zm = MW::a2 * mt, hi = -0.5 * itau;
    double Z0[D], Z[D][D];
#pragma unroll
    for (int l = 0; l < D; l++) {
      Z0[l] = fma(mt, fma(MW::a1, st.U[l], -(MW::b1 * Sc[l])), MW::a1 * Phi[l]);
#pragma unroll
      for (int k = 0; k < D; k++)
        if (k != l) Z[l][k] = fma(zm, T[l][k], MW::a2 * Phi[l]);
    }
    // the rest state: RR, RW of the record, or formed from J and g^ij
    double rw[H + 1], rr[H + 1], mn;
    if constexpr (RREC) {
      mn = mdev - rc[L::RR + H + 1];
    } else {
      double rsum;
      rest_state<Q>(rc, nref, rr, rw, rsum);
      mn = mdev - rsum;
    }
    auto rr_at = [&](int q) -> double { if constexpr (RREC) return rc[L::RR + q]; else return rr[q]; };
    auto rw_at = [&](int q) -> double { if constexpr (RREC) return rc[L::RW + q]; else return rw[q]; };
    dp[0] = d[0] + fma(-itau, fma(-rw_at(0), mn, d[0] - rr_at(0)), (lat_w<Q, double>(0) / w2) * y0);
#pragma unroll
    for (int p = 1; p <= H; p++) {
      const int l = nz_axis<Q>(p, 0), k = nz_axis<Q>(p, 1);
      const int sl = Lat<Q>::c(p, l);
      double e, o;
      if (k < 0) {
        e = wr * (y0 + Y[sym<D>(l, l)]);
        o = sl > 0 ? Z0[l] : -Z0[l];
      } else {
        const int sk = Lat<Q>::c(p, k);
        const double sd = y0 + (Y[sym<D>(l, l)] + Y[sym<D>(k, k)]);
        e = fma((double)(2 * sl * sk), Y[sym<D>(l, k)], sd);
        const double a = sl > 0 ? Z[l][k] : -Z[l][k];
        o = sk > 0 ? a + Z[k][l] : a - Z[k][l];
      }
      const double ne = fma(-rw_at(p), mn, fma(0.5, s[p], -rr_at(p)));
      const double ae = fma(-itau, ne, e), ao = fma(hi, t[p], o);
      dp[p] = d[p] + (ae + ao);
      dp[p + H] = d[p + H] + (ae - ao);
    }
  }
}

// Full local collision: solve the fixed point Phi = J G(Phi / J) of Eq. 27 by
// the chord iteration Phi <- H (Pc - 1/2 m Q(U~)) (see build_record), from the
// start value m times the rest-state force. A step is accepted as converged
// when its change is at most max(tol max(m, |Phi|), 64 eps |Phi|): eps is the
// unit roundoff of R, and Phi is a sum of dozens of rounded terms of its own
// size, so smaller changes are rounding noise. With FINAL, the post-collision
// deviations are formed at the converged Phi.
// rc is the cell's coefficient record (PtrRecord or CellRecord); itau = 1/tau. With REST, d holds e_a = N_a - o_a relative to the
// cell's own rest state (16-bit storage, see CoefLayout), and so does dp.
template <int Q, typename R, bool FINAL, bool REST, bool RREC, bool EXT, bool FR0, typename RC>
__device__ __forceinline__ void collide_f32(const R (&d)[Q], const RC &rc, R nref,
                                             R itau, R tol, int max_iter, R (&dp)[Q],
                                             CollideState<Q, R> &st) {
  static_assert(sizeof(R) == 4, "FP64 goes through collide_f64");
  using L = CoefLayout<Q>;
  constexpr int D = Lat<Q>::D, H = Lat<Q>::H, NS = L::NS, NQ = L::NQ;
  static_assert(D == 2 || NQ % 4 == 0, "row 2 of the chord step is read in 16-byte quads");
  static_assert(!EXT || Q == 19, "extruded meshes are D3Q19's");
  constexpr bool ZERO = EXT && FR0, GRP = EXT && !FR0;   // see map_mono
  constexpr int DI = EXT ? 2 : D;   // components of Phi that are iterated
  const R epsn = sizeof(R) == 4 ? R(64.0 / 16777216.0) : R(64.0 / 9007199254740992.0);
  // pair sums s_p = d_p + d_pbar and differences t_p = d_p - d_pbar
  // (with REST: of e_a; the rest state's part of the s_p enters through SR)
  R sp[H + 1], tp[H + 1];
  R mdev = d[0];
#pragma unroll
  for (int p = 1; p <= H; p++) {
    sp[p] = d[p] + d[p + H];
    tp[p] = d[p] - d[p + H];
    if constexpr (!GRP) mdev += sp[p];
  }
  // sums over the pairs that share link coefficients
  R sg[4], tg[4];
  if constexpr (GRP) {
    sg[0] = sp[1] + (sp[6] + sp[7]);
    sg[1] = sp[2] + (sp[8] + sp[9]);
    tg[0] = tp[1] + (tp[6] + tp[7]);
    tg[1] = tp[2] + (tp[8] + tp[9]);
    sg[2] = sp[4];
    sg[3] = sp[5];
    tg[2] = tp[4];
    tg[3] = tp[5];
    mdev += sp[3] + ((sg[0] + sg[1]) + (sg[2] + sg[3]));
  }
  // m - J, the mass of the flow
  R mn;
  if constexpr (REST) {
    mn = mdev + rc[L::MNV];
    mdev += rc[L::MDV];
  } else {
    mn = RREC ? mdev - rc[L::RR + H + 1] : R(0);   // else formed in form_np
  }
  const R m = nref + mdev;
  // rho = sum f = sum N / J; rho U = sum c f   (Eqs. 14, 15, 17)
  st.rho = m * rc[L::IJ];
  const R im = R(1) / m;
  const R h2m = R(0.5) * im;
  const R hm = R(0.5) * m;
#pragma unroll
  for (int i = 0; i < D; i++) {
    R s = R(0);
    if constexpr (GRP) {
      s = i == 0   ? tg[0] + (tg[2] + tg[3])
          : i == 1 ? tg[1] + (tg[2] - tg[3])
                   : tp[3] + ((tp[6] - tp[7]) + (tp[8] - tp[9]));
    } else {
#pragma unroll
      for (int p = 1; p <= H; p++) {
        const int ci = Lat<Q>::c(p, i);
        if (ci > 0) s += tp[p];
        if (ci < 0) s -= tp[p];
      }
    }
    st.U[i] = s * im;
  }
  // constant part of J F: body force m G, 1/2 sum_a L_a N_a (L_a = -K_abar), the
  // reference part -n_ref sum_a w_a K_a of both sums of Eq. 27 (the largest term,
  // the same every step: formed without rounding error from the split KW + KWL),
  // the parts of -1/2 sum_a K_a N'_a that do not change during the iteration
  // and the terms of the map that depend on U only. Over a pair,
  //   -1/2 (K_pbar d_p + K_p d_pbar) - 1/2 (1 - 1/tau)(K_p d_p + K_pbar d_pbar)
  //     = -(2 - 1/tau)/4 M_p s_p + (1/tau)/4 D_p t_p,
  // whose two weights the record's link coefficients already carry.
  R s[D], pr[D];
#pragma unroll
  for (int i = 0; i < DI; i++) {
    const R kw = rc[L::KW + i];
    pr[i] = nref * kw;
    const R err = two_prod_err(nref, kw, pr[i]) + nref * rc[L::KWL + i];
    s[i] = m * rc[L::BODY + i] - err - R(0.5) * itau * mdev * kw;
    if constexpr (REST) s[i] += rc[L::SR + i];
  }
  {
    // components 0 and 1 in the two lanes of packed FP32 instructions, two
    // partial sums each
    float2 sa = make_float2(s[0], s[1]), sb = make_float2(0.f, 0.f);
    float s2a = D == 3 && !EXT ? s[D - 1] : 0.f, s2b = 0.f;
#pragma unroll
    for (int k = 1; k <= (GRP ? 4 : H); k++) {
      if (ZERO && k == 3) continue;
      const int p = GRP && k > 2 ? k + 1 : k;
      const R sk = GRP ? sg[(k - 1) & 3] : sp[p], tk = GRP ? tg[(k - 1) & 3] : tp[p];
      const float4 q = rc.v4(L::mp(p, 0));   // am M^0, am M^1, ad D^0, ad D^1
      float2 &acc = (k & 1) ? sa : sb;
      acc = __ffma2_rn(make_float2(q.x, q.y), bcast2(sk), acc);
      acc = __ffma2_rn(make_float2(q.z, q.w), bcast2(tk), acc);
      if constexpr (D == 3 && !EXT) {
        const float2 r2 = rc.v2(L::mp(p, 2));   // am M^2, ad D^2
        float &a2 = (p & 1) ? s2a : s2b;
        a2 = fmaf(r2.x, sp[p], a2);
        a2 = fmaf(r2.y, tp[p], a2);
      }
    }
    const float2 st01 = __fadd2_rn(sa, sb);
    s[0] = st01.x;
    s[1] = st01.y;
    if constexpr (D == 3 && !EXT) s[D - 1] = s2a + s2b;
  }
  // Pc = Pb - 1/2 m (CE + (PO1 + LO) U), then Pt = H Pc = Pc + (H - I) Pc
  R Pc[D];
#pragma unroll
  for (int i = 0; i < DI; i++) {
    R u = rc[L::CE + i];
#pragma unroll
    for (int l = 0; l < DI; l++) u = fmar(rc[L::PO1 + i * D + l], st.U[l], u);
    Pc[i] = (s[i] - hm * u) - pr[i];
  }
  R Pt[D];
  {
    float2 x = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < DI; j++) x = __ffma2_rn(rc.v2(L::row(L::HM, D, 0, j)), bcast2(Pc[j]), x);
    const float2 p01 = __fadd2_rn(make_float2(Pc[0], Pc[1]), x);
    Pt[0] = p01.x;
    Pt[1] = p01.y;
    if constexpr (EXT) {
      Pt[2] = m * rc[L::BODY + 2];
    } else if constexpr (D == 3) {
      R y = R(0);
#pragma unroll
      for (int j = 0; j < D; j++) y = fmar(rc[L::row(L::HM, D, 2, j)], Pc[j], y);
      Pt[D - 1] = Pc[D - 1] + y;
    }
  }
  // Start at Pt = H Pc, the fixed point without the polynomial part: it is off by that
  // part, of the order of curvature times U^2 (the rest state's force, the start
  // when only a few evaluations are allowed, by curvature times U), so that one
  // evaluation less reaches the same residual. FR0 (16-bit storage) starts at the latter in
  // any case: a population is rounded to 16 bits after every step, and a last bit of FP32
  // decides which way, so that every other order of the FP32 sums is another sequence of
  // roundings: relative to the uniform reference 1 to 30% of the velocity (large values are
  // stored), relative to the rest state 4e-4 (FP16, 100 steps of a 128^3 channel).
  R Phi[D];
#pragma unroll
  for (int i = 0; i < D; i++) Phi[i] = (max_iter >= 4 && !FR0) || (GRP && i >= DI) ? Pt[i] : m * rc[L::FR + i];
  st.conv = false;
  int it = 0;
  while (it < max_iter) {
    // Phi_new = H Pc - 1/2 m [H PE : U~U~ + H PO2 : (U~^k)^2 U~^l]
    R Ut[D], sq[D], mono[NQ];
#pragma unroll
    for (int i = 0; i < D; i++) {
      Ut[i] = fmar(Phi[i], h2m, st.U[i]);
      sq[i] = Ut[i] * Ut[i];
    }
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = k; l < D; l++) mono[sym<D>(k, l)] = k == l ? sq[k] : Ut[k] * Ut[l];
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = 0; l < D; l++)
        if (k != l) mono[NS + offd<D>(k, l)] = sq[k] * Ut[l];
    R a[D];
    {
      // rows 0 and 1 in the two lanes of packed FP32 instructions, two partial
      // sums per row
      float2 a01a = make_float2(0.f, 0.f), a01b = make_float2(0.f, 0.f);
      float a2a = 0.f, a2b = 0.f;
#pragma unroll
      for (int s2 = 0; s2 < NQ; s2 += 2) {
        if constexpr (EXT) {
          if (!map_mono<EXT, D>(s2) || !map_mono<EXT, D>(s2 + 1)) {
            // one monomial of the two (extruded meshes: never none)
            const int s1 = map_mono<EXT, D>(s2) ? s2 : s2 + 1;
            float2 &acc = (GRP ? (s2 & 2) != 0 : (s1 & 1) == 0) ? a01a : a01b;
            acc = __ffma2_rn(rc.v2(L::QM + 2 * s1), bcast2(mono[s1]), acc);
            continue;
          }
        }
        if (s2 + 1 < NQ) {
          const float4 q = rc.v4(L::QM + 2 * s2);
          a01a = __ffma2_rn(make_float2(q.x, q.y), bcast2(mono[s2]), a01a);
          a01b = __ffma2_rn(make_float2(q.z, q.w), bcast2(mono[s2 + 1]), a01b);
        } else {
          a01a = __ffma2_rn(rc.v2(L::QM + 2 * s2), bcast2(mono[s2]), a01a);
        }
      }
      if constexpr (D == 3 && !EXT) {
#pragma unroll
        for (int s4 = 0; s4 < NQ; s4 += 4) {
          const float4 q = rc.v4(L::row(L::QM, NQ, 2, s4));
          a2a = fmaf(q.x, mono[s4], a2a);
          a2b = fmaf(q.y, mono[s4 + 1], a2b);
          a2a = fmaf(q.z, mono[s4 + 2], a2a);
          a2b = fmaf(q.w, mono[s4 + 3], a2b);
        }
      }
      const float2 a01 = __fadd2_rn(a01a, a01b);
      a[0] = a01.x;
      a[1] = a01.y;
      if constexpr (D == 3 && !EXT) a[D - 1] = a2a + a2b;
    }
    it++;
    // converged when the change is at most max(tol max(m, |Phi|), 64 eps |Phi|)
    R diff = ZERO ? absr(Pt[D - 1] - Phi[D - 1]) : R(0), pmax = EXT ? absr(Phi[D - 1]) : R(0);
    if constexpr (ZERO) Phi[D - 1] = Pt[D - 1];
#pragma unroll
    for (int i = 0; i < DI; i++) {
      const R pn = fmar(-hm, a[i], Pt[i]);
      diff = maxnan(diff, absr(pn - Phi[i]));
      pmax = maxnan(pmax, absr(Phi[i]));
      Phi[i] = pn;
    }
    if (diff <= maxnan(tol * maxnan(m, pmax), epsn * pmax)) {
      st.conv = true;
      break;
    }
  }
  st.iters = it;
  if (FINAL) form_np<Q, R, REST, RREC, EXT, FR0, RC>(d, rc, m, mdev, mn, nref, h2m, st.rho, itau, st.U, Phi, dp);
#pragma unroll
  for (int i = 0; i < D; i++) st.F[i] = Phi[i] * rc[L::IJ];
}

// the local collision in the arithmetic type R
template <int Q, typename R, bool FINAL, bool REST = false, bool RREC = true, typename RC = PtrRecord<R>,
          bool EXT = false, bool FR0 = false>
__device__ __forceinline__ void collide_cell(const R (&d)[Q], const RC &rc, R nref, R itau, R tol, int max_iter,
                                             R (&dp)[Q], CollideState<Q, R> &st) {
  if constexpr (sizeof(R) == 8) {
    static_assert(!REST, "FP64 populations are stored relative to the uniform reference");
    collide_f64<Q, FINAL, EXT, RREC, RC>(d, rc, nref, itau, tol, max_iter, dp, st);
  } else {
    collide_f32<Q, R, FINAL, REST, RREC, EXT, FR0, RC>(d, rc, nref, itau, tol, max_iter, dp, st);
  }
}

}  // namespace vlb
