// vlb_geometry.cu -- FP64 geometry precompute of section 2.1 (done once per
// mesh), mesh diagnostics, the coefficient records the step kernel streams,
// and the equilibrium initialisation of the populations.
#include <type_traits>

#include "vlb_addr.cuh"
#include "vlb_collide.cuh"
#include "vlb_q39.cuh"

namespace vlb {

// ------------------------------------------------------------------ positions
// y <- T_a^k (y), T_a(x) = R_a x + shift_a (inverse for k < 0)
__device__ __noinline__ void apply_period(const MeshDev &m, int ax, int64_t k, double y[3]) {
  const int D = m.dim;
  const double *R = m.rot[ax];
  const double *sh = m.shift[ax];
  for (int64_t t = 0; t < (k > 0 ? k : -k); t++) {
    double z[3] = {y[0], y[1], y[2]};
    if (k > 0) {
      if (m.has_rot[ax])
        for (int i = 0; i < D; i++) {
          double acc = 0.0;
          for (int j = 0; j < D; j++) acc += R[3 * i + j] * z[j];
          y[i] = acc;
        }
      for (int i = 0; i < D; i++) y[i] += sh[i];
    } else {
      for (int i = 0; i < D; i++) z[i] -= sh[i];
      if (m.has_rot[ax]) {
        for (int i = 0; i < D; i++) {
          double acc = 0.0;
          for (int j = 0; j < D; j++) acc += R[3 * j + i] * z[j];
          y[i] = acc;
        }
      } else {
        for (int i = 0; i < D; i++) y[i] = z[i];
      }
    }
  }
}

// position of p whose wall-axis coordinates are in range: wrap the periodic
// axes and apply the image transforms, axis 0 outermost
__device__ __noinline__ void position_periodic(const MeshDev &m, const int64_t p[3], double out[3]) {
  int64_t w[3], k[3];
  for (int a = 0; a < 3; a++) {
    w[a] = p[a];
    k[a] = 0;
    if (a < m.dim && m.bc[a] == VLB_PERIODIC) {
      int64_t q = p[a] / m.n[a];
      if (p[a] < 0 && q * m.n[a] != p[a]) q -= 1;  // floor division
      k[a] = q;
      w[a] = p[a] - q * m.n[a];
    }
  }
  const int64_t idx = (w[0] * m.n[1] + w[1]) * m.n[2] + w[2];
  for (int d = 0; d < 3; d++) out[d] = d < m.dim ? m.x[idx * m.dim + d] : 0.0;
  for (int a = m.dim - 1; a >= 0; a--)
    if (k[a] != 0) apply_period(m, a, k[a], out);
}

// position of any index p: behind a wall, linear extrapolation along that axis
// from the two nearest interior nodes, x(-k) = (1 + k) x(0) - k x(1)
__device__ __noinline__ void position(const MeshDev &m, const int64_t p[3], double out[3]) {
  int wa[3], nw = 0;
  int64_t b0[3], b1[3];
  double c0[3], c1[3];
  for (int a = 0; a < m.dim; a++) {
    if (m.bc[a] != VLB_WALL || (p[a] >= 0 && p[a] < m.n[a])) continue;
    const int64_t k = p[a] < 0 ? -p[a] : p[a] - (m.n[a] - 1);
    wa[nw] = a;
    b0[nw] = p[a] < 0 ? 0 : m.n[a] - 1;
    b1[nw] = p[a] < 0 ? 1 : m.n[a] - 2;
    c0[nw] = 1.0 + (double)k;
    c1[nw] = -(double)k;
    nw++;
  }
  out[0] = out[1] = out[2] = 0.0;
  for (int combo = 0; combo < (1 << nw); combo++) {
    int64_t pp[3] = {p[0], p[1], p[2]};
    double wgt = 1.0;
    for (int t = 0; t < nw; t++) {
      const bool second = (combo >> t) & 1;
      pp[wa[t]] = second ? b1[t] : b0[t];
      wgt *= second ? c1[t] : c0[t];
    }
    double y[3];
    position_periodic(m, pp, y);
    for (int d = 0; d < 3; d++) out[d] += wgt * y[d];
  }
}

__device__ __forceinline__ double nrm(const double v[3]) {
  return sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
}

// tangent basis g_i(p) (Eqs. 1, 3); false on a folded arm (D_i = D_-i)
__device__ __noinline__ bool tangents(const MeshDev &m, const int64_t p[3], double gl[3][3]) {
  const double dx = m.dx > 0.0 ? m.dx : 1.0;
  double x0[3];
  position(m, p, x0);
  bool ok = true;
  for (int i = 0; i < 3; i++)
    for (int d = 0; d < 3; d++) gl[i][d] = 0.0;
  for (int i = 0; i < m.dim; i++) {
    int64_t pp[3] = {p[0], p[1], p[2]}, pm[3] = {p[0], p[1], p[2]};
    pp[i] += 1;
    pm[i] -= 1;
    double xp[3], xm[3], Dp[3], Dm[3], df[3];
    position(m, pp, xp);
    position(m, pm, xm);
    for (int d = 0; d < 3; d++) {
      Dp[d] = xp[d] - x0[d];
      Dm[d] = xm[d] - x0[d];
      df[d] = Dp[d] - Dm[d];
    }
    const double nd = nrm(df);
    if (!(nd > 0.0)) {
      ok = false;
      continue;
    }
    const double beta = (nrm(Dp) + nrm(Dm)) / nd;
    for (int d = 0; d < 3; d++) gl[i][d] = beta * df[d] / (2.0 * dx);
  }
  return ok;
}

// J (Eq. 5) and co-tangents g^i (Eq. 7); in 2D the third tangent is z
__device__ __noinline__ bool dual(int dim, const double gl[3][3], double &J, double gu[3][3]) {
  for (int i = 0; i < 3; i++)
    for (int d = 0; d < 3; d++) gu[i][d] = 0.0;
  if (dim == 2) {
    J = gl[0][0] * gl[1][1] - gl[0][1] * gl[1][0];
    if (!(J > 0.0)) return false;
    gu[0][0] = gl[1][1] / J;
    gu[0][1] = -gl[1][0] / J;
    gu[1][0] = -gl[0][1] / J;
    gu[1][1] = gl[0][0] / J;
    return true;
  }
  double c12[3], c23[3], c31[3];
  auto cross = [](const double *a, const double *b, double *c) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
  };
  cross(gl[0], gl[1], c12);
  cross(gl[1], gl[2], c23);
  cross(gl[2], gl[0], c31);
  J = c12[0] * gl[2][0] + c12[1] * gl[2][1] + c12[2] * gl[2][2];
  if (!(J > 0.0)) return false;
  for (int d = 0; d < 3; d++) {
    gu[0][d] = c23[d] / J;
    gu[1][d] = c31[d] / J;
    gu[2][d] = c12[d] / J;
  }
  return true;
}

// ------------------------------------------------------------------ precompute
// Tangents, J, co-tangents and g^ij of every cell. A cell away from every end of
// an axis reads its 2 D + 1 node positions directly; the others go through position().
template <int Q>
__global__ void __launch_bounds__(128) k_tangents(const MeshDev m, Grid g, int64_t ncell, double *J_out, double *gl_out,
                                                  double *gu_out, double *ginv_out, int *err) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2;
  const int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= ncell) return;
  const Addr<19> ad(g, cell);   // (index coordinates only)
  bool inner = true;
#pragma unroll
  for (int i = 0; i < D; i++) inner = inner && ad.ic[i] > 0 && ad.ic[i] < g.n[i] - 1;
  double gl[3][3], gu[3][3], J = 0.0;
  bool ok = true;
  if (inner) {
    const double dx = m.dx > 0.0 ? m.dx : 1.0;
    const double *x = m.x + cell * D;
    double x0[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int d = 0; d < D; d++) x0[d] = x[d];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int d = 0; d < 3; d++) gl[i][d] = 0.0;
#pragma unroll
    for (int i = 0; i < D; i++) {
      double Dp[3] = {0.0, 0.0, 0.0}, Dm[3] = {0.0, 0.0, 0.0}, df[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int d = 0; d < D; d++) {
        Dp[d] = x[g.s[i] * D + d] - x0[d];
        Dm[d] = x[-g.s[i] * D + d] - x0[d];
        df[d] = Dp[d] - Dm[d];
      }
      const double nd = nrm(df);
      if (!(nd > 0.0)) ok = false;
      const double beta = (nrm(Dp) + nrm(Dm)) / nd;
#pragma unroll
      for (int d = 0; d < D; d++) gl[i][d] = beta * df[d] / (2.0 * dx);
    }
  } else {
    const int64_t q[3] = {ad.ic[0], ad.ic[1], ad.ic[2]};
    ok = tangents(m, q, gl);
  }
  ok = ok && dual(D, gl, J, gu);
  if (!ok) {
    atomicOr(err, ERR_GEOM);
    J = nan("");
  }
  J_out[cell] = J;
  for (int i = 0; i < D; i++)
    for (int d = 0; d < D; d++) {
      gl_out[(cell * D + i) * D + d] = gl[i][d];
      gu_out[(cell * D + i) * D + d] = gu[i][d];
    }
  for (int i = 0; i < D; i++)
    for (int j = i; j < D; j++) {
      double s = 0.0;
      for (int d = 0; d < 3; d++) s += gu[i][d] * gu[j][d];  // g^ij = g^i . g^j (Eq. 8)
      ginv_out[cell * NS + sym<D>(i, j)] = s;
    }
}

// K^i_a = sum_j c^j_a [g_j(q + c_a) - g_j(q)] . g^i(q) = sum_j c^j_a Theta^i_j(q + c_a, q) (Eq. 11), one
// thread per cell and direction, from the stored tangents (links off the mesh: from
// the positions of the image or ghost nodes). Forming the tangents again at every
// neighbour (19 times per cell, each from seven positions) had made the precompute
// 7.0 ms on 492 K general D3Q19 cells; 0.64 ms (tangents) and 1.26 ms (links) so.
template <int Q>
__global__ void __launch_bounds__(256) k_links(const MeshDev m, Grid g, int64_t ncell, const double *gl,
                                               const double *gu, double *K_out, int *err) {
  constexpr int D = Lat<Q>::D;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ncell * Q) return;
  const int64_t cell = t / Q;
  const int a = (int)(t - cell * Q);
  int64_t q[3];
  {
    int64_t r = cell;
    q[2] = r % g.n[2];
    r /= g.n[2];
    q[1] = r % g.n[1];
    q[0] = r / g.n[1];
  }
  int c[3] = {0, 0, 0};
  int64_t p[3] = {q[0], q[1], q[2]};
  bool wall = false, out = false;   // the link leaves through a wall, or at all
  for (int d = 0; d < D; d++) {
    c[d] = Lat<Q>::c(a, d);
    p[d] += c[d];
    if (p[d] >= 0 && p[d] < g.n[d]) continue;
    out = true;
    wall = wall || g.wall[d];
  }
  double Kv[3] = {0.0, 0.0, 0.0};
  // links that cross a wall: zero, or from the ghost-node tangents
  if (a != 0 && (!wall || m.wall_links == VLB_WALL_LINKS_GHOST)) {
    double gp[3][3], de[3] = {0.0, 0.0, 0.0};
    if (out) {
      if (!tangents(m, p, gp)) atomicOr(err, ERR_GEOM);
    } else {
      const double *o = gl + ((p[0] * g.n[1] + p[1]) * g.n[2] + p[2]) * D * D;
      for (int j = 0; j < D; j++)
        for (int d = 0; d < 3; d++) gp[j][d] = d < D ? o[j * D + d] : 0.0;
    }
    for (int j = 0; j < D; j++) {
      if (c[j] == 0) continue;
      for (int d = 0; d < D; d++) de[d] += c[j] * (gp[j][d] - gl[(cell * D + j) * D + d]);
    }
    for (int i = 0; i < D; i++) {
      // (one expression: how its products and sums are contracted shows in the last bit)
      const double *r = gu + (cell * D + i) * D;
      Kv[i] = de[0] * r[0] + de[1] * r[1] + de[2] * (D == 3 ? r[D - 1] : 0.0);
    }
  }
  for (int i = 0; i < D; i++) K_out[t * D + i] = Kv[i];
}

template <int Q>
static void launch_geometry_q(const vlb_mesh *m, int *d_err, cudaStream_t s) {
  const Grid g = make_grid(m);
  k_tangents<Q><<<(unsigned)((m->ncell + 127) / 128), 128, 0, s>>>(m->md, g, m->ncell, m->d_J, m->d_gl, m->d_gu,
                                                                    m->d_ginv, d_err);
  k_links<Q><<<(unsigned)((m->ncell * Q + 255) / 256), 256, 0, s>>>(m->md, g, m->ncell, m->d_gl, m->d_gu, m->d_K,
                                                                     d_err);
}
cudaError_t launch_geometry(const vlb_mesh *m, int *d_err, cudaStream_t s) {
  if (m->md.q == 9)
    launch_geometry_q<9>(m, d_err, s);
  else if (m->md.q == 39)
    launch_geometry_q<39>(m, d_err, s);
  else
    launch_geometry_q<19>(m, d_err, s);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ diagnostics
// per block: [min J, -max J, min f^eq_rest/w, min g^ii, -max g^ii], reduced on the host
template <int Q>
__global__ void k_mesh_stats(const double *J, const double *ginv, int64_t ncell,
                             double *partial) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2, H = Lat<Q>::H;
  __shared__ double sh[5][kStatThreads];
  double v[5] = {1e300, 1e300, 1e300, 1e300, 1e300};
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncell;
       c += (int64_t)gridDim.x * blockDim.x) {
    v[0] = fmin(v[0], J[c]);
    v[1] = fmin(v[1], -J[c]);
    double gi[NS], gd[NS], U[D], Ut[D];
    for (int i = 0; i < NS; i++) gd[i] = gi[i] = ginv[c * NS + i];
    for (int i = 0; i < D; i++) gd[sym<D>(i, i)] -= 1.0;
    for (int i = 0; i < D; i++) U[i] = Ut[i] = 0.0;
    EqParts<Q, double> e;
    eq_parts<Q, double>(gd, U, Ut, e);
    double m = eq_even<Q, double>(e, 0);
#pragma unroll
    for (int p = 1; p <= H; p++) m = fmin(m, eq_even<Q, double>(e, p));
    v[2] = fmin(v[2], m);
    for (int i = 0; i < D; i++) {
      v[3] = fmin(v[3], gi[sym<D>(i, i)]);
      v[4] = fmin(v[4], -gi[sym<D>(i, i)]);
    }
  }
  for (int k = 0; k < 5; k++) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int k = 0; k < 5; k++) sh[k][threadIdx.x] = fmin(sh[k][threadIdx.x], sh[k][threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; k++) partial[blockIdx.x * 5 + k] = sh[k][0];
}

cudaError_t launch_mesh_stats(const vlb_mesh *m, double *d_partial, int64_t nblk, cudaStream_t s) {
  if (m->md.q == 9)
    k_mesh_stats<9><<<(unsigned)nblk, kStatThreads, 0, s>>>(m->d_J, m->d_ginv, m->ncell, d_partial);
  else
    k_mesh_stats<19><<<(unsigned)nblk, kStatThreads, 0, s>>>(m->d_J, m->d_ginv, m->ncell, d_partial);
  return cudaGetLastError();
}

// plane check: does every cell's geometry equal that of the first cell of its
// column along the fastest axis (to 1e-12 relative)? Flag bit 0: no. Bit 1: the columns are
// not those of an extruded mesh (D3Q19; see collide_f32), to the rounding of FP64:
// g^02 = g^12 = 0, K^2_a = 0, and K_a is that of the pair with c^2_a = 0.
__device__ __forceinline__ bool close12(double a, double b) {
  return fabs(a - b) <= 1e-12 * (1.0 + fabs(b));
}

template <int Q>
__global__ void k_plane_check(const double *J, const double *ginv, const double *gu,
                              const double *K, int64_t ncell, int64_t nfast, int *flag) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const int64_t c0 = (c / nfast) * nfast;
  // (a mesh that varies is known to at once: the rest need not be read)
  if (*(volatile int *)flag & 1) return;
  if (c0 == c) {
    if constexpr (Q == 19) {
      const double *k = K + c * Q * D, tiny = 1e-15;
      bool ext = fabs(ginv[c * NS + sym<D>(0, 2)]) <= tiny && fabs(ginv[c * NS + sym<D>(1, 2)]) <= tiny;
      for (int a = 1; a < Q; a++) {
        int b = 0;   // the direction with the same c^0, c^1 and c^2 = 0
        for (int e = 1; e < Q; e++)
          if (Lat<Q>::c(e, 0) == Lat<Q>::c(a, 0) && Lat<Q>::c(e, 1) == Lat<Q>::c(a, 1) && Lat<Q>::c(e, 2) == 0) b = e;
        for (int i = 0; i < 2; i++) {
          const double r = b > 0 ? k[b * D + i] : 0.0;
          ext = ext && fabs(k[a * D + i] - r) <= tiny * (1.0 + fabs(r));
        }
        ext = ext && fabs(k[a * D + 2]) <= tiny;
      }
      if (!ext) atomicOr(flag, 2);
    }
    return;
  }
  bool same = close12(J[c], J[c0]);
  for (int i = 0; i < NS; i++) same = same && close12(ginv[c * NS + i], ginv[c0 * NS + i]);
  for (int i = 0; i < D * D; i++) same = same && close12(gu[c * D * D + i], gu[c0 * D * D + i]);
  for (int i = 0; i < Q * D; i++) same = same && close12(K[c * Q * D + i], K[c0 * Q * D + i]);
  if (!same) atomicOr(flag, 1);
}

cudaError_t launch_plane_check(const vlb_mesh *m, int *d_flag, cudaStream_t s) {
  const int threads = 256;
  const int64_t blocks = (m->ncell + threads - 1) / threads;
  const int64_t nfast = m->md.n[m->md.dim - 1];
  if (m->md.q == 9)
    k_plane_check<9><<<(unsigned)blocks, threads, 0, s>>>(m->d_J, m->d_ginv, m->d_gu, m->d_K,
                                                          m->ncell, nfast, d_flag);
  else
    k_plane_check<19><<<(unsigned)blocks, threads, 0, s>>>(m->d_J, m->d_ginv, m->d_gu, m->d_K,
                                                           m->ncell, nfast, d_flag);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ coefficient records
struct PackArgs {
  MeshDev md;
  Grid g;
  const double *J, *gu, *ginv, *K;
  int64_t nrec, stride, nfast;
  int32_t plane;
  double tau;
  double body[3];
  double wall_u[3][2][3];
  double wall_omega[3][2][3];
  int32_t ref_rest;  // fill the storage-reference offsets (16-bit storage, plane mode)
  double nref;
  CellFactors cf;    // CellLayout records
  float *uw;         // their wall velocities (NULL: no moving walls)
  float *ro;         // (ref_rest) the storage reference per column and pair
};

// wall velocity of a cell: rigid motion of the adjacent wall, at the point halfway
// to the ghost node (zero away from walls)
template <int Q>
__device__ void wall_velocity(const PackArgs &a, int64_t c, double (&uw)[3]) {
  constexpr int D = Lat<Q>::D;
  const Addr<Q> ad(a.g, c);
  uw[0] = uw[1] = uw[2] = 0.0;
  for (int ax = 0; ax < D; ax++) {
    if (!(ad.lo[ax] || ad.hi[ax])) continue;
    const int side = ad.lo[ax] ? 0 : 1;
    int64_t q[3] = {ad.ic[0], ad.ic[1], ad.ic[2]}, gq[3] = {ad.ic[0], ad.ic[1], ad.ic[2]};
    gq[ax] += side ? 1 : -1;
    double x0[3], xg[3], xw[3], u[3];
    position(a.md, q, x0);
    position(a.md, gq, xg);
    for (int d = 0; d < 3; d++) xw[d] = 0.5 * (x0[d] + xg[d]);
    const double *om = a.wall_omega[ax][side];
    u[0] = om[1] * xw[2] - om[2] * xw[1];
    u[1] = om[2] * xw[0] - om[0] * xw[2];
    u[2] = om[0] * xw[1] - om[1] * xw[0];
    for (int d = 0; d < 3; d++) u[d] += a.wall_u[ax][side][d];
    for (int i = 0; i < D; i++) {
      double s = 0.0;
      for (int d = 0; d < D; d++) s += u[d] * a.gu[(c * D + i) * D + d];
      uw[i] = s;
    }
    break;
  }
}

template <int Q, typename R>
__global__ void k_pack_coef(const PackArgs a, R *coef) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2, H = Lat<Q>::H;
  using L = CoefLayout<Q>;
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= a.nrec) return;
  const int64_t c = a.plane ? r * a.nfast : r;
  double K[Q][D], G[D], rec[L::NC];
  for (int av = 0; av < Q; av++)
    for (int i = 0; i < D; i++) K[av][i] = a.K[(c * Q + av) * D + i];
  for (int i = 0; i < D; i++) {
    double s = 0.0;
    for (int d = 0; d < D; d++) s += a.body[d] * a.gu[(c * D + i) * D + d];  // G^i = G . g^i
    G[i] = s;
  }
  build_record<Q>(a.J[c], a.ginv + c * NS, G, K, a.tau, rec);
  // F at rest (rho = 1, U = 0), the start value of the chord iteration
  {
    double gd[NS], U0[D], N[Q], Np[Q];
    for (int i = 0; i < NS; i++) gd[i] = 2.0 * rec[L::GH + i];
    for (int i = 0; i < D; i++) U0[i] = 0.0;
    EqParts<Q, double> e;
    eq_parts<Q, double>(gd, U0, U0, e);
    for (int av = 0; av < Q; av++) {
      const int p = av <= H ? av : av - H;
      N[av] = rec[L::J] * lat_w<Q, double>(av) * eq_even<Q, double>(e, p);
    }
    CollideState<Q, double> cs;
    // chord iteration from F = 0 (the record's FR is still zero here)
    collide_cell<Q, double, false>(N, PtrRecord<double>{rec}, 0.0, 1.0 / a.tau, 1e-15, 400, Np, cs);
    for (int i = 0; i < D; i++) rec[L::FR + i] = cs.conv ? cs.F[i] : 0.0;
  }
  // the local rest state for the final pass: deviations from the uniform
  // reference, their sum over all directions, and the rest weights
  {
    double gd[NS], U0[D], rsum = 0.0;
    for (int i = 0; i < NS; i++) gd[i] = 2.0 * rec[L::GH + i];
    for (int i = 0; i < D; i++) U0[i] = 0.0;
    EqParts<Q, double> e;
    eq_parts<Q, double>(gd, U0, U0, e);
    for (int p = 0; p <= H; p++) {
      const double rwp = lat_w<Q, double>(p) * eq_even<Q, double>(e, p);
      const double r = a.J[c] * rwp - lat_w<Q, double>(p) * a.nref;
      rec[L::RR + p] = r;
      rec[L::RW + p] = rwp;
      rsum += p == 0 ? r : 2.0 * r;
    }
    rec[L::RR + H + 1] = rsum;
  }
  // 16-bit storage relative to the rest state of Eq. 33 at the column that
  // holds each location (the fastest axis never changes the column, so only
  // the other axes decide a wall crossing): the constants and the per-link
  // column differences that let the collision work on N_a - o_a(own)
  if (a.ref_rest) {
    const Addr<Q> ad0(a.g, c);
    double own[Q], osum = 0.0;
    for (int av = 0; av < Q; av++) {
      own[av] = rest_ref<Q>(a.J[c], a.ginv + c * NS, av);
      osum += own[av];
      if (av <= H) a.ro[r * (H + 1) + av] = (float)own[av];   // (an FP32 value already)
    }
    rec[L::MDV] = osum - a.nref;   // the weights sum to one
    rec[L::MNV] = osum - a.J[c];
    for (int i = 0; i < D; i++) {
      double s = 0.0;
      for (int p = 1; p <= H; p++) s += rec[L::mp(p, i)] * 2.0 * (own[p] - lat_w<Q, double>(p) * a.nref);
      rec[L::SR + i] = s;
    }
    for (int av = 0; av < Q; av++) {
      for (int sg = -1; sg <= 1; sg += 2) {
        bool crs = false;
        for (int ax = 0; ax < D - 1; ax++) {
          const int cd = sg * Lat<Q>::c(av, ax);
          if ((cd > 0 && ad0.hi[ax]) || (cd < 0 && ad0.lo[ax])) crs = true;
        }
        const int64_t cb = crs || av == 0 ? c : (ad0.nb(av, sg) / a.nfast) * a.nfast;
        const double ob = rest_ref<Q>(a.J[cb], a.ginv + cb * NS, av);
        if (sg < 0)
          rec[L::DIN + av] = ob - own[av];
        else
          rec[L::DOUT + av] = own[av] - ob;
      }
    }
  }
  // reference-state part of J F as a hi/lo pair
  for (int i = 0; i < D; i++) rec[L::KWL + i] = rec[L::KW + i] - static_cast<double>(static_cast<R>(rec[L::KW + i]));
  R *out = coef + r * a.stride;
  // a per-cell record ends at RR (see CoefLayout::stride)
  for (int k = 0; k < a.stride; k++) out[k] = k < L::NC ? static_cast<R>(rec[k]) : R(0);
  double uw[3];
  wall_velocity<Q>(a, c, uw);
  for (int i = 0; i < D; i++) out[L::UW + i] = static_cast<R>(uw[i]);
}

// Are the entries that the collision of extruded meshes with 16-bit storage leaves out (see
// map_mono) zero in every record? Three groups may keep what is left of FP64 sums whose terms
// cancel, 2^-45 of their block at most (1e-16 of it on the channels here): column 2 of
// H - I and of PO1, and the map's monomials odd in U~^2. A product with such an entry is below the
// last FP32 bit of a sum whose terms do not cancel to 2^-20 of themselves. And H - I may
// keep a last bit of its diagonal, which is added to one. Raises ERR_ZERO_EXT where not.
__global__ void k_zero_entries(const float *coef, int64_t nrec, int64_t stride, int *err) {
  using L = CoefLayout<19>;
  constexpr int D = L::D, H = L::H, NQ = L::NQ;
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrec) return;
  const float *c = coef + r * stride;
  // the largest of the zeros, of the remainders of the map and of PO1, and of those blocks
  float zero = 0.0f, left = 0.0f, map = 0.0f, pleft = 0.0f, po = 0.0f;
  auto see = [&](float &m, int k) { m = maxnan(m, fabsf(c[k])); };
  for (int i = 0; i < 2; i++) {
    see(zero, L::GH + sym<D>(i, 2));
    for (int j = 0; j < D; j++) see(j < 2 ? po : pleft, L::PO1 + i * D + j);
    see(zero, L::row(L::HM, D, 2, i));
    see(zero, L::mp(3, i));
    see(zero, L::dk(3, i));
    for (int k = 0; k < NQ; k++) see(map_mono<true, D>(k) ? map : left, L::row(L::QM, NQ, i, k));
  }
  for (int j = 0; j < D; j++) see(zero, L::PO1 + 2 * D + j);
  for (int k = 0; k < NQ; k++) see(zero, L::row(L::QM, NQ, 2, k));
  for (int q = 1; q <= H; q++) {
    see(zero, L::mp(q, 2));
    see(zero, L::dk(q, 2));
  }
  see(zero, L::KW + 2);
  see(zero, L::KWL + 2);
  see(zero, L::CE + 2);
  see(zero, L::SR + 2);
  float col = 0.0f;
  for (int i = 0; i < 2; i++) see(col, L::row(L::HM, D, i, 2));
  const float tiny = 2.8421709e-14f;   // 2^-45
  const bool ok = zero == 0.0f && left <= tiny * map && pleft <= tiny * po && col <= tiny &&
                  fabsf(c[L::row(L::HM, D, 2, 2)]) <= 1.4901161e-8f;
  if (!ok) atomicOr(err, ERR_ZERO_EXT);
}

cudaError_t launch_zero_entries(const vlb_sim *sim, cudaStream_t s) {
  k_zero_entries<<<(unsigned)((sim->ncoef + 127) / 128), 128, 0, s>>>(static_cast<const float *>(sim->d_coef),
                                                                     sim->ncoef, sim->nc, sim->d_err);
  return cudaGetLastError();
}

// CellLayout records (FP32, one per cell): the entries kept are sums over the
// links formed in FP64 (about 250 operations; the whole record takes ten times that)
// and rounded; the rest state's force, the start value of the chord iteration, is
// solved in FP32 on the finished record. 492 K D3Q19 cells: 2.24 -> 0.33 ms.
template <int Q>
__global__ void __launch_bounds__(128) k_pack_cells(const PackArgs a, float4 *coef) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2, H = Lat<Q>::H;
  using L = CoefLayout<Q>;
  using CL = CellLayout<Q>;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.nrec) return;
  const double itau = 1.0 / a.tau, J = a.J[c];
  CellRecord<Q> r;
  double gd[NS], tr = 0.0, kw[D], ce[D];
#pragma unroll
  for (int i = 0; i < D; i++)
#pragma unroll
    for (int j = i; j < D; j++) {
      gd[sym<D>(i, j)] = a.ginv[c * NS + sym<D>(i, j)] - (i == j ? 1.0 : 0.0);
      r.v[L::GH + sym<D>(i, j)] = (float)(0.5 * gd[sym<D>(i, j)]);
    }
#pragma unroll
  for (int i = 0; i < D; i++) {
    tr += gd[sym<D>(i, i)];
    kw[i] = ce[i] = 0.0;
    double s = 0.0;
#pragma unroll
    for (int d = 0; d < D; d++) s += a.body[d] * a.gu[(c * D + i) * D + d];  // G^i = G . g^i
    r.v[L::BODY + i] = (float)s;
  }
  const double *K = a.K + c * Q * D;
  float N[Q], Np[Q];
  const double am = -0.25 * (2.0 - itau), ad = 0.25 * itau;
#pragma unroll
  for (int p = 1; p <= H; p++) {
    const double w = lat_w<Q, double>(p);
    double cgc = 0.0;
#pragma unroll
    for (int k = 0; k < D; k++)
#pragma unroll
      for (int l = 0; l < D; l++) {
        const int cc = Lat<Q>::c(p, k) * Lat<Q>::c(p, l);
        if (cc != 0) cgc += cc * gd[sym<D>(k, l)];
      }
    // CE^i = T0 sum_kl PE^i_kl gd_kl = itau/2 sum_p w (3 c.gd.c - tr gd) M^i_p; the rest
    // state's populations J w (1 + (3 c.gd.c - tr gd) / 2)
    const double h = w * (3.0 * cgc - tr);
    N[p] = N[p + H] = (float)(J * (w + 0.5 * h));
#pragma unroll
    for (int i = 0; i < D; i++) {
      const double kp = K[p * D + i], km = K[(p + H) * D + i], M = kp + km;
      kw[i] += w * M;
      ce[i] += h * M;
      r.v[L::mp(p, i)] = (float)(am * M);
      r.v[L::dk(p, i)] = (float)(ad * (kp - km));
    }
  }
  N[0] = (float)(J * lat_w<Q, double>(0) * (1.0 - 0.5 * tr));
  r.v[L::J] = (float)J;
  r.v[L::IJ] = (float)(1.0 / J);
#pragma unroll
  for (int i = 0; i < D; i++) {
    r.v[L::KW + i] = (float)kw[i];
    r.v[L::KWL + i] = (float)(kw[i] - (double)(float)kw[i]);
    r.v[L::CE + i] = (float)(0.5 * itau * ce[i]);
    r.v[L::FR + i] = 0.0f;
  }
  r.form(a.cf.k6am, a.cf.kpe, a.cf.ktt);
  CollideState<Q, float> cs;
  collide_cell<Q, float, false>(N, r, 0.0f, (float)itau, 1e-6f, 100, Np, cs);
#pragma unroll
  for (int i = 0; i < D; i++) r.v[L::FR + i] = cs.conv ? cs.F[i] : 0.0f;
  float4 *o = coef + (c >> 5) * (CL::NG * 32) + (c & 31);
#pragma unroll
  for (int g = 0; g < CL::NG; g++) {
    float e[4];
#pragma unroll
    for (int u = 0; u < 4; u++) e[u] = CL::entry(4 * g + u) >= 0 ? r.v[CL::entry(4 * g + u)] : 0.0f;
    o[g * 32] = make_float4(e[0], e[1], e[2], e[3]);
  }
  if (!a.uw) return;
  double uw[3];
  wall_velocity<Q>(a, c, uw);
  for (int i = 0; i < D; i++) a.uw[c * D + i] = (float)uw[i];
}

template <int Q>
static cudaError_t pack_q(const vlb_sim *sim, cudaStream_t s) {
  const vlb_mesh *m = sim->mesh;
  PackArgs a;
  a.md = m->md;
  a.g = make_grid(m);
  a.J = m->d_J;
  a.gu = m->d_gu;
  a.ginv = m->d_ginv;
  a.K = m->d_K;
  a.nrec = sim->ncoef;
  a.stride = sim->nc;
  a.nfast = m->md.n[m->md.dim - 1];
  a.plane = sim->plane;
  a.tau = sim->p.tau;
  a.ref_rest = sim->ref_rest;
  a.nref = sim->nref;
  a.cf = cell_factors(a.tau);
  a.uw = sim->d_uw;
  a.ro = sim->d_ro;
  for (int d = 0; d < 3; d++) a.body[d] = sim->p.body_force[d];
  for (int ax = 0; ax < 3; ax++)
    for (int sd = 0; sd < 2; sd++)
      for (int d = 0; d < 3; d++) {
        a.wall_u[ax][sd][d] = sim->p.wall_u[ax][sd][d];
        a.wall_omega[ax][sd][d] = sim->p.wall_omega[ax][sd][d];
      }
  const int threads = 128;
  const int64_t blocks = (a.nrec + threads - 1) / threads;
  if (sim->cellrec)
    k_pack_cells<Q><<<(unsigned)blocks, threads, 0, s>>>(a, (float4 *)sim->d_coef);
  else if (arith_f64(sim->p.precision))
    k_pack_coef<Q, double><<<(unsigned)blocks, threads, 0, s>>>(a, (double *)sim->d_coef);
  else
    k_pack_coef<Q, float><<<(unsigned)blocks, threads, 0, s>>>(a, (float *)sim->d_coef);
  return cudaGetLastError();
}

cudaError_t launch_pack_coef(const vlb_sim *sim, cudaStream_t s) {
  return sim->mesh->md.q == 9 ? pack_q<9>(sim, s) : pack_q<19>(sim, s);
}

// ------------------------------------------------------------------ initial state
// N_a = J f^eq_a(rho, U, U~ = U), U^i = u . g^i (Eqs. 14, 33), normal layout, in FP64: for FP64
// storage and for 16-bit storage relative to the rest state, whose stored value is what is left of
// N_a after the reference o_a. Bound by the FP64 pipe (some 400 operations a D3Q19 cell); o_a is
// read (RefCtx::o) rather than formed per population, which had doubled them: 128^3 cells, FP16:
// 2.06 -> 0.83 ms.
template <int Q, typename S>
__global__ void k_init(const double *J, const double *gu, const double *ginv, const double *rho,
                       const double *u, int64_t ncell, RefCtx ref, S *f) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2, H = Lat<Q>::H;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  double U[D], gd[NS], zero[D];
  for (int i = 0; i < D; i++) {
    double s = 0.0;
    for (int d = 0; d < D; d++) s += u[c * D + d] * gu[(c * D + i) * D + d];
    U[i] = s;
    zero[i] = 0.0;
  }
  for (int i = 0; i < NS; i++) gd[i] = ginv[c * NS + i];
  for (int i = 0; i < D; i++) gd[sym<D>(i, i)] -= 1.0;
  EqParts<Q, double> e;
  eq_parts<Q, double>(gd, U, zero, e);
  const double r = rho[c], Jc = J[c];
  // stored relative to the storage reference of each location
  f[c] = store_s<S>(Jc * r * lat_w<Q, double>(0) * eq_even<Q, double>(e, 0) - ref_at<Q>(ref, 0, c));
#pragma unroll
  for (int p = 1; p <= H; p++) {
    const double E = eq_even<Q, double>(e, p), O = eq_odd<Q, double>(e, U, p);
    const double w = lat_w<Q, double>(p), rw = Jc * r * w, o = ref_at<Q>(ref, p, c);
    f[p * ncell + c] = store_s<S>(rw * (E + O) - o);
    f[(p + H) * ncell + c] = store_s<S>(rw * (E - O) - o);
  }
}

// The same initial state for FP32 arithmetic (FP32 or 16-bit storage relative
// to the uniform reference n_ref): with J f^eq_a = J rho w_a (1 + x_a),
//   N_a - w_a n_ref = w_a [(J rho - n_ref) + J rho x_a],
// J rho - n_ref is formed in FP64 (one difference of large terms) and the
// bracket x_a in FP32, so every FP32 term is of the size of the deviation.
// (GB300's FP64 rate is a small fraction of its FP32 rate; the FP64 form of
// k_init is bound by it.)
template <int Q>
__device__ __forceinline__ float eq_even_x(const EqParts<Q, float> &e, int a) {
  constexpr int D = Lat<Q>::D;
  float cbc = 0.0f;
#pragma unroll
  for (int i = 0; i < D; i++) {
    const int ci = Lat<Q>::c(a, i);
    if (ci == 0) continue;
#pragma unroll
    for (int j = 0; j < D; j++) {
      const int cj = Lat<Q>::c(a, j);
      if (cj == 0) continue;
      if (ci * cj > 0)
        cbc += e.B[i][j];
      else
        cbc -= e.B[i][j];
    }
  }
  return (3.0f * cbc - e.trB) * 1.5f;
}

template <int Q, typename S>
__global__ void k_init_f32(const double *J, const double *gu, const double *ginv, const double *rho,
                           const double *u, int64_t ncell, double nref, S *f) {
  constexpr int D = Lat<Q>::D, NS = D * (D + 1) / 2, H = Lat<Q>::H;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  float U[D], gd[NS], zero[D];
  for (int i = 0; i < D; i++) {
    float s = 0.0f;
    for (int d = 0; d < D; d++) s = fmaf((float)u[c * D + d], (float)gu[(c * D + i) * D + d], s);
    U[i] = s;
    zero[i] = 0.0f;
  }
  // g^ii - 1 formed in FP64 before rounding
  for (int i = 0; i < D; i++)
    for (int j = i; j < D; j++)
      gd[sym<D>(i, j)] = (float)(ginv[c * NS + sym<D>(i, j)] - (i == j ? 1.0 : 0.0));
  EqParts<Q, float> e;
  eq_parts<Q, float>(gd, U, zero, e);
  const double jr = J[c] * rho[c];
  const float md = (float)(jr - nref), jrf = (float)jr;
  f[c] = store_s<S>(lat_w<Q, float>(0) * fmaf(jrf, eq_even_x<Q>(e, 0), md));
#pragma unroll
  for (int p = 1; p <= H; p++) {
    const float xe = eq_even_x<Q>(e, p), xo = eq_odd<Q, float>(e, U, p), w = lat_w<Q, float>(p);
    f[p * ncell + c] = store_s<S>(w * fmaf(jrf, xe + xo, md));
    f[(p + H) * ncell + c] = store_s<S>(w * fmaf(jrf, xe - xo, md));
  }
}

cudaError_t launch_init(const vlb_sim *sim, const double *d_rho, const double *d_u, cudaStream_t s) {
  const vlb_mesh *m = sim->mesh;
  const int threads = 128;
  const int64_t blocks = (m->ncell + threads - 1) / threads;
  const RefCtx ref = make_ref(sim);
  return with_storage(sim->p.precision, [&](auto tag) {
    using S = typename decltype(tag)::type;
    if constexpr (!std::is_same<S, double>::value) {
      // FP32 arithmetic for the uniform reference (the rest reference of 16-bit storage keeps
      // the FP64 form: what is stored is a small difference, rounded to 16 bits)
      if (!ref.rest) {
        if (m->md.q == 9)
          k_init_f32<9, S><<<(unsigned)blocks, threads, 0, s>>>(m->d_J, m->d_gu, m->d_ginv, d_rho, d_u, m->ncell,
                                                                ref.nref, (S *)sim->d_f);
        else
          k_init_f32<19, S><<<(unsigned)blocks, threads, 0, s>>>(m->d_J, m->d_gu, m->d_ginv, d_rho, d_u, m->ncell,
                                                                 ref.nref, (S *)sim->d_f);
        return cudaGetLastError();
      }
    }
    if constexpr (!std::is_same<S, float>::value) {
      if (m->md.q == 9)
        k_init<9, S><<<(unsigned)blocks, threads, 0, s>>>(m->d_J, m->d_gu, m->d_ginv, d_rho, d_u, m->ncell, ref,
                                                          (S *)sim->d_f);
      else
        k_init<19, S><<<(unsigned)blocks, threads, 0, s>>>(m->d_J, m->d_gu, m->d_ginv, d_rho, d_u, m->ncell, ref,
                                                           (S *)sim->d_f);
    }
    return cudaGetLastError();
  });
}

}  // namespace vlb
