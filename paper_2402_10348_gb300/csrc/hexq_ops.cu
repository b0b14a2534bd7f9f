// Residuals of the three kinds of block on hexahedra, their float64 products at a state that is used
// a few times, and the quadrature-point coefficients of the momentum block, one thread per (element, quadrature point)
// (hexq.cuh); ops.cuh has the equations.
#include "hexq.cuh"
#include "ops_impl.cuh"

namespace fsi {

// R_m, tau and the stresses at a point, tested: E[8 x equation + corner][element], unweighted
__global__ void __launch_bounds__(HQ_THREADS) hq_ns_res_kernel(const __grid_constant__ HexNS H, double* __restrict__ E,
                                                               unsigned e0, unsigned e1) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const int64_t es = H.stride(), at = H.at(l);
  NSPoint p;
  hq_ns_point(H, l, p);
  double S[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int s = 0; s < H.P.ns; ++s) {
    const double a = l.val(H.mat[(2 + s) * H.nn + l.n]) * H.P.muL[H.P.solid_phase[s]];
    const double* b = H.xa + (int64_t)(4 + H.P.N + 6 * s) * H.nn + l.n;
#pragma unroll
    for (int c = 0; c < 6; ++c) S[c] = fma(a, l.val(b[c * H.nn]) - (c < 3 ? 1.0 : 0.0), S[c]);
  }
  const double Rc = p.L[0][0] + p.L[1][1] + p.L[2][2];
  const double iso = p.tau_c * p.rho * Rc - p.p;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double g[3];
    const double tR = p.tau_m * p.R[k];
#pragma unroll
    for (int j = 0; j < 3; ++j)
      g[j] = fma(p.v[j], tR, fma(p.mu, p.L[k][j] + p.L[j][k], S[sym_idx(k, j)])) + (j == k ? iso : 0.0);
    const double c = l.scatter(p.R[k] - p.gp[k], g[0], g[1], g[2]);  // rho (acc_k - g_k)
    if (l.ok) E[(8 * k + l.q) * es + at] = c;
  }
  const double r = p.tau_m * p.rrho;
  const double c = l.scatter(Rc, r * p.R[0], r * p.R[1], r * p.R[2]);
  if (l.ok) E[(24 + l.q) * es + at] = c;
}

__global__ void __launch_bounds__(HQ_THREADS) hq_ac_res_kernel(const __grid_constant__ HexNS H, int phase, double gam,
                                                               double bet, double* __restrict__ E, unsigned e0, unsigned e1) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const Phys& P = H.P;
  double v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = l.val(H.xa[k * H.nn + l.n]);
  const VG<double> ph = l.vg(H.xa[(4 + phase) * H.nn + l.n]);
  const double rate = l.val(H.xd[(4 + phase) * H.nn + l.n]);
  const double phi = ph.v, k_hat = gam * P.eps * P.eps, s_hat = gam * (3.0 * phi * phi - 1.0);
  const double vGv = P.Gd[0] * v[0] * v[0] + P.Gd[1] * v[1] * v[1] + P.Gd[2] * v[2] * v[2];
  const double tau = rsqrt(H.dt2 + vGv + 9.0 * k_hat * k_hat * P.GG + s_hat * s_hat);
  const double R = rate + v[0] * ph.gx + v[1] * ph.gy + v[2] * ph.gz +
                   gam * (phi * phi * phi - phi - bet * (0.5 * fabs(phi * phi - 1.0)));
  const double t = tau * R;
  const double c = l.scatter(R, k_hat * ph.gx + t * v[0], k_hat * ph.gy + t * v[1], k_hat * ph.gz + t * v[2]);
  if (l.ok) E[l.q * H.stride() + H.at(l)] = H.W * c;
}

__global__ void __launch_bounds__(HQ_THREADS) hq_b_res_kernel(const __grid_constant__ HexNS H, int solid,
                                                              double* __restrict__ E, unsigned e0, unsigned e1) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const Phys& P = H.P;
  const int64_t nn = H.nn, es = H.stride(), at = H.at(l);
  double v[3], L[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const VG<double> r = l.vg(H.xa[k * nn + l.n]);
    v[k] = r.v; L[k][0] = r.gx; L[k][1] = r.gy; L[k][2] = r.gz;
  }
  const double al = l.val(H.mat[(2 + solid) * nn + l.n]);
  const double vGv = P.Gd[0] * v[0] * v[0] + P.Gd[1] * v[1] * v[1] + P.Gd[2] * v[2] * v[2];
  const double tau = rsqrt(H.dt2 + vGv);
  const int64_t o = (int64_t)(4 + P.N + 6 * solid) * nn + l.n;
  double B[6], cv[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const VG<double> r = l.vg(H.xa[o + c * nn]);
    B[c] = r.v;
    cv[c] = v[0] * r.gx + v[1] * r.gy + v[2] * r.gz + l.val(H.xd[o + c * nn]);
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int k = sym_k(c), m = sym_l(c);
    double st = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) st += L[k][i] * B[sym_idx(i, m)] + B[sym_idx(k, i)] * L[m][i];
    const double R = H.W * (al * (cv[c] - st) + (1.0 - al) * (B[c] - (c < 3 ? 1.0 : 0.0)));
    const double t = tau * R;
    const double s = l.scatter(R, t * v[0], t * v[1], t * v[2]);
    if (l.ok) E[(8 * c + l.q) * es + at] = s;
  }
}

// Quadrature-point coefficients of the momentum/continuity product (ops.cuh lists them) in
// float64, C[((ez * 8 + q) * NCQ + c) * nxyp + ey * nxp + ex], and/or rounded to float32 in the tiles of
// the float32 product, C[(((ez * tiles + f / 128) * 8 + q) * NCQ + c) * 128 + f % 128], f = ey * nx + ex.  64^3, one
// solid: 3.36 -> 1.17 ms against the tile build, all solids in one pass.
template <bool MANY>
__global__ void __launch_bounds__(HQ_THREADS) hq_ns_coef_kernel(const __grid_constant__ HexNS H, double* __restrict__ c64,
                                                                float* __restrict__ c32, unsigned ne, int elastic) {
  HexLane l;
  l.set(H.g, H.rh, 0, ne);
  NSPoint p;
  hq_ns_point(H, l, p);
  const int64_t b = ((int64_t)l.ez * 8 + l.q) * NCQ * H.nxyp + (int64_t)l.ey * H.nxp + l.ex;
  const unsigned f = (unsigned)l.ey * (unsigned)H.g.nx + (unsigned)l.ex;
  const int64_t b32 = (((int64_t)l.ez * nsq_tiles(H.g) + f / NSQ_TILE) * 8 + l.q) * NCQ * NSQ_TILE + f % NSQ_TILE;
  auto put = [&](int c, double v) {
    if (!l.ok) return;
    if (c64) c64[b + c * H.nxyp] = v;
    if (c32) c32[b32 + c * NSQ_TILE] = (float)v;
  };
  put(0, p.rho);
  put(1, p.mu);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    put(2 + k, p.v[k]);
#pragma unroll
    for (int j = 0; j < 3; ++j) put(5 + 3 * k + j, p.L[k][j]);
    put(14 + k, p.R[k]);
  }
  put(17, p.tau_m);
  put(18, p.tau_c * p.rho);
  put(19, p.tau_m * p.rrho);
  if (!elastic) return;  // (the products then read the first 20)
  double aB[6], aG[6][3];
  hq_elastic<MANY>(H, l, aB, aG);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    put(20 + c, aB[c]);
#pragma unroll
    for (int j = 0; j < 3; ++j) put(26 + 3 * c + j, aG[c][j]);
  }
}

// The product itself for a state that is used a few times: the point's coefficients stay in
// registers.  E as hq_ns_res_kernel.  A product at a new state with its coefficients stored before
// it: 61 x 47 x 35 with two solids 2.97 -> 1.02 ms, 256 x 128 x 64 with nine 216 -> 33 ms.
struct PointCoef {
  const NSPoint& p;
  const double (&aB)[6];
  const double (&aG)[6][3];
  __device__ __forceinline__ double operator()(int i) const {
    if (i == 0) return p.rho;
    if (i == 1) return p.mu;
    if (i < 5) return p.v[i - 2];
    if (i < 14) return p.L[(i - 5) / 3][(i - 5) % 3];
    if (i < 17) return p.R[i - 14];
    if (i == 17) return p.tau_m;
    if (i == 18) return p.tau_c * p.rho;
    if (i == 19) return p.tau_m * p.rrho;
    if (i < 26) return aB[i - 20];
    return aG[(i - 26) / 3][(i - 26) % 3];
  }
};

template <bool MANY>
__global__ void __launch_bounds__(HQ_THREADS) hq_ns_jvp_kernel(const __grid_constant__ HexNS H,
                                                               const double* __restrict__ dx, double* __restrict__ E,
                                                               unsigned e0, unsigned e1, int elastic) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const int64_t es = H.stride(), at = H.at(l);
  NSPoint p;
  hq_ns_point(H, l, p);
  double aB[6] = {}, aG[6][3] = {};
  if (elastic) hq_elastic<MANY>(H, l, aB, aG);
  double dv[3], gd[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const VG<double> r = l.vg(dx[k * H.nn + l.n]);
    dv[k] = r.v; gd[k][0] = r.gx; gd[k][1] = r.gy; gd[k][2] = r.gz;
  }
  const VG<double> d = l.vg(dx[3 * H.nn + l.n]);
  const double dgp[3] = {d.gx, d.gy, d.gz};
  double f[4], g[4][3];
  nsq_point_fg<double>(PointCoef{p, aB, aG}, elastic != 0, dv, gd, d.v, dgp, H.P.alpha, H.P.c_mass, f, g);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double c = l.scatter(f[k], g[k][0], g[k][1], g[k][2]);
    if (l.ok) E[(8 * k + l.q) * es + at] = c;
  }
}

// Allen-Cahn and B products at a state that is used a few times
__global__ void __launch_bounds__(HQ_THREADS) hq_ac_jvp_kernel(const __grid_constant__ HexNS H, int phase, double gam,
                                                               double bet, const double* __restrict__ dx,
                                                               double* __restrict__ E, unsigned e0, unsigned e1) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const Phys& P = H.P;
  double v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = l.val(H.xa[k * H.nn + l.n]);
  const double phi = l.val(H.xa[(4 + phase) * H.nn + l.n]);
  const VG<double> d = l.vg(dx[l.n]);
  const double k_hat = gam * P.eps * P.eps, s_hat = gam * (3.0 * phi * phi - 1.0);
  const double vGv = P.Gd[0] * v[0] * v[0] + P.Gd[1] * v[1] * v[1] + P.Gd[2] * v[2] * v[2];
  const double tau = rsqrt(H.dt2 + vGv + 9.0 * k_hat * k_hat * P.GG + s_hat * s_hat);
  const double p2 = phi * phi - 1.0;
  const double dsF = p2 > 0.0 ? phi : (p2 < 0.0 ? -phi : 0.0);
  const double rp = gam * (3.0 * phi * phi - 1.0 - bet * dsF);
  const double dR = P.c_mass * d.v + P.alpha * (v[0] * d.gx + v[1] * d.gy + v[2] * d.gz + rp * d.v);
  const double t = tau * dR, ka = k_hat * P.alpha;
  const double c = l.scatter(dR, ka * d.gx + t * v[0], ka * d.gy + t * v[1], ka * d.gz + t * v[2]);
  if (l.ok) E[l.q * H.stride() + H.at(l)] = H.W * c;
}

__global__ void __launch_bounds__(HQ_THREADS) hq_b_jvp_kernel(const __grid_constant__ HexNS H, int solid,
                                                              const double* __restrict__ dx, double* __restrict__ E,
                                                              unsigned e0, unsigned e1) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const Phys& P = H.P;
  const int64_t nn = H.nn, es = H.stride(), at = H.at(l);
  double v[3], L[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const VG<double> r = l.vg(H.xa[k * nn + l.n]);
    v[k] = r.v; L[k][0] = r.gx; L[k][1] = r.gy; L[k][2] = r.gz;
  }
  const double al = l.val(H.mat[(2 + solid) * nn + l.n]);
  const double vGv = P.Gd[0] * v[0] * v[0] + P.Gd[1] * v[1] * v[1] + P.Gd[2] * v[2] * v[2];
  const double tau = rsqrt(H.dt2 + vGv);
  double B[6], cv[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const VG<double> r = l.vg(dx[c * nn + l.n]);
    B[c] = P.alpha * r.v;
    cv[c] = P.alpha * (v[0] * r.gx + v[1] * r.gy + v[2] * r.gz) + P.c_mass * r.v;
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int k = sym_k(c), m = sym_l(c);
    double st = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) st += L[k][i] * B[sym_idx(i, m)] + B[sym_idx(k, i)] * L[m][i];
    const double R = H.W * (al * (cv[c] - st) + (1.0 - al) * B[c]);
    const double t = tau * R;
    const double s = l.scatter(R, t * v[0], t * v[1], t * v[2]);
    if (l.ok) E[(8 * c + l.q) * es + at] = s;
  }
}

int ns_build(fsi_mesh* m, unsigned flags, bool f64) {
  const unsigned eflags = flags & FSI_ELASTIC_AUG;
  fsi_mesh::NSCoef& c = f64 ? m->cq64 : m->cq32;
  if (c.gen == m->stage_gen && c.flags == eflags && c.p) return FSI_OK;
  const int nxp = cq_pitch(m);
  const int64_t len = (int64_t)m->g.nz * 8 * NCQ * (f64 ? (int64_t)nxp * m->g.ny : (int64_t)nsq_tiles(m->g) * NSQ_TILE);
  if (c.len < len) {
    cudaFree(c.p);
    c.p = nullptr;
    c.len = 0;
    FSI_CUDA(cudaMalloc(&c.p, (f64 ? sizeof(double) : sizeof(float)) * (size_t)len));
    c.len = len;
  }
  const unsigned ne = (unsigned)m->g.nx * m->g.ny * m->g.nz;
  auto* kernel = m->ns >= HQ_MANY ? &hq_ns_coef_kernel<true> : &hq_ns_coef_kernel<false>;
  FSI_LAUNCH(m, P_NS_BUILD,
             kernel<<<hq_blocks(ne), HQ_THREADS, 0, m->stream>>>(
                 hex_ns(m, nxp), f64 ? static_cast<double*>(c.p) : nullptr, f64 ? nullptr : static_cast<float*>(c.p), ne,
                 eflags && m->ns > 0 ? 1 : 0));
  c.gen = m->stage_gen;
  c.flags = eflags;
  return FSI_OK;
}

// Runs launch(E, H, e0, e1, k0, k1) for every slab of layers: the contributions of the elements [e0, e1) into E, then
// the node planes [k0, k1) that they complete.  E is a ring of layers: the last one before a slab stays for
// the slab's first plane.
template <class F>
static int hq_slabs(fsi_mesh* m, F launch) {
  const Geom& g = m->g;
  const int nxp = cq_pitch(m);
  double* E = nullptr;
  HexNS H = hex_ns(m, nxp);
  if (int rc = elem_layers(m, (int64_t)nxp * g.ny, &E, &H.layers)) return rc;
  const int step = H.layers == g.nz ? g.nz : H.layers - 1;
  for (int z0 = 0; z0 < g.nz; z0 += step) {
    const int z1 = std::min(g.nz, z0 + step);
    if (int rc = launch(E, H, (unsigned)z0 * g.ny * g.nx, (unsigned)z1 * g.ny * g.nx, z0, z1 == g.nz ? z1 + 1 : z1))
      return rc;
  }
  return FSI_OK;
}

// Dirichlet rows: dx, less vD where given
static int hq_ns_sums(fsi_mesh* m, const double* E, const HexNS& H, int k0, int k1, const double* dx, const double* vD,
                      double* y) {
  const Geom& g = m->g;
  const RowLaunch nl = node_launch(g, k0, k1);
  auto* kernel = H.layers < g.nz ? &ns_node_kernel<double, true> : &ns_node_kernel<double, false>;
  FSI_LAUNCH(m, P_NODE_SUM, kernel<<<nl.grid, nl.block, 0, m->stream>>>(E, g.nx, g.ny, g.nz, H.nxp, H.nxyp, H.layers, k0, k1,
                                                                        m->nn, H.W, m->mask, m->pin_active, dx, nullptr, vD,
                                                                        y));
  return FSI_OK;
}

template <int NC>
static int hq_sums(fsi_mesh* m, const double* E, const HexNS& H, int k0, int k1, double* y) {
  const Geom& g = m->g;
  const RowLaunch nl = node_launch(g, k0, k1);
  auto* kernel = H.layers < g.nz ? &em_node_kernel<NC, true> : &em_node_kernel<NC, false>;
  FSI_LAUNCH(m, P_NODE_SUM, kernel<<<nl.grid, nl.block, 0, m->stream>>>(E, g.nx, g.ny, g.nz, H.nxp, H.nxyp, H.layers, k0, k1,
                                                                        m->nn, y));
  return FSI_OK;
}

int hq_ns_jvp(fsi_mesh* m, const double* dx, double* y, unsigned flags) {
  const double ne = (double)m->g.nx * m->g.ny * m->g.nz;
  const int elastic = (flags & FSI_ELASTIC_AUG) && m->ns > 0 ? 1 : 0;
  // algorithmic bytes: the nodal fields once, the contributions written and read, the product
  prof_bytes(m, P_NS_JVP64, ne * 256.0 + (double)m->nn * 8.0 * (13 + (elastic ? 7 * m->ns : 0)));
  prof_bytes(m, P_NODE_SUM, ne * 256.0 + (double)m->nn * 33.0);
  auto* kernel = m->ns >= HQ_MANY ? &hq_ns_jvp_kernel<true> : &hq_ns_jvp_kernel<false>;
  return hq_slabs(m, [&](double* E, const HexNS& H, unsigned e0, unsigned e1, int k0, int k1) -> int {
    FSI_LAUNCH(m, P_NS_JVP64, kernel<<<hq_blocks(e1 - e0), HQ_THREADS, 0, m->stream>>>(H, dx, E, e0, e1, elastic));
    return hq_ns_sums(m, E, H, k0, k1, dx, nullptr, y);
  });
}

int hq_jvp(fsi_mesh* m, const BlockInfo& b, const double* dx, double* y) {
  const double ne = (double)m->g.nx * m->g.ny * m->g.nz;
  prof_bytes(m, P_NODE_SUM, ne * 64 * b.nc + (double)m->nn * 8 * b.nc);
  prof_bytes(m, b.kind == 1 ? P_AC_JVP64 : P_B_JVP64, ne * 64 * b.nc + (double)m->nn * (b.kind == 1 ? 40.0 : 80.0));
  return hq_slabs(m, [&](double* E, const HexNS& H, unsigned e0, unsigned e1, int k0, int k1) -> int {
    if (b.kind == 1) {
      FSI_LAUNCH(m, P_AC_JVP64, hq_ac_jvp_kernel<<<hq_blocks(e1 - e0), HQ_THREADS, 0, m->stream>>>(
                                    H, b.index, m->gamma[b.index], m->beta[b.index], dx, E, e0, e1));
      return hq_sums<1>(m, E, H, k0, k1, y);
    }
    FSI_LAUNCH(m, P_B_JVP64,
               hq_b_jvp_kernel<<<hq_blocks(e1 - e0), HQ_THREADS, 0, m->stream>>>(H, b.index, dx, E, e0, e1));
    return hq_sums<6>(m, E, H, k0, k1, y);
  });
}

int hq_residual(fsi_mesh* m, const BlockInfo& b, double* r) {
  prof_bytes(m, P_NODE_SUM, (double)m->g.nx * m->g.ny * m->g.nz * 64 * b.nc + (double)m->nn * 8 * b.nc);
  return hq_slabs(m, [&](double* E, const HexNS& H, unsigned e0, unsigned e1, int k0, int k1) -> int {
    const unsigned grid = hq_blocks(e1 - e0);
    if (b.kind == 0) {
      FSI_LAUNCH(m, P_NS_RES, hq_ns_res_kernel<<<grid, HQ_THREADS, 0, m->stream>>>(H, E, e0, e1));
      return hq_ns_sums(m, E, H, k0, k1, m->staged_x, m->vD, r);
    }
    if (b.kind == 1) {
      FSI_LAUNCH(m, P_AC_RES, hq_ac_res_kernel<<<grid, HQ_THREADS, 0, m->stream>>>(H, b.index, m->gamma[b.index],
                                                                                  m->beta[b.index], E, e0, e1));
      return hq_sums<1>(m, E, H, k0, k1, r);
    }
    FSI_LAUNCH(m, P_B_RES, hq_b_res_kernel<<<grid, HQ_THREADS, 0, m->stream>>>(H, b.index, E, e0, e1));
    return hq_sums<6>(m, E, H, k0, k1, r);
  });
}

// ------------------------------------------------------------------ gamma, beta
// Sections 2.2.1 and 2.2.2 as CoefOp (ops.cuh) has them: the corner contributions of the lumped
// projection of q = grad phi^T grad v grad phi / |grad phi|^2, unweighted (its denominator is W times
// the node's elements), and the CTA's partial integrals of F' and sqrt F over its elements, added to those
// of the slabs before.
__global__ void __launch_bounds__(HQ_THREADS) hq_coef_kernel(const __grid_constant__ HexNS H, int phase,
                                                             double* __restrict__ E, double* __restrict__ part, unsigned e0,
                                                             unsigned e1) {
  const double* phi = H.xa + (int64_t)(4 + phase) * H.nn;
  const int64_t es = H.stride(), nt = (int64_t)(e1 - e0) * 8;
  double sF = 0.0, sS = 0.0;
  // whole warps stay in the loop together (32 lanes: four elements)
  for (int64_t t = (int64_t)blockIdx.x * HQ_THREADS + threadIdx.x; t - (threadIdx.x & 31) < nt;
       t += (int64_t)gridDim.x * HQ_THREADS) {
    HexLane l;
    l.set(H.g, H.rh, e0, e1, t);
    const VG<double> ph = l.vg(phi[l.n]);
    const double g[3] = {ph.gx, ph.gy, ph.gz};
    double num = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const VG<double> r = l.vg(H.xa[j * H.nn + l.n]);
      num = fma(g[j], r.gx * g[0] + r.gy * g[1] + r.gz * g[2], num);
    }
    const double n2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
    const double c = l.val(n2 < 1e-30 ? 0.0 : num / n2);
    if (l.ok) {
      E[l.q * es + H.at(l)] = c;
      sF += ph.v * ph.v * ph.v - ph.v;
      sS += 0.5 * fabs(ph.v * ph.v - 1.0);
    }
  }
  __shared__ double red[2][HQ_THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sF += __shfl_down_sync(0xffffffffu, sF, o);
    sS += __shfl_down_sync(0xffffffffu, sS, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = sF;
    red[1][threadIdx.x >> 5] = sS;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int i = 0; i < HQ_THREADS / 32; ++i) s += red[threadIdx.x][i];
    double* p = part + 2 * blockIdx.x + threadIdx.x;
    *p = e0 > 0 ? *p + H.W * s : H.W * s;
  }
}

// the CTA's partial sum of squared nodal values and count of nodes in the band |phi| <= 0.9, over the nodes
// [n0, n1) and added to those before
__global__ void __launch_bounds__(NTHREADS) hq_coef_node_kernel(const double* __restrict__ E, int nx, int ny, int nz, int nxp,
                                                                int64_t nxyp, int layers, int64_t n0, int64_t n1,
                                                                const double* __restrict__ phi, double* __restrict__ part) {
  __shared__ double scratch[NTHREADS / 32];
  const int64_t es = (int64_t)layers * nxyp;
  double v2 = 0.0, cnt = 0.0;
  for (int64_t n = n0 + (int64_t)blockIdx.x * NTHREADS + threadIdx.x; n < n1; n += (int64_t)gridDim.x * NTHREADS) {
    if (!(fabs(phi[n]) <= 0.9)) continue;
    const unsigned row = (unsigned)n / (unsigned)(nx + 1);
    const int i = (int)((unsigned)n - row * (unsigned)(nx + 1)), k = (int)(row / (unsigned)(ny + 1));
    const int j = (int)(row - (unsigned)k * (unsigned)(ny + 1));
    double s = 0.0, elems = 0.0;
    for (int az = 1; az >= 0; --az)
      for (int ay = 1; ay >= 0; --ay)
        for (int ax = 1; ax >= 0; --ax) {
          const int ex = i - ax, ey = j - ay, ez = k - az;
          if (ex < 0 || ex >= nx || ey < 0 || ey >= ny || ez < 0 || ez >= nz) continue;
          s += E[(ax + 2 * ay + 4 * az) * es + (int64_t)(ez < layers ? ez : ez % layers) * nxyp + (int64_t)ey * nxp + ex];
          elems += 1.0;
        }
    const double v = fabs(s / elems);
    v2 += v * v;
    cnt += 1.0;
  }
  const double a = block_sum(v2, scratch);
  const double b = block_sum(cnt, scratch);
  if (threadIdx.x == 0) {
    double* p = part + 2 * blockIdx.x;
    p[0] = n0 > 0 ? p[0] + a : a;
    p[1] = n0 > 0 ? p[1] + b : b;
  }
}

// out = {gamma, beta} from the partials of ne element and nn node CTAs, summed in a fixed order
__global__ void __launch_bounds__(NTHREADS) hq_coef_final_kernel(const double* __restrict__ pe, int ne,
                                                                 const double* __restrict__ pn, int nn, double eta,
                                                                 double* __restrict__ out) {
  __shared__ double scratch[NTHREADS / 32];
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < nn; i += NTHREADS) {
    a[0] += pn[2 * i];
    a[1] += pn[2 * i + 1];
  }
  for (int i = threadIdx.x; i < ne; i += NTHREADS) {
    a[2] += pe[2 * i];
    a[3] += pe[2 * i + 1];
  }
  double s[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) s[c] = block_sum(a[c], scratch);
  if (threadIdx.x == 0) {
    out[0] = s[1] > 0.0 ? sqrt(s[0] / s[1]) / eta : 0.0;
    out[1] = s[3] != 0.0 ? s[2] / s[3] : 0.0;
  }
}

int op_coeffs(fsi_mesh* m, int phase, double* gb) {
  if (m->tet) return tet_coeffs(m, phase, gb);
  const Geom& g = m->g;
  const unsigned ne = (unsigned)g.nx * g.ny * g.nz;
  const int ge = (int)std::min<unsigned>(hq_blocks(ne), 152 * 8), gn = (int)std::min<int64_t>((m->nn + NTHREADS - 1) / NTHREADS, 152 * 4);
  if (m->n_partials < ge + gn) {
    cudaFree(m->partials);
    m->partials = nullptr;
    m->n_partials = 0;
    FSI_CUDA(cudaMalloc(&m->partials, sizeof(double) * 4 * (ge + gn)));
    m->n_partials = ge + gn;
  }
  double* pn = m->partials + 2 * ge;
  const double* phi = m->staged_xa + (int64_t)(4 + phase) * m->nn;
  const int64_t plane = (int64_t)(g.nx + 1) * (g.ny + 1);
  const int rc = hq_slabs(m, [&](double* E, const HexNS& H, unsigned e0, unsigned e1, int k0, int k1) -> int {
    FSI_LAUNCH(m, P_COEF, hq_coef_kernel<<<ge, HQ_THREADS, 0, m->stream>>>(H, phase, E, m->partials, e0, e1));
    FSI_LAUNCH(m, P_COEF, hq_coef_node_kernel<<<gn, NTHREADS, 0, m->stream>>>(E, g.nx, g.ny, g.nz, H.nxp, H.nxyp, H.layers,
                                                                             k0 * plane, k1 * plane, phi, pn));
    return FSI_OK;
  });
  if (rc) return rc;
  FSI_LAUNCH(m, P_COEF, hq_coef_final_kernel<<<1, NTHREADS, 0, m->stream>>>(m->partials, ge, pn, gn, m->P.eta, m->red));
  FSI_CUDA(cudaMemcpyAsync(m->red_host, m->red, 2 * sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  FSI_CUDA(cudaStreamSynchronize(m->stream));
  gb[0] = m->red_host[0];
  gb[1] = m->red_host[1];
  return FSI_OK;
}

}  // namespace fsi
