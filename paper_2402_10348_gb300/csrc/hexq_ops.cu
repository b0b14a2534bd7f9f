// Residuals of the three kinds of block on hexahedra, one thread per (element, quadrature point)
// (hexq.cuh); ops.cuh has the equations.
#include "hexq.cuh"
#include "ops_impl.cuh"

namespace fsi {

// R_m, tau and the stresses at a point, tested: E[8 x equation + corner][element], unweighted
__global__ void __launch_bounds__(HQ_THREADS) hq_ns_res_kernel(const __grid_constant__ HexNS H, double* __restrict__ E,
                                                               unsigned ne) {
  HexLane l;
  l.set(H.g, H.rh, H.nxp, 0, ne);
  const int64_t es = (int64_t)H.g.nz * H.nxyp;
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
    if (l.ok) E[(8 * k + l.q) * es + l.e] = c;
  }
  const double r = p.tau_m * p.rrho;
  const double c = l.scatter(Rc, r * p.R[0], r * p.R[1], r * p.R[2]);
  if (l.ok) E[(24 + l.q) * es + l.e] = c;
}

__global__ void __launch_bounds__(HQ_THREADS) hq_ac_res_kernel(const __grid_constant__ HexNS H, int phase, double gam,
                                                               double bet, double* __restrict__ E, unsigned ne) {
  HexLane l;
  l.set(H.g, H.rh, H.nxp, 0, ne);
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
  if (l.ok) E[l.q * (int64_t)H.g.nz * H.nxyp + l.e] = H.W * c;
}

__global__ void __launch_bounds__(HQ_THREADS) hq_b_res_kernel(const __grid_constant__ HexNS H, int solid,
                                                              double* __restrict__ E, unsigned ne) {
  HexLane l;
  l.set(H.g, H.rh, H.nxp, 0, ne);
  const Phys& P = H.P;
  const int64_t nn = H.nn, es = (int64_t)H.g.nz * H.nxyp;
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
    if (l.ok) E[(8 * c + l.q) * es + l.e] = s;
  }
}

int hq_residual(fsi_mesh* m, const BlockInfo& b, double* r) {
  const Geom& g = m->g;
  const int nxp = cq_pitch(m);
  const int64_t nxyp = (int64_t)nxp * g.ny;
  const unsigned ne = (unsigned)g.nx * g.ny * g.nz;
  const int nc = b.kind == 0 ? 4 : b.kind == 1 ? 1 : 6;
  if (int rc = ensure_elem_scratch(m, 8 * nc, nxyp)) return rc;
  const HexNS H = hex_ns(m, nxp);
  const RowLaunch nl = node_launch(g);
  prof_bytes(m, P_NODE_SUM, (double)ne * 64 * nc + (double)m->nn * 8 * nc);
  if (b.kind == 0) {
    FSI_LAUNCH(m, P_NS_RES, hq_ns_res_kernel<<<hq_blocks(ne), HQ_THREADS, 0, m->stream>>>(H, m->ke_e, ne));
    FSI_LAUNCH(m, P_NODE_SUM,
               ns_node_kernel<double><<<nl.grid, nl.block, 0, m->stream>>>(m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp, m->nn, H.W,
                                                                           m->mask, m->pin_active, m->staged_x, nullptr,
                                                                           m->vD, r));
  } else if (b.kind == 1) {
    FSI_LAUNCH(m, P_AC_RES, hq_ac_res_kernel<<<hq_blocks(ne), HQ_THREADS, 0, m->stream>>>(
                                H, b.index, m->gamma[b.index], m->beta[b.index], m->ke_e, ne));
    FSI_LAUNCH(m, P_NODE_SUM,
               em_node_kernel<1><<<nl.grid, nl.block, 0, m->stream>>>(m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp, m->nn, r));
  } else {
    FSI_LAUNCH(m, P_B_RES, hq_b_res_kernel<<<hq_blocks(ne), HQ_THREADS, 0, m->stream>>>(H, b.index, m->ke_e, ne));
    FSI_LAUNCH(m, P_NODE_SUM,
               em_node_kernel<6><<<nl.grid, nl.block, 0, m->stream>>>(m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp, m->nn, r));
  }
  return FSI_OK;
}

}  // namespace fsi
