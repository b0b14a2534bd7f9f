// Float64 instantiations of the element operators and the gamma/beta reduction.
#include "ops_impl.cuh"

namespace fsi {

template int launch_ns<double>(fsi_mesh*, int, const double*, double*, unsigned);

// Element-centric products of the Allen-Cahn element matrices and the B split operator:
// one thread per element (x fastest) gathers its increment values, applies the stored
// operator and writes its 8 (AC) or 48 (B) corner contributions into E[slot][element];
// em_node_kernel then sums, per node, the slots of its up to 8 elements in a fixed order
// (z, y, x).  Each element is evaluated once (no halo recomputation); deterministic.
// Allen-Cahn: c[b] = sum_a K[b][a] x[a]
__global__ void __launch_bounds__(128) ace_elem_kernel(const double* __restrict__ K, const double* __restrict__ dx,
                                                       double* __restrict__ E, int nx, int ny, int nz, int nxp,
                                                       int64_t nxyp) {
  ElemIdx I;
  if (!I.set(nx, ny, nz, nxp, nxyp)) return;
  double x[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) x[a] = __ldg(dx + I.n0 + I.off[a]);
  const double* k = K + (int64_t)I.ez * 64 * nxyp + (int64_t)I.ey * nxp + I.ex;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < 8; ++a) acc += __ldg(k + (int64_t)(b * 8 + a) * nxyp) * x[a];
    E[b * I.es + I.e] = acc;
  }
}

// B split operator of one solid: c[cc][a] = sum_b S[a][b] dB_cc[b]
//   - sum_q Ta_q[a] (L_q dB_q + dB_q L_q^T)_cc   (the stretching coupling at point q)
__global__ void __launch_bounds__(128) be_elem_kernel(const double* __restrict__ K, const double* __restrict__ dx,
                                                      double* __restrict__ E, int nx, int ny, int nz, int nxp,
                                                      int64_t nxyp, int64_t nn) {
  ElemIdx I;
  if (!I.set(nx, ny, nz, nxp, nxyp)) return;
  double x[6][8];
#pragma unroll
  for (int cc = 0; cc < 6; ++cc)
#pragma unroll
    for (int a = 0; a < 8; ++a) x[cc][a] = __ldg(dx + cc * nn + I.n0 + I.off[a]);
  const double* k = K + (int64_t)I.ez * NBK * nxyp + (int64_t)I.ey * nxp + I.ex;
  double c[6][8];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    double s[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) s[b] = __ldg(k + (int64_t)(a * 8 + b) * nxyp);
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) {
      double acc = 0.0;
#pragma unroll
      for (int b = 0; b < 8; ++b) acc += s[b] * x[cc][b];
      c[cc][a] = acc;
    }
  }
#pragma unroll 1
  for (int q = 0; q < 8; ++q) {
    QW<double> w;
    w.set(q);
    const double* kq = k + (int64_t)(64 + 17 * q) * nxyp;
    double dB[6];
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) dB[cc] = interp_v(x[cc], w);
    double L[3][3];
#pragma unroll
    for (int kk = 0; kk < 3; ++kk)
#pragma unroll
      for (int mm = 0; mm < 3; ++mm) L[kk][mm] = __ldg(kq + (int64_t)(8 + 3 * kk + mm) * nxyp);
    double st[6];
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) {
      const int kk = sym_k(cc), l = sym_l(cc);
      double t = 0.0;
#pragma unroll
      for (int mm = 0; mm < 3; ++mm) t += L[kk][mm] * dB[sym_idx(mm, l)] + dB[sym_idx(kk, mm)] * L[l][mm];
      st[cc] = t;
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const double ta = __ldg(kq + (int64_t)a * nxyp);
#pragma unroll
      for (int cc = 0; cc < 6; ++cc) c[cc][a] -= ta * st[cc];
    }
  }
#pragma unroll
  for (int cc = 0; cc < 6; ++cc)
#pragma unroll
    for (int a = 0; a < 8; ++a) E[(8 * cc + a) * I.es + I.e] = c[cc][a];
}

// E[slots][nz * nxyp] scratch of the element-centric products (NS, AC and B in turn)
int ensure_elem_scratch(fsi_mesh* m, int slots, int64_t nxyp) {
  const int64_t elen = (int64_t)slots * m->g.nz * nxyp;
  if (m->ke_e_len < elen) {
    cudaFree(m->ke_e);
    m->ke_e = nullptr;
    m->ke_e_len = 0;
    FSI_CUDA(cudaMalloc(&m->ke_e, sizeof(double) * (size_t)elen));
    m->ke_e_len = elen;
  }
  return FSI_OK;
}

int launch_ace(fsi_mesh* m, int phase, const double* dx, double* y) {
  const int nxp = cq_pitch(m);
  const int64_t nxyp = (int64_t)nxp * m->g.ny;
  const int64_t nn = m->nn;
  if (!m->ake_built) {
    const int64_t len = (int64_t)m->g.nz * 64 * nxyp;
    if (m->ake_len < len) {
      cudaFree(m->ake64);
      m->ake64 = nullptr;
      m->ake_len = 0;
      FSI_CUDA(cudaMalloc(&m->ake64, sizeof(double) * (size_t)len));
      m->ake_len = len;
    }
    ACEBuildOp b;
    memset(&b, 0, sizeof(b));
    const double* xa = m->staged_xa;
    for (int k = 0; k < 3; ++k) put<double>(b.F, k, xa + k * nn);
    put<double>(b.F, 3, xa + (4 + phase) * nn);
    b.nf = 4;
    b.P = m->P;
    fill_common(m, b.rh, &b.W);
    b.gamma = m->gamma[phase];
    b.beta = m->beta[phase];
    b.K = m->ake64;
    b.nxp = nxp;
    b.nxyp = nxyp;
    if (int rc = run_tile(m, b, P_NS_BUILD)) return rc;
    m->ake_built = 1;
  }
  if (int rc = ensure_elem_scratch(m, 8, nxyp)) return rc;
  const Geom& g = m->g;
  const int64_t ne = (int64_t)g.nx * g.ny * g.nz;
  prof_bytes(m, P_AC_JVP64, (double)ne * (64 * 8.0 + 8 * 8.0) + (double)nn * 8.0);
  prof_bytes(m, P_NODE_SUM, (double)ne * 8 * 8.0 + (double)nn * 8.0);
  const RowLaunch el = elem_launch(g), nl = node_launch(g);
  FSI_LAUNCH(m, P_AC_JVP64,
             ace_elem_kernel<<<el.grid, el.block, 0, m->stream>>>(m->ake64, dx, m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp));
  FSI_LAUNCH(m, P_NODE_SUM,
             em_node_kernel<1><<<nl.grid, nl.block, 0, m->stream>>>(m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp, nn, y));
  return FSI_OK;
}

int launch_be(fsi_mesh* m, int solid, const double* dx, double* y) {
  const int nxp = cq_pitch(m);
  const int64_t nxyp = (int64_t)nxp * m->g.ny;
  const int64_t nn = m->nn;
  if (!m->bke_built) {
    const int64_t len = (int64_t)m->g.nz * NBK * nxyp;
    if (m->bke_len < len) {
      cudaFree(m->bke64);
      m->bke64 = nullptr;
      m->bke_len = 0;
      FSI_CUDA(cudaMalloc(&m->bke64, sizeof(double) * (size_t)len));
      m->bke_len = len;
    }
    BEBuildOp b;
    memset(&b, 0, sizeof(b));
    const double* xa = m->staged_xa;
    for (int k = 0; k < 3; ++k) put<double>(b.F, k, xa + k * nn);
    put<double>(b.F, 3, m->mat + (2 + solid) * nn);
    b.nf = 4;
    b.P = m->P;
    fill_common(m, b.rh, &b.W);
    b.K = m->bke64;
    b.nxp = nxp;
    b.nxyp = nxyp;
    if (int rc = run_tile(m, b, P_NS_BUILD)) return rc;
    m->bke_built = 1;
  }
  if (int rc = ensure_elem_scratch(m, 48, nxyp)) return rc;
  const Geom& g = m->g;
  const int64_t ne = (int64_t)g.nx * g.ny * g.nz;
  prof_bytes(m, P_B_JVP64, (double)ne * (NBK * 8.0 + 48 * 8.0) + (double)nn * 48.0);
  prof_bytes(m, P_NODE_SUM, (double)ne * 48 * 8.0 + (double)nn * 48.0);
  const RowLaunch el = elem_launch(g), nl = node_launch(g);
  FSI_LAUNCH(m, P_B_JVP64,
             be_elem_kernel<<<el.grid, el.block, 0, m->stream>>>(m->bke64, dx, m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp,
                                                                nn));
  FSI_LAUNCH(m, P_NODE_SUM,
             em_node_kernel<6><<<nl.grid, nl.block, 0, m->stream>>>(m->ke_e, g.nx, g.ny, g.nz, nxp, nxyp, nn, y));
  return FSI_OK;
}

template int launch_ac<double>(fsi_mesh*, int, int, const double*, double*);
template int launch_b<double>(fsi_mesh*, int, int, const double*, double*);

// Sums the per-CTA partials {sum val^2, n_band, int F', int sqrt F} in a fixed order.
__global__ void coef_finalize(const double* partials, int64_t n, double eta, double* out) {
  __shared__ double s[4][NTHREADS];
  double a[4] = {0, 0, 0, 0};
  for (int64_t i = threadIdx.x; i < n; i += NTHREADS)
    for (int c = 0; c < 4; ++c) a[c] += partials[4 * i + c];
  for (int c = 0; c < 4; ++c) s[c][threadIdx.x] = a[c];
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[4] = {0, 0, 0, 0};
    for (int i = 0; i < NTHREADS; ++i)
      for (int c = 0; c < 4; ++c) t[c] += s[c][i];
    out[0] = t[1] > 0.0 ? sqrt(t[0] / t[1]) / eta : 0.0;  // gamma
    out[1] = t[3] != 0.0 ? t[2] / t[3] : 0.0;             // beta
  }
}

int op_coeffs(fsi_mesh* m, int i, double* gb) {
  static_assert(CoefOp::MINB == 1, "the partial sums are sized for the mesh's own tile grid");
  if (m->tet) return tet_coeffs(m, i, gb);
  CoefOp op;
  memset(&op, 0, sizeof(op));
  const int64_t nn = m->nn;
  for (int k = 0; k < 3; ++k) { op.F.d[k] = m->staged_xa + k * nn; op.F.f[k] = nullptr; }
  op.F.d[3] = m->staged_xa + (4 + i) * nn;
  op.nf = 4;
  fill_common(m, op.rh, &op.W);
  op.phi_node = m->staged_xa + (4 + i) * nn;
  dim3 grid;
  tile_grid(m, &grid);
  op.ncta_xy[0] = grid.x;
  op.ncta_xy[1] = grid.y;
  const int64_t ncta = (int64_t)grid.x * grid.y * grid.z;
  if (m->n_partials < ncta) {
    if (m->partials) cudaFree(m->partials);
    m->partials = nullptr;
    FSI_CUDA(cudaMalloc(&m->partials, sizeof(double) * 4 * ncta));
    m->n_partials = ncta;
  }
  op.partials = m->partials;
  int rc = run_tile(m, op, P_COEF);
  if (rc) return rc;
  FSI_LAUNCH(m, P_COEF, coef_finalize<<<1, NTHREADS, 0, m->stream>>>(m->partials, ncta, m->P.eta, m->red));
  FSI_CUDA(cudaMemcpyAsync(m->red_host, m->red, 2 * sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  FSI_CUDA(cudaStreamSynchronize(m->stream));
  gb[0] = m->red_host[0];
  gb[1] = m->red_host[1];
  return FSI_OK;
}

}  // namespace fsi
