// Assembled float64 Allen-Cahn and B operators: scalar 27-neighbour stencils.
//
// As for the momentum block (nsa.cu) the float64 FMA rate binds a product, so the operators are
// summed into node rows once per solve: 27 FMAs a node for an indicator (64 an element before, in
// element matrices) and 648 for a solid's six components (1,440 an element before).  One product:
// Allen-Cahn 96 x 96 x 192 102 us (0.77 of the float64 FMA rate) against 517 with the node sums, B 64^3
// 323 us (0.88 of it) against 929.  Builds: Allen-Cahn 5.0 ms against 19.3 (and 9.2 for the
// diagonal, 15 for the two products before it), B 3.5 ms against 2.0 (and 2.5 for the diagonal).
//
// Allen-Cahn (Eq. PPV_AC's linearization, gamma, beta and tau_phi frozen): with
//   T_a = N_a + tau v.grad N_a,  R_b = (c_m + alpha gamma (3 phi^2 - 1 - beta dsqrtF)) N_b + alpha v.grad N_b
// the element matrix is sum_q W (T_a R_b + alpha gamma eps^2 grad N_a . grad N_b).
//
// B (Eq. semiCGT's linearization): the six components share a scalar operator S (mass, convection
// and recovery) and are coupled by the stretching terms, which are linear in L = grad v:
//   y_c = S dB_c - sum_m (R_km dB_ml + R_lm dB_km),  c = (k, l),
//   S_ab = sum_q W T_a (al (c_m N_b + alpha v.grad N_b) + (1 - al) alpha N_b),
//   R_km,ab = sum_q W T_a al alpha L_km N_b,   T_a = N_a + tau_B v.grad N_a.
// Stored per neighbour: the diagonal entries S - 2 R_kk (kk), S - R_kk - R_ll (kl) and R_km, k != m.
//
// Layout: tiles of 128 nodes, A[((tile * 27 + o) * NV + value) * 128 + lane], o as in nsa.cu.
#include "hexq.cuh"
#include "ops_impl.cuh"

namespace fsi {

constexpr int ST = 128;

// T and R of the lane's point q for its corners in the order x = corner ^ q: the weights are then constants
// of x and the gradients' signs the lane's own (vr_j = v_j / h_j, signed for the lane's side), and what
// another lane needs of them sits in a register known at compile time.
//   T = W (N + tau v.grad N),   R = mass N + conv v.grad N
__device__ __forceinline__ void test_trial(const HexLane& l, const double (&v)[3], double W, double tau, double mass,
                                           double conv, double (&T)[8], double (&R)[8]) {
  // the lane's own corner lies on the side of its sign: d_j N at the corner q is -sx rhx ... in HexLane's
  // signs (sx turns partner - own into the derivative)
  const double vx = -l.sx * v[0], vy = -l.sy * v[1], vz = -l.sz * v[2];
  const double Wt = W * tau;
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const double wx = (x & 1) ? FSI_G1 : FSI_G0, wy = (x & 2) ? FSI_G1 : FSI_G0, wz = (x & 4) ? FSI_G1 : FSI_G0;
    const double vg = fma((x & 1) ? -wy * wz : wy * wz, vx,
                          fma((x & 2) ? -wx * wz : wx * wz, vy, ((x & 4) ? -wx * wy : wx * wy) * vz));
    T[x] = fma(Wt, vg, W * (wx * wy * wz));
    R[x] = fma(conv, vg, mass * (wx * wy * wz));
  }
}

// M[z] += sum_q T_a(q) R_b(q) for column b = lane and row a = lane ^ z, from all eight points q = lane ^ y
__device__ __forceinline__ void outer_sum(const double (&T)[8], const double (&R)[8], double (&M)[8]) {
#pragma unroll
  for (int y = 0; y < 8; ++y) {
    const double r = hq_shx(R[y], y);
#pragma unroll
    for (int z = 0; z < 8; ++z) M[z] = fma(hq_shx(T[z ^ y], y), r, M[z]);
  }
}

// Element matrices of the layers from e0: K[((ez % slots) * 64 + 8 a + b) * nxyp + ey * nxp + ex].  The
// diffusion part depends on a ^ b alone and is the same for every element (D, from the host).
struct Diffusion {
  double d[8];
};
__global__ void __launch_bounds__(HQ_THREADS) ac_elem_kernel(const __grid_constant__ HexNS H, int phase, double gam,
                                                             double bet, const __grid_constant__ Diffusion D,
                                                             double* __restrict__ K, unsigned e0, unsigned e1, int slots) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const Phys& P = H.P;
  double v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = l.val(H.xa[k * H.nn + l.n]);
  const double phi = l.val(H.xa[(4 + phase) * H.nn + l.n]);
  const double k_hat = gam * P.eps * P.eps, s_hat = gam * (3.0 * phi * phi - 1.0);
  const double vGv = P.Gd[0] * v[0] * v[0] + P.Gd[1] * v[1] * v[1] + P.Gd[2] * v[2] * v[2];
  const double tau = rsqrt(H.dt2 + vGv + 9.0 * k_hat * k_hat * P.GG + s_hat * s_hat);
  const double p2 = phi * phi - 1.0;
  const double dsF = p2 > 0.0 ? phi : (p2 < 0.0 ? -phi : 0.0);
  const double mass = P.c_mass + P.alpha * gam * (3.0 * phi * phi - 1.0 - bet * dsF);
  double T[8], R[8], M[8];
  test_trial(l, v, H.W, tau, mass, P.alpha, T, R);
#pragma unroll
  for (int z = 0; z < 8; ++z) M[z] = D.d[z];
  outer_sum(T, R, M);
  if (!l.ok) return;
  double* out = K + ((int64_t)(l.ez % slots) * 64 + l.q) * H.nxyp + (int64_t)l.ey * H.nxp + l.ex;
#pragma unroll
  for (int z = 0; z < 8; ++z) out[(int64_t)(8 * (l.q ^ z)) * H.nxyp] = M[z];
}

// Ten element matrices of a solid (S, then R_km row-major): layer slots of 640 planes.
__global__ void __launch_bounds__(HQ_THREADS) b_elem_kernel(const __grid_constant__ HexNS H, int solid,
                                                            double* __restrict__ K, unsigned e0, unsigned e1, int slots) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  const Phys& P = H.P;
  const int64_t nn = H.nn;
  double v[3], L[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const VG<double> r = l.vg(H.xa[k * nn + l.n]);
    v[k] = r.v; L[k][0] = r.gx; L[k][1] = r.gy; L[k][2] = r.gz;
  }
  const double al = l.val(H.mat[(2 + solid) * nn + l.n]);
  const double vGv = P.Gd[0] * v[0] * v[0] + P.Gd[1] * v[1] * v[1] + P.Gd[2] * v[2] * v[2];
  const double tau = rsqrt(H.dt2 + vGv);
  const double conv = al * P.alpha;
  double T[8], M[8];
  {
    double R[8];
    test_trial(l, v, H.W, tau, al * P.c_mass + (1.0 - al) * P.alpha, conv, T, R);
#pragma unroll
    for (int z = 0; z < 8; ++z) M[z] = 0.0;
    outer_sum(T, R, M);
  }
  double* out = K + ((int64_t)(l.ez % slots) * 640 + l.q) * H.nxyp + (int64_t)l.ey * H.nxp + l.ex;
  if (l.ok) {
#pragma unroll
    for (int z = 0; z < 8; ++z) out[(int64_t)(8 * (l.q ^ z)) * H.nxyp] = M[z];
  }
  // R_km: the trial side is N_b alone, so the sum over the points is the transposed interpolation: per
  // axis G0 own + G1 of the lane across it, whose row a sits one register bit away
#pragma unroll
  for (int km = 0; km < 9; ++km) {
    const double c = conv * L[km / 3][km % 3];
    double f[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) f[x] = T[x] * c;
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
      double p[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) p[x] = hq_shx(f[x ^ d], d);
#pragma unroll
      for (int x = 0; x < 8; ++x) f[x] = fma(FSI_G1, p[x] - f[x], f[x]);
    }
    if (l.ok) {
#pragma unroll
      for (int z = 0; z < 8; ++z) out[(int64_t)(64 * (km + 1) + 8 * (l.q ^ z)) * H.nxyp] = f[z];
    }
  }
}

// Node rows of NM element matrices (of nk planes per layer slot) on the planes from n0: the sums over
// the up to 8 elements of a node pair, in a fixed order (z, y, x of the element)
template <int NM>
__device__ __forceinline__ void stencil_row(const double* __restrict__ K, int nx, int ny, int nz, int nxp, int64_t nxyp,
                                            int slots, int nk, int i, int j, int k, int dx, int dy, int dz,
                                            double (&acc)[NM]) {
#pragma unroll
  for (int q = 0; q < NM; ++q) acc[q] = 0.0;
  for (int az = dz < 0 ? 1 : 0; az <= (dz > 0 ? 0 : 1); ++az) {
    const int ez = k - az;
    if (ez < 0 || ez >= nz) continue;
    for (int ay = dy < 0 ? 1 : 0; ay <= (dy > 0 ? 0 : 1); ++ay) {
      const int ey = j - ay;
      if (ey < 0 || ey >= ny) continue;
      for (int ax = dx < 0 ? 1 : 0; ax <= (dx > 0 ? 0 : 1); ++ax) {
        const int ex = i - ax;
        if (ex < 0 || ex >= nx) continue;
        const int a = ax + 2 * ay + 4 * az, b = a + dx + 2 * dy + 4 * dz;
        const double* src = K + ((int64_t)(ez % slots) * nk + 8 * a + b) * nxyp + (int64_t)ey * nxp + ex;
#pragma unroll
        for (int q = 0; q < NM; ++q) acc[q] += src[(int64_t)(64 * q) * nxyp];
      }
    }
  }
}

struct NodeIdx {
  int i, j, k;
  __device__ __forceinline__ NodeIdx(int64_t n, int nx, int ny) {
    const unsigned row = (unsigned)n / (unsigned)(nx + 1);
    i = (int)((unsigned)n - row * (unsigned)(nx + 1));
    k = (int)(row / (unsigned)(ny + 1));
    j = (int)(row - (unsigned)k * (unsigned)(ny + 1));
  }
};

// one thread per (node, neighbour): blockIdx.y = o
template <bool B>
__global__ void __launch_bounds__(ST) stencil_gather_kernel(const double* __restrict__ K, int nx, int ny, int nz, int nxp,
                                                            int64_t nxyp, int slots, int64_t n0, int64_t n1,
                                                            double* __restrict__ A) {
  const int64_t n = n0 + (int64_t)blockIdx.x * ST + threadIdx.x;
  if (n >= n1) return;
  const NodeIdx p(n, nx, ny);
  const int o = blockIdx.y, dx = o % 3 - 1, dy = o / 3 % 3 - 1, dz = o / 9 - 1;
  if constexpr (B) {
    double r[10];
    stencil_row<10>(K, nx, ny, nz, nxp, nxyp, slots, 640, p.i, p.j, p.k, dx, dy, dz, r);
    double* out = A + ((n / ST * 27 + o) * 12) * ST + n % ST;
    const double d0 = r[1], d1 = r[5], d2 = r[9];
    out[0 * ST] = r[0] - 2.0 * d0;
    out[1 * ST] = r[0] - 2.0 * d1;
    out[2 * ST] = r[0] - 2.0 * d2;
    out[3 * ST] = r[0] - (d0 + d1);
    out[4 * ST] = r[0] - (d1 + d2);
    out[5 * ST] = r[0] - (d0 + d2);
    out[6 * ST] = r[2];   // R_01
    out[7 * ST] = r[3];   // R_02
    out[8 * ST] = r[4];   // R_10
    out[9 * ST] = r[6];   // R_12
    out[10 * ST] = r[7];  // R_20
    out[11 * ST] = r[8];  // R_21
  } else {
    double r[1];
    stencil_row<1>(K, nx, ny, nz, nxp, nxyp, slots, 64, p.i, p.j, p.k, dx, dy, dz, r);
    A[(n / ST * 27 + o) * ST + n % ST] = r[0];
  }
}

__global__ void __launch_bounds__(ST) ac_apply_kernel(const double* __restrict__ A, const double* __restrict__ x, int nx,
                                                      int ny, int nz, int64_t nn, double* __restrict__ y) {
  const int64_t n = (int64_t)blockIdx.x * ST + threadIdx.x;
  if (n >= nn) return;
  const NodeIdx p(n, nx, ny);
  const int64_t sy = nx + 1, sz = sy * (ny + 1);
  const double* a = A + (int64_t)blockIdx.x * 27 * ST + threadIdx.x;
  double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz) {
    const bool okz = p.k + dz >= 0 && p.k + dz <= nz;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const bool okyz = okz && p.j + dy >= 0 && p.j + dy <= ny;
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        // a missing neighbour's entry is zero and its value is read at the node itself
        const bool ok = okyz && p.i + dx >= 0 && p.i + dx <= nx;
        const int64_t nb = ok ? n + dx + sy * dy + sz * dz : n;
        acc[dx + 1] += __ldcs(a + ((dx + 1) + 3 * (dy + 1) + 9 * (dz + 1)) * ST) * __ldg(x + nb);
      }
    }
  }
  y[n] = acc[0] + acc[1] + acc[2];
}

__global__ void __launch_bounds__(ST) b_apply_kernel(const double* __restrict__ A, const double* __restrict__ x, int nx,
                                                     int ny, int nz, int64_t nn, double* __restrict__ y) {
  const int64_t n = (int64_t)blockIdx.x * ST + threadIdx.x;
  if (n >= nn) return;
  const NodeIdx p(n, nx, ny);
  const int64_t sy = nx + 1, sz = sy * (ny + 1);
  const double* a = A + (int64_t)blockIdx.x * 27 * 12 * ST + threadIdx.x;
  double d[6] = {}, s[6] = {};  // diagonal products, stretching sums (halved for kk)
#pragma unroll 1
  for (int dz = -1; dz <= 1; ++dz) {
    const bool okz = p.k + dz >= 0 && p.k + dz <= nz;
#pragma unroll 1
    for (int dy = -1; dy <= 1; ++dy) {
      const bool okyz = okz && p.j + dy >= 0 && p.j + dy <= ny;
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const bool ok = okyz && p.i + dx >= 0 && p.i + dx <= nx;
        const int64_t nb = ok ? n + dx + sy * dy + sz * dz : n;
        const double* ao = a + ((dx + 1) + 3 * (dy + 1) + 9 * (dz + 1)) * 12 * ST;
        double c[12], u[6];
#pragma unroll
        for (int q = 0; q < 12; ++q) c[q] = __ldcs(ao + q * ST);
#pragma unroll
        for (int q = 0; q < 6; ++q) u[q] = __ldg(x + q * nn + nb);
#pragma unroll
        for (int q = 0; q < 6; ++q) d[q] = fma(c[q], u[q], d[q]);
        // u: 11, 22, 33, 12, 23, 13; c[6..]: R_12, R_13, R_21, R_23, R_31, R_32
        s[0] = fma(c[6], u[3], fma(c[7], u[5], s[0]));
        s[1] = fma(c[8], u[3], fma(c[9], u[4], s[1]));
        s[2] = fma(c[10], u[5], fma(c[11], u[4], s[2]));
        s[3] = fma(c[6], u[1], fma(c[7], u[4], fma(c[8], u[0], fma(c[9], u[5], s[3]))));
        s[4] = fma(c[9], u[2], fma(c[8], u[5], fma(c[11], u[1], fma(c[10], u[3], s[4]))));
        s[5] = fma(c[7], u[2], fma(c[6], u[4], fma(c[10], u[0], fma(c[11], u[3], s[5]))));
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) y[q * nn + n] = d[q] - (q < 3 ? 2.0 * s[q] : s[q]);
}

// the diagonal: value v of the node's own entry for component c
__global__ void stencil_diag_kernel(const double* __restrict__ A, int nv, int nc, int64_t nn, double* __restrict__ d) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  for (int c = 0; c < nc; ++c) d[c * nn + n] = A[((n / ST * 27 + 13) * nv + c) * ST + n % ST];
}

// Element matrices are summed a slab of layers at a time (see nsa_build); small slabs stay in L2
constexpr int64_t STENCIL_SLAB_BYTES = (int64_t)256 << 20;

int stencil_build(fsi_mesh* m, const BlockInfo& b) {
  const bool B = b.kind == 2;
  fsi_mesh::Stencil& S = B ? m->bst : m->acst;
  const double gam = B ? 0.0 : m->gamma[b.index], bet = B ? 0.0 : m->beta[b.index];
  if (S.built && S.gen == m->stage_gen && S.index == b.index && S.gamma == gam && S.beta == bet) return FSI_OK;
  S.built = 0;
  const Geom& g = m->g;
  const int nxp = cq_pitch(m), nk = B ? 640 : 64, nv = B ? 12 : 1;
  const int64_t nxyp = (int64_t)nxp * g.ny, layer = nk * nxyp;
  const int64_t len = (m->nn + ST - 1) / ST * ST * 27 * nv;
  if (S.len < len) {
    cudaFree(S.A);
    S.A = nullptr;
    S.len = 0;
    FSI_CUDA(cudaMalloc(&S.A, sizeof(double) * (size_t)len));
    S.len = len;
  }
  const int slots = (int)std::min<int64_t>(g.nz, std::max<int64_t>(2, STENCIL_SLAB_BYTES / (8 * layer)));
  if (int rc = ensure_elem_matrices(m, slots * layer)) return rc;
  const HexNS H = hex_ns(m, nxp);
  const int64_t plane = (int64_t)(g.nx + 1) * (g.ny + 1);
  const int step = slots == g.nz ? g.nz : slots - 1;
  // alpha gamma eps^2 grad N_a . grad N_b over an element, by a ^ b: 1D factors 1/3 (same side) and 1/6
  Diffusion D;
  for (int x = 0; x < 8; ++x) {
    double s = 0.0;
    for (int j = 0; j < 3; ++j) {
      double t = ((x >> j) & 1) ? -H.rh[j] * H.rh[j] : H.rh[j] * H.rh[j];
      for (int i = 0; i < 3; ++i)
        if (i != j) t *= ((x >> i) & 1) ? 1.0 / 6.0 : 1.0 / 3.0;
      s += t;
    }
    D.d[x] = 8.0 * H.W * gam * m->P.eps * m->P.eps * m->P.alpha * s;
  }
  for (int z0 = 0; z0 < g.nz; z0 += step) {
    const int z1 = std::min(g.nz, z0 + step);
    const unsigned e0 = (unsigned)z0 * g.ny * g.nx, e1 = (unsigned)z1 * g.ny * g.nx;
    const int64_t n0 = z0 * plane, n1 = (z1 == g.nz ? z1 + 1 : z1) * plane;
    const dim3 grid((unsigned)((n1 - n0 + ST - 1) / ST), 27);
    if (B) {
      FSI_LAUNCH(m, P_NS_BUILD, b_elem_kernel<<<hq_blocks(e1 - e0), HQ_THREADS, 0, m->stream>>>(H, b.index, m->ke64, e0, e1,
                                                                                                slots));
      FSI_LAUNCH(m, P_NS_BUILD, stencil_gather_kernel<true><<<grid, ST, 0, m->stream>>>(
                                    m->ke64, g.nx, g.ny, g.nz, nxp, nxyp, slots, n0, n1, S.A));
    } else {
      FSI_LAUNCH(m, P_NS_BUILD, ac_elem_kernel<<<hq_blocks(e1 - e0), HQ_THREADS, 0, m->stream>>>(
                                    H, b.index, gam, bet, D, m->ke64, e0, e1, slots));
      FSI_LAUNCH(m, P_NS_BUILD, stencil_gather_kernel<false><<<grid, ST, 0, m->stream>>>(
                                    m->ke64, g.nx, g.ny, g.nz, nxp, nxyp, slots, n0, n1, S.A));
    }
  }
  S.gen = m->stage_gen;
  S.index = b.index;
  S.gamma = gam;
  S.beta = bet;
  S.built = 1;
  return FSI_OK;
}

int stencil_jvp(fsi_mesh* m, const BlockInfo& b, const double* dx, double* y) {
  if (int rc = stencil_build(m, b)) return rc;
  const Geom& g = m->g;
  const unsigned grid = (unsigned)((m->nn + ST - 1) / ST);
  // algorithmic bytes: the stencil once, the increment in and the product out
  if (b.kind == 2) {
    prof_bytes(m, P_B_JVP64, (double)m->nn * 8.0 * (27 * 12 + 12));
    FSI_LAUNCH(m, P_B_JVP64, b_apply_kernel<<<grid, ST, 0, m->stream>>>(m->bst.A, dx, g.nx, g.ny, g.nz, m->nn, y));
  } else {
    prof_bytes(m, P_AC_JVP64, (double)m->nn * 8.0 * (27 + 2));
    FSI_LAUNCH(m, P_AC_JVP64, ac_apply_kernel<<<grid, ST, 0, m->stream>>>(m->acst.A, dx, g.nx, g.ny, g.nz, m->nn, y));
  }
  return FSI_OK;
}

int stencil_diag(fsi_mesh* m, const BlockInfo& b, double* d) {
  if (int rc = stencil_build(m, b)) return rc;
  const bool B = b.kind == 2;
  FSI_LAUNCH(m, B ? P_B_DIAG : P_AC_DIAG,
             stencil_diag_kernel<<<(unsigned)((m->nn + 255) / 256), 256, 0, m->stream>>>(B ? m->bst.A : m->acst.A, B ? 12 : 1,
                                                                                         B ? 6 : 1, m->nn, d));
  return FSI_OK;
}

}  // namespace fsi
