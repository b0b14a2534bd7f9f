// Assembled float64 momentum/continuity operator: 27 blocks of 4 x 4 per node.
//
// A solve applies the linearized operator hundreds of times on one state.  Float64 FMAs bind it
// (GB300 issues them at 1/64 of the float32 rate), so the form with the fewest is the fastest:
// 432 FMAs a node here, against 1024 an element for element matrices and about 2400 for the
// quadrature-point form, and no element contributions to write and sum.  Bytes: 3,456 a
// node, under the FMA time on this card.  64^3, one product: 221 us (0.86 of the float64 FMA rate
// of 0.628 T/s, 4.3 TB/s) against 586 us with element matrices and their node
// sums; 240 iterations of GMRES(30): 254.4 -> 118.6 ms with the build below.
//
// Layout: tiles of NAT = 128 nodes, A[((tile * 27 + o) * 16 + 4 r + c) * NAT + lane] for row
// (node, r) and column (neighbour o, c), o = (dx+1) + 3 (dy+1) + 9 (dz+1): a warp reads 32
// consecutive doubles and a CTA one contiguous 442 KB stretch.
#include <type_traits>

#include "hexq.cuh"
#include "ops_impl.cuh"

namespace fsi {

constexpr int NAT = 128;

// ------------------------------------------------------------------ element matrices
// The 32 x 32 matrix of an element in the Walsh basis of its corners.  With s = +-1 for the
// upper/lower side, kappa = 1/sqrt3 and chi_u(b) the product of the signs of corner b over the
// axes in the bit set u, a shape function at Gauss point q is
//   N_b(q) = sum_u D_u chi_u(b) chi_u(q),   d_j N_b(q) = (2 / (kappa h_j)) sum_{u with j} D_u chi_u(b) chi_{u-j}(q),
// D_u = kappa^|u| / 8, so a term sum_q c(q) (d_i) N_a (d_j) N_b has the entries
//   D_u D_v m[(u - i) ^ (v - j)],   m[w] = sum_q c(q) chi_w(q):
// a lookup of one of 8 moments instead of 8 products per entry.  Lane v of an element's eight
// holds moment v of every coefficient field and column v of the block being built (registers over
// u); the moments it needs are at lane distance u (shuffles).  Two Walsh transforms, over u in
// registers and over v across the lanes, return to corners.  About 2,300 float64 operations
// a lane against 8,700 when every column is the product of a unit increment.  With the sums
// into node rows 9.0 ms at 64^3, against 38.3 ms for coefficients and matrices before (and 8.5 ms
// for the Jacobi diagonal, which comes with the rows).
struct Walsh {
  int q;
  double sd[3];  // sign of the lane per axis
  double mk[3];  // 1 where the lane's index holds the axis
  __device__ __forceinline__ double moment(double c) const {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double p = hq_shx(c, 1 << d);
      c = fma(-sd[d], p, c);  // lower lane: c + p, upper lane: c - p
    }
    return c;
  }
  // N_a N_b
  __device__ __forceinline__ void nn(double (&T)[8], double m) const {
#pragma unroll
    for (int u = 0; u < 8; ++u) T[u] += hq_shx(m, u);
  }
  // d_j N_a N_b
  template <int J>
  __device__ __forceinline__ void dn(double (&T)[8], double m) const {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u & (1 << J)) T[u] += hq_shx(m, u ^ (1 << J));
  }
  // N_a d_j N_b
  template <int J>
  __device__ __forceinline__ void nd(double (&T)[8], double m) const {
#pragma unroll
    for (int u = 0; u < 8; ++u) T[u] = fma(mk[J], hq_shx(m, u ^ (1 << J)), T[u]);
  }
  // f d_i N_a d_j N_b
  template <int I, int J>
  __device__ __forceinline__ void dd(double (&T)[8], double m, double f) const {
    const double k = f * mk[J];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u & (1 << I)) T[u] = fma(k, hq_shx(m, u ^ (1 << I) ^ (1 << J)), T[u]);
  }
  // to corners, times W D_u D_v; out[a] is entry (a, lane)
  __device__ __forceinline__ void corners(double (&T)[8], double dv) const {
    constexpr double k1 = 0.57735026918962576451;
    // over u: register butterflies that take kappa per axis along
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (!(u & (1 << d))) {
          const double a = T[u], b = T[u | (1 << d)];
          T[u] = fma(-k1, b, a);
          T[u | (1 << d)] = fma(k1, b, a);
        }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      double t = T[a] * dv;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double p = hq_shx(t, 1 << d);
        t = fma(sd[d], p, t);  // lower lane: t - p, upper lane: t + p
      }
      T[a] = t;
    }
  }
};

// Element matrices of the layers [e0, e1) / (nx ny), rows and columns field-major (8 corners of
// dv_x, dv_y, dv_z, dp each): K[((ez % slots) * 1024 + i * 32 + j) * nxyp + ey * nxp + ex],
// times the quadrature weight.  The block of row field r and column field c is the sum of
//   N_a N_b rho (delta cm + al L_rc),  N_a d_j N_b delta rho al v_j,
//   d_j N_a N_b [tau_m rho v_j (delta cm + al L_rc) + delta_jc al tau_m R_r - al aG_rj,c],
//   d_j N_a d_i N_b [delta al (tau_m rho v_j v_i + delta_ij mu + aB_ij)
//                    + delta_jc al (aB_ir + delta_ir mu) + delta_jr delta_ic al tau_c rho]
// for velocities (delta = [r = c]), d_r N_a (-N_b) + d_j N_a d_r N_b tau_m v_j for the pressure
// columns, N_a d_c N_b al + d_j N_a (N_b tau_m (al L_jc + delta_jc cm) + delta_jc tau_m al v.grad N_b)
// for the continuity rows and tau_m / rho grad N_a . grad N_b in their corner (the product's
// linearization at one point, nsq_point_fg, read off by field).
template <bool MANY>
__global__ void __launch_bounds__(HQ_THREADS) nsa_elem_kernel(const __grid_constant__ HexNS H, double* __restrict__ K,
                                                              unsigned e0, unsigned e1, int slots, int elastic) {
  HexLane l;
  l.set(H.g, H.rh, e0, e1);
  Walsh w;
  w.q = l.q;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    w.sd[d] = (l.q >> d) & 1 ? 1.0 : -1.0;
    w.mk[d] = (l.q >> d) & 1 ? 1.0 : 0.0;
  }
  constexpr double k1 = 0.57735026918962576451;
  const int bits = __popc(l.q);
  const double dv = H.W / 64.0 * (bits == 0 ? 1.0 : bits == 1 ? k1 : bits == 2 ? 1.0 / 3.0 : k1 / 3.0);
  // 2 / (kappa h_j): the derivative's factor beside D_u
  const double s[3] = {2.0 / k1 * H.rh[0], 2.0 / k1 * H.rh[1], 2.0 / k1 * H.rh[2]};
  const double al = H.P.alpha, cm = H.P.c_mass;
  NSPoint p;
  hq_ns_point(H, l, p);
  double aB[6], aG[6][3];
  if (elastic) {
    hq_elastic<MANY>(H, l, aB, aG);
  } else {
#pragma unroll
    for (int c = 0; c < 6; ++c) aB[c] = aG[c][0] = aG[c][1] = aG[c][2] = 0.0;
  }
  const double tr = p.tau_m * p.rho;
  double* out = K + (int64_t)(l.ez % slots) * 1024 * H.nxyp + (int64_t)l.ey * H.nxp + l.ex + (int64_t)l.q * H.nxyp;
  auto store = [&](int r, int c, double (&T)[8]) {
    w.corners(T, dv);
    if (l.ok) {
#pragma unroll
      for (int a = 0; a < 8; ++a) out[(int64_t)((8 * r + a) * 32 + 8 * c) * H.nxyp] = T[a];
    }
  };
  // moments that several blocks use, times the derivative factors of their own
  double mtv[3], maB[6];
#pragma unroll
  for (int j = 0; j < 3; ++j) mtv[j] = w.moment(p.tau_m * p.v[j]) * s[j];  // row factor of d_j N_a
#pragma unroll
  for (int c = 0; c < 6; ++c) maB[c] = elastic ? w.moment(al * aB[c]) : 0.0;
  const double mmu = w.moment(al * p.mu), mtc = w.moment(al * p.tau_c * p.rho);
  // the scalar operator of the three diagonal velocity blocks
  double S[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) S[u] = 0.0;
  w.nn(S, w.moment(p.rho * cm));
  {
    const double d0 = w.moment(s[0] * tr * cm * p.v[0]), d1 = w.moment(s[1] * tr * cm * p.v[1]),
                 d2 = w.moment(s[2] * tr * cm * p.v[2]);
    w.dn<0>(S, d0);
    w.dn<1>(S, d1);
    w.dn<2>(S, d2);
    const double ra = p.rho * al;
    w.nd<0>(S, w.moment(s[0] * ra * p.v[0]));
    w.nd<1>(S, w.moment(s[1] * ra * p.v[1]));
    w.nd<2>(S, w.moment(s[2] * ra * p.v[2]));
    const double ta = tr * al;
    const double t00 = w.moment(ta * p.v[0] * p.v[0]) + mmu + maB[0], t11 = w.moment(ta * p.v[1] * p.v[1]) + mmu + maB[1],
                 t22 = w.moment(ta * p.v[2] * p.v[2]) + mmu + maB[2], t01 = w.moment(ta * p.v[0] * p.v[1]) + maB[3],
                 t12 = w.moment(ta * p.v[1] * p.v[2]) + maB[4], t02 = w.moment(ta * p.v[0] * p.v[2]) + maB[5];
    w.dd<0, 0>(S, t00, s[0] * s[0]);
    w.dd<1, 1>(S, t11, s[1] * s[1]);
    w.dd<2, 2>(S, t22, s[2] * s[2]);
    w.dd<0, 1>(S, t01, s[0] * s[1]);
    w.dd<1, 0>(S, t01, s[0] * s[1]);
    w.dd<1, 2>(S, t12, s[1] * s[2]);
    w.dd<2, 1>(S, t12, s[1] * s[2]);
    w.dd<0, 2>(S, t02, s[0] * s[2]);
    w.dd<2, 0>(S, t02, s[0] * s[2]);
  }
  auto velocity = [&](auto kc, auto lc) {
    constexpr int k = decltype(kc)::value, c = decltype(lc)::value;
    double T[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) T[u] = k == c ? S[u] : 0.0;
    const double La = al * p.L[k][c];
    w.nn(T, w.moment(p.rho * La));
    double m[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double t = tr * p.v[j] * La;
      if (j == c) t = fma(al * p.tau_m, p.R[k], t);
      if (elastic) t = fma(-al, aG[sym_idx(k, j)][c], t);
      m[j] = w.moment(s[j] * t);
    }
    w.dn<0>(T, m[0]);
    w.dn<1>(T, m[1]);
    w.dn<2>(T, m[2]);
    w.dd<c, 0>(T, k == 0 ? maB[sym_idx(0, k)] + mmu : maB[sym_idx(0, k)], s[c] * s[0]);
    w.dd<c, 1>(T, k == 1 ? maB[sym_idx(1, k)] + mmu : maB[sym_idx(1, k)], s[c] * s[1]);
    w.dd<c, 2>(T, k == 2 ? maB[sym_idx(2, k)] + mmu : maB[sym_idx(2, k)], s[c] * s[2]);
    w.dd<k, c>(T, mtc, s[k] * s[c]);
    store(k, c, T);
  };
  auto pressure = [&](auto kc) {  // column p of momentum row k
    constexpr int k = decltype(kc)::value;
    double T[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) T[u] = 0.0;
    w.dn<k>(T, l.q == 0 ? -8.0 * s[k] : 0.0);  // the moments of -1
    w.dd<0, k>(T, mtv[0], s[k]);
    w.dd<1, k>(T, mtv[1], s[k]);
    w.dd<2, k>(T, mtv[2], s[k]);
    store(k, 3, T);
  };
  auto continuity = [&](auto lc) {  // column v_c of the continuity row
    constexpr int c = decltype(lc)::value;
    double T[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) T[u] = 0.0;
    w.nd<c>(T, l.q == 0 ? 8.0 * al * s[c] : 0.0);
    double m[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) m[j] = w.moment(s[j] * p.tau_m * (j == c ? fma(al, p.L[j][c], cm) : al * p.L[j][c]));
    w.dn<0>(T, m[0]);
    w.dn<1>(T, m[1]);
    w.dn<2>(T, m[2]);
    const double f = al * s[c];
    w.dd<c, 0>(T, mtv[0], f);
    w.dd<c, 1>(T, mtv[1], f);
    w.dd<c, 2>(T, mtv[2], f);
    store(3, c, T);
  };
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  velocity(I0{}, I0{});
  velocity(I0{}, I1{});
  velocity(I0{}, I2{});
  velocity(I1{}, I0{});
  velocity(I1{}, I1{});
  velocity(I1{}, I2{});
  velocity(I2{}, I0{});
  velocity(I2{}, I1{});
  velocity(I2{}, I2{});
  pressure(I0{});
  pressure(I1{});
  pressure(I2{});
  continuity(I0{});
  continuity(I1{});
  continuity(I2{});
  double T[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) T[u] = 0.0;
  const double mr = w.moment(p.tau_m * p.rrho);
  w.dd<0, 0>(T, mr, s[0] * s[0]);
  w.dd<1, 1>(T, mr, s[1] * s[1]);
  w.dd<2, 2>(T, mr, s[2] * s[2]);
  store(3, 3, T);
}

// Rows of the nodes of the planes [k0, k1): one thread per (node, row field); every entry is the sum
// over the up to 8 elements that hold both nodes, in a fixed order (z, y, x of the element).
// blockDim (NAT, 4), one CTA per 128 nodes.  The neighbour loops stay rolled (unrolled they
// spill: 16^3 84 us, 60 so).
__global__ void __launch_bounds__(4 * NAT) nsa_gather_kernel(const double* __restrict__ K, int nx, int ny, int nz, int nxp,
                                                             int64_t nxyp, int slots, int64_t n0, int64_t n1,
                                                             double* __restrict__ A) {
  const int64_t n = n0 + (int64_t)blockIdx.x * NAT + threadIdx.x;
  if (n >= n1) return;
  const int r = threadIdx.y;
  const unsigned row = (unsigned)(n / (nx + 1));
  const int i = (int)(n - (int64_t)row * (nx + 1)), k = (int)(row / (unsigned)(ny + 1));
  const int j = (int)(row - (unsigned)k * (ny + 1));
  const int64_t dst = ((n / NAT) * 27 * 16 + 4 * r) * NAT + n % NAT;
#pragma unroll 1
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll 1
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll 1
      for (int dx = -1; dx <= 1; ++dx) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        // corner a of the element at node (i, j, k) - a; the neighbour is its corner a + d
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
              const double* src = K + ((int64_t)(ez % slots) * 1024 + (8 * r + a) * 32 + b) * nxyp + (int64_t)ey * nxp + ex;
#pragma unroll
              for (int c = 0; c < 4; ++c) acc[c] += src[(int64_t)(8 * c) * nxyp];
            }
          }
        }
        const int o = (dx + 1) + 3 * (dy + 1) + 9 * (dz + 1);
#pragma unroll
        for (int c = 0; c < 4; ++c) A[dst + (int64_t)(16 * o + c) * NAT] = acc[c];
      }
}

// y = A x: blockDim (NAT, 4), one thread per (node, row field), one tile per CTA.  A missing
// neighbour's block is zero and its values are read at the node itself.  Dirichlet rows (velocity;
// pressure at the pin node when pinned) take the increment itself.
__global__ void __launch_bounds__(4 * NAT) nsa_apply_kernel(const double* __restrict__ A, const double* __restrict__ x,
                                                            int nx, int ny, int nz, int64_t nn,
                                                            const uint8_t* __restrict__ mask, int pin,
                                                            double* __restrict__ y) {
  const int64_t n = (int64_t)blockIdx.x * NAT + threadIdx.x;
  if (n >= nn) return;
  const int r = threadIdx.y;
  const unsigned row = (unsigned)(n / (nx + 1));
  const int i = (int)(n - (int64_t)row * (nx + 1)), k = (int)(row / (unsigned)(ny + 1));
  const int j = (int)(row - (unsigned)k * (ny + 1));
  const int64_t sy = nx + 1, sz = sy * (ny + 1);
  const double* a = A + ((int64_t)blockIdx.x * 27 * 16 + 4 * r) * NAT + threadIdx.x;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const bool okx[3] = {i > 0, true, i < nx};
#pragma unroll 1
  for (int dz = -1; dz <= 1; ++dz) {
    const bool okz = k + dz >= 0 && k + dz <= nz;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const bool okyz = okz && j + dy >= 0 && j + dy <= ny;
#pragma unroll
      for (int ddx = -1; ddx <= 1; ++ddx) {
        const int64_t nb = okyz && okx[ddx + 1] ? n + ddx + sy * dy + sz * dz : n;
        const double* ao = a + (int64_t)16 * ((ddx + 1) + 3 * (dy + 1) + 9 * (dz + 1)) * NAT;
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] += __ldcs(ao + c * NAT) * __ldg(x + c * nn + nb);
      }
    }
  }
  const bool dir = ((mask[n] >> r) & 1) && (r < 3 || pin);
  const int64_t q = (int64_t)r * nn + n;
  y[q] = dir ? x[q] : (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// The same with three threads per (node, row field), one per neighbour plane, summed through shared
// memory: CTAs of 32 nodes.  For meshes whose 128-node CTAs leave SMs idle or with one CTA, where a
// thread's 27 dependent rounds of loads are all of the time.
__global__ void __launch_bounds__(384) nsa_apply_split_kernel(const double* __restrict__ A, const double* __restrict__ x,
                                                              int nx, int ny, int nz, int64_t nn,
                                                              const uint8_t* __restrict__ mask, int pin,
                                                              double* __restrict__ y) {
  __shared__ double part[2][4][32];
  const int64_t n = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int r = threadIdx.y, dz = (int)threadIdx.z - 1;
  double s = 0.0;
  if (n < nn) {
    const unsigned row = (unsigned)n / (unsigned)(nx + 1);
    const int i = (int)((unsigned)n - row * (unsigned)(nx + 1)), k = (int)(row / (unsigned)(ny + 1));
    const int j = (int)(row - (unsigned)k * (unsigned)(ny + 1));
    const int64_t sy = nx + 1, sz = sy * (ny + 1);
    const double* a = A + ((n / NAT * 27 + 9 * (dz + 1)) * 16 + 4 * r) * NAT + n % NAT;
    const bool okz = k + dz >= 0 && k + dz <= nz;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const bool okyz = okz && j + dy >= 0 && j + dy <= ny;
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const bool ok = okyz && i + dx >= 0 && i + dx <= nx;
        const int64_t nb = ok ? n + dx + sy * dy + sz * dz : n;
        const double* ao = a + 16 * ((dx + 1) + 3 * (dy + 1)) * NAT;
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] += __ldg(ao + c * NAT) * __ldg(x + c * nn + nb);
      }
    }
    s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  }
  if (dz != 0) part[dz > 0][r][threadIdx.x] = s;
  __syncthreads();
  if (dz != 0 || n >= nn) return;
  s = part[0][r][threadIdx.x] + s + part[1][r][threadIdx.x];
  const bool dir = ((mask[n] >> r) & 1) && (r < 3 || pin);
  const int64_t q = (int64_t)r * nn + n;
  y[q] = dir ? x[q] : s;
}

// the diagonal of the assembled operator (1 on Dirichlet rows)
__global__ void nsa_diag_kernel(const double* __restrict__ A, int64_t nn, const uint8_t* __restrict__ mask, int pin,
                                double* __restrict__ d) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  const uint8_t mk = mask[n];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const bool dir = ((mk >> r) & 1) && (r < 3 || pin);
    d[(int64_t)r * nn + n] = dir ? 1.0 : A[((n / NAT) * 27 * 16 + 13 * 16 + 5 * r) * NAT + n % NAT];
  }
}

// element matrices kept at a time (they are needed until the node planes on both sides are summed)
constexpr int64_t NSA_SLAB_BYTES = (int64_t)1 << 30;

// scratch of the element matrices (every block in turn)
int ensure_elem_matrices(fsi_mesh* m, int64_t len) {
  if (m->ke_len >= len) return FSI_OK;
  cudaFree(m->ke64);
  m->ke64 = nullptr;
  m->ke_len = 0;
  FSI_CUDA(cudaMalloc(&m->ke64, sizeof(double) * (size_t)len));
  m->ke_len = len;
  return FSI_OK;
}

int nsa_build(fsi_mesh* m, unsigned flags) {
  const unsigned eflags = flags & FSI_ELASTIC_AUG;
  if (m->na_gen == m->stage_gen && m->na_flags == eflags && m->na64) return FSI_OK;
  const Geom& g = m->g;
  const int nxp = cq_pitch(m);
  const int64_t nxyp = (int64_t)nxp * g.ny, layer = 1024 * nxyp;
  const int64_t len = (m->nn + NAT - 1) / NAT * NAT * 27 * 16;
  if (m->na_len < len) {
    cudaFree(m->na64);
    m->na64 = nullptr;
    m->na_len = 0;
    FSI_CUDA(cudaMalloc(&m->na64, sizeof(double) * (size_t)len));
    m->na_len = len;
  }
  const int slots = (int)std::min<int64_t>(g.nz, std::max<int64_t>(2, NSA_SLAB_BYTES / (8 * layer)));
  if (int rc = ensure_elem_matrices(m, slots * layer)) return rc;
  const HexNS H = hex_ns(m, nxp);
  auto* kernel = m->ns >= HQ_MANY ? &nsa_elem_kernel<true> : &nsa_elem_kernel<false>;
  const int elastic = eflags && m->ns > 0 ? 1 : 0;
  const int64_t plane = (int64_t)(g.nx + 1) * (g.ny + 1);
  // a ring of layer slots: after the layers [z0, z1), the planes [z0, z1) are complete, and layer
  // z1 - 1 stays for plane z1
  const int step = slots == g.nz ? g.nz : slots - 1;
  for (int z0 = 0; z0 < g.nz; z0 += step) {
    const int z1 = std::min(g.nz, z0 + step);
    const unsigned e0 = (unsigned)z0 * g.ny * g.nx, e1 = (unsigned)z1 * g.ny * g.nx;
    FSI_LAUNCH(m, P_NS_BUILD,
               kernel<<<hq_blocks(e1 - e0), HQ_THREADS, 0, m->stream>>>(H, m->ke64, e0, e1, slots, elastic));
    const int64_t n0 = z0 * plane, n1 = (z1 == g.nz ? z1 + 1 : z1) * plane;
    FSI_LAUNCH(m, P_NS_BUILD,
               nsa_gather_kernel<<<(unsigned)((n1 - n0 + NAT - 1) / NAT), dim3(NAT, 4), 0, m->stream>>>(
                   m->ke64, g.nx, g.ny, g.nz, nxp, nxyp, slots, n0, n1, m->na64));
  }
  m->na_gen = m->stage_gen;
  m->na_flags = eflags;
  return FSI_OK;
}

// below this many nodes the split kernel is taken
constexpr int64_t NSA_SPLIT_NODES = 152 * 256;

int launch_nsa(fsi_mesh* m, const double* dx, double* y, unsigned flags) {
  if (int rc = nsa_build(m, flags)) return rc;
  const Geom& g = m->g;
  // algorithmic bytes: the blocks once, the increment in, the product out, the mask
  prof_bytes(m, P_NS_JVP64E, (double)m->nn * (27.0 * 16 * 8 + 32 + 32 + 1));
  if (m->nn < NSA_SPLIT_NODES) {
    FSI_LAUNCH(m, P_NS_JVP64E,
               nsa_apply_split_kernel<<<(unsigned)((m->nn + 31) / 32), dim3(32, 4, 3), 0, m->stream>>>(
                   m->na64, dx, g.nx, g.ny, g.nz, m->nn, m->mask, m->pin_active, y));
    return FSI_OK;
  }
  FSI_LAUNCH(m, P_NS_JVP64E,
             nsa_apply_kernel<<<(unsigned)((m->nn + NAT - 1) / NAT), dim3(NAT, 4), 0, m->stream>>>(
                 m->na64, dx, g.nx, g.ny, g.nz, m->nn, m->mask, m->pin_active, y));
  return FSI_OK;
}

int nsa_diag(fsi_mesh* m, double* d, unsigned flags) {
  if (int rc = nsa_build(m, flags)) return rc;
  FSI_LAUNCH(m, P_NS_DIAG,
             nsa_diag_kernel<<<(unsigned)((m->nn + 255) / 256), 256, 0, m->stream>>>(m->na64, m->nn, m->mask,
                                                                                     m->pin_active, d));
  return FSI_OK;
}

}  // namespace fsi
