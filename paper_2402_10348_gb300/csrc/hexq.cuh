// Float64 hexahedral integrals with one thread per (element, quadrature point).
//
// GB300 issues float64 at 1/64 of the float32 rate, so every float64 element kernel here is bound
// by its float64 instruction count, not by memory; shuffles and integer work are almost
// free beside it.  Eight adjacent lanes of a warp share an element: lane q holds the value of
// corner q and ends up with the field at quadrature point q.  The 2 x 2 x 2 interpolation is then
// three butterfly stages (lane distance 1, 2, 4 for x, y, z), each one subtraction and one fused
// multiply-add, G0 u + G1 u' = u + G1 (u' - u), and the difference u' - u is the derivative along
// that axis.  Value and gradient at a point cost 15 float64 operations instead of 32 when one
// thread interpolates the 8 corners for each point by itself, the transposed scatter 18
// instead of 45, and a mesh has 8 times as many threads, which is what small meshes lack.
// Corner contributions leave as E[8 x equation + corner][element]: four adjacent elements
// of a warp fill one 32-byte sector of a plane.  A node kernel sums them in a fixed order; a mesh too
// large for the scratch goes slab by slab of layers.
//
// Against the z-marching tiles (q1_tile.cuh), which evaluate a halo ring twice and give a small
// mesh a handful of CTAs: momentum residual at 64^3 3.88 -> 1.18 ms, at 8^3 444 -> 18 us.
#pragma once
#include "internal.h"

namespace fsi {

__device__ __forceinline__ double hq_shx(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
// G0 own + G1 partner along one axis
__device__ __forceinline__ double hq_mix(double v, int m) { return fma(FSI_G1, hq_shx(v, m) - v, v); }

// The element of this thread: 8 lanes per element, elements numbered x fastest.  Threads past
// the last element work on it again (the shuffles need whole warps) and write nothing.
struct HexLane {
  int q;              // corner and quadrature point of the lane
  bool ok;
  int ex, ey, ez;
  int64_t n;          // the lane's corner node
  double sx, sy, sz;  // 1/h with the sign that turns partner - own into the derivative
  // elements [e0, e1) of the mesh (32-bit: a state of 2^31 elements exceeds the memory)
  __device__ __forceinline__ void set(const Geom& g, const double (&rh)[3], unsigned e0, unsigned e1) {
    set(g, rh, e0, e1, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  }
  __device__ __forceinline__ void set(const Geom& g, const double (&rh)[3], unsigned e0, unsigned e1, int64_t t) {
    q = (int)(t & 7);
    ok = e0 + (t >> 3) < e1;
    const unsigned f = ok ? e0 + (unsigned)(t >> 3) : e1 - 1;
    const unsigned row = f / (unsigned)g.nx;
    ex = (int)(f - row * (unsigned)g.nx);
    ez = (int)(row / (unsigned)g.ny);
    ey = (int)(row - (unsigned)ez * (unsigned)g.ny);
    n = (int64_t)(ex + (q & 1)) + (int64_t)(g.nx + 1) * ((ey + ((q >> 1) & 1)) + (int64_t)(g.ny + 1) * (ez + (q >> 2)));
    sx = (q & 1) ? -rh[0] : rh[0];
    sy = (q & 2) ? -rh[1] : rh[1];
    sz = (q & 4) ? -rh[2] : rh[2];
  }
  __device__ __forceinline__ double val(double u) const { return hq_mix(hq_mix(hq_mix(u, 1), 2), 4); }
  // value and the gradient without its factors sx, sy, sz
  __device__ __forceinline__ VG<double> vg_raw(double u) const {
    const double dx = hq_shx(u, 1) - u, ux = fma(FSI_G1, dx, u);
    const double dy = hq_shx(ux, 2) - ux, uy = fma(FSI_G1, dy, ux);
    const double dz = hq_shx(uy, 4) - uy;
    VG<double> r;
    r.v = fma(FSI_G1, dz, uy);
    r.gx = hq_mix(hq_mix(dx, 2), 4);
    r.gy = hq_mix(dy, 4);
    r.gz = dz;
    return r;
  }
  __device__ __forceinline__ VG<double> vg(double u) const {
    VG<double> r = vg_raw(u);
    r.gx *= sx;
    r.gy *= sy;
    r.gz *= sz;
    return r;
  }
  // the lane's corner of sum_q (N_a f + grad N_a . g), from the lane's point values
  __device__ __forceinline__ double scatter(double f, double gx, double gy, double gz) const {
    const double a = fma(-sz, gz + hq_shx(gz, 4), hq_mix(f, 4));
    const double by = hq_mix(gy, 4), bx = hq_mix(hq_mix(gx, 4), 2);
    const double c = fma(-sy, by + hq_shx(by, 2), hq_mix(a, 2));
    return fma(-sx, bx + hq_shx(bx, 1), hq_mix(c, 1));
  }
};

constexpr int HQ_THREADS = 128;
inline unsigned hq_blocks(int64_t elems) { return (unsigned)((elems * 8 + HQ_THREADS - 1) / HQ_THREADS); }

// Nodal fields of the momentum and continuity equations and what they are evaluated with
struct HexNS {
  const double* xa;   // x^{n+alpha} [ncomp][nn] (p plane: p^{n+1})
  const double* xd;   // dx/dt^{n+alpha_m}
  const double* mat;  // rho, mu, alpha^s
  int64_t nn;
  int nxp;
  int64_t nxyp;
  Geom g;
  Phys P;
  double rh[3];       // 1/h
  double dt2, rtrG;   // 4 / dt^2, 1 / tr G (a float64 division costs tens of instructions)
  double W;           // quadrature weight x |det J|
  int layers;         // layers of elements that the contributions' scratch holds
  __device__ __forceinline__ int64_t stride() const { return (int64_t)layers * nxyp; }  // of its slots
  __device__ __forceinline__ int64_t at(const HexLane& l) const {                       // the lane's element in a slot
    return (int64_t)(l.ez < layers ? l.ez : l.ez % layers) * nxyp + (int64_t)l.ey * nxp + l.ex;
  }
};

// State of the equations at the lane's quadrature point (ops.cuh for the notation)
struct NSPoint {
  double rho, rrho, mu, v[3], L[3][3], gp[3], R[3], tau_m, tau_c, p;  // rrho = 1 / rho
};

__device__ __forceinline__ void hq_ns_point(const HexNS& H, const HexLane& l, NSPoint& s) {
  const Phys& P = H.P;
  const int64_t nn = H.nn, n = l.n;
  s.rho = l.val(H.mat[n]);
  s.mu = l.val(H.mat[nn + n]);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const VG<double> r = l.vg(H.xa[k * nn + n]);
    s.v[k] = r.v; s.L[k][0] = r.gx; s.L[k][1] = r.gy; s.L[k][2] = r.gz;
  }
  const VG<double> pr = l.vg(H.xa[3 * nn + n]);
  s.p = pr.v; s.gp[0] = pr.gx; s.gp[1] = pr.gy; s.gp[2] = pr.gz;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double acc = l.val(H.xd[k * nn + n]) + s.v[0] * s.L[k][0] + s.v[1] * s.L[k][1] + s.v[2] * s.L[k][2];
    s.R[k] = s.rho * acc + s.gp[k] - s.rho * P.grav[k];
  }
  const double vGv = P.Gd[0] * s.v[0] * s.v[0] + P.Gd[1] * s.v[1] * s.v[1] + P.Gd[2] * s.v[2] * s.v[2];
  s.rrho = 1.0 / s.rho;
  const double nu = s.mu * s.rrho;
  const double t2 = H.dt2 + vGv + P.c_i * nu * nu * P.GG;
  s.tau_m = rsqrt(t2);
  s.tau_c = t2 * s.tau_m * H.rtrG;
}

// sum_s a_s B^s and sum_s a_s grad B^s at the lane's point, a_s = alpha^s mu_L^s c_el.  MANY: the sum
// over the solids is taken per corner, C_b = sum_s a_s(q) B^s_b (48 FMAs a solid, the corners' values
// by shuffles), and interpolated once, against interpolating every solid (96): from HQ_MANY
// solids on the fewer operations (a product on the nine-solid ship/ice mesh 47 -> 32.6 ms).
constexpr int HQ_MANY = 4;
template <bool MANY>
__device__ __forceinline__ void hq_elastic(const HexNS& H, const HexLane& l, double (&aB)[6], double (&aG)[6][3]) {
  if constexpr (MANY) {
    double C[6][8];  // entry x: corner q ^ x
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
      for (int x = 0; x < 8; ++x) C[c][x] = 0.0;
    for (int s = 0; s < H.P.ns; ++s) {
      const double a = l.val(H.mat[(2 + s) * H.nn + l.n]) * (H.P.muL[H.P.solid_phase[s]] * H.P.c_el);
      const double* b = H.xa + (int64_t)(4 + H.P.N + 6 * s) * H.nn + l.n;
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const double u = b[c * H.nn];
#pragma unroll
        for (int x = 0; x < 8; ++x) C[c][x] = fma(a, hq_shx(u, x), C[c][x]);
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      // vg_raw in registers: own corner 0, partner along an axis 1
      double dx[4], ux[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        dx[r] = C[c][2 * r + 1] - C[c][2 * r];
        ux[r] = fma(FSI_G1, dx[r], C[c][2 * r]);
      }
      const double dy0 = ux[1] - ux[0], dy1 = ux[3] - ux[2];
      const double uy0 = fma(FSI_G1, dy0, ux[0]), uy1 = fma(FSI_G1, dy1, ux[2]);
      const double gx0 = fma(FSI_G1, dx[1] - dx[0], dx[0]), gx1 = fma(FSI_G1, dx[3] - dx[2], dx[2]);
      const double dz = uy1 - uy0;
      aB[c] = fma(FSI_G1, dz, uy0);
      aG[c][0] = l.sx * fma(FSI_G1, gx1 - gx0, gx0);
      aG[c][1] = l.sy * fma(FSI_G1, dy1 - dy0, dy0);
      aG[c][2] = l.sz * dz;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 6; ++c) aB[c] = aG[c][0] = aG[c][1] = aG[c][2] = 0.0;
    for (int s = 0; s < H.P.ns; ++s) {
      const double a = l.val(H.mat[(2 + s) * H.nn + l.n]) * (H.P.muL[H.P.solid_phase[s]] * H.P.c_el);
      const double* b = H.xa + (int64_t)(4 + H.P.N + 6 * s) * H.nn + l.n;
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const VG<double> r = l.vg_raw(b[c * H.nn]);
        aB[c] = fma(a, r.v, aB[c]);
        aG[c][0] = fma(a, r.gx, aG[c][0]);
        aG[c][1] = fma(a, r.gy, aG[c][1]);
        aG[c][2] = fma(a, r.gz, aG[c][2]);
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      aG[c][0] *= l.sx;
      aG[c][1] *= l.sy;
      aG[c][2] *= l.sz;
    }
  }
}

inline HexNS hex_ns(const fsi_mesh* m, int nxp) {
  HexNS H;
  H.xa = m->staged_xa;
  H.xd = m->xd;
  H.mat = m->mat;
  H.nn = m->nn;
  H.nxp = nxp;
  H.nxyp = (int64_t)nxp * m->g.ny;
  H.g = m->g;
  H.P = m->P;
  H.rh[0] = 1.0 / m->g.hx; H.rh[1] = 1.0 / m->g.hy; H.rh[2] = 1.0 / m->g.hz;
  H.dt2 = 4.0 / (m->P.dt * m->P.dt);
  H.rtrG = 1.0 / m->P.trG;
  H.W = m->g.hx * m->g.hy * m->g.hz / 8.0;
  H.layers = m->g.nz;
  return H;
}

}  // namespace fsi
