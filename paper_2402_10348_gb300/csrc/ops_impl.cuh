// Host-side launchers of the element operators for one compute type T.
// Included by ops_f64.cu (T = double) and ops_f32.cu (T = float).
#pragma once
#include "internal.h"

namespace fsi {

template <typename T>
struct Staged;  // staged-state arrays of the compute type

template <>
struct Staged<double> {
  static const double* xa(const fsi_mesh* m) { return m->staged_xa; }
  static const double* xd(const fsi_mesh* m) { return m->xd; }
  static const double* mat(const fsi_mesh* m) { return m->mat; }
};
template <>
struct Staged<float> {
  static const float* xa(const fsi_mesh* m) { return m->xa32; }
  static const float* xd(const fsi_mesh* m) { return m->xd32; }
  static const float* mat(const fsi_mesh* m) { return m->mat32; }
};

template <typename T>
inline void put(Fields& F, int i, const T* p);
template <>
inline void put<double>(Fields& F, int i, const double* p) { F.d[i] = p; F.f[i] = nullptr; }
template <>
inline void put<float>(Fields& F, int i, const float* p) { F.f[i] = p; F.d[i] = nullptr; }

constexpr size_t SMEM_LIMIT = 232448;

inline void fill_common(const fsi_mesh* m, double rh[3], double* W) {
  rh[0] = 1.0 / m->g.hx; rh[1] = 1.0 / m->g.hy; rh[2] = 1.0 / m->g.hz;
  *W = m->g.hx * m->g.hy * m->g.hz / 8.0;
}

int batch_launch_tiles_impl(fsi_batch* b, const void* ops_dev, size_t smem, int cls, int use_active,
                            const void* kernel);

template <class Op>
int launch_batched(fsi_batch* b, const void* ops_dev, size_t smem, int cls, int use_active);

template <class Op>
void* upload_ops(const BatchRec& r) {
  void* d = nullptr;
  if (cudaMalloc(&d, r.bytes.size()) != cudaSuccess) return nullptr;
  if (cudaMemcpy(d, r.bytes.data(), r.bytes.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaFree(d);
    return nullptr;
  }
  return d;
}

template <class Op>
int record_op(BatchRec* r, const Op& op, int cls) {
  if (r->count > 0 && (r->op_size != sizeof(Op) || r->launch != &launch_batched<Op>))
    return set_error(FSI_EINVAL, "batch: instances need the same operator type (same block and pass count)");
  r->op_size = sizeof(Op);
  r->launch = &launch_batched<Op>;
  r->upload = &upload_ops<Op>;
  r->cls = cls;
  r->smem = std::max(r->smem, tile_smem_bytes<Op>(op.nf));
  const unsigned char* p = reinterpret_cast<const unsigned char*>(&op);
  r->bytes.insert(r->bytes.end(), p, p + sizeof(Op));
  ++r->count;
  return FSI_OK;
}

template <class Op>
int launch_batched(fsi_batch* b, const void* ops_dev, size_t smem, int cls, int use_active) {
  if (int rc = ensure_smem_attr(reinterpret_cast<const void*>(&tile_batch_kernel<Op>), smem)) return rc;
  return batch_launch_tiles_impl(b, ops_dev, smem, cls, use_active,
                                 reinterpret_cast<const void*>(&tile_batch_kernel<Op>));
}

// z-chunking of the tile grid for about `per_sm` x 152 CTAs (the mesh's own geometry
// targets one CTA per SM; operators that fit more CTAs per SM get shorter z-ranges)
inline Geom tile_geom(const fsi_mesh* m, int per_sm, dim3* grid) {
  Geom g = m->g;
  if (per_sm > 1) {
    const int cols = g.ncx * g.ncy;
    const int planes = g.nz + 1;
    const int chunks = std::max(1, std::min(planes, (152 * per_sm + cols / 2) / cols));
    g.zc = (planes + chunks - 1) / chunks;
  }
  *grid = dim3(g.ncx, g.ncy, (g.nz + 1 + g.zc - 1) / g.zc);
  return g;
}

template <class Op>
int run_tile(fsi_mesh* m, const Op& op, int cls) {
  if (m->rec) return record_op(m->rec, op, cls);
  const size_t smem = tile_smem_bytes<Op>(op.nf);
  if (int rc = ensure_smem_attr(reinterpret_cast<const void*>(&tile_kernel<Op>), smem)) return rc;
  dim3 grid;
  const Geom g = tile_geom(m, Op::MINB, &grid);
  FSI_LAUNCH(m, cls, tile_kernel<Op><<<grid, NTHREADS, smem, m->stream>>>(op, g));
  return FSI_OK;
}

template <typename T, int MODE>
constexpr int op_class(int kind) {  // Allen-Cahn (1) and B (2): products, else diagonals
  return MODE == 1 ? (kind == 1 ? (sizeof(T) == 8 ? P_AC_JVP64 : P_AC_JVP32) : (sizeof(T) == 8 ? P_B_JVP64 : P_B_JVP32))
                   : (kind == 1 ? P_AC_DIAG : P_B_DIAG);
}

// The increment of a product: float64 kernels read dx itself, float32 kernels the
// float copy the caller made (m->dx32, same layout).
template <typename T>
inline void put_dx(Fields& F, int i, const fsi_mesh* m, const double* dx, int64_t off) {
  if constexpr (sizeof(T) == 4) put<float>(F, i, m->dx32 + off);
  else put<double>(F, i, dx + off);
}

template <typename T>
inline int solids_per_pass(int nf_fixed) {
  // 3 ring slots x (nf_fixed + 7 s) fields + 4 x 8 x 256 contributions
  const size_t fixed = sizeof(T) * (size_t)(3 * nf_fixed * PP + 4 * 8 * NTHREADS);
  const size_t per = sizeof(T) * (size_t)(3 * 7 * PP);
  if (fixed >= SMEM_LIMIT) return 0;
  return (int)((SMEM_LIMIT - fixed) / per);
}

template <typename T>
int ns_pass(fsi_mesh* m, double* y, unsigned flags, int s0, int s1, bool first) {
  NSOp<T> op;
  memset(&op, 0, sizeof(op));
  const T* xa = Staged<T>::xa(m);
  const T* xd = Staged<T>::xd(m);
  const T* mat = Staged<T>::mat(m);
  const int64_t nn = m->nn;
  if (9 + 7 * (s1 - s0) > MAXF) return set_error(FSI_EINVAL, "NS operator: too many staged fields");
  int f = 0;
  for (int k = 0; k < 3; ++k) put<T>(op.F, f++, xa + k * nn);   // v
  put<T>(op.F, f++, xa + 3 * nn);                                 // p^{n+1}
  for (int k = 0; k < 3; ++k) put<T>(op.F, f++, xd + k * nn);   // dv/dt
  put<T>(op.F, f++, mat);                                         // rho
  put<T>(op.F, f++, mat + nn);                                    // mu
  for (int s = s0; s < s1; ++s) {
    put<T>(op.F, f++, mat + (2 + s) * nn);                        // alpha^s
    const int c0 = 4 + m->N + 6 * s;
    for (int c = 0; c < 6; ++c) put<T>(op.F, f++, xa + (c0 + c) * nn);
  }
  op.nf = f;
  op.s0 = s0;
  op.s1 = s1;
  op.fluid = first ? 1 : 0;
  op.elastic_aug = (flags & FSI_ELASTIC_AUG) ? 1 : 0;
  op.P = m->P;
  fill_common(m, op.rh, &op.W);
  op.out.y = y;
  op.out.mask = m->mask;
  op.out.accumulate = first ? 0 : 1;
  op.out.dirichlet = first ? 1 : 0;
  op.out.pin = m->pin_active;
  op.nn_ = nn;
  return run_tile(m, op, P_NS_DIAG);
}

template <typename T>
int launch_ns_diag(fsi_mesh* m, double* y, unsigned flags) {
  const int ns = (flags & FSI_ELASTIC_AUG) ? m->ns : 0;
  // bounded by shared memory and by the MAXF staged-field slots of Fields
  const int per = std::min(solids_per_pass<T>(9), (MAXF - 9) / 7);
  if (per < 1 && ns > 0) return set_error(FSI_EINVAL, "NS operator: shared memory too small for one solid");
  int s0 = 0;
  bool first = true;
  do {
    const int s1 = ns == 0 ? 0 : std::min(ns, s0 + per);
    if (int rc = ns_pass<T>(m, y, flags, s0, s1, first)) return rc;
    first = false;
    s0 = s1;
  } while (s0 < ns);
  return FSI_OK;
}

// x pitch of the coefficient planes: a multiple of 16 bytes for either compute type
inline int cq_pitch(const fsi_mesh* m) { return (m->g.nx + 3) & ~3; }

// ------------------------------------------------ element-centric products
// One thread per element (x fastest, one CTA row per (ey, ez)) gathers its corner values
// from the nodal vectors and writes its corner contributions into E[slot][element]
// (slot = 8 * component + corner, element index ez * nxyp + ey * nxp + ex); a node
// kernel then sums, per node, the slots of its up to 8 elements in a fixed order
// (z, y, x).  Each element is evaluated once (no halo recomputation); deterministic.
// the thread's position in a row_launch grid: x within the row (*x), row index returned
__device__ __forceinline__ int64_t row_index(int len, int* x) {
  const int nbx = (len + blockDim.x - 1) / blockDim.x;
  const int64_t bxi = blockIdx.x % nbx, byi = blockIdx.x / nbx;
  *x = (int)(bxi * blockDim.x + threadIdx.x);
  return byi * blockDim.y + threadIdx.y;
}

// Launch shape over rows of `len` items (elements or nodes along x), `rows` rows: CTAs of
// bx x by threads (bx the row length rounded up to a warp, at most 128; by = 128 / bx
// rows), numbered x-block fastest in a one-dimensional grid (no 65,535 limit on rows).
struct RowLaunch {
  dim3 grid, block;
};
inline RowLaunch row_launch(int len, int64_t rows) {
  const int bx = std::min(128, (len + 31) / 32 * 32), by = 128 / bx;
  const int64_t nbx = (len + bx - 1) / bx, nby = (rows + by - 1) / by;
  return RowLaunch{dim3((unsigned)(nbx * nby)), dim3(bx, by)};
}
// the nodes of the planes [k0, k1)
inline RowLaunch node_launch(const Geom& g, int k0, int k1) { return row_launch(g.nx + 1, (int64_t)(g.ny + 1) * (k1 - k0)); }

// NS node sums: y = W * sum of the element slots, the Dirichlet rows (velocity; pressure
// at the pin node when pinned) take the increment itself (dx, or its float32 copy dx32), less
// the prescribed velocity vD when that is given (a residual: dx is x^{n+1}).  RING: the planes [k0, k1), and E
// holds `layers` layers of elements, layer ez at ez % layers; else all (the remainders cost 1.3 us of 7 on 14 x 15 x 12).
template <typename T, bool RING>
__global__ void __launch_bounds__(128) ns_node_kernel(const T* __restrict__ E, int nx, int ny, int nz, int nxp,
                                                      int64_t nxyp, int layers, int k0, int k1, int64_t nn, double W,
                                                      const uint8_t* __restrict__ mask,
                                                      int pin, const double* __restrict__ dx,
                                                      const float* __restrict__ dx32, const double* __restrict__ vD,
                                                      double* __restrict__ y) {
  int i;
  if (!RING) layers = nz, k0 = 0, k1 = nz + 1;
  const int64_t jk = row_index(nx + 1, &i) + (int64_t)k0 * (ny + 1);
  if (i > nx || jk >= (int64_t)(ny + 1) * k1) return;
  const int j = (int)(jk % (ny + 1)), k = (int)(jk / (ny + 1));
  const int64_t n = i + (int64_t)(nx + 1) * (j + (int64_t)(ny + 1) * k);
  const int64_t es = (int64_t)layers * nxyp;
  T s[4] = {T(0), T(0), T(0), T(0)};
  // elements (z, y, x) descending; an element outside adds a zero, so that the loads of all eight are in
  // flight together (with early exits the sums of the 64^3 float32 product took 19 us, now 16)
#pragma unroll
  for (int a = 0; a < 8; ++a) {  // this node's corner in element (ex, ey, ez), from 7 down
    const int c = 7 - a, ex = i - (c & 1), ey = j - ((c >> 1) & 1), ez = k - (c >> 2);
    const bool ok = ex >= 0 && ex < nx && ey >= 0 && ey < ny && ez >= 0 && ez < nz;
    const int64_t e = ok ? (int64_t)(RING ? ez % layers : ez) * nxyp + (int64_t)ey * nxp + ex : 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const T v = ok ? E[(8 * f + c) * es + e] : T(0);
      s[f] += v;
    }
  }
  const uint8_t mk = mask[n];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const bool dir = ((mk >> f) & 1) && (f < 3 || pin);
    double v = W * (double)s[f];
    if (dir) {
      v = dx ? dx[f * nn + n] : (double)dx32[f * nn + n];
      if (vD && f < 3) v -= vD[f * nn + n];
    }
    y[f * nn + n] = v;
  }
}

// the same sums of NC components without Dirichlet rows or weight
template <int NC, bool RING>
__global__ void __launch_bounds__(128) em_node_kernel(const double* __restrict__ E, int nx, int ny, int nz, int nxp,
                                                      int64_t nxyp, int layers, int k0, int k1, int64_t nn,
                                                      double* __restrict__ y) {
  int i;
  if (!RING) layers = nz, k0 = 0, k1 = nz + 1;
  const int64_t jk = row_index(nx + 1, &i) + (int64_t)k0 * (ny + 1);
  if (i > nx || jk >= (int64_t)(ny + 1) * k1) return;
  const int j = (int)(jk % (ny + 1)), k = (int)(jk / (ny + 1));
  const int64_t n = i + (int64_t)(nx + 1) * (j + (int64_t)(ny + 1) * k);
  const int64_t es = (int64_t)layers * nxyp;
  double s[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) s[c] = 0.0;
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int q = 7 - a, ex = i - (q & 1), ey = j - ((q >> 1) & 1), ez = k - (q >> 2);
    const bool ok = ex >= 0 && ex < nx && ey >= 0 && ey < ny && ez >= 0 && ez < nz;
    const int64_t e = ok ? (int64_t)(RING ? ez % layers : ez) * nxyp + (int64_t)ey * nxp + ex : 0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double v = ok ? E[(8 * c + q) * es + e] : 0.0;
      s[c] += v;
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) y[c * nn + n] = s[c];
}

template <typename T, int MODE>
int ac_run(fsi_mesh* m, int i, const double* dx, double* y) {
  ACOp<T, MODE> op;
  memset(&op, 0, sizeof(op));
  const T* xa = Staged<T>::xa(m);
  const int64_t nn = m->nn;
  int f = 0;
  if (MODE == 1) put_dx<T>(op.F, f++, m, dx, 0);
  for (int k = 0; k < 3; ++k) put<T>(op.F, f++, xa + k * nn);
  put<T>(op.F, f++, xa + (4 + i) * nn);
  op.nf = f;
  op.P = m->P;
  fill_common(m, op.rh, &op.W);
  op.gamma = m->gamma[i];
  op.beta = m->beta[i];
  op.out.y = y;
  op.nn_ = nn;
  return run_tile(m, op, op_class<T, MODE>(1));
}

template <typename T>
int launch_ac(fsi_mesh* m, int mode, int i, const double* dx, double* y) {
  if (mode == 1) return ac_run<T, 1>(m, i, dx, y);
  return ac_run<T, 2>(m, i, dx, y);
}

template <typename T, int MODE>
int b_run(fsi_mesh* m, int s, const double* dx, double* y) {
  BOp<T, MODE> op;
  memset(&op, 0, sizeof(op));
  const T* xa = Staged<T>::xa(m);
  const T* mat = Staged<T>::mat(m);
  const int64_t nn = m->nn;
  int f = 0;
  if (MODE == 1)
    for (int c = 0; c < 6; ++c) put_dx<T>(op.F, f++, m, dx, c * nn);
  for (int k = 0; k < 3; ++k) put<T>(op.F, f++, xa + k * nn);
  put<T>(op.F, f++, mat + (2 + s) * nn);
  op.nf = f;
  op.P = m->P;
  fill_common(m, op.rh, &op.W);
  op.out.y = y;
  op.nn_ = nn;
  return run_tile(m, op, op_class<T, MODE>(2));
}

template <typename T>
int launch_b(fsi_mesh* m, int mode, int s, const double* dx, double* y) {
  if (mode == 1) return b_run<T, 1>(m, s, dx, y);
  return b_run<T, 2>(m, s, dx, y);
}

}  // namespace fsi
