// Float32 NS product from the quadrature-point coefficients, staged by bulk copies (the FSI_FP32
// product of the NS block inside mixed-precision iterative refinement).
//
// The product is bound by streaming the coefficients (8 points x 44 or 20 float32 values per
// element, Section 2.4's linearization frozen per solve): one thread per element reading 352
// scattered planes keeps too few loads in flight.  Here a CTA owns 128 consecutive elements (x
// fastest) of one layer, whose coefficients lie together, C[(((ez * tiles + tile) * 8 + q) * 44 + c) *
// 128 + element], and receives a point's 44 (or first 20) values of all 128 by one cp.async.bulk
// (22.5 KB) into shared memory, double-buffered on two mbarriers: the copy of point q + 2 runs while
// point q is evaluated.  Thread t evaluates element 128 tile + t (nsq_point on the interpolated
// increment) and writes its 32 corner contributions into E[8 * field + corner][element];
// ns_node_kernel sums them.  With 64 x 2 boxes of a plane layout instead, three quarters of the
// threads and of the bytes in flight were idle on a 16^3 mesh: the product of twelve 16^3-48^3
// cavities took 140 us, now 133; 64^3 62.5 either way.
//
// Every mbarrier wait is bounded; a wait that gives up sets *err, the CTA stops issuing
// copies, waits (bounded) for the copies it has in flight and writes NaN contributions.
#include "ops_impl.cuh"

namespace fsi {
namespace {

constexpr int TBE = NSQ_TILE;  // elements of a CTA's tile, one thread each
constexpr int TSTAGES = 2;
constexpr long long TWAIT = 1LL << 22;

__device__ __forceinline__ uint32_t sptr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  for (long long i = 0; i < TWAIT; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// one point's coefficients into dst (both 16-byte aligned, bytes a multiple of 512); completion on bar
__device__ __forceinline__ void load_point(uint32_t dst, const float* src, uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// coefficient accessor over one element's column of a staged box
struct SmemCoef {
  const float* p;
  __device__ __forceinline__ float operator()(int i) const { return p[i * TBE]; }
};

// One CTA's tile: elements 128 tile .. of layer ez, ncoef coefficients per point staged from the tile's
// coefficients C into `stage` ([TSTAGES][ncoef][TBE]); contributions into E (element plane pitch nxyp).
__device__ __forceinline__ void nsq_tma_tile(float* stage, const float* __restrict__ C, int ncoef,
                                             const float* __restrict__ dx, float* __restrict__ E, int nx, int ny,
                                             int nz, int nxp, int64_t nxyp, int64_t nn, float al, float cmass,
                                             float rhx, float rhy, float rhz, int tile, int ez, int* err) {
  __shared__ __align__(8) uint64_t bar[TSTAGES];
  __shared__ int failed;
  const int SF = ncoef * TBE;  // floats per stage
  const uint32_t SBYTES = (uint32_t)SF * sizeof(float);
  const int tid = threadIdx.x;
  if (tid == 0) {
    failed = 0;
    for (int s = 0; s < TSTAGES; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(sptr(&bar[s])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  if (tid == 0)
    for (int s = 0; s < TSTAGES; ++s) load_point(sptr(stage + s * SF), C + s * NCQ * TBE, sptr(&bar[s]), SBYTES);
  // the increment at the element's corners (while the first boxes arrive)
  const unsigned f0 = (unsigned)tile * TBE + (unsigned)tid;
  const int ey = (int)(f0 / (unsigned)nx), ex = (int)(f0 - (unsigned)ey * (unsigned)nx);
  const bool valid = ey < ny;
  float x[4][8], c[4][8];
  const int64_t sy = nx + 1, sz = (int64_t)(nx + 1) * (ny + 1);
  const int64_t n0 = ex + sy * ey + sz * ez;
  const int64_t off[8] = {0, 1, sy, sy + 1, sz, sz + 1, sz + sy, sz + sy + 1};
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      x[f][a] = valid ? __ldg(dx + f * nn + n0 + off[a]) : 0.0f;
      c[f][a] = 0.0f;
    }
  int q = 0;
  for (; q < 8; ++q) {
    const int s = q % TSTAGES;
    if (!bar_wait(sptr(&bar[s]), (uint32_t)((q / TSTAGES) & 1))) atomicExch(&failed, 1);
    __syncthreads();
    if (failed) break;
    if (valid) {
      QW<float> w;
      w.set(q);
      float dv[3], gd[3][3];
#pragma unroll
      for (int kk = 0; kk < 3; ++kk) {
        const VG<float> r = interp_vg(x[kk], w, rhx, rhy, rhz);
        dv[kk] = r.v; gd[kk][0] = r.gx; gd[kk][1] = r.gy; gd[kk][2] = r.gz;
      }
      const VG<float> dpr = interp_vg(x[3], w, rhx, rhy, rhz);
      const float dgp[3] = {dpr.gx, dpr.gy, dpr.gz};
      nsq_point<float>(SmemCoef{stage + s * SF + tid}, ncoef == NCQ, dv, gd, dpr.v, dgp, al, cmass, w, rhx, rhy, rhz,
                       c);
    }
    __syncthreads();  // every thread is done with stage s
    if (tid == 0 && q + TSTAGES < 8)
      load_point(sptr(stage + s * SF), C + (q + TSTAGES) * NCQ * TBE, sptr(&bar[s]), SBYTES);
  }
  if (failed) {
    // copies issued for points q .. min(q + TSTAGES, 8) - 1 may still be in flight; the
    // product of this tile is NaN, so the solve that uses it stops on a non-finite vector
    if (tid == 0) {
      if (err) *err = 1;
      for (int p = q; p < 8 && p < q + TSTAGES; ++p) bar_wait(sptr(&bar[p % TSTAGES]), (uint32_t)((p / TSTAGES) & 1));
    }
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int a = 0; a < 8; ++a) c[f][a] = __int_as_float(0x7fc00000);
  }
  if (!valid) return;
  const int64_t e = (int64_t)ez * nxyp + (int64_t)ey * nxp + ex;
  const int64_t es = (int64_t)nz * nxyp;
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int a = 0; a < 8; ++a) E[(8 * f + a) * es + e] = c[f][a];
}

__global__ void __launch_bounds__(TBE) nsq_tma_kernel(const float* __restrict__ C, int ncoef, int tiles,
                                                      const float* __restrict__ dx, float* __restrict__ E, int nx, int ny,
                                                      int nz, int nxp, int64_t nxyp, int64_t nn, float al, float cmass,
                                                      float rhx, float rhy, float rhz, int* err) {
  extern __shared__ __align__(128) float stage[];
  const int ez = blockIdx.x / tiles, tile = blockIdx.x - ez * tiles;
  nsq_tma_tile(stage, C + (int64_t)blockIdx.x * 8 * NCQ * TBE, ncoef, dx, E, nx, ny, nz, nxp, nxyp, nn, al, cmass, rhx, rhy,
               rhz, tile, ez, err);
}

// Batched: one CTA per work item (instance, tile, 0, layer); the instance's parameters come from
// its record in global memory.
__global__ void __launch_bounds__(TBE) nsq_tma_batch_kernel(const NSQBatchRec* __restrict__ recs,
                                                            const int4* __restrict__ items, const int* active) {
  extern __shared__ __align__(128) float stage[];
  const int4 it = items[blockIdx.x];
  if (active && !active[it.x]) return;
  const NSQBatchRec& R = recs[it.x];
  const int tiles = (int)(((int64_t)R.nx * R.ny + TBE - 1) / TBE);
  nsq_tma_tile(stage, R.cq32 + ((int64_t)it.w * tiles + it.y) * 8 * NCQ * TBE, R.elastic ? NCQ : NCQ_FLUID, R.dx32, R.E,
               R.nx, R.ny, R.nz, R.nxp, R.nxyp, R.nn, R.al, R.cm, R.rhx, R.rhy, R.rhz, it.y, it.w, R.err);
}

// NS product from the quadrature-point coefficients (see nsq_point) of element (ex, ey, ez)
// into its 32 contribution slots (element-centric)
template <typename T>
__device__ __forceinline__ void nsq_elem_body(const T* __restrict__ cq, const T* __restrict__ dx, T* __restrict__ E,
                                              int nx, int ny, int nz, int nxp, int64_t nxyp, int64_t nn, int elastic,
                                              T al, T cmass, T rhx, T rhy, T rhz, int ex, int ey, int ez) {
  const int64_t sy = nx + 1, sz = (int64_t)(nx + 1) * (ny + 1);
  const int64_t n0 = ex + sy * ey + sz * ez;
  const int64_t off[8] = {0, 1, sy, sy + 1, sz, sz + 1, sz + sy, sz + sy + 1};
  T x[4][8], c[4][8];
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      x[f][a] = __ldg(dx + f * nn + n0 + off[a]);
      c[f][a] = T(0);
    }
  const T* e0 = cq + (int64_t)ez * 8 * NCQ * nxyp + (int64_t)ey * nxp + ex;
#pragma unroll 1
  for (int q = 0; q < 8; ++q) {
    QW<T> w;
    w.set(q);
    T dv[3], gd[3][3];
#pragma unroll
    for (int kk = 0; kk < 3; ++kk) {
      const VG<T> r = interp_vg(x[kk], w, rhx, rhy, rhz);
      dv[kk] = r.v; gd[kk][0] = r.gx; gd[kk][1] = r.gy; gd[kk][2] = r.gz;
    }
    const VG<T> dpr = interp_vg(x[3], w, rhx, rhy, rhz);
    const T dgp[3] = {dpr.gx, dpr.gy, dpr.gz};
    nsq_point<T>(CoefRef<T>{e0 + (int64_t)q * NCQ * nxyp, nxyp}, elastic != 0, dv, gd, dpr.v, dgp, al, cmass, w, rhx,
                 rhy, rhz, c);
  }
  const int64_t e = (int64_t)ez * nxyp + (int64_t)ey * nxp + ex;
  const int64_t es = (int64_t)nz * nxyp;
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int a = 0; a < 8; ++a) E[(8 * f + a) * es + e] = c[f][a];
}

// Batched float64 product from the coefficients (nsq_elem_body): one CTA per (instance, tile, 0,
// layer) work item
__global__ void __launch_bounds__(TBE) nsq_elem_batch_kernel(const NSQBatchRec* __restrict__ recs,
                                                                   const int4* __restrict__ items, const int* active) {
  const int4 it = items[blockIdx.x];
  if (active && !active[it.x]) return;
  const NSQBatchRec& R = recs[it.x];
  const unsigned f = (unsigned)it.y * TBE + threadIdx.x;
  const int ey = (int)(f / (unsigned)R.nx), ex = (int)(f - (unsigned)ey * (unsigned)R.nx);
  if (ey >= R.ny) return;
  nsq_elem_body<double>(R.cq64, R.dx, R.E64, R.nx, R.ny, R.nz, R.nxp, R.nxyp, R.nn, R.elastic, R.al64, R.cm64,
                        R.rh64[0], R.rh64[1], R.rh64[2], ex, ey, it.w);
}

// Batched node sums: one CTA per (instance, 128 consecutive nodes)
template <typename T>
__global__ void __launch_bounds__(128) ns_node_batch_kernel(const NSQBatchRec* __restrict__ recs,
                                                            const int4* __restrict__ items, const int* active) {
  const int4 it = items[blockIdx.x];
  if (active && !active[it.x]) return;
  const NSQBatchRec& R = recs[it.x];
  const int64_t n = (int64_t)it.y * 128 + threadIdx.x;
  if (n >= R.nn) return;
  const int nx = R.nx, ny = R.ny, nz = R.nz;
  const unsigned jk = (unsigned)n / (unsigned)(nx + 1);
  const int i = (int)((unsigned)n - jk * (unsigned)(nx + 1)), k = (int)(jk / (unsigned)(ny + 1));
  const int j = (int)(jk - (unsigned)k * (unsigned)(ny + 1));
  const int64_t es = (int64_t)nz * R.nxyp;
  const T* E = sizeof(T) == 8 ? reinterpret_cast<const T*>(R.E64) : reinterpret_cast<const T*>(R.E);
  T s[4] = {T(0), T(0), T(0), T(0)};
  // as ns_node_kernel: all eight elements' loads in flight
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int c = 7 - a, ex = i - (c & 1), ey = j - ((c >> 1) & 1), ez = k - (c >> 2);
    const bool ok = ex >= 0 && ex < nx && ey >= 0 && ey < ny && ez >= 0 && ez < nz;
    const int64_t e = ok ? (int64_t)ez * R.nxyp + (int64_t)ey * R.nxp + ex : 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const T v = ok ? E[(8 * f + c) * es + e] : T(0);
      s[f] += v;
    }
  }
  const uint8_t mk = R.mask[n];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const bool dir = ((mk >> f) & 1) && (f < 3 || R.pin);
    R.y[f * R.nn + n] = dir ? (R.dx ? R.dx[f * R.nn + n] : (double)R.dx32[f * R.nn + n]) : R.W * (double)s[f];
  }
}

}  // namespace

int check_tma(fsi_mesh* m) {
  if (!m->tma_err) return FSI_OK;
  int e = 0;
  FSI_CUDA(cudaMemcpyAsync(&e, m->tma_err, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
  FSI_CUDA(cudaStreamSynchronize(m->stream));
  if (e) return set_error(FSI_ECUDA, "NS float32 product: a coefficient copy did not complete within its bounded wait");
  return FSI_OK;
}

int nsq_batch_record(fsi_mesh* m, unsigned flags, bool f64, const double* dx, double* y, float* dx32,
                     NSQBatchRec* rec) {
  const unsigned eflags = flags & FSI_ELASTIC_AUG;
  if (int rc = ns_build(m, flags, f64)) return rc;
  const Geom& g = m->g;
  const int nxp = cq_pitch(m);
  const int64_t nxyp = (int64_t)nxp * g.ny;
  if (int rc = ensure_elem_scratch(m, nxyp)) return rc;
  if (!m->tma_err) {
    FSI_CUDA(cudaMalloc(&m->tma_err, sizeof(int)));
    FSI_CUDA(cudaMemsetAsync(m->tma_err, 0, sizeof(int), m->stream));
  }
  const int elastic = (eflags && m->ns > 0) ? 1 : 0;
  memset(rec, 0, sizeof(*rec));
  if (f64) {
    rec->cq64 = static_cast<const double*>(m->cq64.p);
    rec->E64 = m->ke_e;
  } else {
    rec->cq32 = static_cast<const float*>(m->cq32.p);
  }
  rec->al64 = m->P.alpha;
  rec->cm64 = m->P.c_mass;
  rec->rh64[0] = 1.0 / g.hx;
  rec->rh64[1] = 1.0 / g.hy;
  rec->rh64[2] = 1.0 / g.hz;
  rec->dx32 = dx32;
  rec->dx = dx;
  rec->E = reinterpret_cast<float*>(m->ke_e);
  rec->y = y;
  rec->mask = m->mask;
  rec->err = m->tma_err;
  rec->nxyp = nxyp;
  rec->nn = m->nn;
  rec->W = g.hx * g.hy * g.hz / 8.0;
  rec->nx = g.nx;
  rec->ny = g.ny;
  rec->nz = g.nz;
  rec->nxp = nxp;
  rec->pin = m->pin_active;
  rec->elastic = elastic;
  rec->al = (float)m->P.alpha;
  rec->cm = (float)m->P.c_mass;
  rec->rhx = (float)(1.0 / g.hx);
  rec->rhy = (float)(1.0 / g.hy);
  rec->rhz = (float)(1.0 / g.hz);
  return FSI_OK;
}

int nsq_batch_launch(bool f64, const NSQBatchRec* recs, const int4* eitems, int neitems, const int4* nitems,
                     int nnitems, const int* active, cudaStream_t s) {
  if (f64) {
    if (neitems > 0) nsq_elem_batch_kernel<<<neitems, TBE, 0, s>>>(recs, eitems, active);
    if (nnitems > 0) ns_node_batch_kernel<double><<<nnitems, 128, 0, s>>>(recs, nitems, active);
    FSI_CUDA(cudaGetLastError());
    return FSI_OK;
  }
  const size_t smem = sizeof(float) * (size_t)TSTAGES * NCQ * TBE;
  if (neitems > 0) nsq_tma_batch_kernel<<<neitems, TBE, smem, s>>>(recs, eitems, active);
  if (nnitems > 0) ns_node_batch_kernel<float><<<nnitems, 128, 0, s>>>(recs, nitems, active);
  FSI_CUDA(cudaGetLastError());
  return FSI_OK;
}

int launch_nsq32(fsi_mesh* m, const double* dx, double* y, unsigned flags) {
  if (int rc = ns_build(m, flags, false)) return rc;
  const Geom& g = m->g;
  const int nxp = cq_pitch(m);
  const int64_t nxyp = (int64_t)nxp * g.ny, nn = m->nn;
  const int elastic = ((flags & FSI_ELASTIC_AUG) && m->ns > 0) ? 1 : 0;
  if (int rc = ensure_elem_scratch(m, nxyp)) return rc;
  float* E = reinterpret_cast<float*>(m->ke_e);
  if (!m->tma_err) {
    FSI_CUDA(cudaMalloc(&m->tma_err, sizeof(int)));
    FSI_CUDA(cudaMemsetAsync(m->tma_err, 0, sizeof(int), m->stream));
  }
  const int tiles = nsq_tiles(g);
  const int64_t nblk = (int64_t)tiles * g.nz;
  if (nblk > INT32_MAX) return set_error(FSI_EINVAL, "NS float32 product: mesh too large for one launch");
  const int ncoef = elastic ? NCQ : NCQ_FLUID;
  const size_t smem = sizeof(float) * (size_t)TSTAGES * ncoef * TBE;
  const float al = (float)m->P.alpha, cm = (float)m->P.c_mass;
  const float rx = (float)(1.0 / g.hx), ry = (float)(1.0 / g.hy), rz = (float)(1.0 / g.hz);
  // algorithmic bytes: the coefficient planes once per element, the increment once per
  // node, the 32 element contributions written; the node sums read them back and write
  // the product (the mask once per node)
  const double ne = (double)g.nx * g.ny * g.nz;
  prof_bytes(m, P_NS_JVP32, ne * (8.0 * ncoef + 32.0) * 4.0 + (double)nn * 16.0);
  prof_bytes(m, P_NODE_SUM, ne * 32.0 * 4.0 + (double)nn * (32.0 + 1.0));
  FSI_LAUNCH(m, P_NS_JVP32,
             (nsq_tma_kernel<<<(unsigned)nblk, TBE, smem, m->stream>>>(static_cast<const float*>(m->cq32.p), ncoef, tiles,
                                                                       m->dx32, E, g.nx, g.ny, g.nz, nxp, nxyp, nn, al, cm,
                                                                       rx, ry, rz, m->tma_err)));
  const RowLaunch nl = node_launch(g, 0, g.nz + 1);
  FSI_LAUNCH(m, P_NODE_SUM,
             (ns_node_kernel<float, false><<<nl.grid, nl.block, 0, m->stream>>>(
                 E, g.nx, g.ny, g.nz, nxp, nxyp, g.nz, 0, g.nz + 1, nn, g.hx * g.hy * g.hz / 8.0, m->mask, m->pin_active, dx,
                 m->dx32, nullptr, y)));
  return FSI_OK;
}

}  // namespace fsi
