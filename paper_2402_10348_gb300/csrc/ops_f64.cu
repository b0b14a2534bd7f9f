// Float64 instantiations of the element operators and the gamma/beta reduction.
#include "ops_impl.cuh"

namespace fsi {

template int launch_ns_diag<double>(fsi_mesh*, double*, unsigned);

// cudaMalloc that is allowed while a stream is being captured too (it is no part of the graph)
static cudaError_t scratch_malloc(double** p, int64_t len) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
  if (e != cudaSuccess) return e;
  e = cudaMalloc(p, sizeof(double) * (size_t)len);
  cudaThreadExchangeStreamCaptureMode(&mode);
  return e;
}

// Scratch of the element contributions.  Meshes whose largest block (48 slots an element with a solid, else 32)
// fits ELEM_SCRATCH have one for everything, taken at once: its address never changes.  On larger ones
// the float64 products, residuals and gamma/beta go slab by slab of layers through that much of their
// own (they ran without any before they were element-centric), and the products of a whole mesh take
// their 32 slots.
constexpr int64_t ELEM_SCRATCH = (int64_t)1 << 30;
static int most_slots(const fsi_mesh* m) { return m->ns > 0 ? 48 : 32; }
static bool one_scratch(const fsi_mesh* m, int64_t nxyp) { return 8 * most_slots(m) * m->g.nz * nxyp <= ELEM_SCRATCH; }

int ensure_elem_scratch(fsi_mesh* m, int64_t nxyp) {
  if (m->ke_e) return FSI_OK;
  FSI_CUDA(scratch_malloc(&m->ke_e, (int64_t)(one_scratch(m, nxyp) ? most_slots(m) : 32) * m->g.nz * nxyp));
  return FSI_OK;
}

int elem_layers(fsi_mesh* m, int64_t nxyp, double** E, int* layers) {
  *layers = m->g.nz;
  if (one_scratch(m, nxyp)) {
    if (int rc = ensure_elem_scratch(m, nxyp)) return rc;
    *E = m->ke_e;
    return FSI_OK;
  }
  const int64_t layer = most_slots(m) * nxyp;
  *layers = (int)std::min<int64_t>(m->g.nz, std::max<int64_t>(2, ELEM_SCRATCH / (8 * layer)));
  if (!m->ke_s) FSI_CUDA(scratch_malloc(&m->ke_s, *layers * layer));
  *E = m->ke_s;
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

}  // namespace fsi
