// Float64 instantiations of the element operators and the gamma/beta reduction.
#include "ops_impl.cuh"

namespace fsi {

template int launch_ns<double>(fsi_mesh*, int, const double*, double*, unsigned);

// E[slots][nz * nxyp] scratch of the element contributions (NS, AC and B in turn).  Taken for the largest
// block at once: batched launches keep its address between solves.
int ensure_elem_scratch(fsi_mesh* m, int slots, int64_t nxyp) {
  slots = std::max(slots, m->ns > 0 ? 48 : 32);
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
