// Krylov solver of libfsi: restarted right-preconditioned GMRES(m) (the paper's
// linear solver, Section 2.5) on float64 vectors, optionally with a float32 operator
// inside float64 iterative refinement; the inner solves of the refinement keep their
// Arnoldi basis in float32 (Hessenberg, Givens and every residual stay float64).
//
// Basis layout: the vectors V_0..V_m are stored chunk-interleaved, CH = 256
// elements per chunk, all m+1 vectors of a chunk contiguous:
//     V_i[j] = V[(j / CH) * (M1 * CH) + i * CH + j % CH],   M1 = slots per chunk.
// A CTA of the projection kernels walks whole chunks, so it streams one contiguous
// block of k x 2 KiB per chunk instead of k separate streams 8.8 MB apart (measured
// 3.9 vs 2.7 TB/s read on GB300 for 33 vectors of the 64^3 NS block).
//
// Arnoldi step j (D = diag(dinv)), four launches with the operator's one:
//   w = J z, z = D V_j    (z written together with V_j; w: a contiguous work vector
//                          written by the operator)
//   h = V^T w and |w|^2 in one pass over V_0..V_j      (mdot_kernel)
//   w -= V h, |w|^2 and h2 = V^T w (the second pass's projections of the updated w)
//   in one pass                                           (upd_dot_kernel); its last CTA:
//   if |w_new| < |w_old| / sqrt(2) (classical Gram-Schmidt with the DGKS
//   re-orthogonalization test) h += h2 and |w|^2 -= |h2|^2 (summed anew where |h2| is near |w|)
//   V_{j+1} = (w - V h2) / |w| (V h2 only where the test asked for it) into its slot, and
//   z = D V_{j+1} beside it                                (upd_store_kernel); one more CTA: the
//   Givens rotation of the new Hessenberg column and the residual estimate, written to pinned
//   host memory
// In the projection kernels the last CTA to finish adds the per-CTA partial sums (a warp per row, fixed
// order), so no launch follows for them: at small sizes launches are the time.  16^3, one
// iteration: 103 us with ten launches and a copy, 56 with these; 64^3, float32 basis, beside the
// operator: 109 -> 84.
// The host enqueues step j and only then waits for step j-1's residual estimate, so it
// never stalls the GPU between steps; at most one step beyond convergence is computed and
// ignored.  The least-squares solution and x += D V y are device kernels.  One host
// synchronisation per restart recomputes the true residual b - A x.  All reductions use a fixed
// partition and a fixed summation order (bit-reproducible).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.h"
#include "kreduce.cuh"
#include "pcnet.h"

namespace fsi {

constexpr int VB = 256;   // threads per CTA of the vector kernels
constexpr int CH = KCH;   // elements per basis chunk (one per thread)
constexpr int DCH = 16;   // dot products per CTA pass
constexpr int MMAX = 64;  // largest restart length

static int vgrid(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + VB * 4 - 1) / (VB * 4), 152 * 4));
}
// The fused update (float64: upd_dot_kernel, float32: upd_dot2_kernel): one large CTA per SM, whose groups
// of threads take half chunks (float32: chunks) in turn.  What follows the streaming (the CTA's
// reduction, the last CTA's sums over all of them) costs by the CTA: with two CTAs of 128 threads per SM
// (float32: four) it took 10-20 us of a kernel on the 64^3 NS block, more than the streaming at small k.
// 64^3, float64 solve: 111.4 -> 108.5 ms; float32 basis: 1.018 x a solve.  The projections of
// mdot_kernel did not gain from the same grid.  A vector of fewer half chunks gets only the
// groups and CTAs that it fills: an idle group's zeros would be reduced like any other's sums (16^3: 4 % of
// a solve).
constexpr int KG = 152;
constexpr int HCH = 128;         // elements of half a chunk
constexpr int NHG = 3;           // groups of a full CTA (19 elements a thread at 64^3: 1 % of the time is rounding)
constexpr int UDT = NHG * HCH;   // most threads
struct ProjGrid {
  int ctas, threads;
};
static ProjGrid pgrid(int64_t n) {
  const int64_t units = std::max<int64_t>(1, (n + HCH - 1) / HCH);
  const int64_t groups = std::min<int64_t>(NHG, (units + KG - 1) / KG);
  return {(int)std::min<int64_t>(KG, (units + groups - 1) / groups), (int)groups * HCH};
}
// mdot_kernel: two CTAs per SM: each streams enough chunks to amortise its end-of-kernel
// reduction of up to 16 sums (the reduction dominated at four CTAs per SM)
static int cgrid(int64_t nch) { return (int)std::max<int64_t>(1, std::min<int64_t>(nch, 152 * 2)); }
// mdot4_kernel reduces in float32 up to the CTA (cheap): four CTAs per SM keep more loads in flight
static int cgrid4(int64_t nch) { return (int)std::max<int64_t>(1, std::min<int64_t>(nch, 152 * 4)); }
// the basis store: a few chunks of 256 elements per CTA, eight CTAs per SM
static int chunk_grid(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + CH - 1) / CH, 152 * 8)); }

// the second pass with the basis store: `per` chunks a CTA at a time, eight CTAs per SM at most
static int upd_grid(int64_t n, int per) {
  const int64_t groups = ((n + CH - 1) / CH + per - 1) / per;
  return (int)std::max<int64_t>(1, std::min<int64_t>(groups, 152 * 8));
}

// device-resident Arnoldi/Givens state (inside fsi_mesh::kry_dev)
struct KryDev {
  double h[MMAX + 2];      // current column (pass 1), then the accumulated column
  double h2[MMAX + 2];     // second pass
  double H[(MMAX + 1) * MMAX];
  double cs[MMAX], sn[MMAX], g[MMAX + 1], y[MMAX];
  double nrm_fin;          // norm of the new basis vector before scaling
  double bnorm;
  int reorth;              // the second pass is taken
  unsigned counter;        // CTAs done in a projection kernel (back to 0 after each use)
};

template <int K>
__device__ __forceinline__ void block_reduce_store(double (&acc)[K], int kc, double* out, int stride) {
  __shared__ double sm[K][VB / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    double v = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sm[i][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < kc) {
    double s = 0.0;
    for (int wi = 0; wi < VB / 32; ++wi) s += sm[threadIdx.x][wi];
    out[threadIdx.x * stride] = s;
  }
}

// --------------------------------------------------------- basis (chunked) kernels
// The basis type VT is double for float64 solves and float for the inner solves of
// iterative refinement (a float32 operator inside float64 refinement: the inner solve
// only has to reduce its residual by ir_inner_rtol, far above float32 rounding, and the
// refinement's float64 residual removes what the inner solve leaves).  Products, per-thread sums and,
// with a float basis, the sums of a warp are taken in VT, those across warps and CTAs in float64 (or two floats).  The
// work vector w, the preconditioner diagonal and every vector outside the basis stay float64.

// Whether this CTA is the last of `total` to get here; its earlier global writes (and, for the last
// CTA, everybody's) are visible after it.  The counter is back to 0 for the next kernel.
__device__ __forceinline__ bool last_cta(unsigned* counter, unsigned total) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1u) == total - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}
// dst[i] = sum_c part[i * G + c] for i < rows: a warp takes U rows at a time (their loads in flight
// together: this runs in one CTA while the GPU waits), lanes strided, then shuffle trees
template <int U>
__device__ __forceinline__ void sum_rows(const double* part, int G, int rows, double* dst) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int i0 = (threadIdx.x >> 5) * U; i0 < rows; i0 += U * nw) {
    const int cnt = min(U, rows - i0);
    const double* p = part + (int64_t)i0 * G;
    double s[U];
#pragma unroll
    for (int u = 0; u < U; ++u) s[u] = 0.0;
#pragma unroll 4
    for (int c = lane; c < G; c += 32) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u < cnt) s[u] += __ldcg(p + (int64_t)u * G + c);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
      if (lane == 0 && u < cnt) dst[i0 + u] = s[u];
    }
  }
}

// h[i] = V_i . w for i < k, h[k] = w . w (partial sums part[i * G + cta]).  Groups of DCH vectors per
// blockIdx.y; the last group has k mod DCH = R vectors (perhaps none) and takes w . w.
template <int KC, bool SELF>
__device__ __forceinline__ void mdot_group(const double* __restrict__ V, int M1, int ib, const double* __restrict__ w,
                                           int64_t n, double* part) {
  constexpr int NR = KC + (SELF ? 1 : 0);
  const int G = gridDim.x;
  const int64_t nch = (n + CH - 1) / CH;
  const int64_t per = (nch + G - 1) / G;
  const int64_t c0 = blockIdx.x * per, c1 = min(nch, c0 + per);
  double acc[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) acc[i] = 0.0;
  for (int64_t c = c0; c < c1; ++c) {
    const int64_t j = c * CH + threadIdx.x;
    if (j >= n) break;
    const double wj = w[j];
    const double* blk = V + c * (int64_t)M1 * CH + (int64_t)ib * CH + threadIdx.x;
#pragma unroll
    for (int i = 0; i < KC; ++i) acc[i] += blk[i * CH] * wj;
    if (SELF) acc[NR - 1] += wj * wj;
  }
  block_reduce_store_bf<NR, VB>(acc, NR, false, part + (int64_t)ib * G + blockIdx.x, G);
}

template <int R>
__global__ void __launch_bounds__(VB) mdot_kernel(const double* __restrict__ V, int M1, int k, const double* __restrict__ w,
                                                  int64_t n, double* part, KryDev* K) {
  if (blockIdx.y < gridDim.y - 1) mdot_group<DCH, false>(V, M1, blockIdx.y * DCH, w, n, part);
  else mdot_group<R, true>(V, M1, blockIdx.y * DCH, w, n, part);
  if (last_cta(&K->counter, gridDim.x * gridDim.y)) sum_rows<4>(part, gridDim.x, k + 1, K->h);
}

// The float32 basis: the same projections with 16-byte loads.  A CTA works on four
// chunks at a time, a thread on four adjacent elements of one chunk (one float4 per
// basis vector), so a warp moves as many bytes per load as with a float64 basis and
// keeps as many in flight.  Elements at or past n (the ragged end of the last chunk,
// whose basis slots hold stale bytes) are never read.
__global__ void __launch_bounds__(VB, 4) mdot4_kernel(const float* __restrict__ V, int M1, int k,
                                                   const double* __restrict__ w, int64_t n, double* part, KryDev* K) {
  constexpr int KC = DCH, NR = DCH + 1;
  const int G = gridDim.x;
  const int ib = blockIdx.y * KC, kc = min(KC, k - ib);
  const bool self = blockIdx.y == gridDim.y - 1;
  const int64_t nch = (n + CH - 1) / CH;
  const int64_t per = (nch + G - 1) / G;
  const int64_t c0 = blockIdx.x * per, c1 = min(nch, c0 + per);
  const int sub = threadIdx.x >> 6;       // which of the CTA's four chunks
  const int e0 = (threadIdx.x & 63) * 4;  // first of the thread's four elements
  float acc[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) acc[i] = 0.f;
  for (int64_t c = c0 + sub; c < c1; c += 4) {
    const int64_t j = c * CH + e0;
    if (j >= n) break;
    const float* blk = V + c * (int64_t)M1 * CH + (int64_t)ib * CH + e0;
    float w0, w1, w2, w3;
    if (j + 4 <= n) {
      const double2 a = *reinterpret_cast<const double2*>(w + j);
      const double2 b = *reinterpret_cast<const double2*>(w + j + 2);
      w0 = (float)a.x, w1 = (float)a.y, w2 = (float)b.x, w3 = (float)b.y;
#pragma unroll
      for (int i = 0; i < KC; ++i) {
        if (i >= kc) break;
        const float4 v = *reinterpret_cast<const float4*>(blk + i * CH);
        acc[i] += (v.x * w0 + v.y * w1) + (v.z * w2 + v.w * w3);
      }
    } else {
      w0 = (float)w[j];
      w1 = j + 1 < n ? (float)w[j + 1] : 0.f;
      w2 = j + 2 < n ? (float)w[j + 2] : 0.f;
      w3 = 0.f;
#pragma unroll
      for (int i = 0; i < KC; ++i) {
        if (i >= kc) break;
        const float* p = blk + i * CH;
        float t = p[0] * w0;
        if (j + 1 < n) t += p[1] * w1;
        if (j + 2 < n) t += p[2] * w2;
        acc[i] += t;
      }
    }
    if (self) acc[KC] += (w0 * w0 + w1 * w1) + (w2 * w2 + w3 * w3);
  }
  block_reduce_store_f<NR, VB>(acc, kc + (self ? 1 : 0), self, part + (int64_t)ib * G + blockIdx.x, G);
  if (last_cta(&K->counter, gridDim.x * gridDim.y)) sum_rows<4>(part, G, k + 1, K->h);
}

// out[i] = sum_c part[i*G + c] (fixed order), i = blockIdx.x
__global__ void sum_partials(const double* __restrict__ part, int G, double* out) {
  const int i = blockIdx.x;
  double s = 0.0;
  for (int c = threadIdx.x; c < G; c += VB) s += part[(int64_t)i * G + c];
  double acc[1] = {s};
  __shared__ double res;
  block_reduce_store<1>(acc, 1, &res, 1);
  __syncthreads();
  if (threadIdx.x == 0) out[i] = res;
}

// sum_{i<k} hs_i V_i[j] for the element of this thread in chunk blk (8 loads in flight)
template <typename VT>
__device__ __forceinline__ VT lin_comb_chunk(const VT* __restrict__ hs, const VT* __restrict__ blk, int k) {
  VT p[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  int i = 0;
  for (; i + 8 <= k; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) p[u] += hs[i + u] * blk[(i + u) * CH];
  }
  for (; i < k; ++i) p[0] += hs[i] * blk[i * CH];
  return ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
}

// After the fused update, by the last CTA of its kernel: h2 (the second pass's projections of the
// updated w) and |w|^2 summed from the partials, and the DGKS decision.  K->h becomes column j of the
// Hessenberg matrix: h, plus h2 where |w_new| < |w_old| / sqrt(2) asked for the second pass, and
// K->nrm_fin the new norm below it, without a sweep where |h2| is small beside |w| (PYTHAGORAS).
template <typename VT>
__device__ __forceinline__ void orth_step(const double* part, int G, KryDev* K, int j, const double* w, const VT* V, int M1,
                                          int64_t n) {
  __shared__ double c2[MMAX + 2];
  __shared__ bool measure;
  sum_rows<8>(part, G, j + 2, c2);
  __syncthreads();
  if (threadIdx.x < 32) {
    const double w2 = c2[j + 1];
    const bool reorth = sqrt(w2) < sqrt(K->h[j + 1]) * 0.70710678118654752;
    double hh = 0.0;  // |h2|^2
    for (int q = threadIdx.x; q <= j; q += 32) {
      hh = fma(c2[q], c2[q], hh);
      if (reorth) {
        K->h[q] += c2[q];
        K->h2[q] = c2[q];
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
    if (threadIdx.x == 0) {
      measure = reorth && hh > PYTHAGORAS * w2;
      K->nrm_fin = sqrt(reorth && !measure ? w2 - hh : w2);  // a NaN stays one: the host stops on it
      K->reorth = reorth ? 1 : 0;
    }
  }
  __syncthreads();
  if (!measure) return;
  const double s = corrected_norm2<VT, sizeof(VT) == 4>(w, V, M1, j + 1, c2, n);
  if (threadIdx.x == 0) K->nrm_fin = sqrt(s);
}

// The Givens step by one CTA, beside the basis store: column j is rotated by the previous rotations
// (one thread, in shared memory), the new rotation zeroes its subdiagonal entry, and g and the
// residual estimate |g_{j+1}| / |b| follow.  est (pinned host memory): the estimate, then the
// reorth and breakdown flags as ints.
__device__ __forceinline__ void givens_step(KryDev* K, int j, int mm, double* est) {
  __shared__ double col[MMAX + 2], cs[MMAX], sn[MMAX];
  for (int q = threadIdx.x; q <= j; q += blockDim.x) {
    col[q] = K->h[q];
    if (q < j) {
      cs[q] = K->cs[q];
      sn[q] = K->sn[q];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double hn = K->nrm_fin;
    double t = col[0];
    for (int q = 0; q < j; ++q) {
      const double nx = col[q + 1];
      col[q] = fma(sn[q], nx, cs[q] * t);
      t = fma(-sn[q], t, cs[q] * nx);
    }
    const double den = hypot(t, hn);
    const double c = den > 0.0 ? t / den : 1.0;
    const double sj = den > 0.0 ? hn / den : 0.0;
    K->cs[j] = c;
    K->sn[j] = sj;
    col[j] = den;
    col[j + 1] = 0.0;
    const double gj = K->g[j], gn = -sj * gj;
    K->g[j + 1] = gn;
    K->g[j] = c * gj;
    est[0] = fabs(gn) / K->bnorm;
    int* flags = reinterpret_cast<int*>(est + 1);
    flags[0] = K->reorth;
    flags[1] = (hn == 0.0 || den == 0.0 || !isfinite(hn)) ? 1 : 0;
  }
  __syncthreads();
  for (int q = threadIdx.x; q <= j + 1; q += blockDim.x) K->H[q * mm + j] = col[q];
}

// V_slot = (w - sum_{i<k} h2_i V_i) / |w| with the second pass's correction only where the DGKS
// test asked for it (K->reorth), and the next operator input z = dinv V_slot from the stored
// value.  One fused multiply-add per basis element, chained on the element's value of w (no
// partial sums to add up afterwards: float64 adds are scarce on this GPU); the element's
// values of up to UPB basis vectors are loaded ahead of the chain.
constexpr int UPB = 32;
// The last CTA takes the Givens step instead (column k - 1).
__global__ void __launch_bounds__(VB, 2) upd_store_kernel(const double* __restrict__ w, double* V, int M1, int k, KryDev* K,
                                                          int64_t n, const double* __restrict__ dinv,
                                                          double* __restrict__ z, int mm, double* est) {
  if (blockIdx.x == gridDim.x - 1) {
    givens_step(K, k - 1, mm, est);
    return;
  }
  __shared__ double nh[MMAX + 2], s_sh;
  const bool second = K->reorth != 0;
  if (threadIdx.x == 0) s_sh = K->nrm_fin > 0.0 ? 1.0 / K->nrm_fin : 0.0;
  if (second)
    for (int i = threadIdx.x; i < k; i += VB) nh[i] = -K->h2[i];
  __syncthreads();
  const double scale = s_sh;
  const int64_t nch = (n + CH - 1) / CH;
  for (int64_t c = blockIdx.x; c < nch; c += gridDim.x - 1) {
    const int64_t j = c * CH + threadIdx.x;
    if (j >= n) break;
    double* blk = V + c * (int64_t)M1 * CH + threadIdx.x;
    double s = w[j];
    if (second) {
      for (int i0 = 0; i0 < k; i0 += UPB) {
        const int cnt = min(UPB, k - i0);
        double v[UPB];
#pragma unroll
        for (int u = 0; u < UPB; ++u) v[u] = u < cnt ? blk[(int64_t)(i0 + u) * CH] : 0.0;
#pragma unroll
        for (int u = 0; u < UPB; ++u) {
          if (u >= cnt) break;
          s = fma(nh[i0 + u], v[u], s);
        }
      }
    }
    s *= scale;
    blk[(int64_t)k * CH] = s;
    if (z) z[j] = dinv[j] * s;
  }
}

// The same for the float32 basis, laid out as mdot4_kernel: a CTA works on four chunks at a
// time, a thread on four adjacent elements (one float4 per basis vector, two double2 of w); z is the
// float32 operator's increment.
__global__ void __launch_bounds__(VB) upd_store4_kernel(const double* __restrict__ w, float* V, int M1, int k, KryDev* K,
                                                        int64_t n, const double* __restrict__ dinv,
                                                        float* __restrict__ z, int mm, double* est) {
  if (blockIdx.x == gridDim.x - 1) {
    givens_step(K, k - 1, mm, est);
    return;
  }
  __shared__ float hs[MMAX + 2];
  __shared__ double s_sh;
  const bool second = K->reorth != 0;
  if (threadIdx.x == 0) s_sh = K->nrm_fin > 0.0 ? 1.0 / K->nrm_fin : 0.0;
  if (second)
    for (int i = threadIdx.x; i < k; i += VB) hs[i] = (float)K->h2[i];
  __syncthreads();
  // 1 / |w| in two floats: rounded to one, its error would be common to all of V_k
  const float sh = (float)s_sh, sl = (float)(s_sh - (double)sh);
  auto scaled = [&](float x) { return fmaf(x, sh, x * sl); };
  const int64_t nch = (n + CH - 1) / CH;
  const int sub = threadIdx.x >> 6;
  const int e0 = (threadIdx.x & 63) * 4;
  for (int64_t c = (int64_t)blockIdx.x * 4 + sub; c < nch; c += (int64_t)(gridDim.x - 1) * 4) {
    const int64_t j = c * CH + e0;
    if (j >= n) break;
    float* blk = V + c * (int64_t)M1 * CH + e0;
    if (j + 4 <= n) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (second) {
        int i = 0;
#pragma unroll 4
        for (; i + 2 <= k; i += 2) {
          const float4 v0 = *reinterpret_cast<const float4*>(blk + i * CH);
          const float4 v1 = *reinterpret_cast<const float4*>(blk + (i + 1) * CH);
          a.x += hs[i] * v0.x; a.y += hs[i] * v0.y; a.z += hs[i] * v0.z; a.w += hs[i] * v0.w;
          b.x += hs[i + 1] * v1.x; b.y += hs[i + 1] * v1.y; b.z += hs[i + 1] * v1.z; b.w += hs[i + 1] * v1.w;
        }
        if (i < k) {
          const float4 v0 = *reinterpret_cast<const float4*>(blk + i * CH);
          a.x += hs[i] * v0.x; a.y += hs[i] * v0.y; a.z += hs[i] * v0.z; a.w += hs[i] * v0.w;
        }
      }
      const double2 w01 = *reinterpret_cast<const double2*>(w + j);
      const double2 w23 = *reinterpret_cast<const double2*>(w + j + 2);
      float4 v;
      v.x = scaled((float)w01.x - (a.x + b.x));
      v.y = scaled((float)w01.y - (a.y + b.y));
      v.z = scaled((float)w23.x - (a.z + b.z));
      v.w = scaled((float)w23.y - (a.w + b.w));
      *reinterpret_cast<float4*>(blk + (int64_t)k * CH) = v;
      if (z) {
        const double2 d01 = *reinterpret_cast<const double2*>(dinv + j), d23 = *reinterpret_cast<const double2*>(dinv + j + 2);
        *reinterpret_cast<float4*>(z + j) =
            make_float4((float)d01.x * v.x, (float)d01.y * v.y, (float)d23.x * v.z, (float)d23.y * v.w);
      }
    } else {
      for (int e = 0; e < 4 && j + e < n; ++e) {
        float acc = 0.f;
        if (second)
          for (int i = 0; i < k; ++i) acc += hs[i] * blk[i * CH + e];
        const float v = scaled((float)w[j + e] - acc);
        blk[(int64_t)k * CH + e] = v;
        if (z) z[j + e] = (float)dinv[j + e] * v;
      }
    }
  }
}

// Pass-1 update fused with the pass-2 projections: w' = w - sum_{i<k} h_i V_i, the
// partial |w'|^2 and the partial V_i . w' (i < k) of the updated vector, from one read
// of the basis: a thread keeps the k basis values of its element in registers, uses
// them for the update and then for the projections, and accumulates the projections
// in its own shared-memory column; the columns are added once at the end (float64).
// KMAX: k rounded up to a multiple of 8.  Rows of part: i < k the projections, row k
// the norm; part[row * G + cta].
template <int KMAX>
__global__ void __launch_bounds__(UDT) upd_dot_kernel(double* __restrict__ w, const double* __restrict__ V, int M1, int k,
                                                      int64_t n, double* part, KryDev* K) {
  extern __shared__ __align__(16) unsigned char upd_smem[];
  double* sacc = reinterpret_cast<double*>(upd_smem);  // [KMAX + 1][UDT]
  __shared__ double nhs[KMAX];
  const int t = threadIdx.x, NT = blockDim.x;
  for (int i = t; i < KMAX; i += NT) nhs[i] = i < k ? -K->h[i] : 0.0;
  for (int i = 0; i <= KMAX; ++i) sacc[i * UDT + t] = 0.0;
  __syncthreads();
  const int G = gridDim.x;
  const int64_t nu = (n + HCH - 1) / HCH;
  double nrm = 0.0;
  for (int64_t u = blockIdx.x + (int64_t)G * (t / HCH); u < nu; u += (int64_t)G * (blockDim.x / HCH)) {
    const int64_t j = u * HCH + t % HCH;
    if (j >= n) break;
    const double* blk = V + (u >> 1) * (int64_t)M1 * CH + (u & 1) * HCH + t % HCH;
    double v[KMAX];
#pragma unroll
    for (int i = 0; i < KMAX; ++i) v[i] = i < k ? blk[i * CH] : 0.0;
    // one fused multiply-add per basis value, chained on w's value, and none for the
    // padding past k (float64 operations are what this kernel is bound by)
    double ww = w[j];
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i >= k) break;
      ww = fma(nhs[i], v[i], ww);
    }
    w[j] = ww;
    nrm = fma(ww, ww, nrm);
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i >= k) break;
      sacc[i * UDT + t] = fma(v[i], ww, sacc[i * UDT + t]);
    }
  }
  sacc[KMAX * UDT + t] = nrm;
  __syncthreads();
  // one warp per row, lanes on consecutive columns, then a shuffle tree
  const int lane = t & 31;
  for (int i = t >> 5; i <= k; i += NT >> 5) {
    const double* rp = sacc + (i < k ? i : KMAX) * UDT;
    double s = 0.0;
#pragma unroll 4
    for (int c = 0; c < NT >> 5; ++c) s += rp[lane + 32 * c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) part[(int64_t)i * G + blockIdx.x] = s;
  }
  if (last_cta(&K->counter, gridDim.x)) orth_step(part, G, K, k - 1, w, V, M1, n);
}

// The fused update for the float32 basis: a thread takes two adjacent elements of each
// chunk (one float2 per basis vector, one double2 of w), so a warp moves as many bytes
// per load as with a float64 basis, and keeps the projections in registers.  Elements at or past n
// are never read.
template <int KMAX>
constexpr int ud2_threads() { return KMAX <= 32 ? 384 : 256; }
template <int KMAX>
__global__ void __launch_bounds__(ud2_threads<KMAX>()) upd_dot2_kernel(double* __restrict__ w, const float* __restrict__ V,
                                                                       int M1, int k, int64_t n, double* part, KryDev* K) {
  constexpr int NT = ud2_threads<KMAX>();
  __shared__ float nhs[KMAX];
  const int t = threadIdx.x;
  for (int i = t; i < KMAX; i += NT) nhs[i] = i < k ? -(float)K->h[i] : 0.f;
  __syncthreads();
  const int G = gridDim.x;
  const int64_t nch = (n + CH - 1) / CH;
  const int e0 = 2 * (t & 127);
  float acc[KMAX + 1];
#pragma unroll
  for (int i = 0; i <= KMAX; ++i) acc[i] = 0.f;
  for (int64_t c = blockIdx.x + (int64_t)G * (t >> 7); c < nch; c += (int64_t)G * (NT / 128)) {
    const int64_t j = c * CH + e0;
    if (j >= n) break;
    const bool pair = j + 2 <= n;
    const float* blk = V + c * (int64_t)M1 * CH + e0;
    float2 v[KMAX];
    if (pair) {
#pragma unroll
      for (int i = 0; i < KMAX; ++i) v[i] = i < k ? *reinterpret_cast<const float2*>(blk + i * CH) : make_float2(0.f, 0.f);
    } else {
#pragma unroll
      for (int i = 0; i < KMAX; ++i) v[i] = make_float2(i < k ? blk[i * CH] : 0.f, 0.f);
    }
    float sx0 = 0.f, sx1 = 0.f, sy0 = 0.f, sy1 = 0.f;
#pragma unroll
    for (int i = 0; i < KMAX; i += 2) {
      sx0 = fmaf(nhs[i], v[i].x, sx0);
      sx1 = fmaf(nhs[i + 1], v[i + 1].x, sx1);
      sy0 = fmaf(nhs[i], v[i].y, sy0);
      sy1 = fmaf(nhs[i + 1], v[i + 1].y, sy1);
    }
    float wx, wy = 0.f;
    if (pair) {
      const double2 wd = *reinterpret_cast<const double2*>(w + j);
      wx = (float)wd.x + (sx0 + sx1);
      wy = (float)wd.y + (sy0 + sy1);
      *reinterpret_cast<double2*>(w + j) = make_double2((double)wx, (double)wy);
    } else {
      wx = (float)w[j] + (sx0 + sx1);
      w[j] = (double)wx;
    }
    acc[KMAX] += wx * wx + wy * wy;
#pragma unroll
    for (int i = 0; i < KMAX; ++i) acc[i] += v[i].x * wx + v[i].y * wy;
  }
  // rows i < k the projections, row k the norm
  block_reduce_store_f<KMAX + 1, NT>(acc, k + 1, true, part + blockIdx.x, G);
  if (last_cta(&K->counter, gridDim.x)) orth_step(part, G, K, k - 1, w, V, M1, n);
}

template <int KMAX, typename VT>
static int launch_upd_dot(fsi_mesh* m, double* w, const VT* V, int M1, int k, int64_t n) {
  KryDev* K = static_cast<KryDev*>(m->kry_dev);
  if constexpr (sizeof(VT) == 4) {
    const int G = (int)std::max<int64_t>(1, std::min<int64_t>((n + CH - 1) / CH, KG));
    upd_dot2_kernel<KMAX><<<G, ud2_threads<KMAX>(), 0, m->stream>>>(w, V, M1, k, n, m->partials_dot, K);
  } else {
    const ProjGrid g = pgrid(n);
    const size_t smem = sizeof(double) * (size_t)(KMAX + 1) * UDT;
    if (int rc = ensure_smem_attr(reinterpret_cast<const void*>(&upd_dot_kernel<KMAX>), smem)) return rc;
    upd_dot_kernel<KMAX><<<g.ctas, g.threads, smem, m->stream>>>(w, V, M1, k, n, m->partials_dot, K);
  }
  return FSI_OK;
}

template <typename VT>
static int upd_dot(fsi_mesh* m, double* w, const VT* V, int M1, int k, int64_t n) {
  switch ((k + 7) / 8) {
    case 1: return launch_upd_dot<8>(m, w, V, M1, k, n);
    case 2: return launch_upd_dot<16>(m, w, V, M1, k, n);
    case 3: return launch_upd_dot<24>(m, w, V, M1, k, n);
    case 4: return launch_upd_dot<32>(m, w, V, M1, k, n);
    case 5: return launch_upd_dot<40>(m, w, V, M1, k, n);
    case 6: return launch_upd_dot<48>(m, w, V, M1, k, n);
    case 7: return launch_upd_dot<56>(m, w, V, M1, k, n);
    default: return launch_upd_dot<64>(m, w, V, M1, k, n);
  }
}

// V_0 = r / |r|, |r|^2 = *n2; with z, also the next operator input z = dinv V_0 from the stored value
// (the float32 operator's increment when VT is float)
template <typename VT>
__global__ void store_first(VT* __restrict__ V, int M1, const double* __restrict__ r, const double* n2, int64_t n,
                            const double* __restrict__ dinv, VT* __restrict__ z) {
  // the scale once per CTA: float64 division and square root are slow on this GPU
  __shared__ double s_sh;
  if (threadIdx.x == 0) s_sh = 1.0 / sqrt(*n2);
  __syncthreads();
  const double s = s_sh;
  // one chunk of CH = VB elements per CTA pass
  const int64_t nch = (n + CH - 1) / CH;
  for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
    const int64_t j = c * CH + threadIdx.x;
    if (j >= n) continue;
    const VT v = (VT)(r[j] * s);
    V[c * (int64_t)M1 * CH + threadIdx.x] = v;
    if (z) {
      if constexpr (sizeof(VT) == 4) z[j] = (float)dinv[j] * v;
      else z[j] = dinv[j] * v;
    }
  }
}

// z = dinv * V_slot (ZT float: the float32 operator's increment, written directly)
template <typename VT, typename ZT>
__global__ void precond_kernel(const VT* __restrict__ V, int M1, int slot, const double* __restrict__ dinv,
                               ZT* __restrict__ z, int64_t n) {
  const int64_t nch = (n + CH - 1) / CH;
  for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
    const int64_t j = c * CH + threadIdx.x;
    if (j < n) z[j] = (ZT)(dinv[j] * (double)V[c * (int64_t)M1 * CH + (int64_t)slot * CH + threadIdx.x]);
  }
}

// x += dinv * sum_i y_i V_i
__global__ void __launch_bounds__(VB) combine_kernel(double* __restrict__ x, const double* __restrict__ dinv,
                                                     const double* __restrict__ V, int M1, int k,
                                                     const KryDev* __restrict__ K, int64_t n) {
  __shared__ double ys[MMAX];
  for (int i = threadIdx.x; i < k; i += VB) ys[i] = K->y[i];
  __syncthreads();
  const int64_t nch = (n + CH - 1) / CH;
  for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
    const int64_t j = c * CH + threadIdx.x;
    if (j >= n) continue;
    x[j] += dinv[j] * lin_comb_chunk<double>(ys, V + c * (int64_t)M1 * CH + threadIdx.x, k);
  }
}

// the same from the float32 basis, four adjacent elements a thread (upd_store4_kernel's layout), each entry in
// eight sums as lin_comb_chunk has it (30 vectors: 6.3e-8 off, 9.3e-8 in two sums)
__global__ void __launch_bounds__(VB) combine4_kernel(double* __restrict__ x, const double* __restrict__ dinv,
                                                      const float* __restrict__ V, int M1, int k,
                                                      const KryDev* __restrict__ K, int64_t n) {
  __shared__ float ys[MMAX + 8];
  for (int i = threadIdx.x; i < k + 8; i += VB) ys[i] = i < k ? (float)K->y[i] : 0.f;
  __syncthreads();
  const int64_t nch = (n + CH - 1) / CH;
  const int sub = threadIdx.x >> 6, e0 = (threadIdx.x & 63) * 4;
  for (int64_t c = (int64_t)blockIdx.x * 4 + sub; c < nch; c += (int64_t)gridDim.x * 4) {
    const int64_t j = c * CH + e0;
    if (j >= n) break;
    const float* blk = V + c * (int64_t)M1 * CH + e0;
    if (j + 4 <= n) {
      float4 p[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) p[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int i0 = 0; i0 < k; i0 += 8) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          v[u] = i0 + u < k ? *reinterpret_cast<const float4*>(blk + (i0 + u) * CH) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float y = ys[i0 + u];
          p[u].x = fmaf(y, v[u].x, p[u].x);
          p[u].y = fmaf(y, v[u].y, p[u].y);
          p[u].z = fmaf(y, v[u].z, p[u].z);
          p[u].w = fmaf(y, v[u].w, p[u].w);
        }
      }
#pragma unroll
      for (int h = 4; h > 0; h >>= 1)
#pragma unroll
        for (int u = 0; u < h; ++u) {
          p[u].x += p[u + h].x;
          p[u].y += p[u + h].y;
          p[u].z += p[u + h].z;
          p[u].w += p[u + h].w;
        }
      x[j] += dinv[j] * (double)p[0].x;
      x[j + 1] += dinv[j + 1] * (double)p[0].y;
      x[j + 2] += dinv[j + 2] * (double)p[0].z;
      x[j + 3] += dinv[j + 3] * (double)p[0].w;
    } else {
      for (int e = 0; e < 4 && j + e < n; ++e) x[j + e] += dinv[j + e] * (double)lin_comb_chunk<float>(ys, blk + e, k);
    }
  }
}

// z = V_slot (contiguous float64 copy of one basis vector)
template <typename VT>
__global__ void extract_kernel(const VT* __restrict__ V, int M1, int slot, double* __restrict__ z, int64_t n) {
  const int64_t nch = (n + CH - 1) / CH;
  for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
    const int64_t j = c * CH + threadIdx.x;
    if (j < n) z[j] = (double)V[c * (int64_t)M1 * CH + (int64_t)slot * CH + threadIdx.x];
  }
}

// x += sum_i y_i Z_i (flexible GMRES: the stored preconditioned directions)
__global__ void __launch_bounds__(VB) zcombine_kernel(double* __restrict__ x, const double* __restrict__ Z, int k,
                                                      const KryDev* K, int64_t n) {
  __shared__ double ys[MMAX];
  for (int i = threadIdx.x; i < k; i += VB) ys[i] = K->y[i];
  __syncthreads();
  for (int64_t j = blockIdx.x * (int64_t)VB + threadIdx.x; j < n; j += (int64_t)gridDim.x * VB) {
    double s = 0.0;
    for (int i = 0; i < k; ++i) s += ys[i] * Z[(int64_t)i * n + j];
    x[j] += s;
  }
}

// --------------------------------------------------------- small device kernels
// y = R^{-1} g for the first jend columns: the diagonal's reciprocals by all threads (a float64
// division takes most of a microsecond here), then one warp, the entries above the current one
// updated by column in shared memory
__global__ void lsq_kernel(KryDev* K, int jend, int mm) {
  __shared__ double R[MMAX * MMAX], g[MMAX], inv[MMAX];
  for (int q = threadIdx.x; q < jend * jend; q += blockDim.x) R[q] = K->H[(q / jend) * mm + q % jend];
  for (int q = threadIdx.x; q < jend; q += blockDim.x) {
    g[q] = K->g[q];
    const double d = K->H[q * mm + q];
    inv[q] = d != 0.0 ? 1.0 / d : 0.0;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  for (int i = jend - 1; i >= 0; --i) {
    const double y = g[i] * inv[i];
    if (threadIdx.x == 0) K->y[i] = y;
    __syncwarp();
    for (int q = threadIdx.x; q < i; q += 32) g[q] = fma(-R[q * jend + i], y, g[q]);
    __syncwarp();
  }
}

// start of a cycle: g = (|r|, 0, ...)
__global__ void cycle_start(KryDev* K, const double* rn2, int mm) {
  const double b = sqrt(*rn2);
  for (int i = 0; i <= mm; ++i) K->g[i] = 0.0;
  K->g[0] = b;
  K->nrm_fin = b;
}

// --------------------------------------------------------- contiguous vectors
// part[cta] = partial of a . b over a contiguous range
__global__ void __launch_bounds__(VB) dot_kernel(const double* __restrict__ a, const double* __restrict__ b, int64_t n,
                                                 double* part) {
  const int G = gridDim.x;
  const int64_t per = (n + G - 1) / G;
  const int64_t lo = blockIdx.x * per, hi = min(n, lo + per);
  double acc[1] = {0.0};
  for (int64_t j = lo + threadIdx.x; j < hi; j += VB) acc[0] += a[j] * b[j];
  block_reduce_store<1>(acc, 1, part + blockIdx.x, 1);
}
// r = b - t and the partial |r|^2 (the same partition)
__global__ void __launch_bounds__(VB) resid_kernel(const double* __restrict__ b, const double* __restrict__ t,
                                                   double* __restrict__ r, int64_t n, double* part) {
  const int G = gridDim.x;
  const int64_t per = (n + G - 1) / G;
  const int64_t lo = blockIdx.x * per, hi = min(n, lo + per);
  double acc[1] = {0.0};
  for (int64_t j = lo + threadIdx.x; j < hi; j += VB) {
    const double v = b[j] - t[j];
    r[j] = v;
    acc[0] += v * v;
  }
  block_reduce_store<1>(acc, 1, part + blockIdx.x, 1);
}
__global__ void axpby_kernel(double a, const double* __restrict__ x, double b, double* __restrict__ y, int64_t n) {
  for (int64_t j = blockIdx.x * (int64_t)VB + threadIdx.x; j < n; j += (int64_t)gridDim.x * VB) y[j] = a * x[j] + b * y[j];
}
__global__ void mul_kernel(const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ y, int64_t n) {
  for (int64_t j = blockIdx.x * (int64_t)VB + threadIdx.x; j < n; j += (int64_t)gridDim.x * VB) y[j] = a[j] * b[j];
}
__global__ void recip_kernel(const double* __restrict__ a, double* __restrict__ y, int64_t n) {
  for (int64_t j = blockIdx.x * (int64_t)VB + threadIdx.x; j < n; j += (int64_t)gridDim.x * VB) {
    const double v = a[j];
    y[j] = v != 0.0 ? 1.0 / v : 1.0;
  }
}
__global__ void fill_kernel(double* y, double v, int64_t n) {
  for (int64_t j = blockIdx.x * (int64_t)VB + threadIdx.x; j < n; j += (int64_t)gridDim.x * VB) y[j] = v;
}

// ---------------------------------------------------------------- host helpers
static void launch_mdot(fsi_mesh* m, const double* V, int M1, int k, const double* w, int64_t n, KryDev* K) {
  // one group more than the full ones: it holds the rest, or only w . w
  const dim3 grid(cgrid((n + CH - 1) / CH), k / DCH + 1);
  switch (k % DCH) {
    case 0: mdot_kernel<0><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 1: mdot_kernel<1><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 2: mdot_kernel<2><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 3: mdot_kernel<3><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 4: mdot_kernel<4><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 5: mdot_kernel<5><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 6: mdot_kernel<6><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 7: mdot_kernel<7><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 8: mdot_kernel<8><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 9: mdot_kernel<9><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 10: mdot_kernel<10><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 11: mdot_kernel<11><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 12: mdot_kernel<12><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 13: mdot_kernel<13><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    case 14: mdot_kernel<14><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
    default: mdot_kernel<15><<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K); break;
  }
}
static void launch_mdot(fsi_mesh* m, const float* V, int M1, int k, const double* w, int64_t n, KryDev* K) {
  const dim3 grid(cgrid4((n + CH - 1) / CH), k / DCH + 1);
  mdot4_kernel<<<grid, VB, 0, m->stream>>>(V, M1, k, w, n, m->partials_dot, K);
}

// K->h[0..k) = V_i . w for the basis slots i < k, K->h[k] = w . w
template <typename VT>
static int basis_dots(fsi_mesh* m, const VT* V, int M1, int k, const double* w, int64_t n, KryDev* K) {
  FSI_LAUNCH(m, P_KRY_DOT, launch_mdot(m, V, M1, k, w, n, K));
  return FSI_OK;
}

// per-CTA partial sums of the reductions (fixed size, allocated on first use)
static int ensure_partials(fsi_mesh* m) {
  if (m->partials_dot) return FSI_OK;
  FSI_CUDA(cudaMalloc(&m->partials_dot, sizeof(double) * (size_t)(MMAX + 2 + DCH) * 152 * 4));
  return FSI_OK;
}

static int dot_dev(fsi_mesh* m, const double* a, const double* b, int64_t n, double* out) {
  int rc = ensure_partials(m);
  if (rc) return rc;
  const int G = vgrid(n);
  FSI_LAUNCH(m, P_KRY_DOT, dot_kernel<<<G, VB, 0, m->stream>>>(a, b, n, m->partials_dot));
  FSI_LAUNCH(m, P_KRY_DOT, sum_partials<<<1, VB, 0, m->stream>>>(m->partials_dot, G, out));
  return FSI_OK;
}

int vec_dot(fsi_mesh* m, const double* a, const double* b, int64_t n, double* out_host) {
  int rc = dot_dev(m, a, b, n, m->red);
  if (rc) return rc;
  FSI_CUDA(cudaMemcpyAsync(m->red_host, m->red, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  FSI_CUDA(cudaStreamSynchronize(m->stream));
  *out_host = m->red_host[0];
  return FSI_OK;
}

int vec_axpy(fsi_mesh* m, double a, const double* x, double* y, int64_t n) {
  FSI_LAUNCH(m, P_KRYLOV, axpby_kernel<<<vgrid(n), VB, 0, m->stream>>>(a, x, 1.0, y, n));
  return FSI_OK;
}
int vec_scale_copy(fsi_mesh* m, double a, const double* x, double* y, int64_t n) {
  FSI_LAUNCH(m, P_KRYLOV, axpby_kernel<<<vgrid(n), VB, 0, m->stream>>>(a, x, 0.0, y, n));
  return FSI_OK;
}
int vec_mul(fsi_mesh* m, const double* a, const double* b, double* y, int64_t n) {
  FSI_LAUNCH(m, P_KRYLOV, mul_kernel<<<vgrid(n), VB, 0, m->stream>>>(a, b, y, n));
  return FSI_OK;
}
int vec_recip(fsi_mesh* m, const double* a, double* y, int64_t n) {
  FSI_LAUNCH(m, P_KRYLOV, recip_kernel<<<vgrid(n), VB, 0, m->stream>>>(a, y, n));
  return FSI_OK;
}

// basis: nch chunks x (mx + 1) slots x CH; wk: 7 contiguous work vectors
static int ensure_krylov(fsi_mesh* m, int64_t n, int mm) {
  if (m->kry_n >= n && m->kry_m >= mm && m->kry_dev) return FSI_OK;
  const int64_t nn = std::max(n, m->kry_n);
  const int mx = std::max(mm, m->kry_m);
  cudaFree(m->V);
  cudaFree(m->wk);
  cudaFree(m->dinv);
  m->V = m->wk = m->dinv = nullptr;
  const int64_t nch = (nn + CH - 1) / CH;
  FSI_CUDA(cudaMalloc(&m->V, sizeof(double) * (size_t)nch * (mx + 1) * CH));
  FSI_CUDA(cudaMalloc(&m->wk, sizeof(double) * (size_t)7 * nn));
  FSI_CUDA(cudaMalloc(&m->dinv, sizeof(double) * (size_t)nn));
  if (int rc = ensure_partials(m)) return rc;
  if (!m->kry_dev) {
    FSI_CUDA(cudaMalloc(&m->kry_dev, sizeof(KryDev)));
    FSI_CUDA(cudaMemset(m->kry_dev, 0, sizeof(KryDev)));
    FSI_CUDA(cudaMallocHost(&m->kry_est, sizeof(double) * 3 * (MMAX + 1)));
    m->kry_ev.resize(MMAX + 1);
    for (auto& e : m->kry_ev) FSI_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  }
  m->kry_n = nn;
  m->kry_m = mx;
  return FSI_OK;
}

// One GMRES(m) solve A x = b from x = 0 with A = the block operator (flags) and the
// right preconditioner diag(dinv).  VT: the basis type (float exactly when the operator
// is the float32 one, i.e. the inner solves of iterative refinement).
template <typename VT>
static int gmres_core_t(fsi_mesh* m, const BlockInfo& blk, const double* b, double* x, int mm, double rtol,
                        int max_iter, unsigned flags, int* iters, int* restarts, double* rel_out, int* stalled,
                        fsi_pc* pc, fsi_pc* harvest) {
  constexpr bool F32 = sizeof(VT) == 4;
  const bool alternate = (flags & FSI_PC_ALTERNATE) != 0;
  const bool stall_stop = (flags & FSI_NO_STALL_STOP) == 0;
  flags &= ~(FSI_PC_ALTERNATE | FSI_NO_STALL_STOP);
  const int64_t n = blk.n;
  const int M1 = m->kry_m + 1;
  const int G = vgrid(n);
  VT* V = reinterpret_cast<VT*>(m->V);  // the float basis reuses the float64 allocation
  double* r = m->wk;
  double* z = m->wk + n;
  double* t = m->wk + 2 * n;
  double* w = m->wk + 6 * n;
  KryDev* K = static_cast<KryDev*>(m->kry_dev);
  double* est = m->kry_est;  // pinned, 3 slots per step: the estimate, then the reorth and breakdown ints
  FSI_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n, m->stream));
  double bnorm2;
  int rc = vec_dot(m, b, b, n, &bnorm2);
  if (rc) return rc;
  if (!std::isfinite(bnorm2)) return set_error(FSI_ENAN, "GMRES: right-hand side is not finite");
  const double bnorm = std::sqrt(bnorm2);
  *rel_out = 0.0;
  *stalled = 0;
  if (bnorm == 0.0) return FSI_OK;
  FSI_CUDA(cudaMemcpyAsync(&K->bnorm, &bnorm, sizeof(double), cudaMemcpyHostToDevice, m->stream));
  FSI_CUDA(cudaMemcpyAsync(r, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, m->stream));
  double rel = 1.0, cycle_rel = 1.0;
  bool first_cycle = true;
  int n_arnoldi_pairs = 0;
  if ((rc = dot_dev(m, r, r, n, m->red))) return rc;
  while (true) {
    // |r|^2 on the device (m->red); the host needs it for the stopping and stall tests
    FSI_CUDA(cudaMemcpyAsync(m->red_host, m->red, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    FSI_CUDA(cudaStreamSynchronize(m->stream));
    const double beta2 = m->red_host[0];
    if (!std::isfinite(beta2)) return set_error(FSI_ENAN, "GMRES: residual is not finite");
    rel = std::sqrt(beta2) / bnorm;
    if (rel <= rtol || *iters >= max_iter) break;
    if (stall_stop && !first_cycle && rel > 0.99 * cycle_rel) {
      *stalled = 1;
      break;
    }
    first_cycle = false;
    cycle_rel = rel;
    FSI_LAUNCH(m, P_KRY_SMALL, cycle_start<<<1, 1, 0, m->stream>>>(K, m->red, mm));
    // the operator input of the plain (Jacobi) steps: z = dinv V_j, written with V_j
    VT* zn = pc ? nullptr : (F32 ? reinterpret_cast<VT*>(m->dx32) : reinterpret_cast<VT*>(z));
    FSI_LAUNCH(m, P_KRYLOV, store_first<VT><<<chunk_grid(n), VB, 0, m->stream>>>(V, M1, r, m->red, n, m->dinv, zn));
    int jend = 0, enq = 0;
    bool done = false;
    const int jmax = std::min(mm, max_iter - *iters);
    const double vb = (double)sizeof(VT) * (double)n;  // bytes of one basis vector
    const double wb = 8.0 * (double)n;                 // bytes of the float64 work vector
    for (int j = 0; j < jmax && !done; ++j) {
      if (pc) {  // flexible GMRES: z_j = M(v_j), |v_j| = 1
        double* zj = m->Z + (int64_t)j * n;
        if (alternate && (j & 1)) {
          // every other direction is the plain Jacobi one: the least-squares step then
          // weights network and Jacobi directions separately
          FSI_LAUNCH(m, P_KRYLOV, (precond_kernel<VT, double><<<G, VB, 0, m->stream>>>(V, M1, j, m->dinv, zj, n)));
        } else {
          FSI_LAUNCH(m, P_KRYLOV, extract_kernel<VT><<<G, VB, 0, m->stream>>>(V, M1, j, t, n));
          if ((rc = pcn::apply(pc, t, 1.0, m->dinv, zj))) return rc;
        }
        if ((rc = op_jvp(m, blk, zj, w, flags))) return rc;
      } else {
        // z = dinv V_j was written with V_j (the float32 increment straight into the
        // operator's input buffer)
        if (F32) {
          if ((rc = op_jvp(m, blk, nullptr, w, flags | OP_DX32_READY))) return rc;
        } else {
          if ((rc = op_jvp(m, blk, z, w, flags))) return rc;
        }
        // broadband training pairs: A z_j = w exactly for the operator just applied
        // (harvesting solves run with the float64 basis)
        if (!F32 && harvest && j % 8 == 4 && n_arnoldi_pairs < 8) {
          if ((rc = pcn::add_pair(harvest, w, nullptr, z, nullptr, m->dinv))) return rc;
          ++n_arnoldi_pairs;
        }
      }
      // pass 1: h = V^T w and |w|^2 (slot j+1 of h)
      if ((rc = basis_dots(m, V, M1, j + 1, w, n, K))) return rc;
      // pass-1 update fused with the pass-2 projections of the updated vector, then the DGKS test
      FSI_LAUNCH(m, P_KRY_UPD, rc = upd_dot<VT>(m, w, V, M1, j + 1, n));
      if (rc) return rc;
      prof_bytes(m, P_KRY_DOT, (j + 1) * vb + wb);      // j+1 basis vectors and w read once
      prof_bytes(m, P_KRY_UPD, (j + 1) * vb + 2 * wb);  // j+1 basis vectors and w read, w written
      // the pass-2 update (only when the DGKS test asked for it), the new basis vector and the next
      // input; in its last CTA the Givens step and the estimate
      if constexpr (F32) {
        FSI_LAUNCH(m, P_KRY_UPD, upd_store4_kernel<<<upd_grid(n, 4) + 1, VB, 0, m->stream>>>(
                                     w, reinterpret_cast<float*>(V), M1, j + 1, K, n, m->dinv,
                                     reinterpret_cast<float*>(zn), mm, est + 3 * j));
      } else {
        FSI_LAUNCH(m, P_KRY_UPD, upd_store_kernel<<<upd_grid(n, 1) + 1, VB, 0, m->stream>>>(
                                     w, reinterpret_cast<double*>(V), M1, j + 1, K, n, m->dinv,
                                     reinterpret_cast<double*>(zn), mm, est + 3 * j));
      }
      FSI_CUDA(cudaEventRecord(m->kry_ev[j], m->stream));
      prof_bytes(m, P_KRY_UPD, 2 * wb + 2 * vb);  // w and dinv read, V_{j+1} and z written
      ++*iters;
      jend = j + 1;
      enq = j + 1;
      // look at the previous step while this one runs
      if (j >= 1) {
        FSI_CUDA(cudaEventSynchronize(m->kry_ev[j - 1]));
        int bd = 0;
        memcpy(&bd, reinterpret_cast<const char*>(est + 3 * (j - 1)) + sizeof(double) + sizeof(int), sizeof(int));
        const double e = est[3 * (j - 1)];
        if (!std::isfinite(e)) return set_error(FSI_ENAN, "GMRES: Arnoldi vector is not finite");
        if (e <= rtol || bd) {
          jend = j;  // step j was computed for nothing
          done = true;
        }
      }
    }
    FSI_CUDA(cudaEventSynchronize(m->kry_ev[enq - 1]));
    if (!done && !std::isfinite(est[3 * (jend - 1)])) return set_error(FSI_ENAN, "GMRES: Arnoldi vector is not finite");
    for (int j = 0; j < enq; ++j) {  // the second passes that ran
      int ro = 0;
      memcpy(&ro, reinterpret_cast<const char*>(est + 3 * j) + sizeof(double), sizeof(int));
      if (ro) prof_bytes(m, P_KRY_UPD, (j + 1) * vb);
    }
    FSI_LAUNCH(m, P_KRY_SMALL, lsq_kernel<<<1, VB, 0, m->stream>>>(K, jend, mm));
    if (pc) {
      FSI_LAUNCH(m, P_KRYLOV, zcombine_kernel<<<G, VB, 0, m->stream>>>(x, m->Z, jend, K, n));
    } else if constexpr (F32) {
      FSI_LAUNCH(m, P_KRYLOV, combine4_kernel<<<upd_grid(n, 4), VB, 0, m->stream>>>(x, m->dinv, V, M1, jend, K, n));
    } else {
      FSI_LAUNCH(m, P_KRYLOV, combine_kernel<<<upd_grid(n, 1), VB, 0, m->stream>>>(x, m->dinv, V, M1, jend, K, n));
    }
    // true residual r = b - A x
    if ((rc = op_jvp(m, blk, x, t, flags))) return rc;
    FSI_LAUNCH(m, P_KRYLOV, resid_kernel<<<G, VB, 0, m->stream>>>(b, t, r, n, m->partials_dot));
    FSI_LAUNCH(m, P_KRY_DOT, sum_partials<<<1, VB, 0, m->stream>>>(m->partials_dot, G, m->red));
    ++*restarts;
  }
  *rel_out = rel;
  return FSI_OK;
}

static int gmres_core(fsi_mesh* m, const BlockInfo& blk, const double* b, double* x, int mm, double rtol,
                      int max_iter, unsigned flags, int* iters, int* restarts, double* rel_out, int* stalled,
                      fsi_pc* pc = nullptr, fsi_pc* harvest = nullptr) {
  // harvesting solves keep the float64 basis: their Arnoldi pairs and refinement
  // checkpoints are the training data of the learned preconditioner
  if ((flags & FSI_FP32) && !harvest) {
    if (int rc = ensure_dx32(m)) return rc;
    return gmres_core_t<float>(m, blk, b, x, mm, rtol, max_iter, flags, iters, restarts, rel_out, stalled, pc,
                               harvest);
  }
  return gmres_core_t<double>(m, blk, b, x, mm, rtol, max_iter, flags, iters, restarts, rel_out, stalled, pc, harvest);
}

int gmres_solve(fsi_mesh* m, const BlockInfo& blk, const double* rhs, double* x, const fsi_solve_opts& o,
                fsi_solve_info* info) {
  const int mm = o.m;
  if (mm < 1 || mm > MMAX) return set_error(FSI_EINVAL, "GMRES: restart length must be in 1..64");
  const int64_t n = blk.n;
  int rc = ensure_krylov(m, n, mm);
  if (rc) return rc;
  const int64_t a0 = m->applies;
  // the learned preconditioner acts on the NS block only; other blocks use Jacobi
  fsi_pc* pc = (o.precond == FSI_PC_LEARNED && blk.kind == 0) ? m->pc : nullptr;
  if (o.precond == FSI_PC_LEARNED && blk.kind == 0 && !pc)
    return set_error(FSI_EINVAL, "GMRES: FSI_PC_LEARNED without an attached preconditioner (fsi_set_pc)");
  fsi_pc* harvest = ((o.flags & FSI_HARVEST) && blk.kind == 0 && m->pc && m->pc->cap > 0) ? m->pc : nullptr;
  unsigned opflags = o.flags & ~(FSI_HARVEST | FSI_PC_ALTERNATE | FSI_NO_STALL_STOP | FSI_PINNED_SOLVE | OP_DX32_READY |
                                 OP_REUSED);
  // a float64 solve that may take many products (one an iteration, one a cycle for the true residual)
  // assembles the operator before the first one (its diagonal comes with it)
  const int64_t products = o.max_iter + ((int64_t)o.max_iter + mm - 1) / mm;
  if (o.precision == FSI_PREC_FP64 && products > (blk.kind == 0 ? NSA_AFTER : STENCIL_AFTER)) opflags |= OP_REUSED;
  // read by the solver loop only: network/Jacobi alternation, and no stop on stagnation
  const unsigned alt = o.flags & (FSI_PC_ALTERNATE | FSI_NO_STALL_STOP);
  const bool stall_stop = (o.flags & FSI_NO_STALL_STOP) == 0;
  if (pc && (m->Z_n < n * mm || !m->Z)) {
    cudaFree(m->Z);
    m->Z = nullptr;
    FSI_CUDA(cudaMalloc(&m->Z, sizeof(double) * (size_t)(n * mm)));
    m->Z_n = n * mm;
  }
  if (harvest && (rc = pcn::ensure_checkpoints(harvest))) return rc;
  // Jacobi diagonal (also the learned preconditioner's scale), from the operator the
  // inner solves apply: a preconditioner's rounding does not reach the refined solution,
  // and the float64 diagonal costs as much as 20 float32 ones on this GPU
  if (o.precond == FSI_PC_JACOBI || o.precond == FSI_PC_LEARNED || harvest) {
    const unsigned dflags = o.precision == FSI_PREC_FP32_IR ? (opflags | FSI_FP32) : (opflags & ~FSI_FP32);
    if ((rc = op_diag(m, blk, m->wk + 3 * n, dflags))) return rc;
    if ((rc = vec_recip(m, m->wk + 3 * n, m->dinv, n))) return rc;
  }
  if (o.precond == FSI_PC_NONE) {
    FSI_LAUNCH(m, P_KRYLOV, fill_kernel<<<vgrid(n), VB, 0, m->stream>>>(m->dinv, 1.0, n));
  }
  fsi_solve_info inf{};
  double rel = 0.0;
  int nck = 0;  // harvest checkpoints recorded
  auto checkpoint = [&](const double* xk, const double* rk) -> int {
    if (!harvest || nck >= pcn::CKMAX) return FSI_OK;
    FSI_CUDA(cudaMemcpyAsync(harvest->ck + (int64_t)nck * n, xk, sizeof(double) * n, cudaMemcpyDeviceToDevice,
                             m->stream));
    FSI_CUDA(cudaMemcpyAsync(harvest->ck + (int64_t)(pcn::CKMAX + nck) * n, rk, sizeof(double) * n,
                             cudaMemcpyDeviceToDevice, m->stream));
    ++nck;
    return FSI_OK;
  };
  double* rfin = nullptr;  // final true residual (harvest)
  if (o.precision == FSI_PREC_FP64) {
    rc = gmres_core(m, blk, rhs, x, mm, o.rtol, o.max_iter, (opflags & ~FSI_FP32) | alt, &inf.iterations, &inf.restarts,
                    &rel, &inf.stalled, pc, pc ? nullptr : harvest);
    if (rc == FSI_ENAN && pc) {
      // the network produced non-finite directions (corrupted weights, overflow):
      // Jacobi GMRES solves from scratch
      inf.fallback = 1;
      pc = nullptr;
      rc = gmres_core(m, blk, rhs, x, mm, o.rtol, o.max_iter - inf.iterations,
                      (opflags & ~FSI_FP32) | (alt & FSI_NO_STALL_STOP),
                      &inf.iterations, &inf.restarts, &rel, &inf.stalled, nullptr, harvest);
    }
    if (rc) return rc;
    if (pc && rel > o.rtol && inf.iterations < o.max_iter) {
      // fallback: Jacobi GMRES on the remaining residual r = rhs - A x (in wk[0..n))
      double* d = m->wk + 4 * n;
      double* r = m->wk + 5 * n;
      FSI_CUDA(cudaMemcpyAsync(r, m->wk, sizeof(double) * n, cudaMemcpyDeviceToDevice, m->stream));
      double rel2;
      int st2 = 0;
      rc = gmres_core(m, blk, r, d, mm, o.rtol / std::max(rel, 1e-300), o.max_iter - inf.iterations,
                      (opflags & ~FSI_FP32) | (alt & FSI_NO_STALL_STOP), &inf.iterations, &inf.restarts, &rel2, &st2, nullptr);
      if (rc) return rc;
      if ((rc = vec_axpy(m, 1.0, d, x, n))) return rc;
      rel *= rel2;
      inf.stalled = st2;
      inf.fallback = 1;
    }
    rfin = m->wk;  // rhs - A x (the fallback's final residual is the same vector)
    if (harvest) {  // the one checkpoint x_0 = 0, r_0 = rhs
      FSI_CUDA(cudaMemsetAsync(harvest->ck, 0, sizeof(double) * n, m->stream));
      FSI_CUDA(cudaMemcpyAsync(harvest->ck + (int64_t)pcn::CKMAX * n, rhs, sizeof(double) * n,
                               cudaMemcpyDeviceToDevice, m->stream));
      nck = 1;
    }
  } else {
    // x = 0; r = rhs; repeat: solve A32 d = r; x += d; r = rhs - A64 x
    double* d = m->wk + 4 * n;
    double* r = m->wk + 5 * n;
    FSI_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n, m->stream));
    FSI_CUDA(cudaMemcpyAsync(r, rhs, sizeof(double) * n, cudaMemcpyDeviceToDevice, m->stream));
    double b2;
    if ((rc = vec_dot(m, rhs, rhs, n, &b2))) return rc;
    if (!std::isfinite(b2)) return set_error(FSI_ENAN, "IR: right-hand side is not finite");
    const double bnorm = std::sqrt(b2);
    rel = bnorm == 0.0 ? 0.0 : 1.0;
    fsi_pc* inner_pc = pc;
    for (int k = 0; k < std::max(1, o.ir_max) && rel > o.rtol; ++k) {
      if ((rc = checkpoint(x, r))) return rc;
      double inner_rel;
      int inner_stalled;
      rc = gmres_core(m, blk, r, d, mm, o.ir_inner_rtol, o.max_iter - inf.iterations, (opflags | FSI_FP32 | alt),
                      &inf.iterations, &inf.restarts, &inner_rel, &inner_stalled, inner_pc,
                      inner_pc ? nullptr : harvest);
      if (rc == FSI_ENAN && inner_pc) {
        // non-finite network directions: this refinement again, with Jacobi inner solves
        inner_pc = nullptr;
        inf.fallback = 1;
        --k;
        continue;
      }
      if (rc) return rc;
      if ((rc = vec_axpy(m, 1.0, d, x, n))) return rc;
      if ((rc = op_jvp(m, blk, x, d, opflags & ~FSI_FP32))) return rc;
      FSI_CUDA(cudaMemcpyAsync(r, rhs, sizeof(double) * n, cudaMemcpyDeviceToDevice, m->stream));
      if ((rc = vec_axpy(m, -1.0, d, r, n))) return rc;
      double r2;
      if ((rc = vec_dot(m, r, r, n, &r2))) return rc;
      if (!std::isfinite(r2)) return set_error(FSI_ENAN, "IR: residual is not finite");
      const double prev = rel;
      rel = bnorm > 0.0 ? std::sqrt(r2) / bnorm : 0.0;
      inf.refinements = k + 1;
      if (inf.iterations >= o.max_iter) break;
      const bool no_gain = rel > o.rtol && rel > 0.9 * prev;
      if (inner_pc && inner_stalled) {
        // the network failed its job (the inner solve): Jacobi GMRES finishes the
        // solve, retrying this refinement if it did not pay
        inner_pc = nullptr;
        inf.fallback = 1;
        if (no_gain) continue;
      }
      if (no_gain && stall_stop) {
        // the inner solve reached its tolerance but the float64 residual did not
        // follow: the refinement has stopped contracting
        inf.stalled = 1;
        break;
      }
    }
    rfin = r;
    if ((rc = check_tma(m))) return rc;
  }
  if (harvest) {
    // pairs (r_k - r*, x* - x_k): A (x* - x_k) = r_k - r* holds exactly for the
    // float64 operator that computed the residuals
    for (int k = 0; k < nck; ++k)
      if ((rc = pcn::add_pair(harvest, harvest->ck + (int64_t)(pcn::CKMAX + k) * n, rfin, x,
                              harvest->ck + (int64_t)k * n, m->dinv)))
        return rc;
  }
  if (pc && (rc = pcn::check_err(pc))) return rc;
  inf.rel_res = rel;
  inf.applies = (int)(m->applies - a0);
  if (info) *info = inf;
  if (!(rel <= o.rtol)) return set_error(FSI_ENOCONV, "GMRES: tolerance not reached");
  return FSI_OK;
}

}  // namespace fsi
