// Sums across a CTA for the Krylov kernels (krylov.cu, batch.cu).
#pragma once
#include <cuda_runtime.h>

namespace fsi {

// Sums over a CTA of several values a thread, out[i * stride] for i < kc.  Float64 values with few
// float64 adds (this GPU issues them at a small fraction of the float32 rate; a plain shuffle tree
// costs 5 adds a lane per value).
// Inside a warp a transposing butterfly takes the first P values (P the largest power of
// two <= K, at most 32): at shuffle distance 16 a lane keeps half of its values and adds
// its partner's copy of that half, at distance 8 half of that half, and so on; after
// log2 P levels the lane holds value number lane >> (5 - log2 P) summed over the lanes
// that differ from it in the top log2 P bits, and plain shuffles over the remaining bits
// finish the warp's sum (P - 1 + 5 - log2 P adds a lane).  Values past P take plain trees.
// NT: most threads of the CTA; with tail the row kc - 1 is the last value's sum.
template <int K, int NT>
__device__ __forceinline__ void block_reduce_store_bf(double (&acc)[K], int kc, bool tail, double* out, int stride) {
  constexpr int P = K >= 32 ? 32 : K >= 16 ? 16 : K >= 8 ? 8 : K >= 4 ? 4 : K >= 2 ? 2 : 1;
  constexpr int L = P == 32 ? 5 : P == 16 ? 4 : P == 8 ? 3 : P == 4 ? 2 : P == 2 ? 1 : 0;
  __shared__ double smb[K][NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double a[P];
#pragma unroll
  for (int q = 0; q < P; ++q) a[q] = acc[q];
#pragma unroll
  for (int l = 0; l < L; ++l) {
    const int o = 16 >> l;
    const int half = P >> (l + 1);
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < half; ++q) {
      const double send = up ? a[q] : a[q + half];  // the half the partner keeps
      const double keep = up ? a[q + half] : a[q];
      a[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  double s = a[0];
#pragma unroll
  for (int o = 16 >> L; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((lane & ((32 >> L) - 1)) == 0) smb[lane >> (5 - L)][warp] = s;
#pragma unroll
  for (int i = P; i < K; ++i) {
    double v = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) smb[i][warp] = v;
  }
  __syncthreads();
  const int nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < kc; i += blockDim.x) {
    double t = 0.0;
#pragma unroll
    for (int wi = 0; wi < NT / 32; ++wi)
      if (wi < nw) t += smb[tail && i == kc - 1 ? K - 1 : i][wi];
    out[i * stride] = t;
  }
}

// The same in float32 up to the warps' sums, which are added in two floats (Knuth's two-sum) and stored as
// float64: this GPU issues float64 adds at 1/64 of the float32 rate, so a float64 tree over every thread's
// sums costs more than the float32 basis kernel's streaming, and over the warps' it still took 0.7 us of an
// 11 us kernel.  (Added in float32, the 12 warps of a fused update gave |w|^2 of 1.1 M entries an error of
// 4.5e-9 where CTAs of four warps had 1.2e-9; so 1.0e-9.)  Values in groups of 8 by the transposing
// butterfly (9 shuffles a group against 40 for plain trees: with a few basis chunks a thread, the trees took
// as long as the streaming), the last ones by plain trees.
template <int K, int NT>
__device__ __forceinline__ void block_reduce_store_f(float (&acc)[K], int kc, bool tail, double* out, int stride) {
  __shared__ float smf[K][NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int KG = K / 8 * 8;
#pragma unroll
  for (int i0 = 0; i0 < KG; i0 += 8) {
    float a[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = acc[i0 + q];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      const int o = 16 >> l, half = 4 >> l;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int q = 0; q < half; ++q) {
        const float send = up ? a[q] : a[q + half], keep = up ? a[q + half] : a[q];
        a[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    float v = a[0];
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    if ((lane & 3) == 0) smf[i0 + (lane >> 2)][warp] = v;
  }
#pragma unroll
  for (int i = KG; i < K; ++i) {
    float v = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) smf[i][warp] = v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kc; i += NT) {
    const float* row = smf[tail && i == kc - 1 ? K - 1 : i];
    float hi = row[0], lo = 0.f;
#pragma unroll
    for (int wi = 1; wi < NT / 32; ++wi) {
      const float r = row[wi], t = hi + r, b = t - hi;
      lo += (hi - (t - b)) + (r - b);  // what the addition rounded off, exactly
      hi = t;
    }
    out[i * stride] = isfinite(hi) ? (double)hi + (double)lo : (double)hi;  // (of an infinity, lo is a NaN)
  }
}

// |w - V h2|^2 after the second Gram-Schmidt pass.  On an orthonormal basis it is |w|^2 - |h2|^2, which is
// free, but wrong by delta |h2|^2 where V is orthonormal to delta (the basis type's rounding), and all
// rounding where |h2| nears |w|: in an exhausted Krylov space the difference made vectors of length 7e-4 of
// what is left, or 0, a breakdown that is none.  So it is taken up to PYTHAGORAS of |w|^2 only (an
// error of 1e-4 of the basis type's rounding; the solves of the 16^3 to 64^3 cavities stay below); past it
// corrected_norm2 sums the corrected vector itself.
constexpr double PYTHAGORAS = 1e-4;
constexpr int KCH = 256;  // elements of a basis chunk

// By one CTA, for the whole vector (all threads take part; valid in thread 0): the entries that the basis
// store makes, in its order of operations (what is left may be rounding alone), squares in float64.  PAIRS:
// float basis, even and odd vectors in two sums where a group of four elements is whole (upd_store4_kernel),
// else one chain.  w was written by other CTAs of the same launch.
template <typename VT, bool PAIRS>
__device__ __noinline__ double corrected_norm2(const double* w, const VT* __restrict__ V, int M1, int k, const double* h2,
                                               int64_t n) {
  __shared__ VT hs[96];
  __shared__ double sw[32];
  for (int i = threadIdx.x; i < k; i += blockDim.x) hs[i] = (VT)h2[i];
  __syncthreads();
  double s = 0.0;
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    const VT* blk = V + j / KCH * (int64_t)M1 * KCH + j % KCH;
    VT x = (VT)__ldcg(w + j);
    if constexpr (sizeof(VT) == 8) {
#pragma unroll 8
      for (int i = 0; i < k; ++i) x = fma(-hs[i], blk[(int64_t)i * KCH], x);
    } else {
      VT a = 0, b = 0;
      if (PAIRS && (j & ~(int64_t)3) + 4 <= n) {
        int i = 0;
#pragma unroll 4
        for (; i + 2 <= k; i += 2) {
          a = fmaf(hs[i], blk[(int64_t)i * KCH], a);
          b = fmaf(hs[i + 1], blk[(int64_t)(i + 1) * KCH], b);
        }
        if (i < k) a = fmaf(hs[i], blk[(int64_t)i * KCH], a);
      } else {
#pragma unroll 8
        for (int i = 0; i < k; ++i) a = fmaf(hs[i], blk[(int64_t)i * KCH], a);
      }
      x -= a + b;
    }
    s = fma((double)x, (double)x, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < (int)blockDim.x >> 5; ++q) t += sw[q];
  return t;
}

}  // namespace fsi
