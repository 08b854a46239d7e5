// The soft threshold, the objective / KKT pass over the upper triangle and the
// reduction of its partial results, shared by the sweep kernel and the wave form's evaluation.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace concord {

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using V = float4;
  static constexpr int N = 4;
  __device__ static void fma(V& w, float d, const V& s) {
    w.x = fmaf(d, s.x, w.x);
    w.y = fmaf(d, s.y, w.y);
    w.z = fmaf(d, s.z, w.z);
    w.w = fmaf(d, s.w, w.w);
  }
};
template <>
struct Vec16<double> {
  using V = double2;
  static constexpr int N = 2;
  __device__ static void fma(V& w, double d, const V& s) {
    w.x = ::fma(d, s.x, w.x);
    w.y = ::fma(d, s.y, w.y);
  }
};

template <typename T>
__device__ __forceinline__ T soft_threshold(T x, T tau) {
  T a = fabs(x) - tau;
  if (!(a > (T)0)) return (T)0;
  return x > (T)0 ? a : -a;
}

// Block reduction of the per-thread partials into partials[blockIdx.x*kParts+k].
__device__ __forceinline__ void block_reduce_parts(double (&v)[kParts], double* out,
                                                   double (*red)[kParts], int slot) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < kParts; ++k) {
    double x = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      double y = __shfl_down_sync(0xffffffffu, x, o);
      x = (k == kPartKkt || k == kPartDelta) ? fmax(x, y) : x + y;
    }
    if (lane == 0) red[wid][k] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < kParts; ++k) {
      double x = red[0][k];
      for (int w = 1; w < nw; ++w)
        x = (k == kPartKkt || k == kPartDelta) ? fmax(x, red[w][k]) : x + red[w][k];
      out[(size_t)slot * kParts + k] = x;
    }
  }
  __syncthreads();
}

// v += the residual, objective terms and non-finite counts of CTA `cta` of G.
template <typename T, bool MIXED>
__device__ __forceinline__ void kkt_pass(int p, int ld, const T* W, const T* Om, const double* omdiag64,
                                         double lam, int cta, int G, double (&v)[kParts]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // Work unit: an 8-row chunk of a 32 x 32 tile (ta <= tb) of the upper
  // triangle.  Lane l takes column j = tb*32 + l: W_ij comes from row i
  // (coalesced across lanes), W_ji from row j as one 8-element vector, so
  // G_ij = W_ij + W_ji pairs up without a transpose.
  using VT = Vec16<T>;
  using V = typename VT::V;
  constexpr int NV = 8 / VT::N;
  const int nb = (p + kTile - 1) / kTile;
  const double lamd = lam;
  const float lamf = (float)lam;
  const int units = nb * nb * 4;
  const int gwarps = G * (blockDim.x >> 5);
  long long kkt = __double_as_longlong(v[kPartKkt]);
  for (int u = cta * (blockDim.x >> 5) + wid; u < units; u += gwarps) {
    const int tau = u >> 2, r0 = (u & 3) * 8;
    const int ta = tau / nb, tb = tau % nb;
    if (ta > tb) continue;
    const int j = tb * kTile + lane;
    const int i0 = ta * kTile + r0;
    if (i0 >= p) continue;
    T w1[8], om8[8], wt[8];
    const bool jv = j < p;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int i = i0 + r;
      const bool ok = jv && i < p;
      w1[r] = ok ? __ldcg(W + (size_t)i * ld + j) : (T)0;
      om8[r] = ok ? __ldcg(Om + (size_t)i * ld + j) : (T)0;
    }
    if (jv) {
      const V* src = reinterpret_cast<const V*>(W + (size_t)j * ld + i0);
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        V x = __ldcg(src + q);
        if constexpr (VT::N == 4) {
          wt[4 * q + 0] = ((const float*)&x)[0];
          wt[4 * q + 1] = ((const float*)&x)[1];
          wt[4 * q + 2] = ((const float*)&x)[2];
          wt[4 * q + 3] = ((const float*)&x)[3];
        } else {
          wt[2 * q + 0] = ((const double*)&x)[0];
          wt[2 * q + 1] = ((const double*)&x)[1];
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < 8; ++r) wt[r] = (T)0;
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int i = i0 + r;
      if (!jv || i >= j) continue;
      const T om_t = om8[r];
      // FP32 screen: a zero entry whose |G_ij| is clearly below lambda
      // has residual exactly 0 (the margin covers the FP32 rounding of
      // G); every other entry is evaluated in FP64.
      const float w1f = (float)w1[r], w2f = (float)wt[r];
      const float gf = w1f + w2f;
      if (om_t == (T)0 && fabsf(gf) <= lamf - 1e-5f * (1.0f + fabsf(w1f) + fabsf(w2f)))
        continue;
      // |G + lambda sign(om)|, or |G| - lambda where om = 0: one sum on every
      // lane, the maximum of doubles >= 0 as integers (the FP64 pipe issues a
      // warp over 16 cycles; three branches of it took 78 us of a sweep's
      // evaluation at p = 1000)
      const double g = (double)w1[r] + (double)wt[r];
      const bool neg = __double2hiint(g) < 0;
      const bool edge = om_t > (T)0 || om_t < (T)0;
      const double t = g + ((edge ? om_t > (T)0 : neg) ? lamd : -lamd);
      const bool flip = edge ? __double2hiint(t) < 0 : neg;
      const long long res = __double_as_longlong(t) ^ (flip ? 0x8000000000000000ll : 0ll);
      if (res > kkt && res <= 0x7ff0000000000000ll) kkt = res;  // (not a NaN)
      if (om_t != (T)0) {
        v[kPartQuad] += (double)om_t * g;
        v[kPartPen] += fabs((double)om_t);
      }
      if (!isfinite(om_t) || (sizeof(T) == 4 ? !(isfinite(w1[r]) && isfinite(wt[r])) : !isfinite(g)))
        v[kPartBad] += 1.0;
    }
    const int k = lane - r0;  // the diagonal: at most one entry per lane
    if (ta == tb && k >= 0 && k < 8 && jv) {
      double wii = 0.0, oii = 0.0;
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r == k) {
          wii = (double)w1[r];
          oii = (double)om8[r];
        }
      if (MIXED) oii = __ldcg(omdiag64 + j);
      if (oii > 0.0 && isfinite(wii) && isfinite(oii)) {
        kkt = max(kkt, __double_as_longlong(fabs(wii - 1.0 / oii)));
        v[kPartQuad] += oii * wii;
        v[kPartLog] += log(oii);
      } else {
        v[kPartBad] += 1.0;
      }
    }
  }
  v[kPartKkt] = __longlong_as_double(kkt);
}

}  // namespace concord
