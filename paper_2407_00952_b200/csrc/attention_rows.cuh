// Causal attention one row at a time: a warp takes one row (a query, or a key for dK and dV), scores are one key (query)
// per lane, the accumulations one feature per lane with the probability broadcast by shuffle.  Plain fp32 FMA over the
// visible pairs only, in the order of their positions.
#pragma once
#include "common.cuh"

namespace sl {
namespace rows {

constexpr int MAX_DH = 128;
constexpr int DPL = MAX_DH / 32;   // features per lane

template <typename T>
__device__ __forceinline__ float dot_row(const float* a_s, const T* __restrict__ row, int dh) {
  float s = 0.f;
  for (int c = 0; c < dh; ++c) s = fmaf(a_s[c], to_f<T>(row[c]), s);
  return s;
}

// One head of one sequence: `q` is its first query element, keys and values d and 2 d further on, rows `ld` apart; O and
// dO rows are d apart, lse and rowdot 1.
template <typename T> struct Head {
  const T* q; size_t ld; int d, dh, T_; float scale;
  __device__ __forceinline__ Head(const T* qkv, int b, int h, int Tn, int H, int d_)
      : q(qkv + (size_t)b * Tn * 3 * d_ + (size_t)h * (d_ / H)), ld((size_t)3 * d_), d(d_), dh(d_ / H), T_(Tn), scale(rsqrtf((float)(d_ / H))) {}
};

// One row of O and its lse.  s: dh floats of shared memory of the warp's own.
template <typename T>
__device__ __forceinline__ void forward_row(const Head<T>& hd, int i, float* s, T* orow, float* lse) {
  const int lane = threadIdx.x & 31;
  for (int c = lane; c < hd.dh; c += 32) s[c] = to_f<T>(hd.q[(size_t)i * hd.ld + c]);
  __syncwarp();
  float m = -INFINITY, l = 0.f, acc[DPL];
#pragma unroll
  for (int c = 0; c < DPL; ++c) acc[c] = 0.f;
  for (int j0 = 0; j0 <= i; j0 += 32) {
    const int j = j0 + lane;
    float sc = -INFINITY;
    if (j <= i) sc = dot_row<T>(s, hd.q + (size_t)j * hd.ld + hd.d, hd.dh) * hd.scale;
    const float nm = fmaxf(m, warp_max(sc));
    const float p = (j <= i) ? expf(sc - nm) : 0.f;
    const float corr = (m == -INFINITY) ? 0.f : expf(m - nm);
    l = l * corr + warp_sum(p);
#pragma unroll
    for (int c = 0; c < DPL; ++c) acc[c] *= corr;
    const int cnt = min(32, i - j0 + 1);
    for (int jj = 0; jj < cnt; ++jj) {
      const float pj = __shfl_sync(0xffffffffu, p, jj);
      const T* vrow = hd.q + (size_t)(j0 + jj) * hd.ld + 2 * (size_t)hd.d;
#pragma unroll
      for (int c = 0; c < DPL; ++c) {
        const int dim = lane + 32 * c;
        if (dim < hd.dh) acc[c] = fmaf(pj, to_f<T>(vrow[dim]), acc[c]);
      }
    }
    m = nm;
  }
#pragma unroll
  for (int c = 0; c < DPL; ++c) {
    const int dim = lane + 32 * c;
    if (dim < hd.dh) orow[dim] = from_f<T>(acc[c] / l);
  }
  if (lane == 0) *lse = m + logf(l);
  __syncwarp();
}

// One row of dQ from L = lse and D = sum(dO * O) of the row.  s: 2 dh floats.
template <typename T>
__device__ __forceinline__ void dq_row(const Head<T>& hd, const T* dorow, float L, float D, int i, float* s, T* out) {
  const int lane = threadIdx.x & 31;
  float* g = s + hd.dh;
  for (int c = lane; c < hd.dh; c += 32) { s[c] = to_f<T>(hd.q[(size_t)i * hd.ld + c]); g[c] = to_f<T>(dorow[c]); }
  __syncwarp();
  float acc[DPL];
#pragma unroll
  for (int c = 0; c < DPL; ++c) acc[c] = 0.f;
  for (int j0 = 0; j0 <= i; j0 += 32) {
    const int j = j0 + lane;
    float ds = 0.f;
    if (j <= i) {
      const T* krow = hd.q + (size_t)j * hd.ld + hd.d;
      const float p = expf(dot_row<T>(s, krow, hd.dh) * hd.scale - L);
      ds = p * (dot_row<T>(g, krow + hd.d, hd.dh) - D) * hd.scale;
    }
    const int cnt = min(32, i - j0 + 1);
    for (int jj = 0; jj < cnt; ++jj) {
      const float dsj = __shfl_sync(0xffffffffu, ds, jj);
      const T* krow = hd.q + (size_t)(j0 + jj) * hd.ld + hd.d;
#pragma unroll
      for (int c = 0; c < DPL; ++c) {
        const int dim = lane + 32 * c;
        if (dim < hd.dh) acc[c] = fmaf(dsj, to_f<T>(krow[dim]), acc[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < DPL; ++c) {
    const int dim = lane + 32 * c;
    if (dim < hd.dh) out[dim] = from_f<T>(acc[c]);
  }
  __syncwarp();
}

// One row of dK and dV (out, out + d); d_o, lse and rowdot are those of the head's first query.  s: 2 dh floats.
template <typename T>
__device__ __forceinline__ void dkv_row(const Head<T>& hd, const T* d_o, const float* lse, const float* rowdot, int j, float* s, T* out) {
  const int lane = threadIdx.x & 31;
  float* v = s + hd.dh;
  const T* krow = hd.q + (size_t)j * hd.ld + hd.d;
  for (int c = lane; c < hd.dh; c += 32) { s[c] = to_f<T>(krow[c]); v[c] = to_f<T>(krow[hd.d + c]); }
  __syncwarp();
  float dk[DPL], dv[DPL];
#pragma unroll
  for (int c = 0; c < DPL; ++c) { dk[c] = 0.f; dv[c] = 0.f; }
  for (int i0 = j; i0 < hd.T_; i0 += 32) {
    const int i = i0 + lane;
    float p = 0.f, ds = 0.f;
    if (i < hd.T_) {
      p = expf(dot_row<T>(s, hd.q + (size_t)i * hd.ld, hd.dh) * hd.scale - lse[i]);
      ds = p * (dot_row<T>(v, d_o + (size_t)i * hd.d, hd.dh) - rowdot[i]) * hd.scale;
    }
    const int cnt = min(32, hd.T_ - i0);
    for (int ii = 0; ii < cnt; ++ii) {
      const float pi = __shfl_sync(0xffffffffu, p, ii), dsi = __shfl_sync(0xffffffffu, ds, ii);
      const T* qrow = hd.q + (size_t)(i0 + ii) * hd.ld;
      const T* dorow = d_o + (size_t)(i0 + ii) * hd.d;
#pragma unroll
      for (int c = 0; c < DPL; ++c) {
        const int dim = lane + 32 * c;
        if (dim < hd.dh) {
          dv[c] = fmaf(pi, to_f<T>(dorow[dim]), dv[c]);
          dk[c] = fmaf(dsi, to_f<T>(qrow[dim]), dk[c]);
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < DPL; ++c) {
    const int dim = lane + 32 * c;
    if (dim < hd.dh) { out[dim] = from_f<T>(dk[c]); out[hd.d + dim] = from_f<T>(dv[c]); }
  }
  __syncwarp();
}

}  // namespace rows
}  // namespace sl
