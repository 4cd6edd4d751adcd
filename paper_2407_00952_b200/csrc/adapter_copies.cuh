// Compute copies of the adapters of a stand-alone LoRA linear layer, a 16-byte vector per thread.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace sl {

// Vectors that write_copy_vector handles.
inline int64_t adapter_copy_vectors(const AdapterCopyArgs& a) {
  const int n = a.dtype == DT_BF16 ? 8 : 4;
  const int64_t nA = (int64_t)a.ext * a.d_in / n, nB = (int64_t)a.ext * a.d_out / n;
  return a.G * ((a.Acat ? nA : 0) + (a.AcatT ? nA : 0) + (a.Bext ? nB : 0) + (a.BextT ? nB : 0));
}

// One target, padding included, a 16-byte vector per thread: the stand-alone LoRA linear gets a workspace with anything
// in it, and clearing it by memsets first was three or four more operations in front of layers of 10-100 us.
// Vectors in order: Acat [ext, d_in], AcatT [d_in, ext], Bext [d_out, ext], BextT [ext, d_out] of each group (those
// that are wanted); columns (resp. rows) from r on are zero.
template <typename T>
__device__ __forceinline__ void write_copy_vector(const AdapterCopyArgs& a, int64_t idx, int64_t total) {
  constexpr int N = Vec16<T>::N;
  if (idx >= total) return;
  const int64_t nA = (int64_t)a.ext * a.d_in / N, nB = (int64_t)a.ext * a.d_out / N;
  const int64_t per_g = (a.Acat ? nA : 0) + (a.AcatT ? nA : 0) + (a.Bext ? nB : 0) + (a.BextT ? nB : 0);
  const int64_t g = idx / per_g;
  int64_t v = idx % per_g;
  const float* A = a.A + g * a.a_gs;
  const float* B = a.B + g * a.b_gs;
  Vec16<T> o;
  auto by_row = [&](const float* src, int64_t sj, int64_t sc, int n, float scale, void* dst) {     // dst [ext, n]
    const int j = (int)(v * N / n), c = (int)(v * N % n);
#pragma unroll
    for (int i = 0; i < N; ++i) o.set(i, j < a.r ? scale * src[j * sj + (c + i) * sc] : 0.f);
    o.store((T*)dst + (size_t)g * a.ext * n + v * N);
  };
  auto by_column = [&](const float* src, int64_t sj, int64_t sc, int n, float scale, void* dst) {  // dst [n, ext]
    const int c = (int)(v * N / a.ext), j = (int)(v * N % a.ext);
#pragma unroll
    for (int i = 0; i < N; ++i) o.set(i, j + i < a.r ? scale * src[(j + i) * sj + c * sc] : 0.f);
    o.store((T*)dst + (size_t)g * a.ext * n + v * N);
  };
  if (a.Acat) { if (v < nA) { by_row(A, a.d_in, 1, a.d_in, 1.f, a.Acat); return; } v -= nA; }
  if (a.AcatT) { if (v < nA) { by_column(A, a.d_in, 1, a.d_in, 1.f, a.AcatT); return; } v -= nA; }
  if (a.Bext) { if (v < nB) { by_column(B, 1, a.r, a.d_out, a.scale, a.Bext); return; } v -= nB; }
  by_row(B, 1, a.r, a.d_out, a.scale, a.BextT);
}

}  // namespace sl
