// Plain-FMA linear-layer kernel: any shape, fp32 or bf16 storage, fp32 accumulation.
// It is the arithmetic of the fp32 configuration and a second opinion for the tensor-core kernel.
#include "common.cuh"
#include "host_common.h"
#include "kernels.h"
#include "launch.cuh"

namespace sl {

namespace {
constexpr int BM = 64, BN = 64, BK = 16;

template <typename T>
__global__ void __launch_bounds__(256) gemm_simt_kernel(GemmArgs a) {
  overlap_sync();
  __shared__ float As[BK][BM + 4];
  __shared__ float Bs[BK][BN + 4];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int lrow = threadIdx.x / 4, lk = (threadIdx.x % 4) * 4;
  const int g = a.rows_per_group > 0 ? m0 / a.rows_per_group : 0;
  const int w_rows = a.w_rows > 0 ? a.w_rows : a.N;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

  for (int phase = 0; phase < 2; ++phase) {
    const T* X; const T* W; int64_t ldx, ldw; int Kp; int wr;
    if (phase == 0) {
      X = (const T*)a.X; ldx = a.ldx; ldw = a.ldw; Kp = a.K; wr = w_rows;
      W = (const T*)a.W + (a.w_grouped ? (size_t)g * a.N * a.ldw : 0);
    } else {
      if (a.Ke == 0) break;
      X = (const T*)a.Xe; ldx = a.ldxe; ldw = a.ldwe; Kp = a.Ke; wr = a.N;
      W = (const T*)a.We + (a.we_grouped ? (size_t)g * a.N * a.ldwe : 0);
    }
    for (int k0 = 0; k0 < Kp; k0 += BK) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int k = k0 + lk + i;
        int m = m0 + lrow, n = n0 + lrow;
        As[lk + i][lrow] = (m < a.M && k < Kp) ? to_f<T>(X[(size_t)m * ldx + k]) : 0.f;
        Bs[lk + i][lrow] = (n < wr && k < Kp) ? to_f<T>(W[(size_t)n * ldw + k]) : 0.f;
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < BK; ++k) {
        float av[4], bv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) av[i] = As[k][ty * 4 + i];
#pragma unroll
        for (int j = 0; j < 4; ++j) bv[j] = Bs[k][tx * 4 + j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      }
      __syncthreads();
    }
  }

  const T* bias = (const T*)a.bias;
  const T* R = (const T*)a.R;
  T* Y = (T*)a.Y;
  T* Z = (T*)a.Z;
  const bool tanh_form = a.gelu_tanh != 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int m = m0 + ty * 4 + i;
    if (m >= a.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int n = n0 + tx * 4 + j;
      if (n >= a.N) continue;
      float v = acc[i][j];
      if (bias && a.epi != EPI_MUL_GELUGRAD) v += to_f<T>(bias[n]);
      switch (a.epi) {
        case EPI_BIAS_GELU:
          Z[(size_t)m * a.ldz + n] = from_f<T>(v);
          // the activation is applied to the value as it is stored, so that forward and backward agree
          v = gelu_f(to_f<T>(from_f<T>(v)), tanh_form);
          break;
        case EPI_BIAS_RESID: v += to_f<T>(R[(size_t)m * a.ldr + n]); break;
        case EPI_MUL_GELUGRAD: v *= gelu_grad_f(to_f<T>(R[(size_t)m * a.ldr + n]), tanh_form); break;
        default: break;
      }
      Y[(size_t)m * a.ldy + n] = from_f<T>(v);
    }
  }
}
// ------------------------------------------------------------------------------------------
// fp32, 16-byte aligned operands
// ------------------------------------------------------------------------------------------
// A block owns a TM x TN tile and walks the contraction in slabs of SLAB columns through a three-stage ring filled by
// 16-byte asynchronous copies; its KG thread groups each take SLAB / KG columns of every slab (their sums are added in
// order at the end), four rows by four columns per thread.  Operands stay [row][k] in shared memory with rows 4 floats
// longer than the slab, so that the eight rows a quarter-warp reads as float4 lie in different banks.
// What bounds it: at the sizes the fp32 configuration runs (512 tokens, widths 128-1024) the chain of slabs of the few
// tiles, so small outputs take small tiles with the contraction spread over four thread groups.  Against one 64 x 64 tile
// per block with scalar loads and no overlap of loads and products (below), us: 512 x 128 -> 384 13.1 -> 5.4, 128 -> 128
// 13.0 -> 3.7, 512 -> 128 41.4 -> 8.7, 1024 -> 128 79.2 -> 15.6; 4096 x 1024 -> 1024 349 -> 248 (35 TFLOP/s); errors
// against 64 bits halved (four shorter sums) or the same.
template <int TM_, int TN_, int KG_, int SLAB_> struct F32Cfg {
  static constexpr int TM = TM_, TN = TN_, KG = KG_, SLAB = SLAB_, LD = SLAB + 4, STAGES = 3;
  static constexpr int THREADS = KG * (TM / 4) * (TN / 4);
  static constexpr int STAGE_FLOATS = (TM + TN) * LD;
  static constexpr int SMEM = STAGES * STAGE_FLOATS * 4;
  static_assert(KG * TM * (TN + 1) * 4 <= SMEM && SLAB % (4 * KG) == 0 && SLAB % 32 == 0, "");
};

__device__ __forceinline__ void cp_async16_zero(uint32_t dst, const float* src, bool valid) {
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ void store_f32(const GemmArgs& a, int m, int n, float v) {
  if (m >= a.M || n >= a.N) return;
  const bool tanh_form = a.gelu_tanh != 0;
  if (a.bias && a.epi != EPI_MUL_GELUGRAD) v += ((const float*)a.bias)[n];
  switch (a.epi) {
    case EPI_BIAS_GELU:
      ((float*)a.Z)[(size_t)m * a.ldz + n] = v;
      v = gelu_f(v, tanh_form);
      break;
    case EPI_BIAS_RESID: v += ((const float*)a.R)[(size_t)m * a.ldr + n]; break;
    case EPI_MUL_GELUGRAD: v *= gelu_grad_f(((const float*)a.R)[(size_t)m * a.ldr + n], tanh_form); break;
    default: break;
  }
  ((float*)a.Y)[(size_t)m * a.ldy + n] = v;
}

template <class C>
__global__ void __launch_bounds__(C::THREADS) gemm_f32_kernel(GemmArgs a) {
  overlap_sync();
  extern __shared__ __align__(16) float sh[];
  constexpr int TX = C::TN / 4, TY = C::TM / 4, TPG = TX * TY;
  const int m0 = blockIdx.y * C::TM, n0 = blockIdx.x * C::TN;
  const int kg = threadIdx.x / TPG, t = threadIdx.x % TPG, tx = t % TX, ty = t / TX;
  const int g = a.rows_per_group > 0 ? m0 / a.rows_per_group : 0;
  const float* X0 = (const float*)a.X;
  const float* W0 = (const float*)a.W + (a.w_grouped ? (size_t)g * a.N * a.ldw : 0);
  const float* X1 = (const float*)a.Xe;
  const float* W1 = (const float*)a.We + (a.we_grouped ? (size_t)g * a.N * a.ldwe : 0);
  const int w_rows = a.w_rows > 0 ? a.w_rows : a.N;
  const int slabs0 = (a.K + C::SLAB - 1) / C::SLAB, slabs = slabs0 + (a.Ke + C::SLAB - 1) / C::SLAB;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sh);

  auto load = [&](int s) {
    if (s < slabs) {
      const bool ext = s >= slabs0;
      const float* X = ext ? X1 : X0; const float* W = ext ? W1 : W0;
      const int64_t ldx = ext ? a.ldxe : a.ldx, ldw = ext ? a.ldwe : a.ldw;
      const int Kp = ext ? a.Ke : a.K, wr = ext ? a.N : w_rows, k0 = (ext ? s - slabs0 : s) * C::SLAB;
      const uint32_t st = sbase + (uint32_t)((s % C::STAGES) * C::STAGE_FLOATS * 4);
      constexpr int V = C::SLAB / 4;                   // 16-byte pieces per row
#pragma unroll
      for (int i = threadIdx.x; i < (C::TM + C::TN) * V; i += C::THREADS) {
        const int r = i / V, k = k0 + (i % V) * 4;
        const bool isx = r < C::TM;
        const int row = isx ? m0 + r : n0 + r - C::TM;
        const bool ok = k < Kp && row < (isx ? a.M : wr);
        const float* src = isx ? X + (size_t)row * ldx + k : W + (size_t)row * ldw + k;
        cp_async16_zero(st + (uint32_t)((r * C::LD + (i % V) * 4) * 4), ok ? src : X0, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  load(0);
  load(1);
  for (int s = 0; s < slabs; ++s) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();                                   // slab s has arrived, and slab s - 1 has been read by everyone
    load(s + 2);
    const float* As = sh + (s % C::STAGES) * C::STAGE_FLOATS + kg * (C::SLAB / C::KG);
    const float* Bs = As + C::TM * C::LD;
#pragma unroll 2
    for (int k = 0; k < C::SLAB / C::KG; k += 4) {
      float4 av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const float4*>(As + (ty + TY * i) * C::LD + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(Bs + (tx + TX * j) * C::LD + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(av[i].x, bv[j].x, acc[i][j]);
          acc[i][j] = fmaf(av[i].y, bv[j].y, acc[i][j]);
          acc[i][j] = fmaf(av[i].z, bv[j].z, acc[i][j]);
          acc[i][j] = fmaf(av[i].w, bv[j].w, acc[i][j]);
        }
    }
  }
  if constexpr (C::KG == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) store_f32(a, m0 + ty + TY * i, n0 + tx + TX * j, acc[i][j]);
  } else {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sh[(kg * C::TM + ty + TY * i) * (C::TN + 1) + tx + TX * j] = acc[i][j];
    __syncthreads();
    for (int o = threadIdx.x; o < C::TM * C::TN; o += C::THREADS) {
      const int m = o / C::TN, n = o % C::TN;
      float v = sh[m * (C::TN + 1) + n];
#pragma unroll
      for (int q = 1; q < C::KG; ++q) v += sh[(q * C::TM + m) * (C::TN + 1) + n];
      store_f32(a, m0 + m, n0 + n, v);
    }
  }
}

template <class C>
cudaError_t launch_f32(const GemmArgs& a, cudaStream_t st) {
  static PerDeviceOnce once;
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_f32_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  dim3 grid((a.N + C::TN - 1) / C::TN, (a.M + C::TM - 1) / C::TM);
  return launch_overlapped(gemm_f32_kernel<C>, grid, C::THREADS, C::SMEM, st, a);
}

bool f32_vector_ok(const GemmArgs& a) {
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (a.dtype != DT_F32 || a.K % 4 || a.ldx % 4 || a.ldw % 4 || !al(a.X) || !al(a.W)) return false;
  if (a.k_gap_len > 0 || (a.M + 31) / 32 > 65535) return false;
  return a.Ke == 0 || (a.Ke % 4 == 0 && a.ldxe % 4 == 0 && a.ldwe % 4 == 0 && al(a.Xe) && al(a.We));
}

}  // namespace

cudaError_t gemm_simt(const GemmArgs& a, cudaStream_t st) {
  if (a.rows_per_group > 0 && (a.rows_per_group % BM) != 0 && (a.w_grouped || a.we_grouped))
    return cudaErrorInvalidValue;
  if (f32_vector_ok(a)) {
    // 64 x 64 tiles once they fill the chip, else a quarter of the tile and four thread groups along the contraction
    const int64_t tiles = (int64_t)((a.M + 63) / 64) * ((a.N + 63) / 64);
    if (tiles >= num_sms()) return launch_f32<F32Cfg<64, 64, 1, 32>>(a, st);
    // still fewer: halves and quarters of that tile, as long as a block has an SM to itself
    const int64_t small = (int64_t)((a.M + 31) / 32) * ((a.N + 31) / 32);
    if (4 * small <= num_sms()) return launch_f32<F32Cfg<16, 16, 16, 64>>(a, st);
    if (2 * small <= num_sms()) return launch_f32<F32Cfg<32, 16, 8, 64>>(a, st);
    return launch_f32<F32Cfg<32, 32, 4, 64>>(a, st);
  }
  dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM);
  if (a.dtype == DT_BF16) launch_overlapped(gemm_simt_kernel<bf16>, grid, 256, 0, st, a);
  else launch_overlapped(gemm_simt_kernel<float>, grid, 256, 0, st, a);
  return cudaGetLastError();
}

}  // namespace sl
