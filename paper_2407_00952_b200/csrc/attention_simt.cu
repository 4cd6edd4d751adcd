// Causal multi-head attention with plain FMA arithmetic (fp32 or bf16 storage, any shape, head width up to 128): the
// arithmetic of the fp32 configuration and a second opinion for the tensor-core kernels.
// Short sequences take a warp per row (by_rows says which).  Otherwise a block of eight warps owns RT = 32 rows (queries,
// or keys in the dK/dV kernel) of one (sequence, head), four rows per warp, and walks the other side in tiles of 32 rows
// that all its warps share through shared memory.  Scores are one column of the tile per lane; the accumulations are one
// feature per lane, with the tile's probabilities read back as broadcasts from shared memory.  A tile element read from
// shared memory serves four rows, a probability all features.
// What bounds it: shared-memory reads (about five per sixteen products).  Against one warp per row that reads the other side
// from global memory: the fp32 round of 512 tokens (8 sequences of 64, 4 heads of 32) 514 -> 355 us together with the
// sixteen-lane adapter gradients of lora_grad.cu; errors against 64 bits a little smaller.
#include "attention_rows.cuh"
#include "common.cuh"
#include "host_common.h"
#include "kernels.h"
#include "launch.cuh"

namespace sl {
namespace {

constexpr int WARPS = 8, RPW = 4, RT = WARPS * RPW, KT = 32;
constexpr int MAX_DH = rows::MAX_DH;
constexpr int DPL = MAX_DH / 32;   // features per lane

// Shared memory, in floats: two tiles [32][width + 1], width = dh rounded up to 32 so that "one feature per lane" reads
// stay inside a row (the odd stride keeps "one row per lane" reads conflict-free), two row blocks [32][dh rounded up to
// 4] (read as float4 broadcasts, zero past dh), two [32][32] blocks of per-row tile values.
__host__ __device__ constexpr int pad4(int dh) { return (dh + 3) & ~3; }
__host__ __device__ constexpr int tile_stride(int dh) { return ((dh + 31) & ~31) + 1; }
inline size_t smem_bytes(int dh) { return (size_t)(2 * KT * tile_stride(dh) + 2 * RT * pad4(dh) + 2 * RT * KT) * 4; }

struct Tiles {
  float *a, *b, *ra, *rb, *pa, *pb;
  int lt, lr;
  __device__ __forceinline__ Tiles(float* sh, int dh) {
    lr = pad4(dh); lt = tile_stride(dh);
    ra = sh; rb = ra + RT * lr;                        // 16-byte aligned
    pa = rb + RT * lr; pb = pa + RT * KT;
    a = pb + RT * KT; b = a + KT * lt;
  }
};

// rows row0 .. row0 + 31 of a matrix into [32][ld_dst], columns 0 .. width - 1; zero past `rows` and past dh
template <typename T>
__device__ __forceinline__ void load_rows(float* dst, int ld_dst, int width, const T* src, size_t ld, int row0, int rows, int dh) {
  for (int i = threadIdx.x; i < 32 * width; i += WARPS * 32) {
    const int r = i / width, c = i % width;
    dst[r * ld_dst + c] = (row0 + r < rows && c < dh) ? to_f<T>(src[(size_t)(row0 + r) * ld + c]) : 0.f;
  }
}

// out[r] = sum_c row_r[c] * tile[lane][c] for this warp's four rows
__device__ __forceinline__ void dot4(const float* rows, int lr, const float* tile_row, float* out) {
#pragma unroll
  for (int r = 0; r < RPW; ++r) out[r] = 0.f;
#pragma unroll 2
  for (int c = 0; c < lr; c += 4) {
    const float k0 = tile_row[c], k1 = tile_row[c + 1], k2 = tile_row[c + 2], k3 = tile_row[c + 3];
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const float4 q = *reinterpret_cast<const float4*>(rows + r * lr + c);
      out[r] = fmaf(q.w, k3, fmaf(q.z, k2, fmaf(q.y, k1, fmaf(q.x, k0, out[r]))));
    }
  }
}

// acc[r][c] += sum over j0 <= j < j1 (multiples of 4) of p[r][j] * tile[j][lane + 32 c]
__device__ __forceinline__ void accumulate4(float (*acc)[DPL], const float* p, const float* tile, int lt, int lane, int nfeat,
                                            int j0, int j1) {
#pragma unroll 2
  for (int j = j0; j < j1; j += 4) {
    float4 pv[RPW];
#pragma unroll
    for (int r = 0; r < RPW; ++r) pv[r] = *reinterpret_cast<const float4*>(p + r * KT + j);
#pragma unroll
    for (int c = 0; c < DPL; ++c) {
      if (c >= nfeat) break;                           // warp-uniform
      const float* t = tile + j * lt + lane + 32 * c;
      const float v0 = t[0], v1 = t[lt], v2 = t[2 * lt], v3 = t[3 * lt];
#pragma unroll
      for (int r = 0; r < RPW; ++r)
        acc[r][c] = fmaf(pv[r].w, v3, fmaf(pv[r].z, v2, fmaf(pv[r].y, v1, fmaf(pv[r].x, v0, acc[r][c]))));
    }
  }
}

// The 4 x 4 block of the diagonal tile in which the warp's four rows meet their own positions: row r takes the tile rows
// up to the r-th (keys, UP_TO) or from the r-th on (queries).  The pairs that causality hides are left out of the sums
// and not multiplied by a probability of 0, which would turn an inf or NaN of a later key (an earlier query) into NaN.
template <bool UP_TO>
__device__ __forceinline__ void accumulate_diagonal(float (*acc)[DPL], const float* p, const float* tile, int lt, int lane,
                                                    int nfeat, int j) {
  float pv[RPW][4];
#pragma unroll
  for (int r = 0; r < RPW; ++r) *reinterpret_cast<float4*>(pv[r]) = *reinterpret_cast<const float4*>(p + r * KT + j);
#pragma unroll
  for (int c = 0; c < DPL; ++c) {
    if (c >= nfeat) break;
    const float* t = tile + j * lt + lane + 32 * c;
    const float v[4] = {t[0], t[lt], t[2 * lt], t[3 * lt]};
#pragma unroll
    for (int jj = 0; jj < RPW; ++jj)
#pragma unroll
      for (int r = 0; r < RPW; ++r)
        if (UP_TO ? jj <= r : jj >= r) acc[r][c] = fmaf(pv[r][jj], v[jj], acc[r][c]);
  }
}

// What the warp's rows (the w-th four of the block) see of a tile: all of it, or on the diagonal the part up to / from
// their own positions.  Both tile sizes are the same, so the diagonal tile starts where the block's rows do.
static_assert(RT == KT && RPW == 4, "");
template <bool UP_TO>
__device__ __forceinline__ void accumulate_tile(float (*acc)[DPL], const float* p, const float* tile, int lt, int lane,
                                                int nfeat, bool diagonal, int w) {
  if (!diagonal) {
    accumulate4(acc, p, tile, lt, lane, nfeat, 0, KT);
    return;
  }
  if (UP_TO) accumulate4(acc, p, tile, lt, lane, nfeat, 0, w * RPW);
  accumulate_diagonal<UP_TO>(acc, p, tile, lt, lane, nfeat, w * RPW);
  if (!UP_TO) accumulate4(acc, p, tile, lt, lane, nfeat, (w + 1) * RPW, KT);
}

struct Where { int b, h, r0; };
__device__ __forceinline__ Where where(int Tn, int H) {
  const int nt = (Tn + RT - 1) / RT;
  const int64_t item = (int64_t)blockIdx.x / nt;
  return {(int)(item / H), (int)(item % H), (nt - 1 - (int)(blockIdx.x % nt)) * RT};      // long rows first
}

template <typename T>
__global__ void __launch_bounds__(WARPS * 32, 4) attn_fwd_kernel(const T* __restrict__ qkv, int Tn, int H, int d,
                                                              T* __restrict__ o, float* __restrict__ lse) {
  overlap_sync();
  extern __shared__ __align__(16) float sh[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, dh = d / H, nfeat = (dh + 31) / 32;
  const Where at = where(Tn, H);
  Tiles t(sh, dh);
  const float scale = rsqrtf((float)dh);
  const size_t ld = (size_t)3 * d;
  const T* base = qkv + (size_t)at.b * Tn * ld + (size_t)at.h * dh;
  load_rows<T>(t.ra, t.lr, t.lr, base, ld, at.r0, Tn, dh);
  float m[RPW], l[RPW], acc[RPW][DPL];
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < DPL; ++c) acc[r][c] = 0.f;
  }
  const float* rows = t.ra + w * RPW * t.lr;
  float* p_s = t.pa + w * RPW * KT;
  const int row0 = at.r0 + w * RPW;
  for (int j0 = 0; j0 <= at.r0 + RT - 1 && j0 < Tn; j0 += KT) {
    __syncthreads();
    load_rows<T>(t.a, t.lt, t.lr, base + d, ld, j0, Tn, dh);
    load_rows<T>(t.b, t.lt, t.lr, base + 2 * (size_t)d, ld, j0, Tn, dh);
    __syncthreads();
    float s[RPW];
    dot4(rows, t.lr, t.a + lane * t.lt, s);
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const bool vis = j0 + lane <= row0 + r;
      const float sc = vis ? s[r] * scale : -INFINITY;
      const float nm = fmaxf(m[r], warp_max(sc));
      const float p = vis ? expf(sc - nm) : 0.f;
      const float corr = m[r] == -INFINITY ? 0.f : expf(m[r] - nm);
      l[r] = l[r] * corr + warp_sum(p);
#pragma unroll
      for (int c = 0; c < DPL; ++c) acc[r][c] *= corr;
      m[r] = nm;
      p_s[r * KT + lane] = p;
    }
    __syncwarp();
    accumulate_tile<true>(acc, p_s, t.b, t.lt, lane, nfeat, j0 == at.r0, w);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    const int i = row0 + r;
    if (i >= Tn) continue;
    T* orow = o + ((size_t)at.b * Tn + i) * d + (size_t)at.h * dh;
#pragma unroll
    for (int c = 0; c < DPL; ++c) {
      const int dim = lane + 32 * c;
      if (dim < dh) orow[dim] = from_f<T>(acc[r][c] / l[r]);
    }
    if (lane == 0) lse[((size_t)at.b * H + at.h) * Tn + i] = m[r] + logf(l[r]);
  }
}

// dQ, and D[row] = sum(dO * O) of its rows, which the dK/dV kernel (second) reads from `rowdot`
template <typename T>
__global__ void __launch_bounds__(WARPS * 32, 3) attn_bwd_dq_kernel(const T* __restrict__ qkv, const T* __restrict__ o,
                                                                 const float* __restrict__ lse, const T* __restrict__ d_o,
                                                                 float* __restrict__ rowdot, int Tn, int H, int d,
                                                                 T* __restrict__ dqkv) {
  overlap_sync();
  extern __shared__ __align__(16) float sh[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, dh = d / H, nfeat = (dh + 31) / 32;
  const Where at = where(Tn, H);
  Tiles t(sh, dh);
  const float scale = rsqrtf((float)dh);
  const size_t ld = (size_t)3 * d;
  const T* base = qkv + (size_t)at.b * Tn * ld + (size_t)at.h * dh;
  const T* dobase = d_o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  const T* obase = o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  load_rows<T>(t.ra, t.lr, t.lr, base, ld, at.r0, Tn, dh);
  load_rows<T>(t.rb, t.lr, t.lr, dobase, (size_t)d, at.r0, Tn, dh);
  const int row0 = at.r0 + w * RPW;
  const size_t stat = ((size_t)at.b * H + at.h) * Tn;
  float L[RPW], D[RPW], acc[RPW][DPL];
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    const int i = row0 + r;
    float s = 0.f;
    if (i < Tn)
      for (int c = lane; c < dh; c += 32) s = fmaf(to_f<T>(obase[(size_t)i * d + c]), to_f<T>(dobase[(size_t)i * d + c]), s);
    D[r] = warp_sum(s);
    L[r] = i < Tn ? lse[stat + i] : 0.f;
    if (lane == 0 && i < Tn) rowdot[stat + i] = D[r];
#pragma unroll
    for (int c = 0; c < DPL; ++c) acc[r][c] = 0.f;
  }
  const float* qrows = t.ra + w * RPW * t.lr;
  const float* dorows = t.rb + w * RPW * t.lr;
  float* ds_s = t.pa + w * RPW * KT;
  for (int j0 = 0; j0 <= at.r0 + RT - 1 && j0 < Tn; j0 += KT) {
    __syncthreads();
    load_rows<T>(t.a, t.lt, t.lr, base + d, ld, j0, Tn, dh);
    load_rows<T>(t.b, t.lt, t.lr, base + 2 * (size_t)d, ld, j0, Tn, dh);
    __syncthreads();
    float s[RPW], dp[RPW];
    dot4(qrows, t.lr, t.a + lane * t.lt, s);
    dot4(dorows, t.lr, t.b + lane * t.lt, dp);
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const bool vis = j0 + lane <= row0 + r && row0 + r < Tn;
      const float p = vis ? expf(s[r] * scale - L[r]) : 0.f;
      ds_s[r * KT + lane] = vis ? p * (dp[r] - D[r]) * scale : 0.f;
    }
    __syncwarp();
    accumulate_tile<true>(acc, ds_s, t.a, t.lt, lane, nfeat, j0 == at.r0, w);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    if (row0 + r >= Tn) continue;
    T* out = dqkv + ((size_t)at.b * Tn + row0 + r) * ld + (size_t)at.h * dh;
#pragma unroll
    for (int c = 0; c < DPL; ++c) {
      const int dim = lane + 32 * c;
      if (dim < dh) out[dim] = from_f<T>(acc[r][c]);
    }
  }
}

// dK, dV: rows are keys, tiles are queries.  BLOCKS: registers for that many blocks per SM (bwd chooses).
template <typename T, int BLOCKS>
__global__ void __launch_bounds__(WARPS * 32, BLOCKS) attn_bwd_dkv_kernel(const T* __restrict__ qkv, const float* __restrict__ lse,
                                                                  const T* __restrict__ d_o, const float* __restrict__ rowdot,
                                                                  int Tn, int H, int d, T* __restrict__ dqkv) {
  overlap_sync();
  extern __shared__ __align__(16) float sh[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, dh = d / H, nfeat = (dh + 31) / 32;
  const Where at = where(Tn, H);
  Tiles t(sh, dh);
  const float scale = rsqrtf((float)dh);
  const size_t ld = (size_t)3 * d;
  const T* base = qkv + (size_t)at.b * Tn * ld + (size_t)at.h * dh;
  const T* dobase = d_o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  load_rows<T>(t.ra, t.lr, t.lr, base + d, ld, at.r0, Tn, dh);
  load_rows<T>(t.rb, t.lr, t.lr, base + 2 * (size_t)d, ld, at.r0, Tn, dh);
  const int row0 = at.r0 + w * RPW;
  const size_t stat = ((size_t)at.b * H + at.h) * Tn;
  float dk[RPW][DPL], dv[RPW][DPL];
#pragma unroll
  for (int r = 0; r < RPW; ++r)
#pragma unroll
    for (int c = 0; c < DPL; ++c) { dk[r][c] = 0.f; dv[r][c] = 0.f; }
  const float* krows = t.ra + w * RPW * t.lr;
  const float* vrows = t.rb + w * RPW * t.lr;
  float* p_s = t.pa + w * RPW * KT;
  float* ds_s = t.pb + w * RPW * KT;
  for (int i0 = at.r0; i0 < Tn; i0 += KT) {
    __syncthreads();
    load_rows<T>(t.a, t.lt, t.lr, base, ld, i0, Tn, dh);
    load_rows<T>(t.b, t.lt, t.lr, dobase, (size_t)d, i0, Tn, dh);
    __syncthreads();
    const int i = i0 + lane;
    const float L = i < Tn ? lse[stat + i] : 0.f, D = i < Tn ? rowdot[stat + i] : 0.f;
    float s[RPW], dp[RPW];
    dot4(krows, t.lr, t.a + lane * t.lt, s);
    dot4(vrows, t.lr, t.b + lane * t.lt, dp);
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const bool vis = i >= row0 + r && i < Tn;
      const float p = vis ? expf(s[r] * scale - L) : 0.f;
      p_s[r * KT + lane] = p;
      ds_s[r * KT + lane] = vis ? p * (dp[r] - D) * scale : 0.f;
    }
    __syncwarp();
    accumulate_tile<false>(dv, p_s, t.b, t.lt, lane, nfeat, i0 == at.r0, w);
    accumulate_tile<false>(dk, ds_s, t.a, t.lt, lane, nfeat, i0 == at.r0, w);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    if (row0 + r >= Tn) continue;
    T* out = dqkv + ((size_t)at.b * Tn + row0 + r) * ld + (size_t)at.h * dh;
#pragma unroll
    for (int c = 0; c < DPL; ++c) {
      const int dim = lane + 32 * c;
      if (dim < dh) { out[d + dim] = from_f<T>(dk[r][c]); out[2 * (size_t)d + dim] = from_f<T>(dv[r][c]); }
    }
  }
}

// ---- short sequences: a warp per row (attention_rows.cuh) ----
// A tile of 32 rows would be mostly padding, with loads and barriers for the whole of it.
constexpr int ROW_WARPS = 4;

template <typename T>
__global__ void __launch_bounds__(ROW_WARPS * 32) attn_rows_fwd_kernel(const T* __restrict__ qkv, int nseq, int Tn, int H, int d,
                                                                       T* __restrict__ o, float* __restrict__ lse) {
  overlap_sync();
  __shared__ float s[ROW_WARPS][MAX_DH];
  const int64_t w = (int64_t)blockIdx.x * ROW_WARPS + (threadIdx.x >> 5);
  if (w >= (int64_t)nseq * H * Tn) return;
  const int i = (int)(w % Tn), h = (int)((w / Tn) % H), b = (int)(w / ((int64_t)Tn * H));
  const rows::Head<T> hd(qkv, b, h, Tn, H, d);
  rows::forward_row<T>(hd, i, s[threadIdx.x >> 5], o + ((size_t)b * Tn + i) * d + (size_t)h * hd.dh, lse + ((size_t)b * H + h) * Tn + i);
}

// dQ, and D[row] = sum(dO * O) of its row, which the dK/dV kernel (second) reads from `rowdot`
template <typename T>
__global__ void __launch_bounds__(ROW_WARPS * 32) attn_rows_dq_kernel(const T* __restrict__ qkv, const T* __restrict__ o,
                                                                      const float* __restrict__ lse, const T* __restrict__ d_o,
                                                                      float* __restrict__ rowdot, int nseq, int Tn, int H, int d,
                                                                      T* __restrict__ dqkv) {
  overlap_sync();
  __shared__ float s[ROW_WARPS][2 * MAX_DH];
  const int64_t w = (int64_t)blockIdx.x * ROW_WARPS + (threadIdx.x >> 5);
  if (w >= (int64_t)nseq * H * Tn) return;
  const int lane = threadIdx.x & 31, i = (int)(w % Tn), h = (int)((w / Tn) % H), b = (int)(w / ((int64_t)Tn * H));
  const rows::Head<T> hd(qkv, b, h, Tn, H, d);
  const size_t row = ((size_t)b * Tn + i) * d + (size_t)h * hd.dh, stat = ((size_t)b * H + h) * Tn + i;
  float D = 0.f;
  for (int c = lane; c < hd.dh; c += 32) D = fmaf(to_f<T>(o[row + c]), to_f<T>(d_o[row + c]), D);
  D = warp_sum(D);
  if (lane == 0) rowdot[stat] = D;
  rows::dq_row<T>(hd, d_o + row, lse[stat], D, i, s[threadIdx.x >> 5], dqkv + ((size_t)b * Tn + i) * hd.ld + (size_t)h * hd.dh);
}

template <typename T>
__global__ void __launch_bounds__(ROW_WARPS * 32) attn_rows_dkv_kernel(const T* __restrict__ qkv, const float* __restrict__ lse,
                                                                       const T* __restrict__ d_o, const float* __restrict__ rowdot,
                                                                       int nseq, int Tn, int H, int d, T* __restrict__ dqkv) {
  overlap_sync();
  __shared__ float s[ROW_WARPS][2 * MAX_DH];
  const int64_t w = (int64_t)blockIdx.x * ROW_WARPS + (threadIdx.x >> 5);
  if (w >= (int64_t)nseq * H * Tn) return;
  const int j = (int)(w % Tn), h = (int)((w / Tn) % H), b = (int)(w / ((int64_t)Tn * H));
  const rows::Head<T> hd(qkv, b, h, Tn, H, d);
  const size_t stat = ((size_t)b * H + h) * Tn;
  rows::dkv_row<T>(hd, d_o + (size_t)b * Tn * d + (size_t)h * hd.dh, lse + stat, rowdot + stat, j, s[threadIdx.x >> 5],
                   dqkv + ((size_t)b * Tn + j) * hd.ld + d + (size_t)h * hd.dh);
}

// room for the widest head, once per device and kernel
template <typename K> cudaError_t allow_smem(K kernel, PerDeviceOnce& once) {
  const int dev = current_device();
  if (!once.needed(dev)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(MAX_DH));
  if (e == cudaSuccess) once.done(dev);
  return e;
}

template <typename T>
cudaError_t fwd(const void* qkv, unsigned blocks, int T_, int H, int d, void* o, float* lse, cudaStream_t st) {
  static PerDeviceOnce once;
  cudaError_t e = allow_smem(attn_fwd_kernel<T>, once);
  if (e != cudaSuccess) return e;
  return launch_overlapped(attn_fwd_kernel<T>, blocks, WARPS * 32, smem_bytes(d / H), st, (const T*)qkv, T_, H, d, (T*)o, lse);
}

// BLOCKS = 2 where no more blocks than that per SM exist (4 x 64, 8 heads of 32: 20.2 us against 21.8 with registers for
// three), else 3 (42 x 24, 8 heads of 24: 20.9 us against 24.2).  The other kernels: four (forward) and three (dQ).
template <typename T, int BLOCKS>
cudaError_t bwd_blocks(const void* qkv, const void* o, const float* lse, const void* d_o, unsigned blocks, int T_, int H, int d,
                       void* dqkv, float* rowdot, cudaStream_t st) {
  static PerDeviceOnce once_q, once_kv;
  cudaError_t e = allow_smem(attn_bwd_dq_kernel<T>, once_q);
  if (e == cudaSuccess) e = allow_smem(attn_bwd_dkv_kernel<T, BLOCKS>, once_kv);
  if (e != cudaSuccess) return e;
  e = launch_overlapped(attn_bwd_dq_kernel<T>, blocks, WARPS * 32, smem_bytes(d / H), st, (const T*)qkv, (const T*)o, lse,
                      (const T*)d_o, rowdot, T_, H, d, (T*)dqkv);
  if (e != cudaSuccess) return e;
  return launch_overlapped(attn_bwd_dkv_kernel<T, BLOCKS>, blocks, WARPS * 32, smem_bytes(d / H), st, (const T*)qkv, lse, (const T*)d_o,
                         rowdot, T_, H, d, (T*)dqkv);
}

template <typename T>
cudaError_t bwd(const void* qkv, const void* o, const float* lse, const void* d_o, unsigned blocks, int T_, int H, int d,
                void* dqkv, float* rowdot, cudaStream_t st) {
  return (int64_t)blocks <= 2 * num_sms() ? bwd_blocks<T, 2>(qkv, o, lse, d_o, blocks, T_, H, d, dqkv, rowdot, st)
                                          : bwd_blocks<T, 3>(qkv, o, lse, d_o, blocks, T_, H, d, dqkv, rowdot, st);
}

// Whether a warp per row beats tiles of 32 rows: forward up to 10 rows, backward up to 9 (10 up to width 32), and up to 16
// while all the rows are at work at once.  us, forward / backward, rows against tiles, fp32: 8192 heads of 1 x 128 12 / 39
// against 277 / 803; 2048 of 8 x 64 29 / 101 against 45 / 133, of 10 x 64 39 / 142 against 46 / 133, of 12 x 64 51 / 189
// against 47 / 134; 32 of 16 x 64 7.6 / 17 against 7.7 / 19, 128 of them 13 / 41 against 8 / 19.
bool by_rows(int nseq, int T, int H, int d, bool forward) {
  return T <= (forward || d / H <= 32 ? 10 : 9) || (T <= 16 && (int64_t)nseq * H * T <= 4 * num_sms());
}

bool grid_of(int nseq, int T, int H, int d, bool rows, unsigned* blocks) {
  if (d % H != 0 || d / H > MAX_DH) return false;
  const int64_t items = (int64_t)nseq * H, n = rows ? (items * T + ROW_WARPS - 1) / ROW_WARPS : items * ((T + RT - 1) / RT);
  *blocks = (unsigned)n;
  return n <= 0x7fffffff;
}

template <typename T>
cudaError_t fwd_rows(const void* qkv, unsigned blocks, int nseq, int T_, int H, int d, void* o, float* lse, cudaStream_t st) {
  return launch_overlapped(attn_rows_fwd_kernel<T>, blocks, ROW_WARPS * 32, 0, st, (const T*)qkv, nseq, T_, H, d, (T*)o, lse);
}

template <typename T>
cudaError_t bwd_rows(const void* qkv, const void* o, const float* lse, const void* d_o, unsigned blocks, int nseq, int T_, int H,
                     int d, void* dqkv, float* rowdot, cudaStream_t st) {
  cudaError_t e = launch_overlapped(attn_rows_dq_kernel<T>, blocks, ROW_WARPS * 32, 0, st, (const T*)qkv, (const T*)o, lse,
                                    (const T*)d_o, rowdot, nseq, T_, H, d, (T*)dqkv);
  if (e != cudaSuccess) return e;
  return launch_overlapped(attn_rows_dkv_kernel<T>, blocks, ROW_WARPS * 32, 0, st, (const T*)qkv, lse, (const T*)d_o, rowdot, nseq,
                           T_, H, d, (T*)dqkv);
}

}  // namespace

cudaError_t attention_fwd_simt(int dt, const void* qkv, int nseq, int T, int H, int d, void* o, float* lse,
                               cudaStream_t st) {
  unsigned blocks;
  const bool rows = by_rows(nseq, T, H, d, true);
  if (!grid_of(nseq, T, H, d, rows, &blocks)) return cudaErrorInvalidValue;
  if (rows) return dt == DT_BF16 ? fwd_rows<bf16>(qkv, blocks, nseq, T, H, d, o, lse, st) : fwd_rows<float>(qkv, blocks, nseq, T, H, d, o, lse, st);
  return dt == DT_BF16 ? fwd<bf16>(qkv, blocks, T, H, d, o, lse, st) : fwd<float>(qkv, blocks, T, H, d, o, lse, st);
}

cudaError_t attention_bwd_simt(int dt, const void* qkv, const void* o, const float* lse, const void* d_o,
                               int nseq, int T, int H, int d, void* dqkv, float* rowdot, cudaStream_t st) {
  unsigned blocks;
  const bool rows = by_rows(nseq, T, H, d, false);
  if (!grid_of(nseq, T, H, d, rows, &blocks)) return cudaErrorInvalidValue;
  if (rows)
    return dt == DT_BF16 ? bwd_rows<bf16>(qkv, o, lse, d_o, blocks, nseq, T, H, d, dqkv, rowdot, st)
                         : bwd_rows<float>(qkv, o, lse, d_o, blocks, nseq, T, H, d, dqkv, rowdot, st);
  return dt == DT_BF16 ? bwd<bf16>(qkv, o, lse, d_o, blocks, T, H, d, dqkv, rowdot, st)
                       : bwd<float>(qkv, o, lse, d_o, blocks, T, H, d, dqkv, rowdot, st);
}

}  // namespace sl
