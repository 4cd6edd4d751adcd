// Rank-r projections of the LoRA path (h = u A^T, dh = s dy B) as their own kernel: a product whose output is a few dozen
// columns wide, so it is a pass over the rows of X and nothing else.
//   Y[M, ext] = X[M, K] W[ext, K]^T,  W and Y padded per target to rp columns, of which r are used
// X is cut into slabs of at most 1024 columns (for dh: the slices of dqkv that have adapters).  Whole row pieces of a slab,
// 16 rows at a time, are copied into a ring in shared memory; eight warps share the contraction, 32 columns at a time, with
// mma.sync, add their partial sums in shared memory in warp order and write the padded rows of Y.  A CTA walks a
// range of consecutive 16-row tiles and keeps the fragments of W that its warps need in registers all the while (they are
// loaded again where the next client's rows begin).  Both operands' fragments are 16-byte vectors: the contraction index may
// be permuted freely as long as both sides agree, so thread t of a quad takes elements [8 t, 8 t + 8) of 32 for both 16-deep
// steps.  Only the column tiles of 8 that hold adapters are computed, of a slab that is one target's slice only that
// target's; the padding is written as zeros.
// What bounds it: over few rows the latency of one pass; over many rows the read of X, at which the linear-layer kernels'
// narrow tiles are as good or better (LORA_PROJ_ROWS).
// norm_proj_kernel is the forward projection with the norm in front of it: u = LayerNorm(x) (or RMSNorm), h = u A^T.
#include "adapter_copies.cuh"
#include "common.cuh"
#include "host_common.h"
#include "kernels.h"
#include "launch.cuh"
#include "tc_common.cuh"

namespace sl {
namespace {

using namespace tc;

constexpr int WARPS = 8, THREADS = 32 * WARPS; // (a ninth warp for the copies would cost registers: two CTAs of nine take 96 per thread)
constexpr int ROWS = 16;                       // of a tile
constexpr int SLAB = 1024;                     // columns of a slab at most: four chunks of 32 per warp
constexpr int CHUNKS = SLAB / (32 * WARPS);
constexpr int MAX_STAGES = 4;                  // of the ring; as many as leave room for two CTAs per SM (launch)
constexpr int MAX_TILES = 4;                   // column tiles of 8 of Y: slabs * tiles bounds the fragments of W in registers, for two CTAs per SM
constexpr int MAX_EXT = 512;                   // columns of Y, padding included

struct Proj {
  const bf16* X; int64_t ldx;
  const bf16* W; int64_t ldw, w_gs;            // w_gs: elements between the W of two groups (0: shared)
  const float* W32; int w_rows;                // one target's W in fp32, w_rows rows, instead
  bf16* Y;
  int M, rows_per_group, ext;
  int slab_len, last_len, slab_col[4];         // columns of the slabs (and of the last one), first column of each in X and W
  int stages;
  int pitch;                                   // bytes of a row in the ring: an odd number of 64-byte pieces (no bank conflicts)
  int tile_col[MAX_TILES];                     // first output column of each column tile
  int8_t tile_of[MAX_EXT / 8];                  // ext / 8 entries: the tile that holds columns [8 i, 8 i + 8), or -1
  int* status;
};

__device__ __forceinline__ void mma16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 ld16(const bf16* p, bool ok) {
  return ok ? *reinterpret_cast<const uint4*>(p) : make_uint4(0u, 0u, 0u, 0u);
}
// eight fp32 values as bf16
__device__ __forceinline__ uint4 ld8f(const float* p, bool ok) {
  if (!ok) return make_uint4(0u, 0u, 0u, 0u);
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  Vec16<bf16> v;
  v.set(0, a.x); v.set(1, a.y); v.set(2, a.z); v.set(3, a.w); v.set(4, b.x); v.set(5, b.y); v.set(6, b.z); v.set(7, b.w);
  return v.raw;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Adds the eight warps' partial sums of 16 rows in warp order and writes the rows of Y, eight columns (16 bytes) per thread.
template <int TILES>
__device__ __forceinline__ void store_rows(const Proj& p, const float (*red)[ROWS][8 * TILES], int row0) {
  const int per_row = p.ext / 8;
  for (int v = threadIdx.x; v < ROWS * per_row; v += THREADS) {
    const int r = v / per_row, c8 = v % per_row;
    if (row0 + r >= p.M) continue;
    const int n = p.tile_of[c8];
    uint32_t out[4] = {0u, 0u, 0u, 0u};
    if (n >= 0) {
      float sum[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) sum[e] = 0.f;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        const float4* part = reinterpret_cast<const float4*>(&red[w][r][8 * n]);
        const float4 a = part[0], b = part[1];
        sum[0] += a.x; sum[1] += a.y; sum[2] += a.z; sum[3] += a.w;
        sum[4] += b.x; sum[5] += b.y; sum[6] += b.z; sum[7] += b.w;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 o = __floats2bfloat162_rn(sum[2 * e], sum[2 * e + 1]);
        out[e] = *reinterpret_cast<const uint32_t*>(&o);
      }
    }
    *reinterpret_cast<uint4*>(p.Y + (int64_t)(row0 + r) * p.ext + 8 * c8) = make_uint4(out[0], out[1], out[2], out[3]);
  }
}
template <int TILES>
__device__ __forceinline__ void put_partial(float (*mine)[8 * TILES], const float (*acc)[4], int g, int t) {
#pragma unroll
  for (int n = 0; n < TILES; ++n) {
    *reinterpret_cast<float2*>(&mine[g][8 * n + 2 * t]) = make_float2(acc[n][0], acc[n][1]);
    *reinterpret_cast<float2*>(&mine[g + 8][8 * n + 2 * t]) = make_float2(acc[n][2], acc[n][3]);
  }
}

// SLABS of X; N column tiles per slab; SEPARATE: every slab has tiles of its own (N * SLABS in all).
// COPIES: W comes in fp32 (rounded to bf16 on the way, as the compute copies are), and the CTAs past `workers` write the
// layer's compute copies, which the launches after this one need: one launch less in a layer of six.
template <int SLABS, int N, bool SEPARATE, bool COPIES>
__global__ void __launch_bounds__(THREADS, 2)
proj_kernel(const __grid_constant__ Proj p, int workers, const __grid_constant__ AdapterCopyArgs copies, int64_t copy_vectors) {
  constexpr int TILES = SEPARATE ? SLABS * N : N, COLS = 8 * TILES;
  static_assert(SLABS * N <= MAX_TILES, "registers for two CTAs per SM");
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t bars[2 * MAX_STAGES];
  __shared__ __align__(16) float red[2][WARPS][ROWS][COLS];
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint32_t ring = smem_u32(smem), bar = smem_u32(bars);
  auto FULL = [&](int s) { return bar + 8u * s; };
  auto EMPTY = [&](int s) { return bar + 8u * (MAX_STAGES + s); };
  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(FULL(s), 1); mbar_init(EMPTY(s), WARPS); }
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  overlap_sync();
  if constexpr (COPIES) {
    if ((int)blockIdx.x >= workers) {
      write_copy_vector<bf16>(copies, (int64_t)((int)blockIdx.x - workers) * THREADS + threadIdx.x, copy_vectors);
      return;
    }
  }
  const int tiles = (p.M + ROWS - 1) / ROWS;
  const int t0 = (int)((int64_t)tiles * blockIdx.x / workers), t1 = (int)((int64_t)tiles * (blockIdx.x + 1) / workers);
  const uint32_t stage_bytes = (uint32_t)(ROWS * p.pitch);
  auto len = [&](int sl) { return sl == SLABS - 1 ? p.last_len : p.slab_len; };

  // warp 0 copies, one row piece per lane: use `q` of the ring is slab q % SLABS of tile t0 + q / SLABS
  const int uses = (t1 - t0) * SLABS;
  auto copy = [&](int q, int s) {
    const int row0 = (t0 + q / SLABS) * ROWS, rows = min(ROWS, p.M - row0), sl = q % SLABS;
    const uint32_t bytes = (uint32_t)len(sl) * 2u;
    if (lane == 0) mbar_expect_tx(FULL(s), bytes * (uint32_t)rows);
    __syncwarp();
    if (lane < rows) bulk_load(ring + s * stage_bytes + (uint32_t)(lane * p.pitch), p.X + (int64_t)(row0 + lane) * p.ldx + p.slab_col[sl], bytes, FULL(s));
  };
  if (warp == 0)
    for (int q = 0; q < p.stages && q < uses; ++q) copy(q, q);

  uint4 w[SLABS][CHUNKS][N];
  auto load_w = [&](int row0) {
    const int64_t off = p.w_gs ? (int64_t)(row0 / p.rows_per_group) * p.w_gs : 0;
#pragma unroll
    for (int sl = 0; sl < SLABS; ++sl)
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c)
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const int k = (c * WARPS + warp) * 32 + 8 * t, col = p.tile_col[SEPARATE ? sl * N + n : n] + g;
          const int64_t at = off + (int64_t)col * p.ldw + p.slab_col[sl] + k;
          if constexpr (COPIES) w[sl][c][n] = ld8f(p.W32 + at, k < len(sl) && col < p.w_rows);
          else w[sl][c][n] = ld16(p.W + at, k < len(sl));
        }
  };
  int group = -1, q = 0, s = 0, before = 0;    // use, its stage, the stage of the use before
  uint32_t phase = 0, phase_before = 0;
  bool ok = true;
  for (int tile = t0; tile < t1; ++tile) {
    const int row0 = tile * ROWS, gr = p.w_gs ? row0 / p.rows_per_group : 0;
    if (gr != group) { load_w(row0); group = gr; }
    float acc[TILES][4];
#pragma unroll
    for (int n = 0; n < TILES; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll
    for (int sl = 0; sl < SLABS; ++sl) {
      if (warp == 0 && q > 0 && q - 1 + p.stages < uses) {     // into the stage the use before this one has left
        ok = ok && mbar_wait_warp(EMPTY(before), phase_before, abort_flag, p.status, 81);
        if (ok) copy(q - 1 + p.stages, before);
      }
      ok = ok && mbar_wait_warp(FULL(s), phase, abort_flag, p.status, 82);
      const uint8_t* st = smem + s * stage_bytes;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        const int k0 = (c * WARPS + warp) * 32, k = k0 + 8 * t;
        if (k0 >= len(sl)) break;
        uint4 x0 = make_uint4(0u, 0u, 0u, 0u), x1 = x0;
        if (k < len(sl)) {
          x0 = *reinterpret_cast<const uint4*>(st + g * p.pitch + 2 * k);
          x1 = *reinterpret_cast<const uint4*>(st + (g + 8) * p.pitch + 2 * k);
        }
#pragma unroll
        for (int n = 0; n < N; ++n) {
          float* a = acc[SEPARATE ? sl * N + n : n];
          const uint4 v = w[sl][c][n];
          mma16816(a, x0.x, x1.x, x0.y, x1.y, v.x, v.y);
          mma16816(a, x0.z, x1.z, x0.w, x1.w, v.z, v.w);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(EMPTY(s));
      before = s; phase_before = phase; ++q;
      if (++s == p.stages) { s = 0; phase ^= 1u; }
    }
    put_partial<TILES>(red[tile & 1][warp], acc, g, t);
    __syncthreads();                           // (the other buffer's readers are past the barrier before this one)
    store_rows<TILES>(p, red[tile & 1], row0);
  }
  // (a wait that has run out: let the copies in flight land before the CTA exits)
  if (!ok) for (int i = 0; i < 2000; ++i) __nanosleep(1000);
}

// u = norm(x) and Y = u W^T from the rows in shared memory: 16 rows a block, two per warp, each read once into registers (at
// most NV vectors of 8 per lane); the W of the product is asked for before the statistics where its vectors fit in registers.
struct NormIn { const bf16 *x, *g, *b; bf16* u; float *mean, *rstd; int d; float eps; };
template <int NV, int NT, bool RMS>
__global__ void __launch_bounds__(THREADS) norm_proj_kernel(const __grid_constant__ Proj p, const __grid_constant__ NormIn in) {
  overlap_sync();
  extern __shared__ __align__(16) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int row0 = blockIdx.x * 16, d = in.d, ld = d + 32;       // rows an odd number of 64-byte pieces apart: no bank conflicts
  bf16* us = reinterpret_cast<bf16*>(smem);
  const bf16* W = p.W + (p.w_gs ? (int64_t)(row0 / p.rows_per_group) * p.w_gs : 0);
  constexpr bool AHEAD = NV * NT <= 8;
  uint4 w[AHEAD ? NV : 1][NT];
  auto load_w = [&](int it, uint4* dst) {
    const int k = (it * WARPS + warp) * 32 + 8 * t;
#pragma unroll
    for (int n = 0; n < NT; ++n) dst[n] = ld16(W + (int64_t)(p.tile_col[n] + g) * p.ldw + k, k < d);
  };
  if (AHEAD) {
#pragma unroll
    for (int it = 0; it < NV; ++it) load_w(it, w[AHEAD ? it : 0]);
  }
  Vec16<bf16> xv[2][NV];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int row = row0 + 2 * warp + h;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int c = (k * 32 + lane) * 8;
      xv[h][k].raw = ld16(in.x + (int64_t)row * d + c, row < p.M && c < d);
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = 2 * warp + h, row = row0 + r;
    float mu = 0.f, q = 0.f;
    if (!RMS) {
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int i = 0; i < 8; ++i) s += xv[h][k].get(i);
      mu = warp_sum(s) / d;
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      if ((k * 32 + lane) * 8 >= d) break;
#pragma unroll
      for (int i = 0; i < 8; ++i) { const float z = xv[h][k].get(i) - mu; q += z * z; }
    }
    const float rs = rsqrtf(warp_sum(q) / d + in.eps);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int c = (k * 32 + lane) * 8;
      if (c >= d) break;
      Vec16<bf16> gv, bv, o;
      gv.load(in.g + c);
      if (!RMS) bv.load(in.b + c);
#pragma unroll
      for (int i = 0; i < 8; ++i) o.set(i, RMS ? xv[h][k].get(i) * rs * gv.get(i) : (xv[h][k].get(i) - mu) * rs * gv.get(i) + bv.get(i));
      if (row >= p.M) o.raw = make_uint4(0u, 0u, 0u, 0u);
      else o.store(in.u + (int64_t)row * d + c);
      o.store(us + r * ld + c);
    }
    if (lane == 0 && row < p.M) {
      if (!RMS) in.mean[row] = mu;
      in.rstd[row] = rs;
    }
  }
  __syncthreads();
  float acc[NT][4];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll
  for (int it = 0; it < NV; ++it) {
    const int k = (it * WARPS + warp) * 32 + 8 * t;
    uint4* wv = w[AHEAD ? it : 0];
    if (!AHEAD) load_w(it, wv);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    const uint4 x0 = k < d ? *reinterpret_cast<const uint4*>(us + g * ld + k) : z, x1 = k < d ? *reinterpret_cast<const uint4*>(us + (g + 8) * ld + k) : z;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      mma16816(acc[n], x0.x, x1.x, x0.y, x1.y, wv[n].x, wv[n].y);
      mma16816(acc[n], x0.z, x1.z, x0.w, x1.w, wv[n].z, wv[n].w);
    }
  }
  auto red = reinterpret_cast<float (*)[ROWS][8 * NT]>(smem + ROWS * ld * 2);
  put_partial<NT>(red[warp], acc, g, t);
  __syncthreads();
  store_rows<NT>(p, red, row0);
}

// fp32: LayerNorm and the projection of a row by one warp, the row in registers (at most NV vectors of 4 per lane); one dot
// product with a row of W after another.  Over few rows the two launches it replaces were 8 us of a layer's 65.
template <int NV>
__global__ void __launch_bounds__(THREADS) norm_proj_f32_kernel(const float* __restrict__ x, const float* __restrict__ gain, const float* __restrict__ shift,
                                                                float* __restrict__ u, float* __restrict__ mean, float* __restrict__ rstd, float eps,
                                                                const float* __restrict__ W, int64_t w_gs, int rows_per_group, float* __restrict__ Y,
                                                                int M, int d, int ext, int nt, int r, int rp) {
  overlap_sync();
  const int row = (int)blockIdx.x * WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= M) return;
  if (w_gs) W += (int64_t)(row / rows_per_group) * w_gs;
  float4 v[NV];
  float s = 0.f, q = 0.f;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int c = (k * 32 + lane) * 4;
    v[k] = c < d ? *reinterpret_cast<const float4*>(x + (int64_t)row * d + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    s += v[k].x; s += v[k].y; s += v[k].z; s += v[k].w;
  }
  const float mu = warp_sum(s) / d;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    if ((k * 32 + lane) * 4 >= d) break;
    float t;
    t = v[k].x - mu; q += t * t; t = v[k].y - mu; q += t * t; t = v[k].z - mu; q += t * t; t = v[k].w - mu; q += t * t;
  }
  const float rs = rsqrtf(warp_sum(q) / d + eps);
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int c = (k * 32 + lane) * 4;
    if (c >= d) break;
    const float4 gv = *reinterpret_cast<const float4*>(gain + c), bv = *reinterpret_cast<const float4*>(shift + c);
    v[k] = make_float4((v[k].x - mu) * rs * gv.x + bv.x, (v[k].y - mu) * rs * gv.y + bv.y, (v[k].z - mu) * rs * gv.z + bv.z, (v[k].w - mu) * rs * gv.w + bv.w);
    *reinterpret_cast<float4*>(u + (int64_t)row * d + c) = v[k];
  }
  if (lane == 0) { mean[row] = mu; rstd[row] = rs; }
  float mine = 0.f;                              // lane i: component i of nt * r
  for (int i = 0; i < nt * r; ++i) {
    const float* w = W + (int64_t)(i / r * rp + i % r) * d;
    float dot = 0.f;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int c = (k * 32 + lane) * 4;
      if (c >= d) break;
      const float4 a = *reinterpret_cast<const float4*>(w + c);
      dot = fmaf(v[k].w, a.w, fmaf(v[k].z, a.z, fmaf(v[k].y, a.y, fmaf(v[k].x, a.x, dot))));
    }
    dot = warp_sum(dot);
    if (lane == i) mine = dot;
  }
  for (int c0 = 0; c0 < ext; c0 += 32) {
    const int c = c0 + lane, t = c / rp, j = c % rp;
    const bool used = t < nt && j < r;
    const float h = __shfl_sync(0xffffffffu, mine, used ? t * r + j : 0);
    if (c < ext) Y[(int64_t)row * ext + c] = used ? h : 0.f;
  }
}

template <int SLABS, int N, bool SEPARATE, bool COPIES>
cudaError_t launch(Proj p, const AdapterCopyArgs& copies, cudaStream_t st) {
  const auto kernel = proj_kernel<SLABS, N, SEPARATE, COPIES>;
  // two CTAs per SM (228 KB, of which each takes 1 KB and its static part)
  constexpr int STATIC = 2 * WARPS * ROWS * 8 * (SEPARATE ? SLABS * N : N) * 4 + 1024;
  constexpr int ROOM = (228 * 1024) / 2 - 1024 - STATIC;
  p.stages = ROOM / (ROWS * p.pitch);
  p.stages = p.stages > MAX_STAGES ? MAX_STAGES : p.stages;
  const int smem = p.stages * ROWS * p.pitch;
  static_assert(ROOM >= 2 * ROWS * (2 * SLAB + 192), "");
  static PerDeviceOnce once;
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ROOM);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  const int tiles = (p.M + ROWS - 1) / ROWS, slots = 2 * num_sms();
  const int workers = tiles < slots ? tiles : slots;
  const int64_t vectors = COPIES ? adapter_copy_vectors(copies) : 0;
  return launch_overlapped(kernel, (unsigned)(workers + (vectors + THREADS - 1) / THREADS), THREADS, smem, st, p, workers, copies, vectors);
}

struct Shape { int slabs = 0, n = 0; bool separate = false; };
// Slabs and column tiles of a projection (slabs 0: not one of these kernels' shapes).  The fragments of W that a thread keeps
// (four vectors per slab and tile) bound slabs * tiles.
Shape shape_of(const ProjArgs& a) {
  Shape s;
  const int per_target = (a.r + 7) / 8;
  s.separate = a.nt > 1 && a.k_slice > 0;
  s.slabs = s.separate ? a.nt : (a.K + SLAB - 1) / SLAB;
  s.n = s.separate ? per_target : a.nt * per_target;
  const bool fits = s.separate ? a.k_slice <= SLAB && s.slabs <= 3 && s.slabs * s.n <= MAX_TILES : (s.slabs == 1 && s.n <= 4) || (s.slabs == 2 && s.n <= 2) || (s.slabs <= 4 && s.n == 1);
  if (!fits) s.slabs = 0;
  return s;
}

void fill(const ProjArgs& a, const Shape& s, Proj& p) {
  p.X = (const bf16*)a.X; p.ldx = a.ldx; p.W = (const bf16*)a.W; p.ldw = a.ldw;
  p.w_gs = a.rows_per_group > 0 && a.rows_per_group < a.M ? a.w_group_stride : 0;
  p.W32 = nullptr; p.w_rows = a.r;
  p.Y = (bf16*)a.Y; p.M = a.M; p.rows_per_group = a.rows_per_group; p.ext = a.ext;
  p.slab_len = s.separate ? a.k_slice : ((a.K + s.slabs - 1) / s.slabs + 7) / 8 * 8;
  p.last_len = s.separate ? a.k_slice : a.K - (s.slabs - 1) * p.slab_len;
  for (int i = 0; i < 4; ++i) p.slab_col[i] = i >= s.slabs ? 0 : s.separate ? a.slice_col[i] : i * p.slab_len;
  p.pitch = (2 * p.slab_len + 127) / 128 * 128 + 64;
  int n = 0;
  for (int i = 0; i < MAX_EXT / 8; ++i) p.tile_of[i] = -1;
  for (int t = 0; t < a.nt; ++t)
    for (int j = 0; j < a.r; j += 8) {
      p.tile_col[n] = t * a.rp + j;
      p.tile_of[p.tile_col[n] / 8] = (int8_t)n;
      ++n;
    }
  for (; n < MAX_TILES; ++n) p.tile_col[n] = p.tile_col[0];
  p.status = a.status;
}

template <bool COPIES>
cudaError_t launch_plain(const Shape& s, const Proj& p, const AdapterCopyArgs& copies, cudaStream_t st) {
  if (!s.separate) {
    switch (s.slabs * 8 + s.n) {
      case 8 + 1: return launch<1, 1, false, COPIES>(p, copies, st);
      case 8 + 2: return launch<1, 2, false, COPIES>(p, copies, st);
      case 8 + 3: return launch<1, 3, false, COPIES>(p, copies, st);
      case 8 + 4: return launch<1, 4, false, COPIES>(p, copies, st);
      case 16 + 1: return launch<2, 1, false, COPIES>(p, copies, st);
      case 16 + 2: return launch<2, 2, false, COPIES>(p, copies, st);
      case 24 + 1: return launch<3, 1, false, COPIES>(p, copies, st);
      case 32 + 1: return launch<4, 1, false, COPIES>(p, copies, st);
    }
    return cudaErrorInvalidValue;
  }
  if constexpr (!COPIES) {
    switch (s.slabs * 8 + s.n) {
      case 16 + 1: return launch<2, 1, true, false>(p, copies, st);
      case 16 + 2: return launch<2, 2, true, false>(p, copies, st);
      case 24 + 1: return launch<3, 1, true, false>(p, copies, st);
    }
  }
  return cudaErrorInvalidValue;
}
constexpr int norm_proj_smem(int nv, int nt) { return ROWS * (nv * 256 + 32) * 2 + WARPS * ROWS * 8 * nt * 4; }
template <int NV, int NT, bool RMS>
cudaError_t launch_norm(const Proj& p, const NormIn& in, cudaStream_t st) {
  constexpr int SMEM = norm_proj_smem(NV, NT);
  if constexpr (SMEM > 48 * 1024) {
    static PerDeviceOnce once;
    const int dev = current_device();
    if (once.needed(dev)) {
      cudaError_t e = cudaFuncSetAttribute(norm_proj_kernel<NV, NT, RMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
      if (e != cudaSuccess) return e;
      once.done(dev);
    }
  }
  return launch_overlapped(norm_proj_kernel<NV, NT, RMS>, (p.M + ROWS - 1) / ROWS, THREADS, SMEM, st, p, in);
}
template <int NT, bool RMS>
cudaError_t launch_norm_width(const Proj& p, const NormIn& in, cudaStream_t st) {
  switch ((in.d + 255) / 256) {
    case 1: return launch_norm<1, NT, RMS>(p, in, st);
    case 2: return launch_norm<2, NT, RMS>(p, in, st);
    case 3: return launch_norm<3, NT, RMS>(p, in, st);
    default: return launch_norm<4, NT, RMS>(p, in, st);
  }
}
template <bool RMS>
cudaError_t launch_norm_tiles(int n, const Proj& p, const NormIn& in, cudaStream_t st) {
  switch (n) {
    case 1: return launch_norm_width<1, RMS>(p, in, st);
    case 2: return launch_norm_width<2, RMS>(p, in, st);
    case 3: return launch_norm_width<3, RMS>(p, in, st);
    default: return launch_norm_width<4, RMS>(p, in, st);
  }
}

bool with_status(Proj& p) {
  if (!p.status) p.status = library_status_word();
  return p.status != nullptr;
}

}  // namespace

bool lora_proj_supported(const ProjArgs& a) {
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (a.M < 1 || a.K < 8 || a.K % 8 || a.ldx % 8 || a.ldw % 8 || a.w_group_stride % 8 || a.k_slice % 8) return false;
  if (a.r < 1 || a.nt < 1 || a.ext % 8 || a.ext > MAX_EXT || a.rp % 8 || a.r > a.rp || a.nt * a.rp > a.ext) return false;
  if (a.rows_per_group > 0 && a.rows_per_group < a.M && (a.rows_per_group % ROWS || a.M % a.rows_per_group)) return false;
  return al16(a.X) && al16(a.W) && al16(a.Y) && shape_of(a).slabs > 0;
}

cudaError_t lora_proj(const ProjArgs& a, cudaStream_t st) {
  if (!lora_proj_supported(a)) return cudaErrorInvalidValue;
  Proj p;
  fill(a, shape_of(a), p);
  return with_status(p) ? launch_plain<false>(shape_of(a), p, AdapterCopyArgs(), st) : cudaErrorNotSupported;
}

// a.W, ldw, w_group_stride: fp32 [r, K] of the one target
cudaError_t lora_proj_copies(const ProjArgs& a, const AdapterCopyArgs& copies, cudaStream_t st) {
  if (!lora_proj_supported(a) || a.nt != 1 || copies.dtype != DT_BF16) return cudaErrorInvalidValue;
  Proj p;
  fill(a, shape_of(a), p);
  p.W32 = (const float*)a.W; p.W = nullptr;
  return with_status(p) ? launch_plain<true>(shape_of(a), p, copies, st) : cudaErrorNotSupported;
}

// a.X: where the normalised rows go (ldx = K = d), which are also what is projected
bool norm_proj_supported(const ProjArgs& a) {
  const Shape s = shape_of(a);
  return lora_proj_supported(a) && s.slabs == 1 && !s.separate && a.ldx == a.K;
}
cudaError_t norm_proj(bool rms, const void* x, const void* g, const void* b, float* mean, float* rstd, float eps, const ProjArgs& a, cudaStream_t st) {
  if (!norm_proj_supported(a)) return cudaErrorInvalidValue;
  const Shape s = shape_of(a);
  Proj p;
  fill(a, s, p);
  const NormIn in = {(const bf16*)x, (const bf16*)g, (const bf16*)b, (bf16*)const_cast<void*>(a.X), mean, rstd, a.K, eps};
  return rms ? launch_norm_tiles<true>(s.n, p, in, st) : launch_norm_tiles<false>(s.n, p, in, st);
}

bool norm_proj_f32_supported(const ProjArgs& a) {
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  return a.K % 4 == 0 && a.K <= 1024 && a.ldx == a.K && a.ldw == a.K && a.nt * a.r <= 32 && al16(a.X) && al16(a.W) &&
         (a.rows_per_group <= 0 || a.w_group_stride % 4 == 0);
}
cudaError_t norm_proj_f32(const void* x, const void* g, const void* b, float* mean, float* rstd, float eps, const ProjArgs& a, cudaStream_t st) {
  if (!norm_proj_f32_supported(a)) return cudaErrorInvalidValue;
  const int64_t w_gs = a.rows_per_group > 0 && a.rows_per_group < a.M ? a.w_group_stride : 0;
  auto go = [&](auto kernel) {
    return launch_overlapped(kernel, (a.M + WARPS - 1) / WARPS, THREADS, 0, st, (const float*)x, (const float*)g, (const float*)b, (float*)const_cast<void*>(a.X),
                             mean, rstd, eps, (const float*)a.W, w_gs, a.rows_per_group, (float*)a.Y, a.M, a.K, a.ext, a.nt, a.r, a.rp);
  };
  return a.K <= 256 ? go(norm_proj_f32_kernel<2>) : a.K <= 512 ? go(norm_proj_f32_kernel<4>) : go(norm_proj_f32_kernel<8>);
}

}  // namespace sl
