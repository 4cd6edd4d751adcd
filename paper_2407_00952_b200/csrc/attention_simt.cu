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

// Shared memory, in floats: two tiles [32][width + 1], width = dh rounded up to 32 so that "one feature per lane" reads
// stay inside a row (the odd stride keeps "one row per lane" reads conflict-free), two row blocks [32][dh rounded up to
// 4] (read as float4 broadcasts, zero past dh), two [32][32] blocks of per-row tile values.
__host__ __device__ constexpr int pad4(int dh) { return (dh + 3) & ~3; }
__host__ __device__ constexpr int tile_stride(int dh) { return ((dh + 31) & ~31) + 1; }
// (three tiles where the dK/dV blocks read O)
inline size_t smem_bytes(int dh, bool with_o) { return (size_t)((with_o ? 3 : 2) * KT * tile_stride(dh) + 2 * RT * pad4(dh) + 2 * RT * KT) * 4; }

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

// A 32-row block of a matrix on its way from global to shared memory: NF pieces of four columns per thread (NF: head width
// over 32, rounded up), zero past the last row and column.  `vec`: every piece is an aligned vector.
template <typename T, int NF> struct Block {
  float4 v[NF];
  __device__ __forceinline__ void load(const T* src, size_t ld, int row0, int rows, int dh, bool vec) {
    const int per_row = pad4(dh) / 4;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      const int i = threadIdx.x + k * WARPS * 32, r = i / per_row, c = i % per_row * 4;
      v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r >= 32 || row0 + r >= rows) continue;
      const T* p = src + (size_t)(row0 + r) * ld + c;
      if (vec) {
        if constexpr (sizeof(T) == 4) v[k] = *reinterpret_cast<const float4*>(p);
        else {
          const uint2 w = *reinterpret_cast<const uint2*>(p);
          v[k] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
        }
      } else {
        v[k].x = to_f<T>(p[0]);
        if (c + 1 < dh) v[k].y = to_f<T>(p[1]);
        if (c + 2 < dh) v[k].z = to_f<T>(p[2]);
        if (c + 3 < dh) v[k].w = to_f<T>(p[3]);
      }
    }
  }
  // as [32][ld]: rows of float4 (ld a multiple of 4), or a tile of odd stride
  template <bool TILE> __device__ __forceinline__ void put(float* dst, int ld, int dh) const {
    const int per_row = pad4(dh) / 4;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      const int i = threadIdx.x + k * WARPS * 32, r = i / per_row, c = i % per_row * 4;
      if (r >= 32) continue;
      float* p = dst + r * ld + c;
      if constexpr (TILE) { p[0] = v[k].x; p[1] = v[k].y; p[2] = v[k].z; p[3] = v[k].w; }
      else *reinterpret_cast<float4*>(p) = v[k];
    }
  }
};

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
template <int NF>
__device__ __forceinline__ void accumulate4(float (*acc)[NF], const float* p, const float* tile, int lt, int lane, int j0, int j1) {
#pragma unroll 2
  for (int j = j0; j < j1; j += 4) {
    float4 pv[RPW];
#pragma unroll
    for (int r = 0; r < RPW; ++r) pv[r] = *reinterpret_cast<const float4*>(p + r * KT + j);
#pragma unroll
    for (int c = 0; c < NF; ++c) {
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
template <int NF, bool UP_TO>
__device__ __forceinline__ void accumulate_diagonal(float (*acc)[NF], const float* p, const float* tile, int lt, int lane, int j) {
  float pv[RPW][4];
#pragma unroll
  for (int r = 0; r < RPW; ++r) *reinterpret_cast<float4*>(pv[r]) = *reinterpret_cast<const float4*>(p + r * KT + j);
#pragma unroll
  for (int c = 0; c < NF; ++c) {
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
template <int NF, bool UP_TO>
__device__ __forceinline__ void accumulate_tile(float (*acc)[NF], const float* p, const float* tile, int lt, int lane,
                                                bool diagonal, int w) {
  if (!diagonal) {
    accumulate4<NF>(acc, p, tile, lt, lane, 0, KT);
    return;
  }
  if (UP_TO) accumulate4<NF>(acc, p, tile, lt, lane, 0, w * RPW);
  accumulate_diagonal<NF, UP_TO>(acc, p, tile, lt, lane, w * RPW);
  if (!UP_TO) accumulate4<NF>(acc, p, tile, lt, lane, (w + 1) * RPW, KT);
}

struct Where { int b, h, r0; };
__device__ __forceinline__ Where where(int block, int Tn, int H) {
  const int nt = (Tn + RT - 1) / RT;
  const int64_t item = (int64_t)block / nt;
  return {(int)(item / H), (int)(item % H), (nt - 1 - block % nt) * RT};      // long rows first
}

// Widths up to 64: the next tile is asked for while the current one is worked on (wider heads have no registers for it).
template <int NF> constexpr bool AHEAD = NF <= 2;

template <typename T, int NF>
__global__ void __launch_bounds__(WARPS * 32, 4) attn_fwd_kernel(const T* __restrict__ qkv, int Tn, int H, int d,
                                                              T* __restrict__ o, float* __restrict__ lse, bool vec) {
  overlap_sync();
  extern __shared__ __align__(16) float sh[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, dh = d / H;
  const Where at = where((int)blockIdx.x, Tn, H);
  Tiles t(sh, dh);
  const float scale = rsqrtf((float)dh);
  const size_t ld = (size_t)3 * d;
  const T* base = qkv + (size_t)at.b * Tn * ld + (size_t)at.h * dh;
  Block<T, NF> rq, rk, rv;
  rq.load(base, ld, at.r0, Tn, dh, vec);
  auto ask = [&](int j0) { rk.load(base + d, ld, j0, Tn, dh, vec); rv.load(base + 2 * (size_t)d, ld, j0, Tn, dh, vec); };
  if (AHEAD<NF>) ask(0);
  rq.template put<false>(t.ra, t.lr, dh);
  float m[RPW], l[RPW], acc[RPW][NF];
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < NF; ++c) acc[r][c] = 0.f;
  }
  const float* rows = t.ra + w * RPW * t.lr;
  float* p_s = t.pa + w * RPW * KT;
  const int row0 = at.r0 + w * RPW;
  const int end = min(at.r0 + RT, Tn);
  for (int j0 = 0; j0 < end; j0 += KT) {
    if (!AHEAD<NF>) ask(j0);
    __syncthreads();
    rk.template put<true>(t.a, t.lt, dh);
    rv.template put<true>(t.b, t.lt, dh);
    __syncthreads();
    if (AHEAD<NF> && j0 + KT < end) ask(j0 + KT);
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
      for (int c = 0; c < NF; ++c) acc[r][c] *= corr;
      m[r] = nm;
      p_s[r * KT + lane] = p;
    }
    __syncwarp();
    accumulate_tile<NF, true>(acc, p_s, t.b, t.lt, lane, j0 == at.r0, w);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    const int i = row0 + r;
    if (i >= Tn) continue;
    T* orow = o + ((size_t)at.b * Tn + i) * d + (size_t)at.h * dh;
#pragma unroll
    for (int c = 0; c < NF; ++c) {
      const int dim = lane + 32 * c;
      if (dim < dh) orow[dim] = from_f<T>(acc[r][c] / l[r]);
    }
    if (lane == 0) lse[((size_t)at.b * H + at.h) * Tn + i] = m[r] + logf(l[r]);
  }
}

struct Bwd { int Tn, H, d; bool vec; const float* lse; float* rowdot; };

// dQ, and D[row] = sum(dO * O) of its rows, which the dK/dV blocks read from `rowdot` where they run second
template <typename T, int NF>
__device__ __forceinline__ void dq_block(const T* __restrict__ qkv, const T* __restrict__ o, const T* __restrict__ d_o, T* __restrict__ dqkv,
                                         const Bwd& a, int block) {
  extern __shared__ __align__(16) float sh[];
  const int Tn = a.Tn, H = a.H, d = a.d, w = threadIdx.x >> 5, lane = threadIdx.x & 31, dh = d / H;
  const Where at = where(block, Tn, H);
  Tiles t(sh, dh);
  const float scale = rsqrtf((float)dh);
  const size_t ld = (size_t)3 * d;
  const T* base = qkv + (size_t)at.b * Tn * ld + (size_t)at.h * dh;
  const T* dobase = d_o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  const T* obase = o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  Block<T, NF> rk, rv;
  auto ask = [&](int j0) { rk.load(base + d, ld, j0, Tn, dh, a.vec); rv.load(base + 2 * (size_t)d, ld, j0, Tn, dh, a.vec); };
  {
    Block<T, NF> rq, rd;
    rq.load(base, ld, at.r0, Tn, dh, a.vec);
    rd.load(dobase, (size_t)d, at.r0, Tn, dh, a.vec);
    if (AHEAD<NF>) ask(0);
    rq.template put<false>(t.ra, t.lr, dh);
    rd.template put<false>(t.rb, t.lr, dh);
  }
  const int row0 = at.r0 + w * RPW;
  const size_t stat = ((size_t)at.b * H + at.h) * Tn;
  float L[RPW], D[RPW], acc[RPW][NF];
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    const int i = row0 + r;
    float s = 0.f;
    if (i < Tn)
      for (int c = lane; c < dh; c += 32) s = fmaf(to_f<T>(obase[(size_t)i * d + c]), to_f<T>(dobase[(size_t)i * d + c]), s);
    D[r] = warp_sum(s);
    L[r] = i < Tn ? a.lse[stat + i] : 0.f;
    if (lane == 0 && i < Tn) a.rowdot[stat + i] = D[r];
#pragma unroll
    for (int c = 0; c < NF; ++c) acc[r][c] = 0.f;
  }
  const float* qrows = t.ra + w * RPW * t.lr;
  const float* dorows = t.rb + w * RPW * t.lr;
  float* ds_s = t.pa + w * RPW * KT;
  const int end = min(at.r0 + RT, Tn);
  for (int j0 = 0; j0 < end; j0 += KT) {
    if (!AHEAD<NF>) ask(j0);
    __syncthreads();
    rk.template put<true>(t.a, t.lt, dh);
    rv.template put<true>(t.b, t.lt, dh);
    __syncthreads();
    if (AHEAD<NF> && j0 + KT < end) ask(j0 + KT);
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
    accumulate_tile<NF, true>(acc, ds_s, t.a, t.lt, lane, j0 == at.r0, w);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    if (row0 + r >= Tn) continue;
    T* out = dqkv + ((size_t)at.b * Tn + row0 + r) * ld + (size_t)at.h * dh;
#pragma unroll
    for (int c = 0; c < NF; ++c) {
      const int dim = lane + 32 * c;
      if (dim < dh) out[dim] = from_f<T>(acc[r][c]);
    }
  }
}

// sum of a[c] * b[c], added up as dq_block's warp adds its D: 32 strided sums of NF products, then halves upon halves (D of
// both gradients is the same number, and that of the form with a kernel for each; one chain is up to 1.6 % more error in dK)
template <int NF> __device__ __forceinline__ float row_product(const float* a, const float* b, int dh) {
  float half[16];
#pragma unroll
  for (int l = 0; l < 16; ++l) {
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int c = 0; c < NF; ++c) {
      const int c0 = l + 32 * c, c1 = c0 + 16;
      if (c0 < dh) s0 = fmaf(a[c0], b[c0], s0);
      if (c1 < dh) s1 = fmaf(a[c1], b[c1], s1);
    }
    half[l] = s0 + s1;
  }
#pragma unroll
  for (int n = 8; n > 0; n >>= 1)
#pragma unroll
    for (int l = 0; l < n; ++l) half[l] += half[l + n];
  return half[0];
}

// dK, dV: rows are keys, tiles are queries.  OWN_D: D = sum(dO * O) of a tile's queries is formed here, one query per lane,
// from the staged dO and one more tile, of O (behind the others in shared memory).
template <typename T, int NF, bool OWN_D>
__device__ __forceinline__ void dkv_block(const T* __restrict__ qkv, const T* __restrict__ o, const T* __restrict__ d_o, T* __restrict__ dqkv,
                                          const Bwd& a, int block) {
  extern __shared__ __align__(16) float sh[];
  const int Tn = a.Tn, H = a.H, d = a.d, w = threadIdx.x >> 5, lane = threadIdx.x & 31, dh = d / H;
  const Where at = where(block, Tn, H);
  Tiles t(sh, dh);
  float* o_s = t.b + KT * t.lt;
  const float scale = rsqrtf((float)dh);
  const size_t ld = (size_t)3 * d;
  const T* base = qkv + (size_t)at.b * Tn * ld + (size_t)at.h * dh;
  const T* dobase = d_o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  const T* obase = o + (size_t)at.b * Tn * d + (size_t)at.h * dh;
  const int row0 = at.r0 + w * RPW;
  const size_t stat = ((size_t)at.b * H + at.h) * Tn;
  Block<T, NF> rq, rd, ro;
  float L = 0.f, D = 0.f;
  auto ask = [&](int i0) {
    rq.load(base, ld, i0, Tn, dh, a.vec);
    rd.load(dobase, (size_t)d, i0, Tn, dh, a.vec);
    if (OWN_D) ro.load(obase, (size_t)d, i0, Tn, dh, a.vec);
    L = i0 + lane < Tn ? a.lse[stat + i0 + lane] : 0.f;
    if (!OWN_D) D = i0 + lane < Tn ? a.rowdot[stat + i0 + lane] : 0.f;
  };
  {
    Block<T, NF> rk, rv;
    rk.load(base + d, ld, at.r0, Tn, dh, a.vec);
    rv.load(base + 2 * (size_t)d, ld, at.r0, Tn, dh, a.vec);
    if (AHEAD<NF>) ask(at.r0);
    rk.template put<false>(t.ra, t.lr, dh);
    rv.template put<false>(t.rb, t.lr, dh);
  }
  float dk[RPW][NF], dv[RPW][NF];
#pragma unroll
  for (int r = 0; r < RPW; ++r)
#pragma unroll
    for (int c = 0; c < NF; ++c) { dk[r][c] = 0.f; dv[r][c] = 0.f; }
  const float* krows = t.ra + w * RPW * t.lr;
  const float* vrows = t.rb + w * RPW * t.lr;
  float* p_s = t.pa + w * RPW * KT;
  float* ds_s = t.pb + w * RPW * KT;
  for (int i0 = at.r0; i0 < Tn; i0 += KT) {
    if (!AHEAD<NF>) ask(i0);
    __syncthreads();
    rq.template put<true>(t.a, t.lt, dh);
    rd.template put<true>(t.b, t.lt, dh);
    if (OWN_D) ro.template put<true>(o_s, t.lt, dh);
    const float Li = L;
    float Di = D;
    __syncthreads();
    if (AHEAD<NF> && i0 + KT < Tn) ask(i0 + KT);
    if (OWN_D) Di = row_product<NF>(o_s + lane * t.lt, t.b + lane * t.lt, dh);
    const int i = i0 + lane;
    float s[RPW], dp[RPW];
    dot4(krows, t.lr, t.a + lane * t.lt, s);
    dot4(vrows, t.lr, t.b + lane * t.lt, dp);
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const bool vis = i >= row0 + r && i < Tn;
      const float p = vis ? expf(s[r] * scale - Li) : 0.f;
      p_s[r * KT + lane] = p;
      ds_s[r * KT + lane] = vis ? p * (dp[r] - Di) * scale : 0.f;
    }
    __syncwarp();
    accumulate_tile<NF, false>(dv, p_s, t.b, t.lt, lane, i0 == at.r0, w);
    accumulate_tile<NF, false>(dk, ds_s, t.a, t.lt, lane, i0 == at.r0, w);
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < RPW; ++r) {
    if (row0 + r >= Tn) continue;
    T* out = dqkv + ((size_t)at.b * Tn + row0 + r) * ld + (size_t)at.h * dh;
#pragma unroll
    for (int c = 0; c < NF; ++c) {
      const int dim = lane + 32 * c;
      if (dim < dh) { out[d + dim] = from_f<T>(dk[r][c]); out[2 * (size_t)d + dim] = from_f<T>(dv[r][c]); }
    }
  }
}

template <typename T, int NF>
__global__ void __launch_bounds__(WARPS * 32, 3) attn_bwd_dq_kernel(const T* __restrict__ qkv, const T* __restrict__ o, const T* __restrict__ d_o,
                                                                 T* __restrict__ dqkv, Bwd a) {
  overlap_sync();
  dq_block<T, NF>(qkv, o, d_o, dqkv, a, (int)blockIdx.x);
}
// BLOCKS: registers for that many blocks per SM (bwd chooses)
template <typename T, int NF, int BLOCKS>
__global__ void __launch_bounds__(WARPS * 32, BLOCKS) attn_bwd_dkv_kernel(const T* __restrict__ qkv, const T* __restrict__ o, const T* __restrict__ d_o,
                                                                  T* __restrict__ dqkv, Bwd a) {
  overlap_sync();
  dkv_block<T, NF, false>(qkv, o, d_o, dqkv, a, (int)blockIdx.x);
}
// Few blocks: both at once
template <typename T, int NF>
__global__ void __launch_bounds__(WARPS * 32, 2) attn_bwd_kernel(const T* __restrict__ qkv, const T* __restrict__ o, const T* __restrict__ d_o,
                                                              T* __restrict__ dqkv, Bwd a) {
  overlap_sync();
  const int half = (int)gridDim.x / 2;
  if ((int)blockIdx.x < half) dkv_block<T, NF, true>(qkv, o, d_o, dqkv, a, (int)blockIdx.x);
  else dq_block<T, NF>(qkv, o, d_o, dqkv, a, (int)blockIdx.x - half);
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

// room for the widest head of NF, once per device and kernel
template <typename K> cudaError_t allow_smem(K kernel, PerDeviceOnce& once) {
  const int dev = current_device();
  if (!once.needed(dev)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(MAX_DH, true));
  if (e == cudaSuccess) once.done(dev);
  return e;
}
// whether pieces of four columns are aligned vectors
template <typename T> bool vectors(int dh, const void* a, const void* b, const void* c) {
  return dh % 4 == 0 && ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & (4 * sizeof(T) - 1)) == 0;
}

template <typename T, int NF>
cudaError_t fwd_width(const void* qkv, unsigned blocks, int T_, int H, int d, void* o, float* lse, cudaStream_t st) {
  static PerDeviceOnce once;
  cudaError_t e = allow_smem(attn_fwd_kernel<T, NF>, once);
  if (e != cudaSuccess) return e;
  return launch_overlapped(attn_fwd_kernel<T, NF>, blocks, WARPS * 32, smem_bytes(d / H, false), st, (const T*)qkv, T_, H, d, (T*)o, lse,
                           vectors<T>(d / H, qkv, nullptr, nullptr));
}
template <typename T>
cudaError_t fwd(const void* qkv, unsigned blocks, int T_, int H, int d, void* o, float* lse, cudaStream_t st) {
  switch ((d / H + 31) / 32) {
    case 1: return fwd_width<T, 1>(qkv, blocks, T_, H, d, o, lse, st);
    case 2: return fwd_width<T, 2>(qkv, blocks, T_, H, d, o, lse, st);
    case 3: return fwd_width<T, 3>(qkv, blocks, T_, H, d, o, lse, st);
    default: return fwd_width<T, 4>(qkv, blocks, T_, H, d, o, lse, st);
  }
}

// BLOCKS = 2 where no more blocks than that per SM exist (4 x 64, 8 heads of 32: 20.2 us against 21.8 with registers for
// three), else 3 (42 x 24, 8 heads of 24: 20.9 us against 24.2).  The other kernels: four (forward) and three (dQ).
template <typename T, int NF, int BLOCKS>
cudaError_t bwd_blocks(const void* qkv, const void* o, const void* d_o, unsigned blocks, int dh, void* dqkv, const Bwd& a, cudaStream_t st) {
  static PerDeviceOnce once_q, once_kv;
  cudaError_t e = allow_smem(attn_bwd_dq_kernel<T, NF>, once_q);
  if (e == cudaSuccess) e = allow_smem(attn_bwd_dkv_kernel<T, NF, BLOCKS>, once_kv);
  if (e != cudaSuccess) return e;
  e = launch_overlapped(attn_bwd_dq_kernel<T, NF>, blocks, WARPS * 32, smem_bytes(dh, false), st, (const T*)qkv, (const T*)o, (const T*)d_o, (T*)dqkv, a);
  if (e != cudaSuccess) return e;
  return launch_overlapped(attn_bwd_dkv_kernel<T, NF, BLOCKS>, blocks, WARPS * 32, smem_bytes(dh, false), st, (const T*)qkv, (const T*)o, (const T*)d_o, (T*)dqkv, a);
}

template <typename T, int NF>
cudaError_t bwd_width(const void* qkv, const void* o, const void* d_o, unsigned blocks, int dh, void* dqkv, const Bwd& a, cudaStream_t st) {
  const int sms = num_sms();
  if ((int64_t)blocks <= sms) {
    static PerDeviceOnce once;
    cudaError_t e = allow_smem(attn_bwd_kernel<T, NF>, once);
    if (e != cudaSuccess) return e;
    return launch_overlapped(attn_bwd_kernel<T, NF>, 2 * blocks, WARPS * 32, smem_bytes(dh, true), st, (const T*)qkv, (const T*)o, (const T*)d_o, (T*)dqkv, a);
  }
  return (int64_t)blocks <= 2 * sms ? bwd_blocks<T, NF, 2>(qkv, o, d_o, blocks, dh, dqkv, a, st)
                                    : bwd_blocks<T, NF, 3>(qkv, o, d_o, blocks, dh, dqkv, a, st);
}

template <typename T>
cudaError_t bwd(const void* qkv, const void* o, const float* lse, const void* d_o, unsigned blocks, int T_, int H, int d,
                void* dqkv, float* rowdot, cudaStream_t st) {
  const Bwd a = {T_, H, d, vectors<T>(d / H, qkv, o, d_o), lse, rowdot};
  switch ((d / H + 31) / 32) {
    case 1: return bwd_width<T, 1>(qkv, o, d_o, blocks, d / H, dqkv, a, st);
    case 2: return bwd_width<T, 2>(qkv, o, d_o, blocks, d / H, dqkv, a, st);
    case 3: return bwd_width<T, 3>(qkv, o, d_o, blocks, d / H, dqkv, a, st);
    default: return bwd_width<T, 4>(qkv, o, d_o, blocks, d / H, dqkv, a, st);
  }
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
