// Causal multi-head attention on the 5th-generation tensor cores for sequences of any length, bf16, head width 64.  The
// forward kernel is described where it stands; backward, the same two kernels as in attention_t5_bwd.cu (dQ per query tile,
// then dK / dV per key tile, tiles of 128 rows, no atomics, bit-reproducible) with three differences:
//   * Sequences are planes of three-dimensional tensor maps: rows past the end of a sequence arrive as zeros and are
//     clipped on the way out.  A query row past the end carries a row statistic of -1e30, i.e. P = 0.
//   * P and dS enter their products as two bf16 values each (hi + lo, 16 mantissa bits), because lengths off the tile sizes have
//     always held them in more than bf16 (attention_tc.cu).  A 16-column chunk of fp32 scores in tensor memory is replaced by its
//     own 16 elements: 8 columns of hi pairs, 8 of lo pairs; a product over 16 elements is issued once with each.
//   * lse/scale and D enter the score products as three bf16 values (24 bits), exact to fp32.
// With P and dS on top of the scores a half-step (64 columns of S and of dP) takes 128 tensor-memory columns, so three
// half-steps are in flight next to dK and dV: the score products of one, the element-wise work of another, the
// accumulating products of the third.
// A row whose results are not all finite is done again in plain FMA over its visible pairs (attention_rows.cuh), because a
// product multiplies the zero probability of a hidden pair with whatever the tile holds.  (Template KEEP; not backward at
// multiples of 128, where the other form spoils its tiles of 128 rows too.  Odd multiples of 64 used to run in tiles of 64 rows
// and spoil those: keeping the values apart costs 128 sequences of 192, 12 heads 122 -> 129 us, 16 of 960
// 146 -> 147, 8 of 192 with 8 heads 15.0 -> 15.6; in tiles of 64 on mma.sync that one took 23.)
// What bounds them: neither unit by itself.  A half-step is 10 + 16 (dQ: 10 + 8) products [128 x 64 x 16] of 45-48 cycles
// (operand reads from shared memory) next to 512 cycles of exponentials; 16 sequences of 777 tokens, 12 heads, have 80 us of
// products and take 120 us (mma.sync, attention_tc.cu: 336), the tensor pipe active for 36 % (dQ) and 43 % of the cycles.  P and dS
// as single bf16 values (template HILO = false, for lengths that always had that precision) save 15 % (16 x 960, 12 heads 174 -> 148 us);
// with the element-wise warps in two groups on alternate half-steps the time is the same: the chain of barriers, tensor-memory
// loads and stores from a score to its release is what three half-steps in flight do not cover.  Errors against 64 bits agree with
// the mma.sync form's to four digits.
// Few tiles: both kernels run as one launch on their own CTAs (attn64_bwd_t5_kernel), the dK/dV tiles forming D themselves:
// 2 sequences of 256, 16 heads 15.0 -> 9.5 us against the two kernels of attention_t5_bwd.cu.
#include "attention_rows.cuh"
#include "attention_t5.cuh"
#include "host_common.h"
#include "launch.cuh"

namespace sl {
namespace {

using namespace t5;

constexpr int NBUF = 3;                       // half-steps in flight
constexpr int RING = 3;                       // stages of streamed operand tiles
constexpr int EWQ = 4, CW = 16;               // element-wise warps per accumulator lane quarter; columns of each
constexpr int EW_WARPS = 4 * EWQ;
constexpr int ACC_WARP = 2 + EW_WARPS;
constexpr int OUT_WARP0 = ACC_WARP + 1;       // four, one per accumulator lane quarter (warp & 3)
constexpr int STAT_WARP = OUT_WARP0 + 4;      // dK/dV kernel only
constexpr int THREADS_DQ = (OUT_WARP0 + 4) * 32, THREADS_DKV = (STAT_WARP + 1) * 32;
constexpr uint32_t TILE16 = TILE >> 4, AUG16 = AUG_TILE >> 4;
constexpr int REDO_BYTES = 4 * 2 * DH * 4;    // scratch of the rows done again: 2 dh floats per output warp
constexpr float PAST_END = 1e30f;

struct Params {
  int T, H, d, nitems, nq, block, last_halves;   // nq: tiles of 128; block: see Units; last_halves: 64-row halves of the last tile that hold rows
  float scale, scale_log2;
  const float* lse;
  float* rowdot;
  float* lse_out;                             // forward: lse and o
  bf16* o;
  const bf16 *qkv, *d_o;
  bf16* dqkv;
  int* status;
};

// Work units are (tile, item) pairs, item = (sequence, head), in blocks of `block` items whose operands stay in L2 between
// their tiles; inside a block the longest tiles first.  CTA `cta` of `grid` takes one of each round of `grid` units, forwards
// in even rounds and backwards in odd ones, so that all get about the same number of steps.
struct Unit { int tile, item; };              // tile 0: the longest
struct Units {
  int n, nq, nitems, block, grid, cta;
  __device__ __forceinline__ Units(const Params& p, int cta_, int grid_)
      : n(p.nitems * p.nq), nq(p.nq), nitems(p.nitems), block(p.block), grid(grid_), cta(cta_) {}
  __device__ __forceinline__ int index(int k) const { return k * grid + ((k & 1) ? grid - 1 - cta : cta); }
  __device__ __forceinline__ bool has(int k) const { return k * grid < n && index(k) < n; }
  __device__ __forceinline__ Unit at(int k) const {
    const int u = index(k), b0 = u / (block * nq) * block, in = min(block, nitems - b0), rest = u - b0 * nq;
    return {rest / in, b0 + rest % in};
  }
};

// -x as the sum of three bf16 values, the columns [c, c + 3) of an operand row
__device__ __forceinline__ void neg_split3(float x, uint32_t& a, uint32_t& b, uint32_t& c) {
  const __nv_bfloat16 hi = __float2bfloat16_rn(-x);
  const float r1 = -x - __bfloat162float(hi);
  const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
  const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
  a = __bfloat16_as_ushort(hi); b = __bfloat16_as_ushort(mid); c = __bfloat16_as_ushort(lo);
}
// columns 0..2 = -L (for the scores), 3..5 = -D (for dP)
__device__ __forceinline__ uint4 stat_row(float L, float D) {
  uint32_t l0, l1, l2, d0, d1, d2;
  neg_split3(L, l0, l1, l2);
  neg_split3(D, d0, d1, d2);
  return make_uint4(l0 | (l1 << 16), l2 | (d0 << 16), d1 | (d2 << 16), 0u);
}
// zeroes the operand tiles that will carry statistics and writes the two constant tiles: ones in columns 0..2 / 3..5
__device__ __forceinline__ void init_ones(uint8_t* ones_s, uint8_t* ones_d, int rows, uint8_t* zero, int zero_bytes) {
  for (int i = threadIdx.x; i < zero_bytes / 16; i += blockDim.x) reinterpret_cast<uint4*>(zero)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = threadIdx.x; i < rows * 2; i += blockDim.x) {       // 16-byte pieces: row i / 2, columns 0..7 or 8..15
    const uint32_t off = aug_row(i >> 1) + (uint32_t)(i & 1) * 128u;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(ones_s + off) = (i & 1) ? z : make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
    *reinterpret_cast<uint4*>(ones_d + off) = (i & 1) ? z : make_uint4(0u, 0x3F800000u, 0x3F803F80u, 0u);
  }
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// 8 (HILO) or 4 products [128 x 64] += A[128 x 64] * B rows [64 hh, 64 hh + 64), B an MN-major tile used as loaded; A in tensor
// memory at a_tmem, per 16 elements 8 columns of bf16 pairs and, HILO, 8 of what rounding to bf16 left
template <bool HILO>
__device__ __forceinline__ void mma_acc(uint32_t d_tmem, uint32_t a_tmem, uint32_t blo, int hh, bool fresh) {
  const uint32_t b0 = blo + (uint32_t)(512 * hh);
  tc_mma_ts_lo(d_tmem, a_tmem, b0, IDESC_64MN, fresh ? 0u : 1u);
  if constexpr (HILO) tc_mma_ts_lo(d_tmem, a_tmem + 8, b0, IDESC_64MN, 1u);
#pragma unroll
  for (uint32_t k = 1; k < 4; ++k) {
    tc_mma_ts_lo(d_tmem, a_tmem + 16 * k, b0 + 128 * k, IDESC_64MN, 1u);
    if constexpr (HILO) tc_mma_ts_lo(d_tmem, a_tmem + 16 * k + 8, b0 + 128 * k, IDESC_64MN, 1u);
  }
}

// two values as a bf16 pair in w[i] and, HILO, what that rounding leaves in w[8 + i]
template <bool HILO>
__device__ __forceinline__ void put_pair(uint64_t v, uint32_t* w, int i) {
  float a, b;
  unpack2(v, a, b);
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  w[i] = *reinterpret_cast<const uint32_t*>(&h);
  if constexpr (!HILO) return;
  const uint32_t hi = w[i];
  float ra, rb;
  unpack2(add2(v, pack2(__uint_as_float((hi << 16) ^ 0x80000000u), __uint_as_float((hi & 0xffff0000u) ^ 0x80000000u))), ra, rb);
  const __nv_bfloat162 l = __floats2bfloat162_rn(ra, rb);
  w[8 + i] = *reinterpret_cast<const uint32_t*>(&l);
}
template <bool HILO> __device__ __forceinline__ void st_pairs(uint32_t t, const uint32_t* w) {
  if constexpr (HILO) tc_st16(t, w); else tc_st8(t, w);
}

// sum over the 64 columns of row r of a staged tile times the same row in registers (eight 16-byte pieces in order)
__device__ __forceinline__ float row_product(const uint8_t* tile, int r, const uint4* v) {
  float sum = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint4 a = *reinterpret_cast<const uint4*>(tile + r * 128 + ((j ^ (r & 7)) << 4));     // lanes of a warp spread over all banks
    const uint32_t *aw = reinterpret_cast<const uint32_t*>(&a), *vw = reinterpret_cast<const uint32_t*>(&v[j]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      sum = fmaf(__uint_as_float(aw[e] << 16), __uint_as_float(vw[e] << 16), sum);
      sum = fmaf(__uint_as_float(aw[e] & 0xffff0000u), __uint_as_float(vw[e] & 0xffff0000u), sum);
    }
  }
  return sum;
}

// [32 rows x 64] of an accumulator -> bf16 rows of a staged tile; whether one of the values is an inf or NaN
__device__ __forceinline__ bool stage_rows(uint32_t tsrc, uint32_t tile, int r, float mul) {
  uint32_t bad = 0;
#pragma unroll
  for (int c = 0; c < 64; c += 32) {
    float v[32];
    tc_ld32(tsrc + (uint32_t)c, v);
    tc_wait_ld();
#pragma unroll
    for (uint32_t jj = 0; jj < 4; ++jj) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 ob = __floats2bfloat162_rn(v[8 * jj + 2 * e] * mul, v[8 * jj + 2 * e + 1] * mul);
        w[e] = *reinterpret_cast<const uint32_t*>(&ob);
        bad |= ((w[e] & 0x7f807f80u) + 0x00800080u) & 0x80008000u;
      }
      st_row_chunk(tile, r, (uint32_t)(c >> 3) + jj, w);
    }
  }
  return bad != 0;
}
// barrier of the four output warps that tells all of them whether any thread's flag is set
__device__ __forceinline__ bool out_warps_any(bool flag) {
  uint32_t any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(any) : "r"((uint32_t)flag) : "memory");
  return any != 0;
}
__device__ __forceinline__ void out_warps_sync() { asm volatile("barrier.cta.sync 1, 128;" ::: "memory"); }

#define RG_SETUP(NBARS, COUNT, TCOLS)                                                                            \
  extern __shared__ uint8_t smem_raw[];                                                                   \
  const uint32_t raw = smem_u32(smem_raw);                                                                \
  const uint32_t base = (raw + 1023u) & ~1023u;                                                           \
  uint8_t* base_ptr = smem_raw + (base - raw);                                                            \
  const uint32_t bar = base + OFF_BAR;                                                                    \
  auto B = [&](int i) { return bar + 8u * i; };                                                           \
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + OFF_BAR + 8 * NBARS);    \
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + OFF_BAR + 8 * NBARS + 8);         \
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;                                             \
  if (threadIdx.x == 0) {                                                                                 \
    for (int i = 0; i < NBARS; ++i) mbar_init(B(i), COUNT(i));                                            \
    *abort_flag = 0;                                                                                      \
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");                                    \
  }                                                                                                       \
  if (warp == 1) {                                                                                        \
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"                      \
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)TCOLS) : "memory");           \
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");              \
  }

#define RG_SETUP_END()                                                                                    \
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");                                            \
  tc_fence_before();                                                                                      \
  __syncthreads();                                                                                        \
  tc_fence_after();                                                                                       \
  const uint32_t tmem_base = *tmem_slot;                                                                  \
  overlap_sync();

#define RG_TEARDOWN(TCOLS)                                                                                     \
  __syncwarp();                                                                                           \
  if (*abort_flag) { for (int i = 0; i < 2000; ++i) __nanosleep(1000); }                                  \
  tc_fence_before();                                                                                      \
  __syncthreads();                                                                                        \
  if (warp == 1) {                                                                                        \
    tc_fence_after();                                                                                     \
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TCOLS) : "memory"); \
  }

// ==========================================================================================
// dK, dV of a key tile: query tiles i >= kt
// ==========================================================================================
namespace dkv {
enum { KV_FULL = 0 /*+buffer*/, KV_EMPTY = 2, QD_FULL = 4 /*+stage*/, QD_EMPTY = QD_FULL + RING, AUG_READY = QD_EMPTY + RING,
       S_FULL = AUG_READY + RING /*+half-step*/, P_READY = S_FULL + NBUF, P_FREE = P_READY + NBUF, ACC_FULL = P_FREE + NBUF, ACC_FREE,
       N_BARS };
template <bool OWN_D> __device__ __forceinline__ uint32_t count(int i) {
  return i >= QD_EMPTY && i < QD_EMPTY + RING ? 2u : i >= P_READY && i < P_READY + NBUF ? (uint32_t)EW_WARPS
         : i == ACC_FREE || (OWN_D && i >= AUG_READY && i < AUG_READY + RING) ? 4u : 1u;
}
constexpr int OFF_KV = 0;                                  // buffer kb: K, then V
constexpr int OFF_QD = 2 * 2 * TILE;                       // stage s: Q, then dO
constexpr int OFF_OUT = OFF_QD + RING * 2 * TILE;
constexpr int OFF_AUG = OFF_OUT + 2 * TILE;                // ones for S^T, ones for dP^T, one tile per stage
constexpr int OFF_REDO = OFF_AUG + (2 + RING) * AUG_TILE;
constexpr int OFF_BAR = OFF_REDO + REDO_BYTES;
constexpr int SMEM = OFF_BAR + 8 * N_BARS + 16 + 1024;
static_assert(SMEM <= 232448, "");
}  // namespace dkv

// OWN_D: D is not in `rowdot` yet; the output warps, idle until the accumulators are complete, compute it for every step from
// the staged dO rows and the rows of O in global memory, and write the operand rows in the statistics warp's place.
template <bool HILO, bool KEEP, bool OWN_D>
__device__ __forceinline__ void dkv_tiles(const CUtensorMap& mapQKV, const CUtensorMap& mapDO, const CUtensorMap& mapDQKV, const Params& p, int cta, int grid) {
  using namespace dkv;
  RG_SETUP(N_BARS, count<OWN_D>, TMEM_COLS)
  init_ones(base_ptr + OFF_AUG, base_ptr + OFF_AUG + AUG_TILE, BT, base_ptr + OFF_AUG + 2 * AUG_TILE, RING * AUG_TILE);
  RG_SETUP_END()
  const Units units(p, cta, grid);
  const uint32_t tDV = tmem_base + 128u * NBUF, tDK = tDV + 64u;
  auto halves = [&](int i) { return i == p.nq - 1 ? p.last_halves : 2; };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0;                            // ring stage and how often it has been used
    for (int k = 0; units.has(k) && ok; ++k) {
      const Unit u = units.at(k);
      const int kt = u.tile, h = u.item % p.H, b = u.item / p.H, kb = k & 1;
      if (!mbar_wait_warp(B(KV_EMPTY + kb), freed(k >> 1), abort_flag, p.status, 111)) break;
      if (leader) {
        mbar_expect_tx(B(KV_FULL + kb), 2 * TILE);
        const uint32_t kv = base + OFF_KV + kb * 2 * TILE;
        tma_load_3d(kv, &mapQKV, B(KV_FULL + kb), p.d + h * DH, kt * BT, b);
        tma_load_3d(kv + TILE, &mapQKV, B(KV_FULL + kb), 2 * p.d + h * DH, kt * BT, b);
      }
      __syncwarp();
      for (int i = kt; i < p.nq; ++i) {
        if (!mbar_wait_warp(B(QD_EMPTY + s), freed(n), abort_flag, p.status, 112)) { ok = false; break; }
        if (leader) {
          mbar_expect_tx(B(QD_FULL + s), 2 * TILE);
          const uint32_t qd = base + OFF_QD + s * 2 * TILE;
          tma_load_3d(qd, &mapQKV, B(QD_FULL + s), h * DH, i * BT, b);
          tma_load_3d(qd + TILE, &mapDO, B(QD_FULL + s), h * DH, i * BT, b);
        }
        __syncwarp();
        if (++s == RING) { s = 0; ++n; }
      }
    }
  } else if (warp == 1) {
    // ---------------- score products: S^T = K Q^T - lse/scale, dP^T = V dO^T - D ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0, bf = 0, bn = 0;            // ring stage; half-step buffer; how often each has been used
    const uint32_t lo_aug = desc_lo_aug(base + OFF_AUG);
    for (int k = 0; units.has(k) && ok; ++k) {
      const int kt = units.at(k).tile, kb = k & 1;
      const uint32_t lo_k = desc_lo(base + OFF_KV) + (uint32_t)(kb * 2) * TILE16, lo_v = lo_k + TILE16;
      if (!mbar_wait_warp(B(KV_FULL + kb), done(k >> 1), abort_flag, p.status, 113)) break;
      for (int i = kt; i < p.nq && ok; ++i) {
        const uint32_t lo_q = desc_lo(base + OFF_QD) + (uint32_t)(s * 2) * TILE16, lo_do = lo_q + TILE16;
        const uint32_t lo_st = lo_aug + (uint32_t)(2 + s) * AUG16;
        if (!mbar_wait_warp(B(QD_FULL + s), done(n), abort_flag, p.status, 114)) { ok = false; break; }
        if (!mbar_wait_warp(B(AUG_READY + s), done(n), abort_flag, p.status, 115)) { ok = false; break; }
        for (int hh = 0; hh < halves(i); ++hh) {
          if (!mbar_wait_warp(B(P_FREE + bf), freed(bn), abort_flag, p.status, 116)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tS = tmem_base + 128u * (uint32_t)bf;
          if (leader) {
            mma_score_half(tS, lo_k, lo_q, hh);
            tc_mma_aug(tS, lo_aug, lo_st + (uint32_t)(128 * hh), IDESC_64KK);
            mma_score_half(tS + 64u, lo_v, lo_do, hh);
            tc_mma_aug(tS + 64u, lo_aug + AUG16, lo_st + (uint32_t)(128 * hh), IDESC_64KK);
            tc_commit(B(S_FULL + bf));
          }
          __syncwarp();
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
        if (ok && leader) tc_commit(B(QD_EMPTY + s));        // the second arrival comes from the accumulating warp
        __syncwarp();
        if (++s == RING) { s = 0; ++n; }
      }
      if (ok && leader) tc_commit(B(KV_EMPTY + kb));
      __syncwarp();
    }
  } else if (warp == ACC_WARP) {
    // ---------------- accumulating products: dV += P^T dO, dK += dS^T Q ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0, bf = 0, bn = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int kt = units.at(k).tile;
      if (!mbar_wait_warp(B(ACC_FREE), freed(k), abort_flag, p.status, 117)) break;
      for (int i = kt; i < p.nq && ok; ++i) {
        const uint32_t lo_q = desc_lo(base + OFF_QD) + (uint32_t)(s * 2) * TILE16, lo_do = lo_q + TILE16;
        if (!mbar_wait_warp(B(QD_FULL + s), done(n), abort_flag, p.status, 118)) { ok = false; break; }
        for (int hh = 0; hh < halves(i); ++hh) {
          if (!mbar_wait_warp(B(P_READY + bf), done(bn), abort_flag, p.status, 119)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tP = tmem_base + 128u * (uint32_t)bf;
          if (leader) {
            mma_acc<HILO>(tDV, tP, lo_do, hh, i == kt && hh == 0);
            mma_acc<HILO>(tDK, tP + 64u, lo_q, hh, i == kt && hh == 0);
            tc_commit(B(P_FREE + bf));
          }
          __syncwarp();
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
        if (ok && leader) tc_commit(B(QD_EMPTY + s));
        __syncwarp();
        if (++s == RING) { s = 0; ++n; }
      }
      if (ok && leader) tc_commit(B(ACC_FULL));
      __syncwarp();
    }
  } else if (warp < ACC_WARP) {
    // ---------------- element-wise warps: P^T = exp(scale S^T), dS^T = P^T dP^T ----------------
    const int q4 = warp & 3, c = ((warp - 2) >> 2) * CW;
    const int r = q4 * 32 + lane;                // key row inside the tile = accumulator lane
    const uint32_t at = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c;
    const uint64_t sc2 = pack2(p.scale * LOG2E, p.scale * LOG2E);
    bool ok = true;
    int bf = 0, bn = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int kt = units.at(k).tile;
      for (int i = kt; i < p.nq && ok; ++i) {
        for (int hh = 0; hh < halves(i); ++hh) {
          const uint32_t t = at + 128u * (uint32_t)bf;
          const int q0 = hh * 64 + c;            // first query of this thread's 16, inside the tile
          if (!mbar_wait_warp(B(S_FULL + bf), done(bn), abort_flag, p.status, 120)) { ok = false; break; }
          tc_fence_after();
          uint32_t pw[CW], dw[CW];               // 8 words of bf16 pairs, 8 of what rounding left
          // on the diagonal tile only queries >= this key count: chunks wholly before the warp's rows are zero
          if (i != kt || q0 + CW > q4 * 32) {
            float sv[CW], dv[CW];
            tc_ld16(t, sv);
            tc_ld16(t + 64u, dv);
            tc_wait_ld();
            if (i == kt && q0 < q4 * 32 + 32) {  // the mask on the scores: the element loop stays free of tests
#pragma unroll
              for (int e = 0; e < CW; ++e) sv[e] = (q0 + e < r) ? -INFINITY : sv[e];
            }
#pragma unroll
            for (int e = 0; e < CW; e += 2) {
              float a0, a1;
              unpack2(mul2(pack2(sv[e], sv[e + 1]), sc2), a0, a1);
              const uint64_t pv = pack2(ex2(a0), ex2(a1));
              put_pair<HILO>(pv, pw, e >> 1);
              put_pair<HILO>(mul2(pv, pack2(dv[e], dv[e + 1])), dw, e >> 1);
            }
          } else {
#pragma unroll
            for (int e = 0; e < CW; ++e) { pw[e] = 0u; dw[e] = 0u; }
          }
          st_pairs<HILO>(t, pw);
          st_pairs<HILO>(t + 64u, dw);
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(B(P_READY + bf));
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
      }
    }
  } else if (warp == STAT_WARP) {
    if (!OWN_D) {
      // ---------------- -lse/scale and -D of a stage's queries as operand rows ----------------
      const float inv_scale = 1.0f / p.scale;
      bool ok = true;
      int s = 0, n = 0;
      for (int k = 0; units.has(k) && ok; ++k) {
        const Unit u = units.at(k);
        const int kt = u.tile;
        const size_t stat0 = (size_t)u.item * p.T;
        for (int i = kt; i < p.nq; ++i) {
          float L[4], D[4];
  #pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int row = i * BT + lane + 32 * j;
            const bool in = row < p.T;
            L[j] = in ? p.lse[stat0 + row] * inv_scale : PAST_END;
            D[j] = in ? p.rowdot[stat0 + row] : 0.f;
          }
          if (!mbar_wait_warp(B(QD_EMPTY + s), freed(n), abort_flag, p.status, 121)) { ok = false; break; }
          uint8_t* rows = base_ptr + OFF_AUG + (2 + s) * AUG_TILE;
  #pragma unroll
          for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(rows + aug_row(lane + 32 * j)) = stat_row(L[j], D[j]);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(B(AUG_READY + s));
          if (++s == RING) { s = 0; ++n; }
        }
      }
    }
  } else {
    // ---------------- output: dK (scaled) and dV of a finished key tile ----------------
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    bool ok = true;
    int s = 0, n = 0;
    (void)s; (void)n;
    for (int k = 0; units.has(k); ++k) {
      const Unit u = units.at(k);
      const int kt = u.tile, item = u.item, h = item % p.H, b = item / p.H;
      const int row0 = kt * BT + q4 * 32;
      bool bad = false;
      if constexpr (OWN_D) {
        for (int i = kt; i < p.nq && ok; ++i) {
          const int row = i * BT + r;
          const bool in = row < p.T;
          const bf16* orow = p.o + ((size_t)b * p.T + (in ? row : 0)) * p.d + (size_t)h * DH;
          uint4 ov[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) ov[j] = *reinterpret_cast<const uint4*>(orow + 8 * j);
          const float L = in ? p.lse[(size_t)item * p.T + row] * (1.0f / p.scale) : PAST_END;
          if (!mbar_wait_warp(B(QD_FULL + s), done(n), abort_flag, p.status, 123)) { ok = false; break; }
          const float D = in ? row_product(base_ptr + OFF_QD + s * 2 * TILE + TILE, r, ov) : 0.f;
          *reinterpret_cast<uint4*>(base_ptr + OFF_AUG + (2 + s) * AUG_TILE + aug_row(r)) = stat_row(L, D);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(B(AUG_READY + s));
          if (++s == RING) { s = 0; ++n; }
        }
      }
      if (ok && !mbar_wait(B(ACC_FULL), done(k), abort_flag, p.status, 122)) ok = false;
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        tc_fence_after();
        bad = stage_rows(tDK + lane_off, base + OFF_OUT, r, p.scale);
        bad |= stage_rows(tDV + lane_off, base + OFF_OUT + TILE, r, 1.0f);
        bad = bad && row0 + lane < p.T;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(B(ACC_FREE));
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      out_warps_sync();                                          // (always reached by all four)
      const bool storer = ok && warp == OUT_WARP0 && lane == 0;
      if (storer) {
        tma_store_3d(&mapDQKV, base + OFF_OUT, p.d + h * DH, kt * BT, b);
        tma_store_3d(&mapDQKV, base + OFF_OUT + TILE, 2 * p.d + h * DH, kt * BT, b);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      }
      bool redo = false;
      if constexpr (KEEP) redo = out_warps_any(bad); else out_warps_sync();
      if (redo) {
        if (storer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        out_warps_sync();
        if (__any_sync(0xffffffffu, bad)) {
          if constexpr (OWN_D) {                 // D of the rows that are needed: this warp's own copy, the same values as the dQ tiles'
            for (int row = row0 + lane; row < p.T; row += 32) {
              const size_t at = ((size_t)b * p.T + row) * p.d + (size_t)h * DH;
              float D = 0.f;
              for (int c = 0; c < DH; ++c) D = fmaf(__bfloat162float(p.d_o[at + c]), __bfloat162float(p.o[at + c]), D);
              p.rowdot[(size_t)item * p.T + row] = D;
            }
            __syncwarp();
          }
          const rows::Head<bf16> hd(p.qkv, b, h, p.T, p.H, p.d);
          const size_t stat = (size_t)item * p.T;
          float* scratch = reinterpret_cast<float*>(base_ptr + OFF_REDO) + (warp - OUT_WARP0) * 2 * DH;
          for (int row = row0; row < min(row0 + 32, p.T); ++row)
            rows::dkv_row<bf16>(hd, p.d_o + (size_t)b * p.T * p.d + (size_t)h * DH, p.lse + stat, p.rowdot + stat, row, scratch,
                                p.dqkv + ((size_t)b * p.T + row) * hd.ld + p.d + (size_t)h * DH);
        }
      }
    }
    if (warp == OUT_WARP0 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  RG_TEARDOWN(TMEM_COLS)
}

// ==========================================================================================
// dQ of a query tile: key tiles j <= i; also D[row] = sum(dO * O), which the dK/dV kernel reads
// ==========================================================================================
namespace dq {
enum { QO_FULL = 0 /*+buffer*/, QO_EMPTY = 2, AUG_READY = 4, KV_FULL = 6 /*+stage*/, KV_EMPTY = KV_FULL + RING,
       S_FULL = KV_EMPTY + RING /*+half-step*/, P_READY = S_FULL + NBUF, P_FREE = P_READY + NBUF, ACC_FULL = P_FREE + NBUF, ACC_FREE,
       N_BARS };
__device__ __forceinline__ uint32_t count(int i) {
  return i >= KV_EMPTY && i < KV_EMPTY + RING ? 2u : i >= P_READY && i < P_READY + NBUF ? (uint32_t)EW_WARPS
         : i == ACC_FREE || i == AUG_READY || i == AUG_READY + 1 ? 4u : 1u;
}
constexpr int OFF_QO = 0;                                  // buffer qb: Q, dO, O
constexpr int OFF_KV = 2 * 3 * TILE;                       // stage s: K, then V
constexpr int OFF_OUT = OFF_KV + RING * 2 * TILE;
constexpr int OFF_AUG = OFF_OUT + TILE;                    // ones for S and for dP (64 key rows each), one tile per Q buffer
constexpr int OFF_REDO = OFF_AUG + 3 * AUG_TILE;
constexpr int OFF_BAR = OFF_REDO + REDO_BYTES;
constexpr int SMEM = OFF_BAR + 8 * N_BARS + 16 + 1024;
static_assert(SMEM <= 232448, "");
}  // namespace dq

template <bool HILO, bool KEEP>
__device__ __forceinline__ void dq_tiles(const CUtensorMap& mapQKV, const CUtensorMap& mapDO, const CUtensorMap& mapO, const CUtensorMap& mapDQKV,
                                         const Params& p, int cta, int grid) {
  using namespace dq;
  RG_SETUP(N_BARS, count, TMEM_COLS)
  init_ones(base_ptr + OFF_AUG, base_ptr + OFF_AUG + AUG_TILE / 2, 64, base_ptr + OFF_AUG + AUG_TILE, 2 * AUG_TILE);
  RG_SETUP_END()
  const Units units(p, cta, grid);
  const uint32_t tDQ = tmem_base + 128u * NBUF;
  auto halves = [&](int j) { return j == p.nq - 1 ? p.last_halves : 2; };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const Unit u = units.at(k);
      const int i = p.nq - 1 - u.tile, h = u.item % p.H, b = u.item / p.H, qb = k & 1;
      if (!mbar_wait_warp(B(QO_EMPTY + qb), freed(k >> 1), abort_flag, p.status, 131)) break;
      if (leader) {
        mbar_expect_tx(B(QO_FULL + qb), 3 * TILE);
        const uint32_t qo = base + OFF_QO + qb * 3 * TILE;
        tma_load_3d(qo, &mapQKV, B(QO_FULL + qb), h * DH, i * BT, b);
        tma_load_3d(qo + TILE, &mapDO, B(QO_FULL + qb), h * DH, i * BT, b);
        tma_load_3d(qo + 2 * TILE, &mapO, B(QO_FULL + qb), h * DH, i * BT, b);
      }
      __syncwarp();
      for (int j = 0; j <= i; ++j) {
        if (!mbar_wait_warp(B(KV_EMPTY + s), freed(n), abort_flag, p.status, 132)) { ok = false; break; }
        if (leader) {
          mbar_expect_tx(B(KV_FULL + s), 2 * TILE);
          const uint32_t kv = base + OFF_KV + s * 2 * TILE;
          tma_load_3d(kv, &mapQKV, B(KV_FULL + s), p.d + h * DH, j * BT, b);
          tma_load_3d(kv + TILE, &mapQKV, B(KV_FULL + s), 2 * p.d + h * DH, j * BT, b);
        }
        __syncwarp();
        if (++s == RING) { s = 0; ++n; }
      }
    }
  } else if (warp == 1) {
    // ---------------- score products: S = Q K^T - lse/scale, dP = dO V^T - D ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0, bf = 0, bn = 0;
    const uint32_t lo_aug = desc_lo_aug(base + OFF_AUG);
    for (int k = 0; units.has(k) && ok; ++k) {
      const int i = p.nq - 1 - units.at(k).tile, qb = k & 1;
      const uint32_t lo_q = desc_lo(base + OFF_QO) + (uint32_t)(qb * 3) * TILE16, lo_do = lo_q + TILE16;
      const uint32_t lo_st = lo_aug + (uint32_t)(1 + qb) * AUG16;
      if (!mbar_wait_warp(B(QO_FULL + qb), done(k >> 1), abort_flag, p.status, 133)) break;
      for (int j = 0; j <= i && ok; ++j) {
        const uint32_t lo_k = desc_lo(base + OFF_KV) + (uint32_t)(s * 2) * TILE16, lo_v = lo_k + TILE16;
        if (!mbar_wait_warp(B(KV_FULL + s), done(n), abort_flag, p.status, 134)) { ok = false; break; }
        // In a tile's first step the products over the features of all its halves are issued before the rows with -lse/scale
        // and -D are waited for, which the output warps write once Q, dO and O have arrived.
        const int nh = halves(j), b0 = bf;
        auto statistics = [&](int b) {
          const uint32_t tS = tmem_base + 128u * (uint32_t)b;
          if (leader) {
            tc_mma_aug(tS, lo_st, lo_aug, IDESC_64KK);
            tc_mma_aug(tS + 64u, lo_st, lo_aug + AUG16 / 2, IDESC_64KK);
            tc_commit(B(S_FULL + b));
          }
          __syncwarp();
        };
        for (int hh = 0; hh < nh; ++hh) {
          if (!mbar_wait_warp(B(P_FREE + bf), freed(bn), abort_flag, p.status, 135)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tS = tmem_base + 128u * (uint32_t)bf;
          if (leader) {
            mma_score_half(tS, lo_q, lo_k, hh);
            mma_score_half(tS + 64u, lo_do, lo_v, hh);
          }
          __syncwarp();
          if (j > 0) statistics(bf);
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
        if (ok && j == 0) {
          if (!mbar_wait_warp(B(AUG_READY + qb), done(k >> 1), abort_flag, p.status, 136)) { ok = false; break; }
          statistics(b0);
          if (nh > 1) statistics(b0 + 1 == NBUF ? 0 : b0 + 1);
        }
        if (ok && leader) tc_commit(B(KV_EMPTY + s));        // the second arrival comes from the accumulating warp
        __syncwarp();
        if (++s == RING) { s = 0; ++n; }
      }
      if (ok && leader) tc_commit(B(QO_EMPTY + qb));
      __syncwarp();
    }
  } else if (warp == ACC_WARP) {
    // ---------------- accumulating products: dQ += dS K ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0, bf = 0, bn = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int i = p.nq - 1 - units.at(k).tile;
      if (!mbar_wait_warp(B(ACC_FREE), freed(k), abort_flag, p.status, 137)) break;
      for (int j = 0; j <= i && ok; ++j) {
        const uint32_t lo_k = desc_lo(base + OFF_KV) + (uint32_t)(s * 2) * TILE16;
        if (!mbar_wait_warp(B(KV_FULL + s), done(n), abort_flag, p.status, 138)) { ok = false; break; }
        for (int hh = 0; hh < halves(j); ++hh) {
          if (!mbar_wait_warp(B(P_READY + bf), done(bn), abort_flag, p.status, 139)) { ok = false; break; }
          tc_fence_after();
          if (leader) {
            mma_acc<HILO>(tDQ, tmem_base + 128u * (uint32_t)bf, lo_k, hh, j == 0 && hh == 0);
            tc_commit(B(P_FREE + bf));
          }
          __syncwarp();
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
        if (ok && leader) tc_commit(B(KV_EMPTY + s));
        __syncwarp();
        if (++s == RING) { s = 0; ++n; }
      }
      if (ok && leader) tc_commit(B(ACC_FULL));
      __syncwarp();
    }
  } else if (warp < ACC_WARP) {
    // ---------------- element-wise warps: dS = exp(scale S) dP ----------------
    const int q4 = warp & 3, c = ((warp - 2) >> 2) * CW;
    const int r = q4 * 32 + lane;                // query row inside the tile
    const uint32_t at = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c;
    const uint64_t sc2 = pack2(p.scale * LOG2E, p.scale * LOG2E);
    bool ok = true;
    int bf = 0, bn = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int i = p.nq - 1 - units.at(k).tile;
      for (int j = 0; j <= i && ok; ++j) {
        for (int hh = 0; hh < halves(j); ++hh) {
          const uint32_t t = at + 128u * (uint32_t)bf;
          const int k0 = hh * 64 + c;            // first key of this thread's 16, inside the tile
          if (!mbar_wait_warp(B(S_FULL + bf), done(bn), abort_flag, p.status, 140)) { ok = false; break; }
          tc_fence_after();
          uint32_t dw[CW];
          // on the diagonal tile only keys <= this query count: chunks wholly after the warp's rows are zero
          if (j != i || k0 < q4 * 32 + 32) {
            float sv[CW], dv[CW];
            tc_ld16(t, sv);
            tc_ld16(t + 64u, dv);
            tc_wait_ld();
            if (j == i && k0 + CW > q4 * 32 + 1) {
#pragma unroll
              for (int e = 0; e < CW; ++e) sv[e] = (k0 + e > r) ? -INFINITY : sv[e];
            }
#pragma unroll
            for (int e = 0; e < CW; e += 2) {
              float a0, a1;
              unpack2(mul2(pack2(sv[e], sv[e + 1]), sc2), a0, a1);
              put_pair<HILO>(mul2(pack2(ex2(a0), ex2(a1)), pack2(dv[e], dv[e + 1])), dw, e >> 1);
            }
          } else {
#pragma unroll
            for (int e = 0; e < CW; ++e) dw[e] = 0u;
          }
          st_pairs<HILO>(t, dw);
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(B(P_READY + bf));
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
      }
    }
  } else if (warp < OUT_WARP0 + 4) {
    // ---------------- output warps: row statistics of the next tile, dQ (scaled) of a finished one ----------------
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    const float inv_scale = 1.0f / p.scale;
    bool ok = true;
    auto statistics = [&](int k) {
      const Unit u = units.at(k);
      const int i = p.nq - 1 - u.tile, qb = k & 1;
      const int row = i * BT + r;
      const size_t at = (size_t)u.item * p.T + row;
      const float L = row < p.T ? p.lse[at] * inv_scale : PAST_END;
      if (!mbar_wait_warp(B(QO_FULL + qb), done(k >> 1), abort_flag, p.status, 141)) { ok = false; return; }
      uint4 ov[8];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        ov[j] = *reinterpret_cast<const uint4*>(base_ptr + OFF_QO + qb * 3 * TILE + 2 * TILE + r * 128 + ((j ^ (r & 7)) << 4));
      const float D = row_product(base_ptr + OFF_QO + qb * 3 * TILE + TILE, r, ov);
      if (row < p.T) p.rowdot[at] = D;
      *reinterpret_cast<uint4*>(base_ptr + OFF_AUG + (1 + qb) * AUG_TILE + aug_row(r)) = stat_row(L, D);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(B(AUG_READY + qb));
    };
    if (units.has(0)) statistics(0);
    for (int k = 0; units.has(k); ++k) {
      const Unit u = units.at(k);
      const int i = p.nq - 1 - u.tile, item = u.item, h = item % p.H, b = item / p.H;
      const int row0 = i * BT + q4 * 32;
      bool bad = false;
      if (ok && units.has(k + 1)) statistics(k + 1);
      if (ok && !mbar_wait(B(ACC_FULL), done(k), abort_flag, p.status, 142)) ok = false;
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        tc_fence_after();
        bad = stage_rows(tDQ + lane_off, base + OFF_OUT, r, p.scale) && row0 + lane < p.T;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(B(ACC_FREE));
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      out_warps_sync();                                          // (always reached by all four)
      const bool storer = ok && warp == OUT_WARP0 && lane == 0;
      if (storer) {
        tma_store_3d(&mapDQKV, base + OFF_OUT, h * DH, i * BT, b);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      }
      bool redo = false;
      if constexpr (KEEP) redo = out_warps_any(bad); else out_warps_sync();
      if (redo) {
        if (storer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        out_warps_sync();
        if (__any_sync(0xffffffffu, bad)) {
          const rows::Head<bf16> hd(p.qkv, b, h, p.T, p.H, p.d);
          float* scratch = reinterpret_cast<float*>(base_ptr + OFF_REDO) + (warp - OUT_WARP0) * 2 * DH;
          for (int row = row0; row < min(row0 + 32, p.T); ++row) {
            const size_t stat = (size_t)item * p.T + row;
            rows::dq_row<bf16>(hd, p.d_o + ((size_t)b * p.T + row) * p.d + (size_t)h * DH, p.lse[stat], p.rowdot[stat], row, scratch,
                               p.dqkv + ((size_t)b * p.T + row) * hd.ld + (size_t)h * DH);
          }
        }
      }
    }
    if (warp == OUT_WARP0 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  RG_TEARDOWN(TMEM_COLS)
}

template <bool HILO, bool KEEP>
__global__ void __launch_bounds__(THREADS_DKV, 1)
attn64_dkv_t5_kernel(const __grid_constant__ CUtensorMap mapQKV, const __grid_constant__ CUtensorMap mapDO,
                      const __grid_constant__ CUtensorMap mapDQKV, const __grid_constant__ Params p) {
  dkv_tiles<HILO, KEEP, false>(mapQKV, mapDO, mapDQKV, p, (int)blockIdx.x, (int)gridDim.x);
}
template <bool HILO, bool KEEP>
__global__ void __launch_bounds__(THREADS_DQ, 1)
attn64_dq_t5_kernel(const __grid_constant__ CUtensorMap mapQKV, const __grid_constant__ CUtensorMap mapDO,
                     const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapDQKV, const __grid_constant__ Params p) {
  dq_tiles<HILO, KEEP>(mapQKV, mapDO, mapO, mapDQKV, p, (int)blockIdx.x, (int)gridDim.x);
}
// Few tiles: both at once on their own CTAs.  Each kernel by itself is set-up, first loads and a few steps one after another.
template <bool HILO, bool KEEP>
__global__ void __launch_bounds__(THREADS_DKV, 1)
attn64_bwd_t5_kernel(const __grid_constant__ CUtensorMap mapQKV, const __grid_constant__ CUtensorMap mapDO,
                      const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapDQKV, const __grid_constant__ Params p) {
  const int units = p.nitems * p.nq;
  if ((int)blockIdx.x < units) dkv_tiles<HILO, KEEP, true>(mapQKV, mapDO, mapDQKV, p, (int)blockIdx.x, units);
  else dq_tiles<HILO, KEEP>(mapQKV, mapDO, mapO, mapDQKV, p, (int)blockIdx.x - units, units);
}

// ==========================================================================================
// forward of a query tile
// ==========================================================================================
// Two CTAs per SM, one softmax thread per query row as in attention_t5_fwd64.cu, in steps of 32 keys.  A step's score
// products over 16 features each go to accumulators of their own and are added up in fp32 by the thread that reads them:
// the tensor core rounds each step of a chain towards zero, and the log-sum-exp, an fp32 result, shows it (relative error
// against 64 bits 4.3e-8 as a chain at 768 tokens, 2.9e-8 this way).  The one score buffer (four accumulators of 32
// columns) is released as soon as it has been read, so the next step's scores are ready when this step's softmax is done.
// P as hi + lo pairs in two buffers; O stays in tensor memory and is rescaled only when a row's maximum has moved by more
// than 2^2 since the one its exponentials are taken against (2^8 left lse 2 % further off: the exponents' rounding); the row
// sum is compensated.  Bound by the chain of a step (scores, tensor-memory loads, softmax, store, product) of two CTAs per SM:
// 16 sequences of 777 tokens, 12 heads 76 us (mma.sync 114) with the tensor pipe active for 18 % of the cycles.
namespace fwd {
constexpr int HK = 32;                                     // keys per step
constexpr int THREADS = 192;
constexpr int OFF_Q = 0, OFF_K = 2 * TILE, OFF_V = 4 * TILE, OFF_REDO = 6 * TILE, OFF_BAR = OFF_REDO + 4 * DH * 4;
constexpr int COLS = 256;                                  // scores [0, 128), O [128, 192), P [192, 224) and [224, 256)
constexpr float RESCALE_STEP = 2.0f;                       // log2 of the largest P that a stale maximum may produce
constexpr float LN2 = 0.6931471805599453f;
enum { Q_FULL = 0 /*+2*/, Q_EMPTY = 2, K_FULL = 4, K_EMPTY = 6, V_FULL = 8, V_EMPTY = 10, P_READY = 12, P_FREE = 14, S_FULL = 16, S_FREE,
       O_FREE, N_BARS };
__device__ __forceinline__ uint32_t count(int i) { return i == P_READY || i == P_READY + 1 || i == S_FREE || i == O_FREE ? 4u : 1u; }
constexpr int SMEM = OFF_BAR + 8 * N_BARS + 16 + 1024;
static_assert(2 * (SMEM + 1024) <= 228 * 1024, "two CTAs per SM");
constexpr uint32_t IDESC_S = make_idesc(BT, HK);
}  // namespace fwd

__global__ void __launch_bounds__(fwd::THREADS, 2)
attn_rg_fwd_t5_kernel(const __grid_constant__ CUtensorMap mapQKV, const __grid_constant__ Params p) {
  using namespace fwd;
  RG_SETUP(N_BARS, count, COLS)
  RG_SETUP_END()
  const Units units(p, (int)blockIdx.x, (int)gridDim.x);
  const uint32_t tS = tmem_base, tO = tmem_base + 128u, tP = tmem_base + 192u;
  auto steps = [&](int qt) { return min(4 * (qt + 1), (p.T + HK - 1) / HK); };

  if (warp == 0) {
    // ---------------- TMA producer: Q per tile (two buffers), K and V per 128 keys (two stages) ----------------
    const bool leader = elect_one();
    bool ok = true;
    int ks = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const Unit u = units.at(k);
      const int qt = p.nq - 1 - u.tile, h = u.item % p.H, b = u.item / p.H, qs = k & 1;
      if (!mbar_wait_warp(B(Q_EMPTY + qs), freed(k >> 1), abort_flag, p.status, 151)) break;
      if (leader) {
        mbar_expect_tx(B(Q_FULL + qs), TILE);
        tma_load_3d(base + OFF_Q + qs * TILE, &mapQKV, B(Q_FULL + qs), h * DH, qt * BT, b);
      }
      __syncwarp();
      for (int j = 0; j <= qt; ++j, ++ks) {
        const int s = ks & 1;
        if (!mbar_wait_warp(B(K_EMPTY + s), freed(ks >> 1), abort_flag, p.status, 152)) { ok = false; break; }
        if (leader) {
          mbar_expect_tx(B(K_FULL + s), TILE);
          tma_load_3d(base + OFF_K + s * TILE, &mapQKV, B(K_FULL + s), p.d + h * DH, j * BT, b);
        }
        __syncwarp();
        if (!mbar_wait_warp(B(V_EMPTY + s), freed(ks >> 1), abort_flag, p.status, 153)) { ok = false; break; }
        if (leader) {
          mbar_expect_tx(B(V_FULL + s), TILE);
          tma_load_3d(base + OFF_V + s * TILE, &mapQKV, B(V_FULL + s), 2 * p.d + h * DH, j * BT, b);
        }
        __syncwarp();
      }
    }
  } else if (warp == 1) {
    // ---------------- products: S(0), then S(it + 1), P(it) V for it = 0, 1, ... over all tiles ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s_k = 0, s_hs = 0, s_it = 0, s_ks = 0;              // cursor of the score products
    auto issue_s = [&]() -> bool {
      if (!units.has(s_k)) return true;
      const int nhs = steps(p.nq - 1 - units.at(s_k).tile), part = s_hs & 3, st = s_ks & 1, qs = s_k & 1;
      if (s_hs == 0 && !mbar_wait_warp(B(Q_FULL + qs), done(s_k >> 1), abort_flag, p.status, 154)) return false;
      if (part == 0 && !mbar_wait_warp(B(K_FULL + st), done(s_ks >> 1), abort_flag, p.status, 155)) return false;
      if (!mbar_wait_warp(B(S_FREE), freed(s_it), abort_flag, p.status, 156)) return false;
      tc_fence_after();
      const bool last = s_hs == nhs - 1;
      if (leader) {
        const uint32_t a = desc_lo(base + OFF_Q) + (uint32_t)qs * TILE16;
        const uint32_t b = desc_lo(base + OFF_K) + (uint32_t)st * TILE16 + (uint32_t)part * 256u;      // 32 key rows = 4096 bytes
#pragma unroll
        for (uint32_t f = 0; f < 4; ++f) tc_mma_lo(tS + 32u * f, a + 2 * f, b + 2 * f, IDESC_S, 0u);
        if (part == 3 || last) tc_commit(B(K_EMPTY + st));
        if (last) tc_commit(B(Q_EMPTY + qs));
        tc_commit(B(S_FULL));
      }
      __syncwarp();
      ++s_it;
      if (part == 3 || last) ++s_ks;
      if (last) { s_hs = 0; ++s_k; } else ++s_hs;
      return true;
    };
    ok = issue_s();
    int it = 0, ks = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int nhs = steps(p.nq - 1 - units.at(k).tile);
      for (int hs = 0; hs < nhs; ++hs, ++it) {
        const int part = hs & 3, st = ks & 1, pb = it & 1;
        if (!issue_s()) { ok = false; break; }
        if (!mbar_wait_warp(B(P_READY + pb), done(it >> 1), abort_flag, p.status, 157)) { ok = false; break; }
        if (part == 0 && !mbar_wait_warp(B(V_FULL + st), done(ks >> 1), abort_flag, p.status, 158)) { ok = false; break; }
        // the first product of a tile overwrites O: the tile before must have been read
        if (hs == 0 && !mbar_wait_warp(B(O_FREE), freed(k), abort_flag, p.status, 159)) { ok = false; break; }
        tc_fence_after();
        const bool last = hs == nhs - 1;
        if (leader) {
          const uint32_t v = desc_lo(base + OFF_V) + (uint32_t)st * TILE16 + (uint32_t)part * 256u, a = tP + (uint32_t)(pb * 32);
          tc_mma_ts_lo(tO, a, v, IDESC_64MN, hs != 0 ? 1u : 0u);
          tc_mma_ts_lo(tO, a + 8, v, IDESC_64MN, 1u);
          tc_mma_ts_lo(tO, a + 16, v + 128, IDESC_64MN, 1u);
          tc_mma_ts_lo(tO, a + 24, v + 128, IDESC_64MN, 1u);
          tc_commit(B(P_FREE + pb));                        // also says: O holds the products up to this step
          if (part == 3 || last) tc_commit(B(V_EMPTY + st));
        }
        __syncwarp();
        if (part == 3 || last) ++ks;
      }
    }
  } else {
    // ---------------- softmax and output: one thread per query row ----------------
    const int q = warp & 3;
    const int r = q * 32 + lane;                           // row inside the tile = accumulator lane
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    const float scale_log2 = p.scale_log2;
    const uint64_t sc2 = pack2(scale_log2, scale_log2);
    bool ok = true;
    int it = 0;
    // A tile's output is written one step late: its last product still runs when its last P has been handed over, so the
    // next tile's first step goes first.
    auto finish = [&](int k, float m, float l, int it_after) -> bool {
      if (!mbar_wait_warp(B(P_FREE + ((it_after - 1) & 1)), done((it_after - 1) >> 1), abort_flag, p.status, 160)) return false;
      tc_fence_after();
      float acc[DH];
      tc_ld32(tO + lane_off, acc);
      tc_ld32(tO + lane_off + 32u, acc + 32);
      tc_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(B(O_FREE));
      const Unit u = units.at(k);
      const int qt = p.nq - 1 - u.tile, item = u.item, h = item % p.H, b = item / p.H;
      const int row = qt * BT + r;
      const float inv = 1.0f / l;
      uint32_t bad = 0;
      uint4 w[DH / 8];
#pragma unroll
      for (int jj = 0; jj < DH / 8; ++jj) {
        uint32_t* wp = reinterpret_cast<uint32_t*>(&w[jj]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __nv_bfloat162 ob = __floats2bfloat162_rn(acc[8 * jj + 2 * i] * inv, acc[8 * jj + 2 * i + 1] * inv);
          wp[i] = *reinterpret_cast<const uint32_t*>(&ob);
          bad |= ((wp[i] & 0x7f807f80u) + 0x00800080u) & 0x80008000u;
        }
      }
      if (row < p.T) {
        bf16* orow = p.o + ((size_t)b * p.T + row) * p.d + (size_t)h * DH;
#pragma unroll
        for (int jj = 0; jj < DH / 8; ++jj) *reinterpret_cast<uint4*>(orow + 8 * jj) = w[jj];
        // from the maximum as it entered the exponents, so that its rounding cancels
        p.lse_out[(size_t)item * p.T + row] = fmaf(m * scale_log2, LN2, logf(l));
      }
      if (__any_sync(0xffffffffu, bad != 0 && row < p.T)) {
        __syncwarp();
        const rows::Head<bf16> hd(p.qkv, b, h, p.T, p.H, p.d);
        float* scratch = reinterpret_cast<float*>(base_ptr + OFF_REDO) + (warp - 2) * DH;
        const int row0 = qt * BT + q * 32;
        for (int i = row0; i < min(row0 + 32, p.T); ++i)
          rows::forward_row<bf16>(hd, i, scratch, p.o + ((size_t)b * p.T + i) * p.d + (size_t)h * DH, p.lse_out + (size_t)item * p.T + i);
      }
      return true;
    };
    bool pend = false;
    float pend_m = 0.f, pend_l = 1.f;
    int pend_k = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int qt = p.nq - 1 - units.at(k).tile, nhs = steps(qt);
      float m_run = -INFINITY, m_ref = -INFINITY;            // maxima of the unscaled scores; m_ref: the one in the exponents
      float l_run = 0.f, l_rest = 0.f;                       // the row sum, and what its roundings have left (one addition per 32 keys)
      for (int hs = 0; hs < nhs; ++hs, ++it) {
        const int pb = it & 1, e = hs - 4 * qt;            // e: block of 32 keys inside the diagonal tile
        if (!mbar_wait_warp(B(S_FULL), done(it), abort_flag, p.status, 161)) { ok = false; break; }
        tc_fence_after();
        uint32_t pk[32];
        if (e <= q) {                                      // (else all of these keys are hidden from this warp's rows)
          float v[HK], x[HK];
          tc_ld32(tS + lane_off, v);
          tc_ld32(tS + lane_off + 32u, x);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < HK; i += 2) unpack2(add2(pack2(v[i], v[i + 1]), pack2(x[i], x[i + 1])), v[i], v[i + 1]);
          float y[HK];
          tc_ld32(tS + lane_off + 64u, x);
          tc_ld32(tS + lane_off + 96u, y);
          tc_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(B(S_FREE));           // the scores are in registers: the buffer may be overwritten
#pragma unroll
          for (int i = 0; i < HK; i += 2)
            unpack2(add2(add2(pack2(v[i], v[i + 1]), pack2(x[i], x[i + 1])), pack2(y[i], y[i + 1])), v[i], v[i + 1]);
          if (e == q) {
#pragma unroll
            for (int i = 0; i < HK; ++i) v[i] = (i > lane) ? -INFINITY : v[i];
          }
          float m4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
          for (int i = 4; i < HK; i += 4) {
            m4[0] = fmaxf(m4[0], v[i]); m4[1] = fmaxf(m4[1], v[i + 1]); m4[2] = fmaxf(m4[2], v[i + 2]); m4[3] = fmaxf(m4[3], v[i + 3]);
          }
          const float m_new = fmaxf(m_run, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));   // finite: key 0 is visible to every row
          m_run = m_new;
          if (hs == 0) {
            m_ref = m_new;
          } else {
            const bool need = (m_new - m_ref) * scale_log2 > RESCALE_STEP;
            if (__any_sync(0xffffffffu, need)) {
              // O must hold the products up to step it - 1 (the next one waits for P_READY below); that product's commit is
              // the next phase of its P buffer's barrier that this thread has not seen
              if (!mbar_wait_warp(B(P_FREE + ((it - 1) & 1)), done((it - 1) >> 1), abort_flag, p.status, 162)) { ok = false; break; }
              tc_fence_after();
              const float corr = need ? ex2((m_ref - m_new) * scale_log2) : 1.0f;
#pragma unroll
              for (int oc = 0; oc < DH; oc += 32) {
                float ov[32];
                tc_ld32(tO + lane_off + (uint32_t)oc, ov);
                tc_wait_ld();
                uint32_t w[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) w[i] = __float_as_uint(ov[i] * corr);
                tc_st16(tO + lane_off + (uint32_t)oc, w);
                tc_st16(tO + lane_off + (uint32_t)(oc + 16), w + 16);
              }
              l_run *= corr; l_rest *= corr;
              if (need) m_ref = m_new;
            }
          }
          const float k0 = -m_ref * scale_log2;
          const uint64_t k2 = pack2(k0, k0);
          uint64_t ps2[4] = {0, 0, 0, 0};                      // eight chains of four
#pragma unroll
          for (int i = 0; i < HK; i += 2) {
            float a0, a1;
            unpack2(fma2(pack2(v[i], v[i + 1]), sc2, k2), a0, a1);
            const uint64_t pv = pack2(ex2(a0), ex2(a1));
            ps2[(i >> 1) & 3] = add2(ps2[(i >> 1) & 3], pv);
            put_pair<true>(pv, pk, (i >> 4) * 16 + ((i & 15) >> 1));
          }
          float s0, s1;
          unpack2(add2(add2(ps2[0], ps2[1]), add2(ps2[2], ps2[3])), s0, s1);
          const float add = (s0 + s1) + l_rest, sum = l_run + add;
          l_rest = add - (sum - l_run);
          l_run = sum;
        } else {
          __syncwarp();
          if (lane == 0) mbar_arrive(B(S_FREE));
#pragma unroll
          for (int i = 0; i < 32; ++i) pk[i] = 0u;
        }
        // the product that read this P buffer two steps ago must be done
        if (!mbar_wait_warp(B(P_FREE + pb), freed(it >> 1), abort_flag, p.status, 163)) { ok = false; break; }
        tc_fence_after();
        tc_st16(tP + lane_off + (uint32_t)(pb * 32), pk);
        tc_st16(tP + lane_off + (uint32_t)(pb * 32 + 16), pk + 16);
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(B(P_READY + pb));
        if (hs == 0 && pend) {                             // the tile before (its products are done by now)
          if (!finish(pend_k, pend_m, pend_l, it)) { ok = false; break; }
          pend = false;
        }
      }
      pend = true; pend_m = m_ref; pend_l = l_run + l_rest; pend_k = k;
    }
    if (ok && pend) finish(pend_k, pend_m, pend_l, it);
  }
  RG_TEARDOWN(COLS)
}

constexpr int BWD_SMEM = dkv::SMEM > dq::SMEM ? dkv::SMEM : dq::SMEM;
PerDeviceOnce g_once;

bool init_device() {
  const int dev = current_device();
  if (dev < 0 || !tensor_map_encoder()) return false;
  if (!g_once.needed(dev)) return true;
  auto allow = [](const void* kernel, int bytes) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess; };
  if (!allow((const void*)attn_rg_fwd_t5_kernel, fwd::SMEM)) return false;
  if (!allow((const void*)attn64_bwd_t5_kernel<true, true>, BWD_SMEM) || !allow((const void*)attn64_dkv_t5_kernel<true, true>, dkv::SMEM) || !allow((const void*)attn64_dq_t5_kernel<true, true>, dq::SMEM)) return false;
  if (!allow((const void*)attn64_bwd_t5_kernel<false, true>, BWD_SMEM) || !allow((const void*)attn64_dkv_t5_kernel<false, true>, dkv::SMEM) || !allow((const void*)attn64_dq_t5_kernel<false, true>, dq::SMEM)) return false;
  if (!allow((const void*)attn64_bwd_t5_kernel<false, false>, BWD_SMEM) || !allow((const void*)attn64_dkv_t5_kernel<false, false>, dkv::SMEM) || !allow((const void*)attn64_dq_t5_kernel<false, false>, dq::SMEM)) return false;
  g_once.done(dev);
  return true;
}

// a plane of T rows per sequence, box = 64 columns x 128 rows of one plane
bool make_map(CUtensorMap* m, const void* ptr, int nseq, int T, int cols) {
  return cached_map_3d(m, ptr, (uint64_t)nseq, (uint64_t)T, (uint64_t)cols, (uint64_t)cols, (uint64_t)T * cols, 64, (uint32_t)BT,
                       CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

Params shape(int nseq, int T, int H, int d, const void* qkv, int* status) {
  Params p = {};
  p.T = T; p.H = H; p.d = d; p.nitems = nseq * H; p.nq = (T + BT - 1) / BT;
  p.last_halves = T - (p.nq - 1) * BT > 64 ? 2 : 1;
  // q, k, v, o, dO of a block's items: 640 T bytes each, 96 MB together (L2 has 126; in blocks half that size 16 sequences of
  // 777, 12 heads, were 132 us against 123, because every block begins with its longest tiles)
  const int64_t fit = (int64_t)96 * 1024 * 1024 / (640 * (int64_t)T);
  p.block = fit < 1 ? 1 : fit < p.nitems ? (int)fit : p.nitems;
  p.scale = 1.0f / sqrtf((float)DH); p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)DH)); p.qkv = (const bf16*)qkv; p.status = status;
  return p;
}

}  // namespace

bool attention_ragged_t5_supported(int nseq, int T, int H, int d) {
  return H > 0 && d % H == 0 && d / H == DH && T >= 1 && nseq >= 1 && (int64_t)nseq * H * ((T + BT - 1) / BT) < (1 << 30);
}

namespace {
template <bool HILO, bool KEEP>
cudaError_t launch_bwd(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H, int d, void* dqkv,
                       float* rowdot, int* status, cudaStream_t st) {
  if (!attention_ragged_t5_supported(nseq, T, H, d)) return cudaErrorInvalidValue;
  if (!init_device()) return cudaErrorInitializationError;
  const int sms = num_sms();
  if (!status) status = library_status_word();
  if (!status || sms < 1) return cudaErrorInitializationError;
  CUtensorMap mQKV, mDO, mO, mDQKV;
  if (!make_map(&mQKV, qkv, nseq, T, 3 * d) || !make_map(&mDO, d_o, nseq, T, d) || !make_map(&mO, o, nseq, T, d) ||
      !make_map(&mDQKV, dqkv, nseq, T, 3 * d))
    return cudaErrorInvalidValue;
  Params p = shape(nseq, T, H, d, qkv, status);
  p.lse = lse; p.rowdot = rowdot; p.d_o = (const bf16*)d_o; p.dqkv = (bf16*)dqkv; p.o = (bf16*)const_cast<void*>(o);
  const int units = p.nitems * p.nq;
  if (2 * units <= sms) {
    launch_overlapped(attn64_bwd_t5_kernel<HILO, KEEP>, 2 * units, THREADS_DKV, BWD_SMEM, st, mQKV, mDO, mO, mDQKV, p);
    return cudaGetLastError();
  }
  const int grid = units < sms ? units : sms;
  launch_overlapped(attn64_dq_t5_kernel<HILO, KEEP>, grid, THREADS_DQ, dq::SMEM, st, mQKV, mDO, mO, mDQKV, p);
  launch_overlapped(attn64_dkv_t5_kernel<HILO, KEEP>, grid, THREADS_DKV, dkv::SMEM, st, mQKV, mDO, mDQKV, p);
  return cudaGetLastError();
}
}  // namespace

cudaError_t attention_bwd_ragged_t5(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                    int d, void* dqkv, float* rowdot, int* status, cudaStream_t st) {
  return launch_bwd<true, true>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st);
}
cudaError_t attention_bwd_t5_w64(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                 int d, void* dqkv, float* rowdot, int* status, cudaStream_t st) {
  return T % BT != 0 ? launch_bwd<false, true>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st)
                     : launch_bwd<false, false>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st);
}

cudaError_t attention_fwd_ragged_t5(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status, cudaStream_t st) {
  if (!attention_ragged_t5_supported(nseq, T, H, d)) return cudaErrorInvalidValue;
  if (!init_device()) return cudaErrorInitializationError;
  const int sms = num_sms();
  if (!status) status = library_status_word();
  if (!status || sms < 1) return cudaErrorInitializationError;
  CUtensorMap mQKV;
  if (!make_map(&mQKV, qkv, nseq, T, 3 * d)) return cudaErrorInvalidValue;
  Params p = shape(nseq, T, H, d, qkv, status);
  p.o = (bf16*)o; p.lse_out = lse;
  const int units = p.nitems * p.nq;
  launch_overlapped(attn_rg_fwd_t5_kernel, units < 2 * sms ? units : 2 * sms, fwd::THREADS, fwd::SMEM, st, mQKV, p);
  return cudaGetLastError();
}

}  // namespace sl
