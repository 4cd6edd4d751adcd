// Causal multi-head attention backward on the 5th-generation tensor cores for sequences of any length, bf16, head width 64.
// The same two kernels as in attention_t5_bwd.cu (dQ per query tile, then dK / dV per key tile, tiles of 128 rows, no
// atomics, bit-reproducible) with three differences:
//   * Sequences are planes of three-dimensional tensor maps: rows past the end of a sequence arrive as zeros and are
//     clipped on the way out.  A query row past the end carries a row statistic of -1e30, i.e. P = 0.
//   * P and dS enter their products as two bf16 values each (hi + lo, 16 mantissa bits), because these shapes have always
//     held them in more than bf16 (attention_tc.cu).  A 16-column chunk of fp32 scores in tensor memory is replaced by its
//     own 16 elements: 8 columns of hi pairs, 8 of lo pairs; a product over 16 elements is issued once with each.
//   * lse/scale and D enter the score products as three bf16 values (24 bits), exact to fp32.
// With P and dS on top of the scores a half-step (64 columns of S and of dP) takes 128 tensor-memory columns, so three
// half-steps are in flight next to dK and dV: the score products of one, the element-wise work of another, the
// accumulating products of the third.
// A row whose results are not all finite is done again in plain FMA over its visible pairs (attention_rows.cuh), because a
// product multiplies the zero probability of a hidden pair with whatever the tile holds.
// What bounds them: the tensor pipe.  A half-step is 10 + 16 (dQ: 10 + 8) products [128 x 64 x 16] of 45-48 cycles
// (operand reads from shared memory), next to about 512 cycles of exponentials: 80 us for 16 sequences of 777 tokens,
// 12 heads, which take 123 us (mma.sync, attention_tc.cu: 339); errors against 64 bits agree with that form's to four digits.
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
  int T, H, d, nitems, nq, last_halves;       // nq: tiles of 128; last_halves: 64-row halves of the last tile that hold rows
  float scale;
  const float* lse;
  float* rowdot;
  const bf16 *qkv, *d_o;
  bf16* dqkv;
  int* status;
};

// Work units are (tile, item) pairs, item = (sequence, head), longest tiles first; a CTA takes one of each round of gridDim
// units, forwards in even rounds and backwards in odd ones, so that all get about the same number of steps.
struct Units {
  int n, grid, cta;
  __device__ __forceinline__ explicit Units(const Params& p) : n(p.nitems * p.nq), grid((int)gridDim.x), cta((int)blockIdx.x) {}
  __device__ __forceinline__ int at(int k) const { return k * grid + ((k & 1) ? grid - 1 - cta : cta); }
  __device__ __forceinline__ bool has(int k) const { return k * grid < n && at(k) < n; }
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

// 8 products [128 x 64] += (hi + lo of A)[128 x 64] * B rows [64 hh, 64 hh + 64), B an MN-major tile used as loaded; A in
// tensor memory at a_tmem, per 16 elements 8 columns of hi and 8 of lo
__device__ __forceinline__ void mma_acc_hilo(uint32_t d_tmem, uint32_t a_tmem, uint32_t blo, int hh, bool fresh) {
  const uint32_t b0 = blo + (uint32_t)(512 * hh);
  tc_mma_ts_lo(d_tmem, a_tmem, b0, IDESC_64MN, fresh ? 0u : 1u);
  tc_mma_ts_lo(d_tmem, a_tmem + 8, b0, IDESC_64MN, 1u);
#pragma unroll
  for (uint32_t k = 1; k < 4; ++k) {
    tc_mma_ts_lo(d_tmem, a_tmem + 16 * k, b0 + 128 * k, IDESC_64MN, 1u);
    tc_mma_ts_lo(d_tmem, a_tmem + 16 * k + 8, b0 + 128 * k, IDESC_64MN, 1u);
  }
}

// bf16 pairs of two values and of what that rounding leaves
__device__ __forceinline__ void split_pair(uint64_t v, uint32_t& hi, uint32_t& lo) {
  float a, b, ra, rb;
  unpack2(v, a, b);
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  unpack2(add2(v, pack2(__uint_as_float((hi << 16) ^ 0x80000000u), __uint_as_float((hi & 0xffff0000u) ^ 0x80000000u))), ra, rb);
  const __nv_bfloat162 l = __floats2bfloat162_rn(ra, rb);
  lo = *reinterpret_cast<const uint32_t*>(&l);
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

#define RG_SETUP(NBARS, COUNT)                                                                            \
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
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)TMEM_COLS) : "memory");           \
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");              \
  }

#define RG_SETUP_END()                                                                                    \
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");                                            \
  tc_fence_before();                                                                                      \
  __syncthreads();                                                                                        \
  tc_fence_after();                                                                                       \
  const uint32_t tmem_base = *tmem_slot;                                                                  \
  overlap_sync();

#define RG_TEARDOWN()                                                                                     \
  __syncwarp();                                                                                           \
  if (*abort_flag) { for (int i = 0; i < 2000; ++i) __nanosleep(1000); }                                  \
  tc_fence_before();                                                                                      \
  __syncthreads();                                                                                        \
  if (warp == 1) {                                                                                        \
    tc_fence_after();                                                                                     \
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory"); \
  }

// ==========================================================================================
// dK, dV of a key tile: query tiles i >= kt
// ==========================================================================================
namespace dkv {
enum { KV_FULL = 0 /*+buffer*/, KV_EMPTY = 2, QD_FULL = 4 /*+stage*/, QD_EMPTY = QD_FULL + RING, AUG_READY = QD_EMPTY + RING,
       S_FULL = AUG_READY + RING /*+half-step*/, P_READY = S_FULL + NBUF, P_FREE = P_READY + NBUF, ACC_FULL = P_FREE + NBUF, ACC_FREE,
       N_BARS };
__device__ __forceinline__ uint32_t count(int i) {
  return i >= QD_EMPTY && i < QD_EMPTY + RING ? 2u : i >= P_READY && i < P_READY + NBUF ? (uint32_t)EW_WARPS : i == ACC_FREE ? 4u : 1u;
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

__global__ void __launch_bounds__(THREADS_DKV, 1)
attn_rg_dkv_t5_kernel(const __grid_constant__ CUtensorMap mapQKV, const __grid_constant__ CUtensorMap mapDO,
                      const __grid_constant__ CUtensorMap mapDQKV, Params p) {
  using namespace dkv;
  RG_SETUP(N_BARS, count)
  init_ones(base_ptr + OFF_AUG, base_ptr + OFF_AUG + AUG_TILE, BT, base_ptr + OFF_AUG + 2 * AUG_TILE, RING * AUG_TILE);
  RG_SETUP_END()
  const Units units(p);
  const uint32_t tDV = tmem_base + 128u * NBUF, tDK = tDV + 64u;
  auto halves = [&](int i) { return i == p.nq - 1 ? p.last_halves : 2; };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0;                            // ring stage and how often it has been used
    for (int k = 0; units.has(k) && ok; ++k) {
      const int u = units.at(k), kt = u / p.nitems, item = u % p.nitems, h = item % p.H, b = item / p.H, kb = k & 1;
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
      const int kt = units.at(k) / p.nitems, kb = k & 1;
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
      const int kt = units.at(k) / p.nitems;
      if (!mbar_wait_warp(B(ACC_FREE), freed(k), abort_flag, p.status, 117)) break;
      for (int i = kt; i < p.nq && ok; ++i) {
        const uint32_t lo_q = desc_lo(base + OFF_QD) + (uint32_t)(s * 2) * TILE16, lo_do = lo_q + TILE16;
        if (!mbar_wait_warp(B(QD_FULL + s), done(n), abort_flag, p.status, 118)) { ok = false; break; }
        for (int hh = 0; hh < halves(i); ++hh) {
          if (!mbar_wait_warp(B(P_READY + bf), done(bn), abort_flag, p.status, 119)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tP = tmem_base + 128u * (uint32_t)bf;
          if (leader) {
            mma_acc_hilo(tDV, tP, lo_do, hh, i == kt && hh == 0);
            mma_acc_hilo(tDK, tP + 64u, lo_q, hh, i == kt && hh == 0);
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
      const int kt = units.at(k) / p.nitems;
      for (int i = kt; i < p.nq && ok; ++i) {
        for (int hh = 0; hh < halves(i); ++hh) {
          const uint32_t t = at + 128u * (uint32_t)bf;
          const int q0 = hh * 64 + c;            // first query of this thread's 16, inside the tile
          if (!mbar_wait_warp(B(S_FULL + bf), done(bn), abort_flag, p.status, 120)) { ok = false; break; }
          tc_fence_after();
          uint32_t pw[CW], dw[CW];               // 8 words of hi, 8 of lo
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
              split_pair(pv, pw[e >> 1], pw[8 + (e >> 1)]);
              split_pair(mul2(pv, pack2(dv[e], dv[e + 1])), dw[e >> 1], dw[8 + (e >> 1)]);
            }
          } else {
#pragma unroll
            for (int e = 0; e < CW; ++e) { pw[e] = 0u; dw[e] = 0u; }
          }
          tc_st16(t, pw);
          tc_st16(t + 64u, dw);
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(B(P_READY + bf));
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
      }
    }
  } else if (warp == STAT_WARP) {
    // ---------------- -lse/scale and -D of a stage's queries as operand rows ----------------
    const float inv_scale = 1.0f / p.scale;
    bool ok = true;
    int s = 0, n = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int u = units.at(k), kt = u / p.nitems;
      const size_t stat0 = (size_t)(u % p.nitems) * p.T;
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
  } else {
    // ---------------- output: dK (scaled) and dV of a finished key tile ----------------
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    bool ok = true;
    for (int k = 0; units.has(k); ++k) {
      const int u = units.at(k), kt = u / p.nitems, item = u % p.nitems, h = item % p.H, b = item / p.H;
      const int row0 = kt * BT + q4 * 32;
      bool bad = false;
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
      if (out_warps_any(bad)) {
        if (storer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        out_warps_sync();
        if (__any_sync(0xffffffffu, bad)) {
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
  RG_TEARDOWN()
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

__global__ void __launch_bounds__(THREADS_DQ, 1)
attn_rg_dq_t5_kernel(const __grid_constant__ CUtensorMap mapQKV, const __grid_constant__ CUtensorMap mapDO,
                     const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapDQKV, Params p) {
  using namespace dq;
  RG_SETUP(N_BARS, count)
  init_ones(base_ptr + OFF_AUG, base_ptr + OFF_AUG + AUG_TILE / 2, 64, base_ptr + OFF_AUG + AUG_TILE, 2 * AUG_TILE);
  RG_SETUP_END()
  const Units units(p);
  const uint32_t tDQ = tmem_base + 128u * NBUF;
  auto halves = [&](int j) { return j == p.nq - 1 ? p.last_halves : 2; };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, n = 0;
    for (int k = 0; units.has(k) && ok; ++k) {
      const int u = units.at(k), i = p.nq - 1 - u / p.nitems, item = u % p.nitems, h = item % p.H, b = item / p.H, qb = k & 1;
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
      const int i = p.nq - 1 - units.at(k) / p.nitems, qb = k & 1;
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
      const int i = p.nq - 1 - units.at(k) / p.nitems;
      if (!mbar_wait_warp(B(ACC_FREE), freed(k), abort_flag, p.status, 137)) break;
      for (int j = 0; j <= i && ok; ++j) {
        const uint32_t lo_k = desc_lo(base + OFF_KV) + (uint32_t)(s * 2) * TILE16;
        if (!mbar_wait_warp(B(KV_FULL + s), done(n), abort_flag, p.status, 138)) { ok = false; break; }
        for (int hh = 0; hh < halves(j); ++hh) {
          if (!mbar_wait_warp(B(P_READY + bf), done(bn), abort_flag, p.status, 139)) { ok = false; break; }
          tc_fence_after();
          if (leader) {
            mma_acc_hilo(tDQ, tmem_base + 128u * (uint32_t)bf, lo_k, hh, j == 0 && hh == 0);
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
      const int i = p.nq - 1 - units.at(k) / p.nitems;
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
              split_pair(mul2(pack2(ex2(a0), ex2(a1)), pack2(dv[e], dv[e + 1])), dw[e >> 1], dw[8 + (e >> 1)]);
            }
          } else {
#pragma unroll
            for (int e = 0; e < CW; ++e) dw[e] = 0u;
          }
          tc_st16(t, dw);
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(B(P_READY + bf));
          if (++bf == NBUF) { bf = 0; ++bn; }
        }
      }
    }
  } else {
    // ---------------- output warps: row statistics of the next tile, dQ (scaled) of a finished one ----------------
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    const float inv_scale = 1.0f / p.scale;
    bool ok = true;
    auto statistics = [&](int k) {
      const int u = units.at(k), i = p.nq - 1 - u / p.nitems, qb = k & 1;
      const int row = i * BT + r;
      const size_t at = (size_t)(u % p.nitems) * p.T + row;
      const float L = row < p.T ? p.lse[at] * inv_scale : PAST_END;
      if (!mbar_wait_warp(B(QO_FULL + qb), done(k >> 1), abort_flag, p.status, 141)) { ok = false; return; }
      // dO and O tiles have the same swizzle, so 16-byte chunk j of one row holds the same eight columns in both
      const uint8_t* dorow = base_ptr + OFF_QO + qb * 3 * TILE + TILE + r * 128;
      const uint8_t* orow = dorow + TILE;
      float D = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int jj = (j ^ (r & 7)) << 4;       // lanes of a warp spread over all banks
        const uint4 av = *reinterpret_cast<const uint4*>(dorow + jj);
        const uint4 bv = *reinterpret_cast<const uint4*>(orow + jj);
        const uint32_t* aw = reinterpret_cast<const uint32_t*>(&av);
        const uint32_t* bw = reinterpret_cast<const uint32_t*>(&bv);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          D = fmaf(__uint_as_float(aw[e] << 16), __uint_as_float(bw[e] << 16), D);
          D = fmaf(__uint_as_float(aw[e] & 0xffff0000u), __uint_as_float(bw[e] & 0xffff0000u), D);
        }
      }
      if (row < p.T) p.rowdot[at] = D;
      *reinterpret_cast<uint4*>(base_ptr + OFF_AUG + (1 + qb) * AUG_TILE + aug_row(r)) = stat_row(L, D);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(B(AUG_READY + qb));
    };
    if (units.has(0)) statistics(0);
    for (int k = 0; units.has(k); ++k) {
      const int u = units.at(k), i = p.nq - 1 - u / p.nitems, item = u % p.nitems, h = item % p.H, b = item / p.H;
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
      if (out_warps_any(bad)) {
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
  RG_TEARDOWN()
}

PerDeviceOnce g_once;

bool init_device() {
  const int dev = current_device();
  if (dev < 0 || !tensor_map_encoder()) return false;
  if (!g_once.needed(dev)) return true;
  if (cudaFuncSetAttribute(attn_rg_dkv_t5_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dkv::SMEM) != cudaSuccess) return false;
  if (cudaFuncSetAttribute(attn_rg_dq_t5_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dq::SMEM) != cudaSuccess) return false;
  g_once.done(dev);
  return true;
}

// a plane of T rows per sequence, box = 64 columns x 128 rows of one plane
bool make_map(CUtensorMap* m, const void* ptr, int nseq, int T, int cols) {
  return cached_map_3d(m, ptr, (uint64_t)nseq, (uint64_t)T, (uint64_t)cols, (uint64_t)cols, (uint64_t)T * cols, 64, (uint32_t)BT,
                       CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

}  // namespace

bool attention_bwd_ragged_t5_supported(int nseq, int T, int H, int d) {
  return H > 0 && d % H == 0 && d / H == DH && T >= 1 && nseq >= 1 && (int64_t)nseq * H * ((T + BT - 1) / BT) < (1 << 30);
}

cudaError_t attention_bwd_ragged_t5(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                    int d, void* dqkv, float* rowdot, int* status, cudaStream_t st) {
  if (!attention_bwd_ragged_t5_supported(nseq, T, H, d)) return cudaErrorInvalidValue;
  if (!init_device()) return cudaErrorInitializationError;
  const int sms = num_sms();
  if (!status) status = library_status_word();
  if (!status || sms < 1) return cudaErrorInitializationError;
  CUtensorMap mQKV, mDO, mO, mDQKV;
  if (!make_map(&mQKV, qkv, nseq, T, 3 * d) || !make_map(&mDO, d_o, nseq, T, d) || !make_map(&mO, o, nseq, T, d) ||
      !make_map(&mDQKV, dqkv, nseq, T, 3 * d))
    return cudaErrorInvalidValue;
  Params p;
  p.T = T; p.H = H; p.d = d; p.nitems = nseq * H; p.nq = (T + BT - 1) / BT;
  p.last_halves = T - (p.nq - 1) * BT > 64 ? 2 : 1;
  p.scale = 1.0f / sqrtf((float)DH); p.lse = lse; p.rowdot = rowdot; p.qkv = (const bf16*)qkv; p.d_o = (const bf16*)d_o;
  p.dqkv = (bf16*)dqkv; p.status = status;
  const int units = p.nitems * p.nq;
  const int grid = units < sms ? units : sms;
  launch_overlapped(attn_rg_dq_t5_kernel, grid, THREADS_DQ, dq::SMEM, st, mQKV, mDO, mO, mDQKV, p);
  launch_overlapped(attn_rg_dkv_t5_kernel, grid, THREADS_DKV, dkv::SMEM, st, mQKV, mDO, mDQKV, p);
  return cudaGetLastError();
}

}  // namespace sl
