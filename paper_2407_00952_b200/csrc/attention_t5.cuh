// Building blocks of the tcgen05 attention backward kernels: tile sizes, the augmented contraction's operand tiles,
// tensor-memory loads and stores, staging of output rows.
#pragma once
#include "tc_common.cuh"

namespace sl {
namespace t5 {

using namespace tc;

constexpr int DH = 64;
constexpr int BT = 128;                   // rows of a query tile and of a key tile
constexpr int TILE = BT * DH * 2;         // 16 KB: one [128 x 64] bf16 tile
constexpr int OUT_THREADS = 128;

// Operand tiles of an augmented contraction: [128 rows x 16] bf16, K-major without swizzle: 8-row groups of 256 bytes, in
// a group the 16-byte rows of columns 0..7 (128 bytes) and then those of columns 8..15.
constexpr int AUG_TILE = 128 * 16 * 2;
constexpr uint32_t DESC_HI_AUG = (uint32_t)(256 >> 4) | (1u << 14);           // 8-row groups 256 bytes apart, no swizzle
__device__ __forceinline__ uint32_t desc_lo_aug(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | ((uint32_t)(128 >> 4) << 16); }
__device__ __forceinline__ void tc_mma_aug(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, 1, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(DESC_HI_AUG), "r"(idesc) : "memory");
}
// byte offset of row r's columns 0..7 inside such a tile
__device__ __forceinline__ uint32_t aug_row(int r) { return (uint32_t)(r >> 3) * 256u + (uint32_t)(r & 7) * 16u; }

constexpr int TMEM_COLS = 512;
constexpr uint32_t IDESC_64KK = make_idesc(BT, DH);                   // [128 x 64] products, both operands K-major
constexpr uint32_t IDESC_64MN = make_idesc(BT, DH) | (1u << 16);      // [128 x 64] products, right operand MN-major
constexpr float LOG2E = 1.4426950408889634f;

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// 16 consecutive tensor-memory columns of this thread's lane
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// 8 packed words of this thread's lane to 8 consecutive tensor-memory columns
__device__ __forceinline__ void tc_st8(uint32_t taddr, const uint32_t* w) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
      ::"r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1) : "memory");
}
// one row (lane r) of a [128 x 64] bf16 tile in the 128-byte-swizzled layout: 16-byte chunk jj
__device__ __forceinline__ void st_row_chunk(uint32_t tile, int r, uint32_t jj, const uint32_t* w) {
  const uint32_t addr = tile + (uint32_t)r * 128u + ((jj ^ ((uint32_t)r & 7u)) << 4);
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}
// 4 products [128 x 64] = A[128 x 64] * (rows [64h, 64h + 64) of the K-major tile at blo)^T:
// one half (64 columns) of a [128 x 128] score tile.  64 rows of 128 bytes = 512 descriptor units.
__device__ __forceinline__ void mma_score_half(uint32_t d_tmem, uint32_t alo, uint32_t blo, int h, bool fresh = true) {
  const uint32_t b0 = blo + (uint32_t)(512 * h);
  tc_mma_lo(d_tmem, alo, b0, IDESC_64KK, fresh ? 0u : 1u);
  tc_mma_lo_acc(d_tmem, alo + 2, b0 + 2, IDESC_64KK);
  tc_mma_lo_acc(d_tmem, alo + 4, b0 + 4, IDESC_64KK);
  tc_mma_lo_acc(d_tmem, alo + 6, b0 + 6, IDESC_64KK);
}

// parity to wait on for "the n-th completion (0-based) of this barrier has happened"
__device__ __forceinline__ uint32_t done(int n) { return (uint32_t)n & 1u; }
// parity to wait on before the n-th use of a slot whose release is signalled once per use
__device__ __forceinline__ uint32_t freed(int n) { return ((uint32_t)n & 1u) ^ 1u; }

}  // namespace t5
}  // namespace sl
