// Causal multi-head attention on tensor cores (bf16 operands, fp32 softmax and accumulation).
// Flash-style: scores are never written to memory; the forward keeps only the log-sum-exp per row, the
// backward recomputes probabilities.  Two forms of every kernel (template parameter RG):
//   RG = false: head width 64 or 128, sequence length a multiple of 64; P and dS enter their products as bf16.
//   RG = true:  any sequence length and any head width that is a multiple of 8 up to 128 (padded with zeros to
//     DH = 32, 64, 96 or 128 in shared memory; rows past the end of a sequence are zero-filled, never stored,
//     and as queries carry lse = +inf, i.e. P = 0).  These shapes otherwise run on the plain-FMA kernels, which
//     hold P and dS in fp32, so here each of them enters its product as a sum of two bf16 values (hi + lo, 16
//     mantissa bits) against the exact bf16 operand: twice the products of that operand, none of the precision
//     lost (error of o / dqkv against 64 bits over odd T is that of the bf16 output alone, as before).  Measured,
//     16 sequences of 777 tokens, 12 heads of 64, forward + backward: 466 us against 72.9 ms; width 64 now runs on
//     tcgen05 from the lengths and tile counts on that the two dispatches below give (196 us, attention_t5_ragged.cu).
//     Bound by the tensor issue of mma.sync and by ldmatrix traffic (the hi and lo products share one fragment of the
//     right operand).  Shapes that the aligned forms take stay with them.
//   forward : one CTA per (sequence, head, 64-row query tile), 4 warps x 16 rows, K/V tiles double
//             buffered in shared memory with cp.async, online softmax in registers.
//   backward: rowdot = sum(dO*O); a dQ kernel per query tile (loops over key tiles) and a dK/dV
//             kernel per key tile (loops over query tiles).  No atomics: results are bit-reproducible.
// Products use mma.sync m16n8k16 with ldmatrix-fed fragments from XOR-swizzled shared tiles.

#include "attention_rows.cuh"
#include "common.cuh"
#include "host_common.h"
#include "kernels.h"
#include "launch.cuh"

namespace sl {
namespace {

constexpr int BT = 64;            // rows of a query tile and of a key tile
constexpr int NT = 128;           // threads per CTA
constexpr float LOG2E = 1.4426950408889634f;
constexpr float LN2 = 0.6931471805599453f;

template <int DH> struct Sizes {
  static constexpr int TILE = BT * DH * 2;     // bytes of one [64][DH] bf16 tile
  static constexpr int FWD = 5 * TILE, DQ = 6 * TILE, DKV = 6 * TILE + 4 * BT * 4;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of element (r, c) in a [64][DH] bf16 tile; the 16-byte chunks of every 128-byte
// segment of a row are XOR-swizzled by the row index (rows that are an odd number of 64-byte segments: the
// chunks of every 64-byte segment by half the row index, two rows sharing 128 bytes of banks)
template <int DH> __device__ __forceinline__ uint32_t swz(int r, int c) {
  int ch = c >> 3;
  if constexpr (DH % 64 != 0)
    return (uint32_t)(r * (DH * 2) + ((((ch & ~3) | ((ch & 3) ^ ((r >> 1) & 3))) << 4) | ((c & 7) << 1)));
  return (uint32_t)(r * (DH * 2) + ((((ch & ~7) | ((ch & 7) ^ (r & 7))) << 4) | ((c & 7) << 1)));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// 16 bytes, or zeros without touching `src` when !valid
__device__ __forceinline__ void cp_async16_or_zero(uint32_t dst, const void* src, bool valid) {
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 64 x DH bf16 tile, global rows `ld` elements apart -> swizzled shared tile.  RG: only `rows` rows of `dh`
// columns exist, the rest of the tile is zero.
template <int DH, bool RG>
__device__ __forceinline__ void load_tile(uint32_t sbase, const bf16* g, int64_t ld, int rows, int dh) {
  constexpr int CH = DH / 8;
#pragma unroll
  for (int i = threadIdx.x; i < BT * CH; i += NT) {
    int r = i / CH, ch = i % CH;
    if constexpr (RG) {
      const bool ok = r < rows && ch * 8 < dh;
      cp_async16_or_zero(sbase + swz<DH>(r, ch * 8), ok ? g + (size_t)r * ld + ch * 8 : g, ok);
    } else {
      cp_async16(sbase + swz<DH>(r, ch * 8), g + (size_t)r * ld + ch * 8);
    }
  }
}

__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// A fragment (16 x 16) of a row-major [rows][DH] tile at (row0, k0)
template <int DH> __device__ __forceinline__ void load_a(uint32_t* a, uint32_t sbase, int row0, int k0) {
  int l = threadIdx.x & 31;
  ldsm4(a, sbase + swz<DH>(row0 + (l & 7) + ((l >> 3) & 1) * 8, k0 + (l >> 4) * 8));
}
// B fragments for two n-tiles (n0, n0+8) x k16 from a tile stored [n][k]: b[0],b[1] -> n0 ; b[2],b[3] -> n0+8
template <int DH> __device__ __forceinline__ void load_b_nk(uint32_t* b, uint32_t sbase, int n0, int k0) {
  int l = threadIdx.x & 31;
  ldsm4(b, sbase + swz<DH>(n0 + (l & 7) + (l >> 4) * 8, k0 + ((l >> 3) & 1) * 8));
}
// B fragments for two n-tiles (n0, n0+8) x k16 from a tile stored [k][n]
template <int DH> __device__ __forceinline__ void load_b_kn(uint32_t* b, uint32_t sbase, int k0, int n0) {
  int l = threadIdx.x & 31;
  ldsm4t(b, sbase + swz<DH>(k0 + (l & 7) + ((l >> 3) & 1) * 8, n0 + (l >> 4) * 8));
}

// acc[8][4] (16 x 64) += A(16 x DH from `a_tile` rows row0..) * B^T where the B tile is stored [64][DH]
template <int DH>
__device__ __forceinline__ void mma_a_smem_b_nk(float (*acc)[4], uint32_t a_tile, int row0, uint32_t b_tile) {
#pragma unroll
  for (int ks = 0; ks < DH / 16; ++ks) {
    uint32_t a[4];
    load_a<DH>(a, a_tile, row0, ks * 16);
#pragma unroll
    for (int np = 0; np < 4; ++np) {
      uint32_t b[4];
      load_b_nk<DH>(b, b_tile, np * 16, ks * 16);
      mma16816(acc[2 * np], a, b[0], b[1]);
      mma16816(acc[2 * np + 1], a, b[2], b[3]);
    }
  }
}
__device__ __forceinline__ void add2(float& a0, float& a1, float b0, float b1) {
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tadd.rn.f32x2 x, x, y;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}" : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}
// The same with the 16-deep products added up in fp32: the tensor core rounds each accumulation step towards zero, and
// the log-sum-exp, an fp32 result, shows it (relative error at T 500, width 128: 4.6e-8 as a chain of eight steps, 2.9e-8
// this way; 3.6e-8 in plain FMA).
template <int DH>
__device__ __forceinline__ void mma_a_smem_b_nk_rn(float (*acc)[4], uint32_t a_tile, int row0, uint32_t b_tile) {
#pragma unroll
  for (int ks = 0; ks < DH / 16; ++ks) {
    uint32_t a[4];
    load_a<DH>(a, a_tile, row0, ks * 16);
#pragma unroll
    for (int np = 0; np < 4; ++np) {
      uint32_t b[4];
      load_b_nk<DH>(b, b_tile, np * 16, ks * 16);
      if (ks == 0) {
        mma16816(acc[2 * np], a, b[0], b[1]);
        mma16816(acc[2 * np + 1], a, b[2], b[3]);
      } else {
        float p0[4] = {0.f, 0.f, 0.f, 0.f}, p1[4] = {0.f, 0.f, 0.f, 0.f};
        mma16816(p0, a, b[0], b[1]);
        mma16816(p1, a, b[2], b[3]);
        add2(acc[2 * np][0], acc[2 * np][1], p0[0], p0[1]); add2(acc[2 * np][2], acc[2 * np][3], p0[2], p0[3]);
        add2(acc[2 * np + 1][0], acc[2 * np + 1][1], p1[0], p1[1]); add2(acc[2 * np + 1][2], acc[2 * np + 1][3], p1[2], p1[3]);
      }
    }
  }
}
// what bf16 rounding leaves of two values, again as bf16
__device__ __forceinline__ uint32_t pack2_rest(float lo, float hi, uint32_t rounded) {
  return pack2(lo - __uint_as_float(rounded << 16), hi - __uint_as_float(rounded & 0xffff0000u));
}

// acc[DH/8][4] (16 x DH) += P(16 x 64, fp32 accumulator layout, converted to bf16) * B, B tile stored [64][DH].
// RG: P as the sum of two bf16 values; both products use the right operand's fragment while it is in registers.
template <int DH, bool RG>
__device__ __forceinline__ void mma_p_regs_b_kn(float (*acc)[4], const float (*p)[4], uint32_t b_tile) {
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    uint32_t a[4];
    a[0] = pack2(p[2 * ks][0], p[2 * ks][1]);
    a[1] = pack2(p[2 * ks][2], p[2 * ks][3]);
    a[2] = pack2(p[2 * ks + 1][0], p[2 * ks + 1][1]);
    a[3] = pack2(p[2 * ks + 1][2], p[2 * ks + 1][3]);
    uint32_t a2[4];
    if constexpr (RG) {
      a2[0] = pack2_rest(p[2 * ks][0], p[2 * ks][1], a[0]);
      a2[1] = pack2_rest(p[2 * ks][2], p[2 * ks][3], a[1]);
      a2[2] = pack2_rest(p[2 * ks + 1][0], p[2 * ks + 1][1], a[2]);
      a2[3] = pack2_rest(p[2 * ks + 1][2], p[2 * ks + 1][3], a[3]);
    }
#pragma unroll
    for (int np = 0; np < DH / 16; ++np) {
      uint32_t b[4];
      load_b_kn<DH>(b, b_tile, ks * 16, np * 16);
      mma16816(acc[2 * np], a, b[0], b[1]);
      mma16816(acc[2 * np + 1], a, b[2], b[3]);
      if constexpr (RG) {
        mma16816(acc[2 * np], a2, b[0], b[1]);
        mma16816(acc[2 * np + 1], a2, b[2], b[3]);
      }
    }
  }
}

template <int N> __device__ __forceinline__ void zero_acc(float (*a)[4]) {
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) a[i][j] = 0.f;
}

// A product with a 64-row tile multiplies the zero probability of a hidden pair with whatever the tile holds (0 x inf =
// NaN), and an inf with hi + lo where lo may be negative.  So in the RG forms a warp whose results are not all finite does its rows
// again, one by one in plain FMA over the visible pairs, which is how these shapes see values that are not finite
// everywhere else.  Finite rounds pay for a test of the results as they are stored.
// non-zero where one of two bf16 values is an inf or NaN (all exponent bits set)
__device__ __forceinline__ uint32_t not_finite(uint32_t two) { return ((two & 0x7f807f80u) + 0x00800080u) & 0x80008000u; }
__device__ __forceinline__ void redo_forward(const bf16* qkv, bf16* o, float* lse, int b, int h, int row, int end, int T, int H, int d, float* s) {
  const rows::Head<bf16> hd(qkv, b, h, T, H, d);
  for (; row < end; ++row)
    rows::forward_row<bf16>(hd, row, s, o + ((size_t)b * T + row) * d + (size_t)h * hd.dh, lse + ((size_t)b * H + h) * T + row);
}
__device__ __forceinline__ void redo_dq(const bf16* qkv, const bf16* d_o, const float* lse, const float* rowdot, bf16* dqkv, int b, int h, int row,
                                     int end, int T, int H, int d, float* s) {
  const rows::Head<bf16> hd(qkv, b, h, T, H, d);
  for (; row < end; ++row) {
    const size_t stat = ((size_t)b * H + h) * T + row;
    rows::dq_row<bf16>(hd, d_o + ((size_t)b * T + row) * d + (size_t)h * hd.dh, lse[stat], rowdot[stat], row, s,
                       dqkv + ((size_t)b * T + row) * hd.ld + (size_t)h * hd.dh);
  }
}
__device__ __forceinline__ void redo_dkv(const bf16* qkv, const bf16* d_o, const float* lse, const float* rowdot, bf16* dqkv, int b, int h, int row,
                                      int end, int T, int H, int d, float* s) {
  const rows::Head<bf16> hd(qkv, b, h, T, H, d);
  const size_t stat = ((size_t)b * H + h) * T;
  for (; row < end; ++row)
    rows::dkv_row<bf16>(hd, d_o + (size_t)b * T * d + (size_t)h * hd.dh, lse + stat, rowdot + stat, row, s,
                        dqkv + ((size_t)b * T + row) * hd.ld + d + (size_t)h * hd.dh);
}

// ------------------------------------------------------------------------------------------
// forward
// ------------------------------------------------------------------------------------------
// dh: head width (RG only; DH otherwise).  BLOCKS: registers for that many blocks per SM (launch_fwd chooses).
template <int DH, bool RG, int BLOCKS>
__global__ void __launch_bounds__(NT, BLOCKS) attn_fwd_tc_kernel(const bf16* __restrict__ qkv, bf16* __restrict__ o,
                                                         float* __restrict__ lse, int T, int H, int d, int dh,
                                                         float scale, float scale_log2) {
  overlap_sync();
  if (!RG) dh = DH;
  constexpr int TILE_BYTES = Sizes<DH>::TILE;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sQ = smem_u32(smem), sK0 = sQ + TILE_BYTES, sV0 = sQ + 3 * TILE_BYTES;
  const int qt = gridDim.x - 1 - blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t ld = 3 * (int64_t)d;
  const bf16* qbase = qkv + ((size_t)b * T + (size_t)qt * BT) * ld + (size_t)h * dh;
  const bf16* kbase = qkv + (size_t)b * T * ld + d + (size_t)h * dh;
  const bf16* vbase = kbase + d;
  load_tile<DH, RG>(sQ, qbase, ld, T - qt * BT, dh);
  load_tile<DH, RG>(sK0, kbase, ld, T, dh);
  load_tile<DH, RG>(sV0, vbase, ld, T, dh);
  cp_commit();
  float oacc[DH / 8][4];
  zero_acc<DH / 8>(oacc);
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  const int r0 = warp * 16 + g, r1 = r0 + 8;
  for (int j = 0; j <= qt; ++j) {
    const uint32_t sK = sK0 + (j & 1) * TILE_BYTES, sV = sV0 + (j & 1) * TILE_BYTES;
    if (j < qt) {
      load_tile<DH, RG>(sK0 + ((j + 1) & 1) * TILE_BYTES, kbase + (size_t)(j + 1) * BT * ld, ld, T - (j + 1) * BT, dh);
      load_tile<DH, RG>(sV0 + ((j + 1) & 1) * TILE_BYTES, vbase + (size_t)(j + 1) * BT * ld, ld, T - (j + 1) * BT, dh);
      cp_commit();
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    float s[8][4];
    zero_acc<8>(s);
    if constexpr (RG) mma_a_smem_b_nk_rn<DH>(s, sQ, warp * 16, sK);
    else mma_a_smem_b_nk<DH>(s, sQ, warp * 16, sK);
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int col = n * 8 + 2 * t + (e & 1);
        int row = (e < 2) ? r0 : r1;
        float v = RG ? s[n][e] : s[n][e] * scale_log2;      // RG: the maximum of the unscaled scores
        if (j == qt && col > row) v = -INFINITY;
        s[n][e] = v;
        if (e < 2) mx0 = fmaxf(mx0, v); else mx1 = fmaxf(mx1, v);
      }
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)); mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float nm0 = fmaxf(m0, mx0), nm1 = fmaxf(m1, mx1);   // finite: column 0 is never masked
    const float c0 = exp2f(RG ? (m0 - nm0) * scale_log2 : m0 - nm0), c1 = exp2f(RG ? (m1 - nm1) * scale_log2 : m1 - nm1);
    float ps0 = 0.f, ps1 = 0.f;
    const float k0 = -nm0 * scale_log2, k1 = -nm1 * scale_log2;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      if (RG) {                                                // one rounding per exponent
        s[n][0] = exp2f(fmaf(s[n][0], scale_log2, k0)); s[n][1] = exp2f(fmaf(s[n][1], scale_log2, k0));
        s[n][2] = exp2f(fmaf(s[n][2], scale_log2, k1)); s[n][3] = exp2f(fmaf(s[n][3], scale_log2, k1));
      } else {
        s[n][0] = exp2f(s[n][0] - nm0); s[n][1] = exp2f(s[n][1] - nm0);
        s[n][2] = exp2f(s[n][2] - nm1); s[n][3] = exp2f(s[n][3] - nm1);
      }
      ps0 += s[n][0] + s[n][1]; ps1 += s[n][2] + s[n][3];
    }
#pragma unroll
    for (int n = 0; n < DH / 8; ++n) { oacc[n][0] *= c0; oacc[n][1] *= c0; oacc[n][2] *= c1; oacc[n][3] *= c1; }
    l0 = l0 * c0 + ps0; l1 = l1 * c1 + ps1;
    m0 = nm0; m1 = nm1;
    mma_p_regs_b_kn<DH, RG>(oacc, s, sV);
    __syncthreads();
  }
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  const float i0 = 1.f / l0, i1 = 1.f / l1;
  bf16* o0 = o + ((size_t)b * T + (size_t)qt * BT + r0) * d + (size_t)h * dh;
  bf16* o1 = o + ((size_t)b * T + (size_t)qt * BT + r1) * d + (size_t)h * dh;
  const bool v0 = !RG || qt * BT + r0 < T, v1 = !RG || qt * BT + r1 < T;
  uint32_t bad = 0;
#pragma unroll
  for (int n = 0; n < DH / 8; ++n) {
    if (RG && n * 8 >= dh) break;
    const uint32_t w0 = pack2(oacc[n][0] * i0, oacc[n][1] * i0), w1 = pack2(oacc[n][2] * i1, oacc[n][3] * i1);
    if (v0) *reinterpret_cast<uint32_t*>(o0 + n * 8 + 2 * t) = w0;
    if (v1) *reinterpret_cast<uint32_t*>(o1 + n * 8 + 2 * t) = w1;
    if (RG) bad |= not_finite(w0) | not_finite(w1);
  }
  if (t == 0) {
    // RG: from the maximum as it entered the exponents, so that its rounding cancels
    float* lrow = lse + ((size_t)b * H + h) * T + (size_t)qt * BT;
    if (v0) lrow[r0] = RG ? fmaf(m0 * scale_log2, LN2, logf(l0)) : (m0 + log2f(l0)) * LN2;
    if (v1) lrow[r1] = RG ? fmaf(m1 * scale_log2, LN2, logf(l1)) : (m1 + log2f(l1)) * LN2;
  }
  if (RG && __any_sync(0xffffffffu, bad != 0)) {
    const int row = qt * BT + warp * 16;
    redo_forward(qkv, o, lse, b, h, row, min(row + 16, T), T, H, d, reinterpret_cast<float*>(smem) + warp * 2 * dh);
  }
}

// rowdot[b, h, i] = sum_c dO[i, c] O[i, c] over the head's DH columns; DH/8 lanes per row
template <int DH>
__global__ void attn_rowdot_tc_kernel(const bf16* __restrict__ o, const bf16* __restrict__ d_o, int nseq, int T, int H,
                                      int d, float* __restrict__ rowdot) {
  overlap_sync();
  constexpr int LPR = DH / 8;
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t rowhead = idx / LPR;
  int part = (int)(idx % LPR);
  if (rowhead >= (int64_t)nseq * T * H) return;
  int h = (int)(rowhead % H);
  int64_t row = rowhead / H;
  size_t off = (size_t)row * d + (size_t)h * DH + part * 8;
  uint4 a = *reinterpret_cast<const uint4*>(o + off), bb = *reinterpret_cast<const uint4*>(d_o + off);
  const bf16* ap = reinterpret_cast<const bf16*>(&a);
  const bf16* bp = reinterpret_cast<const bf16*>(&bb);
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) s = fmaf(__bfloat162float(ap[i]), __bfloat162float(bp[i]), s);
#pragma unroll
  for (int m = 1; m < LPR; m <<= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
  if (part == 0) {
    int bq = (int)(row / T), i = (int)(row % T);
    rowdot[((size_t)bq * H + h) * T + i] = s;
  }
}

// ------------------------------------------------------------------------------------------
// backward, dQ: one CTA per query tile, loops over key tiles j <= qt
// ------------------------------------------------------------------------------------------
// RG: the kernel also forms D[row] = sum(dO * O) of its own rows (two threads per row) and leaves it in
// `rowdot` for the dK/dV kernel, which runs second; otherwise a small kernel has put it there beforehand.
template <int DH, bool RG>
__global__ void __launch_bounds__(NT, RG ? (DH > 64 ? 1 : 3) : 0) attn_bwd_dq_tc_kernel(const bf16* __restrict__ qkv, const bf16* __restrict__ o,
                                                            const bf16* __restrict__ d_o, const float* __restrict__ lse,
                                                            float* __restrict__ rowdot, bf16* __restrict__ dqkv, int T,
                                                            int H, int d, int dh, float scale) {
  overlap_sync();
  if (!RG) dh = DH;
  constexpr int TILE_BYTES = Sizes<DH>::TILE;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sQ = smem_u32(smem), sdO = sQ + TILE_BYTES, sK0 = sQ + 2 * TILE_BYTES, sV0 = sQ + 4 * TILE_BYTES;
  const int qt = gridDim.x - 1 - blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t ld = 3 * (int64_t)d;
  const bf16* qbase = qkv + ((size_t)b * T + (size_t)qt * BT) * ld + (size_t)h * dh;
  const bf16* kbase = qkv + (size_t)b * T * ld + d + (size_t)h * dh;
  const bf16* vbase = kbase + d;
  const bf16* dobase = d_o + ((size_t)b * T + (size_t)qt * BT) * d + (size_t)h * dh;
  load_tile<DH, RG>(sQ, qbase, ld, T - qt * BT, dh);
  load_tile<DH, RG>(sdO, dobase, d, T - qt * BT, dh);
  load_tile<DH, RG>(sK0, kbase, ld, T, dh);
  load_tile<DH, RG>(sV0, vbase, ld, T, dh);
  cp_commit();
  const int r0 = warp * 16 + g, r1 = r0 + 8;
  const size_t stat = ((size_t)b * H + h) * T + (size_t)qt * BT;
  const bool v0 = !RG || qt * BT + r0 < T, v1 = !RG || qt * BT + r1 < T;
  const float L0 = v0 ? lse[stat + r0] * LOG2E : INFINITY, L1 = v1 ? lse[stat + r1] * LOG2E : INFINITY;
  float D0, D1;
  if constexpr (RG) {
    __shared__ float sD[BT];
    const int dr = threadIdx.x >> 1;
    float acc = 0.f;
    if (qt * BT + dr < T) {
      const size_t off = ((size_t)b * T + (size_t)qt * BT + dr) * d + (size_t)h * dh;
      for (int c = (threadIdx.x & 1) * 8; c < dh; c += 16) {
        const uint4 ov = *reinterpret_cast<const uint4*>(o + off + c), gv = *reinterpret_cast<const uint4*>(d_o + off + c);
        const uint32_t* ow = reinterpret_cast<const uint32_t*>(&ov);
        const uint32_t* gw = reinterpret_cast<const uint32_t*>(&gv);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc = fmaf(__uint_as_float(ow[i] << 16), __uint_as_float(gw[i] << 16), acc);
          acc = fmaf(__uint_as_float(ow[i] & 0xffff0000u), __uint_as_float(gw[i] & 0xffff0000u), acc);
        }
      }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if ((threadIdx.x & 1) == 0) {
      sD[dr] = acc;
      if (qt * BT + dr < T) rowdot[stat + dr] = acc;
    }
    __syncthreads();
    D0 = sD[r0]; D1 = sD[r1];
  } else {
    D0 = rowdot[stat + r0]; D1 = rowdot[stat + r1];
  }
  const float scale_log2 = scale * LOG2E;
  float dq[DH / 8][4];
  zero_acc<DH / 8>(dq);
  for (int j = 0; j <= qt; ++j) {
    const uint32_t sK = sK0 + (j & 1) * TILE_BYTES, sV = sV0 + (j & 1) * TILE_BYTES;
    if (j < qt) {
      load_tile<DH, RG>(sK0 + ((j + 1) & 1) * TILE_BYTES, kbase + (size_t)(j + 1) * BT * ld, ld, T - (j + 1) * BT, dh);
      load_tile<DH, RG>(sV0 + ((j + 1) & 1) * TILE_BYTES, vbase + (size_t)(j + 1) * BT * ld, ld, T - (j + 1) * BT, dh);
      cp_commit();
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    float s[8][4], dp[8][4];
    zero_acc<8>(s);
    mma_a_smem_b_nk<DH>(s, sQ, warp * 16, sK);       // S = Q K^T
    zero_acc<8>(dp);
    mma_a_smem_b_nk<DH>(dp, sdO, warp * 16, sV);     // dP = dO V^T
#pragma unroll
    for (int n = 0; n < 8; ++n) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int col = n * 8 + 2 * t + (e & 1);
        int row = (e < 2) ? r0 : r1;
        float p = exp2f(s[n][e] * scale_log2 - ((e < 2) ? L0 : L1));
        if (j == qt && col > row) p = 0.f;
        s[n][e] = p * (dp[n][e] - ((e < 2) ? D0 : D1));    // dS (without the 1/sqrt(dh) factor)
      }
    }
    mma_p_regs_b_kn<DH, RG>(dq, s, sK);                  // dQ += dS K
    __syncthreads();
  }
  bf16* q0 = dqkv + ((size_t)b * T + (size_t)qt * BT + r0) * ld + (size_t)h * dh;
  bf16* q1 = dqkv + ((size_t)b * T + (size_t)qt * BT + r1) * ld + (size_t)h * dh;
  uint32_t bad = 0;
#pragma unroll
  for (int n = 0; n < DH / 8; ++n) {
    if (RG && n * 8 >= dh) break;
    const uint32_t w0 = pack2(dq[n][0] * scale, dq[n][1] * scale), w1 = pack2(dq[n][2] * scale, dq[n][3] * scale);
    if (v0) *reinterpret_cast<uint32_t*>(q0 + n * 8 + 2 * t) = w0;
    if (v1) *reinterpret_cast<uint32_t*>(q1 + n * 8 + 2 * t) = w1;
    if (RG) bad |= not_finite(w0) | not_finite(w1);
  }
  if (RG && __any_sync(0xffffffffu, bad != 0)) {
    const int row = qt * BT + warp * 16;
    redo_dq(qkv, d_o, lse, rowdot, dqkv, b, h, row, min(row + 16, T), T, H, d, reinterpret_cast<float*>(smem) + warp * 2 * dh);
  }
}

// ------------------------------------------------------------------------------------------
// backward, dK and dV: one CTA per key tile, loops over query tiles i >= kt.
// Works on the transposed score tile S^T = K Q^T so that P^T and dS^T land in the register layout
// the next product needs as its left operand.
// ------------------------------------------------------------------------------------------
template <int DH, bool RG>
__global__ void __launch_bounds__(NT, RG ? (DH > 64 ? 1 : DH > 32 ? 2 : 3) : 0) attn_bwd_dkv_tc_kernel(const bf16* __restrict__ qkv, const bf16* __restrict__ d_o,
                                                             const float* __restrict__ lse, const float* __restrict__ rowdot,
                                                             bf16* __restrict__ dqkv, int T, int H, int d, int dh,
                                                             float scale) {
  overlap_sync();
  if (!RG) dh = DH;
  constexpr int TILE_BYTES = Sizes<DH>::TILE;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sK = smem_u32(smem), sV = sK + TILE_BYTES, sQ0 = sK + 2 * TILE_BYTES, sdO0 = sK + 4 * TILE_BYTES;
  float* sL = reinterpret_cast<float*>(smem + 6 * TILE_BYTES);     // [2][64] lse * log2e
  float* sD = sL + 2 * BT;                                         // [2][64] rowdot
  const int kt = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int nT = RG ? (T + BT - 1) / BT : T / BT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t ld = 3 * (int64_t)d;
  const bf16* qhead = qkv + (size_t)b * T * ld + (size_t)h * dh;
  const bf16* kbase = qhead + (size_t)kt * BT * ld + d;
  const bf16* dohead = d_o + (size_t)b * T * d + (size_t)h * dh;
  const size_t stat = ((size_t)b * H + h) * T;
  load_tile<DH, RG>(sK, kbase, ld, T - kt * BT, dh);
  load_tile<DH, RG>(sV, kbase + d, ld, T - kt * BT, dh);
  load_tile<DH, RG>(sQ0 + (kt & 1) * TILE_BYTES, qhead + (size_t)kt * BT * ld, ld, T - kt * BT, dh);
  load_tile<DH, RG>(sdO0 + (kt & 1) * TILE_BYTES, dohead + (size_t)kt * BT * d, d, T - kt * BT, dh);
  cp_commit();
  auto load_stats = [&](int i) {
    if (threadIdx.x < BT) {
      const int row = i * BT + threadIdx.x;
      const bool ok = !RG || row < T;               // a query past the end of the sequence: P = exp(-inf) = 0
      sL[(i & 1) * BT + threadIdx.x] = ok ? lse[stat + row] * LOG2E : INFINITY;
      sD[(i & 1) * BT + threadIdx.x] = ok ? rowdot[stat + row] : 0.f;
    }
  };
  load_stats(kt);
  const float scale_log2 = scale * LOG2E;
  const int r0 = warp * 16 + g, r1 = r0 + 8;       // key rows of this thread inside the tile
  float dk[DH / 8][4], dv[DH / 8][4];
  zero_acc<DH / 8>(dk); zero_acc<DH / 8>(dv);
  for (int i = kt; i < nT; ++i) {
    const uint32_t sQ = sQ0 + (i & 1) * TILE_BYTES, sdO = sdO0 + (i & 1) * TILE_BYTES;
    const float* Lq = sL + (i & 1) * BT;
    const float* Dq = sD + (i & 1) * BT;
    if (i + 1 < nT) {
      load_tile<DH, RG>(sQ0 + ((i + 1) & 1) * TILE_BYTES, qhead + (size_t)(i + 1) * BT * ld, ld, T - (i + 1) * BT, dh);
      load_tile<DH, RG>(sdO0 + ((i + 1) & 1) * TILE_BYTES, dohead + (size_t)(i + 1) * BT * d, d, T - (i + 1) * BT, dh);
      cp_commit();
      load_stats(i + 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    float st[8][4], dpt[8][4];
    zero_acc<8>(st);
    mma_a_smem_b_nk<DH>(st, sK, warp * 16, sQ);       // S^T = K Q^T   (rows: keys, columns: queries)
    zero_acc<8>(dpt);
    mma_a_smem_b_nk<DH>(dpt, sV, warp * 16, sdO);     // dP^T = V dO^T
#pragma unroll
    for (int n = 0; n < 8; ++n) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int qcol = n * 8 + 2 * t + (e & 1);
        int krow = (e < 2) ? r0 : r1;
        float p = exp2f(st[n][e] * scale_log2 - Lq[qcol]);
        if (i == kt && qcol < krow) p = 0.f;        // causal: query must not precede key
        float ds = p * (dpt[n][e] - Dq[qcol]);      // dS^T (without the 1/sqrt(dh) factor)
        if (RG && i == nT - 1 && i * BT + qcol >= T) p = ds = 0.f;   // also where a key's own values are not finite
        st[n][e] = p;
        dpt[n][e] = ds;
      }
    }
    mma_p_regs_b_kn<DH, RG>(dv, st, sdO);                 // dV += P^T dO
    mma_p_regs_b_kn<DH, RG>(dk, dpt, sQ);                 // dK += dS^T Q
    __syncthreads();
  }
  bf16* k0 = dqkv + ((size_t)b * T + (size_t)kt * BT + r0) * ld + d + (size_t)h * dh;
  bf16* k1 = dqkv + ((size_t)b * T + (size_t)kt * BT + r1) * ld + d + (size_t)h * dh;
  const bool v0 = !RG || kt * BT + r0 < T, v1 = !RG || kt * BT + r1 < T;
  uint32_t bad = 0;
#pragma unroll
  for (int n = 0; n < DH / 8; ++n) {
    if (RG && n * 8 >= dh) break;
    const uint32_t w0 = pack2(dk[n][0] * scale, dk[n][1] * scale), w1 = pack2(dk[n][2] * scale, dk[n][3] * scale);
    const uint32_t x0 = pack2(dv[n][0], dv[n][1]), x1 = pack2(dv[n][2], dv[n][3]);
    if (v0) {
      *reinterpret_cast<uint32_t*>(k0 + n * 8 + 2 * t) = w0;
      *reinterpret_cast<uint32_t*>(k0 + d + n * 8 + 2 * t) = x0;
    }
    if (v1) {
      *reinterpret_cast<uint32_t*>(k1 + n * 8 + 2 * t) = w1;
      *reinterpret_cast<uint32_t*>(k1 + d + n * 8 + 2 * t) = x1;
    }
    if (RG) bad |= not_finite(w0) | not_finite(w1) | not_finite(x0) | not_finite(x1);
  }
  if (RG && __any_sync(0xffffffffu, bad != 0)) {
    const int row = kt * BT + warp * 16;
    redo_dkv(qkv, d_o, lse, rowdot, dqkv, b, h, row, min(row + 16, T), T, H, d, reinterpret_cast<float*>(smem) + warp * 2 * dh);
  }
}

template <int DH, bool RG, int BLOCKS>
cudaError_t launch_fwd_blocks(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, cudaStream_t st) {
  static PerDeviceOnce once;                    // one per instantiation; attributes are per device
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(attn_fwd_tc_kernel<DH, RG, BLOCKS>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sizes<DH>::FWD);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  const int dh = d / H;
  dim3 grid((T + BT - 1) / BT, H, nseq);
  launch_overlapped(attn_fwd_tc_kernel<DH, RG, BLOCKS>, grid, NT, Sizes<DH>::FWD, st, (const bf16*)qkv, (bf16*)o, lse, T, H, d, dh,
                                                              1.0f / sqrtf((float)dh), (float)(1.4426950408889634 / sqrt((double)dh)));
  return cudaGetLastError();
}

// Registers for one block per SM at widths above 64: 4 sequences of 500, 8 heads of 128 33 -> 27.5 us against the
// compiler's own choice.  At width 64 for three, which beats four where a block walks several tiles (8 x 448, 8 heads 14.1
// against 16.2 us) or all blocks are resident at once.  Blocks of one to three tiles mostly wait for their loads: more than
// three per SM of them are better off with four at a time (64 x 64, 16 heads 10.5 -> 9.6 us; 24 x 192, 8 heads 10.7 -> 9.9).
template <int DH, bool RG>
cudaError_t launch_fwd(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, cudaStream_t st) {
  if constexpr (DH > 64) return launch_fwd_blocks<DH, RG, 1>(qkv, nseq, T, H, d, o, lse, st);
  else {
    if constexpr (DH == 64 && !RG) {
      if (T <= 3 * BT && (int64_t)(T / BT) * H * nseq > 3 * num_sms()) return launch_fwd_blocks<DH, RG, 4>(qkv, nseq, T, H, d, o, lse, st);
    }
    return launch_fwd_blocks<DH, RG, 3>(qkv, nseq, T, H, d, o, lse, st);
  }
}

template <int DH, bool RG>
cudaError_t launch_bwd(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H, int d,
                       void* dqkv, float* rowdot, int* status, cudaStream_t st) {
  static PerDeviceOnce once;
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(attn_bwd_dq_tc_kernel<DH, RG>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sizes<DH>::DQ);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attn_bwd_dkv_tc_kernel<DH, RG>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sizes<DH>::DKV);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  const int dh = d / H;
  const float scale = 1.0f / sqrtf((float)dh);
  if constexpr (!RG) {
    int64_t threads = (int64_t)nseq * T * H * (DH / 8);
    launch_overlapped(attn_rowdot_tc_kernel<DH>, (unsigned)((threads + 255) / 256), 256, 0, st, (const bf16*)o, (const bf16*)d_o, nseq, T, H, d, rowdot);
    if (DH == 128 && attention_bwd_t5_128_supported(DT_BF16, T, H, d))
      // dQ, dK, dV on the tcgen05 kernels (they read D[row] from `rowdot`, written just above)
      return attention_bwd_t5_128(qkv, lse, d_o, rowdot, nseq, T, H, d, dqkv, status, st);
  }
  dim3 grid((T + BT - 1) / BT, H, nseq);
  // Few blocks, but more than half as many as SMs: a kernel that starts early is placed where the one before it leaves
  // room, some SMs with three blocks (as many as are resident at once at width 64) and some with none, and then takes as
  // long as the fullest SM.  So these start in order.  Backward us, early -> in order, 64-row sequences of width 64: 16 with
  // 8 heads 11.7 -> 9.7, 24 13.6 -> 11.9, 10 10.1 -> 9.5, but 32 with 12 heads, the end of the range, 14.7 -> 15.7; width 128: 16 x 64, 8 heads
  // 16.8 -> 13.3, 2 x 960, 4 heads 95.8 -> 68.5, 8 x 192, 4 heads 23.7 -> 20.8, 8 heads 29.8 -> 30.6.  (Width 64 comes here at 64 rows
  // only.  The RG forms have no kernel in front of dQ that would upset its placement: 8 x 100 12.7 -> 13.3, so they start early.)
  const int64_t blocks = (int64_t)grid.x * H * nseq, sms = num_sms();
  const bool in_order = !RG && 2 * blocks > sms && blocks <= 3 * sms;
  if (in_order) break_chain();
  launch_overlapped(attn_bwd_dq_tc_kernel<DH, RG>, grid, NT, Sizes<DH>::DQ, st, (const bf16*)qkv, (const bf16*)o, (const bf16*)d_o, lse, rowdot,
                                                                (bf16*)dqkv, T, H, d, dh, scale);
  if (in_order) break_chain();
  launch_overlapped(attn_bwd_dkv_tc_kernel<DH, RG>, grid, NT, Sizes<DH>::DKV, st, (const bf16*)qkv, (const bf16*)d_o, lse, rowdot, (bf16*)dqkv,
                                                                  T, H, d, dh, scale);
  return cudaGetLastError();
}

}  // namespace

bool attention_tc_supported(int dt, int T, int H, int d) {
  return dt == DT_BF16 && H > 0 && d % H == 0 && (d / H == 64 || d / H == 128) && T >= BT && T % BT == 0;
}

// status: device word that receives a code when a bounded wait inside the tcgen05 kernels expires
// (nullptr: the library's own word, see library_status_word).
cudaError_t attention_fwd_tc(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status,
                             cudaStream_t st) {
  if (!attention_tc_supported(DT_BF16, T, H, d)) return cudaErrorInvalidValue;
  if (attention_fwd_t5_supported(DT_BF16, T, H, d)) return attention_fwd_t5(qkv, nseq, T, H, d, o, lse, status, st);
  return d / H == 64 ? launch_fwd<64, false>(qkv, nseq, T, H, d, o, lse, st)
                     : launch_fwd<128, false>(qkv, nseq, T, H, d, o, lse, st);
}

// The two tcgen05 forms of the backward pass at lengths that are multiples of 128.  attention_t5_bwd.cu needs about 0.83 of the
// time per pair of tiles, but shares out whole items: a CTA takes one tile of an item per round, of lengths that rotate.
// attention_t5_ragged.cu shares out single tiles, longest first, and runs both gradients at once where the tiles are few.
// Backward us, whole items -> single tiles: 2 sequences of 256, 16 heads 15.0 -> 9.5; 4 x 128 13.3 -> 8.1; 1 x 2048, 12 heads 70 -> 48;
// 8 x 1024, 8 heads 66 -> 53; 5 x 384, 12 heads 23.3 -> 20.3; 16 x 256, 12 heads 25.4 -> 24.4; 64 x 512, 16 heads 200 -> 233;
// 32 x 512, 12 heads 87 -> 99; 64 x 128, 16 heads 43.5 -> 46.5.
static bool w64_beats_whole_items(int nseq, int T, int H) {
  const int64_t sms = num_sms(), nq = T / 128, items = (int64_t)nseq * H, units = items * nq;
  if (2 * units <= sms) return true;
  if (nq > 64 || sms < nq) return true;                       // (not taken there)
  const int64_t per_round = (units < sms ? units : sms) / nq, rounds = (items + per_round - 1) / per_round;
  int64_t longest = rounds / nq * (nq * (nq + 1) / 2);        // steps of the CTA with the most: whole turns, then the longest tiles
  for (int64_t k = 0; k < rounds % nq; ++k) longest += nq - k;
  const int64_t steps = items * (nq * (nq + 1) / 2), even = (steps + sms - 1) / sms;
  return 12 * (even > nq ? even : nq) < 10 * longest;
}

cudaError_t attention_bwd_tc(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                             int d, void* dqkv, float* rowdot, int* status, cudaStream_t st) {
  if (!attention_tc_supported(DT_BF16, T, H, d)) return cudaErrorInvalidValue;
  if (d / H == 64 && T >= 128 && (T % 128 != 0 || w64_beats_whole_items(nseq, T, H)))
    return attention_bwd_t5_w64(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st);
  if (attention_t5_supported(DT_BF16, T, H, d))
    return attention_bwd_t5(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st);
  return d / H == 64 ? launch_bwd<64, false>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st)
                     : launch_bwd<128, false>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st);
}

// The shapes these kernels take.  The 16-byte copies need every head's first column of every row on a 16-byte boundary (d and the head width
// multiples of 8, aligned bases); sequences and heads are grid dimensions y and z.
bool attention_ragged_supported(int dt, int nseq, int T, int H, int d, const void* qkv, const void* o, const void* d_o,
                                const void* dqkv) {
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (dt != DT_BF16 || H < 1 || d % H != 0 || T < 1 || nseq < 1) return false;
  const int dh = d / H;
  // Many heads of a few rows: the tiles of 64 are padding, and a warp per row (attention_simt.cu) is faster.  us, forward /
  // backward, rows against tiles: 2048 heads of 1 x 64 4.8 / 11 against 19 / 53, of 5 x 64 15 / 47 against 19 / 53, of 6 x
  // 64 20 / 63 against 19 / 53; 8192 of 6 x 64 59 / 211 against 67 / 195; 128 of 1 x 64 4.2 / 10 against 3.6 / 9, 512 4.3 /
  // 10 against 7.1 / 18.
  const int64_t heads = (int64_t)nseq * H, sms = num_sms();
  if ((T <= 5 && heads > 2 * sms) || (T == 6 && !d_o && heads > 16 * sms)) return false;
  return dh % 8 == 0 && dh <= 128 && H <= 65535 && nseq <= 65535 && al16(qkv) && al16(o) && al16(d_o) && al16(dqkv);
}

cudaError_t attention_fwd_ragged(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status, cudaStream_t st) {
  // Tiles of 128 on tcgen05 against tiles of 64 here, us: 16 sequences of 777, 12 heads 114 -> 76; 32 x 288 44 -> 35.5; 5 x 333
  // 17.4 -> 13.8; 4 x 1000, 8 heads 41.5 -> 30.6; 64 x 70, 16 heads 26.8 -> 17.6; with fewer tiles than SMs the longer steps of one CTA
  // show: 1 x 1000, 8 heads 20.5 -> 28.2, 1 x 333 9.1 -> 12.9; up to 64 rows half a tile is padding: 64 x 50, 16 heads 11.1 -> 14.8.
  if (attention_ragged_t5_supported(nseq, T, H, d) && T > 64 && (int64_t)nseq * H * ((T + 127) / 128) > num_sms())
    return attention_fwd_ragged_t5(qkv, nseq, T, H, d, o, lse, status, st);
  switch ((d / H + 31) / 32) {
    case 1: return launch_fwd<32, true>(qkv, nseq, T, H, d, o, lse, st);
    case 2: return launch_fwd<64, true>(qkv, nseq, T, H, d, o, lse, st);
    case 3: return launch_fwd<96, true>(qkv, nseq, T, H, d, o, lse, st);
    case 4: return launch_fwd<128, true>(qkv, nseq, T, H, d, o, lse, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t attention_bwd_ragged(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                 int d, void* dqkv, float* rowdot, int* status, cudaStream_t st) {
  // Tiles of 128 on tcgen05 against tiles of 64 here, backward us: 16 sequences of 777, 12 heads 336 -> 120; 32 x 288 133 -> 62;
  // 5 x 333 44 -> 22; one of 150 with 4 heads 14.2 -> 10.1.  Up to 128 rows a head is one tile there, whose fixed part (set-up,
  // first loads) shows until there are about as many heads as SMs, unless both gradients fit one launch: 64 x 70, 16 heads 79 -> 42;
  // 16 x 100, 8 heads 16.2 -> 15.4; as two kernels 8 x 100 12.3 -> 13.5, 2 x 96, 12 heads 11.8 -> 13.3, which is where the line lies (in
  // one launch, as they would run there now, 9.1 and 8.8).  Up to 64 rows half of that tile is padding: 64 x 50, 16 heads 32.8 -> 37.3.
  if (attention_ragged_t5_supported(nseq, T, H, d) && (T > 128 || (T > 64 && (int64_t)nseq * H * 4 > 3 * (int64_t)num_sms())))
    return attention_bwd_ragged_t5(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, status, st);
  switch ((d / H + 31) / 32) {
    case 1: return launch_bwd<32, true>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, nullptr, st);
    case 2: return launch_bwd<64, true>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, nullptr, st);
    case 3: return launch_bwd<96, true>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, nullptr, st);
    case 4: return launch_bwd<128, true>(qkv, o, lse, d_o, nseq, T, H, d, dqkv, rowdot, nullptr, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace sl
