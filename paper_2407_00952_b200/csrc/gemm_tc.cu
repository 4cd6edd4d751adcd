// Linear-layer kernels for sm_100a: bf16 operands staged in shared memory by TMA, products issued
// with tcgen05.mma from one thread, fp32 accumulators in tensor memory, epilogue read back with
// tcgen05.ld.  Persistent CTAs walk the output tiles; the accumulator is double buffered in tensor
// memory so that the epilogue of one tile overlaps the products of the next.
//
//   Y[M,N] = epilogue( X[M,K] W[N,K]^T  +  Xe[M,Ke] We[N,Ke]^T )
//
// The second term is the rank-r LoRA path: it enters as extra blocks of the contraction, read
// through a second pair of tensor maps whose rows are selected by the row group (client) of the
// tile, so K clients with their own adapters share one pass over the frozen W.
//
// Three kernels (pick_kernel chooses):
//   gemm_tc_pair_kernel   CTA pairs (cluster of 2, tcgen05 cta_group::2): a pair owns a 256 x 256 (or 256 x 128)
//                         tile; each CTA stages its 128 rows of X and one half (128 rows) of the W
//                         tile, the leader issues 256 x 256 x 16 products that read both CTAs'
//                         shared memory and write both CTAs' tensor memory.  32 KB per CTA per
//                         64-deep block (131 FLOP per byte from L2), 6 stages.
//   gemm_tc_kernel<BN, EXACT>    one CTA per tile of 128 x BN (BN 256 / 128 / 64): narrow outputs (the
//                         rank-r down projections) and shapes the pair kernel does not take.
//   gemm_tc_split_kernel  few tiles: one 128 x 64 or 128 x 128 tile per cluster of 1-8 CTAs that share the
//                         contraction.
//
// Warp roles (320 threads): warp 0 = TMA producer, warp 1 = tensor-memory owner + MMA issuer,
// warps 2..9 = epilogue (a warp reads the 32 accumulator lanes its warp id modulo 4 selects; the
// two warps of a lane quarter take one half of the tile's columns each).
// The producer and issuer loops run as whole converged warps and one elected lane issues: in a loop that only one lane
// enters, the operands of every product go to uniform registers one by one, and a 64-deep block cost the issuing
// lane 500 cycles (330 in this form, next to 512 that the pair's four products take); the slack goes to the
// epilogue warps.  Isolated launches at M 32768, before -> after: output projection (bias + residual) 65.4 ->
// 60.2 us, fc1 (GELU) 240 -> 229.5, fc2 212 -> 204, fc2 backward (x GELU') 244 -> 230, QKV + LoRA 151 -> 137,
// plain backward products 193 -> 191 and 54.6 -> 53.1.
// Every wait on an mbarrier is bounded: when it expires the kernel records a code in `status`,
// stops issuing work, waits briefly for copies in flight, frees its tensor memory and returns.
#include "host_common.h"
#include "launch.cuh"
#include "tc_common.cuh"

namespace sl {
namespace {

using namespace tc;

constexpr int NUM_THREADS = 320;

// ------------------------------------------------------------------------------------------
// one CTA per tile
// ------------------------------------------------------------------------------------------
template <int BN> struct Cfg {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  // BN 64 is the HBM-bound rank-r down projection with more tiles than SMs (fewer: gemm_tc_split_kernel): two
  // CTAs per SM (three stages each) keep every SM streaming when the tiles do not fill whole waves of one CTA per SM.
  static constexpr int CTAS_PER_SM = BN == 64 ? 2 : 1;
  static constexpr int STAGES = BN == 64 ? 3 : ((196608 / STAGE_BYTES) > 8 ? 8 : (196608 / STAGE_BYTES));
  static constexpr int TMEM_COLS = 2 * BN < 32 ? 32 : 2 * BN;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_STAGE_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;
  static constexpr uint32_t IDESC = make_idesc(BM, BN);
};

template <int BN, bool EXACT>
__global__ void __launch_bounds__(NUM_THREADS, Cfg<BN>::CTAS_PER_SM)
gemm_tc_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW,
               const __grid_constant__ CUtensorMap mapXe, const __grid_constant__ CUtensorMap mapWe,
               const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapZ, TcParams p) {
  using C = Cfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t epi_base = base + C::STAGES * C::STAGE_BYTES;     // output staging of the epilogue warps
  const uint32_t bar_base = epi_base + EPI_STAGE_BYTES;
  // barrier slots: full[STAGES], empty[STAGES], tmem_full[2], tmem_empty[2]
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::STAGES + s); };
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * C::STAGES + a); };
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * C::STAGES + 2 + a); };
  uint8_t* tail = base_ptr + C::STAGES * C::STAGE_BYTES + EPI_STAGE_BYTES + 8 * (2 * C::STAGES + 4);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 8); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)C::TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  overlap_sync();

  const int num_tiles = p.tiles_m * p.tiles_n;
  const int kb_total = p.num_kb + p.ext_blocks;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const bool leader = elect_one();
    int stage = 0; uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      int tm, tn; tile_coords(tile, p.tiles_m, p.tiles_n, tm, tn);
      const int m0 = tm * BM, n0 = tn * BN;
      const int g = p.rows_per_group > 0 ? m0 / p.rows_per_group : 0;
      const int w_row = g * p.w_group_rows + n0;
      const int we_row = g * p.we_group_rows + n0;
      for (int kb = 0; kb < kb_total; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, abort_flag, p.status, 1)) { ok = false; break; }
        const uint32_t sa = base + stage * C::STAGE_BYTES, sb = sa + C::A_BYTES;
        if (leader) {
          mbar_expect_tx(full_bar(stage), C::STAGE_BYTES);
          if (kb < p.num_kb) {
            const int kc = (kb < p.gap_kb_begin ? kb : kb + p.gap_kb) * BK;
            tma_load_2d(sa, &mapX, full_bar(stage), kc, m0);
            tma_load_2d(sb, &mapW, full_bar(stage), kc, w_row);
          } else {
            const int e = kb - p.num_kb;
            tma_load_2d(sa, &mapXe, full_bar(stage), e * BK, m0);
            tma_load_2d(sb, &mapWe, full_bar(stage), e * BK, we_row);
          }
        }
        __syncwarp();
        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool leader = elect_one();
    int stage = 0; uint32_t phase = 0;
    int as = 0; uint32_t aphase = 0;
    bool ok = true;
    const uint32_t a_lo0 = desc_lo(base);
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      if (!mbar_wait_warp(tempty_bar(as), aphase ^ 1u, abort_flag, p.status, 2)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + (uint32_t)(as * BN);
      // main contraction: four products per block, issued back to back (advancing 16 elements
      // along K inside the swizzled row = +32 bytes = +2 in descriptor units)
      for (int kb = 0; kb < p.num_kb; ++kb) {
        if (!mbar_wait_warp(full_bar(stage), phase, abort_flag, p.status, 3)) { ok = false; break; }
        const uint32_t alo = a_lo0 + (uint32_t)stage * (uint32_t)(C::STAGE_BYTES >> 4);
        const uint32_t blo = alo + (uint32_t)(C::A_BYTES >> 4);
        if (leader) {
          tc_mma_lo(d_tmem, alo, blo, C::IDESC, (uint32_t)kb);
          tc_mma_lo_acc(d_tmem, alo + 2, blo + 2, C::IDESC);
          tc_mma_lo_acc(d_tmem, alo + 4, blo + 4, C::IDESC);
          tc_mma_lo_acc(d_tmem, alo + 6, blo + 6, C::IDESC);
          tc_commit(empty_bar(stage));          // frees the stage once these products have read it
        }
        __syncwarp();
        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      }
      // rank-r extension: the last block may hold fewer than four products
      for (int kb = p.num_kb; kb < kb_total && ok; ++kb) {
        if (!mbar_wait_warp(full_bar(stage), phase, abort_flag, p.status, 3)) { ok = false; break; }
        const uint32_t alo = a_lo0 + (uint32_t)stage * (uint32_t)(C::STAGE_BYTES >> 4);
        const uint32_t blo = alo + (uint32_t)(C::A_BYTES >> 4);
        const int nmma = kb == kb_total - 1 ? p.ext_last_mmas : BK / UMMA_K;
        if (leader) {
#pragma unroll 1
          for (int k = 0; k < nmma; ++k) tc_mma_lo_acc(d_tmem, alo + 2 * k, blo + 2 * k, C::IDESC);
          tc_commit(empty_bar(stage));
        }
        __syncwarp();
        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      if (leader) tc_commit(tfull_bar(as));     // accumulator complete
      __syncwarp();
      if (++as == 2) { as = 0; aphase ^= 1u; }
    }
  } else {
    // ---------------- epilogue ----------------
    const int q = warp & 3;                     // lanes [32q, 32q+32) of tensor memory
    const int half = (warp - 2) >> 2;           // two warps share a lane quarter and split the columns
    const int c_begin = half * (BN / 2), c_end = c_begin + BN / 2;
    int as = 0; uint32_t aphase = 0;
    const bool tanh_form = p.gelu_tanh != 0;
    const uint32_t stage = epi_base + (uint32_t)(warp - 2) * 4096u;   // this warp's two staging buffers
    EpiState est;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      int tm, tn; tile_coords(tile, p.tiles_m, p.tiles_n, tm, tn);
      const int m_warp0 = tm * BM + q * 32;
      const int n0 = tn * BN;
      int m_next = -1, n_next = 0;
      if (tile + (int)gridDim.x < num_tiles) {
        int tm2, tn2; tile_coords(tile + gridDim.x, p.tiles_m, p.tiles_n, tm2, tn2);
        m_next = tm2 * BM + q * 32; n_next = tn2 * BN + c_begin;
      }
      if (!mbar_wait(tfull_bar(as), aphase, abort_flag, p.status, 4)) { ok = false; break; }
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(as * BN);
      if (m_warp0 < p.M) epilogue_tile<EXACT>(p, t_row, m_warp0, lane, n0, c_begin, c_end, m_next, n_next, tanh_form, stage, est, &mapY, &mapZ);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty_bar(as));
      if (++as == 2) { as = 0; aphase ^= 1u; }
    }
    epilogue_drain(lane);
  }

  // ---------------- teardown ----------------
  __syncwarp();
  if (*abort_flag) {
    // give copies and products already in flight time to land before shared / tensor memory go away
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)C::TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------------------------
// CTA pairs
// ------------------------------------------------------------------------------------------
// One kernel per epilogue: with two in one kernel, what one gains from a change of the code the other loses (2-4 %).
// NEED_R: the epilogue has a second operand R (residual, or the pre-activation for GELU').  Its
// [128 x 256] block per CTA tile is brought into shared memory by the producer warp with TMA about
// one tile ahead of its use, so the epilogue never waits on a global load; the room comes from a
// shorter operand ring (4 stages instead of 6).
// BN_: tile columns of the pair.  256, or 128 where tiles of 256 would leave SMs idle.
template <bool NEED_R, int BN_> struct PairCfg {
  static constexpr int BN = BN_;
  static constexpr int A_BYTES = BM * BK * 2;          // this CTA's 128 rows of X
  static constexpr int B_BYTES = (BN / 2) * BK * 2;    // this CTA's half of the W tile
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = BN == 256 ? (NEED_R ? 4 : 6) : (NEED_R ? 6 : 8);
  static constexpr int R_BYTES = NEED_R ? BM * BN * 2 : 0;
  static constexpr int TMEM_COLS = 2 * BN;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + R_BYTES + EPI_STAGE_BYTES + 1024 + 256;
  static constexpr uint32_t IDESC = make_idesc(2 * BM, BN);
};

template <int EPI, bool EXACT, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
gemm_tc_pair_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW,
                    const __grid_constant__ CUtensorMap mapXe, const __grid_constant__ CUtensorMap mapWe,
                    const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapZ,
                    const __grid_constant__ CUtensorMap mapR, TcParams p) {
  constexpr bool NEED_R = EPI == EPI_BIAS_RESID || EPI == EPI_MUL_GELUGRAD;
  using C = PairCfg<NEED_R, BN>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t r_base = base + C::STAGES * C::STAGE_BYTES;       // second epilogue operand of the current tile
  const uint32_t epi_base = r_base + C::R_BYTES;                   // output staging of the epilogue warps
  const uint32_t bar_base = epi_base + EPI_STAGE_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };                         // used in the leader
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::STAGES + s); };          // one per CTA
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * C::STAGES + a); };      // one per CTA
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * C::STAGES + 2 + a); }; // used in the leader
  const uint32_t rfull_bar = bar_base + 8u * (2 * C::STAGES + 4), rempty_bar = rfull_bar + 8u;   // one per CTA
  uint8_t* tail = base_ptr + C::STAGES * C::STAGE_BYTES + C::R_BYTES + EPI_STAGE_BYTES + 8 * (2 * C::STAGES + 6);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();           // 0 = leader of the pair
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 16); }
    mbar_init(rfull_bar, 1); mbar_init(rempty_bar, 8);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    // both CTAs of the pair allocate together
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)C::TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                // the partner's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  overlap_sync();

  const int num_tiles = p.tiles_m * p.tiles_n;       // tiles of 256 x BN
  const int kb_total = p.num_kb + p.ext_blocks;

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    const bool leader = elect_one();
    int stage = 0; uint32_t phase = 0;
    int tcount = 0;                                // tiles this CTA has started
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
      int tm, tn; tile_coords(tile, p.tiles_m, p.tiles_n, tm, tn);
      const int m0 = tm * 2 * BM + (int)rank * BM, n0 = tn * BN + (int)rank * (BN / 2);
      const int g = p.rows_per_group > 0 ? m0 / p.rows_per_group : 0;
      const int w_row = g * p.w_group_rows + n0;
      const int we_row = g * p.we_group_rows + n0;
      // R block of this tile: issued as soon as the epilogue has released the buffer (checked between operand
      // blocks so that the operand ring never waits for it; test_wait: a try_wait here suspends the warp, which
      // cost the tiles with a second operand 20 %)
      bool r_pending = NEED_R;
      auto issue_r = [&](bool blocking) -> bool {
        if (!r_pending) return true;
        const uint32_t par = ((uint32_t)tcount & 1u) ^ 1u;
        if (blocking) { if (!mbar_wait_warp(rempty_bar, par, abort_flag, p.status, 15)) return false; }
        else if (!__all_sync(0xffffffffu, mbar_test(rempty_bar, par))) return true;
        if (leader) {
          mbar_expect_tx(rfull_bar, C::R_BYTES);
#pragma unroll
          for (int j = 0; j < BN / BK; ++j)
            tma_load_2d(r_base + j * (BM * BK * 2), &mapR, rfull_bar, tn * BN + j * BK, m0);
        }
        __syncwarp();
        r_pending = false;
        return true;
      };
      for (int kb = 0; kb < kb_total; ++kb) {
        issue_r(false);
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, abort_flag, p.status, 11)) { ok = false; break; }
        const uint32_t leader_full = map_to_cta(full_bar(stage), 0);
        const uint32_t sa = base + stage * C::STAGE_BYTES, sb = sa + C::A_BYTES;
        if (leader) {
          // the first CTA's barrier collects the bytes of both CTAs' copies
          if (rank == 0) mbar_expect_tx(full_bar(stage), 2 * C::STAGE_BYTES);
          if (kb < p.num_kb) {
            tma_load_2d_pair(sa, &mapX, leader_full, kb * BK, m0);
            tma_load_2d_pair(sb, &mapW, leader_full, kb * BK, w_row);
          } else {
            const int e = kb - p.num_kb;
            tma_load_2d_pair(sa, &mapXe, leader_full, e * BK, m0);
            tma_load_2d_pair(sb, &mapWe, leader_full, e * BK, we_row);
          }
        }
        __syncwarp();
        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      }
      if (ok && !issue_r(true)) ok = false;
      ++tcount;
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (first CTA of the pair only) ----------------
    if (rank == 0) {
      const bool leader = elect_one();
      int stage = 0; uint32_t phase = 0;
      int as = 0; uint32_t aphase = 0;
      bool ok = true;
      const uint32_t a_lo0 = desc_lo(base);
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        if (!mbar_wait_warp(tempty_bar(as), aphase ^ 1u, abort_flag, p.status, 12)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(as * BN);
        for (int kb = 0; kb < p.num_kb; ++kb) {    // four products per block, issued back to back
          if (!mbar_wait_warp(full_bar(stage), phase, abort_flag, p.status, 13)) { ok = false; break; }
          const uint32_t alo = a_lo0 + (uint32_t)stage * (uint32_t)(C::STAGE_BYTES >> 4);
          const uint32_t blo = alo + (uint32_t)(C::A_BYTES >> 4);
          if (leader) {
            tc_mma_pair_lo(d_tmem, alo, blo, C::IDESC, (uint32_t)kb);
            tc_mma_pair_lo_acc(d_tmem, alo + 2, blo + 2, C::IDESC);
            tc_mma_pair_lo_acc(d_tmem, alo + 4, blo + 4, C::IDESC);
            tc_mma_pair_lo_acc(d_tmem, alo + 6, blo + 6, C::IDESC);
            tc_commit_pair(empty_bar(stage), 3);   // frees the stage in both CTAs
          }
          __syncwarp();
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
        for (int kb = p.num_kb; kb < kb_total && ok; ++kb) {   // rank-r extension
          if (!mbar_wait_warp(full_bar(stage), phase, abort_flag, p.status, 13)) { ok = false; break; }
          const uint32_t alo = a_lo0 + (uint32_t)stage * (uint32_t)(C::STAGE_BYTES >> 4);
          const uint32_t blo = alo + (uint32_t)(C::A_BYTES >> 4);
          const int nmma = kb == kb_total - 1 ? p.ext_last_mmas : BK / UMMA_K;
          if (leader) {
#pragma unroll 1
            for (int k = 0; k < nmma; ++k) tc_mma_pair_lo_acc(d_tmem, alo + 2 * k, blo + 2 * k, C::IDESC);
            tc_commit_pair(empty_bar(stage), 3);
          }
          __syncwarp();
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (leader) tc_commit_pair(tfull_bar(as), 3);          // accumulator halves complete in both CTAs
        __syncwarp();
        if (++as == 2) { as = 0; aphase ^= 1u; }
      }
    }
  } else {
    // ---------------- epilogue (both CTAs, own 128 rows) ----------------
    const int q = warp & 3;
    const int half = (warp - 2) >> 2;
    const int c_begin = half * (BN / 2), c_end = c_begin + BN / 2;
    int as = 0; uint32_t aphase = 0;
    const bool tanh_form = p.gelu_tanh != 0;
    const uint32_t stage = epi_base + (uint32_t)(warp - 2) * 4096u;   // this warp's two staging buffers
    int buf = 0, tcount = 0;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += npairs, ++tcount) {
      int tm, tn; tile_coords(tile, p.tiles_m, p.tiles_n, tm, tn);
      const int m_warp0 = tm * 2 * BM + (int)rank * BM + q * 32;
      const int n0 = tn * BN;
      uint4 bfirst[4];
      load_bias_chunk(p, n0 + c_begin, bfirst);       // in flight while the accumulator is awaited
      if (!mbar_wait(tfull_bar(as), aphase, abort_flag, p.status, 14)) { ok = false; break; }
      if (NEED_R && !mbar_wait(rfull_bar, (uint32_t)tcount & 1u, abort_flag, p.status, 16)) { ok = false; break; }
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(as * BN);
      if (m_warp0 < p.M)
        epilogue_tile_smem_r<EXACT, EPI>(p, t_row, m_warp0, lane, n0, c_begin, c_end, tanh_form, stage, buf, &mapY, &mapZ,
                                    NEED_R ? r_base : 0u, q * 32 + lane, bfirst);
      if (NEED_R) { __syncwarp(); if (lane == 0) mbar_arrive(rempty_bar); }   // 8 warps release the R buffer
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_cta(tempty_bar(as), 0));   // 16 arrivals free the stage
      if (++as == 2) { as = 0; aphase ^= 1u; }
    }
    epilogue_drain(lane);
  }

  // ---------------- teardown ----------------
  __syncwarp();
  if (*abort_flag) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                // neither CTA leaves while its partner may still touch it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)C::TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------------------------
// few tiles: one tile per cluster, the contraction split over its CTAs
// ------------------------------------------------------------------------------------------
// S CTAs (a cluster) share one 128 x BN tile: each contracts its range of 64-deep blocks into its own tensor
// memory, then every 32 x 32 piece of the tile is added up by one of them (piece u by CTA u % S), which the
// others have sent their fp32 partial sums to through distributed shared memory, and leaves through that CTA's
// epilogue.  The sums are added in rank order: results do not depend on scheduling.
// What bounds it: the few tiles of a layer over few tokens are a chain (launch, set-up, first loads, blocks one by
// one, epilogue) rather than traffic, so the chain of blocks is cut into S.
template <int BN, int S, int STAGES_> struct SplitCfg {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = STAGES_;
  static constexpr int PIECES = BN / 64;                             // pieces per epilogue warp
  static constexpr int RECV_BYTES = (8 * PIECES / S) * (S - 1) * 4096;
  // the output staging of the epilogue takes the operand ring, which is idle once the accumulator is complete
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + RECV_BYTES + 1024 + 256;
  static constexpr uint32_t IDESC = make_idesc(BM, BN);
  static_assert(STAGES * STAGE_BYTES >= EPI_STAGE_BYTES && (8 * PIECES) % S == 0, "");
};

template <int BN, int S, int STAGES_, bool EXACT>
__global__ void __launch_bounds__(NUM_THREADS, 1)
gemm_tc_split_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW,
                     const __grid_constant__ CUtensorMap mapXe, const __grid_constant__ CUtensorMap mapWe,
                     const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapZ, TcParams p) {
  using C = SplitCfg<BN, S, STAGES_>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t recv_base = base + C::STAGES * C::STAGE_BYTES;
  const uint32_t bar_base = recv_base + C::RECV_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::STAGES + s); };
  const uint32_t tfull_bar = bar_base + 8u * (2 * C::STAGES);
  uint8_t* tail = base_ptr + C::STAGES * C::STAGE_BYTES + C::RECV_BYTES + 8 * (2 * C::STAGES + 1);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = S > 1 ? (int)cluster_ctarank() : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(tfull_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)BN) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (S > 1) cluster_arrive();                       // awaited before the first store to another CTA
  const uint32_t tmem_base = *tmem_slot;
  overlap_sync();

  const int kb_total = p.num_kb + p.ext_blocks;
  const int kb0 = (int)((long long)kb_total * rank / S), kb1 = (int)((long long)kb_total * (rank + 1) / S);
  int tm, tn;
  tile_coords((int)blockIdx.x / S, p.tiles_m, p.tiles_n, tm, tn);
  const int m0 = tm * BM, n0 = tn * BN;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const bool leader = elect_one();
    const int g = p.rows_per_group > 0 ? m0 / p.rows_per_group : 0;
    const int w_row = g * p.w_group_rows + n0;
    const int we_row = g * p.we_group_rows + n0;
    int stage = 0; uint32_t phase = 0;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, abort_flag, p.status, 51)) break;
      const uint32_t sa = base + stage * C::STAGE_BYTES, sb = sa + C::A_BYTES;
      if (leader) {
        mbar_expect_tx(full_bar(stage), C::STAGE_BYTES);
        if (kb < p.num_kb) {
          const int kc = (kb < p.gap_kb_begin ? kb : kb + p.gap_kb) * BK;
          tma_load_2d(sb, &mapW, full_bar(stage), kc, w_row);
          tma_load_2d(sa, &mapX, full_bar(stage), kc, m0);
        } else {
          const int e = kb - p.num_kb;
          tma_load_2d(sb, &mapWe, full_bar(stage), e * BK, we_row);
          tma_load_2d(sa, &mapXe, full_bar(stage), e * BK, m0);
        }
      }
      __syncwarp();
      if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool leader = elect_one();
    int stage = 0; uint32_t phase = 0;
    bool ok = true;
    const uint32_t a_lo0 = desc_lo(base);
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait_warp(full_bar(stage), phase, abort_flag, p.status, 53)) { ok = false; break; }
      const uint32_t alo = a_lo0 + (uint32_t)stage * (uint32_t)(C::STAGE_BYTES >> 4);
      const uint32_t blo = alo + (uint32_t)(C::A_BYTES >> 4);
      const int nmma = kb == kb_total - 1 && p.ext_blocks > 0 ? p.ext_last_mmas : BK / UMMA_K;
      if (leader) {
        tc_mma_lo(tmem_base, alo, blo, C::IDESC, (uint32_t)(kb - kb0));
        if (nmma == 4) {
          tc_mma_lo_acc(tmem_base, alo + 2, blo + 2, C::IDESC);
          tc_mma_lo_acc(tmem_base, alo + 4, blo + 4, C::IDESC);
          tc_mma_lo_acc(tmem_base, alo + 6, blo + 6, C::IDESC);
        } else {
          for (int k = 1; k < nmma; ++k) tc_mma_lo_acc(tmem_base, alo + 2 * k, blo + 2 * k, C::IDESC);
        }
        tc_commit(empty_bar(stage));
      }
      __syncwarp();
      if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
    }
    if (ok && leader) tc_commit(tfull_bar);
  }
  __syncwarp();

  // ---------------- epilogue ----------------
  const int ew = warp - 2;                           // epilogue warp 0..7
  const int q = warp & 3, half = ew >> 2;
  const int m_warp0 = m0 + q * 32;
  const bool need_r = p.epi == EPI_BIAS_RESID || p.epi == EPI_MUL_GELUGRAD;
  const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
  uint4 bcur[C::PIECES][4], rcur[C::PIECES][4];
  bool ok = false;
  // piece j of a warp: columns n0 + half * BN/2 + 32 j; pieces are numbered u = PIECES * (4 half + q) + j
  auto piece = [&](int j) { return C::PIECES * (half * 4 + q) + j; };
  auto column = [&](int j) { return half * (BN / 2) + 32 * j; };
  if (warp >= 2) {
#pragma unroll
    for (int j = 0; j < C::PIECES; ++j) {            // in flight while the accumulator is awaited
      if (S > 1 && piece(j) % S != rank) continue;
      load_bias_chunk(p, n0 + column(j), bcur[j]);
      if (need_r) load_r_chunk(p, m_warp0 + lane, n0 + column(j), rcur[j]);
    }
    ok = mbar_wait(tfull_bar, 0u, abort_flag, p.status, 54);
    tc_fence_after();
  }
  if constexpr (S > 1) {
    cluster_wait();                                  // every CTA of the cluster runs: its shared memory exists
    if (warp >= 2 && ok) {
#pragma unroll
      for (int j = 0; j < C::PIECES; ++j) {
        const int u = piece(j), owner = u % S;
        if (owner == rank || n0 + column(j) >= p.N || m_warp0 >= p.M) continue;
        float v[32];
        tc_ld32(t_row + (uint32_t)column(j), v);
        tc_wait_ld();
        // slot: the owner's (u / S)-th piece, sender number (this rank among the others)
        const int sender = rank < owner ? rank : rank - 1;
        const uint32_t dst = map_to_cta(recv_base + (uint32_t)(((u / S) * (S - 1) + sender) * 4096 + lane * 16), (uint32_t)owner);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(i * 512)), "f"(v[4 * i]),
                       "f"(v[4 * i + 1]), "f"(v[4 * i + 2]), "f"(v[4 * i + 3]) : "memory");
      }
    }
    __syncwarp();
    cluster_sync_all();
  }
  if (warp >= 2) {
    if (ok) {
      const bool tanh_form = p.gelu_tanh != 0;
      const uint32_t stage = base + (uint32_t)ew * 4096u;   // this warp's two staging buffers, in the idle operand ring
      int buf = 0;
#pragma unroll
      for (int j = 0; j < C::PIECES; ++j) {
        const int u = piece(j), n = n0 + column(j);
        if ((S > 1 && u % S != rank) || n >= p.N || m_warp0 >= p.M) continue;
        float v[32];
        tc_ld32(t_row + (uint32_t)column(j), v);
        tc_wait_ld();
        if constexpr (S > 1) {
          // partial sums in rank order: the contribution of rank 0 first
          float acc[32];
#pragma unroll
          for (int r = 0; r < S; ++r) {
            if (r == rank) {
#pragma unroll
              for (int i = 0; i < 32; ++i) acc[i] = r == 0 ? v[i] : acc[i] + v[i];
            } else {
              const int sender = r < rank ? r : r - 1;
              const uint32_t src = recv_base + (uint32_t)(((u / S) * (S - 1) + sender) * 4096 + lane * 16);
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                float x0, x1, x2, x3;
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x0), "=f"(x1), "=f"(x2), "=f"(x3) : "r"(src + (uint32_t)(i * 512)) : "memory");
                acc[4 * i] = r == 0 ? x0 : acc[4 * i] + x0;
                acc[4 * i + 1] = r == 0 ? x1 : acc[4 * i + 1] + x1;
                acc[4 * i + 2] = r == 0 ? x2 : acc[4 * i + 2] + x2;
                acc[4 * i + 3] = r == 0 ? x3 : acc[4 * i + 3] + x3;
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = acc[i];
        }
        epilogue_chunk<EXACT, -1>(p, v, bcur[j], rcur[j], n, tanh_form, stage, buf, &mapY, &mapZ, m_warp0, lane);
      }
    }
    epilogue_drain(lane);
  }

  // ---------------- teardown ----------------
  __syncwarp();
  if (*abort_flag) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)BN) : "memory");
  }
}

// ---- host side -----------------------------------------------------------------------------
// CTA pairs that can be resident at once, per device (0: pair kernel unavailable there)
int g_max_pairs[MAX_DEVICES] = {};
int g_max_split_clusters[MAX_DEVICES][3] = {};      // of 2, 4 and 8 CTAs
PerDeviceOnce g_pair_once;

// 2-D bf16 tensor [rows, cols] with leading dimension ld (elements); box = 64 columns x box_rows rows.
bool make_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows) {
  return cached_map_2d(m, ptr, rows, cols, ld, (uint32_t)BK, box_rows, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

// Output map: bf16 [rows, cols], box = 32 columns x 32 rows, 64-byte swizzle (the epilogue's staging layout).
bool make_out_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld) {
  return cached_map_2d(m, ptr, rows, cols, ld, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

int max_pairs() {
  const int dev = current_device();
  return dev < 0 ? 0 : g_max_pairs[dev];
}
// Clusters of S CTAs of the split kernel that can be resident at once (0: unknown).  Fewer than SMs / S, because a cluster
// stays within one group of SMs: 74, 33 and 15 of 2, 4 and 8 CTAs on 148 SMs.  One tile too many is a second round:
// 36 tiles (384 x 768 -> 768) as clusters of four 10.6 us, as clusters of two 6.2; 16 (2048 x 4096 -> 64) of eight
// 13.3 us, of four 8.4.
int max_split_clusters(int S) {
  const int dev = current_device();
  return dev < 0 ? 0 : g_max_split_clusters[dev][S == 2 ? 0 : S == 4 ? 1 : 2];
}

int pick_bn(const GemmArgs& a) {
  if (a.N % 256 == 0) return 256;
  if (a.N <= 64) return 64;
  if (a.N <= 128) return 128;
  return 256;
}

bool pair_ok(const GemmArgs& a) {
  if (max_pairs() < 1 || a.k_gap_len > 0) return false;
  return a.M > BM && a.N >= 256 && a.rows_per_group % (2 * BM) == 0;     // rows_per_group 0: one group, any M
}

// Which kernel takes a layer: the one with the least estimated time, from the number of rounds its CTAs need on the
// chip, the 64-deep blocks per CTA and each kernel's measured constants (ns; CUDA graph replays over operands that
// exceed L2, M 128-8192, K 768-4096, N 64-4096): a fixed part (launch, set-up, first loads, epilogue of the last
// tile), the time of a block, and for the kernels that are not persistent what every further round starts with.
// The persistent kernels fill the chip from about 60 tiles of 256 x 256 on; below that they leave SMs idle and a
// block takes a lone CTA pair 275 ns whatever the tile.  Measured at M 512 (pair kernel -> this choice): 1024 -> 1024
// 10.9 -> 7.0 us, 1024 -> 3072 11.3 -> 8.4, 4096 -> 1024 24.4 -> 11.8, rank-r projections from 1024 8.6 -> 6.4 and
// (8192 tokens) from 4096 21.5 -> 16.0; 4096 tokens and more of the wide layers stay with the pair kernel
// (1024 -> 1024: 11.6 against 17.4).  Tiles of 128 rows win over pairs where 256-row tiles need a round more: 1152 x 4096
// -> 4096 (144 tiles on 148 SMs, or 80 on 74 pairs) 27.1 us, as pairs 34.3; 2176 x 768 -> 3072 with a residual 19.6, as
// pairs 15.0.
enum Kernel { KERNEL_SINGLE, KERNEL_PAIR, KERNEL_PAIR128, KERNEL_SPLIT64_1, KERNEL_SPLIT64_2, KERNEL_SPLIT64_4, KERNEL_SPLIT64_8, KERNEL_SPLIT128_1,
              KERNEL_SPLIT128_2 };
Kernel pick_kernel(const GemmArgs& a) {
  const int64_t sms = num_sms();
  const int64_t kb = (a.K + BK - 1) / BK + (a.Ke + BK - 1) / BK;
  auto cdiv = [](int64_t x, int64_t y) { return (x + y - 1) / y; };
  Kernel best = KERNEL_SINGLE;
  int64_t best_ns = INT64_MAX;
  auto offer = [&](Kernel k, int64_t ns) { if (ns < best_ns) { best_ns = ns; best = k; } };
  if (pair_ok(a)) offer(KERNEL_PAIR, 5500 + cdiv(cdiv(a.M, 2 * BM) * cdiv(a.N, 256), max_pairs()) * kb * 275);
  // tiles of half the width where those of 256 fill their last round badly: 1665 x 768 -> 3072 with GELU (84 tiles on 74 pairs, or
  // 168) 19.3 -> 16.6 us, its backward 20.2 -> 18.5, 1665 x 1024 -> 3072 16.7 -> 15.7; 2560 x 1024 -> 4096 27.2 as 256, 28.2 as 128
  if (pair_ok(a)) offer(KERNEL_PAIR128, 4500 + cdiv(cdiv(a.M, 2 * BM) * cdiv(a.N, 128), max_pairs()) * kb * 200);
  // (where both take about as many rounds, two CTAs by themselves are 10-20 % slower than a pair, and their epilogue waits
  // for its second operand, 2 us a round, which the pair kernel brings ahead by TMA)
  const int bn = pick_bn(a);
  const int64_t block = bn == 256 ? 330 : bn == 64 ? 200 : 300;
  const bool need_r = a.epi == EPI_BIAS_RESID || a.epi == EPI_MUL_GELUGRAD;
  offer(KERNEL_SINGLE, 5500 + cdiv(cdiv(a.M, BM) * cdiv(a.N, bn), bn == 64 ? 2 * sms : sms) * (kb * block + (need_r ? 2000 : 0)));
  auto split = [&](Kernel k, int bn, int s, int64_t fixed, int64_t block_ns = 190) {
    const int64_t slots = s == 1 ? sms : max_split_clusters(s) > 0 ? max_split_clusters(s) : sms / s;
    const int64_t rounds = cdiv(cdiv(a.M, BM) * cdiv(a.N, bn), slots);
    if (s == 1 || kb >= 2 * s) offer(k, fixed + rounds * cdiv(kb, s) * block_ns + (rounds - 1) * 3000);
  };
  split(KERNEL_SPLIT64_1, 64, 1, 3600);
  split(KERNEL_SPLIT64_2, 64, 2, 4700);
  split(KERNEL_SPLIT64_4, 64, 4, 5000);
  split(KERNEL_SPLIT64_8, 64, 8, 5500);
  split(KERNEL_SPLIT128_1, 128, 1, 4400);
  // 1000 x 4096 -> 1024 17.4 -> 14.2 us (128 tiles of 64 columns, or 64 of 128 in clusters of two), x 2304 -> 768 11.3 -> 10.3
  split(KERNEL_SPLIT128_2, 128, 2, 5350, 230);
  return best;
}

// Fills the parameters both kernels share and encodes the tensor maps; box rows of the W maps differ.
bool prepare(const GemmArgs& a, int* status, int w_box_rows, CUtensorMap* mX, CUtensorMap* mW, CUtensorMap* mXe,
             CUtensorMap* mWe, CUtensorMap* mY, CUtensorMap* mZ, TcParams* p) {
  const int G = a.rows_per_group > 0 ? a.M / a.rows_per_group : 1;
  const int w_rows = a.w_rows > 0 ? a.w_rows : a.N;
  if (!make_map(mX, a.X, a.M, a.K + a.k_gap_len, a.ldx, BM)) return false;
  if (!make_map(mW, a.W, a.w_grouped ? (uint64_t)G * a.N : (uint64_t)w_rows, a.K + a.k_gap_len, a.ldw, w_box_rows)) return false;
  p->M = a.M; p->N = a.N; p->K = a.K; p->num_kb = (a.K + BK - 1) / BK;      // the tail of the last block is zero-filled by the copies
  p->gap_kb = a.k_gap_len / BK;
  p->gap_kb_begin = a.k_gap_len > 0 ? a.k_gap_begin / BK : p->num_kb;
  if (a.Ke > 0) {
    const uint64_t ke_cols = (uint64_t)((a.Ke + BK - 1) / BK) * BK;
    if (!make_map(mXe, a.Xe, a.M, ke_cols, a.ldxe, BM)) return false;
    if (!make_map(mWe, a.We, a.we_grouped ? (uint64_t)G * a.N : (uint64_t)a.N, ke_cols, a.ldwe, w_box_rows)) return false;
    p->ext_blocks = (a.Ke + BK - 1) / BK;
    p->ext_last_mmas = (a.Ke - (p->ext_blocks - 1) * BK) / UMMA_K;
  } else {
    *mXe = *mX; *mWe = *mW;
    p->ext_blocks = 0; p->ext_last_mmas = 0;
  }
  if (!make_out_map(mY, a.Y, a.M, a.N, a.ldy)) return false;
  if (a.epi == EPI_BIAS_GELU) { if (!make_out_map(mZ, a.Z, a.M, a.N, a.ldz)) return false; }
  else *mZ = *mY;
  p->rows_per_group = a.rows_per_group;
  p->w_group_rows = a.w_grouped ? a.N : 0;
  p->we_group_rows = a.we_grouped ? a.N : 0;
  p->epi = a.epi; p->gelu_tanh = a.gelu_tanh;
  p->bias = (const bf16*)a.bias; p->R = (const bf16*)a.R; p->ldr = a.ldr;
  p->Y = (bf16*)a.Y; p->ldy = a.ldy; p->Z = (bf16*)a.Z; p->ldz = a.ldz;
  p->status = status;
  return true;
}

// Off the tile sizes the layers with a tanh-form GELU used to be computed with tanhf (gemm_simt.cu): they keep fp32
// accuracy here (see gelu_sigmoid), for two special-function instructions per element instead of one.
bool exact_gelu(const GemmArgs& a) {
  return (a.epi == EPI_BIAS_GELU || a.epi == EPI_MUL_GELUGRAD) && a.gelu_tanh && (a.M % BM != 0 || a.K % BK != 0);
}

template <int BN, bool EXACT>
cudaError_t launch(const GemmArgs& a, int* status, cudaStream_t st) {
  using C = Cfg<BN>;
  const int sms = num_sms();
  static PerDeviceOnce once;                    // one per instantiation; attributes are per device
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<BN, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  CUtensorMap mX, mW, mXe, mWe, mY, mZ;
  TcParams p;
  if (!prepare(a, status, BN, &mX, &mW, &mXe, &mWe, &mY, &mZ, &p)) return cudaErrorInvalidValue;
  p.tiles_m = (a.M + BM - 1) / BM; p.tiles_n = (a.N + BN - 1) / BN;
  const int tiles = p.tiles_m * p.tiles_n;
  const int slots = sms * C::CTAS_PER_SM;
  const int grid = tiles < slots ? tiles : slots;
  launch_overlapped(gemm_tc_kernel<BN, EXACT>, grid, NUM_THREADS, C::SMEM_BYTES, st, mX, mW, mXe, mWe, mY, mZ, p);
  return cudaGetLastError();
}

template <int BN, int S, int STAGES, bool EXACT>
cudaError_t launch_split(const GemmArgs& a, int* status, cudaStream_t st) {
  using C = SplitCfg<BN, S, STAGES>;
  static PerDeviceOnce once;
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_split_kernel<BN, S, STAGES, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  CUtensorMap mX, mW, mXe, mWe, mY, mZ;
  TcParams p;
  if (!prepare(a, status, BN, &mX, &mW, &mXe, &mWe, &mY, &mZ, &p)) return cudaErrorInvalidValue;
  p.tiles_m = (a.M + BM - 1) / BM; p.tiles_n = (a.N + BN - 1) / BN;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.tiles_m * p.tiles_n * S)); cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = C::SMEM_BYTES; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = chain_attribute(at, 1);
  return cudaLaunchKernelEx(&cfg, gemm_tc_split_kernel<BN, S, STAGES, EXACT>, mX, mW, mXe, mWe, mY, mZ, p);
}

template <int EPI, bool EXACT, int BN>
cudaError_t launch_pair_epi(const GemmArgs& a, int* status, cudaStream_t st) {
  constexpr bool NEED_R = EPI == EPI_BIAS_RESID || EPI == EPI_MUL_GELUGRAD;
  using C = PairCfg<NEED_R, BN>;
  static PerDeviceOnce once;
  const int dev = current_device();
  if (once.needed(dev)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_pair_kernel<EPI, EXACT, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  CUtensorMap mX, mW, mXe, mWe, mY, mZ, mR;
  TcParams p;
  if (!prepare(a, status, C::BN / 2, &mX, &mW, &mXe, &mWe, &mY, &mZ, &p)) return cudaErrorInvalidValue;
  p.tiles_m = (a.M + 2 * BM - 1) / (2 * BM); p.tiles_n = (a.N + C::BN - 1) / C::BN;
  const int tiles = p.tiles_m * p.tiles_n;
  const int pairs = tiles < max_pairs() ? tiles : max_pairs();
  mR = mY;
  if (NEED_R && !make_map(&mR, a.R, a.M, a.N, a.ldr, BM)) return cudaErrorInvalidValue;
  launch_overlapped(gemm_tc_pair_kernel<EPI, EXACT, BN>, 2 * pairs, NUM_THREADS, C::SMEM_BYTES, st, mX, mW, mXe, mWe, mY, mZ, mR, p);
  return cudaGetLastError();
}
template <bool EXACT, int BN>
cudaError_t launch_pair(const GemmArgs& a, int* status, cudaStream_t st) {
  switch (a.epi) {
    case EPI_BIAS_GELU: return launch_pair_epi<EPI_BIAS_GELU, EXACT, BN>(a, status, st);
    case EPI_MUL_GELUGRAD: return launch_pair_epi<EPI_MUL_GELUGRAD, EXACT, BN>(a, status, st);
    case EPI_BIAS_RESID: return launch_pair_epi<EPI_BIAS_RESID, false, BN>(a, status, st);
    default: return launch_pair_epi<EPI_BIAS, false, BN>(a, status, st);
  }
}

template <int S>
int query_split_clusters() {
  using C = SplitCfg<64, S, 8>;
  const auto kernel = gemm_tc_split_kernel<64, S, 8, false>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S); cfg.blockDim = dim3(NUM_THREADS); cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = S; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess ? n : 0;
}

}  // namespace

int gemm_tc_init() {
  if (!tensor_map_encoder()) return -1;
  const int dev = current_device(), sms = num_sms();
  if (dev < 0 || sms < 1) return -1;
  if (!g_pair_once.needed(dev)) return 0;
  // how many CTA pairs fit on this device at once (the pair kernel is persistent: one wave)
  g_max_pairs[dev] = 0;
  if (cudaFuncSetAttribute(gemm_tc_pair_kernel<EPI_BIAS_RESID, false, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<true, 256>::SMEM_BYTES) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sms & ~1); cfg.blockDim = dim3(NUM_THREADS); cfg.dynamicSmemBytes = PairCfg<true, 256>::SMEM_BYTES;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    cfg.attrs = &at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_pair_kernel<EPI_BIAS_RESID, false, 256>, &cfg) == cudaSuccess && n > 0)
      g_max_pairs[dev] = n < sms / 2 ? n : sms / 2;
  }
  g_max_split_clusters[dev][0] = query_split_clusters<2>();
  g_max_split_clusters[dev][1] = query_split_clusters<4>();
  g_max_split_clusters[dev][2] = query_split_clusters<8>();
  cudaGetLastError();
  g_pair_once.done(dev);
  return 0;
}

bool gemm_tc_supported(const GemmArgs& a) {
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (!tensor_map_encoder() || a.dtype != DT_BF16) return false;
  // M and K may be anything the copies' 16-byte rule allows: rows past M and columns past K are zero-filled on the
  // way in, rows past M clipped on the way out (on the plain-FMA kernel instead, a GPT-2-small-shaped round of
  // 5 x 333 tokens takes 22 times as long).  Groups must not share a tile.
  if (a.M < 1 || a.K < 8 || a.K % 8 != 0 || a.N < 8 || a.N % 8 != 0) return false;
  if (a.rows_per_group > 0 && a.rows_per_group < a.M && (a.rows_per_group % BM != 0 || a.M % a.rows_per_group != 0)) return false;
  if (a.k_gap_len > 0 && a.K % BK != 0) return false;
  if (a.ldx % 8 || a.ldw % 8 || a.ldy % 8) return false;
  if (a.k_gap_len < 0 || a.k_gap_begin < 0 || a.k_gap_len % BK || a.k_gap_begin % BK || a.k_gap_begin > a.K) return false;
  if (!al16(a.X) || !al16(a.W) || !al16(a.Y)) return false;
  if (a.bias && !al16(a.bias)) return false;
  if (a.epi == EPI_BIAS_GELU && (!a.Z || a.ldz % 8 || !al16(a.Z))) return false;
  if ((a.epi == EPI_BIAS_RESID || a.epi == EPI_MUL_GELUGRAD) && (!a.R || a.ldr % 8 || !al16(a.R))) return false;
  if (a.Ke > 0) {
    if (a.Ke % UMMA_K != 0 || !a.Xe || !a.We || a.ldxe % 8 || a.ldwe % 8 || !al16(a.Xe) || !al16(a.We)) return false;
    if ((int64_t)((a.Ke + BK - 1) / BK) * BK > a.ldxe || (int64_t)((a.Ke + BK - 1) / BK) * BK > a.ldwe) return false;
  }
  return true;
}

namespace {
template <bool EXACT>
cudaError_t launch_picked(const GemmArgs& a, int* status, cudaStream_t st) {
  switch (pick_kernel(a)) {
    case KERNEL_SPLIT64_1: return launch_split<64, 1, 8, EXACT>(a, status, st);
    case KERNEL_SPLIT64_2: return launch_split<64, 2, 8, EXACT>(a, status, st);
    case KERNEL_SPLIT64_4: return launch_split<64, 4, 8, EXACT>(a, status, st);
    case KERNEL_SPLIT64_8: return launch_split<64, 8, 8, EXACT>(a, status, st);
    case KERNEL_SPLIT128_1: return launch_split<128, 1, 6, EXACT>(a, status, st);
    case KERNEL_SPLIT128_2: return launch_split<128, 2, 6, EXACT>(a, status, st);
    case KERNEL_PAIR: return launch_pair<EXACT, 256>(a, status, st);
    case KERNEL_PAIR128: return launch_pair<EXACT, 128>(a, status, st);
    default: break;
  }
  switch (pick_bn(a)) {
    case 256: return launch<256, EXACT>(a, status, st);
    case 128: return launch<128, EXACT>(a, status, st);
    default: return launch<64, EXACT>(a, status, st);
  }
}
}  // namespace

cudaError_t gemm_tc(const GemmArgs& args, int* status, cudaStream_t st) {
  if (!gemm_tc_supported(args)) return cudaErrorInvalidValue;
  GemmArgs a = args;
  if (a.rows_per_group >= a.M) a.rows_per_group = 0;      // one group
  return exact_gelu(a) ? launch_picked<true>(a, status, st) : launch_picked<false>(a, status, st);
}

}  // namespace sl
