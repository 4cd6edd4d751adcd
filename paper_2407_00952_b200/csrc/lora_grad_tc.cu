// Adapter gradients G_A, G_B (Eq. 4-7) on the tensor cores.  The reduction over tokens
//   out[j][c] = sum_m Wt[m, w0 + j] * Z[m, z0 + c]
// is a product whose contraction index is the row index of BOTH operands, so both are fed to
// tcgen05.mma as MN-major tiles straight from their row-major layout (no transposed copies):
//   D[c, j] (128 x 64, fp32 in tensor memory) += Z_tile^T (128 c x 64 tokens) * Wt_tile (64 tokens x 64 j)
// One CTA owns 128 feature columns and one chunk of the token range; TMA streams 64-token blocks
// through a 4-stage ring, one thread issues the products, four warps read the accumulator back and
// write the wanted columns to scratch, where a second kernel adds the chunks in a fixed order (no float
// atomics), or straight to the gradient where a group's rows are one chunk.  HBM-bound: every Z element is
// read once, the 64-column weight tile is re-read per column tile (from L2).
#include <cuda.h>

#include "common.cuh"
#include "kernels.h"
#include "host_common.h"
#include "launch.cuh"
#include "tc_common.cuh"

namespace sl {
namespace {

using namespace tc;

constexpr int LT_C = 128;           // feature columns per CTA = accumulator lanes
constexpr int LT_K = 64;             // tokens per pipeline stage
constexpr int LT_N = 64;             // weight columns per product (one 128-byte swizzle row)
constexpr int LT_STAGES = 4;
constexpr int LT_ZBOX = LT_K * 64 * 2;                 // one [64 tokens][64 columns] box
constexpr int LT_STAGE = 2 * LT_ZBOX + LT_K * LT_N * 2;
constexpr int LT_THREADS = 192;      // warp 0: TMA, warp 1: MMA, warps 2-5: accumulator read-back
constexpr int LT_OFF_BAR = LT_STAGES * LT_STAGE;
constexpr int LT_SMEM = LT_OFF_BAR + 128 + 1024;
constexpr int LT_TMEM_COLS = 64;
// fp32 accumulate, bf16 x bf16, A and B both MN-major
constexpr uint32_t LT_IDESC = make_idesc(LT_C, LT_N) | (1u << 15) | (1u << 16);

struct LgParams {
  int C, rows_per_chunk, R, r, rp, wsel0;
  float* partial;                                // [layer][chunk][R][C]
  float* out; int64_t out_ls, ogs, ots, osj, osc; float scale;
  int* status;
};
// Up to LT_MAX_JOBS reductions over the same token rows, of several layers, in one launch (blockIdx.z picks layer and
// job): the adapter gradients of a layer, e.g. G_A of all targets from u and G_B of each target from its slice of dy, or
// those of all layers of a side.  One launch instead of one per job: the jobs are short (microseconds to tens of them), so
// their start-up, tail and launch gaps weigh as much as their traffic.
constexpr int LT_MAX_JOBS = LORA_GRAD_MAX_JOBS;
struct LgBatch {
  CUtensorMap mapZ[LT_MAX_JOBS];
  CUtensorMap mapW[LT_MAX_JOBS];
  LgParams p[LT_MAX_JOBS];
  int wx0[LT_MAX_JOBS];
  int njobs;
};
static_assert(sizeof(LgBatch) <= 4000, "kernel parameters");

// MN-major operand stored as [k rows][64 elements] boxes (128-byte rows, 128-byte swizzle): groups
// of 8 k-rows are 1024 bytes apart; `mn_stride` is the distance between consecutive 64-element
// blocks along the MN dimension (unused when the operand is one block wide).
__device__ __forceinline__ uint64_t desc_mn(uint32_t addr, uint32_t mn_stride) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((mn_stride >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// LAYERS: the operands are planes of three-dimensional maps, one per layer (a single layer: two-dimensional ones).  DIRECT:
// one chunk per group, the result goes to the gradient.
template <bool LAYERS, bool DIRECT>
__global__ void __launch_bounds__(LT_THREADS, 2)
lora_grad_tc_kernel(const __grid_constant__ LgBatch bt) {
  const int layer = LAYERS ? (int)blockIdx.z / bt.njobs : 0, job = LAYERS ? (int)blockIdx.z % bt.njobs : (int)blockIdx.z;
  const CUtensorMap& mapZ = bt.mapZ[job];
  const CUtensorMap& mapW = bt.mapW[job];
  const LgParams& p = bt.p[job];
  const int wx0 = bt.wx0[job];
  if ((int)blockIdx.x * LT_C >= p.C) return;             // the grid is as wide as the widest job
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t bar = base + LT_OFF_BAR;
  auto FULL = [&](int s) { return bar + 8u * s; };
  auto EMPTY = [&](int s) { return bar + 8u * (LT_STAGES + s); };
  const uint32_t ACC = bar + 8u * (2 * LT_STAGES);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + LT_OFF_BAR + 8 * (2 * LT_STAGES + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + LT_OFF_BAR + 8 * (2 * LT_STAGES + 1) + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = blockIdx.x * LT_C, chunk = blockIdx.y;
  const int row0 = chunk * p.rows_per_chunk;
  const int kblocks = p.rows_per_chunk / LT_K;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * LT_STAGES + 1; ++i) mbar_init(bar + 8u * i, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"((uint32_t)LT_TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  overlap_sync();

  if (warp == 0) {                       // producer and issuer as converged warps (see gemm_tc.cu)
    const bool leader = elect_one();
    for (int kb = 0; kb < kblocks; ++kb) {
      const int s = kb % LT_STAGES;
      if (!mbar_wait_warp(EMPTY(s), (((uint32_t)(kb / LT_STAGES)) & 1u) ^ 1u, abort_flag, p.status, 40)) break;
      const uint32_t dst = base + s * LT_STAGE;
      const int row = row0 + kb * LT_K;
      if (leader) {
        mbar_expect_tx(FULL(s), LT_STAGE);
        auto load = [&](uint32_t to, const CUtensorMap* map, int c) {
          if constexpr (LAYERS) tma_load_3d(to, map, FULL(s), c, row, layer); else tma_load_2d(to, map, FULL(s), c, row);
        };
        load(dst, &mapZ, c0);
        load(dst + LT_ZBOX, &mapZ, c0 + 64);       // past the last column: zero fill
        load(dst + 2 * LT_ZBOX, &mapW, wx0);
      }
      __syncwarp();
    }
  } else if (warp == 1) {
    const bool leader = elect_one();
    bool ok = true;
    for (int kb = 0; kb < kblocks && ok; ++kb) {
      const int s = kb % LT_STAGES;
      if (!mbar_wait_warp(FULL(s), ((uint32_t)(kb / LT_STAGES)) & 1u, abort_flag, p.status, 41)) { ok = false; break; }
      tc_fence_after();
      const uint32_t a = base + s * LT_STAGE, b = a + 2 * LT_ZBOX;
      if (leader) {
#pragma unroll
        for (int k = 0; k < LT_K / UMMA_K; ++k)     // 16 tokens = two 8-row groups = 2048 bytes
          tc_mma_bf16(tmem_base, desc_mn(a + k * 2048, LT_ZBOX), desc_mn(b + k * 2048, 16), LT_IDESC,
                      (kb | k) != 0 ? 1u : 0u);
        tc_commit(EMPTY(s));
      }
      __syncwarp();
    }
    if (ok && leader) tc_commit(ACC);
  } else {
    // accumulator read-back: lane group (warp % 4) of tensor memory, one feature column per thread
    const int q = warp & 3;
    if (mbar_wait(ACC, 0u, abort_flag, p.status, 42)) {
      tc_fence_after();
      float v[LT_N];
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
      tc_ld32(t_row, v);
      tc_ld32(t_row + 32u, v + 32);
      tc_wait_ld();
      const int c = c0 + q * 32 + lane;
      if (c < p.C) {
        const int sh = p.rp == 16 ? 4 : (p.rp == 32 ? 5 : 6);
        float* out = DIRECT ? p.out + (size_t)layer * p.out_ls + (size_t)chunk * p.ogs + (size_t)c * p.osc
                            : p.partial + ((size_t)layer * gridDim.y + chunk) * p.R * p.C + c;
        const int ots = DIRECT ? (int)p.ots : 0, osj = DIRECT ? (int)p.osj : 0;       // within one adapter pair of one layer
#pragma unroll
        for (int col = 0; col < LT_N; ++col) {
          const int rel = col - p.wsel0;
          const int t = rel >> sh, jj = rel & (p.rp - 1);
          const int j = t * p.r + jj;
          if (rel >= 0 && jj < p.r && j < p.R) {
            if constexpr (DIRECT) out[t * ots + jj * osj] = p.scale * v[col];
            else out[(size_t)j * p.C] = v[col];
          }
        }
      }
    }
  }

  __syncwarp();
  if (*abort_flag) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);     // let copies in flight land before the CTA exits
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)LT_TMEM_COLS) : "memory");
  }
}

PerDeviceOnce g_once;

// `layers` bf16 matrices [rows, cols] with leading dimension ld, ls elements apart; box = 64 columns x 64 rows, 128-byte swizzle
bool make_map(CUtensorMap* m, const void* ptr, uint64_t layers, uint64_t rows, uint64_t cols, uint64_t ld, uint64_t ls) {
  if (layers == 1) return cached_map_2d(m, ptr, rows, cols, ld, 64, (uint32_t)LT_K, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
  return cached_map_3d(m, ptr, layers, rows, cols, ld, ls, 64, (uint32_t)LT_K, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

bool init_device() {
  const int dev = current_device();
  if (dev < 0 || !tensor_map_encoder()) return false;
  if (!g_once.needed(dev)) return true;
  for (auto kernel : {lora_grad_tc_kernel<false, false>, lora_grad_tc_kernel<false, true>, lora_grad_tc_kernel<true, false>, lora_grad_tc_kernel<true, true>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LT_SMEM) != cudaSuccess) return false;
  g_once.done(dev);
  return true;
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

bool lora_grad_tc_supported(int dt, const void* Z, int64_t ldz, int zcol0, int C, const void* Wt, int64_t ldwt,
                            int wcol0, int r, int rp, int nt, int M, int rows_per_group) {
  if (dt != DT_BF16 || !(rp == 16 || rp == 32 || rp == 64) || r < 1 || r > rp || nt < 1) return false;
  // one group: any M (rows past the last are zero-filled by the copies); several: whole 128-row blocks each
  if (rows_per_group > 0 && rows_per_group < M && (rows_per_group % 128 != 0 || M % rows_per_group != 0)) return false;
  if (C % 8 != 0 || ldz % 8 != 0 || zcol0 % 8 != 0 || ldwt % 64 != 0 || !al16(Z) || !al16(Wt)) return false;
  const int wsel0 = wcol0 % LT_N;
  if (wsel0 + (nt - 1) * rp + r > LT_N || wcol0 - wsel0 + LT_N > ldwt) return false;
  return true;
}

// Chunks per group (at most max_chunks) for a grid of `ctas_per_chunk_set` CTAs per chunk: the choice that minimises
// (waves of resident CTAs, two per SM) x (rows per chunk), every chunk a whole number of 128-row blocks.  One chunk needs no second
// kernel, which is worth about 4 us: 1000 rows of a CTA that has an SM's loads to itself, 300 of one among two per SM.
static int pick_chunks(int ctas_per_chunk_set, int rpg, int64_t max_chunks) {
  const int n = num_sms(), sms = n > 0 ? n : 1, resident = 2 * sms;
  const double second_kernel = ctas_per_chunk_set > sms ? 300.0 : 1000.0;
  int best = 1;
  double best_cost = 1e300;
  for (int s = 1; s <= rpg / 128 && s <= (max_chunks > 1 ? max_chunks : 1); ++s) {
    if (rpg % (s * 128) != 0) continue;
    const int ctas = ctas_per_chunk_set * s;
    const double cost = (double)((ctas + resident - 1) / resident) * ((double)rpg / s + 256.0) + (s > 1 ? second_kernel : 0.0);   // 256: a chunk's start-up
    if (cost < best_cost) { best_cost = cost; best = s; }
  }
  return best;
}

// All jobs share M and rows_per_group.  With more than one chunk per group (*chunks_per_group) the partials of job j go to
// partial + offsets[j] as [layer][chunk][R_j][C] (R_j = nt*r) for the caller's second kernel to add.
cudaError_t lora_grad_tc_layers(const LoraGradJob* jobs, int njobs, int layers, int M, int rows_per_group, float* partial,
                                size_t partial_floats, int* status, int* chunks_per_group, size_t* offsets, cudaStream_t st) {
  if (njobs < 1 || njobs > LT_MAX_JOBS || layers < 1) return cudaErrorInvalidValue;
  if (!init_device()) return cudaErrorNotSupported;
  if (!status) status = library_status_word();
  if (!status) return cudaErrorNotSupported;
  const bool one = rows_per_group <= 0 || rows_per_group >= M;
  const int rpg = one ? (M + 127) / 128 * 128 : rows_per_group;
  const int groups = one ? 1 : M / rpg;
  int ctiles = 0, ctiles_sum = 0;
  size_t set_floats = 0;                       // partials of one chunk per group, all jobs and layers
  for (int j = 0; j < njobs; ++j) {
    const int t = (jobs[j].C + LT_C - 1) / LT_C;
    ctiles = t > ctiles ? t : ctiles;
    ctiles_sum += t;
    set_floats += (size_t)layers * groups * jobs[j].nt * jobs[j].r * jobs[j].C;
  }
  const int s = pick_chunks(ctiles_sum * groups * layers, rpg, (int64_t)(partial_floats / set_floats));   // the scratch bounds the number of chunks
  LgBatch bt;
  size_t off = 0;
  for (int j = 0; j < njobs; ++j) {
    const LoraGradJob& jb = jobs[j];
    if (!make_map(&bt.mapZ[j], (const bf16*)jb.Z + jb.zcol0, (uint64_t)layers, (uint64_t)M, (uint64_t)jb.C, (uint64_t)jb.ldz, (uint64_t)jb.z_ls)) return cudaErrorInvalidValue;
    if (!make_map(&bt.mapW[j], jb.Wt, (uint64_t)layers, (uint64_t)M, (uint64_t)jb.ldwt, (uint64_t)jb.ldwt, (uint64_t)jb.wt_ls)) return cudaErrorInvalidValue;
    LgParams& p = bt.p[j];
    p.C = jb.C; p.rows_per_chunk = rpg / s; p.R = jb.nt * jb.r; p.r = jb.r; p.rp = jb.rp; p.wsel0 = jb.wcol0 % LT_N;
    p.partial = partial + off; p.status = status;
    p.out = jb.out; p.out_ls = jb.out_ls; p.ogs = jb.out_group_stride; p.ots = jb.out_target_stride; p.osj = jb.out_sj; p.osc = jb.out_sc;
    p.scale = jb.scale;
    bt.wx0[j] = jb.wcol0 - p.wsel0;
    offsets[j] = off;
    off += (size_t)layers * groups * s * p.R * jb.C;
  }
  for (int j = njobs; j < LT_MAX_JOBS; ++j) { bt.mapZ[j] = bt.mapZ[0]; bt.mapW[j] = bt.mapW[0]; bt.p[j] = bt.p[0]; bt.wx0[j] = bt.wx0[0]; }
  bt.njobs = njobs;
  dim3 grid(ctiles, groups * s, layers * njobs);
  const auto kernel = layers > 1 ? (s > 1 ? lora_grad_tc_kernel<true, false> : lora_grad_tc_kernel<true, true>)
                                 : (s > 1 ? lora_grad_tc_kernel<false, false> : lora_grad_tc_kernel<false, true>);
  launch_overlapped(kernel, grid, LT_THREADS, LT_SMEM, st, bt);
  *chunks_per_group = s;
  return cudaGetLastError();
}

}  // namespace sl
