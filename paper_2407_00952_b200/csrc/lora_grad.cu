// Adapter gradients G_A, G_B (Eq. 4-7): skinny reductions over the tokens of each group,
//   out[g][t][jj][c] = scale * sum_{m in group g} Wt[m, wcol0 + t*rp + jj] * Z[m, zcol0 + c]
// for nt targets of rank r (R = nt*r weight columns) and C feature columns.  HBM-bound: Z is read
// once per 4 weight columns.  A block is 64 column threads (one 16-byte vector each) x 4 or 16 row lanes
// over a chunk of LG_ROWS rows, four blocks per SM so that enough loads are in flight; the row
// lanes are summed through shared memory, chunk partials go to scratch and a second kernel adds
// them in chunk order (no float atomics, so the result does not depend on scheduling).
#include "common.cuh"
#include "host_common.h"
#include "kernels.h"
#include "launch.cuh"

namespace sl {
namespace {

constexpr int LG_ROWS = 128;   // rows per chunk; group sizes must be multiples of it
constexpr int LG_CT = 64;      // column threads per block
constexpr int RJ = 4;          // weight columns per block

// four consecutive weights of one row
template <typename T> __device__ __forceinline__ void load4(const T* p, float* w);
template <> __device__ __forceinline__ void load4<float>(const float* p, float* w) {
  float4 v = *reinterpret_cast<const float4*>(p);
  w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}
template <> __device__ __forceinline__ void load4<bf16>(const bf16* p, float* w) {
  uint2 v = *reinterpret_cast<const uint2*>(p);
  const bf16* b = reinterpret_cast<const bf16*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) w[i] = __bfloat162float(b[i]);
}

// LG_RL: row lanes per block.  Four and four blocks per SM where the chunks fill the chip; sixteen where there are few
// (fp32, 512 tokens: 8 blocks, whose 32 rows per lane one after another took 17 us).
template <typename T, bool VEC4, int LG_RL>
__global__ void __launch_bounds__(LG_CT * LG_RL, LG_RL == 4 ? 4 : 1)
lora_grad_partial_kernel(const T* __restrict__ Z, int64_t ldz, int zcol0, int C, const T* __restrict__ Wt,
                         int64_t ldwt, int wcol0, int r, int rp, int R, int M, float* __restrict__ partial) {
  overlap_sync();
  constexpr int N = Vec16<T>::N;
  __shared__ float red[LG_RL / 2][RJ * N][LG_CT];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int c = (blockIdx.x * LG_CT + tx) * N;
  const int chunk = blockIdx.y;
  const int j0 = blockIdx.z * RJ;
  const int m0 = chunk * LG_ROWS;
  const int m1 = min(m0 + LG_ROWS, M);
  const bool active = c < C;
  int wc[RJ];
#pragma unroll
  for (int j = 0; j < RJ; ++j) {
    int jj = j0 + j;
    wc[j] = jj < R ? wcol0 + (jj / r) * rp + (jj % r) : -1;
  }
  float acc[RJ][N];
#pragma unroll
  for (int j = 0; j < RJ; ++j)
#pragma unroll
    for (int i = 0; i < N; ++i) acc[j][i] = 0.f;
  if (active) {
#pragma unroll 4
    for (int m = m0 + ty; m < m1; m += LG_RL) {
      Vec16<T> v; v.load(Z + (size_t)m * ldz + zcol0 + c);
      float w[RJ];
      if (VEC4) {
        load4<T>(Wt + (size_t)m * ldwt + wc[0], w);     // r % 4 == 0: the four columns are adjacent
      } else {
#pragma unroll
        for (int j = 0; j < RJ; ++j) w[j] = wc[j] >= 0 ? to_f<T>(Wt[(size_t)m * ldwt + wc[j]]) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        float zv = v.get(i);
#pragma unroll
        for (int j = 0; j < RJ; ++j) acc[j][i] = fmaf(w[j], zv, acc[j][i]);
      }
    }
  }
  // add the row lanes pairwise, upper half onto lower half (a fixed order)
#pragma unroll
  for (int half = LG_RL / 2; half > 0; half >>= 1) {
    if (ty >= half && ty < 2 * half) {
#pragma unroll
      for (int j = 0; j < RJ; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) red[ty - half][j * N + i][tx] = acc[j][i];
    }
    __syncthreads();
    if (ty < half) {
#pragma unroll
      for (int j = 0; j < RJ; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) acc[j][i] += red[ty][j * N + i][tx];
    }
    __syncthreads();
  }
  if (ty == 0 && active) {
    // partial layout: [chunk][R][C]
#pragma unroll
    for (int j = 0; j < RJ; ++j) {
      if (j0 + j < R) {
        float* p = partial + ((size_t)chunk * R + (j0 + j)) * C + c;
#pragma unroll
        for (int i = 0; i < N; i += 4)
          *reinterpret_cast<float4*>(p + i) = make_float4(acc[j][i], acc[j][i + 1], acc[j][i + 2], acc[j][i + 3]);
      }
    }
  }
}

// Many outputs (wide models): one output per thread; the chunk partials of a group are added in chunk order (adjacent threads
// read adjacent floats of every partial, so the reads coalesce; no shared memory, no barrier).
constexpr int RED_THREADS = 256;
__global__ void __launch_bounds__(RED_THREADS)
lora_grad_reduce_kernel(const float* __restrict__ partial, int r, int R, int C, int chunks_per_group, float scale,
                        float* __restrict__ out, int64_t out_group_stride, int64_t out_target_stride,
                        int64_t out_sj, int64_t out_sc) {
  overlap_sync();
  const int idx = blockIdx.x * RED_THREADS + threadIdx.x;   // over R*C
  const int g = blockIdx.y;
  if (idx >= R * C) return;
  const size_t rc = (size_t)R * C;
  const float* p = partial + (size_t)g * chunks_per_group * rc + idx;
  float s = 0.f;
#pragma unroll 4
  for (int k = 0; k < chunks_per_group; ++k) s += p[(size_t)k * rc];
  const int j = idx / C, c = idx % C;
  out[(size_t)g * out_group_stride + (size_t)(j / r) * out_target_stride + (size_t)(j % r) * out_sj +
      (size_t)c * out_sc] = scale * s;
}

// Few outputs, many chunks (narrow models, long groups): 32 outputs per block (threadIdx.x) and
// RED_LANES chunk lanes (threadIdx.y), each adding every RED_LANES-th partial, combined in lane order.
constexpr int RED_LANES = 8;
__global__ void __launch_bounds__(32 * RED_LANES)
lora_grad_reduce_lanes_kernel(const float* __restrict__ partial, int r, int R, int C, int chunks_per_group, float scale,
                        float* __restrict__ out, int64_t out_group_stride, int64_t out_target_stride,
                        int64_t out_sj, int64_t out_sc) {
  overlap_sync();
  __shared__ float red[RED_LANES][32];
  const int idx = blockIdx.x * 32 + threadIdx.x;   // over R*C
  const int g = blockIdx.y;
  const bool active = idx < R * C;
  float s = 0.f;
  if (active) {
    const float* p = partial + (size_t)g * chunks_per_group * R * C + idx;
    for (int k = threadIdx.y; k < chunks_per_group; k += RED_LANES) s += p[(size_t)k * R * C];
  }
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && active) {
    float t = 0.f;
#pragma unroll
    for (int l = 0; l < RED_LANES; ++l) t += red[l][threadIdx.x];
    const int j = idx / C, c = idx % C;
    out[(size_t)g * out_group_stride + (size_t)(j / r) * out_target_stride + (size_t)(j % r) * out_sj +
        (size_t)c * out_sc] = scale * t;
  }
}

// The second kernel for a batch of jobs and layers (blockIdx.z): one output per thread, chunks added in order.
struct RedJob { const float* partial; float* out; int r, R, C; float scale; int64_t ols, ogs, ots, osj, osc; };
struct RedBatch { RedJob j[LORA_GRAD_MAX_JOBS]; int njobs; };
__global__ void __launch_bounds__(RED_THREADS)
lora_grad_reduce_batch_kernel(RedBatch b, int chunks_per_group) {
  overlap_sync();
  const int layer = (int)blockIdx.z / b.njobs;
  const RedJob& jb = b.j[(int)blockIdx.z % b.njobs];
  const int idx = blockIdx.x * RED_THREADS + threadIdx.x;   // over R*C
  const int g = blockIdx.y;
  const int C = jb.C;
  if (idx >= jb.R * C) return;
  const size_t rc = (size_t)jb.R * C;
  const float* p = jb.partial + ((size_t)layer * gridDim.y + g) * chunks_per_group * rc + idx;
  float s = 0.f;
#pragma unroll 4
  for (int k = 0; k < chunks_per_group; ++k) s += p[(size_t)k * rc];
  const int j = idx / C, c = idx % C;
  jb.out[(size_t)layer * jb.ols + (size_t)g * jb.ogs + (size_t)(j / jb.r) * jb.ots + (size_t)(j % jb.r) * jb.osj + (size_t)c * jb.osc] = jb.scale * s;
}
cudaError_t launch_reduce_batch(const LoraGradJob* jobs, int njobs, int layers, int groups, int chunks, const float* partial,
                                const size_t* offsets, cudaStream_t st) {
  RedBatch rb;
  int maxRC = 0;
  for (int j = 0; j < LORA_GRAD_MAX_JOBS; ++j) {
    const LoraGradJob& jb = jobs[j < njobs ? j : 0];
    rb.j[j] = {partial + offsets[j < njobs ? j : 0], jb.out, jb.r, jb.nt * jb.r, jb.C, jb.scale, jb.out_ls, jb.out_group_stride,
               jb.out_target_stride, jb.out_sj, jb.out_sc};
    if (jb.nt * jb.r * jb.C > maxRC) maxRC = jb.nt * jb.r * jb.C;
  }
  rb.njobs = njobs;
  launch_overlapped(lora_grad_reduce_batch_kernel, dim3((maxRC + RED_THREADS - 1) / RED_THREADS, groups, layers * njobs), RED_THREADS, 0, st, rb, chunks);
  return cudaGetLastError();
}

// fp32, the jobs of all layers of a side in one launch.  A block: RJ weight columns x 128 feature columns (32 threads of
// four) x one chunk of a group's rows, over 32 row lanes that are summed through shared memory in a fixed order; the result
// goes to the gradient where the chunk is the whole group, else to scratch as [job][layer][chunk][R][C].  What bounds it is
// the number of launches it replaces (two per job and layer, 4-5 us each): 512 tokens of width 128 are 16 loads per lane.
constexpr int LL_CT = 32, LL_RL = 32, LL_ROWS = 512;
struct LayersJob { const float *Z, *Wt; int64_t ldz, zls, ldwt, wls; int r, rp, R, C, jtile0; float* partial; float* out; int64_t ols, ogs, ots, osj, osc; float scale; };
struct LayersBatch { LayersJob j[LORA_GRAD_MAX_JOBS]; int njobs, jtiles, rows_per_group, chunks, chunk_rows, M; };
__global__ void __launch_bounds__(LL_CT * LL_RL) lora_grad_layers_kernel(const __grid_constant__ LayersBatch b) {
  overlap_sync();
  __shared__ float red[LL_RL / 2][RJ * 4][LL_CT];
  const int layer = (int)blockIdx.z / b.jtiles, jt = (int)blockIdx.z % b.jtiles;
  int job = 0;
  while (job + 1 < b.njobs && jt >= b.j[job + 1].jtile0) ++job;
  const LayersJob& jb = b.j[job];
  const int j0 = (jt - jb.jtile0) * RJ;
  const int tx = threadIdx.x, ty = threadIdx.y, c = (blockIdx.x * LL_CT + tx) * 4;
  const int g = (int)blockIdx.y / b.chunks, chunk = (int)blockIdx.y % b.chunks;
  const int m0 = g * b.rows_per_group + chunk * b.chunk_rows;
  const int m1 = min(min(m0 + b.chunk_rows, (g + 1) * b.rows_per_group), b.M);
  const bool active = c < jb.C;
  const float* Z = jb.Z + layer * jb.zls + c;
  const float* Wt = jb.Wt + layer * jb.wls;
  int wc[RJ];
#pragma unroll
  for (int j = 0; j < RJ; ++j) wc[j] = j0 + j < jb.R ? (j0 + j) / jb.r * jb.rp + (j0 + j) % jb.r : -1;
  float acc[RJ][4];
#pragma unroll
  for (int j = 0; j < RJ; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
  if (active) {
#pragma unroll 4
    for (int m = m0 + ty; m < m1; m += LL_RL) {
      const float4 z = *reinterpret_cast<const float4*>(Z + (size_t)m * jb.ldz);
#pragma unroll
      for (int j = 0; j < RJ; ++j) {
        const float w = wc[j] >= 0 ? Wt[(size_t)m * jb.ldwt + wc[j]] : 0.f;
        acc[j][0] = fmaf(w, z.x, acc[j][0]); acc[j][1] = fmaf(w, z.y, acc[j][1]);
        acc[j][2] = fmaf(w, z.z, acc[j][2]); acc[j][3] = fmaf(w, z.w, acc[j][3]);
      }
    }
  }
#pragma unroll
  for (int half = LL_RL / 2; half > 0; half >>= 1) {
    if (ty >= half && ty < 2 * half) {
#pragma unroll
      for (int j = 0; j < RJ; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) red[ty - half][j * 4 + i][tx] = acc[j][i];
    }
    __syncthreads();
    if (ty < half) {
#pragma unroll
      for (int j = 0; j < RJ; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][i] += red[ty][j * 4 + i][tx];
    }
    __syncthreads();
  }
  if (ty != 0 || !active) return;
#pragma unroll
  for (int j = 0; j < RJ; ++j) {
    const int jj = j0 + j;
    if (jj >= jb.R) break;
    if (jb.partial) {
      *reinterpret_cast<float4*>(jb.partial + (((size_t)layer * gridDim.y + blockIdx.y) * jb.R + jj) * jb.C + c) =
          make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
    } else {
      float* o = jb.out + (size_t)layer * jb.ols + (size_t)g * jb.ogs + (size_t)(jj / jb.r) * jb.ots + (size_t)(jj % jb.r) * jb.osj;
#pragma unroll
      for (int i = 0; i < 4; ++i) o[(size_t)(c + i) * jb.osc] = jb.scale * acc[j][i];
    }
  }
}

// picks the second kernel by the number of outputs (both add in a fixed order)
void launch_reduce(const float* partial, int r, int R, int C, int cpg, int groups, float scale, float* out,
                   int64_t out_group_stride, int64_t out_target_stride, int64_t out_sj, int64_t out_sc, cudaStream_t st) {
  if ((int64_t)R * C >= 32768) {
    dim3 g2((R * C + RED_THREADS - 1) / RED_THREADS, groups), b2(RED_THREADS);
    launch_overlapped(lora_grad_reduce_kernel, g2, b2, 0, st, partial, r, R, C, cpg, scale, out, out_group_stride, out_target_stride, out_sj, out_sc);
  } else {
    dim3 g2((R * C + 31) / 32, groups), b2(32, RED_LANES);
    launch_overlapped(lora_grad_reduce_lanes_kernel, g2, b2, 0, st, partial, r, R, C, cpg, scale, out, out_group_stride, out_target_stride, out_sj, out_sc);
  }
}

template <typename T, int RL>
void launch_partial_lanes(dim3 grid, cudaStream_t st, bool vec4, const void* Z, int64_t ldz, int zcol0, int C, const void* Wt,
                          int64_t ldwt, int wcol0, int r, int rp, int R, int M, float* partial) {
  dim3 block(LG_CT, RL);
  if (vec4)
    launch_overlapped(lora_grad_partial_kernel<T, true, RL>, grid, block, 0, st, (const T*)Z, ldz, zcol0, C, (const T*)Wt, ldwt, wcol0, r, rp, R, M, partial);
  else
    launch_overlapped(lora_grad_partial_kernel<T, false, RL>, grid, block, 0, st, (const T*)Z, ldz, zcol0, C, (const T*)Wt, ldwt, wcol0, r, rp, R, M, partial);
}
template <typename T>
void launch_partial(dim3 grid, cudaStream_t st, bool vec4, const void* Z, int64_t ldz, int zcol0, int C, const void* Wt,
                    int64_t ldwt, int wcol0, int r, int rp, int R, int M, float* partial) {
  if constexpr (sizeof(T) == 4) {                      // (16 lanes of bf16 vectors do not fit shared memory)
    if ((int64_t)grid.x * grid.y * grid.z <= num_sms())
      return launch_partial_lanes<T, 16>(grid, st, vec4, Z, ldz, zcol0, C, Wt, ldwt, wcol0, r, rp, R, M, partial);
  }
  launch_partial_lanes<T, 4>(grid, st, vec4, Z, ldz, zcol0, C, Wt, ldwt, wcol0, r, rp, R, M, partial);
}

}  // namespace

size_t lora_grad_scratch_floats(int M, int R, int C) {
  size_t chunks = (size_t)(M + LG_ROWS - 1) / LG_ROWS;
  return chunks * (size_t)R * (size_t)C;
}

cudaError_t lora_grad(int dt, const void* Z, int64_t ldz, int zcol0, int C, const void* Wt, int64_t ldwt, int wcol0,
                      int r, int rp, int nt, int M, int rows_per_group, float scale, float* out,
                      int64_t out_group_stride, int64_t out_target_stride, int64_t out_sj, int64_t out_sc,
                      float* partial, cudaStream_t st, int* status, bool use_tc) {
  if (use_tc && status && dt == DT_BF16 && (rp == 16 || rp == 32 || rp == 64)) {
    // tensor-core path, in windows of the targets whose weight columns share one 64-column tile
    const int tw = 64 / rp;
    bool ok = true;
    for (int t0 = 0; t0 < nt && ok; t0 += tw)
      ok = lora_grad_tc_supported(dt, Z, ldz, zcol0, C, Wt, ldwt, wcol0 + t0 * rp, r, rp, min(tw, nt - t0), M,
                                  rows_per_group);
    if (ok) {
      const int groups = rows_per_group > 0 && rows_per_group < M ? M / rows_per_group : 1;
      for (int t0 = 0; t0 < nt; t0 += tw) {
        const int ntw = min(tw, nt - t0), Rw = ntw * r;
        int cpg = 0;
        LoraGradJob jb;
        jb.Z = Z; jb.ldz = ldz; jb.zcol0 = zcol0; jb.C = C; jb.Wt = Wt; jb.ldwt = ldwt; jb.wcol0 = wcol0 + t0 * rp; jb.r = r; jb.rp = rp; jb.nt = ntw;
        jb.scale = scale; jb.out = out + (size_t)t0 * out_target_stride; jb.out_group_stride = out_group_stride; jb.out_target_stride = out_target_stride;
        jb.out_sj = out_sj; jb.out_sc = out_sc;
        size_t off;
        cudaError_t e = lora_grad_tc_layers(&jb, 1, 1, M, rows_per_group, partial, (size_t)-1, status, &cpg, &off, st);
        if (e != cudaSuccess) return e;
        if (cpg > 1) launch_reduce(partial, r, Rw, C, cpg, groups, scale, out + (size_t)t0 * out_target_stride, out_group_stride,
                      out_target_stride, out_sj, out_sc, st);
      }
      return cudaGetLastError();
    }
  }
  const int R = nt * r;
  const int rpg = rows_per_group > 0 ? rows_per_group : M;
  const int n = dt == DT_BF16 ? 8 : 4;
  const int chunks = (M + LG_ROWS - 1) / LG_ROWS;
  int chunks_per_group, groups;
  if (rpg >= M) { groups = 1; chunks_per_group = chunks; }
  else {
    if (rpg % LG_ROWS != 0 || M % rpg != 0) return cudaErrorInvalidValue;   // chunks must not straddle groups
    groups = M / rpg; chunks_per_group = rpg / LG_ROWS;
  }
  if (C % n != 0 || R < 1) return cudaErrorInvalidValue;
  // vector loads of four adjacent weights need r % 4 == 0 and aligned rows / column offsets
  const bool vec4 = (r % 4 == 0) && (wcol0 % 4 == 0) && (rp % 4 == 0) && (ldwt % 4 == 0);
  const int cvec = C / n;
  dim3 grid((cvec + LG_CT - 1) / LG_CT, chunks, (R + RJ - 1) / RJ);
  if (dt == DT_BF16) launch_partial<bf16>(grid, st, vec4, Z, ldz, zcol0, C, Wt, ldwt, wcol0, r, rp, R, M, partial);
  else launch_partial<float>(grid, st, vec4, Z, ldz, zcol0, C, Wt, ldwt, wcol0, r, rp, R, M, partial);
  launch_reduce(partial, r, R, C, chunks_per_group, groups, scale, out, out_group_stride, out_target_stride, out_sj,
                out_sc, st);
  return cudaGetLastError();
}

bool lora_grad_layers_supported(int dt, const LoraGradJob* jobs, int njobs, int layers, int M, int rows_per_group, bool use_tc) {
  if (njobs < 1 || njobs > LORA_GRAD_MAX_JOBS || layers < 1) return false;
  const int groups = rows_per_group > 0 && rows_per_group < M ? M / rows_per_group : 1;
  int64_t rows = 0;
  for (int j = 0; j < njobs; ++j) {
    const LoraGradJob& jb = jobs[j];
    rows += jb.nt * jb.r;
    if (dt == DT_BF16) {
      if (!use_tc || !lora_grad_tc_supported(dt, jb.Z, jb.ldz, jb.zcol0, jb.C, jb.Wt, jb.ldwt, jb.wcol0, jb.r, jb.rp, jb.nt, M, rows_per_group))
        return false;
    } else if (jb.C % 4 != 0 || jb.ldz % 4 != 0 || jb.zcol0 % 4 != 0 || jb.z_ls % 4 != 0 || jb.C != jobs[0].C || M % groups != 0) {
      return false;
    }
  }
  return (int64_t)layers * rows <= 65535;                   // the grid's third dimension
}

cudaError_t lora_grad_layers(int dt, const LoraGradJob* jobs, int njobs, int layers, int M, int rows_per_group, float* partial,
                             size_t partial_floats, cudaStream_t st, int* status, bool use_tc) {
  if (!lora_grad_layers_supported(dt, jobs, njobs, layers, M, rows_per_group, use_tc)) return cudaErrorInvalidValue;
  const int groups = rows_per_group > 0 && rows_per_group < M ? M / rows_per_group : 1;
  size_t offs[LORA_GRAD_MAX_JOBS];
  int cpg = 0;
  if (dt == DT_BF16) {
    cudaError_t e = lora_grad_tc_layers(jobs, njobs, layers, M, rows_per_group, partial, partial_floats, status, &cpg, offs, st);
    if (e != cudaSuccess || cpg == 1) return e;
    return launch_reduce_batch(jobs, njobs, layers, groups, cpg, partial, offs, st);
  }
  LayersBatch b;
  b.njobs = njobs; b.M = M; b.rows_per_group = M / groups;
  size_t set_floats = 0;
  b.jtiles = 0;
  for (int j = 0; j < njobs; ++j) set_floats += (size_t)layers * groups * jobs[j].nt * jobs[j].r * jobs[j].C;
  cpg = (b.rows_per_group + LL_ROWS - 1) / LL_ROWS;
  if ((size_t)cpg > partial_floats / set_floats) cpg = partial_floats / set_floats > 1 ? (int)(partial_floats / set_floats) : 1;
  b.chunk_rows = (b.rows_per_group + cpg - 1) / cpg;
  b.chunks = cpg;
  size_t off = 0;
  for (int j = 0; j < LORA_GRAD_MAX_JOBS; ++j) {
    const LoraGradJob& jb = jobs[j < njobs ? j : 0];
    const int R = jb.nt * jb.r;
    b.j[j] = {(const float*)jb.Z + jb.zcol0, (const float*)jb.Wt + jb.wcol0, jb.ldz, jb.z_ls, jb.ldwt, jb.wt_ls, jb.r, jb.rp, R, jb.C, b.jtiles,
              cpg > 1 ? partial + off : nullptr, jb.out, jb.out_ls, jb.out_group_stride, jb.out_target_stride, jb.out_sj, jb.out_sc, jb.scale};
    if (j >= njobs) continue;
    offs[j] = off;
    off += (size_t)layers * groups * cpg * R * jb.C;
    b.jtiles += (R + RJ - 1) / RJ;
  }
  const dim3 grid((jobs[0].C / 4 + LL_CT - 1) / LL_CT, groups * cpg, layers * b.jtiles);
  launch_overlapped(lora_grad_layers_kernel, grid, dim3(LL_CT, LL_RL), 0, st, b);
  if (cpg == 1) return cudaGetLastError();
  return launch_reduce_batch(jobs, njobs, layers, groups, cpg, partial, offs, st);
}

cudaError_t lora_grad_batch(int dt, const LoraGradJob* jobs, int njobs, int M, int rows_per_group, float* partial,
                            size_t partial_floats, cudaStream_t st, int* status, bool use_tc) {
  if (dt == DT_BF16 && status && lora_grad_layers_supported(dt, jobs, njobs, 1, M, rows_per_group, use_tc))
    return lora_grad_layers(dt, jobs, njobs, 1, M, rows_per_group, partial, partial_floats, st, status, use_tc);
  for (int j = 0; j < njobs; ++j) {
    const LoraGradJob& jb = jobs[j];
    cudaError_t e = lora_grad(dt, jb.Z, jb.ldz, jb.zcol0, jb.C, jb.Wt, jb.ldwt, jb.wcol0, jb.r, jb.rp, jb.nt, M, rows_per_group,
                              jb.scale, jb.out, jb.out_group_stride, jb.out_target_stride, jb.out_sj, jb.out_sc, partial, st,
                              status, use_tc);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace sl
