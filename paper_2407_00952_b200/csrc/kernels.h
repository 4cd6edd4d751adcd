// Internal launchers of the split-LoRA kernels.  Host-callable, stream-ordered, no allocation.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace sl {

enum { DT_F32 = 0, DT_BF16 = 1 };
static inline size_t dtype_size(int dt) { return dt == DT_BF16 ? 2 : 4; }

// Epilogues of the linear-layer kernels.
enum Epilogue {
  EPI_BIAS = 0,          // Y = acc + bias
  EPI_BIAS_GELU = 1,     // Z = acc + bias ; Y = gelu(Z)
  EPI_BIAS_RESID = 2,    // Y = acc + bias + R
  EPI_MUL_GELUGRAD = 3   // Y = acc * gelu'(R)           (R holds the saved pre-activation)
};

// Width of one block of the rank-r extension of the contraction (elements).
static const int EXT_BLOCK = 64;

// Y[M,N] = epilogue( X[M,K] W[N,K]^T + Xe[M,Ke] We[N,Ke]^T )
// Rows are split into groups of rows_per_group consecutive rows (0: one group).  A grouped operand
// holds one [N, .] matrix per group, stacked along rows.  The extension term is how the rank-r LoRA
// path enters: Xe is the down-projected activation, We the (scaled) up-projection of the row's group.
struct GemmArgs {
  int dtype = DT_BF16;
  const void* X = nullptr; int64_t ldx = 0;
  const void* W = nullptr; int64_t ldw = 0;
  void* Y = nullptr;       int64_t ldy = 0;
  int M = 0, N = 0, K = 0;
  int w_rows = 0;           // number of valid rows of W (rows >= w_rows read as zero); 0 means N
  int rows_per_group = 0;
  int w_grouped = 0;        // W is [G*N, K]
  const void* bias = nullptr;
  int epi = EPI_BIAS;
  const void* R = nullptr; int64_t ldr = 0;
  void* Z = nullptr;       int64_t ldz = 0;
  int gelu_tanh = 1;
  const void* Xe = nullptr; int64_t ldxe = 0;
  const void* We = nullptr; int64_t ldwe = 0;
  int Ke = 0;               // 0: no extension; else a multiple of 16
  int we_grouped = 0;       // We is [G*N, Ke]
  // Columns [k_gap_begin, k_gap_begin + k_gap_len) of X and W are left out of the contraction (both
  // multiples of 64; K counts the contracted columns only).  Single-CTA tensor-core kernel only.
  int k_gap_begin = 0, k_gap_len = 0;
};

// Plain-FMA tiled kernel, any shape, fp32 or bf16 storage with fp32 accumulation.
cudaError_t gemm_simt(const GemmArgs& a, cudaStream_t st);
// tcgen05 / TMEM / TMA kernel (bf16 only).  Shape rules: any M with one group, else rows_per_group % 128 == 0;
// K % 8 == 0, N % 8 == 0, leading dimensions multiples of 8 elements, 16-byte aligned bases.
// status: device word that receives a non-zero code if a bounded wait expires.
bool gemm_tc_supported(const GemmArgs& a);
cudaError_t gemm_tc(const GemmArgs& a, int* status, cudaStream_t st);
int gemm_tc_init();   // resolves the driver entry point for tensor-map encoding; 0 on success

cudaError_t embed(int dt, const int32_t* tokens, const void* wte, const void* wpe, void* out,
                  int M, int T, int d, int vocab, cudaStream_t st);
cudaError_t layernorm_fwd(int dt, const void* x, const void* g, const void* b, void* y, float* mean,
                          float* rstd, int M, int d, float eps, cudaStream_t st);
// dx = resid + dLN(dy)  (resid may be null); gradient w.r.t. the input only.
cudaError_t layernorm_bwd(int dt, const void* dy, const void* x, const void* g, const float* mean,
                          const float* rstd, const void* resid, void* dx, int M, int d, cudaStream_t st);

// Llama-shaped block pieces.  RMSNorm: y = x * rsqrt(mean(x^2) + eps) * g, saves rstd [M];
// backward gives dx = resid + d/dx (resid may be null).
cudaError_t rmsnorm_fwd(int dt, const void* x, const void* g, void* y, float* rstd, int M, int d, float eps,
                        cudaStream_t st);
cudaError_t rmsnorm_bwd(int dt, const void* dy, const void* x, const void* g, const float* rstd, const void* resid,
                        void* dx, int M, int d, cudaStream_t st);
// Rotates the q and k slices of qkv [M, 3d] in place; table [T, d/H/2] of (cos, sin) pairs as
// float2; sign +1 forward, -1 inverse (= gradient).  Needs d/H/2 to be a multiple of the 16-byte
// vector width.
cudaError_t rope_inplace(int dt, void* qkv, const float* table, int M, int T, int H, int d, float sign,
                         cudaStream_t st);
// z [M, 2F] = (gate | up).  act [M, F] = silu(gate) * up;  dz [M, 2F] from dact [M, F].
cudaError_t swiglu_fwd(int dt, const void* z, void* act, int M, int F, cudaStream_t st);
cudaError_t swiglu_bwd(int dt, const void* dact, const void* z, void* dz, int M, int F, cudaStream_t st);

// Cross-entropy over logits [M, ld] (V valid columns): writes per-row losses, then overwrites the
// logits with d loss / d logits (zero in the pad columns) and reduces the mean loss.
// normalizer_override > 0 replaces the count of valid labels (the batch is a shard of a larger one).
cudaError_t cross_entropy(int dt, void* logits, int64_t ld, const int32_t* labels, int M, int V,
                          float* row_loss, int* n_valid, float* loss, int normalizer_override, cudaStream_t st);

// Attention, fused qkv layout [nseq*T, 3d]; heads are contiguous slices of width d/H.
cudaError_t attention_fwd_simt(int dt, const void* qkv, int nseq, int T, int H, int d, void* o, float* lse,
                               cudaStream_t st);
cudaError_t attention_bwd_simt(int dt, const void* qkv, const void* o, const float* lse, const void* d_o,
                               int nseq, int T, int H, int d, void* dqkv, float* rowdot, cudaStream_t st);
// tcgen05 / TMEM attention (bf16, head width 64, T a multiple of 128).  status: device word for the
// code of an expired bounded wait (nullptr: a word inside the library).
bool attention_t5_supported(int dt, int T, int H, int d);
bool attention_fwd_t5_supported(int dt, int T, int H, int d);
bool attention_bwd_t5_128_supported(int dt, int T, int H, int d);
cudaError_t attention_bwd_t5_128(const void* qkv, const float* lse, const void* d_o, const float* rowdot, int nseq,
                                    int T, int H, int d, void* dqkv, int* status, cudaStream_t st);
// head width 64: one softmax thread per row, half-steps of 64 keys (attention_t5_fwd64.cu)
cudaError_t attention_fwd_t5_h64(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status,
                                 cudaStream_t st);
cudaError_t attention_fwd_t5(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status,
                             cudaStream_t st);
cudaError_t attention_bwd_t5(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                             int d, void* dqkv, float* rowdot, int* status, cudaStream_t st);
bool attention_tc_supported(int dt, int T, int H, int d);
cudaError_t attention_fwd_tc(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status,
                             cudaStream_t st);
cudaError_t attention_bwd_tc(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq,
                             int T, int H, int d, void* dqkv, float* rowdot, int* status, cudaStream_t st);

// Attention for the remaining bf16 shapes: any T, head widths that are multiples of 8; P and dS kept to 16 mantissa
// bits (mma.sync in attention_tc.cu, or the tcgen05 form below by the rules there).  Pointers that a direction does not use may be null.
bool attention_ragged_supported(int dt, int nseq, int T, int H, int d, const void* qkv, const void* o, const void* d_o,
                                const void* dqkv);
cudaError_t attention_fwd_ragged(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status, cudaStream_t st);
cudaError_t attention_bwd_ragged(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                 int d, void* dqkv, float* rowdot, int* status, cudaStream_t st);
// Width 64 on tcgen05 (attention_t5_ragged.cu), any length; status as above.  attention_bwd_t5_w64: P and dS as bf16, for the
// lengths that always held them so.
bool attention_ragged_t5_supported(int nseq, int T, int H, int d);
cudaError_t attention_fwd_ragged_t5(const void* qkv, int nseq, int T, int H, int d, void* o, float* lse, int* status, cudaStream_t st);
cudaError_t attention_bwd_t5_w64(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                 int d, void* dqkv, float* rowdot, int* status, cudaStream_t st);
cudaError_t attention_bwd_ragged_t5(const void* qkv, const void* o, const float* lse, const void* d_o, int nseq, int T, int H,
                                    int d, void* dqkv, float* rowdot, int* status, cudaStream_t st);

// Compute copies of the adapters of `layers` layers (G groups), built from fp32 masters.
// Target t of group g has A_t [r, d_in] at A + g*a_gs + t*a_ts and B_t [d_out, r] at B + g*b_gs + t*b_ts.
// With col = t*rp + j the copies are
//   Acat  [G][ext, d_in]  : Acat[col, c]  = A_t[j, c]          AcatT [G][d_in, ext] : its transpose
//   Bext  [G][n_out, ext] : Bext[slice_off[t] + c, col] = scale * B_t[c, j]
//   BextT [G][ext, n_out] : its transpose
// Only live entries are written; the padding must have been zeroed once.
struct AdapterCopyArgs {
  int dtype = 0;
  const float* A = nullptr; int64_t a_gs = 0, a_ts = 0;
  const float* B = nullptr; int64_t b_gs = 0, b_ts = 0;
  int G = 0, n_targets = 0, r = 0, rp = 0, d_in = 0, d_out = 0, n_out = 0, ext = 0;
  int slice_off[4] = {0, 0, 0, 0};
  float scale = 0.f;
  void *Acat = nullptr, *AcatT = nullptr, *Bext = nullptr, *BextT = nullptr;   // any of them may be null (skipped)
  int layers = 1;                      // of layers further on: masters layer_stride, Acat / AcatT acat_ls, Bext / BextT bext_ls elements apart
  int64_t layer_stride = 0, acat_ls = 0, bext_ls = 0;
};
// Rank-r projection of the LoRA path, bf16 (lora_proj.cu): Y[M, ext] = X[M, K] W_g[ext, K]^T where only columns
// t*rp + j, j < r, t < nt of W and Y are used (the others of Y become zero).  W of group g = row / rows_per_group at
// W + g*w_group_stride.  k_slice > 0 and nt > 1: target t's rows of W are zero outside columns [slice_col[t], + k_slice), and
// K is not used.  status: as for the linear layers (nullptr: the library's own word).
struct ProjArgs {
  const void* X = nullptr; int64_t ldx = 0;
  const void* W = nullptr; int64_t ldw = 0, w_group_stride = 0;
  void* Y = nullptr;
  int M = 0, K = 0, rows_per_group = 0, ext = 0, nt = 1, r = 0, rp = 0, k_slice = 0, slice_col[4] = {0, 0, 0, 0};
  int* status = nullptr;
};
bool lora_proj_supported(const ProjArgs& a);
// Rows up to which these kernels beat the linear layers' narrow tiles: (512, 2048 -> 2 x 4 of 32) 8.8 -> 5.5 us from cold
// caches; 12 of 1665 x 1536 149 -> 104, of 16384 x 1536 225 -> 252, 24 of 32768 x 2048 910 -> 966.
constexpr int LORA_PROJ_ROWS = 4096;
cudaError_t lora_proj(const ProjArgs& a, cudaStream_t st);
// The same for one target whose W is the fp32 A [r, K] itself, with the compute copies of write_adapter_copies in the same launch.
cudaError_t lora_proj_copies(const ProjArgs& a, const AdapterCopyArgs& copies, cudaStream_t st);
// The norm in front of it in the same launch: a.X [M, K] receives LayerNorm(x) (RMSNorm: b and mean unused), Y its projection.
bool norm_proj_supported(const ProjArgs& a);
// Whether that pays: it saves a launch and a read of the rows, but two launches overlap, which weighs more where the rows are many
// and wide.  Rounds of 4 blocks, apart -> together, us: width 256, 5120 rows 599 -> 587, 16384 1012 -> 996; 512, 5120 891 -> 874,
// 12288 1475 -> 1463, 16384 1814 -> 1818; 768, 5120 1119 -> 1115, 8192 equal, 12288 2211 -> 2219, 16384 2945 -> 2962; 1024, 8192 equal,
// 12288 3372 -> 3385, 16384 4397 -> 4417; 24 blocks of 512 x 1024 3068 -> 3058, 12 of 1665 x 768 2285 -> 2264.
constexpr int NORM_PROJ_ROWS = 16384;
inline bool norm_proj_pays(int M, int d) { return M <= NORM_PROJ_ROWS && (int64_t)M * d <= 8 << 20; }
// the same in fp32, LayerNorm only
bool norm_proj_f32_supported(const ProjArgs& a);
cudaError_t norm_proj_f32(const void* x, const void* g, const void* b, float* mean, float* rstd, float eps, const ProjArgs& a, cudaStream_t st);
cudaError_t norm_proj(bool rms, const void* x, const void* g, const void* b, float* mean, float* rstd, float eps, const ProjArgs& a, cudaStream_t st);

// Adapter gradients: for nt targets of rank r (weight columns wcol0 + t*rp + jj of Wt),
//   out[g][t][jj][c] = scale * sum_{m in group g} Wt[m, wcol0 + t*rp + jj] * Z[m, zcol0 + c],  c < C,
// stored at out + g*out_group_stride + t*out_target_stride + jj*out_sj + c*out_sc.
// rows_per_group must be a multiple of 128 unless there is one group (0, or >= M).  partial: scratch of at least
// lora_grad_scratch_floats(M, nt*r, C) floats.
size_t lora_grad_scratch_floats(int M, int R, int C);
cudaError_t lora_grad(int dt, const void* Z, int64_t ldz, int zcol0, int C, const void* Wt, int64_t ldwt,
                      int wcol0, int r, int rp, int nt, int M, int rows_per_group, float scale, float* out,
                      int64_t out_group_stride, int64_t out_target_stride, int64_t out_sj, int64_t out_sc,
                      float* partial, cudaStream_t st, int* status = nullptr, bool use_tc = false);
// One reduction of lora_grad as a record, for lora_grad_batch: several of them over the same token rows
// (the adapter gradients of one layer) in one pair of launches.
struct LoraGradJob {
  const void* Z = nullptr; int64_t ldz = 0; int zcol0 = 0, C = 0;
  const void* Wt = nullptr; int64_t ldwt = 0; int wcol0 = 0, r = 0, rp = 0, nt = 1;
  float scale = 1.f; float* out = nullptr;
  int64_t out_group_stride = 0, out_target_stride = 0, out_sj = 0, out_sc = 0;
  int64_t z_ls = 0, wt_ls = 0, out_ls = 0;     // lora_grad_layers: elements between two layers
};
// Up to LORA_GRAD_MAX_JOBS reductions of each of `layers` layers at once (the adapter gradients of a side of the model), all
// with the same C: one launch, or two where the rows of a group are split.  Whether the shapes are taken:
constexpr int LORA_GRAD_MAX_JOBS = 6;
bool lora_grad_layers_supported(int dt, const LoraGradJob* jobs, int njobs, int layers, int M, int rows_per_group, bool use_tc);
cudaError_t lora_grad_layers(int dt, const LoraGradJob* jobs, int njobs, int layers, int M, int rows_per_group, float* partial,
                             size_t partial_floats, cudaStream_t st, int* status, bool use_tc);
// its tcgen05 form: partials of chunks > 1 as [job][layer][chunk][R_j][C], results directly where a group is one chunk
cudaError_t lora_grad_tc_layers(const LoraGradJob* jobs, int njobs, int layers, int M, int rows_per_group, float* partial,
                                size_t partial_floats, int* status, int* chunks_per_group, size_t* offsets, cudaStream_t st);
// partial: scratch of partial_floats floats.  Falls back to one lora_grad per job where the batched
// tensor-core path does not apply.
cudaError_t lora_grad_batch(int dt, const LoraGradJob* jobs, int njobs, int M, int rows_per_group, float* partial,
                            size_t partial_floats, cudaStream_t st, int* status, bool use_tc);
// The reduction as a tcgen05 product with both operands MN-major takes bf16, rp in {16, 32, 64}, ldwt a multiple of 64 and
// the wanted weight columns inside one 64-column tile.  status: device word for an expired bounded wait.
bool lora_grad_tc_supported(int dt, const void* Z, int64_t ldz, int zcol0, int C, const void* Wt, int64_t ldwt,
                            int wcol0, int r, int rp, int nt, int M, int rows_per_group);

struct OptArgs {
  int optimizer; float lr, beta1, beta2, eps, wd; float bc1, bc2;   // bc = 1 - beta^step
};
cudaError_t optimizer_step(float* p, const float* g, float* m, float* v, int64_t n, const OptArgs& o,
                           cudaStream_t st);

// Eq. 8-9 and the write-back: every row of params [K, P] becomes sum_i w[i] params[i, :].
static const int AGG_MAX_CLIENTS = 64;
// zero rank components >= ranks_host[i] in client i's arena of (A [r, d], B [d, r]) pairs (P floats per client)
cudaError_t rank_mask(float* params, int K, int64_t P, int r, int d, const int* ranks_host, cudaStream_t st);
// row_stride: floats between two clients' rows (0: P), so that a column range of a wider arena can be averaged
cudaError_t aggregate(float* params, int K, int64_t P, const float* w_host, cudaStream_t st, int64_t row_stride = 0);
// The same step in two halves, for clients spread over devices: sum [P] = sum_i w[i] params[i, :], and
// (after the caller has added the sums of all devices) every row of params [K, P] = sum.
cudaError_t aggregate_local_sum(const float* params, int K, int64_t P, const float* w_host, float* sum, cudaStream_t st);
cudaError_t aggregate_broadcast(const float* sum, int K, int64_t P, float* params, cudaStream_t st);

// The same for one layer and target (n_targets 1, slice_off 0, n_out = d_out) into uninitialised copies: padding included.
cudaError_t write_adapter_copies(const AdapterCopyArgs& a, cudaStream_t st);
cudaError_t refresh_adapter_copies(const AdapterCopyArgs& a, cudaStream_t st);

cudaError_t transpose(int dt, const void* in, int rows, int cols, void* out, int64_t ldo, cudaStream_t st);
// compressed hand-off (handoff.cu): rows of d values <-> d E4M3 codes + one fp32 scale
cudaError_t handoff_quantize(int dt, const void* x, int64_t M, int d, uint8_t* codes, float* scales, cudaStream_t st);
cudaError_t handoff_dequantize(int dt, const uint8_t* codes, const float* scales, int64_t M, int d, void* y,
                               cudaStream_t st);

}  // namespace sl
