// Stand-alone operator entry points of the C ABI: the grouped LoRA linear layer (forward and
// backward), transposes, raw-buffer aggregation and attention.  Used by kernel-level parity tests
// and by the micro-benchmark sweeps.  Host code only.
#include <cuda_runtime.h>

#include "../../include/splitlora.h"
#include "host_common.h"
#include "kernels.h"
#include "launch.cuh"

using namespace sl;

namespace {
inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

struct LinearPlan {
  int rp, ext;
  size_t off_acat, off_acatT, off_bext, off_bextT, off_h, off_dh, off_scratch, total, scratch_floats;
};

LinearPlan plan_linear(int dtype, int M, int n_in, int n_out, int r, int G) {
  LinearPlan p;
  const size_t es = dtype_size(dtype);
  p.rp = (int)align_up((size_t)r, 16);
  p.ext = (int)align_up((size_t)p.rp, EXT_BLOCK);
  size_t off = 0;
  auto take = [&](size_t bytes) { off = align_up(off, 256); size_t o = off; off += bytes; return o; };
  p.off_acat = take((size_t)G * p.ext * n_in * es);
  p.off_acatT = take((size_t)G * n_in * p.ext * es);
  p.off_bext = take((size_t)G * n_out * p.ext * es);
  p.off_bextT = take((size_t)G * p.ext * n_out * es);
  p.off_h = take((size_t)M * p.ext * es);
  p.off_dh = take((size_t)M * p.ext * es);
  // at least two chunks per group of the wider reduction: dA and dB as one batch
  size_t sc = lora_grad_scratch_floats(M > 256 * G ? M : 256 * G, r, n_in > n_out ? n_in : n_out);
  p.scratch_floats = sc;
  p.off_scratch = take(sc * 4);
  p.total = align_up(off, 256);
  return p;
}

int check_linear(int dtype, int M, int n_in, int n_out, int r, int G) {
  if (dtype != DT_F32 && dtype != DT_BF16) return SPLITLORA_ERR_ARG;
  if (M < 1 || n_in < 8 || n_out < 8 || r < 1 || r > 64 || G < 1 || M % G != 0) return SPLITLORA_ERR_ARG;
  if (n_in % 8 != 0 || n_out % 8 != 0) return SPLITLORA_ERR_ARG;
  if (G > 1 && (M / G) % 128 != 0) return SPLITLORA_ERR_ARG;
  return SPLITLORA_OK;
}

cudaError_t run_gemm(int use_tc, const GemmArgs& a, int* status, cudaStream_t st) {
  if (use_tc && a.dtype == DT_BF16 && gemm_tc_supported(a)) return gemm_tc(a, status, st);
  return gemm_simt(a, st);
}
ProjArgs proj_args(const LinearPlan& p, const void* X, int K, const void* W, void* Y, int M, int r, int G, int* status) {
  ProjArgs a;
  a.X = X; a.ldx = K; a.W = W; a.ldw = K; a.w_group_stride = G > 1 ? (int64_t)p.ext * K : 0; a.Y = Y;
  a.M = M; a.K = K; a.rows_per_group = G > 1 ? M / G : 0; a.ext = p.ext; a.r = r; a.rp = p.rp;
  a.status = status;
  return a;
}
// Y[M, ext] = X[M, K] W_g[ext, K]^T of the LoRA layer with plan p
cudaError_t run_proj(int use_tc, int dtype, const LinearPlan& p, const void* X, int K, const void* W, void* Y, int M, int r, int G,
                     int* status, cudaStream_t st) {
  const ProjArgs a = proj_args(p, X, K, W, Y, M, r, G, status);
  if (use_tc && dtype == DT_BF16 && M <= LORA_PROJ_ROWS && lora_proj_supported(a)) return lora_proj(a, st);
  GemmArgs h;
  h.dtype = dtype; h.X = X; h.ldx = K; h.W = W; h.ldw = K; h.Y = Y; h.ldy = p.ext;
  h.M = M; h.N = p.ext; h.K = K; h.rows_per_group = a.rows_per_group; h.w_grouped = G > 1;
  return run_gemm(use_tc, h, status, st);
}
}  // namespace

extern "C" {

int splitlora_lora_linear_workspace_bytes(int dtype, int M, int n_in, int n_out, int r, int G, size_t* bytes) {
  if (!bytes) return SPLITLORA_ERR_ARG;
  int rc = check_linear(dtype, M, n_in, n_out, r, G);
  if (rc) return rc;
  *bytes = plan_linear(dtype, M, n_in, n_out, r, G).total;
  return SPLITLORA_OK;
}

// The layer's kernels report an expired wait to the library's word, which no launch clears: a word of the workspace would
// have to be cleared first, and the first launch of a call (copies and projection) already has workers that may report to it.

// The compute copies of one direction: Acat and Bext (forward), Acat, AcatT and BextT (backward).
static AdapterCopyArgs copy_args(int dtype, const LinearPlan& p, const float* A, const float* B, float alpha, int n_in,
                                 int n_out, int r, int G, char* ws, bool fwd) {
  AdapterCopyArgs a;
  a.dtype = dtype;
  a.A = A; a.a_gs = (int64_t)r * n_in; a.a_ts = 0;
  a.B = B; a.b_gs = (int64_t)n_out * r; a.b_ts = 0;
  a.G = G; a.n_targets = 1; a.r = r; a.rp = p.rp; a.d_in = n_in; a.d_out = n_out; a.n_out = n_out; a.ext = p.ext;
  a.scale = alpha / (float)r;
  a.Acat = ws + p.off_acat; a.AcatT = fwd ? nullptr : ws + p.off_acatT;
  a.Bext = fwd ? ws + p.off_bext : nullptr; a.BextT = fwd ? nullptr : ws + p.off_bextT;
  return a;
}
// The copies, and h = x A_g^T where `project`: one launch where the projection can take A as it is, else two.
static cudaError_t copies_and_h(int use_tc, AdapterCopyArgs a, bool project, const LinearPlan& p, const void* x, int M, char* ws, int* status, cudaStream_t st) {
  // (16384 rows: 16.5 us as one launch, 10.6 + 4.8 as two)
  if (project && use_tc && M <= LORA_PROJ_ROWS && a.dtype == DT_BF16 && (reinterpret_cast<uintptr_t>(a.A) & 15u) == 0) {
    ProjArgs h = proj_args(p, x, a.d_in, a.A, ws + p.off_h, M, a.r, a.G, status);
    if (a.G > 1) h.w_group_stride = a.a_gs;
    if (lora_proj_supported(h)) {
      a.Acat = nullptr;                        // nothing else reads it
      return lora_proj_copies(h, a, st);
    }
  }
  cudaError_t e = write_adapter_copies(a, st);
  if (e != cudaSuccess || !project) return e;
  return run_proj(use_tc, a.dtype, p, x, a.d_in, ws + p.off_acat, ws + p.off_h, M, a.r, a.G, status, st);
}

int splitlora_lora_linear_fwd(int dtype, int use_tc, const void* x, const void* W, const void* bias, const float* A,
                              const float* B, float alpha, int M, int n_in, int n_out, int r, int G, void* y,
                              void* workspace, size_t workspace_bytes, void* stream) {
  LaunchChain chain;
  return splitlora_lora_linear_fwd_parts(dtype, use_tc, x, W, bias, A, B, alpha, M, n_in, n_out, r, G, y, workspace,
                                         workspace_bytes, stream, 3);
}

int splitlora_lora_linear_fwd_parts(int dtype, int use_tc, const void* x, const void* W, const void* bias, const float* A,
                                    const float* B, float alpha, int M, int n_in, int n_out, int r, int G, void* y,
                                    void* workspace, size_t workspace_bytes, void* stream, int parts) {
  LaunchChain chain;
  int rc = check_linear(dtype, M, n_in, n_out, r, G);
  if (rc) return rc;
  if (parts < 1 || parts > 3) return SPLITLORA_ERR_ARG;
  if (!x || !W || !A || !B || !y || !workspace) return SPLITLORA_ERR_ARG;
  if (!aligned16(x) || !aligned16(W) || !aligned16(y) || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return SPLITLORA_ERR_ALIGN;
  LinearPlan p = plan_linear(dtype, M, n_in, n_out, r, G);
  if (workspace_bytes < p.total) return SPLITLORA_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  int* status = library_status_word();
  if (gemm_tc_init() != 0 || !status) return SPLITLORA_ERR_CUDA;
  const int rpg = G > 1 ? M / G : 0;
  if (parts & 1) {
    if (copies_and_h(use_tc, copy_args(dtype, p, A, B, alpha, n_in, n_out, r, G, ws, true), true, p, x, M, ws, status, st) != cudaSuccess) return SPLITLORA_ERR_CUDA;
  }
  if (!(parts & 2)) return SPLITLORA_OK;
  GemmArgs a;
  a.dtype = dtype; a.X = x; a.ldx = n_in; a.W = W; a.ldw = n_in; a.Y = y; a.ldy = n_out;
  a.M = M; a.N = n_out; a.K = n_in; a.bias = bias; a.rows_per_group = rpg;
  a.Xe = ws + p.off_h; a.ldxe = p.ext; a.We = ws + p.off_bext; a.ldwe = p.ext; a.Ke = p.rp; a.we_grouped = G > 1;
  if (run_gemm(use_tc, a, status, st) != cudaSuccess) return SPLITLORA_ERR_CUDA;
  return SPLITLORA_OK;
}

int splitlora_lora_linear_bwd(int dtype, int use_tc, const void* x, const void* Wt, const void* dy, const float* A,
                              const float* B, float alpha, int M, int n_in, int n_out, int r, int G, void* dx,
                              float* dA, float* dB, void* workspace, size_t workspace_bytes, void* stream) {
  LaunchChain chain;
  return splitlora_lora_linear_bwd_parts(dtype, use_tc, x, Wt, dy, A, B, alpha, M, n_in, n_out, r, G, dx, dA, dB, workspace,
                                         workspace_bytes, stream, 7);
}

int splitlora_lora_linear_bwd_parts(int dtype, int use_tc, const void* x, const void* Wt, const void* dy, const float* A,
                                    const float* B, float alpha, int M, int n_in, int n_out, int r, int G, void* dx,
                                    float* dA, float* dB, void* workspace, size_t workspace_bytes, void* stream, int parts) {
  LaunchChain chain;
  int rc = check_linear(dtype, M, n_in, n_out, r, G);
  if (rc) return rc;
  if (parts < 1 || parts > 7) return SPLITLORA_ERR_ARG;
  if (!x || !Wt || !dy || !A || !B || !dx || !dA || !dB || !workspace) return SPLITLORA_ERR_ARG;
  if (!aligned16(x) || !aligned16(Wt) || !aligned16(dy) || !aligned16(dx) || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return SPLITLORA_ERR_ALIGN;
  LinearPlan p = plan_linear(dtype, M, n_in, n_out, r, G);
  if (workspace_bytes < p.total) return SPLITLORA_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  int* status = library_status_word();
  if (gemm_tc_init() != 0 || !status) return SPLITLORA_ERR_CUDA;
  // h = x A_g^T is recomputed here; the training runtime keeps it from the forward pass
  if (copies_and_h(use_tc, copy_args(dtype, p, A, B, alpha, n_in, n_out, r, G, ws, false), parts & 1, p, x, M, ws, status, st) != cudaSuccess) return SPLITLORA_ERR_CUDA;
  const int rpg = G > 1 ? M / G : 0;
  const float s = alpha / (float)r;
  if (parts & 1) {
    // dh = s dy B_g
    if (run_proj(use_tc, dtype, p, dy, n_out, ws + p.off_bextT, ws + p.off_dh, M, r, G, status, st) != cudaSuccess) return SPLITLORA_ERR_CUDA;
  }
  if (parts & 2) {
    // dx = dy W + dh A_g
    GemmArgs a;
    a.dtype = dtype; a.X = dy; a.ldx = n_out; a.W = Wt; a.ldw = n_out; a.Y = dx; a.ldy = n_in;
    a.M = M; a.N = n_in; a.K = n_out; a.rows_per_group = rpg;
    a.Xe = ws + p.off_dh; a.ldxe = p.ext; a.We = ws + p.off_acatT; a.ldwe = p.ext; a.Ke = p.rp; a.we_grouped = G > 1;
    if (run_gemm(use_tc, a, status, st) != cudaSuccess) return SPLITLORA_ERR_CUDA;
  }
  if (!(parts & 4)) return SPLITLORA_OK;
  // dA = dh^T x and dB = s dy^T h: one pair of launches where the tensor-core path applies
  LoraGradJob jobs[2];
  LoraGradJob &ja = jobs[0], &jb = jobs[1];
  ja.Z = x; ja.ldz = n_in; ja.C = n_in; ja.Wt = ws + p.off_dh; ja.scale = 1.0f; ja.out = dA; ja.out_group_stride = (int64_t)r * n_in;
  ja.out_sj = n_in; ja.out_sc = 1;
  jb.Z = dy; jb.ldz = n_out; jb.C = n_out; jb.Wt = ws + p.off_h; jb.scale = s; jb.out = dB; jb.out_group_stride = (int64_t)n_out * r;
  jb.out_sj = 1; jb.out_sc = r;
  for (LoraGradJob& j : jobs) { j.ldwt = p.ext; j.r = r; j.rp = p.rp; j.nt = 1; }
  if (lora_grad_batch(dtype, jobs, 2, M, rpg, (float*)(ws + p.off_scratch), p.scratch_floats, st, status, use_tc != 0) != cudaSuccess)
    return SPLITLORA_ERR_CUDA;
  return SPLITLORA_OK;
}

int splitlora_library_status(int32_t* code) {
  if (!code) return SPLITLORA_ERR_ARG;
  int* word = library_status_word();
  if (!word) return SPLITLORA_ERR_CUDA;
  if (cudaDeviceSynchronize() != cudaSuccess) return SPLITLORA_ERR_CUDA;
  if (cudaMemcpy(code, word, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SPLITLORA_ERR_CUDA;
  return *code ? SPLITLORA_ERR_TIMEOUT : SPLITLORA_OK;
}

int splitlora_transpose(int dtype, const void* in, int rows, int cols, void* out, void* stream) {
  LaunchChain chain;
  if (!in || !out || rows < 1 || cols < 1 || (dtype != DT_F32 && dtype != DT_BF16)) return SPLITLORA_ERR_ARG;
  return transpose(dtype, in, rows, cols, out, rows, (cudaStream_t)stream) == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}

int splitlora_handoff_quantize(int dtype, const void* x, int64_t M, int d, uint8_t* codes, float* scales, void* stream) {
  LaunchChain chain;
  const int n = dtype == DT_BF16 ? 8 : 4;
  if (!x || !codes || !scales || M < 1 || d < n || d % n != 0 || (dtype != DT_F32 && dtype != DT_BF16)) return SPLITLORA_ERR_ARG;
  if (!aligned16(x) || !aligned16(codes)) return SPLITLORA_ERR_ALIGN;
  return handoff_quantize(dtype, x, M, d, codes, scales, (cudaStream_t)stream) == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}

int splitlora_handoff_dequantize(int dtype, const uint8_t* codes, const float* scales, int64_t M, int d, void* y,
                                 void* stream) {
  LaunchChain chain;
  const int n = dtype == DT_BF16 ? 8 : 4;
  if (!y || !codes || !scales || M < 1 || d < n || d % n != 0 || (dtype != DT_F32 && dtype != DT_BF16)) return SPLITLORA_ERR_ARG;
  if (!aligned16(y) || !aligned16(codes)) return SPLITLORA_ERR_ALIGN;
  return handoff_dequantize(dtype, codes, scales, M, d, y, (cudaStream_t)stream) == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}

int splitlora_aggregate_buffers(float* params, int K, int64_t P, const double* weights, void* stream) {
  LaunchChain chain;
  if (!params || !weights || K < 1 || K > AGG_MAX_CLIENTS || P < 4 || P % 4 != 0) return SPLITLORA_ERR_ARG;
  if (!aligned16(params)) return SPLITLORA_ERR_ALIGN;
  float w[AGG_MAX_CLIENTS];
  for (int i = 0; i < K; ++i) w[i] = (float)weights[i];
  return aggregate(params, K, P, w, (cudaStream_t)stream) == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}

int splitlora_attention_fwd(int dtype, int use_tc, const void* qkv, int nseq, int T, int n_head, int d_model, void* o,
                            float* lse, void* stream) {
  LaunchChain chain;
  if (!qkv || !o || !lse || nseq < 1 || T < 1 || n_head < 1 || d_model % n_head != 0 || d_model / n_head > 128 ||
      (dtype != DT_F32 && dtype != DT_BF16))
    return SPLITLORA_ERR_ARG;
  cudaError_t e;
  if (use_tc && attention_tc_supported(dtype, T, n_head, d_model))
    e = attention_fwd_tc(qkv, nseq, T, n_head, d_model, o, lse, nullptr, (cudaStream_t)stream);
  else if (use_tc && attention_ragged_supported(dtype, nseq, T, n_head, d_model, qkv, o, nullptr, nullptr))
    e = attention_fwd_ragged(qkv, nseq, T, n_head, d_model, o, lse, nullptr, (cudaStream_t)stream);
  else
    e = attention_fwd_simt(dtype, qkv, nseq, T, n_head, d_model, o, lse, (cudaStream_t)stream);
  return e == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}

int splitlora_attention_bwd(int dtype, int use_tc, const void* qkv, const void* o, const float* lse, const void* d_o,
                            int nseq, int T, int n_head, int d_model, void* dqkv, float* rowdot, void* stream) {
  LaunchChain chain;
  if (!qkv || !o || !lse || !d_o || !dqkv || !rowdot || nseq < 1 || T < 1 || n_head < 1 || d_model % n_head != 0 ||
      d_model / n_head > 128 || (dtype != DT_F32 && dtype != DT_BF16))
    return SPLITLORA_ERR_ARG;
  cudaError_t e;
  if (use_tc && attention_tc_supported(dtype, T, n_head, d_model))
    e = attention_bwd_tc(qkv, o, lse, d_o, nseq, T, n_head, d_model, dqkv, rowdot, nullptr, (cudaStream_t)stream);
  else if (use_tc && attention_ragged_supported(dtype, nseq, T, n_head, d_model, qkv, o, d_o, dqkv))
    e = attention_bwd_ragged(qkv, o, lse, d_o, nseq, T, n_head, d_model, dqkv, rowdot, nullptr, (cudaStream_t)stream);
  else
    e = attention_bwd_simt(dtype, qkv, o, lse, d_o, nseq, T, n_head, d_model, dqkv, rowdot, (cudaStream_t)stream);
  return e == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}

}  // extern "C"

// Frozen linear layer with a fused epilogue (steps a4 / a11), stand-alone.
extern "C" int splitlora_linear(int dtype, int use_tc, const void* x, const void* W, const void* bias, int epilogue,
                                const void* r, void* z, int gelu_tanh, int M, int n_in, int n_out, void* y,
                                int* status_word, void* stream) {
  LaunchChain chain;
  if (!x || !W || !y || M < 1 || n_in < 8 || n_out < 8 || n_in % 8 || n_out % 8 || (dtype != DT_F32 && dtype != DT_BF16))
    return SPLITLORA_ERR_ARG;
  if (epilogue < EPI_BIAS || epilogue > EPI_MUL_GELUGRAD) return SPLITLORA_ERR_ARG;
  if ((epilogue == EPI_BIAS_RESID || epilogue == EPI_MUL_GELUGRAD) && !r) return SPLITLORA_ERR_ARG;
  if (epilogue == EPI_BIAS_GELU && !z) return SPLITLORA_ERR_ARG;
  if (use_tc && dtype == DT_BF16 && !status_word) return SPLITLORA_ERR_ARG;
  if (gemm_tc_init() != 0) return SPLITLORA_ERR_CUDA;
  GemmArgs a;
  a.dtype = dtype; a.X = x; a.ldx = n_in; a.W = W; a.ldw = n_in; a.Y = y; a.ldy = n_out;
  a.M = M; a.N = n_out; a.K = n_in; a.bias = bias; a.epi = epilogue; a.R = r; a.ldr = n_out; a.Z = z; a.ldz = n_out;
  a.gelu_tanh = gelu_tanh;
  return run_gemm(use_tc, a, status_word, (cudaStream_t)stream) == cudaSuccess ? SPLITLORA_OK : SPLITLORA_ERR_CUDA;
}
