// Internal launch functions of the CUDA kernels.  All of them only enqueue work on `stream`.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>

#include "../../include/xema.h"

namespace xema {

// Records cudaGetLastError(); returns XEMA_OK or XEMA_ECUDA.
int check_launch();
void set_last_cuda_error(int code);

// One-time launch state (function attributes, SM counts, cluster occupancy) belongs to a device,
// not to the process: these caches are indexed by the current device's ordinal and filled with
// atomic stores, so several host threads, or one process that drives several GPUs, see a
// value only after it was established on that device.  0 means "not known yet".  Ordinals at or
// beyond kMaxDevices are never cached (the value is looked up again on every call).
constexpr int kMaxDevices = 64;
struct PerDeviceInt {
  std::atomic<int> v[kMaxDevices];
  int get(int dev) const { return (dev >= 0 && dev < kMaxDevices) ? v[dev].load(std::memory_order_acquire) : 0; }
  void set(int dev, int value) {
    if (dev >= 0 && dev < kMaxDevices) v[dev].store(value, std::memory_order_release);
  }
};
// Ordinal of the calling thread's current device, or -1.
int current_device();
// Multiprocessor count of the current device (148 on a B200); cached per device.
int sm_count();
// Raises a kernel's dynamic shared-memory limit once per device.  `done` is the kernel's cache.
template <typename Kernel>
int ensure_smem_attr(Kernel kern, int bytes, PerDeviceInt& done) {
  const int dev = current_device();
  if (done.get(dev)) return XEMA_OK;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) {
    set_last_cuda_error((int)e);
    return XEMA_ECUDA;
  }
  done.set(dev, 1);
  return XEMA_OK;
}

// Launches a kernel.  `chained`: it may start while the launch before it in the stream still runs
// (programmatic dependent launch) -- for kernels that call grid_dep_wait() before they touch memory
// which earlier launches use, and whose weights no launch before them in the same forward call
// writes.  The first launch of a forward call is never chained: what the caller enqueued before it, weights
// too, is then complete before any kernel of the call starts.  (A launch that only waits for the work ahead of it and
// copies may itself be chained to that: launch_copy2.)  Measured (B200): without it launches of dependent
// kernels start on a 2.05 us raster, 2 to 4 us after the previous one's last CTA.
template <typename... Params, typename... Args>
int launch_kernel(void (*kern)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, bool chained,
                  const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, Params(args)...);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_last_cuda_error((int)e);
    return XEMA_ECUDA;
  }
  return XEMA_OK;
}

// Features [j_first, j_end) of mod[b, j] = sum_k silu(temb[b, k]) * w[j, k] + bias[j] (mod has n_out features a row).
struct ModArgs {
  const void *temb, *w, *bias;
  float* mod;
  int batch, Dt, n_out, j_first, j_end;
};
int launch_mod(const ModArgs& a, cudaStream_t stream, bool chained = false);
int launch_ln_modulate(const void* in, int in_is_f32, long long in_batch_rows, void* out, const float* shift,
                       const float* scale, long long mod_stride, int batch, int rows, int D, float eps,
                       cudaStream_t stream, bool chained = false, const ModArgs* mod = nullptr);   // mod: beside the rows
constexpr int kLnMaxCarryCols = 3072, kLnMaxCarryCols4 = 2048;   // widths that have an instance for that: 1 and 2 batch elements, more
int launch_rmsnorm_rope(void* x, long long ld, long long batch_rows, const void* g, const float* rope, int pos0,
                        int batch, int rows, int heads, int head_dim, float eps, cudaStream_t stream);

// dst0 <- src0 (n0 bytes) and dst1 <- src1 (n1 bytes); pointers and sizes are multiples of 16 bytes.  `early`: it may be
// launched before the work ahead of it in the stream has finished; it waits for that before its first access.
int launch_copy2(void* dst0, const void* src0, size_t n0, void* dst1, const void* src1, size_t n1, cudaStream_t stream,
                 bool early = false);

// ---- TMA descriptors (encoded on the host once per bound tensor) --------------------------
// bf16 tensor viewed as [batch][rows][cols] with row stride ld and batch stride batch_rows*ld
// (elements); box = 64 columns x box_rows rows x 1, 128-byte swizzle, out-of-range rows and
// columns read as zero.
int encode_tmap_bf16(CUtensorMap* out, const void* base, long long cols, long long rows, long long batch,
                     long long ld, long long batch_rows, int box_rows);
// bf16 or fp32 tensor viewed the same way, its batch stride given in elements; box = 32 columns x 32 rows x 1,
// swizzled over its 64-byte (bf16) or 128-byte (fp32) rows.  The row stride of a single row and the batch
// stride of a single element are not looked at.
int encode_tmap_box32(CUtensorMap* out, const void* base, bool f32, long long cols, long long rows, long long batch,
                      long long ld, long long batch_stride);

// ---- GEMM ------------------------------------------------------------------------------------
struct GemmLaunch {
  CUtensorMap map_a;   // [batch][rows][K], box 64 x 128
  CUtensorMap map_w;   // [1][N][K],       box 64 x block_n (a pair: each CTA half of it)
  CUtensorMap map_out; // [batch][rows][N], box 32 x 32
  CUtensorMap map_res; // the same for the residual (gated epilogues) or for out2
  const void* bias;    // bf16 [N]
  void* out;
  long long ldo, out_batch_rows;
  const void* resid;
  long long ldr, resid_batch_rows;
  const float* gate;
  long long gate_stride;
  int batch, rows, N, K, epilogue, block_n;
  int pair;            // a CTA pair per tile (256 x block_n) or one CTA (128 x block_n)
  const void *a, *w;   // operands as given to gemm_prepare
  long long lda, a_batch_rows, ldw;
  unsigned int* status;
  // XEMA_EPI_BIAS_NORM_ROPE: RMSNorm * gain + RoPE for the heads below column norm_cols
  const void* norm_gain;
  const float* rope;
  int rope_pos0, head_dim, norm_cols;
  float rms_eps;
  float norm_out_scale;   // the normalised, rotated heads are multiplied by this before rounding (1 = as they are)
  // ... and a second result: with cols2 > 0 the first cols2 columns of the product go to out2, normalised with gain2 and
  // multiplied by norm_out_scale2, the others to column 0 on of out (norm_cols counts from the product's first column)
  void* out2;
  long long ldo2, out2_batch_rows;
  const void* norm_gain2;
  float norm_out_scale2;
  int cols2;
};
// Fills the descriptors and the tile (pair, block_n) from plain pointers.  `tile`: {pair, block_n} to take instead
// of the one estimated to be fastest, XEMA_EINVAL where the problem cannot run in it.
int gemm_prepare(GemmLaunch* g, const void* a, long long lda, long long a_batch_rows, const void* w, long long ldw,
                 const int* tile = nullptr);
// The tile alone, on the host (GemmLaunch as for gemm_prepare): fills pair and block_n.
int gemm_tile(GemmLaunch* g);
int launch_gemm(const GemmLaunch& g, cudaStream_t stream, bool chained = false);

// ---- attention -------------------------------------------------------------------------------
struct AttnLaunch {
  CUtensorMap map_q;   // [batch][rows][heads*dh], box 64 x 128
  CUtensorMap map_k;   // [batch][keys][..],       box 64 x 128
  CUtensorMap map_v;
  void* o;             // bf16 [batch][rows][heads*dh]
  float* lse;          // fp32 [batch][heads][rows] or null
  int batch, rows, keys, heads, head_dim;
  // what q k^T is multiplied by to give exponents to base 2: log2(e) / sqrt(head_dim) for a plain
  // q, 1 if q was already multiplied by that (as the fused epilogue of the Q projection does)
  float q_scale;
  unsigned int* status;
  // head_dim 64 only, both or neither: the RMSNorm gains (bf16 [head_dim], device) that q and k
  // went through before their rotation, with q multiplied by log2(e) / sqrt(head_dim) afterwards
  // (q_scale = 1).  A head of q then has norm <= max|gain_q| * log2(e) and a head of k norm <=
  // max|gain_k| * sqrt(head_dim), which bounds every score; where that bound is small the kernel
  // skips its per-score range tracking.  Null: nothing is known about the scores.
  const void* gain_q;
  const void* gain_k;
};
int attn_prepare(AttnLaunch* a, const void* q, long long ldq, long long q_batch_rows, const void* k, const void* v,
                 long long ldkv, long long kv_batch_rows);
int launch_attention(const AttnLaunch& a, cudaStream_t stream, bool chained = false);
constexpr int kAttnKeysPerBlock = 128;   // rows of the K/V TMA boxes

}  // namespace xema
