// Executor and C ABI: binds a plan to arena memory, pre-encodes the TMA descriptors, and
// replays the block's launch list on the caller's stream.  Nothing here allocates, frees or
// synchronises device memory.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <unordered_map>
#include <vector>

#include "kernels.h"
#include "planner.h"

namespace xema {

static thread_local int t_last_cuda_error = 0;
void set_last_cuda_error(int code) { t_last_cuda_error = code; }

int current_device() {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess ? dev : -1;
}

int sm_count() {
  static PerDeviceInt cache;
  const int dev = current_device();
  int n = cache.get(dev);
  if (n > 0) return n;
  if (dev < 0 || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
  cache.set(dev, n);
  return n;
}

int check_launch() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    t_last_cuda_error = (int)e;
    return XEMA_ECUDA;
  }
  return XEMA_OK;
}

// cuTensorMapEncodeTiled is fetched from the driver at run time so the library has no link
// dependency on libcuda and loads on machines without a driver.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres);
    if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !p) {
      t_last_cuda_error = (int)(e != cudaSuccess ? e : cudaErrorUnknown);
      return nullptr;
    }
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

static int encode_tmap(CUtensorMap* out, const void* base, bool f32, long long cols, long long rows, long long batch,
                       long long ld, long long batch_stride, int box_cols, int box_rows, CUtensorMapSwizzle swizzle) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return XEMA_ECUDA;
  const int elem = f32 ? 4 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)(ld * elem), (cuuint64_t)(batch_stride * elem)};
  cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, 1u};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  CUresult r = fn(out, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base),
                  dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    t_last_cuda_error = (int)r;
    return XEMA_ECUDA;
  }
  return XEMA_OK;
}

int encode_tmap_bf16(CUtensorMap* out, const void* base, long long cols, long long rows, long long batch,
                     long long ld, long long batch_rows, int box_rows) {
  if (cols < 64 || rows < 1 || batch < 1 || ld < cols || box_rows < 1 || box_rows > 256) return XEMA_EINVAL;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld & 7)) return XEMA_EALIGN;
  if (batch > 1 && batch_rows < rows) return XEMA_EINVAL;
  return encode_tmap(out, base, false, cols, rows, batch, ld, (batch_rows > 0 ? batch_rows : rows) * ld, 64, box_rows,
                     CU_TENSOR_MAP_SWIZZLE_128B);
}

int encode_tmap_box32(CUtensorMap* out, const void* base, bool f32, long long cols, long long rows, long long batch,
                      long long ld, long long batch_stride) {
  if (cols < 32 || (cols & 7) || rows < 1 || batch < 1) return XEMA_EINVAL;
  if (rows == 1) ld = cols;
  if (batch == 1) batch_stride = rows * ld;
  if (ld < 1 || batch_stride < 1) return XEMA_EINVAL;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld & 7) || (batch_stride & 7)) return XEMA_EALIGN;
  return encode_tmap(out, base, f32, cols, rows, batch, ld, batch_stride, 32, 32,
                     f32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B);
}

// ---------------------------------------------------------------------------------------------
enum OpKind { OP_MOD, OP_LN, OP_ROPE, OP_GEMM, OP_ATTN, OP_FUSED };  // OP_FUSED: done by the previous launch

struct Op {
  OpKind kind;
  char name[8];       // logical op: MOD, LN1A, KV, KROPE, LN1B, Q, QROPE, ATTN, PROJ, LN2, FFN1, FFN2
  int block, chunk;
  double flops;       // algorithmic floating-point operations of this launch
  double bytes;       // algorithmic HBM bytes of this launch (operands read once, results written once)
  // OP_MOD
  const void *temb, *w_mod, *b_mod;
  float* mod;
  // OP_LN
  const void* ln_in;
  int ln_in_f32;
  long long ln_in_batch_rows;
  void* ln_out;
  const float *shift, *scale;
  // OP_ROPE
  void* rope_x;
  long long rope_ld, rope_batch_rows;
  const void* rope_g;
  int pos0;
  // shared
  int rows;
  int batch;          // batch elements this launch covers (OP_LN, OP_ROPE)
  bool reads_ln1a;    // OP_GEMM Q: its input is LN1A's output (LN1B elided)
  size_t mod_op;      // OP_LN LN2, last piece: the next block's MOD op, and LN1A, first piece: its own, where launches may carry it; or 0
  size_t q_op;        // OP_GEMM KV: the Q op that may share its launch (xema_plan::qkv), or 0
  GemmLaunch gemm;
  AttnLaunch attn;
};

// Whether LN launches of up to `rows` rows (batch elements counted) may carry a modulation of `batch` elements.  One launch falls
// away, two get longer by half of its work each.  Speed of stacks of 3 or 8 blocks with it over the same with MOD as a launch of its own
// (repeats differ by 0.01, few by 0.02):
//   1 and 2 elements, whose carrying instances need hardly more registers than the rows: up to 2000 rows 0.99 to 1.07 at every width (8
//   blocks of 1 x 300 x 1024 1.05, of 2 x 500 x 1280 1.05, of 2 x 1000 x 512 1.04, of 2 x 500 x 3072 1.00), at 4000 0.99 to 1.01, at
//   8000 0.98 to 1.01.
//   3 to 6 (5 and more in two passes over the weights), whose instance takes 156 registers, so that fewer blocks of rows fit an SM: 768 and 1024 columns 0.99 to 1.05 up to 2000 rows,
//   0.98 to 1.00 at 3000 and 4000; 1280 and 1536 1.01 to 1.09 up to 640, 1.00 to 1.03 at 1000, 0.98 to 1.01 at 2000; 1792 and 2048 1.01
//   to 1.07 at 300, 0.99 to 1.04 at 500, 0.99 at 640; 2560 0.98 at 300.
//   512 columns and fewer, where MOD by itself is short: 3 and 4 elements 0.99 to 1.03 from 800 to 2000 rows, 0.92 to 1.02 below, 5 and 6
//   0.90 to 1.02; at 512 columns and under 100 rows 3 to 5 elements 0.99 to 1.02.
//   7 and 8: 512 0.93 to 1.01, 1024 0.98 to 1.01, 1536 and 2048 0.97 to 1.02.
static bool ln_may_carry(int batch, long long rows, int D) {
  if (batch <= 2) return D <= kLnMaxCarryCols && rows <= 4096;
  if (batch > 6) return false;
  if (D <= 512) return rows < 800 ? D == 512 && batch <= 5 && rows < 100 : batch <= 4 && rows <= 2048;
  return rows <= (D <= 1024 ? 2048 : D <= 1536 ? 1024 : D <= kLnMaxCarryCols4 ? 512 : 0);
}

// One step of xema_forward_host: a launch, or the arrival / departure of a piece of the block input /
// output (`rows` x `width` bytes at byte offset `offset` of the tensor, rows `pitch` apart).
struct HostStep {
  enum Kind { LAUNCH, COPY_IN, COPY_OUT } kind;
  Op op;
  size_t offset, width, rows, pitch;
};

}  // namespace xema

using namespace xema;

struct xema_plan {
  xema_config cfg;
  int32_t chunks[3];  // key/value, attention, feed-forward phase
  int32_t axes[3];    // XEMA_SPLIT_ROWS or XEMA_SPLIT_BATCH per phase
  Shard shard;        // sequence-parallel shard this plan covers ({0, 1}: the whole sequence)
  uint64_t guard;     // debug layout: bytes kept free after every tensor (0 in a normal plan)
  std::vector<xema_tensor> tensors;
  std::vector<uint64_t> offsets;
  std::unordered_map<std::string, size_t> index;
  uint64_t peak, live;
  uint32_t n_ops;
  bool bound;
  uint8_t* arena;     // as given to xema_plan_bind
  uint8_t *hid_in, *temb_in;   // the inputs' slots in it
  long long own_rows; // token rows of the plan's shard
  const float* rope;
  std::vector<Op> ops;
  std::vector<GemmLaunch> qkv;   // per block: KV and Q in one launch, where the KV op has a q_op
  // xema_forward_host: its launch and copy list, a second stream and events, so that the copies of one
  // piece overlap the launches of its neighbours (made at the first call after a bind; concurrent
  // calls on one plan share the arena and are the caller's error anyway)
  mutable std::vector<HostStep> host_steps;
  mutable int host_pieces_in = 0, host_pieces_out = 0;
  mutable cudaStream_t copy_stream = nullptr;
  mutable std::vector<cudaEvent_t> copy_events;
  ~xema_plan() {
    for (cudaEvent_t e : copy_events) cudaEventDestroy(e);
    if (copy_stream) cudaStreamDestroy(copy_stream);
  }
};

static ModArgs mod_args(const xema_config& c, const Op& op, int j_first, int j_end) {
  return ModArgs{op.temb, op.w_mod, op.b_mod, op.mod, c.batch, c.temb_dim, 6 * c.hidden, j_first, j_end};
}

static int launch_ln(const xema_config& c, const Op& op, cudaStream_t st, bool chained, const ModArgs* mod = nullptr) {
  return launch_ln_modulate(op.ln_in, op.ln_in_f32, op.ln_in_batch_rows, op.ln_out, op.shift, op.scale, 6LL * c.hidden, op.batch,
                            op.rows, c.hidden, c.ln_eps, st, chained, mod);
}

// `chained`: the launch right before this one in the stream is the op before it (see launch_kernel).
static int issue(const xema_plan* pl, const Op& op, cudaStream_t st, bool chained) {
  const xema_config& c = pl->cfg;
  switch (op.kind) {
    case OP_MOD:
      return launch_mod(mod_args(c, op, 0, 6 * c.hidden), st, chained);
    case OP_LN:
      return launch_ln(c, op, st, chained);
    case OP_ROPE:
      return launch_rmsnorm_rope(op.rope_x, op.rope_ld, op.rope_batch_rows, op.rope_g, pl->rope, op.pos0, op.batch,
                                 op.rows, c.heads, c.head_dim, c.rms_eps, st);
    case OP_GEMM:
      return launch_gemm(op.gemm, st, chained);
    case OP_ATTN:
      return launch_attention(op.attn, st, chained);
    case OP_FUSED:
      return XEMA_OK;
  }
  return XEMA_EINVAL;
}

// Whether the copy of the inputs may be launched before the work ahead of it in the stream has finished: not inside a
// stream capture, where the node ahead of it need not be a kernel.
static bool may_open(cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &status) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return status == cudaStreamCaptureStatusNone;
}

static int run_ops(const xema_plan* pl, size_t first, size_t n, void* stream) {
  if (!pl) return XEMA_EINVAL;
  if (!pl->bound) return XEMA_ESTATE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  n = std::min(n, pl->ops.size());
  size_t done = 0;              // the Q op that a launch of KV took along
  size_t carried = 0;           // the MOD op whose first half the LN2 before it took along
  bool chained = false;
  for (size_t i = first; i < n; ++i) {
    if ((done && i == done) || (carried && i == carried)) continue;
    const size_t q_op = pl->ops[i].q_op, mod_op = pl->ops[i].mod_op;
    int rc;
    if (q_op && q_op < n) {
      rc = launch_gemm(pl->qkv[pl->ops[i].block], st, chained);
      done = q_op;
    } else if (mod_op && (mod_op > i ? mod_op + 1 < n : mod_op == carried)) {
      // the shift, scale and gate of the attention half with LN2 of the block before, those of the feed-forward half with LN1A
      const int half = 3 * pl->cfg.hidden;
      const ModArgs mod = mod_args(pl->cfg, pl->ops[mod_op], mod_op > i ? 0 : half, mod_op > i ? half : 2 * half);
      rc = launch_ln(pl->cfg, pl->ops[i], st, chained, &mod);
      carried = mod_op;
    } else {
      rc = issue(pl, pl->ops[i], st, chained);
    }
    if (rc) return rc;
    chained = chained || pl->ops[i].kind != OP_FUSED;
  }
  return XEMA_OK;
}

extern "C" {

int xema_plan_create(const xema_config* cfg, int32_t chunks, xema_plan** out) {
  const int32_t c3[3] = {chunks, chunks, chunks};
  return xema_plan_create_phases(cfg, c3, out);
}

int xema_plan_create_phases(const xema_config* cfg, const int32_t chunks[3], xema_plan** out) {
  if (!chunks) return XEMA_EINVAL;
  xema_mitigation m;
  for (int i = 0; i < 3; ++i) {
    m.chunks[i] = chunks[i];
    m.axis[i] = XEMA_SPLIT_ROWS;
  }
  return xema_plan_create_mitigated(cfg, &m, out);
}

int xema_plan_create_mitigated(const xema_config* cfg, const xema_mitigation* m, xema_plan** out) {
  return xema_plan_create_sharded(cfg, m, 0, 1, out);
}

int xema_plan_create_sharded(const xema_config* cfg, const xema_mitigation* m, int32_t shard, int32_t shards,
                             xema_plan** out) {
  return xema_plan_create_guarded(cfg, m, shard, shards, 0, out);
}

int xema_plan_create_guarded(const xema_config* cfg, const xema_mitigation* m, int32_t shard, int32_t shards,
                             uint64_t guard_bytes, xema_plan** out) {
  if (!cfg || !out || !m) return XEMA_EINVAL;
  if (guard_bytes % 256 || guard_bytes > (1ull << 30)) return XEMA_EINVAL;
  *out = nullptr;
  xema_plan* pl = new (std::nothrow) xema_plan();
  if (!pl) return XEMA_ENOSPC;
  pl->cfg = *cfg;
  const int32_t* chunks = m->chunks;
  for (int i = 0; i < 3; ++i) {
    pl->chunks[i] = m->chunks[i];
    pl->axes[i] = m->axis[i];
  }
  pl->bound = false;
  pl->arena = nullptr;
  pl->rope = nullptr;
  pl->shard.p = shard;
  pl->shard.P = shards;
  int rc = build_trace(*cfg, chunks, pl->axes, pl->shard, pl->tensors, &pl->n_ops);
  pl->guard = guard_bytes;
  if (!rc) {
    pl->offsets.assign(pl->tensors.size(), 0);
    if (guard_bytes == 0) {
      rc = plan_arena(pl->tensors.data(), pl->tensors.size(), pl->offsets.data(), &pl->peak, &pl->live);
    } else {
      // lay out tensors that are guard_bytes larger than they are: the bytes after every tensor
      // then belong to nobody for as long as the tensor lives
      std::vector<xema_tensor> padded(pl->tensors);
      for (xema_tensor& t : padded) t.bytes += guard_bytes;
      uint64_t padded_live = 0;
      rc = plan_arena(padded.data(), padded.size(), pl->offsets.data(), &pl->peak, &padded_live);
      pl->live = max_live(pl->tensors.data(), pl->tensors.size());
    }
  }
  if (rc) {
    delete pl;
    return rc;
  }
  for (size_t i = 0; i < pl->tensors.size(); ++i) pl->index[pl->tensors[i].name] = i;
  *out = pl;
  return XEMA_OK;
}

void xema_plan_destroy(xema_plan* plan) { delete plan; }

int xema_plan_info(const xema_plan* plan, uint64_t* peak_bytes, uint64_t* max_live_bytes, size_t* n_tensors,
                   uint32_t* n_ops, int32_t* chunks) {
  if (!plan) return XEMA_EINVAL;
  if (peak_bytes) *peak_bytes = plan->peak;
  if (max_live_bytes) *max_live_bytes = plan->live;
  if (n_tensors) *n_tensors = plan->tensors.size();
  if (n_ops) *n_ops = plan->n_ops;
  if (chunks) *chunks = std::max(plan->chunks[0], std::max(plan->chunks[1], plan->chunks[2]));
  return XEMA_OK;
}

int xema_plan_phase_chunks(const xema_plan* plan, int32_t chunks[3]) {
  if (!plan || !chunks) return XEMA_EINVAL;
  for (int i = 0; i < 3; ++i) chunks[i] = plan->chunks[i];
  return XEMA_OK;
}

int xema_plan_mitigation(const xema_plan* plan, xema_mitigation* m) {
  if (!plan || !m) return XEMA_EINVAL;
  for (int i = 0; i < 3; ++i) {
    m->chunks[i] = plan->chunks[i];
    m->axis[i] = plan->axes[i];
  }
  return XEMA_OK;
}

int xema_plan_shard(const xema_plan* plan, int32_t* shard, int32_t* shards, int64_t* row0, int64_t* rows) {
  if (!plan) return XEMA_EINVAL;
  if (shard) *shard = plan->shard.p;
  if (shards) *shards = plan->shard.P;
  return shard_rows(plan->cfg, plan->shard, row0, rows);
}

uint64_t xema_plan_guard_bytes(const xema_plan* plan) { return plan ? plan->guard : 0; }

int xema_plan_gather_point(const xema_plan* plan, int32_t block, uint32_t* first_op, uint64_t* kv_offset) {
  if (!plan || block < 0 || block >= plan->cfg.n_blocks) return XEMA_EINVAL;
  const uint32_t per_block = 1 + 3 * (uint32_t)plan->chunks[0] + 5 * (uint32_t)plan->chunks[1] + 3 * (uint32_t)plan->chunks[2];
  if (first_op) *first_op = (uint32_t)block * per_block + 1 + 3 * (uint32_t)plan->chunks[0];
  if (kv_offset) {
    auto it = plan->index.find("kv" + std::to_string(block));
    if (it == plan->index.end()) return XEMA_EINVAL;
    *kv_offset = plan->offsets[it->second];
  }
  return XEMA_OK;
}

int xema_plan_tensor(const xema_plan* plan, const char* name, uint64_t* offset, uint64_t* bytes) {
  if (!plan || !name) return XEMA_EINVAL;
  auto it = plan->index.find(name);
  if (it == plan->index.end()) return XEMA_EINVAL;
  if (offset) *offset = plan->offsets[it->second];
  if (bytes) *bytes = plan->tensors[it->second].bytes;
  return XEMA_OK;
}

int xema_plan_tensor_at(const xema_plan* plan, size_t i, xema_tensor* tensor, uint64_t* offset) {
  if (!plan || i >= plan->tensors.size()) return XEMA_EINVAL;
  if (tensor) *tensor = plan->tensors[i];
  if (offset) *offset = plan->offsets[i];
  return XEMA_OK;
}

int xema_plan_bind(xema_plan* plan, void* arena_dev, uint64_t arena_bytes, const xema_block_weights* weights,
                   const float* rope_dev, void* status_dev) {
  if (!plan || !arena_dev || !weights || !rope_dev) return XEMA_EINVAL;
  if (arena_bytes < plan->peak) return XEMA_ENOSPC;
  if (reinterpret_cast<uintptr_t>(arena_dev) & 255) return XEMA_EALIGN;
  if (reinterpret_cast<uintptr_t>(rope_dev) & 15) return XEMA_EALIGN;
  const xema_config& c = plan->cfg;
  if (c.hidden % 256 || c.ffn % 256 || c.temb_dim % 8 || (c.head_dim != 64 && c.head_dim != 128))
    return XEMA_EINVAL;
  plan->bound = false;
  plan->ops.clear();
  plan->qkv.assign(c.n_blocks > 0 ? c.n_blocks : 0, GemmLaunch{});
  plan->host_steps.clear();
  plan->rope = rope_dev;
  plan->arena = static_cast<uint8_t*>(arena_dev);
  uint8_t* arena = static_cast<uint8_t*>(arena_dev);
  unsigned int* status = static_cast<unsigned int*>(status_dev);

  auto at = [&](const char* stem, int block, int chunk) -> uint8_t* {
    char name[32];
    if (block < 0)
      std::snprintf(name, sizeof(name), "%s", stem);
    else if (chunk < 0)
      std::snprintf(name, sizeof(name), "%s%d", stem, block);
    else
      std::snprintf(name, sizeof(name), "%s%d_%d", stem, block, chunk);
    auto it = plan->index.find(name);
    if (it == plan->index.end()) return nullptr;
    const size_t i = it->second;
    if (plan->offsets[i] + plan->tensors[i].bytes > arena_bytes) return nullptr;
    return arena + plan->offsets[i];
  };

  // S: the token rows this plan covers (the owned rows of its shard; all of them without
  // sharding), row0: the first of them; S_all: every row -- the keys and values of all shards
  const long long S_all = seq_len(c), D = c.hidden, F = c.ffn;
  int64_t row0_ = 0, rows_ = 0;
  if (shard_rows(c, plan->shard, &row0_, &rows_)) return XEMA_EINVAL;
  const long long S = rows_, row0 = row0_;
  const int CA = plan->chunks[0], CB = plan->chunks[1], CC = plan->chunks[2];
  for (int l = 0; l < c.n_blocks; ++l) {
    const xema_block_weights& w = weights[l];
    const void* wp[12] = {w.w_mod, w.b_mod, w.w_qkv, w.b_qkv, w.g_q, w.g_k, w.w_o, w.b_o, w.w_1, w.b_1, w.w_2, w.b_2};
    for (const void* p : wp) {
      if (!p) return XEMA_EINVAL;
      if (reinterpret_cast<uintptr_t>(p) & 15) return XEMA_EALIGN;
    }
    const __nv_bfloat16* w_qkv = static_cast<const __nv_bfloat16*>(w.w_qkv);
    const __nv_bfloat16* b_qkv = static_cast<const __nv_bfloat16*>(w.b_qkv);
    uint8_t* hid = at("hid", l, -1);
    uint8_t* hid_next = at("hid", l + 1, -1);
    float* mod = reinterpret_cast<float*>(at("mod", l, -1));
    uint8_t* kv = at("kv", l, -1);
    uint8_t* res = at("res", l, -1);
    uint8_t* temb = at("temb", -1, -1);
    if (!hid || !hid_next || !mod || !kv || !res || !temb) return XEMA_EINVAL;

    Op op{};
    op.kind = OP_MOD;
    op.temb = temb; op.w_mod = w.w_mod; op.b_mod = w.b_mod; op.mod = mod;
    const double Bd = c.batch, Dd = (double)D, Fd = (double)F, Sd = (double)S_all;
    auto tag = [&](Op& o, const char* nm, int chunk, double flops, double bytes) {
      std::snprintf(o.name, sizeof(o.name), "%s", nm);
      o.block = l; o.chunk = chunk; o.flops = flops; o.bytes = bytes;
    };
    tag(op, "MOD", -1, 2.0 * Bd * 6 * Dd * c.temb_dim, 2.0 * 6 * Dd * c.temb_dim + 24.0 * Bd * Dd);
    plan->ops.push_back(op);

    // A piece of a phase: batch elements [b0, b0 + nb) x rows [r0, r0 + n).
    struct Piece {
      long long b0, r0;
      int nb, n;
    };
    auto piece_of = [&](int phase, int ci) {
      const int C = plan->chunks[phase];
      Piece pc;
      if (plan->axes[phase] == XEMA_SPLIT_BATCH) {
        pc.b0 = (long long)ci * c.batch / C;
        pc.nb = (int)((long long)(ci + 1) * c.batch / C - pc.b0);
        pc.r0 = 0;
        pc.n = (int)S;
      } else {
        pc.b0 = 0;
        pc.nb = c.batch;
        pc.r0 = (long long)ci * S / C;
        pc.n = (int)((long long)(ci + 1) * S / C - pc.r0);
      }
      return pc;
    };
    // byte offset of (batch b0, row r0) in a [B, S, width] tensor over the plan's rows, and in the
    // [B, S_all, 2D] keys-and-values tensor, whose rows are global
    auto at_row = [&](const Piece& pc, long long width, int elem_bytes) { return (pc.b0 * S + pc.r0) * width * elem_bytes; };
    auto at_kv_row = [&](const Piece& pc) { return (pc.b0 * S_all + row0 + pc.r0) * 2 * D * 2; };
    auto ln_op = [&](const void* in, int f32, void* out, const Piece& pc, int which, const char* nm, int chunk) {
      Op o{};
      o.kind = OP_LN;
      const double elems = (double)pc.nb * pc.n;
      tag(o, nm, chunk, 8.0 * elems * Dd, elems * Dd * (f32 ? 6.0 : 4.0));
      o.ln_in = in; o.ln_in_f32 = f32; o.ln_in_batch_rows = S; o.ln_out = out;
      o.shift = mod + pc.b0 * 6 * D + (which == 1 ? 0 : 3 * D);
      o.scale = mod + pc.b0 * 6 * D + (which == 1 ? D : 4 * D);
      o.rows = pc.n;
      o.batch = pc.nb;
      plan->ops.push_back(o);
    };
    auto gemm_op = [&](const void* a, long long lda, long long a_batch_rows, const void* wt, long long ldw,
                       const void* bias, void* out, long long ldo, long long out_batch_rows, const void* resid,
                       long long ldr, long long resid_batch_rows, const float* gate, const Piece& pc, int N, int K,
                       int epi, const char* nm, int chunk, const void* norm_gain = nullptr, int norm_cols = 0,
                       int pos0 = 0, float norm_out_scale = 1.f) -> int {
      const int rows = pc.n;
      const double Bd = (double)pc.nb;
      Op o{};
      o.kind = OP_GEMM;
      o.gemm.norm_gain = norm_gain; o.gemm.rope = rope_dev; o.gemm.rope_pos0 = pos0; o.gemm.head_dim = c.head_dim;
      o.gemm.norm_cols = norm_cols; o.gemm.rms_eps = c.rms_eps; o.gemm.norm_out_scale = norm_out_scale;
      {
        const double out_b = (epi == XEMA_EPI_GATE_RES_F32) ? 4.0 : 2.0;
        const double res_b = (epi == XEMA_EPI_GATE_RES_F32) ? 2.0 : (epi == XEMA_EPI_GATE_RES_BF16 ? 4.0 : 0.0);
        tag(o, nm, chunk, 2.0 * Bd * rows * (double)N * K,
            2.0 * Bd * rows * K + 2.0 * (double)N * K + (out_b + res_b) * Bd * rows * N);
      }
      GemmLaunch& g = o.gemm;
      g.bias = bias; g.out = out; g.ldo = ldo; g.out_batch_rows = out_batch_rows;
      g.resid = resid; g.ldr = ldr; g.resid_batch_rows = resid_batch_rows;
      g.gate = gate; g.gate_stride = 6 * D;
      g.batch = pc.nb; g.rows = rows; g.N = N; g.K = K; g.epilogue = epi; g.status = status;
      int rc = gemm_prepare(&g, a, lda, a_batch_rows, wt, ldw);
      if (rc) return rc;
      plan->ops.push_back(o);
      return XEMA_OK;
    };

    // phase A: keys and values of every piece
    size_t kv_op = 0;               // the last KV op of the phase
    for (int ci = 0; ci < CA; ++ci) {
      const Piece pc = piece_of(0, ci);
      const int n = pc.n;
      uint8_t* h1a = at("h1a", l, ci);
      if (!h1a) return XEMA_EINVAL;
      uint8_t* kv_pc = kv + at_kv_row(pc);
      ln_op(hid + at_row(pc, D, 2), 0, h1a, pc, 1, "LN1A", ci);
      // K half: RMSNorm * g_k + RoPE in the GEMM epilogue; the KROPE op of the trace is then
      // a placeholder (the fused kernel touches a subset of what the trace says is live)
      int rc = gemm_op(h1a, D, n, w_qkv + D * D, D, b_qkv + D, kv_pc, 2 * D, S_all, nullptr, 0, 0, nullptr,
                       pc, (int)(2 * D), (int)D, XEMA_EPI_BIAS_NORM_ROPE, "KV", ci, w.g_k, (int)D, (int)(row0 + pc.r0));
      if (rc) return rc;
      kv_op = plan->ops.size() - 1;
      Op o{};
      o.kind = OP_FUSED;
      tag(o, "KROPE", ci, 0.0, 0.0);
      o.rope_x = kv_pc; o.rope_ld = 2 * D; o.rope_batch_rows = S_all; o.rope_g = w.g_k;
      o.pos0 = (int)(row0 + pc.r0); o.rows = n; o.batch = pc.nb;
      plan->ops.push_back(o);
    }
    // The queries leave their projection already multiplied by log2(e) / sqrt(head_dim), inside the
    // epilogue that rounds them to bf16 (one rounding, as before): the attention's scores are then
    // exponents to base 2 as they come out of the tensor core.
    const float q_scale = 1.4426950408889634f / std::sqrt((float)c.head_dim);
    // phase B: queries, attention and the gated output projection of every piece
    for (int ci = 0; ci < CB; ++ci) {
      const Piece pc = piece_of(1, ci);
      const int n = pc.n;
      const double Bd = (double)pc.nb;
      uint8_t* h1b = at("h1b", l, ci);
      uint8_t* q = at("q", l, ci);
      uint8_t* o_t = at("o", l, ci);
      float* lse = reinterpret_cast<float*>(at("lse", l, ci));
      if (!h1b || !q || !o_t || !lse) return XEMA_EINVAL;
      const uint8_t* hid_pc = hid + at_row(pc, D, 2);
      const uint8_t* kv_b = kv + pc.b0 * S_all * 2 * D * 2;      // keys and values of these batch elements
      ln_op(hid_pc, 0, h1b, pc, 1, "LN1B", ci);
      bool q_follows_kv = false;      // no launch between KV and Q, both read LN1A's output
      // With one piece in both phases LN1B recomputes what LN1A wrote.  When the layout put h1b
      // at h1a's address and nothing was born in between (KROPE allocates nothing, so the only
      // births since the KV op are h1b's own), those bytes are still there: the launch is elided.
      if (CA == 1 && CB == 1 && h1b == at("h1a", l, 0)) {
        bool untouched = true;
        const size_t ia = plan->index.at(std::string("h1a") + std::to_string(l) + "_0");
        const size_t ib = plan->index.at(std::string("h1b") + std::to_string(l) + "_0");
        const xema_tensor& ta = plan->tensors[ia];
        const xema_tensor& tb = plan->tensors[ib];
        for (size_t i = 0; i < plan->tensors.size() && untouched; ++i) {
          if (i == ia || i == ib) continue;
          const xema_tensor& tt = plan->tensors[i];
          const bool born_between = tt.birth >= ta.death && tt.birth <= tb.birth;
          const bool overlaps = plan->offsets[i] < plan->offsets[ia] + ta.bytes && plan->offsets[ia] < plan->offsets[i] + tt.bytes;
          if (born_between && overlaps) untouched = false;
        }
        if (untouched && ta.bytes == tb.bytes) {
          plan->ops.back().kind = OP_FUSED;
          q_follows_kv = true;
          plan->ops.back().flops = 0.0;
          plan->ops.back().bytes = 0.0;
        }
      }
      int rc = gemm_op(h1b, D, n, w_qkv, D, b_qkv, q, D, n, nullptr, 0, 0, nullptr, pc, (int)D, (int)D,
                       XEMA_EPI_BIAS_NORM_ROPE, "Q", ci, w.g_q, (int)D, (int)(row0 + pc.r0), q_scale);
      if (rc) return rc;
      plan->ops.back().reads_ln1a = q_follows_kv;     // ops: LN1A, KV, KROPE (fused), LN1B (elided), Q
      // Q then multiplies the same rows with the weight rows in front of KV's, by the same epilogue: one launch does both where
      // nothing that lives between the two ops lies in q's bytes.  It has one start and end less.  The tile is picked for the 3 D
      // columns, and the product by itself can take longer than the two (by the rule's own figures up to 0.7 us, at 535 to 680 rows of 1280
      // columns, where one wave of 256 x 256 pairs stands against one of 128 x 128 and one of 128 x 64); the saved launch is worth more.  us
      // apart / together, blocks: 640 x 1280 74.8 / 73.7, 879 x 1280 77.5 / 75.7, 796 x 1024 67.1 / 63.8, 1028 x 768 63.4 / 61.6, 535 x 3072
      // 197.1 / 188.8, 2072 x 2816 480.4 / 478.3 (the sizes where the rule's figures speak most against it); 288 x 512 45.3 / 40.7, eight of 333 x
      // 1024 443.5 / 404.8, 1101 x 1536 121.1 / 114.4, 4608 x 3072 and 17776 x 3072 no difference.
      if (q_follows_kv) {
        const size_t q_op = plan->ops.size() - 1;
        const size_t iq = plan->index.at(std::string("q") + std::to_string(l) + "_0");
        const uint64_t q0 = plan->offsets[iq], q1 = q0 + plan->tensors[iq].bytes;
        bool free = true;
        for (size_t i = 0; i < plan->tensors.size() && free; ++i) {
          const xema_tensor& tt = plan->tensors[i];
          free = i == iq || tt.birth > q_op || tt.death <= kv_op || plan->offsets[i] >= q1 || plan->offsets[i] + tt.bytes <= q0;
        }
        if (free) {
          GemmLaunch both = plan->ops[kv_op].gemm;
          both.bias = b_qkv;
          both.N = (int)(3 * D);
          both.norm_cols = (int)(2 * D);
          both.out2 = q; both.ldo2 = D; both.out2_batch_rows = n;
          both.norm_gain2 = w.g_q; both.norm_out_scale2 = q_scale; both.cols2 = (int)D;
          if ((rc = gemm_prepare(&both, both.a, both.lda, both.a_batch_rows, w_qkv, D))) return rc;
          plan->qkv[l] = both;
          plan->ops[kv_op].q_op = q_op;
        }
      }
      Op o{};
      o.kind = OP_FUSED;
      tag(o, "QROPE", ci, 0.0, 0.0);
      o.rope_x = q; o.rope_ld = D; o.rope_batch_rows = n; o.rope_g = w.g_q; o.pos0 = (int)(row0 + pc.r0); o.rows = n;
      o.batch = pc.nb;
      plan->ops.push_back(o);
      Op a{};
      a.kind = OP_ATTN;
      // q and o once, k and v once per launch, lse
      tag(a, "ATTN", ci, 4.0 * Bd * n * Sd * Dd, 4.0 * Bd * n * Dd + 4.0 * Bd * Sd * Dd + 4.0 * Bd * c.heads * n);
      a.attn.o = o_t; a.attn.lse = lse; a.attn.batch = pc.nb; a.attn.rows = n; a.attn.keys = (int)S_all;
      a.attn.heads = c.heads; a.attn.head_dim = c.head_dim; a.attn.status = status; a.attn.q_scale = 1.f;
      a.attn.gain_q = w.g_q; a.attn.gain_k = w.g_k;     // q and k come out of the fused RMSNorm + RoPE epilogues
      rc = attn_prepare(&a.attn, q, D, n, kv_b, kv_b + D * 2, 2 * D, S_all);
      if (rc) return rc;
      plan->ops.push_back(a);
      rc = gemm_op(o_t, D, n, w.w_o, D, w.b_o, res + at_row(pc, D, 4), D, S, hid_pc, D, S,
                   mod + pc.b0 * 6 * D + 2 * D, pc, (int)D, (int)D, XEMA_EPI_GATE_RES_F32, "PROJ", ci);
      if (rc) return rc;
    }
    // phase C: feed-forward of every piece
    for (int ci = 0; ci < CC; ++ci) {
      const Piece pc = piece_of(2, ci);
      const int n = pc.n;
      uint8_t* h2 = at("h2", l, ci);
      uint8_t* g = at("g", l, ci);
      if (!h2 || !g) return XEMA_EINVAL;
      uint8_t* res_pc = res + at_row(pc, D, 4);
      ln_op(res_pc, 1, h2, pc, 2, "LN2", ci);
      int rc = gemm_op(h2, D, n, w.w_1, D, w.b_1, g, F, n, nullptr, 0, 0, nullptr, pc, (int)F, (int)D,
                       XEMA_EPI_BIAS_GELU, "FFN1", ci);
      if (rc) return rc;
      rc = gemm_op(g, F, n, w.w_2, F, w.b_2, hid_next + at_row(pc, D, 2), D, S, res_pc, D, S,
                   mod + pc.b0 * 6 * D + 5 * D, pc, (int)D, (int)F, XEMA_EPI_GATE_RES_BF16, "FFN2", ci);
      if (rc) return rc;
    }
  }
  if (plan->ops.size() != plan->n_ops) return XEMA_EINVAL;
  // The modulation of a later block needs the timestep embedding and the slot of the block before, of which the attention half
  // (shift, scale, gate) has been read when LN2 starts and the rest when the next LN1A does: the blocks of those two launches
  // that have no row work it out, and its own launch falls away.  Where mod<m> lies over nothing but mod<m - 1> from LN2 to
  // MOD and nothing takes the embedding's bytes until LN1A, and where it is faster (ln_may_carry).  Eight blocks of 333 x 1024 in a graph
  // 401.7 -> 385.0 us.
  const size_t per_block = 1 + 3 * (size_t)CA + 5 * (size_t)CB + 3 * (size_t)CC;
  for (int m = 1; m < c.n_blocks; ++m) {
    const size_t mod_op = m * per_block, ln1 = mod_op + 1, ln2 = mod_op - 3;
    const size_t im = plan->index.at("mod" + std::to_string(m)), ib = plan->index.at("mod" + std::to_string(m - 1));
    const size_t it = plan->index.at("temb");
    const long long rows = std::max((long long)plan->ops[ln1].batch * plan->ops[ln1].rows, (long long)plan->ops[ln2].batch * plan->ops[ln2].rows);
    bool free = ln_may_carry(c.batch, rows, (int)D);
    auto overlap = [&](size_t i, size_t j) {
      return plan->offsets[i] < plan->offsets[j] + plan->tensors[j].bytes && plan->offsets[j] < plan->offsets[i] + plan->tensors[i].bytes;
    };
    for (size_t i = 0; i < plan->tensors.size() && free; ++i) {
      const xema_tensor& t = plan->tensors[i];
      if (t.death <= ln2 || t.birth > ln1) continue;
      if (i != im && overlap(i, im) && t.birth <= mod_op) free = i == ib && plan->offsets[ib] == plan->offsets[im];
      if (i != it && overlap(i, it)) free = false;
    }
    if (free) plan->ops[ln2].mod_op = plan->ops[ln1].mod_op = mod_op;
  }
  plan->hid_in = at("hid", 0, -1);
  plan->temb_in = at("temb", -1, -1);
  plan->own_rows = S;
  plan->bound = true;
  return XEMA_OK;
}

int xema_plan_set_inputs(const xema_plan* plan, const void* hid_dev, const void* temb_dev, void* stream) {
  if (!plan || !hid_dev || !temb_dev) return XEMA_EINVAL;
  if (!plan->bound) return XEMA_ESTATE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const xema_config& c = plan->cfg;
  const size_t hid_bytes = (size_t)2 * c.batch * (size_t)plan->own_rows * c.hidden;
  const size_t temb_bytes = (size_t)2 * c.batch * c.temb_dim;
  // The two copies run side by side and in no order of their pieces: a source may be its own slot, but
  // must not overlap a slot otherwise.
  auto overlaps = [](const void* src, size_t n, const uint8_t* slot, size_t m) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src), b = reinterpret_cast<uintptr_t>(slot);
    return a < b + m && b < a + n;
  };
  if ((hid_dev != plan->hid_in && overlaps(hid_dev, hid_bytes, plan->hid_in, hid_bytes)) ||
      (temb_dev != plan->temb_in && overlaps(temb_dev, temb_bytes, plan->temb_in, temb_bytes)) ||
      overlaps(hid_dev, hid_bytes, plan->temb_in, temb_bytes) || overlaps(temb_dev, temb_bytes, plan->hid_in, hid_bytes))
    return XEMA_EINVAL;
  if (((reinterpret_cast<uintptr_t>(hid_dev) | reinterpret_cast<uintptr_t>(temb_dev)) & 15) == 0)
    return launch_copy2(plan->hid_in, hid_dev, hid_bytes, plan->temb_in, temb_dev, temb_bytes, st, may_open(st));
  cudaError_t e = cudaMemcpyAsync(plan->hid_in, hid_dev, hid_bytes, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(plan->temb_in, temb_dev, temb_bytes, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) {
    t_last_cuda_error = (int)e;
    return XEMA_ECUDA;
  }
  return XEMA_OK;
}

int xema_block_forward(const xema_plan* plan, void* stream) {
  if (!plan) return XEMA_EINVAL;
  if (plan->cfg.n_blocks != 1) return XEMA_ESTATE;
  return run_ops(plan, 0, plan->ops.size(), stream);
}

int xema_step_forward(const xema_plan* plan, void* stream) {
  if (!plan) return XEMA_EINVAL;
  return run_ops(plan, 0, plan->ops.size(), stream);
}

// `op` for batch elements [b0, b0 + nb) and rows [r0, r0 + n) of those it covers (rows only where it
// covers one batch element: an LN's output and a chunk's tensors are contiguous over both).
static int sub_op(const xema_config& c, const Op& op, long long b0, int nb, long long r0, int n, Op* out) {
  *out = op;
  if (op.kind == OP_LN) {
    const int elem = op.ln_in_f32 ? 4 : 2;
    out->ln_in = static_cast<const uint8_t*>(op.ln_in) + (b0 * op.ln_in_batch_rows + r0) * c.hidden * elem;
    out->ln_out = static_cast<uint8_t*>(op.ln_out) + (b0 * op.rows + r0) * c.hidden * 2;
    out->shift = op.shift + b0 * 6 * c.hidden;
    out->scale = op.scale + b0 * 6 * c.hidden;
    out->rows = n;
    out->batch = nb;
    return XEMA_OK;
  }
  GemmLaunch& g = out->gemm;
  const int out_elem = g.epilogue == XEMA_EPI_GATE_RES_F32 ? 4 : 2, res_elem = g.epilogue == XEMA_EPI_GATE_RES_BF16 ? 4 : 2;
  g.out = static_cast<uint8_t*>(g.out) + (b0 * g.out_batch_rows + r0) * g.ldo * out_elem;
  if (g.resid) g.resid = static_cast<const uint8_t*>(g.resid) + (b0 * g.resid_batch_rows + r0) * g.ldr * res_elem;
  if (g.out2) g.out2 = static_cast<uint8_t*>(g.out2) + (b0 * g.out2_batch_rows + r0) * g.ldo2 * 2;
  if (g.gate) g.gate += b0 * g.gate_stride;
  g.rope_pos0 += (int)r0;
  g.batch = nb;
  g.rows = n;
  return gemm_prepare(&g, static_cast<const uint8_t*>(g.a) + (b0 * g.a_batch_rows + r0) * g.lda * 2, g.lda, g.a_batch_rows, g.w,
                      g.ldw);
}

// The pieces in which the work of an op on `batch` elements x `rows` token rows follows its copies:
// single batch elements, or, for one element, rows that fill the GPU's CTA pairs with 256 x 256 tiles of
// the D-wide products twice (3072 rows of 3072 columns on 74 pairs), or once where that gives less than two
// pieces; with `fine_begin` the first piece is one wave, because the copies out wait for it, and with `fine_end` a last piece of
// more than one such wave and less than two is halved, because nothing hides its copy, or the work on it (whole pieces stay as
// they are).  Copies under 4 MB are not worth an event.
static std::vector<std::pair<long long, long long>> host_pieces(const xema_config& c, int batch, int rows, bool fine_begin,
                                                               bool fine_end) {
  std::vector<std::pair<long long, long long>> out;      // [begin, end) in elements (batch > 1) or rows
  const long long row_bytes = 2LL * c.hidden, total = batch > 1 ? batch : rows;
  const long long unit_bytes = batch > 1 ? row_bytes * rows : row_bytes;
  const long long least = std::max<long long>(1, (4ll << 20) / unit_bytes);
  long long step = 1, first = 0;
  if (batch == 1) {
    const long long wave = std::max(1, sm_count() / 2 / std::max(1, c.hidden / 256)) * 256ll;
    step = rows >= 4 * wave ? 2 * wave : wave;
    if (fine_begin && step > wave && wave >= least) first = wave;
    fine_end = fine_end && (rows - first) % step > wave;
  } else {
    fine_end = false;
  }
  step = std::max(step, least);
  if (first) out.push_back({0, first});
  for (long long at = first; at < total; at += step) out.push_back({at, std::min(total, at + step)});
  if (out.size() > 1 && out.back().second - out.back().first < least) {   // a remnant joins its neighbour
    out[out.size() - 2].second = total;
    out.pop_back();
  }
  if (fine_end && out.back().second - out.back().first >= 2 * least) {
    const long long b = out.back().first, e = out.back().second, mid = b + (e - b + 1) / 2 / 256 * 256;
    if (mid > b && mid < e) {
      out.back().second = mid;
      out.push_back({mid, e});
    }
  }
  return out;
}

// The launches of the plan with the first block's key/value phase cut so that it can follow the input's
// arrival, and the last block's feed-forward phase so that the output can leave while it is made.  A row's
// bits do not depend on how rows are cut, and every launch stays inside the tensors of its op; where the
// order of the ops changes, the tensors involved are checked to be disjoint.
static int build_host_steps(const xema_plan* plan) {
  const xema_config& c = plan->cfg;
  const std::vector<Op>& ops = plan->ops;
  std::vector<HostStep> steps;
  int n_in = 0, n_out = 0;
  std::vector<bool> done(ops.size(), false);
  uint8_t* out_dev = nullptr;
  {
    char name[32];
    std::snprintf(name, sizeof(name), "hid%d", c.n_blocks);
    auto it = plan->index.find(name);
    if (it == plan->index.end()) return XEMA_EINVAL;
    out_dev = plan->arena + plan->offsets[it->second];
  }
  const size_t row_bytes = (size_t)2 * c.hidden, hid_bytes = (size_t)2 * c.batch * plan->own_rows * c.hidden;
  auto launch = [&](const Op& op) {
    HostStep st{};
    st.kind = HostStep::LAUNCH;
    st.op = op;
    steps.push_back(st);
  };
  auto launch_sub = [&](const Op& op, long long b0, int nb, long long r0, int n) {
    HostStep st{};
    st.kind = HostStep::LAUNCH;
    const int rc = sub_op(c, op, b0, nb, r0, n, &st.op);
    if (!rc) steps.push_back(st);
    return rc;
  };
  // the tensor's rows that `batch` elements x `rows` rows at `dev` cover, elements `batch_rows` apart
  auto copy = [&](HostStep::Kind kind, const uint8_t* tensor, const uint8_t* dev, int batch, int rows, long long batch_rows) {
    HostStep st{};
    st.kind = kind;
    st.offset = (size_t)(dev - tensor);
    st.width = (size_t)rows * row_bytes;
    st.rows = (size_t)batch;
    st.pitch = (size_t)batch_rows * row_bytes;
    steps.push_back(st);
    ++(kind == HostStep::COPY_IN ? n_in : n_out);
  };
  for (size_t i = 0; i < ops.size(); ++i) {
    const Op& op = ops[i];
    if (done[i] || op.kind == OP_FUSED) continue;
    const bool first_ln = op.kind == OP_LN && op.block == 0 && !std::strcmp(op.name, "LN1A");
    const bool last_ln = op.kind == OP_LN && op.block == c.n_blocks - 1 && !std::strcmp(op.name, "LN2");
    if (!first_ln && !last_ln) {
      launch(op);
      continue;
    }
    const bool by_batch = op.batch > 1;
    const bool last_chunk = op.chunk + 1 == plan->chunks[first_ln ? 0 : 2];
    const auto pieces = host_pieces(c, op.batch, op.rows, last_ln && op.chunk == 0, last_chunk);
    // The output is born at the first FFN2 and may lie where h2 of the first chunk was.  The chunk can be cut all the same where
    // every piece's rows of the output end before the rows of h2 that are still to come; otherwise its LN2 and FFN1 stay whole.
    // (17776 x 3072 at 640 MiB, whose copies out take as long as its feed-forward: they begin 0.44 ms earlier, 8486 -> 8175 us.)
    bool apart = true;
    if (last_ln) {
      const GemmLaunch& g = ops[i + 2].gemm;
      const uint8_t *h2 = static_cast<const uint8_t*>(op.ln_out), *out = static_cast<const uint8_t*>(g.out);
      if (!(h2 + (size_t)op.batch * op.rows * row_bytes <= out_dev || out_dev + hid_bytes <= h2))
        for (size_t k = 0; k + 1 < pieces.size(); ++k) {
          const long long end = pieces[k].second;
          const long long out_rows = by_batch ? (end - 1) * g.out_batch_rows + op.rows : end;
          apart = apart && out + out_rows * row_bytes <= h2 + (by_batch ? end * op.rows : end) * row_bytes;
        }
    }
    for (const auto& pc : pieces) {
      const long long b0 = by_batch ? pc.first : 0, r0 = by_batch ? 0 : pc.first;
      const int nb = by_batch ? (int)(pc.second - pc.first) : 1, n = by_batch ? op.rows : (int)(pc.second - pc.first);
      int rc = XEMA_OK;
      if (first_ln) {
        // LN1A, KV and, where it reads LN1A's output too, Q
        copy(HostStep::COPY_IN, plan->hid_in, static_cast<const uint8_t*>(op.ln_in) + (b0 * op.ln_in_batch_rows + r0) * row_bytes,
             nb, n, op.ln_in_batch_rows);
        rc = launch_sub(op, b0, nb, r0, n);
        Op kv = ops[i + 1];
        if (kv.q_op) {
          kv.gemm = plan->qkv[kv.block];
          done[kv.q_op] = true;
        }
        if (!rc) rc = launch_sub(kv, b0, nb, r0, n);
        done[i + 1] = true;
        // (q's bytes are free during KV: whatever lives then lives at the Q op as well)
        if (!rc && !kv.q_op && i + 4 < ops.size() && ops[i + 4].kind == OP_GEMM && ops[i + 4].reads_ln1a) {
          rc = launch_sub(ops[i + 4], b0, nb, r0, n);
          done[i + 4] = true;
        }
      } else {
        // LN2, FFN1, FFN2
        const Op &ffn1 = ops[i + 1], &ffn2 = ops[i + 2];
        if (apart) {
          rc = launch_sub(op, b0, nb, r0, n);
          if (!rc) rc = launch_sub(ffn1, b0, nb, r0, n);
        } else if (pc.first == 0) {
          launch(op);
          launch(ffn1);
        }
        if (!rc) rc = launch_sub(ffn2, b0, nb, r0, n);
        if (!rc)
          copy(HostStep::COPY_OUT, out_dev, static_cast<const uint8_t*>(steps.back().op.gemm.out), nb, n,
               ffn2.gemm.out_batch_rows);
        done[i + 1] = done[i + 2] = true;
      }
      if (rc) return rc;
    }
  }
  plan->host_steps.swap(steps);
  plan->host_pieces_in = n_in;
  plan->host_pieces_out = n_out;
  return XEMA_OK;
}

int xema_forward_host(const xema_plan* plan, const void* hid_in_host, const void* temb_host, void* hid_out_host,
                      void* stream) {
  if (!plan || !hid_in_host || !temb_host || !hid_out_host) return XEMA_EINVAL;
  if (!plan->bound) return XEMA_ESTATE;
  if (plan->shard.P != 1) return XEMA_ESTATE;   // a shard's step needs the caller's exchange in the middle
  const xema_config& c = plan->cfg;
  char out_name[32];
  std::snprintf(out_name, sizeof(out_name), "hid%d", c.n_blocks);
  auto i_out = plan->index.find(out_name);
  if (i_out == plan->index.end()) return XEMA_EINVAL;
  if (plan->host_steps.empty())
    if (int rc = build_host_steps(plan)) return rc;
  // exact sizes (the planned sizes are rounded up to 256 bytes; the caller's buffers are not)
  const size_t temb_bytes = (size_t)2 * c.batch * c.temb_dim;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint8_t* in_dev = plan->hid_in;
  uint8_t* out_dev = plan->arena + plan->offsets[i_out->second];
  const uint8_t* in_host = static_cast<const uint8_t*>(hid_in_host);
  uint8_t* out_host = static_cast<uint8_t*>(hid_out_host);
  cudaError_t e = cudaSuccess;
  auto fail = [&](cudaError_t err) {
    t_last_cuda_error = (int)err;
    return XEMA_ECUDA;
  };
  auto move = [&](const HostStep& s, cudaStream_t on) {
    uint8_t* dev = (s.kind == HostStep::COPY_IN ? in_dev : out_dev) + s.offset;
    const void* src = s.kind == HostStep::COPY_IN ? (const void*)(in_host + s.offset) : dev;
    void* dst = s.kind == HostStep::COPY_IN ? (void*)dev : out_host + s.offset;
    const cudaMemcpyKind kind = s.kind == HostStep::COPY_IN ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
    if (s.rows == 1) return cudaMemcpyAsync(dst, src, s.width, kind, on);
    return cudaMemcpy2DAsync(dst, s.pitch, src, s.pitch, s.width, s.rows, kind, on);
  };

  // Where the input or the output moves in more than one piece, its copies run on the plan's second
  // stream, ordered by events: input piece k + 1 arrives while piece k is worked on, output piece k
  // leaves while piece k + 1 is worked on.  Bits do not depend on it.  One piece is a plain copy on the
  // caller's stream.
  const bool split_in = plan->host_pieces_in > 1, split_out = plan->host_pieces_out > 1;
  const size_t n_events = (split_in ? plan->host_pieces_in : 0) + (split_out ? plan->host_pieces_out : 0) + 2;
  if (split_in || split_out) {
    if (!plan->copy_stream && (e = cudaStreamCreateWithFlags(&plan->copy_stream, cudaStreamNonBlocking)) != cudaSuccess)
      return fail(e);
    while (plan->copy_events.size() < n_events) {
      cudaEvent_t ev;
      if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) return fail(e);
      plan->copy_events.push_back(ev);
    }
  }
  size_t next_event = 0;
  cudaStream_t cs = plan->copy_stream;
  // `later` continues after what `earlier` was given so far
  auto order = [&](cudaStream_t earlier, cudaStream_t later) {
    cudaEvent_t ev = plan->copy_events[next_event++];
    cudaError_t err = cudaEventRecord(ev, earlier);
    return err != cudaSuccess ? err : cudaStreamWaitEvent(later, ev, 0);
  };

  if ((e = cudaMemcpyAsync(plan->temb_in, temb_host, temb_bytes, cudaMemcpyHostToDevice, st)) != cudaSuccess) return fail(e);
  std::vector<cudaEvent_t> arrived;
  if (split_in) {
    // the copy stream starts where the caller's stream stands (the arena may still be in use by work
    // enqueued before this call)
    if ((e = order(st, cs)) != cudaSuccess) return fail(e);
    for (const HostStep& s : plan->host_steps) {
      if (s.kind != HostStep::COPY_IN) continue;
      arrived.push_back(plan->copy_events[next_event++]);
      if ((e = move(s, cs)) != cudaSuccess || (e = cudaEventRecord(arrived.back(), cs)) != cudaSuccess) return fail(e);
    }
  }
  size_t k_in = 0;
  bool chained = false;
  for (const HostStep& s : plan->host_steps) {
    if (s.kind == HostStep::LAUNCH) {
      if (int rc = issue(plan, s.op, st, chained)) return rc;
      chained = true;
      continue;
    }
    chained = false;      // what follows is ordered after a copy or an event, not after a launch alone
    if (s.kind == HostStep::COPY_IN) {
      e = split_in ? cudaStreamWaitEvent(st, arrived[k_in++], 0) : move(s, st);
    } else {
      if (split_out) e = order(st, cs);
      if (e == cudaSuccess) e = move(s, split_out ? cs : st);
    }
    if (e != cudaSuccess) return fail(e);
  }
  // the caller's stream ends after everything the copy stream was given
  if ((split_in || split_out) && (e = order(cs, st)) != cudaSuccess) return fail(e);
  return XEMA_OK;
}

int xema_forward_prefix(const xema_plan* plan, uint32_t n_logical_ops, void* stream) {
  return run_ops(plan, 0, n_logical_ops, stream);
}

int xema_forward_range(const xema_plan* plan, uint32_t first_op, uint32_t end_op, void* stream) {
  if (first_op > end_op) return XEMA_EINVAL;
  return run_ops(plan, first_op, end_op, stream);
}

int xema_plan_op(const xema_plan* plan, uint32_t i, char* name8, int32_t* block, int32_t* chunk, double* flops,
                 double* bytes) {
  if (!plan) return XEMA_EINVAL;
  if (!plan->bound) return XEMA_ESTATE;
  if (i >= plan->ops.size()) return XEMA_EINVAL;
  const Op& o = plan->ops[i];
  if (name8) std::memcpy(name8, o.name, 8);
  if (block) *block = o.block;
  if (chunk) *chunk = o.chunk;
  if (flops) *flops = o.flops;
  if (bytes) *bytes = o.bytes;
  return XEMA_OK;
}

int xema_plan_launch_count(const xema_plan* plan) {
  if (!plan || !plan->bound) return 0;
  int n = 0;
  for (const Op& o : plan->ops) n += o.kind != OP_FUSED;
  return n;
}

int xema_plan_forward_launches(const xema_plan* plan) {
  if (!plan || !plan->bound) return 0;
  int n = xema_plan_launch_count(plan);
  for (const Op& o : plan->ops) n -= (o.q_op != 0) + (o.mod_op != 0 && !std::strcmp(o.name, "LN2"));
  return n;
}

int xema_op_mod(const void* temb, const void* w_mod, const void* b_mod, float* mod, int32_t batch, int32_t temb_dim,
                int32_t n_out, void* stream) {
  if (!temb || !w_mod || !b_mod || !mod) return XEMA_EINVAL;
  return launch_mod(ModArgs{temb, w_mod, b_mod, mod, batch, temb_dim, n_out, 0, n_out}, reinterpret_cast<cudaStream_t>(stream));
}

int xema_op_ln_modulate(const void* in, int32_t in_is_f32, int64_t in_batch_rows, void* out, const float* shift,
                        const float* scale, int64_t mod_stride, int32_t batch, int32_t rows, int32_t D, float eps,
                        void* stream) {
  if (!in || !out || !shift || !scale) return XEMA_EINVAL;
  return launch_ln_modulate(in, in_is_f32, in_batch_rows, out, shift, scale, mod_stride, batch, rows, D, eps,
                            reinterpret_cast<cudaStream_t>(stream));
}

int xema_op_rmsnorm_rope(void* x, int64_t ld, int64_t batch_rows, const void* g, const float* rope, int32_t pos0,
                         int32_t batch, int32_t rows, int32_t heads, int32_t head_dim, float eps, void* stream) {
  if (!x || !g || !rope) return XEMA_EINVAL;
  return launch_rmsnorm_rope(x, ld, batch_rows, g, rope, pos0, batch, rows, heads, head_dim, eps,
                             reinterpret_cast<cudaStream_t>(stream));
}

static GemmLaunch gemm_launch_of(const xema_gemm_args* a, void* status_dev) {
  GemmLaunch g{};
  g.bias = a->bias; g.out = a->out; g.ldo = a->ldo; g.out_batch_rows = a->out_batch_rows;
  g.resid = a->resid; g.ldr = a->ldr; g.resid_batch_rows = a->resid_batch_rows;
  g.gate = a->gate; g.gate_stride = a->gate_stride;
  g.batch = a->batch; g.rows = a->rows; g.N = a->N; g.K = a->K; g.epilogue = a->epilogue;
  g.norm_gain = a->norm_gain; g.rope = a->rope; g.rope_pos0 = a->rope_pos0; g.head_dim = a->head_dim;
  g.norm_cols = a->norm_cols; g.rms_eps = a->rms_eps; g.norm_out_scale = a->norm_out_scale;
  g.status = static_cast<unsigned int*>(status_dev);
  return g;
}

int xema_op_gemm(const xema_gemm_args* a, void* status_dev, void* stream) {
  if (!a) return XEMA_EINVAL;
  GemmLaunch g = gemm_launch_of(a, status_dev);
  int rc = gemm_prepare(&g, a->a, a->lda, a->a_batch_rows, a->w, a->ldw);
  if (rc) return rc;
  return launch_gemm(g, reinterpret_cast<cudaStream_t>(stream));
}

int xema_gemm_tile(const xema_gemm_args* a, int32_t* pair, int32_t* block_n) {
  if (!a || !pair || !block_n) return XEMA_EINVAL;
  GemmLaunch g = gemm_launch_of(a, nullptr);
  int rc = gemm_tile(&g);
  if (rc) return rc;
  *pair = g.pair;
  *block_n = g.block_n;
  return XEMA_OK;
}

int xema_op_gemm_in_tile(const xema_gemm_args* a, int32_t pair, int32_t block_n, void* status_dev, void* stream) {
  if (!a) return XEMA_EINVAL;
  GemmLaunch g = gemm_launch_of(a, status_dev);
  const int tile[2] = {pair, block_n};
  int rc = gemm_prepare(&g, a->a, a->lda, a->a_batch_rows, a->w, a->ldw, tile);
  if (rc) return rc;
  return launch_gemm(g, reinterpret_cast<cudaStream_t>(stream));
}

int xema_op_attention(const void* q, int64_t ldq, int64_t q_batch_rows, const void* k, const void* v, int64_t ldkv,
                      int64_t kv_batch_rows, void* o, float* lse, int32_t batch, int32_t rows, int32_t keys,
                      int32_t heads, int32_t head_dim, float q_scale, void* status_dev, void* stream) {
  if (!(q_scale > 0.f)) return XEMA_EINVAL;
  AttnLaunch a{};
  a.o = o; a.lse = lse; a.batch = batch; a.rows = rows; a.keys = keys; a.heads = heads; a.head_dim = head_dim;
  a.q_scale = q_scale;
  a.status = static_cast<unsigned int*>(status_dev);
  int rc = attn_prepare(&a, q, ldq, q_batch_rows, k, v, ldkv, kv_batch_rows);
  if (rc) return rc;
  return launch_attention(a, reinterpret_cast<cudaStream_t>(stream));
}

int xema_last_cuda_error(void) { return t_last_cuda_error; }

}  // extern "C"
