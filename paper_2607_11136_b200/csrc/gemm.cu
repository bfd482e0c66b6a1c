// bf16 x bf16 -> fp32 GEMM on the 5th-generation tensor cores (tcgen05) with the fused epilogues of
// the DiT block.
//
//   acc[b, i, n] = sum_k A[b, i, k] * W[n, k]          (both operands K-major)
//
// One kernel, two forms.  A persistent grid of 192-thread CTAs walks over output tiles:
//   PAIR    CTA pairs (two neighbouring SMs) share one 256 x 256 or 256 x 128 tile.  Each CTA loads its own
//           128 rows of A and one half of the W tile, so a stage of the wide tile costs 32 KB of shared-
//           memory fill per SM and every MMA reads 8 KB of operands per SM; the even CTA issues
//           tcgen05.mma.cta_group::2 (M = 256), which accumulates 128 rows in the TMEM of each CTA.
//   single  one CTA per 128 x 128, 128 x 64 or (gated epilogues, few rows) 128 x 32 tile.
// pick_tile says which when.
//
//   warp 0    TMA producer: tiles of A and W into a ring of shared-memory stages (128-byte swizzle)
//   warp 1    owns TMEM; converged warp, one elected lane issues tcgen05.mma into one of two fp32
//             accumulators in TMEM and commits stage releases / accumulator-ready
//   warps 2-5 epilogue (thread = output row) of the finished accumulator, while the next tile's main
//             loop fills the other one
// Barriers of the pair form:
//   full[s]        barrier of the even CTA: its producer expects the bytes of both CTAs, and both
//                  CTAs' loads complete on it (an expect-tx arrival sent from the peer CTA for every
//                  stage halved the speed of the whole loop)
//   empty[s]       one barrier per CTA, released for both by a multicast commit
//   tmem_full[a]   one barrier per CTA, same commit form
//   tmem_empty[a]  barrier of the even CTA: the four epilogue warps of both CTAs arrive
//
// The epilogue must not wait for global memory: bias and gate of the tile go to shared memory, the
// residual arrives by TMA in 32-column chunks and the rotation angles in registers, all requested
// while the main loop still runs, and the results leave through shared memory by TMA stores.  With
// plain loads in the chunk loop a 256-column tile took 11 000 (GELU) to 16 000 cycles (RMSNorm + RoPE,
// gated) whatever the shape -- 1300 to 3500 cycles of load latency per chunk -- which is 6 to 8 us at the
// end of every launch.
//
// A row's result depends only on (row, N, K): every form accumulates K in the same order, 16 at a
// time, so outputs are bit-identical however rows are chunked and whichever tile is chosen.
#include <algorithm>

#include "kernels.h"
#include "sm100.cuh"

namespace xema {
using namespace sm100;

namespace {
constexpr int BM = 128;          // rows per CTA
constexpr int BK = 64;
constexpr int GEMM_THREADS = 192;
constexpr int GROUP_M = 8;
constexpr int A_TILE_BYTES = BM * BK * 2;
constexpr int CHUNK = 32;        // columns per epilogue step
constexpr int BUF_BYTES = 4096;  // one staging buffer: 32 rows x 32 columns of fp32, or of bf16 in its first half
constexpr int HALF_BUF = BUF_BYTES / 2;

template <int EPI>
constexpr bool kGated = EPI == XEMA_EPI_GATE_RES_F32 || EPI == XEMA_EPI_GATE_RES_BF16;

// The wide tile has room for five stages and a ring of four residual chunks per epilogue warp, or (DEEP) for six stages
// and two chunks.  The sixth stage keeps the main loop fed over many tiles, the longer ring shortens the epilogue
// of a CTA's last one: 5 + 4 against 6 + 2 with a bf16 residual, K = 3072, N = 3072, us: 4444 rows 76.3 / 77.9, 4608
// 77.0 / 77.9, 8888 149.6 / 145.5, 17776 292 / 283, 36000 575 / 554.  With an fp32 residual (K = 12288) 6 + 2 is 0 to 2 %
// slower at every size.
template <int EPI, int BN, bool PAIR, bool DEEP = false>
struct GemmCfg {
  static constexpr int W_ROWS = PAIR ? BN / 2 : BN;            // rows of W a CTA loads per K block
  static constexpr int W_TILE_BYTES = W_ROWS * BK * 2;
  // K blocks of 64 per stage.  The K block of a smaller tile is short (128 to 256 cycles of MMA), and
  // with a stage per block the barrier round of each one takes longer than that: 8888 x 12288 x 3072 with
  // 64-column tiles 936 us, with two blocks per stage 769 (335 cycles per K block, 73 B/clk of fill).
  static constexpr int KSUB = BN == 256 ? 1 : 2;
  static constexpr int STAGE_BYTES = KSUB * (A_TILE_BYTES + W_TILE_BYTES);
  static constexpr int OFF_W = KSUB * A_TILE_BYTES;            // in a stage
  // staging buffers per epilogue warp: the gated epilogues keep residual chunks in flight
  static constexpr int RING = kGated<EPI> && BN == 256 && !DEEP ? 4 : 2;
  static constexpr int RING_BYTES = 4 * RING * BUF_BYTES;
  static constexpr int STAGES = BN == 256 ? (kGated<EPI> && !DEEP ? 5 : 6) : 196608 / STAGE_BYTES;
  static constexpr int OFF_RING = STAGES * STAGE_BYTES;
  static constexpr int OFF_BIAS = OFF_RING + RING_BYTES;       // float [BN]: bias
  static constexpr int OFF_GATE = OFF_BIAS + BN * 4;           // float [BN]: gate, or [2][128]: RMSNorm gains
  static constexpr int OFF_BAR = OFF_GATE + (kGated<EPI> ? BN * 4 : 1024);
  static constexpr int SMEM_BYTES = OFF_BAR + 384;
  static constexpr int TMEM_COLS = 2 * BN;   // a power of two from 32 on
  static_assert((2 * STAGES + 4 + 4 * RING) * 8 + 8 <= 384, "barrier area");
  static_assert(SMEM_BYTES <= 232448, "shared memory of one SM");
};

struct GemmParams {
  const __nv_bfloat16* bias;
  const float* gate;
  long long gate_stride;
  int batch, rows, N, K;
  int resid_batch, resid_rows;      // 1: the residual has a batch dimension / rows of its own, 0: the same for all
  unsigned int* status;
  // XEMA_EPI_BIAS_NORM_ROPE only: heads that start below column norm_cols get RMSNorm * gain
  // and RoPE in the epilogue (a thread owns whole rows, hence whole heads, of the tile)
  const __nv_bfloat16* norm_gain;   // [head_dim]
  const float* rope;                // [token][head_dim/2][cos, sin]
  int rope_pos0, head_dim, norm_cols;
  float rms_eps, norm_out_scale;
  // the first cols2 columns: another result (map_res), gain and factor
  const __nv_bfloat16* norm_gain2;
  float norm_out_scale2;
  int cols2;
};

__device__ __forceinline__ float gelu_tanh_f(float z) {
  const float u = 0.7978845608028654f * fmaf(0.044715f * z * z, z, z);
  return 0.5f * z * (1.f + tanh_approx(u));
}

// ---- staging buffers: row = lane, 16-byte pieces swizzled as the TMA boxes expect them ---------
// fp32: 128-byte rows, 128-byte swizzle; bf16: 64-byte rows, 64-byte swizzle.
__device__ __forceinline__ uint8_t* piece_f32(uint8_t* buf, int lane, int q) { return buf + lane * 128 + ((q ^ (lane & 7)) << 4); }
__device__ __forceinline__ uint8_t* piece_b16(uint8_t* buf, int lane, int q) {
  return buf + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4);
}
__device__ __forceinline__ void put_b16(uint8_t* buf, int lane, const float (&v)[CHUNK]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    *reinterpret_cast<uint4*>(piece_b16(buf, lane, q)) =
        make_uint4(pack_bf16x2(v[8 * q], v[8 * q + 1]), pack_bf16x2(v[8 * q + 2], v[8 * q + 3]),
                   pack_bf16x2(v[8 * q + 4], v[8 * q + 5]), pack_bf16x2(v[8 * q + 6], v[8 * q + 7]));
}

// Accumulator chunk + bias (broadcast reads of the tile's bias in shared memory).
__device__ __forceinline__ void load_chunk(uint32_t t_addr, const float* bias, float (&v)[CHUNK]) {
  tmem_ld32(t_addr, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
  float4 bb[CHUNK / 4];
#pragma unroll
  for (int q = 0; q < CHUNK / 4; ++q) bb[q] = reinterpret_cast<const float4*>(bias)[q];
  tmem_ld_wait_on(*reinterpret_cast<uint32_t(*)[32]>(&v[0]));
#pragma unroll
  for (int q = 0; q < CHUNK / 4; ++q) {
    v[4 * q + 0] += bb[q].x;
    v[4 * q + 1] += bb[q].y;
    v[4 * q + 2] += bb[q].z;
    v[4 * q + 3] += bb[q].w;
  }
}

struct TileCoord {
  int b, mt, nt;
};
__device__ __forceinline__ TileCoord tile_coord(int tile, int m_tiles, int n_tiles) {
  const int per_batch = m_tiles * n_tiles;
  TileCoord c;
  c.b = tile / per_batch;
  const int t = tile - c.b * per_batch;
  const int group_size = GROUP_M * n_tiles;
  const int g = t / group_size;
  const int first_m = g * GROUP_M;
  const int gm = min(GROUP_M, m_tiles - first_m);
  const int in_group = t - g * group_size;
  c.mt = first_m + in_group % gm;
  c.nt = in_group / gm;
  return c;
}

// Limit of one drain wait after a give-up (about 50 ms): long enough for any copy in flight,
// short enough that several of them in a row stay far below the limit of a regular wait.
constexpr long long kDrainLimitCycles = 100000000ll;

// The narrow single-CTA tiles serve launches of a few microseconds, which meet every line of the epilogue for the first time:
// each costs a trip of the instruction fetch to L2.  Their epilogue warps therefore rehearse one chunk while the CTA waits
// for earlier launches -- the same code on whatever TMEM and the staging ring hold, without waits, global accesses or
// stores.  Block of 288 x 512: 50.2 -> 48.2 us.  The other tiles only lose by it (1101 x 1536, all tiles: 120.3 -> 122.3).
template <int BN, bool PAIR>
constexpr bool kRehearse = !PAIR && BN <= 64;

// One epilogue warp: its staging ring and the chunks of one tile.
template <int EPI, int BN, bool PAIR, bool DEEP>
struct Epilogue {
  using Cfg = GemmCfg<EPI, BN, PAIR, DEEP>;
  static constexpr int RING = Cfg::RING;
  const GemmParams& p;
  const CUtensorMap* map_out;   // of the tile's result
  const CUtensorMap* map_res;
  uint8_t* ring;          // [RING][BUF_BYTES]
  uint64_t* rbar;         // [RING] residual chunk has arrived
  const float* bias;      // [BN], shared memory
  const float* gate;      // [BN] (gated) or the tile's RMSNorm gain
  volatile uint32_t* abort_flag;
  int lane;
  int rlane;              // row of a residual chunk that belongs to this lane
  bool dry = false;       // rehearsal
  float out_scale = 1.f;  // factor of the tile's normalised heads
  int col0 = 0;           // column of the product that is column 0 of the tile's result
  uint32_t used = 0;      // chunks worked on so far (buffer = used % RING)
  uint32_t asked = 0;     // residual chunks requested so far

  __device__ __forceinline__ bool rehearsing() const { return kRehearse<BN, PAIR> && dry; }
  __device__ __forceinline__ void request(int b, int row0, int n0) {   // whole warp; lane 0 acts
    if (lane == 0) {
      uint64_t* bar = rbar + asked % RING;
      mbar_expect_tx(bar, EPI == XEMA_EPI_GATE_RES_F32 ? BUF_BYTES / 2 : BUF_BYTES);
      tma_load_3d(ring + (asked % RING) * BUF_BYTES, map_res, bar, n0, p.resid_rows ? row0 : 0, p.resid_batch ? b : 0);
    }
    __syncwarp();
    ++asked;
  }
  // The chunk in buffer used % RING is complete in shared memory: send it off.
  __device__ __forceinline__ void send(uint8_t* buf, int b, int row0, int n0) {
    fence_proxy_async_smem();
    __syncwarp();
    if (rehearsing()) return;
    if (lane == 0) {
      tma_store_3d(map_out, buf, n0 - col0, row0, b);
      bulk_commit();
    }
    ++used;
  }
  // Buffer for the next chunk of an epilogue without residual: its earlier store has been read.
  __device__ __forceinline__ uint8_t* next_buf() {
    if (lane == 0) bulk_wait_read<RING - 1>();
    __syncwarp();
    // RMSNorm + RoPE: results in the first half of the ring, angles in the second
    static_assert(EPI != XEMA_EPI_BIAS_NORM_ROPE || RING == 2, "two results and one block of angles");
    return ring + (used % RING) * (EPI == XEMA_EPI_BIAS_NORM_ROPE ? HALF_BUF : BUF_BYTES);
  }

  __device__ __forceinline__ bool gated_tile(int b, int row0, int n_base, uint32_t t_addr) {
#pragma unroll 1
    for (int ch = 0; ch < (rehearsing() ? 1 : BN / CHUNK); ++ch) {
      uint8_t* buf = ring + (used % RING) * BUF_BYTES;
      if (!rehearsing() && !mbar_wait_warp(rbar + used % RING, (used / RING) & 1u, abort_flag)) return false;
      float v[CHUNK];
      load_chunk(t_addr + ch * CHUNK, bias + ch * CHUNK, v);
      const float4* g = reinterpret_cast<const float4*>(gate + ch * CHUNK);
      if constexpr (EPI == XEMA_EPI_GATE_RES_F32) {
        // out fp32 = resid(bf16) + gate * v
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 x = *reinterpret_cast<const uint4*>(piece_b16(buf, rlane, q));
          const float4 g0 = g[2 * q], g1 = g[2 * q + 1];
          v[8 * q + 0] = fmaf(g0.x, v[8 * q + 0], bf16_lo(x.x));
          v[8 * q + 1] = fmaf(g0.y, v[8 * q + 1], bf16_hi(x.x));
          v[8 * q + 2] = fmaf(g0.z, v[8 * q + 2], bf16_lo(x.y));
          v[8 * q + 3] = fmaf(g0.w, v[8 * q + 3], bf16_hi(x.y));
          v[8 * q + 4] = fmaf(g1.x, v[8 * q + 4], bf16_lo(x.z));
          v[8 * q + 5] = fmaf(g1.y, v[8 * q + 5], bf16_hi(x.z));
          v[8 * q + 6] = fmaf(g1.z, v[8 * q + 6], bf16_lo(x.w));
          v[8 * q + 7] = fmaf(g1.w, v[8 * q + 7], bf16_hi(x.w));
        }
      } else {
        // out bf16 = resid(fp32) + gate * v
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 x = *reinterpret_cast<const float4*>(piece_f32(buf, rlane, q));
          const float4 gg = g[q];
          v[4 * q + 0] = fmaf(gg.x, v[4 * q + 0], x.x);
          v[4 * q + 1] = fmaf(gg.y, v[4 * q + 1], x.y);
          v[4 * q + 2] = fmaf(gg.z, v[4 * q + 2], x.z);
          v[4 * q + 3] = fmaf(gg.w, v[4 * q + 3], x.w);
        }
      }
      __syncwarp();                                    // every lane has read its residual row
      if constexpr (EPI == XEMA_EPI_GATE_RES_F32) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<float4*>(piece_f32(buf, lane, q)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      } else {
        put_b16(buf, lane, v);
      }
      send(buf, b, row0, n_base + ch * CHUNK);
      // the buffer of the chunk before this one takes the next residual once its store has been read
      if (ch > 0 && ch - 1 + RING < BN / CHUNK) {
        if (lane == 0) bulk_wait_read<1>();
        __syncwarp();
        request(b, row0, n_base + (ch - 1 + RING) * CHUNK);
      }
    }
    return true;
  }

  __device__ __forceinline__ void plain_chunk(int b, int row0, int n_base, int col, uint32_t t_addr) {
    float v[CHUNK];
    uint8_t* buf = next_buf();
    load_chunk(t_addr + col, bias + col, v);
    if constexpr (EPI == XEMA_EPI_BIAS_GELU) {
#pragma unroll
      for (int t = 0; t < CHUNK; ++t) v[t] = gelu_tanh_f(v[t]);
    }
    put_b16(buf, lane, v);
    send(buf, b, row0, n_base + col);
  }

  // The angles of the warp's 32 rows for 32 columns from column c of a head on, 16 per row.  A warp reads four rows of 128 bytes at a
  // time; own_angles hands every lane its row through shared memory.  With a row per lane each load met 32 lines, and the epilogue
  // of the K | V | Q products was bound by that: 8000 rows x 3072 columns, K = 1024, heads of 128, 54.2 -> 48.6 us with 256 x 256
  // tiles, 63.3 -> 58.1 with 128 x 128, heads of 64 48.5 -> 45.8 and 51.0 -> 52.2, with 128 x 64 83.9 -> 72.4.  Heads of 64 in 128 x 128
  // tiles are the one form that can lose: launches chained, 5200 x 2304 x 768 22.5 -> 23.3, 2200 x 2048 x 1024 12.2 -> 12.5, 4650 x 3072 x
  // 1024 29.3 -> 29.9, from K = 1280 on 1 to 3 % faster (3650 x 3840 x 1280 35.1 -> 34.2, 1100 x 6144 x 2048 28.5 -> 28.1).  A row per lane for
  // that form alone gives 22.9, 12.4, 29.6, 35.2 and 27.6: not kept.  The epilogue takes 245 to 249 of 255 registers (226 to 232 before).
  __device__ __forceinline__ void load_angles(int row0, int c, float4 (&cs)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int row = min(row0 + 4 * q + (lane >> 3), p.rows - 1);
      cs[q] = __ldg(reinterpret_cast<const float4*>(p.rope + (size_t)(p.rope_pos0 + row) * p.head_dim + c) + (lane & 7));
    }
  }
  __device__ __forceinline__ void own_angles(float4 (&cs)[8]) {
    uint8_t* buf = ring + BUF_BYTES;
#pragma unroll
    for (int q = 0; q < 8; ++q) *reinterpret_cast<float4*>(piece_f32(buf, 4 * q + (lane >> 3), lane & 7)) = cs[q];
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 8; ++q) cs[q] = *reinterpret_cast<const float4*>(piece_f32(buf, lane, q));
    __syncwarp();
  }
  // acc + bias, RMSNorm over each head, gain, rotation of adjacent pairs by the token's angles.
  // First the head norms from a pass over the accumulator, then 32 columns of every head per
  // step, so that a row's angles are loaded once per tile and not once per head.
  template <int DH>
  __device__ __forceinline__ void norm_rope_tile(int b, int row0, int n_base, uint32_t t_addr, float4 (&cs)[8]) {
    constexpr int HEADS = BN / DH;
    const int norm_heads = min(HEADS, max(0, (p.norm_cols - n_base) / DH));
    float rstd[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int h = 0; h < norm_heads; ++h) {
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 1
      for (int c = 0; c < DH; c += CHUNK) {
        float v[CHUNK];
        load_chunk(t_addr + h * DH + c, bias + h * DH + c, v);
#pragma unroll
        for (int t = 0; t < CHUNK; t += 4) {
          s0 = fmaf(v[t], v[t], s0);
          s1 = fmaf(v[t + 1], v[t + 1], s1);
          s2 = fmaf(v[t + 2], v[t + 2], s2);
          s3 = fmaf(v[t + 3], v[t + 3], s3);
        }
      }
      const float r = rsqrtf(((s0 + s1) + (s2 + s3)) * (1.f / DH) + p.rms_eps) * out_scale;
#pragma unroll
      for (int i = 0; i < 4; ++i) rstd[i] = h == i ? r : rstd[i];
    }
#pragma unroll 1
    for (int c = 0; c < DH; c += CHUNK) {
      if (norm_heads > 0) own_angles(cs);
      // the angles of the next step are requested before this one's heads, which hide the trip to global memory
      // (with the warp index uniform, a step of 8 blocks of 333 x 1024 tokens 483 -> 450 us, a block of 1101 x 1536 129 -> 123,
      // one of 288 x 512 52.6 -> 50.2)
      float4 ahead[8];
      const bool more = c + CHUNK < DH && norm_heads > 0 && !rehearsing();
      if (more) load_angles(row0, c + CHUNK, ahead);
#pragma unroll 1
      for (int h = 0; h < HEADS; ++h) {
        const int col = h * DH + c;
        if (h >= norm_heads) {                     // the V half of a K | V product gets the bias only
          plain_chunk(b, row0, n_base, col, t_addr);
          continue;
        }
        const float r = h == 0 ? rstd[0] : h == 1 ? rstd[1] : h == 2 ? rstd[2] : rstd[3];
        float v[CHUNK];
        uint8_t* buf = next_buf();
        load_chunk(t_addr + col, bias + col, v);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 g = reinterpret_cast<const float4*>(gate + c)[q];
          const float a0 = v[4 * q + 0] * r * g.x, c0 = v[4 * q + 1] * r * g.y;
          const float a1 = v[4 * q + 2] * r * g.z, c1 = v[4 * q + 3] * r * g.w;
          v[4 * q + 0] = a0 * cs[q].x - c0 * cs[q].y;
          v[4 * q + 1] = a0 * cs[q].y + c0 * cs[q].x;
          v[4 * q + 2] = a1 * cs[q].z - c1 * cs[q].w;
          v[4 * q + 3] = a1 * cs[q].w + c1 * cs[q].z;
        }
        put_b16(buf, lane, v);
        send(buf, b, row0, n_base + col);
      }
      if (more) {
#pragma unroll
        for (int q = 0; q < 8; ++q) cs[q] = ahead[q];
      }
    }
  }
};

template <int EPI, int BN, bool PAIR, bool DEEP>
__device__ __forceinline__ void gemm_body(const CUtensorMap& map_a, const CUtensorMap& map_w, const CUtensorMap& map_out,
                                          const CUtensorMap& map_res, const GemmParams& p) {
  using Cfg = GemmCfg<EPI, BN, PAIR, DEEP>;
  constexpr int STAGES = Cfg::STAGES, RING = Cfg::RING, KSUB = Cfg::KSUB;
  constexpr bool GATED = kGated<EPI>;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Cfg::OFF_BAR);
  uint64_t* empty = full + STAGES;
  uint64_t* tmem_full = empty + STAGES;
  uint64_t* tmem_empty = tmem_full + 2;
  uint64_t* res_full = tmem_empty + 2;               // [4][RING]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(res_full + 4 * RING);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0;   // 0: even CTA (issues the MMAs), 1: its peer
  const int worker = PAIR ? blockIdx.x >> 1 : blockIdx.x, n_workers = PAIR ? gridDim.x >> 1 : gridDim.x;
  constexpr int TM = PAIR ? 2 * BM : BM;                // rows per tile
  const int m_tiles = (p.rows + TM - 1) / TM;
  const int n_tiles = p.N / BN;
  const int k_blocks = p.K / BK, k_stages = (k_blocks + KSUB - 1) / KSUB;
  const bool aligned = (smem_u32(smem) & 1023u) == 0;   // the swizzled tiles need a 1024-byte aligned base
  const int total_tiles = aligned ? p.batch * m_tiles * n_tiles : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&tmem_full[s], 1);
      mbar_init(&tmem_empty[s], PAIR ? 8 : 4);
    }
    if (GATED)
      for (int s = 0; s < 4 * RING; ++s) mbar_init(&res_full[s], 1);
    *abort_flag = aligned ? 0u : 1u;
    fence_mbar_init();
    prefetch_tmap(&map_a);
    prefetch_tmap(&map_w);
    prefetch_tmap(&map_out);
    if (GATED || p.cols2) prefetch_tmap(&map_res);
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(tmem_slot, Cfg::TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) {
    cluster_arrive();      // both CTAs' barriers exist before anything arrives on them remotely
    cluster_wait();
  }
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);   // uniform, like the warp index
  if (threadIdx.x == 0) grid_dep_launch();

  if (warp == 0) {
    // ---------------- TMA producer (one per CTA) ----------------
    {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      // ks: stage-sized step along K; the last one may hold fewer K blocks
      auto load_a = [&](int st, const TileCoord& c, int ks) {
        uint8_t* sa = smem + st * Cfg::STAGE_BYTES;
#pragma unroll
        for (int u = 0; u < KSUB; ++u) {
          const int kb = ks * KSUB + u;
          if (KSUB > 1 && kb >= k_blocks) break;
          if constexpr (PAIR)
            tma_load_3d_pair(sa + u * A_TILE_BYTES, &map_a, mapa_shared(smem_u32(&full[st]), 0), kb * BK,
                             (c.mt * 2 + (int)rank) * BM, c.b);
          else
            tma_load_3d(sa + u * A_TILE_BYTES, &map_a, &full[st], kb * BK, c.mt * BM, c.b);
        }
      };
      auto load_w = [&](int st, const TileCoord& c, int ks) {   // with the stage's expected bytes
        uint8_t* sb = smem + st * Cfg::STAGE_BYTES + Cfg::OFF_W;
        const int bytes = min(KSUB, k_blocks - ks * KSUB) * (A_TILE_BYTES + Cfg::W_TILE_BYTES);
        if (!PAIR) mbar_expect_tx(&full[st], bytes);
        else if (rank == 0) mbar_expect_tx(&full[st], 2 * bytes);
#pragma unroll
        for (int u = 0; u < KSUB; ++u) {
          const int kb = ks * KSUB + u;
          if (KSUB > 1 && kb >= k_blocks) break;
          if constexpr (PAIR)
            tma_load_3d_pair(sb + u * Cfg::W_TILE_BYTES, &map_w, mapa_shared(smem_u32(&full[st]), 0), kb * BK,
                             c.nt * BN + (int)rank * (BN / 2), 0);
          else
            tma_load_3d(sb + u * Cfg::W_TILE_BYTES, &map_w, &full[st], kb * BK, c.nt * BN, 0);
        }
      };
      // The weights of the first stages do not depend on earlier launches (see launch_kernel): they
      // are requested before the wait for those, the activations after it.
      const int early = worker < total_tiles ? min(STAGES, k_stages) : 0;
      if (early > 0) {
        const TileCoord c = tile_coord(worker, m_tiles, n_tiles);
        if (elect_one())
          for (int kb = 0; kb < early; ++kb) load_w(kb, c, kb);
        __syncwarp();
        grid_dep_wait();
        if (elect_one())
          for (int kb = 0; kb < early; ++kb) load_a(kb, c, kb);
        __syncwarp();
        if (early == STAGES) phase = 1;
        else stage = early;
      }
      for (int tile = worker; ok && tile < total_tiles; tile += n_workers) {
        const TileCoord c = tile_coord(tile, m_tiles, n_tiles);
        for (int kb = tile == worker ? early : 0; kb < k_stages; ++kb) {
          if (!(ok = mbar_wait_warp(&empty[stage], phase ^ 1, abort_flag))) break;
          if (elect_one()) {
            load_w(stage, c, kb);
            load_a(stage, c, kb);
          }
          __syncwarp();
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      // Tail (pair): the same waits as for STAGES further fills, without filling.  They return once
      // the commits that release this CTA's last fills (arrivals multicast by the even CTA) have
      // landed here, so none of them can reach this CTA's barriers after it has left.
      if constexpr (PAIR) {
        for (int s = 0; ok && s < STAGES; ++s) {
          ok = mbar_wait_warp(&empty[stage], phase ^ 1, abort_flag);
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (!ok) {
        // Gave up.  Copies already issued must land before a CTA leaves.  Pair: all of them complete
        // on the even CTA's full[] barriers, so the even CTA waits (bounded, and without looking
        // at the abort flag) for the latest fill of every stage, which covers the bytes of both CTAs
        // wherever both issued; the closing cluster barrier then keeps the peer until that is done.
        // A short settling time covers loads of a stage that only one of the two CTAs still issued.
        if (rank == 0 && lane == 0) {
          for (int s = 0; s < STAGES; ++s) {
            const int st = (stage + s) % STAGES;                 // oldest outstanding first
            const uint32_t ph = (st < stage) ? phase : (phase ^ 1);
            volatile uint32_t dummy = 0;
            mbar_wait_slow(&full[st], ph, &dummy, kDrainLimitCycles);
          }
        }
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (pair: even CTA only) ----------------
    // The whole warp walks the loop and waits together; one elected lane issues.  (A lone
    // thread of a diverged warp issues MMAs markedly slower than the tensor pipe retires them.)
    if (rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(TM, BN, false, false);
      // Descriptors are built once and advanced by adding constants (the start-address field
      // counts 16-byte units and never carries out of its 14 bits inside shared memory).
      const uint64_t a_desc0 = smem_desc_sw128(smem_u32(smem), 16, 1024);
      const uint64_t b_desc0 = smem_desc_sw128(smem_u32(smem + Cfg::OFF_W), 16, 1024);
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      for (int tile = worker; ok && tile < total_tiles; tile += n_workers) {
        // pair: the peer's epilogue warps arrive from their own CTA, hence the cluster-scope acquire
        if (!(ok = __all_sync(0xffffffffu, mbar_wait_cluster(&tmem_empty[acc], acc_phase ^ 1, abort_flag)))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        uint32_t accumulate = 0;
#pragma unroll 1
        for (int ks = 0; ks < k_stages; ++ks) {
          if (!(ok = mbar_wait_warp(&full[stage], phase, abort_flag))) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t soff = (uint64_t)(stage * (Cfg::STAGE_BYTES >> 4));
            const uint64_t da = a_desc0 + soff, db = b_desc0 + soff;
            auto mma = [&](uint64_t ad, uint64_t bd, uint32_t acc_in) {
              if constexpr (PAIR) mma_ss_pair(d_tmem, ad, bd, idesc, acc_in);
              else mma_ss(d_tmem, ad, bd, idesc, acc_in);
            };
#pragma unroll
            for (int u = 0; u < KSUB; ++u) {
              if (KSUB > 1 && ks * KSUB + u >= k_blocks) break;
              const uint64_t ua = da + (uint64_t)(u * (A_TILE_BYTES >> 4)), ub = db + (uint64_t)(u * (Cfg::W_TILE_BYTES >> 4));
              mma(ua, ub, u > 0 ? 1 : accumulate);
              mma(ua + 2, ub + 2, 1);
              mma(ua + 4, ub + 4, 1);
              mma(ua + 6, ub + 6, 1);
            }
            if constexpr (PAIR) mma_commit_pair(&empty[stage]);
            else mma_commit(&empty[stage]);
          }
          __syncwarp();
          accumulate = 1;
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        if (elect_one()) {
          if (PAIR) mma_commit_pair(&tmem_full[acc]);
          else mma_commit(&tmem_full[acc]);
        }
        __syncwarp();
        if (++acc == 2) { acc = 0; acc_phase ^= 1; }
      }
    }
  } else {
    // ---------------- epilogue (pair: each CTA its own 128 rows) ----------------
    const int quad = warp & 3;           // TMEM lanes [32*quad, 32*quad + 32) belong to this warp
    float* s_bias = reinterpret_cast<float*>(smem + Cfg::OFF_BIAS);
    float* s_gate = reinterpret_cast<float*>(smem + Cfg::OFF_GATE);
    Epilogue<EPI, BN, PAIR, DEEP> ep{p, &map_out, &map_res, smem + Cfg::OFF_RING + quad * RING * BUF_BYTES, res_full + quad * RING,
                               s_bias, s_gate, abort_flag, lane, p.resid_rows ? lane : 0};
    const int et = threadIdx.x - 64;     // 0..127
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    if constexpr (EPI == XEMA_EPI_BIAS_NORM_ROPE) {
      if (et < p.head_dim) {                           // read after the tile's barrier
        s_gate[et] = __bfloat162float(p.norm_gain[et]);
        if (p.cols2) s_gate[128 + et] = __bfloat162float(p.norm_gain2[et]);
      }
    }
    ep.dry = kRehearse<BN, PAIR>;                          // the first round is a rehearsal
    if constexpr (!kRehearse<BN, PAIR>) {
      grid_dep_wait();
    }
    for (int tile = worker; tile < total_tiles;) {
      const bool dry = ep.rehearsing();
      // The four warps meet (the previous tile's bias and gate are no longer read) and agree on going
      // on: a warp that gave up a wait still comes here, so that nobody waits for it.
      if (!(ok = named_barrier_and(1, 128, ok))) break;
      const TileCoord c = tile_coord(tile, m_tiles, n_tiles);
      const int row0 = (c.mt * (TM / BM) + (int)rank) * BM + quad * 32;
      const int n_base = c.nt * BN;
      const bool live = row0 < p.rows;   // rows past the end: nothing to read or store
      // everything the tile needs besides its accumulator, requested while the main loop runs
      if constexpr (GATED) {
        if (lane == 0) bulk_wait_read<0>();
        __syncwarp();
        if (live && !dry)
          for (int ch = 0; ch < (RING < BN / CHUNK ? RING : BN / CHUNK); ++ch) ep.request(c.b, row0, n_base + ch * CHUNK);
      }
      float4 cs[8];
      if constexpr (EPI == XEMA_EPI_BIAS_NORM_ROPE) {
        const bool second = n_base < p.cols2;
        ep.map_out = second ? &map_res : &map_out;
        ep.gate = second ? s_gate + 128 : s_gate;
        ep.out_scale = second ? p.norm_out_scale2 : p.norm_out_scale;
        ep.col0 = second ? 0 : p.cols2;
        if (live && n_base < p.norm_cols && !dry) ep.load_angles(row0, 0, cs);
      }
      for (int i = dry ? BN : et * 2; i < BN; i += 256) {
        const uint32_t bb = __ldg(reinterpret_cast<const uint32_t*>(p.bias + n_base + i));
        *reinterpret_cast<float2*>(s_bias + i) = make_float2(bf16_lo(bb), bf16_hi(bb));
        if constexpr (GATED)
          *reinterpret_cast<float2*>(s_gate + i) =
              ld_f2(p.gate + (size_t)c.b * p.gate_stride + n_base + i);
      }
      named_barrier(1, 128);
      if (!dry) ok = mbar_wait_warp(&tmem_full[acc], acc_phase, abort_flag);
      tc_fence_after();
      const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + (dry ? BN : acc * BN);
      if (live && ok) {
        if constexpr (GATED) {
          ok = ep.gated_tile(c.b, row0, n_base, t_addr);
        } else if constexpr (EPI == XEMA_EPI_BIAS_NORM_ROPE) {
          if (p.head_dim == 64) ep.template norm_rope_tile<64>(c.b, row0, n_base, t_addr, cs);
          else if constexpr (BN >= 128) ep.template norm_rope_tile<128>(c.b, row0, n_base, t_addr, cs);
        } else {
#pragma unroll 1
          for (int col = 0; col < (dry ? CHUNK : BN); col += CHUNK) ep.plain_chunk(c.b, row0, n_base, col, t_addr);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (dry) {
        ep.dry = false;
        grid_dep_wait();
        continue;
      }
      // The issuer asks for this accumulator again for the tile after next.  Without one nobody waits for the release, which in a pair
      // first waits for the warp's own writes (block of 1101 x 1536 112.1 -> 110.4 us, of 1055 x 1280 127.7 -> 126.7).
      if (lane == 0 && tile + 2 * n_workers < total_tiles) {
        if (PAIR) mbar_arrive_cluster(mapa_shared(smem_u32(&tmem_empty[acc]), 0));
        else mbar_arrive(&tmem_empty[acc]);
      }
      if (++acc == 2) { acc = 0; acc_phase ^= 1; }
      tile += n_workers;
    }
    grid_dep_wait();                     // (a CTA without tiles has not waited yet)
    if (GATED && !ok) {
      // gave up: the residual chunks already requested must land before the CTA leaves
      for (uint32_t i = ep.asked > (uint32_t)RING ? ep.asked - RING : 0; i < ep.asked; ++i) {
        volatile uint32_t dummy = 0;
        mbar_wait_slow(ep.rbar + i % RING, (i / RING) & 1u, &dummy, kDrainLimitCycles);
      }
    }
    if (lane == 0) bulk_wait<0>();       // this warp's stores are complete
    __syncwarp();
  }

  // Pair: neither CTA leaves (or frees TMEM) while the other may still read its shared memory, write
  // its TMEM or arrive on its barriers.
  tc_fence_before();
  __syncthreads();
  if (PAIR) {
    cluster_arrive();
    cluster_wait();
  }
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) tmem_dealloc_pair(tmem_base, Cfg::TMEM_COLS);
    else tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status) atomicExch(p.status, STATUS_TIMEOUT_MBARRIER);
}

template <int EPI, int BN>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w,
                 const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_res, const GemmParams p) {
  gemm_body<EPI, BN, false, false>(map_a, map_w, map_out, map_res, p);
}
template <int EPI, int BN, bool DEEP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
gemm_bf16_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w,
                      const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_res,
                      const GemmParams p) {
  gemm_body<EPI, BN, true, DEEP>(map_a, map_w, map_out, map_res, p);
}

// ---------------------------------------------------------------------------------------------
GemmParams make_params(const GemmLaunch& g) {
  GemmParams p;
  p.bias = (const __nv_bfloat16*)g.bias;
  p.gate = g.gate;
  p.gate_stride = g.gate_stride;
  p.batch = g.batch;
  p.rows = g.rows;
  p.N = g.N;
  p.K = g.K;
  p.resid_batch = g.resid_batch_rows * g.ldr != 0;
  p.resid_rows = g.ldr != 0;
  p.status = g.status;
  p.norm_gain = (const __nv_bfloat16*)g.norm_gain;
  p.rope = g.rope;
  p.rope_pos0 = g.rope_pos0;
  p.head_dim = g.head_dim;
  p.norm_cols = g.norm_cols;
  p.rms_eps = g.rms_eps;
  p.norm_out_scale = g.norm_out_scale > 0.f ? g.norm_out_scale : 1.f;
  p.norm_gain2 = (const __nv_bfloat16*)g.norm_gain2;
  p.norm_out_scale2 = g.norm_out_scale2 > 0.f ? g.norm_out_scale2 : 1.f;
  p.cols2 = g.cols2;
  return p;
}

template <int EPI, int BN>
int launch_single(const GemmLaunch& g, cudaStream_t stream, bool chained) {
  using Cfg = GemmCfg<EPI, BN, false>;
  static PerDeviceInt attr_done;
  auto kern = gemm_bf16_kernel<EPI, BN>;
  if (int rc = ensure_smem_attr(kern, Cfg::SMEM_BYTES, attr_done)) return rc;
  const long long tiles = (long long)g.batch * ((g.rows + BM - 1) / BM) * (g.N / BN);
  const int grid = (int)std::min<long long>(tiles, sm_count());
  return launch_kernel(kern, dim3(grid), GEMM_THREADS, Cfg::SMEM_BYTES, stream, chained, g.map_a, g.map_w, g.map_out, g.map_res,
                       make_params(g));
}

template <int EPI, int BN, bool DEEP = false>
int launch_pair(const GemmLaunch& g, cudaStream_t stream, bool chained) {
  using Cfg = GemmCfg<EPI, BN, true, DEEP>;
  static PerDeviceInt attr_done;
  auto kern = gemm_bf16_pair_kernel<EPI, BN, DEEP>;
  if (int rc = ensure_smem_attr(kern, Cfg::SMEM_BYTES, attr_done)) return rc;
  // A persistent grid must be resident all at once: ask how many CTA pairs fit on the device
  // (SMs are handed out to clusters in hardware groups, so it can be fewer than SMs / 2).
  static PerDeviceInt pairs_cache;
  const int dev = current_device();
  int max_pairs = pairs_cache.get(dev);
  if (max_pairs == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (sm_count() / 2), 1, 1);
    cfg.blockDim = dim3(GEMM_THREADS, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM_BYTES;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    if (e != cudaSuccess || n <= 0) {
      set_last_cuda_error((int)e);
      return XEMA_ECUDA;
    }
    max_pairs = std::min(n, sm_count() / 2);
    pairs_cache.set(dev, max_pairs);
  }
  const long long tiles = (long long)g.batch * ((g.rows + 2 * BM - 1) / (2 * BM)) * (g.N / BN);
  const int pairs = (int)std::min<long long>(tiles, max_pairs);
  return launch_kernel(kern, dim3(2 * pairs), GEMM_THREADS, Cfg::SMEM_BYTES, stream, chained, g.map_a, g.map_w, g.map_out,
                       g.map_res, make_params(g));
}

template <int EPI>
int launch_epi(const GemmLaunch& g, cudaStream_t stream, bool chained) {
  if constexpr (EPI == XEMA_EPI_GATE_RES_F32) {
    // six stages from four tiles a pair on (5.7 of them at 8888 rows x 3072 columns are 3 % faster, 2.9 at 4608 1 % slower)
    const long long tiles = (long long)g.batch * ((g.rows + 2 * BM - 1) / (2 * BM)) * (g.N / 256);
    if (g.pair && g.block_n == 256 && tiles > 4LL * (sm_count() / 2)) return launch_pair<EPI, 256, true>(g, stream, chained);
  }
  if (g.pair) return g.block_n == 256 ? launch_pair<EPI, 256>(g, stream, chained) : launch_pair<EPI, 128>(g, stream, chained);
  if (g.block_n == 128) return launch_single<EPI, 128>(g, stream, chained);
  if (g.block_n == 64) return launch_single<EPI, 64>(g, stream, chained);
  if constexpr (kGated<EPI>) return launch_single<EPI, 32>(g, stream, chained);
  return XEMA_EINVAL;
}

// Tile for a problem: the one with the shortest estimated time, waves x K blocks x nanoseconds per K
// block plus what its last tile's epilogue adds.  Measured (B200, shapes from 288 x 512 x 2048 to 8888 x 12288 x
// 3072): a K block takes 370-385 ns with 256 x 256 pair tiles, 212-270 with 256 x 128 pair tiles, 255-290 with
// 128 x 128 and 172-211 with 128 x 64 -- of a single CTA an MMA of 16 along K takes about 26 + operand bytes / 170 clocks (128 x 32 55,
// 128 x 64 62, 128 x 128 73; pairs of 256 x 128 69; without any loads the same) -- so a
// smaller tile is slower per flop and pays only where the larger one leaves SMs idle.  us for 256 x 256 /
// 256 x 128 / 128 x 128 / 128 x 64: 333 x 1024 x 4096 28.8 / 20.2 / 21.9 / 16.5, 1101 x 1536 x 6144 39.1 / 27.3 / 30.9 /
// 37.7, 2222 x 3072 x 3072 41.1 / 37.0 / 43.2 / 56.2, 4444 x 3072 x 3072 58.0 / 65.7 / 78.0 / 104.  128 x 32 exists for the
// gated epilogues, whose products are narrow: 288 x 512 x 2048 12.1 -> 10.4 us, a step of 8 blocks of 333 tokens
// x 1024 521 -> 500.  (Shorter tiles -- 32, 64 or 96 of the 128 rows filled -- are no faster: the MMAs are the same.)
// A pair's ends cost 700 ns more than its epilogue alone (its clusters start and end together): with them counted the pick takes 1.010
// times the best form, without them 1.023, over 447 products back to back (widths 512 to 3072, 170 to 6700 rows; 287 others 1.010 and
// 1.016), and single tiles of 128 x 128 get what is close to a wave either way.  us without / with: eight blocks of 333 x 1024 366.8 /
// 363.8, 1055 x 1280 129.6 / 125.6, 4251 x 768 225.6 / 216.2, two blocks of 4706 x 1280 810 / 800.  (Fitted freely the figures give
// 1.005, but 2.8 % more time for eight blocks of 847 x 2816, whose weights do not stay in L2.)  With every SM at it loads can take
// over: 3 x 680 x 2048 x 8192 52.0 us with 256 x 256 tiles, 44.6 without loads in the steady state (57 B/clk of fill a CTA).
// The 256 x 256 figure was taken under the power cap, as launches that need it run, the small tiles' at full clock, as
// theirs do.  Pairs are counted as SMs / 2, all of which are resident on a B200 (74); where fewer fit, the launch
// takes those and only the estimate is off.  The bits of a row do not depend on the choice.
struct Tile {
  int pair, block_n, block_ns, epilogue_ns;
};
constexpr Tile kTiles[] = {{1, 256, 372, 3700}, {1, 128, 230, 2200}, {0, 128, 265, 1000}, {0, 64, 180, 500}, {0, 32, 150, 400}};

bool tile_fits(const GemmLaunch& g, const Tile& t) {
  if (g.N % t.block_n) return false;
  if (t.block_n < 64 && g.epilogue != XEMA_EPI_GATE_RES_F32 && g.epilogue != XEMA_EPI_GATE_RES_BF16) return false;
  return g.epilogue != XEMA_EPI_BIAS_NORM_ROPE || t.block_n >= g.head_dim;   // whole heads only
}

void pick_tile(GemmLaunch* g) {
  const long long k_blocks = g->K / BK;
  long long best = 0;
  g->block_n = 0;
  for (const Tile& t : kTiles) {
    if (!tile_fits(*g, t)) continue;
    const int rows = t.pair ? 2 * BM : BM;
    const long long n = (long long)g->batch * ((g->rows + rows - 1) / rows) * (g->N / t.block_n);
    const long long workers = std::max(1, t.pair ? sm_count() / 2 : sm_count());
    const long long cost = (n + workers - 1) / workers * k_blocks * t.block_ns + t.epilogue_ns;
    if (!g->block_n || cost < best) {
      best = cost;
      g->block_n = t.block_n;
      g->pair = t.pair;
    }
  }
}

// The sizes and flags of a problem, without its pointers.
int check_shape(const GemmLaunch& g) {
  if (g.batch < 1 || g.rows < 0 || g.N < 128 || (g.N % 128) || g.K < 64 || (g.K % 64)) return XEMA_EINVAL;
  if (g.epilogue < XEMA_EPI_BIAS || g.epilogue > XEMA_EPI_BIAS_NORM_ROPE) return XEMA_EINVAL;
  if (g.epilogue != XEMA_EPI_BIAS_NORM_ROPE) return g.cols2 ? XEMA_EINVAL : XEMA_OK;
  if (g.cols2 < 0 || g.cols2 % 256 || g.cols2 >= g.N) return XEMA_EINVAL;    // whole tiles for either result
  if (g.head_dim != 64 && g.head_dim != 128) return XEMA_EINVAL;
  return g.norm_cols < 0 || g.norm_cols > g.N || g.norm_cols % g.head_dim || g.N % 256 || g.rope_pos0 < 0 ? XEMA_EINVAL : XEMA_OK;
}
}  // namespace

int launch_gemm(const GemmLaunch& g, cudaStream_t stream, bool chained) {
  if (g.rows == 0 || g.batch == 0) return XEMA_OK;
  switch (g.epilogue) {
    case XEMA_EPI_BIAS: return launch_epi<XEMA_EPI_BIAS>(g, stream, chained);
    case XEMA_EPI_BIAS_GELU: return launch_epi<XEMA_EPI_BIAS_GELU>(g, stream, chained);
    case XEMA_EPI_GATE_RES_F32: return launch_epi<XEMA_EPI_GATE_RES_F32>(g, stream, chained);
    case XEMA_EPI_GATE_RES_BF16: return launch_epi<XEMA_EPI_GATE_RES_BF16>(g, stream, chained);
    case XEMA_EPI_BIAS_NORM_ROPE: return launch_epi<XEMA_EPI_BIAS_NORM_ROPE>(g, stream, chained);
    default: return XEMA_EINVAL;
  }
}

int gemm_tile(GemmLaunch* g) {
  if (int rc = check_shape(*g)) return rc;
  pick_tile(g);
  return XEMA_OK;
}

int gemm_prepare(GemmLaunch* g, const void* a, long long lda, long long a_batch_rows, const void* w, long long ldw,
                 const int* tile) {
  if (int rc = check_shape(*g)) return rc;
  if (!a || !w || !g->bias || !g->out) return XEMA_EINVAL;
  const bool gated = g->epilogue == XEMA_EPI_GATE_RES_F32 || g->epilogue == XEMA_EPI_GATE_RES_BF16;
  if (gated && (!g->resid || !g->gate)) return XEMA_EINVAL;
  if (g->epilogue == XEMA_EPI_BIAS_NORM_ROPE) {
    if (!g->norm_gain || !g->rope) return XEMA_EINVAL;
    if ((reinterpret_cast<uintptr_t>(g->norm_gain) & 15) || (reinterpret_cast<uintptr_t>(g->rope) & 15)) return XEMA_EALIGN;
    if (g->cols2) {
      if (!g->out2 || !g->norm_gain2 || g->ldo2 < g->cols2) return XEMA_EINVAL;
      if ((g->ldo2 & 7) || (reinterpret_cast<uintptr_t>(g->out2) & 15)) return XEMA_EALIGN;
    }
  }
  // Result rows lie behind one another; residual rows may be shared (ldr = 0: one row for all,
  // resid_batch_rows = 0: the same rows for every batch element).
  const long long out_cols = g->N - g->cols2;
  if ((g->rows > 1 && g->ldo < out_cols) || (g->batch > 1 && (g->ldo < 1 || g->out_batch_rows < 1))) return XEMA_EINVAL;
  if (gated && (g->ldr < 0 || g->resid_batch_rows < 0)) return XEMA_EINVAL;
  if ((lda & 7) || (ldw & 7) || (g->ldo & 7) || (gated && (g->ldr & 7))) return XEMA_EALIGN;
  auto mis = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) != 0; };
  if (mis(a) || mis(w) || mis(g->bias) || mis(g->out) || (g->resid && mis(g->resid)) || (g->gate && mis(g->gate)))
    return XEMA_EALIGN;
  g->a = a;
  g->w = w;
  g->lda = lda;
  g->a_batch_rows = a_batch_rows;
  g->ldw = ldw;
  if (!tile) {
    pick_tile(g);
  } else {
    g->block_n = 0;
    for (const Tile& t : kTiles)
      if (t.pair == tile[0] && t.block_n == tile[1] && tile_fits(*g, t)) {
        g->pair = t.pair;
        g->block_n = t.block_n;
      }
    if (!g->block_n) return XEMA_EINVAL;
  }
  const long long rows = g->rows > 0 ? g->rows : 1;
  int rc = encode_tmap_bf16(&g->map_a, a, g->K, rows, g->batch, lda, a_batch_rows, BM);
  if (rc) return rc;
  // the pair forms load their W tile as two halves, one per CTA
  rc = encode_tmap_bf16(&g->map_w, w, g->K, g->N, 1, ldw, g->N, g->pair ? g->block_n / 2 : g->block_n);
  if (rc) return rc;
  // results leave, and residuals arrive, as boxes of 32 columns x 32 rows
  rc = encode_tmap_box32(&g->map_out, g->out, g->epilogue == XEMA_EPI_GATE_RES_F32, out_cols, rows, g->batch, g->ldo,
                         g->out_batch_rows * g->ldo);
  if (!rc && g->cols2)
    rc = encode_tmap_box32(&g->map_res, g->out2, false, g->cols2, rows, g->batch, g->ldo2, g->out2_batch_rows * g->ldo2);
  if (rc || !gated) return rc;
  const long long resid_stride = g->resid_batch_rows * g->ldr;
  return encode_tmap_box32(&g->map_res, g->resid, g->epilogue == XEMA_EPI_GATE_RES_BF16, g->N, g->ldr ? rows : 1,
                           resid_stride ? g->batch : 1, g->ldr, resid_stride);
}

}  // namespace xema
