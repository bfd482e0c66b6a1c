// HBM-bound kernels of the block: adaLN modulation GEMV, LayerNorm + modulate, and
// per-head RMSNorm + RoPE.  128-bit coalesced accesses, one warp per token row, warp-shuffle
// reductions, fp32 arithmetic on bf16 storage.
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "sm100.cuh"

namespace xema {

using sm100::bf16_hi;
using sm100::bf16_lo;
using sm100::grid_dep_launch;
using sm100::grid_dep_wait;
using sm100::ld_f4;
using sm100::ld_f8;
using sm100::ld_u4;
using sm100::pack_bf16x2;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------------------
// mod[b, j] = sum_k silu(temb[b,k]) * w[j,k] + bias[j]
// A warp takes kModRows output features at once: their weight rows are requested together, for up to
// 512 inputs before the wait for earlier launches (the weights do not depend on them); silu(temb) for
// all batch elements sits in shared memory, loaded 16 bytes at a time.  Bound by the latency of one trip to HBM for one
// batch element (which has an instance of its own: 80 registers instead of 128, so that three blocks fit an SM, and half of the
// code to fetch), by the products and reductions for several.  us back to back, before these two, the wide load and the
// six-shuffle reduction / with them: 1 x 6144 features 4.7 / 4.2 (as short as launches follow one another), 1 x 9216 5.2 /
// 4.2, 1 x 18432 7.2 / 6.2, 3 x 12288 10.0 / 8.3, 4 x 18432 12.4 / 10.3, 7 x 3072 10.3 / 6.5.
// ---------------------------------------------------------------------------------------
constexpr int kModWarps = 8;
constexpr int kModRows = 4;

// A load of weights that stays where it stands: an __ldg the compiler may move down to its use, behind the wait.
__device__ __forceinline__ uint4 ld_weights(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Features [j_first, j_end) of block `tile` of WARPS * kModRows of them, BATCH batch elements per pass over the weights (ONE_PASS: there
// are no more of them).
template <int WARPS, int BATCH, bool ONE_PASS>
__device__ __forceinline__ void mod_features(const ModArgs& a, int tile) {
  extern __shared__ float s_e[];  // [batch][Dt]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = a.j_first + (tile * WARPS + warp) * kModRows;
  const int n8 = a.Dt / 8;
  const __nv_bfloat16* w = static_cast<const __nv_bfloat16*>(a.w);
  auto weights = [&](int r, int k8) {
    return (j0 + r < a.j_end && k8 < n8) ? ld_weights(reinterpret_cast<const uint4*>(w + (size_t)(j0 + r) * a.Dt) + k8)
                                         : make_uint4(0u, 0u, 0u, 0u);
  };
  uint4 first[2][kModRows];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int r = 0; r < kModRows; ++r) first[u][r] = weights(r, u * 32 + lane);
  // the feature whose sum this lane ends up with, and its bias as it comes (a conversion here would wait for it)
  const int j_own = j0 + lane / 8;
  const unsigned short bias = j_own < a.j_end ? __ldg(static_cast<const unsigned short*>(a.bias) + j_own) : (unsigned short)0;
  grid_dep_launch();
  grid_dep_wait();
  for (int i = threadIdx.x; i < a.batch * n8; i += WARPS * 32) {
    float e[8];
    if ((reinterpret_cast<uintptr_t>(a.temb) & 15) == 0) {
      const uint4 t = ld_u4(static_cast<const uint4*>(a.temb) + i);
      e[0] = bf16_lo(t.x); e[1] = bf16_hi(t.x); e[2] = bf16_lo(t.y); e[3] = bf16_hi(t.y);
      e[4] = bf16_lo(t.z); e[5] = bf16_hi(t.z); e[6] = bf16_lo(t.w); e[7] = bf16_hi(t.w);
    } else {                          // (the operator takes any address; a plan's slot is aligned)
#pragma unroll
      for (int k = 0; k < 8; ++k) e[k] = __bfloat162float(*(static_cast<const volatile __nv_bfloat16*>(a.temb) + i * 8 + k));
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) e[k] = e[k] / (1.f + __expf(-e[k]));
    *reinterpret_cast<float4*>(s_e + i * 8) = make_float4(e[0], e[1], e[2], e[3]);
    *reinterpret_cast<float4*>(s_e + i * 8 + 4) = make_float4(e[4], e[5], e[6], e[7]);
  }
  __syncthreads();
  for (int b0 = 0; b0 < (ONE_PASS ? 1 : a.batch); b0 += BATCH) {
    float acc[kModRows][BATCH];
#pragma unroll
    for (int r = 0; r < kModRows; ++r)
#pragma unroll
      for (int b = 0; b < BATCH; ++b) acc[r][b] = 0.f;
    auto add = [&](const uint4 (&v)[kModRows], int k8) {
#pragma unroll
      for (int b = 0; b < BATCH; ++b) {
        if ((BATCH > 1 && b0 + b >= a.batch) || k8 >= n8) continue;
        const float4 e0 = *reinterpret_cast<const float4*>(s_e + (size_t)(b0 + b) * a.Dt + k8 * 8);
        const float4 e1 = *reinterpret_cast<const float4*>(s_e + (size_t)(b0 + b) * a.Dt + k8 * 8 + 4);
#pragma unroll
        for (int r = 0; r < kModRows; ++r) {
          float c = acc[r][b];
          c = fmaf(bf16_lo(v[r].x), e0.x, c); c = fmaf(bf16_hi(v[r].x), e0.y, c);
          c = fmaf(bf16_lo(v[r].y), e0.z, c); c = fmaf(bf16_hi(v[r].y), e0.w, c);
          c = fmaf(bf16_lo(v[r].z), e1.x, c); c = fmaf(bf16_hi(v[r].z), e1.y, c);
          c = fmaf(bf16_lo(v[r].w), e1.z, c); c = fmaf(bf16_hi(v[r].w), e1.w, c);
          acc[r][b] = c;
        }
      }
    };
    add(first[0], lane);
    add(first[1], 32 + lane);
    for (int k8 = 64 + lane; k8 < n8; k8 += 32) {
      uint4 v[kModRows];
#pragma unroll
      for (int r = 0; r < kModRows; ++r) v[r] = weights(r, k8);
      add(v, k8);
    }
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      if (BATCH > 1 && b0 + b >= a.batch) continue;
      // The four features' sums over the warp at once: after each of the first two steps a lane holds half as many of them.
      // Six shuffles instead of twenty; the values that are added are those of warp_sum, so are the bits.
      static_assert(kModRows == 4, "two halving steps");
      const bool hi = lane & 16, hi2 = lane & 8;
      float u0 = hi ? acc[2][b] : acc[0][b], u1 = hi ? acc[3][b] : acc[1][b];
      u0 += __shfl_xor_sync(0xffffffffu, hi ? acc[0][b] : acc[2][b], 16);
      u1 += __shfl_xor_sync(0xffffffffu, hi ? acc[1][b] : acc[3][b], 16);
      float sum = hi2 ? u1 : u0;
      sum += __shfl_xor_sync(0xffffffffu, hi2 ? u0 : u1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if ((lane & 7) == 0 && j_own < a.j_end) a.mod[(size_t)(b0 + b) * a.n_out + j_own] = sum + __uint_as_float((uint32_t)bias << 16);
    }
  }
}

template <int BATCH>
__global__ void __launch_bounds__(kModWarps * 32, 2) mod_gemv_kernel(const ModArgs a) {
  mod_features<kModWarps, BATCH, BATCH == 1>(a, blockIdx.x);
}

constexpr size_t kModSmemLimit = 48 * 1024;
static int check_mod(const ModArgs& a) {
  if (a.batch < 1 || a.Dt < 8 || (a.Dt & 7) || a.n_out < 1 || a.j_first < 0 || a.j_first >= a.j_end || a.j_end > a.n_out)
    return XEMA_EINVAL;
  return (size_t)a.batch * a.Dt * sizeof(float) > kModSmemLimit ? XEMA_EINVAL : XEMA_OK;
}

int launch_mod(const ModArgs& a, cudaStream_t stream, bool chained) {
  if (int rc = check_mod(a)) return rc;
  const int blocks = (a.j_end - a.j_first + kModWarps * kModRows - 1) / (kModWarps * kModRows);
  return launch_kernel(a.batch == 1 ? mod_gemv_kernel<1> : mod_gemv_kernel<4>, dim3(blocks), kModWarps * 32, (size_t)a.batch * a.Dt * sizeof(float), stream, chained, a);
}

// ---------------------------------------------------------------------------------------
// out = LN(in) * (1 + scale) + shift, one warp per row: no block-wide barrier, the whole row is in
// flight at once (NV 16-byte loads per lane) and stays in registers for the mean, the centred sum of
// squares and the result.  Bound by HBM for many rows, by the latency of load, two reductions and
// store for few.
// bf16 input: lane reads 8 elements (16 B) per step; fp32 input: 4 elements (16 B) per step.
// NV = steps per row (compile-time so the row stays in registers); NV == 0 selects the
// generic variant for rows wider than 4096, which re-reads the row instead.
// ---------------------------------------------------------------------------------------
constexpr int kLnWarps = 4;

template <bool IN_F32>
struct LnIo {
  static constexpr int EPV = IN_F32 ? 4 : 8;  // elements per lane per step
  using Raw = typename std::conditional<IN_F32, float4, uint4>::type;
  __device__ static __forceinline__ Raw load(const void* row, int idx) {
    if constexpr (IN_F32) return ld_f4(reinterpret_cast<const float4*>(row) + idx);
    else return ld_u4(reinterpret_cast<const uint4*>(row) + idx);
  }
  __device__ static __forceinline__ void unpack(const Raw& v, float (&f)[EPV]) {
    if constexpr (IN_F32) {
      f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
    } else {
      f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
      f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
    }
  }
  __device__ static __forceinline__ void store(__nv_bfloat16* row, int idx, const float (&f)[EPV]) {
    if constexpr (IN_F32)
      reinterpret_cast<uint2*>(row)[idx] = make_uint2(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]));
    else
      reinterpret_cast<uint4*>(row)[idx] = make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]),
                                                      pack_bf16x2(f[4], f[5]), pack_bf16x2(f[6], f[7]));
  }
  // sum of a lane's elements of one step; the same of their squares once the mean is off
  __device__ static __forceinline__ float sum(const float (&f)[EPV]) {
    float s = (f[0] + f[1]) + (f[2] + f[3]);
    if constexpr (!IN_F32) s += (f[4] + f[5]) + (f[6] + f[7]);
    return s;
  }
  __device__ static __forceinline__ float centre(float (&f)[EPV], float mean) {
#pragma unroll
    for (int t = 0; t < EPV; ++t) f[t] -= mean;
    float s = fmaf(f[0], f[0], f[1] * f[1]) + fmaf(f[2], f[2], f[3] * f[3]);
    if constexpr (!IN_F32) s += fmaf(f[4], f[4], f[5] * f[5]) + fmaf(f[6], f[6], f[7] * f[7]);
    return s;
  }
  // Scale and shift of one step.  A lane of the bf16 form needs 32 bytes of each: by two 16-byte loads a warp met every line twice,
  // and the L1 was busy with scale and shift for four fifths of a row's time.  `wide`: both rows start on a 32-byte boundary, and
  // one load takes all of it.  us, launches chained: 1101 x 1536 5.1 -> 4.2, 2040 x 2048 6.2 -> 4.8, 4608 x 3072 14.9 -> 12.9, 8888 x 1024
  // 8.5 -> 7.5, 17776 x 2048 31.1 -> 28.5, x 3072 44.3 -> 41.2, x 3328 51.3 -> 46.7, x 3840 57.7 -> 52.5.  It is slower where its registers
  // cost a wave (2961 to 3552 rows of 1536 columns 5.6 -> 6.0, 2000 of 3840 10.4 -> 11.0) and, in LN launches that follow one another
  // with a block an SM or less, by 0.1 (1792 columns) to 1 us (4096) -- not in plans: with narrow loads up to 592 rows, stacks of 1792 to
  // 3072 columns and 68 to 500 rows a launch took 0.99 to 1.01 of the time that they take with wide ones.
  struct Mod {
    float4 a[EPV / 4], c[EPV / 4];
  };
  __device__ static __forceinline__ void load_mod(const float* sc, const float* sh, int idx, bool wide, Mod& m) {
    if constexpr (!IN_F32) {
      if (wide) {
        ld_f8(sc + idx * EPV, m.a[0], m.a[1]);
        ld_f8(sh + idx * EPV, m.c[0], m.c[1]);
        return;
      }
    }
#pragma unroll
    for (int q = 0; q < EPV / 4; ++q) {
      m.a[q] = ld_f4(sc + idx * EPV + 4 * q);
      m.c[q] = ld_f4(sh + idx * EPV + 4 * q);
    }
  }
  __device__ static __forceinline__ void modulate(float (&f)[EPV], float mean, float rstd, const Mod& m) {
#pragma unroll
    for (int q = 0; q < EPV / 4; ++q) {
      f[4 * q + 0] = fmaf((f[4 * q + 0] - mean) * rstd, 1.f + m.a[q].x, m.c[q].x);
      f[4 * q + 1] = fmaf((f[4 * q + 1] - mean) * rstd, 1.f + m.a[q].y, m.c[q].y);
      f[4 * q + 2] = fmaf((f[4 * q + 2] - mean) * rstd, 1.f + m.a[q].z, m.c[q].z);
      f[4 * q + 3] = fmaf((f[4 * q + 3] - mean) * rstd, 1.f + m.a[q].w, m.c[q].w);
    }
  }
};

// CARRY > 0: the first mod_blocks blocks work out features of a modulation (that many batch elements a pass) beside the rows.  For 1 and
// 2 elements one pass is all there is, and the instance needs no more registers than the rows alone or 80.  The instance for 4 loops
// over passes and takes 156: in one pass it needs 80 too, but then its four sums follow one another and few rows wait for it (8
// blocks of 4 x 250 x 1024 462 us with 156 registers, 483 with 80).
// Four blocks an SM for 2816 and 3072 bf16 columns (128 registers, of which 16 and 52 bytes a thread go to local memory), where the
// compiler would take 167, three blocks, and be 15 % slower; three for 4096 (168 registers and 16 bytes), where it would take 247,
// two blocks: us 1200 x 4096 10.3 -> 6.8, 3500 16.6 -> 14.2, 8888 36.5 -> 31.4, 17776 64.6 -> 55.8 (by narrow loads, 166 registers:
// 7.2, 15.3, 34.5, 60.5).  3328 to 3840 columns take 153 to 166 by themselves and are 5 to 22 % slower when told so, fewer than 2816
// stay within 128; told to be six blocks (80 registers) 1536 columns gain 15 % at 3500 rows, which then are one wave, and lose 8 % at
// 1200.
template <bool IN_F32, int NV, int CARRY>
__global__ void __launch_bounds__(kLnWarps * 32, IN_F32 ? 0 : NV == 11 || NV == 12 ? 4 : NV == 16 ? 3 : 0)
ln_modulate_kernel(const void* in, long long in_batch_rows, __nv_bfloat16* out, const float* shift, const float* scale,
                   long long mod_stride, int batch, int rows, int D, float eps, bool wide, const ModArgs mod, int mod_blocks) {
  using Io = LnIo<IN_F32>;
  constexpr int EPV = Io::EPV;
  if constexpr (CARRY > 0) {
    if ((int)blockIdx.x < mod_blocks) {
      mod_features<kLnWarps, CARRY, CARRY <= 2>(mod, blockIdx.x);
      return;
    }
  }
  grid_dep_launch();
  grid_dep_wait();
  const int lane = threadIdx.x & 31;
  const long long total = (long long)batch * rows;
  const float inv_d = 1.f / (float)D;
  const long long r = (long long)(blockIdx.x - (CARRY > 0 ? mod_blocks : 0)) * kLnWarps + (threadIdx.x >> 5);
  if (r >= total) return;
  const int b = (int)(r / rows);
  const int i = (int)(r - (long long)b * rows);
  const size_t in_elem = ((size_t)b * in_batch_rows + i) * D;
  const void* src = IN_F32 ? (const void*)((const float*)in + in_elem) : (const void*)((const __nv_bfloat16*)in + in_elem);
  __nv_bfloat16* dst = out + (size_t)r * D;
  const float* sh = shift + (size_t)b * mod_stride;
  const float* sc = scale + (size_t)b * mod_stride;

  if constexpr (NV > 0) {
    typename Io::Raw raw[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) raw[v] = Io::load(src, v * 32 + lane);
    typename Io::Mod m[2];
    Io::load_mod(sc, sh, lane, wide, m[0]);
    float f[EPV];
    float s = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Io::unpack(raw[v], f);
      s += Io::sum(f);
    }
    const float mean = warp_sum(s) * inv_d;
    float q = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Io::unpack(raw[v], f);
      q += Io::centre(f, mean);
    }
    const float rstd = rsqrtf(warp_sum(q) * inv_d + eps);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (v + 1 < NV) Io::load_mod(sc, sh, (v + 1) * 32 + lane, wide, m[(v + 1) & 1]);
      Io::unpack(raw[v], f);
      Io::modulate(f, mean, rstd, m[v & 1]);
      Io::store(dst, v * 32 + lane, f);
    }
  } else {
    const int nv = D / (32 * EPV);
    float f[EPV];
    float s = 0.f;
    for (int v = 0; v < nv; ++v) {
      Io::unpack(Io::load(src, v * 32 + lane), f);
      s += Io::sum(f);
    }
    const float mean = warp_sum(s) * inv_d;
    float q = 0.f;
    for (int v = 0; v < nv; ++v) {
      Io::unpack(Io::load(src, v * 32 + lane), f);
      q += Io::centre(f, mean);
    }
    const float rstd = rsqrtf(warp_sum(q) * inv_d + eps);
    for (int v = 0; v < nv; ++v) {
      typename Io::Mod m;
      Io::unpack(Io::load(src, v * 32 + lane), f);
      Io::load_mod(sc, sh, v * 32 + lane, wide, m);
      Io::modulate(f, mean, rstd, m);
      Io::store(dst, v * 32 + lane, f);
    }
  }
}

template <bool IN_F32>
static int launch_ln_t(const void* in, long long in_batch_rows, void* out, const float* shift, const float* scale,
                       long long mod_stride, int batch, int rows, int D, float eps, cudaStream_t stream, bool chained,
                       const ModArgs* mod) {
  constexpr int PER = IN_F32 ? 2 : 1;                  // steps per 256 columns
  const long long total = (long long)batch * rows;
  const unsigned blocks = (unsigned)((total + kLnWarps - 1) / kLnWarps);
  const bool wide = ((reinterpret_cast<uintptr_t>(shift) | reinterpret_cast<uintptr_t>(scale)) & 31) == 0 && (batch == 1 || mod_stride % 8 == 0);
  const int per_block = kLnWarps * kModRows;
  const int mod_blocks = mod ? (mod->j_end - mod->j_first + per_block - 1) / per_block : 0;
  const size_t smem = mod ? (size_t)mod->batch * mod->Dt * sizeof(float) : 0;
  auto run = [&](auto kern) {
    return launch_kernel(kern, dim3(blocks + mod_blocks), kLnWarps * 32, smem, stream, chained, in, in_batch_rows,
                         (__nv_bfloat16*)out, shift, scale, mod_stride, batch, rows, D, eps, wide, mod ? *mod : ModArgs{}, mod_blocks);
  };
  if (mod) {
    if (int rc = check_mod(*mod)) return rc;
    switch (D / 256) {
#define XEMA_LN_CASE(N, MOST) \
  case N: return mod->batch == 1   ? run(ln_modulate_kernel<IN_F32, N * PER, 1>) \
                 : mod->batch == 2 ? run(ln_modulate_kernel<IN_F32, N * PER, 2>) \
                 : MOST > 2        ? run(ln_modulate_kernel<IN_F32, N * PER, MOST>) : XEMA_EINVAL;
      XEMA_LN_CASE(1, 4) XEMA_LN_CASE(2, 4) XEMA_LN_CASE(3, 4) XEMA_LN_CASE(4, 4) XEMA_LN_CASE(5, 4) XEMA_LN_CASE(6, 4)
      XEMA_LN_CASE(7, 4) XEMA_LN_CASE(8, 4) XEMA_LN_CASE(9, 2) XEMA_LN_CASE(10, 2) XEMA_LN_CASE(11, 2) XEMA_LN_CASE(12, 2)
#undef XEMA_LN_CASE
      default: return XEMA_EINVAL;
    }
  }
  switch (D / 256) {
#define XEMA_LN_CASE(N) case N: return run(ln_modulate_kernel<IN_F32, N * PER, 0>);
    XEMA_LN_CASE(1) XEMA_LN_CASE(2) XEMA_LN_CASE(3) XEMA_LN_CASE(4) XEMA_LN_CASE(5) XEMA_LN_CASE(6)
    XEMA_LN_CASE(7) XEMA_LN_CASE(8) XEMA_LN_CASE(9) XEMA_LN_CASE(10) XEMA_LN_CASE(11) XEMA_LN_CASE(12)
    XEMA_LN_CASE(13) XEMA_LN_CASE(14) XEMA_LN_CASE(15) XEMA_LN_CASE(16)
#undef XEMA_LN_CASE
    default: return run(ln_modulate_kernel<IN_F32, 0, 0>);
  }
}

int launch_ln_modulate(const void* in, int in_is_f32, long long in_batch_rows, void* out, const float* shift,
                       const float* scale, long long mod_stride, int batch, int rows, int D, float eps,
                       cudaStream_t stream, bool chained, const ModArgs* mod) {
  if (batch < 1 || rows < 0 || D < 256 || (D % 256)) return XEMA_EINVAL;
  if (rows == 0) return mod ? launch_mod(*mod, stream, chained) : XEMA_OK;
  return in_is_f32 ? launch_ln_t<true>(in, in_batch_rows, out, shift, scale, mod_stride, batch, rows, D, eps, stream, chained, mod)
                   : launch_ln_t<false>(in, in_batch_rows, out, shift, scale, mod_stride, batch, rows, D, eps, stream, chained, mod);
}

// ---------------------------------------------------------------------------------------
// In place, per head: x <- RoPE(RMSNorm(x) * g).  One warp per token row; a lane owns 8
// consecutive features (four rotation pairs) of one head; DH/8 lanes share a head.
// ---------------------------------------------------------------------------------------
constexpr int kRopeWarps = 4;

template <int DH>
__global__ void __launch_bounds__(kRopeWarps * 32)
rmsnorm_rope_kernel(__nv_bfloat16* __restrict__ x, long long ld, long long batch_rows,
                    const __nv_bfloat16* __restrict__ g, const float* __restrict__ rope, int pos0, int batch,
                    int rows, int heads, float eps) {
  constexpr int LPH = DH / 8;        // lanes per head
  constexpr int HPW = 32 / LPH;      // heads per warp step
  const int lane = threadIdx.x & 31;
  const long long total = (long long)batch * rows;
  const long long r = (long long)blockIdx.x * kRopeWarps + (threadIdx.x >> 5);
  if (r >= total) return;
  const int b = (int)(r / rows);
  const int i = (int)(r - (long long)b * rows);
  __nv_bfloat16* row = x + ((size_t)b * batch_rows + i) * ld;
  const int e0 = (lane % LPH) * 8;   // first feature of this lane inside its head
  // cos/sin of this lane's four pairs and its eight gains: the same for every head
  const float4* rp = reinterpret_cast<const float4*>(rope + (size_t)(pos0 + i) * DH + e0);
  const float4 cs0 = __ldg(rp), cs1 = __ldg(rp + 1);
  const uint4 gv = __ldg(reinterpret_cast<const uint4*>(g + e0));
  const float gain[8] = {bf16_lo(gv.x), bf16_hi(gv.x), bf16_lo(gv.y), bf16_hi(gv.y),
                         bf16_lo(gv.z), bf16_hi(gv.z), bf16_lo(gv.w), bf16_hi(gv.w)};
  const float cosv[4] = {cs0.x, cs0.z, cs1.x, cs1.z};
  const float sinv[4] = {cs0.y, cs0.w, cs1.y, cs1.w};
  for (int h0 = 0; h0 < heads; h0 += HPW) {
    const int h = h0 + lane / LPH;
    const bool live = h < heads;
    uint4 v = make_uint4(0, 0, 0, 0);
    uint4* p = reinterpret_cast<uint4*>(row + (size_t)h * DH + e0);
    if (live) v = *p;
    float f[8] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y),
                  bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w)};
    float ss = 0.f;
#pragma unroll
    for (int t = 0; t < 8; ++t) ss = fmaf(f[t], f[t], ss);
#pragma unroll
    for (int o = LPH / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float rstd = rsqrtf(ss * (1.f / DH) + eps);
    float y[8];
#pragma unroll
    for (int pr = 0; pr < 4; ++pr) {
      const float a = f[2 * pr] * rstd * gain[2 * pr];
      const float c = f[2 * pr + 1] * rstd * gain[2 * pr + 1];
      y[2 * pr] = a * cosv[pr] - c * sinv[pr];
      y[2 * pr + 1] = a * sinv[pr] + c * cosv[pr];
    }
    if (live)
      *p = make_uint4(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]),
                      pack_bf16x2(y[6], y[7]));
  }
}

int launch_rmsnorm_rope(void* x, long long ld, long long batch_rows, const void* g, const float* rope, int pos0,
                        int batch, int rows, int heads, int head_dim, float eps, cudaStream_t stream) {
  if (batch < 1 || rows < 0 || heads < 1 || (ld & 7)) return XEMA_EINVAL;
  if (rows == 0) return XEMA_OK;
  const long long total = (long long)batch * rows;
  const unsigned blocks = (unsigned)((total + kRopeWarps - 1) / kRopeWarps);
  if (head_dim == 64)
    rmsnorm_rope_kernel<64><<<blocks, kRopeWarps * 32, 0, stream>>>((__nv_bfloat16*)x, ld, batch_rows,
                                                                     (const __nv_bfloat16*)g, rope, pos0, batch, rows,
                                                                     heads, eps);
  else if (head_dim == 128)
    rmsnorm_rope_kernel<128><<<blocks, kRopeWarps * 32, 0, stream>>>((__nv_bfloat16*)x, ld, batch_rows,
                                                                      (const __nv_bfloat16*)g, rope, pos0, batch, rows,
                                                                      heads, eps);
  else
    return XEMA_EINVAL;
  return check_launch();
}

// ---------------------------------------------------------------------------------------
// Two contiguous copies in one launch (a forward call's inputs): 16 bytes per thread and step, four
// loads in flight.  One launch instead of two memory copies takes 2-4 us off a call with small inputs;
// bound by HBM for large ones.  It may be launched before the work ahead of it in the stream has finished, and waits for
// that (calls back to back, a block of 288 x 512 47.1 -> 45.1 us, of 1101 x 1536 123.7 -> 122.2).
// ---------------------------------------------------------------------------------------
constexpr int kCopyThreads = 256;

__device__ __forceinline__ void copy_part(uint8_t* dst, const uint8_t* src, size_t bytes) {
  const size_t n = bytes / 16, stride = (size_t)gridDim.x * kCopyThreads;
  uint4* d = reinterpret_cast<uint4*>(dst);
  const uint4* s = reinterpret_cast<const uint4*>(src);
  for (size_t i = (size_t)blockIdx.x * kCopyThreads + threadIdx.x; i < n; i += 4 * stride) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < n) v[u] = __ldcs(s + i + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < n) d[i + u * stride] = v[u];
  }
}
__global__ void __launch_bounds__(kCopyThreads)
copy2_kernel(uint8_t* dst0, const uint8_t* src0, size_t n0, uint8_t* dst1, const uint8_t* src1, size_t n1) {
  grid_dep_wait();
  copy_part(dst0, src0, n0);
  copy_part(dst1, src1, n1);
}

int launch_copy2(void* dst0, const void* src0, size_t n0, void* dst1, const void* src1, size_t n1, cudaStream_t stream,
                 bool early) {
  const size_t steps = (std::max(n0, n1) / 16 + 4 * kCopyThreads) / (4 * kCopyThreads);
  const unsigned blocks = (unsigned)std::min<size_t>(std::max<size_t>(steps, 1), (size_t)sm_count() * 8);
  return launch_kernel(copy2_kernel, dim3(blocks), kCopyThreads, 0, stream, early, (uint8_t*)dst0, (const uint8_t*)src0, n0,
                       (uint8_t*)dst1, (const uint8_t*)src1, n1);
}

}  // namespace xema
