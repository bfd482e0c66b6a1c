// Non-causal flash-style attention on tcgen05: o = softmax(q k^T / sqrt(dh)) v over all keys.
//
// One persistent CTA per SM walks over work items of up to 256 query rows (two 128-row tiles) of one
// (batch, head) and streams the keys in blocks of 128 from key 0.  Its workspace (shared memory and
// TMEM) depends on the tile only, never on the number of keys.
//
//   warp 0       TMA producer: both Q tiles of an item, then K and V blocks through two rings
//   warps 1, 2   MMA issuers (converged warp, one elected lane issues): dh 64 warp 1 the scores and
//                warp 2 the products, dh 128 warp 1 both.  Warp 1 also owns TMEM
//   warp 3       idle (fills the warpgroup, so that softmax warp w reads TMEM lanes 32 * (w % 4))
//   warps 4-19   softmax: two threads per score row, 64 scores each per block
//
// The softmax threads set the pace (an SM retires 16 exponentials per clock against 4 * dh flop each),
// so their instruction stream is kept short:
//
//   * no running maximum: q arrives multiplied by log2(e) / sqrt(dh) (the Q projection's epilogue does
//     that before its one rounding to bf16), so a score leaves the tensor core as the exponent to base 2
//     of its unnormalised probability and p = 2^(s - reference) is formed whatever its size -- fp32 sums
//     and bf16 probabilities keep their relative precision from 2^-90 to 2^90 -- so O is never rescaled
//     and the two threads of a row need not talk to each other inside the loop.  The reference of a row
//     is 0 for dh 64 and the largest of its first 128 scores for dh 128.  A row that leaves the
//     range (a sum of 2^90 or more, or of 2^-90 or less), or that hands the exponential polynomial an
//     argument outside its range, is flagged, and its item is done again after the CTA's last item, in
//     two more sweeps: one over the scores only, which decides again which rows were at fault and takes
//     their true maximum, and one that repeats the pass with that maximum as the reference of those
//     rows.  Rows that were not at fault repeat exactly what they did before, bit for bit.  A score
//     that is not a number makes its row's maximum one too, and with it the whole row;
//   * dh 64, where the exponentials set the pace: a share of them is evaluated as a polynomial on the
//     FMA pipe (see kPolyPairs);
//   * dh 128, where the threads have issue slots to spare (34 % used without the next two, 45 % with): every
//     exponential on the MUFU, and O is divided by the sum of the probabilities as they were rounded to
//     bf16 (lse takes the unrounded sum), so that the rounding of a dominant key cancels.  Relative error
//     of o against 64 bits, standard normal q and k: 2.24e-3 for 288 keys, 2.32e-3 for 1101, and 1.92e-3 for
//     600 keys with three times the scores; without reference and rounded sum 2.34e-3, 2.35e-3, 2.35e-3; with a
//     running maximum instead 2.29e-3, 2.33e-3, 2.23e-3.  Both together cost 2 % (4608 x 4608 x 24 heads
//     229 -> 233 us, launches in turn on a warm board);
//   * per block a softmax warp runs 212 instructions of arithmetic and, at first, 100 around them.  Warp index and TMEM base are
//     made uniform (barrier and TMEM addresses then stay in uniform registers: no moves there, fewer spills), a wait
//     that gives up does not leave the block (mbar_wait_sticky), three score loads share one wait, P leaves in one store.
//     In turn, cool board / under the power cap: dh 64, 4444 x 17776 x 48 heads 887 -> 861 / 1017 -> 986 us; dh 128, 4608 x
//     4608 x 24 heads 205 -> 190 / 237 -> 221 us.  One arrival per warp instead of one per thread: 1 % slower; 32 / 112
//     registers for helpers / softmax: spills, 4 % slower;
//   * one body for all blocks where there are few: the first time an SM runs a piece of code costs
//     microseconds of instruction fetch, which a call with few keys pays in full.  Keys past the end get
//     the exponent -119 (they add 2^-119 each to a row sum of at least 2^-90; their V rows are zero).
//
// TMEM, per tile 256 columns:
//   dh  64: S [0,128), P [128,192) (bf16 pairs), O [192,256).  S(j+1) is issued as soon as the tile's
//           threads hold S(j) in registers and runs while they work; P(j) is stored once
//           O += P(j-1) V(j-1), which reads the same columns, has finished.
//   dh 128: S [0,128), O [128,256); P(j) lies over S(j), each thread's over its own scores.  S(j+1) is
//           queued behind O += P(j) V(j) in the tensor pipe; the two tiles run half a block apart, so
//           one tile's burst of MMAs runs under the other's softmax.  One warp issues both: with a warp
//           per tile the two bursts shared the pipe and both ended late (a block 3090 cycles against
//           2690).  P goes over in two halves, so half of the product runs under the rest of the softmax.
//
// Measured (B200): dh 64, 4444 x 17776 x 48 heads 845 us; before the overhead instructions went, inside the block, 933 (with one
// CTA per 256 rows and code copies for first and last blocks 970); power-capped 17776-token block 7.28 ms against 7.52.  dh 128, 17776 x
// 17776 x 24 heads 3.38 ms on a warm board (one tile per CTA, two CTAs per SM, 64-key blocks, running maximum:
// 3.79 in turn with it), 4608 x 4608 x 24 heads 235 us (275).  288 x 288 x 8 heads of 64 10.4 us (14.4).
//
// Every decision is per row and keys are always visited in the same order, so a row's bits do not
// depend on how rows are tiled or chunked.
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "sm100.cuh"

namespace xema {
using namespace sm100;

namespace {
constexpr int BM = 128;          // rows per tile
constexpr int TILES = 2;
constexpr int BN = kAttnKeysPerBlock;   // keys per block (128)
constexpr int ATOM_BYTES = 128 * 128;   // 128 rows x 64 bf16, one swizzled column block
constexpr float DANGER = 1.2379400392853803e27f;   // 2^90
constexpr float TINY = 8.077935669463161e-28f;     // 2^-90
constexpr float PAST_END = -119.f;      // score of a key past the end of the sequence
constexpr int MAX_ITEMS = 1024;         // items one CTA can keep a flag for
constexpr int TPR = 2;           // softmax threads per score row
constexpr int COLS = BN / TPR;   // scores per softmax thread and block ...
constexpr int CH = COLS / 4;     // ... worked on in four chunks
constexpr int SOFTMAX_THREADS = TILES * BM * TPR;
constexpr int THREADS = 128 + SOFTMAX_THREADS;
// Registers a thread: the compiler allots 96 to 640 threads; the helper warps give some back to the
// softmax warps.  128 * HELPER + SOFTMAX_THREADS * SOFTMAX must stay within THREADS * 96, or the
// request would wait for ever.
constexpr int REG_HELPER = 64, REG_SOFTMAX = 104;
static_assert(128 * REG_HELPER + SOFTMAX_THREADS * REG_SOFTMAX <= THREADS * 96, "register pool");
// Which of a thread's 32 column pairs evaluate 2^x as a polynomial on the FMA pipe, one bit per pair; the
// others use the MUFU.  dh 64: without any the MUFU sets the pace, with too many the issue slots do, and
// where they stand decides how well the compiler interleaves the two pipes -- the placement is the result of
// a search with this compiler and nothing else.  4444 x 17776 x 48 heads, with the overhead instructions that are gone by
// now: 933 to 1177 us over 125 placements of 6 to 17 bits (this one 933, the next best 945; 9 bits 1000 and more).
// Without them 845; 44 other placements 5.8 % slower to 0.6 % faster.  Accuracy: see exp2_poly; a polynomial of
// degree 4 costs 10 % of the launch.
// dh 128: none.  The MUFU needs no longer for a block than the tensor pipe (2048 cycles each), and 8 pairs on the
// FMA pipe were 2 % slower in turn with none (4608 x 4608 x 24 heads 231 against 226 us).
template <int DH>
constexpr uint32_t kPolyPairs = DH == 64 ? 0xc358a94au : 0u;
static_assert(!(kPolyPairs<64> & 1u), "a row's first key goes through the MUFU, which keeps a NaN");
static_assert(BN == 128 && BM == 128, "the kernel is written for 128-key blocks of 128-row tiles");

// Barriers between softmax threads and issuers per set (s_full to pv_done); the rehearsal uses a second set, none of whose
// phases completes: a wait for the phase before the first returns at once, an arrival has no effect.
constexpr int kDry = 5 * TILES;
constexpr uint32_t kNever = 1u << 19;
constexpr int kRehearseBlocks = 8;       // key blocks a CTA works on, up to which a launch rehearses (see attention_kernel)

template <int DH>
struct Cfg {
  static constexpr bool ALIAS = DH == 128;                 // P over S; otherwise P has its own columns
  static constexpr int ISSUERS = ALIAS ? 1 : 2;            // MMA-issuing warps (from warp 1)
  static constexpr bool FIRST_MAX = DH == 128;             // reference: the largest score of the first block
  static constexpr bool ROUNDED_SUM = DH == 128;           // O over the sum of the rounded probabilities
  static constexpr int ATOMS = DH / 64;
  static constexpr int TILE_BYTES = ATOMS * ATOM_BYTES;    // a Q tile, or a K or V block
  static constexpr int QBUF = DH == 64 ? 2 : 1;
  static constexpr int KS = DH == 64 ? 5 : 2;              // K and V stages
  static constexpr int VS = DH == 64 ? 5 : 3;
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_K = OFF_Q + QBUF * TILES * TILE_BYTES;
  static constexpr int OFF_V = OFF_K + KS * TILE_BYTES;
  static constexpr int OFF_BAR = OFF_V + VS * TILE_BYTES;
  static constexpr int OFF_XCH = OFF_BAR + 512;            // float [TILES][2][BM]
  static constexpr int SMEM_BYTES = OFF_XCH + TILES * 2 * BM * 4;
  static_assert(SMEM_BYTES <= 232448, "shared memory of one SM");
  static constexpr int TM_TILE = 256;
  static constexpr int TM_P = ALIAS ? 0 : 128;
  static constexpr int TM_O = ALIAS ? 128 : 192;
};

struct AttnParams {
  __nv_bfloat16* o;
  float* lse;
  int batch, rows, keys, heads;
  int tiles;          // query tiles per work item (1 or 2)
  int q_items;        // work items per (batch, head)
  int items;
  float q_scale;      // q k^T times this = exponents to base 2 (SCALED kernels only)
  unsigned int* status;
  const __nv_bfloat16 *gain_q, *gain_k;   // RMSNorm gains behind q and k, or null (see AttnLaunch)
};

// 2^x for two values on the FMA pipe instead of the MUFU: round-to-nearest split x = n + r with
// |r| <= 1/2 through the 1.5 * 2^23 trick, a cubic for 2^r, then n added into the exponent field.
// The cubic has the least mean square relative error (4.84e-5) among those of mean 0 that stay within
// 1e-4 of 2^r, a twentieth of the bf16 rounding of the probability it feeds: the errors of a row's keys
// do not add up in its sum.  (The cubic of least largest error, 7.5e-5, has a mean of 5e-6 and a mean square of
// 5.2e-5; lse of 1101 keys 2.8e-6 off with it, 1.7e-6 with this one.)
// Valid for -125 <= x <= 126; CLAMP raises smaller arguments to -125 (2^-125 stands in for zero) and leaves
// the bits of valid ones as they are.
template <bool CLAMP>
__device__ __forceinline__ f32x2 exp2_poly(f32x2 x2) {
  if (CLAMP) x2 = make_float2(fmaxf(x2.x, -125.f), fmaxf(x2.y, -125.f));
  const f32x2 magic = make_float2(12582912.f, 12582912.f);
  const f32x2 neg_magic = make_float2(-12582912.f, -12582912.f);
  const f32x2 neg_one = make_float2(-1.f, -1.f);
  const f32x2 t2 = add_f32x2(x2, magic);                 // integer part lands in the low mantissa bits
  const f32x2 n2 = add_f32x2(t2, neg_magic);             // nearest integer as a float
  const f32x2 r2 = fma_f32x2(n2, neg_one, x2);           // r = x - n
  f32x2 p2 = fma_f32x2(make_float2(0.0551208667f, 0.0551208667f), r2, make_float2(0.242484242f, 0.242484242f));
  p2 = fma_f32x2(p2, r2, make_float2(0.693255842f, 0.693255842f));
  p2 = fma_f32x2(p2, r2, make_float2(0.999933064f, 0.999933064f));
  // (t << 23) + p: written as a plain shift and sum it becomes an IMAD on the pipe of the packed FMAs, which was busy
  // 63 % of the time beside 30 % of the ALU's, where a funnel shift and an add run.  4444 x 17776 x 48 heads 878 -> 846 us,
  // under the power cap 999 -> 971.
  uint32_t nx, ny;
  asm("shf.l.wrap.b32 %0, %1, %2, 23;" : "=r"(nx) : "r"(0u), "r"(__float_as_uint(t2.x)));
  asm("shf.l.wrap.b32 %0, %1, %2, 23;" : "=r"(ny) : "r"(0u), "r"(__float_as_uint(t2.y)));
  return make_float2(__uint_as_float(__float_as_uint(p2.x) + nx), __uint_as_float(__float_as_uint(p2.y) + ny));
}

// Partial sums of one thread's part of a row: of the probabilities, and (ROUNDED_SUM) of what bf16 makes
// of them.
struct RowSums {
  f32x2 plain[4], rounded[2];
};

// p = 2^s for chunk CHUNK of a thread's score columns: packed bf16x2 words, the values added into
// packed partial sums.  CLAMP = false: the polynomial is used as it is and, with TRACK, `poly_abs` collects the
// largest magnitude handed to it, for the caller to check afterwards (without TRACK the caller knows a
// bound on every score beforehand).  CLAMP = true: its arguments are clamped from below first.
template <int DH, int CHUNK, bool CLAMP, bool TRACK>
__device__ __forceinline__ void exp_cols(const float (&s)[CH], uint32_t* pk, RowSums& sums, float& poly_abs) {
#pragma unroll
  for (int t = 0; t < CH; t += 2) {
    const int pair = t >> 1;
    f32x2 e2 = pack_f32x2(s[t], s[t + 1]);
    float e0, e1;
    if (kPolyPairs<DH> >> (CHUNK * (CH / 2) + pair) & 1u) {
      if (TRACK && !CLAMP) poly_abs = max3(poly_abs, fabsf(e2.x), fabsf(e2.y));
      e2 = exp2_poly<CLAMP>(e2);
      unpack_f32x2(e2, e0, e1);
    } else {
      unpack_f32x2(e2, e0, e1);
      e0 = ex2_approx(e0);
      e1 = ex2_approx(e1);
      e2 = pack_f32x2(e0, e1);
    }
    sums.plain[pair & 3] = add_f32x2(sums.plain[pair & 3], e2);
    pk[pair] = pack_bf16x2(e0, e1);
  }
  // (behind the chunk's exponentials: among them the compiler places them 3 % slower)
  if (Cfg<DH>::ROUNDED_SUM) {
#pragma unroll
    for (int i = 0; i < CH / 2; ++i)
      sums.rounded[i & 1] = add_f32x2(sums.rounded[i & 1], make_float2(bf16_lo(pk[i]), bf16_hi(pk[i])));
  }
}
// columns at or beyond `valid` (keys past the end of the sequence) get `value`
__device__ __forceinline__ void mask_tail(float (&s)[CH], int valid, float value) {
#pragma unroll
  for (int t = 0; t < CH; ++t)
    if (t >= valid) s[t] = value;
}
// (a NaN among the values is the result)
__device__ __forceinline__ float row_max(const float (&s)[CH]) {
  float mx = max3_nan(s[0], s[1], s[2]);
#pragma unroll
  for (int t = 3; t + 1 < CH; t += 2) mx = max3_nan(mx, s[t], s[t + 1]);
  return max3_nan(mx, s[CH - 1], s[CH - 1]);
}
__device__ __forceinline__ float sum_partials(const f32x2 (&v)[4]) {
  const f32x2 a = add_f32x2(v[0], v[1]), b = add_f32x2(v[2], v[3]);
  const f32x2 c = add_f32x2(a, b);
  return c.x + c.y;
}
__device__ __forceinline__ float sum_partials(const f32x2 (&v)[2]) {
  const f32x2 c = add_f32x2(v[0], v[1]);
  return c.x + c.y;
}
__device__ __forceinline__ void ld_scores(uint32_t addr, float (&s)[CH]) { tmem_ld16(addr, *reinterpret_cast<uint32_t(*)[CH]>(&s[0])); }
__device__ __forceinline__ void wait_scores(float (&s)[CH]) { tmem_ld_wait_on(*reinterpret_cast<uint32_t(*)[CH]>(&s[0])); }

__device__ __forceinline__ uint4 shfl_xor_u4(uint4 v, int m) {
  return make_uint4(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m),
                    __shfl_xor_sync(0xffffffffu, v.z, m), __shfl_xor_sync(0xffffffffu, v.w, m));
}
// c[k] of lane i in every group of four lanes <- c[i] of the group's lane k
__device__ __forceinline__ void transpose_4x4(uint4 (&c)[4], int lane) {
  const bool odd = lane & 1, high = lane & 2;
  const uint4 ra = shfl_xor_u4(odd ? c[0] : c[1], 1), rb = shfl_xor_u4(odd ? c[2] : c[3], 1);
  const uint4 a0 = odd ? ra : c[0], a1 = odd ? c[1] : ra;     // column (lane & 1) of the pair's two rows
  const uint4 b0 = odd ? rb : c[2], b1 = odd ? c[3] : rb;     // column (lane & 1) + 2
  const uint4 r0 = shfl_xor_u4(high ? a0 : b0, 2), r1 = shfl_xor_u4(high ? a1 : b1, 2);
  c[0] = high ? r0 : a0;
  c[1] = high ? r1 : a1;
  c[2] = high ? b0 : r0;
  c[3] = high ? b1 : r1;
}

// Sweeps of one item: the pass itself; the scores only (flags and true maxima); the repeat.
enum Mode { PASS = 0, PROBE = 1, REPEAT = 2 };

// REHEARSE: a round of the softmax threads' loop before the wait for earlier launches, on whatever TMEM holds and
// without results, so that the first item does not meet every line of the code in an empty instruction cache.  A launch of
// few key blocks gains 0.5 to 3 us by it; the second set of barriers costs the loop 2 %.  us without / with it: block of 288 x 512
// 45.8 / 45.3, 464 x 1792 100.3 / 97.1 (dh 128 105.7 / 101.9), two blocks of 630 x 1536 184.2 / 179.6, eight of 304 x 2304 859.7 /
// 833.7, eight of 333 x 1024 470.9 / 468.7; with 9 key blocks a CTA (1101 x 1536)
// 121.8 / 122.5, with 16 (ragged batch of 3) 799 / 814, with 417 (17776 x 3072) 7129 / 7263.  A CTA that starts when the launch
// before it ends has no time to rehearse in: its scores came 1.8 us after the wait and found the softmax threads at it until 4.8.
// Where an item has one tile the idle warps of the second do it instead: eight of 333 x 1024 382.0 -> 367.4.
// (Registers are given out by the role: what the compiler sees as 96 is short by 4 to 20 bytes a thread in five of the six instances, 20 in
// the plain one of dh 64, which had 8 before the first loads stood behind the wait: 17776 x 3072 7026 / 7052, no difference.)
template <int DH, bool SCALED, bool REHEARSE>
__global__ void __launch_bounds__(THREADS, 1)
attention_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const AttnParams p) {
  using C = Cfg<DH>;
  constexpr int KS = C::KS, VS = C::VS, QBUF = C::QBUF;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint64_t* q_full = bars + 0;     // [QBUF]
  uint64_t* q_empty = bars + 2;    // [QBUF] both tiles' last scores of the item are done
  uint64_t* k_full = bars + 4;     // [KS <= 5]
  uint64_t* k_empty = bars + 9;
  uint64_t* v_full = bars + 14;    // [VS <= 5]
  uint64_t* v_empty = bars + 19;
  uint64_t* s_full = bars + 24;    // [TILES] S(j) of the tile is complete in TMEM
  uint64_t* s_free = bars + 26;    // [TILES] every softmax thread of the tile holds S(j) in registers
  uint64_t* p_half = bars + 28;    // [TILES] the first half of P(j) is complete in TMEM (ALIAS)
  uint64_t* p_full = bars + 30;    // [TILES] P(j) is complete in TMEM
  uint64_t* pv_done = bars + 32;   // [TILES] O += P(j) V(j) has finished (ALIAS: of an item's last block)
  // bars + 34: s_full to pv_done once more, for the rehearsal (kDry)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 44);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  uint32_t* gain_max = tmem_slot + 2;               // [2] bit patterns of max|gain_q|, max|gain_k|
  volatile uint32_t* any_flag = tmem_slot + 4;
  uint32_t* item_flag = tmem_slot + 5;              // [MAX_ITEMS / 32] one bit per item of this CTA
  static_assert((34 + kDry) * 8 + (5 + MAX_ITEMS / 32) * 4 <= 512 && kDry == 10, "barrier area");

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int n_kv = (p.keys + BN - 1) / BN;
  const int n_items = (p.items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // of this CTA

  // The swizzled tiles need a 1024-byte aligned base; refuse to run otherwise.
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0 && p.status) atomicExch(p.status, 0x54310002u);
    return;
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < QBUF; ++s) {
      mbar_init(&q_full[s], 1);
      mbar_init(&q_empty[s], 1);
    }
    for (int s = 0; s < KS; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < VS; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);
    }
    for (int t = 0; t < TILES; ++t) {
      mbar_init(&s_full[t], 1);
      mbar_init(&s_free[t], BM * TPR);   // every softmax thread of the tile arrives
      mbar_init(&p_half[t], BM * TPR);
      mbar_init(&p_full[t], BM * TPR);
      mbar_init(&pv_done[t], 1);
    }
    if (REHEARSE)
      for (int i = 0; i < kDry; ++i) mbar_init(&s_full[kDry + i], kNever);
    *abort_flag = 0;
    *any_flag = 0;
    gain_max[0] = gain_max[1] = 0;
    fence_mbar_init();
    prefetch_tmap(&map_q);
    prefetch_tmap(&map_k);
    prefetch_tmap(&map_v);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if (warp == 3 && lane < MAX_ITEMS / 32) item_flag[lane] = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);   // uniform, like the warp index
  if (threadIdx.x == 0) grid_dep_launch();
  // (the wait for earlier launches stands in the roles, behind the moves of registers)

  struct Item {
    int row0, h, b;
  };
  auto item_at = [&](int i) {
    const int w = (int)blockIdx.x + i * (int)gridDim.x;
    Item it;
    const int bh = w / p.q_items;
    it.row0 = (w - bh * p.q_items) * p.tiles * BM;
    it.b = bh / p.heads;
    it.h = bh - it.b * p.heads;
    return it;
  };
  auto tile_live = [&](const Item& it, int t) { return t < p.tiles && it.row0 + t * BM < p.rows; };

  // ---- per-role state that lives across items and sweeps -------------------------------------
  int k_st = 0, v_st = 0, q_st = 0;                 // ring positions (producer; each MMA warp)
  uint32_t k_ph = 0, v_ph = 0, q_ph = 0;
  int k_issued = 0, v_issued = 0, q_issued = 0;     // producer, for the drain after a give-up
  uint32_t s_ph = 0, pv_ph = 0;                     // softmax: s_full, pv_done
  bool ok = true;

  auto k_next = [&]() { if (++k_st == KS) { k_st = 0; k_ph ^= 1; } };
  auto v_next = [&]() { if (++v_st == VS) { v_st = 0; v_ph ^= 1; } };
  auto q_next = [&]() { if (++q_st == QBUF) { q_st = 0; q_ph ^= 1; } };

  // One item in one sweep, in the roles of the single-warp loops.
  auto load_q = [&](const Item& it) {
    for (int t = 0; t < p.tiles; ++t)
#pragma unroll
      for (int a = 0; a < C::ATOMS; ++a)
        tma_load_3d(smem + C::OFF_Q + (q_st * TILES + t) * C::TILE_BYTES + a * ATOM_BYTES, &map_q, &q_full[q_st],
                    it.h * DH + a * 64, it.row0 + t * BM, it.b);
    ++q_issued;
    q_next();
  };
  // `asked`: the item's queries and first keys are on their way
  auto produce = [&](const Item& it, bool with_v, bool asked) {   // warp 0, one lane
    auto load = [&](uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int row0) {
      mbar_expect_tx(bar, C::TILE_BYTES);
#pragma unroll
      for (int a = 0; a < C::ATOMS; ++a) tma_load_3d(dst + a * ATOM_BYTES, m, bar, it.h * DH + a * 64, row0, it.b);
    };
    auto load_k = [&](int j) {
      if (!(ok = mbar_wait(&k_empty[k_st], k_ph ^ 1, abort_flag))) return;
      load(smem + C::OFF_K + k_st * C::TILE_BYTES, &map_k, &k_full[k_st], j * BN);
      ++k_issued;
      k_next();
    };
    if (!asked) {
      load_k(0);
      if (!ok || !(ok = mbar_wait(&q_empty[q_st], q_ph ^ 1, abort_flag))) return;
      mbar_expect_tx(&q_full[q_st], p.tiles * C::TILE_BYTES);
      load_q(it);
    }
    for (int j = 0; ok && j < n_kv; ++j) {
      if (j + 1 < n_kv) load_k(j + 1);
      if (!ok) return;
      if (with_v) {
        if (!(ok = mbar_wait(&v_empty[v_st], v_ph ^ 1, abort_flag))) return;
        load(smem + C::OFF_V + v_st * C::TILE_BYTES, &map_v, &v_full[v_st], j * BN);
        ++v_issued;
        v_next();
      }
    }
  };

  constexpr uint32_t idesc_s = idesc_bf16_f32(BM, BN, false, false);   // S = Q K^T
  constexpr uint32_t idesc_o = idesc_bf16_f32(BM, DH, false, true);    // O = P V, V is N-major
  // (descriptors: the low words, which hold the address; the high word is the same constant for all)
  const uint32_t q_desc0 = smem_desc_lo(smem_u32(smem + C::OFF_Q), 16);
  const uint32_t k_desc0 = smem_desc_lo(smem_u32(smem + C::OFF_K), 16);
  // V block: rows = keys (the MMA's K), 64 dh per 128-byte row, 16 keys = 2048 bytes; the second
  // 64-wide dh block (dh = 128) starts one atom further (leading byte offset)
  const uint32_t v_desc0 = smem_desc_lo(smem_u32(smem + C::OFF_V), ATOM_BYTES);
  // Scores of one block, tile t.
  auto mma_scores = [&](int t) {   // elected lane
    const uint32_t qd = q_desc0 + (q_st * TILES + t) * (C::TILE_BYTES >> 4);
    const uint32_t kd = k_desc0 + k_st * (C::TILE_BYTES >> 4);
#pragma unroll
    for (int k = 0; k < DH / 16; ++k) {
      const uint32_t off = ((k / 4) * ATOM_BYTES + (k % 4) * 32) >> 4;
      mma_ss_lo(tmem_base + t * C::TM_TILE, qd + off, kd + off, idesc_s, k != 0);
    }
    mma_commit(&s_full[t]);
  };
  // Half of the product of one block: O += P V over 64 keys, 16 keys = 8 packed P columns per step.
  // ALIAS: P of each 64-key half lies over its own scores, and the first
  // (second) 32 keys of both halves are handed over together.
  auto mma_product = [&](int t, int hf, bool init) {   // elected lane
    const uint32_t d = tmem_base + t * C::TM_TILE;
    const uint32_t vd = v_desc0 + v_st * (C::TILE_BYTES >> 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int kk = C::ALIAS ? (i >> 1) * 4 + hf * 2 + (i & 1) : hf * 4 + i;
      const int col = C::ALIAS ? (kk >> 2) * 64 + (kk & 3) * 8 : kk * 8;
      mma_ts_lo(d + C::TM_O, d + C::TM_P + col, vd + kk * (2048 >> 4), idesc_o, !init || i != 0);
    }
  };
  auto wait_k = [&](bool first) {
    if (first && !(ok = mbar_wait_warp(&q_full[q_st], q_ph, abort_flag))) return;
    ok = mbar_wait_warp(&k_full[k_st], k_ph, abort_flag);
    tc_fence_after();
  };
  auto wait_v = [&]() {
    ok = mbar_wait_warp(&v_full[v_st], v_ph, abort_flag);
    tc_fence_after();
  };
  auto wait_phase = [&](uint64_t* bar, uint32_t& ph) {
    ok = mbar_wait_warp(bar, ph, abort_flag);
    ph ^= 1;
    tc_fence_after();
  };
  // whole warp: the block's (and the item's last) scores, or its products, are issued
  auto k_done = [&](bool last) {
    if (elect_one()) {
      mma_commit(&k_empty[k_st]);
      if (last) mma_commit(&q_empty[q_st]);
    }
    __syncwarp();
    k_next();
  };
  auto v_done = [&]() {
    if (elect_one()) mma_commit(&v_empty[v_st]);
    __syncwarp();
    v_next();
  };
  uint32_t s_free_ph[TILES] = {0, 0}, p_full_ph[TILES] = {0, 0}, p_half_ph[TILES] = {0, 0};
  bool s_pending[TILES] = {false, false};     // scores issued whose release has not been waited for yet

  // dh 64, and the score-only sweep: a warp for the scores (it shares an issue port with four softmax warps; with the tiles'
  // checks out of the loop and one election a tile, 4444 x 17776 x 48 heads 857 -> 852 us) ...
  auto issue_scores = [&](const Item& it) {
    const bool two = tile_live(it, 1);
    for (int j = 0; j < n_kv; ++j) {
      wait_k(j == 0);
      if (!ok) return;
      if (s_pending[0]) wait_phase(&s_free[0], s_free_ph[0]);
      if (!ok) return;
      if (elect_one()) {
        mma_scores(0);
        if (!two) {
          mma_commit(&k_empty[k_st]);
          if (j == n_kv - 1) mma_commit(&q_empty[q_st]);
        }
      }
      __syncwarp();
      s_pending[0] = true;
      if (two) {
        if (s_pending[1]) wait_phase(&s_free[1], s_free_ph[1]);
        if (!ok) return;
        if (elect_one()) {
          mma_scores(1);
          mma_commit(&k_empty[k_st]);
          if (j == n_kv - 1) mma_commit(&q_empty[q_st]);
        }
        __syncwarp();
        s_pending[1] = true;
      }
      k_next();
    }
    q_next();
  };
  // ... and one for the products: neither stream waits for the other's barriers.
  auto issue_products = [&](const Item& it) {
    for (int j = 0; j < n_kv; ++j) {
      wait_v();
#pragma unroll
      for (int t = 0; t < TILES; ++t) {
        if (!ok) return;
        if (!tile_live(it, t)) continue;
        wait_phase(&p_full[t], p_full_ph[t]);
        if (!ok) return;
        if (elect_one()) {
          mma_product(t, 0, j == 0);
          mma_product(t, 1, false);
          mma_commit(&pv_done[t]);
        }
        __syncwarp();
      }
      v_done();
    }
  };
  // dh 128, one warp for both tiles: O += P(j) V(j) and S(j+1) of one tile go out in one piece, then
  // those of the other.  (With a warp per tile the two bursts share the tensor pipe and both end late.)
  auto issue_both = [&](const Item& it) {
    const bool live[TILES] = {tile_live(it, 0), tile_live(it, 1)};
    // (after a score-only sweep: its last scores are overwritten without asking)
#pragma unroll
    for (int t = 0; t < TILES; ++t) {
      if (ok && s_pending[t]) wait_phase(&s_free[t], s_free_ph[t]);
      s_pending[t] = false;
    }
    if (!ok) return;
    wait_k(true);
    if (!ok) return;
    if (elect_one()) {
#pragma unroll
      for (int t = 0; t < TILES; ++t)
        if (live[t]) mma_scores(t);
    }
    __syncwarp();
    k_done(n_kv == 1);
    for (int j = 0; j < n_kv; ++j) {
      const bool more = j + 1 < n_kv;
      wait_v();
      if (!ok) return;
#pragma unroll
      for (int t = 0; t < TILES; ++t) {
        if (!live[t]) continue;
        wait_phase(&p_half[t], p_half_ph[t]);
        if (!ok) return;
        if (elect_one()) mma_product(t, 0, j == 0);
        __syncwarp();
        if (more && t == 0) wait_k(false);
        if (!ok) return;
        wait_phase(&p_full[t], p_full_ph[t]);
        if (!ok) return;
        if (elect_one()) {
          mma_product(t, 1, false);
          if (more) mma_scores(t);          // queued behind the product, which reads P from the same columns
          else mma_commit(&pv_done[t]);
        }
        __syncwarp();
      }
      v_done();
      if (more) k_done(j + 2 == n_kv);
    }
    q_next();
  };

  // ---- softmax threads -------------------------------------------------------------------------
  const int tile = ((warp - 4) >> 3) & 1;
  const int half = ((warp - 4) >> 2) & 1;
  const int quad = warp & 3;                               // TMEM lanes [32 * quad, 32 * quad + 32)
  const int r = quad * 32 + lane;                          // query row inside the tile = TMEM lane
  const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16) + tile * C::TM_TILE;
  const uint32_t s_tmem = t_lane + half * COLS;
  uint32_t p_tmem = t_lane + C::TM_P + half * (C::ALIAS ? COLS : COLS / 2);
  const uint32_t o_tmem = t_lane + C::TM_O + half * (DH / TPR);
  int set = 0;                 // offset of the barriers in use (kDry: the rehearsal's) ...
  uint32_t live = 1;           // ... and what their phases advance by
  RowSums sums;
  float poly_abs = 0.f, m_ref = 0.f, m_true = 0.f;
  // The two warps that share 32 rows meet: all of them, with a vote on going on (a warp that gave up
  // still comes here, so that the other does not wait for it) ...
  const int pair_bar = 2 + tile * 4 + quad;
  auto agree = [&]() { ok = named_barrier_and(pair_bar, 64, ok); };
  // ... and one value from each of the two threads of a row; returns the partner's.
  auto exchange = [&](float mine) -> float {
    volatile float* xch = reinterpret_cast<volatile float*>(smem + C::OFF_XCH) + tile * 2 * BM;
    named_barrier(pair_bar, 64);
    xch[half * BM + r] = mine;
    named_barrier(pair_bar, 64);
    return xch[(half ^ 1) * BM + r];
  };

  // The reference of this thread's row from its first block of scores (which has arrived, if ok): the
  // largest of them.  Both threads of a row come here and get the same value.
  auto first_max = [&]() {
    float m = -INFINITY;
    if (ok) {
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        float s[CH];
        ld_scores(s_tmem + c * CH, s);
        wait_scores(s);
        mask_tail(s, p.keys - half * COLS - c * CH, -INFINITY);
        const float mc = row_max(s);
        m = max3_nan(m, mc, mc);
      }
    }
    agree();
    if (!ok) return;
    const float other = exchange(m);
    m_ref = max3_nan(m, other, other);
    if (SCALED) m_ref *= p.q_scale;
  };
  // One key block: this thread's COLS scores in four chunks, the next on its way from TMEM.
  auto run_block = [&](int j, auto mode_tag, auto masked_tag, auto track_tag) {
    constexpr bool MASKED = decltype(masked_tag)::value;   // some keys of the block may lie past the end
    constexpr Mode MODE = decltype(mode_tag)::value;
    constexpr bool TRACK = decltype(track_tag)::value;
    constexpr bool CLAMP = MODE == REPEAT;
    mbar_wait_sticky(&s_full[set + tile], s_ph, abort_flag, ok);
    if (C::FIRST_MAX && MODE != REPEAT && j == 0) first_max();
    tc_fence_after();
    s_ph ^= live;
    const int valid = p.keys - j * BN - half * COLS;     // keys of this thread's columns that exist
    auto adjust = [&](float(&s)[CH], int c) {
      // score -> exponent relative to the row's reference (zero for dh 64 but in the repeat of a flagged row)
      if (SCALED || C::FIRST_MAX || MODE == REPEAT) {
        const f32x2 c2 = make_float2(p.q_scale, p.q_scale), m2 = make_float2(-m_ref, -m_ref);
#pragma unroll
        for (int t = 0; t < CH; t += 2) {
          f32x2 v = pack_f32x2(s[t], s[t + 1]);
          if (!C::FIRST_MAX && MODE != REPEAT) v = __fmul2_rn(v, c2);
          else if (SCALED) v = fma_f32x2(v, c2, m2);
          else v = add_f32x2(v, m2);
          s[t] = v.x;
          s[t + 1] = v.y;
        }
      }
      if (MODE == PROBE) {
        if (MASKED) mask_tail(s, valid - c * CH, -INFINITY);
        const float m = row_max(s);
        m_true = max3_nan(m_true, m, m);
      }
      if (MASKED) mask_tail(s, valid - c * CH, PAST_END);
    };
    uint32_t pk[COLS / 2];                             // packed probabilities
    float b0[CH], b1[CH], b2[CH];
    ld_scores(s_tmem, b0);
    ld_scores(s_tmem + CH, b1);
    ld_scores(s_tmem + 2 * CH, b2);
    tmem_ld_wait();
    tmem_ld_tie(b0);
    tmem_ld_tie(b1);
    tmem_ld_tie(b2);
    adjust(b0, 0);
    exp_cols<DH, 0, CLAMP, TRACK>(b0, &pk[0], sums, poly_abs);
    ld_scores(s_tmem + 3 * CH, b0);
    adjust(b1, 1);
    exp_cols<DH, 1, CLAMP, TRACK>(b1, &pk[CH / 2], sums, poly_abs);
    wait_scores(b0);
    if (C::ALIAS && MODE != PROBE) {
      tmem_st16(p_tmem, *reinterpret_cast<uint32_t(*)[16]>(&pk[0]));   // all scores are in registers
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(&p_half[set + tile]);
    } else {
      tc_fence_before();
      mbar_arrive(&s_free[set + tile]);                         // S(j) is in registers: S(j+1) may land
    }
    adjust(b2, 2);
    exp_cols<DH, 2, CLAMP, TRACK>(b2, &pk[CH], sums, poly_abs);
    adjust(b0, 3);
    exp_cols<DH, 3, CLAMP, TRACK>(b0, &pk[3 * CH / 2], sums, poly_abs);
    if (MODE == PROBE) return;
    if (!C::ALIAS) {
      if (j > 0) {                                        // the previous product reads the same columns
        mbar_wait_sticky(&pv_done[set + tile], pv_ph, abort_flag, ok);
        pv_ph ^= live;
        tc_fence_after();
      }
      tmem_st32(p_tmem, pk);
    } else {
      tmem_st16(p_tmem + COLS / 4, *reinterpret_cast<uint32_t(*)[16]>(&pk[16]));
    }
    tmem_st_wait();
    tc_fence_before();
    mbar_arrive(&p_full[set + tile]);
  };
  // Blocks without keys past the end.  With few of them they all take the masking form, so that
  // only one body has to be fetched.
  const int n_plain = p.keys / BN > 3 ? p.keys / BN : 0;
  auto run_blocks = [&](auto mode_tag, auto track_tag) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sums.plain[i] = make_float2(0.f, 0.f);
    sums.rounded[0] = sums.rounded[1] = make_float2(0.f, 0.f);
    poly_abs = 0.f;
#pragma unroll 1
    for (int j = 0; ok && j < (set ? min(n_plain, 1) : n_plain); ++j) run_block(j, mode_tag, std::false_type{}, track_tag);
#pragma unroll 1
    for (int j = n_plain; ok && j < (set ? min(n_kv, n_plain + 1) : n_kv); ++j) run_block(j, mode_tag, std::true_type{}, track_tag);
  };
  using PassT = std::integral_constant<Mode, PASS>;
  using ProbeT = std::integral_constant<Mode, PROBE>;
  using RepeatT = std::integral_constant<Mode, REPEAT>;
  // Sum of a row over its threads, and whether the row left the range.  Any probability of 2^90 or
  // more shows in the sum: the sums only ever grow, and an overflowed one is infinite or not a number.
  // At or below 2^-90 the row's scores lie so far below zero that the small terms were flushed away.
  // The threads of the row decide the same (an infinity stands for a thread's own flag).
  auto row_sum = [&](bool& flag) -> float {
    const float l = sum_partials(sums.plain);
    float seen = !(l < DANGER) || poly_abs > 120.f ? INFINITY : l;
    const float other = exchange(seen);
    seen += other;
    flag = !(seen < DANGER) || !(seen > TINY);
    return l + other;            // used only where nothing was flagged
  };
  // The accumulator is final once the item's last product has finished: normalise and store.
  // l_row: sum of the row's probabilities, for lse; O goes by the sum of what it was made from.
  auto finish = [&](const Item& it, float l_row) {
    float o_row = l_row;
    if (C::ROUNDED_SUM) {
      const float mine = sum_partials(sums.rounded);
      o_row = mine + exchange(mine);
    }
    ok = mbar_wait_warp(&pv_done[set + tile], pv_ph, abort_flag);
    pv_ph ^= live;
    if (!ok) return;
    tc_fence_after();
    const int row = it.row0 + tile * BM + r;
    const float inv_l = 1.f / o_row;
    // dh 128: four lanes hold 64 bytes of four rows; transposed among themselves, a store covers whole
    // 64-byte pieces of eight rows instead of 16 bytes of 32, which keeps the load/store unit busy for
    // 4000 cycles an item (4608 x 4608 x 24 heads 232 -> 228 us).  The dh 64 kernel gains the same on its
    // short calls (1101 keys 22.4 -> 21.3 us) but its main loop then comes out 2-4 % slower, so it keeps the
    // plain stores.
    constexpr bool TRANSPOSE = DH == 128;
    const int first_row = TRANSPOSE ? row & ~3 : row;
    __nv_bfloat16* orow = p.o + ((size_t)it.b * p.rows + first_row) * ((size_t)p.heads * DH) + (size_t)it.h * DH +
                          half * (DH / TPR) + (TRANSPOSE ? (lane & 3) * 8 : 0);
#pragma unroll 1
    for (int ch = 0; ch < DH / TPR / 32; ++ch) {
      uint32_t o[32];
      tmem_ld32(o_tmem + ch * 32, o);
      tmem_ld_wait_on(o);
      uint4 c[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        c[q] = make_uint4(pack_bf16x2(__uint_as_float(o[8 * q + 0]) * inv_l, __uint_as_float(o[8 * q + 1]) * inv_l),
                          pack_bf16x2(__uint_as_float(o[8 * q + 2]) * inv_l, __uint_as_float(o[8 * q + 3]) * inv_l),
                          pack_bf16x2(__uint_as_float(o[8 * q + 4]) * inv_l, __uint_as_float(o[8 * q + 5]) * inv_l),
                          pack_bf16x2(__uint_as_float(o[8 * q + 6]) * inv_l, __uint_as_float(o[8 * q + 7]) * inv_l));
      if (TRANSPOSE) {
        transpose_4x4(c, lane);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (first_row + k < p.rows) *reinterpret_cast<uint4*>(orow + (size_t)k * p.heads * DH + ch * 32) = c[k];
      } else if (row < p.rows) {
#pragma unroll
        for (int k = 0; k < 4; ++k) reinterpret_cast<uint4*>(orow + ch * 32)[k] = c[k];
      }
    }
    tc_fence_before();     // ordered before this thread's next hand-over, after which O is overwritten
    if (p.lse && half == 0 && row < p.rows)
      p.lse[((size_t)it.b * p.heads + it.h) * p.rows + row] = fmaf(m_ref, 0.6931471805599453f, logf(l_row));
  };

  // All threads meet after the first pass and agree on whether there is a second.
  auto second_pass = [&]() -> bool {
    tc_fence_before();
    const bool go = named_barrier_and(0, THREADS, ok && !*abort_flag) && *any_flag;
    tc_fence_after();
    return go;
  };
  // Calls f(item) for every item of this CTA with a row that left the range.
  auto for_flagged = [&](auto f) {
#pragma unroll 1
    for (int i = 0; i < n_items; ++i) {
      const uint32_t word = ((volatile uint32_t*)item_flag)[i >> 5];
      if (word >> (i & 31) & 1) f(item_at(i));
    }
  };

  // First pass over the CTA's items, then the flagged ones once more in two sweeps.
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_HELPER));
    // The first loads stand right behind the wait, with all that they need worked out: in `produce`, whose code is met for the
    // first time, they came 1.5 to 3.3 us after it, now 0.5 to 1.3.  us: block of 288 x 512 41.2 -> 39.9, of 1101 x 1536 115.0 ->
    // 113.4; one tile an item and few blocks gain the most.
    const Item first = item_at(0);
    if (threadIdx.x == 0) {
      mbar_expect_tx(&k_full[0], C::TILE_BYTES);
      mbar_expect_tx(&q_full[0], p.tiles * C::TILE_BYTES);
    }
    grid_dep_wait();
    if (warp == 0) {
      if (lane == 0) {
#pragma unroll
        for (int a = 0; a < C::ATOMS; ++a)
          tma_load_3d(smem + C::OFF_K + a * ATOM_BYTES, &map_k, &k_full[0], first.h * DH + a * 64, 0, first.b);
        load_q(first);
        ++k_issued;
        k_next();
        for (int i = 0; ok && i < n_items; ++i) produce(i ? item_at(i) : first, true, i == 0);
      }
      __syncwarp();
      const bool again = second_pass();
      if (lane == 0) {
        if (again)
          for_flagged([&](const Item& it) {
#pragma unroll 1
            for (int with_v = 0; ok && with_v < 2; ++with_v) produce(it, with_v != 0, false);
          });
        if (!ok) {
          // gave up: let the copies already issued land before the CTA leaves (the latest fill of
          // each stage; older fills were consumed before their stage was reused)
          auto drain = [&](uint64_t* full, int issued, int stages) {
            for (int i = max(0, issued - stages); i < issued; ++i) {
              volatile uint32_t dummy = 0;
              mbar_wait(&full[i % stages], (uint32_t)(i / stages) & 1u, &dummy);
            }
          };
          drain(q_full, q_issued, QBUF);
          drain(k_full, k_issued, KS);
          drain(v_full, v_issued, VS);
        }
      }
      __syncwarp();
    } else if (warp <= C::ISSUERS) {
      auto issue = [&](const Item& it, Mode mode) {
        if (C::ALIAS) {
          if (mode == PROBE) issue_scores(it);
          else issue_both(it);
        } else if (warp == 1) {
          issue_scores(it);
        } else if (mode != PROBE) {
          issue_products(it);
        }
      };
      // one call site for all sweeps (the loops keep to the helper warps' registers)
      bool again = false;
      Mode mode = PASS;
      for (int i = 0;;) {
        if (again)
          while (i < n_items && !(((volatile uint32_t*)item_flag)[i >> 5] >> (i & 31) & 1)) ++i;
        if (!ok || i >= n_items) {
          if (again || !second_pass()) break;
          again = true;
          mode = PROBE;
          i = 0;
          continue;
        }
        issue(item_at(i), mode);
        if (mode == PROBE) {
          mode = REPEAT;
        } else {
          ++i;
          if (again) mode = PROBE;
        }
      }
    } else {
      second_pass();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REG_SOFTMAX));
    // dh 64: with q and k out of an RMSNorm (gains g), a rotation and, for q, the factor
    // log2(e) / sqrt(dh), a head of q has norm <= max|g_q| * log2(e) and a head of k norm <=
    // sqrt(dh) * max|g_k|: every score lies within +-log2(e) * sqrt(dh) * max|g_q| * max|g_k|
    // (plus the bf16 roundings, under half a percent).  Far inside the polynomial's range nothing
    // needs to be tracked per score.
    constexpr bool POLY = kPolyPairs<DH> != 0;
    bool bounded = !POLY;
    if (POLY && !SCALED && p.gain_q && p.gain_k) {
      const int ts = threadIdx.x - 128;
      if (ts < DH) {
        atomicMax(&gain_max[0], __float_as_uint(fabsf(__bfloat162float(p.gain_q[ts]))));
        atomicMax(&gain_max[1], __float_as_uint(fabsf(__bfloat162float(p.gain_k[ts]))));
      }
      named_barrier(1, SOFTMAX_THREADS);
      const float gq = __uint_as_float(*(volatile uint32_t*)&gain_max[0]);
      const float gk = __uint_as_float(*(volatile uint32_t*)&gain_max[1]);
      static_assert(!POLY || DH == 64, "log2(e) * sqrt(64) below");
      constexpr float factor = 11.55f * 1.01f;
      bounded = gq * gk * factor < 100.f;    // false for a NaN gain
    }
    // Round -1 is the rehearsal: its rows lie past the end (from a multiple of 128 on, because finish stores groups of four
    // rows), its probabilities go where the first product overwrites them (P over S would meet the first scores).
    const uint32_t p_live = p_tmem;
    if (REHEARSE) {
      if (C::ALIAS) p_tmem = o_tmem;
      set = kDry;
      live = 0;
      s_ph = pv_ph = 1;
    } else {
      grid_dep_wait();
    }
    for (int i = REHEARSE ? -1 : 0; i < n_items; ++i) {
      if (REHEARSE && i == 0) {
        grid_dep_wait();
        p_tmem = p_live;
        set = 0;
        live = 1;
        s_ph = pv_ph = 0;
      }
      const Item it = i < 0 ? Item{(p.rows + BM - 1) / BM * BM, 0, 0} : item_at(i);
      // (with one tile an item the second tile's warps, which have nothing else to do, rehearse while the first's go ahead)
      if (i < 0 ? p.tiles == 1 && tile == 0 : !tile_live(it, tile)) continue;
      if (ok) {
        if (bounded) run_blocks(PassT{}, std::false_type{});
        else run_blocks(PassT{}, std::bool_constant<POLY>{});
      }
      agree();
      if (!ok) break;
      bool flag;
      const float l = row_sum(flag);
      if (flag && i >= 0) {
        *any_flag = 1;
        atomicOr(&item_flag[i >> 5], 1u << (i & 31));
      }
      finish(it, l);
    }
    if (second_pass())
      for_flagged([&](const Item& it) {
        if (!tile_live(it, tile)) return;
        bool flag = false;
        m_true = -INFINITY;
        m_ref = 0.f;
        if (ok) run_blocks(ProbeT{}, std::bool_constant<POLY>{});
        agree();
        if (!ok) return;
        row_sum(flag);
        // the true maximum, relative to the reference of the pass; where there is none (a NaN, an
        // infinity) the row has no finite probabilities
        const float other = exchange(m_true);
        m_true = max3_nan(m_true, other, other);
        if (flag) m_ref = fabsf(m_true) < INFINITY ? m_ref + m_true : NAN;
        run_blocks(RepeatT{}, std::false_type{});
        agree();
        if (!ok) return;
        finish(it, row_sum(flag));
        m_ref = 0.f;
      });
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *abort_flag && p.status) atomicExch(p.status, STATUS_TIMEOUT_MBARRIER);
}

// How a launch is divided: tiles an item, items a head, items, CTAs.
struct AttnGrid {
  int tiles, q_items, items, ctas;
};

int attention_grid(const AttnLaunch& a, AttnGrid* g) {
  const long long q_tiles = (a.rows + BM - 1) / BM, bh = (long long)a.heads * a.batch;
  // two tiles per item share their K and V blocks; where every tile can have an SM of its own they
  // are faster apart
  g->tiles = q_tiles * bh <= sm_count() ? 1 : TILES;
  g->q_items = (int)((q_tiles + g->tiles - 1) / g->tiles);
  const long long items = g->q_items * bh;
  if (items > (1ll << 30)) return XEMA_EINVAL;
  g->items = (int)items;
  // one CTA per SM (each takes all of TMEM); more only where a CTA could not keep a flag per item
  g->ctas = std::max((int)std::min<long long>(items, sm_count()), (int)((items + MAX_ITEMS - 1) / MAX_ITEMS));
  return XEMA_OK;
}

template <int DH, bool SCALED, bool REHEARSE>
int launch_attention_t(const AttnLaunch& a, const AttnGrid& g, cudaStream_t stream, bool chained) {
  using C = Cfg<DH>;
  static PerDeviceInt attr_done;
  auto kern = attention_kernel<DH, SCALED, REHEARSE>;
  if (int rc = ensure_smem_attr(kern, C::SMEM_BYTES, attr_done)) return rc;
  AttnParams p;
  p.o = (__nv_bfloat16*)a.o;
  p.lse = a.lse;
  p.batch = a.batch;
  p.rows = a.rows;
  p.keys = a.keys;
  p.heads = a.heads;
  p.q_scale = a.q_scale;
  p.status = a.status;
  p.gain_q = (const __nv_bfloat16*)a.gain_q;
  p.gain_k = (const __nv_bfloat16*)a.gain_k;
  p.tiles = g.tiles;
  p.q_items = g.q_items;
  p.items = g.items;
  return launch_kernel(kern, dim3(g.ctas), THREADS, C::SMEM_BYTES, stream, chained, a.map_q, a.map_k, a.map_v, p);
}
}  // namespace

int launch_attention(const AttnLaunch& a, cudaStream_t stream, bool chained) {
  if (a.rows == 0 || a.batch == 0) return XEMA_OK;
  AttnGrid g;
  if (int rc = attention_grid(a, &g)) return rc;
  // Behind another launch there is a wait to use, and up to kRehearseBlocks key blocks a CTA the gain is the larger.
  const long long rounds = (g.items + g.ctas - 1) / g.ctas;
  const bool rehearse = chained && rounds * ((a.keys + BN - 1) / BN) <= kRehearseBlocks;
  const bool scaled = a.q_scale != 1.f;
  if (a.head_dim == 64)
    return scaled     ? launch_attention_t<64, true, false>(a, g, stream, chained)
           : rehearse ? launch_attention_t<64, false, true>(a, g, stream, chained)
                      : launch_attention_t<64, false, false>(a, g, stream, chained);
  if (a.head_dim == 128)
    return scaled     ? launch_attention_t<128, true, false>(a, g, stream, chained)
           : rehearse ? launch_attention_t<128, false, true>(a, g, stream, chained)
                      : launch_attention_t<128, false, false>(a, g, stream, chained);
  return XEMA_EINVAL;
}

int attn_prepare(AttnLaunch* a, const void* q, long long ldq, long long q_batch_rows, const void* k, const void* v,
                 long long ldkv, long long kv_batch_rows) {
  if (a->batch < 1 || a->rows < 0 || a->keys < 1 || a->heads < 1) return XEMA_EINVAL;
  if (a->head_dim != 64 && a->head_dim != 128) return XEMA_EINVAL;
  if (a->heads > 65535 || a->batch > 65535) return XEMA_EINVAL;
  if (!q || !k || !v || !a->o) return XEMA_EINVAL;
  if ((ldq & 7) || (ldkv & 7)) return XEMA_EALIGN;
  auto mis = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) != 0; };
  if (mis(q) || mis(k) || mis(v) || mis(a->o)) return XEMA_EALIGN;
  const long long width = (long long)a->heads * a->head_dim;
  int rc = encode_tmap_bf16(&a->map_q, q, width, a->rows > 0 ? a->rows : 1, a->batch, ldq, q_batch_rows, BM);
  if (rc) return rc;
  rc = encode_tmap_bf16(&a->map_k, k, width, a->keys, a->batch, ldkv, kv_batch_rows, BN);
  if (rc) return rc;
  return encode_tmap_bf16(&a->map_v, v, width, a->keys, a->batch, ldkv, kv_batch_rows, BN);
}

}  // namespace xema
