// Tensor-core forward kernel for sm_100a: a query tile per CTA at a time, two independent streams of key chunks.
//
// A CTA owns a query tile (128 queries) of one (head, batch row) and walks the live 64-key chunks of its list (laid by the planner
// over the tile's own live keys).  A chunk comes with the class of its two halves for every warp's 32 rows: dead halves are
// skipped, live ones take no element mask.  Two streams share the list, chunk g of the CTA going to stream g % 2; each has its own
// scores and probabilities, and both add to one accumulator, in the order of the list.  320 threads:
//   warps 0-3, 4-7  softmax of stream 0 and 1: thread m of the group owns query slot m (TMEM lane m).  A chunk's 64 scores
//                   come from TMEM in two halves of 32: the plan's element mask, the probabilities (12 to 38 % of the exponentials,
//                   by build, on the FMA pipe by a cubic, the rest on the exponential pipe), and P (packed bf16) over the scores
//                   that have been read.
//   warp 8          Q and the MMAs: once P(g) is complete, O += P(g) [V(g), 1] and S(g + 2) = Q K(g + 2) go out back to back; they
//                   execute in issue order, so that S may overwrite P.  The warp runs converged and what it computes is uniform, so
//                   that descriptors stay in uniform registers (a lane of its own: eight register moves per MMA); one elected lane
//                   issues.
//   warp 9          K and V chunks by tensor-map copies into rings of four stages.
// The row sums are 16 more columns of O: the products take 16 columns of V from a block behind the stages (the leading byte offset of
// V's descriptor) that is 1 where key and column agree modulo 4, and a sum is four of them added up.  (A product shifts its addends
// to the largest exponent and cuts them off there: with ones everywhere 16 addends a step lose up to a bit of the sum each, always
// in the same direction.  Over the 34240 keys of the last 2K step, keys three times as sharp, outputs were too large by 1.0e-4; with
// four addends a step by 1.5e-5, with one too small by 1.9e-5, with sums by additions too small by 1.5e-5.  Time: the same.)  A sum
// by additions is one instruction a score (64, beside the 346 that a warp issues per chunk now, all included).
// Q is a TMEM operand: a step of S = Q K with both operands in shared memory waits for their 6 KB (50 cycles, 32 with Q in TMEM), and
// the two CTAs of an SM share that.
// MANY: a CTA takes several tiles in turn.  Q has two buffers; K and V copies of the next tile go out behind the last ones of this
// one, the softmax warps look the next list up while they wait for their accumulator, and the
// output leaves by tensor-map stores that nobody waits for until the buffer's next use.  What orders the tiles: the first
// P V product of a tile (which overwrites the accumulator) follows the softmax warps' P, which they write after they and the
// warp with the other stream of their rows have read the accumulator; a Q copy follows the stores of the tile that had its buffer.
// Two CTAs per SM, so that every scheduler has four softmax warps of four streams that are in different phases.
// TMEM columns: S and P of stream s at 64 s, O at 128, the row sums at 192, Q at 208.
//
// The reference of a row (probabilities are 2^(score * scale - reference)) is the maximum of the first chunk's first 32 keys
// and stays (0 where none of them is live): bf16 and fp32 have the same exponent range, so P and its sum are as accurate at 2^90 as
// at 1, and a tile's rows need neither a maximum per chunk nor a rescaled accumulator.  The key it is taken from has a probability of
// 1, without rounding, and the larger its weight the more that is worth: error against fp64 (relative L2, N(0, 1) inputs; with the
// maximum of eight keys / of 32 / with two accumulators and a maximum of eight keys for each) 256px step 8 2.306e-3 / 2.282e-3 /
// 2.293e-3, 256px step 10 2.291 / 2.273 / 2.281, 512px step 10 2.324 / 2.316 / 2.322.  The stream with the first chunk hands the
// reference to the other one (which is then a little behind: both streams at the same point of a chunk are 4 to 5 % slower).  Each
// stream's first chunk is a copy of the loop's body in front of it, so that its scores are loaded and masked once: as a case inside
// the loop (with eight keys) / as a load of its own in front of it / as a copy, 256px steps 8, 9 and 10 with 960 units take 24.9 /
// 25.4 / 25.0, 54.4 / 55.4 / 54.4 and 74.4 / 75.1 / 73.9 us, step 9 with 480 30.5 / 31.5 / 30.6, last 512px step 143.0 / 142.8 / 141.0,
// with an 8-bit cache 222.9 / 220.6 / 219.8, 2K step 12 150.9 / 149.9 / 149.0.  At the end a row
// whose sum or output is out of range (kRange, kSmall) sends the CTA through its lists again (`exact`), each list twice: once for
// the rows' maxima, then against them, for the 32 rows of a warp that it belongs to, which are stored then.
//
// What bounds it (ncu, 2K step, full mask): issue slots 70 % busy, exponential pipe 65 %, tensor pipe active 58 %; 5.4 instructions a
// score.  (More warps do not help: three streams of softmax warps, or three score buffers so that none waits for its next scores,
// took as long as before with the sums still added by instructions.)  Measured on B200, in thousand cycles of a launch, with one
// accumulator and sums of its own per stream / shared accumulator and sums by products / and Q in TMEM / and six pairs of a half's
// 16 on the FMA pipe: 2K step with the full mask 8840 / 8100 / 7720 / 7500, window 1/4 2710 / 2540 / 2455 / 2400; last 512px step,
// 288 units 285 / 292 (with one tile per CTA 281) / 271 / 267; last 256px step with 128 units 31.0 / 28.5 / 28.1 / 27.9.  All rows out
// of range, so that every list is walked three times: 2K step, window 1/4, 1365 -> 3660 to 3730 us, last 256px step with 960 units
// 84 -> 200, last 512px step on an 8-bit cache 229 -> 573.
//
// Every wait on an mbarrier is bounded; when one runs out the CTA raises the plan's status word, waits for its copies and products
// in flight, frees its TMEM and returns (the softmax warps still meet the issuing warp for every chunk, so that the named barriers
// complete).  The element mask, the lists and CFG sharing (second store at batch row b + B) are those of the plan (paper
// Sections 2 and 3).
#include <algorithm>
#include <cstring>
#include <mutex>

#include "litevar_tc_ptx.h"

namespace litevar {

using namespace tc;

namespace {

constexpr int kChunkKeys = kBlockN / 2;
constexpr uint32_t kChunkBytes = kChunkKeys * kHeadDim * 2;
constexpr int kStages = 4;                // K ring and V ring; chunk g of the CTA is in stage g % kStages
constexpr int kSumCols = 16;              // of the accumulator, behind O: row sums over the keys that agree with the column modulo 4
constexpr int kThreads = 320;             // two streams of four softmax warps, one warp for the MMAs, one for the copies
// TMEM columns: S (and P over it) of stream s at 64 s, then O and the row sums, then Q
constexpr uint32_t kTmemCols = 256, kColO = 128, kColQ = kColO + kHeadDim + kSumCols;

constexpr unsigned kIdleNs = 200;  // (50 or 500: the same)
constexpr int kPolls = 1 << 23;    // of kIdleNs and more: two seconds
constexpr int kMaxTiles = 1024;  // of a CTA that takes several (MANY)
// A row sum of the first pass outside (2^-64, 2^96) goes to the second pass.  (The lower end keeps the traces of dead keys, 2^-125
// each, below 2^-41 of a sum over the longest list there is, kMaxScales * kMaxScale^2 = 2^20 keys in one accumulator; 2^-46 over the
// 34240 of the last 2K step.)
constexpr float kRange = 79228162514264337593543950336.f, kRangeLow = 5.42101086242752217e-20f;
// So does a row of output that is not finite (sums of P V overflow before those of P), or so small beside its weight, where that is
// above 1, that products P V may have been subnormal (2^-126 each, 2^20 of them: 2^-12 of the smallest output that is kept).
constexpr float kSmall = 5.04870979341447553e-29f;  // 2^-94
static_assert((long long)kMaxScales * kMaxScale * kMaxScale <= 1 << 20, "keys of a list, in kRangeLow and kSmall");

// 8-bit cache build: the codes of a chunk (64 rows of 64 bytes, as the tensor-map copy delivers them, no swizzle) and its rows'
// scales and zero points, on their way into the bf16 stages (empty in the bf16 build).  Chunk g is number g / 2 of stream g % 2.
constexpr uint32_t kCodeBytes = kChunkKeys * kHeadDim;
template <bool KV8>
struct CodeStage {};
template <>
struct CodeStage<true> {
  alignas(128) uint8_t kc[2][2][kCodeBytes];  // [stream][number % 2]
  alignas(128) uint8_t vc[2][kCodeBytes];
  float k_sz[2][2][2][kChunkKeys];  // [stream][number % 2][scale, zero point][row]
  float v_sz[2][2][kChunkKeys];
  uint64_t kc_full[2][2], vc_full[2], vc_free[2];
};

template <bool KV8, bool MANY>
struct WsShared : CodeStage<KV8> {
  alignas(1024) uint8_t q[MANY ? 2 : 1][kTileBytes];  // Q; at the end of a tile the output rows pass through it
  alignas(1024) uint8_t k[kStages][kChunkBytes];
  alignas(1024) uint8_t v[kStages][kChunkBytes];
  alignas(1024) uint8_t ones[16 * kHeadDim * 2];  // 16 keys of the part of V that gives the row sums
  float ref[kBlockM];     // the rows' references, from the stream with the tile's first chunk to the other
  float top[2][kBlockM];  // second pass: the rows' maxima over the keys of each stream
  alignas(8) uint64_t q_full[2], q_free;
  uint64_t k_full[kStages], k_free[kStages], v_full[kStages];
  uint64_t s_full[2], o_full, drained;
  uint32_t held[4][MANY ? kMaxTiles / 32 : 1];  // bit x: the 32 rows of the CTA's tile x are left to the second pass
  int out_of_range[4][2];  // 1 + the last even and odd tile with such rows (a warp is at most one tile ahead of its partner)
  uint32_t tmem_base;
  int abort_flag, redo;
  int met[2];  // 1 + the last chunk of each stream whose P the issuing warp has met
};

// Instruction descriptors (kind::f16).  Fields: D type at bit 4 (1: fp32), A and B type at bits 7 and 10 (1: bf16), B transposed
// (MN-major, as V lies in shared memory) at bit 16, N / 8 at bit 17, M / 16 at bit 24.
constexpr uint32_t kIdescS = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kChunkKeys >> 3) << 17) |
                             ((uint32_t)(kBlockM >> 4) << 24);
constexpr uint32_t kIdescO = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)((kHeadDim + kSumCols) >> 3) << 17) |
                             ((uint32_t)(kBlockM >> 4) << 24);

// 2^x on the FMA pipe for x = score * scale - reference clamped to [-125, 100]: the caller's multiply-add saturates
// y = (100 - x) / 225 to [0, 1].  Dead keys (-inf) give 1 and 2^-125; a NaN saturates to 0 and gives 2^100, which takes the row's
// sum out of range.  x = n + f with n = round(x) and f in [-1/2, 1/2]; 2^f by a cubic fitted to it (relative error 7.5e-5, far
// inside the bf16 rounding of P), 2^n by adding n to the exponent field.
constexpr float kClampHigh = 100.f, kClampSpan = 225.f;
__device__ __forceinline__ float2 exp2_fma2(float2 y) {
  const float2 span = make_float2(-kClampSpan, -kClampSpan);
  const float2 t = __ffma2_rn(y, span, make_float2(12582912.f + kClampHigh, 12582912.f + kClampHigh));  // n in the low mantissa bits
  const float2 m = __fadd2_rn(make_float2(12582912.f + kClampHigh, 12582912.f + kClampHigh), make_float2(-t.x, -t.y));  // 100 - n
  const float2 f = __ffma2_rn(y, span, m);
  float2 z = __ffma2_rn(make_float2(0.05517153441905975f, 0.05517153441905975f), f,
                        make_float2(0.2426111102104187f, 0.2426111102104187f));
  z = __ffma2_rn(z, f, make_float2(0.6932610273361206f, 0.6932610273361206f));
  z = __ffma2_rn(z, f, make_float2(0.9999280571937561f, 0.9999280571937561f));
  return make_float2(__uint_as_float(__float_as_uint(z.x) + (__float_as_uint(t.x) << 23)),
                     __uint_as_float(__float_as_uint(z.y) + (__float_as_uint(t.y) << 23)));
}

// Which of a half's 16 pairs of exponentials take the FMA pipe (of every four keys e .. e + 3 the second pair): six with one tile
// per CTA, two with several on short lists (where the widest tiles are partly masked and the arithmetic is not what a tile waits for),
// three beside the widening of an 8-bit cache, whose arithmetic is on that pipe too.  Measured for 3 / 4 / 5 / 6 / 7 pairs, thousand
// cycles: 2K step 14 2470 / 2455 / 2436 / 2401 / 2426, with the full mask 7800 / 7720 / 7630 / 7500 / 7580; several tiles per CTA, last
// 256px step with 960 units, for 2 / 4 / 5 pairs: 131.8 / 132.6 / 135.5; 8-bit cache, last 512px step, for 3 / 4 / 5 449 / 457 / 460
// (with scales put beside the codes by instructions; 414 with asynchronous copies of them).
template <bool KV8, bool MANY>
__device__ __forceinline__ constexpr bool on_fma_pipe(int e) {
  return KV8 ? (e & 4) != 0 && e != 28 : MANY ? e == 4 || e == 20 : (e & 4) != 0 || (e & 15) == 0;
}

// One elected lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0u;
}
// mma_ts_x4 / mma_commit for a converged warp: one elected lane issues
template <int kAStep, int kBStep>
__device__ __forceinline__ void mma_ts_x4_one(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                              uint32_t accumulate_first) {
  if (elect_one()) mma_ts_x4<kAStep, kBStep>(d_tmem, a_tmem, b_desc, idesc, accumulate_first);
}
// A Q tile as the tensor-map copy left it (128-byte rows, 128-byte swizzle) -> 32 packed columns of TMEM, 16 elements a step.
// Products issued behind it by the same thread read what it wrote.
__device__ __forceinline__ void q_to_tmem(uint32_t taddr, uint64_t desc) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("tcgen05.cp.cta_group::1.128x256b [%0], %1;" ::"r"(taddr + 8 * i), "l"(desc + 2 * i) : "memory");
}
__device__ __forceinline__ void mma_commit_one(uint64_t* bar) {
  if (elect_one()) mma_commit(bar);
}
__device__ __forceinline__ KeyChunk chunk_at(const KeyChunk* c) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(c));
  return KeyChunk{v.x, v.y, v.z, v.w};
}
// mbar_wait_long for a wait of about a step's length with slack behind it: sleeps between the polls, whose instructions (ten each,
// one poll per 112 cycles) the softmax warps of the same scheduler would otherwise wait for.
__device__ __forceinline__ bool mbar_wait_idle(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
#pragma unroll 1
  do {
    if (*abort_flag) return false;
    if (clock64() - t0 > (1ll << 32)) {
      *abort_flag = 1;
      atomicExch(status, 1);
      return false;
    }
    __nanosleep(kIdleNs);
  } while (!mbar_try(bar, parity));
  return true;
}
// four fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
// Largest of 32 scores (dead ones: -inf), four chains of three-way maxima.
__device__ __forceinline__ float largest_score(const uint32_t* r) {
  float top[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) top[i] = fmaxf(__uint_as_float(r[i]), __uint_as_float(r[4 + i]));
#pragma unroll
  for (int e = 8; e < 32; e += 8)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      asm("max.f32 %0, %0, %1, %2;" : "+f"(top[i]) : "f"(__uint_as_float(r[e + i])), "f"(__uint_as_float(r[e + 4 + i])));
  return fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3]));
}
// Until *at >= n, or some seconds.  (One asm block: a loop in C++ here, however cold, costs the one-tile build's hot loop 4 %.)
__device__ __forceinline__ void wait_met(const int* at, int n) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .s32 v, i;\n\tmov.s32 i, 0;\n"
      "AGAIN:\n\tld.volatile.shared.s32 v, [%0];\n\tsetp.ge.s32 p, v, %1;\n\t@p bra MET;\n\tnanosleep.u32 200;\n\t"
      "add.s32 i, i, 1;\n\tsetp.lt.s32 p, i, 16777216;\n\t@p bra AGAIN;\nMET:\n\t}"
      ::"r"(smem_u32(at)), "r"(n)
      : "memory");
}
// Where a chunk's 64 rows are (`map`: 0 raster, else 1 + the patch-tiled key scale's map).
struct ChunkAt {
  int row, col, map, h, b;
};
__device__ __forceinline__ void load_chunk(void* dst, const CUtensorMap* raster, const CUtensorMap* patch, const ChunkAt& c,
                                           uint64_t* bar) {
  mbar_expect_tx(bar, kChunkBytes);
  if (c.map)
    tma_load_5d(dst, patch + (c.map - 1), 0, c.col, c.row, c.h, c.b, bar);
  else
    tma_load_4d(dst, raster, 0, c.row, c.h, c.b, bar);
}

// One chunk of codes -> bf16 rows in the 128-byte swizzle the tensor-map copies of the bf16 path produce (16-byte piece c of row m
// at position c ^ (m & 7)).  Paper Section 4 (8-bit Q/K/V): a row enters the attention as code * s + z, rounded to bf16; the
// arithmetic is widen_codes16's.  128 threads, two pieces of 16 codes each; consecutive threads take consecutive pieces.
__device__ __forceinline__ void widen_chunk(const uint8_t* codes, const float (&sz)[2][kChunkKeys], uint8_t* stage, int t) {
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int id = t + 128 * it, m = id >> 2, c = id & 3;
    const uint4 q = *reinterpret_cast<const uint4*>(codes + id * 16);
    uint4 lo, hi;
    widen_codes16(q, sz[0][m], shifted_zero_point(sz[1][m], sz[0][m]), lo, hi);
    uint8_t* row = stage + m * 128;
    *reinterpret_cast<uint4*>(row + (((2 * c) ^ (m & 7)) << 4)) = lo;
    *reinterpret_cast<uint4*>(row + (((2 * c + 1) ^ (m & 7)) << 4)) = hi;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> the tensor pipe's reads
}

// Scales and zero points of a chunk's 64 rows, two a lane, by asynchronous copies that arrive on `bar` (rows past L_k: 0 and 0;
// their codes arrive as zeros).
__device__ __forceinline__ void load_scales(float (&sz)[2][kChunkKeys], const float* scale, const float* zero, int row, int L_k, int lane,
                                            uint64_t* bar) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int j = lane + 32 * i, bytes = row + j < L_k ? 4 : 0, at = bytes ? row + j : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(&sz[0][j])), "l"(scale + at), "r"(bytes) : "memory");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(&sz[1][j])), "l"(zero + at), "r"(bytes) : "memory");
  }
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <bool KV8, bool MANY>
__global__ void __launch_bounds__(kThreads, 2)
fwd_ws_kernel(const __grid_constant__ TensorMaps tm, const __grid_constant__ FwdParams p, int n_q_tiles, int n_items) {
  static_assert(!(KV8 && MANY), "the code stages leave no room for a second Q buffer");
  constexpr int kQBufs = MANY ? 2 : 1;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  WsShared<KV8, MANY>& sm = *reinterpret_cast<WsShared<KV8, MANY>*>(smem_raw);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // warp-uniform
  // One query tile of one (head, batch row), in the grouped order of work_item, and its list.  A CTA takes items blockIdx.x,
  // blockIdx.x + gridDim.x, ... (MANY; else one).
  struct Item {
    int qt, h, b, n;  // n: chunks
    const KeyChunk* chunks;
    const uint2* mask;
  };
  auto item_at = [&](int w) {
    Item x;
    int unit;
    work_item(p, n_q_tiles, w, x.qt, unit);
    x.h = unit % p.n_heads;
    x.b = unit / p.n_heads;
    const SetDesc sd = p.head_to_set ? p.sets[p.head_to_set[x.h]] : p.set0;
    const int first = __ldg(&sd.chunk_ptr[x.qt]);
    x.n = __ldg(&sd.chunk_ptr[x.qt + 1]) - first;
    x.chunks = sd.chunks + first;
    x.mask = sd.chunk_mask;
    return x;
  };
  // Loop bounds that come from memory, marked as the same in all lanes: the issuing warps' counters and descriptors stay in uniform
  // registers (thousand cycles without / with it: several tiles per CTA, 256px steps 8 / 9 / 10 with 960 units 50.4 / 50.1, 100.7 /
  // 99.6, 134.0 / 131.0; 8-bit cache, last 512px step 417.5 / 414.5).  In the other build they do anyway, and the loop got slower.
  auto uniform = [](int v) { return MANY || KV8 ? __shfl_sync(0xffffffffu, v, 0) : v; };
  const int w_step = MANY ? (int)gridDim.x : n_items;
  const int n_tiles = MANY ? (n_items - (int)blockIdx.x + w_step - 1) / w_step : 1;  // of this CTA
  volatile int* abort_flag = &sm.abort_flag;

  if (warp == 8 && elect_one()) {  // each of the two warps sets up the barriers of its own copies
    mbar_init(&sm.q_full[0], 1);
    mbar_init(&sm.q_full[1], 1);
    mbar_init(&sm.q_free, 8);  // every softmax warp arrives when the tile's output rows have left the buffer
    mbar_init(&sm.s_full[0], 1);
    mbar_init(&sm.s_full[1], 1);
    mbar_init(&sm.o_full, 1);
    mbar_init(&sm.drained, 1);
    sm.abort_flag = 0;
    sm.redo = 0;
    sm.met[0] = sm.met[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 9 && elect_one()) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.k_full[s], KV8 ? 4 : 1);  // 8-bit cache: every softmax warp of the stream arrives
      if constexpr (!KV8) {
        mbar_init(&sm.k_free[s], 1);
        mbar_init(&sm.v_full[s], 1);
      }
    }
    if constexpr (KV8) {
      for (int s = 0; s < 2; ++s) {
        mbar_init(&sm.kc_full[s][0], 33);  // the copy of the codes and every lane's copies of scales
        mbar_init(&sm.kc_full[s][1], 33);
        mbar_init(&sm.vc_full[s], 33);
        mbar_init(&sm.vc_free[s], 4);
      }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (threadIdx.x < 4 * (sizeof(sm.held[0]) / sizeof(uint32_t))) (&sm.held[0][0])[threadIdx.x] = 0u;
  if (threadIdx.x < 8) (&sm.out_of_range[0][0])[threadIdx.x] = 0;
  if (threadIdx.x < sizeof(sm.ones) / 16) {
    // key threadIdx.x / 8: bf16 ones in every fourth column (all 16-byte pieces of a row are the same, wherever the swizzle puts them)
    const uint32_t one = threadIdx.x & 8 ? 0x3f800000u : 0x3f80u, low = threadIdx.x & 16 ? 0u : one, high = threadIdx.x & 16 ? one : 0u;
    reinterpret_cast<uint4*>(sm.ones)[threadIdx.x] = make_uint4(low, high, low, high);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tensor pipe reads them
  }
  // the next kernel of the stream may start its set-up while this grid drains; this grid's set-up ran while the
  // previous one drained.  Nothing an earlier kernel wrote is read before the wait below (the plan is older).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == 4) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const Item item0 = item_at(blockIdx.x);
  // The barriers and the TMEM address are shared here.  The first copies are on their way, and the softmax
  // warps' list and mask words looked up, before the CTA meets: a tile of a short list spends 3000 of its 20000 cycles on the
  // first copies (-2.5 to -5 % with the first reference).  With an 8-bit cache it meets first, which measured 1 % faster.
  auto meet = [&] {
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  };
  if constexpr (KV8) meet();

  bool exact = false;  // second pass over the lists: every tile's list twice, the rows' maxima first
  // Counters that go on from tile to tile and pass to pass, as the barriers' phases do: chunks before the current list, tiles, tiles
  // with a P V product.
  int base = 0, tiles = 0, o_tiles = 0;
  for (;;) {
    const int sweeps = uniform(exact ? 2 : 1), n_lists = n_tiles * sweeps;
    if (warp == 9) {
      // ---------------------------------------------------------------- copies of K and V.  The whole warp runs this code (what it
      // computes is uniform); one elected lane issues.  S(g) complete frees the stage of K(g) and, in issue order, that of
      // V(g - 2): K(g + 4) and V(g + 2) follow.
      int nk = base, nv = base;  // copies issued
      bool ok = true;
      if (!exact) asm volatile("griddepcontrol.wait;" ::: "memory");
      if constexpr (KV8) {
        // the copies bring codes and the rows' scales
        const int end = base + item0.n * sweeps;
        const int64_t row0 = (int64_t)item0.b * p.z_sb + (int64_t)item0.h * p.z_sh;
        const float *k_scale = p.k_scale + row0, *k_zero = p.k_zero + row0, *v_scale = p.v_scale + row0, *v_zero = p.v_zero + row0;
        auto row_of = [&](int g) {  // first cache row of chunk g
          const int j = min(g, end - 1) - base;
          return chunk_at(item0.chunks + (j >= item0.n ? j - item0.n : j)).row;
        };
        auto load_kc = [&](int row) {
          const int st = nk & 1, s = (nk >> 1) & 1;
          load_scales(sm.k_sz[st][s], k_scale, k_zero, row, p.L_k, lane, &sm.kc_full[st][s]);
          if (elect_one()) {
            mbar_expect_tx(&sm.kc_full[st][s], kCodeBytes);
            tma_load_4d(sm.kc[st][s], &tm.kr, 0, row, item0.h, item0.b, &sm.kc_full[st][s]);
          }
          ++nk;
        };
        auto load_vc = [&](int row) {
          const int st = nv & 1;
          load_scales(sm.v_sz[st], v_scale, v_zero, row, p.L_k, lane, &sm.vc_full[st]);
          if (elect_one()) {
            mbar_expect_tx(&sm.vc_full[st], kCodeBytes);
            tma_load_4d(sm.vc[st], &tm.vr, 0, row, item0.h, item0.b, &sm.vc_full[st]);
          }
          ++nv;
        };
        if (item0.n > 0) {
          int row[kStages];
#pragma unroll
          for (int i = 0; i < kStages; ++i) row[i] = row_of(base + i);
#pragma unroll
          for (int i = 0; i < kStages; ++i) {
            if (nk < end) load_kc(row[i]);
            if (i < 2 && nv < end) load_vc(row[i]);
          }
          // K(g) has been widened (behind P(g - 4)): its code buffer takes K(g + 4).  V(g) has (behind P(g - 2)): its buffer takes
          // V(g + 2).
          int k_row = row_of(nk), v_row = row_of(nv);  // looked up a step ahead
          for (int g = base; ok && (nk < end || nv < end); ++g) {
            if (nk < end && (ok = mbar_wait_idle(&sm.k_full[g % kStages], (uint32_t)((g / kStages) & 1), abort_flag, p.status))) {
              load_kc(k_row);
              k_row = row_of(nk);
            }
            if (ok && nv < end && (ok = mbar_wait_idle(&sm.vc_free[g & 1], (uint32_t)((g >> 1) & 1), abort_flag, p.status))) {
              load_vc(v_row);
              v_row = row_of(nv);
            }
          }
        }
      } else {
        // The copies run ahead of the products, into the CTA's next tile where the list ends: `at` is the tile of the next K copy,
        // c its chunk, number j of it.  V copies follow two behind.
        Item at = item0;
        int at_w = blockIdx.x, j = 0, again = sweeps - 1;
        bool more = true;
        ChunkAt c = {}, v0 = {}, v1 = {};  // of K(nk) and the two chunks in front of it
        auto settle = [&] {
          while (j >= at.n) {
            j = 0;
            if (again > 0) {
              --again;
              continue;
            }
            again = sweeps - 1;
            at_w += w_step;
            if (!MANY || at_w >= n_items) {
              more = false;
              return;
            }
            at = item_at(at_w);
          }
          const KeyChunk kc = chunk_at(at.chunks + j);
          c = ChunkAt{kc.row, kc.col, kc.info >> 16, at.h, at.b};
        };
        auto load_k = [&] {
          if (more) {
            const int s = nk % kStages;
            if (elect_one()) load_chunk(sm.k[s], &tm.kr, tm.k2, c, &sm.k_full[s]);
            ++nk;
          }
          v0 = v1;
          v1 = c;
          if (more) {
            ++j;
            settle();
          }
        };
        auto load_v = [&](const ChunkAt& at_v) {
          const int s = nv % kStages;
          if (elect_one()) load_chunk(sm.v[s], &tm.vr, tm.v2, at_v, &sm.v_full[s]);
          ++nv;
        };
        settle();
        for (int i = 0; i < kStages && more; ++i) {
          load_k();
          load_v(v1);
        }
        if (!exact) meet();
        for (int g = base; more || nv < nk; ++g) {
          ok = mbar_wait_idle(&sm.k_free[g % kStages], (uint32_t)((g / kStages) & 1), abort_flag, p.status);
          if (!ok) break;
          const ChunkAt at_v = v0;  // V(g + 2)
          load_k();
          if (g - base >= 2 && nv < nk) load_v(at_v);
          __syncwarp();
        }
      }
      base = nk;
      // Wait (bounded) for the last copies, whose wait in another warp may run out after this one is done.
      int polls = kPolls;
      auto landed = [&](uint64_t* bar, int phase) {
        while (!mbar_try(bar, (uint32_t)(phase & 1)) && --polls > 0) __nanosleep(kIdleNs);
      };
      if constexpr (KV8) {
        for (int i = nk > kStages ? nk - kStages : 0; i < nk; ++i) landed(&sm.kc_full[i & 1][(i >> 1) & 1], i >> 2);
        for (int i = nv > 2 ? nv - 2 : 0; i < nv; ++i) landed(&sm.vc_full[i & 1], i >> 1);
      } else {
        for (int i = nk > kStages ? nk - kStages : 0; i < nk; ++i) landed(&sm.k_full[i % kStages], i / kStages);
        for (int i = nv > kStages ? nv - kStages : 0; i < nv; ++i) landed(&sm.v_full[i % kStages], i / kStages);
      }
    } else if (warp == 8) {
      // ---------------------------------------------------------------- Q and the MMAs.  The whole warp runs this code (descriptors
      // stay in uniform registers); one elected lane issues.  P(g) complete is the event to wait for: O += P(g) V(g) and S(g + 2)
      // go out back to back (they execute in issue order, so that S may overwrite P).
      const uint64_t q_desc0 = make_desc(smem_u32(sm.q[0])), k_desc0 = make_desc(smem_u32(sm.k[0]));
      // V: 64 columns in the stage, the 16 behind them (leading byte offset) in the block of sm.ones
      const uint32_t ones_at = (smem_u32(sm.ones) - smem_u32(sm.v[0])) >> 4;
      const uint64_t v_desc0 = (make_desc(smem_u32(sm.v[0])) & ~(0x3fffull << 16)) | ((uint64_t)ones_at << 16);
      int nq = 0;  // Q copies issued in this pass
      // waits until the tile that had the buffer before has been stored (a pass starts with both buffers free)
      auto load_q = [&] {
        const int i = tiles + nq;
        bool free = true;
        if (MANY && nq >= kQBufs) free = mbar_wait_long(&sm.q_free, (uint32_t)((i - kQBufs) & 1), abort_flag, p.status);
        if (free) {
          int qt = item0.qt, qh = item0.h, qb = item0.b;
          if (MANY && nq > 0) {
            int unit;
            work_item(p, n_q_tiles, (int)blockIdx.x + nq * w_step, qt, unit);
            qh = unit % p.n_heads;
            qb = unit / p.n_heads;
          }
          if (elect_one()) {
            mbar_expect_tx(&sm.q_full[i % kQBufs], kTileBytes);
            load_q_tile(sm.q[i % kQBufs], tm, p, qt, qh, qb, &sm.q_full[i % kQBufs]);
          }
          ++nq;
        }
        return free;
      };
      if (!exact) asm volatile("griddepcontrol.wait;" ::: "memory");
      bool ok = load_q();
      if (MANY && ok && n_tiles > 1) ok = load_q();
      if (!KV8 && !exact) meet();
      const uint32_t tS = sm.tmem_base, tO = tS + kColO, tQ = tS + kColQ;
      int n = item0.n;
      for (int list = 0; list < n_lists; ++list) {
        const int x = exact ? list >> 1 : list, i_q = tiles + x;
        const bool maxima = exact && !(list & 1);
        int n_next = n;
        if (MANY && !maxima && x + 1 < n_tiles) n_next = uniform(item_at((int)blockIdx.x + (x + 1) * w_step).n);
        const int end = base + n;
        if (ok) ok = mbar_wait_long(&sm.q_full[i_q % kQBufs], (uint32_t)((i_q / kQBufs) & 1), abort_flag, p.status);
        // Q to TMEM (32 packed columns): a score product that reads both operands from shared memory waits for the 6 KB of a step.
        // Its last readers, the previous tile's score products, are complete: P(base - 1) was.
        if (ok && maxima == exact) {
          tc_fence_after();
          if (elect_one()) q_to_tmem(tQ, q_desc0 + (uint64_t)((kTileBytes >> 4) * (i_q % kQBufs)));
          __syncwarp();
        }
        for (int g = base - 2; g < end; ++g) {
          const int s = g % kStages, s2 = (g + 2) % kStages;
          if (ok && g + 2 < end) ok = mbar_wait_long(&sm.k_full[s2], (uint32_t)(((g + 2) / kStages) & 1), abort_flag, p.status);
          if (!KV8 && ok && g >= base) ok = mbar_wait_long(&sm.v_full[s], (uint32_t)((g / kStages) & 1), abort_flag, p.status);
          if (g >= base) {
            __syncwarp();
            asm volatile("bar.sync %0, 160;" ::"r"(5 + (g & 1)) : "memory");  // P(g); the softmax warps arrive even when a wait ran out
            *(volatile int*)&sm.met[g & 1] = g + 1;
          }
          if (ok) {
            tc_fence_after();
            if (g >= base && !maxima) {
              // 16 keys per step = 16 rows of 128 B = 2048 B of V (the block for the sums stays) and 8 packed columns of P
              const uint64_t stage = (uint64_t)((kChunkBytes >> 4) * s);
              mma_ts_x4_one<8, (2048 >> 4) - ((2048 >> 4) << 16)>(tO, tS + 64 * (g & 1), v_desc0 + stage - (stage << 16), kIdescO,
                                                                  g > base ? 1u : 0u);
              if (g + 1 == end) mma_commit_one(&sm.o_full);
            }
            if (g + 2 < end) {
              // 16 elements per step = 8 packed columns of Q and 32 B inside the swizzle rows of K
              mma_ts_x4_one<8, 2>(tS + 64 * (g & 1), tQ, k_desc0 + (uint64_t)((kChunkBytes >> 4) * s2), kIdescS, 0u);
              mma_commit_one(&sm.s_full[g & 1]);
              if (!KV8) mma_commit_one(&sm.k_free[s2]);
            }
            // The next tile's Q, once the tile before this one has left its buffer (the first two were copied at the start).  Both
            // streams' warps see to that behind their first chunk: a wait behind the first chunk of one held up the product of the
            // other (256px step 8 with 960 units 25.0 us, 24.2 behind the second).
            if (MANY && g > base && x > 0 && nq == x + 1 && nq < n_tiles) ok = load_q();
            __syncwarp();
          }
        }
        if (MANY && ok && x > 0 && nq == x + 1 && nq < n_tiles) ok = load_q();  // (less than two chunks)
        base = end;
        n = n_next;
      }
      if (*abort_flag) {
        const unsigned long long ts = global_ns();
        for (int i = nq > kQBufs ? nq - kQBufs : 0; i < nq; ++i)
          while (!mbar_try(&sm.q_full[(tiles + i) % kQBufs], (uint32_t)(((tiles + i) / kQBufs) & 1)))
            if (global_ns() - ts > kWaitLimitNs) break;
      }
      tiles += n_tiles;
    } else {
      // ---------------------------------------------------------------- softmax + epilogue.  Chunk g of the CTA belongs to stream g % 2.
      const int st = warp >> 2, lane_group = warp & 3;  // TMEM lanes 32 lane_group .. + 31
      const int m = lane_group * 32 + lane;
      const float sc = p.sm_scale * 1.4426950408889634f;
      const float2 sc2 = make_float2(sc, sc);
      const float sc_y = -sc / kClampSpan;
      int g = base + ((base ^ st) & 1);  // this stream's next chunk
      // Per chunk: class of its two halves for this warp's rows (bits 0 - 1 and 2 - 3: 0 dead, 1 partial, 2 full) and the key bits
      // of this thread's row, looked up one chunk ahead.
      int n = item0.n;
      const int2* infos = reinterpret_cast<const int2*>(&item0.chunks->info);  // {info, mask block} of chunk j at 2 j
      const uint2* mask_row = item0.mask + m;
      int cls = 0, cls_next = 0;
      auto look_up = [&](int j, int& c) {
        uint2 bits = make_uint2(0u, 0u);
        c = 0;
        if (j < n) {
          const int2 inf = __ldg(infos + 2 * j);
          c = (inf.x >> (4 * lane_group)) & 15;
          if (c & 5) bits = __ldg(mask_row + (size_t)inf.y * kBlockM);
          else bits = make_uint2((c & 3) ? ~0u : 0u, (c >> 2) ? ~0u : 0u);
        }
        return bits;
      };
      uint2 mk = look_up(g - base, cls), mk_next = look_up(g - base + 2, cls_next);
      bool bad = false, ok = true;
      if (!KV8 && !exact) meet();
      const uint32_t tlane = sm.tmem_base + ((uint32_t)(lane_group * 32) << 16), tS = tlane + 64 * st;
      // the previous tile's output rows have left their buffer, which the next copy but one (the second pass's next) goes to
      auto stored = [&] {
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          if (MANY) mbar_arrive(&sm.q_free);
        }
      };
      // 8-bit cache: the stream's softmax threads widen its chunks, V(g) before they hand P(g) over and K(g + 4) after it
      const int t = threadIdx.x & 127, pass_end = base + item0.n * sweeps, v_from = pass_end - item0.n;  // (maxima: no V)
      auto widen_k = [&](int i) {
        if constexpr (KV8) {
          if (ok && i < pass_end &&
              (ok = mbar_wait_long(&sm.kc_full[st][(i >> 1) & 1], (uint32_t)((i >> 2) & 1), abort_flag, p.status))) {
            widen_chunk(sm.kc[st][(i >> 1) & 1], sm.k_sz[st][(i >> 1) & 1], sm.k[i % kStages], t);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.k_full[i % kStages]);
          }
        }
      };
      auto widen_v = [&](int i) {
        if constexpr (KV8) {
          if (ok && i < pass_end && (ok = mbar_wait_long(&sm.vc_full[st], (uint32_t)((i >> 1) & 1), abort_flag, p.status))) {
            if (i >= v_from) widen_chunk(sm.vc[st], sm.v_sz[st], sm.v[i % kStages], t);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.vc_free[st]);
          }
        }
      };
      widen_k(g);
      widen_v(g);
      widen_k(g + 2);
      int qt = item0.qt, h = item0.h, b = item0.b;
      float msc = 0.f;      // probabilities are 2^(score * sc - msc)
      float top = 0.f;      // second pass: the row's maximum
      // S(i) complete; in issue order this also means that PV(i - 2) is complete
      auto wait_scores = [&](int i) {
        if (ok) ok = mbar_wait_long(&sm.s_full[st], (uint32_t)((i >> 1) & 1), abort_flag, p.status);
        if (ok) tc_fence_after();
      };
      auto load_scores = [&](int hf, uint32_t* r) {
        tmem_ld32(tS + 32 * hf, r);
        tmem_wait_ld();
        if ((cls >> (2 * hf)) & 1) {  // dead scores of a partially live half become -inf
          const uint32_t w = hf ? mk.y : mk.x;
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (!((w >> e) & 1u)) r[e] = 0xff800000u;
        }
      };
      // probabilities against the reference: scale and shift (packed FMAs), 2^x, bf16, over scores that have been read
      auto store_probabilities = [&](int hf, const uint32_t* r) {
        uint32_t pk[16];
        const float2 nm2 = make_float2(-msc, -msc);
        const float nm_y = fmaf(msc, 1.f / kClampSpan, kClampHigh / kClampSpan);
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const uint32_t* rr = r + e;
          const float2 xa = __ffma2_rn(make_float2(__uint_as_float(rr[0]), __uint_as_float(rr[1])), sc2, nm2);
          const float2 pa = make_float2(fast_exp2(xa.x), fast_exp2(xa.y));
          // some pairs on the FMA pipe: the exponential pipe (16 per clock and SM) is the tighter of the two
          float2 pb;
          if (on_fma_pipe<KV8, MANY>(e)) {
            pb = exp2_fma2(make_float2(__saturatef(fmaf(__uint_as_float(rr[2]), sc_y, nm_y)),
                                       __saturatef(fmaf(__uint_as_float(rr[3]), sc_y, nm_y))));
          } else {
            const float2 xb = __ffma2_rn(make_float2(__uint_as_float(rr[2]), __uint_as_float(rr[3])), sc2, nm2);
            pb = make_float2(fast_exp2(xb.x), fast_exp2(xb.y));
          }
          pk[(e >> 1) + 0] = pack_bf16(pa.x, pa.y);
          pk[(e >> 1) + 1] = pack_bf16(pb.x, pb.y);
        }
        tmem_st16(tS + 16 * hf, pk);
      };
      auto store_zeros = [&](int hf) {
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) pk[e] = 0u;
        tmem_st16(tS + 16 * hf, pk);
      };
      // The row's reference, from the stream with the tile's first chunk (`mx`: the maximum of its first 32 live scores) to the other.
      auto hand_over = [&](float mx) {
        if (g == base) {
          msc = mx != -INFINITY ? mx * sc : 0.f;
          if (n > 1) {
            sm.ref[m] = msc;
            asm volatile("bar.arrive %0, 64;" ::"r"(12 + lane_group) : "memory");
          }
        } else {
          asm volatile("bar.sync %0, 64;" ::"r"(12 + lane_group) : "memory");
          msc = sm.ref[m];
        }
      };
      // P(g) is complete, or of S(g) the maxima: the issuing warp is told, and this warp goes on to its next chunk.
      auto chunk_done = [&](int x, int end, bool first_list) {
        tc_fence_before();
        asm volatile("bar.arrive %0, 160;" ::"r"(5 + st) : "memory");
        if (MANY && x > 0 && g - base < 2 && first_list) stored();
        widen_v(g + 2);
        widen_k(g + 4);
        cls = cls_next;
        mk = mk_next;
        mk_next = look_up(g + 4 - base, cls_next);
        if (g + 2 < end) wait_scores(g + 2);
      };
      for (int list = 0; list < n_lists; ++list) {
        const int x = exact ? list >> 1 : list;
        const bool maxima = exact && !(list & 1);
        const int end = base + n;
        const bool idle = g >= end;
        if (maxima) top = -INFINITY;
        // The slots' first token or cell; a box that starts outside the grid holds no query.  The element is this thread's row.
        int r0 = qt * kBlockM + 32 * lane_group, c0 = 0;
        bool box_live = r0 < p.n_k, row_live = r0 + lane < p.n_k;
        if (p.q_patch) {
          const TileGeom geom = p.q_geom[qt];
          r0 = geom.a + patch_slot_row(32 * lane_group), c0 = geom.b + patch_slot_col(32 * lane_group);
          box_live = r0 < p.s_k && c0 < p.s_k;
          row_live = r0 + (lane >> 3) < p.s_k && c0 + (lane & 7) < p.s_k;
        }
        if (g < end) wait_scores(g);
        if (!exact && g < end) {  // the stream's first chunk, with the rows' references (the warps meet here whether a wait ran out or not)
          if (ok) {
            uint32_t r[32];
            if (cls & 3) {
              load_scores(0, r);
              hand_over(g == base ? largest_score(r) : 0.f);
              store_probabilities(0, r);
            } else {
              hand_over(-INFINITY);
              store_zeros(0);
            }
            if (cls >> 2) {
              load_scores(1, r);
              store_probabilities(1, r);
            } else {
              store_zeros(1);
            }
            tmem_wait_st();
            chunk_done(x, end, true);
            g += 2;
          } else {
            hand_over(-INFINITY);
          }
        }
        for (; g < end && ok; g += 2) {
          if (maxima) {  // second pass: the list once for the rows' maxima
#pragma unroll 1
            for (int hf = 0; hf < 2; ++hf)
              if ((cls >> (2 * hf)) & 3) {
                uint32_t r[32];
                load_scores(hf, r);
                top = fmaxf(top, largest_score(r));
              }
          } else {
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              if ((cls >> (2 * hf)) & 3) {
                uint32_t r[32];
                load_scores(hf, r);
                store_probabilities(hf, r);
              } else {  // no live key for any row of the warp
                store_zeros(hf);
              }
            }
            tmem_wait_st();
          }
          chunk_done(x, end, maxima);
        }
        // A wait ran out.  The issuing warp counts on every chunk's arrival, and the barrier on one of every warp at a time: S(g) says
        // that P(g - 2) has been met, and where no S is waited for any more the issuing warp's note does.
        for (; g < end; g += 2) {
          wait_met(&sm.met[st], g - 1);
          asm volatile("bar.arrive %0, 160;" ::"r"(5 + st) : "memory");
        }
        if (MANY && idle && x > 0 && maxima == exact) stored();
        const int n_here = n, h_here = h, b_here = b;
        base = end;
        if (list + 1 < n_lists) {  // the next list's first classes and masks start travelling
          if (MANY && !maxima) {
            const Item next = item_at((int)blockIdx.x + (x + 1) * w_step);
            n = next.n;
            qt = next.qt;
            h = next.h;
            b = next.b;
            infos = reinterpret_cast<const int2*>(&next.chunks->info);
            mask_row = next.mask + m;
          }
          mk = look_up(g - base, cls);
          mk_next = look_up(g - base + 2, cls_next);
        }
        if (maxima) {  // the two streams of a row agree on its maximum, the reference of the next sweep
          sm.top[st][m] = top;
          asm volatile("bar.sync %0, 64;" ::"r"(1 + lane_group) : "memory");
          top = fmaxf(top, sm.top[st ^ 1][m]);
          msc = top != -INFINITY ? top * sc : 0.f;
          asm volatile("bar.sync %0, 64;" ::"r"(8 + lane_group) : "memory");
          continue;
        }
        // the last PV product (all earlier ones are complete by issue order)
        if (n_here > 0) {
          if (ok) ok = mbar_wait_long(&sm.o_full, (uint32_t)(o_tiles & 1), abort_flag, p.status);
          ++o_tiles;
        }
        uint8_t* slice = sm.q[tiles % kQBufs] + (warp << 11);
        if (ok) {
          tc_fence_after();
          // Row sum: over P as the P V product sees it (rounded to bf16), so that numerator and denominator of a row agree, and a row
          // with one dominant key reproduces that key's V exactly.
          uint32_t r[32], sums[4];
          tmem_ld4(tlane + kColO + kHeadDim, sums);
          tmem_ld32(tlane + kColO + 32 * st, r);
          tmem_wait_ld();
          float l = (__uint_as_float(sums[0]) + __uint_as_float(sums[1])) + (__uint_as_float(sums[2]) + __uint_as_float(sums[3]));
          if (__builtin_expect(!exact && row_live && !(l < kRange && l > kRangeLow), 0)) {  // (a NaN goes this way too)
            bad = true;
            sm.out_of_range[lane_group][x & 1] = x + 1;
          }
          // Against exact maxima a sum is at most the number of keys: a larger one is a score of +inf or NaN.  A row whose maximum
          // is -inf has no finite score.
          if (exact && (!(l < kRange) || top == -INFINITY)) l = NAN;
          // Output columns [32 st, 32 st + 32) of this thread's row.
          // The warp's 32 rows x 64 B pass through its own 2 KB slice of the Q buffer (its last reader, the last score
          // product, is done: every warp has seen it through o_full) to a tensor-map store.  Piece position XOR
          // (row / 2) is the map's swizzle and keeps the writes free of bank conflicts.
          const float inv = 1.f / l;
          const float2 inv2 = make_float2(inv, inv);
          float largest = 0.f;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t o[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const float2 y = __fmul2_rn(make_float2(__uint_as_float(r[16 * c + e]), __uint_as_float(r[16 * c + e + 1])), inv2);
              o[e >> 1] = pack_bf16(y.x, y.y);
              asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(largest) : "f"(fabsf(y.x)), "f"(fabsf(y.y)));
            }
#pragma unroll
            for (int e = 0; e < 2; ++e)
              *reinterpret_cast<uint4*>(slice + lane * 64 + (((2 * c + e) ^ (lane >> 1)) & 3) * 16) =
                  make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
          }
          if (__builtin_expect(!exact && row_live && !(largest < INFINITY && (inv <= 1.f || largest > inv * kSmall)), 0)) {
            bad = true;
            sm.out_of_range[lane_group][x & 1] = x + 1;
          }
        }
        // the pair of warps agrees on what is out of range; the accumulator's rows have been read by both, so that the
        // next tile's may overwrite them
        tc_fence_before();
        asm volatile("bar.sync %0, 64;" ::"r"(8 + lane_group) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        // 32 rows one of which is out of range are not stored, and the second pass stores these rows only: every
        // row is stored once (two bulk stores to one address have no order), and a row of Q that the second pass reads has not been
        // overwritten where the output takes Q's place.
        if (ok && lane == 0) {
          bool store;
          if constexpr (MANY) {
            store = exact ? (sm.held[lane_group][x >> 5] >> (x & 31)) & 1u : *(volatile int*)&sm.out_of_range[lane_group][x & 1] != x + 1;
            if (!exact && !store && st == 0) {
              sm.held[lane_group][x >> 5] |= 1u << (x & 31);
            }
          } else {
            store = exact == (*(volatile int*)&sm.out_of_range[lane_group][0] != 0);
          }
          if (store && box_live) {
            for (int at = b_here;; at = b_here + p.share_offset) {
              if (p.q_patch) tma_store_5d(&tm.o, slice, 32 * st, c0, r0, h_here, at);
              else tma_store_4d(&tm.o, slice, 32 * st, r0, h_here, at);
              if (at != b_here || p.share_offset == 0) break;
            }
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        ++tiles;
      }
      stored();
      if (!exact && __any_sync(0xffffffffu, bad) && lane == 0) sm.redo = 1;
    }
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    tc_fence_after();
    if (uniform(exact || !*(volatile int*)&sm.redo || *abort_flag)) break;
    exact = true;
  }

  // ---------------------------------------------------------------------- teardown (all paths)
  if (*abort_flag) {  // products may be in flight, which read the stages and write TMEM
    if (warp == 8) {
      mma_commit_one(&sm.drained);
      for (int polls = kPolls; !mbar_try(&sm.drained, 0u) && --polls > 0;) __nanosleep(kIdleNs);
    }
    __syncthreads();
  }
  if (warp == 4) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem_base), "r"(kTmemCols) : "memory");
  }
}

template <bool KV8, bool MANY>
litevar_status_t launch_variant(const TensorMaps& tm, const FwdParams& p, int n_q_tiles, int n_ctas, cudaStream_t stream) {
  static std::once_flag attr_once;
  static cudaError_t attr_err = cudaSuccess;
  constexpr int smem_bytes = (int)sizeof(WsShared<KV8, MANY>);
  static_assert(smem_bytes <= 115712, "two CTAs per SM");
  std::call_once(attr_once, [] {
    attr_err = cudaFuncSetAttribute(fwd_ws_kernel<KV8, MANY>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  });
  if (attr_err != cudaSuccess) return LITEVAR_ERR_CUDA;
  const int n_items = n_q_tiles * p.n_heads * p.batch_computed;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(MANY ? n_ctas : n_items));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.overlap_launch ? 1 : 0;  // off when an earlier kernel of the stream writes what the set-up reads
  if (cudaLaunchKernelEx(&cfg, fwd_ws_kernel<KV8, MANY>, tm, p, n_q_tiles, n_items) != cudaSuccess) {
    (void)cudaGetLastError();
    return LITEVAR_ERR_CUDA;
  }
  return LITEVAR_OK;
}

}  // namespace

litevar_status_t launch_forward_ws(const FwdParams& p, int n_q_tiles, cudaStream_t stream) {
  TensorMaps tm;
  if (!encode_tensor_maps(p, &tm, kChunkKeys)) return LITEVAR_ERR_INVALID_ARG;
  // Short lists: a tile spends as long on its first copies, look-ups and output as on 4 to 6 chunks, and CTAs that stay overlap
  // these with the other tiles' work.  What is lost is the balance at the end: a CTA's tiles are fixed, not dealt out.  Measured
  // (thousand cycles, one tile per CTA / staying): 4 chunks at 3.2 tiles per resident CTA 56.2 / 50.6, 6 at 3.2 63.7 / 60.0, at 6.5
  // 113.7 / 100.5, 10 at 3.2 81.4 / 80.6, at 6.5 144.3 / 133.5, 8 at 2.9 60.8 / 60.9, at 5.8 117.1 / 113.1, at 1.5 38.2 / 38.9; 14
  // at 4.9 125.4 / 133.0, at 9.7 236.9 / 244.0; 22 at 7.8 267 / 291, at 15.6 523 / 544; patch tiles of a 48 x 48 step at 11.7 with
  // window 1/4, 1/8, 1/16: 571 / 670, 385 / 433, 304 / 330.  Sets of their own per head make no difference, the average over the
  // heads counts (us, the same step): all keys for one head in eight and 1/8 for the others 263 / 322, 1/4 and 1/8 262 / 313, 1/8 and
  // 1/16 189 / 215, 1/16 and 1/48 155 / 163.
  const long long items = (long long)n_q_tiles * p.n_heads * p.batch_computed, resident = 2ll * current_sm_count();
  const int chunks = p.chunks_per_tile;
  if (chunks > 0 && chunks <= 12 && 2 * items >= 5 * resident && 5 * items >= chunks * resident)
    return launch_variant<false, true>(tm, p, n_q_tiles, (int)std::max(resident, (items + kMaxTiles - 1) / kMaxTiles), stream);
  return launch_variant<false, false>(tm, p, n_q_tiles, 0, stream);
}

litevar_status_t launch_forward_ws_kv8(const FwdParams& p, int n_q_tiles, cudaStream_t stream) {
  TensorMaps tm;
  if (!encode_code_maps(p, &tm, kChunkKeys)) return LITEVAR_ERR_INVALID_ARG;
  return launch_variant<true, false>(tm, p, n_q_tiles, 0, stream);
}

}  // namespace litevar
