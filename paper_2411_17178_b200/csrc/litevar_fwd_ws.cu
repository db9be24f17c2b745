// Tensor-core forward kernel for sm_100a: a query tile per CTA at a time, two independent streams of key chunks.
//
// A CTA owns a query tile (128 queries) of one (head, batch row) and walks the live 64-key chunks of its list (laid by the planner
// over the tile's own live keys).  A chunk comes with the class of its two halves for every warp's 32 rows: dead halves are
// skipped, live ones take no element mask.  Two streams share the list, chunk i going to stream i % 2; each keeps its
// own scores, probabilities, accumulator and reference, and the two results meet at the end.  320 threads:
//   warps 0-3, 4-7  softmax of stream 0 and 1: thread m of the group owns query slot m (TMEM lane m).  A chunk's 64 scores
//                   come from TMEM in two halves of 32 through one rolled copy of the code: the plan's element mask, the
//                   probabilities (19 to 31 % of the exponentials, by build, on the FMA pipe by a cubic, the rest on the
//                   exponential pipe), their sum, and P (packed bf16) over the scores that have been read.
//   warps 8, 9      the stream's copies (K and V chunks by tensor-map copies into rings of two stages) and MMAs: once P(i) is
//                   complete, O += P(i) V(i) and S(i + 1) = Q K(i + 1) go out back to back; they execute in issue order, so
//                   that S may overwrite P.  The warp runs converged and what it computes is uniform, so that descriptors
//                   stay in uniform registers (a lane of its own: eight register moves per MMA); one elected lane issues.
// MANY: a CTA takes several tiles in turn.  Q has two buffers; K and V copies and the first score product of the next tile go out
// behind the last products of this one, the softmax warps look the next list up while they wait for their accumulator, and the
// output leaves by tensor-map stores that nobody waits for until the buffer's next use.  What orders the tiles: the first
// P V product of a tile (which overwrites the accumulator) follows the softmax warps' P, which they write after they and the
// warp with the other stream of their rows have read both accumulators; a Q copy follows the stores of the tile that had its buffer.
// Two CTAs per SM, so that every scheduler has four softmax warps of four streams that are in different phases.
// TMEM columns: S and P of stream s at 64 s, O at 128 + 64 s.
//
// The reference of a row (probabilities are 2^(score * scale - reference)) is the maximum of the first chunk's first eight keys
// and stays (0 where none of them is live): bf16 and fp32 have the same exponent range, so P and its sum are as accurate at 2^90 as
// at 1, and a tile's rows need neither a maximum per chunk nor a rescaled accumulator.  At the end a row whose sum or output is
// out of range (kRange, kSmall) sends the CTA through its lists again, with every chunk's maximum taken first (`exact`), for the 32
// rows of a warp that it belongs to, which are stored then.  The look at the output and the agreement of the two warps of a row on
// it take 1 % of the 2K step and 2 % of a launch with one tile per CTA (0.2 us).  (A reference that followed the chunk sums by powers
// of two from 2^10 on, tested at every chunk: 2 to 3 % slower, 512px step 10 155.6 us against 151.)
//
// What bounds it (ncu, 2K step, full mask / window 1/4): issue slots some 70 % busy, exponential pipe 60 / 50 %, tensor pipe active
// 44 / 41 %; 6.5 instructions a score.  The rest is the hand-off from P to the next S (arrive, issue of eight MMAs, their
// execution, commit, wake: 700 cycles a chunk), which the four streams of an SM cover for one another.
// Measured on B200, with what the kernel with one softmax thread per row and 128-key tiles took before: 2K step with the full
// mask 4.94 ms (6.71), window 1/4 1.48 ms (2.65), 512px steps 10 / 9 / 8 with 288 units 151 / 69 / 30 us (261 / 116 / 47),
// 256px step 10 with 960 units 75 us (117 on the kernel with two threads per row, which this one also replaces).  Steps on
// the way: copy look-ups off the MMA lane -4 %, 64-key streams with uniform issue code -12 %, no maxima -12 %; three stages instead of two: +1 %; chunks from
// a tile's live box on and classes per half and warp (on the fixed grid, one live flag per chunk and warp: 1.69 ms) -7 %.
//
// Every wait on an mbarrier is bounded; when one runs out the CTA raises the plan's status word, drains its copies, frees its
// TMEM and returns (the softmax warps still arrive for every chunk, so that the named barriers complete).  The element mask, the
// lists and CFG sharing (second store at batch row b + B) are those of the plan (paper Sections 2 and 3).
#include <algorithm>
#include <cstring>
#include <mutex>

#include "litevar_tc_ptx.h"

namespace litevar {

using namespace tc;

namespace {

constexpr float kRescaleThreshold = 8.f;  // log2 units: in the second pass the reference moves when a chunk exceeds it by more
constexpr int kChunkKeys = kBlockN / 2;
constexpr uint32_t kChunkBytes = kChunkKeys * kHeadDim * 2;
constexpr int kStages = 2;                // K ring and V ring of a stream
constexpr int kThreads = 320;             // two streams of four softmax warps, one issuing warp each
constexpr uint32_t kTmemCols = 256, kColO = 128;  // S (and P over it) of stream s at 64 s, O at 128 + 64 s

constexpr int kMaxTiles = 1024;  // of a CTA that takes several (MANY)
// A row sum of the first pass outside (2^-64, 2^96) goes to the second pass.  (The lower end keeps the traces of dead keys, 2^-125
// each, 2^-48 below a sum over any number of keys.)
constexpr float kRange = 79228162514264337593543950336.f, kRangeLow = 5.42101086242752217e-20f;
// So does a row of output that is not finite (sums of P V overflow before those of P), or so small beside its weight, where that is
// above 1, that products P V may have been subnormal (2^-126 each, 2^14 of them).
constexpr float kSmall = 7.88860905221011805e-31f;  // 2^-100

// 8-bit cache build: the codes of a chunk (64 rows of 64 bytes, as the tensor-map copy delivers them, no swizzle) and its rows'
// scales and shifted zero points, on their way into the bf16 stages (empty in the bf16 build).
constexpr uint32_t kCodeBytes = kChunkKeys * kHeadDim;
template <bool KV8>
struct CodeStage {};
template <>
struct CodeStage<true> {
  alignas(128) uint8_t kc[2][2][kCodeBytes];  // [stream][chunk % 2]
  alignas(128) uint8_t vc[2][kCodeBytes];
  float k_sz[2][2][2][kChunkKeys];  // [stream][chunk % 2][scale, shifted zero point][row]
  float v_sz[2][2][kChunkKeys];
  uint64_t kc_full[2][2], vc_full[2];
};

template <bool KV8, bool MANY>
struct WsShared : CodeStage<KV8> {
  alignas(1024) uint8_t q[MANY ? 2 : 1][kTileBytes];  // Q; at the end of a tile the output rows pass through it
  alignas(1024) uint8_t k[2][kStages][kChunkBytes];
  alignas(1024) uint8_t v[2][kStages][kChunkBytes];
  alignas(8) float2 ref[2][MANY ? kBlockM : 1];  // reference and row sum of each stream (one tile only: in its idle K stages)
  alignas(8) uint64_t q_full[2], q_free;
  uint64_t k_full[2][kStages], v_full[2][kStages];
  uint64_t s_full[2], o_full[2];
  uint32_t held[4][MANY ? kMaxTiles / 32 : 1];  // bit x: the 32 rows of the CTA's tile x are left to the second pass
  int out_of_range[4][2];  // 1 + the last even and odd tile with such rows (a warp is at most one tile ahead of its partner)
  uint32_t tmem_base;
  int abort_flag, redo;
};

// Instruction descriptors (kind::f16).  Fields: D type at bit 4 (1: fp32), A and B type at bits 7 and 10 (1: bf16), B transposed
// (MN-major, as V lies in shared memory) at bit 16, N / 8 at bit 17, M / 16 at bit 24.
constexpr uint32_t kIdescS = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kChunkKeys >> 3) << 17) |
                             ((uint32_t)(kBlockM >> 4) << 24);
constexpr uint32_t kIdescO = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(kHeadDim >> 3) << 17) |
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

// Which of a half's 16 pairs of exponentials take the FMA pipe (second pair of every four keys e .. e + 3): five with one tile per
// CTA, four on short lists with several, three beside the widening of an 8-bit cache, whose arithmetic is on that pipe too.
// Measured for 3 / 4 / 5 / 6 pairs: 2K step 14 1484 / 1488 / 1451 / 1494 us; 512px step 10 153.6 / 153.3 / 153.8 / 154.4 us; the same
// with an 8-bit cache 227.9 / 229.6 / 233.6 / 237 us.
template <bool KV8, bool MANY>
__device__ __forceinline__ constexpr bool on_fma_pipe(int e) {
  return KV8 ? (e & 4) != 0 && e != 28 : MANY ? (e & 4) != 0 : (e & 4) != 0 || e == 16;
}

// acc += the two bf16 halves of a packed pair: fp32 additions that take a bf16 operand as it is (no unpacking)
__device__ __forceinline__ void add_bf16_pair(float2& acc, uint32_t packed) {
  asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}"
      : "+f"(acc.x), "+f"(acc.y)
      : "r"(packed));
}

// One elected lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0u;
}
// mma_ts_x4 / mma_ss_x4 / mma_commit for a converged warp: one elected lane issues
template <int kAStep, int kBStep>
__device__ __forceinline__ void mma_ts_x4_one(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                              uint32_t accumulate_first) {
  if (elect_one()) mma_ts_x4<kAStep, kBStep>(d_tmem, a_tmem, b_desc, idesc, accumulate_first);
}
template <int kAStep, int kBStep>
__device__ __forceinline__ void mma_ss_x4_one(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                              uint32_t accumulate_first) {
  if (elect_one()) mma_ss_x4<kAStep, kBStep>(d_tmem, a_desc, b_desc, idesc, accumulate_first);
}
__device__ __forceinline__ void mma_commit_one(uint64_t* bar) {
  if (elect_one()) mma_commit(bar);
}
__device__ __forceinline__ KeyChunk chunk_at(const KeyChunk* c) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(c));
  return KeyChunk{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ void load_chunk(void* dst, const CUtensorMap* raster, const CUtensorMap* patch,
                                           const KeyChunk& c, int h, int b, uint64_t* bar) {
  mbar_expect_tx(bar, kChunkBytes);
  if (c.info >> 16)
    tma_load_5d(dst, patch + ((c.info >> 16) - 1), 0, c.col, c.row, h, b, bar);
  else
    tma_load_4d(dst, raster, 0, c.row, h, b, bar);
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
    widen_codes16(q, sz[0][m], sz[1][m], lo, hi);
    uint8_t* row = stage + m * 128;
    *reinterpret_cast<uint4*>(row + (((2 * c) ^ (m & 7)) << 4)) = lo;
    *reinterpret_cast<uint4*>(row + (((2 * c + 1) ^ (m & 7)) << 4)) = hi;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> the tensor pipe's reads
}

// Scales and zero points of a chunk's rows lane and lane + 32 (rows past L_k: 0 and 0; their codes arrive as zeros).
struct RowScales {
  float s[2], z[2];
};
__device__ __forceinline__ RowScales row_scales(const float* scale, const float* zero, int row, int L_k, int lane) {
  RowScales r;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int at = row + lane + 32 * i;
    r.s[i] = at < L_k ? __ldg(scale + at) : 0.f;
    r.z[i] = at < L_k ? __ldg(zero + at) : 0.f;
  }
  return r;
}
__device__ __forceinline__ void put_scales(float (&sz)[2][kChunkKeys], const RowScales& r, int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    sz[0][lane + 32 * i] = r.s[i];
    sz[1][lane + 32 * i] = shifted_zero_point(r.z[i], r.s[i]);
  }
}

template <bool KV8, bool MANY>
__global__ void __launch_bounds__(kThreads, 2)
fwd_ws_kernel(const __grid_constant__ TensorMaps tm, const __grid_constant__ FwdParams p, int n_q_tiles, int n_items) {
  static_assert(!(KV8 && MANY), "the code stages leave no room for a second Q buffer");
  constexpr int kQBufs = MANY ? 2 : 1;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  WsShared<KV8, MANY>& sm = *reinterpret_cast<WsShared<KV8, MANY>*>(smem_raw);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // warp-uniform
  const int st = warp < 8 ? warp >> 2 : warp - 8;  // stream
  // One query tile of one (head, batch row), in the grouped order of work_item, and this stream's share of its list.  A CTA
  // takes items blockIdx.x, blockIdx.x + gridDim.x, ... (MANY; else one).
  struct Item {
    int qt, h, b, n_all, n;  // n: this stream's chunks st, st + 2, ...
    const KeyChunk* chunks;  // the first of them
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
    x.n_all = __ldg(&sd.chunk_ptr[x.qt + 1]) - first;
    x.n = (x.n_all - st + 1) >> 1;
    x.chunks = sd.chunks + first + st;
    x.mask = sd.chunk_mask;
    return x;
  };
  const int w_step = MANY ? (int)gridDim.x : n_items;
  volatile int* abort_flag = &sm.abort_flag;

  if (warp >= 8 && elect_one()) {  // each issuing warp sets up its own stream's barriers
    if (st == 0) {
      mbar_init(&sm.q_full[0], 1);
      mbar_init(&sm.q_full[1], 1);
      mbar_init(&sm.q_free, 8);  // every softmax warp arrives when the tile's output rows have left the buffer
      sm.abort_flag = 0;
      sm.redo = 0;
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.k_full[st][s], KV8 ? 4 : 1);  // 8-bit cache: every softmax warp of the stream arrives
      mbar_init(&sm.v_full[st][s], KV8 ? 4 : 1);
    }
    if constexpr (KV8) {
      mbar_init(&sm.kc_full[st][0], 1);
      mbar_init(&sm.kc_full[st][1], 1);
      mbar_init(&sm.vc_full[st], 1);
    }
    mbar_init(&sm.s_full[st], 1);
    mbar_init(&sm.o_full[st], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (threadIdx.x < 4 * (sizeof(sm.held[0]) / sizeof(uint32_t))) (&sm.held[0][0])[threadIdx.x] = 0u;
  if (threadIdx.x < 8) (&sm.out_of_range[0][0])[threadIdx.x] = 0;
  // the next kernel of the stream may start its set-up while this grid drains; this grid's set-up ran while the
  // previous one drained.  Nothing an earlier kernel wrote is read before the wait below (the plan is older).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == 9) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const Item item0 = item_at(blockIdx.x);
  // The barriers and the TMEM address are shared here.  The issuing warps' first copies are on their way, and the softmax
  // warps' list and mask words looked up, before the CTA meets: a tile of a short list spends 3000 of its 20000 cycles on the
  // first copies (-2.5 to -5 % with the first reference).  With an 8-bit cache it meets first, which measured 1 % faster.
  auto meet = [&] {
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  };
  if constexpr (KV8) meet();

  bool exact = false;  // second pass over the lists, every chunk's maximum taken before its probabilities
  // Counters that go on from tile to tile and pass to pass, as the barriers' phases do: this stream's chunks (`base`: before the
  // current tile), tiles, tiles in which this stream has a chunk.
  int base = 0, tiles = 0, o_tiles = 0;
  for (;;) {
    if (warp >= 8) {
      // ---------------------------------------------------------------- copies and MMAs of the stream.  The whole warp runs
      // this code (what it computes is uniform, so that descriptors and coordinates live in uniform registers); one
      // elected lane issues.  P(i) complete is the event to wait for: PV(i) and S(i + 1) are issued back to back (they
      // execute in issue order, so that S may overwrite P).
      const uint64_t q_desc0 = make_desc(smem_u32(sm.q[0])), k_desc0 = make_desc(smem_u32(sm.k[st][0]));
      const uint64_t v_desc0 = make_desc(smem_u32(sm.v[st][0]));
      // The copies run ahead of the products, into the CTA's next tile where the list ends: `at` is the tile of the next K copy,
      // c_k its chunk, number j of it; V copies follow one step behind (c_v, of head and batch row h_v, b_v).
      Item at = item0;
      int at_w = blockIdx.x, j = 0;
      KeyChunk c_k = {}, c_v = {};
      int h_v = at.h, b_v = at.b;
      int nk = base, nv = base;     // copies issued
      auto settle = [&] {
        while (j >= at.n) {
          if (!MANY) {
            at_w = n_items;
            return;
          }
          at_w += w_step;
          if (at_w >= n_items) return;
          at = item_at(at_w);
          j = 0;
        }
        c_k = chunk_at(at.chunks + 2 * j);
      };
      auto load_k = [&] {
        if (elect_one()) load_chunk(sm.k[st][nk % kStages], &tm.kr, tm.k2, c_k, at.h, at.b, &sm.k_full[st][nk % kStages]);
        ++nk;
        c_v = c_k;
        h_v = at.h;
        b_v = at.b;
        ++j;
        settle();
      };
      auto load_v = [&] {
        if (elect_one()) load_chunk(sm.v[st][nv % kStages], &tm.vr, tm.v2, c_v, h_v, b_v, &sm.v_full[st][nv % kStages]);
        ++nv;
      };
      auto chunk = [&](int i) { return chunk_at(item0.chunks + 2 * min(i, item0.n - 1)); };  // 8-bit cache (one tile)
      int nq = tiles;  // Q copies issued (stream 0)
      const int q_pass = nq;
      // waits until the tile that had the buffer before has been stored (a pass starts with both buffers free)
      auto load_q = [&](int w) {
        bool free = true;
        if (MANY && nq - q_pass >= kQBufs) free = mbar_wait_long(&sm.q_free, (uint32_t)((nq - kQBufs) & 1), abort_flag, p.status);
        if (free) {
          int qt = item0.qt, qh = item0.h, qb = item0.b;
          if (MANY && w != (int)blockIdx.x) {
            int unit;
            work_item(p, n_q_tiles, w, qt, unit);
            qh = unit % p.n_heads;
            qb = unit / p.n_heads;
          }
          if (elect_one()) {
            mbar_expect_tx(&sm.q_full[nq % kQBufs], kTileBytes);
            load_q_tile(sm.q[nq % kQBufs], tm, p, qt, qh, qb, &sm.q_full[nq % kQBufs]);
          }
          ++nq;
        }
        return free;
      };
      // 8-bit cache: the copies bring codes, and the warp puts the rows' scales beside them (looked up a step ahead)
      RowScales rs_k = {}, rs_v = {};
      const float* scales[4] = {};
      if constexpr (KV8) {
        const int64_t row0 = (int64_t)item0.b * p.z_sb + (int64_t)item0.h * p.z_sh;
        scales[0] = p.k_scale + row0;
        scales[1] = p.k_zero + row0;
        scales[2] = p.v_scale + row0;
        scales[3] = p.v_zero + row0;
      }
      auto load_kc = [&](const KeyChunk& c) {
        if constexpr (KV8) {
          const int s = nk & 1;
          put_scales(sm.k_sz[st][s], rs_k, lane);
          __syncwarp();
          if (elect_one()) {
            mbar_expect_tx(&sm.kc_full[st][s], kCodeBytes);
            tma_load_4d(sm.kc[st][s], &tm.kr, 0, c.row, item0.h, item0.b, &sm.kc_full[st][s]);
          }
          ++nk;
        }
      };
      auto load_vc = [&](const KeyChunk& c) {
        if constexpr (KV8) {
          put_scales(sm.v_sz[st], rs_v, lane);
          __syncwarp();
          if (elect_one()) {
            mbar_expect_tx(&sm.vc_full[st], kCodeBytes);
            tma_load_4d(sm.vc[st], &tm.vr, 0, c.row, item0.h, item0.b, &sm.vc_full[st]);
          }
          ++nv;
        }
      };
      if (!exact) asm volatile("griddepcontrol.wait;" ::: "memory");
      bool ok = true;
      if (st == 0) ok = load_q(blockIdx.x);
      if constexpr (KV8) {
        if (item0.n > 0) {
          c_k = chunk(0);
          c_v = chunk(1);
          rs_k = row_scales(scales[0], scales[1], c_k.row, p.L_k, lane);
          rs_v = row_scales(scales[2], scales[3], c_k.row, p.L_k, lane);
          const RowScales rs_k1 = row_scales(scales[0], scales[1], c_v.row, p.L_k, lane);
          load_kc(c_k);
          load_vc(c_k);
          rs_k = rs_k1;
          if (item0.n > 1) load_kc(c_v);
          c_k = chunk(2);
          rs_k = row_scales(scales[0], scales[1], c_k.row, p.L_k, lane);
          rs_v = row_scales(scales[2], scales[3], c_v.row, p.L_k, lane);
        }
      } else {
        settle();
        for (int i = 0; i < kStages && at_w < n_items; ++i) {
          load_k();
          load_v();
        }
      }
      if (MANY && st == 0 && ok && blockIdx.x + w_step < n_items) ok = load_q(blockIdx.x + w_step);
      if (!KV8 && !exact) meet();
      const uint32_t tS = sm.tmem_base + 64 * st, tO = tS + kColO;
      int n = item0.n;
      for (int w = blockIdx.x, x = 0;; w += w_step, ++x) {
        int n_next = 0;
        if (MANY && w + w_step < n_items) n_next = item_at(w + w_step).n;
        const int end = base + n;
        if (ok) ok = mbar_wait_long(&sm.q_full[tiles % kQBufs], (uint32_t)((tiles / kQBufs) & 1), abort_flag, p.status);
        const uint64_t q_desc = q_desc0 + (uint64_t)((kTileBytes >> 4) * (tiles % kQBufs));
        for (int i = base - 1; i < end && n > 0; ++i) {
          const int s = i % kStages, s1 = (i + 1) % kStages;
          if (ok && i + 1 < end) ok = mbar_wait_long(&sm.k_full[st][s1], (uint32_t)(((i + 1) / kStages) & 1), abort_flag, p.status);
          if (i >= base && ok) ok = mbar_wait_long(&sm.v_full[st][s], (uint32_t)((i / kStages) & 1), abort_flag, p.status);
          if constexpr (KV8) {  // K(i + 1) and V(i) are widened: their code buffers take K(i + 3) and V(i + 1)
            if (ok) {
              const KeyChunk c = c_k;
              if (i >= base && nv < end) {
                load_vc(c_v);
                c_v = chunk(nv - base);
                rs_v = row_scales(scales[2], scales[3], c_v.row, p.L_k, lane);
              }
              if (nk < end) {
                load_kc(c);
                c_k = chunk(nk - base);
                rs_k = row_scales(scales[0], scales[1], c_k.row, p.L_k, lane);
              }
            }
          }
          if (i >= base) {
            __syncwarp();
            asm volatile("bar.sync %0, 160;" ::"r"(5 + st) : "memory");  // P(i); the softmax warps arrive even when a wait ran out
          }
          if (ok) {
            tc_fence_after();
            if (i >= base) {
              // 16 keys per step = 16 rows of 128 B = 2048 B of V and 8 packed columns of P
              mma_ts_x4_one<8, (2048 >> 4)>(tO, tS, v_desc0 + (uint64_t)((kChunkBytes >> 4) * s), kIdescO, i > base ? 1u : 0u);
            }
            if (i + 1 < end) {
              // 16 bf16 = 32 B per step inside the swizzle rows of Q and K
              mma_ss_x4_one<2, 2>(tS, q_desc, k_desc0 + (uint64_t)((kChunkBytes >> 4) * s1), kIdescS, 0u);
              mma_commit_one(&sm.s_full[st]);
            } else {
              mma_commit_one(&sm.o_full[st]);
            }
            // P(i) was complete, so S(i) and PV(i - 1) are: K(i + stages) and V(i - 1 + stages) go where K(i) and V(i - 1) were
            if constexpr (!KV8) {
              if (i >= base) {
                if (nv < nk) load_v();
                if (at_w < n_items) load_k();
              }
            }
            // the next tile's Q, once the tile before this one has left its buffer (the first two were copied at the start)
            if (MANY && st == 0 && i == base && x > 0 && w + w_step < n_items) ok = load_q(w + w_step);
            __syncwarp();
          }
        }
        base = end;
        n = n_next;
        ++tiles;
        if (!MANY || w + w_step >= n_items) break;
      }
      if (*abort_flag) {  // wait (bounded) for copies still in flight before the CTA may exit
        const unsigned long long ts = global_ns();
        for (int i = nq > kQBufs ? nq - kQBufs : 0; st == 0 && i < nq; ++i)
          while (!mbar_try(&sm.q_full[i % kQBufs], (uint32_t)((i / kQBufs) & 1)))
            if (global_ns() - ts > kWaitLimitNs) break;
        if constexpr (KV8) {
          for (int i = nk > 2 ? nk - 2 : 0; i < nk; ++i)
            while (!mbar_try(&sm.kc_full[st][i & 1], (uint32_t)((i >> 1) & 1)))
              if (global_ns() - ts > 2 * kWaitLimitNs) break;
          while (nv > 0 && !mbar_try(&sm.vc_full[st], (uint32_t)((nv - 1) & 1)))
            if (global_ns() - ts > 2 * kWaitLimitNs) break;
        } else {
          for (int i = nk > kStages ? nk - kStages : 0; i < nk; ++i)
            while (!mbar_try(&sm.k_full[st][i % kStages], (uint32_t)((i / kStages) & 1)))
              if (global_ns() - ts > 2 * kWaitLimitNs) break;
          for (int i = nv > kStages ? nv - kStages : 0; i < nv; ++i)
            while (!mbar_try(&sm.v_full[st][i % kStages], (uint32_t)((i / kStages) & 1)))
              if (global_ns() - ts > 2 * kWaitLimitNs) break;
        }
      }
    } else {
      // ---------------------------------------------------------------- softmax + epilogue
      const int lane_group = warp & 3;  // TMEM lanes 32 lane_group .. + 31
      const int m = lane_group * 32 + lane;
      const float sc = p.sm_scale * 1.4426950408889634f;
      const float2 sc2 = make_float2(sc, sc);
      const float sc_y = -sc / kClampSpan;
      // Per chunk: class of its two halves for this warp's rows (bits 0 - 1 and 2 - 3: 0 dead, 1 partial, 2 full) and the key bits
      // of this thread's row, looked up one chunk ahead.
      int n = item0.n, n_all = item0.n_all;
      const int2* infos = reinterpret_cast<const int2*>(&item0.chunks->info);  // {info, mask block}, every second chunk is this stream's
      const uint2* mask_row = item0.mask + m;
      int cls = 0, cls_next = 0;
      auto look_up = [&](int j, int& c) {
        uint2 bits = make_uint2(0u, 0u);
        c = 0;
        if (j < n) {
          const int2 inf = __ldg(infos + 4 * j);
          c = (inf.x >> (4 * lane_group)) & 15;
          if (c & 5) bits = __ldg(mask_row + (size_t)inf.y * kBlockM);
          else bits = make_uint2((c & 3) ? ~0u : 0u, (c >> 2) ? ~0u : 0u);
        }
        return bits;
      };
      uint2 mk = look_up(0, cls), mk_next = look_up(1, cls_next);
      bool bad = false, ok = true;
      if (!KV8 && !exact) meet();
      const uint32_t tlane = sm.tmem_base + ((uint32_t)(lane_group * 32) << 16);
      const uint32_t tS = tlane + 64 * st, tO = tlane + kColO + 64 * st;
      // the previous tile's output rows have left their buffer, which the next copy but one (the second pass's next) goes to
      auto stored = [&] {
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          if (MANY) mbar_arrive(&sm.q_free);
        }
      };
      for (int w = blockIdx.x, x = 0;; w += w_step, ++x) {
        const int end = base + n;
        // probabilities are 2^(score * sc - msc); `none` until msc has been set from a live key
        float msc = 0.f;
        bool none = true;
        float2 l2a = make_float2(0.f, 0.f), l2b = make_float2(0.f, 0.f);  // row sum
        uint32_t seen = 0u;  // not 0: this row has had a live key
        // 8-bit cache: the stream's softmax threads widen its chunks, K(i + 2) and V(i + 1) while the products after P(i) run
        const int t = threadIdx.x & 127;
        auto widen_k = [&](int i) {
          if constexpr (KV8) {
            if (ok && i < end && (ok = mbar_wait_long(&sm.kc_full[st][i & 1], (uint32_t)((i >> 1) & 1), abort_flag, p.status))) {
              widen_chunk(sm.kc[st][i & 1], sm.k_sz[st][i & 1], sm.k[st][i % kStages], t);
              __syncwarp();
              if (lane == 0) mbar_arrive(&sm.k_full[st][i % kStages]);
            }
          }
        };
        auto widen_v = [&](int i) {
          if constexpr (KV8) {
            if (ok && i < end && (ok = mbar_wait_long(&sm.vc_full[st], (uint32_t)(i & 1), abort_flag, p.status))) {
              widen_chunk(sm.vc[st], sm.v_sz[st], sm.v[st][i % kStages], t);
              __syncwarp();
              if (lane == 0) mbar_arrive(&sm.v_full[st][i % kStages]);
            }
          }
        };
        widen_k(base);
        widen_v(base);
        widen_k(base + 1);
        for (int j = 0; j < n; ++j) {
          // S(j) complete; in issue order this also means that PV(j - 1) is complete
          if (ok) ok = mbar_wait_long(&sm.s_full[st], (uint32_t)((base + j) & 1), abort_flag, p.status);
          if (!ok) {  // the issuing warp counts on every step's arrival
            asm volatile("bar.arrive %0, 160;" ::"r"(5 + st) : "memory");
            continue;
          }
          tc_fence_after();
          if (j == 0 || exact) {  // a reference first: the chunk's maximum, or in the first pass that of its first eight keys
            float mx = -INFINITY;
            if (cls && !exact) {
              uint32_t r[8];
              tmem_ld8(tS, r);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 8; ++e) mx = fmaxf(mx, (mk.x >> e) & 1u ? __uint_as_float(r[e]) : -INFINITY);
            } else if (cls) {
#pragma unroll 1
              for (int hf = 0; hf < 2; ++hf) {
                const uint32_t w = hf ? mk.y : mk.x;
                uint32_t r[32];
                tmem_ld32(tS + 32 * hf, r);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) mx = fmaxf(mx, (w >> e) & 1u ? __uint_as_float(r[e]) : -INFINITY);
              }
            }
            float alpha = 1.f;
            if (mx != -INFINITY && (none || mx * sc - msc > kRescaleThreshold)) {
              if (!none) {
                alpha = fast_exp2(msc - mx * sc);
                l2a.x *= alpha; l2a.y *= alpha; l2b.x *= alpha; l2b.y *= alpha;
              }
              msc = mx * sc;
              none = false;
            }
            if (exact && __any_sync(0xffffffffu, alpha != 1.f)) {  // the accumulator follows the reference
#pragma unroll 1
              for (int c = 0; c < 4; ++c) {
                uint32_t o[16];
                tmem_ld16(tO + 16 * c, o);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                tmem_st16(tO + 16 * c, o);
              }
            }
          }
#pragma unroll 1
          for (int hf = 0; hf < 2; ++hf) {
            if ((cls >> (2 * hf)) & 3) {
              uint32_t r[32], pk[16];
              tmem_ld32(tS + 32 * hf, r);
              tmem_wait_ld();
              if ((cls >> (2 * hf)) & 1) {  // dead scores of a partially live half become -inf
                const uint32_t w = hf ? mk.y : mk.x;
#pragma unroll
                for (int e = 0; e < 32; ++e)
                  if (!((w >> e) & 1u)) r[e] = 0xff800000u;
              }
              // probabilities against the reference: scale and shift (packed FMAs), 2^x, row sum, bf16
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
                // the row sum adds the probabilities as the PV product sees them (rounded to bf16): numerator and
                // denominator of a row then agree, and a row with one dominant key reproduces that key's V exactly
                const uint32_t ka = pack_bf16(pa.x, pa.y), kb = pack_bf16(pb.x, pb.y);
                add_bf16_pair(l2a, ka);
                add_bf16_pair(l2b, kb);
                pk[(e >> 1) + 0] = ka;
                pk[(e >> 1) + 1] = kb;
              }
              tmem_st16(tS + 16 * hf, pk);  // over scores that have been read
            } else {  // no live key for any row of the warp
              uint32_t pk[16];
#pragma unroll
              for (int e = 0; e < 16; ++e) pk[e] = 0u;
              tmem_st16(tS + 16 * hf, pk);
            }
          }
          tmem_wait_st();  // P and, where it was rescaled, the accumulator
          tc_fence_before();
          asm volatile("bar.arrive %0, 160;" ::"r"(5 + st) : "memory");
          if (MANY && j == 0 && w != (int)blockIdx.x) stored();
          seen |= mk.x | mk.y;
          widen_v(base + j + 1);
          widen_k(base + j + 2);
          cls = cls_next;
          mk = mk_next;
          mk_next = look_up(j + 2, cls_next);
        }
        const int n_here = n;
        const bool both = n_all > 1;  // stream 1 has a chunk
        if (MANY && n == 0 && w != (int)blockIdx.x) stored();
        if (MANY && w + w_step < n_items) {  // the next tile's list and masks start travelling
          const Item next = item_at(w + w_step);
          n = next.n;
          n_all = next.n_all;
          infos = reinterpret_cast<const int2*>(&next.chunks->info);
          mask_row = next.mask + m;
          mk = look_up(0, cls);
          mk_next = look_up(1, cls_next);
        }
        // the last PV product (all earlier ones are complete by issue order)
        if (n_here > 0) {
          if (ok) ok = mbar_wait_long(&sm.o_full[st], (uint32_t)(o_tiles & 1), abort_flag, p.status);
          ++o_tiles;
        }
        float l = (l2a.x + l2a.y) + (l2b.x + l2b.y);
        if (__builtin_expect(!exact && seen && !(l < kRange && l > kRangeLow), 0)) {  // (a NaN goes this way too)
          bad = true;
          sm.out_of_range[lane_group][x & 1] = x + 1;
        }
        // Against exact maxima a sum is at most 2^8 times the number of keys: a larger one is a score of +inf or NaN.
        if (exact && seen && !(l < kRange)) l = NAN;
        // (dead keys leave traces of 2^-125 in l; in the second pass a stream without a reference has scores of -inf only)
        const float own = seen && !(exact && none) ? msc : -INFINITY;
        float2* const ref_own = MANY ? sm.ref[st] : reinterpret_cast<float2*>(sm.k[st][0]);
        const float2* const ref_other = MANY ? sm.ref[st ^ 1] : reinterpret_cast<const float2*>(sm.k[st ^ 1][0]);
        ref_own[m] = make_float2(own, l);
        tc_fence_before();
        asm volatile("bar.sync %0, 64;" ::"r"(1 + lane_group) : "memory");  // the warp with the other stream of these rows
        tc_fence_after();
        uint8_t* slice = sm.q[tiles % kQBufs] + (warp << 11);
        if (ok) {
          // Weights against the larger of the two masses 2^reference * sum.  (Against the larger reference they are wrong: a stream
          // without a live key among its first eight has reference 0, however far below the other's mass its own lies.)
          const float2 other = ref_other[m];
          const float top = fmaxf(own + fast_log2(l), other.x + fast_log2(other.y));
          const float f_own = fast_exp2(own - top), f_other = fast_exp2(other.x - top);
          const float inv = 1.f / (l * f_own + other.y * f_other);
          const float w0 = (st ? f_other : f_own) * inv, w1 = (st ? f_own : f_other) * inv;
          // output columns [32 st, 32 st + 32) of this thread's row: both streams' accumulators, weighted (stream 1's
          // may never have been written).
          // The warp's 32 rows x 64 B pass through its own 2 KB slice of the Q buffer (its last reader, the last score
          // product, is done: every warp of both streams has seen it through o_full) to a tensor-map store.  Piece position XOR
          // (row / 2) is the map's swizzle and keeps the writes free of bank conflicts.
          float largest = 0.f;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t r[16], r1[16];
            tmem_ld16(tlane + kColO + 32 * st + 16 * c, r);
            tmem_ld16(tlane + kColO + 64 + 32 * st + 16 * c, r1);
            tmem_wait_ld();
            uint32_t o[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              float2 x = make_float2(__uint_as_float(r[e]) * w0, __uint_as_float(r[e + 1]) * w0);
              if (both) x = __ffma2_rn(make_float2(__uint_as_float(r1[e]), __uint_as_float(r1[e + 1])), make_float2(w1, w1), x);
              o[e >> 1] = pack_bf16(x.x, x.y);
              asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(largest) : "f"(fabsf(x.x)), "f"(fabsf(x.y)));
            }
#pragma unroll
            for (int e = 0; e < 2; ++e)
              *reinterpret_cast<uint4*>(slice + lane * 64 + (((2 * c + e) ^ (lane >> 1)) & 3) * 16) =
                  make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
          }
          const float weight = fmaxf(w0, w1);
          if (__builtin_expect(!exact && top > -INFINITY && !(largest < INFINITY && (weight <= 1.f || largest > weight * kSmall)), 0)) {
            bad = true;
            sm.out_of_range[lane_group][x & 1] = x + 1;
          }
        }
        // the pair of warps agrees on what is out of range; both streams' accumulators of these rows have been read, so that the
        // next tile's may overwrite them
        tc_fence_before();
        asm volatile("bar.sync %0, 64;" ::"r"(7 + lane_group) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        // 32 rows one of which is out of range in either stream are not stored, and the second pass stores these rows only: every
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
          int qt = item0.qt, h = item0.h, b = item0.b;
          if constexpr (MANY) {
            int unit;
            work_item(p, n_q_tiles, w, qt, unit);
            h = unit % p.n_heads;
            b = unit / p.n_heads;
          }
          // the slots' first token or cell; a box that starts outside the grid holds no query
          const int bs = b + p.share_offset;
          if (p.q_patch) {
            const TileGeom g = p.q_geom[qt];
            const int r0 = g.a + patch_slot_row(32 * lane_group), c0 = g.b + patch_slot_col(32 * lane_group);
            if (store && r0 < p.s_k && c0 < p.s_k) {
              tma_store_5d(&tm.o, slice, 32 * st, c0, r0, h, b);
              if (p.share_offset > 0) tma_store_5d(&tm.o, slice, 32 * st, c0, r0, h, bs);
            }
          } else {
            const int q0 = qt * kBlockM + 32 * lane_group;
            if (store && q0 < p.n_k) {
              tma_store_4d(&tm.o, slice, 32 * st, q0, h, b);
              if (p.share_offset > 0) tma_store_4d(&tm.o, slice, 32 * st, q0, h, bs);
            }
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        base = end;
        ++tiles;
        if (!MANY || w + w_step >= n_items) break;
      }
      stored();
      if (!exact && __any_sync(0xffffffffu, bad) && lane == 0) sm.redo = 1;
    }
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    tc_fence_after();
    if (exact || !*(volatile int*)&sm.redo || *abort_flag) break;
    exact = true;
  }

  // ---------------------------------------------------------------------- teardown (all paths)
  if (warp == 9) {
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
  // (us, one tile per CTA / staying): 10 chunks a tile at 6.5 tiles per resident CTA 83.4 / 75.3, at 2.6 37.6 / 36.9, at 1.7
  // 25.2 / 25.7; 4 chunks at 3.2 29.0 / 24.7, at 1.6 15.3 / 15.9; 14 chunks at 4.9 73.0 / 70.2, at 2.4 39.4 / 40.0; 22 chunks
  // at 7.8 157.3 / 155.5, at 2.9 63.6 / 65.0; 38 chunks at 1.9 66.6 / 73.4; 53 at 3.5 172 / 182; 155 at 13.8 1520 / 1680.
  const long long items = (long long)n_q_tiles * p.n_heads * p.batch_computed, resident = 2ll * current_sm_count();
  const int chunks = p.chunks_per_tile;
  if (chunks > 0 && chunks <= 40 && 2 * items >= 5 * resident && 5 * items >= chunks * resident)
    return launch_variant<false, true>(tm, p, n_q_tiles, (int)std::max(resident, (items + kMaxTiles - 1) / kMaxTiles), stream);
  return launch_variant<false, false>(tm, p, n_q_tiles, 0, stream);
}

litevar_status_t launch_forward_ws_kv8(const FwdParams& p, int n_q_tiles, cudaStream_t stream) {
  TensorMaps tm;
  if (!encode_code_maps(p, &tm, kChunkKeys)) return LITEVAR_ERR_INVALID_ARG;
  return launch_variant<true, false>(tm, p, n_q_tiles, 0, stream);
}

}  // namespace litevar
