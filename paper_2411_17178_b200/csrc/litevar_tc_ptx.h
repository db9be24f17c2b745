// Device-side building blocks of the tensor-core forward kernels (sm_100a): mbarrier, TMA, tcgen05 and TMEM
// wrappers in inline PTX, the shared-memory descriptor, the tensor maps of one launch and the order of its work
// items.  Included by the tensor-core forward kernel and the host code that encodes its maps.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "litevar_internal.h"

namespace litevar {
namespace tc {

constexpr uint32_t kTileBytes = kBlockN * kHeadDim * 2;  // 16 KB: 128 rows of 128 B
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor for a tile of 128-byte rows written by TMA with the 128-byte
// swizzle: 8-row groups are 1024 B apart (stride byte offset); version 1; layout type 2 = SWIZZLE_128B.
// The same encoding serves a K-major operand (Q, K: rows = M/N index, 64 contiguous K elements) and the
// MN-major V operand (rows = keys = K index, 64 contiguous N elements).
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait of a pipeline's role.  Returns false when another role gave up or the time limit passed; the caller then falls
// through to the common teardown.  The polls carry a suspend-time hint (1 ms), so that a waiting
// warp leaves its issue slots to the others (measured on the 2K step: 2.5 % against polls without the hint, although a poll
// takes 112 cycles instead of 74), and the clock is the SM's cycle counter (the global timer costs hundreds of cycles
// per read).  The limit is 2^32 cycles, two seconds or more at any clock the part runs at.
__device__ __forceinline__ uint32_t mbar_try_hint(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000000;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done;
}
__device__ __forceinline__ bool mbar_wait_long(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                               int32_t* status) {
  if (mbar_try_hint(bar, parity)) return true;
  const long long t0 = clock64();
#pragma unroll 1
  while (!mbar_try_hint(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > (1ll << 32)) {
      *abort_flag = 1;
      atomicExch(status, 1);
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}
// Tensor maps of one launch.  q is rank 4 (raster query tiles) or rank 5 (patch query tiles); kr/vr
// cover the raster prefix of the cache; k2/v2[i] cover the grid of the i-th key scale tiled in patches.
struct TensorMaps {
  CUtensorMap o;                   // the output: a warp's 32 query slots x 32 columns
  CUtensorMap q, kr, vr;
  CUtensorMap k2[kMaxPatchScales], v2[kMaxPatchScales];
};

// One warp's 32 output rows x 32 columns from shared memory (64-byte rows, 16-byte piece c of row m at position
// c ^ (m / 2 % 4)); rows outside the tensor are not written.  The caller commits the group.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* src, int x, int y, int z, int w) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(map),
               "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}
__device__ __forceinline__ void tma_store_5d(const CUtensorMap* map, const void* src, int x, int y, int z, int w, int v) {
  asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];" ::"l"(map),
               "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(v)
               : "memory");
}

// Loads of one query tile according to its geometry (patch: four boxes of 4 x 8 cells, in slot order).
__device__ __forceinline__ void load_q_tile(void* dst, const TensorMaps& tm, const FwdParams& p, int qt, int h, int b,
                                            uint64_t* bar) {
  if (!p.q_patch) {
    tma_load_4d(dst, &tm.q, 0, qt * kBlockM, h, b, bar);
    return;
  }
  const TileGeom g = p.q_geom[qt];
#pragma unroll
  for (int w = 0; w < 4; ++w)
    tma_load_5d(static_cast<uint8_t*>(dst) + w * (kTileBytes / 4), &tm.q, 0, g.b + patch_slot_col(32 * w),
                g.a + patch_slot_row(32 * w), h, b, bar);
}
// Four consecutive K = 16 steps of one product in a single instruction sequence: step i reads A at
// a_tmem + i * kAStep (TMEM columns) and B at b_desc + i * kBStep (descriptor units of 16 bytes); the first step
// accumulates only when `accumulate_first` is non-zero, the others always do.  The issuing lane's own
// instruction stream is what a product of small MMAs waits for (the tensor pipe takes 50 to 65 cycles per step
// at N <= 128, a step issued through per-step address arithmetic and predicate set-up costs two to three times
// that), so the offsets are immediates and nothing but the four MMAs depends on anything.
template <int kA1, int kA2, int kA3, int kB1, int kB2, int kB3>
__device__ __forceinline__ void mma_ts_x4_at(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate_first) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 b1, b2, b3;\n\t.reg .b32 a1, a2, a3;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, 1, 0;\n\t"
      "add.u32 a1, %1, %5;\n\tadd.u32 a2, %1, %6;\n\tadd.u32 a3, %1, %7;\n\t"
      "add.s64 b1, %2, %8;\n\tadd.s64 b2, %2, %9;\n\tadd.s64 b3, %2, %10;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a1], b1, %3, q;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a2], b2, %3, q;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a3], b3, %3, q;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate_first), "n"(kA1), "n"(kA2), "n"(kA3),
        "n"(kB1), "n"(kB2), "n"(kB3)
      : "memory");
}
template <int kAStep, int kBStep>
__device__ __forceinline__ void mma_ts_x4(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate_first) {
  mma_ts_x4_at<kAStep, 2 * kAStep, 3 * kAStep, kBStep, 2 * kBStep, 3 * kBStep>(d_tmem, a_tmem, b_desc, idesc,
                                                                               accumulate_first);
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Order of the tensor-core kernel's work items.  The (batch row, head) units are taken in groups of
// p.units_per_group; inside a group the items go query tile by query tile, all
// units of the group side by side.  The K/V of one group is what the CTAs resident at one time read: the host
// sizes the group so that it fits in half of L2, and every K/V tile then comes from DRAM once per step instead of
// once per wave of CTAs.
__device__ __forceinline__ void work_item(const FwdParams& p, int n_ranks, int item, int& rank, int& unit) {
  const int n_units = p.n_heads * p.batch_computed;
  const int g_units = p.units_per_group;
  const int group = item / (g_units * n_ranks);
  const int r = item - group * (g_units * n_ranks);
  const int here = min(g_units, n_units - group * g_units);  // the last group may be smaller
  rank = r / here;
  unit = group * g_units + (r - rank * here);
}

}  // namespace tc

// Fills the tensor maps of a launch from its parameters (host); K and V boxes of `key_rows` rows.  encode_code_maps: kr and vr
// cover the tensors of 8-bit codes (raster tiles only).  False when an encoding fails.
bool encode_tensor_maps(const FwdParams& p, tc::TensorMaps* tm, int key_rows);
bool encode_code_maps(const FwdParams& p, tc::TensorMaps* tm, int key_rows);

}  // namespace litevar
