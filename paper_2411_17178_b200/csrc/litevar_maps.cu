// Tensor maps of the tensor-core forward kernel (host).
#include <cstring>
#include <mutex>

#include "litevar_tc_ptx.h"

namespace litevar {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
    else
      (void)cudaGetLastError();
  });
  return fn;
}

// Rank-4 map over a [batch, head, token, 64] bf16 tensor with element strides; box = box_rows tokens x box_dim elements (64, or
// 32 with the swizzle of 64-byte rows).
bool encode_raster(CUtensorMap* tm, const void* base, int64_t rows, int64_t heads, int64_t batch, int64_t st,
                   int64_t sh, int64_t sb, int box_rows, int box_dim = kHeadDim) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  if (rows < 1) rows = 1;  // no raster tile will use this map
  // a dimension of extent 1 may come with any stride; give it a valid one
  if (heads == 1 && sh < kHeadDim) sh = st * rows;
  if (batch == 1 && sb < kHeadDim) sb = sh * heads;
  cuuint64_t gdim[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)rows, (cuuint64_t)heads, (cuuint64_t)batch};
  cuuint64_t gstr[3] = {(cuuint64_t)st * 2, (cuuint64_t)sh * 2, (cuuint64_t)sb * 2};
  cuuint32_t box[4] = {(cuuint32_t)box_dim, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), gdim, gstr, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, box_dim == kHeadDim ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Rank-4 map over a [batch, head, token, 64] tensor of 8-bit codes with byte strides (multiples of 16); box = box_rows
// tokens x 64 bytes, rows packed in shared memory without swizzle.  Rows past the last one read as zero.
bool encode_codes(CUtensorMap* tm, const void* base, int64_t rows, int64_t heads, int64_t batch, int64_t st,
                  int64_t sh, int64_t sb, int box_rows) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  if (rows < 1) rows = 1;
  if (heads == 1 && sh < kHeadDim) sh = st * rows;
  if (batch == 1 && sb < kHeadDim) sb = sh * heads;
  cuuint64_t gdim[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)rows, (cuuint64_t)heads, (cuuint64_t)batch};
  cuuint64_t gstr[3] = {(cuuint64_t)st, (cuuint64_t)sh, (cuuint64_t)sb};
  cuuint32_t box[4] = {(cuuint32_t)kHeadDim, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(base), gdim, gstr, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Rank-5 map over the side x side grid of one scale inside a [batch, head, token, 64] tensor: dimensions
// (64, column, row, head, batch); box = box_rows rows x box_cols columns x 64, i.e. box_rows box_cols rows of 128 B in shared
// memory in row-major order.  A copy may start at any cell.  Cells outside the grid read as zero and are not written.
bool encode_patch(CUtensorMap* tm, const void* base, int64_t first_token, int64_t side, int64_t heads,
                  int64_t batch, int64_t st, int64_t sh, int64_t sb, int box_rows, int box_cols, int box_dim = kHeadDim) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  if (heads == 1 && sh < kHeadDim) sh = st * side * side;
  if (batch == 1 && sb < kHeadDim) sb = sh * heads;
  const uint16_t* origin = static_cast<const uint16_t*>(base) + first_token * st;
  cuuint64_t gdim[5] = {(cuuint64_t)kHeadDim, (cuuint64_t)side, (cuuint64_t)side, (cuuint64_t)heads, (cuuint64_t)batch};
  cuuint64_t gstr[4] = {(cuuint64_t)st * 2, (cuuint64_t)(st * side) * 2, (cuuint64_t)sh * 2, (cuuint64_t)sb * 2};
  cuuint32_t box[5] = {(cuuint32_t)box_dim, (cuuint32_t)box_cols, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<uint16_t*>(origin), gdim, gstr, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, box_dim == kHeadDim ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// The output: boxes of a warp's 32 query slots x 32 columns (the two stream's warps of a slot store half a row each).
bool encode_out(const FwdParams& p, CUtensorMap* tm) {
  const int64_t batch = p.batch_computed + p.share_offset;
  if (p.q_patch) return encode_patch(tm, p.out, 0, p.s_k, p.n_heads, batch, p.o_st, p.o_sh, p.o_sb, 4, 8, 32);
  return encode_raster(tm, p.out, p.n_k, p.n_heads, batch, p.o_st, p.o_sh, p.o_sb, 32, 32);
}

}  // namespace

bool encode_tensor_maps(const FwdParams& p, tc::TensorMaps* tmp, int key_rows) {
  tc::TensorMaps& tm = *tmp;
  memset(&tm, 0, sizeof(tm));
  bool ok = encode_out(p, &tm.o);
  if (p.q_patch)
    ok = ok && encode_patch(&tm.q, p.q, 0, p.s_k, p.n_heads, p.batch_computed, p.q_st, p.q_sh, p.q_sb, 4, 8);  // a warp's slots
  else
    ok = ok && encode_raster(&tm.q, p.q, p.n_k, p.n_heads, p.batch_computed, p.q_st, p.q_sh, p.q_sb, kBlockM);
  ok = ok && encode_raster(&tm.kr, p.k, p.raster_len, p.n_heads, p.batch_computed, p.k_st, p.k_sh, p.k_sb, key_rows) &&
       encode_raster(&tm.vr, p.v, p.raster_len, p.n_heads, p.batch_computed, p.v_st, p.v_sh, p.v_sb, key_rows);
  for (int i = 0; ok && i < p.n_patch_scales; ++i)
    ok = encode_patch(&tm.k2[i], p.k, p.patch_off[i], p.patch_scale[i], p.n_heads, p.batch_computed, p.k_st, p.k_sh,
                      p.k_sb, kChunkSide, kChunkSide) &&
         encode_patch(&tm.v2[i], p.v, p.patch_off[i], p.patch_scale[i], p.n_heads, p.batch_computed, p.v_st, p.v_sh,
                      p.v_sb, kChunkSide, kChunkSide);
  return ok;
}

bool encode_code_maps(const FwdParams& p, tc::TensorMaps* tmp, int key_rows) {
  tc::TensorMaps& tm = *tmp;
  memset(&tm, 0, sizeof(tm));
  return encode_out(p, &tm.o) && encode_raster(&tm.q, p.q, p.n_k, p.n_heads, p.batch_computed, p.q_st, p.q_sh, p.q_sb, kBlockM) &&
         encode_codes(&tm.kr, p.k8, p.L_k, p.n_heads, p.batch_computed, p.c_st, p.c_sh, p.c_sb, key_rows) &&
         encode_codes(&tm.vr, p.v8, p.L_k, p.n_heads, p.batch_computed, p.c_st, p.c_sh, p.c_sb, key_rows);
}

}  // namespace litevar
