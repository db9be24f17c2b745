// Dynamic min-max quantisation of Q, K or V rows to B-bit integers (paper Section 4, "QKV8"): for every token
// row of a head (64 values) z = (max + min) / 2, s = (max - min) / (2^B - 1),
// code = clamp(round((x - z) / s), -2^(B-1), 2^(B-1) - 1), and the attention runs on code * s + z.  The code is
// the one the correctly rounded fp32 quotient (x - z) / s gives: the quotient is first estimated as
// (x - z) * (1 / s), which is within two units in the last place of it; only an estimate that close to a
// rounding tie (a half-integer) can round to another integer than the quotient does, and those few elements
// take the IEEE division.
//
// In a generation the rows of a step are quantised once, when they are appended to the K/V cache (and Q as it
// is produced); the attention kernels then read the dequantised bf16 rows unchanged.  A row is read
// and written once: eight threads share it (16 bytes each) and take up to four rows at a time (four loads in flight), the row's maximum and minimum come from three shuffles, every thread codes and
// rebuilds its own eight values.  It may run in place.
//
// Bound by instruction issue (ncu, a [64, 30, 680, 64] cache without codes: 77 % of the slots).  That cache with codes (428 MB
// moved) takes 92 us, 4.6 TB/s; it took 135 before: maxima on packed bf16 pairs and three shuffles a row instead of six, the row's
// divisions shared among the threads of a row, index divisions by multiplication, and the code of a row's minimum (a tie by construction, which sent
// every warp through the IEEE divisions of the slow path) decided once per row.
//
// The integer decision is taken in fp32 with one IEEE operation at a time (no contraction into fused
// multiply-adds), so that it can be reproduced exactly.
#include <cuda_runtime.h>

#include "litevar_internal.h"

namespace litevar {

namespace {

constexpr int kQuantThreads = 256;

// Division of an unsigned 31-bit number by a fixed one: multiply and shift (host-computed).
struct FastDiv {
  uint32_t d, mul, shift;
};
FastDiv fast_div(uint32_t d) {
  uint32_t l = 0;
  while (l < 31 && (1u << l) < d) ++l;  // 2^l >= d
  // floor(n / d) = (n mul) >> (31 + l) for n < 2^31 with mul = floor(2^(31 + l) / d) + 1: the error n (mul d - 2^(31 + l)) is
  // at most n d < 2^(31 + l)
  return FastDiv{d, (uint32_t)((1ull << (31 + l)) / d + 1), 31 + l};
}
__device__ __forceinline__ uint32_t div_by(uint32_t n, const FastDiv& f) {
  return (uint32_t)(((uint64_t)n * f.mul) >> f.shift);
}

// One tensor of a launch; its rows go to the groups of eight threads from first_group on.
struct QuantTensor {
  const uint16_t* x;
  uint16_t* dq;  // nullptr: no dequantised output
  int64_t x_sb, x_sh, x_st, d_sb, d_sh, d_st;
  FastDiv n_tokens;
  uint32_t n_rows, first_group;
};
struct QuantArgs {
  QuantTensor t[3];
  int32_t n_tensors;
  FastDiv n_heads;
  float levels, hi;
  int8_t* codes;  // (one tensor only)
  float* scale;
  float* zero;
};

__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float lo_bf16(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float hi_bf16(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// R rows per 8-thread group: that many 16-byte loads in flight per thread (launch_quant has the rule).  MANY: several tensors,
// which have no outputs but the dequantised rows (one tensor: its addresses are read from fixed places).
template <int R, bool MANY>
__global__ void __launch_bounds__(kQuantThreads, 4) quant_rows_kernel(const __grid_constant__ QuantArgs a) {
  // the rows were written by earlier work of the stream; a launch with programmatic serialisation starts early
  asm volatile("griddepcontrol.launch_dependents;");
  constexpr float kMagic = 12582912.f;  // 1.5 * 2^23: a float in [2^23, 2^24) holds an integer in its low mantissa bits
  const int part = threadIdx.x & 7;  // 16-byte column of the row
  // R consecutive rows of a tensor per eight threads, no loop: the grid covers the rows (fewer than 2^31, checked on the
  // host).  Slots past a tensor's last row redo that row and store nothing, so that every lane joins the shuffles.
  const unsigned group = blockIdx.x * (unsigned)(kQuantThreads / 8) + (threadIdx.x >> 3);
  int ti = 0;
  if (MANY && group >= a.t[1].first_group) ti = group >= a.t[2].first_group ? 2 : 1;
  const QuantTensor& tn = a.t[ti];
  const unsigned first = (group - (MANY ? tn.first_group : 0u)) * R;
  int64_t x_off[R], d_off[R];
  uint4 raw[R];
  {
    const unsigned row0 = min(first, tn.n_rows - 1u);
    const unsigned bh = div_by(row0, tn.n_tokens);
    unsigned t = row0 - bh * tn.n_tokens.d;
    unsigned b = div_by(bh, a.n_heads);
    unsigned h = bh - b * a.n_heads.d;
    const bool one_head = t + R <= tn.n_tokens.d;  // the group's rows are tokens of one head (all of them exist)
#pragma unroll
    for (int g = 0; g < R; ++g) {
      if (g > 0 && one_head) {
        x_off[g] = x_off[0] + g * tn.x_st;
        d_off[g] = d_off[0] + g * tn.d_st;
        continue;
      }
      if (g > 0 && first + g < tn.n_rows && ++t == tn.n_tokens.d) {
        t = 0;
        if (++h == a.n_heads.d) {
          h = 0;
          ++b;
        }
      }
      x_off[g] = b * tn.x_sb + h * tn.x_sh + t * tn.x_st + part * 8;
      d_off[g] = b * tn.d_sb + h * tn.d_sh + t * tn.d_st + part * 8;
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
  for (int g = 0; g < R; ++g) raw[g] = *reinterpret_cast<const uint4*>(tn.x + x_off[g]);

  // the row's maximum and minimum: packed bf16 maxima of x and -x (exact), then (max, -min) as one pair through three
  // shuffles; the eight threads of a row are adjacent lanes
  uint32_t top[R];
#pragma unroll
  for (int g = 0; g < R; ++g) {
    const uint4 r = raw[g];
    const uint32_t mx = bf16x2_max(bf16x2_max(r.x, r.y), bf16x2_max(r.z, r.w));
    const uint32_t mn = bf16x2_max(bf16x2_max(r.x ^ 0x80008000u, r.y ^ 0x80008000u),
                                   bf16x2_max(r.z ^ 0x80008000u, r.w ^ 0x80008000u));
    top[g] = bf16x2_max(__byte_perm(mx, mn, 0x5410), __byte_perm(mx, mn, 0x7632));
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1)
#pragma unroll
    for (int g = 0; g < R; ++g) top[g] = bf16x2_max(top[g], __shfl_xor_sync(0xffffffffu, top[g], o));
  // step and its reciprocal, one row per thread (two divisions are a tenth of a thread's work otherwise)
  // The row's minimum is at -(2^B - 1) / 2 of a step, a tie whose rounding takes the exact quotient: its code is decided here,
  // so that no element thread divides for it.  (The maximum is at the opposite tie and ends at the upper clamp either way.)
  float s_row[R], r_row[R], z_row[R], lo_row[R];
  {
    uint32_t mine = top[0];
#pragma unroll
    for (int g = 1; g < R; ++g)
      if ((part & (R - 1)) == g) mine = top[g];
    const float mx = lo_bf16(mine), mn = -hi_bf16(mine);
    const float s = __fdiv_rn(__fsub_rn(mx, mn), a.levels);
    // no step (s = 0, or a row of NaN): estimates of 0, or NaN where x - z is not finite
    const float s1 = s > 0.f ? s : INFINITY;
    const float r = __fdiv_rn(1.f, s1);
    const float z = __fmul_rn(__fadd_rn(mx, mn), 0.5f);
    const float lo = __fsub_rn(__fadd_rn(__fdiv_rn(__fsub_rn(mn, z), s1), kMagic), kMagic);
    const unsigned row = first + (part & (R - 1));
    if (!MANY && part < R && row < tn.n_rows) {
      if (a.scale != nullptr) a.scale[row] = s;
      if (a.zero != nullptr) a.zero[row] = z;
    }
#pragma unroll
    for (int g = 0; g < R; ++g) {
      const int from = (threadIdx.x & 24) + g;
      s_row[g] = R == 1 ? s : __shfl_sync(0xffffffffu, s, from);
      r_row[g] = R == 1 ? r : __shfl_sync(0xffffffffu, r, from);
      lo_row[g] = R == 1 ? lo : __shfl_sync(0xffffffffu, lo, from);
      z_row[g] = __fmul_rn(__fadd_rn(lo_bf16(top[g]), -hi_bf16(top[g])), 0.5f);
    }
  }
#pragma unroll
  for (int g = 0; g < R; ++g) {
    const bool valid = first + g < tn.n_rows;
    const uint32_t u[4] = {raw[g].x, raw[g].y, raw[g].z, raw[g].w};
    const float s = s_row[g], r = r_row[g], z = z_row[g];
    const float2 nz2 = make_float2(-z, -z), r2 = make_float2(r, r);
    const float2 magic2 = make_float2(kMagic, kMagic), nmagic2 = make_float2(-kMagic, -kMagic);
    // Round to nearest even without the conversion pipe: adding 1.5 * 2^23 leaves the integer in the low mantissa bits (|y|
    // stays near 2^(B-1) here), subtracting it again gives it as a float.  The estimate y = (x - z) * (1 / s) is within
    // |y| * 2^-23 < 2^-15.9 of the true quotient and the correctly rounded quotient within 2^-17 of it, so an
    // estimate farther than 2^-14 from a half-integer rounds as the IEEE quotient does; a thread with an estimate
    // closer than that, or that is NaN, redoes its eight values with the division.  So does every thread of a row whose step is so
    // small that its reciprocal is not a normal number.  What has the minimum's difference x - z has its code, and what is above
    // the largest code ends there.
    const float d_min = __fsub_rn(-hi_bf16(top[g]), z), lo = lo_row[g];
    float2 t[4];  // 1.5 * 2^23 + code
    float far = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 dz = __fadd2_rn(make_float2(lo_bf16(u[i]), hi_bf16(u[i])), nz2);
      float2 y = __fmul2_rn(dz, r2);
      y = make_float2(min_nan(dz.x == d_min ? lo : y.x, a.hi), min_nan(dz.y == d_min ? lo : y.y, a.hi));
      t[i] = __fadd2_rn(y, magic2);
      const float2 n = __fadd2_rn(t[i], nmagic2);
      const float2 d = __fadd2_rn(y, make_float2(-n.x, -n.y));
      asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(far) : "f"(fabsf(d.x)), "f"(fabsf(d.y)));
    }
    if (!(far <= 0.5f - 0.00006103515625f) || !((s > 0.f ? s : 1.f) > 1e-30f)) {  // rare (one thread-row in a thousand)
      const float s1 = s > 0.f ? s : 1.f;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        t[i] = make_float2(__fadd_rn(fminf(__fdiv_rn(__fsub_rn(lo_bf16(u[i]), z), s1), a.hi), kMagic),
                           __fadd_rn(fminf(__fdiv_rn(__fsub_rn(hi_bf16(u[i]), z), s1), a.hi), kMagic));
      if (far != far) {  // a NaN takes the lowest code, a row without a step 0
        const float top_code = s > 0.f ? a.hi : 0.f, low_code = s > 0.f ? -1.f - a.hi : 0.f;
        auto code = [&](float x) { return __fadd_rn(fminf(fmaxf(__fdiv_rn(__fsub_rn(x, z), s1), low_code), top_code), kMagic); };
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = make_float2(code(lo_bf16(u[i])), code(hi_bf16(u[i])));
      }
    }
    // (the fast way needs no lower clamp: -(2^B - 1) / 2 rounds to -2^(B-1) at the lowest)
    uint32_t packed[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 c = __fadd2_rn(t[i], nmagic2);
      // two roundings: the packed product and sum were contracted into one multiply-add (measured: other bf16 values)
      const float2 d = make_float2(__fadd_rn(__fmul_rn(c.x, s), z), __fadd_rn(__fmul_rn(c.y, s), z));
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(packed[i]) : "f"(d.y), "f"(d.x));
    }
    if (valid && tn.dq != nullptr)
      *reinterpret_cast<uint4*>(tn.dq + d_off[g]) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    if (!MANY && valid && a.codes != nullptr) {
      uint32_t w[2];
#pragma unroll
      for (int i = 0; i < 2; ++i)  // the low bytes of four codes
        w[i] = __byte_perm(__byte_perm(__float_as_uint(t[2 * i].x), __float_as_uint(t[2 * i].y), 0x0040),
                           __byte_perm(__float_as_uint(t[2 * i + 1].x), __float_as_uint(t[2 * i + 1].y), 0x0040), 0x5410);
      *reinterpret_cast<uint2*>(a.codes + (size_t)(first + g) * kHeadDim + part * 8) = make_uint2(w[0], w[1]);
    }
  }
}

bool quant_strides_ok(const litevar_strides_t* s) {
  return s && s->batch >= 0 && s->head >= 0 && s->token >= kHeadDim && (s->batch % 8) == 0 && (s->head % 8) == 0 &&
         (s->token % 8) == 0;
}

litevar_status_t launch_quant(QuantArgs& a, long long rows, int bits, cudaStream_t stream) {
  a.levels = (float)((1 << bits) - 1);
  a.hi = (float)((1 << (bits - 1)) - 1);
  if (rows >= (1LL << 31)) return LITEVAR_ERR_UNSUPPORTED;  // 2^31 rows of 128 bytes do not fit the device
  // One row per group: more threads and a shorter chain; four: more loads in flight and the row's divisions shared.  Measured (us,
  // one / four): one tensor, 2^15 rows 3.97 / 6.09, 2^16 6.30 / 6.51, 2^17 11.0 / 10.3, 2^18 20.6 / 18.4, 2^21 167 / 136; three
  // tensors, 76 800 rows 7.71 / 7.98, 196 608 16.4 / 15.2, 1.5 million 117 / 98.
  const bool large = rows >= (3LL << 15);
  const int per_group = large ? 4 : 1;
  long long groups = 0;
  for (int i = 0; i < a.n_tensors; ++i) {
    a.t[i].first_group = (uint32_t)groups;
    groups += (a.t[i].n_rows + per_group - 1) / per_group;
  }
  const long long blocks = (groups + kQuantThreads / 8 - 1) / (kQuantThreads / 8);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kQuantThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;  // every thread waits for the previous kernel before its first access
  const bool many = a.n_tensors > 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, large ? (many ? quant_rows_kernel<4, true> : quant_rows_kernel<4, false>)
                                                       : (many ? quant_rows_kernel<1, true> : quant_rows_kernel<1, false>), a);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return LITEVAR_ERR_CUDA;
  }
  return LITEVAR_OK;
}

}  // namespace

}  // namespace litevar

using namespace litevar;

extern "C" litevar_status_t litevar_quantize_rows(const void* x, const litevar_strides_t* sx, int32_t batch,
                                                  int32_t n_heads, int32_t n_tokens, int32_t head_dim, int32_t bits,
                                                  void* x_dq, const litevar_strides_t* sdq, int8_t* codes,
                                                  float* scale, float* zero, void* stream_) {
  if (!x || !quant_strides_ok(sx) || batch < 1 || n_heads < 1 || n_tokens < 1 || bits < 2 || bits > 8)
    return LITEVAR_ERR_INVALID_ARG;
  if (head_dim != kHeadDim) return LITEVAR_ERR_UNSUPPORTED;
  if (x_dq && !quant_strides_ok(sdq)) return LITEVAR_ERR_INVALID_ARG;
  if (((uintptr_t)x | (uintptr_t)x_dq) & 15) return LITEVAR_ERR_INVALID_ARG;
  if (((uintptr_t)codes & 7) || ((uintptr_t)scale & 3) || ((uintptr_t)zero & 3)) return LITEVAR_ERR_INVALID_ARG;
  QuantArgs a = {};
  a.t[0].x = static_cast<const uint16_t*>(x);
  a.t[0].dq = static_cast<uint16_t*>(x_dq);
  a.t[0].x_sb = sx->batch; a.t[0].x_sh = sx->head; a.t[0].x_st = sx->token;
  if (x_dq) { a.t[0].d_sb = sdq->batch; a.t[0].d_sh = sdq->head; a.t[0].d_st = sdq->token; }
  a.t[0].n_tokens = fast_div((uint32_t)n_tokens);
  a.n_tensors = 1;
  a.n_heads = fast_div((uint32_t)n_heads);
  const long long rows = (long long)batch * n_heads * n_tokens;
  a.t[0].n_rows = (uint32_t)rows;
  a.codes = codes; a.scale = scale; a.zero = zero;
  return launch_quant(a, rows, bits, static_cast<cudaStream_t>(stream_));
}

extern "C" litevar_status_t litevar_quantize_qkv(void* q, const litevar_strides_t* sq, int32_t n_q_tokens, void* k,
                                                 const litevar_strides_t* sk, void* v, const litevar_strides_t* sv,
                                                 int32_t n_kv_tokens, int32_t batch, int32_t n_heads,
                                                 int32_t head_dim, int32_t bits, void* stream_) {
  if (!q || !k || !v || !quant_strides_ok(sq) || !quant_strides_ok(sk) || !quant_strides_ok(sv) || batch < 1 ||
      n_heads < 1 || n_q_tokens < 1 || n_kv_tokens < 1 || bits < 2 || bits > 8)
    return LITEVAR_ERR_INVALID_ARG;
  if (head_dim != kHeadDim) return LITEVAR_ERR_UNSUPPORTED;
  if (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v) & 15) return LITEVAR_ERR_INVALID_ARG;
  QuantArgs a = {};
  void* ptr[3] = {q, k, v};
  const litevar_strides_t* st[3] = {sq, sk, sv};
  const int32_t tokens[3] = {n_q_tokens, n_kv_tokens, n_kv_tokens};
  long long rows = 0;
  for (int i = 0; i < 3; ++i) {
    a.t[i].x = static_cast<const uint16_t*>(ptr[i]);
    a.t[i].dq = static_cast<uint16_t*>(ptr[i]);
    a.t[i].x_sb = a.t[i].d_sb = st[i]->batch;
    a.t[i].x_sh = a.t[i].d_sh = st[i]->head;
    a.t[i].x_st = a.t[i].d_st = st[i]->token;
    a.t[i].n_tokens = fast_div((uint32_t)tokens[i]);
    const long long n = (long long)batch * n_heads * tokens[i];
    a.t[i].n_rows = (uint32_t)n;
    rows += n;
  }
  a.n_tensors = 3;
  a.n_heads = fast_div((uint32_t)n_heads);
  return launch_quant(a, rows, bits, static_cast<cudaStream_t>(stream_));
}
