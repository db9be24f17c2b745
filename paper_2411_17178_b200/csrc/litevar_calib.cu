// Window calibration of one step (paper Section 2, steps (1)-(3)): from saved post-softmax attention maps,
// for every part of the step-k map find the smallest window radius w whose share R_w of the part's
// attention mass reaches the threshold R_0.
//
// R_w for all w at once: every map entry (q, t) of part j lies at Chebyshev distance
// d = max(|r' - ctr_j(r)|, |c' - ctr_j(c)|) from the key cell under the query; the window of radius w holds
// exactly the entries with d <= w.  One pass over the maps accumulates the mass per (part, distance); a
// running sum over d then gives the window mass for every w.  The pass is bound by reading the maps once.
//
// A warp owns batches of consecutive (map, query) rows and walks them once per part, so that it needs
// histogram bins for one part at a time: bins[distance][lane] in shared memory (fp32; fp64 for summed maps), private to the lane,
// updated with plain loads and stores.  After at most 256 rows the bins are summed over the lanes in fp64 and
// added to the global histogram with one fp64 add per non-empty bin.
//   Parts of up to 256 keys: a lane reads flat key positions t = 32 * chunk + lane, so every lane of a load is
// used whatever the grid width, and one round takes the same chunk of eight query rows (eight independent
// loads in flight however small the part).
//   Wider parts: lanes sweep the columns of a key row.  In a key row at row distance dr the entries whose
// column distance is smaller fall into bin dr and add up in a register before one shared-memory update per
// key row; the others belong to the bin of their own column distance, which is fixed per lane, so they add up
// in registers over all key rows of the query.
//
// The distance of an entry does not depend on the map, so several maps are added up entry by entry first (sum_maps_kernel, a
// pass at memory speed) and the histogram pass reads one or a few summed maps instead of all of them.  The histogram pass costs
// about 3.5 times what reading its input costs, so this pays from two maps on.  The sums and their histogram are fp64: rounded to
// fp32, a sum over all maps weighs in every entry, where the maps' own histograms average their roundings (error of R_w with fp32
// sums 1.0e-9 to 2.2e-9 rms, 0.8e-10 to 4.0e-10 map by map).  Scratch of at most kScratchBytes (a single 2K map, 2.2 GB, goes to
// the histogram directly, and so do all maps where the scratch cannot be had).
// Measured on B200 (whole calls, us, maps one by one / summed): 64 maps of the last 512px step (587 MB) 338 / 161; 1280 maps of the
// last 256px step (891 MB) 391 / 225; with fp32 sums and bins 158 and 218.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>
#include <vector>

#include "litevar_internal.h"

namespace litevar {

namespace {

constexpr int kCalibWarps = 4;
constexpr int kMaxDist = kMaxScale;   // distances 0 .. s_j - 1
constexpr int kCalibFlushRows = 256;  // rows a lane's fp32 bins take in before they are flushed
constexpr int kCalibMaxRows = 1 << 30;  // (map, query) rows of one launch
constexpr int kSumThreads = 256, kSumPerThread = 4, kSumUnroll = 4;
constexpr size_t kScratchBytes = 64u << 20;    // summed maps of one call, at most

// out[g][i] = sum of maps m in [g * per_group, (g + 1) * per_group) of maps[m][i].  A thread owns kSumPerThread entries, a block's
// width apart (coalesced whatever the alignment of a map), and has kSumPerThread * kSumUnroll loads in flight.  Clears the
// histogram on the way, and lets the histogram pass be launched while the last blocks run (it waits for them).
__global__ void __launch_bounds__(kSumThreads) sum_maps_kernel(const float* __restrict__ maps, int64_t n, int64_t n_maps,
                                                               int64_t per_group, double* __restrict__ out, double* hist) {
  if (blockIdx.y == 0)
    for (int i = blockIdx.x * kSumThreads + threadIdx.x; i < kMaxScales * kMaxDist; i += gridDim.x * kSumThreads) hist[i] = 0.0;
  const int64_t first = (int64_t)blockIdx.x * (kSumThreads * kSumPerThread) + threadIdx.x;
  const int64_t m0 = blockIdx.y * per_group, m1 = min(n_maps, m0 + per_group);
  double acc[kSumPerThread] = {};
  const float* src = maps + m0 * n + first;
  if (first + (kSumPerThread - 1) * kSumThreads < n) {
    int64_t m = m0;
    for (; m + kSumUnroll <= m1; m += kSumUnroll) {
      float v[kSumUnroll][kSumPerThread];
#pragma unroll
      for (int u = 0; u < kSumUnroll; ++u)
#pragma unroll
        for (int e = 0; e < kSumPerThread; ++e) v[u][e] = __ldcs(src + u * n + e * kSumThreads);
#pragma unroll
      for (int u = 0; u < kSumUnroll; ++u)
#pragma unroll
        for (int e = 0; e < kSumPerThread; ++e) acc[e] += v[u][e];
      src += kSumUnroll * n;
    }
    for (; m < m1; ++m, src += n)
#pragma unroll
      for (int e = 0; e < kSumPerThread; ++e) acc[e] += __ldcs(src + e * kSumThreads);
  } else {  // the last block of a map
    for (int64_t m = m0; m < m1; ++m, src += n)
#pragma unroll
      for (int e = 0; e < kSumPerThread; ++e)
        if (first + e * kSumThreads < n) acc[e] += __ldcs(src + e * kSumThreads);
  }
#pragma unroll
  for (int e = 0; e < kSumPerThread; ++e)
    if (first + e * kSumThreads < n) out[blockIdx.y * n + first + e * kSumThreads] = acc[e];
  asm volatile("griddepcontrol.launch_dependents;");
}

// Stream-ordered pool of the calibration scratch, one per device, made on first use.  It keeps at most one call's scratch
// between calls (the device's default pool gives every block back at the synchronisation each call ends with, which made the
// next call pay for a new mapping: 0.3 to 0.9 ms); what overlapping calls took beyond that goes back at their
// synchronisations.  The memory returns to the device when the library is unloaded.
struct ScratchPools {
  std::mutex mu;
  cudaMemPool_t pool[64] = {};
  ~ScratchPools() {
    for (cudaMemPool_t p : pool)
      if (p) (void)cudaMemPoolDestroy(p);
  }
  cudaError_t get(int dev, cudaMemPool_t* out) {
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!pool[dev]) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t p = nullptr;
      cudaError_t e = cudaMemPoolCreate(&p, &props);
      if (e != cudaSuccess) return e;
      uint64_t keep = kScratchBytes + (1u << 20);
      e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
      if (e != cudaSuccess) {
        (void)cudaMemPoolDestroy(p);
        return e;
      }
      pool[dev] = p;
    }
    *out = pool[dev];
    return cudaSuccess;
  }
};

// Wide part (more than 256 keys) of one query row: NC 32-column chunks per key row, 16 loads in flight per round.
template <int NC, typename T>
__device__ __forceinline__ void calib_wide_row(T* bins, int lane, const T* __restrict__ part, int s_j, int cr, int cc) {
  constexpr int KR = 16 / NC;
  int dc[NC];
  T outer[NC];
  bool cv[NC];
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    const int kc = lane + 32 * u;
    cv[u] = kc < s_j;
    dc[u] = abs(kc - cc);
    outer[u] = 0;
  }
  for (int kr0 = 0; kr0 < s_j; kr0 += KR) {
    T a[KR][NC];
#pragma unroll
    for (int v = 0; v < KR; ++v)
#pragma unroll
      for (int u = 0; u < NC; ++u)
        a[v][u] = (cv[u] && kr0 + v < s_j) ? __ldg(part + (kr0 + v) * s_j + lane + 32 * u) : T(0);
#pragma unroll
    for (int v = 0; v < KR; ++v) {
      const int kr = kr0 + v;
      if (kr < s_j) {
        const int dr = abs(kr - cr);
        T inner = 0;
#pragma unroll
        for (int u = 0; u < NC; ++u) {
          if (dc[u] < dr) inner += a[v][u]; else outer[u] += a[v][u];
        }
        bins[(dr << 5) + lane] += inner;
      }
    }
  }
#pragma unroll
  for (int u = 0; u < NC; ++u)
    if (cv[u]) bins[(dc[u] << 5) + lane] += outer[u];
}

// T: float for maps (fp32 bins, at most kCalibFlushRows rows each), double for summed maps (nothing is rounded to fp32 again).
template <typename T>
__global__ void __launch_bounds__(kCalibWarps * 32, sizeof(T) == 4 ? 32 / kCalibWarps : 16 / kCalibWarps)
calib_hist_kernel(Schedule sc, int k0, int first_part, int s_max, const T* __restrict__ maps, int n_rows_total,
                  int q_first /* query index of row 0 */, int rows_per_batch,
                  double* __restrict__ hist /* [kMaxScales][kMaxDist] */) {
  extern __shared__ __align__(8) uint8_t sh[];  // T [warps][s_max][32]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_block_warps = blockDim.x >> 5;
  T* bins = reinterpret_cast<T*>(sh) + (size_t)warp * s_max * 32;
  const int s_k = sc.scale[k0];
  const int n_k = s_k * s_k;
  const int L_k = sc.off[k0 + 1];
  const int n_batches = (n_rows_total + rows_per_batch - 1) / rows_per_batch;
  const int warp_global = blockIdx.x * n_block_warps + warp;
  const int n_warps = gridDim.x * n_block_warps;
  const int flush_every = max(1, kCalibFlushRows / rows_per_batch);
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the summed maps and the cleared histogram

  for (int j = first_part + blockIdx.y; j <= k0; j += gridDim.y) {  // few rows: the parts go to blocks of their own
    const int s_j = sc.scale[j];
    const int n_j = s_j * s_j;
    const int n_chunks = (n_j + 31) >> 5;
    const int step_r = 32 / s_j, step_c = 32 - step_r * s_j;  // a lane's flat key cell moves by this per chunk
    const int r_t0 = lane / s_j, c_t0 = lane - r_t0 * s_j;
    const int off_j = sc.off[j];
    double* hist_j = hist + (size_t)j * kMaxDist;
    for (int d = 0; d < s_j; ++d) bins[(d << 5) + lane] = 0;
    int pending = 0;
    for (int batch = warp_global; batch < n_batches; batch += n_warps) {
      const int row0 = batch * rows_per_batch;
      const int nb = min(rows_per_batch, n_rows_total - row0);
      // lane i holds the co-located key cell of row i of the batch
      int pk;
      {
        const unsigned q = ((unsigned)(q_first + row0 % n_k) + (unsigned)lane) % (unsigned)n_k;
        const int r = (int)q / s_k, c = (int)q - r * s_k;
        pk = (((2 * r + 1) * s_j) / (2 * s_k)) | ((((2 * c + 1) * s_j) / (2 * s_k)) << 16);
      }
      const T* src = maps + (size_t)row0 * L_k + off_j;
      if (n_chunks <= 8) {
        for (int i0 = 0; i0 < nb; i0 += 8) {
          int cr[8], cc[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int p = __shfl_sync(0xffffffffu, pk, (i0 + u) & 31);
            cr[u] = p & 0xffff;
            cc[u] = p >> 16;
          }
          const int ng = nb - i0;
          const T* grp = src + (size_t)i0 * L_k + lane;
          int r_t = r_t0, c_t = c_t0;
          for (int ch = 0; ch < n_chunks; ++ch) {
            const bool tv = (ch << 5) + lane < n_j;
            T a[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u] = (tv && u < ng) ? __ldg(grp + (size_t)u * L_k + (ch << 5)) : T(0);
            if (tv) {
              // rows past the end of the batch carry zeros into a valid bin
#pragma unroll
              for (int u = 0; u < 8; ++u)
                bins[(max(abs(r_t - cr[u]), abs(c_t - cc[u])) << 5) + lane] += a[u];
            }
            r_t += step_r;
            c_t += step_c;
            if (c_t >= s_j) {
              c_t -= s_j;
              ++r_t;
            }
          }
        }
      } else {
        const int nc = (s_j + 31) >> 5;
        for (int i = 0; i < nb; ++i) {
          const int p = __shfl_sync(0xffffffffu, pk, i);
          const int cr = p & 0xffff, cc = p >> 16;
          const T* part = src + (size_t)i * L_k;
          switch (nc) {
            case 1: calib_wide_row<1>(bins, lane, part, s_j, cr, cc); break;
            case 2: calib_wide_row<2>(bins, lane, part, s_j, cr, cc); break;
            case 3: calib_wide_row<3>(bins, lane, part, s_j, cr, cc); break;
            case 4: calib_wide_row<4>(bins, lane, part, s_j, cr, cc); break;
            default: calib_wide_row<8>(bins, lane, part, s_j, cr, cc); break;
          }
        }
      }
      if (++pending == flush_every || batch + n_warps >= n_batches) {
        pending = 0;
        __syncwarp();
        // lane l sums bin d = d0 + l over the 32 lane columns, rotated so that the lanes hit distinct banks
        for (int d0 = 0; d0 < s_j; d0 += 32) {
          const int d = d0 + lane;
          if (d < s_j) {
            double sum = 0.0;
#pragma unroll 8
            for (int i = 0; i < 32; ++i) sum += (double)bins[(d << 5) + ((i + lane) & 31)];
            if (sum != 0.0) atomicAdd(&hist_j[d], sum);
          }
        }
        __syncwarp();
        for (int d = 0; d < s_j; ++d) bins[(d << 5) + lane] = 0;
      }
    }
    __syncwarp();
  }
}

}  // namespace

}  // namespace litevar

using namespace litevar;

extern "C" litevar_status_t litevar_calibrate_windows(const int32_t* scales, int32_t n_scales, int32_t step_k,
                                                      int32_t n_global_scales, const float* maps, int64_t n_maps,
                                                      double r0, int32_t* radius, double* ratio, void* stream_) {
  if (!scales || !maps || !radius) return LITEVAR_ERR_INVALID_ARG;
  if (n_scales < 1 || n_scales > kMaxScales || step_k < 1 || step_k > n_scales || n_maps < 1 ||
      n_global_scales < 0 || !(r0 > 0.0) || r0 > 1.0)
    return LITEVAR_ERR_INVALID_ARG;
  for (int i = 0; i < n_scales; ++i)
    if (scales[i] < 1 || scales[i] > kMaxScale) return LITEVAR_ERR_INVALID_ARG;
  if ((uintptr_t)maps & 3) return LITEVAR_ERR_INVALID_ARG;
  Schedule sc;
  memset(&sc, 0, sizeof(sc));
  sc.n_scales = n_scales;
  for (int i = 0; i < n_scales; ++i) {
    sc.scale[i] = scales[i];
    sc.off[i + 1] = sc.off[i] + scales[i] * scales[i];
  }
  const int k0 = step_k - 1;
  const int first_part = n_global_scales < step_k ? n_global_scales : step_k;
  for (int j = 0; j < n_scales; ++j) radius[j] = -1;
  if (ratio)
    for (int i = 0; i < n_scales * kMaxDist; ++i) ratio[i] = 1.0;
  if (first_part > k0) return LITEVAR_OK;  // every part of this step is global

  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  const size_t hist_bytes = sizeof(double) * kMaxScales * kMaxDist;
  const int n_k = scales[k0] * scales[k0];
  const long long L_k = sc.off[k0 + 1], map_len = (long long)n_k * L_k;
  int dev = 0, n_sm = 148;
  cudaMemPool_t pool = nullptr;
  static ScratchPools pools;
  if (cudaGetDevice(&dev) != cudaSuccess || pools.get(dev, &pool) != cudaSuccess) {
    (void)cudaGetLastError();
    return LITEVAR_ERR_CUDA;
  }
  (void)cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  // groups of maps that are added up: as many as fill the chip with threads
  long long groups = 0, per_group = 0;
  if (n_maps > 1 && map_len <= (long long)(kScratchBytes / sizeof(double))) {
    const long long threads = (map_len + kSumPerThread - 1) / kSumPerThread;
    groups = (2048ll * n_sm + threads - 1) / threads;
    if (groups > (n_maps + 3) / 4) groups = (n_maps + 3) / 4;
    const long long room = (long long)(kScratchBytes / sizeof(double)) / map_len;
    if (groups > room || groups > 65535) groups = 0;  // too much for the scratch: straight to the histogram
    if (groups > 0) {
      per_group = (n_maps + groups - 1) / groups;
      groups = (n_maps + per_group - 1) / per_group;
    }
  }
  char* scratch = nullptr;
  auto allocate = [&] {
    return cudaMallocFromPoolAsync(reinterpret_cast<void**>(&scratch), hist_bytes + (size_t)(groups * map_len) * sizeof(double), pool,
                                   stream);
  };
  cudaError_t got = allocate();
  if (got == cudaErrorMemoryAllocation && groups > 0) {  // no room for the summed maps: straight to the histogram
    (void)cudaGetLastError();
    groups = 0;
    got = allocate();
  }
  if (got != cudaSuccess) {
    (void)cudaGetLastError();
    return LITEVAR_ERR_OOM;
  }
  double* d_hist = reinterpret_cast<double*>(scratch);
  litevar_status_t st = LITEVAR_OK;
  std::vector<double> hist((size_t)kMaxScales * kMaxDist);
  double* summed = nullptr;
  if (groups > 0) {
    summed = reinterpret_cast<double*>(scratch + hist_bytes);
    const long long per_block = kSumThreads * kSumPerThread;
    sum_maps_kernel<<<dim3((unsigned)((map_len + per_block - 1) / per_block), (unsigned)groups), kSumThreads, 0, stream>>>(
        maps, map_len, n_maps, per_group, summed, d_hist);
    if (cudaGetLastError() != cudaSuccess) st = LITEVAR_ERR_CUDA;
    n_maps = groups;
  }
  const long long rows = (long long)n_maps * n_k;
  int s_max = 1;
  for (int j = first_part; j <= k0; ++j) s_max = scales[j] > s_max ? scales[j] : s_max;
  const size_t warp_smem = (groups > 0 ? sizeof(double) : sizeof(float)) * 32 * (size_t)s_max;
  const int block_warps = warp_smem * kCalibWarps > (200u << 10) ? kCalibWarps / 2 : kCalibWarps;  // (fp64 bins, 200 distances and more)
  const size_t smem = warp_smem * block_warps;
  // resident warps: up to 32 per SM (16 with fp64 bins), fewer where the bins of the widest part need the shared memory
  int blocks_per_sm = (int)((200u << 10) / (smem + 1024));
  if (blocks_per_sm > (groups > 0 ? 16 : 32) / kCalibWarps) blocks_per_sm = (groups > 0 ? 16 : 32) / kCalibWarps;
  if (blocks_per_sm < 1) blocks_per_sm = 1;
  const long long n_warps = (long long)n_sm * blocks_per_sm * block_warps;
  if (st != LITEVAR_OK || (groups == 0 && cudaMemsetAsync(d_hist, 0, hist_bytes, stream) != cudaSuccess) ||
      (groups > 0 ? cudaFuncSetAttribute(calib_hist_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                  : cudaFuncSetAttribute(calib_hist_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    st = LITEVAR_ERR_CUDA;
  for (long long first = 0; first < rows && st == LITEVAR_OK; first += kCalibMaxRows) {
    const int n_rows = (int)(rows - first < kCalibMaxRows ? rows - first : kCalibMaxRows);
    // rows per batch: the choice whose batch waves over the resident warps finish first, counting a batch
    // as the mean of its rows (wide parts) and its rows rounded up to groups of eight (small parts)
    int rows_per_batch = 1;
    long long best = 0;
    for (int rpb = 32; rpb >= 1; --rpb) {
      const long long batches = (n_rows + rpb - 1) / rpb;
      const long long span = (batches + n_warps - 1) / n_warps * (rpb + (rpb + 7) / 8 * 8);
      if (best == 0 || span < best) {
        best = span;
        rows_per_batch = rpb;
      }
    }
    const long long n_batches = ((long long)n_rows + rows_per_batch - 1) / rows_per_batch;
    long long blocks = (n_batches + block_warps - 1) / block_warps;
    if (blocks > (long long)n_sm * blocks_per_sm) blocks = (long long)n_sm * blocks_per_sm;
    const unsigned parts = (unsigned)(k0 + 1 - first_part);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, n_batches <= 2 * n_warps ? parts : 1u);
    cfg.blockDim = dim3((unsigned)block_warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = groups > 0 && first == 0 ? 1 : 0;  // behind sum_maps_kernel
    const int q_first = (int)(first % n_k);
    const cudaError_t e =
        groups > 0 ? cudaLaunchKernelEx(&cfg, calib_hist_kernel<double>, sc, k0, first_part, s_max,
                                        static_cast<const double*>(summed + first * L_k), n_rows, q_first, rows_per_batch, d_hist)
                   : cudaLaunchKernelEx(&cfg, calib_hist_kernel<float>, sc, k0, first_part, s_max, maps + first * L_k, n_rows,
                                        q_first, rows_per_batch, d_hist);
    if (e != cudaSuccess)
      st = LITEVAR_ERR_CUDA;
  }
  if (st == LITEVAR_OK && (cudaMemcpyAsync(hist.data(), d_hist, sizeof(double) * kMaxDist * (size_t)step_k, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
                           cudaStreamSynchronize(stream) != cudaSuccess))
    st = LITEVAR_ERR_CUDA;
  (void)cudaFreeAsync(scratch, stream);
  if (st != LITEVAR_OK) {
    (void)cudaGetLastError();
    return st;
  }
  // running sums over the distance: window mass for every radius; smallest radius with mass >= R_0 * total
  for (int j = first_part; j <= k0; ++j) {
    const double* h = hist.data() + (size_t)j * kMaxDist;
    double total = 0.0;
    for (int d = 0; d < scales[j]; ++d) total += h[d];
    double cum = 0.0;
    int w = scales[j] - 1;
    bool found = false;
    for (int d = 0; d < scales[j]; ++d) {
      cum += h[d];
      if (ratio) ratio[(size_t)j * kMaxDist + d] = total > 0.0 ? cum / total : 1.0;
      if (!found && cum >= r0 * total) {
        w = d;
        found = true;
      }
    }
    radius[j] = w;
  }
  return LITEVAR_OK;
}
