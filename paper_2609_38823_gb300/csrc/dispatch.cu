// Dispatch of the routed (token, slot) pairs to the prefix experts: per-tile
// histograms with warp-aggregated shared-memory atomics, a scan, a stable
// rank assignment, and a 128-bit row gather (DecoMoE Algorithm 2: only the
// first K expert MLPs are evaluated, each on the tokens routed to it).
#include <mutex>

#include "dispatch_tile.cuh"

namespace decomoe {

// All threads of the cluster's blocks; release / acquire, so shared memory
// written before the arrive is visible to the cluster after the wait.
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  cluster_arrive();
  cluster_wait();
}
// The int at p's offset in the shared memory of block `rank` of the cluster.
__device__ __forceinline__ int ld_cluster_i32(const int* p, int rank) {
  uint32_t a;
  int v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

// Deferred activated mass (Eq. 11) carried by a dispatch launch: blocks
// [first, first + E) of the grid add up the routing blocks' partial masses,
// one expert each, in the fixed order of mass_finalize_block.
struct MassFinish {
  const double* part = nullptr;  // null: nothing to finish
  int nblocks = 0;
  int E = 0;
  double* mass = nullptr;
};

// Pass 1: histogram of expert ids in each tile of DSP_TILE consecutive pairs
// (blocks [0, ntiles)); blocks from ntiles on finish a deferred mass.
__global__ void __launch_bounds__(DSP_THREADS)
    k_dispatch_hist(const int32_t* __restrict__ idx, int64_t N, int K,
                    int32_t* __restrict__ tile_hist, int32_t* status, int ntiles, MassFinish mf) {
  pdl_enter();
  if (static_cast<int>(blockIdx.x) >= ntiles) {
    mass_finalize_block(mf.part, mf.nblocks, mf.E, static_cast<int>(blockIdx.x) - ntiles, mf.mass);
    return;
  }
  __shared__ int hist[DECOMOE_MAX_E];
  for (int e = threadIdx.x; e < K; e += DSP_THREADS) hist[e] = 0;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t base = static_cast<int64_t>(blockIdx.x) * DSP_TILE + warp * DSP_PER_WARP;
#pragma unroll
  for (int r = 0; r < DSP_PER_WARP / 32; ++r) {
    const int64_t f = base + r * 32 + lane;
    int e = -2;
    if (f < N) {
      e = idx[f];
      if (e < 0 || e >= K) {
        report_status(status, DECOMOE_ERR_BAD_INPUT);
        e = -1;
      }
    }
    const uint32_t grp = __match_any_sync(0xffffffffu, e);
    if (e >= 0 && lane == __ffs(grp) - 1) atomicAdd(&hist[e], __popc(grp));
  }
  __syncthreads();
  for (int e = threadIdx.x; e < K; e += DSP_THREADS)
    tile_hist[static_cast<int64_t>(blockIdx.x) * K + e] = hist[e];
}

// Pass 2: the tile kernel (dispatch_tile). SINGLE: one tile in one block
// that also copies the rows; blocks from 1 on finish a deferred mass.
template <bool SINGLE>
__global__ void __launch_bounds__(DSP_THREADS)
    k_dispatch_scatter(const int32_t* __restrict__ idx, int64_t N, int k, int K,
                       const int32_t* __restrict__ tile_hist, int ntiles,
                       int32_t* __restrict__ counts, int32_t* __restrict__ offsets,
                       int32_t* __restrict__ perm_token, int32_t* __restrict__ inv_slot,
                       int32_t* status = nullptr, const uint4* __restrict__ x = nullptr, int row_vec = 0,
                       uint4* __restrict__ x_perm = nullptr, MassFinish mf = MassFinish{}) {
  pdl_enter();
  if (SINGLE && blockIdx.x > 0) {
    mass_finalize_block(mf.part, mf.nblocks, mf.E, static_cast<int>(blockIdx.x) - 1, mf.mass);
    return;
  }
  dispatch_tile<SINGLE>(idx, N, k, K, tile_hist, ntiles, static_cast<int>(blockIdx.x), counts, offsets, perm_token,
                        inv_slot, status, x, row_vec, x_perm);
}

// Passes 1 and 2 in one launch for up to DSC_MAX_PAIRS pairs: a cluster of
// eight blocks, warp w of block b owning P consecutive pairs (P a multiple of
// 32, at most 32 R). Each warp ranks its pairs as it counts them
// (__match_any_sync per 32-pair round), the block scans its warps' counts per
// expert, and the blocks read each other's counts through distributed shared
// memory: one launch and no histogram in global memory. Blocks from the second
// cluster on finish a deferred mass. Bound by latency: 16384 pairs 11.2 us in two
// launches -> 7.7 (2048-token layer 223.9 -> 222.4 us), 1048 pairs 9.5 -> 5
// (131-token layer 69.7 -> 66.1 us). Eight blocks is the portable cluster; more
// pairs would serialise on them, and the two launches spread over the SMs.
constexpr int DSC_CTAS = 8;
constexpr int DSC_MAX_ROUNDS = 8;
constexpr int64_t DSC_MAX_PAIRS = static_cast<int64_t>(DSC_CTAS) * DSP_WARPS * 32 * DSC_MAX_ROUNDS;  // 16384
template <int R>
__global__ void __launch_bounds__(DSP_THREADS)
    k_dispatch_cluster(const int32_t* __restrict__ idx, int64_t N, int k, int K, int P, int32_t* __restrict__ counts,
                       int32_t* __restrict__ offsets, int32_t* __restrict__ perm_token,
                       int32_t* __restrict__ inv_slot, int32_t* status, MassFinish mf) {
  pdl_enter();
  __shared__ int s_hist[DECOMOE_MAX_E];            // this block's pairs per expert (read by the cluster)
  __shared__ int s_base[DECOMOE_MAX_E];            // first row of this block's pairs of each expert
  __shared__ int s_wcnt[DSP_WARPS][DECOMOE_MAX_E];
  __shared__ int s_wsum[DSP_WARPS];
  if (blockIdx.x >= DSC_CTAS) {
    const int e = static_cast<int>(blockIdx.x) - DSC_CTAS;
    if (e < mf.E) mass_finalize_block(mf.part, mf.nblocks, mf.E, e, mf.mass);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e_t = threadIdx.x;  // one expert per thread (K <= 256 = DSP_THREADS)
  const int64_t base = (static_cast<int64_t>(blockIdx.x) * DSP_WARPS + warp) * P;
  int ex[R], rank[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t f = base + r * 32 + lane;
    const bool in = r * 32 < P && f < N;
    ex[r] = in ? idx[f] : -2;  // -2: no pair here
    if (in && (ex[r] < 0 || ex[r] >= K)) ex[r] = -1;
  }
  for (int e = lane; e < K; e += 32) s_wcnt[warp][e] = 0;
  __syncwarp();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (ex[r] == -1) report_status(status, DECOMOE_ERR_BAD_INPUT);
    const uint32_t grp = __match_any_sync(0xffffffffu, ex[r]);
    if (ex[r] >= 0) rank[r] = s_wcnt[warp][ex[r]] + __popc(grp & ((1u << lane) - 1u));
    __syncwarp();
    if (ex[r] >= 0 && lane == __ffs(grp) - 1) s_wcnt[warp][ex[r]] += __popc(grp);
    __syncwarp();
  }
  __syncthreads();
  if (e_t < K) {  // exclusive scan over the warps
    int run = 0;
#pragma unroll
    for (int w = 0; w < DSP_WARPS; ++w) {
      const int c = s_wcnt[w][e_t];
      s_wcnt[w][e_t] = run;
      run += c;
    }
    s_hist[e_t] = run;
  }
  cluster_sync_all();
  int tot = 0, before = 0;
  if (e_t < K) {
    int v[DSC_CTAS];
#pragma unroll
    for (int b = 0; b < DSC_CTAS; ++b) v[b] = ld_cluster_i32(&s_hist[e_t], b);
#pragma unroll
    for (int b = 0; b < DSC_CTAS; ++b) {
      tot += v[b];
      if (b < static_cast<int>(blockIdx.x)) before += v[b];
    }
  }
  cluster_arrive();  // this block's reads of the others' counts are done
  int incl = tot;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) s_wsum[warp] = incl;
  __syncthreads();
  int wpre = 0;
  for (int w = 0; w < warp; ++w) wpre += s_wsum[w];
  const int excl = wpre + incl - tot;
  if (e_t < K) {
    s_base[e_t] = excl + before;
    if (blockIdx.x == 0) {
      counts[e_t] = tot;
      offsets[e_t] = excl;
      if (e_t == K - 1) offsets[K] = excl + tot;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (ex[r] == -2) continue;
    const int64_t f = base + r * 32 + lane;
    int row = -1;
    if (ex[r] >= 0) {
      row = s_base[ex[r]] + s_wcnt[warp][ex[r]] + rank[r];
      perm_token[row] = static_cast<int32_t>(f / k);
    }
    inv_slot[f] = row;
  }
  cluster_wait();  // no block leaves while another may still read its counts
}

// Pass 3: x_perm[r, :] = x[perm_token[r], :], one warp per row, 16-byte
// vectors, loads of a row issued before its stores.
__global__ void __launch_bounds__(256)
    k_gather_rows(const uint4* __restrict__ x, const int32_t* __restrict__ perm_token,
                  const int32_t* __restrict__ offsets, int K, int vec_per_row,
                  uint4* __restrict__ x_perm) {
  pdl_enter();
  const int rows = offsets[K];
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int r = gw; r < rows; r += nw) {
    const int t = perm_token[r];
    const uint4* src = x + static_cast<int64_t>(t) * vec_per_row;
    uint4* dst = x_perm + static_cast<int64_t>(r) * vec_per_row;
    int c = lane;
    for (; c + 32 * 7 < vec_per_row; c += 32 * 8) {
      uint4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldg(src + c + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u) dst[c + 32 * u] = v[u];
    }
    for (; c < vec_per_row; c += 32) dst[c] = __ldg(src + c);
  }
}

}  // namespace decomoe

using namespace decomoe;

extern "C" {

size_t decomoe_dispatch_workspace_bytes(int64_t T, int k, int K) {
  if (T < 0 || k <= 0 || K <= 0) return 0;
  const int64_t N = T * k;
  const int64_t ntiles = (N + DSP_TILE - 1) / DSP_TILE;
  return align_up(static_cast<size_t>(ntiles > 0 ? ntiles : 1) * K * sizeof(int32_t), 256);
}

int decomoe_gather_rows(const void* x, const int32_t* perm_token, const int32_t* offsets, int K, int64_t N,
                        int d, int dtype, void* x_perm, decomoe_stream_t stream) {
  clear_error();
  DM_ARG_CHECK(N >= 0 && K >= 1 && d > 0 && (dtype == DECOMOE_BF16 || dtype == DECOMOE_F32),
               "gather_rows: bad sizes or dtype");
  if (N == 0) return DECOMOE_OK;
  const size_t row_bytes = static_cast<size_t>(d) * dtype_bytes(dtype);
  DM_ARG_CHECK(x && perm_token && offsets && x_perm, "gather_rows: null pointer");
  DM_ARG_CHECK(row_bytes % 16 == 0 && aligned16(x) && aligned16(x_perm),
               "gather_rows: rows must be 16-byte multiples and 16-byte aligned");
  return launch_gather_rows(x, perm_token, offsets, K, row_bytes, N, x_perm, reinterpret_cast<cudaStream_t>(stream));
}

int decomoe_dispatch(const int32_t* topk_idx, int64_t T, int k, int K, const void* x, int d,
                     int dtype, int32_t* counts, int32_t* offsets, int32_t* perm_token,
                     int32_t* inv_slot, void* x_perm, void* ws, size_t ws_bytes,
                     int32_t* status_dev, decomoe_stream_t stream) {
  clear_error();
  return dispatch_with_mass(topk_idx, T, k, K, x, d, dtype, counts, offsets, perm_token, inv_slot, x_perm, ws,
                            ws_bytes, status_dev, nullptr, 0, 0, nullptr, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"

namespace decomoe {

int dispatch_with_mass(const int32_t* topk_idx, int64_t T, int k, int K, const void* x, int d, int dtype,
                       int32_t* counts, int32_t* offsets, int32_t* perm_token, int32_t* inv_slot, void* x_perm,
                       void* ws, size_t ws_bytes, int32_t* status_dev, const double* mass_part, int mass_blocks,
                       int mass_E, double* mass, cudaStream_t s) {
  MassFinish mf;
  if (mass_part != nullptr && mass_blocks > 0) {
    DM_ARG_CHECK(mass != nullptr && mass_E >= 1 && mass_E <= DECOMOE_MAX_E, "dispatch: bad deferred mass");
    mf.part = mass_part;
    mf.nblocks = mass_blocks;
    mf.E = mass_E;
    mf.mass = mass;
  }
  const int mblocks = mf.part != nullptr ? mf.E : 0;
  DM_ARG_CHECK(T >= 0 && k >= 1 && k <= DECOMOE_MAX_TOPK, "dispatch: bad T=%lld or k=%d", (long long)T, k);
  DM_ARG_CHECK(K >= 1 && K <= DECOMOE_MAX_E, "dispatch: K=%d outside [1, %d]", K, DECOMOE_MAX_E);
  DM_ARG_CHECK(dtype == DECOMOE_BF16 || dtype == DECOMOE_F32, "dispatch: bad dtype");
  DM_ARG_CHECK(counts && offsets, "dispatch: counts/offsets null");
  const int64_t N = T * k;
  DM_ARG_CHECK(N < 0x7fffffffLL, "dispatch: T*k too large");
  DM_ARG_CHECK(N > 0 || mblocks == 0, "dispatch: a deferred mass needs routed pairs");
  if (N == 0) {
    DM_CUDA_CHECK(cudaMemsetAsync(counts, 0, sizeof(int32_t) * K, s));
    DM_CUDA_CHECK(cudaMemsetAsync(offsets, 0, sizeof(int32_t) * (K + 1), s));
    return DECOMOE_OK;
  }
  DM_ARG_CHECK(topk_idx && perm_token && inv_slot, "dispatch: null index array");
  const size_t row_bytes = static_cast<size_t>(d) * dtype_bytes(dtype);
  if (x_perm != nullptr) {
    DM_ARG_CHECK(x != nullptr && d > 0, "dispatch: x null or d <= 0");
    DM_ARG_CHECK(row_bytes % 16 == 0 && aligned16(x) && aligned16(x_perm),
                 "dispatch: rows must be 16-byte multiples and 16-byte aligned");
  }
  if (ws == nullptr || ws_bytes < decomoe_dispatch_workspace_bytes(T, k, K)) {
    set_error("dispatch: workspace needs %zu bytes", decomoe_dispatch_workspace_bytes(T, k, K));
    return DECOMOE_ERR_WORKSPACE;
  }
  const int ntiles = static_cast<int>((N + DSP_TILE - 1) / DSP_TILE);
  int32_t* tile_hist = static_cast<int32_t*>(ws);
  const bool gather_here = ntiles == 1 && x_perm != nullptr && static_cast<size_t>(N) * row_bytes <= 64 * 1024;
  if (gather_here || (x_perm == nullptr && N <= 32)) {
    // one tile with few rows to copy: count, scan, rank and copy in one block.
    // Without the copy only as many pairs as one warp has lanes: the cluster below
    // takes 2.5 us for 8 and for 32 pairs of 128 experts, this 2.2 and 2.4, but 2.6
    // and 4.2 for 128 pairs, 2.8 and 4.2 for 512
    DM_CUDA_CHECK(launch_pdl(k_dispatch_scatter<true>, dim3(1 + mblocks), dim3(DSP_THREADS), 0, s, topk_idx, N,
                             k, K, static_cast<const int32_t*>(nullptr), 1, counts, offsets, perm_token, inv_slot,
                             status_dev, static_cast<const uint4*>(x), static_cast<int>(row_bytes / 16),
                             static_cast<uint4*>(x_perm), mf));
    return DECOMOE_OK;
  }
  if (N <= DSC_MAX_PAIRS) {
    const int P = static_cast<int>((N + DSC_CTAS * DSP_WARPS * 32 - 1) / (DSC_CTAS * DSP_WARPS * 32)) * 32;
    auto kern = P <= 64 ? k_dispatch_cluster<2> : P <= 128 ? k_dispatch_cluster<4> : k_dispatch_cluster<DSC_MAX_ROUNDS>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(DSC_CTAS + (mblocks + DSC_CTAS - 1) / DSC_CTAS * DSC_CTAS);
    cfg.blockDim = dim3(DSP_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = DSC_CTAS;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = pdl_enabled(cfg.gridDim.x) ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    DM_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, topk_idx, N, k, K, P, counts, offsets, perm_token, inv_slot,
                                     status_dev, mf));
  } else {
    DM_CUDA_CHECK(launch_pdl(k_dispatch_hist, dim3(ntiles + mblocks), dim3(DSP_THREADS), 0, s, topk_idx, N, K,
                             tile_hist, status_dev, ntiles, mf));
    DM_CUDA_CHECK(launch_pdl(k_dispatch_scatter<false>, dim3(ntiles), dim3(DSP_THREADS), 0, s, topk_idx, N, k, K,
                             static_cast<const int32_t*>(tile_hist), ntiles, counts, offsets, perm_token, inv_slot,
                             static_cast<int32_t*>(nullptr), static_cast<const uint4*>(nullptr), 0,
                             static_cast<uint4*>(nullptr), MassFinish{}));
  }
  if (x_perm != nullptr) DM_RET(launch_gather_rows(x, perm_token, offsets, K, row_bytes, N, x_perm, s));
  return DECOMOE_OK;
}

int launch_gather_rows(const void* x, const int32_t* perm_token, const int32_t* offsets, int K, size_t row_bytes,
                       int64_t N, void* x_perm, cudaStream_t s) {
  const int vec = static_cast<int>(row_bytes / 16);
  int blocks = static_cast<int>(std::min<int64_t>((N * 32 + 255) / 256, sm_count() * 8LL));
  if (blocks < 1) blocks = 1;
  DM_CUDA_CHECK(launch_pdl(k_gather_rows, dim3(blocks), dim3(256), 0, s, static_cast<const uint4*>(x), perm_token,
                           offsets, K, vec, static_cast<uint4*>(x_perm)));
  return DECOMOE_OK;
}

}  // namespace decomoe

// ---------------------------------------------------------------------------
// Allocation-free dispatch.
//
// Some callers cannot hand the library a workspace: their runtime owns every
// device allocation up front (a serving engine that carves all of HBM into a
// fixed arena at start-up and forbids any later cudaMalloc, because cudaMalloc
// can synchronise the device and fragment that arena). For them this entry
// point keeps the per-tile histograms in a fixed array that is part of the
// library image itself, so the call needs nothing beyond its inputs and
// outputs.
//
// Limit: ceil(T*k / 1024) * K <= DECOMOE_NOALLOC_DISPATCH_SCRATCH_INTS
// (65536 int32 = 256 KiB, e.g. T*k up to 524288 pairs at K = 128). Every GPU
// that loads the library holds this array until the process exits.
// ---------------------------------------------------------------------------
namespace decomoe {

static __device__ __align__(256) int32_t g_noalloc_dispatch_scratch[DECOMOE_NOALLOC_DISPATCH_SCRATCH_INTS];

// Device address of the array, looked up once per device ordinal (host code
// cannot use the symbol itself as a device pointer). The cached address
// belongs to the device's primary context as it was at the first call: it is
// not looked up again after cudaDeviceReset. The first call on a device must
// not be made while `s` is being captured into a graph.
static int noalloc_scratch_ptr(int32_t** out, cudaStream_t s) {
  static std::mutex mu;
  static int32_t* ptrs[64] = {nullptr};
  int dev = 0;
  DM_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("dispatch_noalloc: device ordinal %d out of range", dev);
    return DECOMOE_ERR_UNSUPPORTED;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (ptrs[dev] == nullptr) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    DM_CUDA_CHECK(cudaStreamIsCapturing(s, &cs));
    if (cs != cudaStreamCaptureStatusNone) {
      set_error("dispatch_noalloc: the first call on device %d is inside a stream capture; make one call on "
                "this device before capturing", dev);
      return DECOMOE_ERR_INVALID_ARG;
    }
    void* p = nullptr;
    DM_CUDA_CHECK(cudaGetSymbolAddress(&p, g_noalloc_dispatch_scratch));
    ptrs[dev] = static_cast<int32_t*>(p);
  }
  *out = ptrs[dev];
  return DECOMOE_OK;
}

}  // namespace decomoe

extern "C" int decomoe_dispatch_noalloc(const int32_t* topk_idx, int64_t T, int k, int K, const void* x, int d,
                                        int dtype, int32_t* counts, int32_t* offsets, int32_t* perm_token,
                                        int32_t* inv_slot, void* x_perm, int32_t* status_dev,
                                        decomoe_stream_t stream) {
  using namespace decomoe;
  clear_error();
  DM_ARG_CHECK(T >= 0 && k >= 1 && k <= DECOMOE_MAX_TOPK, "dispatch_noalloc: bad T=%lld or k=%d", (long long)T, k);
  DM_ARG_CHECK(K >= 1 && K <= DECOMOE_MAX_E, "dispatch_noalloc: K=%d outside [1, %d]", K, DECOMOE_MAX_E);
  DM_ARG_CHECK(dtype == DECOMOE_BF16 || dtype == DECOMOE_F32, "dispatch_noalloc: bad dtype");
  DM_ARG_CHECK(counts && offsets, "dispatch_noalloc: counts/offsets null");
  const int64_t N = T * k;
  DM_ARG_CHECK(N < 0x7fffffffLL, "dispatch_noalloc: T*k too large");
  const int64_t ntiles64 = (N + DSP_TILE - 1) / DSP_TILE;
  DM_ARG_CHECK(ntiles64 * K <= DECOMOE_NOALLOC_DISPATCH_SCRATCH_INTS,
               "dispatch_noalloc: ceil(T*k/%d)*K = %lld exceeds the fixed scratch of %d entries; "
               "use decomoe_dispatch with a workspace", DSP_TILE, (long long)(ntiles64 * K),
               DECOMOE_NOALLOC_DISPATCH_SCRATCH_INTS);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (N == 0) {
    DM_CUDA_CHECK(cudaMemsetAsync(counts, 0, sizeof(int32_t) * K, s));
    DM_CUDA_CHECK(cudaMemsetAsync(offsets, 0, sizeof(int32_t) * (K + 1), s));
    return DECOMOE_OK;
  }
  DM_ARG_CHECK(topk_idx && perm_token && inv_slot, "dispatch_noalloc: null index array");
  const size_t row_bytes = static_cast<size_t>(d) * dtype_bytes(dtype);
  if (x_perm != nullptr) {
    DM_ARG_CHECK(x != nullptr && d > 0, "dispatch_noalloc: x null or d <= 0");
    DM_ARG_CHECK(row_bytes % 16 == 0 && aligned16(x) && aligned16(x_perm),
                 "dispatch_noalloc: rows must be 16-byte multiples and 16-byte aligned");
  }
  int32_t* tile_hist = nullptr;
  DM_RET(noalloc_scratch_ptr(&tile_hist, s));
  // k_dispatch_hist writes every entry the scatter pass reads, so nothing
  // left in the array by an earlier call is ever used.
  const int ntiles = static_cast<int>(ntiles64);
  DM_CUDA_CHECK(launch_pdl(k_dispatch_hist, dim3(ntiles), dim3(DSP_THREADS), 0, s, topk_idx, N, K, tile_hist,
                           status_dev, ntiles, MassFinish{}));
  k_dispatch_scatter<false><<<ntiles, DSP_THREADS, 0, s>>>(topk_idx, N, k, K, tile_hist, ntiles, counts, offsets,
                                                    perm_token, inv_slot);
  DM_LAUNCH_CHECK("k_dispatch_scatter");
  if (x_perm != nullptr) DM_RET(launch_gather_rows(x, perm_token, offsets, K, row_bytes, N, x_perm, s));
  return DECOMOE_OK;
}
