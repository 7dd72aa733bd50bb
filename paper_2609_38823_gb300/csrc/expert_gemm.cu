// Grouped expert GEMMs of the prefix-MoE layer (DecoMoE Algorithm 2: evaluate
// only the first K physically contiguous expert MLPs; gate, up and down
// matmuls, Appendix C_expert = 6Kdm) and the bf16 router projection.
//
// bf16, many rows: the tcgen05 kernel on pairs of SMs (ffn_pair.cuh).
// bf16, few rows per expert (decode): the weights-stationary tcgen05 kernel
// k_moe_ws (expert weights as M, the expert's tokens as N) and its one-launch
// form k_ffn_ws. Router: k_router_tc (router rows as M, tokens as N).
// f32: CUDA-core kernels (exact fp32 products, fp32 accumulation).
#include <atomic>
#include <mutex>

#include <cudaTypedefs.h>

#include "decomoe_internal.cuh"
#include "simt_rows.cuh"

// Kernel choice for the bf16 expert GEMMs: the weights-stationary kernels when
// the average expert gets at most DECOMOE_WS_MAX_AVG_ROWS rows (decode sizes:
// every tile streams its own weight slice), the pair kernel otherwise (prefill:
// faster when many rows share an expert's weights).
#ifndef DECOMOE_WS_MAX_AVG_ROWS
#define DECOMOE_WS_MAX_AVG_ROWS 8
#endif

namespace decomoe {

// ------------------------------------------------------------------ TMA maps
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 2-D bf16 tensor [outer, inner] row-major; box = box_outer rows x box_inner
// columns (64 -> 128-byte swizzle, 32 -> 64-byte swizzle), zero fill out of
// bounds.
int make_tmap_bf16(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer,
                          uint32_t box_outer, uint32_t box_inner) {
  auto fn = encode_fn();
  if (fn == nullptr) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return DECOMOE_ERR_CUDA;
  }
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapSwizzle sw = box_inner == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                  estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed (%d): inner=%llu outer=%llu box=%ux%u", (int)r,
              (unsigned long long)inner, (unsigned long long)outer, box_outer, box_inner);
    return DECOMOE_ERR_CUDA;
  }
  return DECOMOE_OK;
}

// 3-D bf16 tensor, dims[0] innermost (contiguous), byte strides of dims 1 and
// 2, box[0] = 64 elements (128-byte swizzle); zero fill out of bounds.
int make_tmap_bf16_3d(CUtensorMap* m, const void* base, const uint64_t dims[3], const uint64_t strides[2],
                      const uint32_t box[3]) {
  auto fn = encode_fn();
  if (fn == nullptr) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return DECOMOE_ERR_CUDA;
  }
  cuuint64_t d[3] = {dims[0], dims[1], dims[2]};
  cuuint64_t st[2] = {strides[0], strides[1]};
  cuuint32_t bx[3] = {box[0], box[1], box[2]};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), d, st, bx, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled (3-D) failed (%d): dims=%llu x %llu x %llu box=%u x %u x %u", (int)r,
              (unsigned long long)dims[0], (unsigned long long)dims[1], (unsigned long long)dims[2], box[0], box[1],
              box[2]);
    return DECOMOE_ERR_CUDA;
  }
  return DECOMOE_OK;
}

// ------------------------------------------------------------------ tile order
// Work item -> (group, M-tile inside the group, N-tile). M-tiles are visited
// alternately from the two ends of the group-ordered list (first, last,
// second, second-to-last, ...), each with all its N-tiles back to back. With
// experts ordered by routed mass, the front holds large experts whose weight
// tiles are shared by many M-tiles (L2 / tensor bound) and the back small
// experts whose weights stream from HBM once; mixing them in every wave keeps
// both HBM and the tensor pipes busy instead of running the two phases one
// after the other.
__device__ __forceinline__ void tile_coords(int tile, int NT, const int* s_mt, int G, int& grp, int& mt,
                                            int& nb) {
  const int mtot = s_mt[G];
  const int j = tile / NT;
  nb = tile - j * NT;
  const int mtg = (j & 1) ? (mtot - 1 - (j >> 1)) : (j >> 1);
  int lo = 0, hi = G - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (s_mt[mid] <= mtg)
      lo = mid;
    else
      hi = mid - 1;
  }
  grp = lo;
  mt = mtg - s_mt[lo];
}

}  // namespace decomoe
#include "ffn_pair.cuh"
namespace decomoe {

// ------------------------------------------------------------------ tensor-core router
// logits[t, e] = sum_k x[t, k] w_r[e, k] (+ bias[e]) with router rows as M (128
// per tile), BN tokens as N and the k loop split into KS slices: work item =
// (128 router rows, BN tokens, slice). Slice s runs k-blocks [s KB, (s + 1) KB)
// and writes its partial sums to out + s * split_stride without the bias; the
// caller adds the slices. Persistent, one CTA per SM: warp 0 streams both
// operands by TMA through an eight-stage ring, warp 1 issues the products,
// eight epilogue warps (two per 32-lane TMEM quarter) store the transposed
// accumulator. Bound by latency up to 4096 tokens, by reading x above. With the
// slices' reduction, d = 2048, E = 128 (the shared GEMM kernel before -> this):
// 131 tokens 7.2 -> 5.7 us, 2048 9.7 -> 8.0, 16384 20.3 -> 15.1.
constexpr int RT_BM = 128, RT_BK = 64, RT_STAGES = 8, RT_EW = 8;
template <int BN>
struct RtCfg {
  static constexpr int A_BYTES = RT_BM * RT_BK * 2;
  static constexpr int B_BYTES = BN * RT_BK * 2;
  static constexpr int ACC_COLS = BN < 32 ? 32 : BN;  // tensor-memory columns per accumulator
  static constexpr int NBARS = 2 * RT_STAGES + 5;
  static constexpr size_t SMEM = 1024 + static_cast<size_t>(RT_STAGES) * (A_BYTES + B_BYTES) + NBARS * 8 + 16;
};
struct RouterArgs {
  int E, n, npad;        // router rows, tokens, tokens rounded up to BN
  int kdim;
  float* out;            // [n, E], slice s at + s * split_stride
  int64_t split_stride;
  const float* bias;     // KS == 1 only
  int32_t* status;
  uint64_t limit_ns;
};

template <int BN, int KS>
__global__ void __launch_bounds__(64 + 32 * RT_EW, 1)
    k_router_tc(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
                const RouterArgs g) {
  using C = RtCfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  uint8_t* smem = smem_raw + pad;
  const uint32_t sA = raw + pad;
  const uint32_t sB = sA + RT_STAGES * C::A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RT_STAGES * (C::A_BYTES + C::B_BYTES));
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(bars + C::NBARS);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars);
  auto FULL = [&](int s) { return bar0 + 8u * s; };
  auto EMPTY = [&](int s) { return bar0 + 8u * (RT_STAGES + s); };
  auto TFULL = [&](int a) { return bar0 + 8u * (2 * RT_STAGES + a); };
  auto TEMPTY = [&](int a) { return bar0 + 8u * (2 * RT_STAGES + 2 + a); };
  const uint32_t DRAIN = bar0 + 8u * (2 * RT_STAGES + 4);

  if (threadIdx.x == 0) {
    *s_abort = 0;
    for (int s = 0; s < RT_STAGES; ++s) {
      mbar_init(FULL(s), 1);
      mbar_init(EMPTY(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(TFULL(a), 1);
      mbar_init(TEMPTY(a), 32 * RT_EW);
    }
    mbar_init(DRAIN, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(s_tmem)), 2 * C::ACC_COLS);
    tmem_relinquish();
  }
  // wait for the earlier kernels' results; the next kernel is released only
  // at the end (its CTAs would otherwise sit resident through this one)
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  const int MT = g.E / RT_BM, total = MT * (g.npad / BN) * KS;
  const int KB = g.kdim / RT_BK / KS;  // k-blocks per work item

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (lane 0)
    if (lane == 0) {
      tma_prefetch_desc(&tma_a);
      tma_prefetch_desc(&tma_b);
      int stage = 0;
      uint32_t ph = 0;
      bool ok = true;
      uint32_t armed = 0, armed_ph = 0;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        const int row0 = t / KS % MT * RT_BM, col0 = t / KS / MT * BN, k0 = t % KS * KB;
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(EMPTY(stage), ph ^ 1u, g.limit_ns, s_abort)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(FULL(stage), C::A_BYTES + C::B_BYTES);
          tma_load_2d(sA + stage * C::A_BYTES, &tma_a, FULL(stage), (k0 + kb) * RT_BK, row0);
          tma_load_2d(sB + stage * C::B_BYTES, &tma_b, FULL(stage), (k0 + kb) * RT_BK, col0);
          armed |= 1u << stage;
          armed_ph = (armed_ph & ~(1u << stage)) | (ph << stage);
          if (++stage == RT_STAGES) {
            stage = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {
        *s_abort = 1;
        report_status(g.status, DECOMOE_ERR_TIMEOUT);
        // let every copy this thread started land before the CTA can exit
        int no_abort = 0;
        for (int s = 0; s < RT_STAGES; ++s)
          if ((armed >> s) & 1u) mbar_wait(FULL(s), (armed_ph >> s) & 1u, g.limit_ns, &no_abort);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (whole warp, one elected thread issues)
    constexpr uint32_t IDESC = idesc_bf16_f32(RT_BM, BN);
    const bool leader = elect_one();
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true, issued = false;
    int n = 0;
    for (int t = blockIdx.x; ok && t < total; t += gridDim.x, ++n) {
      const int acc = n & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(TEMPTY(acc), ((n >> 1) & 1) ^ 1u, g.limit_ns, s_abort))) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t dt = tmem_base + static_cast<uint32_t>(acc * C::ACC_COLS);
      for (int kb = 0; kb < KB; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(FULL(stage), ph, g.limit_ns, s_abort))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t ad = smem_desc_kmajor<RT_BK>(sA + stage * C::A_BYTES);
        const uint64_t bd = smem_desc_kmajor<RT_BK>(sB + stage * C::B_BYTES);
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < RT_BK / 16; ++kk)
            tc_mma_f16(dt, ad + 2u * kk, bd + 2u * kk, IDESC, (kb | kk) != 0 ? 1u : 0u);
          tc_commit(EMPTY(stage));
          if (kb == KB - 1) tc_commit(TFULL(acc));
        }
        issued = true;
        if (++stage == RT_STAGES) {
          stage = 0;
          ph ^= 1u;
        }
      }
    }
    if (!ok && leader) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
      if (issued) {
        int no_abort = 0;
        tc_commit(DRAIN);
        mbar_wait(DRAIN, 0, g.limit_ns, &no_abort);
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------ epilogue: lane = router row
    const int q = warp & 3;          // TMEM lanes [32q, 32q + 32)
    const int wp = (warp - 2) >> 2;  // which of the quarter's two warps
    bool ok = true;
    int n = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++n) {
      const int e = t / KS % MT * RT_BM + q * 32 + lane, n0 = t / KS / MT * BN;
      const int acc = n & 1;
      // decided by the whole warp: the tensor-memory loads below are a warp's
      if (!__all_sync(0xffffffffu, mbar_wait(TFULL(acc), (n >> 1) & 1, g.limit_ns, s_abort))) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t tb =
          tmem_base + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(acc * C::ACC_COLS);
      float* out = g.out + static_cast<int64_t>(t % KS) * g.split_stride + e;
      const float bv = KS == 1 && g.bias != nullptr ? g.bias[e] : 0.f;
      constexpr int CH = BN < 32 ? BN : 32;
#pragma unroll 1
      for (int c0 = CH * wp; c0 < BN; c0 += 2 * CH) {
        uint32_t r[CH];
        if constexpr (CH == 16)
          tmem_ld16(tb + c0, r);
        else
          tmem_ld32(tb + c0, r);
        tc_wait_ld();
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (n0 + c0 + c < g.n) out[static_cast<int64_t>(n0 + c0 + c) * g.E] = __uint_as_float(r[c]) + bv;
      }
      tc_fence_before();
      mbar_arrive(TEMPTY(acc));
    }
    if (!ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
    }
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 2 * C::ACC_COLS);
  }
}

// Logits (KS == 1, with the bias) or KS slices of partial sums, T * E apart.
template <int BN, int KS>
static int launch_router_kernel(const void* x, const void* w_r, const float* bias, int64_t T, int d, int E, float* out,
                                int32_t* status, cudaStream_t s) {
  using C = RtCfg<BN>;
  static_assert(C::SMEM <= 232448, "shared memory budget");
  CUtensorMap ta, tb;
  DM_RET(make_tmap_bf16(&ta, w_r, static_cast<uint64_t>(d), static_cast<uint64_t>(E), RT_BM, RT_BK));
  DM_RET(make_tmap_bf16(&tb, x, static_cast<uint64_t>(d), static_cast<uint64_t>(T), BN, RT_BK));
  RouterArgs g;
  g.E = E;
  g.n = static_cast<int>(T);
  g.npad = static_cast<int>((T + BN - 1) / BN) * BN;
  g.kdim = d;
  g.out = out;
  g.split_stride = T * E;
  g.bias = bias;
  g.status = status;
  g.limit_ns = static_cast<uint64_t>(wait_limit_ns());
  auto kern = k_router_tc<BN, KS>;
  DM_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(C::SMEM)));
  const int64_t total = static_cast<int64_t>(E / RT_BM) * (g.npad / BN) * KS;
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(sm_count(), total)));
  DM_CUDA_CHECK(launch_pdl(kern, dim3(grid), dim3(64 + 32 * RT_EW), C::SMEM, s, ta, tb, g));
  return DECOMOE_OK;
}

// ------------------------------------------------------------------ weights-stationary grouped GEMM
// D[w, t] = sum_k W[e][wrow0 + w, k] * X[row0 + t, k]: the expert's weight rows
// are the M operand (128 per tile, always full) and its tokens the N operand
// (up to 256 per tile, MMA width rounded up to 16). No M padding, so a ragged,
// skewed expert population costs only what it routes; small experts (and the
// decode sizes) become pure weight streaming with every tile reading its own
// 128-row weight slice once. Roles: TMA warp, MMA warp, four epilogue warps;
// double-buffered 256-column TMEM accumulators.
//
// Tiles: per expert e, (wrows / 128) weight blocks x ceil(n_e / 256) token
// chunks, chunk innermost (consecutive tiles share a weight block, so it is
// read from HBM once and from L2 after); the global list is visited
// alternately from both ends (tile_coords).
//
// SwiGLU epilogue: with the 64-row gate/up interleave a weight block holds 64
// gate rows (TMEM lanes 0..63) and the 64 up rows of the same features (lanes
// 64..127). The warps owning lanes 64..127 pass their up values through a
// small double-buffered shared-memory exchange to the warps owning the gate
// lanes of the same features, which write h.
struct WsArgs {
  const int32_t* offsets;  // [G + 1] token row offsets per expert
  int G;                   // experts [0, G)
  int rows;                // token rows of the activation tensor
  int wrows;               // weight rows per expert (2m gate/up, d down)
  int kdim;
  void* out;
  int64_t out_ld;
  int32_t* status;
  uint64_t limit_ns;
  const int32_t* b_rows;  // GATHER_B: token row r is row b_rows[r] of the activation tensor
};

#ifndef DECOMOE_WS_BOX
#define DECOMOE_WS_BOX 32
#endif
constexpr int WS_BM = 128, WS_BK = 64, WS_BOX = DECOMOE_WS_BOX;

// BN: token chunk (the MMA's N), one chunk per (expert, weight block) tile
// when an expert has at most BN rows; smaller chunks leave shared memory for
// a deeper weight-streaming ring.
template <int STAGES, bool SWIGLU, int BN = 256>
struct WsCfg {
  static constexpr int WS_BN = BN;
  static constexpr int A_BYTES = WS_BM * WS_BK * 2;
  static constexpr int B_BYTES = WS_BN * WS_BK * 2;
  static constexpr int BOX_BYTES = WS_BOX * WS_BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 2 * WS_BN;
  static constexpr int MAXG = DECOMOE_MAX_E;
  static constexpr int NBARS = 2 * STAGES + 5;
  static constexpr int XCH_BYTES = SWIGLU ? 2 * 2 * 32 * 32 * 4 : 0;  // up values, double-buffered
  static constexpr int OUT_COLS = SWIGLU ? WS_BM / 2 : WS_BM;            // output features per tile
  static constexpr int STILE_BYTES = 2 * 32 * OUT_COLS * 2;              // [2][32 tokens][OUT_COLS] bf16
  static constexpr size_t SMEM = 1024 + static_cast<size_t>(STAGES) * STAGE_BYTES + XCH_BYTES + STILE_BYTES +
                                 NBARS * 8 + 2 * (MAXG + 1) * 4 + 16;
};

// Most stages of a WsCfg<., SWIGLU, BN> that fit the shared-memory budget.
template <bool SWIGLU, int BN>
constexpr int ws_max_stages() {
  constexpr size_t fixed = WsCfg<1, SWIGLU, BN>::SMEM - WsCfg<1, SWIGLU, BN>::STAGE_BYTES - 2 * 8;
  constexpr size_t per = WsCfg<1, SWIGLU, BN>::STAGE_BYTES + 2 * 8;
  constexpr int n = static_cast<int>((232448 - fixed) / per);
  return n > 12 ? 12 : n;
}

struct WsTile {
  int g, wb, row0, ntok;
};

template <int WS_BN>
__device__ __forceinline__ WsTile ws_tile(int t, int total, const int* s_tt, const int* s_off, int G, int nwb) {
  const int tp = (t & 1) ? (total - 1 - (t >> 1)) : (t >> 1);
  int lo = 0, hi = G - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (s_tt[mid] <= tp)
      lo = mid;
    else
      hi = mid - 1;
  }
  WsTile r;
  r.g = lo;
  const int n = s_off[lo + 1] - s_off[lo];
  const int nch = (n + WS_BN - 1) / WS_BN;
  const int local = tp - s_tt[lo];
  r.wb = local / nch;
  const int c = local - r.wb * nch;
  r.row0 = s_off[lo] + c * WS_BN;
  r.ntok = min(WS_BN, n - c * WS_BN);
  return r;
}


template <bool SWIGLU, int STAGES, bool GATHER_B = false, int BN = 256>
__global__ void __launch_bounds__(192, 1)
    k_moe_ws(const __grid_constant__ CUtensorMap tma_w, const __grid_constant__ CUtensorMap tma_x,
             const WsArgs g) {
  using C = WsCfg<STAGES, SWIGLU, BN>;
  constexpr int WS_BN = BN;
  __shared__ int s_brow[GATHER_B ? WS_BN : 1];
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  uint8_t* smem = smem_raw + pad;
  const uint32_t sA = raw + pad;
  const uint32_t sB = sA + STAGES * C::A_BYTES;
  float* xch = reinterpret_cast<float*>(smem + STAGES * C::STAGE_BYTES);
  __nv_bfloat16* stile = reinterpret_cast<__nv_bfloat16*>(smem + STAGES * C::STAGE_BYTES + C::XCH_BYTES);
  uint64_t* bars =
      reinterpret_cast<uint64_t*>(smem + STAGES * C::STAGE_BYTES + C::XCH_BYTES + C::STILE_BYTES);
  int* s_off = reinterpret_cast<int*>(bars + C::NBARS);
  int* s_tt = s_off + (C::MAXG + 1);
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(s_tt + (C::MAXG + 1));
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars);
#define FULL_BAR(s) (bar0 + 8u * (s))
#define EMPTY_BAR(s) (bar0 + 8u * (STAGES + (s)))
#define TFULL_BAR(a) (bar0 + 8u * (2 * STAGES + (a)))
#define TEMPTY_BAR(a) (bar0 + 8u * (2 * STAGES + 2 + (a)))
#define DRAIN_BAR (bar0 + 8u * (2 * STAGES + 4))

  const int G = g.G;
  const int nwb = g.wrows / WS_BM;
  if (threadIdx.x == 0) {
    *s_abort = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(FULL_BAR(s), 1);
      mbar_init(EMPTY_BAR(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(TFULL_BAR(a), 1);
      mbar_init(TEMPTY_BAR(a), 128);
    }
    mbar_init(DRAIN_BAR, 1);
    fence_mbar_init();
  }
  // wait for the earlier kernels' results; the next kernel is released only
  // at the end (its CTAs would otherwise sit resident through this one)
  pdl_wait();
  for (int i = threadIdx.x; i <= G; i += blockDim.x) s_off[i] = g.offsets[i];
  __syncthreads();
  if (warp == 2) {
    // s_tt[e] = first tile of expert e = sum over earlier experts of nwb * chunks
    const int per = (G + 31) / 32;
    int loc[8];
    int sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      loc[i] = 0;
      const int gi = lane * per + i;
      if (i < per && gi < G) {
        const int n = s_off[gi + 1] - s_off[gi];
        loc[i] = n > 0 ? ((n + WS_BN - 1) / WS_BN) * nwb : 0;
      }
      sum += loc[i];
    }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    int run = incl - sum;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int gi = lane * per + i;
      if (i < per && gi < G) s_tt[gi] = run;
      run += loc[i];
    }
    if (lane == 31) s_tt[G] = incl;
  }
  __syncthreads();
  const int total = s_tt[G];
  if (static_cast<int>(blockIdx.x) >= total) return;

  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(s_tmem)), C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  const int KB = g.kdim / WS_BK;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (lane 0
    // issues; with GATHER_B the warp first reads the tile's token row indices)
    if (lane == 0) {
      tma_prefetch_desc(&tma_w);
      tma_prefetch_desc(&tma_x);
    }
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    uint32_t armed = 0, armed_ph = 0;
    // an expert of one token chunk reads each weight block once: evict-first
    // in L2 (blocks of larger experts are re-read by their next chunks)
    const uint64_t pol_once = policy_evict_first();
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
      const WsTile T = ws_tile<WS_BN>(t, total, s_tt, s_off, G, nwb);
      const int wrow0 = T.g * g.wrows + T.wb * WS_BM;
      const bool once = s_off[T.g + 1] - s_off[T.g] <= WS_BN;
      int nload;       // TMA copies for B per k-block
      uint32_t bytes;  // bytes landing per stage
      if constexpr (GATHER_B) {
        for (int i = lane; i < WS_BN; i += 32)
          s_brow[i] = (i < T.ntok) ? g.b_rows[T.row0 + i] : 0;  // padding rows: any valid row, never stored
        __syncwarp();
        nload = (T.ntok + 3) / 4;
        bytes = C::A_BYTES + nload * 4 * WS_BK * 2;
      } else {
        nload = (T.ntok + WS_BOX - 1) / WS_BOX;
        bytes = C::A_BYTES + nload * C::BOX_BYTES;
      }
      if (lane == 0) {
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(EMPTY_BAR(stage), ph ^ 1u, g.limit_ns, s_abort)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(FULL_BAR(stage), bytes);
          if (once)
            tma_load_2d_hint(sA + stage * C::A_BYTES, &tma_w, FULL_BAR(stage), kb * WS_BK, wrow0, pol_once);
          else
            tma_load_2d(sA + stage * C::A_BYTES, &tma_w, FULL_BAR(stage), kb * WS_BK, wrow0);
          const uint32_t dB = sB + stage * C::B_BYTES;
          if constexpr (GATHER_B) {
            for (int i = 0; i < nload; ++i)
              tma_gather4(dB + i * 4 * WS_BK * 2, &tma_x, FULL_BAR(stage), kb * WS_BK, s_brow[4 * i],
                          s_brow[4 * i + 1], s_brow[4 * i + 2], s_brow[4 * i + 3]);
          } else {
            for (int i = 0; i < nload; ++i)
              tma_load_2d(dB + i * C::BOX_BYTES, &tma_x, FULL_BAR(stage), kb * WS_BK, T.row0 + i * WS_BOX);
          }
          armed |= 1u << stage;
          armed_ph = (armed_ph & ~(1u << stage)) | (ph << stage);
          if (++stage == STAGES) {
            stage = 0;
            ph ^= 1u;
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
    }
    if (lane == 0 && !ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
      int no_abort = 0;
      for (int s = 0; s < STAGES; ++s)
        if ((armed >> s) & 1u) mbar_wait(FULL_BAR(s), (armed_ph >> s) & 1u, g.limit_ns, &no_abort);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (whole warp, one elected thread issues)
    const bool leader = elect_one();
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true, issued = false;
    int it = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
      const WsTile T = ws_tile<WS_BN>(t, total, s_tt, s_off, G, nwb);
      const uint32_t idesc = idesc_bf16_f32(WS_BM, (T.ntok + 15) & ~15);
      const int acc = it & 1;
      const uint32_t aph = (it >> 1) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(TEMPTY_BAR(acc), aph ^ 1u, g.limit_ns, s_abort))) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t dt = tmem_base + static_cast<uint32_t>(acc * WS_BN);
      for (int kb = 0; kb < KB; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(FULL_BAR(stage), ph, g.limit_ns, s_abort))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t ad = smem_desc_kmajor<WS_BK>(sA + stage * C::A_BYTES);
        const uint64_t bd = smem_desc_kmajor<WS_BK>(sB + stage * C::B_BYTES);
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < WS_BK / 16; ++kk)
            tc_mma_f16(dt, ad + 2u * kk, bd + 2u * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          tc_commit(EMPTY_BAR(stage));
        }
        issued = true;
        if (++stage == STAGES) {
          stage = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      if (leader) tc_commit(TFULL_BAR(acc));
    }
    if (!ok && leader) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
      if (issued) {
        int no_abort = 0;
        tc_commit(DRAIN_BAR);
        mbar_wait(DRAIN_BAR, 0, g.limit_ns, &no_abort);
      }
    }
  } else if (warp >= 2) {
    // ------------------------------------------------ epilogue
    const int q = warp & 3;  // TMEM lanes [32q, 32q + 32)
    __nv_bfloat16* out = static_cast<__nv_bfloat16*>(g.out);
    int it = 0;
    int xpar = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
      const WsTile T = ws_tile<WS_BN>(t, total, s_tt, s_off, G, nwb);
      const int acc = it & 1;
      const uint32_t aph = (it >> 1) & 1;
      // a warp whose wait ran out (or that saw another role give up) loads and
      // stores nothing more, but goes on to the barriers, which have no limit
      // and which the other warps may have reached
      if (ok && !__all_sync(0xffffffffu, mbar_wait(TFULL_BAR(acc), aph, g.limit_ns, s_abort))) {
        ok = false;
        *s_abort = 1;
      }
      tc_fence_after();
      const uint32_t tb =
          tmem_base + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(acc * WS_BN);
      // Each 32-token chunk: accumulator columns -> registers -> (SwiGLU) ->
      // bf16 tile [32 tokens][OUT_COLS features] in shared memory -> 16-byte
      // row stores to out[token, feature]. Two named barriers per chunk over
      // the four epilogue warps; the exchange and tile buffers alternate.
      constexpr int OC = C::OUT_COLS;
      const int et = threadIdx.x - 64;  // 0..127 among the epilogue warps
      const int fbase = T.wb * OC;      // first output feature of this tile
#pragma unroll 1
      for (int c0 = 0; c0 < T.ntok; c0 += 32) {
        uint32_t r[32];
        if (ok) {
          tmem_ld32(tb + c0, r);
          tc_wait_ld();
        }
        __nv_bfloat16* st = stile + xpar * (32 * OC);
        if constexpr (SWIGLU) {
          const bool is_gate = q < 2;
          const int pr = q & 1;
          float* xb = xch + (xpar * 2 + pr) * 1024;  // [32 columns][32 lanes]
          if (ok && !is_gate) {
#pragma unroll
            for (int c = 0; c < 32; ++c) xb[c * 32 + lane] = __uint_as_float(r[c]);
          }
          named_bar_sync(1, 128);
          if (ok && is_gate) {
#pragma unroll
            for (int c = 0; c < 32; ++c)
              st[c * OC + pr * 32 + lane] = __float2bfloat16_rn(silu_f(__uint_as_float(r[c])) * xb[c * 32 + lane]);
          }
        } else if (ok) {
#pragma unroll
          for (int c = 0; c < 32; ++c) st[c * OC + q * 32 + lane] = __float2bfloat16_rn(__uint_as_float(r[c]));
        }
        named_bar_sync(1, 128);
        const int nc = min(32, T.ntok - c0);
        constexpr int VPR = OC / 8;  // 16-byte vectors per token row
#pragma unroll
        for (int v = et; v < 32 * VPR; v += 128) {
          const int row = v / VPR, cv = v - row * VPR;
          if (ok && row < nc) {
            const uint4 val = *reinterpret_cast<const uint4*>(st + row * OC + cv * 8);
            *reinterpret_cast<uint4*>(out + static_cast<int64_t>(T.row0 + c0 + row) * g.out_ld + fbase + cv * 8) = val;
          }
        }
        xpar ^= 1;
      }
      tc_fence_before();
      mbar_arrive(TEMPTY_BAR(acc));
    }
    if (!ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
    }
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
#undef FULL_BAR
#undef EMPTY_BAR
#undef TFULL_BAR
#undef TEMPTY_BAR
#undef DRAIN_BAR
}

// ------------------------------------------------------------------ fused decode FFN
// Gate/up and down of the weights-stationary decode path in one persistent
// launch. Work items: every gate/up tile of k_moe_ws<true> first, then every
// down tile of k_moe_ws<false> (each list in k_moe_ws's order), handed out
// round robin. A down tile of expert e reads h rows that the gate/up tiles
// of e write, so after storing its h slice a gate/up tile bumps ready[e]
// (release), and a down tile first issues the loads of its own weight
// k-blocks (they depend on nothing), then waits until ready[e] counts all of
// e's gate/up tiles (acquire, bounded) before loading its h rows. CTAs whose
// first item is a down tile thus stream their weights while the gate/up
// tiles run, and no launch separates the two GEMMs. Deadlock-free with at
// most one CTA per SM and grid <= SMs: gate/up items never wait, and every
// CTA reaches its gate/up items before any down item. ready[] must be zero at
// launch (the layer's routing launch clears it).
struct WsFfnArgs {
  const int32_t* offsets;  // [G + 1] token row offsets per expert
  int G;
  int rows;
  int wrows1, kdim1;  // gate/up: 2m weight rows per expert, K = d
  int wrows2, kdim2;  // down: d weight rows per expert, K = m
  void* h;            // [rows, m] bf16, gate/up output and down input
  int64_t h_ld;
  void* y;  // [rows, d] bf16
  int64_t y_ld;
  int32_t* ready;  // [G] finished gate/up tiles per expert; zero at launch
  int32_t* status;
  uint64_t limit_ns;
};

template <int STAGES, int BN>
struct WsFfnCfg {
  static constexpr int A_BYTES = WS_BM * WS_BK * 2;
  static constexpr int B_BYTES = BN * WS_BK * 2;
  static constexpr int BOX_BYTES = WS_BOX * WS_BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 2 * BN;
  static constexpr int MAXG = DECOMOE_MAX_E;
  static constexpr int NBARS = 2 * STAGES + 5;
  static constexpr int XCH_BYTES = 2 * 2 * 32 * 32 * 4;   // SwiGLU up values, double-buffered
  static constexpr int STILE_BYTES = 2 * 32 * WS_BM * 2;  // [2][32 tokens][128 features] bf16
  static constexpr size_t SMEM = 1024 + static_cast<size_t>(STAGES) * STAGE_BYTES + XCH_BYTES + STILE_BYTES +
                                 NBARS * 8 + 3 * (MAXG + 1) * 4 + 16;
};

template <int BN>
constexpr int ffn_ws_max_stages() {
  constexpr size_t fixed = WsFfnCfg<1, BN>::SMEM - WsFfnCfg<1, BN>::STAGE_BYTES - 2 * 8;
  constexpr size_t per = WsFfnCfg<1, BN>::STAGE_BYTES + 2 * 8;
  constexpr int n = static_cast<int>((232448 - fixed) / per);
  return n > 12 ? 12 : n;
}


template <int STAGES, int BN>
__global__ void __launch_bounds__(192, 1)
    k_ffn_ws(const __grid_constant__ CUtensorMap tma_w1, const __grid_constant__ CUtensorMap tma_x1,
             const __grid_constant__ CUtensorMap tma_w2, const __grid_constant__ CUtensorMap tma_x2,
             const WsFfnArgs g) {
  using C = WsFfnCfg<STAGES, BN>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  uint8_t* smem = smem_raw + pad;
  const uint32_t sA = raw + pad;
  const uint32_t sB = sA + STAGES * C::A_BYTES;
  float* xch = reinterpret_cast<float*>(smem + STAGES * C::STAGE_BYTES);
  __nv_bfloat16* stile = reinterpret_cast<__nv_bfloat16*>(smem + STAGES * C::STAGE_BYTES + C::XCH_BYTES);
  uint64_t* bars =
      reinterpret_cast<uint64_t*>(smem + STAGES * C::STAGE_BYTES + C::XCH_BYTES + C::STILE_BYTES);
  int* s_off = reinterpret_cast<int*>(bars + C::NBARS);
  int* s_tt1 = s_off + (C::MAXG + 1);
  int* s_tt2 = s_tt1 + (C::MAXG + 1);
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(s_tt2 + (C::MAXG + 1));
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars);
#define FULL_BAR(s) (bar0 + 8u * (s))
#define EMPTY_BAR(s) (bar0 + 8u * (STAGES + (s)))
#define TFULL_BAR(a) (bar0 + 8u * (2 * STAGES + (a)))
#define TEMPTY_BAR(a) (bar0 + 8u * (2 * STAGES + 2 + (a)))
#define DRAIN_BAR (bar0 + 8u * (2 * STAGES + 4))

  const int G = g.G;
  const int nwb1 = g.wrows1 / WS_BM, nwb2 = g.wrows2 / WS_BM;
  if (threadIdx.x == 0) {
    *s_abort = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(FULL_BAR(s), 1);
      mbar_init(EMPTY_BAR(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(TFULL_BAR(a), 1);
      mbar_init(TEMPTY_BAR(a), 128);
    }
    mbar_init(DRAIN_BAR, 1);
    fence_mbar_init();
  }
  pdl_wait();
  for (int i = threadIdx.x; i <= G; i += blockDim.x) s_off[i] = g.offsets[i];
  __syncthreads();
  if (warp == 2 || warp == 3) {
    // s_tt1 / s_tt2[e] = first gate/up / down item of expert e
    const int nwb = warp == 2 ? nwb1 : nwb2;
    int* s_tt = warp == 2 ? s_tt1 : s_tt2;
    const int per = (G + 31) / 32;
    int loc[8];
    int sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      loc[i] = 0;
      const int gi = lane * per + i;
      if (i < per && gi < G) {
        const int n = s_off[gi + 1] - s_off[gi];
        loc[i] = n > 0 ? ((n + BN - 1) / BN) * nwb : 0;
      }
      sum += loc[i];
    }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    int run = incl - sum;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int gi = lane * per + i;
      if (i < per && gi < G) s_tt[gi] = run;
      run += loc[i];
    }
    if (lane == 31) s_tt[G] = incl;
  }
  __syncthreads();
  const int total1 = s_tt1[G], total2 = s_tt2[G];
  const int total = total1 + total2;
  if (static_cast<int>(blockIdx.x) >= total) return;

  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(s_tmem)), C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  // work item t -> (down?, tile)
  auto item = [&](int t, bool& dn) -> WsTile {
    dn = t >= total1;
    return dn ? ws_tile<BN>(t - total1, total2, s_tt2, s_off, G, nwb2) : ws_tile<BN>(t, total1, s_tt1, s_off, G, nwb1);
  };

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (lane 0)
    if (lane == 0) {
      tma_prefetch_desc(&tma_w1);
      tma_prefetch_desc(&tma_x1);
      tma_prefetch_desc(&tma_w2);
      tma_prefetch_desc(&tma_x2);
    }
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    uint32_t armed = 0, armed_ph = 0;
    // readiness of a down item, acquire-loaded one item ahead so that its
    // latency hides behind the current item's loads (stale values only send
    // an item down the wait path)
    auto flag_of = [&](int t) -> int {
      if (t < total1 || t >= total) return 0;
      bool d_;
      const WsTile U = item(t, d_);
      return ld_acquire_gpu(g.ready + U.g);
    };
    int flag_cur = lane == 0 ? flag_of(static_cast<int>(blockIdx.x)) : 0;
    const uint64_t pol_once = policy_evict_first();
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
      bool dn;
      const WsTile T = item(t, dn);
      const int flag = flag_cur;
      if (lane == 0) flag_cur = flag_of(t + static_cast<int>(gridDim.x));
      if (lane == 0) {
        const CUtensorMap* tw = dn ? &tma_w2 : &tma_w1;
        const CUtensorMap* tx = dn ? &tma_x2 : &tma_x1;
        const int wrow0 = T.g * (dn ? g.wrows2 : g.wrows1) + T.wb * WS_BM;
        // an expert of one token chunk reads each weight block once: evict-first
        const bool once = s_off[T.g + 1] - s_off[T.g] <= BN;
        const int KB = (dn ? g.kdim2 : g.kdim1) / WS_BK;
        const int nload = (T.ntok + WS_BOX - 1) / WS_BOX;
        const uint32_t bytes = C::A_BYTES + nload * C::BOX_BYTES;
        int pre = 0;  // k-blocks whose weights go out before the dependency is met
        const int need = ((s_off[T.g + 1] - s_off[T.g] + BN - 1) / BN) * nwb1;
        // already met: the ordinary pipeline, weights and h rows together
        const bool met = dn && flag >= need;
        if (met) fence_proxy_async_all();  // h, written by generic stores, read through the tensor map
        if (dn && !met) {
          pre = KB < STAGES ? KB : STAGES;
          const int st0 = stage;
          for (int kb = 0; kb < pre; ++kb) {
            if (!mbar_wait(EMPTY_BAR(stage), ph ^ 1u, g.limit_ns, s_abort)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(FULL_BAR(stage), bytes);
            if (once)
              tma_load_2d_hint(sA + stage * C::A_BYTES, tw, FULL_BAR(stage), kb * WS_BK, wrow0, pol_once);
            else
              tma_load_2d(sA + stage * C::A_BYTES, tw, FULL_BAR(stage), kb * WS_BK, wrow0);
            armed |= 1u << stage;
            armed_ph = (armed_ph & ~(1u << stage)) | (ph << stage);
            if (++stage == STAGES) {
              stage = 0;
              ph ^= 1u;
            }
          }
          if (ok) {
            // every gate/up item of expert T.g has stored its h slice
            const volatile int32_t* rp = g.ready + T.g;
            const uint64_t t0 = globaltimer_ns();
            while (*rp < need) {
              if (*s_abort || globaltimer_ns() - t0 > g.limit_ns) {
                ok = false;
                break;
              }
            }
            __threadfence();
            fence_proxy_async_all();  // the h rows, written by generic stores, read through the tensor map
          }
          if (ok) {
            int st = st0;
            for (int kb = 0; kb < pre; ++kb) {
              const uint32_t dB = sB + st * C::B_BYTES;
              for (int i = 0; i < nload; ++i)
                tma_load_2d(dB + i * C::BOX_BYTES, tx, FULL_BAR(st), kb * WS_BK, T.row0 + i * WS_BOX);
              if (++st == STAGES) st = 0;
            }
          }
        }
        for (int kb = pre; ok && kb < KB; ++kb) {
          if (!mbar_wait(EMPTY_BAR(stage), ph ^ 1u, g.limit_ns, s_abort)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(FULL_BAR(stage), bytes);
          if (once)
            tma_load_2d_hint(sA + stage * C::A_BYTES, tw, FULL_BAR(stage), kb * WS_BK, wrow0, pol_once);
          else
            tma_load_2d(sA + stage * C::A_BYTES, tw, FULL_BAR(stage), kb * WS_BK, wrow0);
          const uint32_t dB = sB + stage * C::B_BYTES;
          for (int i = 0; i < nload; ++i)
            tma_load_2d(dB + i * C::BOX_BYTES, tx, FULL_BAR(stage), kb * WS_BK, T.row0 + i * WS_BOX);
          armed |= 1u << stage;
          armed_ph = (armed_ph & ~(1u << stage)) | (ph << stage);
          if (++stage == STAGES) {
            stage = 0;
            ph ^= 1u;
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
    }
    if (lane == 0 && !ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
      // let the copies this thread started land before the CTA can exit (a
      // stage whose activation rows were never requested runs to the limit)
      int no_abort = 0;
      for (int s = 0; s < STAGES; ++s)
        if ((armed >> s) & 1u) mbar_wait(FULL_BAR(s), (armed_ph >> s) & 1u, g.limit_ns, &no_abort);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (whole warp, one elected thread issues:
    // against one lane of a divergent branch T=40 80.5 -> 76.9 us a layer, T=64 88.8 -> 85.2)
    const bool leader = elect_one();
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true, issued = false;
    int it = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
      bool dn;
      const WsTile T = item(t, dn);
      const int KB = (dn ? g.kdim2 : g.kdim1) / WS_BK;
      const uint32_t idesc = idesc_bf16_f32(WS_BM, (T.ntok + 15) & ~15);
      const int acc = it & 1;
      const uint32_t aph = (it >> 1) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(TEMPTY_BAR(acc), aph ^ 1u, g.limit_ns, s_abort))) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t dt = tmem_base + static_cast<uint32_t>(acc * BN);
      for (int kb = 0; kb < KB; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(FULL_BAR(stage), ph, g.limit_ns, s_abort))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t ad = smem_desc_kmajor<WS_BK>(sA + stage * C::A_BYTES);
        const uint64_t bd = smem_desc_kmajor<WS_BK>(sB + stage * C::B_BYTES);
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < WS_BK / 16; ++kk)
            tc_mma_f16(dt, ad + 2u * kk, bd + 2u * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          tc_commit(EMPTY_BAR(stage));
        }
        issued = true;
        if (++stage == STAGES) {
          stage = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      if (leader) tc_commit(TFULL_BAR(acc));
    }
    if (!ok && leader) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
      if (issued) {
        int no_abort = 0;
        tc_commit(DRAIN_BAR);
        mbar_wait(DRAIN_BAR, 0, g.limit_ns, &no_abort);
      }
    }
  } else if (warp >= 2) {
    // ------------------------------------------------ epilogue (4 warps)
    const int q = warp & 3;  // TMEM lanes [32q, 32q + 32)
    int it = 0;
    int xpar = 0;
    bool ok = true;
    const int et = threadIdx.x - 64;  // 0..127 among the epilogue warps
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
      bool dn;
      const WsTile T = item(t, dn);
      const int acc = it & 1;
      const uint32_t aph = (it >> 1) & 1;
      // as in k_moe_ws: after a wait that ran out, barriers only
      if (ok && !__all_sync(0xffffffffu, mbar_wait(TFULL_BAR(acc), aph, g.limit_ns, s_abort))) {
        ok = false;
        *s_abort = 1;
      }
      tc_fence_after();
      const uint32_t tb = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(acc * BN);
      // as k_moe_ws: 32-token chunks through a bf16 tile in shared memory;
      // gate/up items write silu(gate) * up to h (64 features per item),
      // down items write y (128 features per item)
      const int OC = dn ? WS_BM : WS_BM / 2;
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(dn ? g.y : g.h);
      const int64_t ld = dn ? g.y_ld : g.h_ld;
      const int fbase = T.wb * OC;
#pragma unroll 1
      for (int c0 = 0; c0 < T.ntok; c0 += 32) {
        uint32_t r[32];
        if (ok) {
          tmem_ld32(tb + c0, r);
          tc_wait_ld();
        }
        __nv_bfloat16* st = stile + xpar * (32 * WS_BM);
        if (!dn) {
          const bool is_gate = q < 2;
          const int pr = q & 1;
          float* xb = xch + (xpar * 2 + pr) * 1024;  // [32 columns][32 lanes]
          if (ok && !is_gate) {
#pragma unroll
            for (int c = 0; c < 32; ++c) xb[c * 32 + lane] = __uint_as_float(r[c]);
          }
          named_bar_sync(1, 128);
          if (ok && is_gate) {
#pragma unroll
            for (int c = 0; c < 32; ++c)
              st[c * OC + pr * 32 + lane] = __float2bfloat16_rn(silu_f(__uint_as_float(r[c])) * xb[c * 32 + lane]);
          }
        } else if (ok) {
#pragma unroll
          for (int c = 0; c < 32; ++c) st[c * OC + q * 32 + lane] = __float2bfloat16_rn(__uint_as_float(r[c]));
        }
        named_bar_sync(1, 128);
        const int nc = min(32, T.ntok - c0);
        const int VPR = OC / 8;  // 16-byte vectors per token row
        for (int v = et; v < 32 * VPR; v += 128) {
          const int row = v / VPR, cv = v - row * VPR;
          if (ok && row < nc) {
            const uint4 val = *reinterpret_cast<const uint4*>(st + row * OC + cv * 8);
            *reinterpret_cast<uint4*>(out + static_cast<int64_t>(T.row0 + c0 + row) * ld + fbase + cv * 8) = val;
          }
        }
        xpar ^= 1;
      }
      tc_fence_before();
      mbar_arrive(TEMPTY_BAR(acc));
      if (!dn) {
        // this item's h slice is stored (unless a warp gave up): publish it to the
        // down items of T.g
        fence_proxy_async_all();
        if (named_bar_all(1, 128, ok) && et == 0) {
          __threadfence();
          atomicAdd(g.ready + T.g, 1);
        }
      }
    }
    if (!ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
    }
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
#undef FULL_BAR
#undef EMPTY_BAR
#undef TFULL_BAR
#undef TEMPTY_BAR
#undef DRAIN_BAR
}

template <int STAGES, int BN>
static int launch_ffn_ws_bn(const void* x_perm, int rows, int d, int m, const void* w_gu, const void* w_down,
                            const int32_t* offsets, int G, void* h, void* y, int32_t* ready, int32_t* status,
                            cudaStream_t s) {
  using C = WsFfnCfg<STAGES, BN>;
  CUtensorMap tw1, tx1, tw2, tx2;
  DM_RET(make_tmap_bf16(&tw1, w_gu, static_cast<uint64_t>(d), static_cast<uint64_t>(G) * 2 * m, WS_BM, WS_BK));
  DM_RET(make_tmap_bf16(&tx1, x_perm, static_cast<uint64_t>(d), static_cast<uint64_t>(rows), WS_BOX, WS_BK));
  DM_RET(make_tmap_bf16(&tw2, w_down, static_cast<uint64_t>(m), static_cast<uint64_t>(G) * d, WS_BM, WS_BK));
  DM_RET(make_tmap_bf16(&tx2, h, static_cast<uint64_t>(m), static_cast<uint64_t>(rows), WS_BOX, WS_BK));
  WsFfnArgs g;
  g.offsets = offsets;
  g.G = G;
  g.rows = rows;
  g.wrows1 = 2 * m;
  g.kdim1 = d;
  g.wrows2 = d;
  g.kdim2 = m;
  g.h = h;
  g.h_ld = m;
  g.y = y;
  g.y_ld = d;
  g.ready = ready;
  g.status = status;
  g.limit_ns = static_cast<uint64_t>(wait_limit_ns());
  auto kern = k_ffn_ws<STAGES, BN>;
  static_assert(C::SMEM <= 232448, "shared memory budget");
  static_assert(C::SMEM > 232448 / 2, "one CTA per SM: the dependency waits need every CTA resident");
  DM_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(C::SMEM)));
  const int64_t ub = (static_cast<int64_t>(rows) / BN + G) * ((2 * m + d) / WS_BM);
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(sm_count(), ub)));
  DM_CUDA_CHECK(launch_pdl(kern, dim3(grid), dim3(192), C::SMEM, s, tw1, tx1, tw2, tx2, g));
  return DECOMOE_OK;
}

// Token chunk by row count, as launch_ws_auto.
static int launch_ffn_ws(const void* x_perm, int rows, int d, int m, const void* w_gu, const void* w_down,
                         const int32_t* offsets, int G, void* h, void* y, int32_t* ready, int32_t* status,
                         cudaStream_t s) {
  if (rows <= 256)
    return launch_ffn_ws_bn<ffn_ws_max_stages<32>(), 32>(x_perm, rows, d, m, w_gu, w_down, offsets, G, h, y, ready,
                                                         status, s);
  if (rows <= 512)
    return launch_ffn_ws_bn<ffn_ws_max_stages<64>(), 64>(x_perm, rows, d, m, w_gu, w_down, offsets, G, h, y, ready,
                                                         status, s);
  if (rows <= 1024)
    return launch_ffn_ws_bn<ffn_ws_max_stages<128>(), 128>(x_perm, rows, d, m, w_gu, w_down, offsets, G, h, y,
                                                           ready, status, s);
  return launch_ffn_ws_bn<ffn_ws_max_stages<256>(), 256>(x_perm, rows, d, m, w_gu, w_down, offsets, G, h, y, ready,
                                                         status, s);
}

// ------------------------------------------------------------------ experts on SM pairs
// Clusters of two that the device keeps resident at once (per device ordinal):
// the down tiles wait for gate/up tiles of other clusters.
static std::atomic<int> g_pair_clusters[64];
static int pair_clusters() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = g_pair_clusters[dev].load();
  if (v != 0) return v > 0 ? v : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(PF_THREADS);
  cfg.dynamicSmemBytes = PF_SMEM;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(k_ffn_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(PF_SMEM)) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&v, k_ffn_pair, &cfg) != cudaSuccess)
    v = 0;
  cudaGetLastError();  // a refused query leaves no error behind
  g_pair_clusters[dev].store(v > 0 ? v : -1);
  return v;
}

// Gate/up (h given w_gu), down (w_down) or both over rows grouped by expert:
// a: x_perm, or with perm the token-ordered x (x_copy: receives the grouped
// rows then, or null); see k_ffn_pair.
static int launch_ffn_pair(const void* a, const int32_t* perm, void* x_copy, int64_t rows, int d, int m, const void* w_gu,
                           const void* w_down, const int32_t* offsets, int G, void* h, void* y, int32_t* ready,
                           int32_t* status, cudaStream_t s) {
  const bool gu = w_gu != nullptr, dn = w_down != nullptr;
  CUtensorMap ta1, ta1s, tb1, ta2, ta2s, tb2;
  if (gu) {
    DM_RET(make_tmap_bf16(&tb1, w_gu, static_cast<uint64_t>(d), static_cast<uint64_t>(G) * 2 * m, 128, PF_BK));
    if (perm == nullptr) {
      DM_RET(make_tmap_bf16(&ta1, a, static_cast<uint64_t>(d), static_cast<uint64_t>(rows), PF_BM, PF_BK));
      DM_RET(make_tmap_bf16(&ta1s, a, static_cast<uint64_t>(d), static_cast<uint64_t>(rows), PF_BM / 2, PF_BK));
    } else {
      ta1 = ta1s = tb1;  // rows gathered by index: not used
    }
  }
  if (dn) {
    DM_RET(make_tmap_bf16(&ta2, h, static_cast<uint64_t>(m), static_cast<uint64_t>(rows), PF_BM, PF_BK));
    DM_RET(make_tmap_bf16(&ta2s, h, static_cast<uint64_t>(m), static_cast<uint64_t>(rows), PF_BM / 2, PF_BK));
    DM_RET(make_tmap_bf16(&tb2, w_down, static_cast<uint64_t>(m), static_cast<uint64_t>(G) * d, 128, PF_BK));
  }
  if (!gu) ta1 = ta2, ta1s = ta2s, tb1 = tb2;
  if (!dn) ta2 = ta1, ta2s = ta1s, tb2 = tb1;
  PairArgs g;
  g.offsets = offsets;
  g.G = G;
  g.d = d;
  g.m = m;
  g.gu = gu;
  g.dn = dn;
  g.h = h;
  g.y = y;
  g.ready = ready;
  g.status = status;
  g.limit_ns = static_cast<uint64_t>(wait_limit_ns());
  g.x = perm != nullptr ? static_cast<const uint8_t*>(a) : nullptr;
  g.perm = perm;
  g.x_copy = static_cast<uint8_t*>(x_copy);
  const int64_t ub = (rows / (2 * PF_BM) + std::min<int64_t>(G, rows)) * ((gu ? 2 * m : 0) + (dn ? d : 0)) / PF_BN;
  const int ncl = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(pair_clusters(), ub)));
  DM_CUDA_CHECK(cudaFuncSetAttribute(k_ffn_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(PF_SMEM)));
  DM_CUDA_CHECK(launch_pdl(k_ffn_pair, dim3(2 * ncl), dim3(PF_THREADS), PF_SMEM, s, ta1, tb1, ta2, tb2, ta1s, ta2s, g));
  return DECOMOE_OK;
}

// X: [rows, kdim] token rows grouped by expert, or with GATHER_B the source
// tensor [x_tensor_rows, kdim] whose row b_rows[r] is token row r;
// W: [G * wrows, kdim].
template <bool SWIGLU, int STAGES, bool GATHER_B = false, int BN = 256>
static int launch_ws(const void* X, int rows, int kdim, const void* W, int wrows, const int32_t* offsets, int G,
                     void* out, int64_t out_ld, int32_t* status, cudaStream_t s, const int32_t* b_rows = nullptr,
                     int64_t x_tensor_rows = 0) {
  using C = WsCfg<STAGES, SWIGLU, BN>;
  constexpr int WS_BN = BN;
  CUtensorMap tw, tx;
  DM_RET(make_tmap_bf16(&tw, W, static_cast<uint64_t>(kdim), static_cast<uint64_t>(G) * wrows, WS_BM, WS_BK));
  if (GATHER_B)
    DM_RET(make_tmap_bf16(&tx, X, static_cast<uint64_t>(kdim), static_cast<uint64_t>(x_tensor_rows), 1, WS_BK));
  else
    DM_RET(make_tmap_bf16(&tx, X, static_cast<uint64_t>(kdim), static_cast<uint64_t>(rows), WS_BOX, WS_BK));
  WsArgs g;
  g.offsets = offsets;
  g.G = G;
  g.rows = rows;
  g.wrows = wrows;
  g.kdim = kdim;
  g.out = out;
  g.out_ld = out_ld;
  g.status = status;
  g.limit_ns = static_cast<uint64_t>(wait_limit_ns());
  g.b_rows = b_rows;
  auto kern = k_moe_ws<SWIGLU, STAGES, GATHER_B, BN>;
  static_assert(C::SMEM <= 232448, "shared memory budget");
  DM_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(C::SMEM)));
  const int64_t ub_tiles = (static_cast<int64_t>(rows) / WS_BN + G) * (wrows / WS_BM);
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(sm_count(), ub_tiles)));
  DM_CUDA_CHECK(launch_pdl(kern, dim3(grid), dim3(192), C::SMEM, s, tw, tx, g));
  return DECOMOE_OK;
}

// Weights-stationary launch with the token chunk sized to the row count: an
// expert never gets more rows than there are tokens, and rows = T * k with
// k >= 1, so for rows <= 256 a 32-token chunk usually covers every expert in
// one chunk (decode); smaller chunks buy a deeper weight-streaming ring.
template <bool SWIGLU>
static int launch_ws_auto(const void* X, int rows, int kdim, const void* W, int wrows, const int32_t* offsets,
                          int G, void* out, int64_t out_ld, int32_t* status, cudaStream_t s) {
  if (rows <= 256)
    return launch_ws<SWIGLU, ws_max_stages<SWIGLU, 32>(), false, 32>(X, rows, kdim, W, wrows, offsets, G, out,
                                                                     out_ld, status, s);
  if (rows <= 512)
    return launch_ws<SWIGLU, ws_max_stages<SWIGLU, 64>(), false, 64>(X, rows, kdim, W, wrows, offsets, G, out,
                                                                     out_ld, status, s);
  if (rows <= 1024)
    return launch_ws<SWIGLU, ws_max_stages<SWIGLU, 128>(), false, 128>(X, rows, kdim, W, wrows, offsets, G, out,
                                                                       out_ld, status, s);
  return launch_ws<SWIGLU, 4, false, 256>(X, rows, kdim, W, wrows, offsets, G, out, out_ld, status, s);
}

bool router_tc_supported(int d, int E) { return d % 64 == 0 && (E == 128 || E == 256); }

// Router on the tensor cores with the router rows as the M operand (E = 128
// or 256 rows, one or two M tiles) and the tokens as N tiles of BN columns, so
// that T = 2048 already spreads over 128 CTAs; the epilogue writes the
// transpose, logits[t, e], 32 experts of one token per warp store.
int launch_router_tc(const void* x, const void* w_r, const float* bias, int64_t T, int d, int E,
                     float* logits, int32_t* status, cudaStream_t s) {
  if (T > 0x7fffff00LL) {
    set_error("router_logits: T too large for the tensor-core path");
    return DECOMOE_ERR_UNSUPPORTED;
  }
  const int64_t ctas = sm_count();
  if (T <= 16 * ctas) return launch_router_kernel<16, 1>(x, w_r, bias, T, d, E, logits, status, s);
  if (T <= 32 * ctas) return launch_router_kernel<32, 1>(x, w_r, bias, T, d, E, logits, status, s);
  return launch_router_kernel<64, 1>(x, w_r, bias, T, d, E, logits, status, s);
}

// k-split router: KS k slices of the router GEMM write partial logits
// [KS][T][E] (no bias) to the scratch, then k_router_reduce adds the slices in
// slice order and the bias last: logits = (((p0 + p1) + ...) + p_{KS-1}) + b.
// More CTAs with fewer k-blocks each (and N = 64 tokens per MMA instead of
// 16) than the unsplit kernel at the same token count.
template <int KS>
__global__ void __launch_bounds__(256)
    k_router_reduce(const float4* __restrict__ part, int64_t n4, const float* __restrict__ bias, int E,
                    float4* __restrict__ logits) {
  pdl_enter();
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n4;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    float4 v[KS];
#pragma unroll
    for (int sl = 0; sl < KS; ++sl) v[sl] = __ldcs(part + sl * n4 + i);  // every slice load in flight
    float4 acc = v[0];
#pragma unroll
    for (int sl = 1; sl < KS; ++sl) {
      acc.x += v[sl].x;
      acc.y += v[sl].y;
      acc.z += v[sl].z;
      acc.w += v[sl].w;
    }
    if (bias != nullptr) {
      const int e = static_cast<int>((i * 4) % E);
      acc.x += bias[e];
      acc.y += bias[e + 1];
      acc.z += bias[e + 2];
      acc.w += bias[e + 3];
    }
    logits[i] = acc;
  }
}

int router_split_ks(int64_t T, int d, int E) {
  if (!router_tc_supported(d, E) || d % (64 * 16) != 0) return 1;
  const int64_t tiles = (T + 63) / 64, ctas = sm_count();
  if (tiles * 16 <= ctas) return 16;
  if (tiles * 4 <= ctas) return 4;
  return 1;
}

template <int KS>
static int launch_router_split_ks(const void* x, const void* w_r, const float* bias, int64_t T, int d, int E,
                                  float* logits, float* scratch, int32_t* status, cudaStream_t s) {
  const int64_t n = T * E;
  DM_RET((launch_router_kernel<64, KS>(x, w_r, nullptr, T, d, E, scratch, status, s)));
  const int64_t n4 = n / 4;
  const int blocks = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n4 + 255) / 256, sm_count())));
  DM_CUDA_CHECK(launch_pdl(k_router_reduce<KS>, dim3(blocks), dim3(256), 0, s,
                           reinterpret_cast<const float4*>(scratch), n4, bias, E, reinterpret_cast<float4*>(logits)));
  return DECOMOE_OK;
}

int launch_router_parts(const void* x, const void* w_r, int64_t T, int d, int E, float* scratch, int32_t* status,
                        cudaStream_t s, int* ks_out) {
  const int ks = router_split_ks(T, d, E);
  *ks_out = ks;
  switch (ks) {
    case 16: return launch_router_kernel<64, 16>(x, w_r, nullptr, T, d, E, scratch, status, s);
    case 4: return launch_router_kernel<64, 4>(x, w_r, nullptr, T, d, E, scratch, status, s);
    default:
      return DECOMOE_OK;  // no split at this size: nothing launched
  }
}

int launch_router_split(const void* x, const void* w_r, const float* bias, int64_t T, int d, int E, float* logits,
                        float* scratch, int32_t* status, cudaStream_t s) {
  switch (router_split_ks(T, d, E)) {
    case 16: return launch_router_split_ks<16>(x, w_r, bias, T, d, E, logits, scratch, status, s);
    case 4: return launch_router_split_ks<4>(x, w_r, bias, T, d, E, logits, scratch, status, s);
    default: return launch_router_tc(x, w_r, bias, T, d, E, logits, status, s);
  }
}

// ------------------------------------------------------------------ CUDA-core paths
template <typename T>
__device__ __forceinline__ float ld_f(const T* p);
template <>
__device__ __forceinline__ float ld_f<float>(const float* p) { return *p; }
template <>
__device__ __forceinline__ float ld_f<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}
template <typename T>
__device__ __forceinline__ T from_f(float v);
template <>
__device__ __forceinline__ float from_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ int find_group(const int32_t* __restrict__ offsets, int G, int r) {
  int lo = 0, hi = G - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (offsets[mid] <= r)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// h[r, f] = silu(W_gate[e] x_r)_f * (W_up[e] x_r)_f with the interleaved gate/up
// layout. One thread per (row, feature): the reference of the bf16 experts.
template <typename T>
__global__ void k_simt_gate_up(const T* __restrict__ A, const int32_t* __restrict__ offsets, int G,
                               const T* __restrict__ Wgu, int d, int m, T* __restrict__ H) {
  const int rows = offsets[G];
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= m) return;
  for (int r = blockIdx.y; r < rows; r += gridDim.y) {
    const int e = find_group(offsets, G, r);
    const int blk = f / DECOMOE_GU_BLOCK, i = f % DECOMOE_GU_BLOCK;
    const int64_t grow = static_cast<int64_t>(e) * 2 * m + blk * 2 * DECOMOE_GU_BLOCK + i;
    const T* wg = Wgu + grow * d;
    const T* wu = wg + static_cast<int64_t>(DECOMOE_GU_BLOCK) * d;
    const T* x = A + static_cast<int64_t>(r) * d;
    float ag = 0.f, au = 0.f;
    for (int j = 0; j < d; ++j) {
      const float xv = ld_f(x + j);
      ag = fmaf(xv, ld_f(wg + j), ag);
      au = fmaf(xv, ld_f(wu + j), au);
    }
    const float hv = ag / (1.0f + expf(-ag)) * au;
    H[static_cast<int64_t>(r) * m + f] = from_f<T>(hv);
  }
}

// y[r, n] = sum_f W_down[e][n, f] h[r, f]. One thread per (row, output).
template <typename T>
__global__ void k_simt_down(const T* __restrict__ H, const int32_t* __restrict__ offsets, int G,
                            const T* __restrict__ Wd, int d, int m, T* __restrict__ Y) {
  const int rows = offsets[G];
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d) return;
  for (int r = blockIdx.y; r < rows; r += gridDim.y) {
    const int e = find_group(offsets, G, r);
    const T* w = Wd + (static_cast<int64_t>(e) * d + n) * m;
    const T* h = H + static_cast<int64_t>(r) * m;
    float acc = 0.f;
    for (int f = 0; f < m; ++f) acc = fmaf(ld_f(h + f), ld_f(w + f), acc);
    Y[static_cast<int64_t>(r) * d + n] = from_f<T>(acc);
  }
}

// fp32 experts: a warp takes up to F32_RT rows of one expert and four features
// (a gate and an up row each) or eight outputs. 128 routed rows over ten
// experts of d = 256, m = 128: gate/up 39.4 -> 5.9 us, down 20.4 ->
// 4.5 us against one thread per result.
constexpr int F32_RT = 8, F32_WARPS = 4;
template <int VEC>
__global__ void __launch_bounds__(32 * F32_WARPS)
    k_f32_gate_up(const float* __restrict__ A, const int32_t* __restrict__ offsets, int G,
                  const float* __restrict__ Wgu, int d, int m, float* __restrict__ H,
                  const int32_t* __restrict__ a_rows) {
  pdl_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int e, r0, r1;
  if (!chunk_rows<F32_RT>(offsets, G, blockIdx.x, lane, e, r0, r1)) return;
  const float* a[F32_RT];
#pragma unroll
  for (int r = 0; r < F32_RT; ++r) {
    const int row = min(r0 + r, r1 - 1);  // a short chunk repeats its last row
    a[r] = A + static_cast<int64_t>(a_rows ? a_rows[row] : row) * d;
  }
  for (int f0 = (blockIdx.y * F32_WARPS + warp) * 4; f0 < m; f0 += gridDim.y * F32_WARPS * 4) {
    const float* w[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int f = f0 + i;
      const int64_t grow = static_cast<int64_t>(e) * 2 * m + f / DECOMOE_GU_BLOCK * 2 * DECOMOE_GU_BLOCK +
                           f % DECOMOE_GU_BLOCK;
      w[2 * i] = Wgu + grow * d;
      w[2 * i + 1] = w[2 * i] + static_cast<int64_t>(DECOMOE_GU_BLOCK) * d;
    }
    float acc[F32_RT * 8];
    rows_dot<float, VEC>(a, w, d, lane, acc);
    warp_scatter_sum(acc, lane);  // lane 4 r + i: gate and up of row r, feature i
    const float ag = acc[0], au = acc[1];
    const int row = r0 + (lane >> 2);
    if (row < r1) H[static_cast<int64_t>(row) * m + f0 + (lane & 3)] = ag / (1.0f + expf(-ag)) * au;
  }
}

template <int VEC>
__global__ void __launch_bounds__(32 * F32_WARPS)
    k_f32_down(const float* __restrict__ H, const int32_t* __restrict__ offsets, int G, const float* __restrict__ Wd,
               int d, int m, float* __restrict__ Y) {
  pdl_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int e, r0, r1;
  if (!chunk_rows<F32_RT>(offsets, G, blockIdx.x, lane, e, r0, r1)) return;
  const float* a[F32_RT];
#pragma unroll
  for (int r = 0; r < F32_RT; ++r) a[r] = H + static_cast<int64_t>(min(r0 + r, r1 - 1)) * m;
  for (int n0 = (blockIdx.y * F32_WARPS + warp) * 8; n0 < d; n0 += gridDim.y * F32_WARPS * 8) {
    const float* w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = Wd + (static_cast<int64_t>(e) * d + min(n0 + i, d - 1)) * m;
    float acc[F32_RT * 8];
    rows_dot<float, VEC>(a, w, m, lane, acc);
    warp_scatter_sum(acc, lane);  // lane 4 r + i: outputs 2 i and 2 i + 1 of row r
    const int row = r0 + (lane >> 2), n = n0 + 2 * (lane & 3);
    if (row < r1) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (n + u < d) Y[static_cast<int64_t>(row) * d + n + u] = acc[u];
    }
  }
}

// Row chunks of R rows in K groups (at most) and the features' blocks.
static dim3 f32_grid(int64_t R, int K, int outs, int per_warp) {
  const int64_t chunks = (R + F32_RT - 1) / F32_RT + std::min<int64_t>(K, R);
  const int per_block = F32_WARPS * per_warp;
  return dim3(static_cast<unsigned>(chunks), static_cast<unsigned>(std::min((outs + per_block - 1) / per_block, 65535)));
}
static int launch_f32_gate_up(const float* x, const int32_t* offsets, int64_t R, int K, int d, int m, const float* wgu,
                              float* h, const int32_t* rows, cudaStream_t s) {
  const bool vec = d % 4 == 0 && aligned16(x) && aligned16(wgu);
  DM_CUDA_CHECK(launch_pdl(vec ? k_f32_gate_up<4> : k_f32_gate_up<1>, f32_grid(R, K, m, 4), dim3(32 * F32_WARPS), 0, s,
                           x, offsets, K, wgu, d, m, h, rows));
  return DECOMOE_OK;
}

// ------------------------------------------------------------------ weight layout
__global__ void k_weight_layout(const uint4* __restrict__ wg, const uint4* __restrict__ wu,
                                uint4* __restrict__ wgu, int E, int m, int vec) {
  const int64_t rows_out = static_cast<int64_t>(E) * 2 * m;
  const int lane = threadIdx.x & 31;
  const int64_t gw = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t ro = gw; ro < rows_out; ro += nw) {
    const int64_t e = ro / (2 * m);
    const int rr = static_cast<int>(ro - e * 2 * m);
    const int blk = rr / (2 * DECOMOE_GU_BLOCK), w = rr % (2 * DECOMOE_GU_BLOCK);
    const bool is_up = w >= DECOMOE_GU_BLOCK;
    const int f = blk * DECOMOE_GU_BLOCK + (is_up ? w - DECOMOE_GU_BLOCK : w);
    const uint4* src = (is_up ? wu : wg) + (e * m + f) * vec;
    uint4* dst = wgu + ro * vec;
    for (int c = lane; c < vec; c += 32) dst[c] = src[c];
  }
}

}  // namespace decomoe

using namespace decomoe;

extern "C" {

int decomoe_weight_layout(const void* w_gate, const void* w_up, void* w_gate_up, int E, int d, int m,
                          int dtype, decomoe_stream_t stream) {
  clear_error();
  DM_ARG_CHECK(w_gate && w_up && w_gate_up, "weight_layout: null pointer");
  DM_ARG_CHECK(E > 0 && d > 0 && m > 0, "weight_layout: bad sizes");
  DM_ARG_CHECK(m % DECOMOE_GU_BLOCK == 0, "weight_layout: m=%d must be a multiple of %d", m, DECOMOE_GU_BLOCK);
  DM_ARG_CHECK(dtype == DECOMOE_BF16 || dtype == DECOMOE_F32, "weight_layout: bad dtype");
  const size_t row_bytes = static_cast<size_t>(d) * dtype_bytes(dtype);
  DM_ARG_CHECK(row_bytes % 16 == 0 && aligned16(w_gate) && aligned16(w_up) && aligned16(w_gate_up),
               "weight_layout: rows must be 16-byte multiples, pointers 16-byte aligned");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int blocks = sm_count() * 8;
  k_weight_layout<<<blocks, 256, 0, s>>>(static_cast<const uint4*>(w_gate), static_cast<const uint4*>(w_up),
                                         static_cast<uint4*>(w_gate_up), E, m,
                                         static_cast<int>(row_bytes / 16));
  DM_LAUNCH_CHECK("k_weight_layout");
  return DECOMOE_OK;
}

static int expert_check(const char* name, const void* a, const int32_t* offsets, int64_t rows, int K, int d,
                        int m, int dtype, const void* w, void* out) {
  DM_ARG_CHECK(rows >= 0 && rows < 0x7fffffffLL, "%s: rows out of range", name);
  DM_ARG_CHECK(K >= 1 && K <= DECOMOE_MAX_E, "%s: K=%d outside [1, %d]", name, K, DECOMOE_MAX_E);
  DM_ARG_CHECK(d > 0 && m > 0, "%s: bad d/m", name);
  DM_ARG_CHECK(dtype == DECOMOE_BF16 || dtype == DECOMOE_F32, "%s: bad dtype", name);
  DM_ARG_CHECK(m % DECOMOE_GU_BLOCK == 0, "%s: m must be a multiple of %d", name, DECOMOE_GU_BLOCK);
  if (rows == 0) return DECOMOE_OK;
  DM_ARG_CHECK(a && offsets && w && out, "%s: null pointer", name);
  if (dtype == DECOMOE_BF16) {
    // tensor-core tiles: 256 output columns (gate/up interleaved 2m, down d)
    DM_ARG_CHECK(m % 128 == 0, "%s: bf16 needs m %% 128 == 0 (m=%d)", name, m);
    DM_ARG_CHECK(d % 256 == 0, "%s: bf16 needs d %% 256 == 0 (d=%d)", name, d);
    DM_ARG_CHECK(aligned16(a) && aligned16(w) && aligned16(out), "%s: pointers must be 16-byte aligned", name);
  }
  return DECOMOE_OK;
}

int decomoe_expert_gate_up(const void* x_perm, const int32_t* offsets, int64_t rows, int K, int d, int m,
                           int dtype, const void* w_gate_up, void* h, int32_t* status_dev, int32_t* sched_dev,
                           decomoe_stream_t stream) {
  clear_error();
  DM_RET(expert_check("expert_gate_up", x_perm, offsets, rows, K, d, m, dtype, w_gate_up, h));
  if (rows == 0) return DECOMOE_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int R = static_cast<int>(rows);
  if (dtype == DECOMOE_F32)
    return launch_f32_gate_up(static_cast<const float*>(x_perm), offsets, R, K, d, m,
                              static_cast<const float*>(w_gate_up), static_cast<float*>(h), nullptr, s);
  if (static_cast<int64_t>(R) <= static_cast<int64_t>(DECOMOE_WS_MAX_AVG_ROWS) * K)
    return launch_ws_auto<true>(x_perm, R, d, w_gate_up, 2 * m, offsets, K, h, m, status_dev, s);
  (void)sched_dev;  // the pair kernel hands its tiles out in a fixed order
  return launch_ffn_pair(x_perm, nullptr, nullptr, R, d, m, w_gate_up, nullptr, offsets, K, h, nullptr, nullptr, status_dev, s);
}

int decomoe_expert_down(const void* h, const int32_t* offsets, int64_t rows, int K, int d, int m, int dtype,
                        const void* w_down, void* y_perm, int32_t* status_dev, int32_t* sched_dev,
                        decomoe_stream_t stream) {
  clear_error();
  DM_RET(expert_check("expert_down", h, offsets, rows, K, d, m, dtype, w_down, y_perm));
  if (rows == 0) return DECOMOE_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int R = static_cast<int>(rows);
  if (dtype == DECOMOE_F32) {
    const bool vec = m % 4 == 0 && aligned16(h) && aligned16(w_down);
    DM_CUDA_CHECK(launch_pdl(vec ? k_f32_down<4> : k_f32_down<1>, f32_grid(R, K, d, 8), dim3(32 * F32_WARPS), 0, s,
                             static_cast<const float*>(h), offsets, K, static_cast<const float*>(w_down), d, m,
                             static_cast<float*>(y_perm)));
    return DECOMOE_OK;
  }
  if (static_cast<int64_t>(R) <= static_cast<int64_t>(DECOMOE_WS_MAX_AVG_ROWS) * K)
    return launch_ws_auto<false>(h, R, m, w_down, d, offsets, K, y_perm, d, status_dev, s);
  (void)sched_dev;
  return launch_ffn_pair(nullptr, nullptr, nullptr, R, d, m, nullptr, w_down, offsets, K, const_cast<void*>(h), y_perm, nullptr,
                           status_dev, s);
}

int decomoe_expert_gate_up_gather(const void* x, int64_t T, const int32_t* perm_token, const int32_t* offsets,
                                  int64_t rows, int K, int d, int m, int dtype, const void* w_gate_up, void* h,
                                  int32_t* status_dev, int32_t* sched_dev, decomoe_stream_t stream) {
  (void)sched_dev;  // the gathered form keeps the static tile order
  clear_error();
  DM_RET(expert_check("expert_gate_up_gather", x, offsets, rows, K, d, m, dtype, w_gate_up, h));
  if (rows == 0) return DECOMOE_OK;
  DM_ARG_CHECK(perm_token != nullptr && T > 0 && T < 0x7fffffffLL, "expert_gate_up_gather: bad perm_token or T");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int R = static_cast<int>(rows);
  if (dtype == DECOMOE_F32)
    return launch_f32_gate_up(static_cast<const float*>(x), offsets, R, K, d, m, static_cast<const float*>(w_gate_up),
                              static_cast<float*>(h), perm_token, s);
  if (static_cast<int64_t>(R) <= static_cast<int64_t>(DECOMOE_WS_MAX_AVG_ROWS) * K)
    return launch_ws<true, 4, true>(x, R, d, w_gate_up, 2 * m, offsets, K, h, m, status_dev, s, perm_token, T);
  return launch_ffn_pair(x, perm_token, nullptr, R, d, m, w_gate_up, nullptr, offsets, K, h, nullptr, nullptr, status_dev, s);
}

int decomoe_expert_swiglu_gather(const void* x, int64_t T, const int32_t* perm_token, const int32_t* offsets,
                                 int64_t rows, int K, int d, int m, int dtype, const void* w_gate_up,
                                 const void* w_down, void* h_ws, void* y_perm, int32_t* status_dev,
                                 int32_t* sched_dev, decomoe_stream_t stream) {
  DM_RET(decomoe_expert_gate_up_gather(x, T, perm_token, offsets, rows, K, d, m, dtype, w_gate_up, h_ws,
                                       status_dev, sched_dev, stream));
  return decomoe_expert_down(h_ws, offsets, rows, K, d, m, dtype, w_down, y_perm, status_dev, sched_dev, stream);
}

int decomoe_expert_swiglu(const void* x_perm, const int32_t* offsets, int64_t rows, int K, int d, int m,
                          int dtype, const void* w_gate_up, const void* w_down, void* h_ws, void* y_perm,
                          int32_t* status_dev, int32_t* sched_dev, decomoe_stream_t stream) {
  DM_RET(decomoe_expert_gate_up(x_perm, offsets, rows, K, d, m, dtype, w_gate_up, h_ws, status_dev, sched_dev,
                                stream));
  return decomoe_expert_down(h_ws, offsets, rows, K, d, m, dtype, w_down, y_perm, status_dev, sched_dev, stream);
}

// Reference CUDA-core path for bf16 (same math as the tensor-core path: bf16
// products, fp32 accumulation, h rounded to bf16). Not part of the public
// header; used by tests to localise disagreements between the tensor-core
// kernels and the oracle.
int decomoe_expert_swiglu_ref(const void* x_perm, const int32_t* offsets, int64_t rows, int K, int d, int m,
                               const void* w_gate_up, const void* w_down, void* h_ws, void* y_perm,
                               decomoe_stream_t stream) {
  clear_error();
  DM_ARG_CHECK(rows >= 0 && rows < 0x7fffffffLL && K >= 1 && K <= DECOMOE_MAX_E && d > 0 && m > 0,
               "expert_swiglu_ref: bad sizes");
  if (rows == 0) return DECOMOE_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int R = static_cast<int>(rows);
  dim3 g1((m + 127) / 128, static_cast<unsigned>(std::min(R, 65535)));
  k_simt_gate_up<__nv_bfloat16><<<g1, 128, 0, s>>>(static_cast<const __nv_bfloat16*>(x_perm), offsets, K,
                                                    static_cast<const __nv_bfloat16*>(w_gate_up), d, m,
                                                    static_cast<__nv_bfloat16*>(h_ws));
  DM_LAUNCH_CHECK("k_simt_gate_up<bf16>");
  dim3 g2((d + 127) / 128, static_cast<unsigned>(std::min(R, 65535)));
  k_simt_down<__nv_bfloat16><<<g2, 128, 0, s>>>(static_cast<const __nv_bfloat16*>(h_ws), offsets, K,
                                                 static_cast<const __nv_bfloat16*>(w_down), d, m,
                                                 static_cast<__nv_bfloat16*>(y_perm));
  DM_LAUNCH_CHECK("k_simt_down<bf16>");
  return DECOMOE_OK;
}

}  // extern "C"

namespace decomoe {

// Rows from which the fused launch is taken (with fewer, the gate/up tiles
// leave SMs idle and the fused form gains nothing).
#ifndef DECOMOE_FFN_FUSED_MIN_ROWS
#define DECOMOE_FFN_FUSED_MIN_ROWS 16
#endif
// Rows up to which it is taken: FFN_FUSED_MAX_ROWS. Its down tiles wait for gate/up tiles of other
// blocks, so the launch needs all its blocks on the device together: other
// long-running work on the device holds it up, and a second launch of the kind
// on another stream, each with part of the SMs, would end both in a timeout.
// Two launches need nothing of other blocks. A layer (d = 2048, m = 768, top 8) in
// one launch and in two: 4097 tokens, 128 experts 342 and 349 us, 8000 tokens 566
// and 557, 16384 tokens 1050 and 1005.
// Which one-launch form the expert FFN takes: FFN_FUSED_NONE (two launches:
// fp32, fewer than DECOMOE_FFN_FUSED_MIN_ROWS rows or more than
// FFN_FUSED_MAX_ROWS), FFN_FUSED_WS (at most 8 rows per expert on average) or
// FFN_FUSED_PAIR (above).
int expert_ffn_fused_kind(int64_t rows, int K, int dtype) {
  constexpr int64_t min_rows = DECOMOE_FFN_FUSED_MIN_ROWS;
  if (dtype != DECOMOE_BF16 || rows < min_rows || rows > FFN_FUSED_MAX_ROWS || K <= 0) return FFN_FUSED_NONE;
  return rows <= static_cast<int64_t>(DECOMOE_WS_MAX_AVG_ROWS) * K ? FFN_FUSED_WS : FFN_FUSED_PAIR;
}

int launch_expert_ffn_fused(const void* x_perm, const int32_t* offsets, int64_t rows, int K, int d, int m, int dtype,
                            const void* w_gate_up, const void* w_down, void* h, void* y_perm, int32_t* ready,
                            int32_t* status, cudaStream_t s, bool* launched, const void* gather_x,
                            const int32_t* perm, bool copy_rows) {
  *launched = false;
  const int kind = expert_ffn_fused_kind(rows, K, dtype);
  DM_ARG_CHECK(gather_x == nullptr || kind == FFN_FUSED_PAIR, "expert ffn: the row gather needs the pair form");
  if (kind == FFN_FUSED_NONE) return DECOMOE_OK;
  DM_RET(expert_check("expert_gate_up", x_perm, offsets, rows, K, d, m, dtype, w_gate_up, h));
  DM_RET(expert_check("expert_down", h, offsets, rows, K, d, m, dtype, w_down, y_perm));
  DM_ARG_CHECK(ready != nullptr, "expert ffn: null ready counters");
  if (gather_x != nullptr)
    DM_ARG_CHECK(perm != nullptr && aligned16(gather_x), "expert ffn: gather needs perm and a 16-byte aligned x");
  if (kind == FFN_FUSED_WS)
    DM_RET(launch_ffn_ws(x_perm, static_cast<int>(rows), d, m, w_gate_up, w_down, offsets, K, h, y_perm, ready,
                         status, s));
  else
    DM_RET(launch_ffn_pair(gather_x != nullptr ? gather_x : x_perm, gather_x != nullptr ? perm : nullptr,
                           copy_rows ? const_cast<void*>(x_perm) : nullptr, rows, d, m, w_gate_up, w_down, offsets, K, h, y_perm, ready, status, s));
  *launched = true;
  return DECOMOE_OK;
}

// int32 counters the fused expert launch needs (zero at launch): one per
// expert (decode kernel) or two per 256-row tile (pair kernel).
size_t expert_ffn_sync_ints(int64_t rows, int E) { return 2 * static_cast<size_t>(rows / 128 + E + 1); }

}  // namespace decomoe

extern "C" {

size_t decomoe_expert_swiglu_ready_ints(int64_t rows, int K) {
  return rows < 0 || K <= 0 ? 0 : decomoe::expert_ffn_sync_ints(rows, K);
}

int decomoe_expert_swiglu_fused(const void* x_perm, const int32_t* offsets, int64_t rows, int K, int d, int m,
                                int dtype, const void* w_gate_up, const void* w_down, void* h_ws, void* y_perm,
                                int32_t* ready, int32_t* status_dev, decomoe_stream_t stream) {
  using namespace decomoe;
  clear_error();
  bool fused = false;
  DM_RET(launch_expert_ffn_fused(x_perm, offsets, rows, K, d, m, dtype, w_gate_up, w_down, h_ws, y_perm, ready,
                                 status_dev, reinterpret_cast<cudaStream_t>(stream), &fused));
  if (fused) return DECOMOE_OK;
  return decomoe_expert_swiglu(x_perm, offsets, rows, K, d, m, dtype, w_gate_up, w_down, h_ws, y_perm, status_dev,
                               nullptr, stream);
}

int decomoe_expert_swiglu_fused_gather(const void* x, int64_t T, const int32_t* perm_token, const int32_t* offsets,
                                       int64_t rows, int K, int d, int m, int dtype, const void* w_gate_up,
                                       const void* w_down, void* x_perm, void* h_ws, void* y_perm, int32_t* ready,
                                       int32_t* status_dev, decomoe_stream_t stream) {
  using namespace decomoe;
  clear_error();
  DM_ARG_CHECK(x != nullptr && perm_token != nullptr && T >= 0, "expert_swiglu_fused_gather: null pointer");
  DM_ARG_CHECK(expert_ffn_fused_kind(rows, K, dtype) == FFN_FUSED_PAIR,
               "expert_swiglu_fused_gather: %lld rows at K=%d take no one-launch tokens-as-M form",
               (long long)rows, K);
  bool fused = false;
  DM_RET(launch_expert_ffn_fused(x_perm, offsets, rows, K, d, m, dtype, w_gate_up, w_down, h_ws, y_perm, ready,
                                 status_dev, reinterpret_cast<cudaStream_t>(stream), &fused, x, perm_token, true));
  return fused ? DECOMOE_OK : DECOMOE_ERR_UNSUPPORTED;
}

}  // extern "C"
