// Router logits (CUDA-core path) and prefix-restricted top-k routing with the
// activated-mass reduction of RCEP (DecoMoE Section 3.3, Eqs. 10-12,
// Algorithm 2).
#include <cfloat>
#include <cstdint>

#include "dispatch_tile.cuh"
#include "route_common.cuh"
#include "simt_rows.cuh"

namespace decomoe {

// ------------------------------------------------------------ router, CUDA cores
// logits[t, e] = sum_j x[t, j] * w_r[e, j] + bias[e] for fp32 storage and
// shapes the tensor-core kernel does not take: a warp per RS_RT tokens and
// RS_NR experts, four warps per block (64 tokens, 16 experts, d = 256: 21.6 ->
// 4.9 us against one thread per logit).
constexpr int RS_RT = 4, RS_NR = 4, RS_WARPS = 4;
template <typename T, int VEC>
__global__ void __launch_bounds__(32 * RS_WARPS)
    k_router_rows(const T* __restrict__ x, const T* __restrict__ w_r, const float* __restrict__ bias, int64_t Tn, int d,
                  int E, float* __restrict__ logits) {
  pdl_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * RS_RT;
  const T* a[RS_RT];
#pragma unroll
  for (int r = 0; r < RS_RT; ++r) a[r] = x + (t0 + r < Tn ? t0 + r : Tn - 1) * d;
  for (int e0 = (blockIdx.y * RS_WARPS + warp) * RS_NR; e0 < E; e0 += gridDim.y * RS_WARPS * RS_NR) {
    const T* w[RS_NR];
#pragma unroll
    for (int j = 0; j < RS_NR; ++j) w[j] = w_r + static_cast<int64_t>(min(e0 + j, E - 1)) * d;
    float acc[RS_RT * RS_NR];
    rows_dot<T, VEC>(a, w, d, lane, acc);
    warp_scatter_sum(acc, lane);  // lanes 2 i and 2 i + 1: token i / RS_NR, expert i % RS_NR
    const int64_t t = t0 + (lane >> 1) / RS_NR;
    const int e = e0 + (lane >> 1) % RS_NR;
    if ((lane & 1) == 0 && t < Tn && e < E) logits[t * E + e] = acc[0] + (bias != nullptr ? bias[e] : 0.f);
  }
}

// Router for few tokens (decode) on CUDA cores: fp32 dot products of the bf16
// router rows and token rows. The router matrix is read from HBM once and
// spread over many SMs instead of one tensor-core tile.
#ifndef DECOMOE_ROUTER_GEMV_MAX_T
#define DECOMOE_ROUTER_GEMV_MAX_T 6  // token counts up to which the router runs on CUDA cores
#endif
static constexpr int64_t router_gemv_max_t() { return DECOMOE_ROUTER_GEMV_MAX_T; }
// One block per expert row and GEMV_TPB tokens: the block's 128 threads split
// the row's 16-byte vectors (thread i takes vectors i, i + 128, ...), so a
// row's loads are spread over four warps and the E rows over E blocks (one per
// SM at decode sizes) instead of piling every row of a block onto one SM; all
// of a thread's loads are issued before its first multiply. Partial dots are
// reduced by warp shuffles, then over the four warps in a fixed order.
__global__ void __launch_bounds__(GEMV_THREADS)
    k_router_gemv(const uint4* __restrict__ x, const uint4* __restrict__ w_r, const float* __restrict__ bias,
                  int64_t Tn, int vpr, int E, float* __restrict__ logits) {
  pdl_enter();
  __shared__ float red[GEMV_THREADS / 32][GEMV_TPB];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.y) * GEMV_TPB;
  const int nt = Tn - t0 < GEMV_TPB ? static_cast<int>(Tn - t0) : GEMV_TPB;
  const uint4* wr = w_r + static_cast<int64_t>(e) * vpr;
  float acc[GEMV_TPB];
#pragma unroll
  for (int j = 0; j < GEMV_TPB; ++j) acc[j] = 0.f;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  for (int c0 = 0; c0 < vpr; c0 += GEMV_THREADS * GEMV_VPT) {
    uint4 wv[GEMV_VPT], xv[GEMV_TPB][GEMV_VPT];
#pragma unroll
    for (int i = 0; i < GEMV_VPT; ++i) {
      const int c = c0 + static_cast<int>(threadIdx.x) + GEMV_THREADS * i;
      wv[i] = (c < vpr) ? __ldg(wr + c) : zero;
#pragma unroll
      for (int j = 0; j < GEMV_TPB; ++j) xv[j][i] = (c < vpr && j < nt) ? __ldg(x + (t0 + j) * vpr + c) : zero;
    }
#pragma unroll
    for (int i = 0; i < GEMV_VPT; ++i)
#pragma unroll
      for (int j = 0; j < GEMV_TPB; ++j) acc[j] = dot8_bf16(wv[i], xv[j][i], acc[j]);
  }
#pragma unroll
  for (int j = 0; j < GEMV_TPB; ++j) {
    float v = acc[j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) red[warp][j] = v;
  }
  __syncthreads();
  if (static_cast<int>(threadIdx.x) < nt) {
    const int j = threadIdx.x;
    float v = red[0][j];
#pragma unroll
    for (int w = 1; w < GEMV_THREADS / 32; ++w) v += red[w][j];
    logits[(t0 + j) * E + e] = v + (bias != nullptr ? bias[e] : 0.f);
  }
}

// ------------------------------------------------------------ routing
// One warp per token; lane l holds logits l, l+32, ... (E <= 256, 8 per lane)
// in registers. A pass of k rounds of warp arg-max picks the k largest of a
// range (ties: lower expert index); pick j ends in lane j. Weights are the
// softmax over the k picks (equal to prefix softmax + top-k + renormalise,
// because the prefix denominator cancels).
//
// With a mass buffer the same launch also computes the activated mass of
// Eq. 11 over the full pool [0, E): the full-pool picks are found first; if
// they all lie inside [0, K) they are also the prefix picks, else a second
// pass runs over [0, K). Each block writes its tokens' fp32 full-pool weights
// per expert, summed in token order, to part[block][e]; k_mass_finalize sums
// the blocks in a fixed order in fp64, so the mass is bit-reproducible.
constexpr int ROUTE_THREADS = 256;
constexpr int ROUTE_TPB = ROUTE_TOKENS_PER_BLOCK;  // tokens per block: one per warp

// NP: 1 reads plain logit rows; NP > 1 reads NP k slices of the split
// router (src), each warp loading its row's slices as coalesced 16-byte
// vectors (all NP in flight), adding them in slice order and the bias last,
// storing the sums to src.logits_out and, through shared memory, into the
// key layout (E % 4 == 0, 16-byte aligned rows).
// rd.counts set (one block, T <= ROUTE_TPB): after routing, the block
// dispatches its own picks (dispatch_tile over the T*k pairs).
static_assert(ROUTE_THREADS == DSP_THREADS, "the routing block runs the dispatch tile");
// NSL: key slots per lane (32 NSL >= E): 4 for pools of up to 128 experts halve
// the compares of a pick, which bound many tokens (2048 4.1 -> 3.3 us, 16384
// 16.6 -> 11.5).
template <int NP, int NSL>
__global__ void __launch_bounds__(ROUTE_THREADS)
    k_route(const float* __restrict__ logits, int64_t Tn, int E, int64_t ld, int K, int k,
            int32_t* __restrict__ idx_out, float* __restrict__ w_out, double* __restrict__ part,
            const int32_t* __restrict__ K_dev, int64_t skip_at, int64_t skip_len, RouteSrc src, RouteDispatch rd,
            int32_t* __restrict__ zero_ints, int n_zero) {
  pdl_enter();
  // block 0 clears a small int array for a later launch of the caller's chain
  if (zero_ints != nullptr && blockIdx.x == 0)
    for (int i = threadIdx.x; i < n_zero; i += ROUTE_THREADS) zero_ints[i] = 0;
  if (K_dev != nullptr) K = *K_dev;  // prefix chosen on the device (k <= K <= E by construction)
  // a token's logits (NP > 1), then its full-pool weights by expert (mass): one
  // read per token and expert, where each thread looked for its expert among the
  // block's 64 picks (with the mass 131 tokens 6.8 -> 5.9 us, 16384 23.3 -> 20.4)
  __shared__ __align__(16) float s_row[ROUTE_TPB][32 * NSL];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = static_cast<int64_t>(blockIdx.x) * ROUTE_TPB + warp;
  const bool mass = part != nullptr;
  if (t < Tn) {
    // token t reads logit row t, or t + skip_len from skip_at on (the text
    // tokens around a removed visual block)
    const int64_t roff = (t < skip_at ? t : t + skip_len) * ld;
    const float* row = logits + roff;
    const int lim = mass ? E : K;
    uint32_t v[NSL];  // order-preserving keys of the row's logits
    if constexpr (NP == 1) {
#pragma unroll
      for (int i = 0; i < NSL; ++i) {
        const int e = lane + 32 * i;
        v[i] = (e < lim) ? fkey(row[e]) : 0u;
      }
    } else {
      // partial sums of the k-split router, added in slice order, bias last
      const float4* r4 = reinterpret_cast<const float4*>(row);
      const int64_t s4 = src.part_stride / 4;
      for (int c = lane; c < E / 4; c += 32) {
        float4 p[NP];
#pragma unroll
        for (int sl = 0; sl < NP; ++sl) p[sl] = __ldcs(r4 + sl * s4 + c);
        float4 a = p[0];
#pragma unroll
        for (int sl = 1; sl < NP; ++sl) {
          a.x += p[sl].x;
          a.y += p[sl].y;
          a.z += p[sl].z;
          a.w += p[sl].w;
        }
        if (src.bias != nullptr) {
          const float4 b = reinterpret_cast<const float4*>(src.bias)[c];
          a.x += b.x;
          a.y += b.y;
          a.z += b.z;
          a.w += b.w;
        }
        if (src.logits_out != nullptr) reinterpret_cast<float4*>(src.logits_out + roff)[c] = a;
        reinterpret_cast<float4*>(s_row[warp])[c] = a;
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < NSL; ++i) {
        const int e = lane + 32 * i;
        v[i] = (e < lim) ? fkey(s_row[warp][e]) : 0u;
      }
    }
    if (mass) {
      __syncwarp();
      for (int e = lane; e < E; e += 32) s_row[warp][e] = 0.f;
    }
    float my_v;
    int my_i;
    warp_topk_n<NSL>(v, lim, k, lane, my_v, my_i);
    if (mass) {
      const float wf = pick_weight(my_v, lane, k);
      __syncwarp();
      if (lane < k && my_i >= 0 && my_i < E) s_row[warp][my_i] = wf;
      // full-pool picks all inside the prefix: they are the prefix picks too
      const bool inside = __all_sync(0xffffffffu, lane >= k || my_i < K);
      if (!inside) warp_topk_n<NSL>(v, K, k, lane, my_v, my_i);
    }
    if (idx_out != nullptr || w_out != nullptr) {
      const float w = pick_weight(my_v, lane, k);
      if (lane < k) {
        if (idx_out != nullptr) idx_out[t * k + lane] = my_i;
        if (w_out != nullptr) w_out[t * k + lane] = w;
      }
    }
  }
  if (mass) {
    __syncthreads();
    const int ntok = static_cast<int>(Tn - static_cast<int64_t>(blockIdx.x) * ROUTE_TPB < ROUTE_TPB
                                          ? Tn - static_cast<int64_t>(blockIdx.x) * ROUTE_TPB
                                          : ROUTE_TPB);
    for (int e = threadIdx.x; e < E; e += ROUTE_THREADS) {
      float acc = 0.f;
#pragma unroll
      for (int tt = 0; tt < ROUTE_TPB; ++tt)
        if (tt < ntok) acc += s_row[tt][e];  // token order; a token that did not pick e adds zero
      part[static_cast<int64_t>(blockIdx.x) * E + e] = static_cast<double>(acc);
    }
  }
  if (rd.counts != nullptr) {
    __syncthreads();  // the block's picks in idx_out are visible to all its threads
    dispatch_tile<true>(idx_out, Tn * k, k, rd.Kd, nullptr, 1, 0, rd.counts, rd.offsets, rd.perm_token, rd.inv_slot,
                        rd.status, static_cast<const uint4*>(rd.x), rd.row_vec, static_cast<uint4*>(rd.x_perm));
  }
}

// mass[e] = sum over blocks of part[b][e]: one block per expert, each thread
// sums a fixed strided subset of blocks in order, then a fixed-shape tree in
// shared memory combines the 256 thread sums (bit-reproducible).
__global__ void __launch_bounds__(256)
    k_mass_finalize(const double* __restrict__ part, int nblocks, int E, double* __restrict__ mass) {
  pdl_enter();
  mass_finalize_block(part, nblocks, E, static_cast<int>(blockIdx.x), mass);
}

// Eq. 12 by one block of DECOMOE_MAX_E threads on the mass in shared memory,
// thread e on the sum of the first e + 1 masses: the K of
// decomoe_select_prefix bit for bit. fp64 is what this costs (a dependent add
// takes tens of cycles here: one thread adding and dividing took 13.4 us for
// 128 experts), so the sums are formed as integers where that is exact: the
// masses are sums of fp32 weights, and when all of them are multiples of
// 2^-sh with a total below 2^(53 - sh) every sequential fp64 sum is exact, in
// whatever order it is formed. Otherwise one thread adds them up in order. A
// ratio is divided out only where the product p * total leaves it open.
// s_cum: E doubles of scratch.
__device__ __forceinline__ int select_prefix_block(const double* s_mass, double* s_cum, int E, int k, double p) {
  constexpr int NW = DECOMOE_MAX_E / 32;
  __shared__ float s_tf[NW];
  __shared__ uint64_t s_wsum[NW];
  __shared__ int s_first;
  const int e = threadIdx.x, warp = e >> 5, lane = e & 31;
  const uint64_t bits = e < E ? static_cast<uint64_t>(__double_as_longlong(s_mass[e])) : 0ull;
  const int ex = static_cast<int>(bits >> 52);  // sign and exponent
  // the total, to fix the scale (truncated to fp32 by hand; other exponents
  // than fp32's are left to the sequential sum)
  bool odd = bits != 0 && (ex < 1023 - 126 || ex > 1023 + 100);
  float tf = (odd || bits == 0) ? 0.f
                                : __uint_as_float((static_cast<uint32_t>(ex - 1023 + 127) << 23) |
                                                  static_cast<uint32_t>((bits >> 29) & 0x7FFFFFu));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) tf += __shfl_xor_sync(0xffffffffu, tf, off);
  if (lane == 0) s_tf[warp] = tf;
  if (e == 0) s_first = E;  // none reaches p (or p >= 1): the whole pool
  __syncthreads();
  tf = 0.f;
#pragma unroll
  for (int w = 0; w < NW; ++w) tf += s_tf[w];
  const int te = static_cast<int>(__float_as_uint(tf) >> 23) - 127;  // total < 2^(te + 2)
  const int shift = ex - 1075 + (51 - te);                           // scale sh = 51 - te
  uint64_t v = 0;
  if (!odd && bits != 0) {
    const uint64_t mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    if (shift >= 0) {
      v = mant << shift;  // below 2^53, as the total is
    } else if (shift > -53) {
      v = mant >> -shift;
      odd = (v << -shift) != mant;
    } else {
      odd = true;
    }
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint64_t u = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += u;
  }
  if (lane == 31) s_wsum[warp] = v;
  double cum, tot;
  if (!__syncthreads_or(odd)) {
    uint64_t all = 0, before = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      if (w == warp) before = all;
      all += s_wsum[w];
    }
    cum = __ull2double_rn(v + before);
    tot = __ull2double_rn(all);
  } else {
    if (e == 0) {
      double acc = 0.0;
      for (int i = 0; i < E; ++i) {
        acc = __dadd_rn(acc, s_mass[i]);
        s_cum[i] = acc;
      }
    }
    __syncthreads();
    cum = e < E ? s_cum[e] : 0.0;
    tot = s_cum[E - 1];
  }
  if (p < 1.0 && e < E) {
    // |p * tot rounded - p * tot| <= 2^-53 of it, and the quotient is rounded
    // by as little: outside 2^-50 of p * tot the comparison is decided
    const double t = p * tot;
    bool reached;
    if (p > 1e-280 && t < 1e280 && tot > 1e-280 && cum > fma(t, 0x1p-50, t))
      reached = true;
    else if (p > 1e-280 && t < 1e280 && tot > 1e-280 && cum < fma(t, -0x1p-50, t))
      reached = false;
    else
      reached = __ddiv_rn(cum, tot) >= p;
    if (reached) atomicMin(&s_first, e + 1);
  }
  __syncthreads();
  return tot > 0.0 && s_first > k ? s_first : k;
}

__global__ void __launch_bounds__(DECOMOE_MAX_E)
    k_select_prefix(const double* __restrict__ mass, int E, int k, double p, int32_t* __restrict__ K_dev) {
  pdl_enter();
  __shared__ double s_mass[DECOMOE_MAX_E], s_cum[DECOMOE_MAX_E];
  if (E > DECOMOE_MAX_E) {  // larger than any pool routed here: one thread
    if (threadIdx.x == 0) *K_dev = select_prefix_seq(mass, E, k, p);
    return;
  }
  for (int e = threadIdx.x; e < E; e += blockDim.x) s_mass[e] = mass[e];
  __syncthreads();
  const int K = select_prefix_block(s_mass, s_cum, E, k, p);
  if (threadIdx.x == 0) *K_dev = K;
}

// k_mass_finalize and k_select_prefix in one block, for at most MS_MAX_BLOCKS
// routing blocks: a thread per expert holds the partials that threads 0, 1,
// ... of mass_finalize_block would, and adds them in the same tree (its other
// leaves are zero, which change nothing), so the bits are the same. fp64 adds
// are the cost (an SM issues about two a cycle, so a warp's takes 16 cycles
// whatever its lanes do): a warp per expert with shuffles took 33 us at 17
// blocks of 128 experts, and above 64 blocks E blocks of their own are faster.
constexpr int MS_MAX_BLOCKS = 64;
__global__ void __launch_bounds__(DECOMOE_MAX_E)
    k_mass_select(const double* __restrict__ part, int nblocks, int E, double* __restrict__ mass, int k, double p,
                  int32_t* __restrict__ K_dev) {
  pdl_enter();
  __shared__ double s_mass[DECOMOE_MAX_E], s_cum[DECOMOE_MAX_E];
  const int e = threadIdx.x;
  if (e < E) {
    double a[MS_MAX_BLOCKS];
#pragma unroll
    for (int b = 0; b < MS_MAX_BLOCKS; ++b)
      if (b < nblocks) a[b] = part[static_cast<int64_t>(b) * E + e];
#pragma unroll
    for (int w = MS_MAX_BLOCKS / 2; w > 0; w >>= 1)
#pragma unroll
      for (int i = 0; i < w; ++i)
        if (i + w < nblocks) a[i] += a[i + w];
    mass[e] = a[0];
    s_mass[e] = a[0];
  }
  __syncthreads();
  const int K = select_prefix_block(s_mass, s_cum, E, k, p);
  if (threadIdx.x == 0) *K_dev = K;
}

int launch_mass_select(const double* part, int nblocks, int E, double* mass, int k, double p, int32_t* K_dev,
                       cudaStream_t s) {
  if (nblocks > MS_MAX_BLOCKS) {
    DM_CUDA_CHECK(launch_pdl(k_mass_finalize, dim3(E), dim3(256), 0, s, part, nblocks, E, mass));
    return decomoe_select_prefix_device(mass, E, k, p, K_dev, reinterpret_cast<decomoe_stream_t>(s));
  }
  DM_CUDA_CHECK(launch_pdl(k_mass_select, dim3(1), dim3(DECOMOE_MAX_E), 0, s, part, nblocks, E, mass, k, p, K_dev));
  return DECOMOE_OK;
}

// Activated mass (Eq. 11) over n tokens whose logit rows skip a block:
// token t reads row t, or t + skip_len from skip_at on. part needs
// ceil(n / ROUTE_TPB) * E doubles.
int launch_skip_mass(const float* logits, int64_t n, int E, int64_t ld, int k, int64_t skip_at, int64_t skip_len,
                     double* part, double* mass, cudaStream_t s) {
  const int64_t nblocks = (n + ROUTE_TPB - 1) / ROUTE_TPB;
  auto kern = E <= 128 ? k_route<1, 4> : k_route<1, 8>;
  kern<<<static_cast<unsigned>(nblocks), ROUTE_THREADS, 0, s>>>(logits, n, E, ld, E, k, nullptr, nullptr, part, nullptr,
                                                                skip_at, skip_len, RouteSrc{}, RouteDispatch{}, nullptr,
                                                                0);
  DM_LAUNCH_CHECK("k_route");
  k_mass_finalize<<<E, 256, 0, s>>>(part, static_cast<int>(nblocks), E, mass);
  DM_LAUNCH_CHECK("k_mass_finalize");
  return DECOMOE_OK;
}

}  // namespace decomoe

using namespace decomoe;

extern "C" {

int decomoe_router_logits(const void* x, const void* w_r, const float* bias, int64_t T, int d,
                          int E, int dtype, float* logits, int32_t* status_dev,
                          decomoe_stream_t stream) {
  clear_error();
  DM_ARG_CHECK(T >= 0 && d > 0 && E > 0, "router_logits: bad sizes T=%lld d=%d E=%d", (long long)T, d, E);
  DM_ARG_CHECK(dtype == DECOMOE_BF16 || dtype == DECOMOE_F32, "router_logits: bad dtype %d", dtype);
  if (T == 0) return DECOMOE_OK;
  DM_ARG_CHECK(x && w_r && logits, "router_logits: null pointer");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (dtype == DECOMOE_BF16 && T <= router_gemv_max_t() && d % 8 == 0 && aligned16(x) && aligned16(w_r)) {
    const dim3 grid(static_cast<unsigned>(E), static_cast<unsigned>((T + GEMV_TPB - 1) / GEMV_TPB));
    DM_CUDA_CHECK(launch_pdl(k_router_gemv, grid, dim3(GEMV_THREADS), 0, s, static_cast<const uint4*>(x),
                             static_cast<const uint4*>(w_r), bias, static_cast<int64_t>(T), d / 8, E, logits));
    return DECOMOE_OK;
  }
  if (dtype == DECOMOE_BF16 && router_tc_supported(d, E)) {
    DM_ARG_CHECK(aligned16(x) && aligned16(w_r) && aligned16(logits),
                 "router_logits: pointers must be 16-byte aligned");
    return launch_router_tc(x, w_r, bias, T, d, E, logits, status_dev, s);
  }
  const bool f32 = dtype == DECOMOE_F32;
  const bool vec = d % (f32 ? 4 : 8) == 0 && aligned16(x) && aligned16(w_r);
  const dim3 grid(static_cast<unsigned>((T + RS_RT - 1) / RS_RT),
                  static_cast<unsigned>(std::min((E + RS_WARPS * RS_NR - 1) / (RS_WARPS * RS_NR), 65535)));
  auto go = [&](auto kern, auto type) -> int {
    using S = decltype(type);
    DM_CUDA_CHECK(launch_pdl(kern, grid, dim3(32 * RS_WARPS), 0, s, static_cast<const S*>(x),
                             static_cast<const S*>(w_r), bias, T, d, E, logits));
    return DECOMOE_OK;
  };
  if (f32) return go(vec ? k_router_rows<float, 4> : k_router_rows<float, 1>, 0.f);
  return go(vec ? k_router_rows<__nv_bfloat16, 8> : k_router_rows<__nv_bfloat16, 1>, __nv_bfloat16());
}

size_t decomoe_router_logits_ws_bytes(int64_t T, int d, int E) {
  if (T <= 0 || d <= 0 || E <= 0) return 0;
  if (T <= router_gemv_max_t()) return 0;
  const int ks = router_split_ks(T, d, E);
  return ks > 1 ? align_up(static_cast<size_t>(ks) * T * E * sizeof(float), 256) : 0;
}

int decomoe_router_logits_ws(const void* x, const void* w_r, const float* bias, int64_t T, int d, int E, int dtype,
                             float* logits, void* ws, size_t ws_bytes, int32_t* status_dev, decomoe_stream_t stream) {
  clear_error();
  const size_t need = decomoe_router_logits_ws_bytes(T, d, E);
  if (dtype != DECOMOE_BF16 || need == 0 || T <= router_gemv_max_t())
    return decomoe_router_logits(x, w_r, bias, T, d, E, dtype, logits, status_dev, stream);
  DM_ARG_CHECK(x && w_r && logits, "router_logits_ws: null pointer");
  DM_ARG_CHECK(aligned16(x) && aligned16(w_r) && aligned16(logits) && aligned16(ws),
               "router_logits_ws: pointers must be 16-byte aligned");
  if (ws == nullptr || ws_bytes < need) {
    set_error("router_logits_ws: workspace needs %zu bytes", need);
    return DECOMOE_ERR_WORKSPACE;
  }
  return launch_router_split(x, w_r, bias, T, d, E, logits, static_cast<float*>(ws), status_dev,
                             reinterpret_cast<cudaStream_t>(stream));
}

size_t decomoe_route_workspace_bytes(int64_t T, int E) {
  if (T < 0 || E <= 0) return 0;
  const int64_t nblocks = (T + ROUTE_TPB - 1) / ROUTE_TPB;
  return align_up(static_cast<size_t>(nblocks > 0 ? nblocks : 1) * E * sizeof(double), 256);
}

int decomoe_route_prefix(const float* logits, int64_t T, int E, int64_t ld, int K, int k,
                         int32_t* topk_idx, float* topk_w, double* mass_out, void* ws,
                         size_t ws_bytes, decomoe_stream_t stream) {
  clear_error();
  return route_prefix_src(logits, RouteSrc{}, T, E, ld, K, k, topk_idx, topk_w, mass_out, ws, ws_bytes, false,
                          nullptr, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"

namespace decomoe {

int route_prefix_src(const float* logits, const RouteSrc& src, int64_t T, int E, int64_t ld, int K, int k,
                     int32_t* topk_idx, float* topk_w, double* mass_out, void* ws, size_t ws_bytes,
                     bool defer_finalize, int* mass_blocks, cudaStream_t s, const int32_t* K_dev,
                     const RouteDispatch* rd, int32_t* zero_ints, int n_zero) {
  if (mass_blocks != nullptr) *mass_blocks = 0;
  DM_ARG_CHECK(T >= 0, "route_prefix: T < 0");
  DM_ARG_CHECK(E >= 1 && E <= DECOMOE_MAX_E, "route_prefix: E=%d outside [1, %d]", E, DECOMOE_MAX_E);
  DM_ARG_CHECK(k >= 1 && k <= DECOMOE_MAX_TOPK, "route_prefix: k=%d outside [1, %d]", k, DECOMOE_MAX_TOPK);
  DM_ARG_CHECK(K_dev != nullptr || (K >= k && K <= E), "route_prefix: need k <= K <= E (k=%d K=%d E=%d)", k, K, E);
  DM_ARG_CHECK(K_dev == nullptr || mass_out == nullptr, "route_prefix: a device prefix takes no mass");
  DM_ARG_CHECK(ld >= E, "route_prefix: ld < E");
  DM_ARG_CHECK(src.nparts == 1 || ((src.nparts == 4 || src.nparts == 16) && E % 4 == 0 && ld == E &&
                                    src.part_stride % 4 == 0 && aligned16(logits) &&
                                    (src.bias == nullptr || aligned16(src.bias)) &&
                                    (src.logits_out == nullptr || aligned16(src.logits_out))),
               "route_prefix: logit slices need 4 or 16 slices of 16-byte aligned rows");
  if (T == 0) {
    if (mass_out) DM_CUDA_CHECK(cudaMemsetAsync(mass_out, 0, sizeof(double) * E, s));
    return DECOMOE_OK;
  }
  DM_ARG_CHECK(logits != nullptr, "route_prefix: logits is null");
  const int64_t nblocks = (T + ROUTE_TPB - 1) / ROUTE_TPB;
  DM_ARG_CHECK(nblocks <= 0x7fffffff, "route_prefix: T too large");
  double* part = nullptr;
  if (mass_out != nullptr) {
    if (ws == nullptr || ws_bytes < decomoe_route_workspace_bytes(T, E)) {
      set_error("route_prefix: workspace needs %zu bytes", decomoe_route_workspace_bytes(T, E));
      return DECOMOE_ERR_WORKSPACE;
    }
    // one routing block: its partial is the mass itself (the fixed-order
    // finalize would only add zeros), so it is written in place
    part = nblocks == 1 ? mass_out : static_cast<double*>(ws);
  }
  RouteDispatch rdv;
  if (rd != nullptr && rd->counts != nullptr) {
    DM_ARG_CHECK(nblocks == 1 && topk_idx != nullptr && T * k <= DSP_TILE,
                 "route_prefix: dispatch in the routing block needs T <= %d", ROUTE_TPB);
    rdv = *rd;
  }
  auto kern = E <= 128 ? (src.nparts == 16 ? k_route<16, 4> : src.nparts == 4 ? k_route<4, 4> : k_route<1, 4>)
                       : (src.nparts == 16 ? k_route<16, 8> : src.nparts == 4 ? k_route<4, 8> : k_route<1, 8>);
  DM_CUDA_CHECK(launch_pdl(kern, dim3(static_cast<unsigned>(nblocks)), dim3(ROUTE_THREADS), 0, s, logits, T, E, ld,
                           K, k, topk_idx, topk_w, part, K_dev, INT64_MAX, static_cast<int64_t>(0), src, rdv,
                           zero_ints, n_zero));
  if (mass_out != nullptr && nblocks > 1) {
    if (defer_finalize && mass_blocks != nullptr) {
      *mass_blocks = static_cast<int>(nblocks);  // the caller's next kernel adds the partials up
    } else {
      DM_CUDA_CHECK(launch_pdl(k_mass_finalize, dim3(E), dim3(256), 0, s, static_cast<const double*>(part),
                               static_cast<int>(nblocks), E, mass_out));
    }
  }
  return DECOMOE_OK;
}

}  // namespace decomoe

extern "C" {


int decomoe_select_prefix_device(const double* mass, int E, int k, double p, int32_t* K_dev,
                                 decomoe_stream_t stream) {
  clear_error();
  DM_ARG_CHECK(mass && K_dev, "select_prefix_device: null pointer");
  DM_ARG_CHECK(E >= 1 && k >= 1 && k <= E, "select_prefix_device: need 1 <= k <= E");
  DM_ARG_CHECK(p > 0.0 && p <= 1.0, "select_prefix_device: p must lie in (0, 1]");
  DM_CUDA_CHECK(launch_pdl(k_select_prefix, dim3(1), dim3(DECOMOE_MAX_E), 0, reinterpret_cast<cudaStream_t>(stream), mass, E, k,
                           p, K_dev));
  return DECOMOE_OK;
}

int decomoe_route_prefix_dk(const float* logits, int64_t T, int E, int64_t ld, const int32_t* K_dev, int k,
                            int32_t* topk_idx, float* topk_w, decomoe_stream_t stream) {
  clear_error();
  DM_ARG_CHECK(T >= 0 && E >= 1 && E <= DECOMOE_MAX_E && k >= 1 && k <= DECOMOE_MAX_TOPK && k <= E && ld >= E,
               "route_prefix_dk: bad sizes");
  if (T == 0) return DECOMOE_OK;
  DM_ARG_CHECK(logits && K_dev, "route_prefix_dk: null pointer");
  return route_prefix_src(logits, RouteSrc{}, T, E, ld, E, k, topk_idx, topk_w, nullptr, nullptr, 0, false, nullptr,
                          reinterpret_cast<cudaStream_t>(stream), K_dev);
}

}  // extern "C"
