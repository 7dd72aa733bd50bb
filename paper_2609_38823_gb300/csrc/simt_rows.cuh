// CUDA-core matrix products of a few rows with row-major weights (fp32
// storage, and bf16 router shapes that the tensor cores do not take): every
// product is a row of A with a row of W, both contiguous. A warp takes RT
// rows and NR weight rows; its lanes split the inner dimension in VEC-element
// vectors (16 bytes where rows and pointers allow), so every load is
// coalesced and each is used by RT or NR products; the RT x NR partial sums
// of the 32 lanes are then added by a halving butterfly (RT*NR values in
// about RT*NR shuffles instead of five each). fp32 products and sums: 32
// interleaved partial sums per result, then a tree.
//
// Bound at these sizes: latency (a few loads deep); what counts is that the
// work spreads over the SMs. One thread per result with a serial inner loop
// over uncoalesced weight rows took, for the 64-token layer with d = 256,
// m = 128 and 16 experts, 21.6 us (router), 39.4 (gate/up) and 20.4 (down).
#pragma once

#include "decomoe_internal.cuh"

namespace decomoe {

// VEC consecutive elements as fp32 (VEC > 1: one 16-byte load).
template <typename T, int VEC>
__device__ __forceinline__ void load_row_vec(const T* __restrict__ p, float (&v)[VEC]) {
  if constexpr (VEC == 1) {
    if constexpr (sizeof(T) == 2)
      v[0] = __bfloat162float(*p);
    else
      v[0] = *p;
  } else {
    static_assert(VEC * sizeof(T) == 16, "one 16-byte vector");
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    if constexpr (sizeof(T) == 2) {
      v[0] = bf16_lo(u.x), v[1] = bf16_hi(u.x), v[2] = bf16_lo(u.y), v[3] = bf16_hi(u.y);
      v[4] = bf16_lo(u.z), v[5] = bf16_hi(u.z), v[6] = bf16_lo(u.w), v[7] = bf16_hi(u.w);
    } else {
      v[0] = __uint_as_float(u.x), v[1] = __uint_as_float(u.y);
      v[2] = __uint_as_float(u.z), v[3] = __uint_as_float(u.w);
    }
  }
}

// acc[r * NR + w] = this lane's part of a_r . w_w over n elements.
template <typename T, int VEC, int RT, int NR>
__device__ __forceinline__ void rows_dot(const T* const (&a)[RT], const T* const (&w)[NR], int n, int lane,
                                         float (&acc)[RT * NR]) {
#pragma unroll
  for (int i = 0; i < RT * NR; ++i) acc[i] = 0.f;
  for (int c = lane * VEC; c < n; c += 32 * VEC) {
    float av[RT][VEC], wv[NR][VEC];
#pragma unroll
    for (int r = 0; r < RT; ++r) load_row_vec<T, VEC>(a[r] + c, av[r]);
#pragma unroll
    for (int j = 0; j < NR; ++j) load_row_vec<T, VEC>(w[j] + c, wv[j]);
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int j = 0; j < NR; ++j)
#pragma unroll
        for (int i = 0; i < VEC; ++i) acc[r * NR + j] = fmaf(av[r][i], wv[j][i], acc[r * NR + j]);
  }
}

// Sums acc[i] over the warp's lanes; with N = 32 M results lane l ends with
// results l*M .. l*M + M-1 in acc[0..M). N < 32: lanes l with equal
// l / (32 / N) all hold result l / (32 / N) in acc[0].
template <int N>
__device__ __forceinline__ void warp_scatter_sum(float (&acc)[N], int lane) {
  static_assert((N & (N - 1)) == 0, "a power of two");
  int n = N;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool hi = (lane & off) != 0;
#pragma unroll
      for (int i = 0; i < N / 2; ++i)
        if (i < n) {
          const float send = hi ? acc[i] : acc[i + n];
          const float keep = hi ? acc[i + n] : acc[i];
          acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    } else {
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
    }
  }
}

// Group and first row of row chunk c (RT rows at most, within one group) of
// the grouped rows [offsets[g], offsets[g + 1]), g < G <= 256; one warp, lane
// l counts groups 8 l .. 8 l + 7. Returns false past the last chunk.
template <int RT>
__device__ __forceinline__ bool chunk_rows(const int32_t* __restrict__ offsets, int G, int64_t c, int lane, int& g,
                                           int& r0, int& r1) {
  int o[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) o[i] = offsets[min(8 * lane + i, G)];
  int64_t mine = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) mine += (o[i + 1] - o[i] + RT - 1) / RT;
  int64_t before = mine;  // inclusive scan over the lanes
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int64_t v = __shfl_up_sync(0xffffffffu, before, off);
    if (lane >= off) before += v;
  }
  const uint32_t past = __ballot_sync(0xffffffffu, before > c);
  if (past == 0u) return false;
  const int src = __ffs(past) - 1;
  int64_t left = c - (before - mine);
  int gg = 0, lo = 0, hi = 0;
  if (lane == src) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int n = (o[i + 1] - o[i] + RT - 1) / RT;
      if (left >= 0 && left < n) {
        gg = 8 * lane + i;
        lo = o[i] + static_cast<int>(left) * RT;
        hi = min(lo + RT, o[i + 1]);
      }
      left -= n;
    }
  }
  g = __shfl_sync(0xffffffffu, gg, src);
  r0 = __shfl_sync(0xffffffffu, lo, src);
  r1 = __shfl_sync(0xffffffffu, hi, src);
  return true;
}

}  // namespace decomoe
