// Expert FFN on pairs of SMs (tcgen05 cta_group::2): gate/up with SwiGLU, down,
// or both in one persistent launch. Included by expert_gemm.cu.
//
// A cluster of two CTAs computes one tile of 256 rows x 256 weight rows. CTA r
// holds rows [128 r, 128 r + 128) of the row tile (A) and weight rows [128 r,
// 128 r + 128) (B). A row tile of at most 128 rows is an M = 128 product with 64
// rows per CTA: its k-blocks take as long in the tensor pipe (a gate/up item
// 20200 cycles against 19900), but half the row traffic (T = 2048, K = 64 184 us
// a layer, with full tiles throughout 194). One thread of CTA 0 issues M = 256,
// N = 256 products that read both CTAs' operands, and each CTA's tensor memory
// receives its 128 rows x 256 columns. Why pairs: at 128 x 256 on one SM a 64-deep k-block moves 48 KB
// into shared memory and the products read 48 KB back, 768 cycles of its 128
// bytes a cycle against 512 of tensor work; half the weights per SM make that
// 512 against 512, and six k-blocks are on their way instead of four. Weights and
// rows have rings of their own, filled by different threads: weights stream on
// while rows wait for h or for their token numbers.
//
// Rows of the gate/up operand come from x by index (gather mode: four warps
// copy them with cp.async, coalesced, in the swizzle the TMA would produce: no
// gathered copy of x is written or read) or from grouped rows by TMA.
//
// Per k-block each CTA's loads complete on its own barriers; a relay thread in
// each passes them on to CTA 0's LOADED, the one barrier its MMA warp waits
// for. The commits arrive on both CTAs' EMPTY and TFULL
// barriers; both CTAs' epilogue warps arrive on CTA 0's TEMPTY. All waits are
// bounded: on expiry the role reports, its CTA's other roles stop, the peer's
// waits run out, in-flight copies and products are waited for, and both CTAs
// meet at the closing cluster barrier, so neither leaves while the other can
// still reach its shared memory.
//
// What bounds it: with weights in L2 and 4096 rows an expert (d = 2048, m = 768)
// gate/up runs at 1805 TFLOP/s and down at 1560, against 1547 and 1148 of the
// one-SM kernels before, near the power limit; with few rows an expert the
// weight stream. The MMA warp's loop decides: issued by one thread of a divergent
// branch with two barriers per k-block, the same kernel took 637 cycles per
// k-block (gate/up 1576 TFLOP/s) instead of 512, and an arrival with cluster
// release 1900. Layer against the one-SM kernels: T = 2048, K = 64 222 -> 187 us;
// 4096 361 -> 282; 16384, K = 128 1272 -> 1029 (two launches); 1552, K = 128 237 -> 216; 272, K =
// 57 114 -> 106; 131, K = 64 97.6 -> 91.3. With one ring for both operands it had
// been 199, 301, 1037 (in one launch), 228, 109 and 93.7; with eight slots for weights and four
// for rows gate/up from L2 ran at 1654 TFLOP/s instead of 1805.
#pragma once

namespace decomoe {

constexpr int PF_BM = 128;                  // rows per CTA (256 per tile)
constexpr int PF_BN = 256;                  // weight rows per tile (128 per CTA)
constexpr int PF_BK = 64;
constexpr int PF_NB = 6, PF_NA = 6;         // ring slots for weights and for rows
static_assert(PF_NA <= PF_NB, "the rows' slots are freed through the weights' barriers");
constexpr int PF_HALF = 128 * PF_BK * 2;    // A or B of one k-block and CTA (16 KB)
constexpr int PF_EW = 8;                    // epilogue warps
constexpr int PF_GW = 4;                    // gather warps
constexpr int PF_THREADS = 96 + 32 * (PF_EW + PF_GW);  // TMA, MMA, relay, epilogue and gather warps
constexpr int PF_STG = 32 * 64;             // store staging per epilogue warp: 32 rows x 64 bytes
constexpr int PF_NBARS = 3 * PF_NB + 2 * PF_NA + 5;
constexpr size_t PF_SMEM = 1024 + static_cast<size_t>(PF_NA + PF_NB) * PF_HALF + PF_EW * PF_STG + PF_NBARS * 8 +
                           2 * (DECOMOE_MAX_E + 1) * 4 + 16;
static_assert(PF_SMEM <= 232448, "shared memory budget");
static_assert(PF_SMEM > 232448 / 2, "one CTA per SM: the dependency waits need every CTA resident");

struct PairArgs {
  const int32_t* offsets;  // [G + 1]
  int G;
  int d, m;
  int gu, dn;           // which halves of the FFN this launch computes
  void* h;              // [rows, m] bf16
  void* y;              // [rows, d] bf16
  int32_t* ready;       // gate/up and down together: per 128-row half tile, gate/up tiles stored (zero at launch)
  int32_t* status;
  uint64_t limit_ns;
  const uint8_t* x;     // gather mode: [tokens, d] bf16, else null (grouped rows by TMA)
  const int32_t* perm;  // gather mode: [rows] token of each grouped row
  uint8_t* x_copy;      // gather mode: receives the grouped rows [rows, d] too, or null
};

// ---- cluster and cta_group::2 wrappers
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrive (count 1) on the barrier at `bar`'s offset in CTA `rank` of the pair.
// What the arrival passes on was written by copies whose completion this
// thread has observed, or is tensor memory read before the tcgen05 fence: no
// cluster-scope release is needed, which would wait for every store of the
// thread's SM in flight (1430 cycles per k-block).
__device__ __forceinline__ void mbar_arrive_rank(uint32_t bar, uint32_t rank) {
  asm volatile(
      "{\n\t.reg .b32 ra;\n\t"
      "mapa.shared::cluster.u32 ra, %0, %1;\n\t"
      "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}" ::"r"(bar),
      "r"(rank)
      : "memory");
}
// mbar_wait of a whole warp with time to spare: it sleeps between tests (they
// read shared memory, whose bandwidth the products need).
__device__ __forceinline__ bool mbar_wait_idle(uint32_t bar, uint32_t parity, uint64_t limit_ns, volatile int* abort,
                                               uint32_t sleep_ns) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    __nanosleep(sleep_ns);
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if (__any_sync(0xffffffffu, *abort != 0 || globaltimer_ns() - t0 > limit_ns)) return false;
  }
}
__device__ __forceinline__ void tc2_mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on `bar` in both CTAs when all prior products of this thread completed.
__device__ __forceinline__ void tc2_commit_both(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}
__device__ __forceinline__ void tmem2_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem2_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem2_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PF_THREADS, 1)
    k_ffn_pair(const __grid_constant__ CUtensorMap tma_a1, const __grid_constant__ CUtensorMap tma_b1,
               const __grid_constant__ CUtensorMap tma_a2, const __grid_constant__ CUtensorMap tma_b2,
               const __grid_constant__ CUtensorMap tma_a1s, const __grid_constant__ CUtensorMap tma_a2s,
               const PairArgs g) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;  // the same in both CTAs: one kernel, one layout
  uint8_t* smem = smem_raw + pad;
  const uint32_t sA = raw + pad;
  const uint32_t sB = sA + PF_NA * PF_HALF;
  uint8_t* stg = smem + (PF_NA + PF_NB) * PF_HALF;
  uint64_t* bars = reinterpret_cast<uint64_t*>(stg + PF_EW * PF_STG);
  int* s_off = reinterpret_cast<int*>(bars + PF_NBARS);
  int* s_mt = s_off + (DECOMOE_MAX_E + 1);
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(s_mt + (DECOMOE_MAX_E + 1));
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const uint32_t bar0 = smem_u32(bars);
  // k-block c (counted over the CTA's items) has its weights in slot c % PF_NB
  // and its rows in slot c % PF_NA
  auto FULLB = [&](int s) { return bar0 + 8u * s; };                     // weights loaded (this CTA)
  auto LOADED = [&](int s) { return bar0 + 8u * (PF_NB + s); };          // CTA 0: the k-block is loaded in both CTAs
  auto EMPTY = [&](int s) { return bar0 + 8u * (2 * PF_NB + s); };       // products have read the k-block of weight slot s
  auto FULLA = [&](int s) { return bar0 + 8u * (3 * PF_NB + s); };       // rows loaded by TMA (this CTA)
  auto ROWS = [&](int s) { return bar0 + 8u * (3 * PF_NB + PF_NA + s); };  // rows gathered (this CTA)
  auto TFULL = [&](int a) { return bar0 + 8u * (3 * PF_NB + 2 * PF_NA + a); };
  auto TEMPTY = [&](int a) { return bar0 + 8u * (3 * PF_NB + 2 * PF_NA + 2 + a); };  // CTA 0: both epilogues are done
  const uint32_t DRAIN = bar0 + 8u * (3 * PF_NB + 2 * PF_NA + 4);

  const int G = g.G;
  if (threadIdx.x == 0) {
    *s_abort = 0;
    for (int s = 0; s < PF_NB; ++s) {
      mbar_init(FULLB(s), 1);
      mbar_init(LOADED(s), 2);
      mbar_init(EMPTY(s), 1);
    }
    for (int s = 0; s < PF_NA; ++s) {
      mbar_init(FULLA(s), 1);
      mbar_init(ROWS(s), 32 * PF_GW);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(TFULL(a), 1);
      mbar_init(TEMPTY(a), 2 * PF_EW);
    }
    mbar_init(DRAIN, 1);
    fence_mbar_init();
  }
  pdl_wait();
  for (int i = threadIdx.x; i <= G; i += PF_THREADS) s_off[i] = g.offsets[i];
  __syncthreads();
  if (warp == 2) {
    // exclusive scan of 256-row tiles per group: s_mt[e] = first tile of e
    const int per = (G + 31) / 32;  // <= 8
    int loc[8];
    int sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      loc[i] = 0;
      const int gi = lane * per + i;
      if (i < per && gi < G) {
        const int n = s_off[gi + 1] - s_off[gi];
        loc[i] = n > 0 ? (n + 2 * PF_BM - 1) / (2 * PF_BM) : 0;
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
      if (i < per && gi < G) s_mt[gi] = run;
      run += loc[i];
    }
    if (lane == 31) s_mt[G] = incl;
  }
  __syncthreads();
  const int NT1 = 2 * g.m / PF_BN, NT2 = g.d / PF_BN;
  const int total1 = g.gu ? s_mt[G] * NT1 : 0;
  const int total = total1 + (g.dn ? s_mt[G] * NT2 : 0);
  const int cid = static_cast<int>(blockIdx.x) >> 1, ncl = static_cast<int>(gridDim.x) >> 1;
  if (cid >= total) return;  // both CTAs of the pair, before any cluster barrier, TMEM or TMA use

  if (warp == 1) {
    tmem2_alloc(smem_u32(const_cast<uint32_t*>(s_tmem)), 512);
    tmem2_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  pair_sync();  // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  struct Item {
    bool dn;
    int grp, nb, mtg;  // group, N-tile, row tile (over all groups)
    bool half;         // M = 128 tile (64 rows per CTA): a row tile of at most 128 rows
    int row0, nrow;    // this CTA's first row and how many of its 128 (64) exist
  };
  auto item = [&](int t) -> Item {
    Item r;
    int mt;
    r.dn = t >= total1;
    tile_coords(r.dn ? t - total1 : t, r.dn ? NT2 : NT1, s_mt, G, r.grp, mt, r.nb);
    r.mtg = s_mt[r.grp] + mt;
    const int first = s_off[r.grp] + 2 * mt * PF_BM, end = s_off[r.grp + 1];
    r.half = end - first <= PF_BM;
    const int mine = r.half ? PF_BM / 2 : PF_BM;
    r.row0 = first + static_cast<int>(rank) * mine;
    r.nrow = min(max(end - r.row0, 0), mine);
    return r;
  };
  const bool gather = g.x != nullptr;
  const bool dep = g.gu && g.dn;  // down tiles wait for the gate/up tiles of this launch

  if (warp == 0) {
    // ------------------------------------------------ weights by TMA (lane 0)
    if (lane == 0) {
      tma_prefetch_desc(&tma_b1);
      tma_prefetch_desc(&tma_b2);
      int stage = 0;
      uint32_t ph = 0;
      bool ok = true;
      uint32_t armed = 0, armed_ph = 0;
      const uint64_t pol_once = policy_evict_first();
      for (int t = cid; ok && t < total; t += ncl) {
        const Item it = item(t);
        const CUtensorMap* tb = it.dn ? &tma_b2 : &tma_b1;
        const int brow = it.grp * (it.dn ? g.d : 2 * g.m) + it.nb * PF_BN + static_cast<int>(rank) * 128;
        const int KB = (it.dn ? g.m : g.d) / PF_BK;
        // weights that one row tile reads go to L2 as evict-first
        const bool once = s_mt[it.grp + 1] - s_mt[it.grp] == 1;
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(EMPTY(stage), ph ^ 1u, g.limit_ns, s_abort)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(FULLB(stage), PF_HALF);
          if (once)
            tma_load_2d_hint(sB + stage * PF_HALF, tb, FULLB(stage), kb * PF_BK, brow, pol_once);
          else
            tma_load_2d(sB + stage * PF_HALF, tb, FULLB(stage), kb * PF_BK, brow);
          armed |= 1u << stage;
          armed_ph = (armed_ph & ~(1u << stage)) | (ph << stage);
          if (++stage == PF_NB) {
            stage = 0;
            ph ^= 1u;
          }
        }
      }
      int no_abort = 0;
      if (!ok) {
        *s_abort = 1;
        report_status(g.status, DECOMOE_ERR_TIMEOUT);
        for (int s = 0; s < PF_NB; ++s)
          if ((armed >> s) & 1u) mbar_wait(FULLB(s), (armed_ph >> s) & 1u, g.limit_ns, &no_abort);
      } else {
        // the last products' arrivals land here before the CTA may leave
        for (int s = 0; s < PF_NB; ++s)
          if ((armed >> s) & 1u) mbar_wait(EMPTY(s), (armed_ph >> s) & 1u, g.limit_ns, s_abort);
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ------------------------------------------------ MMA issuer: the whole
      // warp runs the loop (its values stay in uniform registers), one elected
      // thread issues. One barrier to wait for per k-block: at 512 cycles of
      // products each, what this loop spends between them is lost.
      const bool leader = elect_one();
      const uint64_t ad0 = smem_desc_kmajor<PF_BK>(sA), bd0 = smem_desc_kmajor<PF_BK>(sB);
      int stage = 0, rows = 0;  // weight slot, row slot
      uint32_t ph = 0;
      bool ok = true, issued = false;
      int n = 0;
      bool half = item(cid).half, half_next = false;
      for (int t = cid; ok && t < total; t += ncl, ++n) {
        const int KB = (t >= total1 ? g.m : g.d) / PF_BK;
        const uint32_t idesc = half ? idesc_bf16_f32(PF_BM, PF_BN) : idesc_bf16_f32(2 * PF_BM, PF_BN);
        const int acc = n & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(TEMPTY(acc), ((n >> 1) & 1) ^ 1u, g.limit_ns, s_abort))) {
          ok = false;
          break;
        }
        const uint32_t dt = tmem_base + static_cast<uint32_t>(acc * PF_BN);
        for (int kb = 0; kb < KB; ++kb) {
          if (!__all_sync(0xffffffffu, mbar_wait(LOADED(stage), ph, g.limit_ns, s_abort))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = ad0 + static_cast<uint32_t>(rows * (PF_HALF >> 4));
          const uint64_t bd = bd0 + static_cast<uint32_t>(stage * (PF_HALF >> 4));
          if (leader) {
            tc2_mma_f16(dt, ad, bd, idesc, kb != 0 ? 1u : 0u);
#pragma unroll
            for (int kk = 1; kk < PF_BK / 16; ++kk) tc2_mma_f16(dt, ad + 2u * kk, bd + 2u * kk, idesc, 1u);
            tc2_commit_both(EMPTY(stage));
            if (kb == KB - 1) tc2_commit_both(TFULL(acc));
          }
          if (kb == 0) half_next = t + ncl < total && item(t + ncl).half;  // while the products run
          issued = true;
          if (++rows == PF_NA) rows = 0;
          if (++stage == PF_NB) {
            stage = 0;
            ph ^= 1u;
          }
        }
        half = half_next;
      }
      if (!ok && leader) {
        *s_abort = 1;
        report_status(g.status, DECOMOE_ERR_TIMEOUT);
        if (issued) {
          int no_abort = 0;
          tc2_commit_both(DRAIN);
          mbar_wait(DRAIN, 0, g.limit_ns, &no_abort);
        }
      }
    }
  } else if (warp == PF_EW + PF_GW + 2) {
    // ------------------------------------------------ relay: this CTA's part of
    // each k-block is in shared memory
    if (lane == 0) {
      uint32_t b = 0, a = 0, pb = 0;  // weight slot, row slot, the weight ring's phase
      uint32_t pt = 0, pg = 0;        // phase per row slot: rows by TMA, gathered
      bool ok = true;
      for (int t = cid; ok && t < total; t += ncl) {
        const bool rows = gather && t < total1;
        const int KB = (t >= total1 ? g.m : g.d) / PF_BK;
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(FULLB(b), pb, g.limit_ns, s_abort) ||
              !(rows ? mbar_wait(ROWS(a), pg >> a & 1u, g.limit_ns, s_abort)
                     : mbar_wait(FULLA(a), pt >> a & 1u, g.limit_ns, s_abort))) {
            ok = false;
            break;
          }
          if (rows) {
            fence_proxy_async_smem();  // cp.async rows, read by the tensor cores
            pg ^= 1u << a;
          } else {
            pt ^= 1u << a;
          }
          mbar_arrive_rank(LOADED(b), 0);
          if (++a == PF_NA) a = 0;
          if (++b == PF_NB) b = 0, pb ^= 1u;
        }
      }
      if (!ok) {
        *s_abort = 1;
        report_status(g.status, DECOMOE_ERR_TIMEOUT);
      }
    }
  } else if (warp < 2 + PF_EW) {
    // ------------------------------------------------ epilogue
    const int q = warp & 3;               // tensor-memory lane quarter
    const int wp = (warp - 2) >> 2;       // which of the quarter's two warps
    uint8_t* my = stg + (warp - 2) * PF_STG;
    bool ok = true;
    int n = 0;
    for (int t = cid; t < total; t += ncl, ++n) {
      const Item it = item(t);
      const int acc = n & 1;
      if (ok && g.x_copy != nullptr && !it.dn) {
        // the grouped rows are wanted too: this item's share (rows dealt over
        // the row tile's gate/up items), while its accumulator is computed
        const int vec = g.d / 8, per = (it.nrow + NT1 - 1) / NT1;
        const int a = min(it.nb * per, it.nrow), nv = (min(a + per, it.nrow) - a) * vec;
        for (int i0 = threadIdx.x - 64; i0 < nv; i0 += 32 * PF_EW * 4) {
          uint4 v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 32 * PF_EW;
            if (i < nv)
              v[u] = __ldg(reinterpret_cast<const uint4*>(g.x) +
                           static_cast<int64_t>(g.perm[it.row0 + a + i / vec]) * vec + i % vec);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 32 * PF_EW;
            if (i < nv) reinterpret_cast<uint4*>(g.x_copy)[(static_cast<int64_t>(it.row0) + a) * vec + i] = v[u];
          }
        }
        __syncwarp();
      }
      // a warp whose wait ran out stores nothing more, but goes on to the barrier
      // that the others may have reached
      if (ok && !mbar_wait_idle(TFULL(acc), (n >> 1) & 1, g.limit_ns, s_abort, 100)) {
        ok = false;
        *s_abort = 1;
      }
      tc_fence_after();
      const uint32_t tb = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(acc * PF_BN);
      // lanes 32 q ..: rows 32 q .. of the CTA's 128 and all 256 columns; of an M
      // = 128 tile rows 32 (q & 1) .. of its 64 and columns 128 (q >> 1) ..
      const int r0 = it.half ? (q & 1) * 32 : q * 32;
      const int col0 = it.half ? (q >> 1) * (PF_BN / 2) : 0;
      const int ncol = it.half ? PF_BN / 2 : PF_BN;
      const int nmine = it.nrow - r0;  // rows of this warp that exist
      // 32 rows x 32 bf16 columns (pk: this lane's row) to out, whole 64-byte
      // segments: through the warp's staging rows, eight rows per store
      auto store = [&](const uint32_t (&pk)[16], __nv_bfloat16* out, int64_t ld) {
        uint4* w = reinterpret_cast<uint4*>(my + lane * 64);
#pragma unroll
        for (int v = 0; v < 4; ++v)
          w[v ^ ((lane >> 1) & 3)] = make_uint4(pk[4 * v], pk[4 * v + 1], pk[4 * v + 2], pk[4 * v + 3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = 8 * i + (lane >> 2), v = lane & 3;
          const uint4 u = reinterpret_cast<const uint4*>(my + r * 64)[v ^ ((r >> 1) & 3)];
          if (r < nmine) *reinterpret_cast<uint4*>(out + r * ld + 8 * v) = u;
        }
        __syncwarp();
      };
      if (ok && nmine > 0) {
        const int64_t row = it.row0 + r0;
        if (!it.dn) {
          constexpr int GU = DECOMOE_GU_BLOCK;
          __nv_bfloat16* out = static_cast<__nv_bfloat16*>(g.h) + row * g.m + it.nb * (PF_BN / 2) + col0 / 2;
#pragma unroll 1
          for (int cc = 32 * wp; cc < ncol / 2; cc += 64) {
            const int half = cc / GU, c = cc % GU;
            uint32_t gr[32], ur[32];
            tmem_ld32(tb + half * 2 * GU + c, gr);
            tmem_ld32(tb + half * 2 * GU + GU + c, ur);
            tc_wait_ld();
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float g0 = __uint_as_float(gr[2 * i]), g1 = __uint_as_float(gr[2 * i + 1]);
              const float u0 = __uint_as_float(ur[2 * i]), u1 = __uint_as_float(ur[2 * i + 1]);
              pk[i] = pack_bf16x2(silu_f(g0) * u0, silu_f(g1) * u1);
            }
            store(pk, out + cc, g.m);
          }
        } else {
          __nv_bfloat16* out = static_cast<__nv_bfloat16*>(g.y) + row * g.d + it.nb * PF_BN + col0;
#pragma unroll 1
          for (int c = 32 * wp; c < ncol; c += 64) {
            uint32_t r[32];
            tmem_ld32(tb + c, r);
            tc_wait_ld();
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) pk[i] = pack_bf16x2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
            store(pk, out + c, g.d);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_rank(TEMPTY(acc), 0);
      if (!it.dn && dep) {
        // this CTA's h columns of the tile are stored: publish them to the down tiles
        fence_proxy_async_all();
        named_bar_sync(1, 32 * PF_EW);
        if (ok && warp == 2 && lane == 0) {
          __threadfence();
          atomicAdd(g.ready + 2 * it.mtg + rank, 1);
        }
      }
    }
    if (!ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
    }
  } else {
    // ------------------------------------------------ rows: gate/up items by
    // index (four warps; eight lanes take one row's 128 bytes of the k-block,
    // four rows per copy), grouped rows and h by TMA (one thread)
    const int gw = warp - 2 - PF_EW;
    // k-block c takes row slot a once the products of k-block c - PF_NA are
    // done, which the barrier of that one's weight slot eb says. It cannot be a
    // phase ahead of this wait: that would need k-block c's products.
    uint32_t a = 0, eb = 0, pe = 0;
    int unused = PF_NA;  // slots not taken yet
    auto slot_next = [&]() {
      if (++a == PF_NA) a = 0;
      if (unused > 0) {
        --unused;
      } else if (++eb == PF_NB) {
        eb = 0;
        pe ^= 1u;
      }
    };
    bool ok = true;
    int t = cid;
    const int sub = lane >> 3, ch = lane & 7;
    // an item's rows and tokens are looked up half an item ahead: the ring holds
    // less time than that chain of loads takes (gate/up by index 1559 -> 1660
    // TFLOP/s with weights in L2, T = 16384 1023 -> 1000 us a layer)
    Item it = item(t), it_next = it;
    int tok[8];
    auto tokens = [&](const Item& i2, bool any) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = 32 * gw + 4 * i + sub;
        tok[i] = any && r < i2.nrow ? g.perm[i2.row0 + r] : -1;
      }
    };
    if (gather && t < total1) tokens(it, true);
    for (; gather && ok && t < total1; t += ncl) {
      it = it_next;
      const uint8_t* src[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        src[i] = tok[i] >= 0 ? g.x + (static_cast<int64_t>(tok[i]) * g.d + 8 * ch) * 2 : nullptr;
      const int KB = g.d / PF_BK;
      for (int kb = 0; kb < KB; ++kb, slot_next()) {
        if (kb == KB / 2 && t + ncl < total) {
          it_next = item(t + ncl);
          tokens(it_next, t + ncl < total1);
        }
        if (unused == 0 && !mbar_wait_idle(EMPTY(eb), pe, g.limit_ns, s_abort, 20)) {
          ok = false;
          break;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (src[i] != nullptr) {
            const int r = 32 * gw + 4 * i + sub;
            cp_async16(sA + a * PF_HALF + r * 128 + ((ch ^ (r & 7)) << 4), src[i] + kb * (PF_BK * 2));
          }
        cp_async_mbar_arrive_noinc(ROWS(a));
      }
    }
    cp_async_wait_all();
    if (ok && gw == 0 && lane == 0) {
      tma_prefetch_desc(&tma_a1);
      tma_prefetch_desc(&tma_a2);
      uint32_t armed = 0, pt = 0;  // slots with a copy in flight; phase per slot
      // readiness of this CTA's rows of a down item, acquire-loaded one item
      // ahead (an acquire holds up the thread's later loads)
      auto ready_of = [&](const Item& i2) -> bool {
        if (!(dep && i2.dn && i2.nrow > 0)) return true;
        if (ld_acquire_gpu(g.ready + 2 * i2.mtg + rank) < NT1) return false;
        fence_proxy_async_all();  // h, written by generic stores, is read through TMA
        return true;
      };
      bool ready_next = t < total ? ready_of(it_next) : true;
      for (; ok && t < total; t += ncl) {
        it = it_next;
        const bool ready = ready_next;
        const CUtensorMap* ta = it.half ? (it.dn ? &tma_a2s : &tma_a1s) : (it.dn ? &tma_a2 : &tma_a1);
        const uint32_t bytes = it.half ? PF_HALF / 2 : PF_HALF;
        const int KB = (it.dn ? g.m : g.d) / PF_BK;
        if (!ready) {  // wait until every gate/up tile of these rows has stored its h
          const volatile int32_t* rp = g.ready + 2 * it.mtg + rank;
          const uint64_t t0 = globaltimer_ns();
          while (*rp < NT1) {
            if (*s_abort || globaltimer_ns() - t0 > g.limit_ns) {
              ok = false;
              break;
            }
          }
          if (!ok) break;
          __threadfence();
          fence_proxy_async_all();
        }
        for (int kb = 0; kb < KB; ++kb, slot_next()) {
          if (kb == 0 && t + ncl < total) {
            it_next = item(t + ncl);
            ready_next = ready_of(it_next);
          }
          if (unused == 0 && !mbar_wait(EMPTY(eb), pe, g.limit_ns, s_abort)) {
            ok = false;
            break;
          }
          if (it.nrow > 0) {
            mbar_arrive_expect_tx(FULLA(a), bytes);
            tma_load_2d(sA + a * PF_HALF, ta, FULLA(a), kb * PF_BK, it.row0);
            armed |= 1u << a;
          } else {
            mbar_arrive(FULLA(a));  // no rows of this CTA in the tile
            armed &= ~(1u << a);
          }
          pt ^= 1u << a;
        }
      }
      int no_abort = 0;
      if (!ok)
        for (int s = 0; s < PF_NA; ++s)
          if ((armed >> s) & 1u) mbar_wait(FULLA(s), ~(pt >> s) & 1u, g.limit_ns, &no_abort);
    }
    if (!ok) {
      *s_abort = 1;
      report_status(g.status, DECOMOE_ERR_TIMEOUT);
    }
  }
  __syncwarp();
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  pair_sync();  // neither CTA's shared or tensor memory is in use any more
  tc_fence_after();
  if (warp == 1) tmem2_dealloc(tmem_base, 512);
}

}  // namespace decomoe
