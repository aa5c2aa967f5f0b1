// y = x W^T for many activation rows (or, from 33 rows on, a large matrix).
//
// Two CTAs on two SMs form one MMA unit (tcgen05 cta_group::2): the pair owns a [256 weight rows x BNT
// activation rows] tile of y^T.  Each CTA loads its own 128 weight rows and only HALF of the activation tile per
// k-step (the MMA reads the B operand from both CTAs' shared memory), which halves the shared-memory fill per
// flop compared with the one-CTA kernel; the accumulator lives in both CTAs' TMEM (128 lanes each).
// The kernel is persistent: one cluster per SM pair walks a static list of tiles; two TMEM accumulators
// alternate so the epilogue of one tile (tcgen05.ld -> global stores) overlaps the main loop of the next.
//
//   warp 0   TMA producer (both CTAs; both signal the LEADER CTA's "full" barrier)
//   warp 1   TMEM allocation (both CTAs), MMA issue + commits (leader CTA only, one thread)
//   warps 2..9  epilogue (both CTAs, their own 128 accumulator lanes): two warps per TMEM lane quarter take alternate groups
//               of 16 accumulator columns
// No TMA load is multicast; the only cluster-wide signal is tcgen05.commit to both CTAs' barriers.
//
// A pipeline stage holds TWO 64-column k-steps (64 KB per CTA at 256-wide tiles, three stages): every barrier round of
// the MMA thread (wait for "full", commit to "empty") costs the tensor pipe about 150 clocks whatever the order of the
// operations, so it is paid once per eight MMAs instead of once per four.  (Three k-steps per stage leave room for two
// stages only: 1 291 against 1 331 TFLOP/s on M = 2048, n_out = 25600, K = 5120.)
//
// On M = 2048, n_out = 25600, K = 5120, SM clocks per 256 x 256 x 16
// instruction (the arithmetic needs 128): MMA issue alone, no barrier at all 128; one k-step per stage 167 alone and
// 182 with loads and read-out; two k-steps per stage 146 and 160 (with eight epilogue warps and elect.sync: 145, the tensor pipe
// 92 % busy).
#include "common.cuh"
#include "kernels.h"

#include <cstdio>
#include <cstdlib>
#include <cstring>

namespace hspec {

namespace {

constexpr int TILE_K = 64;
// Eight epilogue warps: with four, reading a 256-column tile out (a TMEM load, then 16 stores, per 16 columns and warp, one
// after the other) was slow enough to show at the end of every launch.  Burst us, four -> eight warps:
// M = 512, n_out = 28672, K = 4096 (SwiGLU) 114 -> 107; M = 2048, n_out = 51200, K = 5120 770 -> 760.
constexpr int EPI_WARPS = 8, EPI_THREADS = 32 * EPI_WARPS, GEMM2_THREADS = 64 + EPI_THREADS;
constexpr uint32_t A_BYTES = 128 * TILE_K * 2;     // 16 KiB: this CTA's 128 weight rows

struct Gemm2Args {
  int M, N_out, K;
  int BNT;                 // activation rows per cluster tile (a multiple of 16, at most 256); each CTA stages BNT/2
  uint32_t acc_cols;       // TMEM columns per accumulator: BNT rounded up to a power of two
  int k_tiles, stages;
  int ksub;                // 64-column k-steps per pipeline stage (1 or 2): one barrier round per stage
  GemmRaster raster;
  // Work units: the first n_full_tiles tiles run whole (full waves of the SM pairs); each of the remaining "tail" tiles
  // is cut into tail_splits K-slices so that the last, partly filled wave keeps every pair busy.  A slice stores an
  // fp32 partial tile to `part` ([tail tile][slice][activation row][256 weight rows]); a second kernel sums them.
  int n_full_tiles, tail_splits, k_tiles_per_split;
  float* part;
  int f16, mode;
  int early_w;             // the weights may be read before the previous kernel of the stream has finished
  void* out;
  long long ldo;
  float* logits;
  unsigned long long* keys;
  uint32_t* status;
};

struct __align__(16) Tail2 {
  uint64_t full[GEMM_MAX_STAGES];
  uint64_t empty[GEMM_MAX_STAGES];
  uint64_t tmem_full[2];
  uint64_t tmem_empty[2];
  uint32_t tmem_base;
  uint32_t abort_flag;
  float4 best[EPI_WARPS][32];   // LM head: what each column of a warp's share has to reach to matter
};

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tmem_alloc_2sm(uint32_t smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_2sm() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_2sm(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// TMA load issued by either CTA of the pair; the byte count is credited to the barrier at the same offset in
// the leader CTA (rank bit of the shared::cluster address cleared).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const void* tmap, int c0, int c1, uint32_t bar_local,
                                                 uint64_t policy) {
  const uint32_t bar_leader = bar_local & 0xFEFFFFFFu;
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;"
      ::"r"(dst), "l"(tmap), "r"(c0), "r"(c1), "r"(bar_leader), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void umma_2sm(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives (once every MMA issued so far has finished) on the barrier at this offset in BOTH CTAs of the pair
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask)
               : "memory");
}
__device__ __forceinline__ uint32_t idesc_m256(uint32_t n, bool f16) {
  const uint32_t fmt = f16 ? 0u : 1u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((n >> 3) << 17) | ((256u >> 4) << 24);
}

// ARGMAX: the LM head's epilogue, apart so that the other launches do not carry its registers (96 for all of them instead of 64).
template <bool ARGMAX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM2_THREADS, 1)
gemm_2sm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, Gemm2Args g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t b_bytes = uint32_t(g.BNT / 2) * TILE_K * 2;
  const uint32_t sub_bytes = A_BYTES + b_bytes;                    // one k-step: this CTA's weight rows + its half of the activations
  const uint32_t stage_bytes = uint32_t(g.ksub) * sub_bytes;
  Tail2* tail = reinterpret_cast<Tail2*>(smem + size_t(g.stages) * stage_bytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
  const int total_tiles = g.raster.n_tiles_w * g.raster.n_tiles_m;
  const int total_units = g.n_full_tiles + (total_tiles - g.n_full_tiles) * g.tail_splits;
  // unit u < n_full_tiles: tile u, all of K; else tail tile n_full_tiles + v / tail_splits, K-slice v % tail_splits
  auto decode = [&](int u, int& tile, int& sp, int& kt_begin, int& kt_end) {
    if (u < g.n_full_tiles) { tile = u; sp = -1; kt_begin = 0; kt_end = g.k_tiles; return; }
    const int v = u - g.n_full_tiles;
    tile = g.n_full_tiles + v / g.tail_splits;
    sp = g.tail_splits > 1 ? v % g.tail_splits : -1;          // -1: the unit is a whole tile with the real epilogue
    kt_begin = (v % g.tail_splits) * g.k_tiles_per_split;
    kt_end = min(g.k_tiles, kt_begin + g.k_tiles_per_split);
  };
  const uint32_t tmem_cols = 2u * g.acc_cols;                // two accumulators

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(smem_u32(&tail->full[s]), 1);
      mbar_init(smem_u32(&tail->empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tail->tmem_full[a]), 1);
      mbar_init(smem_u32(&tail->tmem_empty[a]), 2 * EPI_WARPS);   // one arrival per epilogue warp of each CTA (leader's copy is used)
    }
    tail->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_2sm(smem_u32(&tail->tmem_base), tmem_cols);
    tmem_relinquish_2sm();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = tail->tmem_base;
  volatile uint32_t* abort_flag = &tail->abort_flag;

  if (warp == 0) {
    if (elect_one()) {
      // Weights at normal L2 priority, activations evict-last.  Evict-first weights ran a few percent faster in
      // short isolated runs, but ncu showed 2.4x the algorithmic DRAM reads (the clusters that share a weight tile
      // drift apart and fetch it again), and in a long power-capped step the extra DRAM traffic costs clock:
      // 13.5 vs 13.75 ms per step at conc128_32b.
      // (With a single activation tile nobody shares a weight tile: the weights stream through once, evict-first.)
      const uint64_t pol_w = g.raster.n_tiles_m == 1 ? policy_evict_first() : policy_evict_normal(), pol_x = policy_evict_last();
      // The weights do not depend on the kernels in front: the first stages' boxes are requested while those still run.
      uint32_t early = 0;
      if (g.early_w) {
        int tile, sp, kt_begin, kt_end;
        decode(cluster_id, tile, sp, kt_begin, kt_end);
        int tn, tm;
        g.raster.tile_at(tile, tn, tm);
        for (int kt = kt_begin; kt < kt_end && early < uint32_t(g.stages); kt += g.ksub, ++early) {
          const int n_sub = min(g.ksub, kt_end - kt);
          const uint32_t full = smem_u32(&tail->full[early]);
          if (rank == 0) mbar_expect_tx(full, 2 * uint32_t(n_sub) * sub_bytes);
          for (int sub = 0; sub < n_sub; ++sub)
            tma_load_2d_pair(smem_u32(smem + size_t(early) * stage_bytes + size_t(sub) * sub_bytes), &tmA, (kt + sub) * TILE_K,
                             tn * 256 + int(rank) * 128, full, pol_w);
        }
      }
      pdl_wait();
      pdl_trigger();
      uint32_t it = 0;
      bool ok = true;
      for (int unit = cluster_id; unit < total_units && ok; unit += n_clusters) {
        int tile, sp, kt_begin, kt_end;
        decode(unit, tile, sp, kt_begin, kt_end);
        int tn, tm;
        g.raster.tile_at(tile, tn, tm);
        for (int kt = kt_begin; kt < kt_end; kt += g.ksub, ++it) {
          const int s = it % g.stages;
          const uint32_t lap = it / g.stages;
          if (lap > 0 && !mbar_wait(smem_u32(&tail->empty[s]), (lap - 1) & 1)) {
            atomicExch(g.status, STATUS_TIMEOUT_PRODUCER);
            *abort_flag = 1;
            ok = false;
            break;
          }
          const int n_sub = min(g.ksub, kt_end - kt);
          const uint32_t full = smem_u32(&tail->full[s]);
          if (rank == 0 && it >= early) mbar_expect_tx(full, 2 * uint32_t(n_sub) * sub_bytes);   // both CTAs' bytes land on the leader's barrier
          for (int sub = 0; sub < n_sub; ++sub) {
            uint8_t* sa = smem + size_t(s) * stage_bytes + size_t(sub) * sub_bytes;
            if (it >= early) tma_load_2d_pair(smem_u32(sa), &tmA, (kt + sub) * TILE_K, tn * 256 + int(rank) * 128, full, pol_w);
            tma_load_2d_pair(smem_u32(sa + A_BYTES), &tmB, (kt + sub) * TILE_K, tm * g.BNT + int(rank) * (g.BNT / 2), full, pol_x);
          }
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = idesc_m256(uint32_t(g.BNT), g.f16 != 0);
      uint32_t it = 0, tile_count = 0;
      bool ok = true;
      for (int unit = cluster_id; unit < total_units && ok; unit += n_clusters, ++tile_count) {
        int tile, sp, kt_begin, kt_end;
        decode(unit, tile, sp, kt_begin, kt_end);
        const uint32_t acc = tile_count & 1, use = tile_count >> 1;
        if (use > 0 && !mbar_wait(smem_u32(&tail->tmem_empty[acc]), (use - 1) & 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_acc = tmem_base + acc * g.acc_cols;
        for (int kt = kt_begin; kt < kt_end; kt += g.ksub, ++it) {
          const int s = it % g.stages;
          const uint32_t lap = it / g.stages;
          // (every barrier round in this thread costs the tensor pipe ~150 clocks: with two k-steps per stage it is
          // paid once per eight MMAs instead of once per four)
          if (!mbar_wait(smem_u32(&tail->full[s]), lap & 1)) { ok = false; break; }
          tc_fence_after();
          const int n_sub = min(g.ksub, kt_end - kt);
          for (int sub = 0; sub < n_sub; ++sub) {
            const uint32_t sa = smem_u32(smem + size_t(s) * stage_bytes + size_t(sub) * sub_bytes);
            const uint64_t da = umma_desc_kmajor_sw128(sa), db = umma_desc_kmajor_sw128(sa + A_BYTES);
#pragma unroll
            for (int kk = 0; kk < TILE_K / 16; ++kk)
              umma_2sm(tmem_acc, da + uint64_t(kk * 2), db + uint64_t(kk * 2), idesc, (kt > kt_begin || sub > 0 || kk > 0) ? 1u : 0u);
          }
          umma_commit_pair(smem_u32(&tail->empty[s]));
        }
        if (ok) umma_commit_pair(smem_u32(&tail->tmem_full[acc]));
      }
      if (!ok) { atomicExch(g.status, STATUS_TIMEOUT_MMA); *abort_flag = 1; }
    }
  } else {
    // ---------------------------------------------------------------- epilogue (both CTAs)
    pdl_wait();                                  // nothing is read or written before the kernels in front have finished
    const int q = warp & 3;
    uint32_t tile_count = 0;
    bool ok = true;
    const uint32_t empty_leader0 = mapa_rank(smem_u32(&tail->tmem_empty[0]), 0);
    const uint32_t empty_leader1 = mapa_rank(smem_u32(&tail->tmem_empty[1]), 0);
    for (int unit = cluster_id; unit < total_units && ok; unit += n_clusters, ++tile_count) {
      int tile, sp, kt_begin, kt_end;
      decode(unit, tile, sp, kt_begin, kt_end);
      int tn, tm;
      g.raster.tile_at(tile, tn, tm);
      const int mode = sp >= 0 ? EPI_PARTIAL_F32 : g.mode;
      if constexpr (ARGMAX) {
        // The rows' maxima over the tiles that are done by now, asked for while this one is still computed.  They only grow, so an older value costs
        // a reduction too many at worst.
        float* best = reinterpret_cast<float*>(tail->best[warp - 2]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = ((warp - 2) >> 2) * 16 + (2 * i + (lane >> 4)) * 32 + (lane & 15), m = tm * g.BNT + c;
          best[i * 32 + lane] = c < g.BNT && m < g.M ? argmax_key_value(__ldcg(g.keys + m)) : INFINITY;
        }
        __syncwarp();
      }
      const uint32_t acc = tile_count & 1, use = tile_count >> 1;
      if (!mbar_wait(smem_u32(&tail->tmem_full[acc]), use & 1)) {
        atomicExch(g.status, STATUS_TIMEOUT_EPILOGUE);
        ok = false;
        break;
      }
      tc_fence_after();
      const int tile_n128 = tn * 2 + int(rank);               // 128-row weight tile of this CTA
      const int n = tile_n128 * 128 + q * 32 + lane;
      const bool n_ok = n < g.N_out;
      const int m0 = tm * g.BNT;
      const uint32_t tmem_acc = tmem_base + acc * g.acc_cols + (uint32_t(q * 32) << 16);
      for (int c0 = ((warp - 2) >> 2) * 16; c0 < g.BNT; c0 += EPI_WARPS * 4) {
        if (m0 + c0 >= g.M) break;                          // rows past M: nothing to store (warp-uniform)
        uint32_t r[16];
        tmem_ld16(tmem_acc + uint32_t(c0), r);
        tmem_ld_wait();
        if constexpr (ARGMAX) {
          // A lane that does not reach its row's maximum so far has nothing to say about the arg-max, and after the first few of a
          // row's tiles hardly one does: the reduction network (64 shuffles for 16 rows) runs for the few groups with one that reaches it.  (For
          // every group it cost the LM head 4 %, mostly as clock under the power cap; one redux.sync maximum + ballot per column more still.  Logits that rise along the
          // vocabulary still run it for every group, equal ones too: within 1 % of the form without the test, 77 rows of 152 064 256 -> 255.5 and 255 -> 254.7 us.)
          const float4* best = tail->best[warp - 2] + (c0 >> 5) * 4;
          bool reached = false;
#pragma unroll
          for (int j = 0; j < 16; j += 4) {
            const float4 t = best[j >> 2];
            const float tj[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int m = m0 + c0 + j + e;
              const float x = __uint_as_float(r[j + e]);
              if (g.logits != nullptr && n_ok && m < g.M) g.logits[size_t(m) * g.ldo + n] = x;
              reached |= !(x < tj[e]);
            }
          }
          if (__any_sync(0xffffffffu, reached && n_ok)) {
            float v[16];
            int vi[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) { v[j] = argmax_value(__uint_as_float(r[j]), n_ok); vi[j] = n; }
            int row = 0;
            warp_argmax16(v, vi, lane, row);
            const int m = m0 + c0 + row;
            if ((lane & 1) == 0 && m < g.M && vi[0] < g.N_out && !(v[0] < reinterpret_cast<const float*>(best)[row]))
              atomicMax(g.keys + m, argmax_key(v[0], vi[0]));
          }
        } else if (mode == EPI_PARTIAL_F32) {
          // slice of a tail tile: [tail tile][slice][activation row of the tile][256 weight rows of the pair]
          float* out = g.part + (size_t(tile - g.n_full_tiles) * g.tail_splits + sp) * size_t(g.BNT) * 256 +
                       int(rank) * 128 + q * 32 + lane;
#pragma unroll
          for (int j = 0; j < 16; ++j) out[size_t(c0 + j) * 256] = __uint_as_float(r[j]);
        } else if (mode == EPI_STORE_F32) {
          float* out = reinterpret_cast<float*>(g.out);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int m = m0 + c0 + j;
            if (n_ok && m < g.M) out[size_t(m) * g.ldo + n] = __uint_as_float(r[j]);
          }
        } else if (mode == EPI_ACCUM_F32) {
          // Residual stream: y += acc as a reduction in the L2 (one rounding of old + acc, as in registers; every element is
          // met once per launch, so the result does not depend on any order).  No thread waits for the old value.
          // Burst us, loads and adds -> reductions: M = 8192, n_out = K = 4096 242 -> 227; M = 512 28.7 -> 25.2 (280 and 33.7
          // before both this and the eight warps).
          float* out = reinterpret_cast<float*>(g.out);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int m = m0 + c0 + j;
            if (n_ok && m < g.M) red_add_f32(out + size_t(m) * g.ldo + n, __uint_as_float(r[j]));
          }
        } else if (mode == EPI_SWIGLU_F16 || mode == EPI_SWIGLU_BF16) {
          const int f = tile_n128 * 64 + q * 16 + (lane & 15);
          swiglu_store16(r, g.out, mode == EPI_SWIGLU_BF16, g.ldo, m0 + c0, g.M, f, 2 * f < g.N_out, lane, g.status);
        } else if (mode == EPI_STORE_F16) {
          __half* out = reinterpret_cast<__half*>(g.out);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int m = m0 + c0 + j;
            if (n_ok && m < g.M) out[size_t(m) * g.ldo + n] = f16_sat(__uint_as_float(r[j]), g.status);
          }
        } else if (mode == EPI_STORE_BF16) {
          __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(g.out);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int m = m0 + c0 + j;
            if (n_ok && m < g.M) out[size_t(m) * g.ldo + n] = __float2bfloat16_rn(__uint_as_float(r[j]));
          }
        }
      }
      // accumulator drained: hand it back to the MMA issuer in the leader CTA
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc ? empty_leader1 : empty_leader0);
    }
  }
  tc_fence_before();
  cluster_sync_all();           // neither CTA may leave while its pair still reads its shared memory or TMEM
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_2sm(tmem_base, tmem_cols);
  }
}

// Sums the K-slices of the tail tiles in slice order (deterministic) and applies the real epilogue.
// Block = (tail tile, group of 4 activation rows); thread = one of the pair's 256 weight rows; all slices' loads are
// issued before the first add.
constexpr int TAIL_MAX_SPLITS = 8, TAIL_ROWS = 4;
__global__ void __launch_bounds__(256)
gemm2_tail_reduce_kernel(Gemm2Args g) {
  pdl_wait();
  pdl_trigger();
  const int tail = blockIdx.x, tile = g.n_full_tiles + tail;
  int tn, tm;
  g.raster.tile_at(tile, tn, tm);
  const int n = tn * 256 + threadIdx.x;
  const int m_base = tm * g.BNT + blockIdx.y * TAIL_ROWS;
  if (m_base >= g.M) return;
  const float* src = g.part + size_t(tail) * g.tail_splits * g.BNT * 256 + size_t(blockIdx.y) * TAIL_ROWS * 256 + threadIdx.x;
  float v[TAIL_MAX_SPLITS][TAIL_ROWS];
#pragma unroll
  for (int sp = 0; sp < TAIL_MAX_SPLITS; ++sp)
#pragma unroll
    for (int j = 0; j < TAIL_ROWS; ++j)
      v[sp][j] = (sp < g.tail_splits && m_base + j < g.M) ? __ldcs(src + (size_t(sp) * g.BNT + j) * 256) : 0.f;
  const int lane = threadIdx.x & 31;
  // SwiGLU epilogue: weight rows are interleaved in blocks of 16 (gate | up), so lanes l and l ^ 16 of a warp hold the
  // gate and the up projection of feature f
  const int f = (tn * 2 + (threadIdx.x >> 7)) * 64 + ((threadIdx.x >> 5) & 3) * 16 + (lane & 15);
#pragma unroll
  for (int j = 0; j < TAIL_ROWS; ++j) {
    const int m = m_base + j;
    if (m >= g.M) break;                                    // uniform over the block
    float acc = 0.f;
#pragma unroll
    for (int sp = 0; sp < TAIL_MAX_SPLITS; ++sp)
      if (sp < g.tail_splits) acc += v[sp][j];
    if (g.mode == EPI_SWIGLU_F16 || g.mode == EPI_SWIGLU_BF16) {
      const float up = __shfl_xor_sync(0xffffffffu, acc, 16);
      if (lane < 16 && 2 * f < g.N_out) store_act16(g.out, size_t(m) * g.ldo + f, silu_f(acc) * up, g.mode == EPI_SWIGLU_BF16, g.status);
      continue;
    }
    if (n >= g.N_out) continue;
    const size_t o = size_t(m) * g.ldo + n;
    if (g.mode == EPI_STORE_F32) reinterpret_cast<float*>(g.out)[o] = acc;
    else if (g.mode == EPI_ACCUM_F32) reinterpret_cast<float*>(g.out)[o] += acc;
    else if (g.mode == EPI_STORE_F16) reinterpret_cast<__half*>(g.out)[o] = f16_sat(acc, g.status);
    else reinterpret_cast<__nv_bfloat16*>(g.out)[o] = __float2bfloat16_rn(acc);
  }
}

bool g_attr_done2[MAX_DEVICES] = {};
int g_smem_optin2[MAX_DEVICES] = {};

}  // namespace

bool gemm2_preferred(int M, int n_out) {
  static const bool off = [] { const char* e = getenv("HSPEC_GEMM_1SM"); return e && e[0] == '1'; }();
  static const int min_m = [] { const char* e = getenv("HSPEC_GEMM2_MIN_M"); return e ? atoi(e) : 0; }();   // measurements only
  if (off) return false;
  if (min_m > 0) return M >= min_m;
  // Above 128 rows always: the one-CTA kernel's 256-wide accumulator leaves it one CTA per SM and half the weights in flight
  // (us, one CTA / pair: 160 rows, n_out = K = 4096 35 / 22, n_out = 28672 68 / 51; 255 rows 46 / 21 and 87 / 65).  From 33 rows on
  // for matrices of about a wave of pair tiles or more, where the pair kernel streams weights at least as fast (n_out = 17536:
  // 16 rows 26.5 / 26.7, 48 rows 30.3 / 27.1, 128 rows 40.3 / 29.6; n_out = 262144: 316 / 324, 339 / 320, 434 / 370; the LM head of
  // 152 064 rows, K = 5120, logits written: 246 / 239, 260 / 248, 328 / 291).  Smaller matrices keep the one-CTA kernel and its
  // K-slices in a cluster (n_out = 4096, K = 14336: 21.5 / 25.1, 23.6 / 25.7, 27.9 / 28.0).
  return M > 128 || (M > 32 && n_out >= 64 * 256);
}

// Tile width (activation rows per pair tile) and the number of K-slices for the tiles of the last, partly filled wave,
// by a simple model: full waves of the 74 SM pairs x k-steps x cost of a k-step, plus the tail wave (k-steps / slices),
// a fixed cost per wave (pipeline fill, the last epilogue) and, with slices, the pass that sums the partial tiles.
// One cost unit ~ 2.2 ns (a k-step of a 256-wide pair tile = 256 units ~ 0.56 us).
// The rows are spread evenly over the tiles, in steps of 16, so that the last one is not mostly padding: 549 rows are three tiles of 192
// and not of 256 (n_out = 28672, K = 4096: 134 -> 122 us; n_out = 4096, K = 14336: 70 -> 66 us).
void gemm2_pick(int M, int n_out, int K, int mode, int* bnt_out, int* splits_out) {
  const int tw = (n_out + 255) / 256;
  const int k_tiles = (K + TILE_K - 1) / TILE_K;
  const bool may_split = mode != EPI_ARGMAX;            // every other epilogue can be applied after the slices are summed
  double best_cost = 1e30;
  int best_bnt = 256, best_s = 1;
  for (int widest = 256; widest >= 128; widest -= 32) {
    const int nm = (M + widest - 1) / widest;
    const int bnt = ((M + nm - 1) / nm + 15) / 16 * 16;
    const int tiles = tw * nm;
    const int full_waves = tiles / 74, tail = tiles % 74;
    // a k-step fills 16 KB of weights and BNT x 64 bytes of activations per SM: below 256 rows it is this fill that sets the
    // pace (measured, a 128-wide tile runs 1.5x slower per flop than a 256-wide one)
    const double kstep = 128.0 + 0.5 * bnt;
    for (int s = 1; s <= 8; ++s) {
      if (s > 1 && (!may_split || tail == 0 || tail * s > 74 || k_tiles / s < 8)) continue;
      const int kps = (k_tiles + s - 1) / s;
      if (s > 1 && kps * (s - 1) >= k_tiles) continue;         // an empty last slice
      double cost = double(full_waves) * (k_tiles * kstep + 1500.0);
      if (tail > 0) cost += kps * kstep + 1500.0;
      // (the pass that sums the slices: its bytes at 4 TB/s plus 2 us; with 4, 8, 12 or 20 us fewer launches are sliced and
      // the 256-row steps get slower, 1.93 -> 1.95 / 2.02 / 2.07 / 2.10 ms at paper_8b; no difference at 2048 rows)
      if (s > 1) cost += (double(s + 2) * tail * bnt * 256 * 4.0 / 4.0e6 + 2.0) * 455.0;
      if (cost < best_cost) { best_cost = cost; best_bnt = bnt; best_s = s; }
    }
  }
  *bnt_out = best_bnt;
  *splits_out = best_s;
}

// Scratch for the tail tiles' partials: at most one wave of pair tiles, each up to 256 x 256 fp32, times the slices.
size_t gemm2_tail_bytes() { return size_t(74) * 256 * 256 * 4; }

cudaError_t gemm2_launch(const GemmCall& c, cudaStream_t stream, Tracker* trk, std::string* err) {
  {
    const cudaError_t e = once_per_device(g_attr_done2, [](int dev) {
      cudaError_t e2 = cudaDeviceGetAttribute(&g_smem_optin2[dev], cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      if (e2 != cudaSuccess) return e2;
      e2 = cudaFuncSetAttribute(gemm_2sm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, g_smem_optin2[dev]);
      return e2 != cudaSuccess ? e2 : cudaFuncSetAttribute(gemm_2sm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, g_smem_optin2[dev]);
    });
    if (e != cudaSuccess) return e;
  }
  const int smem_optin2 = g_smem_optin2[current_device()];
  Gemm2Args g{};
  g.M = c.M; g.N_out = c.n_out; g.K = c.K;
  int splits = 1;
  gemm2_pick(c.M, c.n_out, c.K, c.mode, &g.BNT, &splits);
  g.acc_cols = g.BNT > 128 ? 256 : (g.BNT > 64 ? 128 : 64);
  g.k_tiles = (c.K + TILE_K - 1) / TILE_K;
  g.raster.n_tiles_w = (c.n_out + 255) / 256;
  g.raster.n_tiles_m = (c.M + g.BNT - 1) / g.BNT;
  // Groups of at most 16 activation tiles, evenly: with all 32 of M = 8192 inside one weight tile a wave was 32 x 2.3 tiles, its activations
  // (67 MB at K = 4096) did not stay in the L2 - 1.5 GB read from DRAM where 0.2 were needed - and the power that took came off the
  // clock.  us (burst / sustained), 32 tiles together, groups of 16, 11, 8: n_out 28672, K 4096 1531 / 1780, 1413 / 1557, 1417 / 1551,
  // 1442 / 1618; n_out 4096, K 14336 846 / 956, 779 / 882, 762 / 911, 756 / 895.  M = 4096 (16 tiles): whole 699 / 776, two groups of
  // eight 717 / 796.
  const int n_groups = (g.raster.n_tiles_m + 15) / 16;
  g.raster.group = (g.raster.n_tiles_m + n_groups - 1) / n_groups;
  const int tiles = g.raster.n_tiles_w * g.raster.n_tiles_m;
  const int tail = tiles % 74;
  if (c.splits > 0) splits = c.splits;                    // the caller fixed the number of K-slices (of the tail tiles)
  if (c.mode == EPI_ARGMAX || tail == 0) splits = 1;
  if (splits > g.k_tiles) splits = g.k_tiles;
  if (splits > TAIL_MAX_SPLITS) splits = TAIL_MAX_SPLITS;
  while (splits > 1 && size_t(tail) * splits * g.BNT * 256 * 4 > c.splitk_ws_bytes) --splits;   // never more than the scratch holds
  if (c.splitk_ws == nullptr) splits = 1;
  g.k_tiles_per_split = (g.k_tiles + splits - 1) / splits;
  splits = (g.k_tiles + g.k_tiles_per_split - 1) / g.k_tiles_per_split;   // no empty slice
  g.tail_splits = splits;
  g.n_full_tiles = splits > 1 ? tiles - tail : tiles;
  g.part = reinterpret_cast<float*>(c.splitk_ws);
  g.early_w = c.w_stable ? 1 : 0;
  g.f16 = c.f16 ? 1 : 0; g.mode = c.mode; g.out = c.out; g.ldo = c.ldo;
  if (c.addend != nullptr) { if (err) *err = "the 2-SM kernel has no addend epilogue"; return cudaErrorInvalidValue; }
  g.logits = c.logits; g.keys = c.keys; g.status = c.status;
  static const int ksub_env = [] { const char* e = getenv("HSPEC_GEMM2_KSUB"); return e ? atoi(e) : 0; }();   // measurements only
  g.ksub = (ksub_env == 1 || ksub_env == 2) ? ksub_env : 2;
  const size_t stage_bytes = size_t(g.ksub) * (A_BYTES + size_t(g.BNT / 2) * TILE_K * 2);
  const size_t fixed = sizeof(Tail2) + 1024;
  int stages = int((size_t(smem_optin2) - fixed) / stage_bytes);
  if (stages > GEMM_MAX_STAGES) stages = GEMM_MAX_STAGES;
  if (stages < 2) { if (err) *err = "shared memory too small for the 2-SM GEMM pipeline"; return cudaErrorInvalidValue; }
  g.stages = stages;
  CUtensorMap tmB;
  if (!make_tmap_16bit_2d(&tmB, c.x, c.M, c.K, c.ldx, g.BNT / 2, c.f16, err)) return cudaErrorInvalidValue;
  const int total = g.n_full_tiles + (tiles - g.n_full_tiles) * splits;
  const int clusters = total < 74 ? total : 74;
  const size_t smem = size_t(stages) * stage_bytes + fixed;
  // profile name "gemm2:<what>" tells this kernel's launches from the one-CTA kernel's "gemm:<what>"
  char label[40] = "gemm2:";
  if (c.label) {
    const char* colon = strchr(c.label, ':');
    strncat(label, colon ? colon + 1 : c.label, sizeof(label) - 7);
  }
  trk_begin(trk, label, 2.0 * c.M * c.n_out * c.K, 2.0 * c.n_out * c.K,
            gemm_io_bytes(c.M, c.n_out, c.K, c.mode, c.logits != nullptr));
  cudaError_t e = launch_pdl(c.mode == EPI_ARGMAX ? gemm_2sm_kernel<true> : gemm_2sm_kernel<false>, dim3(2 * clusters), dim3(GEMM2_THREADS), smem, stream,
                             *c.tmW, tmB, g);
  trk_end(trk);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (c.defer_tail) *c.defer_tail = GemmTail{};
  if (e == cudaSuccess && splits > 1 && c.defer_tail && (c.mode == EPI_ACCUM_F32 || c.mode == EPI_STORE_F32)) {
    *c.defer_tail = GemmTail{g.part, g.raster, g.n_full_tiles, g.BNT, splits};
    return e;
  }
  if (e == cudaSuccess && splits > 1) {
    trk_begin(trk, "gemm2_tail_reduce", 0, double(splits + 1) * tail * g.BNT * 256 * 4);
    e = launch_pdl(gemm2_tail_reduce_kernel, dim3(tail, g.BNT / TAIL_ROWS), dim3(256), 0, stream, g);
    trk_end(trk);
  }
  return e;
}

}  // namespace hspec
