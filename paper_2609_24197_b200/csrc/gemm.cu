// bf16 GEMM y = x W^T on the 5th-generation tensor cores (tcgen05 + TMEM + TMA), sm_100a.
//
// Every dense map of the draft step is "few activation rows times a tall weight matrix".  The
// weight rows therefore sit on the MMA's M side (128 output features per CTA = 128 TMEM lanes) and
// the activation rows on its N side (BN = 16..256 rows = BN TMEM columns), so a step with one
// request and a step with 256 requests run the same kernel: the accumulator tile is y^T.
//
//   warp 0 : TMA producer  (weights [128 x 64] and activations [BN x 64] per stage, 128-byte swizzle)
//   warp 1 : allocates TMEM, issues tcgen05.mma (one elected thread), commits stages back
//   warps 2..5 : epilogue, one TMEM lane quarter each: tcgen05.ld -> registers -> global
//
// Epilogues: fp32 / fp16 / bf16 store, fp32 accumulate-into (residual), SwiGLU, and the LM-head form that reduces each
// activation row's (max, index) over the CTA's 128 vocabulary rows.
//
// K-slices: where a matrix has fewer tiles than the chip has SMs, the slices of a tile are the CTAs of one cluster.  Each leaves
// its accumulator in its own shared memory (the ring is free by then), and each sums its share of the columns over all of them
// through distributed shared memory, in slice order (deterministic), and applies the epilogue.  (Slices written to global memory and
// summed by a second kernel cost a launch and a pass each: 11 of a one-request step's 51 launches.  16 rows, residual epilogue, back
// to back: n_out 4096, K 4096 13.9 -> 11.0 us, K 14336 28.7 -> 21.6 us; 128 rows, K 8192 36.8 -> 20.2 us.)
#include "common.cuh"
#include "kernels.h"

#include <cuda.h>

#include <cstdio>
#include <cstdlib>

namespace hspec {

namespace {

constexpr int TILE_W = 128;       // weight rows per CTA (UMMA M)
constexpr int TILE_K = 64;        // bf16 elements per stage along K = one 128-byte swizzle row
constexpr int UMMA_K = 16;
constexpr uint32_t A_STAGE_BYTES = TILE_W * TILE_K * 2;   // 16 KiB

struct __align__(8) GemmSmemTail {
  uint64_t full[GEMM_MAX_STAGES];
  uint64_t empty[GEMM_MAX_STAGES];
  uint64_t tmem_full;
  uint32_t tmem_base;
  uint32_t abort_flag;
  float red_val[4][256];   // LM-head epilogue: per lane-quarter (max, index) of each activation row
  int red_idx[4][256];
};

__global__ void __launch_bounds__(192, 2)
gemm_tcgen05_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmArgs g) {
  extern __shared__ uint8_t smem_raw[];
  // 128-byte swizzle needs 1024-byte aligned tiles
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t b_stage_bytes = g.BN * TILE_K * 2;
  const uint32_t stage_bytes = A_STAGE_BYTES + b_stage_bytes;
  GemmSmemTail* tail = reinterpret_cast<GemmSmemTail*>(smem + size_t(g.stages) * stage_bytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile_m = blockIdx.x;            // activation-row tile (fastest: CTAs sharing a weight tile run together)
  const int tile_n = blockIdx.y;            // 128-row weight tile
  const int split = blockIdx.z, n_splits = gridDim.z;      // the slices of a tile form one cluster
  const int kt_begin = split * g.k_tiles_per_split;
  const int kt_end = min(g.k_tiles_total, kt_begin + g.k_tiles_per_split);
  const int n_kt = kt_end - kt_begin;       // >= 1 by construction of the grid
  const uint32_t tmem_cols = g.tmem_cols;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(smem_u32(&tail->full[s]), 1);
      mbar_init(smem_u32(&tail->empty[s]), 1);
    }
    mbar_init(smem_u32(&tail->tmem_full), 1);
    tail->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tail->tmem_base), tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_acc = tail->tmem_base;

  if (warp == 0) {
    if (elect_one()) {
      // weights are streamed once per step, unless the caller runs the same matrix again right away
      const uint64_t pol_w = g.keep_w ? policy_evict_last() : policy_evict_first();
      const uint64_t pol_x = policy_evict_last();    // activations are re-read by every weight tile
      // The weights do not depend on the kernels in front: the first stages' boxes are requested while those still run.
      int early = 0;
      for (; g.early_w && early < n_kt && early < g.stages; ++early) {
        const uint32_t full = smem_u32(&tail->full[early]);
        mbar_expect_tx(full, stage_bytes);
        tma_load_2d(smem_u32(smem + size_t(early) * stage_bytes), &tmA, (kt_begin + early) * TILE_K, tile_n * TILE_W, full, pol_w);
      }
      pdl_wait();
      pdl_trigger();
      for (int i = 0; i < n_kt; ++i) {
        const int s = i % g.stages;
        const uint32_t round = i / g.stages;
        if (round > 0 && !mbar_wait(smem_u32(&tail->empty[s]), (round - 1) & 1)) {
          atomicExch(g.status, STATUS_TIMEOUT_PRODUCER);
          atomicExch(&tail->abort_flag, 1u);
          break;
        }
        const uint32_t full = smem_u32(&tail->full[s]);
        uint8_t* sa = smem + size_t(s) * stage_bytes;
        if (i >= early) {
          mbar_expect_tx(full, stage_bytes);
          tma_load_2d(smem_u32(sa), &tmA, (kt_begin + i) * TILE_K, tile_n * TILE_W, full, pol_w);
        }
        tma_load_2d(smem_u32(sa + A_STAGE_BYTES), &tmB, (kt_begin + i) * TILE_K, tile_m * g.BN, full, pol_x);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t idesc = umma_idesc_m128(g.BN, g.f16 != 0);
      bool ok = true;
      for (int i = 0; i < n_kt && ok; ++i) {
        const int s = i % g.stages;
        const uint32_t round = i / g.stages;
        if (!mbar_wait(smem_u32(&tail->full[s]), round & 1)) {
          atomicExch(g.status, STATUS_TIMEOUT_MMA);
          atomicExch(&tail->abort_flag, 1u);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + size_t(s) * stage_bytes);
        const uint64_t da = umma_desc_kmajor_sw128(sa), db = umma_desc_kmajor_sw128(sa + A_STAGE_BYTES);
#pragma unroll
        for (int kk = 0; kk < TILE_K / UMMA_K; ++kk) {
          // advancing K inside the swizzle row: +32 bytes = +2 in the descriptor's 16-byte units
          umma_bf16(tmem_acc, da + uint64_t(kk * 2), db + uint64_t(kk * 2), idesc, (i > 0 || kk > 0) ? 1u : 0u);
        }
        umma_commit(smem_u32(&tail->empty[s]));   // stage reusable once these MMAs have read it
      }
      // accumulator complete (or aborted: release the epilogue either way)
      if (ok) umma_commit(smem_u32(&tail->tmem_full));
      else mbar_arrive(smem_u32(&tail->tmem_full));
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    const int q = warp & 3;                         // TMEM lane quarter this warp may read
    pdl_wait();                                     // nothing else is read or written before the kernels in front have finished
    if (g.addend != nullptr && g.mode == EPI_ARGMAX) {
      // the addend rows of this tile do not depend on the accumulator: pull this warp's 128-byte piece of every
      // row into L2 while the main loop runs (one line per lane and pass)
      const int n_w = tile_n * TILE_W + q * 32;
      if (n_w < g.N_out)
        for (int c = lane; c < g.BN; c += 32) {
          const int m = tile_m * g.BN + c;
          if (m < g.M) asm volatile("prefetch.global.L2 [%0];" ::"l"(g.addend + size_t(m) * g.ld_add + n_w));
        }
    }
    bool ok = mbar_wait(smem_u32(&tail->tmem_full), 0);
    if (!ok) atomicExch(g.status, STATUS_TIMEOUT_EPILOGUE);
    tc_fence_after();
    if (*reinterpret_cast<volatile uint32_t*>(&tail->abort_flag)) ok = false;
    const int m0 = tile_m * g.BN;
    const int n = tile_n * TILE_W + q * 32 + lane;  // output feature (weight row) of this thread
    const bool n_ok = n < g.N_out;
    if (n_splits > 1) {
      // this slice's accumulator -> this CTA's shared memory, [column][128 weight rows] (every stage of the ring has been read)
      float* mine = reinterpret_cast<float*>(smem) + q * 32 + lane;
      for (int c0 = 0; c0 < g.BN; c0 += 16) {
        uint32_t r[16];
        tmem_ld16(tmem_acc + (uint32_t(q * 32) << 16) + uint32_t(c0), r);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) mine[(c0 + j) * TILE_W] = ok ? __uint_as_float(r[j]) : 0.f;
      }
    }
    // Addend of the arg-max epilogue (the causal-correction head): the loads of the next 16 columns are issued before
    // this batch is reduced.  Measured on that head's CTAs (K = 256, 128 requests): the epilogue
    // takes 23 000 of a CTA's 29 000 clocks - 10 000 with neither addend nor reduction, +6 000 for the reduction network,
    // +7 500 for the addend - and a queue of 64 loads per thread instead of 16 changes nothing: with two CTAs of four
    // epilogue warps per SM it is the warps' instruction latency, not memory, that sets the pace.
    float add_next[16];
    auto load_addend = [&](int c_first) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int m = m0 + c_first + j;
        add_next[j] = (n_ok && c_first < g.BN && m < g.M) ? __ldcs(g.addend + size_t(m) * g.ld_add + n) : 0.f;
      }
    };
    const bool with_addend = g.mode == EPI_ARGMAX && g.addend != nullptr;
    if (with_addend && ok) load_addend(0);

    for (int c0 = 0; c0 < g.BN && ok && n_splits == 1; c0 += 16) {
      uint32_t r[16];
      tmem_ld16(tmem_acc + (uint32_t(q * 32) << 16) + uint32_t(c0), r);
      tmem_ld_wait();
      if (g.mode == EPI_STORE_F32) {
        float* out = reinterpret_cast<float*>(g.out);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          if (n_ok && m < g.M) out[size_t(m) * g.ldo + n] = __uint_as_float(r[j]);
        }
      } else if (g.mode == EPI_ACCUM_F32) {
        // residual stream: y += acc as a reduction in the L2, no thread waits for the old value
        float* out = reinterpret_cast<float*>(g.out);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          if (n_ok && m < g.M) red_add_f32(out + size_t(m) * g.ldo + n, __uint_as_float(r[j]));
        }
      } else if (g.mode == EPI_STORE_BF16) {
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(g.out);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          if (n_ok && m < g.M) out[size_t(m) * g.ldo + n] = __float2bfloat16_rn(__uint_as_float(r[j]));
        }
      } else if (g.mode == EPI_SWIGLU_F16 || g.mode == EPI_SWIGLU_BF16) {
        const int f = tile_n * 64 + q * 16 + (lane & 15);
        swiglu_store16(r, g.out, g.mode == EPI_SWIGLU_BF16, g.ldo, m0 + c0, g.M, f, 2 * f < g.N_out, lane, g.status);
      } else if (g.mode == EPI_STORE_F16) {
        __half* out = reinterpret_cast<__half*>(g.out);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          if (n_ok && m < g.M) out[size_t(m) * g.ldo + n] = f16_sat(__uint_as_float(r[j]), g.status);
        }
      } else {  // EPI_ARGMAX: logits optional, (max, lowest index) over this warp's 32 vocabulary rows
        float add[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) add[j] = with_addend ? add_next[j] : 0.f;
        if (with_addend) load_addend(c0 + 16);
        float v[16];
        int vi[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int m = m0 + c0 + j;
          const float x = __uint_as_float(r[j]) + add[j];
          if (g.logits != nullptr && n_ok && m < g.M) g.logits[size_t(m) * g.ldo + n] = x;
          v[j] = argmax_value(x, n_ok);
          vi[j] = n;
        }
        int row = 0;
        warp_argmax16(v, vi, lane, row);
        if ((lane & 1) == 0) { tail->red_val[q][c0 + row] = v[0]; tail->red_idx[q][c0 + row] = vi[0]; }
      }
    }
    if (g.mode == EPI_ARGMAX) {
      asm volatile("bar.sync 1, 128;" ::: "memory");      // the four epilogue warps only
      const int t = threadIdx.x - 64;                     // 0..127
      for (int c = t; c < g.BN; c += 128) {
        const int m = m0 + c;
        if (m >= g.M) continue;
        float v = tail->red_val[0][c];
        int idx = tail->red_idx[0][c];
#pragma unroll
        for (int qq = 1; qq < 4; ++qq) {
          const float ov = tail->red_val[qq][c];
          const int oi = tail->red_idx[qq][c];
          if (ov > v || (ov == v && oi < idx)) { v = ov; idx = oi; }
        }
        if (!ok) { v = -INFINITY; idx = 0x7fffffff; }
        if (g.keys != nullptr) {
          if (idx != 0x7fffffff) atomicMax(g.keys + m, argmax_key(v, idx));
          continue;
        }
        g.part_val[size_t(tile_n) * g.M + m] = v;
        g.part_idx[size_t(tile_n) * g.M + m] = idx;
      }
    }
    tc_fence_before();
  }
  if (n_splits > 1) {
    cluster_sync_all();                             // every slice's accumulator lies in its CTA's shared memory
    // CTA `split` finishes the columns split, split + n_splits, ...: four groups of 32 weight rows x the warps 2..5
    if (warp >= 2) {
      const int q = warp & 3;
      const int n = tile_n * TILE_W + q * 32 + lane;
      const bool n_ok = n < g.N_out;
      const uint32_t base = smem_u32(smem) + uint32_t(q * 32 + lane) * 4;
      constexpr int U = 4;                          // columns in flight
      uint32_t peer[GEMM_MAX_SPLITS];
#pragma unroll
      for (int s = 0; s < GEMM_MAX_SPLITS; ++s) peer[s] = s < n_splits ? mapa_rank(base, uint32_t(s)) : 0u;
      for (int c0 = split; c0 < g.BN && tile_m * g.BN + c0 < g.M; c0 += U * n_splits) {
        float v[U][GEMM_MAX_SPLITS];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int s = 0; s < GEMM_MAX_SPLITS; ++s) {
            const int c = c0 + u * n_splits;
            v[u][s] = (s < n_splits && c < g.BN) ? ld_cluster_f32(peer[s] + uint32_t(c) * (TILE_W * 4)) : 0.f;
          }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int c = c0 + u * n_splits, m = tile_m * g.BN + c;
          if (c >= g.BN || m >= g.M) break;         // warp-uniform
          float acc = v[u][0];
#pragma unroll
          for (int s = 1; s < GEMM_MAX_SPLITS; ++s)
            if (s < n_splits) acc += v[u][s];
          const size_t o = size_t(m) * g.ldo + n;
          if (epi_is_swiglu(g.mode)) {
            const float up = __shfl_xor_sync(0xffffffffu, acc, 16);       // lanes l and l + 16 hold gate and up of one feature
            const int f = tile_n * 64 + q * 16 + lane;
            if (lane < 16 && 2 * f < g.N_out) store_act16(g.out, size_t(m) * g.ldo + f, silu_f(acc) * up, g.mode == EPI_SWIGLU_BF16, g.status);
          } else if (n_ok) {
            if (g.mode == EPI_STORE_F32) reinterpret_cast<float*>(g.out)[o] = acc;
            else if (g.mode == EPI_ACCUM_F32) red_add_f32(reinterpret_cast<float*>(g.out) + o, acc);
            else if (g.mode == EPI_STORE_F16) reinterpret_cast<__half*>(g.out)[o] = f16_sat(acc, g.status);
            else reinterpret_cast<__nv_bfloat16*>(g.out)[o] = __float2bfloat16_rn(acc);
          }
        }
      }
    }
    cluster_sync_all();                             // no CTA leaves while another still reads its shared memory
  } else {
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_acc, tmem_cols);
  }
}

__global__ void __launch_bounds__(256)
argmax_init_kernel(unsigned long long* keys, int M) {
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x * 256 + threadIdx.x;
  if (m < M) keys[m] = 0;
}

// A row that no tile has finished (a wait that gave up) has no id: 0x7fffffff.  (A key per row against (value, index) pairs per tile and row
// that a kernel reduces: LM head of 152 064 rows, 77 requests 279 against 282 us.  Letting the GEMM's last CTA write the ids instead
// costs a fence, a ticket and a read-back at its end, more than this launch: test-sized drafter 65.3 -> 66.6 us per step.)
__global__ void __launch_bounds__(256)
argmax_ids_kernel(const unsigned long long* keys, int M, int* ids, const int* id_map) {
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x * 256 + threadIdx.x;
  if (m >= M) return;
  const unsigned long long key = keys[m];
  const int idx = key ? int(0xffffffffu - uint32_t(key)) : 0x7fffffff;
  ids[m] = id_map && idx != 0x7fffffff ? id_map[idx] : idx;
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

bool g_attr_done[MAX_DEVICES] = {};
int g_smem_optin[MAX_DEVICES] = {};

}  // namespace

// 2-D bf16/fp16 row-major [rows, cols] tensor, box [box_rows x 64 columns], 128-byte swizzle, zero fill.
bool make_tmap_16bit_2d(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld_elems,
                        int box_rows, bool f16, std::string* err) {
  EncodeTiledFn enc = get_encode();
  if (!enc) { if (err) *err = "cuTensorMapEncodeTiled is not available from the CUDA driver"; return false; }
  if ((reinterpret_cast<uintptr_t>(base) & 15) || ((ld_elems * 2) & 15)) {
    if (err) *err = "TMA operand needs a 16-byte aligned base and row pitch";
    return false;
  }
  cuuint64_t dims[2] = {cuuint64_t(cols), cuuint64_t(rows)};
  cuuint64_t strides[1] = {cuuint64_t(ld_elems) * 2};
  cuuint32_t box[2] = {cuuint32_t(TILE_K), cuuint32_t(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(tm, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (err) *err = "cuTensorMapEncodeTiled failed with CUresult " + std::to_string(int(r));
    return false;
  }
  return true;
}

int gemm_pick_bn(int M) {
  if (M >= 256) return 256;
  return ((M + 15) / 16) * 16;
}

int gemm_pick_splits(int M, int n_out, int K, int num_sms, int mode) {
  if (gemm2_preferred(M, n_out)) {
    int bnt = 256, s = 1;
    gemm2_pick(M, n_out, K, mode, &bnt, &s);
    return s;
  }
  // Weight streaming (few rows): keep every SM fed.  Many rows: one slice (tensor-bound, no reduction pass).
  const int k_tiles = (K + TILE_K - 1) / TILE_K;
  const int tiles = ((n_out + TILE_W - 1) / TILE_W) * ((M + 255) / 256);
  if (tiles >= num_sms || k_tiles < 8) return 1;
  // One wave, two CTAs per SM - but a cluster lives in one GPC, and clusters stop fitting before the last of the 296 places is taken:
  // 48 tiles (n_out = 6144, K = 4096, 16 rows) 5 slices 12.0 us, 6 17.3; 40 tiles (5120 x 5120, 96 rows) 6 17.1, 7 26.3; 64 tiles
  // 4 17.6, 5 24.1; 96 tiles 2 23.8, 3 29.9.  Clusters of two still fit at 274 CTAs (137 tiles: 1 slice 26.9 us, 2 25.7, 3 31.7).
  int want = 256 * num_sms / 148 / tiles;
  if (want < 2 && 2 * tiles <= 276 * num_sms / 148) want = 2;
  // (down to one K-tile per slice: the cluster's read-out, a slice's share of the columns in turn, is longer than a short K loop, and it is more
  // slices that shorten it.  K = 512, n_out = 256, 2 / 4 / 8 slices: 128 rows 18.4 / 11.8 / 9.2 us, 64 11.8 / 8.2 / 6.6, 16 6.6 / 5.6 / 5.1)
  int s = want < k_tiles ? want : k_tiles;
  if (s > GEMM_MAX_SPLITS) s = GEMM_MAX_SPLITS;
  return s < 1 ? 1 : s;
}

// Launches y = x W^T.  tmW must describe W with box rows 128; x is described here (box rows BN).
cudaError_t gemm_launch(const GemmCall& c, cudaStream_t stream, Tracker* trk, std::string* err) {
  if (c.addend == nullptr && gemm2_preferred(c.M, c.n_out)) return gemm2_launch(c, stream, trk, err);
  {
    // the opt-in shared-memory limit is a per-device function attribute
    const cudaError_t e = once_per_device(g_attr_done, [](int dev) {
      cudaError_t e2 = cudaDeviceGetAttribute(&g_smem_optin[dev], cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      if (e2 != cudaSuccess) return e2;
      return cudaFuncSetAttribute(gemm_tcgen05_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, g_smem_optin[dev]);
    });
    if (e != cudaSuccess) return e;
  }
  const int smem_optin = g_smem_optin[current_device()];
  GemmArgs g{};
  g.M = c.M; g.N_out = c.n_out; g.K = c.K;
  g.BN = gemm_pick_bn(c.M);
  g.k_tiles_total = (c.K + TILE_K - 1) / TILE_K;
  int splits = c.splits < 1 ? 1 : (c.splits > GEMM_MAX_SPLITS ? GEMM_MAX_SPLITS : c.splits);
  if (splits > g.k_tiles_total) splits = g.k_tiles_total;
  g.k_tiles_per_split = (g.k_tiles_total + splits - 1) / splits;
  splits = (g.k_tiles_total + g.k_tiles_per_split - 1) / g.k_tiles_per_split;   // no empty slice
  const int n_tiles_w = (c.n_out + TILE_W - 1) / TILE_W;
  uint32_t cols = 32;
  while (cols < uint32_t(g.BN)) cols <<= 1;
  g.tmem_cols = cols;
  const size_t stage_bytes = A_STAGE_BYTES + size_t(g.BN) * TILE_K * 2;
  const size_t fixed = sizeof(GemmSmemTail) + 1024;
  // Weight streaming (narrow activation tile): size the ring so that TWO CTAs fit on an SM; one CTA's prologue and
  // epilogue then overlap the other's stream.  Wide tiles take the whole SM.
  const size_t budget = (g.BN <= 128) ? size_t(smem_optin) / 2 - 1024 : size_t(smem_optin);
  int stages = int((budget - fixed) / stage_bytes);
  if (stages > GEMM_MAX_STAGES) stages = GEMM_MAX_STAGES;
  if (stages > g.k_tiles_per_split) stages = g.k_tiles_per_split < 2 ? 2 : g.k_tiles_per_split;
  if (stages < 2) { if (err) *err = "shared memory too small for the GEMM pipeline"; return cudaErrorInvalidValue; }
  g.stages = stages;
  g.status = c.status;
  g.f16 = c.f16 ? 1 : 0;
  g.logits = c.logits; g.addend = c.addend; g.ld_add = c.ld_add; g.keys = c.keys; g.part_val = c.part_val; g.part_idx = c.part_idx;
  g.keep_w = c.keep_weights_in_l2 ? 1 : 0;
  g.early_w = c.w_stable ? 1 : 0;
  g.ldo = c.ldo;
  if (splits > 1 && c.mode == EPI_ARGMAX) { if (err) *err = "LM-head epilogue cannot be K-sliced"; return cudaErrorInvalidValue; }
  if (splits > 1 && size_t(stages) * stage_bytes < size_t(g.BN) * TILE_W * 4) {
    if (err) *err = "K-slices: the accumulator does not fit where the pipeline was";
    return cudaErrorInvalidValue;
  }
  g.mode = c.mode; g.out = c.out;
  CUtensorMap tmB;
  if (!make_tmap_16bit_2d(&tmB, c.x, c.M, c.K, c.ldx, g.BN, c.f16, err)) return cudaErrorInvalidValue;
  dim3 grid((c.M + g.BN - 1) / g.BN, n_tiles_w, splits);
  const size_t smem = size_t(stages) * stage_bytes + fixed;
  trk_begin(trk, c.label ? c.label : "gemm", 2.0 * c.M * c.n_out * c.K, 2.0 * c.n_out * c.K,
            gemm_io_bytes(c.M, c.n_out, c.K, c.mode, c.logits != nullptr));
  if (c.defer_tail) *c.defer_tail = GemmTail{};
  cudaError_t e = launch_pdl_cluster(gemm_tcgen05_kernel, grid, dim3(192), dim3(1, 1, splits), smem, stream, *c.tmW, tmB, g);
  trk_end(trk);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t argmax_init_launch(unsigned long long* keys, int M, cudaStream_t stream) {
  const cudaError_t e = launch_pdl(argmax_init_kernel, dim3((M + 255) / 256), dim3(256), 0, stream, keys, M);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t argmax_ids_launch(const unsigned long long* keys, int M, int* ids, const int* id_map, cudaStream_t stream, Tracker* trk) {
  trk_begin(trk, "argmax_ids", 0, double(M) * 12);
  const cudaError_t e = launch_pdl(argmax_ids_kernel, dim3((M + 255) / 256), dim3(256), 0, stream, keys, M, ids, id_map);
  trk_end(trk);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace hspec
