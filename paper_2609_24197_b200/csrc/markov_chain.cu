// The causal-correction head over all k positions of a block in one launch (Sec. 3.3.3; up to 128 requests).
//
// Position i needs the token chosen at i - 1, so the positions run one after the other: logits'[b, i, :] = logits[b, i, :] +
// W_out x_b with x_b = W_in[token at i - 1], then the arg-max.  What a position has to move is W_out (78 MB at a vocabulary of
// 152 064 and rank 256; it stays in the L2 for the next position) and the batch's logits rows (read, and written back when the
// caller wants them).  As one GEMM and one reduction launch per position it took 47.6 + 8.9 us at 32 requests and that
// vocabulary and 44 + 9.8 us at 96 requests and 32 000 rows: CTAs too short to fill their pipelines, a reduction network per
// 16 columns, and a launch boundary on each side.  As one launch for all positions: 20 and 14 us per position (and 46 against 64 at
// 128 requests and 152 064 rows, logits not written; with few rows to go over and 97 requests or more it is 12 us of gathers, barriers and
// reductions a position, where two launches took 10).
//
// Here one cooperative kernel (one CTA per SM) walks the positions with a grid barrier between them:
//   warp 16       producer: 64-column boxes of W_out (128 vocabulary rows each) through a ring of 16 KB stages; it does not
//                 depend on the tokens and runs on into the next position while the grid barrier is under way
//   warp 17       one thread issues the MMAs: A = W_out tile (vocabulary rows = TMEM lanes), B = the requests' factor rows
//                 (resident in shared memory for the whole position), into one of two accumulators
//   warps 0..15   four warps per TMEM lane quarter, 8 columns (requests) per chunk.  A thread owns one vocabulary row of every
//                 tile and keeps the running (max, tile) of its requests in registers over all tiles of the position: the
//                 reduction across lanes, warps and CTAs happens once per position and not once per tile.  The logits of
//                 the next tile (at the end the next position's first) are requested as soon as a chunk's registers are free.
// The maxima meet in a 64-bit key per request, (ordered value, ~index), through atomic maxima: the result does not depend on
// any order, and ties go to the lowest index.  Every wait is bounded, the grid barrier's included.
#include "common.cuh"
#include "kernels.h"

#include <cstdlib>

namespace hspec {

namespace {

constexpr int EPI_WARPS = 16, EPI_THREADS = EPI_WARPS * 32, CHAIN_THREADS = EPI_THREADS + 64;
constexpr int TILE_W = 128, TILE_K = 64;
constexpr uint32_t W_STAGE = TILE_W * TILE_K * 2;
constexpr int MAX_STAGES = 8;
constexpr int MAX_B = 128;

struct ChainArgs {
  float* logits;
  long long ld;
  const uint16_t* W_in;
  const int* last_token;
  const int* id_map;
  int* ids;
  unsigned long long* keys;   // [3][B], zeroed before the launch
  unsigned int* arrived;      // grid barrier, zeroed before the launch
  uint32_t* status;
  int B, BN, k, Vd, r, kt, stages, n_tiles, write_logits, f16;
  uint32_t tmem_cols;
};

struct __align__(8) ChainTail {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t x_ready;
  unsigned long long key[4][MAX_B];   // per TMEM lane quarter
  int token[MAX_B];
  uint32_t tmem_base;
  uint32_t epi_abort;
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory"); }

__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long v, int off) {
  const uint32_t lo = __shfl_xor_sync(0xffffffffu, uint32_t(v), off), hi = __shfl_xor_sync(0xffffffffu, uint32_t(v >> 32), off);
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}
// 8 columns x 32 lanes -> the maximum of column `col` in every fourth lane (each round a lane hands half of its columns over)
__device__ __forceinline__ unsigned long long max_over_lanes8(unsigned long long (&v)[8], int lane, int& col) {
#pragma unroll
  for (int half = 4, off = 16; half >= 1; half >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (t >= half) break;
      const unsigned long long send = up ? v[t] : v[t + half], keep = up ? v[t + half] : v[t];
      const unsigned long long got = shfl_xor_u64(send, off);
      v[t] = keep > got ? keep : got;
    }
  }
#pragma unroll
  for (int off = 2; off >= 1; off >>= 1) {
    const unsigned long long got = shfl_xor_u64(v[0], off);
    v[0] = v[0] > got ? v[0] : got;
  }
  col = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
  return v[0];
}

// NCH = chunks of 8 requests per epilogue warp (4 warps share a lane quarter): 32 NCH requests
template <int NCH>
__global__ void __launch_bounds__(CHAIN_THREADS, 1)
markov_chain_kernel(const __grid_constant__ CUtensorMap tmW, ChainArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sX = smem;                                            // [kt][BN rows x 64 columns], K-major, 128-byte swizzle
  uint8_t* sW = smem + size_t(a.kt) * a.BN * 128;
  ChainTail* tail = reinterpret_cast<ChainTail*>(sW + size_t(a.stages) * W_STAGE);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grid = int(gridDim.x), cta = int(blockIdx.x);
  const int n_my = (a.n_tiles - cta + grid - 1) / grid;          // >= 1: the grid is never larger than the tile count

  if (tid == 0) {
    tma_prefetch_desc(&tmW);
    for (int s = 0; s < a.stages; ++s) { mbar_init(smem_u32(&tail->full[s]), 1); mbar_init(smem_u32(&tail->empty[s]), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&tail->acc_full[i]), 1); mbar_init(smem_u32(&tail->acc_empty[i]), EPI_WARPS); }
    mbar_init(smem_u32(&tail->x_ready), EPI_WARPS);
    tail->epi_abort = 0;
    fence_mbar_init();
  }
  if (warp == 17) {
    tmem_alloc(smem_u32(&tail->tmem_base), a.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tail->tmem_base;

  if (warp == 16) {
    if (elect_one()) {
      const uint64_t pol = policy_evict_last();                  // every position reads the same matrix
      uint32_t it = 0;
      bool ok = true;
      for (int pos = 0; pos < a.k && ok; ++pos)
        for (int t = 0; t < n_my && ok; ++t)
          for (int kt = 0; kt < a.kt; ++kt, ++it) {
            const int s = it % a.stages;
            const uint32_t lap = it / a.stages;
            if (lap > 0 && !mbar_wait(smem_u32(&tail->empty[s]), (lap - 1) & 1)) {
              atomicExch(a.status, STATUS_TIMEOUT_PRODUCER);
              ok = false;
              break;
            }
            const uint32_t full = smem_u32(&tail->full[s]);
            mbar_expect_tx(full, W_STAGE);
            tma_load_2d(smem_u32(sW + size_t(s) * W_STAGE), &tmW, kt * TILE_K, (cta + t * grid) * TILE_W, full, pol);
          }
    }
  } else if (warp == 17) {
    if (elect_one()) {
      const uint32_t idesc = umma_idesc_m128(a.BN, a.f16 != 0);
      uint32_t it = 0, gt = 0;
      bool ok = true;
      for (int pos = 0; pos < a.k && ok; ++pos) {
        if (!mbar_wait(smem_u32(&tail->x_ready), pos & 1, 4000000000ull)) { ok = false; break; }
        tc_fence_after();
        for (int t = 0; t < n_my && ok; ++t, ++gt) {
          const uint32_t acc = gt & 1, use = gt >> 1;
          if (use > 0 && !mbar_wait(smem_u32(&tail->acc_empty[acc]), (use - 1) & 1)) { ok = false; break; }
          tc_fence_after();
          for (int kt = 0; kt < a.kt; ++kt, ++it) {
            const int s = it % a.stages;
            if (!mbar_wait(smem_u32(&tail->full[s]), (it / a.stages) & 1)) { ok = false; break; }
            tc_fence_after();
            const uint64_t da = umma_desc_kmajor_sw128(smem_u32(sW + size_t(s) * W_STAGE));
            const uint64_t db = umma_desc_kmajor_sw128(smem_u32(sX + size_t(kt) * a.BN * 128));
#pragma unroll
            for (int kk = 0; kk < TILE_K / 16; ++kk)
              umma_bf16(tmem + acc * a.BN, da + uint64_t(kk * 2), db + uint64_t(kk * 2), idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            umma_commit(smem_u32(&tail->empty[s]));
          }
          if (ok) umma_commit(smem_u32(&tail->acc_full[acc]));
        }
      }
      if (!ok) atomicExch(a.status, STATUS_TIMEOUT_MMA);
    }
  } else {
    const int q = warp & 3, cg = warp >> 2;
    const int row_in_tile = q * 32 + lane;
    bool ok = true;                                              // a warp that gave up skips its work but keeps the barriers
    uint32_t gt = 0;
    // factor rows of the batch's previous tokens -> shared memory (zeros past B and past r)
    auto gather = [&](auto token_of) {
      const int chunks = a.kt * 8;                               // 16-byte pieces of a row
      for (int i = tid; i < a.BN * chunks; i += EPI_THREADS) {
        const int b = i / chunks, c = i % chunks;
        const bool valid = b < a.B && c * 8 < a.r;
        const uint16_t* src = valid ? a.W_in + size_t(token_of(b)) * a.r + c * 8 : a.W_in;
        cp_async16(smem_u32(sX) + (c >> 3) * a.BN * 128 + (b >> 3) * 1024 + (b & 7) * 128 + (((c & 7) ^ (b & 7)) << 4), src, valid);
      }
      cp_async_commit();
      cp_async_wait<0>();
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&tail->x_ready));
    };
    // Logits on their way: AQ chunks (of the NCH a tile has), refilled as they are used.  With four chunks of maxima 96 registers have
    // room for one: a spilled logit waits for its load on the spot (us per position at 128 requests, V = 152 064: one chunk 62.8,
    // two 77.5, four 93.8).
    constexpr int AQ = NCH == 4 ? 1 : NCH;
    static_assert(AQ == NCH || AQ == 1, "the refill below knows these two");
    float add[AQ * 8];
    const size_t req_stride = size_t(a.k) * a.ld;                // from request to request in the block's logits
    // (the empty asm keeps the walk a chain of additions: as base + j x stride the offsets of all columns were kept in registers
    // across the tiles, and the logits spilled: 18.8 -> 14.0 us per position at 96 requests, 119 -> 94 at 128)
    auto step_row = [&](auto*& p) { p += req_stride; asm volatile("" : "+l"(p)); };
    auto load_add = [&](int u, int pos, int t) {                 // chunk u of this CTA's t-th tile at position pos
      const int n = (cta + t * grid) * TILE_W + row_in_tile, c0 = (u * 4 + cg) * 8;
      const float* src = a.logits + size_t(pos) * a.ld + n + size_t(c0) * req_stride;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        add[u % AQ * 8 + j] = (n < a.Vd && c0 + j < a.B) ? __ldcs(src) : 0.f;
        step_row(src);
      }
    };
    // With a single chunk in flight the others' lines are at least in the L2: a warp's 32 columns of a tile are 32 lines, one per lane.  (128
    // requests, rank 256, us per position, logits not written / written, without -> with: V = 32 000 19.6 / 20.9 -> 17.2 / 18.3, 152 064 52 / 63 -> 46 / 52.)
    auto prefetch_add = [&](int pos, int t) {
      const int n = (cta + t * grid) * TILE_W + q * 32, c = (lane >> 3) * 32 + cg * 8 + (lane & 7);
      if (n < a.Vd && c < a.B) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.logits + size_t(pos) * a.ld + n + size_t(c) * req_stride));
    };
    if (AQ < NCH) prefetch_add(0, 0);
#pragma unroll
    for (int u = 0; u < AQ; ++u) load_add(u, 0, 0);
    gather([&](int b) { return a.last_token[b]; });

    for (int pos = 0; pos < a.k; ++pos) {
      float best[NCH * 8];
      uint32_t ord[NCH * 2];                                     // ordinal of the best tile, four 8-bit values per register
#pragma unroll
      for (int j = 0; j < NCH * 8; ++j) best[j] = -INFINITY;
#pragma unroll
      for (int j = 0; j < NCH * 2; ++j) ord[j] = 0;
      for (int t = 0; t < n_my; ++t, ++gt) {
        const uint32_t acc = gt & 1;
        const int n = (cta + t * grid) * TILE_W + row_in_tile;
        const bool n_ok = n < a.Vd;
        const bool more = t + 1 < n_my || pos + 1 < a.k;
        const int pos2 = t + 1 < n_my ? pos : pos + 1, t2 = t + 1 < n_my ? t + 1 : 0;
        if (AQ < NCH && more) prefetch_add(pos2, t2);
        if (ok && !mbar_wait(smem_u32(&tail->acc_full[acc]), (gt >> 1) & 1, 6000000000ull)) {
          atomicExch(a.status, STATUS_TIMEOUT_EPILOGUE);
          ok = false;
        }
        if (!ok) continue;
        tc_fence_after();
#pragma unroll
        for (int u = 0; u < NCH; ++u) {
          const int c0 = (u * 4 + cg) * 8;
          if (c0 >= a.BN) break;                                 // warp-uniform
          uint32_t r[8];
          tmem_ld8(tmem + (uint32_t(q * 32) << 16) + acc * a.BN + c0, r);
          tmem_ld_wait();
          float* dst = a.logits + size_t(pos) * a.ld + n + size_t(c0) * req_stride;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float v = __uint_as_float(r[j]) + add[u % AQ * 8 + j];
            if (n_ok && c0 + j < a.B) {
              if (a.write_logits) __stcs(dst, v);
              if (v > best[u * 8 + j]) {                         // ascending tiles, strict: the lowest index wins ties, NaN never does
                best[u * 8 + j] = v;
                uint32_t& o = ord[(u * 8 + j) >> 2];             // byte j % 4 becomes t
                o = __byte_perm(o, uint32_t(t), j % 4 == 0 ? 0x3214 : j % 4 == 1 ? 0x3240 : j % 4 == 2 ? 0x3410 : 0x4210);
              }
            }
            step_row(dst);
          }
          // refill: the chunk's own successor in the next tile, or, with a single chunk in flight, the next one this warp has (a warp's last
          // chunk can lie past the batch: 112 columns are 14 chunks for 4 x 4 places)
          if (AQ == NCH) {
            if (more) load_add(u, pos2, t2);
          } else if (u + 1 < NCH && c0 + 32 < a.BN) {
            load_add(u + 1, pos, t);
          } else if (more) {
            load_add(0, pos2, t2);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tail->acc_empty[acc]));
      }
      // ---- this position's maxima: lanes, then the four lane quarters, then the CTAs
#pragma unroll
      for (int u = 0; u < NCH; ++u) {
        const int c0 = (u * 4 + cg) * 8;
        if (c0 >= a.BN) break;
        unsigned long long v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t o = (ord[(u * 8 + j) >> 2] >> ((j & 3) * 8)) & 0xffu;
          const int n = (cta + int(o) * grid) * TILE_W + row_in_tile;
          v[j] = n < a.Vd ? argmax_key(best[u * 8 + j], n) : 0ull;
        }
        int col;
        const unsigned long long m = max_over_lanes8(v, lane, col);
        if ((lane & 3) == 0) tail->key[q][c0 + col] = m;         // (one warp per quarter and chunk: written once a position)
      }
      if (!ok && lane == 0) *reinterpret_cast<volatile uint32_t*>(&tail->epi_abort) = 1;
      epi_sync();
      unsigned long long* gkeys = a.keys + size_t(pos % 3) * a.B;
      if (tid < a.B) {
        unsigned long long m = tail->key[0][tid];
#pragma unroll
        for (int i = 1; i < 4; ++i) m = m > tail->key[i][tid] ? m : tail->key[i][tid];
        if (m) atomicMax(gkeys + tid, m);
        __threadfence();
      }
      epi_sync();
      const bool last = pos + 1 == a.k;
      if (tid == 0) {
        __threadfence();
        atomicAdd(a.arrived, 1u);
        const unsigned int want = unsigned(grid) * unsigned(pos + 1);
        uint64_t t0 = 0;
        for (uint32_t i = 0; !(last && cta != 0); ++i) {         // (after the last position only CTA 0 reads the result)
          unsigned int seen;
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.arrived) : "memory");
          if (seen >= want) break;
          if ((i & 255u) == 255u) {
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > 8000000000ull) {
              atomicExch(a.status, STATUS_TIMEOUT_EPILOGUE);
              *reinterpret_cast<volatile uint32_t*>(&tail->epi_abort) = 1;
              break;
            }
          }
        }
        __threadfence();
      }
      epi_sync();
      if (*reinterpret_cast<volatile uint32_t*>(&tail->epi_abort)) break;      // (written before a barrier all have passed)
      if (last && cta != 0) break;
      if (tid < a.B) {
        const uint32_t idx = 0xffffffffu - uint32_t(__ldcg(gkeys + tid));
        const int row = idx < uint32_t(a.Vd) ? int(idx) : 0;
        const int tok = a.id_map ? a.id_map[row] : row;
        tail->token[tid] = tok;
        if (cta == 0) {
          a.ids[size_t(tid) * a.k + pos] = tok;
          // the keys of position pos - 1 were read by everybody before this barrier: clear them for position pos + 2
          a.keys[size_t((pos + 2) % 3) * a.B + tid] = 0ull;
        }
      }
      if (last) break;
      epi_sync();
      gather([&](int b) { return tail->token[b]; });
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 17) {
    tc_fence_after();
    tmem_dealloc(tmem, a.tmem_cols);
  }
}

bool g_chain_attr[4][MAX_DEVICES] = {};
int g_chain_smem[MAX_DEVICES] = {}, g_chain_sms[MAX_DEVICES] = {};

template <int NCH>
cudaError_t chain_launch_n(const CUtensorMap* tm, const ChainArgs& a, int grid, size_t smem, cudaStream_t stream) {
  const cudaError_t e = once_per_device(g_chain_attr[NCH - 1], [](int dev) {
    return cudaFuncSetAttribute(markov_chain_kernel<NCH>, cudaFuncAttributeMaxDynamicSharedMemorySize, g_chain_smem[dev]);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(CHAIN_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, markov_chain_kernel<NCH>, *tm, a);
}

bool g_chain_dev[MAX_DEVICES] = {};

// Shared memory and SMs of the current device, looked up once.  (The SM count is the context's where a limit is set from outside.)
cudaError_t chain_device(int* dev) {
  const cudaError_t e = once_per_device(g_chain_dev, [](int d) {
    cudaError_t e2 = cudaDeviceGetAttribute(&g_chain_smem[d], cudaDevAttrMaxSharedMemoryPerBlockOptin, d);
    if (e2 == cudaSuccess) e2 = cudaDeviceGetAttribute(&g_chain_sms[d], cudaDevAttrMultiProcessorCount, d);
    return e2;
  });
  *dev = current_device();
  return e == cudaSuccess && *dev < 0 ? cudaErrorInvalidDevice : e;
}

}  // namespace

size_t markov_chain_bytes(int B) { return size_t(3) * B * 8 + 16; }

// Up to 128 requests whose factor rows leave room for at least four stages of W_out (rank 256 at 128 requests does), up to 2^21 vocabulary
// rows, and no more tiles per CTA than their ordinals' byte counts.
bool markov_chain_supported(int B, int Vd, int r) {
  const size_t x = size_t((r + TILE_K - 1) / TILE_K) * ((B + 15) / 16 * 16) * 128;
  int dev = -1;
  return B <= MAX_B && x <= 128 * 1024 && Vd <= (1 << 21) && chain_device(&dev) == cudaSuccess && (Vd + TILE_W - 1) / TILE_W <= 255 * g_chain_sms[dev];
}

cudaError_t markov_chain_launch(const MarkovCall& c, cudaStream_t stream, Tracker* trk) {
  static const bool refuse = [] { const char* e = getenv("HSPEC_NO_COOPERATIVE"); return e && e[0] == '1'; }();
  if (refuse) return cudaErrorCooperativeLaunchTooLarge;
  int dev = -1;
  const cudaError_t e0 = chain_device(&dev);
  if (e0 != cudaSuccess) return e0;
  ChainArgs a{};
  a.logits = c.logits; a.ld = c.ld; a.W_in = reinterpret_cast<const uint16_t*>(c.W_in); a.last_token = c.last_token;
  a.id_map = c.id_map; a.ids = c.ids; a.status = c.status;
  a.keys = reinterpret_cast<unsigned long long*>(c.ws);
  a.arrived = reinterpret_cast<unsigned int*>(a.keys + size_t(3) * c.B);
  a.B = c.B; a.BN = (c.B + 15) / 16 * 16; a.k = c.k; a.Vd = c.Vd; a.r = c.r; a.kt = (c.r + TILE_K - 1) / TILE_K;
  a.n_tiles = (c.Vd + TILE_W - 1) / TILE_W; a.write_logits = c.write_logits; a.f16 = c.f16 ? 1 : 0;
  a.tmem_cols = 32;
  while (a.tmem_cols < uint32_t(2 * a.BN)) a.tmem_cols <<= 1;
  const size_t x_bytes = size_t(a.kt) * a.BN * 128, fixed = x_bytes + sizeof(ChainTail) + 1024;
  a.stages = int((size_t(g_chain_smem[dev]) - fixed) / W_STAGE);
  if (a.stages > MAX_STAGES) a.stages = MAX_STAGES;
  // a full SM's shared memory, so that one CTA sits on each SM
  const size_t smem = fixed + size_t(a.stages) * W_STAGE;
  const int grid = a.n_tiles < g_chain_sms[dev] ? a.n_tiles : g_chain_sms[dev];
  cudaError_t e = cudaMemsetAsync(c.ws, 0, markov_chain_bytes(c.B), stream);
  if (e != cudaSuccess) return e;
  trk_begin(trk, "markov_chain", 2.0 * c.B * c.k * double(c.Vd) * c.r, double(c.k) * c.Vd * c.r * 2,
            double(c.k) * c.B * c.Vd * (c.write_logits ? 8 : 4));
  if (a.BN <= 32) e = chain_launch_n<1>(c.tmW_out, a, grid, smem, stream);
  else if (a.BN <= 64) e = chain_launch_n<2>(c.tmW_out, a, grid, smem, stream);
  else if (a.BN <= 96) e = chain_launch_n<3>(c.tmW_out, a, grid, smem, stream);
  else e = chain_launch_n<4>(c.tmW_out, a, grid, smem, stream);
  trk_end(trk);
  if (e != cudaSuccess) cudaGetLastError();                      // (the code is returned; left behind, the next call would find it)
  if ((e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) && trk) trk->drop_last();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace hspec
