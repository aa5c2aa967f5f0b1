// Work list of the tcgen05 attention kernel: shared between attention_tc.cu, which walks it, and the kernel that opens a draft
// step and builds it there once for all layers (the list depends on the context lengths only).
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace hspec {

constexpr int ATTN_KT = 128;         // keys per tile

// Geometry of one work item's key range, computed identically by every role.
struct AttnRange {
  int base;        // first position of the visible prefix, rounded down to a page boundary
  int n_chunks;
  int p_begin;     // first position of this chunk
  int n_full;      // 128-key tiles fetched by TMA
  int rem;         // valid prefix keys after the full tiles (only in the last chunk)
  int n_manual;    // 0, 1 or 2 hand-loaded tiles (ragged end and/or the block's own keys)
  int T;           // tiles in total
  bool last;
};

__device__ __forceinline__ AttnRange make_range(int ctx, int window, int chunk, int c, int k) {
  AttnRange g;
  const int lo0 = (window > 0) ? max(0, ctx - window + 1) : 0;
  g.base = lo0 & ~15;
  const int len = ctx - g.base;
  g.n_chunks = max(1, (len + chunk - 1) / chunk);
  g.last = (c == g.n_chunks - 1);
  g.p_begin = g.base + c * chunk;
  const int p_end = min(ctx, g.p_begin + chunk);
  const int span = max(0, p_end - g.p_begin);
  g.n_full = span / ATTN_KT;
  g.rem = span - g.n_full * ATTN_KT;
  g.n_manual = g.last ? ((g.rem + k <= ATTN_KT) ? 1 : 2) : 0;
  g.T = g.n_full + g.n_manual;
  return g;
}

// One item per (request, KV head, context chunk, 128-row tile), longest first (bucketed by tile count), heads of one request and
// chunk next to each other so the CTAs that run them at the same time read neighbouring bytes of the same pages.  The order
// inside a bucket depends on atomics; every item is computed independently, so results do not.  Run by one block; `bucket` and
// `offset` are 64 ints of its shared memory each.
__device__ __forceinline__ void attn_build_plan(const AttnPlan& a, int* bucket, int* offset) {
  const int per_chunk = a.Hkv * a.n_row_tiles;
  const int pairs = a.B * a.max_chunks;            // one thread per (request, chunk slot); slots past n_chunks are skipped
  auto length = [&](int b) { return min(max(a.ctx_lens[b], 0), a.max_ctx); };
  for (int i = threadIdx.x; i < 64; i += blockDim.x) bucket[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < pairs; i += blockDim.x) {
    const int b = i / a.max_chunks, c = i % a.max_chunks;
    if (c == 0 && a.ctx_lens[b] != length(b)) atomicAdd(a.status + STATUS_WORD_BAD_INPUT, 1u);
    const AttnRange g = make_range(length(b), a.window, a.chunk, c, a.k);
    if (c < g.n_chunks) atomicAdd(&bucket[min(g.T, 63)], per_chunk);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int off = 0;
    for (int T = 63; T >= 0; --T) { offset[T] = off; off += bucket[T]; }
    *a.count = off;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < pairs; i += blockDim.x) {
    const int b = i / a.max_chunks, c = i % a.max_chunks;
    const int ctx = length(b);
    const AttnRange g = make_range(ctx, a.window, a.chunk, c, a.k);
    if (c >= g.n_chunks) continue;
    int at = atomicAdd(&offset[min(g.T, 63)], per_chunk);
    for (int kvh = 0; kvh < a.Hkv; ++kvh)
      for (int rt = 0; rt < a.n_row_tiles; ++rt) a.items[at++] = make_int4(b, kvh | (rt << 16), c, ctx);
  }
}

}  // namespace hspec
