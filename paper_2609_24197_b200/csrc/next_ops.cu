// Steps next to the draft block: the acceptance rule of App. A, the draft probability it divides by, and the
// causal correction of Sec. 3.3.3 (a first-order dependency between adjacent draft positions applied to the logits).
#include "common.cuh"
#include "kernels.h"

#include <cstdlib>

namespace hspec {

namespace {

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// ------------------------------------------------------------------ acceptance rule (App. A)
// One warp per request: n[b] = number of leading positions with min(1, P_T / P_D) >= alpha, all in fp32 with IEEE
// division.  0 / 0 (NaN) rejects; P_D = 0 with P_T > 0 (+inf) accepts.
__global__ void accept_kernel(const float* __restrict__ pt, const float* __restrict__ pd, const float* __restrict__ alpha,
                              int* __restrict__ n_accept, int B, int k) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= B) return;
  int n = k;
  for (int base = 0; base < k; base += 32) {
    const int i = base + lane;
    bool ok = true;
    if (i < k) {
      const float r = __fdiv_rn(pt[size_t(b) * k + i], pd[size_t(b) * k + i]);
      ok = !(r != r) && fminf(1.0f, r) >= alpha[size_t(b) * k + i];
    }
    const unsigned bad = __ballot_sync(0xffffffffu, !ok);
    if (bad != 0u) { n = base + __ffs(bad) - 1; break; }
  }
  if (lane == 0) n_accept[b] = n;
}

// ------------------------------------------------------------------ softmax probability of one token per row
// A cluster of S blocks per row (S = 1, 2, 4 or 8), one pass over the fp32 logits: every thread keeps a running (max, sum of
// exp) over its share, 16 values at a time with their loads in flight together; the warps, then the blocks (through the first
// block's shared memory) merge theirs; p = exp(z[id] - max) / sum.
// One request's block is 16 rows: with a block per row 132 of the 148 SMs had nothing to read.  2048 rows of 152 064: 201 -> 188 us
// (6.6 TB/s) from the four loads in flight.
__global__ void __launch_bounds__(512)
token_probs_kernel(const float* __restrict__ logits, long long ld, const int* __restrict__ ids, float* __restrict__ p, int V, int S) {
  pdl_wait();
  pdl_trigger();
  if (S > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int m = blockIdx.x / S, part = blockIdx.x % S;
  const float* z = logits + size_t(m) * ld;
  float mx = -INFINITY, sum = 0.f;
  auto add = [&](float v) {                       // (-inf entries contribute nothing, also while the maximum is still -inf)
    if (v > mx) { sum = sum * __expf(mx - v) + 1.f; mx = v; }
    else if (v > -INFINITY) sum += __expf(v - mx);
  };
  const bool vec = ((reinterpret_cast<uintptr_t>(z) & 15) == 0);
  const int V4 = vec ? (V >> 2) : 0;
  const int per = (V4 + S - 1) / S, end4 = min(V4, (part + 1) * per);
  constexpr int U = 4;                            // 16-byte loads in flight per thread
  for (int i0 = part * per + threadIdx.x; i0 < end4; i0 += U * int(blockDim.x)) {
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * int(blockDim.x);
      v[u] = i < end4 ? __ldcs(reinterpret_cast<const float4*>(z) + i) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    }
    // local maximum first: one rescale per sixteen elements
    float mu = -INFINITY;
#pragma unroll
    for (int u = 0; u < U; ++u) mu = fmaxf(mu, fmaxf(fmaxf(v[u].x, v[u].y), fmaxf(v[u].z, v[u].w)));
    if (mu > mx) { sum *= __expf(mx - mu); mx = mu; }
    if (mx > -INFINITY) {
#pragma unroll
      for (int u = 0; u < U; ++u) sum += (__expf(v[u].x - mx) + __expf(v[u].y - mx)) + (__expf(v[u].z - mx) + __expf(v[u].w - mx));
    }
  }
  for (int i = V4 * 4 + part * int(blockDim.x) + threadIdx.x; i < V; i += S * int(blockDim.x)) add(z[i]);
  auto merge = [&](float omx, float osum) {
    const float nm = fmaxf(mx, omx);
    if (nm == -INFINITY) return;
    sum = (mx > -INFINITY ? sum * __expf(mx - nm) : 0.f) + (omx > -INFINITY ? osum * __expf(omx - nm) : 0.f);
    mx = nm;
  };
  for (int off = 16; off > 0; off >>= 1) {
    const float omx = __shfl_xor_sync(0xffffffffu, mx, off);
    const float osum = __shfl_xor_sync(0xffffffffu, sum, off);
    merge(omx, osum);
  }
  __shared__ float smx[32], ssum[32];
  __shared__ float cmx[8], csum[8];               // in the cluster's first block: one pair per block
  if ((threadIdx.x & 31) == 0) { smx[threadIdx.x >> 5] = mx; ssum[threadIdx.x >> 5] = sum; }
  if (S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every block of the cluster runs by now
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nw = blockDim.x >> 5;
    mx = threadIdx.x < nw ? smx[threadIdx.x] : -INFINITY;
    sum = threadIdx.x < nw ? ssum[threadIdx.x] : 0.f;
    for (int off = 16; off > 0; off >>= 1) {
      const float omx = __shfl_xor_sync(0xffffffffu, mx, off);
      const float osum = __shfl_xor_sync(0xffffffffu, sum, off);
      merge(omx, osum);
    }
    if (S > 1 && threadIdx.x == 0) {
      uint32_t r_mx, r_sum;
      asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r_mx) : "r"(smem_u32(cmx + part)));
      asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r_sum) : "r"(smem_u32(csum + part)));
      asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r_mx), "f"(mx) : "memory");
      asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r_sum), "f"(sum) : "memory");
    }
  }
  if (S > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (part == 0 && threadIdx.x == 0) {
      mx = cmx[0]; sum = csum[0];
      for (int i = 1; i < S; ++i) merge(cmx[i], csum[i]);
    }
  }
  if (part == 0 && threadIdx.x == 0) p[m] = expf(z[ids[m]] - mx) / sum;
}

// ------------------------------------------------------------------ Markov head (Sec. 3.3.3)
// x[b, :] = W_in[prev[b], :] (16-bit rows copied as they are): the predecessor's factor row, the activation of the
// position's rank-r product with W_out.
__global__ void markov_gather_kernel(const uint16_t* __restrict__ W_in, const int* __restrict__ prev, long long prev_stride,
                                     uint16_t* __restrict__ x, int r) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x;
  const uint16_t* src = W_in + size_t(prev[size_t(b) * prev_stride]) * r;
  for (int i = threadIdx.x; i < (r >> 3); i += blockDim.x)
    reinterpret_cast<uint4*>(x + size_t(b) * r)[i] = reinterpret_cast<const uint4*>(src)[i];
}

// Position i of every request: lowest index among the per-tile maxima -> ids[b * k + i] (mapped to a token id when the
// drafter's vocabulary is pruned), and the factor row of that token -> x[b, :] for position i + 1.
// The partials are [tile][request]: a block takes eight consecutive requests, thread (tid % 8, tid / 8) walks every
// 128th tile of its request, so that eight neighbouring threads read one 32-byte sector (1024 threads: there are only
// B / 8 blocks, and the kernel sits between two dependent GEMMs, so its latency counts).
__global__ void __launch_bounds__(1024)
markov_reduce_gather_kernel(const float* __restrict__ pv, const int* __restrict__ pi, int n_tiles, int B,
                            int* __restrict__ ids, int k, int i, const int* __restrict__ id_map,
                            const uint16_t* __restrict__ W_in, uint16_t* __restrict__ x, int r, int gather) {
  pdl_wait();
  pdl_trigger();
  const int rr = threadIdx.x & 7, b = blockIdx.x * 8 + rr;
  float v = -INFINITY;
  int idx = 0x7fffffff;
  auto take = [&](float ov, int oi) { if (ov > v || (ov == v && oi < idx)) { v = ov; idx = oi; } };
  if (b < B) {
    for (int t = threadIdx.x >> 3; t < n_tiles; t += 256) {          // two tiles' loads in flight per step
      const int t2 = t + 128;
      const float v1 = pv[size_t(t) * B + b], v2 = t2 < n_tiles ? pv[size_t(t2) * B + b] : -INFINITY;
      const int i1 = pi[size_t(t) * B + b], i2 = t2 < n_tiles ? pi[size_t(t2) * B + b] : 0x7fffffff;
      take(v1, i1);
      take(v2, i2);
    }
  }
  for (int off = 8; off < 32; off <<= 1) take(__shfl_xor_sync(0xffffffffu, v, off), __shfl_xor_sync(0xffffffffu, idx, off));
  __shared__ float sv[32][8];
  __shared__ int si[32][8];
  __shared__ int token[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane < 8) { sv[warp][lane] = v; si[warp][lane] = idx; }
  __syncthreads();
  if (threadIdx.x < 8) {
    int tok = 0;
    if (b < B) {
      v = sv[0][rr]; idx = si[0][rr];
      for (int w = 1; w < 32; ++w) take(sv[w][rr], si[w][rr]);
      if (idx == 0x7fffffff) idx = 0;                     // (a wait that gave up: the next position still needs a factor row)
      tok = id_map ? id_map[idx] : idx;
      ids[size_t(b) * k + i] = tok;
    }
    token[rr] = tok;
  }
  __syncthreads();
  if (gather) {
    // warp w copies the factor row of request blockIdx.x * 8 + w (16 bytes per lane and step)
    const int bw = blockIdx.x * 8 + warp;
    if (warp < 8 && bw < B) {
      const uint16_t* src = W_in + size_t(token[warp]) * r;
      for (int j = lane; j < (r >> 3); j += 32)
        reinterpret_cast<uint4*>(x + size_t(bw) * r)[j] = reinterpret_cast<const uint4*>(src)[j];
    }
  }
}

}  // namespace

cudaError_t accept_launch(const float* pt, const float* pd, const float* alpha, int* n_accept, int B, int k, cudaStream_t stream) {
  const cudaError_t e = launch_pdl(accept_kernel, dim3((B + 7) / 8), dim3(256), 0, stream, pt, pd, alpha, n_accept, B, k);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t token_probs_launch(const float* logits, long long ld, const int* ids, float* p, int M, int V, cudaStream_t stream) {
  // enough blocks for two per SM, as long as a block still has a few KB to read
  int S = 1;
  while (S < 8 && M * S < 2 * 148 && V / (2 * S) >= 4096) S *= 2;
  return launch_pdl_cluster(token_probs_kernel, dim3(unsigned(M) * S), dim3(512), dim3(S), 0, stream, logits, ld, ids, p, V, S);
}

size_t markov_workspace_bytes(int B, int Vd, int r) {
  const size_t vt = (size_t(Vd) + 127) / 128;
  return round_up(size_t(B) * r * 2, 256) + 2 * round_up(vt * B * 4, 256) + round_up(markov_chain_bytes(B), 256) + 256;
}

// Up to 128 requests all positions run in one launch (markov_chain.cu; us per position with the logits written, GEMM + reduction against
// it: 32 requests, V = 151 936 48 / 21, 96, 32 000 34 / 14, 64, 152 064 69 / 30, 1, 32 000 10.4 / 7.6); above that, and where that launch
// is refused, one GEMM and one reduction per position.
cudaError_t markov_launch(const MarkovCall& c, cudaStream_t stream, Tracker* trk, std::string* err) {
  if (markov_chain_supported(c.B, c.Vd, c.r)) {
    const cudaError_t e = markov_chain_launch(c, stream, trk);
    if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) return e;
  }
  const size_t vt = (size_t(c.Vd) + 127) / 128;
  uint8_t* ws = reinterpret_cast<uint8_t*>(c.ws);
  uint16_t* x = reinterpret_cast<uint16_t*>(ws);
  float* part_val = reinterpret_cast<float*>(ws + round_up(size_t(c.B) * c.r * 2, 256));
  int* part_idx = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(part_val) + round_up(vt * c.B * 4, 256));
  trk_begin(trk, "markov_gather");
  markov_gather_kernel<<<c.B, 32, 0, stream>>>(reinterpret_cast<const uint16_t*>(c.W_in), c.last_token, 1, x, c.r);
  trk_end(trk);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int i = 0; i < c.k; ++i) {
    GemmCall g{};
    g.tmW = c.tmW_out; g.x = x; g.ldx = c.r; g.M = c.B; g.n_out = c.Vd; g.mode = EPI_ARGMAX;
    g.f16 = c.f16; g.K = c.r; g.splits = 1;
    g.addend = c.logits + size_t(i) * c.ld;                 // row b of this GEMM is row b * k + i of the block's logits
    g.ld_add = (long long)c.k * c.ld;
    g.logits = c.write_logits ? c.logits + size_t(i) * c.ld : nullptr;
    g.ldo = (long long)c.k * c.ld;
    g.part_val = part_val; g.part_idx = part_idx; g.status = c.status;
    g.keep_weights_in_l2 = true;                            // W_out (78 MB at V = 152 064, r = 256) serves every position
    g.label = "markov";
    e = gemm_launch(g, stream, trk, err);
    if (e != cudaSuccess) return e;
    trk_begin(trk, "markov_reduce");
    e = launch_pdl(markov_reduce_gather_kernel, dim3((c.B + 7) / 8), dim3(1024), 0, stream, (const float*)part_val, (const int*)part_idx,
                   int(vt), c.B, c.ids, c.k, i, c.id_map, reinterpret_cast<const uint16_t*>(c.W_in), x, c.r, int(i + 1 < c.k));
    trk_end(trk);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace hspec
