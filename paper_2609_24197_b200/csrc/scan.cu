// Mamba-2 mixer core over the k block rows, started from the injected state (paper Sec. 3.3.1).
//
// Because the recurrence S_i = a_i S_{i-1} + dt_i x_i B_i^T is linear, all k positions are evaluated in one
// pass without carrying the state:
//   y_t = exp(c_t) * (S_init C_t)  +  sum_{s<=t} exp(c_t - c_s) dt_s (C_t . B_s) x_s  +  D x_t,
//   c_t = sum_{r<=t} dt_r A   (inclusive prefix sum over the block positions, one warp shuffle scan).
// S_init (fp16 [P, N] per head) is read from HBM exactly once; it is the largest operand where N is large.  The causal
// depthwise conv + SiLU of x, B, C (zero left context), softplus(dt), the D skip and the SiLU(z) gate are part of it.
// Forms, as scan_launch() chooses them:
//   P = 64, N = 128 with scratch     scan_conv_kernel, then mamba_scan_stream_kernel (one warp per head, tensor-core fragments)
//   the same without scratch         mamba_scan_mma_kernel, everything in one
//   N <= 16                          scan_small_state_kernel, the state in registers; with the gated norm where a cluster holds a request
//   everything else                  mamba_scan_kernel / mamba_scan_five_kernel, one CTA per (request, head), the state staged in fp32
#include "common.cuh"
#include "kernels.h"

namespace hspec {

namespace {

constexpr int SCAN_THREADS = 128;
constexpr int KMAX = 32;

struct ScanArgs {
  const float* zxbcdt; long long ld_in;
  const float* dt_raw;
  const uint16_t* dt_w;   // [H, dt_rank] fp16 (or bf16): the dt columns of zxbcdt are dt_rank wide and expanded here; null: they are not
  int dt_rank, dt_bf16;
  int w_stable;           // no kernel in front writes the weights: they may be read before it has finished
  const __half* s_init;
  const float *conv_w, *conv_b, *dt_bias, *A_log, *Dskip;
  float* y;
  int B, k, Di, P, N, G, H, d_conv, d_xBC;
  int shared_rows;  // zxbcdt (and dt_raw) hold B + 1 rows: row b is position 0 of request b, row B every later position
  // row of zxbcdt / dt_raw that belongs to position i of request b
  __device__ __forceinline__ size_t in_row(int b, int i) const {
    return shared_rows ? size_t(i == 0 ? b : B) : size_t(b) * k + i;
  }
  // dt of head h before the bias, at position i of request b
  __device__ __forceinline__ float dt_pre(int b, int i, int h) const {
    const size_t row = in_row(b, i);
    if (dt_raw) return dt_raw[row * H + h];
    const float* x = zxbcdt + row * ld_in + Di + d_xBC;
    if (!dt_w) return x[h];
    const uint16_t* wr = dt_w + size_t(h) * dt_rank;
    float s = 0.f;
#pragma unroll 16
    for (int r = 0; r < dt_rank; ++r) s += x[r] * (dt_bf16 ? __uint_as_float(uint32_t(wr[r]) << 16) : __half2float(__ushort_as_half(wr[r])));
    return s;
  }
  int NP;          // padded N (row pitch of the staged state in floats)
};

// The gated norm behind the scan, where one kernel does both.
struct ScanNorm {
  const float* w;      // [Di]
  uint16_t* u;         // [B * k, Di] fp16 or bf16
  float eps;
  int bf16_out;
  uint32_t* status;
};

__device__ __forceinline__ float softplus_f(float v) { return v > 20.f ? v : log1pf(expf(v)); }

__device__ __forceinline__ void scan_general(const ScanArgs& a) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x;
  const int h = blockIdx.x, b = blockIdx.y;
  const int g = h / (a.H / a.G);
  const int k = a.k, P = a.P, N = a.N;
  float* xs = sm;                    // [k][P]
  float* Bs = xs + KMAX * P;         // [k][N]
  float* Cs = Bs + KMAX * N;         // [k][N]
  float* Wm = Cs + KMAX * N;         // [k][k]  exp(c_t - c_s) dt_s (C_t . B_s), s <= t
  float* dec = Wm + KMAX * KMAX;     // [k]     exp(c_t)
  float* dts = dec + KMAX;           // [k]
  float* cum = dts + KMAX;           // [k]
  float* Ss = cum + KMAX;            // [P][NP] staged S_init (fp32)
  const size_t row0 = size_t(b) * k;

  // ---- conv + SiLU for this head's x channels and its group's B, C channels
  const int n_ch = P + 2 * N;
  for (int idx = tid; idx < k * n_ch; idx += SCAN_THREADS) {
    const int i = idx / n_ch, cc = idx % n_ch;
    int ch;                          // channel inside xBC
    if (cc < P) ch = h * P + cc;
    else if (cc < P + N) ch = a.Di + g * N + (cc - P);
    else ch = a.Di + a.G * N + g * N + (cc - P - N);
    float acc = a.conv_b[ch];
    for (int j = 0; j < a.d_conv; ++j) {
      const int src = i - (a.d_conv - 1) + j;
      if (src >= 0) acc += a.conv_w[ch * a.d_conv + j] * a.zxbcdt[a.in_row(b, src) * a.ld_in + a.Di + ch];
    }
    const float v = silu_f(acc);
    if (cc < P) xs[i * P + cc] = v;
    else if (cc < P + N) Bs[i * N + (cc - P)] = v;
    else Cs[i * N + (cc - P - N)] = v;
  }
  // ---- dt, cumulative log-decay (warp 0: inclusive shuffle scan over the k <= 32 positions)
  if (tid < 32) {
    float dt = 0.f, dA = 0.f;
    if (tid < k) {
      const float raw = a.dt_pre(b, tid, h);
      dt = softplus_f(raw + a.dt_bias[h]);
      dA = dt * (-expf(a.A_log[h]));
    }
    float c = dA;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float up = __shfl_up_sync(0xffffffffu, c, off);
      if (tid >= off) c += up;
    }
    if (tid < k) { dts[tid] = dt; cum[tid] = c; dec[tid] = expf(c); }
  }
  // ---- stage S_init[b, h] (fp16 -> fp32), 16-byte loads
  if (a.s_init != nullptr) {
    const __half* src = a.s_init + (size_t(b) * a.H + h) * P * N;
    if ((N & 7) == 0 && (reinterpret_cast<uintptr_t>(a.s_init) & 15) == 0) {
      const int vec = P * N / 8;
      for (int idx = tid; idx < vec; idx += SCAN_THREADS) {
        const uint4 raw = reinterpret_cast<const uint4*>(src)[idx];
        const int p = (idx * 8) / N, n = (idx * 8) % N;
        float* d = Ss + p * a.NP + n;
        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
          d[2 * e] = f.x;
          d[2 * e + 1] = f.y;
        }
      }
    } else {
      for (int idx = tid; idx < P * N; idx += SCAN_THREADS)
        Ss[(idx / N) * a.NP + idx % N] = __half2float(src[idx]);
    }
  }
  __syncthreads();
  // ---- W[t][s] = exp(c_t - c_s) dt_s (C_t . B_s) for s <= t
  for (int idx = tid; idx < k * k; idx += SCAN_THREADS) {
    const int t = idx / k, s = idx % k;
    float w = 0.f;
    if (s <= t) {
      float dot = 0.f;
      for (int n = 0; n < N; ++n) dot += Cs[t * N + n] * Bs[s * N + n];
      w = expf(cum[t] - cum[s]) * dts[s] * dot;
    }
    Wm[t * KMAX + s] = w;
  }
  __syncthreads();
  // ---- outputs: thread owns head channel p for all k positions
  const float Dh = a.Dskip[h];
  for (int p = tid; p < P; p += SCAN_THREADS) {
    float acc[KMAX];
#pragma unroll
    for (int t = 0; t < KMAX; ++t) acc[t] = 0.f;
    if (a.s_init != nullptr) {
      const float* srow = Ss + p * a.NP;
      for (int n = 0; n < N; ++n) {
        const float sv = srow[n];
#pragma unroll
        for (int t = 0; t < KMAX; ++t)
          if (t < k) acc[t] += Cs[t * N + n] * sv;
      }
    }
#pragma unroll
    for (int t = 0; t < KMAX; ++t) {
      if (t < k) {
        float y = dec[t] * acc[t] + Dh * xs[t * P + p];
        for (int s = 0; s <= t; ++s) y += Wm[t * KMAX + s] * xs[s * P + p];
        const size_t row = row0 + t;
        const float z = a.zxbcdt[a.in_row(b, t) * a.ld_in + h * P + p];
        a.y[row * a.Di + h * P + p] = y * silu_f(z);
      }
    }
  }
}

// The compiler's own choice: 128 registers, many loads of a block in flight, four blocks to an SM.
__global__ void __launch_bounds__(SCAN_THREADS)
mamba_scan_kernel(ScanArgs a) { scan_general(a); }

// 96 registers, five blocks to an SM: 1.1 to 1.5 times slower over the same number of waves, but 593 to 740 blocks are one wave
// instead of two.  Us, the kernel above / this one, 608 blocks of 8 positions: P = 64, N = 20 30.7 / 24.6, P = 24, N = 64 55.3 / 42.6,
// P = 128, N = 24 36.9 / 32.8; 736 of 12, P = 64, N = 20 38.8 / 28.2; 1184 blocks of 8, P = 64, N = 20 38.9 / 47.1; 4480 of 4 90.1 / 103.
__global__ void __launch_bounds__(SCAN_THREADS, 5)
mamba_scan_five_kernel(ScanArgs a) { scan_general(a); }

// ---------------------------------------------------------------------------------------------------
// Small states (N <= 16: the paper's own drafter has N = 4).  The state of a channel fits in registers, so a thread owns one
// (request, head, channel) and walks the block positions with the plain recurrence S <- a_t S + dt_t x_t B_t, y_t = S C_t + D x_t.
// A block is the channels of up to four heads of one B/C group: the group's B and C rows (conv + SiLU) and the heads' dt and decay
// are computed once per block into shared memory while the threads' own inputs (x and z of eight positions) are in flight.
// The operands are a few MB, so latency is what counts: the general kernel above takes 33 us at the paper's shape
// (32 requests, 48 heads, 8 positions), this one 5.  (Event times less the 6 us an empty pair of events reads: 39.4 -> 10.8.)
// NORM: the gated RMSNorm over all Di channels behind the scan happens here too, without a launch of its own and without the fp32 rows
// in between: a request's blocks are one cluster (eight at most) and add up their rows' sums of squares through distributed
// shared memory, in a fixed order.  Together with the dt expansion (dt_pre) this takes three launches out of a step of the test-sized
// drafter and one per layer out of the paper's: 69.1 -> 67.4 and 1507 -> 1495 us per step; before the wait for the kernels in front
// the block already reads what the layer's weights give.
template <int NMAX, bool NORM>
__global__ void __launch_bounds__(512)
scan_small_state_kernel(ScanArgs a, int hb, ScanNorm nm) {
  if (!a.w_stable) { pdl_wait(); pdl_trigger(); }
  extern __shared__ __align__(16) float sm[];
  const int k = a.k, P = a.P, N = a.N, tid = threadIdx.x;
  const int h0 = blockIdx.x * hb, b = blockIdx.y, g = h0 / (a.H / a.G);
  float* Bs = sm;                    // [k][NMAX], zero past N
  float* Cs = Bs + k * NMAX;         // [k][NMAX]
  float* dts = Cs + k * NMAX;        // [k][hb]
  float* dec = dts + k * hb;         // [k][hb]
  float* part = dec + k * hb;        // NORM: [k] this block's sums of squares, then ys
  float* ys = part + k;              // NORM: [k][hb * P] the gated outputs
  const size_t row0 = size_t(b) * k;
  const int hl = tid / P, p = tid % P, h = h0 + hl;
  const bool act = hl < hb;
  constexpr int CH = 8;              // positions whose inputs are in flight together
  const int ch = act ? h * P + p : 0;
  // ---- what the layer's weights give, before the kernels in front have finished: the taps of the thread's own channel and of the B or C
  // channel it convolves below (always the same one: the block is a multiple of 2 NMAX wide)
  const int is_c = tid % (2 * NMAX) / NMAX, nb_c = tid % NMAX;
  const int cb = a.Di + is_c * a.G * N + g * N + (nb_c < N ? nb_c : 0);    // channel inside xBC
  float w[4], wb[4];                 // right-aligned taps
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const bool tap = j >= 4 - a.d_conv;
    w[j] = tap ? a.conv_w[ch * a.d_conv + j - (4 - a.d_conv)] : 0.f;
    wb[j] = tap ? a.conv_w[cb * a.d_conv + j - (4 - a.d_conv)] : 0.f;
  }
  const float bias = a.conv_b[ch], bias_b = a.conv_b[cb];
  const float gain = NORM ? nm.w[ch] : 0.f;
  const float Dh = a.Dskip[act ? h : h0];
  const float dtb = a.dt_bias[h0 + tid % hb], Ah = -expf(a.A_log[h0 + tid % hb]);   // (of the first dt the thread computes)
  if (a.w_stable) { pdl_wait(); pdl_trigger(); }
  // (plain loads from here on: the read-only form __ldg may be moved up past the wait, and did)
  float xr[CH], zr[CH], S[NMAX];
  auto fetch = [&](int t0) {
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const bool ok = act && t0 + i < k;
      const float* row = a.zxbcdt + a.in_row(b, ok ? t0 + i : 0) * a.ld_in;
      xr[i] = ok ? row[a.Di + ch] : 0.f;
      zr[i] = ok ? row[ch] : 0.f;
    }
  };
  fetch(0);
  {
    const __half* s0 = a.s_init + ((size_t(b) * a.H + (act ? h : h0)) * P + p) * N;
    const bool have = act && a.s_init != nullptr;
    if (N == NMAX && (reinterpret_cast<uintptr_t>(a.s_init) & 7) == 0) {   // whole rows of 8 or 32 bytes
#pragma unroll
      for (int n = 0; n < NMAX; n += 4) {
        const uint2 v = have ? *reinterpret_cast<const uint2*>(s0 + n) : make_uint2(0, 0);
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&v.x)), hi = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
        S[n] = lo.x; S[n + 1] = lo.y; S[n + 2] = hi.x; S[n + 3] = hi.y;
      }
    } else {
#pragma unroll
      for (int n = 0; n < NMAX; ++n) S[n] = have && n < N ? __half2float(s0[n]) : 0.f;
    }
  }
  for (int idx = tid; idx < k * 2 * NMAX; idx += blockDim.x) {
    const int i = idx / (2 * NMAX);
    float x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = i - 3 + j >= 0 ? a.zxbcdt[a.in_row(b, i - 3 + j) * a.ld_in + a.Di + cb] : 0.f;
    const float v = silu_f(bias_b + wb[0] * x[0] + wb[1] * x[1] + wb[2] * x[2] + wb[3] * x[3]);
    (is_c ? Cs : Bs)[i * NMAX + nb_c] = nb_c < N ? v : 0.f;
  }
  for (int idx = tid; idx < k * hb; idx += blockDim.x) {
    const int i = idx / hb, hh = h0 + idx % hb;
    const bool first = idx == tid;
    const float dt = softplus_f(a.dt_pre(b, i, hh) + (first ? dtb : a.dt_bias[hh]));
    dts[idx] = dt;
    dec[idx] = expf(dt * (first ? Ah : -expf(a.A_log[hh])));
  }
  __syncthreads();
  if (!NORM && !act) return;
  float c1 = 0.f, c2 = 0.f, c3 = 0.f;                              // the three rows before this one (zero left context)
  for (int t0 = 0; act && t0 < k; t0 += CH) {
    if (t0 > 0) fetch(t0);
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int t = t0 + i;
      if (t >= k) break;
      const float x = silu_f(bias + w[0] * c3 + w[1] * c2 + w[2] * c1 + w[3] * xr[i]);
      c3 = c2; c2 = c1; c1 = xr[i];
      const float at = dec[t * hb + hl], dx = dts[t * hb + hl] * x;
      float y[4] = {Dh * x, 0.f, 0.f, 0.f};                        // (four sums: one would be a chain of N products)
#pragma unroll
      for (int n = 0; n < NMAX; n += 4) {
        const float4 bv = *reinterpret_cast<const float4*>(Bs + t * NMAX + n), cv = *reinterpret_cast<const float4*>(Cs + t * NMAX + n);
        S[n] = at * S[n] + dx * bv.x;             y[0] += S[n] * cv.x;
        S[n + 1] = at * S[n + 1] + dx * bv.y;     y[1] += S[n + 1] * cv.y;
        S[n + 2] = at * S[n + 2] + dx * bv.z;     y[2] += S[n + 2] * cv.z;
        S[n + 3] = at * S[n + 3] + dx * bv.w;     y[3] += S[n + 3] * cv.w;
      }
      const float out = ((y[0] + y[1]) + (y[2] + y[3])) * silu_f(zr[i]);
      if (NORM) ys[t * hb * P + tid] = out;
      else a.y[(row0 + t) * a.Di + ch] = out;
    }
  }
  if constexpr (NORM) {
    __syncthreads();
    const int lane = tid & 31, nb = int(gridDim.x), n = hb * P;
    for (int t = tid >> 5; t < k; t += blockDim.x >> 5) {
      float ss = 0.f;
      for (int d = lane; d < n; d += 32) ss += ys[t * n + d] * ys[t * n + d];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      if (lane == 0) part[t] = ss;
    }
    if (nb > 1) cluster_sync_all(); else __syncthreads();
    float* inv = dec;                                              // [k]; the decays are no longer needed
    // eight lanes per row, one per block of the cluster
    for (int idx = tid; idx < (k * 8 + 31) / 32 * 32; idx += blockDim.x) {
      const int t = min(idx >> 3, k - 1), r = idx & 7;
      float v = r >= nb ? 0.f : nb > 1 ? ld_cluster_f32(mapa_rank(smem_u32(part + t), r)) : part[t];
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (r == 0) inv[t] = rsqrtf(v / float(a.Di) + nm.eps);
    }
    if (nb > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // this block has read the others' sums
    __syncthreads();
    if (act)
      for (int t = 0; t < k; ++t) store_act16(nm.u + (row0 + t) * a.Di, ch, ys[t * n + tid] * inv[t] * gain, nm.bf16_out != 0, nm.status);
    if (nb > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // no block leaves while another reads its sums
  }
}

// ---------------------------------------------------------------------------------------------------
// Fast path for the serving shapes (P = 64, N = 128 here; any N % 32 == 0, P % 8 == 0 instantiation):
// one warp per head, HPC heads of one B/C group per CTA.  The state term  Y[t, p] = sum_n C[t, n] S[p, n]
// is a [k x N] x [N x P] contraction per head and runs on mma.sync m16n8k16 (fp16 in, fp32 out):
//   * S_init goes from HBM straight into the B fragments: each lane loads 16 contiguous bytes
//     S[p = 8j + lane/4][32 kp + 8 (lane%4) .. +7], which feed TWO k-steps; the contraction index is
//     permuted accordingly (a sum does not care), and the A fragments of C use the same permutation;
//   * no shared-memory staging of the state, every byte of S_init is read exactly once.
// The conv + SiLU of the group's B and C is computed once per CTA and shared by its heads; the k x k
// intra-block term, the decay prefix sums (warp shuffle scan), the D skip and the SiLU(z) gate stay fp32.
template <int P, int N, int MT>
__global__ void __launch_bounds__(128)
mamba_scan_mma_kernel(ScanArgs a) {
  pdl_wait();
  pdl_trigger();
  constexpr int HPC = 4;                 // heads (= warps) per CTA
  constexpr int NT = P / 8;              // n-tiles of the MMA (head channels)
  constexpr int KP = N / 32;             // k-step pairs
  constexpr int ROWS = MT * 16;          // padded block positions
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int h0 = blockIdx.x * HPC, b = blockIdx.y;
  const int hpg = a.H / a.G;
  const int g = h0 / hpg;
  const int k = a.k;
  float* Bs = sm;                                    // [ROWS][N+1]
  float* Cs = Bs + ROWS * (N + 1);                   // [ROWS][N+1]
  float* CB = Cs + ROWS * (N + 1);                   // [ROWS][ROWS+1]   C_t . B_s
  float* xs = CB + ROWS * (ROWS + 1);                // [ROWS][HPC*P]
  float* Wm = xs + ROWS * HPC * P;                   // [HPC][ROWS][ROWS+1]
  float* dts = Wm + HPC * ROWS * (ROWS + 1);         // [HPC][ROWS]
  float* cum = dts + HPC * ROWS;                     // [HPC][ROWS]
  __half* C16 = reinterpret_cast<__half*>(cum + HPC * ROWS);   // [ROWS][N] fp16 head of C (rows >= k are zero)
  __half* C16lo = C16 + ROWS * N;                              // [ROWS][N] fp16 of the remainder C - head
  const size_t row0 = size_t(b) * k;

  // ---- phase 1: causal conv + SiLU for x of the CTA's heads and B, C of their group
  constexpr int NCH = HPC * P + 2 * N;
  for (int idx = tid; idx < ROWS * NCH; idx += 128) {
    const int i = idx / NCH, cc = idx % NCH;
    float v = 0.f;
    if (i < k) {
      int ch;
      if (cc < HPC * P) ch = h0 * P + cc;
      else if (cc < HPC * P + N) ch = a.Di + g * N + (cc - HPC * P);
      else ch = a.Di + a.G * N + g * N + (cc - HPC * P - N);
      float acc = a.conv_b[ch];
      for (int j = 0; j < a.d_conv; ++j) {
        const int src = i - (a.d_conv - 1) + j;
        if (src >= 0) acc += a.conv_w[ch * a.d_conv + j] * a.zxbcdt[a.in_row(b, src) * a.ld_in + a.Di + ch];
      }
      v = silu_f(acc);
    }
    if (cc < HPC * P) xs[i * HPC * P + cc] = v;
    else if (cc < HPC * P + N) Bs[i * (N + 1) + (cc - HPC * P)] = v;
    else {
      // C = hi + lo with both parts fp16: the tensor-core contraction then carries ~22 bits of C
      const __half hi = __float2half_rn(v);
      Cs[i * (N + 1) + (cc - HPC * P - N)] = v;
      C16[i * N + (cc - HPC * P - N)] = hi;
      C16lo[i * N + (cc - HPC * P - N)] = __float2half_rn(v - __half2float(hi));
    }
  }
  // ---- per head (warp): dt, inclusive prefix sum of dt * A over the block positions
  const int h = h0 + warp;
  {
    float dt = 0.f, dA = 0.f;
    if (lane < k) {
      const float raw = a.dt_pre(b, lane, h);
      dt = softplus_f(raw + a.dt_bias[h]);
      dA = dt * (-expf(a.A_log[h]));
    }
    float c = dA;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float up = __shfl_up_sync(0xffffffffu, c, off);
      if (lane >= off) c += up;
    }
    if (lane < ROWS) { dts[warp * ROWS + lane] = dt; cum[warp * ROWS + lane] = c; }
  }
  __syncthreads();
  // ---- phase 2: CB[t][s] = C_t . B_s (shared by the CTA's heads), s <= t
  for (int idx = tid; idx < ROWS * ROWS; idx += 128) {
    const int t = idx / ROWS, s2 = idx % ROWS;
    float dot = 0.f;
    if (s2 <= t && t < k) {
      const float* cr = Cs + t * (N + 1);
      const float* br = Bs + s2 * (N + 1);
#pragma unroll 8
      for (int n = 0; n < N; ++n) dot += cr[n] * br[n];
    }
    CB[t * (ROWS + 1) + s2] = dot;
  }
  __syncthreads();
  // ---- per head: W[t][s] = exp(c_t - c_s) dt_s CB[t][s]
  float* Wh = Wm + warp * ROWS * (ROWS + 1);
  for (int idx = lane; idx < ROWS * ROWS; idx += 32) {
    const int t = idx / ROWS, s2 = idx % ROWS;
    float w = 0.f;
    if (s2 <= t && t < k) w = expf(cum[warp * ROWS + t] - cum[warp * ROWS + s2]) * dts[warp * ROWS + s2] * CB[t * (ROWS + 1) + s2];
    Wh[t * (ROWS + 1) + s2] = w;
  }
  __syncwarp();

  // ---- phase 3: state term on the tensor cores, S_init read once from global into the B fragments
  const int gq = lane >> 2, tq = lane & 3;
  float acc[MT][NT][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int j = 0; j < NT; ++j) { acc[mt][j][0] = acc[mt][j][1] = acc[mt][j][2] = acc[mt][j][3] = 0.f; }
  if (a.s_init != nullptr) {
    const __half* S = a.s_init + (size_t(b) * a.H + h) * P * N;
#pragma unroll
    for (int kp = 0; kp < KP; ++kp) {
      uint4 sv[NT];
#pragma unroll
      for (int j = 0; j < NT; ++j)
        sv[j] = *reinterpret_cast<const uint4*>(S + size_t(j * 8 + gq) * N + kp * 32 + tq * 8);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        const uint4 c_lo = *reinterpret_cast<const uint4*>(C16 + (mt * 16 + gq) * N + kp * 32 + tq * 8);
        const uint4 c_hi = *reinterpret_cast<const uint4*>(C16 + (mt * 16 + gq + 8) * N + kp * 32 + tq * 8);
        const uint4 r_lo = *reinterpret_cast<const uint4*>(C16lo + (mt * 16 + gq) * N + kp * 32 + tq * 8);
        const uint4 r_hi = *reinterpret_cast<const uint4*>(C16lo + (mt * 16 + gq + 8) * N + kp * 32 + tq * 8);
        const uint32_t a0[4] = {c_lo.x, c_hi.x, c_lo.y, c_hi.y};     // first virtual k-step
        const uint32_t a1[4] = {c_lo.z, c_hi.z, c_lo.w, c_hi.w};     // second virtual k-step
        const uint32_t e0[4] = {r_lo.x, r_hi.x, r_lo.y, r_hi.y};     // the same two k-steps of the remainder
        const uint32_t e1[4] = {r_lo.z, r_hi.z, r_lo.w, r_hi.w};
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          mma_f16_16816(acc[mt][j], a0, sv[j].x, sv[j].y);
          mma_f16_16816(acc[mt][j], a1, sv[j].z, sv[j].w);
          mma_f16_16816(acc[mt][j], e0, sv[j].x, sv[j].y);
          mma_f16_16816(acc[mt][j], e1, sv[j].z, sv[j].w);
        }
      }
    }
  }
  // ---- epilogue: decay, intra-block term, D skip, gate
  const float Dh = a.Dskip[h];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int t = mt * 16 + gq + half * 8;
      if (t >= k) continue;
      const float dec = expf(cum[warp * ROWS + t]);
      float y[NT][2];
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const float2 xv = *reinterpret_cast<const float2*>(xs + t * HPC * P + warp * P + j * 8 + tq * 2);
        y[j][0] = dec * acc[mt][j][half * 2] + Dh * xv.x;
        y[j][1] = dec * acc[mt][j][half * 2 + 1] + Dh * xv.y;
      }
      for (int s2 = 0; s2 <= t; ++s2) {
        const float w = Wh[t * (ROWS + 1) + s2];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          const float2 xv = *reinterpret_cast<const float2*>(xs + s2 * HPC * P + warp * P + j * 8 + tq * 2);
          y[j][0] += w * xv.x;
          y[j][1] += w * xv.y;
        }
      }
      const size_t row = row0 + t;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int col = h * P + j * 8 + tq * 2;
        const float2 z = *reinterpret_cast<const float2*>(a.zxbcdt + a.in_row(b, t) * a.ld_in + col);
        *reinterpret_cast<float2*>(a.y + row * a.Di + col) = make_float2(y[j][0] * silu_f(z.x), y[j][1] * silu_f(z.y));
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------------
// Two-kernel form of the fast path (used when the caller provides scratch): the small per-position
// operands are prepared once per request and group, so the kernel that streams S_init has no
// block-wide phases in front of its loads.
//   scan_conv_kernel   causal depthwise conv + SiLU of every xBC channel (thread = 4 channels x 4 positions); for the B and C channels
//                      of a group one block does all positions, writes C as fp16 head + fp16 remainder for the tensor-core
//                      contraction and CB[b, g, t, s] = C_t . B_s for s <= t
//   mamba_scan_stream_kernel  one warp per head: everything it needs is fetched up front (cp.async for the
//                      shared operands, 32-byte loads of S_init straight into the MMA fragments)
constexpr int CONV_ROWS = 4;                                 // block positions per thread
// thread = (VEC adjacent channels, group of four block positions): the filter reads raw inputs only, so the groups are
// independent; a thread's seven (vector) loads are in flight together and it needs few registers.  VEC = 4 (16-byte
// loads and stores) when every channel offset and row stride is a multiple of four, else 1.  (One thread per channel
// walking all k rows held 72 registers, three blocks per SM, and reached 25 % of the DRAM peak with its warps waiting
// on loads; one channel and four rows per thread was bound by the instruction issue, 85 %, most of it set-up.)
// conv + SiLU of channels ch .. ch + VEC - 1 at positions i0 .. i0 + CONV_ROWS - 1 (those past the block are left as they come)
template <int VEC>
__device__ __forceinline__ void conv_rows(const ScanArgs& a, int b, int i0, int ch, float (&out)[CONV_ROWS][VEC]) {
  float w[VEC][4], bias[VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    if (VEC == 4 && a.d_conv == 4) {                         // a channel's four taps in one 16-byte load
      const float4 t = reinterpret_cast<const float4*>(a.conv_w)[ch + v];
      w[v][0] = t.x; w[v][1] = t.y; w[v][2] = t.z; w[v][3] = t.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) w[v][j] = (j >= 4 - a.d_conv) ? a.conv_w[(ch + v) * a.d_conv + j - (4 - a.d_conv)] : 0.f;   // right-aligned taps
    }
  }
  if (VEC == 4) {
    const float4 t = *reinterpret_cast<const float4*>(a.conv_b + ch);
    bias[0] = t.x; bias[VEC > 1 ? 1 : 0] = t.y; bias[VEC > 1 ? 2 : 0] = t.z; bias[VEC > 1 ? 3 : 0] = t.w;
  } else {
    bias[0] = a.conv_b[ch];
  }
  float in[CONV_ROWS + 3][VEC];                              // rows i0 - 3 .. i0 + 3 (zero left context before the block)
#pragma unroll
  for (int j = 0; j < CONV_ROWS + 3; ++j) {
    const int i = i0 - 3 + j;
    const bool ok = i >= 0 && i < a.k;
    const float* src = a.zxbcdt + a.in_row(b, ok ? i : 0) * a.ld_in + a.Di + ch;
    if (VEC == 4) {
      const float4 t = ok ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
      in[j][0] = t.x; in[j][VEC > 1 ? 1 : 0] = t.y; in[j][VEC > 1 ? 2 : 0] = t.z; in[j][VEC > 1 ? 3 : 0] = t.w;
    } else {
      in[j][0] = ok ? *src : 0.f;
    }
  }
#pragma unroll
  for (int r = 0; r < CONV_ROWS; ++r)
#pragma unroll
    for (int v = 0; v < VEC; ++v)
      out[r][v] = silu_f(bias[v] + w[v][0] * in[r][v] + w[v][1] * in[r + 1][v] + w[v][2] * in[r + 2][v] + w[v][3] * in[r + 3][v]);
}

// Blocks x < G: the B and C channels of one group and, from shared memory, their products CB (a launch of its own before that read
// both back from memory: conv 8 us + CB 4 us at 32 requests of the 8B-class shapes, k = 16).  The rows are padded by four floats
// so that the 16-byte reads of a warp's threads spread over the banks.  Blocks x >= G: 256 VEC channels of x at CONV_ROWS positions.
template <int VEC>
__global__ void __launch_bounds__(256)
scan_conv_kernel(ScanArgs a, float* __restrict__ xact, __half* __restrict__ c16, float* __restrict__ cb) {
  pdl_wait();
  pdl_trigger();
  const int k = a.k, N = a.N, n_grp = (k + CONV_ROWS - 1) / CONV_ROWS;
  const int b = blockIdx.y / n_grp, grp = blockIdx.y % n_grp;
  const size_t row0 = size_t(b) * k;
  float o[CONV_ROWS][VEC];
  if (int(blockIdx.x) >= a.G) {
    const int ch = ((blockIdx.x - a.G) * 256 + threadIdx.x) * VEC, i0 = grp * CONV_ROWS;
    if (ch >= a.Di) return;
    conv_rows<VEC>(a, b, i0, ch, o);
#pragma unroll
    for (int r = 0; r < CONV_ROWS; ++r) {
      if (i0 + r >= k) break;
      float* dst = xact + (row0 + i0 + r) * a.Di + ch;
      if (VEC == 4) *reinterpret_cast<float4*>(dst) = make_float4(o[r][0], o[r][VEC > 1 ? 1 : 0], o[r][VEC > 1 ? 2 : 0], o[r][VEC > 1 ? 3 : 0]);
      else dst[0] = o[r][0];
    }
    return;
  }
  if (grp != 0) return;
  extern __shared__ __align__(16) float cb_sm[];
  const int g = blockIdx.x, ldr = N + 4, GN = a.G * N;
  float* Bs = cb_sm;                 // [k][N + 4]
  float* Cs = cb_sm + k * ldr;       // [k][N + 4]
  for (int idx = threadIdx.x; idx < n_grp * (2 * N / VEC); idx += 256) {
    const int i0 = idx / (2 * N / VEC) * CONV_ROWS, c = idx % (2 * N / VEC) * VEC, is_c = c >= N, n = is_c ? c - N : c;
    conv_rows<VEC>(a, b, i0, a.Di + is_c * GN + g * N + n, o);
#pragma unroll
    for (int r = 0; r < CONV_ROWS; ++r) {
      const int i = i0 + r;
      if (i >= k) break;
      float* dst = (is_c ? Cs : Bs) + i * ldr + n;
#pragma unroll
      for (int v = 0; v < VEC; ++v) dst[v] = o[r][v];
      if (is_c) {
        __half hi[VEC], lo[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) { hi[v] = __float2half_rn(o[r][v]); lo[v] = __float2half_rn(o[r][v] - __half2float(hi[v])); }
        __half* d_hi = c16 + ((row0 + i) * 2 + 0) * GN + g * N + n;
        __half* d_lo = c16 + ((row0 + i) * 2 + 1) * GN + g * N + n;
        if (VEC == 4) {
          *reinterpret_cast<uint2*>(d_hi) = *reinterpret_cast<const uint2*>(hi);
          *reinterpret_cast<uint2*>(d_lo) = *reinterpret_cast<const uint2*>(lo);
        } else {
          d_hi[0] = hi[0];
          d_lo[0] = lo[0];
        }
      }
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < k * k; idx += 256) {
    const int t = idx / k, s2 = idx % k;
    float dot = 0.f;
    if (s2 <= t) {
      const float4* cr = reinterpret_cast<const float4*>(Cs + t * ldr);
      const float4* br = reinterpret_cast<const float4*>(Bs + s2 * ldr);
      for (int n4 = 0; n4 < N / 4; ++n4) {
        const float4 c = cr[n4], bb = br[n4];
        dot += c.x * bb.x; dot += c.y * bb.y; dot += c.z * bb.z; dot += c.w * bb.w;
      }
    }
    cb[((size_t(b) * a.G + g) * KMAX + t) * KMAX + s2] = dot;
  }
}

template <int P, int N, int MT>
__global__ void __launch_bounds__(128, MT == 1 ? 4 : 3)
mamba_scan_stream_kernel(ScanArgs a, const float* __restrict__ xact, const __half* __restrict__ c16,
                         const float* __restrict__ cb) {
  constexpr int HPC = 4, NT = P / 8, ROWS = MT * 16;
  constexpr int XS = P + 8;                                    // floats per x row in shared memory (padded: the fragment reads
                                                               // of rows tq and columns gq then fall on 32 different banks)
  constexpr int CS = 2 * N + 8;                                // halves per C row (hi | lo | 16 bytes of padding: the 16-byte
                                                               // fragment reads, 32 bytes apart along a row, of rows gq and gq + 1
                                                               // then fall on different banks)
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int h0 = blockIdx.x * HPC, b = blockIdx.y;
  const int hpg = a.H / a.G, g = h0 / hpg, k = a.k, GN = a.G * N;
  const int h = h0 + warp;
  const size_t row0 = size_t(b) * k;
  __half* C16 = reinterpret_cast<__half*>(sm);                 // [ROWS][CS]  (hi, lo), rows >= k zero
  float* CB = sm + ROWS * CS / 2;                                   // [ROWS][ROWS]
  float* xs = CB + ROWS * ROWS + warp * (ROWS * XS);           // per warp [ROWS][XS]
  float* Wh = CB + ROWS * ROWS + HPC * ROWS * XS + warp * ROWS * (ROWS + 1);   // per warp [ROWS][ROWS+1]

  // ---- state fragments of the first two k-step pairs: issued before anything else, and before the wait for the kernel in front: that
  // kernel (the conv) started its dependents only once everything ahead of it, the state's producer included, had finished
  const int gq = lane >> 2, tq = lane & 3;
  const __half* S = a.s_init ? a.s_init + (size_t(b) * a.H + h) * P * N : nullptr;
  // (32-byte loads: the four lanes of a row then cover a whole 128-byte line per instruction; with 16-byte loads every
  // line was touched twice, and the state's loads were a quarter of the L1's work)
  uint4 sv0[NT][2];
  if (S != nullptr) {
#pragma unroll
    for (int j = 0; j < NT; ++j) ldg_nc_32B(S + size_t(j * 8 + gq) * N + tq * 16, sv0[j][0], sv0[j][1]);
  }
  pdl_wait();
  pdl_trigger();
  // ---- shared operands (C halves, CB) and this head's x rows: cp.async, zero fill for the padding rows
  for (int idx = tid; idx < ROWS * 2 * N / 8; idx += 128) {
    const int r = idx / (2 * N / 8), rest = idx % (2 * N / 8), half = rest / (N / 8), c8 = rest % (N / 8);
    cp_async16(smem_u32(C16 + r * CS + half * N + c8 * 8), c16 + ((row0 + min(r, k - 1)) * 2 + half) * GN + g * N + c8 * 8, r < k);
  }
  for (int idx = tid; idx < ROWS * ROWS / 4; idx += 128) {
    const int r = idx / (ROWS / 4), c4 = idx % (ROWS / 4);
    cp_async16(smem_u32(CB + r * ROWS + c4 * 4), cb + ((size_t(b) * a.G + g) * KMAX + r) * KMAX + c4 * 4, true);
  }
  for (int idx = lane; idx < ROWS * P / 4; idx += 32) {
    const int r = idx / (P / 4), c4 = idx % (P / 4);
    cp_async16(smem_u32(xs + r * XS + c4 * 4), xact + (row0 + min(r, k - 1)) * a.Di + h * P + c4 * 4, r < k);
  }
  cp_async_commit();
  // ---- dt, inclusive prefix sum of dt * A over the block positions (one warp shuffle scan per head)
  float dt = 0.f, dA = 0.f;
  if (lane < k) {
    const float raw = a.dt_pre(b, lane, h);
    dt = softplus_f(raw + a.dt_bias[h]);
    dA = dt * (-expf(a.A_log[h]));
  }
  float cum = dA;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float up = __shfl_up_sync(0xffffffffu, cum, off);
    if (lane >= off) cum += up;
  }
  cp_async_wait<0>();
  __syncthreads();
  // ---- W[t][s] = exp(c_t - c_s) dt_s CB[t][s] for s <= t, plus the skip weight D on the diagonal: lane s owns
  // column s; the rows past k are zero
  const float Dh = a.Dskip[h];
  for (int t = 0; t < ROWS; ++t) {
    const float ct = __shfl_sync(0xffffffffu, cum, t & 31);
    float w = 0.f;
    if (t < k && lane <= t) w = __expf(ct - cum) * dt * CB[t * ROWS + lane];
    if (t < k && lane == t) w += Dh;
    if (lane < ROWS) Wh[t * (ROWS + 1) + lane] = w;
  }
  __syncwarp();
  // ---- state term on the tensor cores
  float acc[MT][NT][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int j = 0; j < NT; ++j) { acc[mt][j][0] = acc[mt][j][1] = acc[mt][j][2] = acc[mt][j][3] = 0.f; }
  if (S != nullptr) {
#pragma unroll
    // the contraction index is permuted (the same way for C and for the state): within a chunk of 64, lane tq's 16
    // consecutive elements serve four k-steps, four elements each
    for (int kq = 0; kq < N / 64; ++kq) {
      uint4 sv[NT][2];
      if (kq >= 1) {
#pragma unroll
        for (int j = 0; j < NT; ++j) ldg_nc_32B(S + size_t(j * 8 + gq) * N + kq * 64 + tq * 16, sv[j][0], sv[j][1]);
      } else {
#pragma unroll
        for (int j = 0; j < NT; ++j) { sv[j][0] = sv0[j][0]; sv[j][1] = sv0[j][1]; }
      }
#pragma unroll
      for (int piece = 0; piece < 2; ++piece) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          const __half* c0 = C16 + (mt * 16 + gq) * CS + kq * 64 + tq * 16 + piece * 8;
          const __half* c1 = C16 + (mt * 16 + gq + 8) * CS + kq * 64 + tq * 16 + piece * 8;
          const uint4 c_lo = *reinterpret_cast<const uint4*>(c0), c_hi = *reinterpret_cast<const uint4*>(c1);
          const uint4 r_lo = *reinterpret_cast<const uint4*>(c0 + N), r_hi = *reinterpret_cast<const uint4*>(c1 + N);
          const uint32_t a0[4] = {c_lo.x, c_hi.x, c_lo.y, c_hi.y}, a1[4] = {c_lo.z, c_hi.z, c_lo.w, c_hi.w};
          const uint32_t e0[4] = {r_lo.x, r_hi.x, r_lo.y, r_hi.y}, e1[4] = {r_lo.z, r_hi.z, r_lo.w, r_hi.w};
#pragma unroll
          for (int j = 0; j < NT; ++j) {
            mma_f16_16816(acc[mt][j], a0, sv[j][piece].x, sv[j][piece].y);
            mma_f16_16816(acc[mt][j], a1, sv[j][piece].z, sv[j][piece].w);
            mma_f16_16816(acc[mt][j], e0, sv[j][piece].x, sv[j][piece].y);
            mma_f16_16816(acc[mt][j], e1, sv[j][piece].z, sv[j][piece].w);
          }
        }
      }
    }
  }
  // ---- decay of the state term: row t of the accumulator times exp(c_t)
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const float d_lo = __expf(__shfl_sync(0xffffffffu, cum, (mt * 16 + gq) & 31));
    const float d_hi = __expf(__shfl_sync(0xffffffffu, cum, (mt * 16 + gq + 8) & 31));
#pragma unroll
    for (int j = 0; j < NT; ++j) { acc[mt][j][0] *= d_lo; acc[mt][j][1] *= d_lo; acc[mt][j][2] *= d_hi; acc[mt][j][3] *= d_hi; }
  }
  // ---- intra-block term and D skip, y_t += sum_{s <= t} W[t][s] x_s, as a [ROWS x ROWS] x [ROWS x P] product on the
  // tensor cores: tf32 operands keep fp32's range (W is a product of exponentials, dt and a 128-term dot product), and
  // each operand is split in two tf32 parts, three products per k-step, for ~21 bits.  (The scalar form read x from
  // shared memory once per (t, s) pair and thread, and the kernel ran at the L1's limit.)
#pragma unroll
  for (int ks = 0; ks < ROWS / 8; ++ks) {
    uint32_t ah[MT][4], al[MT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      const float* wr = Wh + (mt * 16 + gq) * (ROWS + 1) + ks * 8 + tq;
      split_tf32(wr[0], ah[mt][0], al[mt][0]);
      split_tf32(wr[8 * (ROWS + 1)], ah[mt][1], al[mt][1]);
      split_tf32(wr[4], ah[mt][2], al[mt][2]);
      split_tf32(wr[8 * (ROWS + 1) + 4], ah[mt][3], al[mt][3]);
    }
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      uint32_t bh[2], bl[2];
      split_tf32(xs[(ks * 8 + tq) * XS + j * 8 + gq], bh[0], bl[0]);
      split_tf32(xs[(ks * 8 + tq + 4) * XS + j * 8 + gq], bh[1], bl[1]);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        if (ks * 8 > mt * 16 + 15) continue;                   // W is lower triangular: nothing in this k-step for these rows
        mma_tf32_1688(acc[mt][j], al[mt], bh[0], bh[1]);
        mma_tf32_1688(acc[mt][j], ah[mt], bl[0], bl[1]);
        mma_tf32_1688(acc[mt][j], ah[mt], bh[0], bh[1]);
      }
    }
  }
  // ---- gate and store
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int t = mt * 16 + gq + half * 8;
      if (t >= k) continue;
      const size_t row = row0 + t;
      float2 z[NT];
#pragma unroll
      for (int j = 0; j < NT; ++j) z[j] = *reinterpret_cast<const float2*>(a.zxbcdt + a.in_row(b, t) * a.ld_in + h * P + j * 8 + tq * 2);
#pragma unroll
      for (int j = 0; j < NT; ++j)
        *reinterpret_cast<float2*>(a.y + row * a.Di + h * P + j * 8 + tq * 2) =
            make_float2(acc[mt][j][half * 2] * silu_f(z[j].x), acc[mt][j][half * 2 + 1] * silu_f(z[j].y));
    }
  }
}

template <int MT>
size_t scan_stream_smem() {
  constexpr int P = 64, N = 128, HPC = 4, ROWS = MT * 16;
  return sizeof(__half) * ROWS * (2 * N + 8) + sizeof(float) * (ROWS * ROWS + HPC * ROWS * (P + 8) + HPC * ROWS * (ROWS + 1));
}

template <int MT>
size_t scan_mma_smem() {
  constexpr int P = 64, N = 128, HPC = 4, ROWS = MT * 16;
  return sizeof(float) * (2 * ROWS * (N + 1) + ROWS * (ROWS + 1) + ROWS * HPC * P + HPC * ROWS * (ROWS + 1) + 2 * HPC * ROWS) +
         sizeof(__half) * 2 * ROWS * N;
}

}  // namespace

size_t scan_workspace_bytes(int B, int k, int Di, int N, int G) {
  const size_t M = size_t(B) * k, d_xBC = size_t(Di) + 2 * size_t(G) * N;
  return M * d_xBC * 4 + size_t(B) * G * KMAX * KMAX * 4 + M * 2 * size_t(G) * N * 2 + 256;
}

namespace {
constexpr size_t SMALL_STATE_SMEM = sizeof(float) * KMAX * (2 * (16 + 8) + 1 + 512);   // the most a call with the norm can ask for
// Heads per block of the small-state kernel: heads of one group share a block while they fit 256 threads; when the norm follows, up to
// eight heads and 512 threads, so that a request's blocks fit a cluster of eight.
int small_state_heads(const ScanCall& c) {
  const int H = c.Di / c.P, hpg = H / c.G;
  int hb = 1;
  while (hb < 4 && hpg % (2 * hb) == 0 && 2 * hb * c.P <= 256) hb *= 2;
  if (c.norm_w != nullptr)
    for (int n = hb; n <= 8 && n * c.P <= 512; ++n)
      if (hpg % n == 0 && H / n <= 8) return n;
  return hb;
}
}  // namespace

bool scan_does_norm(const ScanCall& c) {
  return c.norm_w != nullptr && c.N <= 16 && c.Di / c.P / small_state_heads(c) <= 8;
}

// An expansion of the dt columns inside the scan reads every column once per head through the L1; past a few million products the
// tensor-core GEMM is the better one although it takes two launches more.
bool scan_expands_dt(int B, int k, int H, int dt_rank) { return dt_rank <= 64 && (long long)B * k * H * dt_rank <= (1 << 22); }

cudaError_t scan_launch(const ScanCall& c, cudaStream_t stream, Tracker* trk, std::string* err) {
  if (c.k < 1 || c.k > KMAX) { if (err) *err = "scan: k out of range"; return cudaErrorInvalidValue; }
  if (c.Di % c.P) { if (err) *err = "scan: Di must be a multiple of P"; return cudaErrorInvalidValue; }
  ScanArgs a{};
  a.zxbcdt = c.zxbcdt; a.ld_in = c.ld_in; a.dt_raw = c.dt_raw; a.dt_w = (const uint16_t*)c.dt_w; a.dt_rank = c.dt_rank; a.dt_bf16 = c.dt_bf16 ? 1 : 0;
  a.s_init = (const __half*)c.s_init;
  a.conv_w = c.conv_w; a.conv_b = c.conv_b; a.dt_bias = c.dt_bias; a.A_log = c.A_log; a.Dskip = c.Dskip;
  a.y = c.y_gated; a.B = c.B; a.k = c.k; a.Di = c.Di; a.P = c.P; a.N = c.N; a.G = c.G; a.H = c.Di / c.P;
  a.d_conv = c.d_conv; a.d_xBC = c.Di + 2 * c.G * c.N;
  a.shared_rows = c.shared_rows ? 1 : 0;
  a.w_stable = c.w_stable ? 1 : 0;
  a.NP = c.N + 1;                                    // odd pitch: threads of a warp own consecutive p
  if (a.H % c.G) { if (err) *err = "scan: heads must divide into groups"; return cudaErrorInvalidValue; }
  // serving shapes: tensor-core paths.  z and y are read and written in pairs; the state comes by 32-byte loads with scratch (which is read in
  // 16-byte copies) and by 16-byte ones without.  What is off these boundaries takes the general kernel.
  const bool mma = c.P == 64 && c.N == 128 && (a.H / c.G) % 4 == 0 && c.ld_in % 2 == 0 &&
                   ((reinterpret_cast<uintptr_t>(c.zxbcdt) | reinterpret_cast<uintptr_t>(c.y_gated)) & 7) == 0 &&
                   (reinterpret_cast<uintptr_t>(c.s_init) & 15) == 0;
  if (mma && c.ws != nullptr && (reinterpret_cast<uintptr_t>(c.s_init) & 31) == 0 && (reinterpret_cast<uintptr_t>(c.ws) & 15) == 0 &&
      c.ws_bytes >= scan_workspace_bytes(c.B, c.k, c.Di, c.N, c.G)) {
    const bool two = c.k > 16;
    const size_t M = size_t(c.B) * c.k;
    float* xact = reinterpret_cast<float*>(c.ws);
    float* cbw = xact + M * a.d_xBC;
    __half* c16 = reinterpret_cast<__half*>(cbw + size_t(c.B) * c.G * KMAX * KMAX);
    trk_begin(trk, "scan_conv", 0, double(M) * (a.d_xBC + a.Di) * 4);
    const bool vec4 = a.Di % 4 == 0 && (c.G * c.N) % 4 == 0 && a.ld_in % 4 == 0 &&
                      ((reinterpret_cast<uintptr_t>(a.zxbcdt) | reinterpret_cast<uintptr_t>(c.ws) | reinterpret_cast<uintptr_t>(a.conv_w) |
                        reinterpret_cast<uintptr_t>(a.conv_b)) & 15) == 0;
    const dim3 grid_c(c.G + (a.Di / (vec4 ? 4 : 1) + 255) / 256, c.B * ((c.k + CONV_ROWS - 1) / CONV_ROWS));
    const size_t smem_c = size_t(2) * c.k * (c.N + 4) * sizeof(float);
    const cudaError_t e_conv = launch_pdl(vec4 ? scan_conv_kernel<4> : scan_conv_kernel<1>, grid_c, dim3(256), smem_c, stream, a, xact, c16, cbw);
    trk_end(trk);
    if (e_conv != cudaSuccess) return e_conv;        // (the stream kernel reads the state early on the strength of this launch in front of it)
    const size_t smem_s = two ? scan_stream_smem<2>() : scan_stream_smem<1>();
    static bool sset[2][MAX_DEVICES] = {};
    {
      const cudaError_t e = once_per_device(sset[two ? 1 : 0], [two, smem_s](int) {
        return two ? cudaFuncSetAttribute(mamba_scan_stream_kernel<64, 128, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_s))
                   : cudaFuncSetAttribute(mamba_scan_stream_kernel<64, 128, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_s));
      });
      if (e != cudaSuccess) return e;
    }
    dim3 grid_s(a.H / 4, c.B);
    trk_begin(trk, "mamba_scan", 2.0 * c.B * c.k * a.H * c.P * c.N, double(c.B) * a.H * c.P * c.N * 2);
    const cudaError_t e = launch_pdl(two ? mamba_scan_stream_kernel<64, 128, 2> : mamba_scan_stream_kernel<64, 128, 1>, grid_s, dim3(128), smem_s, stream, a,
                                     (const float*)xact, (const __half*)c16, (const float*)cbw);
    trk_end(trk);
    return e;
  }
  if (mma) {
    const bool two = c.k > 16;
    const size_t smem_f = two ? scan_mma_smem<2>() : scan_mma_smem<1>();
    static bool fset[2][MAX_DEVICES] = {};
    {
      const cudaError_t e = once_per_device(fset[two ? 1 : 0], [two, smem_f](int) {
        return two ? cudaFuncSetAttribute(mamba_scan_mma_kernel<64, 128, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_f))
                   : cudaFuncSetAttribute(mamba_scan_mma_kernel<64, 128, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_f));
      });
      if (e != cudaSuccess) return e;
    }
    dim3 grid_f(a.H / 4, c.B);
    trk_begin(trk, "mamba_scan", 2.0 * c.B * c.k * a.H * c.P * c.N, double(c.B) * a.H * c.P * c.N * 2);
    const cudaError_t e = launch_pdl(two ? mamba_scan_mma_kernel<64, 128, 2> : mamba_scan_mma_kernel<64, 128, 1>, grid_f, dim3(128), smem_f, stream, a);
    trk_end(trk);
    return e;
  }
  if (c.N <= 16) {
    const int hb = small_state_heads(c), threads = (hb * c.P + 31) / 32 * 32, nmax = c.N <= 4 ? 4 : 16;
    const bool norm = scan_does_norm(c);
    const size_t smem_n = sizeof(float) * (size_t(c.k) * 2 * (nmax + hb) + (norm ? size_t(c.k) * (1 + hb * c.P) : 0));
    const dim3 grid_n(a.H / hb, c.B);
    const ScanNorm nm{c.norm_w, (uint16_t*)c.u_16, c.norm_eps, c.bf16_out ? 1 : 0, c.status};
    auto kernel = nmax == 4 ? (norm ? scan_small_state_kernel<4, true> : scan_small_state_kernel<4, false>)
                            : (norm ? scan_small_state_kernel<16, true> : scan_small_state_kernel<16, false>);
    if (norm) {
      static bool nset[2][MAX_DEVICES] = {};
      const cudaError_t e = once_per_device(nset[nmax == 4 ? 0 : 1], [kernel](int) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SMALL_STATE_SMEM));
      });
      if (e != cudaSuccess) return e;
    }
    trk_begin(trk, norm ? "mamba_scan_norm" : "mamba_scan", 0, double(c.B) * a.H * c.P * c.N * 2);
    cudaError_t e = launch_pdl_cluster(kernel, grid_n, dim3(threads), dim3(norm ? grid_n.x : 1), smem_n, stream, a, hb, nm);
    trk_end(trk);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  const size_t smem = sizeof(float) * (size_t(KMAX) * c.P + 2 * size_t(KMAX) * c.N + KMAX * KMAX + 3 * KMAX +
                                       size_t(c.P) * a.NP);
  // one wave of five blocks to an SM, each with its shared memory and 1 KB of the 228 KB, where four would need two
  const size_t blocks = size_t(a.H) * c.B;
  const bool five = 5 * (smem + 1024) <= 228 * 1024 && blocks > 4 * 148 && blocks <= 5 * 148;
  if (smem > 48 * 1024) {            // (never with `five`)
    // the largest size asked for so far, per device (the attribute is a per-device property of the function)
    static size_t smem_set[MAX_DEVICES] = {};
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(device_setup_mutex());
    if (smem > smem_set[dev]) {
      cudaError_t e = cudaFuncSetAttribute(mamba_scan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
      if (e != cudaSuccess) { if (err) *err = "scan: state tile does not fit in shared memory"; return e; }
      smem_set[dev] = smem;
    }
  }
  dim3 grid(a.H, c.B);
  trk_begin(trk, "mamba_scan", 0, double(c.B) * a.H * c.P * c.N * 2);
  const cudaError_t e = launch_pdl(five ? mamba_scan_five_kernel : mamba_scan_kernel, grid, dim3(SCAN_THREADS), smem, stream, a);
  trk_end(trk);
  return e;
}

}  // namespace hspec
