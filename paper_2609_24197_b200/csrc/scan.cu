// Mamba-2 mixer core over the k block rows, started from the injected state (paper Sec. 3.3.1).
//
// One CTA per (request, head).  Because the recurrence S_i = a_i S_{i-1} + dt_i x_i B_i^T is linear,
// all k positions are evaluated in one pass without carrying the state:
//   y_t = exp(c_t) * (S_init C_t)  +  sum_{s<=t} exp(c_t - c_s) dt_s (C_t . B_s) x_s  +  D x_t,
//   c_t = sum_{r<=t} dt_r A   (inclusive prefix sum over the block positions, one warp shuffle scan).
// S_init (fp16 [P, N] per head) is read from HBM exactly once with 16-byte loads; it is the only
// large operand, so the kernel is bound by that read.  The causal depthwise conv + SiLU of x, B, C
// (zero left context), softplus(dt), the D skip and the SiLU(z) gate are fused around it.
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
    if ((N & 7) == 0) {
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
// The serving shapes with scratch, as two kernels:
//   scan_prep_kernel   per request and group: conv + SiLU of the B and C channels, C as fp16 head + fp16 remainder in the form of a tensor-core
//                      operand tile, C_t . B_s in fp32; dt and the prefix sums of dt A of the group's heads
//   scan_tc_kernel     state term of two heads at a time on tcgen05; conv of x, intra-block term, skip and gate with one thread per channel
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

// Where the prepared operands lie in the scratch (rows = block positions padded to 16 or 32).
struct ScanPrep {
  uint8_t* c;     // [B][G][head, remainder][2 halves of 64 n] tiles of [rows x 64] fp16, K-major, 128-byte swizzle
  float* cb;      // [B][G] C_t . B_s, quads of neighbouring s up to the diagonal, row after row (tri_quad); zero for s > t and for t >= k
  float* dt;      // [B][H][rows], zero past k
  float* cum;     // [B][H][rows]
};

// Quads (t; 4 s4 .. 4 s4 + 3) of a lower triangle, row after row: row t has t / 4 + 1 of them.
__host__ __device__ constexpr int tri_quad(int t, int s4) { return 2 * (t / 4) * (t / 4 + 1) + (t & 3) * (t / 4 + 1) + s4; }
__host__ __device__ constexpr int tri_quads(int rows) { return tri_quad(rows, 0); }

// Blocks x < G: B, C and their products of a group; x >= G: dt of eight warps' heads, one to four each.  (As part
// of a kernel that also activated x and wrote it back for the scan to read: 184 us at 256 requests of 32 positions, 128 heads.)  The
// rows are padded by four floats so that the 16-byte reads of a warp's threads spread over the banks.
template <int VEC, int MT>
__global__ void __launch_bounds__(256)
scan_prep_kernel(ScanArgs a, ScanPrep sp, int heads_per_warp) {
  constexpr int N = 128, LDR = N + 4, ROWS = MT * 16, HW = 4;
  extern __shared__ __align__(16) float cb_sm[];
  const int k = a.k, n_grp = (k + CONV_ROWS - 1) / CONV_ROWS, g = blockIdx.x, b = blockIdx.y, GN = a.G * N;
  if (!a.w_stable) { pdl_wait(); pdl_trigger(); }
  if (g >= a.G) {
    // a lane per position; what the weights give before the wait for the kernel in front
    const int lane = threadIdx.x & 31, h0 = ((g - a.G) * 8 + (threadIdx.x >> 5)) * heads_per_warp;
    float bias[HW], A[HW], raw[HW];
#pragma unroll
    for (int i = 0; i < HW; ++i) {
      const bool on = i < heads_per_warp && h0 + i < a.H;
      bias[i] = on ? a.dt_bias[h0 + i] : 0.f;
      A[i] = on ? -expf(a.A_log[h0 + i]) : 0.f;
    }
    if (a.w_stable) { pdl_wait(); pdl_trigger(); }
#pragma unroll
    for (int i = 0; i < HW; ++i) raw[i] = i < heads_per_warp && h0 + i < a.H && lane < k ? a.dt_pre(b, lane, h0 + i) : 0.f;
#pragma unroll
    for (int i = 0; i < HW; ++i) {
      if (i >= heads_per_warp || h0 + i >= a.H) break;         // (the same for the warp)
      const float dt = lane < k ? softplus_f(raw[i] + bias[i]) : 0.f;
      float cum = dt * A[i];
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float up = __shfl_up_sync(0xffffffffu, cum, off);
        if (lane >= off) cum += up;
      }
      if (lane < ROWS) {
        sp.dt[(size_t(b) * a.H + h0 + i) * ROWS + lane] = dt;
        sp.cum[(size_t(b) * a.H + h0 + i) * ROWS + lane] = cum;
      }
    }
    return;
  }
  if (a.w_stable) {
    const int c = threadIdx.x & (2 * N - 1), ch = a.Di + (c >= N ? GN : 0) + g * N + (c & (N - 1));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a.conv_w + size_t(ch) * a.d_conv));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a.conv_b + ch));
    pdl_wait();
    pdl_trigger();
  }
  float* Bs = cb_sm;                 // [k][LDR]
  float* Cs = cb_sm + k * LDR;       // [k][LDR]
  uint8_t* ct = sp.c + (size_t(b) * a.G + g) * (4 * ROWS * 128);
  for (int idx = threadIdx.x; idx < n_grp * (2 * N / VEC); idx += 256) {
    const int i0 = idx / (2 * N / VEC) * CONV_ROWS, c = idx % (2 * N / VEC) * VEC, is_c = c >= N, n = is_c ? c - N : c;
    float o[CONV_ROWS][VEC];
    conv_rows<VEC>(a, b, i0, a.Di + is_c * GN + g * N + n, o);
#pragma unroll
    for (int r = 0; r < CONV_ROWS; ++r) {
      const int i = i0 + r;
      if (i >= k) break;
      float* dst = (is_c ? Cs : Bs) + i * LDR + n;
#pragma unroll
      for (int v = 0; v < VEC; ++v) dst[v] = o[r][v];
      if (is_c) {
        __half hi[VEC], lo[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) { hi[v] = __float2half_rn(o[r][v]); lo[v] = __float2half_rn(o[r][v] - __half2float(hi[v])); }
        uint8_t* tile = ct + (n >> 6) * ROWS * 128 + (i >> 3) * 1024 + (i & 7) * 128 + ((((n >> 3) & 7) ^ (i & 7)) << 4);
        __half *d_hi = reinterpret_cast<__half*>(tile) + (n & 7), *d_lo = reinterpret_cast<__half*>(tile + 2 * ROWS * 128) + (n & 7);
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
  // C_t . B_s: a thread makes MT x MT neighbouring products, so that 136 of them have work either way (two by two from four rows of shared
  // memory: with one product per thread and 32 positions the reads of the rows set the kernel's pace)
  float* cbt = sp.cb + (size_t(b) * a.G + g) * tri_quads(ROWS) * 4;
  for (int idx = threadIdx.x; idx < 16 * 17 / 2; idx += 256) {
    int tb = int((sqrtf(8.f * float(idx) + 1.f) - 1.f) * 0.5f);
    if ((tb + 1) * (tb + 2) / 2 <= idx) ++tb;
    if (tb * (tb + 1) / 2 > idx) --tb;
    const int t = MT * tb, s0 = MT * (idx - tb * (tb + 1) / 2);
    float d[MT][MT];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < MT; ++j) d[i][j] = 0.f;
    if (t < k) {
      const float4 *cr[MT], *br[MT];
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        cr[i] = reinterpret_cast<const float4*>(Cs + min(t + i, k - 1) * LDR);
        br[i] = reinterpret_cast<const float4*>(Bs + min(s0 + i, k - 1) * LDR);
      }
#pragma unroll 4
      for (int n4 = 0; n4 < N / 4; ++n4) {
        float4 cv[MT], bv[MT];
#pragma unroll
        for (int i = 0; i < MT; ++i) { cv[i] = cr[i][n4]; bv[i] = br[i][n4]; }
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int j = 0; j < MT; ++j) {
            d[i][j] += cv[i].x * bv[j].x; d[i][j] += cv[i].y * bv[j].y; d[i][j] += cv[i].z * bv[j].z; d[i][j] += cv[i].w * bv[j].w;
          }
      }
    }
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      float* row = cbt + tri_quad(t + i, s0 >> 2) * 4;
#pragma unroll
      for (int j = 0; j < MT; ++j) row[(s0 & 3) + j] = t + i < k && s0 + j <= t + i ? d[i][j] : 0.f;
      if (s0 + MT > t)                                         // the places behind the diagonal's block in its quad
        for (int e = (s0 & 3) + MT; e < 4; ++e) row[e] = 0.f;
    }
  }
}

// A tile is two heads of one group of one request (128 channels); a CTA per SM walks a contiguous stretch of the tiles.
//   warp 0        producer: the tile's state rows (32 KB, two boxes [128 channels x 64 n], 128-byte swizzle) through a ring of four stages; the
//                 group's C (head and remainder, both operand tiles as the preparation left them) when the group changes
//   warp 1        state term  D[p, t] = sum_n S[p, n] C[t, n]: A = state (M = 128 channels), B = C (N = 16 or 32 positions), head and remainder into
//                 the same accumulator (~22 bits of C), one of four in tensor memory
//   warps 2..13   three groups of four warps take the tiles in turn; a thread owns a channel (= TMEM lane) with all its positions in registers:
//                 conv + SiLU of x, then  y_t = e^{c_t} D_t + sum_{s <= t} W[t][s] x_s,  W[t][s] = exp(c_t - c_s) dt_s (C_t . B_s) (+ skip on the
//                 diagonal) in fp32 from a table in shared memory that the head's two warps make together, gate, store.
// What has to move is the state, x, z and y, once each (1.34 GB at 256 requests of 32 positions and 128 heads, 205 us at the copy peak); the issue of
// the channel threads' instructions comes next (about 1 900 per warp and tile).  Before, the products were mma.sync fragments (1 600 clocks of a
// scheduler per 32 channels, and as many instructions again for the lanes' pieces of C and x), and a kernel of its own activated x and wrote it
// back.  Us of both kernels, before -> now, requests x positions, 128 heads: 1 x 16 9.6 -> 6.8, 5 x 7 9.7 -> 8.3, 16 x 1 13.7 -> 11.7, 32 x 16
// 35.0 -> 24.3, 61 x 9 52.3 -> 33.3, 256 x 32 514 -> 317; 160 heads: 128 x 16 147 -> 114, 40 x 32 116 -> 71.
constexpr int TC_BUFS = 4, TC_GROUPS = 3, TC_THREADS = 64 + TC_GROUPS * 128;
constexpr uint32_t TC_S_BYTES = 128 * 128 * 2;
constexpr int TC_MAX_STAGES = 5;
struct __align__(8) ScanTcBars {
  uint64_t s_full[TC_MAX_STAGES], s_empty[TC_MAX_STAGES], x_full[TC_MAX_STAGES], x_empty[TC_MAX_STAGES], c_full[2], c_empty[2], d_full[TC_BUFS], d_empty[TC_BUFS];
  uint32_t tmem_base;
};
// Shared memory: bars, [6 heads' tables], [2][C], [NS][state], [NX][slot].
template <int MT>
struct ScanTcSmem {
  static constexpr int ROWS = MT * 16, NS = MT == 1 ? 3 : 2, NX = MT == 1 ? 5 : 3;       // most stages of the state, of the rest
  static constexpr int C_BYTES = 4 * ROWS * 128, X_BYTES = ROWS * 512, CB_BYTES = tri_quads(ROWS) * 16, W_FLOATS = tri_quads(ROWS) * 4 + ROWS;
  // a slot: x, z, the group's table, prefix sums and dt of the two heads
  static constexpr int SLOT = 2 * X_BYTES + CB_BYTES + 4 * ROWS * 4;
  static constexpr int W_AT = 512, C_AT = (W_AT + 2 * TC_GROUPS * W_FLOATS * 4 + 1023) / 1024 * 1024, S_AT = C_AT + 2 * C_BYTES;
  static_assert(sizeof(ScanTcBars) <= W_AT, "");
  static constexpr size_t BYTES = S_AT + NS * size_t(TC_S_BYTES) + NX * size_t(SLOT) + 1024;
};
static_assert(ScanTcSmem<1>::BYTES <= 227 * 1024 && ScanTcSmem<2>::BYTES <= 227 * 1024, "shared memory of an SM");

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ float exp_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x * 1.4426950408889634f));
  return y;
}

// TMA_X: x and z come by TMA as well (rows of 16-byte multiples), else by plain loads of their channel's thread.
template <int MT, bool TMA_X>
__global__ void __launch_bounds__(TC_THREADS, 1)
scan_tc_kernel(const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmX, ScanArgs a, ScanPrep sp, int n_tiles, uint32_t* status) {
  using L = ScanTcSmem<MT>;
  constexpr int P = 64, ROWS = L::ROWS, NS = L::NS, NX = L::NX;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  ScanTcBars* bars = reinterpret_cast<ScanTcBars*>(smem);
  uint8_t *sC = smem + L::C_AT, *sS = smem + L::S_AT, *sX = sS + NS * TC_S_BYTES;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = a.k;
  const int t_begin = int((long long)n_tiles * blockIdx.x / gridDim.x), n_my = int((long long)n_tiles * (blockIdx.x + 1) / gridDim.x) - t_begin;
  const int per_group = a.H / a.G / 2, per_req = a.H / 2;      // tiles of a group and of a request
  const bool has_state = a.s_init != nullptr;
  constexpr uint32_t TMEM_COLS = TC_BUFS * ROWS;               // 64 or 128

  if (threadIdx.x == 0) {
    if (has_state) tma_prefetch_desc(&tmS);
    if (TMA_X) tma_prefetch_desc(&tmX);
    for (int i = 0; i < NS; ++i) { mbar_init(smem_u32(&bars->s_full[i]), 1); mbar_init(smem_u32(&bars->s_empty[i]), 1); }
    for (int i = 0; i < NX; ++i) { mbar_init(smem_u32(&bars->x_full[i]), 1); mbar_init(smem_u32(&bars->x_empty[i]), 4); }
    for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&bars->c_full[i]), 1); mbar_init(smem_u32(&bars->c_empty[i]), 1); }
    for (int i = 0; i < TC_BUFS; ++i) { mbar_init(smem_u32(&bars->d_full[i]), 1); mbar_init(smem_u32(&bars->d_empty[i]), 4); }
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  if (warp == 0) {
    if (elect_one()) {
      const uint64_t pol = policy_evict_first();
      bool ok = true;
      int n_c = 0;                                             // groups so far
      auto load_state = [&](int i) {
        const uint32_t dst = smem_u32(sS + (i % NS) * TC_S_BYTES), full = smem_u32(&bars->s_full[i % NS]);
        mbar_expect_tx(full, TC_S_BYTES);
        tma_load_2d(dst, &tmS, 0, (t_begin + i) * 128, full, pol);
        tma_load_2d(dst + TC_S_BYTES / 2, &tmS, 64, (t_begin + i) * 128, full, pol);
      };
      auto load_x = [&](int i) {
        const int b = (t_begin + i) / per_req, c = (t_begin + i - b * per_req) * 128;
        const uint32_t dst = smem_u32(sX + (i % NX) * L::SLOT), full = smem_u32(&bars->x_full[i % NX]);
        const int n = !TMA_X ? 0 : !a.shared_rows ? k : k > 1 ? 2 : 1;
        mbar_expect_tx(full, n * 1024 + L::CB_BYTES + 4 * ROWS * 4);
        if (!TMA_X) return;
        if (a.shared_rows) {                                   // boxes of one row: position 0, every later position
          for (int r = 0; r < n; ++r) {
            tma_load_2d(dst + r * 512, &tmX, a.Di + c, r == 0 ? b : a.B, full, pol);
            tma_load_2d(dst + L::X_BYTES + r * 512, &tmX, c, r == 0 ? b : a.B, full, pol);
          }
        } else {
          tma_load_2d(dst, &tmX, a.Di + c, b * k, full, pol);
          tma_load_2d(dst + L::X_BYTES, &tmX, c, b * k, full, pol);
        }
      };
      auto load_prep = [&](int i) {                            // what the kernel in front makes
        const int tile = t_begin + i;
        const uint32_t dst = smem_u32(sX + (i % NX) * L::SLOT) + 2 * L::X_BYTES, full = smem_u32(&bars->x_full[i % NX]);
        bulk_load(dst, sp.cb + size_t(tile / per_group) * (L::CB_BYTES / 4), L::CB_BYTES, full);
        bulk_load(dst + L::CB_BYTES, sp.cum + size_t(tile) * 2 * ROWS, 2 * ROWS * 4, full);
        bulk_load(dst + L::CB_BYTES + 2 * ROWS * 4, sp.dt + size_t(tile) * 2 * ROWS, 2 * ROWS * 4, full);
      };
      // The kernel in front (the preparation) started this one only after everything ahead of it had finished: state and in-projection are there.
      const int early_s = has_state ? min(NS, n_my) : 0, early_x = min(NX, n_my);
      for (int i = 0; i < early_s; ++i) load_state(i);
      for (int i = 0; i < early_x; ++i) load_x(i);
      pdl_wait();
      pdl_trigger();
      for (int i = 0; i < n_my && ok; ++i) {
        if (has_state) {
          const int tile = t_begin + i;
          if (i == 0 || tile % per_group == 0) {               // a group's first tile here
            const int cb = n_c & 1;
            if (n_c >= 2 && !mbar_wait(smem_u32(&bars->c_empty[cb]), ((n_c >> 1) - 1) & 1)) { ok = false; break; }
            mbar_expect_tx(smem_u32(&bars->c_full[cb]), L::C_BYTES);
            bulk_load(smem_u32(sC + cb * L::C_BYTES), sp.c + size_t(tile / per_group) * L::C_BYTES, L::C_BYTES, smem_u32(&bars->c_full[cb]));
            ++n_c;
          }
          if (i >= early_s) {
            if (!mbar_wait(smem_u32(&bars->s_empty[i % NS]), (i / NS - 1) & 1)) { ok = false; break; }
            load_state(i);
          }
        }
        if (i >= early_x) {
          if (!mbar_wait(smem_u32(&bars->x_empty[i % NX]), (i / NX - 1) & 1)) { ok = false; break; }
          load_x(i);
        }
        load_prep(i);
      }
      if (!ok) atomicExch(status, STATUS_TIMEOUT_PRODUCER);
    }
  } else if (warp == 1) {
    if (has_state && elect_one()) {
      const uint32_t idesc = umma_idesc_m128(ROWS, true);
      bool ok = true;
      int n_c = 0;
      for (int i = 0; i < n_my && ok; ++i) {
        const int tile = t_begin + i, s = i % NS, d = i % TC_BUFS;
        if (i == 0 || tile % per_group == 0) {
          ok = mbar_wait(smem_u32(&bars->c_full[n_c & 1]), (n_c >> 1) & 1);
          ++n_c;
        }
        ok = ok && mbar_wait(smem_u32(&bars->s_full[s]), (i / NS) & 1);
        if (ok && i >= TC_BUFS) ok = mbar_wait(smem_u32(&bars->d_empty[d]), (i / TC_BUFS - 1) & 1);
        if (!ok) break;
        tc_fence_after();
        const uint32_t st = smem_u32(sS + s * TC_S_BYTES), sc = smem_u32(sC + ((n_c - 1) & 1) * L::C_BYTES);
#pragma unroll
        for (int hl = 0; hl < 2; ++hl)
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            const uint64_t da = umma_desc_kmajor_sw128(st + (kk >> 2) * (TC_S_BYTES / 2)) + uint64_t((kk & 3) * 2);
            const uint64_t db = umma_desc_kmajor_sw128(sc + (hl * 2 + (kk >> 2)) * ROWS * 128) + uint64_t((kk & 3) * 2);
            umma_bf16(tmem + d * ROWS, da, db, idesc, (hl > 0 || kk > 0) ? 1u : 0u);
          }
        umma_commit(smem_u32(&bars->s_empty[s]));
        umma_commit(smem_u32(&bars->d_full[d]));
        if ((tile + 1) % per_group == 0) umma_commit(smem_u32(&bars->c_empty[(n_c - 1) & 1]));
      }
      if (!ok) atomicExch(status, STATUS_TIMEOUT_MMA);
    }
  } else {
    const int wg = (warp - 2) >> 2, q = warp & 3, pair = q >> 1;          // TMEM lane quarter; head of the tile
    float* Wt = reinterpret_cast<float*>(smem + L::W_AT) + (wg * 2 + pair) * L::W_FLOATS;     // triangle, then exp(c_t)
    float* dec = Wt + tri_quads(ROWS) * 4;
    const int bar_id = 1 + wg * 2 + pair, j64 = (q & 1) * 32 + lane;
    bool ok = true;
    // this thread's quads of the table: t and s4
    constexpr int QUADS = tri_quads(ROWS), ITS = (QUADS + 63) / 64;
    int q_t[ITS], q_s[ITS];
#pragma unroll
    for (int it = 0; it < ITS; ++it) {
      const int i = min(it * 64 + j64, QUADS - 1);
      int r = 0;
      while (2 * (r + 1) * (r + 2) <= i) ++r;                  // group of four rows with r + 1 quads each
      const int rem = i - 2 * r * (r + 1);
      q_t[it] = 4 * r + rem / (r + 1);
      q_s[it] = rem % (r + 1);
    }
    // taps, bias and skip weight of the thread's channel, a tile ahead
    float w[4], bias, Dh;
    auto load_taps = [&](int i) {
      const int tile = t_begin + i, h = (tile % per_req) * 2 + pair, ch = h * P + j64;
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = j >= 4 - a.d_conv ? a.conv_w[ch * a.d_conv + j - (4 - a.d_conv)] : 0.f;   // right-aligned
      bias = a.conv_b[ch];
      Dh = a.Dskip[h];
    };
    if (a.w_stable && wg < n_my) load_taps(wg);
    pdl_wait();
    if (!a.w_stable && wg < n_my) load_taps(wg);
    for (int i = wg; i < n_my; i += TC_GROUPS) {
      const int tile = t_begin + i, b = tile / per_req, ch = ((tile - b * per_req) * 2 + pair) * P + j64;
      // ---- raw x and gate of the channel at every position
      float x[ROWS], z[ROWS];
      const int sx = i % NX;
      const uint8_t* slot = sX + sx * L::SLOT;
      if (ok && !mbar_wait(smem_u32(&bars->x_full[sx]), (i / NX) & 1)) {
        atomicExch(status, STATUS_TIMEOUT_EPILOGUE);
        ok = false;
      }
      if constexpr (TMA_X) {
        const float* px = reinterpret_cast<const float*>(slot) + q * 32 + lane;
        if (a.shared_rows) {
          x[0] = px[0]; z[0] = px[ROWS * 128];
          const float x1 = px[128], z1 = px[ROWS * 128 + 128];
#pragma unroll
          for (int t = 1; t < ROWS; ++t) { x[t] = x1; z[t] = z1; }
        } else {
#pragma unroll
          for (int t = 0; t < ROWS; ++t) { x[t] = px[t * 128]; z[t] = px[ROWS * 128 + t * 128]; }
        }
      } else {
        const float* row = a.zxbcdt + a.in_row(b, 0) * a.ld_in + ch;
        const size_t first_step = a.shared_rows ? size_t(a.B - b) * a.ld_in : size_t(a.ld_in), step = a.shared_rows ? 0 : size_t(a.ld_in);
#pragma unroll
        for (int t = 0; t < ROWS; ++t) {
          x[t] = t < k ? ld_stream(row + a.Di) : 0.f;
          z[t] = t < k ? ld_stream(row) : 0.f;
          row += t == 0 ? first_step : step;
        }
      }
      // ---- the head's table, by its 64 threads.  (The products are zero for s > t and for t >= k; the decay only must not overflow there.)
      {
        const float* cbt = reinterpret_cast<const float*>(slot + 2 * L::X_BYTES);
        const float *cum = reinterpret_cast<const float*>(slot + 2 * L::X_BYTES + L::CB_BYTES) + pair * ROWS, *dts = cum + 2 * ROWS;
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
          if (QUADS % 64 != 0 && it == ITS - 1 && it * 64 + j64 >= QUADS) break;
          const int t = q_t[it], s4 = q_s[it], d = t - s4 * 4;
          const float4 cb = *reinterpret_cast<const float4*>(cbt + (it * 64 + j64) * 4);
          const float4 cs = *reinterpret_cast<const float4*>(cum + s4 * 4), ds = *reinterpret_cast<const float4*>(dts + s4 * 4);
          const float c = cum[t];
          float4 v;
          v.x = exp_ftz(fminf(c - cs.x, 0.f)) * ds.x * cb.x + (d == 0 ? Dh : 0.f);
          v.y = exp_ftz(fminf(c - cs.y, 0.f)) * ds.y * cb.y + (d == 1 ? Dh : 0.f);
          v.z = exp_ftz(fminf(c - cs.z, 0.f)) * ds.z * cb.z + (d == 2 ? Dh : 0.f);
          v.w = exp_ftz(fminf(c - cs.w, 0.f)) * ds.w * cb.w + (d == 3 ? Dh : 0.f);
          *reinterpret_cast<float4*>(Wt + (it * 64 + j64) * 4) = v;
        }
        if (j64 < ROWS) dec[j64] = exp_ftz(cum[j64]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->x_empty[sx]));
      asm volatile("bar.sync %0, 64;" ::"r"(bar_id) : "memory");
      // ---- conv + SiLU of x, zero left context
      {
        float c1 = 0.f, c2 = 0.f, c3 = 0.f;
#pragma unroll
        for (int t = 0; t < ROWS; ++t) {
          const float in = x[t];
          x[t] = silu_f(bias + w[0] * c3 + w[1] * c2 + w[2] * c1 + w[3] * in);
          c3 = c2; c2 = c1; c1 = in;
        }
      }
      if (i + TC_GROUPS < n_my) load_taps(i + TC_GROUPS);
      // ---- state term
      float acc[ROWS];
      if (has_state) {
        const int d = i % TC_BUFS;
        if (ok && !mbar_wait(smem_u32(&bars->d_full[d]), (i / TC_BUFS) & 1)) {
          atomicExch(status, STATUS_TIMEOUT_EPILOGUE);
          ok = false;
        }
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < ROWS; c0 += 16)
          tmem_ld16(tmem + (uint32_t(q * 32) << 16) + d * ROWS + c0, *reinterpret_cast<uint32_t(*)[16]>(acc + c0));
        tmem_ld_wait();
#pragma unroll
        for (int t = 0; t < ROWS; ++t) asm volatile("" : "+f"(acc[t]));     // (no use of the registers ahead of the wait)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->d_empty[d]));
      } else {
#pragma unroll
        for (int t = 0; t < ROWS; ++t) acc[t] = 0.f;
      }
      // ---- four positions at a time
      float* yr = a.y + size_t(b) * k * a.Di + ch;
#pragma unroll
      for (int t0 = 0; t0 < ROWS; t0 += 4) {
        if (t0 >= k) break;
        const float4 dc = *reinterpret_cast<const float4*>(dec + t0);
        float y[4] = {dc.x * acc[t0], dc.y * acc[t0 + 1], dc.z * acc[t0 + 2], dc.w * acc[t0 + 3]};
#pragma unroll
        for (int s4 = 0; s4 <= t0 / 4; ++s4)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float4 v = *reinterpret_cast<const float4*>(Wt + tri_quad(t0 + r, s4) * 4);
            const int s = s4 * 4, t = t0 + r;
            y[r] += v.x * x[s];
            if (s + 1 <= t) y[r] += v.y * x[s + 1];
            if (s + 2 <= t) y[r] += v.z * x[s + 2];
            if (s + 3 <= t) y[r] += v.w * x[s + 3];
          }
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (t0 + r < k && ok) { *yr = y[r] * silu_f(z[t0 + r]); yr += a.Di; }
      }
      asm volatile("bar.sync %0, 64;" ::"r"(bar_id) : "memory");           // the table may be written again
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// rows of a request's prepared operands: block positions padded to a tile of the tensor-core products
int unit_rows(int k) { return k > 16 ? 32 : 16; }

template <int MT>
size_t scan_mma_smem() {
  constexpr int P = 64, N = 128, HPC = 4, ROWS = MT * 16;
  return sizeof(float) * (2 * ROWS * (N + 1) + ROWS * (ROWS + 1) + ROWS * HPC * P + HPC * ROWS * (ROWS + 1) + 2 * HPC * ROWS) +
         sizeof(__half) * 2 * ROWS * N;
}

}  // namespace

size_t scan_workspace_bytes(int B, int k, int Di, int N, int G) {
  const size_t rows = size_t(unit_rows(k));
  return size_t(B) * (G * (rows * 2 * N * 2 + size_t(tri_quads(int(rows))) * 16) + size_t(Di / 64) * 2 * rows * 4) + 256;
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
  // serving shapes: tcgen05 path (16-byte copies of the state and of the scratch)
  if (c.P == 64 && c.N == 128 && (a.H / c.G) % 4 == 0 && c.ws != nullptr && c.status != nullptr &&
      ((reinterpret_cast<uintptr_t>(c.s_init) | reinterpret_cast<uintptr_t>(c.ws)) & 15) == 0 &&
      c.ws_bytes >= scan_workspace_bytes(c.B, c.k, c.Di, c.N, c.G)) {
    // (a grid of the conv that this path once had: calls past its limit stay refused)
    if ((long long)c.B * ((c.k + CONV_ROWS - 1) / CONV_ROWS) > 65535) return cudaErrorInvalidConfiguration;
    const bool two = c.k > 16;
    const int rows = unit_rows(c.k);
    ScanPrep sp{};
    sp.c = reinterpret_cast<uint8_t*>(c.ws);
    sp.cb = reinterpret_cast<float*>(sp.c + size_t(c.B) * c.G * rows * 2 * c.N * 2);
    sp.dt = sp.cb + size_t(c.B) * c.G * tri_quads(rows) * 4;
    sp.cum = sp.dt + size_t(c.B) * a.H * rows;
    const bool vec4 = a.ld_in % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.zxbcdt) | reinterpret_cast<uintptr_t>(a.conv_w) |
                                            reinterpret_cast<uintptr_t>(a.conv_b)) & 15) == 0;
    CUtensorMap tmS{}, tmX{};
    if (c.s_init != nullptr && !make_tmap_16bit_2d(&tmS, c.s_init, int64_t(c.B) * a.H * c.P, c.N, c.N, 128, true, err)) return cudaErrorInvalidValue;
    const bool tma_x = a.ld_in % 4 == 0 && (reinterpret_cast<uintptr_t>(a.zxbcdt) & 15) == 0;
    if (tma_x && !make_tmap_f32_2d(&tmX, a.zxbcdt, a.shared_rows ? c.B + 1 : int64_t(c.B) * c.k, a.ld_in, 128, a.shared_rows ? 1 : c.k, err))
      return cudaErrorInvalidValue;
    trk_begin(trk, "scan_prep", 0, double(c.B) * c.k * (2 * c.G * c.N + a.H) * 4);
    auto prep = two ? (vec4 ? scan_prep_kernel<4, 2> : scan_prep_kernel<1, 2>) : (vec4 ? scan_prep_kernel<4, 1> : scan_prep_kernel<1, 1>);
    const int hw = (long long)c.B * a.H > 148 * 32 ? 4 : 1;    // one head per warp while the blocks for them fit the chip at once
    const cudaError_t e_prep = launch_pdl(prep, dim3(c.G + (a.H + 8 * hw - 1) / (8 * hw), c.B), dim3(256), size_t(2) * c.k * (c.N + 4) * sizeof(float), stream,
                                          a, sp, hw);
    trk_end(trk);
    if (e_prep != cudaSuccess) return e_prep;        // (the next kernel reads the state early on the strength of this launch in front of it)
    const int n_tiles = c.B * (a.H / 2), ctas = n_tiles < 148 ? n_tiles : 148;
    const size_t smem_t = two ? ScanTcSmem<2>::BYTES : ScanTcSmem<1>::BYTES;
    auto kernel = two ? (tma_x ? scan_tc_kernel<2, true> : scan_tc_kernel<2, false>) : (tma_x ? scan_tc_kernel<1, true> : scan_tc_kernel<1, false>);
    static bool tset[4][MAX_DEVICES] = {};
    const cudaError_t e0 = once_per_device(tset[two * 2 + tma_x], [kernel](int) {
      return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    });
    if (e0 != cudaSuccess) return e0;
    trk_begin(trk, "mamba_scan", 2.0 * c.B * c.k * a.H * c.P * c.N, double(c.B) * a.H * c.P * c.N * 2);
    const cudaError_t e = launch_pdl(kernel, dim3(ctas), dim3(TC_THREADS), smem_t, stream, tmS, tmX, a, sp, n_tiles, c.status);
    trk_end(trk);
    return e;
  }
  if (c.P == 64 && c.N == 128 && (a.H / c.G) % 4 == 0 && c.ld_in % 2 == 0 && c.Di % 2 == 0) {
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
