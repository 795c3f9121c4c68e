// Recurrent-step kernels (one step, K steps) and the bounded-wait self-test,
// with what the scan kernels share. The path is elementwise and memory-bound:
// no tensor cores; 16-byte accesses along the channels, the gate arithmetic
// fused into the loads, float32 state.
#pragma once

#include <cuda.h>
#include <limits.h>

#include "blr_device.cuh"

namespace blr {

constexpr unsigned kFull = 0xffffffffu;

// The first step of row b's sequence: 0, or L - lengths[b] (lengths clamped to
// [0, L]) when the rows carry their own lengths; the steps before it are
// padding (Sec. 3.3's left padding), never read and never written.
__device__ __forceinline__ int64_t row_start(const int32_t* lengths, int64_t b, int64_t L) {
  if (lengths == nullptr) return 0;
  int64_t n = lengths[b];
  n = n < 0 ? 0 : (n > L ? L : n);
  return L - n;
}

struct StepArgs {
  int64_t B, D;
  float c;
  int64_t n_vgroups;  // blocks along the channel vectors
  const float* h_prev;
  const void* x;
  const void* gl;
  const float* lambda;
  float* h_t;
};

// ------------------------------------------------------------ recurrent step
//
// h_t = alpha h_prev + beta x for B rows of D channels. A persistent grid: a
// block covers blockDim.x channel vectors and computes k = -c softplus(Lambda)
// for them once; each thread then walks rows ROWS at a time, with a stride of
// the grid's row threads, loading the next rows' inputs before the current
// rows' arithmetic so that every thread keeps loads in flight.

constexpr int kStepBlocksPerSm = 3;

template <typename T, int VEC, class M, int ROWS>
__global__ void __launch_bounds__(256, kStepBlocksPerSm) step_kernel(const StepArgs a) {
  using IO = Io<T, VEC>;
  __shared__ float s_k[64 * 8];
  pdl_wait();
  pdl_release();
  const int64_t vg = blockIdx.x % a.n_vgroups;
  const int64_t rg = blockIdx.x / a.n_vgroups;
  const int64_t n_rg = gridDim.x / a.n_vgroups;  // the grid launches whole channel groups
  const int64_t dblock = vg * blockDim.x * VEC;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  for (int j = tid; j < (int)blockDim.x * VEC; j += blockDim.x * blockDim.y)
    if (dblock + j < a.D) s_k[j] = decay_rate(a.c, a.lambda[dblock + j]);
  __syncthreads();
  const int64_t d0 = dblock + threadIdx.x * VEC;
  if (d0 >= a.D) return;
  float k[VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) k[v] = s_k[threadIdx.x * VEC + v];
  const T* x = static_cast<const T*>(a.x);
  const T* gl = static_cast<const T*>(a.gl);
  const int64_t rstride = n_rg * blockDim.y * ROWS;  // rows the grid takes per step of the walk
  float hp[ROWS][VEC], xv[ROWS][VEC], rv[ROWS][VEC], iv[ROWS][VEC];
  auto load = [&](int64_t r0) {
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int64_t bb = r0 + r;
      if (bb < a.B) {
        load_f32<VEC>(a.h_prev + bb * a.D + d0, hp[r]);
        IO::unpack(IO::load_raw(x + bb * a.D + d0), xv[r]);
        IO::unpack(IO::load_raw(gl + bb * 2 * a.D + d0), rv[r]);
        IO::unpack(IO::load_raw(gl + bb * 2 * a.D + a.D + d0), iv[r]);
      }
    }
  };
  int64_t r0 = (rg * blockDim.y + threadIdx.y) * ROWS;
  if (r0 < a.B) load(r0);
  for (; r0 < a.B; r0 += rstride) {
    float ch[ROWS][VEC], cx[ROWS][VEC], cr[ROWS][VEC], ci[ROWS][VEC];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        ch[r][v] = hp[r][v];
        cx[r][v] = xv[r][v];
        cr[r][v] = rv[r][v];
        ci[r][v] = iv[r][v];
      }
    }
    if (r0 + rstride < a.B) load(r0 + rstride);  // in flight during this rows' arithmetic
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int64_t bb = r0 + r;
      if (bb < a.B) {
        float out[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          const float rr = M::sigmoid(cr[r][v]);
          const float i = M::sigmoid(ci[r][v]);
          const float e = M::expm1_any(k[v] * rr);
          out[v] = fmaf(1.0f + e, ch[r][v], M::sqrt(-e * (2.0f + e)) * i * cx[r][v]);
        }
#pragma unroll
        for (int j = 0; j < VEC; j += 4)
          __stcs(reinterpret_cast<float4*>(a.h_t + bb * a.D + d0 + j),
                 make_float4(out[j], out[j + 1], out[j + 2], out[j + 3]));
      }
    }
  }
}

// ------------------------------------------------------- K recurrent steps
//
// h_j = alpha_j h_{j-1} + beta_j x_j for j = 1..K and every (row, channel), from
// h_0 = h_prev: a thread owns VEC channels of one row at a time and walks its K
// steps serially with the state in float32 registers, whatever the state dtype
// in memory (a bfloat16 state is rounded once, when it is stored).
//
// A persistent grid (as the single step's): a thread goes on to its next row
// without a gap. Its inputs come through steps_ahead register sets, each
// refilled as soon as its step is done, across the ends of rows, so that loads
// are always in flight; the next row's state is requested a row ahead. The
// arithmetic runs on pairs of channels, and k is computed once a block.
// 65536 x 8 x 64 bfloat16 with all states written: 47.6 us (0.88 of the
// measured copy rate); one row a thread, its loads in batches of four steps and
// the arithmetic unpaired took 55.7.
// float32, whose loads are half as many values each, wants more threads and fewer
// sets: 3 blocks an SM and 2 sets against 2 and 4, 65536 x 2 x 64 20.2 against 24.3
// us, x 4 44.3 / 48.6. From kStepsRowK steps on it runs steps_row_kernel.

struct StepsArgs {
  int64_t B, K, D;
  float c;
  int64_t n_vgroups;   // blocks along the channel vectors
  const void* h_prev;  // (B, D), state dtype
  const void* x;       // (B, K, D), io dtype
  const void* gl;      // (B, K, 2D), io dtype
  const float* lambda;
  void* h_out;         // (B, D), state dtype
  void* h_seq;         // (B, K, D), io dtype, or NULL
};

template <typename T>
__host__ __device__ constexpr int steps_ahead() { return sizeof(T) == 4 ? 2 : 4; }
template <typename T>
__host__ __device__ constexpr int steps_blocks_per_sm() { return sizeof(T) == 4 ? 3 : 2; }

// One step of a pair of channels from its raw inputs (a bfloat16 word, its logits
// halved on the packed pair, or two floats): h <- alpha h + sqrt(1 - alpha^2) i x.
// kp: k/2 of the channels for bfloat16, k for float32.
template <bool POLY>
__device__ __forceinline__ void step_pair(uint32_t x, uint32_t r, uint32_t i, float2 kp, float2& h) {
  const float2 e = expm1_neg2<POLY>(__ffma2_rn(kp, tanh2(bf2_scaled(r, kBf2Half)), kp));
  const float2 m2 = __fmul2_rn(e, __fadd2_rn(e, f2(2.0f)));  // -(1 - alpha^2)
  // i and x apart ((x/2) tanh(iota/2) + x/2 is nan at an infinite x)
  const float2 si = __ffma2_rn(f2(0.5f), tanh2(bf2_scaled(i, kBf2Half)), f2(0.5f));
  const float2 u = __fmul2_rn(make_float2(sqrt_approx(-m2.x), sqrt_approx(-m2.y)), __fmul2_rn(si, bf2_unpack(x)));
  h = __ffma2_rn(__fadd2_rn(f2(1.0f), e), h, u);
}
template <bool POLY>
__device__ __forceinline__ void step_pair(float2 x, float2 r, float2 i, float2 kp, float2& h) {
  const float2 e = expm1_neg2_precise<POLY>(__fmul2_rn(kp, sigmoid2(r)));
  const float2 m2 = __fmul2_rn(e, __fadd2_rn(e, f2(2.0f)));
  const float2 u = __fmul2_rn(make_float2(sqrt_approx(-m2.x), sqrt_approx(-m2.y)),
                              __fmul2_rn(sigmoid2(i), x));
  h = __ffma2_rn(__fadd2_rn(f2(1.0f), e), h, u);
}
__device__ __forceinline__ uint32_t raw_pair(const uint4& v, int p) {
  return p == 0 ? v.x : p == 1 ? v.y : p == 2 ? v.z : v.w;
}
__device__ __forceinline__ float2 raw_pair(const float4& v, int p) {
  return p == 0 ? make_float2(v.x, v.y) : make_float2(v.z, v.w);
}

template <typename S, int VEC>
__device__ __forceinline__ void load_state(const S* p, float (&h)[VEC]) {
  if constexpr (sizeof(S) == 4)
    load_f32<VEC>(reinterpret_cast<const float*>(p), h);
  else
    Io<__nv_bfloat16, VEC>::unpack(Io<__nv_bfloat16, VEC>::load_raw(p), h);
}
template <typename S, int VEC>
__device__ __forceinline__ void store_state(S* p, const float (&h)[VEC]) {
  if constexpr (sizeof(S) == 4) {
#pragma unroll
    for (int j = 0; j < VEC; j += 4)
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + j) =
          make_float4(h[j], h[j + 1], h[j + 2], h[j + 3]);
  } else {
    Io<__nv_bfloat16, VEC>::store(p, h);
  }
}

template <typename T, typename S, int VEC, bool POLY>
__device__ __forceinline__ void steps_walk(const StepsArgs& a, const float2 (&kp)[VEC / 2], int64_t d0,
                                           int64_t r, int64_t rstride) {
  using IO = Io<T, VEC>;
  using Raw = typename IO::Raw;
  constexpr int A = steps_ahead<T>(), P = VEC / 2;
  if (r >= a.B) return;
  // where the next inputs are: row lr, step lj
  int64_t lr = r, lj = 0;
  const T* px = static_cast<const T*>(a.x) + r * a.K * a.D + d0;
  const T* pg = static_cast<const T*>(a.gl) + r * a.K * 2 * a.D + d0;
  const int64_t row_x = (rstride * a.K - a.K + 1) * a.D;  // from a row's last step to the next row's first
  Raw rx[A], rr[A], ri[A];
  auto request = [&](int u) {
    if (lr < a.B) {
      rx[u] = IO::load_raw(px);
      rr[u] = IO::load_raw(pg);
      ri[u] = IO::load_raw(pg + a.D);
      const bool turn = ++lj == a.K;
      if (turn) {
        lj = 0;
        lr += rstride;
      }
      px += turn ? row_x : a.D;
      pg += turn ? 2 * row_x : 2 * a.D;
    }
  };
#pragma unroll
  for (int u = 0; u < A; ++u) request(u);
  const S* hp = static_cast<const S*>(a.h_prev) + d0;
  S* ho = static_cast<S*>(a.h_out) + d0;
  T* hs = a.h_seq != nullptr ? static_cast<T*>(a.h_seq) + r * a.K * a.D + d0 : nullptr;
  float hv[VEC], hn[VEC];
  load_state<S, VEC>(hp + r * a.D, hv);
  float2 h[P];
#pragma unroll
  for (int p = 0; p < P; ++p) h[p] = make_float2(hv[2 * p], hv[2 * p + 1]);
  if (r + rstride < a.B) load_state<S, VEC>(hp + (r + rstride) * a.D, hn);
  for (int64_t j = 0;;) {
#pragma unroll
    for (int u = 0; u < A; ++u) {
#pragma unroll
      for (int p = 0; p < P; ++p)
        step_pair<POLY>(raw_pair(rx[u], p), raw_pair(rr[u], p), raw_pair(ri[u], p), kp[p], h[p]);
      request(u);
#pragma unroll
      for (int p = 0; p < P; ++p) {
        hv[2 * p] = h[p].x;
        hv[2 * p + 1] = h[p].y;
      }
      const bool turn = ++j == a.K;
      if (hs != nullptr) {
        IO::store(hs, hv);
        hs += turn ? row_x : a.D;
      }
      if (turn) {
        store_state<S, VEC>(ho + r * a.D, hv);
        j = 0;
        r += rstride;
        if (r >= a.B) return;
#pragma unroll
        for (int p = 0; p < P; ++p) h[p] = make_float2(hn[2 * p], hn[2 * p + 1]);
        if (r + rstride < a.B) load_state<S, VEC>(hp + (r + rstride) * a.D, hn);
      }
    }
  }
}

template <typename T, typename S, int VEC>
__global__ void __launch_bounds__(256, steps_blocks_per_sm<T>()) steps_kernel(const StepsArgs a) {
  __shared__ float s_k[64 * 8];
  pdl_wait();
  pdl_release();
  const int64_t vg = blockIdx.x % a.n_vgroups;
  const int64_t rg = blockIdx.x / a.n_vgroups;
  const int64_t n_rg = gridDim.x / a.n_vgroups;  // the grid launches whole channel groups
  const int64_t dblock = vg * blockDim.x * VEC;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  bool poly = true;
  for (int j = tid; j < (int)blockDim.x * VEC; j += blockDim.x * blockDim.y) {
    const float k = dblock + j < a.D ? decay_rate(a.c, a.lambda[dblock + j]) : 0.0f;
    s_k[j] = k;
    poly = poly && k >= -kExpm1Series;
  }
  poly = __syncthreads_and(poly);
  const int64_t d0 = dblock + threadIdx.x * VEC;
  if (d0 >= a.D) return;
  float2 kp[VEC / 2];
  constexpr float f = sizeof(T) == 4 ? 1.0f : 0.5f;
#pragma unroll
  for (int p = 0; p < VEC / 2; ++p)
    kp[p] = make_float2(f * s_k[threadIdx.x * VEC + 2 * p], f * s_k[threadIdx.x * VEC + 2 * p + 1]);
  const int64_t r = rg * blockDim.y + threadIdx.y, rstride = n_rg * blockDim.y;
  if (poly)
    steps_walk<T, S, VEC, true>(a, kp, d0, r, rstride);
  else
    steps_walk<T, S, VEC, false>(a, kp, d0, r, rstride);
}

// float32 with kStepsRowK steps or more: one row a thread, its inputs in batches of
// kStepsRowBatch steps, whose gates are independent work. With rows this long a
// thread needs no next one, and with few rows the gates' latency binds, which the
// walk above takes step by step (us, walk / rows: 65536 x 8 x 64 85.3 / 83.0, the
// measured copy rate, x 12 126.9 / 123.6, 1000 x 50 x 64 23.1 / 18.0, 100000 x 12 x
// 16 53.9 / 52.0; but 20000 x 8 x 64 22.5 / 24.7, 65536 x 4 x 64 44.3 / 45.9, x 2
// 20.2 / 32.1).
constexpr int64_t kStepsRowK = 8;
constexpr int kStepsRowBatch = 4;

template <typename S>
__global__ void __launch_bounds__(256) steps_row_kernel(const StepsArgs a) {
  using IO = Io<float, 4>;
  using M = MathPrecise;
  constexpr int A = kStepsRowBatch;
  pdl_wait();
  pdl_release();
  const int64_t nv = a.D / 4;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= a.B * nv) return;
  const int64_t b = idx / nv, d0 = (idx - b * nv) * 4;
  float k[4], h[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) k[v] = decay_rate(a.c, a.lambda[d0 + v]);
  load_state<S, 4>(static_cast<const S*>(a.h_prev) + b * a.D + d0, h);
  const float* x = static_cast<const float*>(a.x) + b * a.K * a.D + d0;
  const float* gl = static_cast<const float*>(a.gl) + b * a.K * 2 * a.D + d0;
  float* hs = a.h_seq != nullptr ? static_cast<float*>(a.h_seq) + b * a.K * a.D + d0 : nullptr;
  for (int64_t j0 = 0; j0 < a.K; j0 += A) {
    float4 rx[A], rr[A], ri[A];
#pragma unroll
    for (int u = 0; u < A; ++u) {
      const int64_t j = j0 + u;
      if (j < a.K) {
        rx[u] = IO::load_raw(x + j * a.D);
        rr[u] = IO::load_raw(gl + j * 2 * a.D);
        ri[u] = IO::load_raw(gl + j * 2 * a.D + a.D);
      }
    }
#pragma unroll
    for (int u = 0; u < A; ++u) {
      const int64_t j = j0 + u;
      if (j < a.K) {
        float xv[4], rv[4], iv[4];
        IO::unpack(rx[u], xv);
        IO::unpack(rr[u], rv);
        IO::unpack(ri[u], iv);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const float e = M::expm1_any(k[v] * M::sigmoid(rv[v]));
          h[v] = fmaf(1.0f + e, h[v], M::sqrt(-e * (2.0f + e)) * M::sigmoid(iv[v]) * xv[v]);
        }
        if (hs != nullptr) IO::store(hs + j * a.D, h);
      }
    }
  }
  store_state<S, 4>(static_cast<S*>(a.h_out) + b * a.D + d0, h);
}

// ------------------------------------------------------------ bounded-wait test

__global__ void selftest_wait_kernel(const uint32_t* flag, uint32_t* err, uint64_t timeout_ns) {
  (void)wait_word(flag, err, timeout_ns);
}

}  // namespace blr
