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
// h_0 = h_prev: a thread owns VEC channels of one row and walks its K steps
// serially with the state in float32 registers, whatever the state dtype in
// memory (a bfloat16 state is rounded once, when it is stored). The loads of
// kStepsAhead steps are issued before the first of them is used.

struct StepsArgs {
  int64_t B, K, D;
  float c;
  const void* h_prev;  // (B, D), state dtype
  const void* x;       // (B, K, D), io dtype
  const void* gl;      // (B, K, 2D), io dtype
  const float* lambda;
  void* h_out;         // (B, D), state dtype
  void* h_seq;         // (B, K, D), io dtype, or NULL
};

constexpr int kStepsAhead = 4;

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

template <typename T, typename S, int VEC, class M>
__global__ void __launch_bounds__(256) steps_kernel(const StepsArgs a) {
  using IO = Io<T, VEC>;
  using Raw = typename IO::Raw;
  const int64_t nv = a.D / VEC;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= a.B * nv) return;
  const int64_t b = idx / nv;
  const int64_t d0 = (idx - b * nv) * VEC;
  float k[VEC], h[VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) k[v] = decay_rate(a.c, a.lambda[d0 + v]);
  load_state<S, VEC>(static_cast<const S*>(a.h_prev) + b * a.D + d0, h);
  const T* x = static_cast<const T*>(a.x) + b * a.K * a.D + d0;
  const T* gl = static_cast<const T*>(a.gl) + b * a.K * 2 * a.D + d0;
  T* hs = a.h_seq != nullptr ? static_cast<T*>(a.h_seq) + b * a.K * a.D + d0 : nullptr;
  for (int64_t j0 = 0; j0 < a.K; j0 += kStepsAhead) {
    Raw rx[kStepsAhead], rr[kStepsAhead], ri[kStepsAhead];
#pragma unroll
    for (int u = 0; u < kStepsAhead; ++u) {
      const int64_t j = j0 + u;
      if (j < a.K) {
        rx[u] = IO::load_raw(x + j * a.D);
        rr[u] = IO::load_raw(gl + j * 2 * a.D);
        ri[u] = IO::load_raw(gl + j * 2 * a.D + a.D);
      }
    }
#pragma unroll
    for (int u = 0; u < kStepsAhead; ++u) {
      const int64_t j = j0 + u;
      if (j < a.K) {
        float xv[VEC], rv[VEC], iv[VEC];
        IO::unpack(rx[u], xv);
        IO::unpack(rr[u], rv);
        IO::unpack(ri[u], iv);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          const float r = M::sigmoid(rv[v]);
          const float i = M::sigmoid(iv[v]);
          const float e = M::expm1_any(k[v] * r);
          h[v] = fmaf(1.0f + e, h[v], M::sqrt(-e * (2.0f + e)) * i * xv[v]);
        }
        if (hs != nullptr) IO::store(hs + j * a.D, h);
      }
    }
  }
  store_state<S, VEC>(static_cast<S*>(a.h_out) + b * a.D + d0, h);
}

// ------------------------------------------------------------ bounded-wait test

__global__ void selftest_wait_kernel(const uint32_t* flag, uint32_t* err, uint64_t timeout_ns) {
  (void)wait_word(flag, err, timeout_ns);
}

}  // namespace blr
