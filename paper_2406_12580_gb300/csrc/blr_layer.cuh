// Kernels of the gated recurrent layer (Alg. 1) around the scan: the causal
// depthwise Conv1d and SiLU of one half of the expansion's output, and the
// float32 linear projections with their gradients.
#pragma once

#include "blr_device.cuh"

namespace blr {

// ------------------------------------------------------ convolution and SiLU
//
// in (B, L, 2C) is the expansion's output H_x | H_z. Forward: x = SiLU(conv(H_x))
// with conv_t = b + sum_k w_k in_{t-3+k} (width kConvWidth, causal: rows before
// the sequence are zero), and z = H_z as a tensor of its own, which the scan
// takes. Backward: with g_t = dx_t SiLU'(conv_t) (conv recomputed),
// d in_t = sum_k w_k g_{t+3-k}, d w_k = sum_t g_t in_{t-3+k}, d b = sum_t g_t, and
// dz goes into its half of d in.
//
// A thread owns VEC channels (16 bytes in float32, 8 in bfloat16) and walks
// kConvRows rows of one sequence with the window of inputs in registers, so every
// element is read and written once but for the halo of 3 (backward 6) rows. Memory-bound:
// 256 x 200 x 128 float32 moves 105 MB forward and 184 MB backward. As separate
// operators (transposing copies, a depthwise convolution, SiLU, and their
// gradients and the halves' concatenation) the forward took 150 us and the
// backward 330 us.

constexpr int kConvWidth = 4;
constexpr int kConvRows = 16;
constexpr int kConvThreads = 128;

struct ConvArgs {
  int64_t B, L, C;
  int64_t n_chunk;  // chunks of kConvRows rows per sequence
  const void* in;   // (B, L, 2C)
  const void* w;    // (C, kConvWidth)
  const void* b;    // (C)
  void* x;          // forward: (B, L, C) outputs; backward: their gradients dx, dz (inputs)
  void* z;
  void* din;        // backward: (B, L, 2C)
  float* part;      // backward: per block, (C, kConvWidth + 1) sums of dw | db
};

// The accurate exponential: these kernels stand in for accurate operators.
__device__ __forceinline__ float sigmoid_full(float v) { return __fdividef(1.0f, 1.0f + expf(-v)); }

template <typename T>
__device__ __forceinline__ float as_float(T v) {
  if constexpr (sizeof(T) == 4) return v;
  else return __bfloat162float(v);
}

template <typename T, int VEC>
struct ConvTaps {
  float w[kConvWidth][VEC], b[VEC];
  __device__ __forceinline__ void load(const ConvArgs& a, int64_t c0) {
    const T* wp = static_cast<const T*>(a.w) + c0 * kConvWidth;
    const T* bp = static_cast<const T*>(a.b) + c0;
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
#pragma unroll
      for (int k = 0; k < kConvWidth; ++k) w[k][v] = as_float(wp[v * kConvWidth + k]);
      b[v] = as_float(bp[v]);
    }
  }
};

template <typename T, int VEC>
__global__ void __launch_bounds__(kConvThreads, 4) conv_silu_fwd_kernel(const ConvArgs a) {
  using IO = Io<T, VEC>;
  constexpr int H = kConvWidth - 1;
  pdl_wait();
  pdl_release();
  const int64_t nv = a.C / VEC;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t unit = idx / nv, c0 = (idx - unit * nv) * VEC;
  if (unit >= a.B * a.n_chunk) return;
  const int64_t b = unit / a.n_chunk, t0 = (unit - b * a.n_chunk) * kConvRows;
  const int64_t t1 = min(t0 + kConvRows, a.L);
  ConvTaps<T, VEC> f;
  f.load(a, c0);
  const int64_t pitch = 2 * a.C;
  const T* in = static_cast<const T*>(a.in) + b * a.L * pitch + c0;
  T* x = static_cast<T*>(a.x) + b * a.L * a.C + c0;
  T* z = static_cast<T*>(a.z) + b * a.L * a.C + c0;
  float win[H][VEC];  // the inputs of steps t-3, t-2, t-1
#pragma unroll
  for (int k = 0; k < H; ++k) {
#pragma unroll
    for (int v = 0; v < VEC; ++v) win[k][v] = 0.0f;
    if (t0 - H + k >= 0) IO::unpack(IO::load_raw(in + (t0 - H + k) * pitch), win[k]);
  }
  constexpr int U = 4;  // rows in flight
  for (int64_t t = t0; t < t1; t += U) {
    typename IO::Raw rx[U], rz[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (t + u < t1) {
        rx[u] = IO::load_raw(in + (t + u) * pitch);
        rz[u] = IO::load_raw(in + (t + u) * pitch + a.C);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (t + u < t1) {
        float cur[VEC], zv[VEC], out[VEC];
        IO::unpack(rx[u], cur);
        IO::unpack(rz[u], zv);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          float s = f.b[v];
#pragma unroll
          for (int k = 0; k < H; ++k) s = fmaf(f.w[k][v], win[k][v], s);
          s = fmaf(f.w[H][v], cur[v], s);
          out[v] = s * sigmoid_full(s);
#pragma unroll
          for (int k = 0; k + 1 < H; ++k) win[k][v] = win[k + 1][v];
          win[H - 1][v] = cur[v];
        }
        IO::store(x + (t + u) * a.C, out);
        IO::store(z + (t + u) * a.C, zv);
      }
    }
  }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(kConvThreads, 3) conv_silu_bwd_kernel(const ConvArgs a) {
  using IO = Io<T, VEC>;
  constexpr int W = kConvWidth, H = W - 1;
  constexpr int NS = (W + 1) * VEC;  // a thread's sums: dw and db of its channels
  __shared__ float red[kConvThreads][VEC];
  pdl_wait();
  pdl_release();
  const int64_t nv = a.C / VEC;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t unit = idx / nv, c0 = (idx - unit * nv) * VEC;
  float sum[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) sum[i] = 0.0f;
  if (unit < a.B * a.n_chunk) {
    const int64_t b = unit / a.n_chunk, t0 = (unit - b * a.n_chunk) * kConvRows;
    const int64_t t1 = min(t0 + kConvRows, a.L);
    ConvTaps<T, VEC> f;
    f.load(a, c0);
    const int64_t pitch = 2 * a.C;
    const T* in = static_cast<const T*>(a.in) + b * a.L * pitch + c0;
    const T* dx = static_cast<const T*>(a.x) + b * a.L * a.C + c0;
    const T* dz = static_cast<const T*>(a.z) + b * a.L * a.C + c0;
    T* din = static_cast<T*>(a.din) + b * a.L * pitch + c0;
    float win[H][VEC], g[H][VEC];  // inputs of steps t-3 .. t-1, and g of them (g of steps before t0: unused)
#pragma unroll
    for (int k = 0; k < H; ++k) {
#pragma unroll
      for (int v = 0; v < VEC; ++v) win[k][v] = g[k][v] = 0.0f;
      if (t0 - H + k >= 0) IO::unpack(IO::load_raw(in + (t0 - H + k) * pitch), win[k]);
    }
    // step t gives g_t and completes d in_{t-3}; steps up to t1 + 2 (zero past
    // the sequence) complete the chunk's
    constexpr int U = 4;
    for (int64_t t = t0; t < t1 + H; t += U) {
      typename IO::Raw ri[U], rd[U], rz[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (t + u < a.L && t + u < t1 + H) {
          ri[u] = IO::load_raw(in + (t + u) * pitch);
          rd[u] = IO::load_raw(dx + (t + u) * a.C);
          if (t + u < t1) rz[u] = IO::load_raw(dz + (t + u) * a.C);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t s = t + u;
        if (s < t1 + H) {
          float cur[VEC], gc[VEC], out[VEC];
#pragma unroll
          for (int v = 0; v < VEC; ++v) cur[v] = gc[v] = 0.0f;
          if (s < a.L) {
            IO::unpack(ri[u], cur);
            IO::unpack(rd[u], gc);
          }
#pragma unroll
          for (int v = 0; v < VEC; ++v) {
            float q = f.b[v];
#pragma unroll
            for (int k = 0; k < H; ++k) q = fmaf(f.w[k][v], win[k][v], q);
            q = fmaf(f.w[H][v], cur[v], q);
            const float sg = sigmoid_full(q);
            gc[v] *= sg * fmaf(q, 1.0f - sg, 1.0f);
            if (s < t1) {
#pragma unroll
              for (int k = 0; k < H; ++k) sum[k * VEC + v] = fmaf(gc[v], win[k][v], sum[k * VEC + v]);
              sum[H * VEC + v] = fmaf(gc[v], cur[v], sum[H * VEC + v]);
              sum[W * VEC + v] += gc[v];
            }
            // d in_{s-3} = w_3 g_{s-3} + w_2 g_{s-2} + w_1 g_{s-1} + w_0 g_s
            float o = f.w[0][v] * gc[v];
#pragma unroll
            for (int k = 0; k < H; ++k) o = fmaf(f.w[H - k][v], g[k][v], o);
            out[v] = o;
#pragma unroll
            for (int k = 0; k + 1 < H; ++k) {
              win[k][v] = win[k + 1][v];
              g[k][v] = g[k + 1][v];
            }
            win[H - 1][v] = cur[v];
            g[H - 1][v] = gc[v];
          }
          if (s >= t0 + H) IO::store(din + (s - H) * pitch, out);
          if (s < t1) {
            float zv[VEC];
            IO::unpack(rz[u], zv);
            IO::store(din + s * pitch + a.C, zv);
          }
        }
      }
    }
  }
  // The block's sums per channel, in thread order: threads idx and idx + nv hold
  // the same channels. (A block need not start at channel 0: thread j's channels
  // start at ((block start + j) % nv) * VEC.)
  const int64_t first = blockIdx.x * (int64_t)blockDim.x % nv;
  float* part = a.part + blockIdx.x * a.C * (W + 1);
  for (int i = 0; i < W + 1; ++i) {
    __syncthreads();
#pragma unroll
    for (int v = 0; v < VEC; ++v) red[threadIdx.x][v] = sum[i * VEC + v];
    __syncthreads();
    for (int64_t c = threadIdx.x; c < a.C; c += blockDim.x) {
      const int64_t cv = c / VEC;
      float t = 0.0f;
      for (int64_t j = (cv - first + nv) % nv; j < blockDim.x; j += nv) t += red[j][c - cv * VEC];
      part[c * (W + 1) + i] = t;
    }
  }
}

// Sums n parts of `size` values each (32 interleaved float32 sums, then those).
// cols > 1: value i is column i % cols of row i / cols, the last column goes to
// `b`, the others to `a`.
// cols == 0: the first `split` values go to `a`, the rest to `b`.
struct SumArgs {
  const float* part;
  int64_t n, size, split;
  int cols;
  void* a;
  void* b;
};

constexpr int kSumThreads = 1024;  // 32 values a block, 32 threads each

template <typename T>
__global__ void __launch_bounds__(kSumThreads) sum_parts_kernel(const SumArgs s_) {
  const float* part = s_.part;
  const int64_t n = s_.n, size = s_.size;
  const int cols = s_.cols;
  T* a = static_cast<T*>(s_.a);
  T* b = static_cast<T*>(s_.b);
  __shared__ float red[kSumThreads / 32][33];
  pdl_wait();
  pdl_release();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t i = blockIdx.x * (int64_t)32 + tx;
  float s = 0.0f;
  if (i < size) {
#pragma unroll 4
    for (int64_t p = ty; p < n; p += kSumThreads / 32) s += part[p * size + i];
  }
  red[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && i < size) {
#pragma unroll
    for (int k = 1; k < kSumThreads / 32; ++k) s += red[k][tx];
    T* out;
    if (cols > 1) {
      const int64_t row = i / cols;
      const int col = (int)(i - row * cols);
      out = col == cols - 1 ? b + row : a + row * (cols - 1) + col;
    } else {
      out = i < s_.split ? a + i : b + (i - s_.split);
    }
    if constexpr (sizeof(T) == 4) *out = s;
    else *out = __float2bfloat16_rn(s);
  }
}

// ------------------------------------------------------- float32 projections
//
// C (M, N) = sum over k of A(m, k) B(n, k), float32 throughout (multiply-adds on
// pairs of columns, no tensor cores: the layer's float32 means float32). Blocks
// of 128 threads compute 128 x 64 tiles, 8 x 8 a thread, from double-buffered
// 16-deep slices of A and B in shared memory, k-major.
//   kNT: A (M, K), B (N, K), both k-contiguous: y = x W^T + bias
//   kNN: A (M, K) k-contiguous, B (K, N) n-contiguous: dx = dy W
//   kTN: A (K, M), B (K, N): dW = dy^T x, the long sum over rows split over
//        grid.z, with the column sums of A (the bias gradient) beside it
// The layer's projections are thin (64 to 512 columns) over many rows. At
// 51200 rows cuBLAS ran them at 7 to 40 TFLOP/s, with a separate pass for the bias
// (53 us for 256 columns) and another for its gradient (70 us). There is no split
// of kNT's and kNN's sums: few rows of wide projections are latency-bound (128 rows,
// 1024 x 512: forward 32 us against cuBLAS's 13, input gradient 61 / 17), and callers
// choose by size.

enum GemmForm { kNT, kNN, kTN };

struct GemmArgs {
  int64_t M, N, K;
  int64_t k_split;    // kTN: rows of the sum per grid.z
  const float* A;
  const float* B;
  const float* bias;  // kNT: (N) or NULL
  float* C;           // kTN: grid.z parts of M N values and the M column sums of A
  int add;            // kNN: C += instead of C =
};

constexpr int kGemmM = 128, kGemmN = 64, kGemmK = 16;

template <int FORM>
__global__ void __launch_bounds__(128, 3) gemm_f32_kernel(const GemmArgs a) {
  constexpr int BM = kGemmM, BN = kGemmN, BK = kGemmK;
  constexpr int PA = BM + 4, PB = BN + 4;  // row pitches: 16-byte aligned, transposing stores spread over banks
  __shared__ __align__(16) float sA[2][BK][PA];
  __shared__ __align__(16) float sB[2][BK][PB];
  pdl_wait();
  pdl_release();
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
  const int64_t k_lo = FORM == kTN ? blockIdx.z * a.k_split : 0;
  const int64_t k_hi = FORM == kTN ? min(k_lo + a.k_split, a.K) : a.K;

  if (FORM == kNN && a.add) {  // the values to add to, wanted at the end
    const int64_t m = m0 + tid;
    if (m < a.M) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(a.C + m * a.N + n0));
      if (n0 + 32 < a.N) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.C + m * a.N + n0 + 32));
    }
  }
  float4 ra[4], rb[2];
  const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  // Sizes are multiples of 4 (checked on the host): a vector is in or out whole.
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      ra[i] = zero;
      if constexpr (FORM == kTN) {  // 16 rows of 32 vectors
        const int64_t k = k0 + ty / 4 + 4 * i, m = m0 + 4 * (tid & 31);
        if (k < k_hi && m < a.M) ra[i] = *reinterpret_cast<const float4*>(a.A + k * a.M + m);
      } else {  // 128 rows of 4 vectors
        const int64_t m = m0 + (tid >> 2) + 32 * i, k = k0 + 4 * (tid & 3);
        if (m < a.M && k < k_hi) ra[i] = *reinterpret_cast<const float4*>(a.A + m * a.K + k);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      rb[i] = zero;
      if constexpr (FORM == kNT) {  // 64 rows of 4 vectors
        const int64_t n = n0 + (tid >> 2) + 32 * i, k = k0 + 4 * (tid & 3);
        if (n < a.N && k < k_hi) rb[i] = *reinterpret_cast<const float4*>(a.B + n * a.K + k);
      } else {  // 16 rows of 16 vectors
        const int64_t k = k0 + (tid >> 4) + 8 * i, n = n0 + 4 * (tid & 15);
        if (k < k_hi && n < a.N) rb[i] = *reinterpret_cast<const float4*>(a.B + k * a.N + n);
      }
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (FORM == kTN) {
        *reinterpret_cast<float4*>(&sA[buf][ty / 4 + 4 * i][4 * (tid & 31)]) = ra[i];
      } else {
        const int m = (tid >> 2) + 32 * i, k = 4 * (tid & 3);
        sA[buf][k][m] = ra[i].x;
        sA[buf][k + 1][m] = ra[i].y;
        sA[buf][k + 2][m] = ra[i].z;
        sA[buf][k + 3][m] = ra[i].w;
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if constexpr (FORM == kNT) {
        const int n = (tid >> 2) + 32 * i, k = 4 * (tid & 3);
        sB[buf][k][n] = rb[i].x;
        sB[buf][k + 1][n] = rb[i].y;
        sB[buf][k + 2][n] = rb[i].z;
        sB[buf][k + 3][n] = rb[i].w;
      } else {
        *reinterpret_cast<float4*>(&sB[buf][(tid >> 4) + 8 * i][4 * (tid & 15)]) = rb[i];
      }
    }
  };

  // Thread (ty, tx): rows 4 ty .. + 3 and 64 + 4 ty .. + 3, columns likewise of 32.
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
  }
  float colsum = 0.0f;  // kTN: thread tid's column of A
  const bool sums = FORM == kTN && blockIdx.y == 0;
  fetch(k_lo);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = k_lo; k0 < k_hi; k0 += BK) {
    const bool more = k0 + BK < k_hi;
    if (more) fetch(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&sA[buf][k][4 * ty]);
      const float4 a1 = *reinterpret_cast<const float4*>(&sA[buf][k][64 + 4 * ty]);
      const float4 b0 = *reinterpret_cast<const float4*>(&sB[buf][k][4 * tx]);
      const float4 b1 = *reinterpret_cast<const float4*>(&sB[buf][k][32 + 4 * tx]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                            make_float2(b1.z, b1.w)};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          acc[i][j] = __ffma2_rn(make_float2(av[i], av[i]), bv[j], acc[i][j]);
      }
    }
    if (sums) {
#pragma unroll
      for (int k = 0; k < BK; ++k) colsum += sA[buf][k][tid];
    }
    if (more) {
      stash(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
  float* C = a.C + (FORM == kTN ? (int64_t)blockIdx.z * (a.M * a.N + a.M) : 0);
  float4 bias[2] = {zero, zero};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t n = n0 + 32 * h + 4 * tx;
    if (FORM == kNT && a.bias != nullptr && n < a.N) bias[h] = *reinterpret_cast<const float4*>(a.bias + n);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t m = m0 + (i < 4 ? 4 * ty + i : 60 + 4 * ty + i);
    if (m >= a.M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t n = n0 + 32 * h + 4 * tx;
      if (n < a.N) {
        float4* to = reinterpret_cast<float4*>(C + m * a.N + n);
        const float4 base = FORM == kNN && a.add ? *to : bias[h];
        *to = make_float4(acc[i][2 * h].x + base.x, acc[i][2 * h].y + base.y,
                          acc[i][2 * h + 1].x + base.z, acc[i][2 * h + 1].y + base.w);
      }
    }
  }
  if (sums && m0 + tid < a.M) C[a.M * a.N + m0 + tid] = colsum;
}

}  // namespace blr
