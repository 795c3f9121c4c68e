// Serial scan kernels: the BD-LRU scan when a problem has enough independent
// (batch row, channel group) chains to fill the GPU by itself.
//
// One warp (one thread block) owns CHW = 32 * VEC consecutive channels of one
// batch row (a 128-byte row segment; bfloat16's narrow form, VEC = 1, a 64-byte
// one, for problems with few chains or few channels: plan_narrow) and walks the
// whole sequence: each lane
// runs the recurrence h_t = alpha_t h_{t-1} + beta_t x_t of Sec. 3.2 serially
// for its VEC channels, one multiply-add per element, with the state in
// registers. There is no cross-lane or cross-block combine and no second pass.
//
// Data movement is TMA both ways. The inputs stream through a ring of
// shared-memory stages, one box of R rows per tensor; each lane writes
// its outputs over its own, already consumed, inputs in the stage, and one TMA
// store per output tensor sends the stage's outputs to global memory, clipped
// to the tensor's extent (sequence and channel tails need no masking). A stage
// is refilled at the start of the next iteration, once its store has read it,
// so two stages already double-buffer.
//
// The forward also keeps the state after every RB steps, which the backward
// uses as its starting points: the backward walks the sequence from the end in
// sub-blocks of RB steps, recomputes the sub-block's gates and states forward
// from the kept state (holding E = alpha - 1, 1 / sqrt(1 - alpha^2) and
// h_{t-1} per element in registers; bfloat16 lanes: alpha, sqrt(1 - alpha^2)
// and the d l factor), then runs the reverse recurrence
// g_t = dh_t + alpha_{t+1} g_{t+1} through it, writing dx, d rho and d iota and
// accumulating d Lambda. bfloat16 lanes carry their two channels as packed
// float pairs (paired multiply-adds).
//
// The forward's first block also restarts the workspace bookkeeping (error
// word, problem tag, the backward's exit counter and d Lambda partial sums), so
// no preparation kernel runs before either scan. Both kernels set their
// barriers up and then wait for the kernel before them on the stream
// (programmatic dependent launch), so that back-to-back calls do not pay the
// launch: 256 x 200 x 64 float32 fwd + bwd 41.9 -> 37.7 us, 1000 x 200 x 64
// bfloat16 with lengths 67.0 -> 60.5. They release the next kernel when their
// last row is done, not at their start: a grid let in early fills the SMs that
// have room first and runs unevenly (1500 x 800 x 64 bfloat16 364 against
// 292 us).
#pragma once

#include "blr_kernels.cuh"

namespace blr {

constexpr int kSeqMaxStages = 8;   // ring stages per warp
// Rings of at least this many stages may refill a consumed stage after the
// next stage's arithmetic rather than before it (the kernels' LATE form;
// measured on GB300: float32 rings of 4-8 stages up to 5 % faster that way; of
// the bfloat16 kernels the forward without the merge from 3 stages, 1500 x 800
// x 64 111 -> 99 us, and the narrow form's, with the merge 650 x 400 x 64 107.3 ->
// 105.6; the others 3-7 % slower).
constexpr int kSeqLateRefillStages = 4, kSeqLateRefillStagesBf16 = 3;

// Tensor maps: (channels, time, batch) views with boxes of 32 * VEC channels x
// R steps x 1 row. gate_logits is seen as two views of D channels each
// (rho: columns [0, D), iota: columns [D, 2D)), so that boxes clip at D.
struct SeqFwdArgs {
  CUtensorMap tm_x;
  CUtensorMap tm_r;
  CUtensorMap tm_i;
  CUtensorMap tm_h;  // h, or y = h SiLU(z) when gated; unused when NULL
  CUtensorMap tm_z;  // gated: z, the merge gate's input
  Plan p;
  const int32_t* lengths;  // NULL, or row b's sequence is its last lengths[b] steps
  const float* lambda;
  const float* h0;
  float* h_last;
  unsigned char* ws;
  int stages;
  int write_h;
};

struct SeqBwdArgs {
  CUtensorMap tm_dh;
  CUtensorMap tm_x;
  CUtensorMap tm_r;
  CUtensorMap tm_i;
  CUtensorMap tm_dx;
  CUtensorMap tm_dr;
  CUtensorMap tm_di;
  CUtensorMap tm_z;   // gated: z
  CUtensorMap tm_dz;  // gated: dz
  Plan p;
  const int32_t* lengths;  // as SeqFwdArgs
  const float* dh_last;
  const float* lambda;
  const float* h0;
  float* dlambda;
  float* dh0;
  unsigned char* ws;
  int stages;
};

__device__ __forceinline__ unsigned char* align128(unsigned char* p) {
  const uint32_t a = smem_addr(p);
  return p + (((a + 127u) & ~127u) - a);
}

// Dynamic shared memory of a serial kernel: `stages` stages of NB boxes, one
// mbarrier per stage, and slack for the 128-byte alignment of the boxes.
template <typename T, int VEC, int R>
__host__ __device__ constexpr uint32_t seq_box_bytes() {
  return (uint32_t)(R * 32 * VEC * sizeof(T));
}
template <typename T, int VEC, int R>
inline size_t seq_smem_bytes(int stages, int nb) {
  return (size_t)stages * nb * seq_box_bytes<T, VEC, R>() + (size_t)stages * sizeof(uint64_t) + 128;
}

// Per-lane channel constants: k = -c softplus(Lambda), kh = k / 2, and whether
// every channel of the warp keeps l = k r inside the series' range.
template <int VEC>
__device__ __forceinline__ bool seq_rates(const float* lambda, float c, int64_t d0, bool ch_ok,
                                          float (&k)[VEC], float (&kh)[VEC]) {
  bool poly = true;
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    k[v] = ch_ok ? decay_rate(c, lambda[d0 + v]) : 0.0f;
    kh[v] = 0.5f * k[v];
    poly = poly && k[v] >= -kExpm1Series;
  }
  return __all_sync(kFull, poly);
}

// The ring: stage i holds NB boxes, then the S mbarriers. Block-uniform
// bookkeeping of which stage holds which box and when it may be refilled.
template <int NB, uint32_t BOX>
struct SeqRing {
  unsigned char* base;
  uint64_t* bars;
  int S;
  __device__ __forceinline__ unsigned char* stage(int st) const { return base + (size_t)st * NB * BOX; }
};

// Kernel modes: the plain scan, or rows with lengths.
constexpr int kSeqPlain = 0, kSeqVarlen = 1;

// Restarts the workspace bookkeeping for a forward (one block, one warp):
// clears the error word, the backward's exit counter and the d Lambda partial
// sums, and tags the workspace with the problem.
__device__ __forceinline__ void seq_reset_workspace(unsigned char* ws, const Plan& p, uint32_t tag,
                                                    int lane) {
  FwdHeader* fh = reinterpret_cast<FwdHeader*>(ws + p.off_fhdr);
  BwdHeader* bh = reinterpret_cast<BwdHeader*>(ws + p.off_bhdr);
  double* acc = reinterpret_cast<double*>(ws + p.off_dlam);
  for (int64_t i = lane; i < (int64_t)kStripes * p.D; i += 32) acc[i] = 0.0;
  if (lane == 0) {
    fh->err = 0u;
    bh->exited = 0u;
    bh->set = 0u;
    fh->tag = tag;
    fh->complete = 1u;
  }
}

// ------------------------------------------------------------------ forward

// seq_fwd_stage for a bfloat16 lane under GatesFast: the same arithmetic in
// the same order, on packed pairs.
template <bool POLY, bool FULL, int R, int RB, bool GATED>
__device__ __forceinline__ void seq_fwd_stage_bf16x2(unsigned char* sb, int rows, float2 kh,
                                                     float2& hc, float* carry, int64_t& cidx,
                                                     int64_t n_carry, int64_t BD, bool ch_ok) {
  constexpr uint32_t ROWB = 128;
  constexpr uint32_t BOX = R * ROWB;
  float2 al[R], uu[R];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    if (FULL || s < rows) {
      const float2 hx = bf2_scaled(*reinterpret_cast<const uint32_t*>(sb + s * ROWB), kBf2Half);
      const float2 hr = bf2_scaled(*reinterpret_cast<const uint32_t*>(sb + BOX + s * ROWB), kBf2Half);
      const float2 hi = bf2_scaled(*reinterpret_cast<const uint32_t*>(sb + 2 * BOX + s * ROWB), kBf2Half);
      const float2 e = expm1_neg2<POLY>(__ffma2_rn(kh, tanh2(hr), kh));  // l = kh tanh(rho/2) + kh
      al[s] = __fadd2_rn(f2(1.0f), e);
      const float2 m2 = __fmul2_rn(e, __fadd2_rn(e, f2(2.0f)));  // -(1 - alpha^2)
      const float2 n = make_float2(sqrt_approx(-m2.x), sqrt_approx(-m2.y));
      uu[s] = __fmul2_rn(n, __ffma2_rn(hx, tanh2(hi), hx));  // sqrt(1 - alpha^2) i x
    }
  }
#pragma unroll
  for (int s = 0; s < R; ++s) {
    if (FULL || s < rows) {
      hc = __ffma2_rn(al[s], hc, uu[s]);
      float2 out = hc;
      if constexpr (GATED) {  // y = h SiLU(z), off the gates' dependency chains
        const float2 hz = bf2_scaled(*reinterpret_cast<const uint32_t*>(sb + 3 * BOX + s * ROWB), kBf2Half);
        out = __fmul2_rn(hc, __ffma2_rn(hz, tanh2(hz), hz));
      }
      *reinterpret_cast<uint32_t*>(sb + s * ROWB) = bf2_pack(out);
      if ((s + 1) % RB == 0) {  // a kept state: after step (cidx + 1) RB - 1
        if (cidx < n_carry && ch_ok) *reinterpret_cast<float2*>(carry + cidx * BD) = hc;
        ++cidx;
      }
    }
  }
}

// One stage, rows [0, rows) (all R when FULL). Phase 1 evaluates the
// gates of every row (independent work), phase 2 runs the recurrence and
// writes h over x in the stage (GATED: y = h SiLU(z), the merge of the gated
// recurrent layer, Alg. 1, with z the stage's fourth box). `cidx` is the index
// of the next kept state.
template <class IO, class G, bool POLY, bool FULL, int R, int RB, bool GATED>
__device__ __forceinline__ void seq_fwd_stage(unsigned char* sb, int rows,
                                              const float (&k)[IO::VEC], const float (&kh)[IO::VEC],
                                              float (&hc)[IO::VEC], float* carry, int64_t& cidx,
                                              int64_t n_carry, int64_t BD, bool ch_ok) {
  using Raw = typename IO::Raw;
  constexpr int V = IO::VEC;
  constexpr uint32_t ROWB = 32 * V * sizeof(typename IO::T);
  constexpr uint32_t BOX = R * ROWB;
  float al[R][V], uu[R][V];
#pragma unroll
  for (int s = 0; s < R; ++s) {
    if (FULL || s < rows) {
      float xv[V], rv[V], iv[V];
      if constexpr (G::kHalfInputs) {
        IO::unpack_half(*reinterpret_cast<const Raw*>(sb + s * ROWB), xv);
        IO::unpack_half(*reinterpret_cast<const Raw*>(sb + BOX + s * ROWB), rv);
        IO::unpack_half(*reinterpret_cast<const Raw*>(sb + 2 * BOX + s * ROWB), iv);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const float e = expm1_neg<G::kDeg, POLY>(G::decay_log_half(rv[v], kh[v]));
          al[s][v] = 1.0f + e;
          uu[s][v] = G::sqrt(-e * (e + 2.0f)) * G::gated_x_half(iv[v], xv[v]);
        }
      } else {
        IO::unpack(*reinterpret_cast<const Raw*>(sb + s * ROWB), xv);
        IO::unpack(*reinterpret_cast<const Raw*>(sb + BOX + s * ROWB), rv);
        IO::unpack(*reinterpret_cast<const Raw*>(sb + 2 * BOX + s * ROWB), iv);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const float e = expm1_neg<G::kDeg, POLY>(G::decay_log(rv[v], k[v], kh[v]));
          al[s][v] = 1.0f + e;
          uu[s][v] = G::sqrt(-e * (e + 2.0f)) * (G::sigmoid(iv[v]) * xv[v]);
        }
      }
    }
  }
#pragma unroll
  for (int s = 0; s < R; ++s) {
    if (FULL || s < rows) {
      float out[V];
      // SiLU(z) here rather than with the gates: off the gates' dependency
      // chains, it overlaps the recurrence (measured faster).
      float sz[V];
      if constexpr (GATED) {
        float zv[V];
        if constexpr (G::kHalfInputs)
          IO::unpack_half(*reinterpret_cast<const Raw*>(sb + 3 * BOX + s * ROWB), zv);
        else
          IO::unpack(*reinterpret_cast<const Raw*>(sb + 3 * BOX + s * ROWB), zv);
#pragma unroll
        for (int v = 0; v < V; ++v) sz[v] = G::silu(zv[v]);
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        hc[v] = fmaf(al[s][v], hc[v], uu[s][v]);
        if constexpr (GATED)
          out[v] = hc[v] * sz[v];
        else
          out[v] = hc[v];
      }
      IO::store_smem(sb + s * ROWB, out);
      if ((s + 1) % RB == 0) {  // a kept state: after step (cidx + 1) RB - 1
        if (cidx < n_carry && ch_ok) {
#pragma unroll
          for (int v = 0; v < V; ++v) carry[cidx * BD + v] = hc[v];
        }
        ++cidx;
      }
    }
  }
}

// MODE kSeqVarlen: the rows carry lengths (a.lengths) and each chain starts
// at its first real step. kSeqPlain keeps the plain scan's code.
// LATE: refill a consumed stage after the next stage's arithmetic (deep rings).
template <typename T, class M, int VEC, int R, int RB, bool GATED, int MODE, bool LATE>
__global__ void __launch_bounds__(32) seq_fwd_kernel(const __grid_constant__ SeqFwdArgs a) {
  constexpr bool VARLEN = MODE == kSeqVarlen;
  using IO = Io<T, VEC>;
  using G = typename GatePolicy<M>::type;
  constexpr int CHW = 32 * VEC;
  constexpr int NB = GATED ? 4 : 3;  // boxes per stage: x, rho, iota (, z)
  constexpr uint32_t BOX = seq_box_bytes<T, VEC, R>();
  static_assert(R % RB == 0, "kept states must fall on stage rows");
  // bfloat16 lanes run their arithmetic on packed pairs with the merge, whose
  // instructions fill the scheduler, and one channel at a time without it: a
  // paired instruction holds the one pipe that has it for two cycles, and the
  // few warps of a scheduler wait for it (fwd, us, paired / single: 1000 x 200 x 64
  // 24.1 / 21.8, 700 x 200 x 64 23.8 / 21.2; with the merge 2048 x 50 x 64
  // 19.4 / 19.7).
  constexpr bool kPacked = G::kHalfInputs && VEC == 2 && GATED;
  const Plan& p = a.p;
  extern __shared__ unsigned char seq_smem[];
  SeqRing<NB, BOX> ring{align128(seq_smem), nullptr, a.stages};
  ring.bars = reinterpret_cast<uint64_t*>(ring.stage(ring.S));

  const int lane = threadIdx.x;
  const int64_t n_g = (p.D + CHW - 1) / CHW;
  const int64_t chain = blockIdx.x;
  const int64_t b = chain / n_g;
  const int64_t g = chain - b * n_g;
  const int64_t d0 = g * CHW + lane * VEC;
  const bool ch_ok = d0 < p.D;  // D % 8 == 0: a lane's VEC channels are all in or all out
  const int64_t BD = p.B * p.D;
  FwdHeader* fh = reinterpret_cast<FwdHeader*>(a.ws + p.off_fhdr);

  if (lane == 0) {
    for (int s = 0; s < ring.S; ++s) mbar_init(&ring.bars[s], 1);
    fence_mbar_init();
    tensormap_prefetch(&a.tm_x);
    tensormap_prefetch(&a.tm_r);
    tensormap_prefetch(&a.tm_i);
    if constexpr (GATED) tensormap_prefetch(&a.tm_z);
    if (a.write_h) tensormap_prefetch(&a.tm_h);
  }
  pdl_wait();
  if (blockIdx.x == 0) seq_reset_workspace(a.ws, p, p.tag, lane);

  float k[VEC], kh[VEC], hc[VEC];
  const bool poly = seq_rates<VEC>(a.lambda, p.c, d0, ch_ok, k, kh);
#pragma unroll
  for (int v = 0; v < VEC; ++v) hc[v] = (ch_ok && a.h0 != nullptr) ? a.h0[b * p.D + d0 + v] : 0.0f;

  // The chain's steps: [t0, t0 + len) (all of them unless the rows carry lengths).
  const int64_t t0 = VARLEN ? row_start(a.lengths, b, p.L) : 0;
  const int64_t len = p.L - t0;
  const int64_t nblk = (len + R - 1) / R;
  const int cd = (int)(g * CHW), cb = (int)b;
  auto issue = [&](int st, int64_t j) {
    unsigned char* dst = ring.stage(st);
    const int t = (int)(t0 + j * R);
    mbar_arrive_expect_tx(&ring.bars[st], NB * BOX);
    tma_load_3d(dst, &a.tm_x, &ring.bars[st], cd, t, cb);
    tma_load_3d(dst + BOX, &a.tm_r, &ring.bars[st], cd, t, cb);
    tma_load_3d(dst + 2 * BOX, &a.tm_i, &ring.bars[st], cd, t, cb);
    if constexpr (GATED) tma_load_3d(dst + 3 * BOX, &a.tm_z, &ring.bars[st], cd, t, cb);
  };
  if (lane == 0) {
    for (int s = 0; s < ring.S && s < nblk; ++s) issue(s, s);
  }
  __syncwarp();

  float* carry = reinterpret_cast<float*>(a.ws + p.off_kept) + b * p.D + d0;
  int64_t cidx = 0;
  const int64_t n_carry = p.n_carry;
  int st = 0, prev = ring.S - 1;
  uint32_t phase = 0;
  for (int64_t j = 0; j < nblk; ++j) {
    mbar_wait(&ring.bars[st], phase, &fh->err);
    // Shallow rings refill the previous stage at the top of the iteration, deep
    // ones after this stage's arithmetic (as the backward).
    if (!LATE && lane == 0 && j > 0 && j - 1 + ring.S < nblk) {
      if (a.write_h) bulk_wait_read<0>();
      issue(prev, j - 1 + ring.S);
    }
    unsigned char* sb = ring.stage(st);
    unsigned char* lb = sb + lane * VEC * sizeof(T);
    const int64_t left = len - j * R;
    const int rows = (int)(left < R ? left : R);
    if constexpr (kPacked) {
      float2 hc2 = make_float2(hc[0], hc[1]);
      const float2 kh2 = make_float2(kh[0], kh[1]);
      if (rows == R) {
        if (poly)
          seq_fwd_stage_bf16x2<true, true, R, RB, GATED>(lb, rows, kh2, hc2, carry, cidx, n_carry, BD, ch_ok);
        else
          seq_fwd_stage_bf16x2<false, true, R, RB, GATED>(lb, rows, kh2, hc2, carry, cidx, n_carry, BD, ch_ok);
      } else {
        seq_fwd_stage_bf16x2<false, false, R, RB, GATED>(lb, rows, kh2, hc2, carry, cidx, n_carry, BD, ch_ok);
      }
      hc[0] = hc2.x;
      hc[1] = hc2.y;
    } else if (rows == R) {
      if (poly)
        seq_fwd_stage<IO, G, true, true, R, RB, GATED>(lb, rows, k, kh, hc, carry, cidx, n_carry, BD, ch_ok);
      else
        seq_fwd_stage<IO, G, false, true, R, RB, GATED>(lb, rows, k, kh, hc, carry, cidx, n_carry, BD, ch_ok);
    } else {
      seq_fwd_stage<IO, G, false, false, R, RB, GATED>(lb, rows, k, kh, hc, carry, cidx, n_carry, BD, ch_ok);
    }
    fence_proxy_async_smem();  // the stage's h rows, visible to the TMA store
    __syncwarp();
    if (lane == 0) {
      if (LATE && j > 0 && j - 1 + ring.S < nblk) {
        if (a.write_h) bulk_wait_read<0>();
        issue(prev, j - 1 + ring.S);
      }
      if (a.write_h) {
        tma_store_3d(&a.tm_h, sb, cd, (int)(t0 + j * R), cb);
        bulk_commit();
      }
    }
    prev = st;
    if (++st == ring.S) {
      st = 0;
      phase ^= 1u;
    }
  }
  pdl_release();
  if (lane == 0 && a.write_h) bulk_wait_all();
  if (a.h_last != nullptr && ch_ok) {
#pragma unroll
    for (int v = 0; v < VEC; ++v) a.h_last[b * p.D + d0 + v] = hc[v];
  }
}

// ----------------------------------------------------------------- backward

// One sub-block of RB steps (rows [0, srows) when not FULL) starting at row
// `row0` of the stage, float32: forward recompute from the state hc, then the reverse
// recurrence carrying w = alpha g. dx, d rho and d iota overwrite dh, rho and
// iota of the same rows in the stage. GATED: the first box holds dy, the
// gradient of y = h SiLU(z) (Alg. 1), so dh = dy SiLU(z), and
// dz = dy h SiLU'(z) overwrites z in the fifth box.
template <class IO, class G, bool POLY, bool FULL, int R, int RB, bool GATED>
__device__ __forceinline__ void seq_bwd_sub(unsigned char* lb, int row0, int srows,
                                            const float (&k)[IO::VEC], const float (&kh)[IO::VEC],
                                            float (&hc)[IO::VEC], float (&w)[IO::VEC],
                                            float (&dlr)[IO::VEC]) {
  using Raw = typename IO::Raw;
  constexpr int V = IO::VEC;
  constexpr uint32_t ROWB = 32 * V * sizeof(typename IO::T);
  constexpr uint32_t BOX = R * ROWB;
  // boxes of a backward stage: dh (dy), x, rho, iota (, z)
  unsigned char* s_dh = lb + row0 * ROWB;
  const unsigned char* s_x = s_dh + BOX;
  unsigned char* s_r = s_dh + 2 * BOX;
  unsigned char* s_i = s_dh + 3 * BOX;
  unsigned char* s_z = s_dh + 4 * BOX;
  float E[RB][V], RS[RB][V], HP[RB][V];
#pragma unroll
  for (int s = 0; s < RB; ++s) {
    if (FULL || s < srows) {
      float xv[V], rv[V], iv[V], ix[V], l[V];
      IO::unpack(*reinterpret_cast<const Raw*>(s_x + s * ROWB), xv);
      IO::unpack(*reinterpret_cast<const Raw*>(s_r + s * ROWB), rv);
      IO::unpack(*reinterpret_cast<const Raw*>(s_i + s * ROWB), iv);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        l[v] = G::decay_log(rv[v], k[v], kh[v]);
        ix[v] = G::sigmoid(iv[v]) * xv[v];
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float e = expm1_neg<G::kDeg, POLY>(l[v]);
        const float q = -e * (e + 2.0f);
        const float rs = rsqrt_approx(fmaxf(q, 1e-30f));  // 1/sqrt(q); finite at q = 0
        E[s][v] = e;
        RS[s][v] = rs;
        HP[s][v] = hc[v];
        hc[v] = fmaf(1.0f + e, hc[v], (q * rs) * ix[v]);
      }
    }
  }
#pragma unroll
  for (int s = RB - 1; s >= 0; --s) {
    if (FULL || s < srows) {
      float gv[V], xv[V], rv[V], iv[V], ox[V], orho[V], oiota[V], sf[V], sdf[V], oz[V];
      IO::unpack(*reinterpret_cast<const Raw*>(s_dh + s * ROWB), gv);
      if constexpr (GATED) {
        float zv[V];
        IO::unpack(*reinterpret_cast<const Raw*>(s_z + s * ROWB), zv);
#pragma unroll
        for (int v = 0; v < V; ++v) G::silu_grad(zv[v], sf[v], sdf[v]);
      }
      IO::unpack(*reinterpret_cast<const Raw*>(s_x + s * ROWB), xv);
      IO::unpack(*reinterpret_cast<const Raw*>(s_r + s * ROWB), rv);
      IO::unpack(*reinterpret_cast<const Raw*>(s_i + s * ROWB), iv);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float e = E[s][v], rs = RS[s][v];
        const float alpha = 1.0f + e;
        const float q = -e * (e + 2.0f);
        const float r = G::sigmoid(rv[v]), i = G::sigmoid(iv[v]);
        float dhv = gv[v];
        if constexpr (GATED) dhv *= sf[v];
        const float g = dhv + w[v];
        w[v] = alpha * g;
        const float ix = i * xv[v];
        const float u = (q * rs) * ix;
        if constexpr (GATED) oz[v] = (gv[v] * fmaf(alpha, HP[s][v], u)) * sdf[v];  // dy h_t SiLU'
        ox[v] = (g * (q * rs)) * i;
        oiota[v] = (g * u) * (1.0f - i);
        // d/dl of h_t: alpha g (h_{t-1} - alpha u / q), with alpha g = w and
        // u / q = i x rs
        const float dl = w[v] * (HP[s][v] - (alpha * rs) * ix);
        orho[v] = (dl * k[v]) * fmaf(-r, r, r);
        dlr[v] = fmaf(dl, r, dlr[v]);
      }
      IO::store_smem(s_dh + s * ROWB, ox);
      IO::store_smem(s_r + s * ROWB, orho);
      IO::store_smem(s_i + s * ROWB, oiota);
      if constexpr (GATED) IO::store_smem(s_z + s * ROWB, oz);
    }
  }
}

// seq_bwd_sub for a bfloat16 lane of two channels under GatesFast, on packed
// pairs. The forward recompute keeps, per step, alpha, -sqrt(1 - alpha^2)
// and c = h_{t-1} - alpha i x / sqrt(1 - alpha^2) (so that d l = alpha g c);
// the reverse recurrence re-reads the step's inputs for i and r, and uses
// r (1 - r) = (1 - tanh(rho/2)^2) / 4, so d rho = d l (k/4) (1 - tanh^2).
// kq = k/4 and nkq = -k/4 per channel. GATED: the recompute also forms
// dz = dy h SiLU'(z), rounded to the bfloat16 it is written as (one register a
// step, where h itself would take two).
template <bool POLY, bool FULL, int R, int RB, bool GATED>
__device__ __forceinline__ void seq_bwd_sub_bf16x2(unsigned char* lb, int row0, int srows, float2 kh,
                                                   float2 kq, float2 nkq, float2& hc, float2& w,
                                                   float2& dlr) {
  constexpr uint32_t ROWB = 128;
  constexpr uint32_t BOX = R * ROWB;
  unsigned char* s_dh = lb + row0 * ROWB;
  const unsigned char* s_x = s_dh + BOX;
  unsigned char* s_r = s_dh + 2 * BOX;
  unsigned char* s_i = s_dh + 3 * BOX;
  unsigned char* s_z = s_dh + 4 * BOX;
  float2 AL[RB], NQ[RB], CP[RB];
  uint32_t DZ[GATED ? RB : 1];
#pragma unroll
  for (int s = 0; s < RB; ++s) {
    if (FULL || s < srows) {
      const float2 nhx = bf2_scaled(*reinterpret_cast<const uint32_t*>(s_x + s * ROWB), kBf2NegHalf);
      const float2 hr = bf2_scaled(*reinterpret_cast<const uint32_t*>(s_r + s * ROWB), kBf2Half);
      const float2 hi = bf2_scaled(*reinterpret_cast<const uint32_t*>(s_i + s * ROWB), kBf2Half);
      const float2 e = expm1_neg2<POLY>(__ffma2_rn(kh, tanh2(hr), kh));
      const float2 m2 = __fmul2_rn(e, __fadd2_rn(e, f2(2.0f)));  // -(1 - alpha^2)
      const float2 rs = make_float2(rsqrt_approx(fmaxf(-m2.x, 1e-30f)), rsqrt_approx(fmaxf(-m2.y, 1e-30f)));
      const float2 al = __fadd2_rn(f2(1.0f), e);
      const float2 nq = __fmul2_rn(m2, rs);                // -sqrt(1 - alpha^2)
      const float2 nix = __ffma2_rn(nhx, tanh2(hi), nhx);  // -i x
      AL[s] = al;
      NQ[s] = nq;
      CP[s] = __ffma2_rn(__fmul2_rn(al, rs), nix, hc);
      hc = __ffma2_rn(al, hc, __fmul2_rn(nq, nix));  // alpha h + sqrt(1 - alpha^2) i x
      if constexpr (GATED) {  // with hz = z/2 and th = tanh(hz) as silu_grad
        const float2 hz = bf2_scaled(*reinterpret_cast<const uint32_t*>(s_z + s * ROWB), kBf2Half);
        const float2 th = tanh2(hz);
        const float2 sg = __ffma2_rn(f2(0.5f), th, f2(0.5f));
        const float2 df = __ffma2_rn(sg, __ffma2_rn(__fmul2_rn(f2(-1.0f), hz), th, hz), sg);
        const float2 dy = bf2_unpack(*reinterpret_cast<const uint32_t*>(s_dh + s * ROWB));
        DZ[s] = bf2_pack(__fmul2_rn(__fmul2_rn(dy, hc), df));
      }
    }
  }
#pragma unroll
  for (int s = RB - 1; s >= 0; --s) {
    if (FULL || s < srows) {
      float2 dh = bf2_unpack(*reinterpret_cast<const uint32_t*>(s_dh + s * ROWB));
      if constexpr (GATED) {  // dh = dy SiLU(z)
        const float2 hz = bf2_scaled(lds_again(s_z + s * ROWB), kBf2Half);
        dh = __fmul2_rn(dh, __ffma2_rn(hz, tanh2(hz), hz));
        *reinterpret_cast<uint32_t*>(s_z + s * ROWB) = DZ[s];
      }
      const float2 nhx = bf2_scaled(lds_again(s_x + s * ROWB), kBf2NegHalf);
      const float2 thr = tanh2(bf2_scaled(lds_again(s_r + s * ROWB), kBf2Half));
      const float2 thi = tanh2(bf2_scaled(lds_again(s_i + s * ROWB), kBf2Half));
      const float2 g = __fadd2_rn(dh, w);
      w = __fmul2_rn(AL[s], g);
      const float2 gnq = __fmul2_rn(g, NQ[s]);                    // -g sqrt(1 - alpha^2)
      const float2 ni = __ffma2_rn(f2(-0.5f), thi, f2(-0.5f));    // -i
      const float2 omi = __ffma2_rn(f2(-0.5f), thi, f2(0.5f));    // 1 - i
      const float2 nix = __ffma2_rn(nhx, thi, nhx);               // -i x
      const float2 ox = __fmul2_rn(gnq, ni);                      // g sqrt(1 - alpha^2) i
      const float2 oi = __fmul2_rn(__fmul2_rn(gnq, nix), omi);    // g u (1 - i)
      const float2 dl = __fmul2_rn(w, CP[s]);
      const float2 orho = __fmul2_rn(dl, __ffma2_rn(nkq, __fmul2_rn(thr, thr), kq));
      dlr = __ffma2_rn(dl, __ffma2_rn(f2(0.5f), thr, f2(0.5f)), dlr);  // += d l r
      *reinterpret_cast<uint32_t*>(s_dh + s * ROWB) = bf2_pack(ox);
      *reinterpret_cast<uint32_t*>(s_r + s * ROWB) = bf2_pack(orho);
      *reinterpret_cast<uint32_t*>(s_i + s * ROWB) = bf2_pack(oi);
    }
  }
}

// The same for a lane of one bfloat16 channel: the recompute also keeps the
// step's inputs and gates (there are registers for them).
template <bool POLY, bool FULL, int R, int RB, bool GATED>
__device__ __forceinline__ void seq_bwd_sub_bf16(unsigned char* lb, int row0, int srows, float kh,
                                                 float kq, float& hc, float& w, float& dlr) {
  using IO = Io<__nv_bfloat16, 1>;
  using G = GatesFast;
  constexpr uint32_t ROWB = 64;
  constexpr uint32_t BOX = R * ROWB;
  unsigned char* s_dh = lb + row0 * ROWB;
  const unsigned char* s_x = s_dh + BOX;
  unsigned char* s_r = s_dh + 2 * BOX;
  unsigned char* s_i = s_dh + 3 * BOX;
  unsigned char* s_z = s_dh + 4 * BOX;
  auto full = [](const unsigned char* p) {
    float v[1];
    IO::unpack(*reinterpret_cast<const uint16_t*>(p), v);
    return v[0];
  };
  auto put = [](unsigned char* p, float v) {
    const float t[1] = {v};
    IO::store_smem(p, t);
  };
  float AL[RB], NQ[RB], CP[RB], NX[RB], TR[RB], TI[RB], DH[RB];
#pragma unroll
  for (int s = 0; s < RB; ++s) {
    if (FULL || s < srows) {
      const float nhx = -0.5f * full(s_x + s * ROWB);
      TR[s] = tanh_approx(0.5f * full(s_r + s * ROWB));
      TI[s] = tanh_approx(0.5f * full(s_i + s * ROWB));
      const float e = expm1_neg<G::kDeg, POLY>(fmaf(kh, TR[s], kh));
      const float m2 = e * (e + 2.0f);  // -(1 - alpha^2)
      const float rs = rsqrt_approx(fmaxf(-m2, 1e-30f));
      AL[s] = 1.0f + e;
      NQ[s] = m2 * rs;                    // -sqrt(1 - alpha^2)
      NX[s] = fmaf(nhx, TI[s], nhx);      // -i x
      CP[s] = fmaf(AL[s] * rs, NX[s], hc);
      hc = fmaf(AL[s], hc, NQ[s] * NX[s]);  // alpha h + sqrt(1 - alpha^2) i x
      DH[s] = full(s_dh + s * ROWB);
      if constexpr (GATED) {
        float f, df;
        G::silu_grad(0.5f * full(s_z + s * ROWB), f, df);
        put(s_z + s * ROWB, (DH[s] * hc) * df);  // dz = dy h SiLU'(z)
        DH[s] *= f;
      }
    }
  }
#pragma unroll
  for (int s = RB - 1; s >= 0; --s) {
    if (FULL || s < srows) {
      const float g = DH[s] + w;
      w = AL[s] * g;
      const float gnq = g * NQ[s];                                      // -g sqrt(1 - alpha^2)
      const float dl = w * CP[s];
      put(s_dh + s * ROWB, gnq * fmaf(-0.5f, TI[s], -0.5f));            // g sqrt(1 - alpha^2) i
      put(s_i + s * ROWB, (gnq * NX[s]) * fmaf(-0.5f, TI[s], 0.5f));    // g u (1 - i)
      put(s_r + s * ROWB, dl * fmaf(-kq, TR[s] * TR[s], kq));
      dlr = fmaf(dl, fmaf(0.5f, TR[s], 0.5f), dlr);                     // += d l r
    }
  }
}

// MODE as seq_fwd_kernel's.
template <typename T, class M, int VEC, int R, int RB, bool GATED, int MODE, bool LATE>
__global__ void __launch_bounds__(32, sizeof(T) == 4 ? 8 : 16) seq_bwd_kernel(const __grid_constant__ SeqBwdArgs a) {
  constexpr bool VARLEN = MODE == kSeqVarlen;
  using IO = Io<T, VEC>;
  using G = typename GatePolicy<M>::type;
  constexpr int CHW = 32 * VEC;
  constexpr int NB = GATED ? 5 : 4;  // boxes per stage: dh (dy), x, rho, iota (, z)
  constexpr uint32_t BOX = seq_box_bytes<T, VEC, R>();
  constexpr int NSUB = R / RB;
  static_assert(R % RB == 0, "sub-blocks must tile a stage");
  constexpr bool kBf16 = sizeof(T) == 2, kPacked = kBf16 && VEC == 2;  // bfloat16, on packed pairs
  const Plan& p = a.p;
  extern __shared__ unsigned char seq_smem[];
  SeqRing<NB, BOX> ring{align128(seq_smem), nullptr, a.stages};
  ring.bars = reinterpret_cast<uint64_t*>(ring.stage(ring.S));

  const int lane = threadIdx.x;
  FwdHeader* fh = reinterpret_cast<FwdHeader*>(a.ws + p.off_fhdr);
  BwdHeader* bh = reinterpret_cast<BwdHeader*>(a.ws + p.off_bhdr);
  if (lane == 0) {
    for (int s = 0; s < ring.S; ++s) mbar_init(&ring.bars[s], 1);
    fence_mbar_init();
    tensormap_prefetch(&a.tm_dh);
    tensormap_prefetch(&a.tm_x);
    tensormap_prefetch(&a.tm_r);
    tensormap_prefetch(&a.tm_i);
    if constexpr (GATED) tensormap_prefetch(&a.tm_z);
  }
  pdl_wait();
  {
    int ok = 0;
    if (lane == 0) {
      const uint32_t tag = __ldcg(&fh->tag), complete = __ldcg(&fh->complete);  // one round trip
      ok = tag == p.tag && complete == 1u;
      if (!ok) atomicOr(&fh->err, kErrWorkspace);
    }
    if (!__shfl_sync(kFull, ok, 0)) return;  // no forward states for this problem: write nothing
  }
  const int64_t n_g = (p.D + CHW - 1) / CHW;
  const int64_t chain = blockIdx.x;
  const int64_t b = chain / n_g;
  const int64_t g = chain - b * n_g;
  const int64_t d0 = g * CHW + lane * VEC;
  const bool ch_ok = d0 < p.D;
  const int64_t BD = p.B * p.D;

  // The start states of the next QD sub-blocks, loaded QD sub-blocks ahead of
  // use (one ahead for bfloat16, whose registers are fully used).
  constexpr int QD = sizeof(T) == 4 ? 4 : 1;
  float k[VEC], kh[VEC], w[VEC], dlr[VEC], sq[QD][VEC];
  const bool poly = seq_rates<VEC>(a.lambda, p.c, d0, ch_ok, k, kh);
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    w[v] = (ch_ok && a.dh_last != nullptr) ? a.dh_last[b * p.D + d0 + v] : 0.0f;
    dlr[v] = 0.0f;
  }
  const int64_t t0 = VARLEN ? row_start(a.lengths, b, p.L) : 0;
  const int64_t len = p.L - t0;
  const int64_t nblk = (len + R - 1) / R;
  const float* carry = reinterpret_cast<const float*>(a.ws + p.off_kept) + b * p.D + d0;
  // the state before sub-block m: h0 for the chain's first, else kept state m - 1
  auto load_start = [&](int64_t m, float (&out)[VEC]) {
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      out[v] = 0.0f;
      if (ch_ok) {
        if (m > 0)
          out[v] = __ldcg(carry + (m - 1) * BD + v);
        else if (a.h0 != nullptr)
          out[v] = a.h0[b * p.D + d0 + v];
      }
    }
  };
  const int cd = (int)(g * CHW), cb = (int)b;
  auto issue = [&](int st, int64_t j) {
    unsigned char* dst = ring.stage(st);
    const int t = (int)(t0 + j * R);
    mbar_arrive_expect_tx(&ring.bars[st], NB * BOX);
    tma_load_3d(dst, &a.tm_dh, &ring.bars[st], cd, t, cb);
    tma_load_3d(dst + BOX, &a.tm_x, &ring.bars[st], cd, t, cb);
    tma_load_3d(dst + 2 * BOX, &a.tm_r, &ring.bars[st], cd, t, cb);
    tma_load_3d(dst + 3 * BOX, &a.tm_i, &ring.bars[st], cd, t, cb);
    if constexpr (GATED) tma_load_3d(dst + 4 * BOX, &a.tm_z, &ring.bars[st], cd, t, cb);
  };
  if (lane == 0) {
    for (int s = 0; s < ring.S && s < nblk; ++s) issue(s, nblk - 1 - s);
  }
  __syncwarp();

  int64_t m = (len + RB - 1) / RB - 1;  // the sub-block processed next (-1: none)
#pragma unroll
  for (int u = 0; u < QD; ++u) {
#pragma unroll
    for (int v = 0; v < VEC; ++v) sq[u][v] = 0.0f;
    if (m - u >= 0) load_start(m - u, sq[u]);
  }
  int st = 0, prev = ring.S - 1;
  uint32_t phase = 0;
  for (int64_t i = 0; i < nblk; ++i) {
    const int64_t j = nblk - 1 - i;
    mbar_wait(&ring.bars[st], phase, &fh->err);
    // Shallow rings refill the previous stage as soon as its stores have read
    // it, at the top of the iteration; deep ones after this stage's arithmetic,
    // when those stores are long done and the wait costs nothing.
    if (!LATE && lane == 0 && i > 0 && i - 1 + ring.S < nblk) {
      bulk_wait_read<0>();
      issue(prev, nblk - 1 - (i - 1 + ring.S));
    }
    unsigned char* sb = ring.stage(st);
    unsigned char* lb = sb + lane * VEC * sizeof(T);
    const int64_t left = len - j * R;
    const int rows = (int)(left < R ? left : R);
#pragma unroll
    for (int q = NSUB - 1; q >= 0; --q) {
      const int row0 = q * RB;
      if (row0 < rows) {
        const int srows = rows - row0 < RB ? rows - row0 : RB;
        float hc[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) hc[v] = sq[0][v];
#pragma unroll
        for (int u = 0; u + 1 < QD; ++u) {
#pragma unroll
          for (int v = 0; v < VEC; ++v) sq[u][v] = sq[u + 1][v];
        }
        if (m - QD >= 0) load_start(m - QD, sq[QD - 1]);  // in flight for QD sub-blocks
        if constexpr (kPacked) {
          float2 hc2 = make_float2(hc[0], hc[1]), w2 = make_float2(w[0], w[1]);
          float2 dlr2 = make_float2(dlr[0], dlr[1]);
          const float2 kh2 = make_float2(kh[0], kh[1]);
          const float2 kq = make_float2(0.25f * k[0], 0.25f * k[1]);
          const float2 nkq = make_float2(-kq.x, -kq.y);
          if (srows == RB) {
            if (poly)
              seq_bwd_sub_bf16x2<true, true, R, RB, GATED>(lb, row0, srows, kh2, kq, nkq, hc2, w2, dlr2);
            else
              seq_bwd_sub_bf16x2<false, true, R, RB, GATED>(lb, row0, srows, kh2, kq, nkq, hc2, w2, dlr2);
          } else {
            seq_bwd_sub_bf16x2<false, false, R, RB, GATED>(lb, row0, srows, kh2, kq, nkq, hc2, w2, dlr2);
          }
          w[0] = w2.x;
          w[1] = w2.y;
          dlr[0] = dlr2.x;
          dlr[1] = dlr2.y;
        } else if constexpr (kBf16) {
          const float kq = 0.25f * k[0];
          if (srows == RB) {
            if (poly)
              seq_bwd_sub_bf16<true, true, R, RB, GATED>(lb, row0, srows, kh[0], kq, hc[0], w[0], dlr[0]);
            else
              seq_bwd_sub_bf16<false, true, R, RB, GATED>(lb, row0, srows, kh[0], kq, hc[0], w[0], dlr[0]);
          } else {
            seq_bwd_sub_bf16<false, false, R, RB, GATED>(lb, row0, srows, kh[0], kq, hc[0], w[0], dlr[0]);
          }
        } else if (srows == RB) {
          if (poly)
            seq_bwd_sub<IO, G, true, true, R, RB, GATED>(lb, row0, srows, k, kh, hc, w, dlr);
          else
            seq_bwd_sub<IO, G, false, true, R, RB, GATED>(lb, row0, srows, k, kh, hc, w, dlr);
        } else {
          seq_bwd_sub<IO, G, false, false, R, RB, GATED>(lb, row0, srows, k, kh, hc, w, dlr);
        }
        --m;
      }
    }
    fence_proxy_async_smem();  // the stage's outputs, visible to the TMA stores
    __syncwarp();
    if (lane == 0) {
      if (LATE && i > 0 && i - 1 + ring.S < nblk) {
        bulk_wait_read<0>();
        issue(prev, nblk - 1 - (i - 1 + ring.S));
      }
      const int t = (int)(t0 + j * R);
      tma_store_3d(&a.tm_dx, sb, cd, t, cb);
      tma_store_3d(&a.tm_dr, sb + 2 * BOX, cd, t, cb);
      tma_store_3d(&a.tm_di, sb + 3 * BOX, cd, t, cb);
      if constexpr (GATED) tma_store_3d(&a.tm_dz, sb + 4 * BOX, cd, t, cb);
      bulk_commit();
    }
    prev = st;
    if (++st == ring.S) {
      st = 0;
      phase ^= 1u;
    }
  }
  pdl_release();
  if (lane == 0) bulk_wait_all();

  double* acc = reinterpret_cast<double*>(a.ws + p.off_dlam);
  if (ch_ok) {
    if (a.dh0 != nullptr) {
#pragma unroll
      for (int v = 0; v < VEC; ++v) a.dh0[b * p.D + d0 + v] = w[v];
    }
#pragma unroll
    for (int v = 0; v < VEC; ++v) atomicAdd(acc + (b % kStripes) * p.D + d0 + v, (double)dlr[v]);
  }
  // The last block out turns the partial sums into dLambda and clears them
  // (and the exit counter) for the next backward.
  __syncwarp();
  int last = 0;
  if (lane == 0) {
    __threadfence();
    last = atomicAdd(&bh->exited, 1u) == gridDim.x - 1;
  }
  if (__shfl_sync(kFull, last, 0)) {
    __threadfence();
    for (int64_t d = lane; d < p.D; d += 32) {
      double sum = 0.0;
      for (int s2 = 0; s2 < kStripes; ++s2) {
        sum += __ldcg(&acc[s2 * p.D + d]);
        acc[s2 * p.D + d] = 0.0;
      }
      const double lam = (double)a.lambda[d];
      const double sig = 1.0 / (1.0 + exp(-lam));  // d softplus / d Lambda
      a.dlambda[d] = (float)(-(double)p.c * sig * sum);
    }
    if (lane == 0) bh->exited = 0u;
  }
}

}  // namespace blr
