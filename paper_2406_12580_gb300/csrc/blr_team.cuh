// Team kernels: what the forward (blr_team_fwd.cuh) and the backward
// (blr_team_bwd.cuh) share.
//
// They scan a problem in tiles of `ts` consecutive steps of one chain (a
// 128-byte row segment, 32 float32 or 64 bfloat16 channels of one batch row).
// A block, one per SM, holds kTeamWarps compute warps as kTeams independent
// teams of kTeamWidth warps; a team takes one tile at a time, each of its warps
// a slice of kTeamSlice steps of it, and has a scanner warp of its own that
// finds its tiles and carries the state from tile to tile. Two teams a block
// keep the SM busy while one waits for its carry.
//
// Two tile orders (Plan::lookback):
//   local     a team owns whole chains and walks the tiles of each in scan
//             order; its scanner keeps the carry in registers. Nothing waits
//             on another block. For problems with enough chains for all teams.
//   look-back tiles are numbered time-major (from the start of the sequence
//             forward, from its end backward) and team j takes tiles j,
//             j + teams, ...; the carry comes from the tiles before it in the
//             same chain by a decoupled look-back over per-(tile, channel)
//             records. All blocks are resident (a cooperative launch), and a
//             tile only waits on tiles of smaller number. For few, long chains.
//
// Products of alphas are carried as their difference from one (m = A - 1):
// with slow decays a product of a few alphas lies within 1e-3 of one, where a
// float32 holds only a few significant digits of 1 - A, which the large states
// of slow decays then multiply. A map h -> A h + U is applied as
// (m h + h) + U, and two maps compose as m = m1 + m2 + m1 m2 (the operator of
// Sec. 3.3).
//
// Records validate themselves: a record is one relaxed 32- or 64-bit store of
// a value that is never the all-ones pattern the records hold
// before the scan (A - 1 lies in [-1, 0]; a float state is never that NaN).
//
// Rows with lengths: a row's tiles count from its first real step, so padding
// is neither loaded nor stored; time blocks a row does not have are skipped.
//
// What bounds them: HBM bandwidth for float32 (8 x 8192 x 512 fwd + bwd 261 us,
// 0.84 of the measured copy rate on the compulsory bytes), and for bfloat16 a
// mix of issue slots (60 % of cycles) and bandwidth (8 x 32768 x 512 fwd + bwd
// 530 us, 0.82; with the merge 671 us, 0.83). Slices of 16 steps: the fixed cost
// of a slice (waits, TMEM transfers, map, addresses) is spread over twice the
// steps of an 8-step slice, and the kept states take half the bytes. 8 warps a
// team: one 16-warp team of 8-step slices idles whenever its carry is late.
// Loops over a slice's parts are not unrolled: unrolled, both passes and their
// variants overflow the instruction cache (forward 224 against 215 us). One base
// register and constant offsets address a team's shared memory: with a pointer
// per region the bfloat16 backward spilled in its inner loop (119 k against
// 106 k instructions a scheduler at 8 x 8192 x 512).
#pragma once

#include "blr_seq.cuh"

namespace blr {

constexpr int kTeamMeta = 4;        // tiles' coordinates and rates kept (a ring by tile)
constexpr int kTeamSlots = 2;       // maps, start values and TMEM slots of a team

constexpr int kTeams = kTeamWarps / kTeamWidth;              // teams of a block
constexpr int kTeamThreads = (kTeamWarps + kTeams) * 32;      // compute warps, a scanner warp per team
// Registers per thread: each of the SM's 4 schedulers holds a quarter of the
// 65536 registers and a quarter of the warps (rounded up); rounded down to the
// allocation granule of 8.
constexpr int kTeamMaxRegs = (16384 / (((kTeamThreads / 32 + 3) / 4) * 32)) / 8 * 8;
// Shared-memory bytes of one box: a tile's rows of 128 bytes.
constexpr uint32_t kTeamBox = kTeamWidth * kTeamSlice * 128;

template <typename T>
__host__ __device__ constexpr int team_vec() { return sizeof(T) == 4 ? 1 : 2; }
// TMEM columns a warp uses per slot: two 32-bit values per step and channel.
template <typename T>
__host__ __device__ constexpr uint32_t team_cols() { return 2u * kTeamSlice * team_vec<T>(); }
template <typename T>
__host__ __device__ constexpr uint32_t team_tmem_cols() {  // 4 warps share each lane quarter
  return 4u * kTeamSlots * team_cols<T>();
}

// The map h -> (1 + m) h + U applied to a pair of finite h, and the composition of
// the minus-one parts of two maps' products.
__device__ __forceinline__ float2 map_apply2(float2 m, float2 h, float2 U) {
  return __fadd2_rn(__ffma2_rn(m, h, h), U);
}
__device__ __forceinline__ float m_compose(float m1, float m2) { return fmaf(m1, m2, m1 + m2); }

// Infinite values. At h = +-inf the map is h + U, but m h + h is -inf + inf. The
// maps between slices and tiles test h; a slice that an infinite value enters adds
// it to its parked states (team_enter_any), so that the loop over its steps need not
// (fwd + bwd, us, without / with the tests: 12 x 1031 x 200 bfloat16 43.5 / 43.8, 8 x
// 32768 x 512 530 / 532, with the merge 674 / 669; 8 x 8192 x 512 float32 260.2 / 259.6).
__device__ __forceinline__ bool is_inf(float v) { return fabsf(v) == __int_as_float(0x7f800000); }
__device__ __forceinline__ bool all_finite(float2 v) {
  return fabsf(v.x) <= 3.402823466e38f && fabsf(v.y) <= 3.402823466e38f;
}
__device__ __forceinline__ float map_apply_any(float m, float h, float U) {
  return fmaf(m, is_inf(h) ? 0.0f : h, h) + U;
}
// The values entering a slice when they need not be finite: v, which enters the
// tile, through the n slices before this one (`maps`, CHW * dir apart). What is
// infinite of it is added to the slice's parked states (TMEM columns from tcol
// on: state and A - 1 in turn, by channels), and returned as zero.
template <typename T>
__device__ __forceinline__ float2 team_enter_any(uint32_t tcol, const float2* maps, int n, int dir, float2 v) {
  constexpr bool F32 = sizeof(T) == 4;
  constexpr int VEC = F32 ? 1 : 2, NP = 2 * kTeamSlice * VEC / 16;
#pragma unroll 1
  for (int o = 0; o < n; ++o, maps += dir * 32 * VEC) {
    v.x = map_apply_any(maps[0].x, v.x, maps[0].y);
    v.y = map_apply_any(maps[VEC - 1].x, v.y, maps[VEC - 1].y);
  }
  const bool ix = is_inf(v.x), iy = is_inf(v.y);
  __syncwarp();
#pragma unroll 1
  for (int part = 0; part < NP; ++part) {
    uint32_t r[16];
    float park[16];
    tmem_ld16_start(tcol + part * 16, r);
    tmem_ld_wait(r);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      park[j] = __uint_as_float(r[j]);
      if (j % 2 == 0) {
        if (F32 || j % 4 == 0) park[j] += ix ? v.x : -0.0f;
        else park[j] += iy ? v.y : -0.0f;
      }
    }
    tmem_st16(tcol + part * 16, park);
  }
  tmem_wait_st();
  return make_float2(ix ? 0.0f : v.x, iy ? 0.0f : v.y);
}

// ------------------------------------------------------------------ look-back

// Empties a lane's records of one tile in a set no scan uses meanwhile.
template <int VEC>
__device__ __forceinline__ void clear_records(unsigned char* set, const Plan& p, int64_t rec) {
  uint32_t* inc = reinterpret_cast<uint32_t*>(set) + rec;
  unsigned long long* agg = reinterpret_cast<unsigned long long*>(set + (p.off_cagg - p.off_cinc)) + rec;
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    inc[v] = kEmpty;
    agg[v] = ~0ull;
  }
}

// One channel's walk over the tile's nprev predecessors, nearest first: the
// q-th has its records at inc[q * step] and agg[q * step] (step = -BD when
// the predecessors are the earlier time blocks, as in the forward; +BD when
// they are the later ones, as in the backward). W predecessors are
// read in one round trip; the walk folds aggregates until it meets a published
// state. The farthest predecessor publishes only its state, so every walk ends.

template <int W>
struct LookWindow {
  uint32_t in[W];
  unsigned long long ag[W];
  __device__ __forceinline__ void load(const unsigned long long* agg, const uint32_t* inc, int64_t step,
                                       int nprev, int q0) {
#pragma unroll
    for (int q = 0; q < W; ++q) {
      in[q] = kEmpty;
      ag[q] = ~0ull;
      if (q0 + q < nprev) {
        in[q] = ld_record(inc + (q0 + q) * step);
        ag[q] = ld_record(agg + (q0 + q) * step);
      }
    }
  }
};

// The value entering the tile (its predecessors' state, or adjoint, carried
// through them), starting from the window `w` already loaded for q0 = 0. On an
// expired wait (recorded in *err) it returns what it has.
template <int W>
__device__ __forceinline__ float look_walk(const unsigned long long* agg, const uint32_t* inc,
                                           int64_t step, int nprev, uint32_t* err, LookWindow<W>& w) {
  float em = 0.0f, eu = 0.0f;  // the fold of the aggregates walked so far: h -> (1 + em) h + eu
  int q0 = 0;
  for (;;) {
    int adv = W;
    bool open = true;
#pragma unroll
    for (int q = 0; q < W; ++q) {
      if (open) {
        if (w.in[q] != kEmpty) return map_apply_any(em, __uint_as_float(w.in[q]), eu);
        if (agg_empty(w.ag[q])) {  // nothing published yet: wait for it, then re-read from it
          open = false;
          adv = q;
        } else {
          eu = map_apply_any(em, __uint_as_float((uint32_t)(w.ag[q] >> 32)), eu);
          em = m_compose(em, __uint_as_float((uint32_t)w.ag[q]));
        }
      }
    }
    q0 += adv;
    if (q0 >= nprev) return eu;  // no predecessor left (cannot happen: the farthest publishes its state)
    if (!open && !wait_record(inc + q0 * step, agg + q0 * step, err, kWaitTimeoutNs))
      return eu;  // the wait expired (recorded): finish with what is known
    w.load(agg, inc, step, nprev, q0);
  }
}

// The whole walk, kFarWindow predecessors a round trip: few chains, whose
// tiles of one round are many predecessors deep.
__device__ __noinline__ float look_far(const unsigned long long* agg, const uint32_t* inc, int64_t step,
                                       int nprev, uint32_t* err) {
  LookWindow<kFarWindow> w;
  w.load(agg, inc, step, nprev, 0);
  return look_walk<kFarWindow>(agg, inc, step, nprev, err, w);
}

// The values entering a tile for a lane's VEC channels; `meanwhile` runs while
// the first reads are on their way.
template <int VEC, typename F>
__device__ __forceinline__ void team_lookback(const unsigned long long* agg, const uint32_t* inc,
                                              int64_t step, int nprev, bool wide, uint32_t* err,
                                              float (&out)[VEC], F&& meanwhile) {
  LookWindow<kNearWindow> w[VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) w[v].load(agg + v, inc + v, step, wide ? 0 : nprev, 0);
  meanwhile();
  if (wide) {
#pragma unroll 1
    for (int v = 0; v < VEC; ++v) {
      const float t = look_far(agg + v, inc + v, step, nprev, err);
      if (v == 0) out[0] = t;
      else out[VEC - 1] = t;
    }
  } else {
#pragma unroll
    for (int v = 0; v < VEC; ++v) out[v] = look_walk<kNearWindow>(agg + v, inc + v, step, nprev, err, w[v]);
  }
}

// ----------------------------------------------------------------- tile order

struct TileMeta {
  int t0;    // the tile's first row in the tensors
  int b;     // batch row
  int d;     // first channel
  int rel0;  // its first step, counted from the row's first real step
  int len;   // the row's steps
  int tb;    // time block, counted from the row's first real step
  int ntb;   // time blocks of the row (at least one)
  int end;   // no tile: the team is done
};

// The team's position in its tile order. REV: the backward's order.
constexpr uint32_t kTeamIdle = 0xffffffffu;
template <bool REV>
struct TileWalk {
  uint32_t chain, q;       // the next tile: its chain and time block in scan order
  uint32_t step_q, step_r;  // look-back: teams = step_q chains' worth of tiles + step_r
  uint32_t teams, n_g;

  __device__ __forceinline__ TileWalk(const Plan& p, uint32_t team, uint32_t teams_, uint32_t n_g_)
      : chain(team), q(0), step_q(0), step_r(0), teams(teams_), n_g(n_g_) {
    const uint32_t C = (uint32_t)p.n_chain;
    if (team >= teams_) {
      q = kTeamIdle;
    } else if (p.lookback) {
      step_q = teams_ / C;
      step_r = teams_ - step_q * C;
      q = team / C;
      chain = team - q * C;
    }
  }

  __device__ __forceinline__ TileMeta next(const Plan& p, const int32_t* lengths) {
    TileMeta m;
    m.t0 = m.b = m.d = m.rel0 = m.len = m.tb = m.ntb = 0;
    m.end = 1;
    const uint32_t C = (uint32_t)p.n_chain, ts = (uint32_t)p.ts;
    for (;;) {
      if (q == kTeamIdle) return m;
      if (p.lookback ? q >= (uint32_t)p.n_tc : chain >= C) return m;
      const uint32_t ch = chain, tq = q;
      const uint32_t b = ch / n_g;
      uint32_t start = 0, ntb = (uint32_t)p.n_tc;
      if (lengths != nullptr) {
        start = (uint32_t)row_start(lengths, b, p.L);
        ntb = ((uint32_t)p.L - start + ts - 1) / ts;
        if (ntb == 0) ntb = 1;
      }
      if (p.lookback) {
        q += step_q;
        chain += step_r;
        if (chain >= C) {
          chain -= C;
          ++q;
        }
      } else if (++q >= ntb) {  // the chain's last tile: on to the team's next chain
        q = 0;
        chain += teams;
      }
      if (tq >= ntb) continue;  // look-back: a time block this row does not have
      m.tb = (int)(REV ? ntb - 1 - tq : tq);
      m.b = (int)b;
      m.d = (int)(ch - b * n_g) * 32 * p.sv;
      m.rel0 = m.tb * (int)ts;
      m.t0 = (int)start + m.rel0;
      m.len = (int)((uint32_t)p.L - start);
      m.ntb = (int)ntb;
      m.end = 0;
      return m;
    }
  }
};

// ----------------------------------------------------------------- gate pairs
//
// A bfloat16 lane's two channels of one row, or a float32 lane's channel in
// two consecutive rows.

__device__ __forceinline__ float2 lds_rows2(const unsigned char* p) {  // a channel's two rows
  return make_float2(*reinterpret_cast<const float*>(p), *reinterpret_cast<const float*>(p + 128));
}
__device__ __forceinline__ uint32_t lds_u32(const unsigned char* p) {
  return *reinterpret_cast<const uint32_t*>(p);
}

// Decay constants of a lane's channels as the gate pairs take them: bfloat16
// (k/2 of both channels), float32 (k twice); both as stored by the scanner.
template <typename T>
__device__ __forceinline__ float2 team_rate(float k0, float k1) {
  if constexpr (sizeof(T) == 4) return make_float2(k0, k0);
  return make_float2(0.5f * k0, 0.5f * k1);
}

}  // namespace blr
