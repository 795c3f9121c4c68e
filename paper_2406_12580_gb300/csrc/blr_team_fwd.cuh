// Team forward: the BD-LRU forward scan (and the gated layer's merge) in
// tiles, reading every input once and writing every output once.
//
// The life of a tile in its team:
//   scanner   loads x, rho and iota into one of the team's kTfStages ring
//             stages by TMA, with the tile's decay constants and coordinates;
//   pass A    every warp evaluates the gates of Sec. 3.2 for its slice, folds
//             it serially from a zero state (hl_t, and am_t = the product of
//             the alphas so far minus one, so that h_t = hl_t + (1 + am_t)
//             h_in), parks (hl_t, am_t) in tensor memory, off the register
//             file, and publishes the slice's map;
//   scanner   refills the stage, composes the slice maps, finds the state
//             entering the tile (its own carry, or the look-back) and hands
//             every slice its entering state;
//   pass C    one tile later: h_t = hl_t + (1 + am_t) h_in is written from
//             registers (coalesced 128-byte rows), with the state after every
//             kTeamSlice-th step kept for the backward. GATED: y = h SiLU(z)
//             instead, z read here (its box was prefetched into L2 with the
//             tile's loads).
#pragma once

#include "blr_team.cuh"

namespace blr {

constexpr int kTfStages = 2;  // ring stages of a team

struct TeamFwdArgs {
  CUtensorMap tm_x;
  CUtensorMap tm_r;
  CUtensorMap tm_i;
  CUtensorMap tm_z;  // gated: z (prefetched by box)
  Plan p;
  const int32_t* lengths;  // NULL, or row b's sequence is its last lengths[b] steps
  const float* lambda;
  const float* h0;
  const void* z;
  void* h;  // h, or y when gated; NULL: kept states and h_last only
  float* h_last;
  unsigned char* ws;
  uint32_t tag;
  uint32_t teams;  // teams at work: the stride of a team's tiles (or chains)
};

// A team's shared memory (offsets from a 128-byte aligned base; every region
// 16-byte aligned). One base register and constant offsets address all of it.
template <typename T>
struct TeamFwdSmem {
  static constexpr int NW = kTeamWidth, CHW = 32 * team_vec<T>();
  static constexpr uint32_t ring = 0;  // [stages][x, rho, iota]
  static constexpr uint32_t maps = kTfStages * 3 * kTeamBox;              // float2 [slots][NW][CHW]
  static constexpr uint32_t carry = maps + kTeamSlots * NW * CHW * 8;           // float [slots][CHW]
  static constexpr uint32_t rates = carry + kTeamSlots * CHW * 4;           // float2 [meta][32]
  static constexpr uint32_t meta = rates + kTeamMeta * 32 * 8;                  // TileMeta [meta]
  static constexpr uint32_t poly = meta + kTeamMeta * sizeof(TileMeta);         // int [meta]
  static constexpr uint32_t bars = poly + kTeamMeta * 4;                        // full, maps_ready, carry_ready, maps_read
  static constexpr uint32_t team = (bars + (kTfStages + 3 * kTeamSlots) * 8 + 127) / 128 * 128;
  static constexpr uint32_t tmem = kTeams * team;  // the block's TMEM address
  static constexpr size_t bytes = tmem + 16 + 128;
  static_assert(bytes <= 232448, "an SM's shared memory");
};

// Pass A, one part of a slice (16 TMEM columns): the gates of its rows from
// the stage, then the fold continued from (H, M), the state and the product of
// alphas minus one after the slice's earlier rows. bfloat16: 4 rows, two
// channels a lane; park[4r ..] = (H.x, M.x, H.y, M.y).
template <bool POLY, uint32_t BOX>
__device__ __forceinline__ void team_fold_bf16(const unsigned char* lb, float2 kh, float2& H,
                                               float2& M, float (&park)[16]) {
  float2 u[4], e[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const float2 hx = bf2_scaled(lds_u32(lb + s * 128), kBf2Half);
    const float2 hr = bf2_scaled(lds_u32(lb + BOX + s * 128), kBf2Half);
    const float2 hi = bf2_scaled(lds_u32(lb + 2 * BOX + s * 128), kBf2Half);
    // l = kh tanh(rho/2) + kh, e = e^l - 1
    e[s] = expm1_neg2<POLY>(__ffma2_rn(kh, tanh2(hr), kh));
    // 1 - alpha^2 = -e (e + 2); u = sqrt(1 - alpha^2) i x with i x = (x/2) tanh(iota/2) + x/2
    const float2 m2 = __fmul2_rn(e[s], __fadd2_rn(e[s], f2(2.0f)));
    u[s] = __fmul2_rn(make_float2(sqrt_approx(-m2.x), sqrt_approx(-m2.y)),
                      __ffma2_rn(hx, tanh2(hi), hx));
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const float2 alpha = __fadd2_rn(f2(1.0f), e[s]);
    H = __ffma2_rn(alpha, H, u[s]);
    M = __ffma2_rn(alpha, M, e[s]);  // alpha (1 + M) - 1
    park[4 * s] = H.x;
    park[4 * s + 1] = M.x;
    park[4 * s + 2] = H.y;
    park[4 * s + 3] = M.y;
  }
}
// float32: 8 rows of one channel, gates by row pairs; park[2r ..] = (H, M).
template <bool POLY, uint32_t BOX>
__device__ __forceinline__ void team_fold_f32(const unsigned char* lb, float2 k, float& H, float& M,
                                              float (&park)[16]) {
  float2 u[4], e[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 x = lds_rows2(lb + j * 256);
    const float2 r = sigmoid2(lds_rows2(lb + BOX + j * 256));
    const float2 i = sigmoid2(lds_rows2(lb + 2 * BOX + j * 256));
    e[j] = expm1_neg2_precise<POLY>(__fmul2_rn(k, r));
    const float2 m2 = __fmul2_rn(e[j], __fadd2_rn(e[j], f2(2.0f)));
    u[j] = __fmul2_rn(make_float2(sqrt_approx(-m2.x), sqrt_approx(-m2.y)), __fmul2_rn(i, x));
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 alpha = __fadd2_rn(f2(1.0f), e[j]);
    H = fmaf(alpha.x, H, u[j].x);
    M = fmaf(alpha.x, M, e[j].x);
    park[4 * j] = H;
    park[4 * j + 1] = M;
    H = fmaf(alpha.y, H, u[j].y);
    M = fmaf(alpha.y, M, e[j].y);
    park[4 * j + 2] = H;
    park[4 * j + 3] = M;
  }
}

template <bool V>
struct BoolC {
  static constexpr bool value = V;
};

template <typename T, bool GATED>
__global__ void __maxnreg__(kTeamMaxRegs)
    team_fwd_kernel(const __grid_constant__ TeamFwdArgs a) {
  using SM = TeamFwdSmem<T>;
  constexpr bool F32 = sizeof(T) == 4;
  constexpr int VEC = team_vec<T>(), CHW = 32 * VEC, NW = kTeamWidth;
  constexpr int S = kTfStages, MS = kTeamSlots, TS = kTeamSlice;
  constexpr uint32_t BOX = kTeamBox;
  constexpr uint32_t COLS = team_cols<T>();
  constexpr int NP = COLS / 16, PR = TS / NP;  // TMEM parts of a slice, rows per part
  static_assert(NP % 2 == 0, "pass C takes two parts at a time");
  const Plan& p = a.p;
  extern __shared__ unsigned char team_smem[];
  unsigned char* base = align128(team_smem);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(base + SM::tmem);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool scanner = warp >= kTeamWarps;
  const int team = scanner ? warp - kTeamWarps : warp / NW;
  const int ns = p.ts / TS;  // slices of a tile: the team's warps at work
  unsigned char* tb = base + (uint32_t)team * SM::team;
  unsigned char* ring = tb + SM::ring;
  float2* maps = reinterpret_cast<float2*>(tb + SM::maps);
  float* carries = reinterpret_cast<float*>(tb + SM::carry);
  float2* rates = reinterpret_cast<float2*>(tb + SM::rates);
  TileMeta* meta = reinterpret_cast<TileMeta*>(tb + SM::meta);
  int* polys = reinterpret_cast<int*>(tb + SM::poly);
  uint64_t* full = reinterpret_cast<uint64_t*>(tb + SM::bars);
  uint64_t* maps_ready = full + S;
  uint64_t* carry_ready = maps_ready + MS;
  uint64_t* maps_read = carry_ready + MS;  // pass C has read the slot's maps: it may be refilled
  const int64_t BD = p.B * p.D;
  uint32_t* err = &reinterpret_cast<FwdHeader*>(a.ws + p.off_fhdr)->err;

  if (warp == 0) {  // the block's TMEM, freed by this warp after the final barrier
    tmem_alloc(tslot, team_tmem_cols<T>());
    tmem_fence_before_sync();
  }
  if (scanner && lane == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&full[s], 1);
    for (int m = 0; m < MS; ++m) {
      mbar_init(&maps_ready[m], ns);
      mbar_init(&carry_ready[m], 1);
      mbar_init(&maps_read[m], ns);
    }
    fence_mbar_init();
    tensormap_prefetch(&a.tm_x);
    tensormap_prefetch(&a.tm_r);
    tensormap_prefetch(&a.tm_i);
    if constexpr (GATED) tensormap_prefetch(&a.tm_z);
  }
  __syncthreads();  // the roles part here and meet again at the end
  pdl_wait();
  pdl_release();
  if (blockIdx.x == 0 && warp == 0) seq_reset_workspace(a.ws, p, a.tag, lane);

  if (scanner) {
    const uint32_t teams = a.teams;
    const uint32_t n_g = (uint32_t)((p.D + CHW - 1) / CHW);
    TileWalk<false> walk(p, blockIdx.x + team * gridDim.x, teams, n_g);
    unsigned long long* agg = reinterpret_cast<unsigned long long*>(a.ws + p.off_cagg);
    uint32_t* inc = reinterpret_cast<uint32_t*>(a.ws + p.off_cinc);
    // The tile to be loaded next, and its decay constants: found ahead of time.
    TileMeta nm;
    float nk[VEC], nkh[VEC];
    bool npoly = true;
    int rgroup = -1;  // the channel group they belong to
    bool more = true;
    auto prepare = [&]() {
      nm = walk.next(p, a.lengths);
      if (!nm.end && nm.d != rgroup) {
        rgroup = nm.d;
        const int64_t d0 = nm.d + lane * VEC;
        npoly = seq_rates<VEC>(a.lambda, p.c, d0, d0 < p.D, nk, nkh);
      }
    };
    auto load = [&](uint32_t n) {  // the prepared tile, as tile n of the team
      if (!more) return;
      const uint32_t s = n % S, r = n % kTeamMeta;
      if (nm.end) {
        more = false;
        if (lane == 0) {
          meta[r].end = 1;
          mbar_arrive(&full[s]);
        }
        __syncwarp();
        return;
      }
      rates[r * 32 + lane] = team_rate<T>(nk[0], nk[VEC - 1]);
      if (lane == 0) {
        meta[r] = nm;
        polys[r] = npoly;
      }
      __syncwarp();
      if (lane == 0) {  // the arrival releases the constants and coordinates with the stage
        unsigned char* dst = ring + (size_t)s * 3 * BOX;
        mbar_arrive_expect_tx(&full[s], 3u * (uint32_t)p.ts * 128u);
        tma_load_3d(dst, &a.tm_x, &full[s], nm.d, nm.t0, nm.b);
        tma_load_3d(dst + BOX, &a.tm_r, &full[s], nm.d, nm.t0, nm.b);
        tma_load_3d(dst + 2 * BOX, &a.tm_i, &full[s], nm.d, nm.t0, nm.b);
        if constexpr (GATED) tma_prefetch_3d(&a.tm_z, nm.d, nm.t0, nm.b);
      }
    };
    prepare();
    for (int s = 0; s < S; ++s) {
      load(s);
      if (more) prepare();
    }
    float carry[VEC];  // the state after the team's last tile
#pragma unroll
    for (int v = 0; v < VEC; ++v) carry[v] = 0.0f;
    __syncwarp();
    for (uint32_t n = 0;; ++n) {
      const TileMeta tm = meta[n % kTeamMeta];
      if (tm.end) break;
      const uint32_t m = n % MS;
      const int64_t d0 = tm.d + lane * VEC;
      const bool ch_ok = d0 < p.D;
      const int64_t ch0 = (int64_t)tm.b * p.D + d0;
      float hs[VEC];
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        hs[v] = 0.0f;
        if (tm.tb == 0 && ch_ok && a.h0 != nullptr) hs[v] = a.h0[ch0 + v];
      }
      mbar_wait(&maps_ready[m], (n / MS) & 1u, err);
      float TM[VEC], TU[VEC];  // the tile's map h -> (1 + TM) h + TU
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        TM[v] = TU[v] = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const float2 e = w < ns ? maps[(m * NW + w) * CHW + lane * VEC + v] : make_float2(0.0f, 0.0f);
          TU[v] = map_apply_any(e.x, TU[v], e.y);
          TM[v] = m_compose(TM[v], e.x);
        }
      }
      const bool records = p.lookback && ch_ok, last = tm.tb + 1 == tm.ntb;  // no tile reads the last's
      const int64_t rec = (int64_t)tm.tb * BD + ch0;
      if (records && tm.tb > 0 && !last) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) st_record(&agg[rec + v], pack_agg(TM[v], TU[v]));
      }
      // pass A is done with the stage: refilled while the look-back's first reads are on their way
      auto refill = [&]() { load(n + S); };
      if (p.lookback) {
        const int64_t near = rec - BD;  // predecessors: time blocks tb - 1, tb - 2, ..., 0
        const int nprev = ch_ok ? tm.tb : 0;
        if (tm.tb == 0)
          refill();
        else
          team_lookback<VEC>(agg + near, inc + near, -BD, nprev, p.far_window != 0, err, hs, refill);
        if (records && !last) {
#pragma unroll
          for (int v = 0; v < VEC; ++v)
            st_record(&inc[rec + v], __float_as_uint(map_apply_any(TM[v], hs[v], TU[v])));
        }
      } else {
        refill();
        if (tm.tb > 0) {  // the state after the team's last tile
#pragma unroll
          for (int v = 0; v < VEC; ++v) hs[v] = carry[v];
        }
      }
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        carries[m * CHW + lane * VEC + v] = hs[v];
        carry[v] = map_apply_any(TM[v], hs[v], TU[v]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&carry_ready[m]);
      if (records) clear_records<VEC>(a.ws + p.off_cend, p, rec);  // the backward's set
      if (tm.len == 0 && a.h_last != nullptr && ch_ok) {  // an empty row: the state is unchanged
#pragma unroll
        for (int v = 0; v < VEC; ++v) a.h_last[ch0 + v] = a.h0 != nullptr ? a.h0[ch0 + v] : 0.0f;
      }
      if (more) prepare();
    }
  } else if (warp - team * NW < ns) {
    // Pass A of tile n, then pass C of tile n - 1: the scanner has tile n - 1's
    // carry ready by then, and its states' TMEM stores have long completed.
    tmem_fence_after_sync();
    const int w = warp - team * NW;
    const uint32_t tq = *tslot + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * (MS * COLS);
    float* kept = reinterpret_cast<float*>(a.ws + p.off_kept);
    const uint32_t loff = (uint32_t)w * TS * 128u + lane * 4u;  // this lane's first word
    for (uint32_t n = 0;; ++n) {
      tmem_wait_st();  // tile n - 1's park stores, before they are loaded
      const uint32_t s = n % S, m = n % MS;
      mbar_wait(&full[s], (n / S) & 1u, err);
      const bool last = meta[n % kTeamMeta].end != 0;
      if (!last) {
        // ---- A
        const unsigned char* lb = ring + s * (3 * BOX) + loff;
        const float2 k = rates[(n % kTeamMeta) * 32 + lane];
        const bool poly = polys[n % kTeamMeta] != 0;
        float2 H = f2(0.0f), M = f2(0.0f);
        __syncwarp();
#pragma unroll 1
        for (int part = 0; part < NP; ++part) {
          float park[16];
          const unsigned char* lp = lb + part * PR * 128;
          if constexpr (F32) {
            if (poly)
              team_fold_f32<true, BOX>(lp, k, H.x, M.x, park);
            else
              team_fold_f32<false, BOX>(lp, k, H.x, M.x, park);
          } else {
            if (poly)
              team_fold_bf16<true, BOX>(lp, k, H, M, park);
            else
              team_fold_bf16<false, BOX>(lp, k, H, M, park);
          }
          __syncwarp();
          tmem_st16(tq + m * COLS + part * 16, park);
        }
        if (n >= MS) mbar_wait(&maps_read[m], (n / MS - 1) & 1u, err);
        float2* mp = maps + (m * NW + w) * CHW + lane * VEC;
        mp[0] = make_float2(M.x, H.x);
        if constexpr (!F32) mp[1] = make_float2(M.y, H.y);
        __syncwarp();
        if (lane == 0) mbar_arrive(&maps_ready[m]);  // the stage is read and the map published
      }
      if (n > 0) {
        // ---- C: tile n - 1
        const uint32_t q = n - 1, mq = q % MS;
        const TileMeta tm = meta[q % kTeamMeta];
        const int rel = tm.rel0 + w * TS;
        const int rows = min(tm.len - rel, TS);
        const int d0 = tm.d + lane * VEC;
        const bool ch_ok = d0 < p.D;
        const int wrows = ch_ok && a.h != nullptr ? rows : 0;  // rows to write
        const bool whole = __all_sync(kFull, wrows == TS);
        const int64_t off = (((int64_t)tm.b * p.L + tm.t0 + w * TS) * p.D + d0) * (int64_t)sizeof(T);
        const int64_t pitch = p.D * (int64_t)sizeof(T);
        // the raw words of z of two parts' rows, a part's loads at a time
        uint32_t z0[PR], z1[PR];
        [[maybe_unused]] const unsigned char* zp = static_cast<const unsigned char*>(a.z) + off;
        [[maybe_unused]] auto z_load = [&](int part, uint32_t(&zw)[PR]) {
          if (whole) {
#pragma unroll
            for (int r = 0; r < PR; ++r) {
              zw[r] = __ldcs(reinterpret_cast<const uint32_t*>(zp));
              zp += pitch;
            }
          } else {
#pragma unroll
            for (int r = 0; r < PR; ++r) {
              zw[r] = part * PR + r < wrows ? __ldcs(reinterpret_cast<const uint32_t*>(zp)) : 0u;
              zp += pitch;
            }
          }
        };
        if constexpr (GATED) {
          z_load(0, z0);
          z_load(1, z1);
        }
        uint32_t pr0[16], pr1[16];
        __syncwarp();  // tcgen05 accesses are warp-collective
        tmem_ld16_start(tq + mq * COLS, pr0);
        mbar_wait(&carry_ready[mq], (q / MS) & 1u, err);
        // the state entering the slice: the tile's, through the slices before it
        float2 hs;
        hs.x = carries[mq * CHW + lane * VEC];
        hs.y = F32 ? hs.x : carries[mq * CHW + lane * VEC + VEC - 1];
        const float2* mp = maps + mq * NW * CHW + lane * VEC;
        for (int o = 0; o < w; ++o) {
          const float2 e0 = mp[o * CHW], e1 = mp[o * CHW + VEC - 1];
          hs = map_apply2(make_float2(e0.x, e1.x), hs, make_float2(e0.y, e1.y));
        }
        if (__any_sync(kFull, !all_finite(hs))) {
          tmem_ld_wait(pr0);
          const float2 in = make_float2(carries[mq * CHW + lane * VEC], carries[mq * CHW + lane * VEC + VEC - 1]);
          hs = team_enter_any<T>(tq + mq * COLS, mp, w, 1, in);
          tmem_ld16_start(tq + mq * COLS, pr0);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&maps_read[mq]);
        const int64_t row0 = (int64_t)tm.b * p.D + d0;  // (batch row, channel) offset of a state
        unsigned char* ph = static_cast<unsigned char*>(a.h) + off;
        float2 fin = hs;  // the state after the slice's last row
        // Parts two at a time, the next one's states on their way meanwhile; not
        // unrolled further (the instruction cache holds both passes).
        auto rows_out = [&](auto whole_c, const uint32_t(&pk)[16], int part, const uint32_t* zw) {
          constexpr bool WHOLE = decltype(whole_c)::value;
#pragma unroll
          for (int j = 0; j < 4; ++j) {  // pairs: bfloat16 row j, float32 rows 2j and 2j + 1
            const float2 o = map_apply2(
                make_float2(__uint_as_float(pk[4 * j + 1]), __uint_as_float(pk[4 * j + 3])), hs,
                make_float2(__uint_as_float(pk[4 * j]), __uint_as_float(pk[4 * j + 2])));
            float2 y = o;
            if constexpr (F32) {
              const int r = part * PR + 2 * j;
              if constexpr (GATED) {
                const float2 zv = make_float2(__uint_as_float(zw[2 * j]), __uint_as_float(zw[2 * j + 1]));
                y = __fmul2_rn(o, __fmul2_rn(zv, sigmoid2(zv)));
              }
              if (WHOLE || r < wrows) __stcs(reinterpret_cast<float*>(ph), y.x);
              ph += pitch;
              if (WHOLE || r + 1 < wrows) __stcs(reinterpret_cast<float*>(ph), y.y);
              ph += pitch;
              if (WHOLE || r + 1 < rows) fin.x = o.y;
              else if (r < rows) fin.x = o.x;
            } else {
              const int r = part * PR + j;
              if constexpr (GATED) {
                const float2 hz = bf2_scaled(zw[j], kBf2Half);
                y = __fmul2_rn(o, __ffma2_rn(hz, tanh2(hz), hz));
              }
              if (WHOLE || r < wrows) __stcs(reinterpret_cast<unsigned int*>(ph), bf2_pack(y));
              ph += pitch;
              if (WHOLE || r < rows) fin = o;
            }
          }
        };
        auto sweep = [&](auto whole_c) {
#pragma unroll 1
          for (int part = 0; part < NP; part += 2) {
            __syncwarp();
            tmem_ld_wait(pr0);
            tmem_ld16_start(tq + mq * COLS + (part + 1) * 16, pr1);
            rows_out(whole_c, pr0, part, z0);
            if constexpr (GATED) {
              if (part + 2 < NP) z_load(part + 2, z0);
            }
            __syncwarp();
            tmem_ld_wait(pr1);
            if (part + 2 < NP) tmem_ld16_start(tq + mq * COLS + (part + 2) * 16, pr0);
            rows_out(whole_c, pr1, part + 1, z1);
            if constexpr (GATED) {
              if (part + 2 < NP) z_load(part + 3, z1);
            }
          }
        };
        if (whole)
          sweep(BoolC<true>{});
        else
          sweep(BoolC<false>{});
        if (ch_ok && rows > 0) {
          const int64_t mk = rel / TS;  // the kept state of a whole slice
          if (rows == TS && mk < p.n_carry) {
            float* kp = kept + mk * BD + row0;
            if constexpr (F32)
              kp[0] = fin.x;
            else
              *reinterpret_cast<float2*>(kp) = fin;
          }
          if (a.h_last != nullptr && rel + rows == tm.len) {
            a.h_last[row0] = fin.x;
            if constexpr (!F32) a.h_last[row0 + 1] = fin.y;
          }
        }
      }
      if (last) break;
    }
    tmem_fence_before_sync();
  }
  __syncthreads();  // every role is done with the block's TMEM
  if (warp == 0) {
    tmem_fence_after_sync();
    tmem_dealloc(*tslot, team_tmem_cols<T>());
  }
}

}  // namespace blr
