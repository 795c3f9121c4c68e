// Team backward: the BD-LRU backward scan (and the gated layer's merge) in the
// forward's tiles, last tile of a chain first, reading every input from HBM
// once and writing every output once.
//
// With g_t the total derivative with respect to h_t and w_t = alpha_t g_t the
// adjoint passed to step t - 1, the reverse recurrence g_t = dh_t + w_{t+1}
// (w_L = dh_last) is again a first-order linear scan (Sec. 3.3's operator,
// run from the end): over a run of steps, w leaving its left end is an affine
// map w -> A w + W of the w entering its right end, A the product of the run's
// alphas. The life of a tile in its team:
//   scanner   announces the tile (its coordinates and decay constants) two
//             tiles ahead;
//   pass A    every warp evaluates the alphas of its slice and folds the
//             reverse recurrence from a zero adjoint, last step first (gl_t,
//             and sm_t = the product of the alphas after step t within the
//             slice minus one, so that g_t = gl_t + (1 + sm_t) w_in), parks
//             both in tensor memory and publishes the slice's map. Every warp
//             has its own slice of dh and rho (GATED: dy, rho and z; ring A),
//             and requests the next tile's as soon as it has read it;
//   scanner   composes the slice maps and finds the adjoint entering the tile
//             (the carry of the team's last tile, or the look-back);
//   pass C    one tile later, forward in time from the forward's kept state:
//             each step's gates once, h_{t-1}, g_t and every output (dx,
//             d rho, d iota and the d Lambda terms) in one sweep, the outputs
//             written over the step's consumed inputs. Every warp has its own
//             slice of x, rho and iota (ring C) and moves it by itself: a TMA
//             store sends the outputs out, and during the next pass A, when
//             the store has read them, the next tile's slice is requested.
//             GATED: dz = dy SiLU'(z) h is written directly, dy SiLU'(z) having
//             been parked by pass A.
// The gradient formulas are those of the serial backward kernels (the chain
// rule of Sec. 3.2's definitions).
//
// Rings a warp moves by itself: a warp that has read its slice requests the
// next at once, where a tile-wide stage waits for its slowest warp (8 x 32768 x
// 512 bfloat16: 386 -> 340 us; 8 x 8192 x 512 float32: 193 -> 172). No L2
// prefetches of the tiles ahead: at 128-byte rows the TMA units bind, and the
// prefetches slow the loads that are needed sooner (float32 193 against 172 us).
// d Lambda: a warp sums its channels over its tiles in float64 in shared
// memory, and teams stay within one channel group where they can, so that a
// team adds to the workspace once: with an atomic per slice, 300 x 1500 x 64
// (512 addresses) took 158 us against 92.
#pragma once

#include "blr_team_fwd.cuh"

namespace blr {

struct TeamBwdArgs {
  CUtensorMap tm_dh;  // dh, or dy when gated; all in boxes of one slice
  CUtensorMap tm_x;
  CUtensorMap tm_r;
  CUtensorMap tm_i;
  CUtensorMap tm_z;  // gated: z
  CUtensorMap tm_dx;
  CUtensorMap tm_dr;
  CUtensorMap tm_di;
  Plan p;
  const int32_t* lengths;  // as TeamFwdArgs
  void* dz;                // gated
  const float* dh_last;
  const float* lambda;
  const float* h0;
  float* dlambda;
  float* dh0;
  unsigned char* ws;
  uint32_t tag;
  uint32_t teams;  // as TeamFwdArgs
};

// A team's shared memory, as TeamFwdSmem.
template <typename T, bool GATED>
struct TeamBwdSmem {
  static constexpr int NW = kTeamWidth, CHW = 32 * team_vec<T>();
  static constexpr int NBA = GATED ? 3 : 2;                                     // boxes of ring A
  static constexpr uint32_t ringA = 0;                                          // [dh, rho (, z)]
  static constexpr uint32_t ringC = NBA * kTeamBox;                       // [x, rho, iota]
  static constexpr uint32_t maps = ringC + 3 * kTeamBox;                  // float2 [slots][NW][CHW]
  static constexpr uint32_t carry = maps + kTeamSlots * NW * CHW * 8;           // float [slots][CHW]
  static constexpr uint32_t dsum = carry + kTeamSlots * CHW * 4;            // double [NW][CHW]
  static constexpr uint32_t rates = dsum + NW * CHW * 8;                        // float2 [meta][32]
  static constexpr uint32_t meta = rates + kTeamMeta * 32 * 8;                  // TileMeta [meta]
  static constexpr uint32_t poly = meta + kTeamMeta * sizeof(TileMeta);         // int [meta]
  static constexpr uint32_t bars = poly + kTeamMeta * 4;  // fullA, fullC, known, maps_ready, carry_ready, maps_read
  static constexpr uint32_t team = (bars + (kTeamMeta + 2 * NW + 3 * kTeamSlots) * 8 + 127) / 128 * 128;
  static constexpr uint32_t tmem = kTeams * team;  // the block's TMEM address
  static constexpr size_t bytes = tmem + 16 + 128;
  static_assert(bytes <= 232448, "an SM's shared memory");
};

// Pass A, one part of a slice (16 TMEM columns), last row first; rows from
// `valid` on lie past the sequence and act as the identity (alpha = 1,
// dh = 0). (w, m): the fold of the slice's later rows, zero at the slice's
// end; on return the map of the rows folded so far. GATED: dh = dy SiLU(z), and
// merge gets dy SiLU'(z) of every element. bfloat16: 4 rows, two channels a
// lane, park[4r ..] = (g.x, sm.x, g.y, sm.y). ROUND: the merge as an operator of
// its own would hand dh on, with the sigmoid of float32 data and dh rounded to
// bfloat16: so the float32 gradients (d Lambda, dh0) of small problems, whose
// merge is defined that way, do not depend on how it is computed (with tanh and
// an unrounded dh they lie up to 3e-3 elsewhere).
template <bool FAST, bool GATED, bool ROUND, uint32_t BOX>
__device__ __forceinline__ void team_rfold_bf16(const unsigned char* lb, float2 kh, int valid,
                                                float2& w, float2& m, float (&park)[16],
                                                float (&merge)[8]) {
#pragma unroll
  for (int r = 3; r >= 0; --r) {
    float2 dh = bf2_unpack(lds_u32(lb + r * 128));
    if constexpr (ROUND) {
      const float2 z = bf2_unpack(lds_u32(lb + 2 * BOX + r * 128)), sg = sigmoid2(z), f = __fmul2_rn(z, sg);
      const float2 pd = __fmul2_rn(dh, __ffma2_rn(sg, __ffma2_rn(f2(-1.0f), f, z), sg));
      merge[2 * r] = pd.x;
      merge[2 * r + 1] = pd.y;
      dh = bf2_unpack(bf2_pack(__fmul2_rn(dh, f)));
    } else if constexpr (GATED) {  // with hz = z/2 and th = tanh(hz), as silu_grad
      const float2 hz = bf2_scaled(lds_u32(lb + 2 * BOX + r * 128), kBf2Half), th = tanh2(hz);
      const float2 sg = __ffma2_rn(f2(0.5f), th, f2(0.5f));
      const float2 f = __ffma2_rn(hz, th, hz);
      const float2 df = __ffma2_rn(sg, __ffma2_rn(__fmul2_rn(f2(-1.0f), hz), th, hz), sg);
      const float2 pd = __fmul2_rn(dh, df);
      merge[2 * r] = pd.x;
      merge[2 * r + 1] = pd.y;
      dh = __fmul2_rn(dh, f);
    }
    const float2 hr = bf2_scaled(lds_u32(lb + BOX + r * 128), kBf2Half);
    float2 e = expm1_neg2<FAST>(__ffma2_rn(kh, tanh2(hr), kh));
    if (!FAST && r >= valid) {
      e = f2(0.0f);
      dh = f2(0.0f);
    }
    const float2 g = __fadd2_rn(dh, w);
    park[4 * r] = g.x;
    park[4 * r + 1] = m.x;
    park[4 * r + 2] = g.y;
    park[4 * r + 3] = m.y;
    const float2 alpha = __fadd2_rn(f2(1.0f), e);
    m = __ffma2_rn(alpha, m, e);  // alpha (1 + m) - 1
    w = __fmul2_rn(alpha, g);
  }
}
// float32: 8 rows of one channel by row pairs; park[2r ..] = (g, sm).
template <bool FAST, bool GATED, uint32_t BOX>
__device__ __forceinline__ void team_rfold_f32(const unsigned char* lb, float2 k, int valid,
                                               float& w, float& m, float (&park)[16],
                                               float (&merge)[8]) {
#pragma unroll
  for (int j = 3; j >= 0; --j) {
    float2 dh = lds_rows2(lb + j * 256);
    if constexpr (GATED) {
      const float2 z = lds_rows2(lb + 2 * BOX + j * 256), sg = sigmoid2(z), f = __fmul2_rn(z, sg);
      const float2 pd = __fmul2_rn(dh, __ffma2_rn(sg, __ffma2_rn(f2(-1.0f), f, z), sg));
      merge[2 * j] = pd.x;
      merge[2 * j + 1] = pd.y;
      dh = __fmul2_rn(dh, f);
    }
    float2 e = expm1_neg2_precise<FAST>(__fmul2_rn(k, sigmoid2(lds_rows2(lb + BOX + j * 256))));
    if (!FAST && 2 * j >= valid) e.x = dh.x = 0.0f;
    if (!FAST && 2 * j + 1 >= valid) e.y = dh.y = 0.0f;
    const float2 alpha = __fadd2_rn(f2(1.0f), e);
    float g = dh.y + w;
    park[4 * j + 2] = g;
    park[4 * j + 3] = m;
    m = fmaf(alpha.y, m, e.y);
    w = alpha.y * g;
    g = dh.x + w;
    park[4 * j] = g;
    park[4 * j + 1] = m;
    m = fmaf(alpha.x, m, e.x);
    w = alpha.x * g;
  }
}

// Pass C, one part of a slice: its rows forward in time from the state hp
// before them (updated), with the parked (gl, sm) in pr and the adjoint win
// entering the slice; dx, d rho and d iota overwrite x, rho and iota in the
// stage (the TMA store clips rows past the sequence); rows from `rows` on are
// not summed. Adds the d Lambda terms dl_t r_t to dlr. Gated: dz rows to `dz`,
// moved on. FAST: the whole slice
// inside the sequence and every l in the series' range.
template <bool FAST, bool GATED, uint32_t BOX>
__device__ __forceinline__ void team_rows_bf16(unsigned char* lb, const uint32_t (&pr)[16], float2 win,
                                               float2 kh, int rows, float2& hp, float2& dlr,
                                               const uint32_t (&merge)[8], unsigned char*& dz, int64_t pitch) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float2 gl = make_float2(__uint_as_float(pr[4 * r]), __uint_as_float(pr[4 * r + 2]));
    const float2 sm = make_float2(__uint_as_float(pr[4 * r + 1]), __uint_as_float(pr[4 * r + 3]));
    const float2 nhx = bf2_scaled(lds_u32(lb + r * 128), kBf2NegHalf);
    const float2 thr = tanh2(bf2_scaled(lds_u32(lb + BOX + r * 128), kBf2Half));
    const float2 thi = tanh2(bf2_scaled(lds_u32(lb + 2 * BOX + r * 128), kBf2Half));
    const float2 l = __ffma2_rn(kh, thr, kh);  // log alpha = k r
    const float2 e = expm1_neg2<FAST>(l);
    const float2 alpha = __fadd2_rn(f2(1.0f), e);
    const float2 m2 = __fmul2_rn(e, __fadd2_rn(e, f2(2.0f)));  // -(1 - alpha^2)
    const float2 rs = make_float2(rsqrt_approx(fmaxf(-m2.x, 1e-30f)), rsqrt_approx(fmaxf(-m2.y, 1e-30f)));
    const float2 nq = __fmul2_rn(m2, rs);                // -sqrt(1 - alpha^2)
    const float2 nix = __ffma2_rn(nhx, thi, nhx);        // -i x
    const float2 g = map_apply2(sm, win, gl);            // g_t = gl_t + (1 + sm_t) w_in
    const float2 w = __fmul2_rn(alpha, g);
    const float2 gnq = __fmul2_rn(g, nq);                // -g sqrt(1 - alpha^2)
    const float2 ni = __ffma2_rn(f2(-0.5f), thi, f2(-0.5f));  // -i
    const float2 omi = __ffma2_rn(f2(-0.5f), thi, f2(0.5f));  // 1 - i
    // dx = g sqrt(1 - alpha^2) i; d iota = g u (1 - i);
    // d l = alpha g (h_{t-1} - alpha i x / sqrt(1 - alpha^2)); d rho = d l k r (1 - r) = d l l (1 - r)
    const float2 ox = __fmul2_rn(gnq, ni);
    const float2 oi = __fmul2_rn(__fmul2_rn(gnq, nix), omi);
    const float2 dl = __fmul2_rn(w, __ffma2_rn(__fmul2_rn(alpha, rs), nix, hp));
    const float2 orho = __fmul2_rn(__fmul2_rn(dl, l), __ffma2_rn(f2(-0.5f), thr, f2(0.5f)));
    hp = __ffma2_rn(alpha, hp, __fmul2_rn(nq, nix));  // alpha h + sqrt(1 - alpha^2) i x
    *reinterpret_cast<uint32_t*>(lb + r * 128) = bf2_pack(ox);
    *reinterpret_cast<uint32_t*>(lb + BOX + r * 128) = bf2_pack(orho);
    *reinterpret_cast<uint32_t*>(lb + 2 * BOX + r * 128) = bf2_pack(oi);
    if (FAST || r < rows) {
      dlr = __ffma2_rn(dl, __ffma2_rn(f2(0.5f), thr, f2(0.5f)), dlr);  // += d l r
      if constexpr (GATED) {  // dz = dy SiLU'(z) h
        const float2 pd = make_float2(__uint_as_float(merge[2 * r]), __uint_as_float(merge[2 * r + 1]));
        __stcs(reinterpret_cast<unsigned int*>(dz), bf2_pack(__fmul2_rn(pd, hp)));
      }
    }
    if constexpr (GATED) dz += pitch;
  }
}
template <bool FAST, bool GATED, uint32_t BOX>
__device__ __forceinline__ void team_rows_f32(unsigned char* lb, const uint32_t (&pr)[16], float win,
                                              float2 k, int rows, float& hp, float& dlr,
                                              const uint32_t (&merge)[8], unsigned char*& dz, int64_t pitch) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 gl = make_float2(__uint_as_float(pr[4 * j]), __uint_as_float(pr[4 * j + 2]));
    const float2 sm = make_float2(__uint_as_float(pr[4 * j + 1]), __uint_as_float(pr[4 * j + 3]));
    const float2 x = lds_rows2(lb + j * 256);
    const float2 r = sigmoid2(lds_rows2(lb + BOX + j * 256));
    const float2 i = sigmoid2(lds_rows2(lb + 2 * BOX + j * 256));
    const float2 e = expm1_neg2_precise<FAST>(__fmul2_rn(k, r));
    const float2 alpha = __fadd2_rn(f2(1.0f), e);
    const float2 m2 = __fmul2_rn(e, __fadd2_rn(e, f2(2.0f)));  // -(1 - alpha^2)
    const float2 rs = make_float2(rsqrt_approx(fmaxf(-m2.x, 1e-30f)), rsqrt_approx(fmaxf(-m2.y, 1e-30f)));
    const float2 n = make_float2(-m2.x * rs.x, -m2.y * rs.y);  // sqrt(1 - alpha^2)
    const float2 ix = __fmul2_rn(i, x);
    const float2 u = __fmul2_rn(n, ix);
    const float2 g = map_apply2(sm, f2(win), gl);
    const float2 w = __fmul2_rn(alpha, g);
    const float h0 = hp, h1 = fmaf(alpha.x, h0, u.x);
    hp = fmaf(alpha.y, h1, u.y);
    const float2 ox = __fmul2_rn(__fmul2_rn(g, n), i);
    const float2 oi = __fmul2_rn(__fmul2_rn(g, u), __ffma2_rn(f2(-1.0f), i, f2(1.0f)));
    const float2 ars = __fmul2_rn(alpha, rs);
    const float2 dl = make_float2(w.x * fmaf(-ars.x, ix.x, h0), w.y * fmaf(-ars.y, ix.y, h1));
    const float2 orho = __fmul2_rn(__fmul2_rn(dl, k), make_float2(fmaf(-r.x, r.x, r.x), fmaf(-r.y, r.y, r.y)));
    float* sx = reinterpret_cast<float*>(lb + j * 256);
    sx[0] = ox.x;
    sx[32] = ox.y;
    float* sr = reinterpret_cast<float*>(lb + BOX + j * 256);
    sr[0] = orho.x;
    sr[32] = orho.y;
    float* si = reinterpret_cast<float*>(lb + 2 * BOX + j * 256);
    si[0] = oi.x;
    si[32] = oi.y;
    float2 oz = f2(0.0f);
    if constexpr (GATED) {  // dz = dy SiLU'(z) h
      const float2 pd = make_float2(__uint_as_float(merge[2 * j]), __uint_as_float(merge[2 * j + 1]));
      oz = __fmul2_rn(pd, make_float2(h1, hp));
    }
    if (FAST || 2 * j < rows) {
      dlr = fmaf(dl.x, r.x, dlr);
      if constexpr (GATED) __stcs(reinterpret_cast<float*>(dz), oz.x);
    }
    if constexpr (GATED) dz += pitch;
    if (FAST || 2 * j + 1 < rows) {
      dlr = fmaf(dl.y, r.y, dlr);
      if constexpr (GATED) __stcs(reinterpret_cast<float*>(dz), oz.y);
    }
    if constexpr (GATED) dz += pitch;
  }
}

// ROUND: as team_rfold_bf16 (bfloat16 with the merge only).
template <typename T, bool GATED, bool ROUND>
__global__ void __maxnreg__(kTeamMaxRegs)
    team_bwd_kernel(const __grid_constant__ TeamBwdArgs a) {
  using SM = TeamBwdSmem<T, GATED>;
  constexpr bool F32 = sizeof(T) == 4;
  constexpr int VEC = team_vec<T>(), CHW = 32 * VEC, NW = kTeamWidth;
  constexpr int MS = kTeamSlots, TS = kTeamSlice, NBA = SM::NBA;
  constexpr uint32_t BOX = kTeamBox;
  // TMEM columns of a slot: the parked (gl, sm), and dy SiLU'(z) when gated. Two
  // slots let pass C run a tile behind pass A; the gated bfloat16 states take
  // more than half of the TMEM, so there pass C follows its own pass A and the
  // block's other team fills the wait for the carry.
  constexpr uint32_t COLS = team_cols<T>() + (GATED ? TS * VEC : 0);
  constexpr int LAG = GATED && !F32 ? 0 : 1;
  constexpr uint32_t TSLOTS = LAG + 1;
  constexpr uint32_t TCOLS = 4 * TSLOTS * COLS <= 256 ? 256 : 512;
  constexpr int NP = team_cols<T>() / 16, PR = TS / NP;  // TMEM parts of a slice, rows per part
  static_assert(PR * VEC == 8 && 4 * TSLOTS * COLS <= TCOLS, "a part's merge values are 8 columns");
  const Plan& p = a.p;
  extern __shared__ unsigned char team_smem[];
  unsigned char* base = align128(team_smem);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(base + SM::tmem);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool scanner = warp >= kTeamWarps;
  const int team = scanner ? warp - kTeamWarps : warp / NW;
  const int ns = p.ts / TS;  // slices of a tile: the team's warps at work
  unsigned char* tb = base + (uint32_t)team * SM::team;
  float2* maps = reinterpret_cast<float2*>(tb + SM::maps);
  float* carries = reinterpret_cast<float*>(tb + SM::carry);
  float2* rates = reinterpret_cast<float2*>(tb + SM::rates);
  TileMeta* meta = reinterpret_cast<TileMeta*>(tb + SM::meta);
  int* polys = reinterpret_cast<int*>(tb + SM::poly);
  uint64_t* fullA = reinterpret_cast<uint64_t*>(tb + SM::bars);
  uint64_t* fullC = fullA + NW;   // one of each per warp
  uint64_t* known = fullC + NW;   // a tile's coordinates and decay constants are written
  uint64_t* maps_ready = known + kTeamMeta;
  uint64_t* carry_ready = maps_ready + MS;
  uint64_t* maps_read = carry_ready + MS;  // pass C has read the slot's maps: it may be refilled
  const int64_t BD = p.B * p.D;
  FwdHeader* fh = reinterpret_cast<FwdHeader*>(a.ws + p.off_fhdr);
  BwdHeader* bh = reinterpret_cast<BwdHeader*>(a.ws + p.off_bhdr);
  uint32_t* err = &fh->err;

  if (scanner && lane == 0) {
    for (int w = 0; w < NW; ++w) {
      mbar_init(&fullA[w], 1);
      mbar_init(&fullC[w], 1);
    }
    for (int r = 0; r < kTeamMeta; ++r) mbar_init(&known[r], 1);
    for (int m = 0; m < MS; ++m) {
      mbar_init(&maps_ready[m], ns);
      mbar_init(&carry_ready[m], 1);
      mbar_init(&maps_read[m], ns);
    }
    fence_mbar_init();
    tensormap_prefetch(&a.tm_dh);
    tensormap_prefetch(&a.tm_x);
    tensormap_prefetch(&a.tm_r);
    tensormap_prefetch(&a.tm_i);
    if constexpr (GATED) tensormap_prefetch(&a.tm_z);
  }
  pdl_wait();
  pdl_release();
  __shared__ uint32_t s_set;  // the record set to use; changed by the last block out only
  {
    __shared__ int s_ok;
    if (threadIdx.x == 0) {  // one round trip: no load waits for another
      const uint32_t tag = __ldcg(&fh->tag), complete = __ldcg(&fh->complete), set = __ldcg(&bh->set);
      s_ok = tag == a.tag && complete == 1u;
      s_set = set & 1u;
      if (!s_ok) atomicOr(&fh->err, kErrWorkspace);
    }
    __syncthreads();
    if (!s_ok) return;  // no forward states for this problem: write nothing
  }
  if (warp == 0) {  // the block's TMEM, freed by this warp after the final barrier
    tmem_alloc(tslot, TCOLS);
    tmem_fence_before_sync();
  }
  __syncthreads();  // the roles part here and meet again at the end

  double* acc = reinterpret_cast<double*>(a.ws + p.off_dlam);
  double* dsums = reinterpret_cast<double*>(tb + SM::dsum);  // [NW][CHW]
  int dgroup = -1;  // compute warps: the channel group of their d Lambda sums
  // Sums of a lane's channels into the workspace (striped over teams).
  auto dlam_add = [&](double* to, int d0, const double* sum) {
    if (d0 < p.D) {
      double* ad = to + ((blockIdx.x + team * gridDim.x) % kStripes) * p.D + d0;
#pragma unroll
      for (int v = 0; v < VEC; ++v) atomicAdd(ad + v, sum[v]);  // reductions without a result
    }
  };

  if (scanner) {
    const uint32_t teams = a.teams;
    const uint32_t n_g = (uint32_t)((p.D + CHW - 1) / CHW);
    TileWalk<true> walk(p, blockIdx.x + team * gridDim.x, teams, n_g);
    const uint32_t set = s_set;
    unsigned char* recs = a.ws + (set ? p.off_cinc : p.off_cend);
    unsigned char* spare = a.ws + (set ? p.off_cend : p.off_cinc);  // emptied for the next backward
    uint32_t* inc = reinterpret_cast<uint32_t*>(recs);
    unsigned long long* agg = reinterpret_cast<unsigned long long*>(recs + (p.off_cagg - p.off_cinc));
    TileMeta nm;  // the tile to be loaded next, and its decay constants
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
    auto announce = [&](uint32_t n) {  // the prepared tile, as tile n of the team
      if (!more) return;
      const uint32_t r = n % kTeamMeta;
      more = !nm.end;
      if (more) rates[r * 32 + lane] = team_rate<T>(nk[0], nk[VEC - 1]);
      if (lane == 0) {
        meta[r] = nm;
        polys[r] = npoly;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&known[r]);
    };
    prepare();
    for (int s = 0; s < 2; ++s) {
      announce(s);
      if (more) prepare();
    }
    float carry[VEC];  // the adjoint leaving the team's last tile
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
      float ws[VEC];
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        ws[v] = 0.0f;
        if (tm.tb == tm.ntb - 1 && ch_ok && a.dh_last != nullptr)  // the row's last tile
          ws[v] = a.dh_last[ch0 + v];
      }
      mbar_wait(&maps_ready[m], (n / MS) & 1u, err);
      float TM[VEC], TU[VEC];  // the tile's map: its slices from the last to the first
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        TM[v] = TU[v] = 0.0f;
#pragma unroll
        for (int w = NW - 1; w >= 0; --w) {
          const float2 e = w < ns ? maps[(m * NW + w) * CHW + lane * VEC + v] : make_float2(0.0f, 0.0f);
          TU[v] = map_apply_any(e.x, TU[v], e.y);
          TM[v] = m_compose(TM[v], e.x);
        }
      }
      const bool records = p.lookback && ch_ok, last = tm.tb == 0;  // no tile reads the last's
      const int64_t rec = (int64_t)tm.tb * BD + ch0;
      const int nprev = tm.ntb - 1 - tm.tb;  // predecessors: time blocks tb + 1, tb + 2, ..., ntb - 1
      if (records && nprev > 0 && !last) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) st_record(&agg[rec + v], pack_agg(TM[v], TU[v]));
      }
      // tile n + 2 is announced while the look-back's first reads are on their way
      auto ahead = [&]() { announce(n + 2); };
      if (p.lookback) {
        const int64_t near = rec + BD;
        if (nprev == 0)
          ahead();
        else
          team_lookback<VEC>(agg + near, inc + near, BD, ch_ok ? nprev : 0, p.far_window != 0, err, ws, ahead);
        if (records && !last) {
#pragma unroll
          for (int v = 0; v < VEC; ++v)
            st_record(&inc[rec + v], __float_as_uint(map_apply_any(TM[v], ws[v], TU[v])));
        }
      } else {
        ahead();
        if (nprev > 0) {  // the adjoint leaving the team's last tile
#pragma unroll
          for (int v = 0; v < VEC; ++v) ws[v] = carry[v];
        }
      }
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        carries[m * CHW + lane * VEC + v] = ws[v];
        carry[v] = map_apply_any(TM[v], ws[v], TU[v]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&carry_ready[m]);
      if (records) clear_records<VEC>(spare, p, rec);
      if (last && a.dh0 != nullptr && ch_ok) {  // the adjoint leaving the row's first step
#pragma unroll
        for (int v = 0; v < VEC; ++v) a.dh0[ch0 + v] = carry[v];
      }
      if (more) prepare();
    }
  } else if (warp - team * NW < ns) {
    // Pass A of tile n, then pass C of tile n - 1 (as the forward).
    tmem_fence_after_sync();
    const int w = warp - team * NW;
    const uint32_t tq = *tslot + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * (TSLOTS * COLS);
    const float* kept = reinterpret_cast<const float*>(a.ws + p.off_kept);
    unsigned char* wb = tb + (uint32_t)w * (TS * 128u);  // this warp's slices of the rings
    auto load_a = [&](uint32_t n) {  // tile n's dh and rho (gated: dy, rho and z), if there is one
      mbar_wait(&known[n % kTeamMeta], (n / kTeamMeta) & 1u, err);
      const TileMeta* t = &meta[n % kTeamMeta];
      if (t->end) {
        mbar_arrive(&fullA[w]);
        return;
      }
      const int row = t->t0 + w * TS, d = t->d, b = t->b;
      mbar_arrive_expect_tx(&fullA[w], (uint32_t)NBA * TS * 128u);
      tma_load_3d(wb + SM::ringA, &a.tm_dh, &fullA[w], d, row, b);
      tma_load_3d(wb + SM::ringA + BOX, &a.tm_r, &fullA[w], d, row, b);
      if constexpr (GATED) tma_load_3d(wb + SM::ringA + 2 * BOX, &a.tm_z, &fullA[w], d, row, b);
    };
    auto load_c = [&](uint32_t n) {  // tile n's x, rho and iota
      const TileMeta* t = &meta[n % kTeamMeta];
      const int row = t->t0 + w * TS, d = t->d, b = t->b;
      mbar_arrive_expect_tx(&fullC[w], 3u * TS * 128u);
      tma_load_3d(wb + SM::ringC, &a.tm_x, &fullC[w], d, row, b);
      tma_load_3d(wb + SM::ringC + BOX, &a.tm_r, &fullC[w], d, row, b);
      tma_load_3d(wb + SM::ringC + 2 * BOX, &a.tm_i, &fullC[w], d, row, b);
    };
    if (lane == 0) load_a(0);
    __syncwarp();
    float2 hp = f2(0.0f);  // tile n - 1: the state before this slice
    for (uint32_t n = 0;; ++n) {
      tmem_wait_st();  // tile n - 1's park stores, before they are loaded
      const uint32_t m = n % MS;
      mbar_wait(&fullA[w], n & 1u, err);
      const TileMeta tm = meta[n % kTeamMeta];
      float2 nhp = f2(0.0f);
      if (lane == 0) {
        if (n == 0 && !tm.end) load_c(0);
        if (LAG == 1 && tm.end && n >= 2) {  // no pass A left to hide this in
          bulk_wait_read<0>();
          load_c(n - 1);
        }
      }
      __syncwarp();
      if (!tm.end) {
        // ---- A
        const int rel = tm.rel0 + w * TS;
        const int valid = min(max(tm.len - rel, 0), TS);
        // the state before this slice, for its pass C: kept state rel / TS - 1 (h0 for the first)
        const int d0 = tm.d + lane * VEC;
        if (d0 < p.D && valid > 0) {
          const int64_t row0 = (int64_t)tm.b * p.D + d0;
          const float* src = rel > 0 ? kept + (int64_t)(rel / TS - 1) * BD + row0
                                     : (a.h0 != nullptr ? a.h0 + row0 : nullptr);
          if (src != nullptr) {
            nhp.x = __ldcg(src);
            if constexpr (!F32) nhp.y = __ldcg(src + 1);
          }
        }
        const unsigned char* lb = wb + SM::ringA + lane * 4u;
        const float2 k = rates[(n % kTeamMeta) * 32 + lane];
        const bool poly = polys[n % kTeamMeta] != 0;
        float2 W = f2(0.0f), M = f2(0.0f);
        auto fold = [&](auto fast_c) {
          constexpr bool FAST = decltype(fast_c)::value;
#pragma unroll 1  // the instruction cache holds both passes
          for (int part = NP - 1; part >= 0; --part) {
            float park[16], merge[8];
            const unsigned char* lp = lb + part * PR * 128;
            if constexpr (F32)
              team_rfold_f32<FAST, GATED, BOX>(lp, k, valid - part * PR, W.x, M.x, park, merge);
            else
              team_rfold_bf16<FAST, GATED, ROUND, BOX>(lp, k, valid - part * PR, W, M, park, merge);
            __syncwarp();
            const uint32_t to = tq + (n % TSLOTS) * COLS;
            tmem_st16(to + part * 16, park);
            if constexpr (GATED) tmem_st8(to + team_cols<T>() + part * 8, merge);
            // the outputs of the last pass C have been read by now: the next one's inputs
            if (part == NP / 2 && n >= 1 + LAG && lane == 0) {
              bulk_wait_read<0>();
              load_c(n - LAG);
            }
          }
        };
        __syncwarp();
        if (poly && valid == TS)
          fold(BoolC<true>{});
        else
          fold(BoolC<false>{});
        if (n >= MS) mbar_wait(&maps_read[m], (n / MS - 1) & 1u, err);
        float2* mp = maps + (m * NW + w) * CHW + lane * VEC;
        mp[0] = make_float2(M.x, W.x);
        if constexpr (!F32) mp[1] = make_float2(M.y, W.y);
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&maps_ready[m]);
          load_a(n + 1);  // the slice of ring A is read
        }
        __syncwarp();
      }
      if (LAG == 0 ? !tm.end : n > 0) {
        // ---- C: tile n - LAG
        const uint32_t q = n - LAG, mq = q % MS;
        if (LAG == 0) hp = nhp;
        const TileMeta tc = meta[q % kTeamMeta];
        const int rel = tc.rel0 + w * TS;
        const int d0 = tc.d + lane * VEC;
        const bool ch_ok = d0 < p.D;
        const int rows = ch_ok ? min(tc.len - rel, TS) : 0;
        const bool fast = polys[q % kTeamMeta] != 0 && __all_sync(kFull, rows == TS);
        [[maybe_unused]] const int64_t pitch = p.D * (int64_t)sizeof(T);
        [[maybe_unused]] unsigned char* dz =
            static_cast<unsigned char*>(a.dz) + ((int64_t)tc.b * p.L + tc.t0 + w * TS) * pitch + d0 * (int64_t)sizeof(T);
        uint32_t pr[16], merge[8];
        if constexpr (LAG == 0) tmem_wait_st();
        __syncwarp();  // tcgen05 accesses are warp-collective
        const uint32_t from = tq + (q % TSLOTS) * COLS;
        tmem_ld16_start(from, pr);
        if constexpr (GATED) tmem_ld8_start(from + team_cols<T>(), merge);
        mbar_wait(&carry_ready[mq], (q / MS) & 1u, err);
        // the adjoint entering the slice: the tile's, through the slices after it
        float2 win;
        win.x = carries[mq * CHW + lane * VEC];
        win.y = F32 ? win.x : carries[mq * CHW + lane * VEC + VEC - 1];
        const float2* mp = maps + mq * NW * CHW + lane * VEC;
        for (int o = ns - 1; o > w; --o) {
          const float2 e0 = mp[o * CHW], e1 = mp[o * CHW + VEC - 1];
          win = map_apply2(make_float2(e0.x, e1.x), win, make_float2(e0.y, e1.y));
        }
        if (__any_sync(kFull, !all_finite(win))) {
          tmem_ld_wait(pr);
          if constexpr (GATED) tmem_ld8_ready(merge);
          const float2 in = make_float2(carries[mq * CHW + lane * VEC], carries[mq * CHW + lane * VEC + VEC - 1]);
          win = team_enter_any<T>(from, mp + (ns - 1) * CHW, ns - 1 - w, -1, in);
          tmem_ld16_start(from, pr);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&maps_read[mq]);
        const float2 k = rates[(q % kTeamMeta) * 32 + lane];
        float2 dlr = f2(0.0f);
        mbar_wait(&fullC[w], q & 1u, err);
        unsigned char* lb = wb + SM::ringC + lane * 4u;
        auto sweep = [&](auto fast_c) {
          constexpr bool FAST = decltype(fast_c)::value;
#pragma unroll 1
          for (int part = 0; part < NP; ++part) {
            __syncwarp();
            tmem_ld_wait(pr);
            if constexpr (GATED) tmem_ld8_ready(merge);
            unsigned char* lp = lb + part * PR * 128;
            const int pv = rows - part * PR;
            if constexpr (F32)
              team_rows_f32<FAST, GATED, BOX>(lp, pr, win.x, k, pv, hp.x, dlr.x, merge, dz, pitch);
            else
              team_rows_bf16<FAST, GATED, BOX>(lp, pr, win, k, pv, hp, dlr, merge, dz, pitch);
            if (part + 1 < NP) {
              __syncwarp();
              tmem_ld16_start(from + (part + 1) * 16, pr);
              if constexpr (GATED) tmem_ld8_start(from + team_cols<T>() + (part + 1) * 8, merge);
            }
          }
        };
        if (fast)
          sweep(BoolC<true>{});
        else
          sweep(BoolC<false>{});
        fence_proxy_async_smem();  // this thread's outputs in the slice, visible to the TMA stores
        __syncwarp();
        if (lane == 0 && rel < tc.len) {  // a slice past the sequence has none
          tma_store_3d(&a.tm_dx, wb + SM::ringC, tc.d, tc.t0 + w * TS, tc.b);
          tma_store_3d(&a.tm_dr, wb + SM::ringC + BOX, tc.d, tc.t0 + w * TS, tc.b);
          tma_store_3d(&a.tm_di, wb + SM::ringC + 2 * BOX, tc.d, tc.t0 + w * TS, tc.b);
          bulk_commit();
        }
        // d Lambda: this slice's terms into the warp's own float64 sums, which go to
        // the workspace's when the channel group changes (and at the end)
        double* ds = dsums + w * CHW + lane * VEC;
        if (tc.d != dgroup) {
          if (dgroup >= 0) dlam_add(acc, dgroup + lane * VEC, ds);
          dgroup = tc.d;
#pragma unroll
          for (int v = 0; v < VEC; ++v) ds[v] = 0.0;
        }
        if (rows > 0) {
          ds[0] += (double)dlr.x;
          if constexpr (!F32) ds[VEC - 1] += (double)dlr.y;
        }
      }
      if (LAG == 1) hp = nhp;
      if (tm.end) break;
    }
    if (lane == 0) bulk_wait_all();  // every store complete before the block ends
    __syncwarp();
    tmem_fence_before_sync();
  }
  __syncthreads();  // every role is done with the block's TMEM
  if (warp == 0) {
    tmem_fence_after_sync();
    tmem_dealloc(*tslot, TCOLS);
  }
  // The warps' last d Lambda sums: added up per team, one reduction per team
  // and channel.
  {
    const int w = warp - team * NW;
    if (warp < kTeamWarps && w == 0 && dgroup >= 0) {
      double sum[VEC];
#pragma unroll
      for (int v = 0; v < VEC; ++v) sum[v] = 0.0;
      for (int o = 0; o < ns; ++o) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) sum[v] += dsums[o * CHW + lane * VEC + v];
      }
      dlam_add(acc, dgroup + lane * VEC, sum);
    }
    __syncthreads();
  }
  // The last block out turns the partial sums into d Lambda and clears them
  // (and the exit counter) for the next backward.
  __shared__ int s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&bh->exited, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int64_t d = threadIdx.x; d < p.D; d += blockDim.x) {
      double sum = 0.0;
      for (int s2 = 0; s2 < kStripes; ++s2) {
        sum += __ldcg(&acc[s2 * p.D + d]);
        acc[s2 * p.D + d] = 0.0;
      }
      const double lam = (double)a.lambda[d];
      const double sig = 1.0 / (1.0 + exp(-lam));  // d softplus / d Lambda
      a.dlambda[d] = (float)(-(double)p.c * sig * sum);
    }
    if (threadIdx.x == 0) {
      bh->exited = 0u;
      bh->set = s_set ^ 1u;
    }
  }
}

}  // namespace blr
