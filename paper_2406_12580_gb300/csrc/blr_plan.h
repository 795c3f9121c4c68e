// Plan and workspace layout of the BD-LRU scan kernels (host and device).
//
// A chain is a 128-byte row segment, 32 float32 or 64 bfloat16 channels of one
// batch row (in the narrow serial kernels 32 bfloat16 ones), followed through
// time. Problems with many chains run the serial
// kernels (blr_seq.cuh): one warp walks one chain through the whole sequence.
// The others run the team kernels (blr_team.cuh): teams of warps scan tiles of
// `ts` steps of a chain, whole chains at a time (local order) or tiles of all
// chains in time order, chained by a decoupled look-back.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace blr {

constexpr int kStripes = 8;                // dlambda float64 partial-sum stripes
constexpr size_t kAlign = 256;             // alignment of every workspace region

// Error bits recorded in FwdHeader::err.
constexpr uint32_t kErrTimeout = 1u;
constexpr uint32_t kErrWorkspace = 2u;
// The look-back's records validate themselves: they hold this all-ones pattern
// (a negative NaN with a full payload, which float arithmetic never produces)
// before a scan, and a record is published by one 32- or 64-bit store.
// There are two sets. The forward uses the first, which a memset fills before the
// call, and fills the second for the backward; each backward fills the one it
// does not use, for a backward that may follow it on the same workspace. So the
// backward needs no memset (fwd + bwd, us, with one / without: 12 x 1031 x 200
// bfloat16 45.6 / 42.0, 8 x 8192 x 512 float32 260.6 / 257.3, 1 x 2000 x 64 34.9 / 31.9).
constexpr uint32_t kEmpty = 0xffffffffu;

// Upper bound of every inter-block wait.
constexpr uint64_t kWaitTimeoutNs = 1000000000ull;  // 1 s
constexpr uint32_t kMaxWaitIters = 1u << 23;

struct FwdHeader {     // restarted by every forward
  uint32_t pad0[2];    // (with err first, the gated bfloat16 team backward spills 28 B instead of 8)
  uint32_t err;        // error bits (forward and backward timeouts, workspace misuse)
  uint32_t tag;        // hash of the problem, written by the forward
  uint32_t complete;   // 1 once a forward has run
  uint32_t pad[3];
};

struct BwdHeader {
  uint32_t set;            // look-back: the record set the next backward uses (0: the second)
  uint32_t exited;         // blocks of the backward that are done
  uint32_t selftest_flag;  // a flag nothing sets (blr_selftest_wait_timeout)
  uint32_t pad[5];
};

// Shape classes that blr_scan_family reports: at least kManyChains chains, or
// bfloat16 sequences of at least kSegMinL steps with kSegMinElems elements or
// kSegLongL steps, or the rest.
constexpr int64_t kManyChains = 256;
constexpr int64_t kSegMinL = 2048;
constexpr int64_t kSegMinElems = (int64_t)8 << 20;
constexpr int64_t kSegLongL = 16384;

constexpr int64_t kSeqTallRowsMinL = 1024;

// float32 problems with at least this many chains run the serial kernels, one
// warp a chain; the GPU's 608 schedulers are then close to one warp each or
// above. Measured on GB300 (fwd + bwd, us, serial / team kernels): 600 chains x
// 800 steps 119 / 124, x 3000 399 / 431, 400 x 3000 320 / 297, 512 x 2048 251 / 274.
constexpr int64_t kSeqMinChainsF32 = 512;
// Its backward without lengths from somewhat fewer on, where the rows are long, on
// the states a team forward kept (they lie the same way): the team backward takes
// two rounds of whole chains from 305 to 608 of them however many, a serial one
// grows by the chain. Rows whose last chain is not full, and wide ones, whose d Lambda
// the serial kernel's last warp adds up by itself, stay with the teams (backward, us
// over us, serial / team: D = 32, L = 800 430 chains 0.95, 460 0.90, 511 0.90, L =
// 2000 0.94, 0.91, 0.87; D = 64 1.03, 0.96, 0.94 and 1.00, 0.95, 0.92; D = 128 1.04,
// 1.00, 0.96 and 1.01, 0.96, 0.94; D = 256 1.15, 1.07, 1.06; D = 16 1.12, 1.03, 0.88 and
// 1.25, 1.17, 1.08; L = 373 D = 32 1.07, 1.02, 1.02, D = 128 1.17, 1.09, 1.12. With the
// merge D = 32, L = 800 416 chains 0.88, 488 0.81, D = 64 0.93, 0.85, D = 128 0.94, 0.87;
// 488 chains, L = 400, 512, 700 D = 32 0.91, 0.86, 0.85, D = 64 0.95, 0.93, 0.90, D = 128
// 0.99, 0.96, 0.94, at L = 420 1.03). Rows with lengths share the teams' work better
// and stay with them (fwd + bwd 456 x 400 51.2 / 47.8 us, x 2000 206 / 158).
inline bool plan_seq_bwd_f32(int64_t chains, int64_t L, int64_t D, bool gated) {
  if (D % 32 != 0 || D > 128) return false;
  if (gated) return (chains >= 416 && L >= 800) || (chains >= 488 && L >= (D <= 64 ? 385 : 512));
  return chains >= 456 && L >= 800;
}

// Team kernels: kTeamWarps compute warps a block, in teams of kTeamWidth;
// a warp takes kTeamSlice steps of a tile. The plan (and with it the workspace)
// depends on the problem alone, so it counts teams of the GB300's 152 SMs.
constexpr int kTeamWarps = 16;
constexpr int kTeamWidth = 8;
constexpr int kTeamSlice = 16;
constexpr int64_t kPlanTeams = 152 * (kTeamWarps / kTeamWidth);

// bfloat16: a chain of the serial kernels is 64 channels, two a lane, or, in
// their narrow form, 32, one a lane: twice the warps with about 0.6 of the
// instructions each. `wide` and `narrow` count a problem's chains either way.
//
// Serial from this many wide chains, and from one a team where the sequences
// are no longer than 5/4 of that number: a serial chain takes its steps one by
// one however few chains there are, the team kernels' time follows the work
// (fwd + bwd, us, narrow serial / team kernels: 330 chains x 50 steps 19.4 / 21.6, x
// 400 72 / 73, x 800 136 / 98; 450 x 50 20.4 / 23.5, x 800 140 / 123; 700 x 200
// 52 / 65, x 800 170 / 176, x 2000 407 / 374; 780 x 200 53 / 71, x 2000 415 / 417;
// with the merge 450 x 200 50.0 / 54.3, 700 x 800 204 / 224, x 2000 490 / 464).
constexpr int64_t kSeqMinChainsBf16 = 780;
inline bool plan_seq_bf16(int64_t wide, int64_t L) {
  return wide >= kSeqMinChainsBf16 || (wide >= kPlanTeams && 4 * L <= 5 * wide);
}
// Forward and backward choose by themselves: the states kept between them lie
// the same way. Both are narrow up to three narrow warps a scheduler (608 of
// them), the backward of short sequences up to four. Up to there the busiest
// scheduler has less to walk; beyond, the wide form has the fewer instructions
// (fwd + bwd, us, wide / narrow: 650 wide chains x 200 steps 57.8 / 52.5, with the
// merge 74.8 / 61.8; 850 x 200 58.8 / 53.4; forward alone 950 x 200 20.1 / 21.6, x 800
// 67.9 / 80.3; backward narrow after a wide forward 950 x 50 26.4 / 24.7, 1216 x 50
// 28.7 / 26.6, with the merge 33.7 / 30.9, 1000 x 200 with lengths 56.0 / 57.1, 950 x
// 800 202.6 / 205.3, 1500 x 200 80.0 / 92.7). And wherever a third or more of the wide
// lanes lie past D (1000 x 200 x 32 62.4 / 43.9, 4000 x 50 x 32 with the merge
// 76 / 48, 1500 x 100 x 96 81.3 / 70.6, 3000 x 50 x 96 82.2 / 80.7).
constexpr int64_t kSeqMaxNarrow = 3 * 608, kSeqMaxNarrowBwd = 4 * 608, kSeqNarrowBwdL = 128;
inline bool plan_narrow(int64_t wide, int64_t narrow, int64_t most = kSeqMaxNarrow) {
  return narrow <= most || 2 * narrow <= 3 * wide;
}
inline bool plan_narrow_bwd(int64_t wide, int64_t narrow, int64_t L) {
  return plan_narrow(wide, narrow, L <= kSeqNarrowBwdL ? kSeqMaxNarrowBwd : kSeqMaxNarrow);
}
// With the merge the wide forward's rings fit 13 blocks an SM. Where there are more
// chains than that, some wait for a place, and the narrow form, two blocks of half
// the size, is faster again for short ones (fwd + bwd, us, wide / narrow forward, L =
// 50: 913 x 64 27.6 / 27.7, 1400 36.0 / 36.0, 1600 37.6 / 37.4, 1824 39.9 / 41.2, 1950
// 41.5 / 44.1, 2000 46.8 / 44.8, 2048 47.1 / 44.8, 2600 62.9 / 61.7, 3500 77.1 / 76.0,
// 8000 142.8 / 141.3; x 100 1950 70.1 / 73.4, 2048 76.4 / 73.8; but 3000 x 160 171 /
// 177, 1500 x 200 99 / 101). For longer ones it is where a sixth or more of the wide
// lanes lie past D (700 x 200 x 160 137.6 / 122.9, 3000 x 50 x 160 144.2 / 140.2; but
// 2100 x 800 x 160 1337 / 1347).
constexpr int64_t kSeqWideMergeMost = 13 * 152;
inline bool plan_narrow_merge(int64_t wide, int64_t narrow, int64_t L) {
  return (wide > kSeqWideMergeMost && L <= 100) ||
         (wide >= kSeqMaxNarrow && L <= 256 && 3 * narrow <= 5 * wide);
}

// The look-back reads this many predecessors a round trip; kFarWindow where the
// chains are so few (kFarChains) that the tiles scanned at one time are many
// predecessors deep.
constexpr int kNearWindow = 2, kFarWindow = 8;
constexpr int64_t kFarChains = 19;

struct Plan {
  int64_t B, L, D;
  int io;           // 0 = float32, 1 = bfloat16
  float c;
  int seq;          // 1: serial kernels, 0: team kernels
  int seq_bwd[2];   // without lengths, plain and gated: 1: the serial backward all the same
  int sv;           // channels per lane (a chain is a row segment of 32 * sv channels)
  int rb;           // steps between the forward's kept states
  int sr, srb;      // serial: rows per TMA box, forward and backward (multiples of rb)
  int ts;           // team: steps per tile (a multiple of kTeamSlice)
  int lookback;     // team: 1 look-back order, 0 local order
  int far_window;   // team: the look-back's window
  int segmented;    // the shape class BLR_FAMILY_SEGMENTED
  int64_t n_chain;  // chains = B * ceil(D / (32 * sv))
  int64_t n_carry;  // kept states per chain = ceil(L / rb) - 1
  int64_t n_tc;     // team: tiles per chain
  uint32_t tag;
  // Workspace byte offsets: headers, dlambda partial sums, kept states (one per
  // rb steps, batch row and channel) and, in the look-back order, one record per
  // tile and channel: the state after it (off_cinc, 32-bit) and its map
  // (off_cagg, 64-bit), rec_set bytes up to off_cend; the second set of them
  // follows.
  size_t off_fhdr, off_bhdr, off_dlam, off_kept, off_cinc, off_cagg, off_cend, rec_set, bytes;
};

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline uint32_t fnv1a(uint32_t h, uint64_t v) {
  for (int i = 0; i < 8; ++i) {
    h ^= (uint32_t)(v & 0xff);
    h *= 16777619u;
    v >>= 8;
  }
  return h;
}

// Whether the team kernels take the look-back order: when the tiles of the
// busiest team, spread over all teams, plus the look-back's own cost (about
// 5 % a tile, and its records and cooperative launch, worth about 2 tiles) still
// come to less than whole chains a team. Measured on GB300 (fwd + bwd, us,
// look-back / local): bfloat16 20 chains x 300 steps 31.2 / 37.8 (the forward alone 13.5 /
// 12.6), 30 x 500 31.7 / 47.2, with the merge 33.4 / 55.9, 100 x 600 39.3 / 55.3, 150 x
// 800 57.0 / 75.1, 200 x 130 38 / 33, 300 x 800 94 / 84, 700 x 3000 547 / 588;
// float32 400 x 3000 297 / 326.
inline bool plan_lookback(int64_t chains, int64_t tiles) {
  const int64_t local = (chains + kPlanTeams - 1) / kPlanTeams * tiles;
  const int64_t spread = (chains * tiles + kPlanTeams - 1) / kPlanTeams;
  return tiles > 1 && 20 * local > 21 * spread + 38;
}

// Fills `p` for a validated problem (B, L, D >= 1, D % 8 == 0). local_only
// keeps the team kernels in the local order, whose workspace has no records.
inline void make_plan(int64_t B, int64_t L, int64_t D, int io, float c, bool local_only, Plan* p) {
  p->B = B;
  p->L = L;
  p->D = D;
  p->io = io;
  p->c = c;
  uint32_t h = 2166136261u;
  h = fnv1a(h, (uint64_t)B);
  h = fnv1a(h, (uint64_t)L);
  h = fnv1a(h, (uint64_t)D);
  h = fnv1a(h, (uint64_t)io);
  uint32_t cbits;
  __builtin_memcpy(&cbits, &c, 4);
  h = fnv1a(h, cbits);
  p->tag = h | 1u;  // never 0, the value of a cleared header
  p->sv = io == 0 ? 1 : 2;
  p->n_chain = B * ((D + 32 * p->sv - 1) / (32 * p->sv));
  p->seq = io == 0 ? p->n_chain >= kSeqMinChainsF32 : plan_seq_bf16(p->n_chain, L);
  for (int g = 0; g < 2; ++g)
    p->seq_bwd[g] = p->seq || (io == 0 && plan_seq_bwd_f32(p->n_chain, L, D, g != 0));
  p->segmented = p->n_chain < kManyChains && io == 1 && L >= kSegMinL &&
                 (B * L * D >= kSegMinElems || L >= kSegLongL);
  // Long float32 sequences stream the serial forward in 32-row boxes (fewer,
  // larger TMA loads per chain); shorter ones in 16-row boxes, which reach the
  // first rows sooner.
  p->sr = (io == 0 && L >= kSeqTallRowsMinL) ? 32 : 16;
  p->srb = p->sv == 1 ? 16 : 8;
  p->rb = !p->seq ? kTeamSlice : io == 0 ? 16 : 8;
  p->n_carry = (L + p->rb - 1) / p->rb - 1;
  // Tiles of equal height, as few as cover L.
  const int64_t most = (int64_t)kTeamWidth * kTeamSlice;
  const int64_t n = (L + most - 1) / most;
  p->ts = (int)(((L + n - 1) / n + kTeamSlice - 1) / kTeamSlice * kTeamSlice);
  p->n_tc = (L + p->ts - 1) / p->ts;
  p->lookback = !p->seq && !local_only && plan_lookback(p->n_chain, p->n_tc) ? 1 : 0;
  p->far_window = p->n_chain <= kFarChains ? 1 : 0;
  const size_t BD = (size_t)B * (size_t)D;
  const size_t rec = p->lookback ? (size_t)p->n_tc * BD : 0;
  size_t o = 0;
  p->off_fhdr = o;
  o = align_up(o + sizeof(FwdHeader), kAlign);
  p->off_bhdr = o;
  o = align_up(o + sizeof(BwdHeader), kAlign);
  p->off_dlam = o;
  o = align_up(o + 8 * (size_t)kStripes * (size_t)D, kAlign);
  p->off_kept = o;
  o = align_up(o + 4 * (size_t)p->n_carry * BD, kAlign);
  p->off_cinc = o;
  o = align_up(o + 4 * rec, kAlign);
  p->off_cagg = o;
  o = align_up(o + 8 * rec, kAlign);
  p->off_cend = o;
  p->rec_set = o - p->off_cinc;
  p->bytes = o + p->rec_set;
}

// The teams that work, of `teams` launched: a multiple of the channel groups, if
// that idles few of them (a team then stays within one group, and the backward adds
// its d Lambda sums up once) and gives the busiest no further chain to walk.
inline uint32_t plan_teams(const Plan& p, uint32_t teams) {
  const int64_t n_g = p.n_chain / p.B;
  if (teams < 8 * n_g) return teams;
  const uint32_t whole = teams - teams % (uint32_t)n_g;
  const bool longer = (p.n_chain + whole - 1) / whole > (p.n_chain + teams - 1) / teams;
  return !p.lookback && longer ? teams : whole;
}

}  // namespace blr
