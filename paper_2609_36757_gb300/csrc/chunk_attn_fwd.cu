// Chunk-causal attention forward for sm_103a (Sec. 3.1, Eq. 1): tcgen05
// tensor cores with TMEM accumulators, TMA-staged tiles, fp32 online softmax.
//
// Masking acts at chunk granularity and a call attends one chunk's queries,
// so every key of the visible segments is visible to every query: the host
// enumerates only visible cache ranges (block-causal skipping happens before
// launch, invisible chunks are never loaded) and the only in-kernel mask is
// the ragged end of a segment.
//
// One CTA owns two 128-row query tiles of one (batch, head), or one where a
// launch has few, and streams the visible keys in 128-key tiles:
//   warp 8      TMA producer of the Q tiles (once) and the K ring (3 deep);
//   warp 10     TMA producer of the V ring (2 deep); all tiles are
//               128-byte swizzled boxes of 64 columns.
//   warp 11     relay: observes the TMA completions and hands each K/V ring
//               stage to the MMA warp through a named barrier.
//   warp 9      MMA issuer (the warp runs converged, an elected lane
//               issues): S = Q_t K^T into TMEM, then O_t += P_t V with P_t
//               read from TMEM; order per key tile j: QK_0(j), PV_0(j-1),
//               QK_1(j), PV_1(j-1).
//   warps 0-3   softmax of query tile 0, one thread per row (TMEM lane);
//   warps 4-7   softmax of query tile 1.
// TMEM (512 columns): S (shared by the two tiles) | P_0 | P_1 | O_0 | O_1,
// 128 + 64 + 64 + 128 + 128 columns (d = 64: S_0 | S_1 | P_0 | P_1 | O_0 |
// O_1, 128 + 128 + 4 x 64).  S only lives until the softmax warps
// have loaded it (they release it before the row max), so the next QK^T of
// either tile can follow at once; each tile's PV runs one key tile behind,
// which gives its softmax three MMA steps to store P_t.  The MMA warp never
// polls a shared-memory barrier: every hand-off to it (S read, P_t stored,
// K/V stage landed) is a named barrier, whose arrivals are made on every
// path (also after a failed wait: handoff.h), since a named barrier has no time
// limit.
//
// Online softmax in the exp2 domain: each row keeps a reference m (a lower
// bound of its running max) and exponentiates against it; m moves, and O is
// rescaled, only when a tile's max exceeds m by more than 8 (P stays <= 256,
// finite in bf16 and fp32).  The final O / l is the same for any reference,
// so this is exact up to rounding.  Before storing P_t(j) the softmax waits
// until PV_t(j-1) has completed, so O_t is current for the rare rescale.
//
// Epilogue: a whole unit's softmax warps stage O_t / l as bf16 in the Q_t
// buffer (free once every MMA has completed) and one thread per tile writes
// it with tiled TMA stores; a split unit's key ranges write fp32 partials
// and the log2-domain LSE for the merge kernel.  The TMA loads carry L2
// policies: evict_first for the query tiles (one CTA reads them),
// evict_last for K/V (every unit of the head reads them).
//
// Every mbarrier wait is bounded: past the limit the kernel records
// FASTVR timeout in the control word, no role starts new copies or takes up
// new work, the hand-offs are made to the end (the MMA warp, if it had begun,
// runs on over undefined data), in-flight TMA loads and MMAs are drained, TMEM
// is released and the CTA exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <float.h>
#include <math.h>

#include <algorithm>

#include "fastvr_internal.h"
#include "handoff.h"
#include "sm100_ptx.cuh"

namespace fastvr {
namespace {

using namespace sm100;

constexpr int kBM = 128;        // query rows per tile (one TMEM lane each)
constexpr int kBN = 128;        // keys per tile
constexpr int kQTiles = 2;      // query tiles per CTA
constexpr int kKStages = handoff::kFwdKStages;  // depth of the K ring
constexpr int kVStages = handoff::kFwdVStages;  // depth of the V ring
constexpr int kThreads = 384;   // 8 softmax warps, K and V producers, MMA,
                                // relay
constexpr int kBox = 128 * 128; // one TMA box: 128 rows x 64 bf16 (bytes)
constexpr uint32_t kTmemCols = 512;
// TMEM columns.  d = 128: one S tile shared by the two query tiles, P_0 and
// P_1 (bf16 pairs, 64 columns each), O_0 and O_1 (128 columns each), all 512.
// d = 64: O needs half the columns, and each query tile has an S of its own:
// its QK^T then waits for its own softmax alone, which keeps the two tiles'
// softmax warps apart in time (with a shared S each tile's S came a whole
// hand-off after the other tile had read its own; d = 64 chunk step, 48 heads
// of 3465 x 10395: 429.2 -> 415.4 us together with the early look at p_free).
template <int D>
struct Tmem {
  static constexpr bool kOwnS = D == 64;
  __host__ __device__ static constexpr uint32_t s(int t) {
    return kOwnS ? t * 128u : 0u;
  }
  __host__ __device__ static constexpr uint32_t p(int t) {
    return (kOwnS ? 256u : 128u) + t * 64u;
  }
  __host__ __device__ static constexpr uint32_t o(int t) {
    return kOwnS ? 384u + t * 64u : 256u + t * 128u;
  }
};
static_assert(Tmem<128>::o(1) + 128 == kTmemCols &&
                  Tmem<64>::o(1) + 64 == kTmemCols,
              "TMEM columns");
constexpr float kRescaleThreshold = 8.0f;      // log2 units
constexpr int kMinTilesPerPart = 4;             // key tiles per split part
constexpr uint64_t kDefaultWaitLimitNs = 4000000000ull;  // 4 s per wait
// Threads of a generation of the hand-offs' named barriers (which of them are
// which, and their order: handoff.h).
constexpr int kHandoff = handoff::kFwdSoftmaxWarps * 32;
constexpr int kRelay = handoff::kRelayWarps * 32;
// Named barrier of a query tile's four softmax warps: their rows of O are
// staged for the tile's TMA store.
constexpr int kBarOStaged0 = 9;  // + t

struct TcParams {
  CUtensorMap q_map;                  // {d, Lq, H, B}
  CUtensorMap o_map;                  // the output, the same form as q_map
  CUtensorMap k_map[kMaxSegments];    // {d, segment end, H, B} of the cache
  CUtensorMap v_map[kMaxSegments];
  uint16_t* o;
  float* lse;
  Strides o_str;
  int32_t q_tokens, heads;
  int32_t seg_start[kMaxSegments];
  int32_t seg_len[kMaxSegments];
  int32_t seg_tiles0;   // tiles of segment 0
  int32_t total_tiles;
  float scale_log2;
  int* status;
  uint64_t wait_limit_ns;
  int32_t inject_stall;
  // Work split: units of two query tiles, (b, h, pair) with the pair index
  // fastest, a head's last pair that holds one query tile only (pair
  // long_pairs) after all others, or in its place (long_pairs = q_pairs); the
  // first units_full run whole, the tail_units after them are cut into `split`
  // key-tile ranges, equal ones or, with cut > 0, [0, cut) and the rest, whose
  // partial results go to the workspace.
  int32_t q_pairs, long_pairs, units_full, tail_units, split, cut;
  int32_t unit_rows;  // query rows of a unit: two tiles, or one (few units)
  int32_t sms;  // SM count: CTA index / sms is a CTA's wave
  float* ws;      // partial O: [part][d][kUnitRows]
  float* ws_lse;  // partial log2-domain LSE: [part][kUnitRows]
  int32_t ws_parts;  // partial results the workspace holds
  int64_t o_elems;   // elements of o (B Lq H d), for the debug index checks
  // One-shot (training-form) launches: the whole sequence of seq_tokens
  // tokens, chunks of chunk_tokens tokens, window W (-1: unbounded).
  int32_t seq_tokens, chunk_tokens, window, batch;
};

// The work of one CTA.
struct Work {
  int q0, h, b;
  int j0, n;   // first key tile (index into the visible tiles) and count
  int nqt;     // query tiles with at least one row in the chunk (1 or 2)
  int part;    // -1: whole unit, final output; else workspace slot
  int kv0, kv1;  // one-shot: the unit's key token range [kv0, kv1)
  bool rev;    // walk the key tiles last to first
};

// Whole units in odd waves (CTA index / SM count) walk their key tiles last
// to first.  Consecutive units of a head run together, so a head whose units
// straddle two waves is streamed by the second wave right after the first:
// walking back, that wave starts on the tiles the first one loaded last,
// which are still in L2, instead of on the oldest ones.  The online softmax
// does not depend on the order (up to rounding).
__device__ __forceinline__ bool odd_wave(const TcParams& p) {
  return ((int)blockIdx.x / p.sms) & 1;
}

// One-shot launches: the query pairs are grouped from the end of the
// sequence into blocks of kOneShotBlock pairs; unit x takes block
// x / (kOneShotBlock H B) (the units with the most keys start first), then
// (b, h) and a pair within the block with the pair fastest, so that the CTAs
// of one wave stream the keys of a few heads, each shared by up to
// kOneShotBlock CTAs, rather than of every head at once.  A unit's keys are
// the union of what its rows see: chunks max(0, c_lo - W) .. c_hi of its
// first and last rows (Eq. 1 with window W).
constexpr int kOneShotBlock = 32;

__device__ __forceinline__ Work oneshot_work(const TcParams& p) {
  Work w;
  const int hb = p.heads * p.batch;
  const int blk = blockIdx.x / (kOneShotBlock * hb);
  const int x = blockIdx.x % (kOneShotBlock * hb);
  const int in_blk = min(kOneShotBlock, p.q_pairs - blk * kOneShotBlock);
  const int bh = x / in_blk;
  const int pair = p.q_pairs - 1 - blk * kOneShotBlock - x % in_blk;
  w.h = bh % p.heads;
  w.b = bh / p.heads;
  w.q0 = pair * p.unit_rows;
  const int rows = min(p.unit_rows, p.q_tokens - w.q0);
  w.nqt = rows > kBM ? 2 : 1;
  const int c_lo = w.q0 / p.chunk_tokens;
  const int c_hi = w.q0 + rows - 1;
  const int chunk_hi = c_hi / p.chunk_tokens;
  w.kv0 = p.window < 0 ? 0 : max(0, c_lo - p.window) * p.chunk_tokens;
  w.kv1 = min((chunk_hi + 1) * p.chunk_tokens, p.seq_tokens);
  w.j0 = 0;
  w.n = (w.kv1 - w.kv0 + kBN - 1) / kBN;
  w.part = -1;
  w.rev = odd_wave(p);
  return w;
}

// Streaming: query pair and (b, h) of a unit; the short units come last, or,
// with long_pairs = q_pairs, in their place.
__device__ __forceinline__ void unit_coord(const TcParams& p, int unit,
                                           int& pair, int& bh) {
  const int n_long = p.long_pairs * p.heads * p.batch;
  if (unit < n_long) {
    pair = unit % p.long_pairs;
    bh = unit / p.long_pairs;
  } else {
    pair = p.long_pairs;
    bh = unit - n_long;
  }
}

// The tail's CTAs go range by range, the longer range first: the CTAs that
// run together then stream the same keys of a head.
template <bool kOneShot>
__device__ __forceinline__ Work cta_work(const TcParams& p) {
  if (kOneShot) return oneshot_work(p);
  Work w;
  w.kv0 = w.kv1 = 0;
  w.j0 = 0;
  w.n = p.total_tiles;
  int unit = blockIdx.x, part = -1;
  if (unit >= p.units_full) {
    const int k = unit - p.units_full;
    const int u = k % p.tail_units, idx = k / p.tail_units;
    unit = p.units_full + u;
    part = u * p.split + idx;
    if (p.cut > 0) {
      w.j0 = idx ? p.cut : 0;
      w.n = idx ? p.total_tiles - p.cut : p.cut;
    } else {
      w.j0 = (int)((int64_t)idx * p.total_tiles / p.split);
      w.n = (int)((int64_t)(idx + 1) * p.total_tiles / p.split) - w.j0;
    }
  }
  int pair, bh;
  unit_coord(p, unit, pair, bh);
  w.h = bh % p.heads;
  w.b = bh / p.heads;
  w.q0 = pair * p.unit_rows;
  w.nqt = min(p.unit_rows, p.q_tokens - w.q0) > kBM ? 2 : 1;
  w.part = part;
  w.rev = part < 0 && odd_wave(p);
  return w;
}

struct Shared {
  uint64_t q_full;
  uint64_t k_full[kKStages], k_empty[kKStages];
  uint64_t v_full[kVStages], v_empty[kVStages];
  uint64_t s_full[kQTiles], p_free[kQTiles];
  uint64_t o_full, drain;
  uint32_t tmem_base;
  int abort;
  uint64_t wait_limit_ns;
};

template <int D>
struct Layout {
  static constexpr int kNB = D / 64;  // boxes per tile
  __host__ __device__ static constexpr int q(int t, int bx) { return (t * kNB + bx) * kBox; }
  __host__ __device__ static constexpr int k(int s, int bx) {
    return ((kQTiles + s) * kNB + bx) * kBox;
  }
  __host__ __device__ static constexpr int v(int s, int bx) {
    return ((kQTiles + kKStages + s) * kNB + bx) * kBox;
  }
  static constexpr int shared_off = (kQTiles + kKStages + kVStages) * kNB * kBox;
  static constexpr int bytes = shared_off + 1024 /*Shared*/ + 1024 /*align*/;
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Bounded wait.  Returns false when this wait timed out or another role
// already aborted; the first timeout records the error.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity,
                                      Shared* S, int* status) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*reinterpret_cast<volatile int*>(&S->abort)) return false;
    if (global_timer_ns() - t0 > S->wait_limit_ns) {
      *reinterpret_cast<volatile int*>(&S->abort) = 1;
      if (status != nullptr) atomicExch(status, kDevTimeout);
      return false;
    }
  }
}

// Bounded wait that ignores the abort flag (draining in-flight work).
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity,
                                           const Shared* S) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > S->wait_limit_ns) return;
  }
}

// One-shot: key tile j of the unit range [kv0, kv1) (map 0).
__device__ __forceinline__ void oneshot_tile(int kv0, int kv1, int j,
                                             int& seg, int& tok0, int& valid) {
  seg = 0;
  tok0 = kv0 + j * kBN;
  valid = min(kBN, kv1 - tok0);
}

__device__ __forceinline__ void tile_coord(const TcParams& p, int j, int& seg,
                                           int& tok0, int& valid) {
  seg = j < p.seg_tiles0 ? 0 : 1;
  const int jj = seg ? j - p.seg_tiles0 : j;
  tok0 = p.seg_start[seg] + jj * kBN;
  valid = min(kBN, p.seg_len[seg] - jj * kBN);
}

// TMA producers, one thread each: the K producer also loads the query tiles.
// K and V advance independently, so a slow V slot never holds back the next
// K tile (QK^T of tile j+1 is issued before PV of tile j completes).
template <int D, bool kIsK, bool kOneShot>
__device__ void producer(const TcParams& p, uint8_t* smem, Shared* S,
                         const Work& w) {
  const int h = w.h, b = w.b;
  using L = Layout<D>;
  constexpr int kStages = kIsK ? kKStages : kVStages;
  uint64_t* full = kIsK ? S->k_full : S->v_full;
  uint64_t* empty = kIsK ? S->k_empty : S->v_empty;
  // The query tiles are read by this CTA alone (evict first); the K and V
  // tiles of a head are read by every unit of the head (evict last).
  const uint64_t keep = l2_policy_evict_last();
  if (kIsK) {
    tma_prefetch_desc(&p.q_map);
    const uint64_t once = l2_policy_evict_first();
    mbar_arrive_expect_tx(&S->q_full, w.nqt * L::kNB * kBox);
    for (int t = 0; t < w.nqt; ++t)
      for (int bx = 0; bx < L::kNB; ++bx)
        tma_load_4d_hint(&p.q_map, smem + L::q(t, bx), &S->q_full, bx * 64,
                         w.q0 + t * kBM, h, b, once);
  }
  for (int s = 0; s < kMaxSegments; ++s)
    tma_prefetch_desc(kIsK ? &p.k_map[s] : &p.v_map[s]);
  int issued = 0;
  for (int j = 0; j < w.n; ++j) {
    const int st = j % kStages;
    const uint32_t ph = (j / kStages) & 1;
    int seg, tok0, valid;
    const int jt = w.rev ? w.n - 1 - j : j;
    if (kOneShot)
      oneshot_tile(w.kv0, w.kv1, jt, seg, tok0, valid);
    else
      tile_coord(p, w.j0 + jt, seg, tok0, valid);
    if (!wait_bar(&empty[st], ph ^ 1, S, p.status)) break;
    mbar_arrive_expect_tx(&full[st], L::kNB * kBox);
    for (int bx = 0; bx < L::kNB; ++bx)
      tma_load_4d_hint(kIsK ? &p.k_map[seg] : &p.v_map[seg],
                       smem + (kIsK ? L::k(st, bx) : L::v(st, bx)), &full[st],
                       bx * 64, tok0, h, b, keep);
    ++issued;
  }
  // Every issued load has landed before the CTA may exit (a no-op wait in
  // normal operation: consumers already waited for them).
  if (kIsK) drain_wait(&S->q_full, 0, S);
  for (int i = max(0, issued - kStages); i < issued; ++i)
    drain_wait(&full[i % kStages], (i / kStages) & 1, S);
}

// The issuing warp's waits: every lane polls and each decision (phase
// complete, abort seen, time limit passed) is a warp vote, so the warp
// never diverges and reaches the elected MMA instructions converged.  A
// phase that has already completed costs one try_wait and one vote.
__device__ __forceinline__ bool wait_bar_warp(uint64_t* bar, uint32_t parity,
                                              Shared* S, int* status) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = global_timer_ns();
  while (true) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const bool aborted = *reinterpret_cast<volatile int*>(&S->abort) != 0;
    const bool late = global_timer_ns() - t0 > S->wait_limit_ns;
    if (__any_sync(0xffffffffu, aborted)) return false;
    if (__any_sync(0xffffffffu, late)) {
      if ((threadIdx.x & 31) == 0) {
        *reinterpret_cast<volatile int*>(&S->abort) = 1;
        if (status != nullptr) atomicExch(status, kDevTimeout);
      }
      __syncwarp();
      return false;
    }
  }
}

// The waits of a warp that makes the arrivals it owes after a failed wait
// (handoff.h): deaf to the abort flag; past the limit, which only a stopped
// tensor pipe reaches, the warp waits no more.
struct OwedWaits {
  bool pipe_runs = true;
  __device__ __forceinline__ void wait(uint64_t* bar, uint32_t parity) {
    const uint64_t t0 = global_timer_ns();
    while (pipe_runs) {
      const bool late = global_timer_ns() - t0 > kDefaultWaitLimitNs;
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return;
      pipe_runs = !__any_sync(0xffffffffu, late);
    }
  }
};

// A commit of the MMA warp; with nothing issued, an arrival.
template <bool kIssue>
__device__ __forceinline__ void commit_step(uint64_t* bar) {
  if (kIssue) {
    mma_commit_warp(bar);
  } else {
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
    __syncwarp();  // converged at the next named barrier
  }
}

// Hand-offs from the softmax warps to the MMA warp go through named
// barriers, which live in hardware rather than in shared memory: an mbarrier
// poll is a shared-memory access, and while SMEM x SMEM MMAs are queued every
// such access waits behind their operand reads (~200 clk), which the issuer
// cannot afford several times per key tile.  A named barrier has no time
// limit: after a failed wait a role still makes the arrivals that it owes, in
// step with the MMA warp (handoff.h says how).
__device__ __forceinline__ void named_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kHandoff) : "memory");
}
__device__ __forceinline__ void named_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kHandoff) : "memory");
}
__device__ __forceinline__ void relay_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kRelay) : "memory");
}
// The four softmax warps of one query tile (128 threads), and no other warp.
__device__ __forceinline__ void tile_sync(int id) {
  asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void relay_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kRelay) : "memory");
}

// The relay warp observes the TMA completions in the order the MMA warp
// needs them (K(j), then V(j - 1)) and hands each over through the named
// barrier of its ring stage, so the MMA warp itself never polls a
// shared-memory barrier.  A stage's barrier cannot be arrived at twice
// before the MMA warp has synced on it: the producer refills the stage only
// after the MMAs that read it.
__device__ void relay_role(const TcParams& p, Shared* S, int n) {
  struct Ops {
    Shared* S;
    int* status;
    OwedWaits owed;
    __device__ __forceinline__ bool wait_k(int j) {
      return wait_bar_warp(&S->k_full[j % kKStages], (j / kKStages) & 1, S,
                           status);
    }
    __device__ __forceinline__ bool wait_v(int j) {
      return wait_bar_warp(&S->v_full[j % kVStages], (j / kVStages) & 1, S,
                           status);
    }
    __device__ __forceinline__ void wait_k_slot(int j) {
      owed.wait(&S->k_empty[j % kKStages], ((j / kKStages) & 1) ^ 1);
    }
    __device__ __forceinline__ void wait_v_slot(int j) {
      owed.wait(&S->v_empty[j % kVStages], ((j / kVStages) & 1) ^ 1);
    }
    __device__ __forceinline__ void arrive(int id) { relay_arrive(id); }
  } ops{S, p.status, {}};
  handoff::fwd_relay_steps(n, ops);
}

// What the MMA warp does between its hand-offs (handoff::fwd_mma_steps); with
// kIssue false, after a wait that failed before the first MMA, the commits
// alone.
//
// One warp issues every MMA (an elected lane, the warp kept converged) and
// a tcgen05.mma takes it ~54 clk to issue against 64 clk of tensor work
// (M128 N128 K16), so the issue loop carries no descriptor arithmetic: the
// descriptor words are formed once and each MMA only adds a constant
// offset (16-byte units) to the low word.
template <int D, bool kIssue>
struct MmaOps {
  using L = Layout<D>;
  using T = Tmem<D>;
  static constexpr uint32_t kIdescQK = idesc_bf16_f32(kBM, kBN, 0);
  static constexpr uint32_t kIdescPV = idesc_bf16_f32(kBM, D, 1);
  static constexpr uint32_t kStage16 = (uint32_t)(L::kNB * kBox) >> 4;
  Shared* S;
  uint32_t tmem, hi, q_lo, k_lo, v_lo;

  __device__ __forceinline__ void relay_sync(int id) {
    fastvr::relay_sync(id);
  }
  __device__ __forceinline__ void softmax_sync(int id) { named_sync(id); }
  // S_t = Q_t K^T: both operands K-major, 128-byte
  // swizzle; a K step of 16 elements is 32 bytes inside a 64-column box.
  __device__ __forceinline__ void qk(int t, int st, bool last_use) {
    tc_fence_after();
    const uint32_t a0 = q_lo + (uint32_t)(L::q(t, 0) >> 4);
    const uint32_t b0 = k_lo + (uint32_t)st * kStage16;
#pragma unroll
    for (int ks = 0; kIssue && ks < D / 16; ++ks) {
      const uint32_t off = (uint32_t)((ks / 4) * kBox + (ks % 4) * 32) >> 4;
      mma_ss_warp(tmem + T::s(t), a0 + off, b0 + off, hi, kIdescQK, ks > 0);
    }
    commit_step<kIssue>(&S->s_full[t]);
    if (last_use) commit_step<kIssue>(&S->k_empty[st]);
  }
  // O_t += P_t V: P_t from its TMEM columns (8 per 16 keys), V MN-major (d
  // contiguous): 16 keys are two 8-row groups (2048 bytes), the two 64-column
  // halves of d are one box apart.
  __device__ __forceinline__ void pv(int t, int st, bool acc, bool last_use) {
    tc_fence_after();
    const uint32_t b0 = v_lo + (uint32_t)st * kStage16;
#pragma unroll
    for (int kk = 0; kIssue && kk < kBN / 16; ++kk)
      mma_ts_warp(tmem + T::o(t), tmem + T::p(t) + kk * 8,
                  b0 + (uint32_t)(kk * 2048 >> 4), hi, kIdescPV,
                  (acc | kk) != 0);
    commit_step<kIssue>(&S->p_free[t]);
    if (last_use) commit_step<kIssue>(&S->v_empty[st]);
  }
};

// Issue order per key tile j: QK_0(j), PV_0(j-1), QK_1(j), PV_1(j-1).  A
// tile's PV runs one key tile behind its QK^T, so the softmax of S_t(j)
// has the MMAs of three other steps (about 2000 clk) to produce P_t(j)
// before the pipe needs it, while S, which only has to survive until the
// softmax has loaded it, alternates between the tiles.
template <int D>
__device__ void mma_issuer(const TcParams& p, uint8_t* smem, Shared* S,
                           uint32_t tmem, const Work& w) {
  using L = Layout<D>;
  const uint32_t sbase = smem_addr(smem);
  // Test hook: o_full receives no arrival before the end of the stream, so
  // this wait runs out and exercises the abort path.
  bool ok = !p.inject_stall || wait_bar_warp(&S->o_full, 0, S, p.status);
  ok = ok && wait_bar_warp(&S->q_full, 0, S, p.status);
  if (ok) {
    MmaOps<D, true> ops{S, tmem, desc_hi_sw128(1024),
                        desc_lo(sbase + L::q(0, 0), 16),
                        desc_lo(sbase + L::k(0, 0), 16),
                        desc_lo(sbase + L::v(0, 0), kBox)};
    handoff::fwd_mma_steps(w.n, w.nqt == 2, Tmem<D>::kOwnS, ops);
    mma_commit_warp(&S->o_full);
  } else {
    MmaOps<D, false> ops{S};
    handoff::fwd_mma_steps(w.n, w.nqt == 2, Tmem<D>::kOwnS, ops);
  }
  mma_commit_warp(&S->drain);
  if ((threadIdx.x & 31) == 0) drain_wait(&S->drain, 0, S);
  __syncwarp();
}

__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// P = 2^(s * scale_log2 - m) for the 32 columns of s[c] (a packed FFMA per
// pair, one MUFU ex2 per element), packed as 16 bf16 pairs; the row sums go
// to four independent packed accumulators.
__device__ __forceinline__ void exp_pack32(const uint32_t (&sc)[32],
                                           uint64_t sl2x2, uint64_t neg2,
                                           uint32_t (&pk)[16],
                                           uint64_t (&acc)[4]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint64_t x2 = f2_fma(f2_pack(__uint_as_float(sc[2 * i]),
                                       __uint_as_float(sc[2 * i + 1])),
                               sl2x2, neg2);
    float x0, x1;
    f2_unpack(x2, x0, x1);
    const float p0 = ex2(x0), p1 = ex2(x1);
    acc[i & 3] = f2_add(acc[i & 3], f2_pack(p0, p1));
    pk[i] = pack_bf16(p0, p1);
  }
}

__device__ __forceinline__ float acc_total(const uint64_t (&acc)[4]) {
  float a0, a1, b0, b1, c0, c1, d0, d1;
  f2_unpack(acc[0], a0, a1);
  f2_unpack(acc[1], b0, b1);
  f2_unpack(acc[2], c0, c1);
  f2_unpack(acc[3], d0, d1);
  return ((a0 + a1) + (b0 + b1)) + ((c0 + c1) + (d0 + d1));
}

// Mask the columns of s[c] outside [lo, hi) (relative to the tile).
__device__ __forceinline__ void mask32(uint32_t (&sc)[32], int c, int lo,
                                       int hi) {
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (c * 32 + i < lo || c * 32 + i >= hi) sc[i] = 0xff800000u;  // -inf
}

// Fold the row max of s[c] into four independent accumulators.
__device__ __forceinline__ void max32(const uint32_t (&sc)[32],
                                      float (&mx)[4]) {
#pragma unroll
  for (int i = 0; i < 16; ++i)
    mx[i & 3] = max3(mx[i & 3], __uint_as_float(sc[2 * i]),
                     __uint_as_float(sc[2 * i + 1]));
}

// Streaming: j0, n index the launch's visible tiles.  One-shot: the tiles of
// [kv0, kv1); a row of chunk c sees keys of chunks max(0, c - W) .. c, so a
// row can be fully masked in a tile (its reference then stays as it was).
// Per key tile: read S (at d = 128 one buffer for both query tiles, at d = 64
// one each) into registers and release it at once, exponentiate, wait until the previous PV of this tile
// has consumed P_t (and brought O_t up to date), rescale O_t if the
// reference moved, then store P_t.
template <int D, bool kOneShot>
__device__ void softmax_role(const TcParams& p, Shared* S, uint32_t tmem,
                             int t, int nqt, int wq, int lane, int j0, int n,
                             int kv0, int kv1, int q0, bool rev) {
  const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
  using T = Tmem<D>;
  const uint32_t tS = tmem + T::s(t) + lane_off;
  const uint32_t tP = tmem + T::p(t) + lane_off;
  const uint32_t tO = tmem + T::o(t) + lane_off;
  const float sl2 = p.scale_log2;
  const uint64_t sl2x2 = f2_pack(sl2, sl2);
  // exp2-domain reference (scaled scores).  It starts at the lowest finite
  // value: a row that has seen no visible key yet, or none with a score above
  // -inf (one that overflowed), then exponentiates -inf, to 0, and not
  // -inf + inf.
  float m_ref = -FLT_MAX;
  float l = 0.f;
  // Each wait is decided per warp, by a vote whose latency passes behind the
  // loads or the exponentials that follow the wait: the TMEM accesses and the
  // named barriers are warp-wide, so lanes must not part after a failed wait.
  bool ok = true;
  const int s_expected = handoff::fwd_s_arrivals(n, t, nqt, T::kOwnS);
  int s_done = n;  // "S read" arrivals made
  int vis_lo = 0, vis_hi = 0;  // one-shot: this row's visible key tokens
  if (kOneShot) {
    const int row = min(q0 + t * kBM + wq * 32 + lane, p.q_tokens - 1);
    const int c = row / p.chunk_tokens;
    vis_lo = p.window < 0 ? 0 : max(0, c - p.window) * p.chunk_tokens;
    vis_hi = min((c + 1) * p.chunk_tokens, p.seq_tokens);
  }
  // Few tiles need a mask: streaming, the ragged ends of the two segments (at
  // most one tile each); one-shot, tiles that cross a chunk edge.  Whether
  // this one does is settled before S is waited for and decided once per
  // tile: worked out after the wait, with a test per 32 columns, it stood in
  // the chain from S to P (d = 64 chunk step, 48 heads of 3465 x 10395, with
  // one S for both query tiles as it then was: 433.7 -> 429.2 us).
  const int rag0_n = p.seg_len[0] % kBN, rag1_n = p.seg_len[1] % kBN;
  const int rag0 = rag0_n ? p.seg_tiles0 - 1 - j0 : -1;
  const int rag1 = rag1_n ? p.total_tiles - 1 - j0 : -1;
  int j = 0;  // and, after the loop, "P stored" arrivals made
  for (; j < n; ++j) {
    const int jt = rev ? n - 1 - j : j;  // the producers' order
    int lo = 0, hi = kBN;  // the columns of the tile that the row sees
    bool masked;
    if (kOneShot) {
      const int tok0 = kv0 + jt * kBN;
      lo = vis_lo - tok0;
      hi = min(vis_hi, kv1) - tok0;
      masked = __any_sync(0xffffffffu, lo > 0 || hi < kBN);
    } else {
      masked = jt == rag0 || jt == rag1;
      if (jt == rag0) hi = rag0_n;
      if (jt == rag1) hi = rag1_n;
    }
    const bool s_ok = wait_bar(&S->s_full[t], j & 1, S, p.status);
    tc_fence_after();
    uint32_t s[4][32];
#pragma unroll
    for (int c = 0; c < 4; ++c) tmem_ld32(tS + 32 * c, s[c]);
    ok = __all_sync(0xffffffffu, s_ok);
    tmem_wait_ld();
    if (!ok) {
      s_done = j;
      break;
    }
    // S is in registers: the next QK^T (of either tile) may overwrite it.
    tc_fence_before();
    if (j < s_expected) named_arrive(handoff::fwd_s_free(t, T::kOwnS));
    // At d = 64 the softmax warps set the pace (about 2000 clk per key tile
    // against 1040 of MMAs): a first look at p_free is sent off here, so that
    // its latency passes behind the row max.  At d = 128 it gained nothing.
    const bool p_is_free =
        T::kOwnS && j > 0 && mbar_test_wait(&S->p_free[t], (j - 1) & 1);
    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    if (masked) {
#pragma unroll
      for (int c = 0; c < 4; ++c) mask32(s[c], c, lo, hi);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) max32(s[c], mx);
    const float mrow = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]) * sl2;
    // The reference moves only when a row max passes it by more than the
    // threshold (decided per warp: TMEM accesses are warp-wide).
    const bool rescale =
        __any_sync(0xffffffffu, mrow > m_ref + kRescaleThreshold);
    float alpha = 1.f;
    if (rescale) {
      const float m_new = fmaxf(m_ref, mrow);
      alpha = ex2(m_ref - m_new);
      l *= alpha;
      m_ref = m_new;
    }
    const uint64_t neg2 = f2_pack(-m_ref, -m_ref);
    uint64_t acc[4] = {0, 0, 0, 0};
    uint32_t pk[2][16];
#pragma unroll
    for (int c = 0; c < 2; ++c) exp_pack32(s[c], sl2x2, neg2, pk[c], acc);
    // P_t(j - 1) has been consumed and O_t holds PV_t(0 .. j-1) (PV_t(j-1)
    // was issued right after this S, so this normally does not wait).
    const bool p_ok = j == 0 || p_is_free ||
                      wait_bar(&S->p_free[t], (j - 1) & 1, S, p.status);
    tc_fence_after();
    if (rescale && j > 0) {
      // Scale O_t in place before PV_t(j) accumulates against the new
      // reference.
#pragma unroll 1
      for (int c = 0; c < D / 8; ++c) {
        uint32_t r[8];
        tmem_ld8(tO + c * 8, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; ++i)
          r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
        tmem_st8(tO + c * 8, r);
      }
    }
    tmem_st16(tP, pk[0]);
    tmem_st16(tP + 16, pk[1]);
#pragma unroll
    for (int c = 2; c < 4; ++c) {
      exp_pack32(s[c], sl2x2, neg2, pk[c - 2], acc);
      tmem_st16(tP + 16 * c, pk[c - 2]);
    }
    l += acc_total(acc);
    ok = __all_sync(0xffffffffu, p_ok);
    tmem_wait_st();
    tc_fence_before();
    if (!ok) {
      s_done = j + 1;
      break;
    }
    named_arrive(handoff::fwd_p_full(t));
  }
  if (!ok) {
    struct Ops {
      Shared* S;
      int t;
      OwedWaits owed;
      __device__ __forceinline__ void wait_s(int j) {
        owed.wait(&S->s_full[t], j & 1);
      }
      __device__ __forceinline__ void wait_p(int j) {
        owed.wait(&S->p_free[t], j & 1);
      }
      __device__ __forceinline__ void arrive(int id) { named_arrive(id); }
    };
    handoff::fwd_softmax_rest(n, t, T::kOwnS, s_expected, s_done, j,
                              Ops{S, t, {}});
  }
  const bool have = ok && wait_bar_warp(&S->o_full, 0, S, p.status);
  const Work w = cta_work<kOneShot>(p);
  const int r_unit = t * kBM + wq * 32 + lane;  // row within the unit
  const int row = w.q0 + r_unit;
  // A part may hold nothing but scores of -inf for a row: its O is then 0, and
  // its log-sum-exp of -inf gives it no weight in the merge.  (A NaN l stays.)
  const float inv_l = w.part >= 0 && l == 0.f ? 0.f : 1.f / l;
  if (w.part >= 0) {
    // Partial result of a key range: O / l in fp32 (transposed, so a warp's
    // stores are contiguous) and the log2-domain log-sum-exp.
    if (!have) return;
    tc_fence_after();
    float* ws_o = p.ws + (size_t)w.part * D * kUnitRows;
    float* ws_l = p.ws_lse + (size_t)w.part * kUnitRows;
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
      uint32_t r[32];
      tmem_ld32(tO + c * 32, r);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const int64_t x = (int64_t)w.part * D * kUnitRows +
                          (int64_t)(c * 32 + i) * kUnitRows + r_unit;
        if (in_bounds(x, (int64_t)p.ws_parts * D * kUnitRows, p.status))
          ws_o[(c * 32 + i) * kUnitRows + r_unit] = __uint_as_float(r[i]) * inv_l;
      }
    }
    if (in_bounds((int64_t)w.part * kUnitRows + r_unit,
                  (int64_t)p.ws_parts * kUnitRows, p.status))
      ws_l[r_unit] = m_ref + __log2f(l);
    return;
  }
  // Whole unit: the tile's rows of O / l, as bf16, are staged in its Q tile
  // (free: every MMA has completed) as 128-byte-swizzled [128 x 64] boxes,
  // and leave as TMA tile stores (rows past the chunk fall outside the map
  // and are not written), instead of each thread writing 16-byte pieces of
  // its row at a stride of H d elements.  Every thread of the tile reaches
  // the barrier, also after a failed wait.
  uint8_t* tile = reinterpret_cast<uint8_t*>(S) - Layout<D>::shared_off +
                  Layout<D>::q(t, 0);
  const int rt = wq * 32 + lane;  // row within the tile
  if (have) {
    tc_fence_after();
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
      uint32_t r[32];
      tmem_ld32(tO + c * 32, r);
      tmem_wait_ld();
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 16; ++i)
        pk[i] = pack_bf16(__uint_as_float(r[2 * i]) * inv_l,
                          __uint_as_float(r[2 * i + 1]) * inv_l);
      uint8_t* line = tile + (c / 2) * kBox + rt * 128;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(line + ((((c % 2) * 4 + q) ^ (rt & 7)) << 4)) =
            make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
    }
    fence_proxy_async_smem();
  }
  tile_sync(kBarOStaged0 + t);
  if (wq == 0 && lane == 0 && have &&
      !*reinterpret_cast<volatile int*>(&S->abort)) {
    for (int bx = 0; bx < Layout<D>::kNB; ++bx)
      tma_store_4d(&p.o_map, tile + bx * kBox, bx * 64, w.q0 + t * kBM, w.h,
                   w.b);
    bulk_commit_group();
    bulk_wait_group0();
  }
  const int64_t lse_i = ((int64_t)w.b * p.heads + w.h) * p.q_tokens + row;
  if (have && p.lse != nullptr && row < p.q_tokens &&
      in_bounds(lse_i, (int64_t)p.batch * p.heads * p.q_tokens, p.status))
    p.lse[lse_i] = (m_ref + __log2f(l)) * 0.6931471805599453f;
}

// Merge the partial results of the split units: weights 2^(lse_i - m),
// O = sum_i w_i O_i / sum_i w_i, LSE = m + log2(sum_i w_i) (natural log out).
// A CTA merges a block of 32 query rows x 32 columns of one unit: thread
// (r, g) accumulates columns [4 g, 4 g + 4) of the block for row r, so a
// warp reads 32 consecutive rows of one column of a part (coalesced).  The
// parts are walked once, kPartUnroll at a time with all their loads issued
// together, the reference max moving with each group (what was accumulated
// is rescaled by 2^(m_old - m_new)): the merge reads tens of MB that are
// mostly still in L2, and it is the latency of those reads, not their
// volume, that sets its time.  The bf16 rows are written contiguously
// through shared memory.
constexpr int kMergeRows = 32;
constexpr int kMergeCols = 32;
constexpr int kMergeThreads = kMergeRows * kMergeCols / 4;  // 256
constexpr int kPartUnroll = 16;

template <int D>
__global__ void __launch_bounds__(kMergeThreads)
combine_kernel(const __grid_constant__ TcParams p) {
  constexpr int kCols = 4;  // columns per thread
  __shared__ __align__(16) uint16_t tile[kMergeRows][kMergeCols + 8];
  pdl_trigger();
  pdl_wait();  // the partial results of the attention kernel are complete
  const int ut = blockIdx.x;
  const int r = threadIdx.x % kMergeRows;
  const int g = threadIdx.x / kMergeRows;
  const int r_unit = blockIdx.y * kMergeRows + r;
  const int col0 = blockIdx.z * kMergeCols + g * kCols;
  int pair, bh;
  unit_coord(p, p.units_full + ut, pair, bh);
  const int h = bh % p.heads, b = bh / p.heads;
  const int row0 = pair * kQTiles * kBM + blockIdx.y * kMergeRows;
  if (row0 >= p.q_tokens) return;  // the whole block is past the chunk end
  const int k0 = ut * p.split;
  // every part this block reads lies in the workspace
  if (!in_bounds(k0 + p.split - 1, p.ws_parts, p.status)) return;
  const float* lse = p.ws_lse + (size_t)k0 * kUnitRows + r_unit;
  float m = -INFINITY;  // reference: the max of the parts seen so far
  float acc[kCols];
#pragma unroll
  for (int x = 0; x < kCols; ++x) acc[x] = 0.f;
  float wsum = 0.f;
  const float* src0 = p.ws + ((size_t)k0 * D + col0) * kUnitRows + r_unit;
  for (int i0 = 0; i0 < p.split; i0 += kPartUnroll) {
    float w8[kPartUnroll], v[kPartUnroll][kCols];
#pragma unroll
    for (int u = 0; u < kPartUnroll; ++u) {
      const bool have = i0 + u < p.split;
      w8[u] = have ? lse[(size_t)(i0 + u) * kUnitRows] : -INFINITY;
      const float* src = src0 + (size_t)(i0 + u) * D * kUnitRows;
#pragma unroll
      for (int x = 0; x < kCols; ++x)
        v[u][x] = have ? src[(size_t)x * kUnitRows] : 0.f;
    }
    float mg = m;
#pragma unroll
    for (int u = 0; u < kPartUnroll; ++u) mg = fmaxf(mg, w8[u]);
    if (mg == -INFINITY) continue;  // nothing finite yet
    // 0 on the first finite group (nothing accumulated), else <= 1
    const float sc = m == -INFINITY ? 0.f : ex2(m - mg);
    wsum *= sc;
#pragma unroll
    for (int x = 0; x < kCols; ++x) acc[x] *= sc;
    m = mg;
#pragma unroll
    for (int u = 0; u < kPartUnroll; ++u) {
      const float wi = ex2(w8[u] - m);  // 0 for the missing parts
      wsum += wi;
#pragma unroll
      for (int x = 0; x < kCols; ++x) acc[x] = fmaf(wi, v[u][x], acc[x]);
    }
  }
  const float inv = 1.f / wsum;
#pragma unroll
  for (int x = 0; x < kCols; x += 2)
    *reinterpret_cast<uint32_t*>(&tile[r][g * kCols + x]) =
        pack_bf16(acc[x] * inv, acc[x + 1] * inv);
  const int64_t lse_i = ((int64_t)b * p.heads + h) * p.q_tokens + row0 + r;
  if (blockIdx.z == 0 && g == 0 && p.lse != nullptr && row0 + r < p.q_tokens &&
      in_bounds(lse_i, (int64_t)p.batch * p.heads * p.q_tokens, p.status))
    p.lse[lse_i] = (m + __log2f(wsum)) * 0.6931471805599453f;
  __syncthreads();
  // Each row of the block is 32 bf16 = 4 16-byte pieces; one piece per
  // thread of the first 128.
  if (threadIdx.x < kMergeRows * kMergeCols / 8) {
    const int rr = threadIdx.x / (kMergeCols / 8);
    const int piece = threadIdx.x % (kMergeCols / 8);
    const int row = row0 + rr;
    const int64_t x = (int64_t)b * p.o_str.batch + (int64_t)row * p.o_str.token +
                      (int64_t)h * p.o_str.head + blockIdx.z * kMergeCols +
                      piece * 8;
    if (row < p.q_tokens && in_bounds(x, p.o_elems - 7, p.status))
      *reinterpret_cast<uint4*>(p.o + x) =
          *reinterpret_cast<const uint4*>(&tile[rr][piece * 8]);
  }
}

// The same merge for at most kFewParts parts per unit: many units then,
// and little to do for each, so a thread takes four rows x eight columns with
// 16-byte loads and writes each row's 16 bytes straight out, and a CTA takes
// all 256 rows of a unit x 32 columns.  (Blocks of 32 rows with 4-byte loads,
// as above: 2688 of them for 84 units, 11.1 us against 8.3; 56 units, 12.8
// against 7.8.  With fewer blocks than SMs this form loses: 4 units, 5.4 us
// against 4.6.)
constexpr int kFewParts = 4;
constexpr int kFewCols = 8;  // columns per thread
constexpr int kFewThreads = kUnitRows / 4 * (kMergeCols / kFewCols);  // 256

template <int D>
__global__ void __launch_bounds__(kFewThreads)
combine_few_kernel(const __grid_constant__ TcParams p) {
  pdl_trigger();
  pdl_wait();  // the partial results of the attention kernel are complete
  const int ut = blockIdx.x;
  const int r0 = threadIdx.x % (kUnitRows / 4) * 4;
  const int col0 = blockIdx.y * kMergeCols + threadIdx.x / (kUnitRows / 4) * kFewCols;
  const int parts = p.split;
  int pair, bh;
  unit_coord(p, p.units_full + ut, pair, bh);
  const int row0 = pair * kQTiles * kBM + r0;
  if (row0 >= p.q_tokens) return;
  const int k0 = ut * parts;
  // every part this block reads lies in the workspace
  if (!in_bounds(k0 + parts - 1, p.ws_parts, p.status)) return;
  const float* lse = p.ws_lse + (size_t)k0 * kUnitRows + r0;
  float w[kFewParts][4], m[4], wsum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int r = 0; r < 4; ++r) m[r] = -INFINITY;
#pragma unroll
  for (int u = 0; u < kFewParts; ++u) {
    float4 l = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (u < parts)
      l = *reinterpret_cast<const float4*>(lse + (size_t)u * kUnitRows);
    w[u][0] = l.x, w[u][1] = l.y, w[u][2] = l.z, w[u][3] = l.w;
#pragma unroll
    for (int r = 0; r < 4; ++r) m[r] = fmaxf(m[r], w[u][r]);
  }
#pragma unroll
  for (int u = 0; u < kFewParts; ++u)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      // 0 for the missing parts, and where no part has anything finite
      w[u][r] = ex2(w[u][r] - (m[r] == -INFINITY ? 0.f : m[r]));
      wsum[r] += w[u][r];
    }
  float acc[kFewCols][4] = {};
  const float* src = p.ws + ((size_t)k0 * D + col0) * kUnitRows + r0;
#pragma unroll
  for (int u = 0; u < kFewParts; ++u) {
    if (u >= parts) break;
#pragma unroll
    for (int x = 0; x < kFewCols; ++x) {
      const float4 v = *reinterpret_cast<const float4*>(
          src + ((size_t)u * D + x) * kUnitRows);
      acc[x][0] = fmaf(w[u][0], v.x, acc[x][0]);
      acc[x][1] = fmaf(w[u][1], v.y, acc[x][1]);
      acc[x][2] = fmaf(w[u][2], v.z, acc[x][2]);
      acc[x][3] = fmaf(w[u][3], v.w, acc[x][3]);
    }
  }
  const int h = bh % p.heads, b = bh / p.heads;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = row0 + r;
    if (row >= p.q_tokens) return;
    const float inv = 1.f / wsum[r];
    const int64_t x = (int64_t)b * p.o_str.batch + (int64_t)row * p.o_str.token +
                      (int64_t)h * p.o_str.head + col0;
    if (in_bounds(x, p.o_elems - 7, p.status))
      *reinterpret_cast<uint4*>(p.o + x) =
          make_uint4(pack_bf16(acc[0][r] * inv, acc[1][r] * inv),
                     pack_bf16(acc[2][r] * inv, acc[3][r] * inv),
                     pack_bf16(acc[4][r] * inv, acc[5][r] * inv),
                     pack_bf16(acc[6][r] * inv, acc[7][r] * inv));
    const int64_t lse_i = ((int64_t)b * p.heads + h) * p.q_tokens + row;
    if (col0 == 0 && p.lse != nullptr &&
        in_bounds(lse_i, (int64_t)p.batch * p.heads * p.q_tokens, p.status))
      p.lse[lse_i] = (m[r] + __log2f(wsum[r])) * 0.6931471805599453f;
  }
}

template <int D, bool kOneShot>
__global__ void __launch_bounds__(kThreads, 1)
chunk_attn_tc_kernel(const __grid_constant__ TcParams p) {
  using L = Layout<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Shared* S = reinterpret_cast<Shared*>(smem + L::shared_off);
  const int warp = threadIdx.x / 32;
  const int lane = threadIdx.x % 32;
  const Work w = cta_work<kOneShot>(p);

  if (warp == 9) {
    tmem_alloc(&S->tmem_base, kTmemCols);
    tmem_relinquish();
  }
  if (threadIdx.x == 256) {
    mbar_init(&S->q_full, 1);
    for (int s = 0; s < kKStages; ++s) {
      mbar_init(&S->k_full[s], 1);
      mbar_init(&S->k_empty[s], 1);
    }
    for (int s = 0; s < kVStages; ++s) {
      mbar_init(&S->v_full[s], 1);
      mbar_init(&S->v_empty[s], 1);
    }
    for (int t = 0; t < kQTiles; ++t) {
      mbar_init(&S->s_full[t], 1);
      mbar_init(&S->p_free[t], 1);
    }
    mbar_init(&S->o_full, 1);
    mbar_init(&S->drain, 1);
    S->abort = 0;
    S->wait_limit_ns = p.wait_limit_ns ? p.wait_limit_ns : kDefaultWaitLimitNs;
    fence_barrier_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S->tmem_base;
  // Set-up above touched no global memory; Q, K, V and the outputs may
  // belong to the previous kernel on the stream until it has completed.
  pdl_trigger();
  pdl_wait();

  if (warp == 8) {
    if (lane == 0) producer<D, true, kOneShot>(p, smem, S, w);
    __syncwarp();
  } else if (warp == 10) {
    if (lane == 0) producer<D, false, kOneShot>(p, smem, S, w);
    __syncwarp();
  } else if (warp == 9) {
    mma_issuer<D>(p, smem, S, tmem, w);
  } else if (warp == 11) {
    relay_role(p, S, w.n);
  } else {
    // A query tile that lies past the end of the chunk has no work.
    if (warp / 4 < w.nqt)
      softmax_role<D, kOneShot>(p, S, tmem, warp / 4, w.nqt, warp % 4, lane,
                                w.j0, w.n, w.kv0, w.kv1, w.q0, w.rev);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// ------------------------------------------------------------------ host

// 4-D bf16 map over (x = d, token, head, batch) with a box of 64 x 128
// (one 128-byte swizzled row per token); element strides in bytes.
int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// How a launch's units of two query tiles are spread over the SMs.
struct Split {
  int units_full;  // units that run whole, a CTA each
  int split;       // parts of each unit after those
  int cut;         // 0: equal parts; else the key tiles of the first of two
  int unit_rows;   // query rows of a unit
};

// Time of a key tile with one query tile, in units of one with two: its QK^T,
// softmax and PV follow one another (480p, 25 to 199 key tiles: 0.72-0.78).
constexpr double kOneTileCost = 0.75;

// Launches whose units have at most this many key tiles run a head's unit of
// one query tile after all others: it is the cheaper one to have left over
// (480p, chunk of 25 tiles: 49.5 -> 43.1 us; 3180 queries, 12, 24 or 48 heads,
// d = 64 and 128: 63 tiles 0.6-4 % faster, 157 and 243 tiles 0.2-2 %).  Run
// there, away from its head's other units, it reads the head's keys once more.
// Past the line that goes either way: the same queries over 313 and 454 tiles
// would gain 0.4-1.4 %, 720p's 7200 queries x 12 heads over 450 tiles lost
// 0.7 %; it stays in its place there.
constexpr int kShortsLastTiles = 256;

// Whole waves of units run whole; the units of a last partial wave are cut
// along the keys where that ends sooner.  Counted in key tiles of two query
// tiles (about 1.1 us at d = 128): a CTA costs its tiles and kCtaCost (set-up,
// first loads, filling and draining the pipeline, epilogue: 10.8k clk against
// 2240 per tile), the merge of the parts kMergeCost (its launch, here and on
// the host, and its fixed time) and 1 / kPartsPerTile for each.  Equal parts
// may take more than one round on the SMs.  Where most of the SMs have a unit
// already, two unequal parts: one for a CTA on each of `rem` SMs, the others go
// round the rest, at most q on one SM, and the cut lies where both end
// together.  (Equal parts in one round at most left 68 of 152 SMs idle for a
// 480p frame, 84 units of 63 tiles: 76.8 us, now 65.9 with the merge.)
//
// max_parts is what the allocation-free entry point's scratch holds, so that
// both entry points split alike, and it ends the second form early at d = 128:
// 95 units of 63 tiles are cut (66 us), 96 would need 192 parts of the 190 and
// run whole (76 us).
//
// Where twice the units still fit the SMs, units of one query tile are the
// other way to use more of them, and cost no merge (chunk of 600 queries x 2400
// keys, 12 heads, d = 64: 26.4 -> 21.2 us).
Split split_units(int units, int one_tile_units, int tiles, int sms,
                  int max_parts) {
  constexpr double kCtaCost = 5.0, kMergeCost = 6.0, kPartsPerTile = 40.0;
  const int rem = units % sms;
  Split best = {units, 1, 0, kUnitRows};
  if (rem == 0) return best;
  double best_cost = tiles + kCtaCost;
  auto merge = [&](int s) { return kMergeCost + rem * s / kPartsPerTile; };
  for (int s = 2; s * kMinTilesPerPart <= tiles && rem * s <= max_parts; ++s) {
    const int rounds = (rem * s + sms - 1) / sms;
    const double cost = rounds * ((tiles + s - 1) / s + kCtaCost) + merge(s);
    if (cost < best_cost) {
      best_cost = cost;
      best = {units - rem, s, 0, kUnitRows};
    }
  }
  if (2 * rem > sms && 2 * rem <= max_parts) {
    const int q = (rem + sms - rem - 1) / (sms - rem);
    const int cut = (int)ceil((q * (tiles + kCtaCost) - kCtaCost) / (1 + q));
    if (cut >= kMinTilesPerPart && tiles - cut >= kMinTilesPerPart &&
        cut + kCtaCost + merge(2) < best_cost) {
      best_cost = cut + kCtaCost + merge(2);
      best = {units - rem, 2, cut, kUnitRows};
    }
  }
  if (one_tile_units > units && one_tile_units <= sms &&
      kOneTileCost * tiles + kCtaCost < best_cost)
    best = {one_tile_units, 1, 0, kBM};
  return best;
}

// Units of a head.
int units_of(int q_tokens, int unit_rows) {
  return (q_tokens + unit_rows - 1) / unit_rows;
}

// Query pairs of a head with rows in both of their tiles.
int long_pairs(int q_tokens) {
  return (q_tokens + kBM - 1) / (kQTiles * kBM);
}

bool make_map(CUtensorMap* m, const void* base, int d, int64_t tokens,
              int heads, int batch, int64_t token_stride_b,
              int64_t head_stride_b, int64_t batch_stride_b) {
  EncodeTiledFn enc = encode_tiled_fn();
  if (enc == nullptr) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)tokens,
                              (cuuint64_t)heads, (cuuint64_t)batch};
  const cuuint64_t strides[3] = {(cuuint64_t)token_stride_b,
                                 (cuuint64_t)head_stride_b,
                                 (cuuint64_t)batch_stride_b};
  const cuuint32_t box[4] = {64, 128, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base),
             dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
cudaError_t launch_d(const AttnParams& a, cudaStream_t stream, int* launches) {
  TcParams p;
  memset(&p, 0, sizeof(p));
  const int64_t es = 2;  // bytes per bf16
  if (!make_map(&p.q_map, a.q, D, a.q_tokens, a.heads, a.batch,
                a.q_str.token * es, a.q_str.head * es, a.q_str.batch * es) ||
      !make_map(&p.o_map, a.o, D, a.q_tokens, a.heads, a.batch,
                a.q_str.token * es, a.q_str.head * es, a.q_str.batch * es))
    return cudaErrorInvalidValue;
  int tiles = 0;
  for (int s = 0; s < kMaxSegments; ++s) {
    if (s >= a.num_segments) {  // never read: seg_len stays 0
      p.k_map[s] = p.k_map[0];
      p.v_map[s] = p.v_map[0];
      continue;
    }
    // The map ends where the segment ends: keys past it read as zeros.
    const int64_t end = a.seg_start[s] + a.seg_len[s];
    if (!make_map(&p.k_map[s], a.k, D, end, a.heads, a.batch,
                  a.kv_str.token * es, a.kv_str.head * es, a.kv_str.batch * es) ||
        !make_map(&p.v_map[s], a.v, D, end, a.heads, a.batch,
                  a.kv_str.token * es, a.kv_str.head * es, a.kv_str.batch * es))
      return cudaErrorInvalidValue;
    p.seg_start[s] = (int32_t)a.seg_start[s];
    p.seg_len[s] = a.seg_len[s];
    const int t = (p.seg_len[s] + kBN - 1) / kBN;
    if (s == 0) p.seg_tiles0 = t;
    tiles += t;
  }
  p.total_tiles = tiles;
  p.o = a.o;
  p.lse = a.lse;
  p.o_str = a.q_str;
  p.o_elems = a.q_str.batch * a.batch;
  p.q_tokens = a.q_tokens;
  p.heads = a.heads;
  p.batch = a.batch;
  p.ws_parts = a.workspace_parts;
  p.scale_log2 = a.scale_log2;
  p.status = a.status;
  p.wait_limit_ns = a.wait_limit_ns;
  p.inject_stall = a.inject_stall;
  p.ws = a.workspace;

  const int bh = a.heads * a.batch;
  const int units = units_of(a.q_tokens, kUnitRows) * bh;
  p.sms = sm_count();
  const Split sp = split_units(units, units_of(a.q_tokens, kBM) * bh, tiles,
                               p.sms, split_parts(D));
  p.unit_rows = sp.unit_rows;
  p.q_pairs = units_of(a.q_tokens, sp.unit_rows);
  p.long_pairs = sp.unit_rows == kUnitRows && tiles <= kShortsLastTiles
                     ? long_pairs(a.q_tokens)
                     : p.q_pairs;
  p.units_full = sp.units_full;
  p.tail_units = p.q_pairs * bh - sp.units_full;
  p.split = sp.split;
  p.cut = sp.cut;
  p.ws_lse = p.ws + (size_t)a.workspace_parts * D * kUnitRows;
  const int grid = p.units_full + p.tail_units * p.split;
  const int smem = Layout<D>::bytes;
  cudaError_t e = cudaFuncSetAttribute(
      chunk_attn_tc_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(chunk_attn_tc_kernel<D, false>, dim3(grid), dim3(kThreads),
                 smem, stream, p);
  if (e != cudaSuccess) return e;
  *launches = 1;
  if (p.split > 1) {
    const bool few =
        p.split <= kFewParts && p.tail_units * (D / kMergeCols) >= p.sms;
    e = few ? launch_pdl(combine_few_kernel<D>,
                         dim3(p.tail_units, D / kMergeCols),
                         dim3(kFewThreads), 0, stream, p)
            : launch_pdl(combine_kernel<D>,
                         dim3(p.tail_units, kUnitRows / kMergeRows,
                              D / kMergeCols),
                         dim3(kMergeThreads), 0, stream, p);
    if (e != cudaSuccess) return e;
    *launches = 2;
  }
  return cudaSuccess;
}

// One unit per pair of query tiles, no key splitting: the units differ in
// length (later chunks see more keys) and run longest first.
template <int D>
cudaError_t launch_oneshot_d(const OneShotParams& a, cudaStream_t stream) {
  TcParams p;
  memset(&p, 0, sizeof(p));
  const int64_t es = 2;
  const int64_t tok = (int64_t)a.heads * D, bat = (int64_t)a.seq_tokens * tok;
  if (!make_map(&p.q_map, a.q, D, a.seq_tokens, a.heads, a.batch, tok * es,
                D * es, bat * es) ||
      !make_map(&p.k_map[0], a.k, D, a.seq_tokens, a.heads, a.batch, tok * es,
                D * es, bat * es) ||
      !make_map(&p.v_map[0], a.v, D, a.seq_tokens, a.heads, a.batch, tok * es,
                D * es, bat * es) ||
      !make_map(&p.o_map, a.o, D, a.seq_tokens, a.heads, a.batch, tok * es,
                D * es, bat * es))
    return cudaErrorInvalidValue;
  p.k_map[1] = p.k_map[0];
  p.v_map[1] = p.v_map[0];
  p.o = a.o;
  p.lse = a.lse;
  p.o_str.token = tok;
  p.o_str.head = D;
  p.o_str.batch = bat;
  p.o_elems = bat * a.batch;
  p.q_tokens = a.seq_tokens;
  p.heads = a.heads;
  p.batch = a.batch;
  p.scale_log2 = a.scale_log2;
  p.status = a.status;
  p.inject_stall = a.inject_stall;
  p.wait_limit_ns = a.wait_limit_ns;
  p.seq_tokens = a.seq_tokens;
  p.chunk_tokens = a.chunk_tokens;
  p.window = a.window;
  p.sms = sm_count();
  // Units of one query tile where twice the units still fit the SMs: 9000
  // tokens, 2 heads, no window: 98.1 -> 75.2 us; 2400 tokens, 8 heads, W = 1:
  // 32.0 -> 23.7.  (With more units they would take a second round.)
  p.unit_rows = units_of(a.seq_tokens, kBM) * a.heads * a.batch <= p.sms
                    ? kBM
                    : kUnitRows;
  p.q_pairs = units_of(a.seq_tokens, p.unit_rows);
  p.split = 1;
  const int grid = p.q_pairs * a.heads * a.batch;
  p.units_full = grid;
  const int smem = Layout<D>::bytes;
  cudaError_t e = cudaFuncSetAttribute(
      chunk_attn_tc_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(chunk_attn_tc_kernel<D, true>, dim3(grid), dim3(kThreads),
                    smem, stream, p);
}

}  // namespace

cudaError_t launch_blockcausal_attn(const OneShotParams& p, cudaStream_t stream) {
  if (p.head_dim == 64) return launch_oneshot_d<64>(p, stream);
  if (p.head_dim == 128) return launch_oneshot_d<128>(p, stream);
  return cudaErrorInvalidValue;
}

cudaError_t launch_chunk_attn(const AttnParams& p, cudaStream_t stream,
                              int* launches) {
  *launches = 0;
  if (p.head_dim == 64) return launch_d<64>(p, stream, launches);
  if (p.head_dim == 128) return launch_d<128>(p, stream, launches);
  return cudaErrorInvalidValue;
}

// Resolved once; C++ initialises the function-local static exactly once even
// when several host threads make their first call at the same time.
EncodeTiledFn encode_tiled_fn() {
  static const EncodeTiledFn fn = []() -> EncodeTiledFn {
    cudaDriverEntryPointQueryResult q;
    void* ptr = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                         cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(ptr);
    cudaGetLastError();
    return nullptr;
  }();
  return fn;
}

}  // namespace fastvr
