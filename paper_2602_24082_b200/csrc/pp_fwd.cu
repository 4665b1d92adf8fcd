// Forward kernel: O = softmax(mask(scale Q K^T)) V and LSE over the plan's visible tiles.
//
// Persistent, warp-specialised CTA (one per SM):
//   warp 0      TMA producer: draws and decodes the work units (the only reader of the plan's
//               tile list; the other roles get a decoded record through shared memory), loads
//               the Q tiles of the unit's two query heads, then the K / V tiles of every
//               visible key tile in two-deep stages {V(j), K(j + 1)} (one barrier pair each)
//   warp 1      MMA issuer (one thread): S = Q K^T and O += P V with tcgen05.mma, fp32 in TMEM
//   warps 2-9   softmax warps of slot 0: two threads per query row (= TMEM lane), 64 key
//               columns each
//   warps 10-17 softmax warps of slot 1
//   warps 18-19 optional: clear the backward's fp32 dQ accumulator for the unit's rows
// A work unit is (query tile, KV head, pair of query heads of that KV head): both slots see
// the same keys and the same mask, so every K / V tile staged in shared memory feeds two
// S tiles.  The last head of an odd number of heads per KV head, and every head where there is one
// per KV head, takes two query tiles of a segment into the slots (kPaired below) or leaves slot 1 empty.
// While one slot's warpgroup does its exponentials the tensor core works on the other slot (order: PV_0(j), QK_0(j+1), PV_1(j), QK_1(j+1), ...).  P (bf16) overwrites columns
// [0,32) and [64,96) of its S tile in tensor memory (each half-row thread inside the columns it
// has read itself) and is the A operand of the second MMA; V is
// its MN-major B operand straight from the TMA layout.  O is rescaled lazily: only when a
// row's running maximum grew by more than 2^8 since the value used for scaling.
// TMEM: S0 | S1 | O0 | O1, 128 columns each.  At D = 64 narrower accumulators leave room for P beside S
// (kOwnP below): S0 | S1 | P0 | P1 | O0 | O1, and a slot's next QK is issued as soon as its scores are read.
// Query tiles are those of the segments or, with many short ones, mixed tiles (kMixed below).
#include <algorithm>
#include <type_traits>

#include "pp_dev.cuh"

namespace pp {
namespace {

struct FwdParams {
  int32_t* header;
  const Tile* tiles;       // tiles of the segments
  const uint8_t* tile_unit;  // (paired tiles)
  const QTile* qtiles;     // (mixed tiles)
  const int32_t* key_end;  // (mixed tiles)
  const int32_t* order;    // the tiles, longest work first
  __nv_bfloat16* o;
  float* lse;
  float* dq_clear;  // optional: the backward's fp32 dQ accumulator [T][Hq][D], cleared here
  int T, Hq, Hkv;
  float scale_log2;  // softmax scale * log2(e)
};

constexpr int kFwdThreads = 640;
constexpr uint32_t kFwdTmemCols = 512;
constexpr float kRescaleThreshold = 8.f;  // log2 units
constexpr int kEarlySteps = 3;            // of a half row's four 16-key steps of P, those handed over first

enum FwdBar : int {
  kQFull = 0,   // [2] per slot
  kQEmpty = 2,  // [2]
  kKFull = 4,   // [2] per K / V stage: full
  kKEmpty = 6,  // [2]                 empty
  kSFull = 8,   // [2] per slot
  kPFull = 10,
  kODone = 12,
  kOFree = 14,
  kSchedFullF = 16,   // [2] unit ids handed from the producer to the other roles
  kSchedEmptyF = 18,  // [2] 17 arrivals: MMA thread + 16 softmax warps (+ 2 clearing warps)
  kPRest = 20,        // [2] per slot: the late columns of P (kPFull: the early ones)
  kSFree = 22,        // [2] per slot, with columns of its own for P: the scores are read
  kPFree = 24,        // [2]                                          PV has read P
  kNumFwdBars = 26
};

template <int D>
struct FwdSmem {
  static constexpr int kTileBytes = 128 * D * 2;
  static constexpr int kQ = 0, kK = 2 * kTileBytes, kV = 4 * kTileBytes, kBars = 6 * kTileBytes;
  static constexpr int kSched = kBars + 256;          // two decoded unit records of 8 ints
  static constexpr int kXch = kSched + 64;            // float [2 slots][3 buffers][128 rows][2 halves]
  static constexpr int kTotal = kXch + 6144 + 1024;   // + slack to align the base to 1024 B
};

struct KvTile {
  int start, len;
  bool diag;
};

template <typename T>
__device__ __forceinline__ KvTile kv_tile_of(const T& t, int j, int n0, int n1) {
  KvTile k;
  if (j < n0) {
    k.start = t.kv0_start + j * kTile;
    k.len = min(kTile, t.kv0_len - j * kTile);
    k.diag = false;
  } else if (j < n0 + n1) {
    k.start = t.kv1_start + (j - n0) * kTile;
    k.len = min(kTile, t.kv1_len - (j - n0) * kTile);
    k.diag = false;
  } else {
    k.start = t.start;
    k.len = t.len;
    k.diag = true;
  }
  return k;
}

// What the slots of a unit hold: two query heads of a tile, or of a tile that may have rows of several
// segments (kMixed), or (kPaired) for the head left over by an odd number of heads per KV head two tiles of a
// segment, one behind the other: slot 1 has the unit's tile, slot 0 the one before it, whose keys are those of
// slot 1 but the last tile.
enum FwdMode : int { kPlain, kMixedTiles, kPairedTiles };

template <int kMode>
struct Unit {
  std::conditional_t<kMode == kMixedTiles, QTile, Tile> tile;
  int h0, kvh, nslots, n0, n1, ntiles;
  bool paired;
};

// Units are handed out dynamically in the plan's longest-work-first order: a CTA starts with the
// unit of its own index, for later ones the producer draws from a global counter (header[4]) when
// the CTA is ready for more; it passes them on through a two-entry shared-memory ring; header[6] counts
// finished CTAs and the last one resets both counters for the next launch.
constexpr int kHdrFwdNext = 4, kHdrFwdDone = 6;

// (a unit may be empty: no slots)
template <int kMode>
__device__ __forceinline__ bool get_unit(const FwdParams& prm, int u, int ntiles_total, Unit<kMode>& un) {
  const int r = prm.Hq / prm.Hkv, npairs = (r + 1) >> 1, per_tile = prm.Hkv * npairs;
  const int ord = u / per_tile;
  if (ord >= ntiles_total) return false;
  const int rem = u - ord * per_tile;
  un.kvh = rem / npairs;
  const int pair = rem - un.kvh * npairs;
  un.h0 = un.kvh * r + 2 * pair;
  un.nslots = (2 * pair + 1 < r) ? 2 : 1;
  const int t = prm.order[ord];
  if constexpr (kMode == kMixedTiles) un.tile = prm.qtiles[t];
  else un.tile = prm.tiles[t];
  un.paired = false;
  if (kMode == kPairedTiles && un.nslots == 1) {
    un.nslots = prm.tile_unit[t];
    un.paired = un.nslots == 2;
  }
  un.n0 = (un.tile.kv0_len + kTile - 1) / kTile;
  un.n1 = (un.tile.kv1_len + kTile - 1) / kTile;
  un.ntiles = un.n0 + un.n1 + 1;
  return true;
}

// D: head dimension of the shared-memory tiles (64 or 128); DV <= D: head dimension of the
// tensors in global memory.  For DV < D (96 in tiles of 128) the TMA loads fill the columns
// past DV with zeros, so only the loops over the head dimension, the N of the second GEMM and
// everything that addresses global memory know about DV.
// kMode: see FwdMode.  With mixed tiles the masks of a tile's own keys and of the first rows' response
// change.  (A template parameter because the more general masks take registers from the loop: 3.5 %
// on two rows of 32768 tokens in one instance for all.)
template <int D, int kMode, int DV = D>
__global__ void __launch_bounds__(kFwdThreads, 1)
fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
           const __grid_constant__ CUtensorMap tm_v, FwdParams prm) {
  using L = FwdSmem<D>;
  constexpr bool kMixed = kMode == kMixedTiles, kPaired = kMode == kPairedTiles;
  // P in columns of its own: the chain of a slot is then softmax -> QK -> softmax, without PV.
  // 16384 tokens, 32 / 8 heads 214 -> 205 us, 12000, 16 / 16 heads 184 -> 170, 28 / 4 190 -> 180.  Not with
  // mixed tiles, whose units are short: 12000 tokens in short segments, 32 / 8 heads 98.3 -> 100.4.
  constexpr bool kOwnP = D == 64 && !kMixed;
  constexpr uint32_t kTmemP = kOwnP ? 256 : 0, kTmemPStep = kOwnP ? 64 : 128, kPHalf = kOwnP ? 32 : 64;
  constexpr uint32_t kTmemO = kOwnP ? 384 : 256, kTmemOStep = kOwnP ? 64 : 128;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (known to be uniform in the warp)

  dependency_wait();
  if (prm.header[0] != kStatusOk) return;
  const int ntiles_total = prm.header[kMixed ? kHdrNumQTiles : kHdrNumTiles];
#ifdef PP_DEBUG_COUNTERS
  const long long t_kernel0 = clock64();
#endif

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t sQ = base + L::kQ, sK = base + L::kK, sV = base + L::kV;
  const uint32_t bars = base + L::kBars;
  auto bar = [&](int i) { return bars + 8u * uint32_t(i); };
  const uint32_t tmem_slot = bars + 8 * kNumFwdBars;
  volatile uint32_t* tmem_slot_p = reinterpret_cast<volatile uint32_t*>(gbase + L::kBars + 8 * kNumFwdBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kBars + 8 * kNumFwdBars + 8);

  if (tid == 0) {
    for (int i = 0; i < kNumFwdBars; ++i) {
      const bool wg_count = (i >= kPFull && i < kPFull + 2) || (i >= kOFree && i < kOFree + 2) ||
                            (i >= kPRest && i < kPFree);
      const bool sched_empty = (i >= kSchedEmptyF && i < kSchedEmptyF + 2);
      // unit records are released by the MMA thread, the 16 softmax warps and, when the dQ
      // accumulator is cleared here, the two clearing warps
      mbar_init(bar(i), wg_count ? 256 : (sched_empty ? (prm.dq_clear ? 19 : 17) : 1));
    }
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, kFwdTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_p;
  // Ring of two decoded unit records (producer -> MMA thread and softmax warps): the producer
  // alone reads the plan's tile list; the other roles get what they need from shared memory.
  volatile int* sched = reinterpret_cast<volatile int*>(gbase + L::kSched);
  bool first_draw = true;
  auto fetch_unit = [&](uint32_t n, Unit<kMode>& un) -> bool {  // producer thread
    wait_bar(bar(kSchedEmptyF + (n & 1)), ((n >> 1) & 1) ^ 1, abort_flag, prm.header, 90);
    bool ok;
    do {
      // after a wait has given up, no more work is drawn: the end marker goes out instead
      const int u = *abort_flag  ? 0x7fffffff
                    : first_draw ? int(blockIdx.x)
                                 : int(gridDim.x) + atomicAdd(&prm.header[kHdrFwdNext], 1);
      first_draw = false;
      ok = get_unit<kMode>(prm, u, ntiles_total, un);
    } while (kPaired && ok && un.nslots == 0);
    volatile int* e = sched + (n & 1) * 8;
    e[0] = un.tile.start;
    if constexpr (kMixed) e[1] = un.tile.len | un.tile.first_rows << 8;
    else e[1] = un.tile.len;
    e[2] = un.h0;
    e[3] = ok ? un.nslots | (kPaired && un.paired ? 4 : 0) : 0;  // 0 slots marks the end of the work list
    e[4] = un.n0;
    e[5] = un.n1;
    e[6] = un.tile.kv0_len - (un.n0 - 1) * kTile;
    e[7] = un.tile.kv1_len - (un.n1 - 1) * kTile;
    mbar_arrive(bar(kSchedFullF + (n & 1)));
    return ok;
  };
  // Consumers: read the record into plain scalars (kept in registers) and release the entry.
#define PP_TAKE_UNIT(n, whole_warp)                                                              \
  const bool u_ok = wait_bar(bar(kSchedFullF + ((n) & 1)), ((n) >> 1) & 1, abort_flag, prm.header, 91); \
  const volatile int* u_e = sched + ((n) & 1) * 8;                                               \
  const int u_start = u_e[0], u_len1 = u_e[1], u_len = kMixed ? u_len1 & 255 : u_len1;           \
  const int u_h0 = u_e[2], u_slots = u_ok ? u_e[3] : 0;                                          \
  const int u_nslots = kPaired ? u_slots & 3 : u_slots;                                          \
  const bool u_paired = kPaired && (u_slots & 4);                                                \
  const int u_n0 = u_e[4], u_n1 = u_e[5], u_last0 = u_e[6], u_last1 = u_e[7];                    \
  const int u_ntiles = u_n0 + u_n1 + 1;                                                          \
  if (whole_warp) {                                                                              \
    __syncwarp();                                                                                \
    if (lane == 0) mbar_arrive(bar(kSchedEmptyF + ((n) & 1)));                                   \
  } else {                                                                                       \
    mbar_arrive(bar(kSchedEmptyF + ((n) & 1)));                                                  \
  }                                                                                              \
  (void)u_start, (void)u_len, (void)u_h0, (void)u_paired;                                        \
  /* keys of visible key tile j: only the last tile of a full range and the diagonal tile */    \
  /* can be shorter than 128 */                                                                  \
  auto u_klen = [=](int j) -> int {                                                              \
    return (j + 1 == u_n0) ? u_last0 : (j + 1 == u_n0 + u_n1) ? u_last1 : (j + 1 == u_ntiles) ? u_len : kTile; \
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (elect_one()) {
      uint32_t kc = 0, qc[2] = {0, 0};
      Unit<kMode> un;
      for (uint32_t un_i = 0; fetch_unit(un_i, un); ++un_i) {
        for (int s = 0; s < un.nslots; ++s) {
          wait_bar(bar(kQEmpty + s), (qc[s] & 1) ^ 1, abort_flag, prm.header, 20 + s);
          mbar_expect_tx(bar(kQFull + s), L::kTileBytes);
          for (int b = 0; b < D / 64; ++b)
            tma_load_3d(sQ + s * L::kTileBytes + b * kBoxBytes, &tm_q, b * 64, un.paired ? un.h0 : un.h0 + s,
                        un.paired && s == 0 ? un.tile.start - kTile : un.tile.start, bar(kQFull + s));
          ++qc[s];
        }
        // K and V travel in stages {V(j), K(j + 1)} -- what one period of the MMA thread
        // consumes -- with ONE full / empty barrier pair per stage (the first stage of a unit
        // holds only K(0), the last only V(last)): every barrier operation costs the MMA
        // thread 100 - 150 cycles of tensor-pipe time, so it gets one wait and one commit per
        // period instead of two of each.  Stage n uses the K and V buffers n & 1.
        auto load_stage = [&](int jv, int jk) {   // key tile of V and of K in this stage, or -1
          const uint32_t st = kc & 1;
          wait_bar(bar(kKEmpty + st), ((kc >> 1) & 1) ^ 1, abort_flag, prm.header, 22);
          mbar_expect_tx(bar(kKFull + st), (jv >= 0 && jk >= 0 ? 2 : 1) * L::kTileBytes);
          if (jk >= 0) {
            const KvTile kt = kv_tile_of(un.tile, jk, un.n0, un.n1);
            for (int b = 0; b < D / 64; ++b)
              tma_load_3d(sK + st * L::kTileBytes + b * kBoxBytes, &tm_k, b * 64, un.kvh, kt.start,
                          bar(kKFull + st));
          }
          if (jv >= 0) {
            const KvTile kt = kv_tile_of(un.tile, jv, un.n0, un.n1);
            for (int b = 0; b < D / 64; ++b)
              tma_load_3d(sV + st * L::kTileBytes + b * kBoxBytes, &tm_v, b * 64, un.kvh, kt.start,
                          bar(kKFull + st));
          }
          ++kc;
        };
        load_stage(-1, 0);
        for (int j = 0; j < un.ntiles && !*abort_flag; ++j)
          load_stage(j, j + 1 < un.ntiles ? j + 1 : -1);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The tensor pipe takes about two MMAs ahead of the one it executes, so whatever the issuing
    // thread does between two groups of MMAs beyond that is idle tensor-pipe time: the loop
    // below keeps it to a minimum (descriptors and instruction descriptors precomputed, barrier
    // addresses and parities kept in registers, one branch for the common case of full 128-key
    // tiles).  The branch is an elect.sync and not `lane == 0`: with the latter eight MMAs took
    // the thread 494 cycles to issue whatever their N (62 each: operands moved to uniform
    // registers one by one), with the former 402 at N = 128 and 322 at N = 64.  A launch on two
    // rows of 32768 tokens (Hq / Hkv 32 / 8, D 128) went from 11.3 to 10.4 M cycles, eight
    // 1100-token rows from 143 to 132 us, head_dim 64 from 248 to 227 us.
    if (elect_one()) {
      uint32_t kc = 0, tc0 = 0, tc1 = 0, uc0 = 0, uc1 = 0;
      constexpr uint32_t idesc_o = make_idesc(128, DV, 0, 1);
      constexpr uint32_t idesc_full = make_idesc(128, 128, 0, 0);
      constexpr uint32_t kStageStep = uint32_t(L::kTileBytes >> 4);
      const uint32_t dq0 = kmajor_base(sQ), dk0 = kmajor_base(sK), dv0 = mnmajor_base(sV);
      // length of key tile j of a unit: only the last tile of each visible range and the
      // diagonal tile can be shorter than 128
      auto issue_qk = [&](int s, uint32_t kstage, int k_len) {
        const uint32_t a = dq0 + s * kStageStep, b = dk0 + kstage * kStageStep;
        const uint32_t tS = tmem + s * 128;
        if (k_len == kTile) {
#pragma unroll
          for (int kk = 0; kk < DV / 16; ++kk)
            mma_ss(tS, a + kmajor_off(kk), b + kmajor_off(kk), idesc_full, kk > 0);
        } else {
          const uint32_t idesc_s = make_idesc(128, 0, 0, 0) | (uint32_t(((k_len + 15) >> 4) << 1) << 17);
#pragma unroll
          for (int kk = 0; kk < DV / 16; ++kk)
            mma_ss(tS, a + kmajor_off(kk), b + kmajor_off(kk), idesc_s, kk > 0);
        }
        mma_commit(bar(kSFull + s));
      };
      // P arrives in two parts: of the four k-steps (16 keys each) of each half row the first
      // kEarlySteps, then the others
      auto issue_pv = [&](int s, uint32_t vstage, int k_len, bool first, bool last, uint32_t par) {
        const uint32_t b = dv0 + vstage * kStageStep;
        const uint32_t tP = tmem + kTmemP + s * kTmemPStep, tO = tmem + kTmemO + s * kTmemOStep;
        auto p_at = [&](int kk) { return tP + (kk < 4 ? kk * 8 : kPHalf + (kk - 4) * 8); };
        if (k_len == kTile && !first) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            if ((kk & 3) < kEarlySteps)
              mma_ts(tO, p_at(kk), b + mnmajor_off(kk), idesc_o, 1);
          wait_bar(bar(kPRest + s), par, abort_flag, prm.header, 39);
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            if ((kk & 3) >= kEarlySteps)
              mma_ts(tO, p_at(kk), b + mnmajor_off(kk), idesc_o, 1);
        } else {
          const int ksteps = (k_len + 15) >> 4;
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            if ((kk & 3) < kEarlySteps && kk < ksteps)
              mma_ts(tO, p_at(kk), b + mnmajor_off(kk), idesc_o,
                     !first || (kk > 0));
          wait_bar(bar(kPRest + s), par, abort_flag, prm.header, 39);
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            if ((kk & 3) >= kEarlySteps && kk < ksteps)
              mma_ts(tO, p_at(kk), b + mnmajor_off(kk), idesc_o, 1);
        }
        // the accumulator is only waited for after the unit's last PV (the lazy rescale, rare,
        // runs after S of the next tile is complete, whose commit covers this PV as well)
        if (kOwnP) mma_commit(bar(kPFree + s));
        if (last) mma_commit(bar(kODone + s));
      };
      for (uint32_t un_i = 0;; ++un_i) {
        PP_TAKE_UNIT(un_i, false)
        if (u_nslots == 0) break;
        const bool two = u_nslots == 2;
        const int nt0 = u_ntiles - int(u_paired);   // key tiles of slot 0
        wait_bar(bar(kQFull + 0), uc0 & 1, abort_flag, prm.header, 30);
        if (two) wait_bar(bar(kQFull + 1), uc1 & 1, abort_flag, prm.header, 31);
        int cur_len = u_klen(0);
        wait_bar(bar(kKFull + (kc & 1)), (kc >> 1) & 1, abort_flag, prm.header, 32);
        tc_fence_after();
        issue_qk(0, kc & 1, cur_len);
        if (nt0 == 1) mma_commit(bar(kQEmpty + 0));
        if (two) {
          issue_qk(1, kc & 1, cur_len);
          if (u_ntiles == 1) mma_commit(bar(kQEmpty + 1));
        }
        mma_commit(bar(kKEmpty + (kc & 1)));
        ++kc;
        for (int j = 0; j < u_ntiles; ++j) {
          const bool has_next = j + 1 < u_ntiles;
          const int nx_len = has_next ? u_klen(j + 1) : 0;
          const uint32_t vst = kc & 1, kst = kc & 1;   // stage {V(j), K(j + 1)}
          wait_bar(bar(kKFull + kst), (kc >> 1) & 1, abort_flag, prm.header, 33);
          if (!kPaired || j < nt0) {   // slot 0
            const bool has_next0 = j + 1 < nt0;
            if (kOwnP && has_next0) {
              wait_bar(bar(kSFree + 0), tc0 & 1, abort_flag, prm.header, 27);
              tc_fence_after();
              issue_qk(0, kst, nx_len);
              if (j + 2 == nt0) mma_commit(bar(kQEmpty + 0));
            }
            wait_bar(bar(kPFull + 0), tc0 & 1, abort_flag, prm.header, 35);
            if (j == 0) wait_bar(bar(kOFree + 0), (uc0 & 1) ^ 1, abort_flag, prm.header, 37);
            tc_fence_after();
            issue_pv(0, vst, cur_len, j == 0, !has_next0, tc0 & 1);
            ++tc0;
            if (!kOwnP && has_next0) {
              issue_qk(0, kst, nx_len);
              if (j + 2 == nt0) mma_commit(bar(kQEmpty + 0));
            }
          }
          if (two) {
            if (kOwnP && has_next) {
              wait_bar(bar(kSFree + 1), tc1 & 1, abort_flag, prm.header, 28);
              tc_fence_after();
              issue_qk(1, kst, nx_len);
              if (j + 2 == u_ntiles) mma_commit(bar(kQEmpty + 1));
            }
            wait_bar(bar(kPFull + 1), tc1 & 1, abort_flag, prm.header, 36);
            if (j == 0) wait_bar(bar(kOFree + 1), (uc1 & 1) ^ 1, abort_flag, prm.header, 38);
            tc_fence_after();
            issue_pv(1, vst, cur_len, j == 0, !has_next, tc1 & 1);
            ++tc1;
            if (!kOwnP && has_next) {
              issue_qk(1, kst, nx_len);
              if (j + 2 == u_ntiles) mma_commit(bar(kQEmpty + 1));
            }
          }
          mma_commit(bar(kKEmpty + kst));
          ++kc;
          cur_len = nx_len;
        }
        ++uc0;
        if (two) ++uc1;
      }
    }
  } else if (warp >= 18) {
    // ------------------------------------------------------------ clearing warps (optional)
    // The kernel is compute-bound and leaves most of the memory bandwidth idle: when the
    // caller passes the backward's scratch, these two warps write zeros over the rows of the
    // fp32 dQ accumulator that belong to the unit's query tile and heads, so that the
    // backward needs no clearing pass.  Every (token, query head) row belongs to exactly one
    // unit and slot.
    if (prm.dq_clear) {
      const int cl = (warp - 18) * 32 + lane;  // 0..63
      for (uint32_t un_i = 0;; ++un_i) {
        PP_TAKE_UNIT(un_i, true)
        if (u_nslots == 0) break;
        constexpr int kChunks = DV / 4;  // 16-byte chunks per row
        for (int sl = 0; sl < u_nslots; ++sl) {
          const bool before = u_paired && sl == 0;   // the tile before the unit's
          const int total = (before ? kTile : u_len) * kChunks;
          float* base = prm.dq_clear + (size_t(before ? u_start - kTile : u_start) * prm.Hq +
                                        (u_paired ? u_h0 : u_h0 + sl)) * DV;
          for (int c = cl; c < total; c += 64) {
            const int r = c / kChunks, col = c - r * kChunks;
            *reinterpret_cast<float4*>(base + size_t(r) * prm.Hq * DV + col * 4) =
                make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------ softmax warps
    // Eight warps per slot: two threads share a query row (= TMEM lane), each owning 64 of
    // the tile's 128 key columns and D/2 of the output columns.  Halving the work per thread
    // keeps one slot's softmax shorter than the other slot's MMA phase, so the two slots'
    // exponentials do not pile up on the same MUFU at the same time.  The two halves of a row
    // exchange their partial maxima (every tile) and sums (once per unit) through shared
    // memory, guarded by a 64-thread named barrier per (slot, lane quarter).
    const int lw = warp - 2;                  // 0..15
    const int s = lw >> 3;                    // slot
    const int half = (lw >> 2) & 1;           // column half of the row
    const int qd = warp & 3;                  // lane quarter this warp may touch
    const int row = 32 * qd + lane;
    const int bar_id = 1 + s * 4 + qd;        // named barrier shared with the partner warp
    const uint32_t lane_base = tmem + (uint32_t(32 * qd) << 16);
    const uint32_t tS = lane_base + s * 128 + half * 64;   // my S columns; P goes to their start
    const uint32_t tP = lane_base + kTmemP + s * kTmemPStep + half * kPHalf;   //   or to its own
    const uint32_t tO = lane_base + kTmemO + s * kTmemOStep + half * (D / 2);
    // What the two halves of a row exchange, one buffer each for the largest exponentials, the maxima
    // and the row sums: a value is then only overwritten behind a barrier, or a wait for a tile that
    // needs the partner's P, that follows the partner's read.
    float* const xch_exp = reinterpret_cast<float*>(gbase + L::kXch) + s * 768 + row * 2;
    float* const xch_max = xch_exp + 256, * const xch_sum = xch_exp + 512;
    uint32_t tcS = 0, ucS = 0;
    for (uint32_t un_i = 0;; ++un_i) {
      PP_TAKE_UNIT(un_i, true)
      if (u_nslots == 0) break;
      if (s >= u_nslots) continue;
      // what this slot holds
      const bool my_before = u_paired && s == 0;
      const int my_start = my_before ? u_start - kTile : u_start, my_len = my_before ? kTile : u_len;
      const int my_ntiles = my_before ? u_ntiles - 1 : u_ntiles;
      float m_used = -INFINITY, l_part = 0.f;
      // Rows of several segments: of the tile's own keys up to its own position, a row sees the
      // prompt's, [0, pr), and those of its own segment, from `lo` on.  A segment ends where the
      // visibility of its keys does.
      const int u_first = kMixed ? (u_len1 >> 8) & (kQTilePrompt - 1) : u_len;
      const bool one_segment = !kMixed || u_first == u_len;
      int pr = 0, lo = 0;
      if (!one_segment) {
        int end[4];
#pragma unroll
        for (int b = 0; b < 4; ++b)
          end[b] = prm.key_end[u_start + min(32 * b + lane, u_len - 1)];
        lo = pr = (u_len1 >> 8) & kQTilePrompt ? u_first : 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          uint32_t m = __ballot_sync(0xffffffffu, 32 * b + lane < u_len && end[b] == u_start + 32 * b + lane + 1);
          if (b == qd) m &= (1u << lane) - 1u;   // segments that end before this row
          if (b <= qd && m) lo = max(lo, 32 * (b + 1) - __clz(m));
        }
      }
      for (int j = 0; j < my_ntiles; ++j) {
        KvTile kt;
        kt.len = u_klen(j);
        kt.diag = j + 1 == my_ntiles;
        wait_bar(bar(kSFull + s), tcS & 1, abort_flag, prm.header, 40 + s);
        tc_fence_after();
        const bool full = !kt.diag && kt.len == kTile && (one_segment || j < u_n0);
        // visible columns of this half: [0, col_lim) in the half's own numbering
        const int col_lim = (kt.diag ? min(kt.len, row + 1) : kMixed && j >= u_n0 && row >= u_first ? 0 : kt.len) -
                            64 * half;
        uint32_t vis[2];   // mixed tiles: one bit each
        if (kMixed) {
          auto below = [&](int x) { return ~__funnelshift_lc(0u, ~0u, max(x, 0)); };   // bits below x
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int at = 64 * half + 32 * c;
            vis[c] = below(col_lim - 32 * c);
            if (kt.diag) vis[c] &= below(pr - at) | ~below(lo - at);
          }
        }
        auto visible = [&](int col) -> bool {
          return kMixed ? (vis[col >> 5] >> (col & 31)) & 1u : col < col_lim;
        };
        // The 64 scores of this thread are handled as two chunks of 32 (fewer live registers).
        // max over the visible scores of one chunk
        auto chunk_max = [&](const uint32_t (&w)[32], int c, float m) -> float {
          if (full) {
            float m1 = -INFINITY;
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              m = max3(m, __uint_as_float(w[i]), __uint_as_float(w[i + 1]));
              m1 = max3(m1, __uint_as_float(w[i + 2]), __uint_as_float(w[i + 3]));
            }
            return fmaxf(m, m1);
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) m = fmaxf(m, visible(32 * c + i) ? __uint_as_float(w[i]) : -INFINITY);
          return m;
        };
        // maximum over the row's visible scores, in base-2 units
        auto row_max = [&]() -> float {
          float mx = -INFINITY;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t w[32];
            tmem_ld32(tS + 32 * c, w);
            tmem_wait_ld();
            mx = chunk_max(w, c, mx);
          }
          xch_max[half] = mx;
          named_barrier_sync(bar_id, 64);
          return fmaxf(mx, xch_max[half ^ 1]) * prm.scale_log2;
        };
        // First tile of the unit: the reference maximum is needed before the exponentials -- with a
        // guessed one the largest P of a row would not be exactly 1, and rows that see one or two
        // keys would lose the exact cancellation in dP - Delta.  Later tiles use the reference of
        // the tiles before; only if a row has outgrown it by more than the rescale threshold (rare)
        // is the accumulator rescaled and the tile redone from the S values, which stay in tensor
        // memory until P is stored.
        if (j == 0) m_used = row_max();
        // The 64 scores go through in four pieces of 16, the tensor-memory load of the next piece
        // in flight under the exponentials of this one.  The first kEarlySteps pieces of P are
        // handed to the MMA thread before the exponentials of the last are formed: their share of
        // PV then runs under the rest of the softmax, which shortens the chain softmax -> PV -> QK
        // that is one slot's period and bounds this kernel (two rows of 32768 tokens, Hq / Hkv
        // 32 / 8, D 128: 7890 -> 7360 us; sixteen thousand tokens, 64 / 8: 535 -> 513; with two
        // pieces early 7550 and 519).  Whether the row has outgrown its reference has to be known
        // by then: the largest exponential tells for the early pieces (its max3 rides in the
        // MUFU-bound loop for free), the largest exponent for the last.
        uint32_t pk[32];
        uint64_t sum2;
        float x[16];   // exponents of the late piece
        bool redone = j == 0;
        for (;;) {
          const float neg_m = -m_used;
          const uint64_t sc2 = pack2(prm.scale_log2, prm.scale_log2), nm2 = pack2(neg_m, neg_m);
          sum2 = pack2(0.f, 0.f);
          float pm0 = 0.f, pm1 = 0.f, xm = -INFINITY;
          uint32_t wa[16], wb[16];
          auto exp16 = [&](const uint32_t (&w)[16], int piece, auto masked_c) {
            constexpr bool kMasked = decltype(masked_c)::value;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float x0, x1;
              unpack2(fma2(pack2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1])), sc2, nm2), x0, x1);
              float p0 = ex2(x0), p1 = ex2(x1);
              if (kMasked) {
                p0 = visible(16 * piece + 2 * i) ? p0 : 0.f;
                p1 = visible(16 * piece + 2 * i + 1) ? p1 : 0.f;
              }
              sum2 = add2(sum2, pack2(p0, p1));
              if (i & 1) pm1 = max3(pm1, p0, p1); else pm0 = max3(pm0, p0, p1);
              pk[8 * piece + i] = pack_bf16(p0, p1);
            }
          };
          auto arg16 = [&](const uint32_t (&w)[16], int piece, auto masked_c) {
            constexpr bool kMasked = decltype(masked_c)::value;
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
              unpack2(fma2(pack2(__uint_as_float(w[i]), __uint_as_float(w[i + 1])), sc2, nm2), x[i], x[i + 1]);
              if (kMasked) {
                x[i] = visible(16 * piece + i) ? x[i] : -INFINITY;
                x[i + 1] = visible(16 * piece + i + 1) ? x[i + 1] : -INFINITY;
              }
              xm = max3(xm, x[i], x[i + 1]);
            }
          };
          auto pieces = [&](auto masked_c) {
            tmem_ld16(tS, wa);
            tmem_wait_ld();
            tmem_ld16(tS + 16, wb);
            exp16(wa, 0, masked_c);
            tmem_wait_ld();
            tmem_ld16(tS + 32, wa);
            exp16(wb, 1, masked_c);
            tmem_wait_ld();
            tmem_ld16(tS + 48, wb);
            exp16(wa, 2, masked_c);
            tmem_wait_ld();
            arg16(wb, 3, masked_c);
          };
          if (full) pieces(std::false_type{}); else pieces(std::true_type{});
          if (redone) break;
          const float pmax = fmaxf(fmaxf(pm0, pm1), ex2(xm));
          xch_exp[half] = pmax;
          named_barrier_sync(bar_id, 64);
          const float hi = fmaxf(pmax, xch_exp[half ^ 1]);
          // Rows past the tile's end hold whatever follows in memory: they must not steer the
          // warp-wide decision, or a row's rounding would depend on its neighbours' data.
          const bool need = row < my_len && !(hi <= exp2f(kRescaleThreshold));
          if (!__any_sync(0xffffffffu, need)) break;   // same rows, same values in the partner warp
          const float m_new = fmaxf(m_used, row_max());
          const float alpha = ex2(m_used - m_new);
          // PV of the previous tile is complete: the commit that announced this tile's S was
          // issued after it and covers every earlier MMA of the issuing thread (but with columns of P's own
          // that QK came first)
          if (kOwnP) {
            wait_bar(bar(kPFree + s), (tcS & 1) ^ 1, abort_flag, prm.header, 48);
            tc_fence_after();
          }
#pragma unroll 1
          for (int c = 0; c < D / 16; ++c) {  // eight columns at a time
            uint32_t w[8];
            tmem_ld8(tO + c * 8, w);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) w[i] = __float_as_uint(__uint_as_float(w[i]) * alpha);
            tmem_st8(tO + c * 8, w);
          }
          l_part *= alpha;
          m_used = m_new;
          redone = true;
        }
        if (kOwnP) {
          tc_fence_before();
          mbar_arrive(bar(kSFree + s));
          wait_bar(bar(kPFree + s), (tcS & 1) ^ 1, abort_flag, prm.header, 48);   // (long complete)
          tc_fence_after();
        }
        // P over the first half of my own S columns, or to its own
        tmem_st16(tP, pk);
        tmem_st8(tP + 16, pk + 16);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar(kPFull + s));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float p0 = ex2(x[2 * i]), p1 = ex2(x[2 * i + 1]);
          sum2 = add2(sum2, pack2(p0, p1));
          pk[24 + i] = pack_bf16(p0, p1);
        }
        float s0, s1;
        unpack2(sum2, s0, s1);
        l_part += s0 + s1;
        tmem_st8(tP + 24, pk + 24);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar(kPRest + s));
        ++tcS;
      }
      // ---- epilogue: row sum from both halves, O / l -> bf16, release the accumulator, store
      xch_sum[half] = l_part;
      named_barrier_sync(bar_id, 64);
      const float l_run = l_part + xch_sum[half ^ 1];
      wait_bar(bar(kODone + s), ucS & 1, abort_flag, prm.header, 44 + s);
      ++ucS;
      tc_fence_after();
      const float inv_l = 1.f / l_run;
      uint32_t ob[D / 4];
#pragma unroll
      for (int c = 0; c < D / 64; ++c) {
        uint32_t w[32];
        // (columns at and past DV hold nothing and are not stored: the zeros only fill ob)
        if (DV == D || half * (D / 2) + c * 32 < DV) {
          tmem_ld32(tO + c * 32, w);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) w[i] = 0u;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
          ob[c * 16 + i] = pack_bf16(__uint_as_float(w[2 * i]) * inv_l, __uint_as_float(w[2 * i + 1]) * inv_l);
      }
      tc_fence_before();
      mbar_arrive(bar(kOFree + s));
      const int h = u_paired ? u_h0 : u_h0 + s;
      if (half == 0 && row < my_len)
        prm.lse[size_t(h) * prm.T + my_start + row] = (m_used + log2f(l_run)) * 0.69314718055994531f;
      // A thread holds kCh 16-byte chunks of one row; transposing them inside groups of kCh
      // lanes gives every lane the same chunk of kCh consecutive rows, so that one store
      // instruction of the warp writes whole contiguous half-rows instead of 32 scattered
      // 16-byte pieces.
      constexpr int kCh = D / 16;
      auto exchange = [&](auto dist) {
        constexpr int d = decltype(dist)::value;
        if constexpr (d < kCh) {
          const bool hi = (lane & d) != 0;
#pragma unroll
          for (int i = 0; i < kCh; ++i) {
            if ((i & d) == 0) {
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const uint32_t send = hi ? ob[4 * i + c] : ob[4 * (i | d) + c];
                const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, d);
                if (hi) ob[4 * i + c] = recv; else ob[4 * (i | d) + c] = recv;
              }
            }
          }
        }
      };
      exchange(std::integral_constant<int, 4>{});
      exchange(std::integral_constant<int, 2>{});
      exchange(std::integral_constant<int, 1>{});
      {
        const int grp = lane / kCh, chunk = lane % kCh;
#pragma unroll
        for (int i = 0; i < kCh; ++i) {
          const int r = 32 * qd + grp * kCh + i;
          if (r < my_len && (DV == D || half * (D / 2) + chunk * 8 < DV)) {
            uint4* dst = reinterpret_cast<uint4*>(
                prm.o + ((size_t(my_start) + r) * prm.Hq + h) * DV + half * (D / 2) + chunk * 8);
            *dst = make_uint4(ob[4 * i], ob[4 * i + 1], ob[4 * i + 2], ob[4 * i + 3]);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // After a wait that gave up, copies and MMAs issued without their barriers may still be in
  // flight: give them time to land before the CTA's shared and tensor memory are released.
  if (*abort_flag)
    for (int i = 0; i < 50; ++i) __nanosleep(1000);
  if (warp == 0) tmem_dealloc(tmem, kFwdTmemCols);
  if (tid == 0) {  // the last CTA to finish re-arms the unit counter for the next launch
    __threadfence();
    if (atomicAdd(&prm.header[kHdrFwdDone], 1) == int(gridDim.x) - 1) {
      prm.header[kHdrFwdNext] = 0;
      prm.header[kHdrFwdDone] = 0;
    }
  }
#ifdef PP_DEBUG_COUNTERS
  if (blockIdx.x == 0 && tid == 0) g_wait_cycles[127] = (unsigned long long)(clock64() - t_kernel0);
  if (tid == 0) g_cta_cycles[blockIdx.x & 255] = (unsigned long long)(clock64() - t_kernel0);
#endif
}

#ifdef PP_DEBUG_COUNTERS
}  // namespace
}  // namespace pp
extern "C" int pp_debug_fwd_cta_cycles(unsigned long long* out) {
  return cudaMemcpyFromSymbol(out, pp::g_cta_cycles, sizeof(unsigned long long) * 256) == cudaSuccess ? 0 : -5;
}
extern "C" int pp_debug_fwd_wait_cycles(unsigned long long* out, int reset) {
  if (out && cudaMemcpyFromSymbol(out, pp::g_wait_cycles, sizeof(unsigned long long) * 128) != cudaSuccess)
    return -5;
  if (reset) {
    static unsigned long long zeros[128] = {};
    if (cudaMemcpyToSymbol(pp::g_wait_cycles, zeros, sizeof zeros) != cudaSuccess) return -5;
  }
  return 0;
}
namespace pp {
namespace {
#endif

template <int D, int DV = D>
cudaError_t launch_fwd_t(const pp_plan* plan, const CUtensorMap& tq, const CUtensorMap& tk,
                         const CUtensorMap& tv, const FwdParams& prm, cudaStream_t stream) {
  static DeviceSetup setup[kMaxDevices];
  DeviceSetup* dev = device_setup(setup);
  if (!dev) return cudaErrorInvalidDevice;
  if (dev->cc_major != 10) return cudaErrorNotSupported;
  using Kernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, FwdParams);
  const Kernel kerns[3] = {fwd_kernel<D, kPlain, DV>, fwd_kernel<D, kMixedTiles, DV>, fwd_kernel<D, kPairedTiles, DV>};
  if (!dev->configured) {
    for (Kernel k : kerns) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem<D>::kTotal);
      if (e != cudaSuccess) return e;
    }
    dev->configured = true;
  }
  const int num_sms = dev->num_sms;
  const pp_problem& pb = plan->prob;
  const int r = pb.num_q_heads / pb.num_kv_heads;
  const long long units = (long long)plan->max_tiles * pb.num_kv_heads * ((r + 1) / 2);
  const Kernel kern = kerns[plan->mixed ? kMixedTiles : plan->paired ? kPairedTiles : kPlain];
  dim3 grid(unsigned(std::min<long long>(units, num_sms)));
  ProfileEvents& ev = profile_events();
  const int slot = int(ev.fwd_count % kProfileRing);
  if (ev.on && ev.fwd_on) profile_record(ev.fwd0[slot], stream);
  const cudaError_t le = launch_kernel(units <= (long long)kOverlapUnits * num_sms, kern, grid,
                                       dim3(kFwdThreads), FwdSmem<D>::kTotal, stream, tq, tk, tv, prm);
  if (ev.on && ev.fwd_on) {
    profile_record(ev.fwd1[slot], stream);
    ++ev.fwd_count;
  }
  return le;
}

}  // namespace

cudaError_t launch_fwd(const pp_plan* plan, const void* q, const void* k, const void* v, float scale,
                       void* o, float* lse, float* dq_clear, cudaStream_t stream, int* launches) {
  const pp_problem& pb = plan->prob;
  CUtensorMap tq, tk, tv;
  if (!encode_thd(&tq, q, pb.total_tokens, pb.num_q_heads, pb.head_dim, kTile) ||
      !encode_thd(&tk, k, pb.total_tokens, pb.num_kv_heads, pb.head_dim, kTile) ||
      !encode_thd(&tv, v, pb.total_tokens, pb.num_kv_heads, pb.head_dim, kTile))
    return cudaErrorNotSupported;
  FwdParams prm;
  prm.header = reinterpret_cast<int32_t*>(plan->ws + plan->lay.header);
  prm.tiles = reinterpret_cast<const Tile*>(plan->ws + plan->lay.tiles);
  prm.tile_unit = reinterpret_cast<const uint8_t*>(plan->ws + plan->lay.tile_unit);
  prm.qtiles = reinterpret_cast<const QTile*>(plan->ws + plan->lay.qtiles);
  prm.key_end = reinterpret_cast<const int32_t*>(plan->ws + plan->lay.key_end);
  prm.order = reinterpret_cast<const int32_t*>(plan->ws + (plan->mixed ? plan->lay.qorder : plan->lay.fwd_order));
  prm.o = static_cast<__nv_bfloat16*>(o);
  prm.lse = lse;
  prm.dq_clear = dq_clear;
  prm.T = pb.total_tokens;
  prm.Hq = pb.num_q_heads;
  prm.Hkv = pb.num_kv_heads;
  prm.scale_log2 = scale * 1.4426950408889634f;
  cudaError_t e = pb.head_dim == 128  ? launch_fwd_t<128>(plan, tq, tk, tv, prm, stream)
                  : pb.head_dim == 96 ? launch_fwd_t<128, 96>(plan, tq, tk, tv, prm, stream)
                                      : launch_fwd_t<64>(plan, tq, tk, tv, prm, stream);
  if (e == cudaSuccess && launches) *launches += 1;
  return e;
}

}  // namespace pp
