// Internal definitions shared by the plan builder, the kernels and the C ABI.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/pp_attn.h"

namespace pp {

constexpr int kTile = 128;  // query-tile and key-tile length in tokens

// One tile of a segment (prompt or response).  Read as a query tile it lists the keys it
// sees; read as a key tile it lists the queries that see it.
struct Tile {
  int32_t start;      // first token
  int32_t len;        // 1..128 tokens
  int32_t kv0_start;  // FULL range 0: prompt keys visible to every row of the tile
  int32_t kv0_len;    //   (for a prompt tile: the prompt keys before the tile)
  int32_t kv1_start;  // FULL range 1: own-response keys before the tile (0 for prompt tiles)
  int32_t kv1_len;
  int32_t vis_end;    // queries [start, vis_end) see this tile's keys (causally inside the tile)
  int32_t work;       // forward work estimate in key tiles (backward: derived)
};
static_assert(sizeof(Tile) == 32, "tile record is 32 bytes");
// What the forward does with a query tile of a segment where it takes them by twos: nothing (the tile
// behind it has it), this tile alone (a segment's last, and the longest: pair_pays), or the tile before it
// and this one.
enum kTileUnit : uint8_t { kTileNone = 0, kTileAlone = 1, kTileWithLast = 2 };
__host__ __device__ constexpr uint8_t tile_unit_of(int rel, int count) {   // tile `rel` of a segment's `count`
  return rel & 1 ? kTileWithLast : rel + 1 == count ? kTileAlone : kTileNone;
}

// One key tile of the backward pass.  The backward cuts each GROUP (prompt and responses as one
// token range) into tiles of 128 tokens from the group's start, so a tile may straddle segment
// boundaries: short segments then leave no ragged tile each, only the group's last tile is
// short.  Key j of the tile is seen by the queries [j, key_end[j]); the query tiles of the unit
// are the tiles of the same grid from this one on, up to vis_end.
struct BTile {
  int32_t start;      // first token
  int32_t len;        // 1..128 tokens
  int32_t vis_end;    // largest key_end of the tile's keys: queries [start, vis_end) see some key
  int32_t dep_lo;     // read as a query tile: besides the prompt tiles [0, npc), the key tiles
                      //   [dep_lo, own index] of the group's grid add to its dQ
  int32_t grp_start;  // first token of the group (also the group's identity)
  int32_t grp_end;    // one past the last token of the group
  int32_t work;       // number of query tiles: 1 + ceil((vis_end - start - len) / 128)
  int32_t npc;        // tiles of the group that hold prompt keys: ceil(prompt length / 128)
};
static_assert(sizeof(BTile) == 32, "backward tile record is 32 bytes");

// One query tile of the forward where it does not run over the tiles of the segments
// (fwd_mixed_tiles below): a tile of the group's grid, whose rows may belong to several segments,
// or a copy of a segment's tile.
struct QTile {
  int32_t start, len;
  int32_t kv0_start, kv0_len;  // prompt keys before the tile: every row sees them
  int32_t kv1_start, kv1_len;  // the first rows' own response before the tile: only they see it
  int32_t first_rows;          // rows of the first segment, and kQTilePrompt if it is the prompt
  int32_t work;                // key tiles of both ranges, and the tile itself
};
constexpr int kQTilePrompt = 256;

// Words of the plan header (int32[16]).
constexpr int kHdrStatus = 0, kHdrDetail = 1, kHdrNumTiles = 2, kHdrNumSegments = 3,
              kHdrNumBTiles = 8, kHdrNumQTiles = 9,
              kHdrSchedTail = 10,   // (multi-kernel plan) tiles of the last of the smaller blocks
              kHdrFwdWork = 12;     // ... and the forward tiles' works, 64 bits

// Status word values written by device code.
enum : int32_t {
  kStatusOk = 0,
  kStatusBadDescriptor = 1,  // detail = index of the offending group / response
  kStatusTokenMismatch = 2,  // detail = token count found
  kStatusWaitExpired = 3,    // detail = site id
};

// Device part of a plan: offsets (bytes) into the caller's workspace.
struct PlanLayout {
  size_t header;     // int32[16]: status, detail, num_tiles, num_segments, counters, num_btiles
  size_t desc;       // device copy of the descriptor arrays (when given on host)
  size_t seg_start;  // int32[nseg + 1]
  size_t seg_tile0;  // int32[nseg + 1]  first tile of each segment
  size_t tiles;      // Tile[max_tiles]
  size_t tile_unit;  // uint8[max_tiles]  kTileUnit below
  size_t fwd_order;  // int32[max_tiles]
  size_t grp_btile0; // int32[G + 1]  first backward tile of each group
  size_t btiles;     // BTile[max_tiles]  (at most max_btiles_of of them)
  size_t bwd_order;  // int32[max_tiles]  backward tiles, longest work first
  size_t tile_gwork; // int32[max_tiles]  backward work of the backward tile's whole group
  size_t tile_block; // int32[max_tiles] super-group (block of consecutive groups) or, for the smaller blocks,
                     //   tiles of the groups behind the tile's
  size_t bwd_units;  // int32[max_tiles * Hkv]  (kv head << 24) | backward tile, processing order
                     //   (in super-groups or, with bwd_takes_sched, in smaller blocks)
  size_t bwd_units_det;  // the same units, one (group, KV head) set after the other and inside a
                         //   set by descending tile index: the order of the deterministic backward
  size_t key_end;    // int32[T]
  // only where the forward runs over mixed tiles
  size_t qtiles;     // QTile[max_tiles]  a group's tiles from its first segment tile's index on
  size_t qorder;     // int32[max_tiles]  the query tiles, longest work first
  size_t grid_gain;  // int64[G]  forward work over the segments' tiles less that over the grid's
  size_t total;
};

}  // namespace pp

struct pp_plan {
  pp_problem prob;  // descriptor pointers are rewritten to the copies in the workspace
  // Descriptors given on the device: the caller's arrays, which the first plan kernel copies
  // into the workspace (null when the host path has staged them already).
  const int32_t* src_desc[4] = {nullptr, nullptr, nullptr, nullptr};
  int nseg;
  int max_tiles;
  char* ws;
  pp::PlanLayout lay;
  // scratch sizes
  size_t fwd_scratch, bwd_scratch;
  bool mixed;     // the forward runs over mixed query tiles (fwd_mixed_tiles)
  bool paired;    // ... takes tiles of a segment by twos (fwd_paired_tiles)
  int lg_split;   // log2 of the parts each backward unit is cut into (bwd_split_log2)
  // backward scratch whose dQ accumulator the latest forward on this plan has cleared
  mutable const void* cleared_scratch = nullptr;
};

namespace pp {

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

inline int max_tiles_of(const pp_problem& p) {
  // sum over segments of ceil(len / 128) <= T / 128 + number of segments
  return p.total_tokens / kTile + p.num_groups + p.num_responses;
}
// The backward's tiles, cut per group: ceil(length / 128) each.
inline int max_btiles_of(const pp_problem& p) { return p.total_tokens / kTile + p.num_groups; }

// The forward's query tiles: those of the segments, or tiles of each group's 128-token grid, whose
// rows may belong to several segments (a group keeps its segments' tiles where they are less
// work).  Short segments leave their own tiles nearly empty: 41 groups of 106 tokens in 5 segments
// have 165 tiles and 297 key tiles to visit, on the grid 52 and 89.  The plan then takes one more
// order and the forward the more general masks, 2 - 4 us a step, which pays where segments add
// more than 0.3 to the number of tiles and there are more units than run in two waves anyway.
// Whole steps, segments -> grid, at (added tiles, units per SM): (2.6, 5) 139 -> 97 us, (1.4, 8)
// 148 -> 118, (0.42, 54) 1805 -> 1524, (0.45, 13) 326 -> 289, (0.72, 1.8) 66 -> 63; but (0.27, 9)
// 170 -> 173, (0.36, 1.6) 105 -> 112, (1.25, 0.4) 49 -> 52.  By sizes alone, 148 SMs whatever part of a
// device there is, so that every way of running a problem sums in the same order.
inline bool fwd_mixed_tiles(const pp_problem& p) {
  const int pairs = (p.num_q_heads / p.num_kv_heads + 1) / 2;
  const double grid = p.total_tokens / double(kTile) + 0.5 * p.num_groups, added = 0.5 * p.num_responses;
  return added > 0.3 * grid && (grid + added) * p.num_kv_heads * pairs > 1.75 * 148;
}

// Whether the forward takes two tiles of a segment into a unit's slots for the last head of an odd number
// of heads per KV head (each row's arithmetic is the same either way).  A unit with both slots filled
// takes 1.4 times one with slot 1 empty, so it pays once there is more work per SM than the
// longest such unit, in key tiles estimated from the mean group (the plan, which knows the groups, leaves
// those alone that are longer: pair_pays there): 12000 tokens in 3000-token groups, 16 / 16 heads, D 128
// 291 -> 204 us, 2600-token groups, D 96 225 -> 165; but 8000-token groups, 2 / 2 heads 166 -> 182.  With three and
// more heads per KV head the other units take that long anyway: 20187 tokens, 28 / 4 631 -> 594.
inline bool fwd_paired_tiles(const pp_problem& p, int sms) {
  const int r = p.num_q_heads / p.num_kv_heads;
  const double tiles = p.total_tokens / double(kTile) + 0.5 * (p.num_groups + p.num_responses);
  const double m = double((p.total_tokens / p.num_groups + kTile - 1) / kTile);
  if (!(r & 1) || tiles * p.num_kv_heads * ((r + 1) / 2) <= sms) return false;
  return r > 1 || tiles * p.num_kv_heads * (m + 1) / 2 > 1.4 * sms * m * (p.num_groups > 1 ? 1.5 : 1.0);
}

inline PlanLayout plan_layout(const pp_problem& p) {
  PlanLayout l{};
  int nseg = p.num_groups + p.num_responses;
  int mt = max_tiles_of(p);
  size_t off = 0;
  l.header = off;    off = align_up(off + 64, 256);
  l.desc = off;
  off = align_up(off + sizeof(int32_t) * (size_t(p.num_rows) + 1 + p.num_groups +
                                           (p.num_groups + 1) + p.num_responses), 256);
  l.seg_start = off; off = align_up(off + sizeof(int32_t) * (nseg + 1), 256);
  l.seg_tile0 = off; off = align_up(off + sizeof(int32_t) * (nseg + 1), 256);
  l.tiles = off;     off = align_up(off + sizeof(Tile) * size_t(mt), 256);
  l.tile_unit = off; off = align_up(off + size_t(mt), 256);
  l.fwd_order = off; off = align_up(off + sizeof(int32_t) * size_t(mt), 256);
  l.grp_btile0 = off; off = align_up(off + sizeof(int32_t) * (size_t(p.num_groups) + 1), 256);
  l.btiles = off;    off = align_up(off + sizeof(BTile) * size_t(mt), 256);
  l.bwd_order = off; off = align_up(off + sizeof(int32_t) * size_t(mt), 256);
  l.tile_gwork = off; off = align_up(off + sizeof(int32_t) * size_t(mt), 256);
  l.tile_block = off; off = align_up(off + sizeof(int32_t) * size_t(mt), 256);
  l.bwd_units = off; off = align_up(off + sizeof(int32_t) * size_t(mt) * size_t(p.num_kv_heads), 256);
  l.bwd_units_det = off;
  off = align_up(off + sizeof(int32_t) * size_t(mt) * size_t(p.num_kv_heads), 256);
  l.key_end = off;   off = align_up(off + sizeof(int32_t) * size_t(p.total_tokens), 256);
  l.qtiles = off;    off = align_up(off + sizeof(QTile) * size_t(mt), 256);
  l.qorder = off;    off = align_up(off + sizeof(int32_t) * size_t(mt), 256);
  l.grid_gain = off; off = align_up(off + sizeof(int64_t) * size_t(p.num_groups), 256);
  l.total = off;
  return l;
}

// Backward scratch: fp32 dQ accumulator [T][Hq][D], Delta [Hq][T], LSE*log2(e) [Hq][T]; where units
// are cut into parts (below), the parts' fp32 dV and dK tiles; and, last because only the
// deterministic variant has them, the turn counters, four per (query tile of the backward grid,
// query head): one for each warp's 32 rows
struct BwdScratch {
  size_t dq_acc, delta, lse2, parts, sem, sem_bytes, total;
};

// A backward unit (a key tile and KV head against every (query tile, query head) that sees them)
// is a serial chain, so in small batches a few CTAs run long ones while the others idle: eight heads
// on one KV head and a 276-token group make three units of up to 24 iterations.  There each unit is
// cut into 2^n parts by query heads, which CTAs process independently; each part leaves its dV and
// dK in fp32 in the scratch and the finalize kernel adds them up in order.  n minimises the
// estimated time in iterations, the longer of the longest part and everything's share per SM, with
// two iterations of overhead for a unit and three for a part; it depends on sizes alone (148 SMs
// whatever part of a device there is), so that every way of running a problem sums in the same order.
// It knows the mean group, not the longest: one long group among many short ones may get fewer parts
// than would suit it.  Whole steps, units whole -> cut (us):
// 276 tokens, 8 heads on 1 KV head 99 -> 56; 573, 32 on 4 102 -> 53; 8999, 7 on 1 183 -> 114; 3999,
// 4 on 1 in one group 251 -> 113; 2753, 2 on 1 50 -> 44.  From about 148 units' worth of balanced
// work on, parts only add their overhead and fp32 traffic, and the rule leaves units whole.
constexpr int kPartShift = 21;   // tile, part and KV head of a part in one word: 21, 3 and 7 bits
inline int bwd_split_log2(const pp_problem& p) {
  const int heads = p.num_q_heads / p.num_kv_heads;
  const double r = heads, groups = p.num_groups;
  const double m = double((p.total_tokens / p.num_groups + kTile - 1) / kTile);   // tiles of a mean group
  const double units = (p.total_tokens / double(kTile) + groups / 2) * p.num_kv_heads;
  const double longest = r * m * (p.num_groups > 1 ? 1.5 : 1.0);
  const double total = units * r * (m + 1) / 2;
  int best = 0;
  double best_time = 0;
  for (int n = 0; n <= 3 && (1 << n) <= heads && max_btiles_of(p) < (1 << kPartShift); ++n) {
    const double parts = units * (1 << n), share = (total + (n ? 3 : 2) * parts) / 148;
    const double time = share > longest / (1 << n) + 2 ? share : longest / (1 << n) + 2;
    if (n == 0 || time < 0.95 * best_time) {
      best = n;
      best_time = time;
    }
  }
  return best;
}

// Which order the backward takes its units in.  Both go through the groups by decreasing work, in
// blocks of groups inside which the longest units come first.  With blocks of 600 units
// (super-groups) the 148 units that run at a time may be the longest of all of a block's groups, and with r
// query heads per KV head a block's Q, dO and dQ accumulator are 600 r * 128 KB at D 128: far beyond
// L2, so that a (query tile, head) is fetched, and its accumulator written back, for nearly every
// other key tile.  Blocks of 150 units with a larger last one to balance the end (sched_tail in the plan)
// move less where the groups are small against L2.  DRAM traffic of the main kernel, 600s -> these: 9241
// tokens, 32 / 8 heads 0.93 -> 0.52 GB, 16384, 64 / 8 5.36 -> 3.31; 20187 in four long groups, 28 / 4, where the
// last block grows to what it was, 5.90 -> 5.95; two rows of 32768 in groups as large as a block, 32 / 8,
// between -15 and +3 %.  Times of it: 9241 tokens 262 -> 250 us; 16384, 64 / 8 1361 -> 1230; 16384, 32 / 8, D 64
// 456 -> 400; 36000 in short groups, 16 / 2 277 -> 243; 16760, 32 / 8 307 -> 272; two rows of 32768, 32 / 8
// 19320 -> 19220.  With one and two heads per KV head a block's data is that much smaller, and the smaller blocks
// only cost balance: 8 / 8 258 -> 265, 16 / 8 278 -> 276, 754 -> 740.  Up to 200 units both are one block.
constexpr int kSuperGroupUnits = 600, kSchedBlockUnits = 150, kSchedTailUnits = 200;
inline bool bwd_takes_sched(const pp_problem& p) {
  return p.num_q_heads / p.num_kv_heads >= 3 && (long long)max_btiles_of(p) * p.num_kv_heads > kSchedTailUnits;
}

inline BwdScratch bwd_scratch_layout(const pp_problem& p, int lg_split) {
  BwdScratch s{};
  size_t T = p.total_tokens, Hq = p.num_q_heads, D = p.head_dim;
  size_t off = 0;
  s.dq_acc = off; off = align_up(off + 4 * T * Hq * D, 256);
  s.delta = off;  off = align_up(off + 4 * T * Hq, 256);
  s.lse2 = off;   off = align_up(off + 4 * T * Hq, 256);
  s.parts = off;
  if (lg_split) {
    const size_t parts = size_t(max_btiles_of(p)) * p.num_kv_heads << lg_split;
    off = align_up(off + parts * 2 * kTile * D * 4, 256);
  }
  s.sem = off;
  s.sem_bytes = 16 * size_t(max_btiles_of(p)) * Hq;
  off = align_up(off + s.sem_bytes, 256);
  s.total = off;
  return s;
}
inline BwdScratch bwd_scratch_layout(const pp_problem& p) { return bwd_scratch_layout(p, bwd_split_log2(p)); }

// Device arena of pp_attn_step_host: inputs, outputs, plan workspace, backward scratch.  The
// step is cut into at most kStepChunks runs of whole groups, each with its own plan, scratch and
// LSE block inside the shared regions; the regions carry the alignment slack that costs.
constexpr int kStepChunks = 8;
struct StepArena {
  size_t q, k, v, d_o, o, lse, dq, dk, dv, plan, scratch, total;
};
inline StepArena step_arena_layout(const pp_problem& p) {
  StepArena a{};
  const size_t T = p.total_tokens, D = p.head_dim;
  const size_t qb = T * p.num_q_heads * D * 2, kb = T * p.num_kv_heads * D * 2;
  size_t off = 0;
  auto take = [&](size_t n) { size_t o = off; off = align_up(off + n, 256); return o; };
  a.q = take(qb); a.k = take(kb); a.v = take(kb); a.d_o = take(qb);
  a.o = take(qb); a.lse = take(T * p.num_q_heads * 4 + 256 * kStepChunks);
  a.dq = take(qb); a.dk = take(kb); a.dv = take(kb);
  a.plan = take(plan_layout(p).total + size_t(16384) * kStepChunks);
  a.scratch = take(bwd_scratch_layout(p).total + size_t(4096) * kStepChunks);
  a.total = off;
  return a;
}

// Per-device launch state of a kernel family: the opt-in to large dynamic shared memory is a
// per-device function attribute, and the SM count differs between devices, so a process that
// drives several GPUs must set up each of them.
constexpr int kMaxDevices = 64;
struct DeviceSetup {
  bool configured = false;
  int num_sms = 0;
  int cc_major = 0;
};
// Entry for the current device in `table` (kMaxDevices entries), or null.
inline DeviceSetup* device_setup(DeviceSetup* table) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  DeviceSetup* d = table + dev;
  if (!d->num_sms &&
      (cudaDeviceGetAttribute(&d->cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
       cudaDeviceGetAttribute(&d->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess))
    return nullptr;
  return d;
}
// The kernels are sm_100a code (tcgen05, tensor memory): any other device is refused before a
// launch is attempted.  Checked once per device.
inline int sm100_sms() {   // SMs of the current device; 0 if it is another kind
  static DeviceSetup probe[kMaxDevices];
  DeviceSetup* d = device_setup(probe);
  return d && d->cc_major == 10 ? d->num_sms : 0;
}

// Launches a kernel, with `overlap` so that it may start before the kernel in front of it on the
// stream has ended (programmatic dependent launch): it calls dependency_wait before it touches global
// memory, and its launch (in the backward also barrier set-up, tensor-map fetches and tensor-memory
// allocation) runs under the tail of the one before, or under all of it where that calls
// launch_dependents first thing (plan, preprocess, finalize).  (Kernels that know nothing of this, in
// front or behind, see ordinary stream order.)
// Such a kernel is resident while the one in front still writes what it will read: its pointers carry no
// __restrict__, which would promise that those values do not change meanwhile.
// The main kernels take it up to kOverlapUnits units per SM: steps of 60 - 100 us gain 5 -
// 9 % (144 ... 1054 tokens), one of 180 us 2.5 %, one of 500 us nothing, and a forward and
// backward of 2600 and 1100 units (T 16384, 32 / 8 heads, D 64) lost 2 %.  Preprocess and finalize always take it,
// 3 - 5 us a step: 144 tokens, 1 / 1 heads 30.0 -> 27.4 us in a row of steps, 40.0 -> 36.4 alone; 374, 28 / 4,
// D 64 39.4 -> 35.1; 1000, 8 / 2 59.8 -> 56.2; 3000, 16 / 8 104.9 -> 100.4; 28626 in short groups, 4 / 1
// 169.3 -> 165; 12000, 32 / 8 427 -> 422.  The main kernels in front of them do not call
// launch_dependents: early blocks of the stream crowd the SMs that free up first (with it and more than
// two blocks per SM 1000 tokens, 8 / 1 55 -> 61, preprocess 30 -> 38 us at T 9241, and even
// with fewer 144 tokens 30.1 instead of 27.4).
constexpr int kOverlapUnits = 4;
template <typename... P, typename... A>
cudaError_t launch_kernel(bool overlap, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Optional event pairs around the forward kernel and the backward main kernel.
// A ring of pairs per kernel, so that a benchmark can time many steps and read the durations
// afterwards instead of synchronising after every step.
constexpr int kProfileRing = 64;
struct ProfileEvents {
  bool on = false;
  bool fwd_on = false;  // forward events wanted too (mode 1); mode 2 times the backward only
  cudaEvent_t fwd0[kProfileRing] = {}, fwd1[kProfileRing] = {}, bwd0[kProfileRing] = {},
              bwd1[kProfileRing] = {};
  long long fwd_count = 0, bwd_count = 0;   // launches recorded since the events were enabled
};
ProfileEvents& profile_events();
// Records a profiling event.  On a capturing stream the record becomes a node of the graph
// that marks the event at every replay (an ordinary record would only order the capture).
inline void profile_record(cudaEvent_t ev, cudaStream_t stream) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &st) == cudaSuccess && st == cudaStreamCaptureStatusActive)
    cudaEventRecordWithFlags(ev, stream, cudaEventRecordExternal);
  else
    cudaEventRecord(ev, stream);
}
bool profile_enable(int mode);
bool profile_read(float* fwd_ms, float* bwd_ms);
bool profile_read_all(float* fwd_ms, float* bwd_ms, int capacity, int* n_fwd, int* n_bwd);

// launchers (defined in the .cu files); all return a cudaError_t
// host_desc: the four descriptor arrays on the host, or null when they are on the device
cudaError_t launch_plan(const pp_plan* plan, const int32_t* const* host_desc, cudaStream_t stream,
                        int* launches);
cudaError_t launch_fwd(const pp_plan* plan, const void* q, const void* k, const void* v, float scale,
                       void* o, float* lse, float* dq_clear, cudaStream_t stream, int* launches);
cudaError_t launch_bwd(const pp_plan* plan, const void* q, const void* k, const void* v,
                       const void* o, const float* lse, const void* d_o, float scale, void* dq,
                       void* dk, void* dv, void* scratch, int lg_split, bool dq_cleared,
                       bool deterministic, cudaStream_t stream, int* launches);

// Row builder (csrc/pp_rows.cu).
size_t rows_workspace_bytes(int num_groups);
cudaError_t launch_build_rows(int G, int N, const int32_t* prompt_len, const int32_t* resp_off,
                              const int32_t* resp_len, int capacity, void* ws, int32_t* order,
                              int32_t* row_group_off, int32_t* num_rows, long long* row_tokens,
                              long long* row_cost, int32_t* out_prompt_len, int32_t* out_resp_off,
                              int32_t* out_resp_len, int32_t* status, cudaStream_t stream,
                              int* launches);

cudaError_t launch_assign_rows(int R, const long long* row_cost, int ranks, int32_t* order,
                               int32_t* rank_of_row, long long* rank_cost, cudaStream_t stream,
                               int* launches);

// Size of the scratch array built into the library image for pp_attn_bwd_noalloc.
constexpr size_t kStaticScratchBytes = size_t(32) << 20;
cudaError_t launch_bwd_static(const pp_plan* plan, const void* q, const void* k, const void* v,
                              const void* o, const float* lse, const void* d_o, float scale,
                              void* dq, void* dk, void* dv, cudaStream_t stream, int* launches);

cudaError_t launch_position_ids(const pp_plan* plan, int32_t* pos, cudaStream_t stream);
cudaError_t launch_rope(const pp_plan* plan, void* q, void* k, float base, cudaStream_t stream);

cudaError_t launch_preference_loss(const pp_plan* plan, const float* logp, const float* ref,
                                   float beta, float* resp_logp, float* resp_reward,
                                   float* grp_loss, float* d_logp, cudaStream_t stream);

}  // namespace pp
