// Device-side plan builder: segment descriptors -> tiles, visible key/query ranges, orders.
//
// The packing mask (paper Sec. 3.2) has a simple structure once tokens are grouped by
// segment: a key j is seen by the contiguous queries [j, end_j) where end_j is the end of
// j's group for a prompt key and the end of j's own response otherwise; a query sees at
// most two contiguous key ranges (its group's prompt, and its own segment up to itself).
// Forward tiles are cut per segment (aligned to the segment start), so a tile never straddles
// two segments and only its own diagonal block needs element-wise causal masking.  The
// backward has its own key tiles, cut per group (see BTile): its masks are two comparisons per
// element with per-key bounds, so straddling costs nothing there and short segments leave no
// ragged tiles.
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "pp_internal.h"
#include "pp_ptx.cuh"

namespace pp {
namespace {

struct PlanPtrs {
  int32_t* header;
  // descriptors given on the device: the caller's arrays (null otherwise) and the workspace
  // block they are copied into, which is what row_group_off .. resp_len below point at
  const int32_t* src_desc[4];
  int32_t* desc_copy;
  const int32_t* row_group_off;
  const int32_t* grp_prompt_len;
  const int32_t* grp_resp_off;
  const int32_t* resp_len;
  int32_t* seg_start;
  int32_t* seg_tile0;
  Tile* tiles;
  uint8_t* tile_unit;   // null: not wanted
  int sms;
  int pair_cost, unit_cost;  // tenths per key tile of a unit with two tiles and of all units of a query
                             //   tile and KV head (see pair_pays)
  int32_t* grp_btile0;
  BTile* btiles;
  int32_t* fwd_order;
  int32_t* bwd_order;
  int32_t* tile_gwork;
  int32_t* tile_block;
  int32_t* bwd_units;
  bool sched;           // in the smaller blocks (bwd_takes_sched)
  int32_t* bwd_units_det;
  int Hkv;
  int32_t* key_end;
  QTile* qtiles;        // null: not wanted
  int32_t* qorder;
  long long* grid_gain;
  int32_t* work_at;     // per work: how many query tiles have it, then where the next of them goes
                        // (multi-kernel plan; the space of bwd_units_det, which is written last)
  int det_asc_max;  // deterministic order: sets of at most this many tiles are handed out longest first
  int num_rows, G, N, T, nseg, max_tiles;
};

// Works that are told apart in the order of the query tiles: all that there can be.
__device__ __forceinline__ int work_slots(const PlanPtrs& p) { return min(p.max_tiles, p.T / kTile + 4); }

__device__ __forceinline__ void set_status(int32_t* header, int32_t status, int32_t detail) {
  if (atomicCAS(&header[0], kStatusOk, status) == kStatusOk) header[1] = detail;
}

// Segment order: group 0 prompt, group 0 responses, group 1 prompt, ...  so the prompt of
// group g is segment g + resp_off[g] and response x (global index) of group g is g + 1 + x.

// One block of 1024 threads.  Validates, writes segment lengths, scans them into seg_start /
// seg_tile0.  Returns (uniformly) whether the descriptors were accepted.
__device__ __forceinline__ bool plan_scan_body(const PlanPtrs& p) {
  __shared__ int32_t s_tok[1024];
  __shared__ int32_t s_til[1024];
  __shared__ int32_t s_carry[2];
  const int tid = threadIdx.x;

  // Descriptors handed over on the device are copied into the workspace first: everything
  // after this call -- the later plan kernels, position ids, rotary embedding, the loss -- reads
  // the copy, so the caller's arrays are free again once this kernel has run.
  if (p.src_desc[0]) {
    const int n[4] = {p.num_rows + 1, p.G, p.G + 1, p.N};
    int32_t* dst = p.desc_copy;
    for (int a = 0; a < 4; ++a) {
      for (int i = tid; i < n[a]; i += blockDim.x) dst[i] = p.src_desc[a][i];
      dst += n[a];
    }
    __syncthreads();
  }
  if (tid == 0) {
    p.header[0] = kStatusOk;
    p.header[1] = 0;
    p.header[2] = 0;
    p.header[3] = p.nseg;
    for (int i = 4; i < 16; ++i) p.header[i] = 0;  // [4,8): dynamic-scheduling counters
    if (p.row_group_off[0] != 0 || p.row_group_off[p.num_rows] != p.G)
      set_status(p.header, kStatusBadDescriptor, -1);
    if (p.grp_resp_off[0] != 0 || p.grp_resp_off[p.G] != p.N)
      set_status(p.header, kStatusBadDescriptor, -2);
    s_carry[0] = 0;
    s_carry[1] = 0;
  }
  __syncthreads();
  for (int r = tid; r < p.num_rows; r += blockDim.x)
    if (p.row_group_off[r + 1] < p.row_group_off[r]) set_status(p.header, kStatusBadDescriptor, r);
  // segment lengths (stored in seg_start, scanned in place below)
  for (int g = tid; g < p.G; g += blockDim.x) {
    int lo = p.grp_resp_off[g], hi = p.grp_resp_off[g + 1];
    bool ok = p.grp_prompt_len[g] >= 1 && hi > lo && lo >= 0 && hi <= p.N;
    if (!ok) {
      set_status(p.header, kStatusBadDescriptor, g);
      continue;
    }
    p.seg_start[g + lo] = p.grp_prompt_len[g];
    for (int x = lo; x < hi; ++x) {
      int len = p.resp_len[x];
      if (len < 1) set_status(p.header, kStatusBadDescriptor, p.G + x);
      p.seg_start[g + 1 + x] = len;
    }
  }
  __syncthreads();
  if (p.header[0] != kStatusOk) return false;

  // chunked exclusive scan of lengths and tile counts
  for (int base = 0; base < p.nseg; base += blockDim.x) {
    int s = base + tid;
    int len = s < p.nseg ? p.seg_start[s] : 0;
    // guard against overflow from absurd lengths
    if (len > p.T) len = p.T + 1;
    int til = (len + kTile - 1) / kTile;
    s_tok[tid] = len;
    s_til[tid] = til;
    __syncthreads();
    for (int d = 1; d < (int)blockDim.x; d <<= 1) {
      int a = tid >= d ? s_tok[tid - d] : 0;
      int b = tid >= d ? s_til[tid - d] : 0;
      __syncthreads();
      // saturate so a corrupted descriptor cannot wrap around
      s_tok[tid] = min(s_tok[tid] + a, 0x3fffffff);
      s_til[tid] += b;
      __syncthreads();
    }
    if (s < p.nseg) {
      p.seg_start[s] = s_carry[0] + s_tok[tid] - len;
      p.seg_tile0[s] = s_carry[1] + s_til[tid] - til;
    }
    __syncthreads();
    if (tid == blockDim.x - 1) {
      s_carry[0] = min(s_carry[0] + s_tok[tid], 0x3fffffff);
      s_carry[1] += s_til[tid];
    }
    __syncthreads();
  }
  if (tid == 0) {
    p.seg_start[p.nseg] = s_carry[0];
    p.seg_tile0[p.nseg] = s_carry[1];
    if (s_carry[0] != p.T) {
      set_status(p.header, kStatusTokenMismatch, s_carry[0]);
    } else {
      p.header[2] = p.header[kHdrNumQTiles] = s_carry[1];  // number of tiles
    }
  }
  __syncthreads();
  if (p.header[0] != kStatusOk) return false;

  // backward tiles: ceil(group length / 128) per group, exclusive scan over the groups
  if (tid == 0) s_carry[1] = 0;
  if (p.qtiles)
    for (int g = tid; g < p.G; g += blockDim.x) p.grid_gain[g] = 0;
  __syncthreads();
  for (int base = 0; base < p.G; base += blockDim.x) {
    const int g = base + tid;
    int til = 0;
    if (g < p.G) {
      const int gs = p.seg_start[g + p.grp_resp_off[g]];
      const int ge = p.seg_start[(g + 1) + p.grp_resp_off[g + 1]];
      til = (ge - gs + kTile - 1) / kTile;
    }
    s_til[tid] = til;
    __syncthreads();
    for (int d = 1; d < (int)blockDim.x; d <<= 1) {
      int b = tid >= d ? s_til[tid - d] : 0;
      __syncthreads();
      s_til[tid] += b;
      __syncthreads();
    }
    if (g < p.G) p.grp_btile0[g] = s_carry[1] + s_til[tid] - til;
    __syncthreads();
    if (tid == blockDim.x - 1) s_carry[1] += s_til[tid];
    __syncthreads();
  }
  if (tid == 0) {
    p.grp_btile0[p.G] = s_carry[1];
    p.header[kHdrNumBTiles] = s_carry[1];
  }
  __syncthreads();
  return true;
}

__global__ void __launch_bounds__(1024) plan_scan_kernel(PlanPtrs p) { plan_scan_body(p); }

// largest s in [0, n) with a[s] <= x  (a is non-decreasing, a[0] <= x)
__device__ __forceinline__ int upper_segment(const int32_t* a, int n, int x) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (a[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

// group of segment s: the largest g with g + resp_off[g] <= s
__device__ __forceinline__ int group_of_segment(const PlanPtrs& p, int s) {
  int lo = 0, hi = p.G;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (mid + p.grp_resp_off[mid] <= s) lo = mid; else hi = mid;
  }
  return lo;
}

// Query tile of the grid, from the group's start, the prompt's end, and start and end of the
// segment of the first row.
__device__ __forceinline__ QTile grid_query_tile(int start, int len, int gs, int pe, int ss, int se) {
  const bool prompt = start < pe;
  QTile q;
  q.start = start;
  q.len = len;
  q.kv0_start = gs;
  q.kv0_len = prompt ? start - gs : pe - gs;
  q.kv1_start = prompt ? start : ss;
  q.kv1_len = prompt ? 0 : start - ss;
  q.first_rows = min(len, se - start) + (prompt ? kQTilePrompt : 0);
  q.work = (q.kv0_len + kTile - 1) / kTile + (q.kv1_len + kTile - 1) / kTile + 1;
  return q;
}
// a segment's tile as query tile: rows of one segment
__device__ __forceinline__ QTile segment_query_tile(const Tile& t) {
  return {t.start, t.len, t.kv0_start, t.kv0_len, t.kv1_start, t.kv1_len, t.len, t.work};
}
// Work of a query tile in the choice between the two: its key tiles, and one for its beginning and
// end.
__device__ __forceinline__ int tile_cost(int work) { return work + 1; }
__device__ __forceinline__ void add_grid_gain(const PlanPtrs& p, int g, int gain) {
  atomicAdd(reinterpret_cast<unsigned long long*>(p.grid_gain + g),
            static_cast<unsigned long long>(static_cast<long long>(gain)));
}

// Whether two query tiles of a segment go into one unit, by the key tiles of the second and of the whole
// forward: such a unit takes 1.4 times as long as that tile alone (1.6 times at head_dim 64), which must not
// be longer than every SM's share of everything.  So the longest tiles of uneven batches stay alone.  All by
// twos -> none -> by this rule: one group of 6000 tokens and thirty of 600, 3 / 3 heads, D 64 69.6 -> 53.2 -> 51.2
// us; 14384 and forty of 600, 2 / 2, D 128 161.9 -> 149.5 -> 145.4; 20000 and a hundred of 300, 1 / 1
// 212.8 -> 188.5 -> 188.4; the same, 2 / 2 225.4 -> 253.9 -> 204.8.  Even batches go by twos as before.
__device__ __forceinline__ bool pair_pays(const PlanPtrs& p, int work, long long all_work) {
  return (long long)p.pair_cost * p.sms * work <= p.Hkv * all_work * p.unit_cost;
}
// ... for a tile of `work` of which tile_unit_of says `unit` (the tile behind it has one key tile more)
__device__ __forceinline__ uint8_t settled_unit(const PlanPtrs& p, uint8_t unit, int work, long long all_work) {
  return pair_pays(p, work + (unit == kTileNone), all_work) ? unit : uint8_t(kTileAlone);
}

__device__ __forceinline__ int plan_tile_body(const PlanPtrs& p, int t) {
  int s = upper_segment(p.seg_tile0, p.nseg, t);
  // segments with zero tiles cannot exist (len >= 1), so seg_tile0 is strictly increasing
  int g = group_of_segment(p, s);
  int sp = g + p.grp_resp_off[g];             // the group's prompt segment
  int gs = p.seg_start[sp];
  int P = p.grp_prompt_len[g];
  int gend = p.seg_start[(g + 1) + p.grp_resp_off[g + 1]];  // next group's prompt (or T)
  int ss = p.seg_start[s], se = p.seg_start[s + 1];
  int start = ss + (t - p.seg_tile0[s]) * kTile;
  Tile tl;
  tl.start = start;
  tl.len = min(kTile, se - start);
  if (s == sp) {
    tl.kv0_start = gs;  tl.kv0_len = start - gs;
    tl.kv1_start = start; tl.kv1_len = 0;
    tl.vis_end = gend;
  } else {
    tl.kv0_start = gs;  tl.kv0_len = P;
    tl.kv1_start = ss;  tl.kv1_len = start - ss;
    tl.vis_end = se;
  }
  tl.work = (tl.kv0_len + kTile - 1) / kTile + (tl.kv1_len + kTile - 1) / kTile + 1;
  p.tiles[t] = tl;
  if (p.tile_unit) p.tile_unit[t] = tile_unit_of(t - p.seg_tile0[s], p.seg_tile0[s + 1] - p.seg_tile0[s]);
  if (p.qtiles) add_grid_gain(p, g, tile_cost(tl.work));
  return tl.work;
}

__global__ void plan_tiles_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (p.qtiles && t < work_slots(p)) p.work_at[t] = 0;
  const int work = t < p.header[2] ? plan_tile_body(p, t) : 0;
  if (p.tile_unit) {
    const int sum = __reduce_add_sync(0xffffffffu, work);
    if ((threadIdx.x & 31) == 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(p.header + kHdrFwdWork), static_cast<unsigned long long>(sum));
  }
}

__device__ __forceinline__ void plan_key_end_body(const PlanPtrs& p, int j) {
  int s = upper_segment(p.seg_start, p.nseg, j);
  int g = group_of_segment(p, s);
  bool prompt = (s == g + p.grp_resp_off[g]);
  p.key_end[j] = prompt ? p.seg_start[(g + 1) + p.grp_resp_off[g + 1]] : p.seg_start[s + 1];
}

__global__ void plan_key_end_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < p.T) plan_key_end_body(p, j);
}

// Backward tile t: tile k of its group's 128-token grid.
__device__ __forceinline__ void plan_btile_body(const PlanPtrs& p, int t) {
  const int g = upper_segment(p.grp_btile0, p.G, t);
  const int sp = g + p.grp_resp_off[g];  // the group's prompt segment
  const int gs = p.seg_start[sp];
  const int pe = p.seg_start[sp + 1];    // end of the prompt
  const int ge = p.seg_start[(g + 1) + p.grp_resp_off[g + 1]];
  BTile b;
  b.start = gs + (t - p.grp_btile0[g]) * kTile;
  b.len = min(kTile, ge - b.start);
  b.grp_start = gs;
  b.grp_end = ge;
  // segments of the first and of the last key
  const int s_first = upper_segment(p.seg_start, p.nseg, b.start);
  const int s_last = upper_segment(p.seg_start, p.nseg, b.start + b.len - 1);
  // key_end is the group's end for prompt keys and the own response's end otherwise; along
  // the tile it is: (group end for the prompt part,) then increasing response ends
  b.vis_end = (s_first == sp) ? ge : p.seg_start[s_last + 1];
  b.work = 1 + (b.vis_end - (b.start + b.len) + kTile - 1) / kTile;
  b.npc = (pe - gs + kTile - 1) / kTile;
  // Read as a QUERY tile: the key tiles that add to its dQ are the prompt tiles [0, npc) and
  // the tiles [dep_lo, own index] -- from the one holding the start of the first row's own
  // response on (earlier tiles past the prompt hold only earlier responses' keys).
  const int k_rel = (b.start - gs) / kTile;
  b.dep_lo = k_rel;
  if (b.start >= pe) b.dep_lo = max(b.npc, (p.seg_start[s_first] - gs) / kTile);
  p.btiles[t] = b;
  if (p.qtiles)
    add_grid_gain(p, g, -tile_cost(grid_query_tile(b.start, b.len, gs, pe, p.seg_start[s_first],
                                                   p.seg_start[s_first + 1]).work));
}

// Query tile t: a group's tiles stand where the tiles of its segments do, those of the grid (never
// more of them) followed by empty ones of no work.
__device__ __forceinline__ void plan_qtile_body(const PlanPtrs& p, int t) {
  const int g = group_of_segment(p, upper_segment(p.seg_tile0, p.nseg, t));
  if (p.grid_gain[g] <= 0) {
    p.qtiles[t] = segment_query_tile(p.tiles[t]);
    return;
  }
  const int sp = g + p.grp_resp_off[g], i = t - p.seg_tile0[sp];
  QTile q{};
  if (i < p.grp_btile0[g + 1] - p.grp_btile0[g]) {
    const BTile b = p.btiles[p.grp_btile0[g] + i];
    const int s = upper_segment(p.seg_start, p.nseg, b.start);
    q = grid_query_tile(b.start, b.len, b.grp_start, p.seg_start[sp + 1], p.seg_start[s], p.seg_start[s + 1]);
  } else {
    atomicSub(&p.header[kHdrNumQTiles], 1);
  }
  p.qtiles[t] = q;
}

__global__ void plan_btiles_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < p.header[kHdrNumBTiles]) plan_btile_body(p, t);
}

// Longest-work-first orders by rank counting (tile counts are small: T/128 + segments).
__device__ __forceinline__ void plan_fwd_order_body(const PlanPtrs& p, int t, int n) {
  const int wf = p.tiles[t].work;
  int rf = 0;
  for (int u = 0; u < n; ++u) {
    const int of = p.tiles[u].work;
    rf += (of > wf) || (of == wf && u < t);
  }
  p.fwd_order[rf] = t;
  if (p.tile_unit)
    p.tile_unit[t] = settled_unit(p, p.tile_unit[t], wf, *reinterpret_cast<const long long*>(p.header + kHdrFwdWork));
}

// The query tiles' order by counting: tiles per work (plan_fwd_order_kernel), where each work begins
// (plan_gwork_kernel), and the tiles into their places (plan_sgroup_kernel).  Counting every
// tile's rank as above is quadratic, and with many short segments that cost the plan more than the mixed
// tiles save the forward of a head or two: 600 groups of 64 short responses 2073 us without them, 2947
// with, now 2135; 2048 groups of eight 8-token responses 971, 1362, 1007; 64 groups of 64 responses 292,
// 383, 302.  Tiles of equal work stand in the order their warps come.
// Adds one to the count of this thread's work (if it has one) and gives its old value.  Whole warps call:
// one atomic for all lanes with the same work.
__device__ __forceinline__ int count_work(const PlanPtrs& p, bool has, int work) {
  const uint32_t all = __ballot_sync(0xffffffffu, has);
  if (!has) return 0;
  const int slot = min(work, work_slots(p) - 1), lane = threadIdx.x & 31;
  const uint32_t same = __match_any_sync(all, slot);
  const int first = __ffs(same) - 1;
  int base = 0;
  if (lane == first) base = atomicAdd(&p.work_at[slot], __popc(same));
  return __shfl_sync(same, base, first) + __popc(same & ((1u << lane) - 1u));
}
// One block: the counts become the places of the first tiles, largest work first.
__device__ __forceinline__ void plan_work_places(const PlanPtrs& p) {
  __shared__ int32_t s_sum[32];
  const int n = work_slots(p), per = (n + blockDim.x - 1) / blockDim.x;
  const int hi = n - int(threadIdx.x) * per, lo = max(hi - per, 0);   // thread 0 has the largest
  int sum = 0;
  for (int i = lo; i < hi; ++i) sum += p.work_at[i];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int before = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, before, d);
    if (lane >= d) before += x;
  }
  if (lane == 31) s_sum[warp] = before;
  __syncthreads();
  for (int w = 0; w < warp; ++w) before += s_sum[w];
  before -= sum;
  for (int i = hi - 1; i >= lo; --i) {
    const int c = p.work_at[i];
    p.work_at[i] = before;
    before += c;
  }
}

__global__ void plan_fwd_order_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  const int n = p.header[kHdrNumTiles];
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) plan_fwd_order_body(p, t, n);
  if (p.qtiles) {
    if (t < n) plan_qtile_body(p, t);
    count_work(p, t < n, t < n ? p.qtiles[t].work : 0);
  }
}

// Backward processing order, built for L2 reuse and balance.  Key tiles of one group stream
// the same Q / dO tiles, so groups are taken in order of decreasing work and consecutive
// groups are merged into super-groups of about kSuperGroupUnits units (cut from the end of
// the list, so the last block is a full one); inside a super-group
// units are ordered longest first (all KV heads of a tile adjacent).  Small problems collapse
// into one super-group, i.e. a plain longest-first list; large ones keep the working set of the
// concurrently running units near one group's Q / dO.  Dynamic scheduling in the kernel does
// the balancing.  A tile's group is identified by the group's first token.

// The blocks of the order that the kernel takes with several query heads per KV head
// (bwd_takes_sched, which has the reasons).  The last block begins with the first group behind which
// there are fewer than kSchedTailUnits units, or not enough work to balance its longest unit: with less
// than two thirds of that unit behind it for each of 148 SMs, 12000 tokens in four groups (28 / 4 heads, D 64,
// 384 units) took 490 us, all in one block 455.  But for that it does not grow beyond a super-group: of 21883
// tokens, 10844 in one group, at 32 / 8 heads, D 96, it took all 1424 units, whose data L2 does not hold: main
// kernel and streams 1648 us, with the limit 1580; 8000 tokens and eight groups of 1000, 32 / 8 1355 -> 1295.
// `later`, `later_work` = tiles of the groups ranked behind a group of `tiles` tiles, and their work.
__device__ __forceinline__ bool sched_tail(const PlanPtrs& p, int later, int later_work, int tiles) {
  return p.Hkv * later < kSchedTailUnits || ((long long)p.Hkv * later_work < 100LL * tiles &&
                                             p.Hkv * (later + tiles) <= kSuperGroupUnits);
}
// `tail` = tiles of the groups in the last block, `total` = of all.  (At most 1007 blocks -- the divisor is
// rounded down and at least 150 --, which the one-block plan's sort keys have room for.)
__device__ __forceinline__ int sched_block(const PlanPtrs& p, int later, int tail, int total) {
  return later < tail ? 0 : 1 + p.Hkv * (later - tail) / max(kSchedBlockUnits, p.Hkv * total / 1000);
}
// The values [lo, hi) of `later` that fall into the same block.  (The plan of several kernels compares every
// pair of tiles: with a division for each, and groups' works added up tile by tile, a plan of 300000 tokens in
// 1000 groups took 981 us, now 685.)
__device__ __forceinline__ void sched_block_range(int Hkv, int later, int tail, int total, int& lo, int& hi) {
  lo = 0, hi = tail;
  if (later < tail) return;
  const int unit = max(kSchedBlockUnits, Hkv * total / 1000), q = Hkv * (later - tail) / unit;
  lo = tail + (q * unit + Hkv - 1) / Hkv;
  hi = tail + ((q + 1) * unit + Hkv - 1) / Hkv;
}

// bwd_order (plain longest-first list of the backward tiles) and each tile's group work
__device__ __forceinline__ void plan_gwork_body(const PlanPtrs& p, int t, int n) {
  const BTile me = p.btiles[t];
  int gw = 0, rb = 0;
  for (int u = 0; u < n; ++u) {
    const BTile o = p.btiles[u];
    gw += (o.grp_start == me.grp_start) ? o.work : 0;
    rb += (o.work > me.work) || (o.work == me.work && u < t);
  }
  p.tile_gwork[t] = gw;
  p.bwd_order[rb] = t;
}

__device__ __forceinline__ void plan_sgroup_body(const PlanPtrs& p, int t, int n) {
  const BTile me = p.btiles[t];
  const int gw = p.tile_gwork[t];
  // tiles and work of the groups that come later
  int later = 0, later_work = 0;
#pragma unroll 4
  for (int g = 0; g < p.G; ++g) {
    const int first = p.grp_btile0[g], ow = p.tile_gwork[first];
    if (ow < gw || (ow == gw && first > t)) {
      later += p.grp_btile0[g + 1] - first;
      later_work += ow;
    }
  }
  const int own = (me.grp_end - me.grp_start + kTile - 1) / kTile, rest = later + own;
  if (!p.sched) {
    // counted from the END of the list, so the last block is never a small leftover whose
    // long units would start late: blocks are processed in decreasing index
    p.tile_block[t] = (p.Hkv * rest - 1) / kSuperGroupUnits;
  } else {
    p.tile_block[t] = later;
    if (sched_tail(p, later, later_work, own)) atomicMax(&p.header[kHdrSchedTail], rest);
  }
}

__device__ __forceinline__ void plan_units_body(const PlanPtrs& p, int t, int n) {
  const int wb = p.btiles[t].work, mine = p.tile_block[t];
  int lo = mine, hi = mine + 1;   // the values of tile_block in this tile's block
  if (p.sched) sched_block_range(p.Hkv, mine, p.header[kHdrSchedTail], n, lo, hi);
  int pos = 0;
  for (int u = 0; u < n; ++u) {
    const int other = p.tile_block[u], ob = p.btiles[u].work;
    pos += (other >= hi) || (other >= lo && ((ob > wb) || (ob == wb && u < t)));
  }
  for (int kvh = 0; kvh < p.Hkv; ++kvh) p.bwd_units[p.Hkv * pos + kvh] = (kvh << 24) | t;
  // Deterministic order: one (group, KV head) set after the other, groups by decreasing work.
  // The tiles add to a query tile's dQ in descending order, so a unit waits for the unit of the
  // next tile.  Inside a set the units go out in ascending tile order (longest first, as in the
  // default order) when the set is small against the grid: only the one set at the frontier of
  // the list can have units waiting for a unit that has not been handed out yet, so fewer than
  // det_asc_max CTAs can be held up that way and the others keep drawing.  Larger sets go out
  // in DESCENDING tile order, where every unit follows the units it waits for.
  const int gs = p.btiles[t].grp_start, gw = p.tile_gwork[t];
  int before = 0, ng = 0;  // tiles of groups ranked earlier; tiles of this group
  for (int u = 0; u < n; ++u) {
    const int ogs = p.btiles[u].grp_start, ow = p.tile_gwork[u];
    before += (ow > gw) || (ow == gw && ogs < gs);
    ng += (ogs == gs);
  }
  const int k_rel = (p.btiles[t].start - gs) / kTile;
  const int slot = ng <= p.det_asc_max ? k_rel : ng - 1 - k_rel;
  for (int kvh = 0; kvh < p.Hkv; ++kvh)
    p.bwd_units_det[p.Hkv * before + kvh * ng + slot] = (kvh << 24) | t;
}

__global__ void plan_gwork_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  const int n = p.header[kHdrNumBTiles];
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) plan_gwork_body(p, t, n);
  if (p.qtiles && blockIdx.x == gridDim.x - 1) plan_work_places(p);
}

__global__ void plan_sgroup_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  const int n = p.header[kHdrNumBTiles];
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (p.qtiles) {
    const bool there = t < p.header[kHdrNumTiles];
    const int at = count_work(p, there, there ? p.qtiles[t].work : 0);
    if (there) p.qorder[at] = t;
  }
  if (t < n) plan_sgroup_body(p, t, n);
}

__global__ void plan_units_kernel(PlanPtrs p) {
  if (p.header[0] != kStatusOk) return;
  const int n = p.header[kHdrNumBTiles];
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) plan_units_body(p, t, n);
}

// ---------------------------------------------------------------- host descriptors
template <size_t N>
struct DescBlock {
  int32_t v[N];
};
constexpr size_t kDescSmall = 960, kDescFused = 4104, kDescLarge = 7168;

void fill_desc(const int32_t* const* src, const size_t (&n)[4], int32_t* dst) {
  for (int i = 0; i < 4; ++i) {
    memcpy(dst, src[i], n[i] * sizeof(int32_t));
    dst += n[i];
  }
}

template <size_t N>
__global__ void stage_desc_kernel(const __grid_constant__ DescBlock<N> blk, int n, int32_t* dst) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = blk.v[i];
}

// ---------------------------------------------------------------- the whole plan in one block
// Used when the problem is small enough that one block's latency beats eight dependent launches.
// It is all latency: a few thousand integers through a chain of dependent steps.  So everything
// that is read back -- descriptors, segment and tile offsets, works -- stays in shared memory (a
// dependent read costs 30 cycles there instead of 300 - 700), host descriptors arrive as a kernel
// argument without a staging kernel in front, scans are two barriers, the block has no more
// threads than the plan has use for (idle warps take issue slots from the others), and the orders
// come from 32-bit keys, work and index in one word: up to kRankTiles tiles by counting the
// smaller keys (n^2 comparisons spread over the block: 300 cycles for 128 keys), beyond by a
// bitonic sort (66 steps for 2048).  Eight 1100-token groups 17.4 -> 8.2 us, four 4800-token
// groups 27 -> 12, two rows of 32768 tokens 118 -> 32, 40000 tokens in 1330 short segments
// 194 -> 52.
constexpr int kRankTiles = 512;
constexpr int kFusedSmallTiles = 256;  // blocks of 256 threads up to here, 1024 beyond
constexpr int kFusedMaxTiles = 2048;   // tiles; also bounds the segments, and twice the groups

// kMixed: with the forward's mixed query tiles (an instance of its own: carried along, their code
// and space cost the plans without them 1 us)
template <bool kMixed>
struct FusedSmem {
  union alignas(16) {   // (keys are read as uint4)
    uint32_t sort[2][kMixed ? 4 : 3][kFusedMaxTiles];
    struct {
      uint32_t key[kMixed ? 5 : 4][kRankTiles];      // forward tiles, backward tiles, groups, backward units,
      int32_t rank[kMixed ? 5 : 4][kRankTiles];      //   query tiles (groups: backward tiles of the groups before)
    } r;
  } o;
  int32_t desc[kDescFused];
  int32_t seg_start[kFusedMaxTiles + 1];
  int32_t seg_tile0[kFusedMaxTiles + 1];
  int32_t btile0[kFusedMaxTiles / 2 + 1];
  int32_t tile[3][kFusedMaxTiles];      // start, end, vis_end of the forward tiles
  int32_t gwork[kFusedMaxTiles / 2];    // backward work of each group
  int32_t before[kFusedMaxTiles / 2];   // backward tiles of the groups ranked before it
  uint16_t seg_grp[kFusedMaxTiles];
  uint16_t wb[kFusedMaxTiles];          // work and group of the backward tiles
  uint16_t bgrp[kFusedMaxTiles];
  int32_t grid_gain[kMixed ? kFusedMaxTiles / 2 : 1];
  uint16_t qwork[kMixed ? kFusedMaxTiles : 2];       // work of the query tiles, 0 where there is none
  uint16_t unit_tile[kFusedMaxTiles];   // backward tiles in the order of their units
  int32_t warp_sum[2][32];
  int32_t status, detail, no_qtile, sched_tail, fwd_work;
};

// Inclusive sums of two values over the block.
__device__ __forceinline__ void block_scan2(int& a, int& b, int32_t (&s_warp)[2][32]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto warp_scan = [&](int& x, int& y) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int xa = __shfl_up_sync(0xffffffffu, x, d), yb = __shfl_up_sync(0xffffffffu, y, d);
      if (lane >= d) {
        x += xa;
        y += yb;
      }
    }
  };
  warp_scan(a, b);
  if (lane == 31) {
    s_warp[0][warp] = a;
    s_warp[1][warp] = b;
  }
  __syncthreads();
  if (warp == 0) {
    const bool there = lane < int(blockDim.x >> 5);
    int x = there ? s_warp[0][lane] : 0, y = there ? s_warp[1][lane] : 0;
    warp_scan(x, y);
    s_warp[0][lane] = x;
    s_warp[1][lane] = y;
  }
  __syncthreads();
  if (warp) {
    a += s_warp[0][warp - 1];
    b += s_warp[1][warp - 1];
  }
}

// rank[t] += (weight of the) keys below key t, for m <= kRankTiles keys: the block's threads form
// slices of a power of two >= m threads, each counts over its part of the keys (read four at a
// time, the same ones by all lanes of a warp).  Keys are padded to a multiple of four with ~0.
template <bool kWeighted>
__device__ __forceinline__ void rank_count(const uint32_t* key, int m, int32_t* rank, const int32_t* off) {
  int lg = 5;
  while ((1 << lg) < m) ++lg;
  const int t = threadIdx.x & ((1 << lg) - 1), slice = threadIdx.x >> lg, slices = blockDim.x >> lg;
  const int quads = (m + 3) >> 2, per = (quads + slices - 1) / slices;
  const int lo = slice * per, hi = min(lo + per, quads);
  if (t >= m || lo >= hi) return;
  const uint32_t mine = key[t];
  int count = 0;
#pragma unroll 2
  for (int i = lo; i < hi; ++i) {
    const uint4 k = reinterpret_cast<const uint4*>(key)[i];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (kk[c] < mine) count += kWeighted ? off[4 * i + c + 1] - off[4 * i + c] : 1;
  }
  if (count) atomicAdd(&rank[t], count);
}

// Ascending bitonic sort of kArrays arrays of `n2` (1024 or 2048) keys in a block of 1024 threads,
// key tid + 1024 r of each in v[.][r].  Distances below 32 are shuffles, 1024 is inside the thread,
// the others go through shared memory (two buffers in turn: one barrier per distance).
template <int kArrays, int kBufs>
__device__ __forceinline__ void bitonic_sort(uint32_t (&v)[kArrays][2], int n2,
                                             uint32_t (&buf)[2][kBufs][kFusedMaxTiles]) {
  const int tid = threadIdx.x;
  const bool two = n2 > 1024;
  int turn = 0;
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j == 1024) {   // k = 2048: ascending throughout
#pragma unroll
        for (int a = 0; a < kArrays; ++a) {
          const uint32_t lo = min(v[a][0], v[a][1]), hi = max(v[a][0], v[a][1]);
          v[a][0] = lo;
          v[a][1] = hi;
        }
        continue;
      }
      // the lower key of a pair keeps the smaller one where the run ascends, and vice versa
      const bool small0 = ((tid & j) == 0) == ((tid & k) == 0);
      const bool small1 = ((tid & j) == 0) == (((tid + 1024) & k) == 0);
      if (j >= 32) {
#pragma unroll
        for (int a = 0; a < kArrays; ++a) {
          buf[turn][a][tid] = v[a][0];
          if (two) buf[turn][a][tid + 1024] = v[a][1];
        }
        __syncthreads();
#pragma unroll
        for (int a = 0; a < kArrays; ++a) {
          const uint32_t o = buf[turn][a][tid ^ j];
          v[a][0] = small0 ? min(v[a][0], o) : max(v[a][0], o);
          if (two) {
            const uint32_t q = buf[turn][a][(tid ^ j) + 1024];
            v[a][1] = small1 ? min(v[a][1], q) : max(v[a][1], q);
          }
        }
        turn ^= 1;
      } else {
#pragma unroll
        for (int a = 0; a < kArrays; ++a) {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, v[a][0], j);
          v[a][0] = small0 ? min(v[a][0], o) : max(v[a][0], o);
          if (two) {
            const uint32_t q = __shfl_xor_sync(0xffffffffu, v[a][1], j);
            v[a][1] = small1 ? min(v[a][1], q) : max(v[a][1], q);
          }
        }
      }
    }
  }
}

template <size_t kDesc, bool kMixed>
__global__ void __launch_bounds__(1024)
plan_fused_kernel(const __grid_constant__ DescBlock<kDesc> blk, PlanPtrs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FusedSmem<kMixed>& sm = *reinterpret_cast<FusedSmem<kMixed>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nthr = blockDim.x;
  const int n_rgo = p.num_rows + 1, n_all = n_rgo + p.G + p.G + 1 + p.N;
  launch_dependents();
  // ---- descriptors -> shared memory, and the copy that later kernels read
  if (kDesc > 1) {
    for (int i = tid; i < n_all; i += nthr) sm.desc[i] = blk.v[i];
  } else {
    dependency_wait();
    const int n[4] = {n_rgo, p.G, p.G + 1, p.N};
    int at = 0;
    for (int a = 0; a < 4; ++a) {
      for (int i = tid; i < n[a]; i += nthr) sm.desc[at + i] = p.src_desc[a][i];
      at += n[a];
    }
  }
  if (tid == 0) {
    sm.status = kStatusOk;
    sm.detail = sm.no_qtile = sm.sched_tail = sm.fwd_work = 0;
  }
  if (kDesc > 1) dependency_wait();   // (the workspace may still be in use up to here)
  __syncthreads();
  for (int i = tid; i < n_all; i += nthr) p.desc_copy[i] = sm.desc[i];
  const int32_t* rgo = sm.desc;
  const int32_t* gpl = rgo + n_rgo;
  const int32_t* gro = gpl + p.G;
  const int32_t* rlen = gro + p.G + 1;
  auto fail = [&](int32_t status, int32_t detail) {
    if (atomicCAS(&sm.status, kStatusOk, status) == kStatusOk) sm.detail = detail;
  };
  auto give_up = [&]() {   // the header of a plan that was refused
    if (tid < 16)
      p.header[tid] = tid == kHdrStatus ? sm.status
                      : tid == kHdrDetail ? sm.detail : tid == kHdrNumSegments ? p.nseg : 0;
  };
  // ---- validation, segment lengths
  if (tid == 0) {
    if (rgo[0] != 0 || rgo[p.num_rows] != p.G) fail(kStatusBadDescriptor, -1);
    if (gro[0] != 0 || gro[p.G] != p.N) fail(kStatusBadDescriptor, -2);
  }
  __syncthreads();
  for (int r = tid; r < p.num_rows; r += nthr)
    if (rgo[r + 1] < rgo[r]) fail(kStatusBadDescriptor, r);
  for (int g = tid; g < p.G; g += nthr) {
    const int lo = gro[g], hi = gro[g + 1];
    if (!(gpl[g] >= 1 && hi > lo && lo >= 0 && hi <= p.N)) {
      fail(kStatusBadDescriptor, g);
      continue;
    }
    sm.seg_start[g + lo] = gpl[g];
    sm.seg_grp[g + lo] = uint16_t(g);
    for (int x = lo; x < hi; ++x) {
      const int len = rlen[x];
      if (len < 1) fail(kStatusBadDescriptor, p.G + x);
      sm.seg_start[g + 1 + x] = len;
      sm.seg_grp[g + 1 + x] = uint16_t(g);
    }
  }
  __syncthreads();
  if (sm.status != kStatusOk) {
    give_up();
    return;
  }
  // ---- first token and first tile of every segment: two segments per thread
  {
    const int s0 = 2 * tid, s1 = s0 + 1;
    // (a length beyond T is a mismatch anyway; clamped, 2048 of them cannot overflow)
    const int l0 = s0 < p.nseg ? min(sm.seg_start[s0], p.T + 1) : 0;
    const int l1 = s1 < p.nseg ? min(sm.seg_start[s1], p.T + 1) : 0;
    const int c0 = (l0 + kTile - 1) / kTile, c1 = (l1 + kTile - 1) / kTile;
    int tok = l0 + l1, til = c0 + c1;
    block_scan2(tok, til, sm.warp_sum);
    // (the barriers inside the scan order these writes behind the reads above)
    if (s0 <= p.nseg) {
      sm.seg_start[s0] = tok - l0 - l1;
      sm.seg_tile0[s0] = til - c0 - c1;
    }
    if (s1 <= p.nseg) {
      sm.seg_start[s1] = tok - l1;
      sm.seg_tile0[s1] = til - c1;
    }
    if (tid == nthr - 1) {
      if (p.nseg == 2 * nthr) {   // (entry nseg is past the last pair)
        sm.seg_start[p.nseg] = tok;
        sm.seg_tile0[p.nseg] = til;
      }
      if (tok != p.T) fail(kStatusTokenMismatch, tok);
    }
  }
  __syncthreads();
  if (sm.status != kStatusOk) {
    give_up();
    return;
  }
  const int n = sm.seg_tile0[p.nseg];
  // ---- first backward tile of every group
  {
    int til = 0, unused = 0;
    if (tid < p.G)
      til = (sm.seg_start[tid + 1 + gro[tid + 1]] - sm.seg_start[tid + gro[tid]] + kTile - 1) / kTile;
    const int mine = til;
    block_scan2(til, unused, sm.warp_sum);
    if (tid < p.G) {
      sm.btile0[tid] = til - mine;
      if (kMixed) sm.grid_gain[tid] = 0;
    }
    if (tid == p.G - 1) sm.btile0[p.G] = til;
  }
  if constexpr (kMixed) __syncthreads();
  // ---- forward tiles
  const bool by_rank = n <= kRankTiles;   // (there are at most as many backward tiles as forward
                                          // tiles, and fewer groups)
  // keys of tile (group) tid + nthr r: forward tiles, backward tiles, groups, query tiles
  constexpr int kOrders = kMixed ? 4 : 3;
  uint32_t key[kOrders][2];
  for (int a = 0; a < kOrders; ++a) key[a][0] = key[a][1] = ~0u;
  uint8_t unit[2];
  int work = 0;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int t = tid + nthr * r;
    if (t < n) {
      const int s = upper_segment(sm.seg_tile0, p.nseg, t), g = sm.seg_grp[s];
      const int sp = g + gro[g], gs = sm.seg_start[sp];
      const int ss = sm.seg_start[s], se = sm.seg_start[s + 1];
      Tile tl;
      tl.start = ss + (t - sm.seg_tile0[s]) * kTile;
      tl.len = min(kTile, se - tl.start);
      tl.kv0_start = gs;
      if (s == sp) {
        tl.kv0_len = tl.start - gs;
        tl.kv1_start = tl.start;
        tl.kv1_len = 0;
        tl.vis_end = sm.seg_start[g + 1 + gro[g + 1]];
      } else {
        tl.kv0_len = gpl[g];
        tl.kv1_start = ss;
        tl.kv1_len = tl.start - ss;
        tl.vis_end = se;
      }
      tl.work = (tl.kv0_len + kTile - 1) / kTile + (tl.kv1_len + kTile - 1) / kTile + 1;
      p.tiles[t] = tl;
      unit[r] = tile_unit_of(t - sm.seg_tile0[s], sm.seg_tile0[s + 1] - sm.seg_tile0[s]);
      sm.tile[0][t] = tl.start;
      sm.tile[1][t] = tl.start + tl.len;
      sm.tile[2][t] = tl.vis_end;
      key[0][r] = uint32_t(0xffff - tl.work) << 16 | uint32_t(t);
      if constexpr (kMixed) atomicAdd(&sm.grid_gain[g], tile_cost(tl.work));
      work += tl.work;
    }
  }
  if (!kMixed && p.tile_unit) {
    work = __reduce_add_sync(0xffffffffu, work);
    if (lane == 0) atomicAdd(&sm.fwd_work, work);
  }
  for (int s = tid; s <= p.nseg; s += nthr) p.seg_start[s] = sm.seg_start[s];
  __syncthreads();
  const int nb = sm.btile0[p.G];
  if (!kMixed && p.tile_unit) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (tid + nthr * r < n)
        p.tile_unit[tid + nthr * r] = settled_unit(p, unit[r], 0xffff - int(key[0][r] >> 16), sm.fwd_work);
  }
  QTile q[2];
  // ---- backward tiles; key_end (every key of a forward tile ends its visibility at vis_end)
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int t = tid + nthr * r;
    if (t >= nb) break;
    const int g = upper_segment(sm.btile0, p.G, t);
    const int sp = g + gro[g], s_end = g + 1 + gro[g + 1];   // the group's segments [sp, s_end)
    const int gs = sm.seg_start[sp], pe = sm.seg_start[sp + 1], ge = sm.seg_start[s_end];
    const int k_rel = t - sm.btile0[g];
    BTile b;
    b.start = gs + k_rel * kTile;
    b.len = min(kTile, ge - b.start);
    b.grp_start = gs;
    b.grp_end = ge;
    // (key_end and query-tile readings: see plan_btile_body)
    const int s_first = sp + upper_segment(sm.seg_start + sp, s_end - sp, b.start);
    const int s_last = sp + upper_segment(sm.seg_start + sp, s_end - sp, b.start + b.len - 1);
    b.vis_end = s_first == sp ? ge : sm.seg_start[s_last + 1];
    b.work = 1 + (b.vis_end - (b.start + b.len) + kTile - 1) / kTile;
    b.npc = (pe - gs + kTile - 1) / kTile;
    b.dep_lo = b.start >= pe ? max(b.npc, (sm.seg_start[s_first] - gs) / kTile) : k_rel;
    p.btiles[t] = b;
    sm.wb[t] = uint16_t(b.work);
    sm.bgrp[t] = uint16_t(g);
    key[1][r] = uint32_t(0xffff - b.work) << 16 | uint32_t(t);
    if constexpr (kMixed) {
      q[r] = grid_query_tile(b.start, b.len, gs, pe, sm.seg_start[s_first], sm.seg_start[s_first + 1]);
      atomicSub(&sm.grid_gain[g], tile_cost(q[r].work));
    }
  }
  for (int t = wid; t < n; t += nthr >> 5) {
    const int left = sm.tile[1][t] - sm.tile[0][t] - lane, vis_end = sm.tile[2][t];
    int32_t* at = p.key_end + sm.tile[0][t] + lane;
#pragma unroll
    for (int c = 0; c < kTile; c += 32)
      if (c < left) at[c] = vis_end;
  }
  __syncthreads();
  // ---- query tiles (see plan_qtile_body)
  if constexpr (kMixed) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int t = tid + nthr * r;
      if (t < n) {
        const int g = sm.seg_grp[upper_segment(sm.seg_tile0, p.nseg, t)];
        const int i = t - sm.seg_tile0[g + gro[g]], ng = sm.btile0[g + 1] - sm.btile0[g];
        if (sm.grid_gain[g] <= 0) {
          const QTile own = segment_query_tile(p.tiles[t]);
          p.qtiles[t] = own;
          sm.qwork[t] = uint16_t(own.work);
        } else if (i >= ng) {
          sm.qwork[t] = 0;
          atomicAdd(&sm.no_qtile, 1);
        }
      }
      if (t < nb) {
        const int g = sm.bgrp[t], at = sm.seg_tile0[g + gro[g]] + t - sm.btile0[g];
        if (sm.grid_gain[g] > 0) {
          p.qtiles[at] = q[r];
          sm.qwork[at] = uint16_t(q[r].work);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int t = tid + nthr * r;
      if (t < n) key[3][r] = uint32_t(0xffff - sm.qwork[t]) << 16 | uint32_t(t);
    }
  }
  // ---- work of every group (a warp each), groups in order of decreasing work
  for (int g = wid; g < p.G; g += nthr >> 5) {
    int w = 0;
    for (int t = sm.btile0[g] + lane; t < sm.btile0[g + 1]; t += 32) w += sm.wb[t];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) w += __shfl_xor_sync(0xffffffffu, w, d);
    if (lane == 0) sm.gwork[g] = w;
  }
  __syncthreads();
  // at most 2048 * 2049 / 2 < 2^22 units of work in a group, at most 1024 groups
  if (tid < p.G) key[2][0] = uint32_t(0x3fffff - sm.gwork[tid]) << 10 | uint32_t(tid);
  // super-groups or blocks (see above), inside one the longest tiles first; Hkv * nb / 600 < 512 and a
  // tile's work is 1 .. 2048
  auto unit_key = [&](int t, int ranked_before) {
    const int g = sm.bgrp[t], rest = nb - ranked_before, later = rest - (sm.btile0[g + 1] - sm.btile0[g]);
    const int block = p.sched ? sched_block(p, later, sm.sched_tail, nb) : (p.Hkv * rest - 1) / kSuperGroupUnits;
    return uint32_t(1023 - block) << 22 | uint32_t(2048 - sm.wb[t]) << 11 | uint32_t(t);
  };
  if (by_rank) {   // (blocks of 256 threads have at most 256 tiles: one per thread)
    for (int t = tid; t < kRankTiles; t += nthr) {
      sm.o.r.key[0][t] = t == tid ? key[0][0] : ~0u;
      sm.o.r.key[1][t] = t == tid ? key[1][0] : ~0u;
      sm.o.r.key[2][t] = t == tid ? key[2][0] : ~0u;
      sm.o.r.key[3][t] = ~0u;
      sm.o.r.rank[0][t] = sm.o.r.rank[1][t] = sm.o.r.rank[2][t] = sm.o.r.rank[3][t] = 0;
      if constexpr (kMixed) {
        sm.o.r.key[4][t] = t == tid ? key[3][0] : ~0u;
        sm.o.r.rank[4][t] = 0;
      }
    }
    __syncthreads();
    rank_count<false>(sm.o.r.key[0], n, sm.o.r.rank[0], nullptr);
    rank_count<false>(sm.o.r.key[1], nb, sm.o.r.rank[1], nullptr);
    rank_count<true>(sm.o.r.key[2], p.G, sm.o.r.rank[2], sm.btile0);
    if constexpr (kMixed) rank_count<false>(sm.o.r.key[4], n, sm.o.r.rank[4], nullptr);
    __syncthreads();
    if (p.sched) {
      if (tid < p.G) {
        const uint32_t mine = sm.o.r.key[2][tid];
        int later_work = 0;
        for (int g = 0; g < p.G; ++g) later_work += sm.o.r.key[2][g] > mine ? sm.gwork[g] : 0;
        const int rest = nb - sm.o.r.rank[2][tid], own = sm.btile0[tid + 1] - sm.btile0[tid];
        if (sched_tail(p, rest - own, later_work, own)) atomicMax(&sm.sched_tail, rest);
      }
      __syncthreads();
    }
    if (tid < n) p.fwd_order[sm.o.r.rank[0][tid]] = tid;
    if constexpr (kMixed)
      if (tid < n) p.qorder[sm.o.r.rank[4][tid]] = tid;
    if (tid < nb) {
      p.bwd_order[sm.o.r.rank[1][tid]] = tid;
      sm.o.r.key[3][tid] = unit_key(tid, sm.o.r.rank[2][sm.bgrp[tid]]);
    }
    if (tid < p.G) sm.before[tid] = sm.o.r.rank[2][tid];
    __syncthreads();
    rank_count<false>(sm.o.r.key[3], nb, sm.o.r.rank[3], nullptr);
    __syncthreads();
    if (tid < nb) sm.unit_tile[sm.o.r.rank[3][tid]] = uint16_t(tid);
    __syncthreads();
  } else {
    int n2 = 1024;
    while (n2 < n) n2 <<= 1;
    bitonic_sort(key, n2, sm.o.sort);
    // tiles of the groups ranked before each group
    int cnt = 0, work = 0, g = 0;
    if (tid < p.G) {
      g = int(key[2][0] & 1023u);
      cnt = sm.btile0[g + 1] - sm.btile0[g];
      work = sm.gwork[g];
    }
    const int mine = cnt;
    block_scan2(cnt, work, sm.warp_sum);
    const int all_work = sm.warp_sum[1][(nthr >> 5) - 1];
    if (tid < p.G) {
      sm.before[g] = cnt - mine;
      if (sched_tail(p, nb - cnt, all_work - work, mine)) atomicMax(&sm.sched_tail, nb - cnt + mine);
    }
    __syncthreads();
    uint32_t ukey[1][2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int t = tid + nthr * r;
      if (t < n) p.fwd_order[t] = int32_t(key[0][r] & 0xffffu);
      if constexpr (kMixed)
        if (t < n) p.qorder[t] = int32_t(key[3][r] & 0xffffu);
      if (t < nb) p.bwd_order[t] = int32_t(key[1][r] & 0xffffu);
      ukey[0][r] = t < nb ? unit_key(t, sm.before[sm.bgrp[t]]) : ~0u;
    }
    bitonic_sort(ukey, n2, sm.o.sort);
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (tid + nthr * r < nb) sm.unit_tile[tid + nthr * r] = uint16_t(ukey[0][r] & 2047u);
    __syncthreads();
  }
  // ---- backward units, in both orders
  for (int e = tid; e < nb * p.Hkv; e += nthr) {
    const int i = e / p.Hkv, kvh = e - i * p.Hkv;
    p.bwd_units[e] = (kvh << 24) | int(sm.unit_tile[i]);
    // deterministic backward: set after set (see plan_units_body)
    const int g = sm.bgrp[i], ng = sm.btile0[g + 1] - sm.btile0[g], k_rel = i - sm.btile0[g];
    const int slot = ng <= p.det_asc_max ? k_rel : ng - 1 - k_rel;
    p.bwd_units_det[p.Hkv * sm.before[g] + kvh * ng + slot] = (kvh << 24) | i;
  }
  if (tid < 16)   // (words 4 to 7: dynamic-scheduling counters)
    p.header[tid] = tid == kHdrNumTiles ? n
                    : tid == kHdrNumSegments ? p.nseg : tid == kHdrNumBTiles ? nb
                    : kMixed && tid == kHdrNumQTiles ? n - sm.no_qtile : 0;
}

}  // namespace

ProfileEvents& profile_events() {
  static ProfileEvents ev;
  return ev;
}

bool profile_enable(int mode) {
  ProfileEvents& ev = profile_events();
  const bool on = mode != 0;
  if (on && ev.on) {  // already on: the choice of kernels can change, and the counts restart
    ev.fwd_on = mode == 1;
    ev.fwd_count = ev.bwd_count = 0;
    return true;
  }
  if (on == ev.on) return true;
  if (on) {
    bool ok = true;
    for (int i = 0; i < kProfileRing && ok; ++i)
      ok = cudaEventCreate(&ev.fwd0[i]) == cudaSuccess && cudaEventCreate(&ev.fwd1[i]) == cudaSuccess &&
           cudaEventCreate(&ev.bwd0[i]) == cudaSuccess && cudaEventCreate(&ev.bwd1[i]) == cudaSuccess;
    ev.on = ok;
    ev.fwd_on = mode == 1;
    ev.fwd_count = ev.bwd_count = 0;
    return ok;
  }
  for (int i = 0; i < kProfileRing; ++i) {
    cudaEventDestroy(ev.fwd0[i]); cudaEventDestroy(ev.fwd1[i]);
    cudaEventDestroy(ev.bwd0[i]); cudaEventDestroy(ev.bwd1[i]);
  }
  ev = ProfileEvents();
  return true;
}

// Durations of the most recent launches, oldest first (at most kProfileRing are kept).
bool profile_read_all(float* fwd_ms, float* bwd_ms, int capacity, int* n_fwd, int* n_bwd) {
  ProfileEvents& ev = profile_events();
  if (!ev.on || capacity < 0) return false;
  bool ok = true;
  auto dump = [&](float* out, int* n_out, long long count, cudaEvent_t* e0, cudaEvent_t* e1) {
    const int n = int(std::min<long long>(std::min<long long>(count, kProfileRing), capacity));
    if (n_out) *n_out = n;
    if (!out) return;
    for (int i = 0; i < n; ++i) {
      const long long idx = count - n + i;
      ok = ok && cudaEventElapsedTime(&out[i], e0[idx % kProfileRing], e1[idx % kProfileRing]) == cudaSuccess;
    }
  };
  dump(fwd_ms, n_fwd, ev.fwd_count, ev.fwd0, ev.fwd1);
  dump(bwd_ms, n_bwd, ev.bwd_count, ev.bwd0, ev.bwd1);
  return ok;
}

bool profile_read(float* fwd_ms, float* bwd_ms) {
  ProfileEvents& ev = profile_events();
  if (!ev.on) return false;
  bool ok = true;
  if (fwd_ms) {
    const long long i = (ev.fwd_count - 1) % kProfileRing;
    ok = ok && ev.fwd_count > 0 && cudaEventElapsedTime(fwd_ms, ev.fwd0[i], ev.fwd1[i]) == cudaSuccess;
  }
  if (bwd_ms) {
    const long long i = (ev.bwd_count - 1) % kProfileRing;
    ok = ok && ev.bwd_count > 0 && cudaEventElapsedTime(bwd_ms, ev.bwd0[i], ev.bwd1[i]) == cudaSuccess;
  }
  return ok;
}

cudaError_t launch_plan(const pp_plan* plan, const int32_t* const* host_desc, cudaStream_t stream,
                        int* launches) {
  PlanPtrs p;
  char* ws = plan->ws;
  const PlanLayout& l = plan->lay;
  p.header = reinterpret_cast<int32_t*>(ws + l.header);
  for (int a = 0; a < 4; ++a) p.src_desc[a] = plan->src_desc[a];
  p.desc_copy = reinterpret_cast<int32_t*>(ws + l.desc);
  p.row_group_off = plan->prob.row_group_off;
  p.grp_prompt_len = plan->prob.grp_prompt_len;
  p.grp_resp_off = plan->prob.grp_resp_off;
  p.resp_len = plan->prob.resp_len;
  p.seg_start = reinterpret_cast<int32_t*>(ws + l.seg_start);
  p.seg_tile0 = reinterpret_cast<int32_t*>(ws + l.seg_tile0);
  p.tiles = reinterpret_cast<Tile*>(ws + l.tiles);
  p.tile_unit = plan->paired ? reinterpret_cast<uint8_t*>(ws + l.tile_unit) : nullptr;
  p.grp_btile0 = reinterpret_cast<int32_t*>(ws + l.grp_btile0);
  p.btiles = reinterpret_cast<BTile*>(ws + l.btiles);
  p.fwd_order = reinterpret_cast<int32_t*>(ws + l.fwd_order);
  p.bwd_order = reinterpret_cast<int32_t*>(ws + l.bwd_order);
  p.tile_gwork = reinterpret_cast<int32_t*>(ws + l.tile_gwork);
  p.tile_block = reinterpret_cast<int32_t*>(ws + l.tile_block);
  p.bwd_units = reinterpret_cast<int32_t*>(ws + l.bwd_units);
  p.sched = bwd_takes_sched(plan->prob);
  p.bwd_units_det = reinterpret_cast<int32_t*>(ws + l.bwd_units_det);
  p.Hkv = plan->prob.num_kv_heads;
  p.key_end = reinterpret_cast<int32_t*>(ws + l.key_end);
  p.qtiles = plan->mixed ? reinterpret_cast<QTile*>(ws + l.qtiles) : nullptr;
  p.qorder = reinterpret_cast<int32_t*>(ws + l.qorder);
  p.work_at = p.bwd_units_det;
  p.grid_gain = reinterpret_cast<long long*>(ws + l.grid_gain);
  p.num_rows = plan->prob.num_rows;
  p.G = plan->prob.num_groups;
  p.N = plan->prob.num_responses;
  p.T = plan->prob.total_tokens;
  p.nseg = plan->nseg;
  p.max_tiles = plan->max_tiles;
  // a third of the SMs (the backward runs one CTA per SM), at most 48 tiles = 6144 tokens
  static DeviceSetup setup[kMaxDevices];
  DeviceSetup* dev = device_setup(setup);
  if (!dev) return cudaErrorInvalidDevice;
  // (a set of the backward is held up with all its parts)
  p.det_asc_max = std::min(48, dev->num_sms / 3) >> plan->lg_split;
  p.sms = dev->num_sms;
  p.pair_cost = plan->prob.head_dim == 64 ? 16 : 14;   // (two heads in a unit: as much)
  p.unit_cost = 10 + p.pair_cost * (plan->prob.num_q_heads / plan->prob.num_kv_heads / 2);

  const int mt = plan->max_tiles;
  // Host descriptors: up to kDescLarge entries travel as a kernel argument, which keeps the call
  // asynchronous (a cudaMemcpyAsync from pageable host memory would first wait on the host for
  // everything already in the stream); longer sets are copied into the workspace.
  const size_t n_desc[4] = {size_t(p.num_rows) + 1, size_t(p.G), size_t(p.G) + 1, size_t(p.N)};
  const size_t n_all = n_desc[0] + n_desc[1] + n_desc[2] + n_desc[3];
  if (mt <= kFusedMaxTiles && p.T <= (1 << 18)) {
    // rows <= G <= N and G + N <= 2048: kDescFused entries always suffice
    cudaError_t e = cudaSuccess;
    if (!dev->configured) {
      auto opt_in = [&](auto kern, size_t bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      };
      auto both = [&](auto n_c) {
        constexpr size_t kN = decltype(n_c)::value;
        opt_in(plan_fused_kernel<kN, false>, sizeof(FusedSmem<false>));
        opt_in(plan_fused_kernel<kN, true>, sizeof(FusedSmem<true>));
      };
      both(std::integral_constant<size_t, 1>{});
      both(std::integral_constant<size_t, kDescSmall>{});
      both(std::integral_constant<size_t, kDescFused>{});
      if (e != cudaSuccess) return e;
      dev->configured = true;
    }
    auto go = [&](auto n_c) {
      constexpr size_t kN = decltype(n_c)::value;
      DescBlock<kN> blk;
      if (host_desc) fill_desc(host_desc, n_desc, blk.v);
      const dim3 threads(mt <= kFusedSmallTiles ? 256 : 1024);
      e = plan->mixed ? launch_kernel(true, plan_fused_kernel<kN, true>, dim3(1), threads,
                                      sizeof(FusedSmem<true>), stream, blk, p)
                      : launch_kernel(true, plan_fused_kernel<kN, false>, dim3(1), threads,
                                      sizeof(FusedSmem<false>), stream, blk, p);
    };
    if (!host_desc) go(std::integral_constant<size_t, 1>{});
    else if (n_all <= kDescSmall) go(std::integral_constant<size_t, kDescSmall>{});
    else go(std::integral_constant<size_t, kDescFused>{});
    if (launches) *launches = 1;
    return e;
  }
  int n_launch = 8;
  if (host_desc) {
    if (n_all <= kDescLarge) {
      DescBlock<kDescLarge> blk;
      fill_desc(host_desc, n_desc, blk.v);
      stage_desc_kernel<kDescLarge><<<1, 256, 0, stream>>>(blk, int(n_all), p.desc_copy);
      ++n_launch;
    } else {
      int32_t* at = p.desc_copy;
      for (int i = 0; i < 4; ++i) {
        cudaError_t e = cudaMemcpyAsync(at, host_desc[i], n_desc[i] * sizeof(int32_t),
                                        cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess) return e;
        at += n_desc[i];
      }
    }
  }
  plan_scan_kernel<<<1, 1024, 0, stream>>>(p);
  plan_tiles_kernel<<<(mt + 255) / 256, 256, 0, stream>>>(p);
  plan_key_end_kernel<<<(p.T + 255) / 256, 256, 0, stream>>>(p);
  plan_btiles_kernel<<<(mt + 255) / 256, 256, 0, stream>>>(p);
  plan_fwd_order_kernel<<<(mt + 127) / 128, 128, 0, stream>>>(p);
  plan_gwork_kernel<<<(mt + 127) / 128, 128, 0, stream>>>(p);
  plan_sgroup_kernel<<<(mt + 127) / 128, 128, 0, stream>>>(p);
  plan_units_kernel<<<(mt + 127) / 128, 128, 0, stream>>>(p);
  if (launches) *launches = n_launch;
  return cudaGetLastError();
}

}  // namespace pp
