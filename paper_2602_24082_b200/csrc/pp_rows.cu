// Row builder: the step before the attention path (paper Sec. 2.2, used with preference
// packing in Sec. 5.2).  Preference groups [prompt | responses] of varying length are ordered by
// total length, longest first with ties in their original order (batch sorting: samples of
// similar length end up together), and consecutive groups of that order are concatenated into
// rows of at most `capacity` tokens (batch packing: next fit).  The outputs are
// the order, the rows, each row's tokens and visible query-key pairs (the attention cost of
// Sec. 3.2.1, for balancing data-parallel ranks) and the descriptor arrays in row order, ready
// for pp_build_plan with descriptors on the device.  Integer work only; microseconds.
#include <algorithm>
#include <type_traits>

#include "pp_internal.h"
#include "pp_ptx.cuh"

namespace pp {
namespace {

enum : int32_t { kRowsOk = 0, kRowsBadGroup = 1, kRowsTooLong = 2 };

struct RowsPtrs {
  int G, N, capacity;
  const int32_t* prompt_len;
  const int32_t* resp_off;
  const int32_t* resp_len;
  int2* tok;         // [G] tokens (negative: why the group is refused, kTokBad or kTokTooLong) and responses
                     //   per group; in the space of nxt and jump_a
  long long* cost;   // [G] visible pairs per group
  // in sorted order:
  long long* pre;    // [G] tokens, then (where they do not fit shared memory) their inclusive prefix sums
  long long* pre_cost;  // [G] ... and visible pairs
  int32_t* nxt;      // [G] end of the row that would start at each sorted position
  int32_t* jump_a;   // [G] pointer-doubling buffers, used when they do not fit shared memory
  int32_t* jump_b;   // [G]
  int32_t* mark;     // [G] 1 = a row starts here
  int32_t* order;
  int32_t* row_group_off;
  int32_t* num_rows;
  long long* row_tokens;
  long long* row_cost;
  int32_t* out_prompt_len;
  int32_t* out_resp_off;
  int32_t* out_resp_len;
  int32_t* status;   // [2]: code, detail
};

constexpr int32_t kTokBad = -1, kTokTooLong = -2;

// tokens and visible pairs of every group: P (P + 1) / 2 for the causal prompt, and
// R P + R (R + 1) / 2 for a response that sees the whole prompt and itself causally
__global__ void rows_measure_kernel(RowsPtrs p) {
  launch_dependents();
  dependency_wait();
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= p.G) return;
  const long long P = p.prompt_len[g];
  const int x0 = p.resp_off[g], x1 = p.resp_off[g + 1];
  bool ok = !(P < 1 || x1 <= x0 || x0 < 0 || x1 > p.N);
  long long t = P, u = P * (P + 1) / 2;
  if (ok) {
#pragma unroll 4
    for (int x = x0; x < x1; ++x) {
      const long long R = p.resp_len[x];
      ok = ok && R >= 1;
      t += R;
      u += R * P + R * (R + 1) / 2;
    }
  }
  const int32_t tok = !ok ? kTokBad : t > p.capacity ? kTokTooLong : int32_t(t);
  p.tok[g] = make_int2(tok, tok > 0 ? x1 - x0 : 0);
  p.cost[g] = u;
}

// Position of every key in the order "largest first, ties by index", by rank counting.  The count
// is quadratic, so what matters is to spread it: a block ranks 32 keys, each of its 32 warps
// counts a slice of every staged chunk (all lanes read the same key: broadcast reads), and the
// partial counts are added at the end.  (One thread per key and 256 keys per block left 132 SMs
// idle: 72 us for 4096 groups, now 7.)  For groups the responses before each are counted along, and the
// group goes to its place here, on many SMs: one block that gathered it in sorted order was bound by its
// SM's memory pipe.
constexpr int kRankKeys = 32, kRankSlices = 32, kRankChunk = 2048;
__device__ __forceinline__ long long key_of(long long k) { return k; }
__device__ __forceinline__ int32_t key_of(int2 k) { return k.x; }
// what a key before mine adds: 1, and in the upper half its responses
__device__ __forceinline__ int32_t weight_of(long long) { return 1; }
__device__ __forceinline__ long long weight_of(int2 k) { return static_cast<long long>(k.y) << 32 | 1; }

template <typename Item>
__global__ void __launch_bounds__(kRankKeys * kRankSlices)
rank_kernel(int n, const Item* items, int32_t* order, RowsPtrs p) {
  constexpr bool kGroups = sizeof(Item) == sizeof(int2) && !std::is_same_v<Item, long long>;
  using Key = decltype(key_of(Item{}));
  using Sum = decltype(weight_of(Item{}));
  __shared__ Item s_item[kRankChunk];
  __shared__ Sum s_sum[kRankSlices][kRankKeys];
  __shared__ int3 s_copy[kRankKeys];   // first response, number of them, where they go
  launch_dependents();
  dependency_wait();
  const int tid = threadIdx.x, item = tid % kRankKeys, slice = tid / kRankKeys;
  const int first = blockIdx.x * kRankKeys, g = first + item;
  const bool emits = tid < kRankKeys && g < n;
  const Key mine = g < n ? key_of(items[g]) : Key(0);
  int32_t prompt = 0, x0 = 0, n_resp = 0;
  long long cost = 0;
  if (kGroups && emits) {
    prompt = p.prompt_len[g];
    x0 = p.resp_off[g];
    n_resp = p.tok[g].y;
    cost = p.cost[g];
  }
  Sum sum = 0;
  for (int base = 0; base < n; base += kRankChunk) {
    const int here = min(kRankChunk, n - base);
    for (int i = tid; i < here; i += kRankKeys * kRankSlices) s_item[i] = items[base + i];
    __syncthreads();
    constexpr int kPer = kRankChunk / kRankSlices;
    const int lo = slice * kPer, hi = min(lo + kPer, here);
    if (base + hi <= first) {          // slices before or behind my block's keys: one comparison
#pragma unroll 16
      for (int i = lo; i < hi; ++i) sum += key_of(s_item[i]) >= mine ? weight_of(s_item[i]) : 0;
    } else if (base + lo >= first + kRankKeys) {
#pragma unroll 16
      for (int i = lo; i < hi; ++i) sum += key_of(s_item[i]) > mine ? weight_of(s_item[i]) : 0;
    } else {
      for (int i = lo; i < hi; ++i)
        sum += key_of(s_item[i]) > mine || (key_of(s_item[i]) == mine && base + i < g) ? weight_of(s_item[i]) : 0;
    }
    __syncthreads();
  }
  s_sum[slice][item] = sum;
  if (kGroups && tid < kRankKeys) s_copy[tid] = make_int3(0, 0, 0);
  __syncthreads();
  if (emits) {
    Sum before = 0;
#pragma unroll
    for (int k = 0; k < kRankSlices; ++k) before += s_sum[k][tid];
    const int rank = int(before & 0xffffffff);
    order[rank] = g;
    if constexpr (kGroups) {
      const int y0 = int(before >> 32);
      p.pre[rank] = mine;
      p.pre_cost[rank] = cost;
      p.out_prompt_len[rank] = prompt;
      p.out_resp_off[rank] = y0;
      if (rank == n - 1) p.out_resp_off[n] = y0 + n_resp;
      // (only with a refused group elsewhere can the sum of the others go beyond N)
      s_copy[tid] = make_int3(x0, y0 >= 0 ? max(min(n_resp, p.N - y0), 0) : 0, y0);
    }
  }
  if constexpr (kGroups) {
    __syncthreads();
    const int3 c = s_copy[slice];   // a warp per group
    for (int x = item; x < c.y; x += 32) p.out_resp_len[c.z + x] = p.resp_len[c.x + x];
  }
}

// Inclusive block-wide sums of one or two values per thread of a block of 1024 (two barriers).
template <int kN>
struct Sums {
  long long v[kN];
};
template <int kN>
__device__ __forceinline__ Sums<kN> warp_scan(Sums<kN> s) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
    for (int a = 0; a < kN; ++a) {
      const long long x = __shfl_up_sync(0xffffffffu, s.v[a], d);
      if (lane >= d) s.v[a] += x;
    }
  }
  return s;
}
// `all` receives the block's totals.
template <int kN>
__device__ __forceinline__ Sums<kN> block_scan(Sums<kN> s, Sums<kN>* s_warp, Sums<kN>& all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  s = warp_scan(s);
  __syncthreads();   // (s_warp may still be read from the scan before)
  if (lane == 31) s_warp[warp] = s;
  __syncthreads();
  const Sums<kN> w = warp_scan(s_warp[lane]);   // every warp for itself
#pragma unroll
  for (int a = 0; a < kN; ++a) {
    const long long before = __shfl_sync(0xffffffffu, w.v[a], warp ? warp - 1 : 0);
    if (warp) s.v[a] += before;
    all.v[a] = __shfl_sync(0xffffffffu, w.v[a], 31);
  }
  return s;
}

// One block: prefix sums over the sorted groups, next-fit rows, row costs.  Bound by what one SM's
// shared-memory pipe and barriers allow, so the sums come from kPer consecutive positions per thread, read as
// vectors and scanned once for 1024 kPer of them; searches and jumps take neighbouring positions in
// neighbouring lanes, kPer of them side by side; and up to kPackSmemGroups groups all that is
// searched or chased lives in shared memory (28 bytes each).  4096 groups: 38 us with
// gathers and every phase strided over global memory and scans of 1024, now 18.
constexpr int kPackSmemGroups = 8192;
constexpr size_t pack_smem(int G) { return size_t(16) * ((G + 1) & ~1) + size_t(12) * G; }

template <int kPer, bool kSmem>
__global__ void __launch_bounds__(1024) rows_pack_kernel(RowsPtrs p) {
  extern __shared__ __align__(16) long long s_tables[];
  __shared__ Sums<2> s_warp[32];
  __shared__ Sums<1> s_warp1[32];
  __shared__ int32_t s_bad;
  const int tid = threadIdx.x, G = p.G;
  constexpr int kThreads = 1024, kChunk = kThreads * kPer;
  const int Gp = (G + 1) & ~1;   // (tables begin on 16 bytes)
  long long* pre = kSmem ? s_tables : p.pre;
  long long* pre_cost = kSmem ? s_tables + Gp : p.pre_cost;
  int32_t* s_int = reinterpret_cast<int32_t*>(s_tables + 2 * Gp);
  int32_t* ja = kSmem ? s_int : p.jump_a;
  int32_t* jb = kSmem ? s_int + G : p.jump_b;
  int32_t* mark = kSmem ? s_int + 2 * G : p.mark;
  if (tid == 0) s_bad = 0x7fffffff;
  launch_dependents();
  dependency_wait();
  // (refused groups have negative tokens and stand last)
  if (p.pre[G - 1] < 0) {
    __syncthreads();
    for (int g = tid; g < G; g += kThreads)
      if (p.tok[g].x < 0) atomicMin(&s_bad, g);
    __syncthreads();
    if (tid == 0) {
      p.status[0] = p.tok[s_bad].x == kTokBad ? kRowsBadGroup : kRowsTooLong;
      p.status[1] = s_bad;
      *p.num_rows = 0;
    }
    return;
  }
  // inclusive sums of tokens and pairs
  Sums<2> carry = {};
  for (int base = 0; base < G; base += kChunk) {
    const int i0 = base + tid * kPer;
    long long t[kPer], c[kPer];
    if (kPer > 1 && i0 + kPer <= G) {
#pragma unroll
      for (int k = 0; k < kPer; k += 2) {
        const longlong2 a = *reinterpret_cast<const longlong2*>(p.pre + i0 + k);
        const longlong2 b = *reinterpret_cast<const longlong2*>(p.pre_cost + i0 + k);
        t[k] = a.x;
        t[k + 1] = a.y;
        c[k] = b.x;
        c[k + 1] = b.y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        t[k] = i0 + k < G ? p.pre[i0 + k] : 0;
        c[k] = i0 + k < G ? p.pre_cost[i0 + k] : 0;
      }
    }
#pragma unroll
    for (int k = 1; k < kPer; ++k) {
      t[k] += t[k - 1];
      c[k] += c[k - 1];
    }
    Sums<2> all;
    const Sums<2> w = block_scan<2>({t[kPer - 1], c[kPer - 1]}, s_warp, all);
    const long long t0 = carry.v[0] + w.v[0] - t[kPer - 1], c0 = carry.v[1] + w.v[1] - c[kPer - 1];
    if (kPer > 1 && i0 + kPer <= G) {
#pragma unroll
      for (int k = 0; k < kPer; k += 2) {
        *reinterpret_cast<longlong2*>(pre + i0 + k) = make_longlong2(t0 + t[k], t0 + t[k + 1]);
        *reinterpret_cast<longlong2*>(pre_cost + i0 + k) = make_longlong2(c0 + c[k], c0 + c[k + 1]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (i0 + k < G) {
          pre[i0 + k] = t0 + t[k];
          pre_cost[i0 + k] = c0 + c[k];
        }
    }
    carry.v[0] += all.v[0];
    carry.v[1] += all.v[1];
  }
  __syncthreads();
  // Next fit in parallel.  The row that starts at sorted position s ends at the largest e whose tokens
  // still fit (every group fits alone, so e > s).  The row starts are
  // the positions reachable from 0 that way; they are marked by pointer doubling (after
  // round r every start within 2^r hops is marked), then numbered by a prefix count.
  const int top = 1 << (31 - __clz(G));
  for (int base = 0; base < G; base += kChunk) {
    int at[kPer];
    long long limit[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      at[k] = min(base + tid + kThreads * k, G);
      limit[k] = (at[k] ? pre[at[k] - 1] : 0) + p.capacity;
    }
    for (int w = top; w > 0; w >>= 1) {
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (at[k] + w <= G && pre[at[k] + w - 1] <= limit[k]) at[k] += w;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int s = base + tid + kThreads * k;
      if (s < G) {
        p.nxt[s] = at[k];
        ja[s] = at[k];
        mark[s] = s == 0;
      }
    }
  }
  __syncthreads();
  // (marking runs along with the doubling: a mark set in this round by another thread only
  // marks further positions that are reachable as well; once the doubled hop from 0 has left the
  // list, all are marked)
  for (bool last = false; !last;) {
    last = ja[0] >= G;
#pragma unroll 4
    for (int s = tid; s < G; s += kThreads) {
      const int to = ja[s], m = mark[s];
      jb[s] = to < G ? ja[to] : G;
      if (to < G && m) mark[to] = 1;
    }
    __syncthreads();
    int32_t* t = ja;
    ja = jb;
    jb = t;
  }
  // number the marked positions (exclusive scan of the marks) and emit the rows
  int32_t rows = 0;
  for (int base = 0; base < G; base += kChunk) {
    const int i0 = base + tid * kPer;
    int32_t m[kPer], mine = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      m[k] = i0 + k < G ? mark[i0 + k] : 0;
      mine += m[k];
    }
    Sums<1> all;
    const Sums<1> w = block_scan<1>({mine}, s_warp1, all);
    int r = rows + int(w.v[0]) - mine;
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (m[k]) {
        const int i = i0 + k, e = p.nxt[i] - 1;
        p.row_group_off[r] = i;
        p.row_tokens[r] = pre[e] - (i ? pre[i - 1] : 0);
        p.row_cost[r] = pre_cost[e] - (i ? pre_cost[i - 1] : 0);
        ++r;
      }
    rows += int(all.v[0]);
  }
  if (tid == 0) {
    p.row_group_off[rows] = G;
    *p.num_rows = rows;
    p.status[0] = kRowsOk;
    p.status[1] = 0;
  }
}

// ---------------------------------------------------------------- rows -> data-parallel ranks
// Longest-processing-time assignment: rows in order of decreasing cost (ties by index), each to
// the rank with the least cost so far (ties to the lowest rank).  The order comes from rank
// counting over all rows; the greedy pass is sequential by nature and runs in one block: in rounds
// (assign_batch_kernel below) or, where the sums are too large for those, one row at a time in one warp.  What
// bounds the latter is the chain from one row's assignment to the next one's, so the ranks are kept
// sorted by (load, rank) across the lanes' registers, kPerLane entries each: a step takes the
// first entry, adds the row's cost and inserts it again -- every lane compares its entries with
// the new one and keeps, shifts or replaces them -- so the chain is one broadcast, one add and
// one compare.  Rows are fetched and results written 32 at a time.  (67 ns a row with up to 32 ranks, 98
// with 64, 120 with 128; searching all loads in shared memory for the least one, as beyond 128, 345.)
constexpr int kMaxAssignRanks = 1024;

template <int kPerLane>
__device__ __forceinline__ void assign_one_by_one(int R, int ranks, const long long* cost,
                                                  const int32_t* order,
                                                  int32_t* rank_of_row,
                                                  long long* rank_cost) {
  constexpr long long kInf = 0x7fffffffffffffffLL;
  const int lane = threadIdx.x;
  long long load[kPerLane];
  int id[kPerLane];
#pragma unroll
  for (int j = 0; j < kPerLane; ++j) {   // entry lane * kPerLane + j of the sorted list
    id[j] = lane * kPerLane + j;
    load[j] = id[j] < ranks ? 0 : kInf;
  }
  int row_next = lane < R ? order[lane] : 0;
  long long cost_next = lane < R ? cost[row_next] : 0;
  for (int base = 0; base < R; base += 32) {
    const int row = row_next;
    const long long c_mine = cost_next;
    const int ahead = base + 32 + lane;
    row_next = ahead < R ? order[ahead] : 0;
    cost_next = ahead < R ? cost[row_next] : 0;
    int my_rank = 0;
    const int here = min(32, R - base);
    for (int i = 0; i < here; ++i) {
      const long long v = __shfl_sync(0xffffffffu, load[0], 0) + __shfl_sync(0xffffffffu, c_mine, i);
      const int r = __shfl_sync(0xffffffffu, id[0], 0);
      // the entry behind my last one
      long long up_load = __shfl_down_sync(0xffffffffu, load[0], 1);
      const int up_id = __shfl_down_sync(0xffffffffu, id[0], 1);
      if (lane == 31) up_load = kInf;
      if (lane == i) my_rank = r;
      // before(e): entry e stays in front of the new one
      auto before = [&](long long l, int k) { return l < v || (l == v && k < r); };
      bool mine_before = lane == 0 || before(load[0], id[0]);   // (entry 0 of lane 0 is taken out)
#pragma unroll
      for (int j = 0; j < kPerLane; ++j) {
        const long long nl = j + 1 < kPerLane ? load[j + 1] : up_load;
        const int ni = j + 1 < kPerLane ? id[j + 1] : up_id;
        const bool next_before = before(nl, ni);
        if (next_before) {           // everything up to the next entry moves forward
          load[j] = nl;
          id[j] = ni;
        } else if (mine_before) {    // the new entry belongs here
          load[j] = v;
          id[j] = r;
        }
        mine_before = next_before;
      }
    }
    if (base + lane < R) rank_of_row[row] = my_rank;
  }
#pragma unroll
  for (int j = 0; j < kPerLane; ++j)
    if (id[j] < ranks) rank_cost[id[j]] = load[j];
}
// Up to 128 ranks: a round assigns as many rows as the sorted order of the ranks allows at once.  Row i of
// the round goes to the rank at place i while that rank is still before all the ranks that have got
// a row in this round -- with loads closer together than a row's cost, as they soon are, that is
// every rank.  A thread keeps one rank, whose load and number are one 64-bit word (for sums of costs
// below 2^56, else one row at a time); its place is the number of words before its own, all kN read from shared
// memory side by side.  Bound by that chain, word -> place -> cost -> word.  972 rows to 8 ranks:
// 35 us with the list sorted again every round, now 32; building and dealing out to 64 ranks 177 us with
// one row at a time, now 68.
// Where ranks lie further apart than the rows are long, only the first few are in time: with more than 32 of
// them a round that assigned less than a fifth of its places is followed by a stretch of rows one at a time, first
// kStretchFirst, twice as many each time the round behind it is no better.  Rounds alone -> so: 300 rows, few long
// ones, 33 ranks 98 -> 38 us (one at a time: 50), 3000 that fall by a ninth each, 100 ranks 636 -> 240 (350);
// even costs are as fast as before with up to 64 ranks and 1 to 4 % slower with more.
constexpr int kBatchRows = 1024, kBatchThreads = 256, kStretchFirst = 16, kStretchLast = 128;
// One warp: the next rows one at a time.  `sorted`: the 32 kPerLane words in order, kPerLane to a lane; a row
// takes the first, adds its cost and inserts it again.  The words return to key_of_rank.
template <int kPerLane>
__device__ __noinline__ void one_by_one_sorted(int rows, const unsigned long long* sorted, const unsigned long long* cost,
                                                  const int32_t* row, int32_t* rank_of_row,
                                                  unsigned long long* key_of_rank) {
  constexpr unsigned long long kInf = ~0ull;
  const int lane = threadIdx.x;
  unsigned long long e[kPerLane];
#pragma unroll
  for (int j = 0; j < kPerLane; ++j) e[j] = sorted[lane * kPerLane + j];
  for (int i = 0; i < rows; ++i) {
    const unsigned long long least = __shfl_sync(0xffffffffu, e[0], 0), v = least + cost[i];
    unsigned long long up = __shfl_down_sync(0xffffffffu, e[0], 1);   // the word behind my last one
    if (lane == 31) up = kInf;
    if (lane == 0) rank_of_row[row[i]] = int(least & 127u);
    bool mine_before = lane == 0 || e[0] < v;   // (word 0 of lane 0 is taken out)
#pragma unroll
    for (int j = 0; j < kPerLane; ++j) {
      const unsigned long long next = j + 1 < kPerLane ? e[j + 1] : up;
      const bool next_before = next < v;
      if (next_before) e[j] = next;
      else if (mine_before) e[j] = v;
      mine_before = next_before;
    }
  }
#pragma unroll
  for (int j = 0; j < kPerLane; ++j)
    if (e[j] != kInf) key_of_rank[e[j] & 127u] = e[j];
}

template <int kN>   // ranks at most; a multiple of 32 threads work, one warp without barriers
__global__ void __launch_bounds__(kBatchThreads)
assign_batch_kernel(int R, int ranks, const long long* cost,
                    const int32_t* order, int32_t* rank_of_row,
                    long long* rank_cost) {
  using Key = unsigned long long;
  constexpr int kWork = kN < 32 ? 32 : kN;
  __shared__ Key s_cost[kBatchRows];
  __shared__ int32_t s_row[kBatchRows];
  __shared__ alignas(16) Key s_key[kN];
  __shared__ alignas(16) Key s_next[kN];
  __shared__ int32_t s_count;
  dependency_wait();
  const int tid = threadIdx.x;
  if (R > 0 && (cost[order[R - 1]] < 0 || cost[order[0]] >= (1LL << 56) / R)) {
    if (tid < 32) assign_one_by_one<(kN + 31) / 32>(R, ranks, cost, order, rank_of_row, rank_cost);
    return;
  }
  auto sync = [&]() {
    if constexpr (kWork == 32) __syncwarp(); else named_barrier_sync(1, kWork);
  };
  const bool mine = tid < ranks;
  Key key = mine ? Key(tid) : ~Key(0);
  int count, stretch = 0, stretch_end;   // rows of the last round; rows one at a time, and their end
  for (int base = 0; base < R; base += kBatchRows) {
    const int m = min(kBatchRows, R - base);
    __syncthreads();
    for (int i = tid; i < m; i += kBatchThreads) {
      s_row[i] = order[base + i];
      s_cost[i] = Key(cost[s_row[i]]) << 7;
    }
    __syncthreads();
    if (tid >= kWork) continue;
    count = kN;   // (the last round of a chunk says nothing)
    stretch_end = -1;
    for (int pos = 0; pos < m;) {
      if (tid < kN) s_key[tid] = key;
      if (tid == 0) s_count = min(ranks, m - pos);
      sync();
      int place = 0;
#pragma unroll 16
      for (int i = 0; i < kN; i += 2) {
        const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(&s_key[i]);
        place += int(o.x < key) + int(o.y < key);
      }
      if constexpr (kN > 32) {
        if (count < kN / 5) {
          stretch = pos - count == stretch_end ? min(2 * stretch, kStretchLast) : kStretchFirst;
          count = kN;
          s_next[mine ? place : tid] = key;
          sync();
          const int rows = min(stretch, m - pos);
          if (tid < 32) one_by_one_sorted<kN / 32>(rows, s_next, s_cost + pos, s_row + pos, rank_of_row, s_key);
          sync();
          if (mine) key = s_key[tid];
          pos += rows;
          stretch_end = pos;
          sync();
          continue;
        }
      }
      const bool there = mine && pos + place < m;
      const Key next = there ? key + s_cost[pos + place] : key;
      // every rank is in time if all that get a row end up behind the last one
      bool all_in_time = false;
      if constexpr (kWork == 32) {
        const int last = __ffs(__ballot_sync(0xffffffffu, mine && place == ranks - 1)) - 1;
        const Key last_key = __shfl_sync(0xffffffffu, key, last);
        all_in_time = __all_sync(0xffffffffu, !there || next > last_key);
      }
      count = min(ranks, m - pos);
      if (!all_in_time) {
        if (mine) s_next[place] = there ? next : ~Key(0);
        sync();
        Key least = ~Key(0);   // of the ranks that get a row before this one
#pragma unroll 16
        for (int i = 0; i < kN; i += 2) {
          const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(&s_next[i]);
          if (i < place && o.x < least) least = o.x;
          if (i + 1 < place && o.y < least) least = o.y;
        }
        if (there && key > least) atomicMin(&s_count, place);
        sync();
        count = s_count;
      }
      if (there && place < count) {
        rank_of_row[s_row[pos + place]] = tid;
        key = next;
      }
      pos += count;
      sync();
    }
  }
  if (mine) rank_cost[tid] = static_cast<long long>(key >> 7);
}

// One rank: all rows and their sum.
__global__ void __launch_bounds__(1024)
assign_single_kernel(int R, const long long* cost, int32_t* rank_of_row,
                     long long* rank_cost) {
  __shared__ unsigned long long s_sum;
  if (threadIdx.x == 0) s_sum = 0;
  dependency_wait();
  __syncthreads();
  unsigned long long sum = 0;
  for (int i = threadIdx.x; i < R; i += blockDim.x) {
    sum += static_cast<unsigned long long>(cost[i]);
    rank_of_row[i] = 0;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, sum);
  __syncthreads();
  if (threadIdx.x == 0) *rank_cost = static_cast<long long>(s_sum);
}

// More ranks than the lanes' registers hold: the loads in shared memory, the lanes sharing the
// search for the least one.
__global__ void __launch_bounds__(32)
assign_greedy_smem_kernel(int R, int ranks, const long long* cost,
                          const int32_t* order, int32_t* rank_of_row,
                          long long* rank_cost) {
  __shared__ long long s_load[kMaxAssignRanks];
  dependency_wait();
  const int lane = threadIdx.x;
  for (int k = lane; k < ranks; k += 32) s_load[k] = 0;
  __syncwarp();
  // (fetched ahead: the loads may not pass the stores of the row before; 3000 rows, 129 ranks 1264 -> 1115 us)
  int row = order[0], row_next = R > 1 ? order[1] : 0;
  long long c = cost[row];
  for (int i = 0; i < R; ++i) {
    const long long c_next = i + 1 < R ? cost[row_next] : 0;
    const int row_after = i + 2 < R ? order[i + 2] : 0;
    long long best = 0x7fffffffffffffffLL;
    int best_k = ranks;
    for (int k = lane; k < ranks; k += 32) {   // ascending k: the first minimum is kept
      const long long l = s_load[k];
      if (l < best) {
        best = l;
        best_k = k;
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, best, d);
      const int ok = __shfl_xor_sync(0xffffffffu, best_k, d);
      if (ob < best || (ob == best && ok < best_k)) {
        best = ob;
        best_k = ok;
      }
    }
    if (lane == 0) {
      rank_of_row[row] = best_k;
      s_load[best_k] = best + c;
    }
    row = row_next;
    row_next = row_after;
    c = c_next;
    __syncwarp();
  }
  for (int k = lane; k < ranks; k += 32) rank_cost[k] = s_load[k];
}

}  // namespace

cudaError_t launch_assign_rows(int R, const long long* row_cost, int ranks, int32_t* order,
                               int32_t* rank_of_row, long long* rank_cost, cudaStream_t stream,
                               int* launches) {
  const unsigned blocks = unsigned((R + kRankKeys - 1) / kRankKeys);
  cudaError_t e = launch_kernel(true, rank_kernel<long long>, dim3(blocks), dim3(kRankKeys * kRankSlices), 0,
                                stream, R, row_cost, order, RowsPtrs{});
  if (e != cudaSuccess) return e;
  if (ranks == 1) {
    e = launch_kernel(true, assign_single_kernel, dim3(1), dim3(1024), 0, stream, R, row_cost, rank_of_row, rank_cost);
  } else {
    auto greedy = ranks <= 8     ? assign_batch_kernel<8>
                  : ranks <= 32  ? assign_batch_kernel<32>
                  : ranks <= 64  ? assign_batch_kernel<64>
                  : ranks <= 128 ? assign_batch_kernel<128>
                                 : assign_greedy_smem_kernel;
    e = launch_kernel(true, greedy, dim3(1), dim3(ranks <= 128 ? kBatchThreads : 32), 0, stream, R, ranks, row_cost,
                      order, rank_of_row, rank_cost);
  }
  if (launches) *launches = 2;
  return e;
}

size_t rows_workspace_bytes(int G) {
  return align_up(size_t(8) * G, 256) * 3 + align_up(size_t(4) * G, 256) * 5;
}

cudaError_t launch_build_rows(int G, int N, const int32_t* prompt_len, const int32_t* resp_off,
                              const int32_t* resp_len, int capacity, void* ws, int32_t* order,
                              int32_t* row_group_off, int32_t* num_rows, long long* row_tokens,
                              long long* row_cost, int32_t* out_prompt_len, int32_t* out_resp_off,
                              int32_t* out_resp_len, int32_t* status, cudaStream_t stream,
                              int* launches) {
  RowsPtrs p;
  p.G = G;
  p.N = N;
  p.capacity = capacity;
  p.prompt_len = prompt_len;
  p.resp_off = resp_off;
  p.resp_len = resp_len;
  char* w = static_cast<char*>(ws);
  const size_t a8 = align_up(size_t(8) * G, 256);
  p.cost = reinterpret_cast<long long*>(w);
  p.pre = reinterpret_cast<long long*>(w + a8);
  p.pre_cost = reinterpret_cast<long long*>(w + 2 * a8);
  const size_t a4 = align_up(size_t(4) * G, 256);
  p.nxt = reinterpret_cast<int32_t*>(w + 3 * a8);
  p.jump_a = reinterpret_cast<int32_t*>(w + 3 * a8 + a4);
  p.jump_b = reinterpret_cast<int32_t*>(w + 3 * a8 + 2 * a4);
  p.mark = reinterpret_cast<int32_t*>(w + 3 * a8 + 3 * a4);
  p.tok = reinterpret_cast<int2*>(w + 3 * a8);
  p.order = order;
  p.row_group_off = row_group_off;
  p.num_rows = num_rows;
  p.row_tokens = row_tokens;
  p.row_cost = row_cost;
  p.out_prompt_len = out_prompt_len;
  p.out_resp_off = out_resp_off;
  p.out_resp_len = out_resp_len;
  p.status = status;
  // per device: the opt-in to more than 48 KB of dynamic shared memory
  static DeviceSetup setup[kMaxDevices];
  DeviceSetup* dev = device_setup(setup);
  if (!dev) return cudaErrorInvalidDevice;
  cudaError_t e = cudaSuccess;
  if (!dev->configured) {
    for (auto kern : {rows_pack_kernel<1, true>, rows_pack_kernel<2, true>, rows_pack_kernel<4, true>,
                      rows_pack_kernel<8, true>}) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(pack_smem(kPackSmemGroups)));
      if (e != cudaSuccess) return e;
    }
    dev->configured = true;
  }
  e = launch_kernel(true, rows_measure_kernel, dim3((G + 255) / 256), dim3(256), 0, stream, p);
  if (e == cudaSuccess)
    e = launch_kernel(true, rank_kernel<int2>, dim3((G + kRankKeys - 1) / kRankKeys),
                      dim3(kRankKeys * kRankSlices), 0, stream, G, p.tok, order, p);
  auto pack = G <= 1024            ? rows_pack_kernel<1, true>
              : G <= 2048            ? rows_pack_kernel<2, true>
              : G <= 4096            ? rows_pack_kernel<4, true>
              : G <= kPackSmemGroups ? rows_pack_kernel<8, true>
                                     : rows_pack_kernel<8, false>;
  if (e == cudaSuccess)
    e = launch_kernel(true, pack, dim3(1), dim3(1024), G <= kPackSmemGroups ? pack_smem(G) : 0, stream, p);
  if (launches) *launches = 3;
  return e;
}

}  // namespace pp
