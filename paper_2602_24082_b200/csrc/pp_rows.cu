// Row builder: the step before the attention path (paper Sec. 2.2, used with preference
// packing in Sec. 5.2).  Preference groups [prompt | responses] of varying length are ordered by
// total length, longest first with ties in their original order (batch sorting: samples of
// similar length end up together), and consecutive groups of that order are concatenated into
// rows of at most `capacity` tokens (batch packing: next fit).  The outputs are
// the order, the rows, each row's tokens and visible query-key pairs (the attention cost of
// Sec. 3.2.1, for balancing data-parallel ranks) and the descriptor arrays in row order, ready
// for pp_build_plan with descriptors on the device.  Integer work only; microseconds.
#include "pp_internal.h"

namespace pp {
namespace {

enum : int32_t { kRowsOk = 0, kRowsBadGroup = 1, kRowsTooLong = 2 };

struct RowsPtrs {
  int G, N, capacity;
  const int32_t* prompt_len;
  const int32_t* resp_off;
  const int32_t* resp_len;
  int32_t* tok;      // [G] tokens per group, saturated (a group above the capacity is an error)
  long long* cost;   // [G] visible pairs per group
  long long* pre;    // [G] inclusive prefix sums of the sorted groups' tokens
  long long* pre_cost;  // [G] ... and of their visible pairs
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

__device__ __forceinline__ void rows_fail(int32_t* status, int32_t code, int32_t detail) {
  if (atomicCAS(&status[0], kRowsOk, code) == kRowsOk) status[1] = detail;
}

// tokens and visible pairs of every group: P (P + 1) / 2 for the causal prompt, and
// R P + R (R + 1) / 2 for a response that sees the whole prompt and itself causally
__global__ void rows_measure_kernel(RowsPtrs p) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= p.G) return;
  const long long P = p.prompt_len[g];
  const int x0 = p.resp_off[g], x1 = p.resp_off[g + 1];
  if (P < 1 || x1 <= x0 || x0 < 0 || x1 > p.N) {
    rows_fail(p.status, kRowsBadGroup, g);
    p.tok[g] = 0;
    p.cost[g] = 0;
    return;
  }
  long long t = P, u = P * (P + 1) / 2;
  for (int x = x0; x < x1; ++x) {
    const long long R = p.resp_len[x];
    if (R < 1) rows_fail(p.status, kRowsBadGroup, g);
    t += R;
    u += R * P + R * (R + 1) / 2;
  }
  if (t > p.capacity) rows_fail(p.status, kRowsTooLong, g);
  p.tok[g] = int32_t(t < 0x7fffffff ? t : 0x7fffffff);
  p.cost[g] = u;
}

// Position of every key in the order "largest first, ties by index", by rank counting.  The count
// is quadratic, so what matters is to spread it: a block ranks 32 keys, each of its 32 warps
// counts a slice of every staged chunk (all lanes read the same key: broadcast reads), and the
// partial counts are added at the end.  (One thread per key and 256 keys per block left 132 SMs
// idle: 72 us for 4096 groups, now 7.)
constexpr int kRankKeys = 32, kRankSlices = 32, kRankChunk = 2048;

template <typename Key>
__global__ void __launch_bounds__(kRankKeys * kRankSlices)
rank_kernel(int n, const Key* __restrict__ keys, int32_t* __restrict__ order) {
  __shared__ Key s_key[kRankChunk];
  __shared__ int32_t s_count[kRankSlices][kRankKeys];
  const int tid = threadIdx.x, item = tid % kRankKeys, slice = tid / kRankKeys;
  const int first = blockIdx.x * kRankKeys, g = first + item;
  const Key mine = g < n ? keys[g] : 0;
  int count = 0;
  for (int base = 0; base < n; base += kRankChunk) {
    const int here = min(kRankChunk, n - base);
    for (int i = tid; i < here; i += kRankKeys * kRankSlices) s_key[i] = keys[base + i];
    __syncthreads();
    constexpr int kPer = kRankChunk / kRankSlices;
    const int lo = slice * kPer, hi = min(lo + kPer, here);
    if (base + hi <= first) {          // slices before or behind my block's keys: one comparison
#pragma unroll 16
      for (int i = lo; i < hi; ++i) count += s_key[i] >= mine;
    } else if (base + lo >= first + kRankKeys) {
#pragma unroll 16
      for (int i = lo; i < hi; ++i) count += s_key[i] > mine;
    } else {
      for (int i = lo; i < hi; ++i) count += s_key[i] > mine || (s_key[i] == mine && base + i < g);
    }
    __syncthreads();
  }
  s_count[slice][item] = count;
  __syncthreads();
  if (tid < kRankKeys && g < n) {
    int rank = 0;
#pragma unroll
    for (int k = 0; k < kRankSlices; ++k) rank += s_count[k][tid];
    order[rank] = g;
  }
}

// Inclusive block-wide sums of three values per thread (two barriers).
struct Sum3 {
  long long a, b;
  int32_t c;
};
__device__ __forceinline__ Sum3 block_scan(Sum3 v, Sum3* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const long long a = __shfl_up_sync(0xffffffffu, v.a, d), b = __shfl_up_sync(0xffffffffu, v.b, d);
    const int32_t c = __shfl_up_sync(0xffffffffu, v.c, d);
    if (lane >= d) {
      v.a += a;
      v.b += b;
      v.c += c;
    }
  }
  if (lane == 31) s_warp[warp] = v;
  __syncthreads();
  if (warp == 0) {   // the block has 32 warps
    Sum3 w = s_warp[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const long long a = __shfl_up_sync(0xffffffffu, w.a, d), b = __shfl_up_sync(0xffffffffu, w.b, d);
      const int32_t c = __shfl_up_sync(0xffffffffu, w.c, d);
      if (lane >= d) {
        w.a += a;
        w.b += b;
        w.c += c;
      }
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  if (warp) {
    v.a += s_warp[warp - 1].a;
    v.b += s_warp[warp - 1].b;
    v.c += s_warp[warp - 1].c;
  }
  return v;
}

// One block: prefix sums over the sorted groups, next-fit rows, row costs, reordered
// descriptors.  It is all latency, so dependent loads are issued for several groups at once and
// whatever is searched or chased -- the token sums, the pointer-doubling tables -- lives in
// shared memory up to kPackSmemGroups groups (20 bytes each).  4096 groups: 47 us with the tables
// in global memory and shared-memory scans of ten rounds per 1024 groups, now 38.
constexpr int kPackSmemGroups = 8192;

__global__ void __launch_bounds__(1024) rows_pack_kernel(RowsPtrs p, int tables_in_smem) {
  extern __shared__ long long s_tables[];
  __shared__ Sum3 s_warp[32];
  __shared__ Sum3 s_total;
  const int tid = threadIdx.x, nthr = blockDim.x;
  if (p.status[0] != kRowsOk) {
    if (tid == 0) *p.num_rows = 0;
    return;
  }
  long long* pre = tables_in_smem ? s_tables : p.pre;
  int32_t* s_int = reinterpret_cast<int32_t*>(s_tables + p.G);
  int32_t* ja = tables_in_smem ? s_int : p.jump_a;
  int32_t* jb = tables_in_smem ? s_int + p.G : p.jump_b;
  int32_t* mark = tables_in_smem ? s_int + 2 * p.G : p.mark;
  // tokens, pairs and response counts in sorted order
#pragma unroll 4
  for (int i = tid; i < p.G; i += nthr) {
    const int g = p.order[i];
    pre[i] = p.tok[g];
    p.pre_cost[i] = p.cost[g];
    p.out_prompt_len[i] = p.prompt_len[g];
    const int x0 = p.resp_off[g];
    ja[i] = x0;
    jb[i] = p.resp_off[g + 1] - x0;
  }
  // inclusive scans of tokens and pairs and exclusive scan of response counts, in sorted order
  // (every thread scans what it has gathered itself: no barrier in between)
  Sum3 carry = {0, 0, 0};
  for (int base = 0; base < p.G; base += nthr) {
    const int i = base + tid;
    Sum3 v = {0, 0, 0};
    if (i < p.G) v = {pre[i], p.pre_cost[i], jb[i]};
    const int32_t n_resp = v.c;
    const Sum3 w = block_scan(v, s_warp);
    if (i < p.G) {
      pre[i] = carry.a + w.a;
      p.pre_cost[i] = carry.b + w.b;
      p.out_resp_off[i] = carry.c + w.c - n_resp;
    }
    if (tid == nthr - 1) s_total = w;
    __syncthreads();
    carry.a += s_total.a;
    carry.b += s_total.b;
    carry.c += s_total.c;
  }
  if (tid == 0) p.out_resp_off[p.G] = carry.c;
  // the responses' lengths, four loads in flight per thread
  for (int i = tid; i < p.G; i += nthr) {
    const int x0 = ja[i], n = jb[i], y0 = p.out_resp_off[i];
#pragma unroll 4
    for (int x = 0; x < n; ++x) p.out_resp_len[y0 + x] = p.resp_len[x0 + x];
  }
  __syncthreads();
  // Next fit in parallel.  nxt[s] = where the row that starts at sorted position s ends: the
  // largest e whose tokens still fit (every group fits alone, so e > s).  The row starts are
  // the positions reachable from 0 through nxt; they are marked by pointer doubling (after
  // round r every start within 2^r hops is marked), then numbered by a prefix count.
  for (int s = tid; s < p.G; s += nthr) {
    const long long base = s ? pre[s - 1] : 0;
    int lo = s + 1, hi = p.G;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (pre[mid - 1] - base <= p.capacity) lo = mid; else hi = mid - 1;
    }
    p.nxt[s] = lo;
    ja[s] = lo;
    mark[s] = (s == 0);
  }
  for (int hop = 1; hop < p.G; hop <<= 1) {
    __syncthreads();
    for (int s = tid; s < p.G; s += nthr) {
      const int to = ja[s];
      jb[s] = to < p.G ? ja[to] : p.G;
    }
    // (marking runs along with the doubling: a mark set in this round by another thread only
    // marks further positions that are reachable as well)
    for (int s = tid; s < p.G; s += nthr)
      if (mark[s] && ja[s] < p.G) mark[ja[s]] = 1;
    __syncthreads();
    int32_t* t = ja;
    ja = jb;
    jb = t;
  }
  __syncthreads();
  // number the marked positions (exclusive scan of the marks) and emit the rows
  int32_t rows = 0;
  for (int base = 0; base < p.G; base += nthr) {
    const int i = base + tid;
    const int32_t m = i < p.G ? mark[i] : 0;
    const Sum3 w = block_scan({0, 0, m}, s_warp);
    if (m) {
      const int r = rows + w.c - 1, e = p.nxt[i] - 1;
      p.row_group_off[r] = i;
      p.row_tokens[r] = pre[e] - (i ? pre[i - 1] : 0);
      p.row_cost[r] = p.pre_cost[e] - (i ? p.pre_cost[i - 1] : 0);
    }
    if (tid == nthr - 1) s_total = w;
    __syncthreads();
    rows += s_total.c;
  }
  if (tid == 0) {
    p.row_group_off[rows] = p.G;
    *p.num_rows = rows;
  }
}

// ---------------------------------------------------------------- rows -> data-parallel ranks
// Longest-processing-time assignment: rows in order of decreasing cost (ties by index), each to
// the rank with the least cost so far (ties to the lowest rank).  The order comes from rank
// counting over all rows; the greedy pass is sequential by nature and runs in one warp.  What
// bounds it is the chain from one row's assignment to the next one's, so the ranks are kept
// sorted by (load, rank) across the lanes' registers, kPerLane entries each: a step takes the
// first entry, adds the row's cost and inserts it again -- every lane compares its entries with
// the new one and keeps, shifts or replaces them -- so the chain is one broadcast, one add and
// one compare.  Rows are fetched and results written 32 at a time.  (Searching all loads in shared
// memory for the least one with a five-step butterfly took 345 ns a row, now 67 with up to 32 ranks, 98 with 64, 120 with 128.)
constexpr int kMaxAssignRanks = 1024;

template <int kPerLane>
__device__ __forceinline__ void assign_one_by_one(int R, int ranks, const long long* __restrict__ cost,
                                                  const int32_t* __restrict__ order,
                                                  int32_t* __restrict__ rank_of_row,
                                                  long long* __restrict__ rank_cost) {
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
template <int kPerLane>
__global__ void __launch_bounds__(32)
assign_greedy_kernel(int R, int ranks, const long long* __restrict__ cost,
                     const int32_t* __restrict__ order, int32_t* __restrict__ rank_of_row,
                     long long* __restrict__ rank_cost) {
  assign_one_by_one<kPerLane>(R, ranks, cost, order, rank_of_row, rank_cost);
}

// Up to 32 ranks: a round assigns as many rows as the sorted list of ranks allows at once.  Row i of
// the round goes to rank i of the list while that rank is still before all the ranks that have got
// a row in this round -- with loads closer together than a row's cost, as they soon are, that is
// every rank.  Load and rank are one 64-bit word (for sums of costs below 2^58, else one row at a
// time); the list is sorted again by counting, every lane comparing its word with the others', kN at
// most, read from shared memory in one go.  Bound by that chain.
// Building the rows of 4096 groups and dealing the 972 rows out to 8 ranks took 150 us with one row
// at a time, now 126 (122 rounds instead of 972 steps).
constexpr int kBatchRows = 1024, kBatchThreads = 256;
template <int kN>
__global__ void __launch_bounds__(kBatchThreads)
assign_batch_kernel(int R, int ranks, const long long* __restrict__ cost,
                    const int32_t* __restrict__ order, int32_t* __restrict__ rank_of_row,
                    long long* __restrict__ rank_cost) {
  using Key = unsigned long long;
  __shared__ Key s_cost[kBatchRows];
  __shared__ int32_t s_row[kBatchRows];
  __shared__ alignas(16) Key s_key[32];
  __shared__ Key s_sorted[32];
  const int tid = threadIdx.x, lane = tid & 31;
  if (R > 0 && (cost[order[R - 1]] < 0 || cost[order[0]] >= (1LL << 58) / R)) {
    if (tid < 32) assign_one_by_one<1>(R, ranks, cost, order, rank_of_row, rank_cost);
    return;
  }
  Key key = lane < ranks ? Key(lane) : ~Key(0);
  for (int base = 0; base < R; base += kBatchRows) {
    const int m = min(kBatchRows, R - base);
    __syncthreads();
    for (int i = tid; i < m; i += kBatchThreads) {
      s_row[i] = order[base + i];
      s_cost[i] = Key(cost[s_row[i]]) << 5;
    }
    __syncthreads();
    if (tid >= 32) continue;
    auto exchange = [&]() {   // the list sorted again: my place is the number of words before mine
      __syncwarp();
      s_key[lane] = key;
      __syncwarp();
      int before = 0;
#pragma unroll
      for (int i = 0; i < kN; i += 2) {
        const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(&s_key[i]);
        before += int(o.x < key) + int(o.y < key);
      }
      if (lane < ranks) s_sorted[before] = key;
      __syncwarp();
      if (lane < ranks) key = s_sorted[lane];
    };
    Key c = lane < m ? s_cost[lane] : 0;
    for (int pos = 0; pos < m;) {
      const bool there = lane < ranks && pos + lane < m;
      const Key next = key + c, last = __shfl_sync(0xffffffffu, key, ranks - 1);
      int count = ranks;
      // every rank is in time if the last one is before all that have got a row
      if (!__all_sync(0xffffffffu, lane >= ranks || (there && next > last))) {
        __syncwarp();
        s_key[lane] = there ? next : ~Key(0);
        __syncwarp();
        bool in_time = there;
        for (int i = 0; i < ranks - 1; ++i) in_time = in_time && (i >= lane || key < s_key[i]);
        const uint32_t fits = __ballot_sync(0xffffffffu, in_time);
        count = fits == 0xffffffffu ? 32 : __ffs(~fits) - 1;   // (the first row always fits)
      }
      if (lane < count) {
        rank_of_row[s_row[pos + lane]] = int(key & 31u);
        key = next;
      }
      pos += count;
      c = pos + lane < m ? s_cost[pos + lane] : 0;
      exchange();
    }
  }
  if (tid < ranks) rank_cost[key & 31u] = static_cast<long long>(key >> 5);
}

// More ranks than the lanes' registers hold: the loads in shared memory, the lanes sharing the
// search for the least one.
__global__ void __launch_bounds__(32)
assign_greedy_smem_kernel(int R, int ranks, const long long* __restrict__ cost,
                          const int32_t* __restrict__ order, int32_t* __restrict__ rank_of_row,
                          long long* __restrict__ rank_cost) {
  __shared__ long long s_load[kMaxAssignRanks];
  const int lane = threadIdx.x;
  for (int k = lane; k < ranks; k += 32) s_load[k] = 0;
  __syncwarp();
  for (int i = 0; i < R; ++i) {
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
      const int row = order[i];
      rank_of_row[row] = best_k;
      s_load[best_k] = best + cost[row];
    }
    __syncwarp();
  }
  for (int k = lane; k < ranks; k += 32) rank_cost[k] = s_load[k];
}

}  // namespace

cudaError_t launch_assign_rows(int R, const long long* row_cost, int ranks, int32_t* order,
                               int32_t* rank_of_row, long long* rank_cost, cudaStream_t stream,
                               int* launches) {
  rank_kernel<long long><<<(R + kRankKeys - 1) / kRankKeys, kRankKeys * kRankSlices, 0, stream>>>(
      R, row_cost, order);
  auto greedy = ranks <= 8     ? assign_batch_kernel<8>
                : ranks <= 32  ? assign_batch_kernel<32>
                : ranks <= 64  ? assign_greedy_kernel<2>
                : ranks <= 128 ? assign_greedy_kernel<4>
                               : assign_greedy_smem_kernel;
  greedy<<<1, ranks <= 32 ? kBatchThreads : 32, 0, stream>>>(R, ranks, row_cost, order, rank_of_row, rank_cost);
  if (launches) *launches = 2;
  return cudaGetLastError();
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
  p.tok = reinterpret_cast<int32_t*>(w + 3 * a8 + 4 * a4);
  p.order = order;
  p.row_group_off = row_group_off;
  p.num_rows = num_rows;
  p.row_tokens = row_tokens;
  p.row_cost = row_cost;
  p.out_prompt_len = out_prompt_len;
  p.out_resp_off = out_resp_off;
  p.out_resp_len = out_resp_len;
  p.status = status;
  cudaError_t e = cudaMemsetAsync(status, 0, 8, stream);
  if (e != cudaSuccess) return e;
  rows_measure_kernel<<<(G + 255) / 256, 256, 0, stream>>>(p);
  rank_kernel<int32_t><<<(G + kRankKeys - 1) / kRankKeys, kRankKeys * kRankSlices, 0, stream>>>(
      G, p.tok, order);
  // per device: the opt-in to more than 48 KB of dynamic shared memory
  static DeviceSetup setup[kMaxDevices];
  DeviceSetup* dev = device_setup(setup);
  if (!dev) return cudaErrorInvalidDevice;
  if (!dev->configured) {
    e = cudaFuncSetAttribute(rows_pack_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             20 * kPackSmemGroups);
    if (e != cudaSuccess) return e;
    dev->configured = true;
  }
  const bool in_smem = G <= kPackSmemGroups;
  rows_pack_kernel<<<1, 1024, in_smem ? size_t(20) * G : 0, stream>>>(p, in_smem);
  if (launches) *launches = 3;
  return cudaGetLastError();
}

}  // namespace pp
