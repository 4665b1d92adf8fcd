// Backward kernels: dQ, dK, dV of preference-packed attention.
//
//   preprocess : Delta_i = sum_d dO_id O_id and LSE * log2(e), per (query head, token)
//   main       : one CTA per (key tile, KV head).  K and V stay in shared memory; dK and dV
//                stay in tensor memory while the CTA walks over every query tile that sees
//                the key tile -- its own diagonal tile, then the contiguous range of later
//                queries (for prompt keys: the rest of the prompt and every response) -- and
//                over the query heads sharing the KV head.  So the prompt keys' gradients
//                gather all responses' contributions inside one accumulator, with no atomics.
//                Per query tile: S^T = K Q^T and dP^T = V dO^T (tensor memory), P^T =
//                exp2(S^T - LSE), dS^T = P^T (dP^T - Delta) in registers (thread = key row),
//                dV += P^T dO, dK += dS^T Q, dQ_tile = dS K.  Only dQ leaves the CTA per tile:
//                it is added into an fp32 accumulator with TMA reductions.
//   finalize   : dQ = bf16(scale * accumulator)
#include <algorithm>
#include <mutex>

#include <type_traits>

#include "pp_dev.cuh"

namespace pp {
namespace {

struct BwdParams {
  int32_t* header;
  const BTile* tiles;       // the backward's key tiles (cut per group)
  const int32_t* order;
  const int32_t* key_end;   // [T] first query that cannot see key j
  const float* delta;  // [Hq][T]
  const float* lse2;   // [Hq][T]  LSE * log2(e)
  float* dq_acc;       // [T][Hq][D] fp32
  int32_t* dq_sem;     // deterministic variant: turn counters [backward tile][Hq][4 row quarters]; else null
  __nv_bfloat16* dk;
  __nv_bfloat16* dv;
  int T, Hq, Hkv;
  float scale, scale_log2;
  // where units are cut into parts
  float4* parts;       // dV, dK of the parts [part][2][D / 4][128 rows]
  int lg_split;        // log2 of the parts per unit
};

// ---------------------------------------------------------------- preprocess
// Delta = sum_d dO * O per (token, query head) row, the LSE in base-2 units, and the row of
// the fp32 dQ accumulator cleared (so no separate memset pass over it is needed) unless the
// forward has already cleared it (kClear = false).  A pure stream over O and dO, bound by
// memory: D / 8 lanes per row with 16-byte loads, kUnroll rows per lane group in flight.  A warp
// takes kUnroll * kRows consecutive tokens of one head, so that the statistics [Hq][T] leave as
// one store of consecutive words; the block index runs over the heads fastest, so that the blocks
// running at the same time read whole tokens of [T][Hq][D].  Without the clearing the
// tokens go from the last to the first, so that the end of O that the forward left in L2 is read
// before it is evicted, and O, not read again in the step, is marked evict-first: in a step, 33.8
// -> 27.6 us at T = 9241, Hq = 32, D = 128 (151 MB, part of it from L2), 101 -> 92 at T = 16384,
// Hq = 64 (with the clearing, beyond 640 MB, either cost 2 %).  No row index is divided: a version
// that derived (token, head) from a 64-bit row number, two divisions per row and lane, took 40 us
// where this takes 30 (T = 9241, Hq = 32, D = 128: 151 MB), 129 against 92 at T = 16384, Hq = 64,
// and with the clearing 488 against 330 at T = 65536, Hq = 32 (2.1 GB, 6.5 TB/s).
// lanes that share a row: D / 8 (16 bytes of bf16 per lane), rounded up to a power of two
__host__ __device__ constexpr int pre_lanes(int d) { return d == 96 ? 16 : d / 8; }
constexpr int kPreUnroll = 4, kPreWarps = 8;
// tokens per block
__host__ __device__ constexpr int pre_tokens(int d) { return kPreWarps * kPreUnroll * (32 / pre_lanes(d)); }

template <int D, bool kClear>
__global__ void __launch_bounds__(32 * kPreWarps)
bwd_preprocess_kernel(const __nv_bfloat16* o, const __nv_bfloat16* d_o,
                      const float* lse, float* delta,
                      float* lse2, float* dq_acc, int T, int Hq, int4* sem, unsigned sem_n4) {
  launch_dependents();
  dependency_wait();
  constexpr int kLanes = pre_lanes(D);    // lanes per row (D / 8 of them hold data)
  constexpr int kRows = 32 / kLanes;      // rows per warp and step
  const int lane = threadIdx.x & 31, sub = lane % kLanes, rin = lane / kLanes;
  const int block = int(kClear ? blockIdx.x : gridDim.x - 1 - blockIdx.x), chunk = block / Hq, h = block - chunk * Hq;
  const int t0 = chunk * pre_tokens(D) + (threadIdx.x >> 5) * (kPreUnroll * kRows);
  // lane (rin, sub = u) writes the statistics of token t0 + u * kRows + rin
  const int t_stat = t0 + sub * kRows + rin;
  const bool writes = sub < kPreUnroll && t_stat < T;
  const size_t stat = size_t(h) * T + t_stat;
  const float my_lse = writes ? lse[stat] : 0.f;
  const size_t row0 = (size_t(t0 + rin) * Hq + h) * D + sub * 8, step = size_t(kRows) * Hq * D;
  uint4 a[kPreUnroll], b[kPreUnroll];
#pragma unroll
  for (int u = 0; u < kPreUnroll; ++u) {
    a[u] = b[u] = make_uint4(0u, 0u, 0u, 0u);
    if (t0 + u * kRows + rin < T && sub < D / 8) {
      const uint4* po = reinterpret_cast<const uint4*>(o + row0 + u * step);
      a[u] = kClear ? *po : __ldcs(po);
      b[u] = *reinterpret_cast<const uint4*>(d_o + row0 + u * step);
    }
  }
  float mine = 0.f;
#pragma unroll
  for (int u = 0; u < kPreUnroll; ++u) {
    const uint32_t aw[4] = {a[u].x, a[u].y, a[u].z, a[u].w}, bw[4] = {b[u].x, b[u].y, b[u].z, b[u].w};
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[i]));
      const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[i]));
      acc = fmaf(x.x, y.x, fmaf(x.y, y.y, acc));
    }
#pragma unroll
    for (int sft = kLanes / 2; sft > 0; sft >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, sft);
    if (sub == u) mine = acc;
    if (kClear && t0 + u * kRows + rin < T && sub < D / 8) {
      float4* z = reinterpret_cast<float4*>(dq_acc + row0 + u * step);
      z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
      z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < sem_n4; i += gridDim.x * blockDim.x)
    sem[i] = make_int4(0, 0, 0, 0);   // turn counters (deterministic variant)
  if (writes) {
    delta[stat] = mine;
    lse2[stat] = my_lse * 1.4426950408889634f;
  }
}

// ---------------------------------------------------------------- finalize
// dQ = bf16(scale * accumulator) in the first `dq_blocks` blocks: a stream bound by memory, four
// 16-byte loads per thread in flight and, as neither side is read again here, both marked
// evict-first, which leaves more of the accumulator's tail from the backward in L2.  T = 9241,
// Hq = 32, D = 128 (227 MB): 44 us with one load per thread and a grid-stride loop, 38 / 33 with
// 2 / 4 loads, 30 with the hints (7.5 TB/s, part of it from L2); T = 16384, Hq = 64: 154 -> 116.
// Where units are cut into parts, the blocks behind these add up the parts of a (backward tile, KV
// head), 32 rows of dV or dK each, with the loads of four or eight parts in flight (fin_parts).
constexpr int kFinUnroll = 4;
// Eight parts in flight shorten the sums, but take 78 registers instead of 40, which the whole stream pays
// for: eight only where there are as many and the stream is about one wave of such blocks.
// Whole steps, four -> eight: 251 tokens, 8 / 1 heads 33.9 -> 33.2 us, 1556 69.5 -> 68.7; backward with
// preprocess and finalize, eight everywhere -> this rule: 14381 tokens, 14 / 2, D 96 212 -> 208, 5000, 28 / 4
// 452 -> 448.
inline int fin_parts(int lg_split, unsigned dq_blocks, int num_sms) {
  return lg_split == 0 ? 0 : lg_split == 3 && dq_blocks <= 4u * num_sms ? 8 : 4;
}
struct SumParts {
  const float4* parts;
  const int32_t* header;
  const BTile* tiles;
  __nv_bfloat16* dk;
  __nv_bfloat16* dv;
  int lg_split, Hkv, D;
};

template <int kParts>   // (0: an instance of its own, the stream alone needs 26 registers)
__global__ void __launch_bounds__(256)
bwd_finalize_kernel(const float4* acc, uint2* dq, size_t n4, float scale,
                    unsigned dq_blocks, SumParts sp) {
  launch_dependents();
  dependency_wait();
  if (!kParts || blockIdx.x < dq_blocks) {
    const size_t i0 = size_t(blockIdx.x) * (256 * kFinUnroll) + threadIdx.x;
    float4 a[kFinUnroll];
#pragma unroll
    for (int u = 0; u < kFinUnroll; ++u)
      if (i0 + u * 256 < n4) a[u] = __ldcs(acc + i0 + u * 256);
#pragma unroll
    for (int u = 0; u < kFinUnroll; ++u)
      if (i0 + u * 256 < n4) {
        uint2 w;
        w.x = pack_bf16(a[u].x * scale, a[u].y * scale);
        w.y = pack_bf16(a[u].z * scale, a[u].w * scale);
        __stcs(dq + i0 + u * 256, w);
      }
    return;
  }
  __shared__ uint2 s_out[32][33];
  const int b = int(blockIdx.x - dq_blocks), quarter = b & 3, which = (b >> 2) & 1, unit = b >> 3;
  const int tidx = unit / sp.Hkv, kvh = unit - tidx * sp.Hkv;
  if (sp.header[0] != kStatusOk || tidx >= sp.header[kHdrNumBTiles]) return;
  const BTile tile = sp.tiles[tidx];
  const int rows = min(32, tile.len - 32 * quarter), c4s = sp.D / 4;
  if (rows <= 0) return;
  const int lane = threadIdx.x & 31;
  const float f = which ? scale : 1.f;
  for (int c = threadIdx.x >> 5; c < c4s; c += 8) {
    const float4* src = sp.parts + ((size_t(unit) << sp.lg_split) * 2 + which) * (c4s * kTile) +
                        c * kTile + 32 * quarter + lane;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    constexpr int kIn = kParts ? kParts : 1;
#pragma unroll 1
    for (int first = 0; first < (1 << sp.lg_split); first += kIn) {
      float4 x[kIn];
#pragma unroll
      for (int p = 0; p < kIn; ++p)
        if (first + p < (1 << sp.lg_split)) x[p] = src[size_t(first + p) * 2 * c4s * kTile];
#pragma unroll
      for (int p = 0; p < kIn; ++p)
        if (first + p < (1 << sp.lg_split)) {
          s.x += x[p].x;
          s.y += x[p].y;
          s.z += x[p].z;
          s.w += x[p].w;
        }
    }
    s_out[lane][c] = make_uint2(pack_bf16(s.x * f, s.y * f), pack_bf16(s.z * f, s.w * f));
  }
  __syncthreads();
  __nv_bfloat16* out = which ? sp.dk : sp.dv;
  for (int i = threadIdx.x; i < rows * c4s; i += blockDim.x) {
    const int r = i / c4s, c = i - r * c4s;
    *reinterpret_cast<uint2*>(out + ((size_t(tile.start) + 32 * quarter + r) * sp.Hkv + kvh) * sp.D + 4 * c) =
        s_out[r][c];
  }
}

// ---------------------------------------------------------------- main
// Persistent, warp-specialised CTA (one per SM), 512 threads in four warpgroups:
//   warp 0       producer: K, V once per unit; per query tile Q and dO by TMA (two-stage rings)
//                and the tile's LSE*log2(e) / Delta into shared memory
//   warp 1       MMA issuer (one thread); warps 2, 3 idle
//   warps 4-7    compute warpgroup 0: thread = key row, query columns 0..63 of the tile
//   warps 8-11   compute warpgroup 1: query columns 64..127
//   warps 12-15  dQ warpgroup: thread = query row; takes each dQ tile out of tensor memory as a
//                whole and adds it to the fp32 accumulator, every warp its own 32 rows through its
//                own two swizzled staging boxes with TMA reduce-adds (whole 128-byte lines per
//                row instead of per-thread 16-byte reductions, which saturate the L2 atomic units)
// What bounds it (two rows of 32768 tokens, Hq / Hkv 32 / 8, D 128; cycles per query tile and
// head): 2560 of MMAs; 3100 - 3400 with every load and reduction taken out, the MMA thread's own
// waits; 3850 as it is, because an iteration moves 64 KB of Q and dO and 64 KB of reductions
// between the SM and L2.  Before, at 4070, the thread waited for two chains on top: dQ drained in
// two halves with the staging of the first in between (1015 cycles to 200 now that 152 registers
// hold the tile), and dS (1350 to 1000: P kept in fp32 registers instead of unpacked from bf16, no
// selects on full tiles, the next columns loaded under the arithmetic of these).  The kernel went
// from 26.9 to 25.8 M cycles there, 2.64 to 2.49 on four 4800-token groups (28 / 4 heads), 2.13 to
// 2.01 on sixteen thousand tokens (64 / 8 heads), 757 to 726 thousand at D 64.
// Tensor-memory map (columns): [0,128) S^T, overwritten by P^T (bf16: columns [0,32) and
// [64,96), each warpgroup inside the columns it has read itself); [128,256) dP^T, then the
// dQ tile; [256,256+D) dV; [384,384+D) dK.
// MMA order per query tile i:  dP(i)  dV(i)  S(i+1)  dQ(i)  dK(i).  The exponentials of tile
// i+1 run under dQ(i), dK(i), dP(i+1); dS(i) is computed under dV(i), S(i+1); the dQ tile is
// drained under dK(i), so the dP/dQ columns are free again when dP(i+1) is issued.
constexpr int kBwdThreads = 512;
// Registers per thread behind the split: warpgroup 0 (producer, MMA issuer), 1 and 2 (compute), 3
// (dQ).  They have to add up to what the launch allocates.
constexpr int kBwdRegsLaunch = 65536 / kBwdThreads;  // 128
constexpr int kBwdRegsIssue = 104, kBwdRegsCompute = 128, kBwdRegsDq = 152;
static_assert(kBwdRegsIssue + 2 * kBwdRegsCompute + kBwdRegsDq == 4 * kBwdRegsLaunch, "register split");
constexpr uint32_t kBwdTmemCols = 512;

enum BwdBar : int {
  kKvFull = 0,
  kKvEmpty,
  kQFullB,       // [2]   33 arrivals: TMA transaction + 32 producer lanes (LSE / Delta)
  kQEmptyB = 4,  // [2]
  kDoFull = 6,   // dO is single-buffered: free after dV(i), needed again at dP(i+1)
  kDoEmpty = 8,
  kSFullB = 10,
  kPReady,       // 8: one arrival per compute warp
  kDpFull,
  kDsReady,      // 8
  kDqFull,
  kDqDrained,    // 4: one arrival per dQ warp
  kDkvFull,
  kDkvFree,      // 8
  kSchedFull,    // [2]  unit ids handed from the producer warp to the other roles
  kSchedEmpty = kSchedFull + 2,  // [2]  13 arrivals: MMA thread + 8 compute warps + 4 dQ warps
  kNumBwdBars = kSchedEmpty + 2
};

template <int D>
struct BwdSmem {
  static constexpr int kTileBytes = 128 * D * 2;
  static constexpr int kStageBytes = 32 * 128;  // one {32 floats x 32 rows} box of a dQ tile; two per dQ warp
  static constexpr int kK = 0, kV = kTileBytes, kQ = 2 * kTileBytes, kdO = 4 * kTileBytes,
                       kStg = 5 * kTileBytes, kdS = kStg + 8 * kStageBytes,
                       kStats = kdS + 128 * 128 * 2, kBars = kStats + 2 * 256 * 4;
  static constexpr int kUsed = kBars + 8 * kNumBwdBars + 32;
  // The declared 1024-byte alignment of the dynamic shared memory leaves no slack to spend at
  // D = 128 (227 KB limit); the kernel checks the base and reports if it is not aligned.
  static constexpr int kTotal = kUsed + (kUsed + 1024 <= 232448 ? 1024 : 0);
};

struct BwdUnit {
  BTile tile;
  int kvh, nq, n_it, tidx;
  int part, h0, nh;   // part of the unit: query heads [h0, h0 + nh) of the KV head
};

// Units are handed out dynamically: the producer warp draws the next index of the plan's
// longest-work-first order from a global counter whenever the CTA is ready for more (list
// scheduling), and passes its entry to the other roles through a two-entry shared-memory ring.
// header[5] is that counter, header[7] counts finished CTAs; the last one resets both, so a
// plan can be used by any number of launches without a memset in between.
constexpr int kHdrBwdNext = 5, kHdrBwdDone = 7;

// `packed` = (kv head << 24) | backward tile, negative at the end of the work list; with units cut
// into parts also (part << kPartShift).  (kSplit is a template parameter all the way down: with the
// parts' heads worked out at run time, steps whose units stay whole lost 1 - 4 % to other code
// around the issue loops.)
template <bool kSplit>
__device__ __forceinline__ bool get_bwd_unit(const BwdParams& prm, int packed, BwdUnit& un) {
  if (packed < 0) return false;
  un.kvh = packed >> 24;
  un.tidx = packed & (kSplit ? (1 << kPartShift) - 1 : 0xffffff);
  un.tile = prm.tiles[un.tidx];
  un.nq = un.tile.work;
  if (kSplit) {
    const int heads = prm.Hq / prm.Hkv;
    un.part = (packed >> kPartShift) & ((1 << (24 - kPartShift)) - 1);
    un.h0 = (heads * un.part) >> prm.lg_split;
    un.nh = ((heads * (un.part + 1)) >> prm.lg_split) - un.h0;
    un.h0 += un.kvh * heads;
    un.n_it = un.nq * un.nh;
  } else {
    un.n_it = un.nq * (prm.Hq / prm.Hkv);
  }
  return true;
}
// query heads the (part of the) unit walks
template <bool kSplit>
__device__ __forceinline__ int unit_heads(const BwdParams& prm, const BwdUnit& un) {
  return kSplit ? un.nh : prm.Hq / prm.Hkv;
}

// Query tile qt of a unit: tile qt of the group's 128-token grid counted from the key tile
// itself.  Key j of the unit sees query i iff j <= i < key_end[j].
struct QTile {
  int h, start, len;
};

// (query tile, head) position inside a unit, advanced without divisions: the query tiles from the
// key tile itself upwards and for each query tile all query heads of the KV head -- or, from
// kChunkedHeads heads on, kHeadChunk heads at a time, walking the query tiles once per chunk.
// The key tiles of a group, in different CTAs, walk the same (query tile, head) sequence one query
// tile apart, so a Q / dO tile and its dQ accumulator are wanted again after one query tile's
// worth of iterations; 148 CTAs move 128 KB each per iteration, 150 MB in eight, and by then they
// have left L2.  Chunks of two against all heads: 3740 instead of 3880 thousand cycles on three
// 6000-token groups with eight heads per KV head, 858 instead of 911 on 800-token groups, 611
// instead of 676 with seven heads on 2000-token groups, 1992 instead of 2088 on two rows of 8192
// tokens with eight; four heads and fewer were within 2 % either way.
// In the deterministic variant the turns need all heads of a query tile before the next one.
constexpr int kChunkedHeads = 6, kHeadChunk = 2;
struct QIter {
  int hh = 0, qt = 0, h0 = 0;
};
template <bool kDet>
__device__ __forceinline__ void q_advance(QIter& s, int heads, int nq) {
  const int h1 = kDet || heads < kChunkedHeads ? heads : min(s.h0 + kHeadChunk, heads);
  if (++s.hh == h1) {
    s.hh = s.h0;
    ++s.qt;
    if (!kDet && s.qt == nq) {
      s.qt = 0;
      s.hh = s.h0 = h1;
    }
  }
}
template <bool kSplit>
__device__ __forceinline__ QTile q_tile_at(const BwdParams& prm, const BwdUnit& un, const QIter& s) {
  QTile q;
  q.h = kSplit ? un.h0 + s.hh : un.kvh * (prm.Hq / prm.Hkv) + s.hh;
  q.start = un.tile.start + s.qt * kTile;
  q.len = min(kTile, un.tile.grp_end - q.start);
  return q;
}

// D: head dimension of the shared-memory tiles; DV <= D: head dimension of the tensors in
// global memory (96 in tiles of 128: the TMA loads zero-fill the columns past DV, so only the
// loops over the head dimension, the N of dV / dK / dQ and global addressing know about DV).
template <int D, bool kDet, bool kSplit, int DV = D>
__global__ void __launch_bounds__(kBwdThreads, 1)
bwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
           const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
           const __grid_constant__ CUtensorMap tm_dq, BwdParams prm) {
  using L = BwdSmem<D>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (known to be uniform in the warp)

#ifdef PP_DEBUG_COUNTERS
  const long long t_kernel0 = clock64();
#endif

  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  if (base - raw + L::kUsed > L::kTotal) {  // cannot happen with an aligned base
    dependency_wait();
    if (tid == 0 && atomicCAS(&prm.header[0], kStatusOk, kStatusWaitExpired) == kStatusOk)
      prm.header[1] = 99;
    return;
  }
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t sK = base + L::kK, sV = base + L::kV, sQ = base + L::kQ, sdO = base + L::kdO,
                 sdS = base + L::kdS;
  float* stats = reinterpret_cast<float*>(gbase + L::kStats);  // [stage][lse2 128 | delta 128]
  const uint32_t bars = base + L::kBars;
  auto bar = [&](int i) { return bars + 8u * uint32_t(i); };
  const uint32_t tmem_slot = bars + 8 * kNumBwdBars;
  volatile uint32_t* tmem_slot_p = reinterpret_cast<volatile uint32_t*>(gbase + L::kBars + 8 * kNumBwdBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kBars + 8 * kNumBwdBars + 8);

  if (tid == 0) {
    for (int i = 0; i < kNumBwdBars; ++i) {
      uint32_t cnt = 1;
      if (i == kQFullB || i == kQFullB + 1) cnt = 33;
      if (i == kPReady || i == kDsReady || i == kDkvFree) cnt = 8;
      if (i == kDqDrained) cnt = 4;
      if (i == kSchedEmpty || i == kSchedEmpty + 1) cnt = 13;
      mbar_init(bar(i), cnt);
    }
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
    tma_prefetch_desc(&tm_do);
    tma_prefetch_desc(&tm_dq);
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, kBwdTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_p;
  dependency_wait();
  constexpr uint32_t tS = 0, tdP = 128, tdV = 256, tdK = 384;
  volatile int* sched = reinterpret_cast<volatile int*>(gbase + L::kBars + 8 * kNumBwdBars + 16);
  // other roles: read the n-th unit; `whole_warp` = all 32 lanes are calling
  auto take_unit = [&](uint32_t n, bool whole_warp) -> int {
    const bool ok = wait_bar(bar(kSchedFull + (n & 1)), (n >> 1) & 1, abort_flag, prm.header, 91);
    const int u = ok ? sched[n & 1] : -1;
    if (whole_warp) {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kSchedEmpty + (n & 1)));
    } else {
      mbar_arrive(bar(kSchedEmpty + (n & 1)));
    }
    return u;
  };

  if (warp < 4) {
    set_max_registers<kBwdRegsIssue, kBwdRegsLaunch>();
    if (warp == 0) {
    // ------------------------------------------------------------ producer
    uint32_t qc = 0, ucnt = 0;
    BwdUnit un;
    // (a refused plan has no work)
    const int num_units = prm.header[0] == kStatusOk ? prm.header[kHdrNumBTiles] * prm.Hkv : 0;
    const int num_parts = kSplit ? num_units << prm.lg_split : num_units;
    // all lanes: draw the n-th (part of a) unit of this CTA, publish it to the other roles
    auto fetch_unit = [&](uint32_t n) -> int {
      int packed = -1;
      if (lane == 0) {
        wait_bar(bar(kSchedEmpty + (n & 1)), ((n >> 1) & 1) ^ 1, abort_flag, prm.header, 90);
        // after a wait has given up, no more work is drawn: the end marker goes out instead
        // (The first unit is the one of the CTA's own index.  Not in the deterministic variant: a
        // CTA that starts late must not hold a unit that running CTAs wait for.)
        const int u = *abort_flag        ? num_parts
                      : !kDet && n == 0 ? int(blockIdx.x)
                                         : (kDet ? 0 : int(gridDim.x)) + atomicAdd(&prm.header[kHdrBwdNext], 1);
        if (u < num_parts)
          packed = kSplit ? prm.order[u >> prm.lg_split] | (u & ((1 << prm.lg_split) - 1)) << kPartShift
                          : prm.order[u];
        sched[n & 1] = packed;
        mbar_arrive(bar(kSchedFull + (n & 1)));
      }
      return __shfl_sync(0xffffffffu, packed, 0);
    };
    for (; get_bwd_unit<kSplit>(prm, fetch_unit(ucnt), un); ++ucnt) {
      if (lane == 0) {
        wait_bar(bar(kKvEmpty), (ucnt & 1) ^ 1, abort_flag, prm.header, 50);
        mbar_expect_tx(bar(kKvFull), 2 * L::kTileBytes);
        for (int b = 0; b < D / 64; ++b) {
          tma_load_3d(sK + b * kBoxBytes, &tm_k, b * 64, un.kvh, un.tile.start, bar(kKvFull));
          tma_load_3d(sV + b * kBoxBytes, &tm_v, b * 64, un.kvh, un.tile.start, bar(kKvFull));
        }
      }
      QIter qi;
      for (int it = 0; it < un.n_it && !*abort_flag; ++it, ++qc, q_advance<kDet>(qi, unit_heads<kSplit>(prm, un), un.nq)) {
        const QTile qt = q_tile_at<kSplit>(prm, un, qi);
        const uint32_t st = qc & 1, par = ((qc >> 1) & 1) ^ 1;
        // per-query statistics, fetched before the stage is known to be free and handed on
        // NEGATED (the compute warps add them in packed two-lane instructions);
        // +inf LSE and zero Delta switch off columns past the tile's end
        const size_t row0 = size_t(qt.h) * prm.T + qt.start;
        float r_lse[4], r_del[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = lane + 32 * i;
          r_lse[i] = c < qt.len ? prm.lse2[row0 + c] : INFINITY;
          r_del[i] = c < qt.len ? prm.delta[row0 + c] : 0.f;
        }
        wait_bar(bar(kQEmptyB + st), par, abort_flag, prm.header, 51);
        if (lane == 0) {
          mbar_expect_tx(bar(kQFullB + st), L::kTileBytes);
          for (int b = 0; b < D / 64; ++b)
            tma_load_3d(sQ + st * L::kTileBytes + b * kBoxBytes, &tm_q, b * 64, qt.h, qt.start,
                        bar(kQFullB + st));
        }
        float* sl = stats + st * 256;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          sl[lane + 32 * i] = -r_lse[i];
          sl[128 + lane + 32 * i] = -r_del[i];
        }
        mbar_arrive(bar(kQFullB + st));
        if (lane == 0) {
          wait_bar(bar(kDoEmpty), (qc & 1) ^ 1, abort_flag, prm.header, 52);
          mbar_expect_tx(bar(kDoFull), L::kTileBytes);
          for (int b = 0; b < D / 64; ++b)
            tma_load_3d(sdO + b * kBoxBytes, &tm_do, b * 64, qt.h, qt.start, bar(kDoFull));
        }
      }
    }
    } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // (elect.sync, not `lane == 0`: see the forward's issuer.  Here two rows of 32768 tokens went
    // from 32.8 to 26.9 M cycles and from 21.2 to 19.4 ms -- the clock settles lower under the
    // power limit --, eight 1100-token rows from 281 to 261 us, head_dim 64 from 554 to 432 us.)
    if (elect_one()) {
      uint32_t gc = 0, ucnt = 0;
      constexpr uint32_t idesc_kv = make_idesc(128, DV, 0, 1);  // dV, dK : K-major A, MN-major B
      constexpr uint32_t idesc_dq = make_idesc(128, DV, 1, 1);  // dQ     : MN-major A and B
      BwdUnit un;
      const uint32_t dK_k = kmajor_base(sK), dV_k = kmajor_base(sV), dK_mn = mnmajor_base(sK);
      const uint32_t dS_k = kmajor_base(sdS), dS_mn = mnmajor_base(sdS);
      constexpr uint32_t kStageStep = uint32_t(L::kTileBytes >> 4);
      auto issue_s = [&](uint32_t st, int q_len) {
        const uint32_t idesc = make_idesc(128, ((q_len + 15) >> 4) << 4, 0, 0);
        const uint32_t dq_k = kmajor_base(sQ) + st * kStageStep;
#pragma unroll
        for (int k = 0; k < DV / 16; ++k)
          mma_ss(tmem + tS, dK_k + kmajor_off(k), dq_k + kmajor_off(k), idesc, k > 0);
        mma_commit(bar(kSFullB));
      };
      for (; get_bwd_unit<kSplit>(prm, take_unit(ucnt, false), un); ++ucnt) {
        const int ksteps = (un.tile.len + 15) >> 4;
        wait_bar(bar(kKvFull), ucnt & 1, abort_flag, prm.header, 60);
        QIter qi;
        QTile qt = q_tile_at<kSplit>(prm, un, qi);
        wait_bar(bar(kQFullB + (gc & 1)), (gc >> 1) & 1, abort_flag, prm.header, 61);
        tc_fence_after();
        issue_s(gc & 1, qt.len);
        for (int it = 0; it < un.n_it; ++it) {
          const uint32_t g = gc + it, st = g & 1, par = g & 1;
          const int qsteps = (qt.len + 15) >> 4;
          const uint32_t dq_mn = mnmajor_base(sQ) + st * kStageStep;
          const uint32_t ddo_k = kmajor_base(sdO), ddo_mn = mnmajor_base(sdO);
          // dP^T(it) = V dO^T
          wait_bar(bar(kDoFull), par, abort_flag, prm.header, 62);
          if (g > 0) wait_bar(bar(kDqDrained), (g - 1) & 1, abort_flag, prm.header, 63);
          tc_fence_after();
          {
            const uint32_t idesc = make_idesc(128, qsteps << 4, 0, 0);
#pragma unroll
            for (int k = 0; k < DV / 16; ++k)
              mma_ss(tmem + tdP, dV_k + kmajor_off(k), ddo_k + kmajor_off(k), idesc, k > 0);
            mma_commit(bar(kDpFull));
          }
          // (the next tile's coordinates and descriptors are worked out here, while the pipe is
          // still busy with dP, not between dV and S)
          QTile nx = qt;
          const bool has_next = it + 1 < un.n_it;
          if (has_next) {
            q_advance<kDet>(qi, unit_heads<kSplit>(prm, un), un.nq);
            nx = q_tile_at<kSplit>(prm, un, qi);
          }
          const uint32_t idesc_s_next = make_idesc(128, ((nx.len + 15) >> 4) << 4, 0, 0);
          const uint32_t dq_k_next = kmajor_base(sQ) + ((g + 1) & 1) * kStageStep;
          // dV += P^T dO
          wait_bar(bar(kPReady), par, abort_flag, prm.header, 64);
          if (it == 0) wait_bar(bar(kDkvFree), (ucnt & 1) ^ 1, abort_flag, prm.header, 65);
          tc_fence_after();
          // (the k-step count and the accumulate flag are decided once per group: a branch or
          // a run-time predicate in front of every MMA costs the issuing thread more than the
          // MMA takes)
          auto issue_dv = [&](auto full_c, auto acc_c) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (decltype(full_c)::value || k < qsteps)
                mma_ts(tmem + tdV, tmem + tS + (k < 4 ? k * 8 : 64 + (k - 4) * 8),
                       ddo_mn + mnmajor_off(k), idesc_kv, (decltype(acc_c)::value || k > 0) ? 1u : 0u);
          };
          if (qsteps == 8) {
            if (it > 0) issue_dv(std::true_type{}, std::true_type{});
            else issue_dv(std::true_type{}, std::false_type{});
          } else {
            if (it > 0) issue_dv(std::false_type{}, std::true_type{});
            else issue_dv(std::false_type{}, std::false_type{});
          }
          mma_commit(bar(kDoEmpty));
          // S^T(it+1) = K Q^T
          if (has_next) {
            const uint32_t g1 = g + 1;
            wait_bar(bar(kQFullB + (g1 & 1)), (g1 >> 1) & 1, abort_flag, prm.header, 66);
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < DV / 16; ++k)
              mma_ss(tmem + tS, dK_k + kmajor_off(k), dq_k_next + kmajor_off(k), idesc_s_next, k > 0);
            mma_commit(bar(kSFullB));
          }
          // dQ(it) = dS K, then dK += dS^T Q
          wait_bar(bar(kDsReady), par, abort_flag, prm.header, 67);
          tc_fence_after();
          if (ksteps == 8) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              mma_ss(tmem + tdP, dS_mn + mnmajor_off(k), dK_mn + mnmajor_off(k), idesc_dq, k > 0);
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (k < ksteps)
                mma_ss(tmem + tdP, dS_mn + mnmajor_off(k), dK_mn + mnmajor_off(k), idesc_dq, k > 0);
          }
          mma_commit(bar(kDqFull));
          auto issue_dk = [&](auto full_c, auto acc_c) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (decltype(full_c)::value || k < qsteps)
                mma_ss(tmem + tdK, dS_k + kmajor_off(k), dq_mn + mnmajor_off(k), idesc_kv,
                       (decltype(acc_c)::value || k > 0) ? 1u : 0u);
          };
          if (qsteps == 8) {
            if (it > 0) issue_dk(std::true_type{}, std::true_type{});
            else issue_dk(std::true_type{}, std::false_type{});
          } else {
            if (it > 0) issue_dk(std::false_type{}, std::true_type{});
            else issue_dk(std::false_type{}, std::false_type{});
          }
          mma_commit(bar(kQEmptyB + st));
          qt = nx;
        }
        mma_commit(bar(kDkvFull));
        mma_commit(bar(kKvEmpty));
        gc += un.n_it;
      }
    }
    }
  } else if (warp < 12) {
    // ------------------------------------------------------------ compute warpgroups
    set_max_registers<kBwdRegsCompute, kBwdRegsLaunch>();
    const int wg = (warp - 4) >> 2;       // column half
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_base = tmem + (uint32_t(32 * (warp & 3)) << 16);
    const int cb = 64 * wg;
    const uint64_t sc2 = pack2(prm.scale_log2, prm.scale_log2);
    const uint32_t ds_row = sdS + wg * kBoxBytes + row * 128;   // dS^T row `row` in box wg
    uint32_t gc = 0, ucnt = 0;
    BwdUnit un;
    for (; get_bwd_unit<kSplit>(prm, take_unit(ucnt, true), un); ++ucnt) {
      const bool row_ok = row < un.tile.len;
      // my key j = tile.start + row is seen by the queries [j, key_end[j])
      const int key_lo = un.tile.start + row;
      const int key_hi = row_ok ? prm.key_end[key_lo] : key_lo;
      QIter qi;
      for (int it = 0; it < un.n_it; ++it, q_advance<kDet>(qi, unit_heads<kSplit>(prm, un), un.nq)) {
        const QTile qt = q_tile_at<kSplit>(prm, un, qi);
        const uint32_t g = gc + it, st = g & 1, par = g & 1;
        const float* sl = stats + st * 256 + cb;
        // Fast path: both tiles complete and every key row of this warp sees either the whole
        // query tile or none of it -- true for all query tiles behind the key tile except
        // where a segment ends inside them, also when the key tile itself straddles segments
        // (its prompt / earlier-response keys then see everything, the others nothing).  The
        // unmasked arithmetic runs and an unseen row's P (hence dS) is set to zero afterwards.
        const int lo = key_lo - qt.start, hi = key_hi - qt.start;
        const bool row_all = lo <= 0 && hi >= kTile, row_none = hi <= 0 || lo >= kTile;
        const bool full = qt.len == kTile && un.tile.len == kTile &&
                          __all_sync(0xffffffffu, row_all || row_none);
        wait_bar(bar(kQFullB + st), (g >> 1) & 1, abort_flag, prm.header, 70);
        wait_bar(bar(kSFullB), par, abort_flag, prm.header, 71);
        tc_fence_after();
        // P stays in fp32 registers for dS; its bf16 form goes to tensor memory
        float p[64];
        const float4* sl4 = reinterpret_cast<const float4*>(sl);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t v[32], pk[16];
          tmem_ld32(lane_base + tS + cb + 32 * hf, v);
          tmem_wait_ld();
          float* ph = p + 32 * hf;
          if (full) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 l = sl4[8 * hf + i];   // -LSE * log2(e)
              float x0, x1, x2, x3;
              unpack2(fma2(pack2(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1])), sc2,
                           pack2(l.x, l.y)), x0, x1);
              unpack2(fma2(pack2(__uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])), sc2,
                           pack2(l.z, l.w)), x2, x3);
              ph[4 * i] = ex2(x0);
              ph[4 * i + 1] = ex2(x1);
              ph[4 * i + 2] = ex2(x2);
              ph[4 * i + 3] = ex2(x3);
            }
            if (!row_all) {
#pragma unroll
              for (int i = 0; i < 32; ++i) ph[i] = 0.f;
            }
          } else {
            // query column c is visible iff key_lo <= qt.start + c < key_hi (an absent key row
            // has an empty range; key_hi never exceeds the group's end, so c < qt.len follows)
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const int c = cb + 32 * hf + i;
              const float e = ex2(fmaf(__uint_as_float(v[i]), prm.scale_log2, sl[32 * hf + i]));
              ph[i] = (c >= lo && c < hi) ? e : 0.f;
            }
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(ph[2 * i], ph[2 * i + 1]);
          tmem_st16(lane_base + tS + cb + 16 * hf, pk);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kPReady));

        wait_bar(bar(kDpFull), par, abort_flag, prm.header, 72);
        tc_fence_after();
        // dS = P (dP - Delta), in pieces of 16 columns: the load of the next one in flight under
        // the arithmetic of this one
        auto ds16 = [&](const uint32_t (&d)[16], int piece, auto masked_c) {
          uint32_t ds[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 dl = sl4[32 + 4 * piece + i];   // -Delta
            const float* pp = p + 16 * piece + 4 * i;
            float d0, d1, d2, d3;
            unpack2(mul2(pack2(pp[0], pp[1]),
                         add2(pack2(__uint_as_float(d[4 * i]), __uint_as_float(d[4 * i + 1])),
                              pack2(dl.x, dl.y))), d0, d1);
            unpack2(mul2(pack2(pp[2], pp[3]),
                         add2(pack2(__uint_as_float(d[4 * i + 2]), __uint_as_float(d[4 * i + 3])),
                              pack2(dl.z, dl.w))), d2, d3);
            if (decltype(masked_c)::value) {  // stale tensor-memory columns may hold anything
              d0 = pp[0] != 0.f ? d0 : 0.f;
              d1 = pp[1] != 0.f ? d1 : 0.f;
              d2 = pp[2] != 0.f ? d2 : 0.f;
              d3 = pp[3] != 0.f ? d3 : 0.f;
            }
            ds[2 * i] = pack_bf16(d0, d1);
            ds[2 * i + 1] = pack_bf16(d2, d3);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const uint32_t chunk = uint32_t(piece * 2 + i) ^ uint32_t(row & 7);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ds_row + chunk * 16),
                         "r"(ds[4 * i]), "r"(ds[4 * i + 1]), "r"(ds[4 * i + 2]), "r"(ds[4 * i + 3])
                         : "memory");
          }
        };
        auto ds_all = [&](auto masked_c) {
          const uint32_t t = lane_base + tdP + cb;
          uint32_t da[16], db[16];
          tmem_ld16(t, da);
          tmem_wait_ld();
          tmem_ld16(t + 16, db);
          ds16(da, 0, masked_c);
          tmem_wait_ld();
          tmem_ld16(t + 32, da);
          ds16(db, 1, masked_c);
          tmem_wait_ld();
          tmem_ld16(t + 48, db);
          ds16(da, 2, masked_c);
          tmem_wait_ld();
          ds16(db, 3, masked_c);
        };
        if (full) ds_all(std::false_type{}); else ds_all(std::true_type{});
        fence_proxy_async_smem();
        tc_fence_before();   // (the dQ tile overwrites the columns dP was loaded from)
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kDsReady));
      }
      gc += un.n_it;
      // ---- unit epilogue: warpgroup 0 stores dV, warpgroup 1 stores scale * dK
      wait_bar(bar(kDkvFull), ucnt & 1, abort_flag, prm.header, 73);
      tc_fence_after();
      if constexpr (kSplit) {   // a part: fp32, 128 rows side by side per four columns
        const size_t slot = (size_t(un.tidx) * prm.Hkv + un.kvh) << prm.lg_split | size_t(un.part);
        float4* dst = prm.parts + (slot * 2 + wg) * (DV / 4 * kTile) + row;
#pragma unroll 1
        for (int c = 0; c < DV / 16; ++c) {
          uint32_t w[16];
          tmem_ld16(lane_base + (wg ? tdK : tdV) + c * 16, w);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 4; ++i)
            dst[(c * 4 + i) * kTile] = make_float4(__uint_as_float(w[4 * i]), __uint_as_float(w[4 * i + 1]),
                                                   __uint_as_float(w[4 * i + 2]), __uint_as_float(w[4 * i + 3]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kDkvFree));
        continue;
      }
      const uint32_t tsrc = wg ? tdK : tdV;
      const float f = wg ? prm.scale : 1.f;
      uint32_t ob[D / 2];
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t w[32];
        if (DV == D || c * 32 < DV) {
          tmem_ld32(lane_base + tsrc + c * 32, w);
          tmem_wait_ld();
        } else {  // columns past DV hold nothing and are not stored
#pragma unroll
          for (int i = 0; i < 32; ++i) w[i] = 0u;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
          ob[c * 16 + i] = pack_bf16(__uint_as_float(w[2 * i]) * f, __uint_as_float(w[2 * i + 1]) * f);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kDkvFree));
      // A thread holds one row as 16-byte chunks; transposing each group of eight chunks
      // (128 bytes) inside groups of eight lanes gives every lane the same chunk of eight
      // consecutive rows, so that one store instruction of the warp writes four whole
      // 128-byte lines instead of 32 scattered 16-byte pieces (which kept the SM's memory
      // pipe busy for thousands of cycles at every unit boundary).
#pragma unroll
      for (int hb = 0; hb < D / 64; ++hb) {
        uint32_t* x = ob + 32 * hb;
        auto exchange = [&](auto dist) {
          constexpr int d = decltype(dist)::value;
          const bool hi = (lane & d) != 0;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if ((i & d) == 0) {
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const uint32_t send = hi ? x[4 * i + c] : x[4 * (i | d) + c];
                const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, d);
                if (hi) x[4 * i + c] = recv; else x[4 * (i | d) + c] = recv;
              }
            }
          }
        };
        exchange(std::integral_constant<int, 4>{});
        exchange(std::integral_constant<int, 2>{});
        exchange(std::integral_constant<int, 1>{});
      }
      {
        __nv_bfloat16* out = wg ? prm.dk : prm.dv;
        const int grp = lane >> 3, chunk = lane & 7;
#pragma unroll
        for (int hb = 0; hb < D / 64; ++hb) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = 32 * (warp & 3) + grp * 8 + i;
            if (r < un.tile.len && (DV == D || hb * 64 + chunk * 8 < DV)) {
              uint4* dst = reinterpret_cast<uint4*>(
                  out + ((size_t(un.tile.start) + r) * prm.Hkv + un.kvh) * DV + hb * 64 + chunk * 8);
              *dst = make_uint4(ob[32 * hb + 4 * i], ob[32 * hb + 4 * i + 1], ob[32 * hb + 4 * i + 2],
                                ob[32 * hb + 4 * i + 3]);
            }
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------ dQ warpgroup
    set_max_registers<kBwdRegsDq, kBwdRegsLaunch>();
    const int row = 32 * (warp & 3) + lane;
    const int quarter = warp & 3;   // rows [32 quarter, + 32) of the tile
    const bool leader = lane == 0;
    const uint32_t lane_base = tmem + (uint32_t(32 * (warp & 3)) << 16);
    const uint32_t stg = base + L::kStg + (warp - 12) * (2 * L::kStageBytes);
    uint32_t gc = 0, chunk = 0, ucnt = 0;
    BwdUnit un;
    for (; get_bwd_unit<kSplit>(prm, take_unit(ucnt, true), un); ++ucnt) {
      QIter qi;
      // Deterministic variant: the key tiles that add to a (query tile, head) do so in
      // DESCENDING tile order: the query tile's own key tile first, then the tiles below it
      // down to dep_lo of the query tile, then the prompt tiles from npc - 1 down to 0.  With
      // every unit walking its query tiles upwards from its own tile, that is the order in
      // which the units reach a query tile anyway (tile k gets there one query tile's worth
      // of iterations after tile k + 1), so in the steady state nobody waits.  The counter of
      // the pair holds 1 + the group-relative index of the last key tile that has added (0:
      // none yet).  Units are handed out set by set and inside a set in descending tile order
      // (the plan's second unit list), so the tile waited for is always running or done and
      // the waits cannot lock up.
      const int k_rel = (un.tile.start - un.tile.grp_start) / kTile;
      int dep_lo = 0;
      // Passing the turn on needs the reductions of the tile to be complete (a wait of a
      // microsecond or two), so it is deferred: the counter of iteration i is published in
      // iteration i + 1, as soon as that tile is out of tensor memory and before this unit can come
      // to wait for its own turn -- the next key tile gets to the same query tile a whole query
      // tile's worth of iterations later.
      int32_t* pend = nullptr;
      // What the turns order are reductions of the async proxy.  Ours are complete, and so visible to
      // this thread, behind the bulk wait; the release hands that on, and the next unit issues
      // its own behind the acquire that sees it and a proxy fence.  Release and acquire cost this
      // warp about a thousand cycles each, the first while the tile behind it waits in registers and
      // not in tensor memory (with the release at the end of the iteration four 4800-token groups,
      // 28 / 4 heads, take 2306 us, here 2207; eight 1100-token groups, 32 / 8, 438 and 415).  It is this
      // variant's longest chain: two rows of 32768 tokens take 25.6 ms, by default 20.0.
      auto publish = [&](int32_t* p) { store_release_gpu(p, k_rel + 1); };
      for (int it = 0; it < un.n_it; ++it, q_advance<kDet>(qi, unit_heads<kSplit>(prm, un), un.nq)) {
        const QTile qt = q_tile_at<kSplit>(prm, un, qi);
        const uint32_t g = gc + it;
        int32_t* sem = nullptr;
        int seen_early = -1;
        if (kDet && leader) {
          sem = prm.dq_sem + (size_t(un.tidx + qi.qt) * prm.Hq + qt.h) * 4 + quarter;
          // the last prompt tile follows the lowest response tile that adds to this query tile
          if (qi.hh == 0 && qi.qt > 0 && k_rel == un.tile.npc - 1 && k_rel + qi.qt >= un.tile.npc)
            dep_lo = prm.tiles[un.tidx + qi.qt].dep_lo;
          // read the counter now, under the wait for the tile (normally it has the expected value)
          seen_early = load_acquire_gpu(sem);
        }
        wait_bar(bar(kDqFull), g & 1, abort_flag, prm.header, 80);
        tc_fence_after();
        // The whole tile goes to registers at once and the dP/dQ columns back to the MMA thread,
        // before any wait on the staging buffers: the next dP has to wait for this.
        uint32_t w[D];
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          if (c * 32 < DV) {   // (no such columns in global memory: the box is not reduced either)
            tmem_ld32(lane_base + tdP + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&w[c * 32]));
          }
        }
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kDqDrained));
        if (kDet && leader) {
          if (pend) {
            bulk_wait_group<0>();
            publish(pend);
          }
          pend = sem;
        }
        if (row >= qt.len) {  // rows past the tile's end belong to other tokens: add zero
#pragma unroll
          for (int i = 0; i < DV; ++i) w[i] = 0u;
        }
#pragma unroll
        for (int c = 0; c < DV / 32; ++c, ++chunk) {
          const uint32_t buf = stg + (chunk & 1) * L::kStageBytes;
          // the reduce issued two boxes ago must have finished reading this buffer
          if (leader) bulk_wait_group_read<1>();
          __syncwarp();
          const uint32_t row_addr = buf + lane * 128;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t ch = uint32_t(i) ^ uint32_t(lane & 7);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row_addr + ch * 16),
                         "r"(w[c * 32 + 4 * i]), "r"(w[c * 32 + 4 * i + 1]),
                         "r"(w[c * 32 + 4 * i + 2]), "r"(w[c * 32 + 4 * i + 3])
                         : "memory");
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (leader) {
            if (kDet && sem && c == 0) {  // wait for this unit's turn (bounded)
              const int expect =
                  qi.qt == 0 ? 0
                             : ((k_rel == un.tile.npc - 1 && k_rel + qi.qt >= un.tile.npc) ? dep_lo + 1
                                                                                          : k_rel + 2);
              bool ok = seen_early == expect;
              for (uint32_t spin = 0; !ok && spin < (1u << 22); ++spin) {
                if (load_acquire_gpu(sem) == expect) {
                  ok = true;
                  break;
                }
                if ((spin & 0xff) == 0xff && *abort_flag) break;
                __nanosleep(20);
              }
              if (!ok && !*abort_flag) {
                if (atomicCAS(&prm.header[0], kStatusOk, kStatusWaitExpired) == kStatusOk)
                  prm.header[1] = 81;
                *abort_flag = 1;
              }
              fence_proxy_async_global();
            }
            if (32 * quarter < qt.len) tma_reduce_add_3d(&tm_dq, buf, c * 32, qt.h, qt.start + 32 * quarter);
            bulk_commit_group();
          }
        }
      }
      if (kDet && pend) {
        bulk_wait_group<0>();
        publish(pend);
      }
      gc += un.n_it;
    }
    if (leader) bulk_wait_group<0>();
  }

  tc_fence_before();
  __syncthreads();
  // After a wait that gave up, copies, reductions and MMAs issued without their barriers may
  // still be in flight: give them time to land before shared and tensor memory are released.
  if (*abort_flag)
    for (int i = 0; i < 50; ++i) __nanosleep(1000);
  if (warp == 0) tmem_dealloc(tmem, kBwdTmemCols);
  if (tid == 0) {  // the last CTA to finish re-arms the unit counter for the next launch
    __threadfence();
    if (atomicAdd(&prm.header[kHdrBwdDone], 1) == int(gridDim.x) - 1) {
      prm.header[kHdrBwdNext] = 0;
      prm.header[kHdrBwdDone] = 0;
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
extern "C" int pp_debug_bwd_cta_cycles(unsigned long long* out) {
  return cudaMemcpyFromSymbol(out, pp::g_cta_cycles, sizeof(unsigned long long) * 256) == cudaSuccess ? 0 : -5;
}
extern "C" int pp_debug_bwd_wait_cycles(unsigned long long* out, int reset) {
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
cudaError_t launch_bwd_t(const pp_plan* plan, const void* o, const float* lse, const void* d_o,
                         void* dq, const CUtensorMap& tq, const CUtensorMap& tk,
                         const CUtensorMap& tv, const CUtensorMap& tdo, const CUtensorMap& tdq,
                         const BwdParams& prm, bool dq_cleared, cudaStream_t stream,
                         int* launches) {
  static DeviceSetup setup[kMaxDevices];
  DeviceSetup* dev = device_setup(setup);
  if (!dev) return cudaErrorInvalidDevice;
  if (dev->cc_major != 10) return cudaErrorNotSupported;
  using Kernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, BwdParams);
  const Kernel kerns[4] = {bwd_kernel<D, false, false, DV>, bwd_kernel<D, false, true, DV>,
                           bwd_kernel<D, true, false, DV>, bwd_kernel<D, true, true, DV>};
  const Kernel kern = kerns[(prm.dq_sem ? 2 : 0) + (prm.lg_split ? 1 : 0)];
  if (!dev->configured) {
    for (Kernel k : kerns) {
      cudaError_t ce = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<D>::kTotal);
      if (ce != cudaSuccess) return ce;
    }
    dev->configured = true;
  }
  const pp_problem& pb = plan->prob;
  const size_t T = pb.total_tokens, Hq = pb.num_q_heads;
  const int num_sms = dev->num_sms;
  const unsigned sem_n4 = prm.dq_sem ? unsigned(max_btiles_of(pb)) * pb.num_q_heads : 0;   // 16 bytes each
  const unsigned pre_blocks = unsigned(Hq * ((T + pre_tokens(DV) - 1) / pre_tokens(DV)));
  auto pre = dq_cleared ? bwd_preprocess_kernel<DV, false> : bwd_preprocess_kernel<DV, true>;
  cudaError_t e = launch_kernel(true, pre, dim3(pre_blocks), dim3(32 * kPreWarps), 0, stream,
                                static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(d_o), lse,
                                const_cast<float*>(prm.delta), const_cast<float*>(prm.lse2), prm.dq_acc, int(T),
                                int(Hq), reinterpret_cast<int4*>(prm.dq_sem), sem_n4);
  const long long units = ((long long)plan->max_tiles * pb.num_kv_heads) << prm.lg_split;
  dim3 grid(unsigned(std::min<long long>(units, num_sms)));
  ProfileEvents& ev = profile_events();
  const int slot = int(ev.bwd_count % kProfileRing);
  if (ev.on) profile_record(ev.bwd0[slot], stream);
  if (e == cudaSuccess)
    e = launch_kernel(units <= (long long)kOverlapUnits * num_sms, kern, grid, dim3(kBwdThreads),
                      BwdSmem<D>::kTotal, stream, tq, tk, tv, tdo, tdq, prm);
  if (ev.on) {
    profile_record(ev.bwd1[slot], stream);
    ++ev.bwd_count;
  }
  const size_t n4 = T * Hq * DV / 4;
  unsigned fb = unsigned((n4 + 256 * kFinUnroll - 1) / (256 * kFinUnroll));
  const SumParts sp = {prm.parts, prm.header, prm.tiles, prm.dk, prm.dv, prm.lg_split, pb.num_kv_heads, DV};
  const unsigned sum_blocks = prm.lg_split ? unsigned(max_btiles_of(pb)) * pb.num_kv_heads * 8 : 0;
  const int parts = fin_parts(prm.lg_split, fb, num_sms);
  auto fin = parts == 8 ? bwd_finalize_kernel<8> : parts == 4 ? bwd_finalize_kernel<4> : bwd_finalize_kernel<0>;
  if (e == cudaSuccess)
    e = launch_kernel(true, fin, dim3(fb + sum_blocks), dim3(256), 0, stream,
                      reinterpret_cast<const float4*>(prm.dq_acc), static_cast<uint2*>(dq), n4, prm.scale, fb, sp);
  if (launches) *launches += 3;
  return e;
}

}  // namespace

cudaError_t launch_bwd(const pp_plan* plan, const void* q, const void* k, const void* v,
                       const void* o, const float* lse, const void* d_o, float scale, void* dq,
                       void* dk, void* dv, void* scratch, int lg_split, bool dq_cleared,
                       bool deterministic, cudaStream_t stream, int* launches) {
  const pp_problem& pb = plan->prob;
  CUtensorMap tq, tk, tv, tdo;
  if (!encode_thd(&tq, q, pb.total_tokens, pb.num_q_heads, pb.head_dim, kTile) ||
      !encode_thd(&tk, k, pb.total_tokens, pb.num_kv_heads, pb.head_dim, kTile) ||
      !encode_thd(&tv, v, pb.total_tokens, pb.num_kv_heads, pb.head_dim, kTile) ||
      !encode_thd(&tdo, d_o, pb.total_tokens, pb.num_q_heads, pb.head_dim, kTile))
    return cudaErrorNotSupported;
  const BwdScratch sl = bwd_scratch_layout(pb, lg_split);
  char* sc = static_cast<char*>(scratch);
  BwdParams prm;
  prm.header = reinterpret_cast<int32_t*>(plan->ws + plan->lay.header);
  prm.tiles = reinterpret_cast<const BTile*>(plan->ws + plan->lay.btiles);
  prm.order = reinterpret_cast<const int32_t*>(
      plan->ws + (deterministic ? plan->lay.bwd_units_det : plan->lay.bwd_units));
  prm.key_end = reinterpret_cast<const int32_t*>(plan->ws + plan->lay.key_end);
  prm.delta = reinterpret_cast<float*>(sc + sl.delta);
  prm.lse2 = reinterpret_cast<float*>(sc + sl.lse2);
  prm.dq_acc = reinterpret_cast<float*>(sc + sl.dq_acc);
  prm.parts = reinterpret_cast<float4*>(sc + sl.parts);
  prm.lg_split = lg_split;
  prm.dq_sem = nullptr;
  if (deterministic) prm.dq_sem = reinterpret_cast<int32_t*>(sc + sl.sem);
  prm.dk = static_cast<__nv_bfloat16*>(dk);
  prm.dv = static_cast<__nv_bfloat16*>(dv);
  prm.T = pb.total_tokens;
  prm.Hq = pb.num_q_heads;
  prm.Hkv = pb.num_kv_heads;
  prm.scale = scale;
  prm.scale_log2 = scale * 1.4426950408889634f;
  CUtensorMap tdq;
  if (!encode_thd_f32(&tdq, prm.dq_acc, pb.total_tokens, pb.num_q_heads, pb.head_dim))
    return cudaErrorNotSupported;
  if (pb.head_dim == 128)
    return launch_bwd_t<128>(plan, o, lse, d_o, dq, tq, tk, tv, tdo, tdq, prm, dq_cleared, stream,
                             launches);
  if (pb.head_dim == 96)
    return launch_bwd_t<128, 96>(plan, o, lse, d_o, dq, tq, tk, tv, tdo, tdq, prm, dq_cleared,
                                 stream, launches);
  return launch_bwd_t<64>(plan, o, lse, d_o, dq, tq, tk, tv, tdo, tdq, prm, dq_cleared, stream,
                          launches);
}

// ---------------------------------------------------------------- built-in scratch
// Backward scratch for callers that cannot allocate device memory (pp_attn_bwd_noalloc).
// The array is part of the library image: every device that loads the library holds
// kStaticScratchBytes until the process exits, and every call on a device shares it.
static __device__ __align__(256) unsigned char g_static_bwd_scratch[kStaticScratchBytes];

// In host code `g_static_bwd_scratch` is only a stand-in for the symbol, not a device
// address, so the address is looked up once per device (with that device current) and kept.
// The array used must be the one on the device that holds the plan (and so the tensors): the
// current device has to be that device, otherwise the call is refused instead of handing the
// kernels another GPU's array.
static cudaError_t static_scratch_address(const pp_plan* plan, void** out) {
  static std::mutex mu;
  static void* ptrs[kMaxDevices] = {};
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  cudaPointerAttributes attr;
  e = cudaPointerGetAttributes(&attr, plan->ws);
  if (e != cudaSuccess) return e;
  if (attr.type != cudaMemoryTypeDevice || attr.device != dev) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!ptrs[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_bwd_scratch);
    if (e != cudaSuccess) return e;
    if (!p) return cudaErrorInvalidSymbol;
    ptrs[dev] = p;
  }
  *out = ptrs[dev];
  return cudaSuccess;
}

cudaError_t launch_bwd_static(const pp_plan* plan, const void* q, const void* k, const void* v,
                              const void* o, const float* lse, const void* d_o, float scale,
                              void* dq, void* dk, void* dv, cudaStream_t stream, int* launches) {
  void* scratch = nullptr;
  cudaError_t e = static_scratch_address(plan, &scratch);
  if (e != cudaSuccess) return e;
  // launch_bwd zeroes the fp32 dQ accumulator inside the scratch on every call and rewrites
  // Delta and the scaled LSE, so nothing of an earlier call's contents is read.
  const int lg_split =
      bwd_scratch_layout(plan->prob, plan->lg_split).sem <= kStaticScratchBytes ? plan->lg_split : 0;
  return launch_bwd(plan, q, k, v, o, lse, d_o, scale, dq, dk, dv, scratch, lg_split, false, false,
                    stream, launches);
}

}  // namespace pp
