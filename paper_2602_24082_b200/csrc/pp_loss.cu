// Loss-side consumer on the packed layout (paper Sec. 2.1): per-response sequence
// log-probabilities and the pairwise preference loss over the ranked responses of a group.
//
// The packed row is split back into its responses here: s_k = sum of the token log-probs of
// response k (prompt tokens do not count).  Reward r_k = beta * (s_k - s_k_ref) (DPO; the
// paper prints the ratio without the logarithm -- the log-ratio of Rafailov et al. is used),
// or beta * s_k when no reference is given.  Responses are ranked as in the paper's Sec. 3.1:
// response a is preferred over response b for a > b.  Group loss = mean over the pairs a > b
// of -log sigmoid(r_a - r_b) (the paper's Bradley-Terry expression with the usual minus sign);
// the optional gradient is d(sum of group losses) / d token_logp.
// 4 bytes per token read per log-prob array, 4 written for the gradient: a few microseconds of
// memory time, so what counts is how many loads are in flight.  One block per group, its warps
// split into teams that take one response at a time -- a team is as wide as the batch's mean
// segment asks for, so that two long responses keep all warps busy and many short ones are
// summed at the same time.  (One warp per group took 47 us on 7 groups of 9400 tokens, this
// 16.)
#include "pp_internal.h"

namespace pp {
namespace {

struct LossPtrs {
  const int32_t* header;
  const int32_t* seg_start;
  const int32_t* grp_resp_off;
  int G;
};

__device__ __forceinline__ float log_sigmoid(float x) {
  return fminf(x, 0.f) - log1pf(expf(-fabsf(x)));
}
__device__ __forceinline__ float sigmoid(float x) { return 1.f / (1.f + expf(-x)); }

constexpr int kLossThreads = 512, kLossWarps = kLossThreads / 32;

// f(t) for the tokens of [a, b) that warp w of a team of nw covers, four per lane in flight
template <typename F>
__device__ __forceinline__ void for_tokens(int a, int b, int w, int nw, F f) {
  const int step = nw * 32;
#pragma unroll 4
  for (int t = a + w * 32 + (threadIdx.x & 31); t < b; t += step) f(t);
}

__global__ void __launch_bounds__(kLossThreads)
preference_loss_kernel(LossPtrs p, const float* __restrict__ logp, const float* __restrict__ ref,
                       float beta, float* __restrict__ resp_logp, float* resp_reward,
                       float* __restrict__ grp_loss, float* __restrict__ d_logp, int team_warps) {
  __shared__ double s_sum[kLossWarps], s_ref[kLossWarps];
  __shared__ float s_grad[kLossWarps];
  if (p.header[0] != kStatusOk) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = blockIdx.x;
  const int x0 = p.grp_resp_off[g], x1 = p.grp_resp_off[g + 1], n = x1 - x0;
  const int sp = g + x0;  // the group's prompt segment; response x is segment g + 1 + x
  const int teams = kLossWarps / team_warps, team = warp / team_warps, in_team = warp % team_warps;
  // 1. sequence log-probs and rewards, `teams` responses at a time.  A lane's own terms, a few dozen,
  // are added in fp32, everything above in fp64: a reward is the small difference of two large sums, and
  // every rounding of those is many times larger in it.
  for (int first = x0; first < x1; first += teams) {
    const int x = first + team;
    float s = 0.f, sr = 0.f;
    if (x < x1) {
      const int a = p.seg_start[g + 1 + x], b = p.seg_start[g + 2 + x];
      if (ref)
        for_tokens(a, b, in_team, team_warps, [&](int t) {
          s += logp[t];
          sr += ref[t];
        });
      else
        for_tokens(a, b, in_team, team_warps, [&](int t) { s += logp[t]; });
    }
    double sum = s, sum_ref = sr;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
      sum_ref += __shfl_xor_sync(0xffffffffu, sum_ref, o);
    }
    if (lane == 0) {
      s_sum[warp] = sum;
      s_ref[warp] = sum_ref;
    }
    __syncthreads();
    if (in_team == 0 && lane == 0 && x < x1) {
      for (int w = 1; w < team_warps; ++w) {
        sum += s_sum[warp + w];
        sum_ref += s_ref[warp + w];
      }
      resp_logp[x] = float(sum);
      resp_reward[x] = float(beta * (sum - sum_ref));
    }
    __syncthreads();
  }
  // 2. pairwise loss over ranked pairs (a preferred over b for a > b) and d loss / d reward
  const int npairs = n * (n - 1) / 2;
  const float inv = npairs > 0 ? 1.f / float(npairs) : 0.f;
  if (warp == 0) {
    float loss = 0.f;
    for (int a = 1 + lane; a < n; a += 32)
      for (int b = 0; b < a; ++b) loss -= log_sigmoid(resp_reward[x0 + a] - resp_reward[x0 + b]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) grp_loss[g] = loss * inv;
  }
  if (!d_logp) return;
  // 3. gradient: prompt tokens get 0; tokens of response k get beta * dL/dr_k
  for_tokens(p.seg_start[sp], p.seg_start[sp + 1], warp, kLossWarps, [&](int t) { d_logp[t] = 0.f; });
  for (int first = 0; first < n; first += teams) {
    const int k = first + team;
    if (k < n && in_team == 0) {
      const float rk = resp_reward[x0 + k];
      float gk = 0.f;
      for (int j = lane; j < n; j += 32) {
        if (j == k) continue;
        const float rj = resp_reward[x0 + j];
        // k preferred over j (k > j): d/dr_k of -log sig(r_k - r_j) = -sig(r_j - r_k)
        // j preferred over k (j > k): d/dr_k of -log sig(r_j - r_k) = +sig(r_k - r_j)
        gk += (k > j) ? -sigmoid(rj - rk) : sigmoid(rk - rj);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) gk += __shfl_xor_sync(0xffffffffu, gk, o);
      if (lane == 0) s_grad[team] = beta * gk * inv;
    }
    __syncthreads();
    if (k < n) {
      const float gt = s_grad[team];
      for_tokens(p.seg_start[g + 1 + x0 + k], p.seg_start[g + 2 + x0 + k], in_team, team_warps,
                 [&](int t) { d_logp[t] = gt; });
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_preference_loss(const pp_plan* plan, const float* logp, const float* ref,
                                   float beta, float* resp_logp, float* resp_reward,
                                   float* grp_loss, float* d_logp, cudaStream_t stream) {
  LossPtrs p;
  p.header = reinterpret_cast<const int32_t*>(plan->ws + plan->lay.header);
  p.seg_start = reinterpret_cast<const int32_t*>(plan->ws + plan->lay.seg_start);
  p.grp_resp_off = plan->prob.grp_resp_off;
  p.G = plan->prob.num_groups;
  // a warp has 128 tokens in flight: a team covers the mean segment in about one round
  const int mean = plan->prob.total_tokens / plan->nseg;
  int team_warps = 1;
  while (team_warps < kLossWarps && team_warps * 128 < mean) team_warps *= 2;
  preference_loss_kernel<<<p.G, kLossThreads, 0, stream>>>(p, logp, ref, beta, resp_logp, resp_reward,
                                                           grp_loss, d_logp, team_warps);
  return cudaGetLastError();
}

}  // namespace pp
