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
// memory time, so what counts is how many loads are in flight.  A gang of 1 - 16 warps works on a group,
// as many as fill the chip with the batch's groups (loss_gang_warps below), and inside a gang teams
// of warps take one response at a time -- a team is as wide as the batch's mean segment asks for, so
// that two long responses keep all warps busy and many short ones are summed at the same time.
// (Device time, always one warp per group -> gangs: 7 groups of 9400 tokens 23 -> 8 us; always sixteen ->
// gangs: 8192 groups of 70 tokens 53 -> 14.)
#include "pp_internal.h"
#include "pp_ptx.cuh"

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

// Warps per group: the largest power of two that leaves the batch at 32 warps per SM, half of what
// fits; or 64 where groups have many responses, whose pairs take more time than their tokens.  (2048
// groups of 820 tokens, 2 responses: 12.4 us, with 64 per SM 14.9; 600 groups of 64 short responses 47
// and 36.)
int loss_gang_warps(const pp_problem& p, int num_sms) {
  const long long limit = (long long)num_sms * (p.num_responses / p.num_groups >= 16 ? 64 : 32);
  int w = kLossWarps;
  while (w > 1 && p.num_groups * w > limit) w /= 2;
  return w;
}

// f(t) for the tokens of [a, b) that warp w of a team of nw covers, four per lane in flight
template <typename F>
__device__ __forceinline__ void for_tokens(int a, int b, int w, int nw, F f) {
  const int step = nw * 32;
#pragma unroll 4
  for (int t = a + w * 32 + (threadIdx.x & 31); t < b; t += step) f(t);
}

template <int kGang>
__global__ void __launch_bounds__(kLossThreads)
preference_loss_kernel(LossPtrs p, const float* logp, const float* ref,
                       float beta, float* resp_logp, float* resp_reward,
                       float* grp_loss, float* d_logp, int team_warps) {
  dependency_wait();
  // (two buffers each, in turn: one barrier per round)
  __shared__ double s_sum[2][kLossWarps], s_ref[2][kLossWarps];
  __shared__ float s_grad[2][kLossWarps];
  if (p.header[0] != kStatusOk) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gang = warp / kGang, in_gang = warp % kGang;
  const int g = blockIdx.x * (kLossWarps / kGang) + gang;
  if (g >= p.G) return;
  auto sync = [&]() {
    if (kGang == 1) __syncwarp();
    else if (kGang == kLossWarps) __syncthreads();
    else named_barrier_sync(1 + gang, 32 * kGang);
  };
  if (kGang == 1) team_warps = 1;
  const int x0 = p.grp_resp_off[g], x1 = p.grp_resp_off[g + 1], n = x1 - x0;
  const int sp = g + x0;  // the group's prompt segment; response x is segment g + 1 + x
  const int teams = kGang / team_warps, team = in_gang / team_warps, in_team = in_gang % team_warps;
  // 1. sequence log-probs and rewards, `teams` responses at a time.  A lane's own terms, a few dozen,
  // are added in fp32, everything above in fp64: a reward is the small difference of two large sums, and
  // every rounding of those is many times larger in it.
  int buf = 0;
  for (int first = x0; first < x1; first += teams, buf ^= 1) {
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
    if (team_warps > 1) {
      if (lane == 0) {
        s_sum[buf][warp] = sum;
        s_ref[buf][warp] = sum_ref;
      }
      sync();
      if (in_team == 0 && lane == 0)
        for (int w = 1; w < team_warps; ++w) {
          sum += s_sum[buf][warp + w];
          sum_ref += s_ref[buf][warp + w];
        }
    }
    if (in_team == 0 && lane == 0 && x < x1) {
      resp_logp[x] = float(sum);
      resp_reward[x] = float(beta * (sum - sum_ref));
    }
  }
  sync();
  // 2. pairwise loss over ranked pairs (a preferred over b for a > b) and d loss / d reward
  const int npairs = n * (n - 1) / 2;
  const float inv = npairs > 0 ? 1.f / float(npairs) : 0.f;
  if (in_gang == 0) {
    float loss = 0.f;
    for (int a = 1 + lane; a < n; a += 32)
      for (int b = 0; b < a; ++b) loss -= log_sigmoid(resp_reward[x0 + a] - resp_reward[x0 + b]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) grp_loss[g] = loss * inv;
  }
  if (!d_logp) return;
  // 3. gradient: prompt tokens get 0; tokens of response k get beta * dL/dr_k
  for_tokens(p.seg_start[sp], p.seg_start[sp + 1], in_gang, kGang, [&](int t) { d_logp[t] = 0.f; });
  for (int first = 0; first < n; first += teams, buf ^= 1) {
    const int k = first + team;
    float gk = 0.f;
    if (k < n && in_team == 0) {
      const float rk = resp_reward[x0 + k];
      for (int j = lane; j < n; j += 32) {
        if (j == k) continue;
        const float rj = resp_reward[x0 + j];
        // k preferred over j (k > j): d/dr_k of -log sig(r_k - r_j) = -sig(r_j - r_k)
        // j preferred over k (j > k): d/dr_k of -log sig(r_j - r_k) = +sig(r_k - r_j)
        gk += (k > j) ? -sigmoid(rj - rk) : sigmoid(rk - rj);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) gk += __shfl_xor_sync(0xffffffffu, gk, o);
      gk = beta * gk * inv;
      if (team_warps > 1 && lane == 0) s_grad[buf][warp] = gk;
    }
    if (team_warps > 1) {
      sync();
      gk = s_grad[buf][warp - in_team];
    }
    if (k < n)
      for_tokens(p.seg_start[g + 1 + x0 + k], p.seg_start[g + 2 + x0 + k], in_team, team_warps,
                 [&](int t) { d_logp[t] = gk; });
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
  static DeviceSetup setup[kMaxDevices];
  const DeviceSetup* dev = device_setup(setup);
  if (!dev) return cudaErrorInvalidDevice;
  const int gang_warps = loss_gang_warps(plan->prob, dev->num_sms);
  // a warp has 128 tokens in flight: a team covers the mean segment in about one round
  const int mean = plan->prob.total_tokens / plan->nseg;
  int team_warps = 1;
  while (team_warps < gang_warps && team_warps * 128 < mean) team_warps *= 2;
  const int gangs = kLossWarps / gang_warps;
  auto kern = gang_warps == 16  ? preference_loss_kernel<16>
              : gang_warps == 8 ? preference_loss_kernel<8>
              : gang_warps == 4 ? preference_loss_kernel<4>
              : gang_warps == 2 ? preference_loss_kernel<2>
                                : preference_loss_kernel<1>;
  return launch_kernel(true, kern, dim3((p.G + gangs - 1) / gangs), dim3(kLossThreads), 0, stream, p, logp, ref, beta,
                       resp_logp, resp_reward, grp_loss, d_logp, team_warps);
}

}  // namespace pp
