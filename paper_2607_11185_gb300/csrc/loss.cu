// loss.cu - the token-level RL objective over packed segments (App. C.2), sm_103a.
//
// For every segment token t (trajectory b(t), advantage A = adv[b(t)], loss
// mask m_t from the segment builder):
//   rho = exp(logp - old_logp)
//   o   = min(rho A, clip(rho, 1 - eps_l, 1 + eps_h) A), and for A < 0 also
//         o = max(o, c A)   (the clip-ratio cap c)
//   k   = exp(r) - r - 1 with r = ref_logp - logp   (per-token KL estimate)
//   loss   = (1/N_traj) sum_t m_t (-o + lambda k)
//   dlogp  = (m_t/N_traj) (-do/dlogp + lambda (1 - exp(r))),  do/dlogp = rho A
//            on the rho-dependent branch, 0 where o is clipped to a constant.
// The branch is taken in float32; the per-token terms are float32 and the sum
// is accumulated in double, per block and then over the blocks in a fixed
// order (the result does not depend on scheduling).
//
// HBM-bound: the mask byte and the fp32 gradient of every token, three fp32 inputs of a
// trainable one, plus a log2(num_segments) lookup of a token's segment in cu_seqlens
// (L1-resident).
#include <cstdint>

#include "internal.h"

namespace vcs {
namespace {

constexpr int kThreads = 256;
constexpr int kPerThread = 8;
constexpr int kChunk = kThreads * kPerThread;  // tokens per block
constexpr int kMaxBlocks = 152 * 8;

__device__ __forceinline__ void set_status(int32_t* status, int32_t code) { atomicCAS(status, 0, code); }

// last s in [0, num_segments) with cu[s] <= t (t < cu[num_segments])
__device__ __forceinline__ int segment_of(const int32_t* __restrict__ cu, int num_segments, int t) {
  int lo = 0, hi = num_segments;  // invariant: cu[lo] <= t < cu[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(&cu[mid]) <= t) lo = mid;
    else hi = mid;
  }
  return lo;
}

struct LossArgs {
  const float* logp;
  const float* old_logp;
  const float* ref_logp;
  const uint8_t* mask;
  const int32_t* cu_seqlens;
  const int32_t* seg_traj;
  int32_t num_segments, num_tokens;
  const float* adv;
  int32_t num_traj;
  float lo, hi, cap, kl_coef, inv_ntraj;
  float* dlogp;
  double* partial;
  double inv_ntraj64;
  double* loss;
  int32_t* status;
  uint32_t* done;  // blocks that have written their partial sum
};

// Gradient of trainable token t of segment s; its loss term is added to acc.
__device__ __forceinline__ float loss_token(const LossArgs& a, int t, int s, double& acc) {
  const int b = __ldg(&a.seg_traj[s]);
  if (b < 0 || b >= a.num_traj) {
    set_status(a.status, VCS_ERR_DEVICE_CHECK);
    return 0.f;
  }
  const float A = __ldg(&a.adv[b]);
  const float lp = __ldg(&a.logp[t]);
  const float rho = expf(lp - __ldg(&a.old_logp[t]));
  float o, dobj;
  if (A >= 0.f) {
    if (rho <= a.hi) { o = rho * A; dobj = o; }
    else { o = a.hi * A; dobj = 0.f; }
  } else {
    if (rho < a.lo) { o = a.lo * A; dobj = 0.f; }
    else if (rho > a.cap) { o = a.cap * A; dobj = 0.f; }
    else { o = rho * A; dobj = o; }
  }
  const float r = __ldg(&a.ref_logp[t]) - lp;
  const float em1 = expm1f(r);
  acc += (double)(-o + a.kl_coef * (em1 - r));
  return (-dobj - a.kl_coef * em1) * a.inv_ntraj;
}

// Four consecutive tokens a thread: one mask word, one gradient store (VEC: the mask 4-byte and
// dlogp 16-byte aligned), one segment look-up for a group with trainable tokens.  The block that
// finishes last adds the blocks' sums, in block order, so the loss does not depend on scheduling.
// 2.0 M tokens, L2 flushed, events around the call: 18.1 us, 20.1 with a token a thread and a second
// launch for the sum.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) grpo_loss_tokens(const __grid_constant__ LossArgs a) {
  double acc = 0.0;
  for (int64_t base = (int64_t)blockIdx.x * kChunk; base < a.num_tokens; base += (int64_t)gridDim.x * kChunk) {
#pragma unroll
    for (int i = 0; i < kPerThread / 4; ++i) {
      const int64_t t0 = base + i * (kThreads * 4) + threadIdx.x * 4;
      if (t0 >= a.num_tokens) break;
      const int n = (int)(a.num_tokens - t0 < 4 ? a.num_tokens - t0 : 4);
      uint32_t m = 0;
      if (VEC && n == 4) {
        m = __ldg(reinterpret_cast<const uint32_t*>(a.mask + t0));
      } else {
        for (int u = 0; u < n; ++u) m |= (uint32_t)__ldg(&a.mask[t0 + u]) << (8 * u);
      }
      float g[4] = {0.f, 0.f, 0.f, 0.f};
      if (m != 0) {
        int s = segment_of(a.cu_seqlens, a.num_segments, (int)t0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int t = (int)t0 + u;
          if (((m >> (8 * u)) & 0xffu) == 0) continue;
          while (s + 1 < a.num_segments && __ldg(&a.cu_seqlens[s + 1]) <= t) ++s;
          g[u] = loss_token(a, t, s, acc);
        }
      }
      if (a.dlogp != nullptr) {
        if (VEC && n == 4) {
          *reinterpret_cast<float4*>(a.dlogp + t0) = make_float4(g[0], g[1], g[2], g[3]);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (u < n) a.dlogp[t0 + u] = g[u];
        }
      }
    }
  }
  // block sum (double) in a fixed order
  __shared__ double red[kThreads / 32];
  __shared__ bool last;
  auto block_sum = [&](double x) {  // thread 0 holds it
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    double sum = 0.0;
    if (threadIdx.x == 0)
      for (int w = 0; w < kThreads / 32; ++w) sum += red[w];
    return sum;
  };
  const double sum = block_sum(acc);
  if (threadIdx.x == 0) {
    a.partial[blockIdx.x] = sum;
    __threadfence();
    last = atomicAdd(a.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double x = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += kThreads) x += __ldcg(&a.partial[i]);
  const double total = block_sum(x);
  if (threadIdx.x == 0) *a.loss = total * a.inv_ntraj64;
}

// Mean and population standard deviation in double.  One warp per group: a group's latency (one group of
// 8: 8.9 us with events around the call, nearly all of it the launch; 10.9 with a thread per group).
__global__ void __launch_bounds__(256) group_advantage_warp(const float* __restrict__ rewards, int64_t num_groups,
                                                              int32_t group_size, float eps, float* __restrict__ adv) {
  const int lane = threadIdx.x & 31;
  auto warp_sum = [](double x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
  };
  for (int64_t gi = blockIdx.x * 8ll + (threadIdx.x >> 5); gi < num_groups; gi += (int64_t)gridDim.x * 8) {
    const float* r = rewards + gi * group_size;
    double sum = 0.0;
    for (int j = lane; j < group_size; j += 32) sum += r[j];
    const double mean = warp_sum(sum) / group_size;
    double var = 0.0;
    for (int j = lane; j < group_size; j += 32) {
      const double d = r[j] - mean;
      var += d * d;
    }
    const double den = sqrt(warp_sum(var) / group_size) + (double)eps;
    for (int j = lane; j < group_size; j += 32) adv[gi * group_size + j] = (float)((r[j] - mean) / den);
  }
}

// One thread per group: every lane's double arithmetic, which bounds many groups, is another group's.
__global__ void group_advantage_thread(const float* __restrict__ rewards, int64_t num_groups, int32_t group_size,
                                       float eps, float* __restrict__ adv) {
  for (int64_t gi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gi < num_groups;
       gi += (int64_t)gridDim.x * blockDim.x) {
    const float* r = rewards + gi * group_size;
    double mean = 0.0;
    for (int j = 0; j < group_size; ++j) mean += r[j];
    mean /= group_size;
    double var = 0.0;
    for (int j = 0; j < group_size; ++j) {
      const double d = r[j] - mean;
      var += d * d;
    }
    const double den = sqrt(var / group_size) + (double)eps;
    for (int j = 0; j < group_size; ++j) adv[gi * group_size + j] = (float)((r[j] - mean) / den);
  }
}

int loss_blocks(int64_t num_tokens) {
  int64_t b = (num_tokens + kChunk - 1) / kChunk;
  if (b < 1) b = 1;
  return (int)(b < kMaxBlocks ? b : kMaxBlocks);
}

}  // namespace

size_t grpo_loss_ws_bytes(int64_t num_tokens) { return kWsHeader + (size_t)loss_blocks(num_tokens) * sizeof(double); }

cudaError_t launch_grpo_loss(const float* logp, const float* old_logp, const float* ref_logp, const uint8_t* mask,
                             const int32_t* cu_seqlens, const int32_t* seg_traj, int32_t num_segments,
                             int32_t num_tokens, const float* adv, int32_t num_traj, float lo, float hi,
                             float clip_cap, float kl_coef, double* loss, float* dlogp, void* ws, cudaStream_t st) {
  int32_t* status = static_cast<int32_t*>(ws);
  double* partial = reinterpret_cast<double*>(static_cast<char*>(ws) + kWsHeader);
  const int nb = loss_blocks(num_tokens);
  // the status word and the count of finished blocks
  if (cudaError_t e = cudaMemsetAsync(status, 0, 2 * sizeof(int32_t), st); e != cudaSuccess) return e;
  LossArgs a;
  a.logp = logp;
  a.old_logp = old_logp;
  a.ref_logp = ref_logp;
  a.mask = mask;
  a.cu_seqlens = cu_seqlens;
  a.seg_traj = seg_traj;
  a.num_segments = num_segments;
  a.num_tokens = num_tokens;
  a.adv = adv;
  a.num_traj = num_traj;
  a.lo = lo;
  a.hi = hi;
  a.cap = clip_cap;
  a.kl_coef = kl_coef;
  a.inv_ntraj = 1.f / (float)num_traj;
  a.dlogp = dlogp;
  a.partial = partial;
  a.inv_ntraj64 = 1.0 / (double)num_traj;
  a.loss = loss;
  a.status = status;
  a.done = reinterpret_cast<uint32_t*>(status + 1);
  const bool vec = (reinterpret_cast<uintptr_t>(mask) & 3u) == 0 && (reinterpret_cast<uintptr_t>(dlogp) & 15u) == 0;
  if (vec)
    grpo_loss_tokens<true><<<nb, kThreads, 0, st>>>(a);
  else
    grpo_loss_tokens<false><<<nb, kThreads, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_group_advantage(const float* rewards, int64_t num_groups, int32_t group_size, float eps,
                                   float* adv, cudaStream_t st) {
  if (num_groups == 0) return cudaSuccess;
  // Measured up to 1 M groups: a warp a group takes 1.8 + 1.1 ceil(group_size / 32) ns a group, a thread a
  // group 1,140 ns a member until the groups fill the chip, so the line is where the two are equal (8 a
  // group, us, warp / thread: 12 / 16 at 2,048 groups, 20 / 16 at 4,096, 2,950 / 295 at 1 M).  Past 512
  // members a warp, whose loads are whole lines, is no slower at any count (32,768 of 1,024: 1,120 / 1,165).
  const bool thread = group_size <= 512 && num_groups >= 11400ll * group_size / (18 + 11 * ((group_size + 31) / 32));
  int64_t blocks = thread ? (num_groups + 255) / 256 : (num_groups + 7) / 8;
  if (blocks > 152 * 8) blocks = 152 * 8;
  (thread ? group_advantage_thread : group_advantage_warp)<<<(unsigned)blocks, 256, 0, st>>>(rewards, num_groups,
                                                                                            group_size, eps, adv);
  return cudaGetLastError();
}

}  // namespace vcs
