// segments.cu - the Visual Context Segmentation layout builder (Sec. 3.4,
// Algorithm 1; App. C.1), as integer scans and a per-token expansion.
//
// Algorithm 1 keeps a running token stream per rollout and prunes it when the
// screenshot count exceeds K + delta.  Because a prune depends only on the
// number of steps seen, the segment boundaries have a closed form per
// trajectory (K = keep, delta = window, steps 1-based):
//   first segment: new steps 1..min(K+delta, T), screenshots for all of them;
//   segment j >= 1: new steps s_j = K+delta+(j-1)*delta+1 .. e_j =
//   min(s_j+delta-1, T); screenshots for a_j = max(1, s_j-K) .. e_j; steps
//   before a_j appear as their response tokens only (the fresh, re-tokenised
//   stream after a prune).
// Segment j's length is therefore
//   L_j = sum_{t<a_j} txt_t + sum_{t=a_j..e_j} (img_t + txt_t),
// which two global exclusive scans over the steps give in O(1).
//
// Kernels (all on the caller's stream, no host synchronisation):
//   seg_plan    one warp per trajectory: prefix sums of img+txt and txt over its steps, segment
//               count, tokens, max length; then one block: scans over trajectories, totals,
//               overflow and capacity checks, the vcs_sizes record and, for up to kOneBlock
//               trajectories, the segment tables
//   seg_write   (more trajectories) the segment tables: cu_seqlens, seg_traj and the per-segment
//               step bounds used by the expansion
//   seg_expand  gather index, source step, position, loss mask of every segment token, streamed
//               run by run (one run per step of the segment), 32 consecutive tokens per store
// A small batch is bound by launches, so up to kOneBlock trajectories take one block and one
// launch, and nothing needs clearing first.
#include <climits>
#include <cstdint>

#include "internal.h"
#include "sm100.cuh"

namespace vcs {
namespace {

constexpr int kScanThreads = 1024;
// Up to this many trajectories one block does the whole plan: 8 rollouts of 50 steps 3.9 us in one
// launch against 13 us in three; at 128 the passes of its 32 warps cost about what a second launch
// and the memset of the counters would.
constexpr int kOneBlock = 128;

// Inclusive block-wide scan of two int64 values per thread; *tot receives the block totals.
__device__ void block_scan2(long long& a, long long& b, long long& tot_a, long long& tot_b) {
  __shared__ long long sa[32], sb[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    long long ta = __shfl_up_sync(0xffffffffu, a, o);
    long long tb = __shfl_up_sync(0xffffffffu, b, o);
    if (lane >= o) {
      a += ta;
      b += tb;
    }
  }
  if (lane == 31) {
    sa[warp] = a;
    sb[warp] = b;
  }
  __syncthreads();
  if (warp == 0) {
    long long xa = lane < nwarps ? sa[lane] : 0, xb = lane < nwarps ? sb[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      long long ta = __shfl_up_sync(0xffffffffu, xa, o);
      long long tb = __shfl_up_sync(0xffffffffu, xb, o);
      if (lane >= o) {
        xa += ta;
        xb += tb;
      }
    }
    sa[lane] = xa;
    sb[lane] = xb;
  }
  __syncthreads();
  if (warp > 0) {
    a += sa[warp - 1];
    b += sb[warp - 1];
  }
  tot_a = sa[nwarps - 1];
  tot_b = sb[nwarps - 1];
  __syncthreads();
}

// totals[3] holds the status; of several errors inconsistent data comes first, then overflow, then
// capacity, which is their numeric order.
__device__ __forceinline__ void fail(int64_t* totals, int code) {
  static_assert(VCS_ERR_DEVICE_CHECK > VCS_ERR_OVERFLOW && VCS_ERR_OVERFLOW > VCS_ERR_CAPACITY, "order of errors");
  atomicMax(reinterpret_cast<unsigned long long*>(&totals[3]), (unsigned long long)code);
}

// Segment j of a T-step trajectory: 1-based (a, s, e).
__device__ __forceinline__ void seg_bounds(int j, int T, int keep, int window, int& a, int& s, int& e) {
  if (j == 0) {
    s = 1;
    e = min(keep + window, T);
  } else {
    s = keep + window + (j - 1) * window + 1;
    e = min(s + window - 1, T);
  }
  a = max(1, s - keep);
}

__device__ __forceinline__ int seg_count(int T, int keep, int window) {
  if (T <= 0) return 0;
  if (T <= keep + window) return 1;
  return 1 + (T - keep - window + window - 1) / window;
}

// Exclusive prefix of a trajectory-local inclusive prefix array at step u (g0 the first step).
__device__ __forceinline__ int64_t pre(const int64_t* inc, int64_t g0, int64_t u) { return u > g0 ? inc[u - 1] : 0; }

// Tokens of segment (a, s, e) (1-based) of the trajectory whose steps start at g0.
__device__ __forceinline__ long long seg_len(const SegWorkspace& w, int64_t g0, int a, int e) {
  return pre(w.txt_inc, g0, g0 + a - 1) + (w.step_inc[g0 + e - 1] - pre(w.step_inc, g0, g0 + a - 1));
}

// Segment tables of trajectory b, by one warp: 32 segments at a time, their starts by a warp scan.
__device__ void write_segments(int b, int g0, int T, int window, int keep, int32_t* __restrict__ cu_seqlens,
                               int32_t* __restrict__ seg_traj, const SegWorkspace& w, int lane) {
  const int nseg = seg_count(T, keep, window);
  int64_t base = w.tok_base[b];
  const int64_t seg0 = w.seg_base[b];
  for (int j0 = 0; j0 < nseg; j0 += 32) {
    const int j = j0 + lane;
    int a = 1, s = 1, e = 1;
    long long len = 0;
    if (j < nseg) {
      seg_bounds(j, T, keep, window, a, s, e);
      len = seg_len(w, g0, a, e);
    }
    long long x = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (j < nseg) {
      const int64_t seg = seg0 + j, start = base + x - len;
      cu_seqlens[seg] = (int32_t)start;
      if (seg_traj != nullptr) seg_traj[seg] = b;
      w.seg_start[seg] = start;
      w.seg_traj[seg] = b;
      w.seg_full[seg] = g0 + a - 1;
      w.seg_new[seg] = g0 + s - 1;
      w.seg_last[seg] = g0 + e - 1;
    }
    base += __shfl_sync(0xffffffffu, x, 31);
  }
}

// BUILD: also the segment tables (one block only).
template <bool BUILD>
__global__ void __launch_bounds__(kScanThreads)
    seg_plan(const int32_t* __restrict__ cu_steps, int32_t num_traj, int64_t num_steps,
             const int32_t* __restrict__ step_img, const int32_t* __restrict__ step_txt, int32_t window, int32_t keep,
             int64_t seg_capacity, int64_t tok_capacity, vcs_sizes* sizes, int32_t* __restrict__ cu_seqlens,
             int32_t* __restrict__ seg_traj, SegWorkspace w) {
  __shared__ int smax[32];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (gridDim.x == 1) {
    if (threadIdx.x == 0) w.totals[3] = 0;
    __syncthreads();
  }
  // ---- each trajectory: prefix sums and its segments' sizes
  const int nwarps = gridDim.x * (kScanThreads / 32);
  for (int b = blockIdx.x * (kScanThreads / 32) + warp; b < num_traj; b += nwarps) {
    const int64_t g0 = cu_steps[b], g1 = cu_steps[b + 1];
    const bool ok =
        g0 >= 0 && g1 >= g0 && g1 <= num_steps && (b > 0 || g0 == 0) && (b < num_traj - 1 || g1 == num_steps);
    long long ntok = 0, maxlen = 0, ca = 0, cb = 0;
    int nseg = 0;
    if (!ok) {
      if (lane == 0) fail(w.totals, VCS_ERR_DEVICE_CHECK);
    } else {
      for (int64_t i0 = g0; i0 < g1; i0 += 32) {
        const int64_t i = i0 + lane;
        int im = 0, tx = 0;
        if (i < g1) {
          im = step_img[i];
          tx = step_txt[i];
          if (im < 0 || tx < 0) {
            fail(w.totals, VCS_ERR_DEVICE_CHECK);
            im = im < 0 ? 0 : im;
            tx = tx < 0 ? 0 : tx;
          }
        }
        long long xa = (long long)im + tx, xb = tx;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long ya = __shfl_up_sync(0xffffffffu, xa, o), yb = __shfl_up_sync(0xffffffffu, xb, o);
          if (lane >= o) {
            xa += ya;
            xb += yb;
          }
        }
        if (i < g1) {
          w.step_inc[i] = ca + xa;
          w.txt_inc[i] = cb + xb;
        }
        ca += __shfl_sync(0xffffffffu, xa, 31);
        cb += __shfl_sync(0xffffffffu, xb, 31);
      }
      __syncwarp();
      const int T = (int)(g1 - g0);
      nseg = seg_count(T, keep, window);
      for (int j = lane; j < nseg; j += 32) {
        int a, s, e;
        seg_bounds(j, T, keep, window, a, s, e);
        const long long len = seg_len(w, g0, a, e);
        ntok += len;
        maxlen = len > maxlen ? len : maxlen;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ntok += __shfl_xor_sync(0xffffffffu, ntok, o);
        const long long y = __shfl_xor_sync(0xffffffffu, maxlen, o);
        maxlen = y > maxlen ? y : maxlen;
      }
      if (lane == 0 && maxlen > INT_MAX) fail(w.totals, VCS_ERR_OVERFLOW);
    }
    if (lane == 0) {
      w.seg_base[b] = nseg;
      w.tok_base[b] = ntok;
      w.traj_base[b] = ca;
      w.traj_maxlen[b] = (int32_t)(maxlen > INT_MAX ? INT_MAX : maxlen);
    }
  }
  if (num_traj == 0) {  // steps that belong to no trajectory are still checked
    for (int64_t i = threadIdx.x; i < num_steps; i += kScanThreads)
      if (step_img[i] < 0 || step_txt[i] < 0) fail(w.totals, VCS_ERR_DEVICE_CHECK);
  }
  // ---- one block (the last to get here): scans over the trajectories
  __threadfence();
  __syncthreads();
  if (gridDim.x > 1) {
    if (threadIdx.x == 0)
      last = atomicAdd(reinterpret_cast<unsigned long long*>(&w.totals[4]), 1ull) == gridDim.x - 1 ? 1 : 0;
    __syncthreads();
    if (!last) return;
    __threadfence();
  }
  int mx = 0;
  long long c_seg = 0, c_tok = 0, c_traj = 0;
  for (int64_t base = 0; base < num_traj; base += kScanThreads) {
    const int64_t i = base + threadIdx.x;
    const bool in = i < num_traj;
    const long long a = in ? __ldcg(&w.seg_base[i]) : 0, b = in ? __ldcg(&w.tok_base[i]) : 0;
    const long long c = in ? __ldcg(&w.traj_base[i]) : 0;
    if (in) mx = max(mx, __ldcg(&w.traj_maxlen[i]));
    long long ia = a, ib = b, ic = c, id = 0, ta, tb, tc, td;
    block_scan2(ia, ib, ta, tb);
    block_scan2(ic, id, tc, td);
    if (in) {
      w.seg_base[i] = c_seg + ia - a;
      w.tok_base[i] = c_tok + ib - b;
      w.traj_base[i] = c_traj + ic - c;
    }
    c_seg += ta;
    c_tok += tb;
    c_traj += tc;
  }
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) smax[warp] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kScanThreads / 32; ++i) mx = max(mx, smax[i]);
    w.seg_base[num_traj] = c_seg;
    w.tok_base[num_traj] = c_tok;
    if (c_tok > INT_MAX || c_traj > INT_MAX) fail(w.totals, VCS_ERR_OVERFLOW);
    if (seg_capacity >= 0 && (c_seg > seg_capacity || c_tok > tok_capacity)) fail(w.totals, VCS_ERR_CAPACITY);
    w.totals[0] = c_seg;
    w.totals[1] = c_tok;
    w.totals[2] = mx;
    const int64_t status = atomicAdd(reinterpret_cast<unsigned long long*>(&w.totals[3]), 0ull);
    sizes->num_segments = c_seg;
    sizes->num_tokens = c_tok;
    sizes->max_seqlen = mx;
    sizes->status = (int32_t)status;
    last = status == 0;
    if (BUILD && status == 0) {
      cu_seqlens[c_seg] = (int32_t)c_tok;
      w.seg_start[c_seg] = c_tok;
    }
  }
  if constexpr (BUILD) {
    __syncthreads();
    if (!last) return;
    for (int b = warp; b < num_traj; b += kScanThreads / 32) {
      const int g0 = cu_steps[b];
      write_segments(b, g0, cu_steps[b + 1] - g0, window, keep, cu_seqlens, seg_traj, w, lane);
    }
  }
}

__global__ void __launch_bounds__(256) seg_write(const int32_t* __restrict__ cu_steps, int32_t num_traj,
                                                 int32_t window, int32_t keep, int32_t* __restrict__ cu_seqlens,
                                                 int32_t* __restrict__ seg_traj, SegWorkspace w) {
  if (w.totals[3] != 0) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    cu_seqlens[w.totals[0]] = (int32_t)w.totals[1];
    w.seg_start[w.totals[0]] = w.totals[1];
  }
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= num_traj) return;
  const int g0 = cu_steps[b];
  write_segments(b, g0, cu_steps[b + 1] - g0, window, keep, cu_seqlens, seg_traj, w, threadIdx.x & 31);
}

// Largest index u in [lo, hi] with arr[u] <= x (arr non-decreasing, arr[lo] <= x).
__device__ __forceinline__ int64_t last_le(const int64_t* __restrict__ arr, int64_t lo, int64_t hi, int64_t x) {
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (__ldg(&arr[mid]) <= x)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}
// Smallest index u in [lo, hi] with inc[u] > x (inc non-decreasing, inc[hi] > x).
__device__ __forceinline__ int64_t first_gt(const int64_t* __restrict__ inc, int64_t lo, int64_t hi, int64_t x) {
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (__ldg(&inc[mid]) > x)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo;
}

// One warp per chunk of consecutive segment tokens.  A segment is a sequence of runs, one per
// step: the response tokens of each step before a_j (text-only history), then the
// screenshot-and-response tokens of each step a_j..e_j; inside a run the gather index, the position
// and the mask follow from the run's start, so the warp finds the run of its first token once (two
// binary searches, uniform across the lanes) and then streams the runs in order, the lanes writing
// 32 consecutive tokens per store.  A chunk is at most 4,096 tokens (13 bytes each, HBM-bound: 5.8
// TB/s of writes on 126 M tokens) and shrinks to 256 so that a small layout still fills the GPU
// (130 k tokens: 32 warps of 4,096 took 15 us).
constexpr int kExpandChunk = 4096, kExpandMin = 256;

__global__ void __launch_bounds__(256) seg_expand(const int32_t* __restrict__ cu_steps,
                                                  const int32_t* __restrict__ step_img,
                                                  int32_t* __restrict__ tok_gather, int32_t* __restrict__ tok_src_step,
                                                  int32_t* __restrict__ tok_pos, uint8_t* __restrict__ tok_loss_mask,
                                                  SegWorkspace w) {
  if (w.totals[3] != 0) return;
  const int64_t nseg = w.totals[0], ntok = w.totals[1];
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  int64_t chunk = (ntok / warps + kExpandMin - 1) / kExpandMin * kExpandMin;
  chunk = chunk < kExpandMin ? kExpandMin : chunk > kExpandChunk ? kExpandChunk : chunk;
  for (int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c * chunk < ntok; c += warps) {
    int64_t n = c * chunk;
    const int64_t nend = min(n + chunk, ntok);
    int64_t seg = last_le(w.seg_start, 0, nseg - 1, n);
    while (n < nend) {
      while (w.seg_start[seg + 1] <= n) ++seg;  // skip segments without tokens
      const int64_t start = w.seg_start[seg], next = w.seg_start[seg + 1];
      const int b = w.seg_traj[seg];
      const int64_t g0 = cu_steps[b], A = w.seg_full[seg], S = w.seg_new[seg], E = w.seg_last[seg];
      const int64_t tb = w.traj_base[b];  // the trajectory's first row
      const int64_t H = pre(w.txt_inc, g0, A), f0 = pre(w.step_inc, g0, A);
      // the run (step u) of position p = n - start, and its bounds [lo, hi) in the segment
      const int64_t p = n - start;
      int64_t u = p < H ? first_gt(w.txt_inc, g0, A - 1, p) : first_gt(w.step_inc, A, E, f0 + (p - H));
      const int64_t send = min(next, nend);
      while (n < send) {
        const bool hist = u < A;
        const int64_t off = pre(w.step_inc, g0, u);
        const int64_t lo = hist ? pre(w.txt_inc, g0, u) : H + (off - f0);
        const int64_t hi = hist ? w.txt_inc[u] : H + (w.step_inc[u] - f0);
        const int64_t img = step_img[u];
        // token at position q of the run's step: history tokens are the step's response
        // tokens (after its screenshot); a full step's tokens start with the screenshot
        const int64_t g_base = tb + off + (hist ? img : 0) - lo;
        const bool trainable_step = !hist && u >= S;
        const int64_t rend = min(start + hi, send);
        for (int64_t m = n + lane; m < rend; m += 32) {
          const int64_t q = m - start;
          tok_gather[m] = (int32_t)(g_base + q);
          tok_src_step[m] = (int32_t)u;
          tok_pos[m] = (int32_t)q;
          if (tok_loss_mask != nullptr) tok_loss_mask[m] = (trainable_step && q - lo >= img) ? 1 : 0;
        }
        n = max(n, rend);
        ++u;
      }
      ++seg;
    }
  }
}

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

size_t seg_workspace_bytes(int32_t num_traj, int64_t num_steps) {
  const size_t S = (size_t)num_steps, B = (size_t)num_traj;
  size_t n = 0;
  n += align256((S + 1) * 8) * 2;       // step_inc, txt_inc
  n += align256(B * 4) * 2;             // traj_maxlen; as much is reserved, so that the size stays as callers know it
  n += align256(B * 8);                 // traj_base
  n += align256((B + 1) * 8) * 2;       // seg_base, tok_base
  n += align256((S + 1) * 8);           // seg_start
  n += align256(S * 4) * 4;             // seg_full/new/last, seg_traj
  n += align256(5 * 8);                 // totals
  return n;
}

SegWorkspace seg_workspace_carve(void* ws, int32_t num_traj, int64_t num_steps) {
  const size_t S = (size_t)num_steps, B = (size_t)num_traj;
  char* p = static_cast<char*>(ws);
  auto take = [&](size_t bytes) {
    char* r = p;
    p += align256(bytes);
    return r;
  };
  SegWorkspace w;
  w.totals = reinterpret_cast<int64_t*>(take(5 * 8));
  w.step_inc = reinterpret_cast<int64_t*>(take((S + 1) * 8));
  w.txt_inc = reinterpret_cast<int64_t*>(take((S + 1) * 8));
  w.traj_maxlen = reinterpret_cast<int32_t*>(take(B * 4));
  take(B * 4);  // reserved
  w.traj_base = reinterpret_cast<int64_t*>(take(B * 8));
  w.seg_base = reinterpret_cast<int64_t*>(take((B + 1) * 8));
  w.tok_base = reinterpret_cast<int64_t*>(take((B + 1) * 8));
  w.seg_start = reinterpret_cast<int64_t*>(take((S + 1) * 8));
  w.seg_full = reinterpret_cast<int32_t*>(take(S * 4));
  w.seg_new = reinterpret_cast<int32_t*>(take(S * 4));
  w.seg_last = reinterpret_cast<int32_t*>(take(S * 4));
  w.seg_traj = reinterpret_cast<int32_t*>(take(S * 4));
  return w;
}

// One launch that plans and, up to kOneBlock trajectories, writes the segment tables; cu_seqlens
// nullptr only plans.
static cudaError_t launch_plan(const int32_t* cu_steps, int32_t num_traj, int64_t num_steps, const int32_t* step_img,
                               const int32_t* step_txt, int32_t window, int32_t keep, int64_t seg_capacity,
                               int64_t tok_capacity, vcs_sizes* sizes, int32_t* cu_seqlens, int32_t* seg_traj,
                               const SegWorkspace& w, cudaStream_t st) {
  if (num_traj <= kOneBlock) {
    if (cu_seqlens != nullptr)
      seg_plan<true><<<1, kScanThreads, 0, st>>>(cu_steps, num_traj, num_steps, step_img, step_txt, window, keep,
                                                 seg_capacity, tok_capacity, sizes, cu_seqlens, seg_traj, w);
    else
      seg_plan<false><<<1, kScanThreads, 0, st>>>(cu_steps, num_traj, num_steps, step_img, step_txt, window, keep,
                                                  seg_capacity, tok_capacity, sizes, nullptr, nullptr, w);
    return cudaGetLastError();
  }
  // status and the count of finished blocks
  const cudaError_t e = cudaMemsetAsync(w.totals, 0, 5 * sizeof(int64_t), st);
  if (e != cudaSuccess) return e;
  const int nb = (num_traj + 31) / 32 < 152 ? (num_traj + 31) / 32 : 152;
  seg_plan<false><<<nb, kScanThreads, 0, st>>>(cu_steps, num_traj, num_steps, step_img, step_txt, window, keep,
                                               seg_capacity, tok_capacity, sizes, nullptr, nullptr, w);
  return cudaGetLastError();
}

cudaError_t launch_seg_plan(const int32_t* cu_steps, int32_t num_traj, int64_t num_steps, const int32_t* step_img,
                            const int32_t* step_txt, int32_t window, int32_t keep, vcs_sizes* sizes,
                            const SegWorkspace& w, cudaStream_t st) {
  return launch_plan(cu_steps, num_traj, num_steps, step_img, step_txt, window, keep, -1, -1, sizes, nullptr, nullptr,
                     w, st);
}

cudaError_t launch_seg_build(const int32_t* cu_steps, int32_t num_traj, int64_t num_steps, const int32_t* step_img,
                             const int32_t* step_txt, int32_t window, int32_t keep, int64_t seg_capacity,
                             int64_t tok_capacity, int32_t* cu_seqlens, int32_t* seg_traj, int32_t* tok_gather,
                             int32_t* tok_src_step, int32_t* tok_pos, uint8_t* tok_loss_mask, vcs_sizes* sizes,
                             const SegWorkspace& w, cudaStream_t st) {
  const cudaError_t e = launch_plan(cu_steps, num_traj, num_steps, step_img, step_txt, window, keep, seg_capacity,
                                    tok_capacity, sizes, cu_seqlens, seg_traj, w, st);
  if (e != cudaSuccess) return e;
  if (num_traj > kOneBlock)
    seg_write<<<(num_traj + 7) / 8, 256, 0, st>>>(cu_steps, num_traj, window, keep, cu_seqlens, seg_traj, w);
  // a warp per 256 tokens of the capacity, at most 16 blocks an SM
  int64_t blocks = (tok_capacity + 8 * kExpandMin - 1) / (8 * kExpandMin);
  blocks = blocks < 1 ? 1 : blocks > 152 * 16 ? 152 * 16 : blocks;
  seg_expand<<<(unsigned)blocks, 256, 0, st>>>(cu_steps, step_img, tok_gather, tok_src_step, tok_pos, tok_loss_mask, w);
  return cudaGetLastError();
}

}  // namespace vcs
