// gather.cu - packed segment rows from trajectory rows.
//
// After a prune, Algorithm 1 (Sec. 3.4) re-tokenises the retained history into
// a fresh stream: every segment token is a token of its trajectory, so the
// packed Q/K/V of a segment are rows of the trajectory-layout tensors at the
// builder's gather map.  The copy is HBM-bound: every 16-byte chunk of every
// destination row is read once and written once, with consecutive threads on
// consecutive chunks (coalesced on both sides whenever consecutive segment
// tokens map to consecutive trajectory tokens, which is the common case).
#include <cstdint>

#include "internal.h"
#include "sm100.cuh"

namespace vcs {
namespace {

constexpr int kThreads = 256;
constexpr int kUnroll = 4;

__device__ __forceinline__ int4 ld_stream(const int4* p) {
  int4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}
__device__ __forceinline__ void st_stream(int4* p, int4 v) {
  asm volatile("st.global.cs.v4.s32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

// Copies chunks lane, lane + 32, ... of a row, kUnroll loads in flight per lane.
template <typename Chunk>
__device__ __forceinline__ void copy_row(const int4* __restrict__ src, int4* __restrict__ dst, Chunk chunks, int lane) {
  Chunk c = lane;
  for (; c + 32 * (kUnroll - 1) < chunks; c += 32 * kUnroll) {
    int4 v[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) v[u] = ld_stream(src + c + 32 * u);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) st_stream(dst + c + 32 * u, v[u]);
  }
  for (; c < chunks; c += 32) st_stream(dst + c, ld_stream(src + c));
}

// One warp per segment token, for rows of at least kNarrow chunks: its Q, K and V rows in one launch.
// The token's index is loaded a token ahead; per row there is no division and one address each (a
// chunk-per-thread form with a 64-bit division per chunk, launched once per tensor, took 1.19 ms for
// the 3.5 GB of a long-horizon rollout, this form 1.06: 6.7 TB/s read and written; 8 loads in flight a
// lane 1.12).  Chunk: int, or int64_t for rows of 2^30 chunks and more (1.2 M tokens at 8/2/128 take
// 1,200 us with it, 1,116 with int).
template <typename Chunk>
__global__ void __launch_bounds__(kThreads)
    gather_rows(const int4* __restrict__ q_src, const int4* __restrict__ k_src, const int4* __restrict__ v_src,
                int64_t traj_tokens, const int32_t* __restrict__ tok_gather, int64_t num_tokens, Chunk q_chunks,
                Chunk kv_chunks, int4* __restrict__ q, int4* __restrict__ k, int4* __restrict__ v, int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kThreads / 32);
  int64_t n = blockIdx.x * (int64_t)(kThreads / 32) + (threadIdx.x >> 5);
  int32_t next = n < num_tokens ? __ldg(&tok_gather[n]) : 0;
  for (; n < num_tokens; n += warps) {
    const int64_t s = next;
    if (n + warps < num_tokens) next = __ldg(&tok_gather[n + warps]);
    if (s < 0 || s >= traj_tokens) {
      if (lane == 0) dev::set_status(status, VCS_ERR_DEVICE_CHECK);
      continue;
    }
    copy_row(q_src + s * q_chunks, q + n * q_chunks, q_chunks, lane);
    if (kv_chunks > 0) {
      copy_row(k_src + s * kv_chunks, k + n * kv_chunks, kv_chunks, lane);
      copy_row(v_src + s * kv_chunks, v + n * kv_chunks, kv_chunks, lane);
    }
  }
}

// Rows of fewer than kNarrow chunks: a warp takes `per_warp` tokens, lane t holding token t's index, and
// copies them tensor by tensor as one run of chunks of the destination, 32 a step, so that every lane
// has a chunk whatever the row's width and kUnroll steps, of any of the three tensors, are in flight.
// 1.2 M tokens, us, for a chunk a thread with a launch a tensor / a warp a token / this form: heads 1/1 of
// 8 dims 34.8 / 393 / 28.7, 1/1/64 190 / 446 / 170, 14/2/64 1,001 / 1,114 / 971.  From kNarrow chunks on a
// warp a token is the faster (8/2/128: 1,364 / 1,116 / 1,288; 28/4/128: 3,829 / 3,331 / 3,762).
constexpr int kNarrow = 128;
// chunk f of a run of rows of c chunks lies in row f * (2^24 / c + 1) >> 24, exactly for f < 2^24 / c
constexpr int kMagicShift = 24;
static_assert((32 * kNarrow + 32) * kNarrow <= 1 << kMagicShift, "row of a chunk");

template <int UNROLL>
__global__ void __launch_bounds__(kThreads)
    gather_narrow(const int4* __restrict__ q_src, const int4* __restrict__ k_src, const int4* __restrict__ v_src,
                  int64_t traj_tokens, const int32_t* __restrict__ tok_gather, int64_t num_tokens, int q_chunks,
                  int kv_chunks, uint32_t q_magic, uint32_t kv_magic, int per_warp, int4* __restrict__ q,
                  int4* __restrict__ k, int4* __restrict__ v, int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * (kThreads / 32) * per_warp;
  int64_t n0 = (blockIdx.x * (int64_t)(kThreads / 32) + (threadIdx.x >> 5)) * per_warp;
  for (; n0 < num_tokens; n0 += stride) {
    const int m = (int)(num_tokens - n0 < per_warp ? num_tokens - n0 : per_warp);
    int row = lane < m ? __ldg(&tok_gather[n0 + lane]) : -1;  // source row of token n0 + lane, -1: none
    if (lane < m && (row < 0 || row >= traj_tokens)) {
      dev::set_status(status, VCS_ERR_DEVICE_CHECK);
      row = -1;
    }
    const int q_steps = (m * q_chunks + 31) / 32, kv_steps = (m * kv_chunks + 31) / 32;
    const int steps = q_steps + 2 * kv_steps;
    for (int i = 0; i < steps; i += UNROLL) {
      int4 x[UNROLL];
      int4* to[UNROLL];
      bool live[UNROLL];
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        const bool is_q = i + u < q_steps, is_v = i + u >= q_steps + kv_steps;
        const int c = is_q ? q_chunks : kv_chunks;
        const uint32_t f = 32 * (i + u - (is_q ? 0 : is_v ? q_steps + kv_steps : q_steps)) + lane;
        const uint32_t t = f * (is_q ? q_magic : kv_magic) >> kMagicShift;
        const int s = __shfl_sync(0xffffffffu, row, t & 31);
        live[u] = i + u < steps && f < (uint32_t)(m * c) && s >= 0;
        to[u] = (is_q ? q : is_v ? v : k) + n0 * c + f;
        if (live[u]) x[u] = ld_stream((is_q ? q_src : is_v ? v_src : k_src) + (int64_t)s * c + (f - t * c));
      }
#pragma unroll
      for (int u = 0; u < UNROLL; ++u)
        if (live[u]) st_stream(to[u], x[u]);
    }
  }
}

}  // namespace

cudaError_t launch_gather(const void* q_src, const void* k_src, const void* v_src, int64_t traj_tokens,
                          const int32_t* tok_gather, int64_t num_tokens, int64_t q_row_bytes, int64_t kv_row_bytes,
                          void* q, void* k, void* v, int32_t* dev_status, cudaStream_t st) {
  if (num_tokens == 0) return cudaSuccess;
  const int64_t cap = 152 * 16;
  const int64_t q_chunks = q_row_bytes / 16, kv_chunks = kv_row_bytes / 16;
  if (q_chunks < kNarrow && kv_chunks < kNarrow) {
    // At most 32 tokens a warp, and as many as divide the tokens evenly over whole passes of the 32 warps an
    // SM holds (174,000 tokens at 4/4/64: 102 us, 127 with 32 a warp, which leave a second pass nearly
    // empty; 111 for a chunk a thread), in fours where they are many, whose chunks fill whole steps more
    // often, but no fewer than fill a step.
    const int64_t slots = 152 * 32, passes = (num_tokens + slots * 32 - 1) / (slots * 32);
    int64_t per_warp = (num_tokens + slots * passes - 1) / (slots * passes);
    if (per_warp > 16) per_warp = (per_warp + 3) / 4 * 4;
    if (per_warp * q_chunks < 32) per_warp = (31 + q_chunks) / q_chunks;
    if (per_warp > 32) per_warp = 32;
    const bool few_steps = q_chunks + 2 * kv_chunks < kUnroll;
    int64_t blocks = ((num_tokens + per_warp - 1) / per_warp + kThreads / 32 - 1) / (kThreads / 32);
    if (few_steps && blocks > cap) blocks = cap;
    auto magic = [](int64_t c) { return c > 0 ? (1u << kMagicShift) / (uint32_t)c + 1 : 0u; };
    // of a few steps a pass none waits for another, and more warps fit (Q alone, a chunk a row: 20.5 -> 16.4 us)
    const auto kernel = few_steps ? gather_narrow<1> : gather_narrow<kUnroll>;
    kernel<<<(unsigned)blocks, kThreads, 0, st>>>(
        static_cast<const int4*>(q_src), static_cast<const int4*>(k_src), static_cast<const int4*>(v_src), traj_tokens,
        tok_gather, num_tokens, (int)q_chunks, (int)kv_chunks, magic(q_chunks), magic(kv_chunks), (int)per_warp,
        static_cast<int4*>(q), static_cast<int4*>(k), static_cast<int4*>(v), dev_status);
    return cudaGetLastError();
  }
  int64_t blocks = (num_tokens + kThreads / 32 - 1) / (kThreads / 32);
  if (blocks > cap) blocks = cap;
  auto launch = [&](auto kernel, auto qc, auto kvc) {
    kernel<<<(unsigned)blocks, kThreads, 0, st>>>(
        static_cast<const int4*>(q_src), static_cast<const int4*>(k_src), static_cast<const int4*>(v_src), traj_tokens,
        tok_gather, num_tokens, qc, kvc, static_cast<int4*>(q), static_cast<int4*>(k), static_cast<int4*>(v),
        dev_status);
  };
  if (q_chunks < 1 << 30 && kv_chunks < 1 << 30)
    launch(gather_rows<int>, (int)q_chunks, (int)kv_chunks);
  else
    launch(gather_rows<int64_t>, q_chunks, kv_chunks);
  return cudaGetLastError();
}

}  // namespace vcs
