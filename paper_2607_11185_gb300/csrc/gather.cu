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
__device__ __forceinline__ void copy_row(const int4* __restrict__ src, int4* __restrict__ dst, int chunks, int lane) {
  int c = lane;
  for (; c + 32 * (kUnroll - 1) < chunks; c += 32 * kUnroll) {
    int4 v[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) v[u] = ld_stream(src + c + 32 * u);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) st_stream(dst + c + 32 * u, v[u]);
  }
  for (; c < chunks; c += 32) st_stream(dst + c, ld_stream(src + c));
}

// One warp per segment token: its Q, K and V rows in one launch.  The token's index is loaded a token
// ahead; per row there is no division and one address each (a chunk-per-thread form with a 64-bit
// division per chunk, launched once per tensor, took 1.19 ms for the 3.5 GB of a long-horizon rollout,
// this form 1.06: 6.7 TB/s read and written; 8 loads in flight a lane 1.12).
__global__ void __launch_bounds__(kThreads)
    gather_rows(const int4* __restrict__ q_src, const int4* __restrict__ k_src, const int4* __restrict__ v_src,
                int64_t traj_tokens, const int32_t* __restrict__ tok_gather, int64_t num_tokens, int q_chunks,
                int kv_chunks, int4* __restrict__ q, int4* __restrict__ k, int4* __restrict__ v, int32_t* status) {
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

}  // namespace

cudaError_t launch_gather(const void* q_src, const void* k_src, const void* v_src, int64_t traj_tokens,
                          const int32_t* tok_gather, int64_t num_tokens, int64_t q_row_bytes, int64_t kv_row_bytes,
                          void* q, void* k, void* v, int32_t* dev_status, cudaStream_t st) {
  if (num_tokens == 0) return cudaSuccess;
  if (q_row_bytes / 16 > INT32_MAX || kv_row_bytes / 16 > INT32_MAX) return cudaErrorInvalidValue;
  int64_t blocks = (num_tokens + kThreads / 32 - 1) / (kThreads / 32);
  const int64_t cap = 152 * 16;
  if (blocks > cap) blocks = cap;
  gather_rows<<<(unsigned)blocks, kThreads, 0, st>>>(
      static_cast<const int4*>(q_src), static_cast<const int4*>(k_src), static_cast<const int4*>(v_src), traj_tokens,
      tok_gather, num_tokens, (int)(q_row_bytes / 16), (int)(kv_row_bytes / 16), static_cast<int4*>(q),
      static_cast<int4*>(k), static_cast<int4*>(v), dev_status);
  return cudaGetLastError();
}

}  // namespace vcs
