// stream.cu - Algorithm 1's token-ID stream fields over the segment layout
// (App. C.1) and the ordered list of trainable tokens, sm_103a.
//
//   ids[n]  = traj_ids[tok_gather[n]]
//   logp[n] = tok_loss_mask[n] ? traj_logp[tok_gather[n]] : 0
// (trainable response tokens keep their rollout log-probability; observation
// tokens and the re-tokenised history of a fresh stream carry 0), and
//   idx = the n with tok_loss_mask[n] = 1, in increasing order.
//
// Both are HBM-bound on large streams and launch-bound on small ones.  The stream fields
// take four tokens a thread where the buffers' alignment allows it.  The compaction is two
// launches (2.0 M tokens: 14.0 us against 30.3 for a byte a thread, a scan launch and a block scan
// per 256 tokens): per-chunk counts of 4,096 mask bytes (16 a thread), then per chunk the sum of the
// counts before it, one block scan and the indices in order; above kSumChunks chunks, where
// summing the counts per chunk would be quadratic, a launch between them scans the counts.
#include <cstdint>

#include "internal.h"

namespace vcs {
namespace {

constexpr int kThreads = 256;
constexpr int kChunk = kThreads * 16;  // tokens per compaction block
// Chunks up to which each block sums the counts before it: 4,096 chunks (16.8 M tokens) are at most
// 16 loads a thread, about what the scan's launch costs.
constexpr int64_t kSumChunks = 4096;

__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  if (status != nullptr) atomicCAS(status, 0, code);
}

__global__ void __launch_bounds__(kThreads) stream_fields_kernel(const int32_t* __restrict__ traj_ids,
                                                                 const float* __restrict__ traj_logp,
                                                                 int64_t traj_tokens,
                                                                 const int32_t* __restrict__ tok_gather,
                                                                 const uint8_t* __restrict__ mask, int64_t num_tokens,
                                                                 int32_t* __restrict__ ids, float* __restrict__ logp,
                                                                 int32_t* status) {
  for (int64_t n = blockIdx.x * (int64_t)kThreads + threadIdx.x; n < num_tokens; n += (int64_t)gridDim.x * kThreads) {
    const int32_t g = __ldg(&tok_gather[n]);
    if (g < 0 || g >= traj_tokens) {
      set_status(status, VCS_ERR_DEVICE_CHECK);
      ids[n] = 0;
      logp[n] = 0.f;
      continue;
    }
    ids[n] = __ldg(&traj_ids[g]);
    logp[n] = __ldg(&mask[n]) != 0 ? __ldg(&traj_logp[g]) : 0.f;
  }
}

// Four consecutive tokens a thread: the gather index, mask, ids and log-probabilities in one access
// each (16-byte aligned buffers, 4-byte aligned mask).  2.0 M tokens, L2 flushed, events around the
// call: 13.1 us against 17.0 for a token a thread.
__global__ void __launch_bounds__(kThreads) stream_fields_kernel4(const int32_t* __restrict__ traj_ids,
                                                                  const float* __restrict__ traj_logp,
                                                                  int64_t traj_tokens,
                                                                  const int32_t* __restrict__ tok_gather,
                                                                  const uint8_t* __restrict__ mask, int64_t num_tokens,
                                                                  int32_t* __restrict__ ids, float* __restrict__ logp,
                                                                  int32_t* status) {
  const int64_t quads = num_tokens / 4;
  const int64_t i0 = blockIdx.x * (int64_t)kThreads + threadIdx.x, stride = (int64_t)gridDim.x * kThreads;
  for (int64_t i = i0; i < quads; i += stride) {
    const int4 g4 = __ldg(reinterpret_cast<const int4*>(tok_gather) + i);
    const uint32_t m4 = __ldg(reinterpret_cast<const uint32_t*>(mask) + i);
    const int32_t g[4] = {g4.x, g4.y, g4.z, g4.w};
    int32_t id[4];
    float lp[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool ok = g[u] >= 0 && g[u] < traj_tokens;
      if (!ok) set_status(status, VCS_ERR_DEVICE_CHECK);
      id[u] = ok ? __ldg(&traj_ids[g[u]]) : 0;
      lp[u] = ok && ((m4 >> (8 * u)) & 0xffu) != 0 ? __ldg(&traj_logp[g[u]]) : 0.f;
    }
    reinterpret_cast<int4*>(ids)[i] = make_int4(id[0], id[1], id[2], id[3]);
    reinterpret_cast<float4*>(logp)[i] = make_float4(lp[0], lp[1], lp[2], lp[3]);
  }
  const int64_t n = 4 * quads + i0;  // the last 1 .. 3 tokens
  if (i0 < num_tokens - 4 * quads) {
    const int32_t g = __ldg(&tok_gather[n]);
    const bool ok = g >= 0 && g < traj_tokens;
    if (!ok) set_status(status, VCS_ERR_DEVICE_CHECK);
    ids[n] = ok ? __ldg(&traj_ids[g]) : 0;
    logp[n] = ok && __ldg(&mask[n]) != 0 ? __ldg(&traj_logp[g]) : 0.f;
  }
}

// Bit u set when mask byte n0 + u is not zero (0 past num_tokens), n0 a multiple of 16; VEC: the mask
// is 16-byte aligned.
template <bool VEC>
__device__ __forceinline__ uint32_t mask_bits16(const uint8_t* __restrict__ mask, int64_t n0, int64_t num_tokens) {
  uint32_t bits = 0;
  if (VEC && n0 + 16 <= num_tokens) {
    const uint4 m = __ldg(reinterpret_cast<const uint4*>(mask + n0));
    const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t ones = __vminu4(w[i], 0x01010101u);         // 1 per non-zero byte
      bits |= ((ones * 0x01020408u) >> 24 & 0xfu) << (4 * i);  // byte u of the word to bit u
    }
  } else {
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (n0 + u < num_tokens && __ldg(&mask[n0 + u]) != 0) bits |= 1u << u;
  }
  return bits;
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads) compact_count(const uint8_t* __restrict__ mask, int64_t num_tokens,
                                                          int64_t* __restrict__ counts, int32_t* status) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *status = VCS_OK;  // compact_write reports into it
  int c = __popc(mask_bits16<VEC>(mask, blockIdx.x * (int64_t)kChunk + 16 * threadIdx.x, num_tokens));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) c += __shfl_down_sync(0xffffffffu, c, off);
  __shared__ int red[kThreads / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < kThreads / 32; ++w) s += red[w];
    counts[blockIdx.x] = s;
  }
}

// exclusive scan of the chunk counts in place (one block); total -> *count
__global__ void __launch_bounds__(kThreads) compact_scan(int64_t* __restrict__ counts, int nchunks,
                                                         int64_t* __restrict__ count) {
  __shared__ int64_t carry;
  __shared__ int64_t warp_sum[kThreads / 32];
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nchunks; base += kThreads) {
    const int i = base + threadIdx.x;
    const int64_t v = i < nchunks ? counts[i] : 0;
    int64_t x = v;  // inclusive scan within the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, x, off);
      if ((threadIdx.x & 31) >= off) x += y;
    }
    if ((threadIdx.x & 31) == 31) warp_sum[threadIdx.x >> 5] = x;
    __syncthreads();
    int64_t before = carry;
    for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += warp_sum[w];
    if (i < nchunks) counts[i] = before + x - v;
    __syncthreads();
    if (threadIdx.x == kThreads - 1) carry = before + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) *count = carry;
}

// SCANNED: counts hold the chunks' offsets (compact_scan); otherwise the chunk counts, which the
// block sums up to its own, and the last block writes *count.
template <bool VEC, bool SCANNED>
__global__ void __launch_bounds__(kThreads) compact_write(const uint8_t* __restrict__ mask, int64_t num_tokens,
                                                          const int64_t* __restrict__ counts,
                                                          int32_t* __restrict__ idx, int64_t capacity,
                                                          int64_t* __restrict__ count, int32_t* status) {
  __shared__ int64_t before[kThreads / 32];
  __shared__ int warp_cnt[kThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n0 = blockIdx.x * (int64_t)kChunk + 16 * threadIdx.x;
  uint32_t bits = mask_bits16<VEC>(mask, n0, num_tokens);
  const int mine = __popc(bits);
  int64_t sum = 0;
  if (!SCANNED)
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kThreads) sum += counts[i];
  int x = mine;  // inclusive scan within the warp
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
    if (!SCANNED) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  }
  if (lane == 31) warp_cnt[warp] = x;
  if (lane == 0) before[warp] = sum;
  __syncthreads();
  int64_t out = SCANNED ? counts[blockIdx.x] : 0;
  int total = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) {
    if (!SCANNED) out += before[w];
    if (w < warp) out += warp_cnt[w];
    total += warp_cnt[w];
  }
  if (!SCANNED && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *count = out + total;  // warp 0: out is the chunk's offset
  out += x - mine;
  bool over = false;
  while (bits != 0) {
    const int u = __ffs(bits) - 1;
    bits &= bits - 1;
    if (out < capacity) idx[out] = (int32_t)(n0 + u);
    else over = true;
    ++out;
  }
  if (over) set_status(status, VCS_ERR_CAPACITY);
}

}  // namespace

cudaError_t launch_stream_fields(const int32_t* traj_ids, const float* traj_logp, int64_t traj_tokens,
                                 const int32_t* tok_gather, const uint8_t* mask, int64_t num_tokens, int32_t* ids,
                                 float* logp, int32_t* status, cudaStream_t st) {
  if (num_tokens == 0) return cudaSuccess;
  const bool vec = ((reinterpret_cast<uintptr_t>(tok_gather) | reinterpret_cast<uintptr_t>(ids) |
                     reinterpret_cast<uintptr_t>(logp)) & 15u) == 0 &&
                   (reinterpret_cast<uintptr_t>(mask) & 3u) == 0;
  const int64_t threads = vec ? (num_tokens + 3) / 4 : num_tokens;
  int64_t blocks = (threads + kThreads - 1) / kThreads;
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (vec)
    stream_fields_kernel4<<<(unsigned)blocks, kThreads, 0, st>>>(traj_ids, traj_logp, traj_tokens, tok_gather, mask,
                                                                 num_tokens, ids, logp, status);
  else
    stream_fields_kernel<<<(unsigned)blocks, kThreads, 0, st>>>(traj_ids, traj_logp, traj_tokens, tok_gather, mask,
                                                                num_tokens, ids, logp, status);
  return cudaGetLastError();
}

size_t compact_ws_bytes(int64_t num_tokens) {
  const int64_t nchunks = (num_tokens + kChunk - 1) / kChunk;
  return kWsHeader + (size_t)(nchunks > 0 ? nchunks : 1) * sizeof(int64_t);
}

cudaError_t launch_compact(const uint8_t* mask, int64_t num_tokens, int32_t* idx, int64_t capacity, int64_t* count,
                           void* ws, cudaStream_t st) {
  int32_t* status = static_cast<int32_t*>(ws);
  int64_t* counts = reinterpret_cast<int64_t*>(static_cast<char*>(ws) + kWsHeader);
  const int64_t nchunks = (num_tokens + kChunk - 1) / kChunk;
  if (nchunks == 0) {
    if (cudaMemsetAsync(status, 0, sizeof(int32_t), st) != cudaSuccess) return cudaErrorUnknown;
    return cudaMemsetAsync(count, 0, sizeof(int64_t), st);
  }
  const bool vec = (reinterpret_cast<uintptr_t>(mask) & 15u) == 0;
  const bool scanned = nchunks > kSumChunks;
  const unsigned nb = (unsigned)nchunks;
  (vec ? compact_count<true> : compact_count<false>)<<<nb, kThreads, 0, st>>>(mask, num_tokens, counts, status);
  if (scanned) compact_scan<<<1, kThreads, 0, st>>>(counts, (int)nchunks, count);
  (vec ? (scanned ? compact_write<true, true> : compact_write<true, false>)
       : (scanned ? compact_write<false, true> : compact_write<false, false>))<<<nb, kThreads, 0, st>>>(
      mask, num_tokens, counts, idx, capacity, count, status);
  return cudaGetLastError();
}

}  // namespace vcs
