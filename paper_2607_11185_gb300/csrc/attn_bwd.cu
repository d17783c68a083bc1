// attn_bwd.cu - backward of the packed-segment causal GQA attention, sm_103a.
//
// For an upstream gradient dO of o_i = sum_j P_ij v_j (P the causal softmax of
// s_ij = scale <q_i, k_j> within one segment):
//   D_i   = <dO_i, o_i>
//   dP_ij = <dO_i, v_j>,   dS_ij = P_ij (dP_ij - D_i)
//   dq_i  = scale sum_j dS_ij k_j
//   dk_j  = scale sum_{h in group} sum_i dS_ij q_i
//   dv_j  = sum_{h in group} sum_i P_ij dO_i
// P is recomputed from the forward's log-sum-exp: P_ij = exp(s_ij - lse_i).
//
// Three kernels on the caller's stream:
//   bwd_pre     D = rowsum(dO * O) (fp32, [hq, N]) and zeroes the fp32 dQ accumulator
//   bwd_main    one CTA per (segment, 128-key tile n, kv-head g); loops over the
//               G query heads of the group and the query tiles m >= n.  dK and
//               dV of the tile accumulate in TMEM across the whole loop (GQA head
//               sharing: the K/V tile is loaded once for all G heads); the dQ
//               contribution of every (m, h) is added to the fp32 accumulator
//               with reductions.
//   bwd_dq_cvt  fp32 dQ accumulator -> bf16 dq
// Gathered: the accumulators of dQ, dK and dV are in trajectory layout (zeroed by a memset),
// bwd_main adds to them at the tokens' trajectory rows, and bwd_dq_cvt converts all three.
#include <cfloat>
#include <cstdint>

#include "internal.h"
#include "sm100.cuh"

namespace vcs {
namespace {

using namespace dev;

constexpr int kPreThreads = 256;

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// ------------------------------------------------------------------ bwd_pre
// One 16-byte chunk (8 elements) per thread; D/8 consecutive threads share a row.  dq_acc
// nullptr (gathered: its accumulator is in trajectory layout) zeroes nothing.
template <int D>
__global__ void __launch_bounds__(kPreThreads) bwd_pre(const __nv_bfloat16* __restrict__ o,
                                                       const __nv_bfloat16* __restrict__ dout, int64_t rows,
                                                       int32_t hq, int64_t num_tokens, float* __restrict__ dvec,
                                                       float* __restrict__ dq_acc, int32_t* status) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *status = VCS_OK;  // the call's first kernel
  constexpr int CPR = D / 8;  // chunks per row
  const int64_t total = rows * CPR;
  for (int64_t c = blockIdx.x * (int64_t)kPreThreads + threadIdx.x; c - threadIdx.x < total;
       c += (int64_t)gridDim.x * kPreThreads) {
    float acc = 0.f;
    if (c < total) {
      const uint4 a = __ldg(reinterpret_cast<const uint4*>(o) + c);
      const uint4 b = __ldg(reinterpret_cast<const uint4*>(dout) + c);
      const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 fa = __bfloat1622float2(pa[e]);
        const float2 fb = __bfloat1622float2(pb[e]);
        acc = fmaf(fa.x, fb.x, acc);
        acc = fmaf(fa.y, fb.y, acc);
      }
      if (dq_acc != nullptr) {
        float4* z = reinterpret_cast<float4*>(dq_acc) + 2 * c;
        z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int off = CPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (c < total && (c % CPR) == 0) {
      const int64_t row = c / CPR;           // row = token * hq + head
      const int64_t tok = row / hq;
      const int64_t h = row - tok * hq;
      dvec[h * num_tokens + tok] = acc;
    }
  }
}

// ------------------------------------------------------------------ bwd_dq_cvt
__global__ void __launch_bounds__(256) bwd_dq_cvt(const float* __restrict__ acc, __nv_bfloat16* __restrict__ dq,
                                                  int64_t n8) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n8; c += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(acc) + 2 * c);
    const float4 b = __ldg(reinterpret_cast<const float4*>(acc) + 2 * c + 1);
    uint4 r;
    r.x = pack_bf16(a.x, a.y);
    r.y = pack_bf16(a.z, a.w);
    r.z = pack_bf16(b.x, b.y);
    r.w = pack_bf16(b.z, b.w);
    reinterpret_cast<uint4*>(dq)[c] = r;
  }
}

// ------------------------------------------------------------------ bwd_main
// One CTA: key tile n of a (segment, kv head); tile u of its loop is one 128-row query tile of
// one head of the group.  Two chains of dependent steps alternate on the tensor pipe, so that
// each one's MMAs run under the other's arithmetic:
//   S^T(u) -> P^T(u) (compute warps) -> dV += P^T dO
//   dP^T(u) -> dS^T(u) (compute warps) -> dK += dS^T Q, dQ(u) -> drain
// Two warps issue MMAs, one for each chain, so that a barrier wait of one (about 250 cycles while the
// pipe streams from shared memory) is covered by the other's MMAs.
// d = 128: the order on the pipe is dP^T(u), dV(u), S^T(u+1), dK(u), dQ(u): dP^T(u) follows the
// drain's read of dQ(u-1), whose columns it overwrites, dV(u) and S^T(u+1) run while dS^T(u) is
// computed, and P^T(u+1) is computed while dK(u), dQ(u) and that read run.
// What bounds it is the shared-memory pipe: per tile at d = 128 the MMAs read 256 KB (2,048 cycles
// at 128 B/clk), TMA writes 64 KB (512), dS^T and the row terms take 512 and the dQ reductions about
// 990 (measured against a stream of shared loads).  Before, S^T and dP^T were issued together, one
// pass of the compute warps made P^T and dS^T of both, and dQ left through shared memory by TMA
// reduce-adds, whose engine also carries the tile loads (64 KB at 25.5 B/clk + 64 KB at 62 B/clk).
// vcs_attn_bwd, 40/8/128, four segments of 8,192: 6.18 ms before, 5.31 now (892 -> 1,035 TFLOP/s
// credited).
// d = 64: the MMAs need about 1,400 cycles a tile; the compute warps' two passes (about 1,000 and
// 1,100, mostly latencies of one warp's chain: neither leaving out the reductions nor the stores of
// dS^T shortens them) bound it, so everything they wait for is issued a step ahead: TMEM has room
// for dQ and P^T in columns of their own, so S^T(u+1) is issued when S^T(u) has been read, not when
// dV(u) has, and dP^T(u+1) right behind dK(u), not behind the drain's read.  14/2/64, sixteen of
// 4,096: 3.89 ms for the serial loop with 16-byte reductions of 32 different rows that was here
// first, 1.42 for the order of d = 128, 1.35 with dP^T ahead, 1.29 with S^T ahead too, 1.27 with the
// drain's pace set again, 1.26 now (247 -> 767 TFLOP/s credited).
//   WG0   warp 0: TMA producer (K and V once, NST tiles of Q and dO in flight)
//         warp 1: TMEM allocation, MMAs of S^T and dV;  warp 2: MMAs of dP^T, dK and dQ;  warp 3: row terms
//         (both run warp-uniformly up to an elected lane's issue, which keeps descriptors in uniform
//         registers: 7.6 -> 6.7 ms on the case above while it was being built)
//   WG1/2 compute: warpgroup k takes query columns [32k, 32k+32) of each half of the tile (so that the
//         halves' K steps, and with them dK's sum, run in order), a thread one key row.  P^T stays
//         in fp32 registers between its two passes; its bf16 copy goes to TMEM (the A operand of
//         dV += P^T dO), dS^T over the dP^T columns the thread has read (A of dK += dS^T Q) and to
//         shared memory (for dQ)
//   WG3   dQ drain: TMEM -> registers -> fp32 reductions into the accumulator.  An SM sends 32 B a
//         clock to L2 and a 128-byte line costs a fifth flit, so 25.5 B/clk (2,570 cycles for
//         64 KB) is the ceiling for TMA bulk reduce-adds and register reductions alike, if a warp's
//         reduction covers whole lines (16-byte pieces of 32 rows: 11-16 B/clk).  d = 128: the
//         product is taken transposed, dQ^T = K^T dS, so that a warp holds 32 consecutive head
//         dims of one query and a scalar reduction is one line.  d = 64 (M = 64 would halve the
//         rate): dQ = dS^T K, and two rounds of lane exchanges make 8 lanes hold a 128-byte row
//         piece.
// TMEM (512 columns): dV, dK (D each), S^T (128), dP^T/dS^T (128).  d = 128: P^T goes over the S^T
// columns and dQ over the dP^T columns (dK(u) reads dS^T there first, in pipe order).  d = 64: dQ
// and P^T have 64 columns each.
// Pipe order: the MMAs one thread issues are taken to execute in issue order.  PTX states that for MMAs
// of one shape on one accumulator; here it is relied on where an MMA overwrites the TMEM operand of the
// one before it, across accumulators and, at d = 64, across shapes: S^T(u+1) over the P^T that dV(u)
// reads and dQ(u) over the dS^T that dK(u) reads (d = 128, all N = 128), dP^T(u+1) (N = 128) over the
// dS^T that dK(u) (N = 64) reads (d = 64).  No completed barrier stands between them; the comparisons
// with the oracle are what shows a violation.

// TMEM loads / stores of N consecutive 32-bit columns of the warp's 32 lanes.
template <int N>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[N]) {
  static_assert(N == 16 || N == 32, "16 or 32 columns");
  if constexpr (N == 32) tmem_ld_32x32b_x32(taddr, r);
  else tmem_ld_32x32b_x16(taddr, r);
}

__device__ __forceinline__ void red_add(float* p, float a) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(a) : "memory");
}

template <int D>
struct Bwd {
  static constexpr int BM = 128;                 // key rows of the tile
  static constexpr int BQ = 128;                 // query rows per tile
  static constexpr int KB = D / 64;              // 64-column blocks of a row
  static constexpr int NST = D == 128 ? 2 : 4;   // Q/dO pairs in flight (227 KB leaves two at d = 128)
  static constexpr int THREADS = 512;
  static constexpr int TILE = 128 * D * 2;
  static constexpr int BLOCK = 128 * 128;        // one 64-column block of a 128-row tile
  static constexpr int OFF_K = 0;
  static constexpr int OFF_V = TILE;
  static constexpr int OFF_QD = 2 * TILE;
  static constexpr int OFF_DS = OFF_QD + 2 * NST * TILE;  // dS^T [128 keys][128 queries], two 64-query blocks
  static constexpr int NDS = D == 128 ? 1 : 2;              // buffers of dS^T, by tile parity
  static constexpr int OFF_ROW = OFF_DS + NDS * 2 * BLOCK;  // [tile parity][WG k]: -lse*log2e of 64 queries, -D (* scale)
  static constexpr int OFF_BAR = OFF_ROW + 2 * 2 * 128 * 4;
  static constexpr int BAR_BYTES = 512;
  static constexpr int SMEM = OFF_BAR + BAR_BYTES;
  static constexpr int TM_DV = 0, TM_DK = D, TM_S = 2 * D, TM_P = 2 * D + 128;
  static constexpr bool OWN_DQ = D == 64;
  static constexpr int TM_DQ = OWN_DQ ? TM_P + 128 : TM_P;
  static constexpr bool OWN_PT = D == 64;
  static constexpr int TM_PT = OWN_PT ? TM_DQ + 64 : TM_S;
  static constexpr int PT_WG = OWN_PT ? 16 : 32;  // columns from one warpgroup's half of P^T to the next's
  // queries [16kk, 16kk+16) of P^T / dS^T: 8 columns of bf16 pairs (a warpgroup's 16 words of a
  // half are at the start of its 32 columns, or alone in P^T's own)
  __host__ __device__ static constexpr uint32_t pt_col(int kk) { return TM_PT + PT_WG * (kk >> 1) + 8 * (kk & 1); }
  __host__ __device__ static constexpr uint32_t ds_col(int kk) { return TM_P + 32 * (kk >> 1) + 8 * (kk & 1); }
  // Row terms staged by warp 3, or by the compute warps.  d = 64, which the compute warps bound: 1.34
  // ms against 1.29 (14/2/64, sixteen segments of 4,096); d = 128: 0.5% slower by a warp of its own.
  static constexpr bool ROW_WARP = D == 64;
  static constexpr bool SCALED_D = D == 128;
  static constexpr int REG_CTRL = ROW_WARP ? 96 : 80, REG_COMPUTE = ROW_WARP ? 136 : 144, REG_DRAIN = 144;
  static constexpr int REG_LAUNCH = 65536 / THREADS;
  // Tile u's Q and dO take the slots 2(u % NST) and the next, in turn: dO(u) is released well
  // before Q(u), and S^T needs Q(u+NST) before dV and dP^T need dO(u+NST), so Q(u+NST) goes where
  // dO(u) was and dO(u+NST) where Q(u) was, and both loads have about a tile's time.
  __device__ static uint32_t q_off(int u) { return (2 * (u % NST) + ((u / NST) & 1)) * TILE; }
  __device__ static uint32_t do_off(int u) { return (2 * (u % NST) + 1 - ((u / NST) & 1)) * TILE; }
  static constexpr uint32_t IDESC_S = idesc_bf16(128, 128, 0, 0);   // K or V (K-major) x Q or dO (K-major)
  static constexpr uint32_t IDESC_KV = idesc_bf16(128, D, 0, 1);    // P^T / dS^T (TMEM) x dO / Q (MN-major)
  // d = 128: K^T (MN-major, M = dims) x dS (MN-major, N = queries); d = 64: dS^T x K (both MN-major)
  static constexpr uint32_t IDESC_DQ = D == 128 ? idesc_bf16(128, 128, 1, 1) : idesc_bf16(128, D, 1, 1);
};
static_assert(Bwd<64>::SMEM <= 232448 && Bwd<128>::SMEM <= 232448, "shared memory budget");
template <int D>
constexpr bool regs_fit() {
  return Bwd<D>::REG_CTRL + 2 * Bwd<D>::REG_COMPUTE + Bwd<D>::REG_DRAIN <= 4 * Bwd<D>::REG_LAUNCH;
}
static_assert(regs_fit<64>() && regs_fit<128>(), "setmaxnreg targets exceed the registers the block is launched with");

struct BwdBars {
  uint64_t kv_full;
  uint64_t q_full[4], q_done[4];     // Q(u) landed; its last reader dK(u) complete
  uint64_t do_full[4], do_done[4];   // dO(u) landed; its readers dV(u) and dP^T(u) complete
  uint64_t s_full;                   // S^T(u) complete (ROW_WARP: and its row terms staged)
  uint64_t rt_free[2];               // ROW_WARP: the row terms of the tile of this parity no longer needed
  uint64_t s_read;                   // d = 64: S^T(u) read out of TMEM
  uint64_t p_full;                   // P^T(u) written, dP^T(u) issued (so that dV(u) does not run ahead of it)
  uint64_t dp_full;                  // dP^T(u) complete
  uint64_t ds_full[2];               // dS^T(u): columns [0,32) / [32,64) of each warpgroup written
  uint64_t dq_full;                  // dK(u), dQ(u) complete
  uint64_t dq_free;                  // dQ(u) read out of TMEM
  uint64_t acc_done;
  uint32_t tmem_base;
  int32_t abort;
};
static_assert(sizeof(BwdBars) <= Bwd<64>::BAR_BYTES && sizeof(BwdBars) <= Bwd<128>::BAR_BYTES, "barrier space");

// d = 64: v holds the warp's 32 query rows in the 16x256b layout of its two 16-row halves g: words
// 4b + 2*half of v[g] are row 16g + 8*half + lane/4, columns 8b + 2*(lane%4) and the next.  One
// exchange with lane^1 makes 4 consecutive columns of 64-byte row pieces, one with lane^4 makes
// 128-byte pieces: 8 lanes a row, 4 rows a reduction.  row(i, live) gives the accumulator row of the
// warp's query i and whether its values are added (else 0 is).  Four reductions (16 lines of 128
// bytes) a warp every 200 cycles: 1.268 ms (14/2/64, 16 segments of 4,096) against 1.293 at full
// speed and 1.273 and 1.288 with 300 and 400.
// Rows past the segment's end add 0 as well: leaving groups of them out put a branch between the
// reductions that cost full tiles 8% (1.255 -> 1.356 ms).
template <typename RowFn>
__device__ __forceinline__ void drain_d64(const uint32_t (&v)[2][32], int lane, RowFn row) {
  const bool odd = lane & 1, oddr = lane & 4;
  const uint32_t t0 = clock();
  const int coff = (lane & 1) * 8 + ((lane >> 1) & 1) * 4 + (oddr ? 16 : 0);
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int rr = 16 * g + 8 * half + ((lane >> 2) & 6);
      bool le, lo;
      float* pe = row(rr, le);
      float* po = row(rr + 1, lo);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint32_t a[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t x0 = v[g][4 * (4 * i + 2 * j) + 2 * half], y0 = v[g][4 * (4 * i + 2 * j) + 2 * half + 1];
          const uint32_t x1 = v[g][4 * (4 * i + 2 * j + 1) + 2 * half],
                         y1 = v[g][4 * (4 * i + 2 * j + 1) + 2 * half + 1];
          const uint32_t rx = __shfl_xor_sync(0xffffffffu, odd ? x0 : x1, 1);
          const uint32_t ry = __shfl_xor_sync(0xffffffffu, odd ? y0 : y1, 1);
          a[j][0] = odd ? rx : x0;
          a[j][1] = odd ? ry : y0;
          a[j][2] = odd ? x1 : rx;
          a[j][3] = odd ? y1 : ry;
        }
        float e[4], o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t r = __shfl_xor_sync(0xffffffffu, oddr ? a[0][c] : a[1][c], 4);
          e[c] = le ? __uint_as_float(oddr ? r : a[0][c]) : 0.f;
          o[c] = lo ? __uint_as_float(oddr ? a[1][c] : r) : 0.f;
        }
        red_add_v4(pe + 32 * i + coff, e[0], e[1], e[2], e[3]);
        red_add_v4(po + 32 * i + coff, o[0], o[1], o[2], o[3]);
      }
      if (g == 0 || half == 0)
        while ((uint32_t)clock() - t0 < (uint32_t)(200 * (2 * g + half + 1))) {
        }
    }
}

// GATHER: Q, K and V are trajectory-layout tensors read through tok_gather, one warp per
// tile (TMA gather4 with the 2-D maps tm_q/k/v, or tiled loads with the 3-D maps
// tm_qr/kr/vr and tm_qs/ks/vs, 128- and 32-row boxes, where a tile or a 32-row group is one
// run of consecutive trajectory rows), and dQ, dK, dV are added in fp32 to trajectory-layout
// accumulators (dq_acc, dk_acc, dv_acc) at row tok_gather[token]; otherwise segment-layout tiled
// loads, dq_acc in segment layout, bf16 dK, dV, and the other maps unused.
template <int D, bool GATHER>
__global__ void __launch_bounds__(Bwd<D>::THREADS, 1)
    bwd_main(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
             const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
             const int32_t* __restrict__ cu_seqlens, int32_t num_segments, int32_t num_tokens, int32_t max_seqlen,
             int32_t hq, int32_t hkv, int32_t tail_groups, float scale, float scale_log2,
             const float* __restrict__ lse, const float* __restrict__ dvec, float* __restrict__ dq_acc, __nv_bfloat16* __restrict__ dk,
             __nv_bfloat16* __restrict__ dv, int32_t* status, const int32_t* __restrict__ tok_gather,
             int32_t traj_tokens, float* __restrict__ dk_acc, float* __restrict__ dv_acc,
             const __grid_constant__ CUtensorMap tm_qr, const __grid_constant__ CUtensorMap tm_kr,
             const __grid_constant__ CUtensorMap tm_vr, const __grid_constant__ CUtensorMap tm_qs,
             const __grid_constant__ CUtensorMap tm_ks, const __grid_constant__ CUtensorMap tm_vs) {
  using C = Bwd<D>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw;
  BwdBars* bars = reinterpret_cast<BwdBars*>(smem + C::OFF_BAR);

  // x = key tile (fastest), so the CTAs resident at one time mostly belong to one (segment, kv head).
  // The last tail_groups of those go key tile by key tile instead, the first (longest) of every
  // group first: in turn, the last groups' longest CTAs would start when little else is left.
  int sg = (int)(blockIdx.z * 65535u + blockIdx.y);
  const int ngroups = num_segments * hkv;
  if (sg >= ngroups) return;
  int n = blockIdx.x;  // key tile
  if (sg >= ngroups - tail_groups) {
    const int64_t t = (int64_t)(sg - (ngroups - tail_groups)) * gridDim.x + n;
    n = (int)(t / tail_groups);
    sg = ngroups - tail_groups + (int)(t % tail_groups);
  }
  const int seg = sg / hkv;
  const int g = sg - seg * hkv;
  const int start = cu_seqlens[seg];
  const int end = cu_seqlens[seg + 1];
  if (start < 0 || end < start || end > num_tokens || end - start > max_seqlen ||
      (seg == 0 && start != 0) || (seg == num_segments - 1 && end != num_tokens)) {
    if (threadIdx.x == 0 && n == 0 && g == 0) set_status(status, VCS_ERR_DEVICE_CHECK);
    return;
  }
  const int L = end - start;
  if (n * C::BM >= L) return;
  // The tiles' 128-byte swizzle wants 1,024-byte aligned blocks.  A kernel without static shared
  // memory gets its dynamic shared memory so aligned; there is no room to align it here.
  if (smem_u32(smem) & 1023u) {
    if (threadIdx.x == 0) set_status(status, VCS_ERR_CUDA);
    return;
  }
  // once any CTA of this launch has given up on a wait, the rest stand down (read only by the
  // CTAs that have a key tile)
  if (*reinterpret_cast<volatile int32_t*>(status) == VCS_ERR_DEVICE_TIMEOUT) return;
  const int G = hq / hkv;
  const int nsub = (L - n * C::BM + C::BQ - 1) / C::BQ;  // 128-row query tiles at or after this key tile
  const int U = G * nsub;
  // Tile u covers query rows n*BM + sub*BQ ... +BQ-1 of one head.  d = 128: swept from the segment
  // end toward the key tile with the G heads of one row block in turn, so that the key tiles of one
  // (segment, kv head) running together meet the same Q/dO/dQ lines in L2.  d = 64: head by head
  // from the key tile to the segment end, which is the order dK and dV are summed in, and the key
  // tiles that run together are on different rows of dQ.
  struct Walk {  // tile u's row block and head, stepped without divisions
    int sub, head, first, count;  // first head and heads (d = 128); row blocks and last head + 1 (d = 64)
    __device__ __forceinline__ void next() {
      if constexpr (D == 64) {
        if (++sub == first) {
          sub = 0;
          ++head;
        }
      } else if (++head == first + count) {
        head = first;
        --sub;
      }
    }
    __device__ __forceinline__ bool live() const { return D == 64 ? head < count : sub >= 0; }
  };
  const Walk walk0 = D == 64 ? Walk{0, g * G, nsub, g * G + G} : Walk{nsub - 1, g * G, g * G, G};
  // lse and D of query i of w's tile, as loaded: scaled only where they are staged
  auto row_terms = [&](const Walk& w, int i, bool mine, float& l, float& dd) {
    l = __int_as_float(0x7f800000);  // +inf: query outside the segment -> P = 0
    dd = 0.f;
    const int q = n * C::BM + w.sub * C::BQ + i;
    if (w.live() && mine && q < L) {
      const size_t j = (size_t)w.head * num_tokens + start + q;
      l = __ldg(&lse[j]);
      dd = __ldg(&dvec[j]);
    }
  };

  // -D, scaled at d = 128, where dS = P fma(dP, scale, -D scale).  d = 64 keeps the exact difference,
  // dS = P (dP - D) scale: a rounded D scale would leave a residue where dP and D cancel.
  auto nd_of = [&](float dd) { return C::SCALED_D ? -dd * scale : -dd; };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_u32(smem);

  if (threadIdx.x == 0) {
    mbar_init(&bars->kv_full, 1);
    for (int i = 0; i < C::NST; ++i) {
      mbar_init(&bars->q_full[i], 1);
      mbar_init(&bars->q_done[i], 1);
      mbar_init(&bars->do_full[i], 1);
      mbar_init(&bars->do_done[i], 2);
    }
    mbar_init(&bars->s_full, C::ROW_WARP ? 2 : 1);
    for (int i = 0; i < 2; ++i) mbar_init(&bars->rt_free[i], 8);
    mbar_init(&bars->s_read, 8);
    mbar_init(&bars->p_full, 256 + 1);
    mbar_init(&bars->dp_full, 1);
    for (int i = 0; i < 2; ++i) mbar_init(&bars->ds_full[i], 256);
    mbar_init(&bars->dq_full, 1);
    mbar_init(&bars->dq_free, 128);
    mbar_init(&bars->acc_done, 2);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  auto abort_now = [&]() {
    set_status(status, VCS_ERR_DEVICE_TIMEOUT);
    *reinterpret_cast<volatile int32_t*>(&bars->abort) = 1;
  };
  auto aborted_now = [&]() { return *reinterpret_cast<volatile int32_t*>(&bars->abort) != 0; };

  if (warp < 4) {
    setmaxnreg_dec<C::REG_CTRL>();
    if (warp == 0 && (GATHER || lane == 0)) {
      // ---------------------------------------------------------- producer
      // gathered: the whole warp loads K, V and each tile's Q; lane 0 posts the bytes, waits for
      // free slots and loads dO
      if (lane == 0) {
        tma_prefetch_desc(&tm_q);
        tma_prefetch_desc(&tm_k);
        tma_prefetch_desc(&tm_v);
        tma_prefetch_desc(&tm_do);
        mbar_arrive_expect_tx(&bars->kv_full, 2 * C::TILE);
      }
      Walk wq = walk0, wd = walk0;  // of the next Q and the next dO to load
      auto load_q = [&](int u) {
        const int h = wq.head, row = start + n * C::BM + wq.sub * C::BQ;
        wq.next();
        uint8_t* dst = smem + C::OFF_QD + C::q_off(u);
        uint64_t* bar = &bars->q_full[u % C::NST];
        if (lane == 0) mbar_arrive_expect_tx(bar, C::TILE);
        if constexpr (GATHER) {
          __syncwarp();
          load_traj_tile<C::KB, C::BLOCK>(dst, &tm_q, &tm_qr, &tm_qs, bar, h, D, row, end - 1, tok_gather,
                                          traj_tokens, status, lane);
        } else {
#pragma unroll
          for (int kb = 0; kb < C::KB; ++kb)
            tma_load_3d(dst + kb * C::BLOCK, &tm_q, bar, kb * 64, h, row);
        }
      };
      auto load_do = [&](int u) {
        const int h = wd.head, row = start + n * C::BM + wd.sub * C::BQ;
        wd.next();
        if (lane != 0) return;
        uint64_t* bar = &bars->do_full[u % C::NST];
        mbar_arrive_expect_tx(bar, C::TILE);
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
          tma_load_3d(smem + C::OFF_QD + C::do_off(u) + kb * C::BLOCK, &tm_do, bar, kb * 64, h, row);
      };
      // a bounded wait whose outcome is the producer's (lane 0 waits and broadcasts)
      auto wait_free = [&](uint64_t* bar, uint32_t parity) -> bool {
        int go = 1;
        if (lane == 0) {
          if (!mbar_wait(bar, parity)) {
            abort_now();
            go = 0;
          } else if (aborted_now()) {
            go = 0;
          }
        }
        if constexpr (GATHER) go = __shfl_sync(0xffffffffu, go, 0);
        return go != 0;
      };
      if constexpr (GATHER) {
        __syncwarp();
        load_traj_tile<C::KB, C::BLOCK>(smem + C::OFF_K, &tm_k, &tm_kr, &tm_ks, &bars->kv_full, g, D,
                                        start + n * C::BM, end - 1, tok_gather, traj_tokens, status, lane);
        load_q(0);
        load_traj_tile<C::KB, C::BLOCK>(smem + C::OFF_V, &tm_v, &tm_vr, &tm_vs, &bars->kv_full, g, D,
                                        start + n * C::BM, end - 1, tok_gather, traj_tokens, status, lane);
      } else {
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
          tma_load_3d(smem + C::OFF_K + kb * C::BLOCK, &tm_k, &bars->kv_full, kb * 64, g, start + n * C::BM);
        load_q(0);
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
          tma_load_3d(smem + C::OFF_V + kb * C::BLOCK, &tm_v, &bars->kv_full, kb * 64, g, start + n * C::BM);
      }
      for (int u = 0; u < C::NST && u < U; ++u) {
        if (u > 0) load_q(u);
        load_do(u);
      }
      for (int v = 0; v + C::NST < U; ++v) {
        if (!wait_free(&bars->do_done[v % C::NST], (v / C::NST) & 1)) break;
        load_q(v + C::NST);
        if (!wait_free(&bars->q_done[v % C::NST], (v / C::NST) & 1)) break;
        load_do(v + C::NST);
      }
    } else if (warp == 1 || warp == 2) {
      // ---------------------------------------------------------- MMA issuers
      // descriptors built once; the issue loops only add compile-time offsets
      const uint64_t k_kmaj = smem_desc(sbase + C::OFF_K, 16, 1024);
      const uint64_t k_mnmaj = smem_desc(sbase + C::OFF_K, C::BLOCK, 1024);
      const uint64_t qd_kmaj = desc_at(k_kmaj, C::OFF_QD), qd_mnmaj = desc_at(k_mnmaj, C::OFF_QD);
      auto issue_kmaj = [&](uint32_t tm, uint64_t a, uint64_t b) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t o = (kk >> 2) * C::BLOCK + (kk & 3) * 32;
          tc_mma_ss(tm, desc_at(a, o), desc_at(b, o), C::IDESC_S, kk > 0);
        }
      };
      // A wait can run out, and another role give up, between two lanes' reads, so no lane's answer
      // decides where the warp goes: every lane runs every tile, one that has given up waits no more, and
      // the elected lane issues as long as its own waits were met.
      bool ok = mbar_wait(&bars->kv_full, 0);
      if (warp == 1) {
        // S^T and dV.  d = 128: S^T(u+1) overwrites P^T(u), which dV(u), issued before, reads first.
        // d = 64: P^T has columns of its own, so S^T(u+1) is issued as soon as S^T(u) is read; its
        // barrier is then completed by dV(u), which also frees P^T's columns.
        auto issue_s = [&](int u) {
          ok = ok && mbar_wait(&bars->q_full[u % C::NST], (u / C::NST) & 1);
          if (C::OWN_PT && u > 0) ok = ok && mbar_wait(&bars->s_read, (u - 1) & 1);
          tc_fence_after();
          if (elect_one() && ok) {
            issue_kmaj(tmem + C::TM_S, k_kmaj, desc_at(qd_kmaj, C::q_off(u)));
            if (!C::OWN_PT || u == 0) tc_commit(&bars->s_full);
          }
          __syncwarp();
        };
        issue_s(0);
        for (int u = 0; u < U; ++u) {
          if (C::OWN_PT && u + 1 < U) issue_s(u + 1);
          ok = ok && mbar_wait(&bars->do_full[u % C::NST], (u / C::NST) & 1) && mbar_wait(&bars->p_full, u & 1) &&
               !aborted_now();
          tc_fence_after();
          if (elect_one() && ok) {
            const uint64_t dmn = desc_at(qd_mnmaj, C::do_off(u));
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              tc_mma_ts(tmem + C::TM_DV, tmem + C::pt_col(kk), desc_at(dmn, kk * 2048), C::IDESC_KV,
                        (u > 0 || kk > 0) ? 1u : 0u);
            tc_commit(&bars->do_done[u % C::NST]);
            if (C::OWN_PT && u + 1 < U) tc_commit(&bars->s_full);
          }
          __syncwarp();
          if (!C::OWN_PT && u + 1 < U) issue_s(u + 1);
        }
      } else {
        // dP^T, dK and dQ.  d = 128: dP^T(u) goes where dQ(u-1) was, dQ(u) where dS^T(u) was, which
        // dK(u), issued before, reads first.  d = 64: dQ(u) goes where dQ(u-1) was, in columns of its
        // own, so dP^T(u+1) need not wait for it and is issued ahead (what the compute warps wait for
        // next); dS^T in shared memory then takes two buffers.
        const uint64_t v_kmaj = desc_at(k_kmaj, C::OFF_V);
        const uint64_t ds_mnmaj = desc_at(k_mnmaj, C::OFF_DS);
        auto issue_dp = [&](int u) {
          ok = ok && mbar_wait(&bars->do_full[u % C::NST], (u / C::NST) & 1);
          if (!C::OWN_DQ && u > 0) ok = ok && mbar_wait(&bars->dq_free, (u - 1) & 1);
          ok = ok && !aborted_now();
          tc_fence_after();
          if (elect_one() && ok) {
            issue_kmaj(tmem + C::TM_P, v_kmaj, desc_at(qd_kmaj, C::do_off(u)));
            tc_commit(&bars->dp_full);
            mbar_arrive(&bars->p_full);
            tc_commit(&bars->do_done[u % C::NST]);
          }
          __syncwarp();
        };
        if (C::OWN_DQ) issue_dp(0);
        for (int u = 0; u < U; ++u) {
          if (!C::OWN_DQ) issue_dp(u);
          const uint64_t qmn = desc_at(qd_mnmaj, C::q_off(u));
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            ok = ok && mbar_wait(&bars->ds_full[hf], u & 1);
            tc_fence_after();
            if (elect_one() && ok) {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int kk = 4 * hf + j;
                tc_mma_ts(tmem + C::TM_DK, tmem + C::ds_col(kk), desc_at(qmn, kk * 2048), C::IDESC_KV,
                          (u > 0 || hf > 0 || j > 0) ? 1u : 0u);
              }
            }
            __syncwarp();
          }
          if (C::OWN_DQ) {
            if (u + 1 < U) issue_dp(u + 1);
            if (u > 0) ok = ok && mbar_wait(&bars->dq_free, (u - 1) & 1);
            tc_fence_after();
          }
          if (elect_one() && ok) {
            const uint64_t ds = desc_at(ds_mnmaj, (u % C::NDS) * 2 * C::BLOCK);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              tc_mma_ss(tmem + C::TM_DQ, desc_at(D == 128 ? k_mnmaj : ds, kk * 2048),
                        desc_at(D == 128 ? ds : k_mnmaj, kk * 2048), C::IDESC_DQ, kk > 0 ? 1u : 0u);
            tc_commit(&bars->dq_full);
          }
          __syncwarp();
        }
      }
      if (elect_one()) tc_commit(&bars->acc_done);
      __syncwarp();
      if (!ok) abort_now();
    } else if (C::ROW_WARP && warp == 3) {
      // ---------------------------------------------------------- row terms
      // Stages -lse*log2e and -D of each tile's 128 queries for the compute warps, loaded a tile
      // ahead (behind the drain's reductions a load can take more than a tile's time), and joins S^T's
      // barrier, so that the compute warps wait once for both.
      Walk w = walk0;
      float l[4], dd[4];
      auto load = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) row_terms(w, 32 * i + lane, true, l[i], dd[i]);
        w.next();
      };
      load();
      bool ok = true;
      float* rows = reinterpret_cast<float*>(smem + C::OFF_ROW);
      for (int u = 0; u < U; ++u) {
        if (u >= 2 && !mbar_wait_warp(&bars->rt_free[u & 1], ((u >> 1) - 1) & 1)) { ok = false; break; }
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // half i/2 of warpgroup i%2's 64 queries: nl, then nd
          float* r = rows + (u & 1) * 256 + (i & 1) * 128 + (i >> 1) * 32 + lane;
          r[0] = -l[i] * 1.4426950408889634f;
          r[64] = nd_of(dd[i]);
        }
        load();
        __syncwarp();
        // S^T(u-1) has completed the phase before
        if (u > 0 && !mbar_wait_warp(&bars->s_full, (u - 1) & 1)) { ok = false; break; }
        if (lane == 0) mbar_arrive(&bars->s_full);
        if (__any_sync(0xffffffffu, aborted_now())) break;
      }
      if (!ok) abort_now();
    }
  } else if (warp < 12) {
    // ------------------------------------------------------------ compute
    setmaxnreg_inc<C::REG_COMPUTE>();
    // query columns [32k, 32k+32) of each 64-column half of the tile: columns 0..31 and 32..63 below
    const int k = (warp - 4) >> 2;
    const int quad = warp & 3;
    const int r = quad * 32 + lane;  // TMEM lane: key row
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    // row terms of the warpgroup's 64 queries: nl = -lse*log2e, then nd (nd_of D); two buffers
    const uint32_t rt_u32 = smem_u32(smem + C::OFF_ROW) + k * 512;
    const uint32_t ds_row = sbase + C::OFF_DS + r * 128;
    const uint64_t sl2 = f2pack(scale_log2, scale_log2), sc2 = f2pack(scale, scale);
    Walk wc = walk0;  // of the tile computed
    bool ok = true;
    // without a warp for them: the row terms of the warpgroup's queries, loaded two tiles ahead
    const int tw = threadIdx.x - 128 - k * 128;
    float* rt_s = reinterpret_cast<float*>(smem + C::OFF_ROW) + k * 128;
    Walk wr = walk0;
    float l0, d0, l1, d1;
    auto next_terms = [&](float& l, float& dd) {
      row_terms(wr, 64 * (tw >> 5) + 32 * k + (tw & 31), tw < 64, l, dd);
      wr.next();
    };
    if constexpr (!C::ROW_WARP) {
      next_terms(l0, d0);
      next_terms(l1, d1);
    }
    for (int u = 0; u < U; ++u) {
      // the query rows are the key tile's own: mask keys after queries (column c of the
      // warpgroup's half hf is hidden from key row r when c < dlim - 64 hf)
      const int dlim = wc.sub == 0 ? r - 32 * k : 0;
      wc.next();
      const uint32_t rt = rt_u32 + (u & 1) * 1024;
      if constexpr (!C::ROW_WARP) {
        if (tw < 64) {
          rt_s[(u & 1) * 256 + tw] = -l0 * 1.4426950408889634f;
          rt_s[(u & 1) * 256 + 64 + tw] = nd_of(d0);
        }
        l0 = l1;
        d0 = d1;
        next_terms(l1, d1);
        // the row terms are staged and everyone is done with the other buffer's; go on only if every
        // thread got the tile before and no other role has given up
        if (!named_bar_and(1 + k, 128, ok && !aborted_now())) { ok = false; break; }
      }
      uint4 rq[2][4];  // the row terms of 16 columns, and of the next 16
      auto first_terms = [&](uint32_t at) {
#pragma unroll
        for (int j = 0; j < 4; ++j) rq[0][j] = ld_shared_v4(at + 16 * j);
      };
      if (!C::ROW_WARP) first_terms(rt);
      // each wait's outcome is the warp's (the TMEM loads below are warp-collective); without ROW_WARP
      // the warpgroup decides together at the barrier that opens the next tile
      if (!mbar_wait_warp(&bars->s_full, u & 1)) {
        ok = false;
        if (C::ROW_WARP) break;
        continue;
      }
      tc_fence_after();
      if (C::ROW_WARP) first_terms(rt);
      // P^T = 2^(S^T * scale*log2e - lse*log2e), fp32 in p, bf16 over the S^T columns just read
      uint32_t p[2][32];
      tmem_ld_cols<32>(trow + C::TM_S + 32 * k, p[0]);
      tmem_ld_cols<32>(trow + C::TM_S + 32 * k + 64, p[1]);
      tmem_ld_wait();
      reg_fence<32>(p[0]);
      reg_fence<32>(p[1]);
      if constexpr (C::OWN_PT) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->s_read);
      }
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        if (ch < 3) {
#pragma unroll
          for (int j = 0; j < 4; ++j) rq[(ch + 1) & 1][j] = ld_shared_v4(rt + 64 * (ch + 1) + 16 * j);
        }
        uint32_t(&x)[32] = p[ch >> 1];
        const int x0 = 16 * (ch & 1);
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const uint4 t = rq[ch & 1][c / 4];
          float a, b;
          f2unpack(ffma2(f2pack(__uint_as_float(x[x0 + c]), __uint_as_float(x[x0 + c + 1])), sl2,
                         f2pack(__uint_as_float(c & 2 ? t.z : t.x), __uint_as_float(c & 2 ? t.w : t.y))),
                   a, b);
          x[x0 + c] = __float_as_uint(ex2(a));
          x[x0 + c + 1] = __float_as_uint(ex2(b));
        }
        const int hide = dlim - 64 * (ch >> 1) - x0;
        if (hide > 0) {
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (c < hide) x[x0 + c] = 0u;
        }
        uint32_t pk[8];
#pragma unroll
        for (int c2 = 0; c2 < 8; ++c2)
          pk[c2] = pack_bf16(__uint_as_float(x[x0 + 2 * c2]), __uint_as_float(x[x0 + 2 * c2 + 1]));
        tmem_st_32x32b_x8(trow + C::TM_PT + C::PT_WG * (k + (ch & 2)) + 8 * (ch & 1), pk);
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(&bars->p_full);
      first_terms(rt + 256);
      if (!mbar_wait_warp(&bars->dp_full, u & 1)) {
        ok = false;
        if (C::ROW_WARP) break;
        continue;
      }
      tc_fence_after();
      // dS^T = P^T (dP^T - D) scale, 16 columns at a time, the next ones' loads in flight
      uint32_t dp[2][16];
      tmem_ld_cols<16>(trow + C::TM_P + 32 * k, dp[0]);
      tmem_ld_wait();
      reg_fence<16>(dp[0]);
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const int cur = ch & 1;
        if (ch < 3) {
          tmem_ld_cols<16>(trow + C::TM_P + 32 * k + 64 * ((ch + 1) >> 1) + 16 * ((ch + 1) & 1), dp[cur ^ 1]);
#pragma unroll
          for (int j = 0; j < 4; ++j) rq[cur ^ 1][j] = ld_shared_v4(rt + 256 + 64 * (ch + 1) + 16 * j);
        }
        uint32_t wd[8];
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const uint4 t = rq[cur][c / 4];
          const uint64_t x = f2pack(__uint_as_float(dp[cur][c]), __uint_as_float(dp[cur][c + 1]));
          const uint64_t nd = f2pack(__uint_as_float(c & 2 ? t.z : t.x), __uint_as_float(c & 2 ? t.w : t.y));
          const int pc = 16 * (ch & 1) + c;
          const uint64_t pp = f2pack(__uint_as_float(p[ch >> 1][pc]), __uint_as_float(p[ch >> 1][pc + 1]));
          float a, b;
          f2unpack(C::SCALED_D ? fmul2(pp, ffma2(x, sc2, nd)) : fmul2(fmul2(pp, fadd2(x, nd)), sc2), a, b);
          wd[c / 2] = pack_bf16(a, b);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
          st_shared_v4(ds_row + ((u % C::NDS) * 2 + (ch >> 1)) * C::BLOCK + (uint32_t)(((4 * k + 2 * (ch & 1) + j) ^ (r & 7)) << 4),
                       wd[4 * j], wd[4 * j + 1], wd[4 * j + 2], wd[4 * j + 3]);
        tmem_st_32x32b_x8(trow + C::TM_P + 32 * k + 64 * (ch >> 1) + 8 * (ch & 1), wd);
        if (ch & 1) {
          // dQ, the only reader of dS^T in shared memory, is issued after both halves' barriers, so
          // the second half's fence serves both (each costs the warp a drain of its stores: one
          // fewer, 14/2/64 ragged forward and backward 2.935 -> 2.921 ms)
          if (ch == 3) fence_proxy_async_smem();
          tmem_st_wait();
          tc_fence_before();
          mbar_arrive(&bars->ds_full[ch >> 1]);
        }
        if (ch < 3) {
          tmem_ld_wait();
          reg_fence<16>(dp[cur ^ 1]);
        }
      }
      if constexpr (C::ROW_WARP) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->rt_free[u & 1]);
      }
    }
    if (ok) ok = mbar_wait_warp(&bars->acc_done, 0);
    if (!ok) {
      abort_now();
    } else if (n * C::BM + quad * 32 < L) {  // the warp has rows in the segment
      tc_fence_after();
      // warpgroup 1 writes dK, warpgroup 2 writes dV (key row r on the TMEM lane)
      const uint32_t col = k == 0 ? C::TM_DK : C::TM_DV;
      if constexpr (GATHER) {  // fp32 add at the key's trajectory row
        const int kpos = n * C::BM + r;
        float* accp = nullptr;
        if (kpos < L) {
          const int t = tok_gather[start + kpos];
          if (t >= 0 && t < traj_tokens) accp = (k == 0 ? dk_acc : dv_acc) + ((size_t)t * hkv + g) * D;
        }
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t v32[32];
          tmem_ld_32x32b_x32(trow + col + c * 32, v32);
          tmem_ld_wait();
          reg_fence<32>(v32);
          if (accp != nullptr) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
              red_add_v4(accp + c * 32 + e * 4, __uint_as_float(v32[e * 4]), __uint_as_float(v32[e * 4 + 1]),
                         __uint_as_float(v32[e * 4 + 2]), __uint_as_float(v32[e * 4 + 3]));
          }
        }
      } else if constexpr (D == 64) {
        const int kpos = n * C::BM + r;
        __nv_bfloat16* outp = (k == 0 ? dk : dv) + ((size_t)(start + kpos) * hkv + g) * D;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t v32[32];
          tmem_ld_32x32b_x32(trow + col + c * 32, v32);
          tmem_ld_wait();
          reg_fence<32>(v32);
          if (kpos < L) {
            uint4* d4 = reinterpret_cast<uint4*>(outp + c * 32);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              d4[q] = make_uint4(pack_bf16(__uint_as_float(v32[q * 8 + 0]), __uint_as_float(v32[q * 8 + 1])),
                                 pack_bf16(__uint_as_float(v32[q * 8 + 2]), __uint_as_float(v32[q * 8 + 3])),
                                 pack_bf16(__uint_as_float(v32[q * 8 + 4]), __uint_as_float(v32[q * 8 + 5])),
                                 pack_bf16(__uint_as_float(v32[q * 8 + 6]), __uint_as_float(v32[q * 8 + 7])));
          }
        }
      } else {
        // the warp's 32 rows pass through its part of the K or V buffer (every MMA is complete), so
        // that 8 lanes store a row's 128 bytes instead of a thread its own row in 16-byte pieces (8
        // short rollouts 6.88 -> 6.75 ms, 32 segments of 1,024 0.327 -> 0.304; at d = 64 it cost 1%)
        const uint32_t stage = sbase + (k == 0 ? C::OFF_K : C::OFF_V);
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t v32[32];
          tmem_ld_32x32b_x32(trow + col + c * 32, v32);
          tmem_ld_wait();
          reg_fence<32>(v32);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            st_shared_v4(stage + (c / 2) * C::BLOCK + r * 128 + (uint32_t)((((c & 1) * 4 + q) ^ (r & 7)) << 4),
                         pack_bf16(__uint_as_float(v32[q * 8 + 0]), __uint_as_float(v32[q * 8 + 1])),
                         pack_bf16(__uint_as_float(v32[q * 8 + 2]), __uint_as_float(v32[q * 8 + 3])),
                         pack_bf16(__uint_as_float(v32[q * 8 + 4]), __uint_as_float(v32[q * 8 + 5])),
                         pack_bf16(__uint_as_float(v32[q * 8 + 6]), __uint_as_float(v32[q * 8 + 7])));
        }
        asm volatile("" ::: "memory");
        __syncwarp();
        asm volatile("" ::: "memory");
        const int row0 = quad * 32 + (lane >> 3), chunk = lane & 7;
        __nv_bfloat16* dst = (k == 0 ? dk : dv) + ((size_t)(start + n * C::BM + row0) * hkv + g) * D + chunk * 8;
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int ri = row0 + 4 * i;
            const uint4 v = ld_shared_v4(stage + kb * C::BLOCK + ri * 128 + (uint32_t)((chunk ^ (ri & 7)) << 4));
            if (n * C::BM + ri < L) *reinterpret_cast<uint4*>(dst + (size_t)(4 * i) * hkv * D + kb * 64) = v;
          }
      }
    }
  } else {
    // ------------------------------------------------------------ dQ drain
    setmaxnreg_inc<C::REG_DRAIN>();
    const int quad = warp & 3;
    const int dw = threadIdx.x - 12 * 32;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const size_t row_stride = (size_t)hq * D;
    Walk w = walk0;
    bool ok = true;
    for (int u = 0; u < U; ++u) {
      const int q0 = n * C::BM + w.sub * C::BQ;
      const int qn = min(C::BQ, L - q0);  // valid query rows
      float* base = dq_acc + (size_t)w.head * D;
      w.next();
      if (!mbar_wait_warp(&bars->dq_full, u & 1)) { ok = false; break; }
      tc_fence_after();
      // Q(u)'s last reader, dK(u), is complete: its slot may be refilled
      if (dw == 0) mbar_arrive(&bars->q_done[u % C::NST]);
      if constexpr (D == 128) {
        uint32_t v[128];  // head dim dw of the tile's 128 queries
#pragma unroll
        for (int c = 0; c < 4; ++c)
          tmem_ld_32x32b_x32(trow + C::TM_DQ + 32 * c, *reinterpret_cast<uint32_t(*)[32]>(&v[32 * c]));
        tmem_ld_wait();
        reg_fence<128>(v);
        tc_fence_before();
        mbar_arrive(&bars->dq_free);
        base += dw;
        // 16 reductions a warp, then a pause until 20 cycles have passed for each: issued as fast as
        // the SM takes them (22 cycles each) they hold up the compute warps' shared-memory accesses.
        // No branch per reduction (it would double the kernel's time): rows past the segment end, and
        // gather indices out of range, add 0 to a row in range; a burst wholly past the end is left out.
        const uint32_t t0 = clock();
        auto burst = [&](int c, auto add) {
#pragma unroll
          for (int i = 0; i < 16; ++i) add(16 * c + i);
          if (c < 7)
            while ((uint32_t)clock() - t0 < (uint32_t)(16 * 20 * (c + 1))) {
            }
        };
        bool run = qn == C::BQ;  // the tile's rows are consecutive rows of the accumulator
        int tok[4] = {0, 0, 0, 0};
        bool live[4];
        if constexpr (GATHER) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int q = 32 * j + lane;
            tok[j] = __ldg(&tok_gather[start + q0 + min(q, qn - 1)]);
            live[j] = q < qn && tok[j] >= 0 && tok[j] < traj_tokens;
            if (!live[j]) tok[j] = 0;
          }
          const int first = __shfl_sync(0xffffffffu, tok[0], 0);
#pragma unroll
          for (int j = 0; j < 4; ++j) run = run && live[j] && tok[j] == first + 32 * j + lane;
          run = __all_sync(0xffffffffu, run);
          if (run) base += (size_t)first * row_stride;
        } else {
          base += (size_t)(start + q0) * row_stride;
        }
        if (run) {
#pragma unroll
          for (int c = 0; c < 8; ++c)
            burst(c, [&](int q) { red_add(base + q * row_stride, __uint_as_float(v[q])); });
        } else if constexpr (GATHER) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if (16 * c >= qn) break;
            const unsigned lives = __ballot_sync(0xffffffffu, live[c / 2]);
            burst(c, [&](int q) {
              const int t = __shfl_sync(0xffffffffu, tok[q / 32], q % 32);
              red_add(base + (size_t)t * row_stride, (lives >> (q % 32)) & 1 ? __uint_as_float(v[q]) : 0.f);
            });
          }
        } else {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if (16 * c >= qn) break;
            burst(c, [&](int q) {
              red_add(base + min(q, qn - 1) * row_stride, q < qn ? __uint_as_float(v[q]) : 0.f);
            });
          }
        }
      } else {
        uint32_t v[2][32];
#pragma unroll
        for (int i = 0; i < 2; ++i) tmem_ld_16x256b_x8(trow + ((uint32_t)(16 * i) << 16) + C::TM_DQ, v[i]);
        tmem_ld_wait();
        reg_fence<32>(v[0]);
        reg_fence<32>(v[1]);
        tc_fence_before();
        mbar_arrive(&bars->dq_free);
        const int qr = 32 * quad;  // the warp's first query row
        if constexpr (GATHER) {
          int tok = __ldg(&tok_gather[start + q0 + min(qr + lane, qn - 1)]);
          const bool live = qr + lane < qn && tok >= 0 && tok < traj_tokens;
          if (tok < 0 || tok >= traj_tokens) tok = 0;
          const unsigned lives = __ballot_sync(0xffffffffu, live);
          drain_d64(v, lane, [&](int i, bool& l) -> float* {
            l = (lives >> i) & 1;
            return base + (size_t)__shfl_sync(0xffffffffu, tok, i) * row_stride;
          });
        } else {
          base += (size_t)(start + q0) * row_stride;
          drain_d64(v, lane, [&](int i, bool& l) -> float* {
            l = qr + i < qn;
            return base + min(qr + i, qn - 1) * row_stride;
          });
        }
      }
      if (__any_sync(0xffffffffu, aborted_now())) { ok = false; break; }
    }
    if (!ok) abort_now();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

template <int D, bool GATHER>
cudaError_t launch_bwd_d(const AttnArgs& a, const void* o, const float* lse, const void* dout, void* dq, void* dk,
                         void* dv, void* ws, cudaStream_t st) {
  using C = Bwd<D>;
  char* w = static_cast<char*>(ws) + kWsHeader;
  float* dvec = reinterpret_cast<float*>(w);
  float* dq_acc = reinterpret_cast<float*>(w + align256((size_t)a.hq * a.num_tokens * 4));
  // gathered: fp32 trajectory-layout accumulators of dQ, dK, dV behind the (unused) segment-layout dQ
  float *dq_t = nullptr, *dk_t = nullptr, *dv_t = nullptr;
  const int64_t rows = a.num_tokens * a.hq;
  if (GATHER) {
    char* t0 = reinterpret_cast<char*>(dq_acc) + align256((size_t)a.num_tokens * a.hq * D * 4);
    const size_t qb = align256((size_t)a.traj_tokens * a.hq * D * 4), kb = align256((size_t)a.traj_tokens * a.hkv * D * 4);
    dq_t = reinterpret_cast<float*>(t0);
    dk_t = reinterpret_cast<float*>(t0 + qb);
    dv_t = reinterpret_cast<float*>(t0 + qb + kb);
    if (cudaMemsetAsync(t0, 0, qb + 2 * kb, st) != cudaSuccess) return cudaErrorUnknown;
  }
  {
    const int64_t total = rows * (D / 8);
    int64_t blocks = (total + kPreThreads - 1) / kPreThreads;
    if (blocks > 152 * 32) blocks = 152 * 32;
    bwd_pre<D><<<(unsigned)blocks, kPreThreads, 0, st>>>(static_cast<const __nv_bfloat16*>(o),
                                                         static_cast<const __nv_bfloat16*>(dout), rows, a.hq,
                                                         a.num_tokens, dvec, GATHER ? nullptr : dq_acc, a.status);
  }
  alignas(64) CUtensorMap tq, tk, tv, tdo, tqr, tkr, tvr, tqs, tks, tvs;
  if (GATHER) {
    if (!encode_tma_rows_bf16(&tq, a.q, (uint64_t)a.hq * D, a.traj_tokens) ||
        !encode_tma_rows_bf16(&tk, a.k, (uint64_t)a.hkv * D, a.traj_tokens) ||
        !encode_tma_rows_bf16(&tv, a.v, (uint64_t)a.hkv * D, a.traj_tokens) ||
        !encode_tma_3d_bf16(&tqr, a.q, D, a.hq, a.traj_tokens, 64, 128) ||
        !encode_tma_3d_bf16(&tkr, a.k, D, a.hkv, a.traj_tokens, 64, 128) ||
        !encode_tma_3d_bf16(&tvr, a.v, D, a.hkv, a.traj_tokens, 64, 128) ||
        !encode_tma_3d_bf16(&tqs, a.q, D, a.hq, a.traj_tokens, 64, 32) ||
        !encode_tma_3d_bf16(&tks, a.k, D, a.hkv, a.traj_tokens, 64, 32) ||
        !encode_tma_3d_bf16(&tvs, a.v, D, a.hkv, a.traj_tokens, 64, 32))
      return cudaErrorInvalidValue;
  } else if (!encode_tma_3d_bf16(&tq, a.q, D, a.hq, a.num_tokens, 64, 128) ||
             !encode_tma_3d_bf16(&tk, a.k, D, a.hkv, a.num_tokens, 64, 128) ||
             !encode_tma_3d_bf16(&tv, a.v, D, a.hkv, a.num_tokens, 64, 128)) {
    return cudaErrorInvalidValue;
  }
  if (!encode_tma_3d_bf16(&tdo, dout, D, a.hq, a.num_tokens, 64, 128)) return cudaErrorInvalidValue;
  const int ntiles = (a.max_seqlen + C::BM - 1) / C::BM;
  const int64_t gx = (int64_t)a.num_segments * a.hkv;
  if (gx > (int64_t)65535 * 65535) return cudaErrorInvalidConfiguration;
  dim3 grid((unsigned)ntiles, (unsigned)(gx < 65535 ? gx : 65535), (unsigned)((gx + 65534) / 65535));
  // Tail: a group of t key tiles is about G t^2 / 2 tiles of work, shared by 152 SMs, and its longest
  // CTA G t of them; the last `tail_groups` groups are half of what keeps all SMs busy for as long as
  // the longest CTA of the launch takes (the CTAs before them cover the rest).  8 short rollouts,
  // 28/4/128: 6.94 ms without, 6.89 / 6.75 / 6.99 / 7.6 with half / this / twice / four times as many
  // (more groups at once share less in L2); forward + backward at 14/2/64 3.36 -> 3.22.
  const double tavg = (double)a.num_tokens / ((double)a.num_segments * C::BM);
  double tail_groups = 152.0 * ntiles / (tavg < 1.0 ? 1.0 : tavg * tavg);
  if (tail_groups < 1.0) tail_groups = 1.0;
  if (tail_groups > (double)gx) tail_groups = (double)gx;
  if (ntiles > 0) {
    static std::atomic<int> regs_cache{-1};
    bool regs_ok = false;
    if (cudaError_t e = launch_regs_match(reinterpret_cast<const void*>(bwd_main<D, GATHER>), C::REG_LAUNCH,
                                          &regs_cache, &regs_ok);
        e != cudaSuccess)
      return e;
    if (!regs_ok) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(bwd_main<D, GATHER>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    bwd_main<D, GATHER><<<grid, C::THREADS, C::SMEM, st>>>(
        tq, tk, tv, tdo, a.cu_seqlens, a.num_segments, (int32_t)a.num_tokens, a.max_seqlen, a.hq, a.hkv,
        (int32_t)tail_groups, a.scale, a.scale * 1.4426950408889634f, lse, dvec, GATHER ? dq_t : dq_acc, static_cast<__nv_bfloat16*>(dk),
        static_cast<__nv_bfloat16*>(dv), a.status, a.tok_gather, (int32_t)a.traj_tokens, dk_t, dv_t,
        GATHER ? tqr : tq, GATHER ? tkr : tk, GATHER ? tvr : tv, GATHER ? tqs : tq, GATHER ? tks : tk,
        GATHER ? tvs : tv);
  }
  auto convert = [&](const float* acc, void* out, int64_t elems) {
    const int64_t n8 = elems / 8;
    int64_t blocks = (n8 + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (n8 > 0) bwd_dq_cvt<<<(unsigned)blocks, 256, 0, st>>>(acc, static_cast<__nv_bfloat16*>(out), n8);
  };
  if (GATHER) {
    convert(dq_t, dq, a.traj_tokens * a.hq * D);
    convert(dk_t, dk, a.traj_tokens * a.hkv * D);
    convert(dv_t, dv, a.traj_tokens * a.hkv * D);
  } else {
    convert(dq_acc, dq, rows * D);
  }
  return cudaGetLastError();
}

}  // namespace

size_t attn_bwd_ws_bytes(const AttnArgs& a) {
  if (a.num_tokens < 0 || a.hq <= 0 || a.hkv <= 0 || a.d <= 0 || a.traj_tokens < 0) return kWsHeader;
  size_t b = kWsHeader + align256((size_t)a.hq * a.num_tokens * 4) + align256((size_t)a.num_tokens * a.hq * a.d * 4);
  // gathered: fp32 trajectory-layout dQ, dK, dV accumulators.  The size callers know, vcs_attn_bwd's plus
  // these, stays: its segment-layout dQ term is unused space then.
  if (a.traj_tokens > 0)
    b += align256((size_t)a.traj_tokens * a.hq * a.d * 4) + 2 * align256((size_t)a.traj_tokens * a.hkv * a.d * 4);
  return b;
}

cudaError_t launch_attn_bwd(const AttnArgs& a, const void* o, const float* lse, const void* dout, void* dq, void* dk,
                            void* dv, void* ws, cudaStream_t st) {
  if (a.tok_gather != nullptr) {
    if (a.d == 64) return launch_bwd_d<64, true>(a, o, lse, dout, dq, dk, dv, ws, st);
    return launch_bwd_d<128, true>(a, o, lse, dout, dq, dk, dv, ws, st);
  }
  if (a.d == 64) return launch_bwd_d<64, false>(a, o, lse, dout, dq, dk, dv, ws, st);
  return launch_bwd_d<128, false>(a, o, lse, dout, dq, dk, dv, ws, st);
}

}  // namespace vcs
