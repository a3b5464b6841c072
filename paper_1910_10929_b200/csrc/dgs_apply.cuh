// Kernels of the server's apply and of the pull without secondary compression.  Apart from dgs_kernels.cuh, which the module
// of the short vectors' kernels includes too.
#pragma once
#include "dgs_kernels.cuh"

namespace dgs {

// ---- pull without secondary compression: every nonzero entry of D_w -------------------
// The stream pass has run with the bound 1 for every layer (key >= 1 <=> the value is not zero),
// so the candidate buffer lists all nonzero entries of D_w in index order, part after part.
// This kernel copies the first `capacity` of them into the packet, clears them in D_w (Eq. 4:
// v_k becomes M), adds them to theta_w if kept (Eq. 5), and writes the count.
constexpr int kStatusLimit = -6;   // = DGS_ELIMIT
__global__ void __launch_bounds__(kThreads) k_emit_all(Workspace ws, float* __restrict__ D,
                                                       float* __restrict__ theta_local,
                                                       uint32_t* __restrict__ blk_max, uint32_t* __restrict__ out_idx,
                                                       float* __restrict__ out_val, uint32_t* __restrict__ out_count,
                                                       uint32_t capacity, int packet_format) {
  __shared__ uint32_t pre[kMaxParts + 1];
  __shared__ unsigned long long warp_scan[kWarps];
  const uint32_t parts = ld_volatile(ws.sync + kParts);
  number_parts<kMaxParts>(ws, parts, pre, warp_scan);
  const uint32_t C = pre[parts];
  const bool all = C <= capacity;          // every nonzero entry is sent: D_w is zero afterwards
  const uint32_t take = all ? C : capacity;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *out_count = take;
    if (!all) atomicMin(ws.status, kStatusLimit);
    atomicAdd(ws.stats + 2, (unsigned long long)C);
  }
  for (uint32_t p = blockIdx.x * kThreads + threadIdx.x; p < take; p += gridDim.x * kThreads) {
    const uint32_t part = part_of(pre, 0, parts - 1u, p), slot = __ldcg(ws.part_slot0 + part) + (p - pre[part]);
    const uint32_t i = __ldcg(ws.cand_idx + slot);
    const float v = __ldcg(ws.cand_val + slot);
    const float q = round16(v, packet_format);
    out_idx[p] = i;
    out_val[p] = q;
    D[i] = __fsub_rn(v, q);      // zero with float32 packets; else what rounding left behind stays (Eq. 6b)
    if (theta_local != nullptr) theta_local[i] = __fadd_rn(theta_local[i], q);
    // the block's bound was made exact by the pass (a block without a nonzero entry already has bound 0);
    // with everything sent unrounded the whole block is zero now
    if (all && packet_format == 0 && blk_max != nullptr) blk_max[i / kWarpTile] = 0;
  }
  // the pass has counted the candidates in the layers' histograms: nobody reads them here
  const size_t words = (size_t)ws.num_segs * kBins1;
  for (size_t w = (size_t)blockIdx.x * kThreads + threadIdx.x; w < words; w += (size_t)gridDim.x * kThreads) ws.hist1[w] = 0;
}

// ---- server apply (see PacketLog) ---------------------------------------------------
// Keeps a block's bound an upper bound on the magnitudes in the block.  Bounds only rise while
// packets are being subtracted, so a bound already read as high enough needs no atomic.
__device__ __forceinline__ void raise_bound(uint32_t* bound, uint32_t key) {
  if (key > __ldcg(bound)) atomicMax(bound, key);
}

// First position in the sorted idx[0, count) whose entry is >= key, found by a whole warp: 32 probes at a time, so
// that a packet of 2^15 entries takes three trips to memory and not fifteen.
__device__ __forceinline__ uint32_t warp_lower_bound(const uint32_t* __restrict__ idx, uint32_t count, uint64_t key, int lane) {
  uint32_t l = 0, r = count;                     // the answer lies in [l, r]
  while (r - l > 32) {
    const uint32_t step = (r - l + 32) / 33, q = l + step * (lane + 1) - 1;
    const bool less = q < r && (uint64_t)__ldg(idx + q) < key;
    const uint32_t c = __popc(__ballot_sync(kFull, less));   // sorted: the first c probes are below the key
    const uint32_t qc = l + step * (c + 1) - 1;
    if (c < 32 && qc < r) r = qc;
    l += step * c;
  }
  const bool less = l + lane < r && (uint64_t)__ldg(idx + l + lane) < key;
  return l + __popc(__ballot_sync(kFull, less));
}

// theta -= packet, and a copy of the packet into slot `slot` of the log: CTAs [0, copy_ctas).
// Each of the remaining CTAs finds where kThreads blocks of the vector begin in this packet: the packet's part that
// falls into them is found by two searches, its entries are counted per block in shared memory, and a prefix sum
// gives the positions.
__global__ void __launch_bounds__(kThreads) k_apply_log(const uint32_t* __restrict__ idx,
                                                        const float* __restrict__ val, uint32_t count,
                                                        float* __restrict__ theta, uint64_t n, int* status,
                                                        PacketLog lg, uint32_t slot, uint32_t row, uint32_t copy_ctas) {
  if (blockIdx.x >= copy_ctas) {
    __shared__ uint32_t s_cnt[kThreads], s_end[2];
    __shared__ unsigned long long s_warp[kWarps];
    const uint32_t b0 = (blockIdx.x - copy_ctas) * kThreads, warp = threadIdx.x >> 5;
    s_cnt[threadIdx.x] = 0;
    if (warp < 2) {
      const uint32_t at = warp_lower_bound(idx, count, (uint64_t)(b0 + warp * kThreads) * kWarpTile, threadIdx.x & 31);
      if ((threadIdx.x & 31) == 0) s_end[warp] = at;
    }
    __syncthreads();
    const uint32_t lo = s_end[0], hi = s_end[1];
    for (uint32_t j = lo + threadIdx.x; j < hi; j += kThreads) {
      const uint32_t b = __ldg(idx + j) / kWarpTile - b0;
      if (b < (uint32_t)kThreads) atomicAdd(s_cnt + b, 1u);
    }
    __syncthreads();
    unsigned long long total;
    const uint32_t before = (uint32_t)block_excl_scan(s_cnt[threadIdx.x], s_warp, total);
    const uint32_t b = b0 + threadIdx.x;
    if (b < lg.pos_rows) {
      lg.pos[(uint64_t)b * lg.ring + slot] = lo + before;
      const uint32_t next = row == lg.ring ? 0u : row + 1u;       // `row`: as of the packet before
      lg.sum[(uint64_t)next * lg.sum_stride + b] = __ldcg(lg.sum + (uint64_t)row * lg.sum_stride + b) + s_cnt[threadIdx.x];
    }
    return;
  }
  const uint32_t j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= count) return;
  const uint32_t i = idx[j];
  const float v = val[j];
  lg.ent[(uint64_t)slot * lg.stride + j] = make_uint2(i, __float_as_uint(v));
  if (i >= n || (j + 1 < count && idx[j + 1] <= i)) atomicMin(status, -2000);   // out of range, or not ascending
  if (i >= n) return;
  theta[i] = __fsub_rn(theta[i], v);
}

// Eager form, for a packet that is too long for the log (any count): buffer q < N is D_q, buffer N is theta.  Indices of
// one packet ascend, so every (buffer, entry) pair is touched by exactly one thread: plain load / subtract / store.  A
// packet that does not ascend is reported.
__global__ void __launch_bounds__(kThreads) k_scatter_sub(const uint32_t* __restrict__ idx,
                                                          const float* __restrict__ val, uint32_t count,
                                                          float* __restrict__ theta, float* __restrict__ D,
                                                          uint64_t d_stride, uint32_t num_workers, uint64_t n,
                                                          int* status, uint32_t* __restrict__ blk_max,
                                                          uint64_t blk_stride) {
  const uint32_t j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= count) return;
  const uint32_t i = idx[j];
  const float v = val[j];
  const uint32_t q = blockIdx.y;
  if (q == 0 && (i >= n || (j + 1 < count && idx[j + 1] <= i))) atomicMin(status, -2000);   // out of range, or not ascending
  if (i >= n) return;
  float* p = (q == num_workers ? theta : D + (uint64_t)q * d_stride) + i;
  const float r = __fsub_rn(*p, v);
  *p = r;
  if (q < num_workers) raise_bound(blk_max + (uint64_t)q * blk_stride + i / kWarpTile, key_of(r));
}

}  // namespace dgs
