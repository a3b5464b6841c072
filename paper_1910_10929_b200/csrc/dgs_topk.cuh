// Top-k + encode of one short flat vector in one kernel (dgs_topk_encode_static).
//
// One cluster of up to 16 CTAs does the whole selection: its CTAs are resident together and meet at the hardware
// barrier of the cluster, and their histograms are added up in the shared memory of the first of them.  What bounds it
// is the chain of those meetings, not the bytes (4 MB at the most).
// Measured against the copy, histogram pass, pick, stream pass and cooperative finalize it stands for: 65536 elements,
// 0.1 %: 10.3 us for 41.7; 1000003 elements, 5 %: 24.1 us for 49.2 (reading and listing is half of that).
//   sample      every CTA takes the same sample of at most kTopkSample elements, evenly spaced over the vector, and
//               from it a bound L that very likely admits at least k elements and not many more.  No meeting: all
//               CTAs find the same bound.
//   list        every warp reads its tiles of the vector and lists the elements whose key is at least L, in index order,
//               in shared memory; they are counted in bins above L.
//   exact       the few elements of the k-th's bin go to the first CTA, which compares each with all the others: the k-th
//               largest key T and the number r of entries equal to T that still fit.
//   emit        counts of (key > T, key == T) per warp, prefix sums over warps and CTAs, packet in index order.
// If the bin holds too many elements, radix levels (11 + 10 + 10 key bits) take the place of the exact step.  A warp whose
// list overflows visits its tiles again in every later step instead.  If fewer than k elements are at least L (the sample
// said nothing about the vector), all warps visit all their elements.  The vector is then read six times instead of once;
// if what is left is all zeros, three times.  The result never depends on the sample.
#pragma once
#include <cooperative_groups.h>

#include <type_traits>

#include "dgs_kernels.cuh"

namespace dgs {

// Two variants.  Short vectors take 512 threads a CTA and fine bins with one exact step; the barriers of fewer warps are
// shorter (65536 elements, 0.1 %: 10.3 us, 11.6 us with 1024 threads).  Long ones take 1024 threads, which list faster, and
// three radix levels, since a bin of many candidates holds too many to compare (1000003 elements, 5 %: 24.1 us; 28.0 us
// with 512 threads).
constexpr uint32_t kTopkFine = 1u << 18;   // longest vector that takes the first
__host__ __device__ constexpr int topk_threads(bool fine) { return fine ? 512 : 1024; }
constexpr uint32_t kTopkMaxCluster = 16;   // (more than 8 is not portable to every GPU: the launch asks for it)
constexpr int kBins2 = 1024;               // levels 2 and 3 (level 1: kBins1, the top 11 key bits)
constexpr uint32_t kTopkSample = 1024;
constexpr uint32_t kTopkShort = 512;       // most elements in the k-th's bin that are ranked by comparing them
constexpr uint32_t kTopkTurns = 4;         // most turns in which the tiles are dealt out
// most elements a warp can list: 184 KB of lists per CTA
__host__ __device__ constexpr uint32_t topk_cap(bool fine) { return 736u * 1024u / topk_threads(fine); }
constexpr int kStatusRank = -1002;         // an entry got a rank that cannot be

// Outcome of the last call's kernel on the device: 0, or a negative word if its packet is not complete.
__device__ int g_topk_status;

struct TopkShared {
  uint32_t hist[kBins1];                     // this CTA's counts of the level in hand
  uint32_t sum1[kBins1], again1[kBins1];     // first CTA of the cluster: counts of all CTAs, level 1 (lists; slices)
  uint32_t sum2[kBins2], sum3[kBins2];       //                                               levels 2 and 3
  uint32_t warp_sum[32];
  uint32_t list_end[kTopkTurns][32];         // elements on each warp's list after each turn
  uint2 warp_tot[kTopkTurns][32];            // (key > T, key == T) of each warp
  uint2 cta_tot[kTopkTurns][kTopkMaxCluster];   // of each CTA of the cluster
  uint32_t together;                         // the large elements of the sample lie together
  uint32_t short_cnt, short_at;              // elements of this CTA in the k-th's bin; where they go
  uint32_t short_all;                        // first CTA: of all CTAs
  uint32_t res[3];                           // of this CTA's own pick
  uint4 told;                                // what the first CTA found: bin, entries needed of it, total, entries in
                                             // the bin; in the end T and r
};

// From a histogram of B bins in shared memory, counting from the top bin down, the bin that
// holds the k-th entry and how many entries of that bin are needed.  Returns the total count; bin and need are valid
// if it is at least k.  The same for every thread of the CTA.
template <int B, int kTopkThreads>
__device__ uint32_t topk_pick(const uint32_t* hist, uint32_t k, uint32_t& bin, uint32_t& need, TopkShared& sh) {
  constexpr int PER = B / kTopkThreads;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t c[PER], sum = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    c[j] = hist[B - 1 - (int)threadIdx.x * PER - j];
    sum += c[j];
  }
  uint32_t incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) sh.warp_sum[warp] = incl;
  __syncthreads();
  const uint32_t w = lane < kTopkThreads / 32 ? sh.warp_sum[lane] : 0u;
  uint32_t winc = w;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, winc, d);
    if (lane >= d) winc += o;
  }
  const uint32_t total = __shfl_sync(kFull, winc, 31);
  uint32_t above = __shfl_sync(kFull, winc - w, warp) + incl - sum;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if (above < k && k <= above + c[j]) {
      sh.res[0] = B - 1 - threadIdx.x * PER - j;
      sh.res[1] = k - above;
      sh.res[2] = c[j];
    }
    above += c[j];
  }
  __syncthreads();
  bin = sh.res[0];
  need = sh.res[1];
  return total;
}

// From the bound on: lists, selection, packet.  DEALT: where the large elements of the sample lie together (a layer with
// large updates, a sorted vector) the tiles of 512 are dealt out to the warps in turns, so that no list overflows; else every
// warp has a run of tiles (of units of 32 where there are not enough tiles).  (Sorted, 2^20 elements, 0.1 % / 10 %: 27 us dealt
// out, 54 / 74 in runs.  Not sorted, 10 %: 32 us dealt out, 27 in runs.  One body for both, with DEALT in a register, cost the runs 2 to 4 us.)
template <bool FINE, bool DEALT>
__device__ __forceinline__ void topk_rest(const float* __restrict__ x, uint32_t n, uint32_t k, uint32_t* __restrict__ out_idx,
                                          float* __restrict__ out_val, uint32_t cap, uint32_t L, TopkShared& sh, unsigned char* lists) {
  constexpr int kTopkThreads = topk_threads(FINE);
  constexpr uint32_t kTopkWarps = kTopkThreads / 32;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t C = gridDim.x, cta = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, lt = lanemask_lt();
  uint32_t* const my_idx = reinterpret_cast<uint32_t*>(lists) + warp * 2u * cap;
  float* const my_val = reinterpret_cast<float*>(my_idx + cap);
  const uint32_t lw = 31u - __clz(C * kTopkWarps), g = cta * kTopkWarps + warp;   // 2^lw warps
  const uint32_t turns = DEALT ? ((n - 1u) >> (9u + lw)) + 1u : 1u;
  const uint32_t unit = n >= 512u << lw ? 512u : 32u, units = (n + unit - 1u) / unit;
  const uint32_t i0 = (g * units >> lw) * unit, i1 = min(n, ((g + 1u) * units >> lw) * unit);   // (n <= 2^20)

  // list
  uint32_t listed = 0;
  const float Lf = __uint_as_float(L);   // |x| >= Lf  <=>  key(x) >= L for finite x (no flush-to-zero)
  {
    uint32_t from = DEALT ? g << 9 : i0, turn = 0;
    const uint32_t stop = DEALT ? n : i1, step = DEALT ? 512u << lw : 512u;
    // 512 elements at a time, 16 bytes a lane: lane order is element order inside each of the four pieces of 128, so
    // four counts of a lane travel as four bytes through one prefix sum over the lanes
    float4 v[4], next[4];
    auto load = [&](uint32_t at) {
#pragma unroll
      for (int j = 0; j < 4; ++j) next[j] = __ldg(reinterpret_cast<const float4*>(x + at) + j * 32 + lane);
    };
    auto take = [&]() {                        // (the next tile is on its way while this one is listed)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = next[j];
      if (from + step + 512u <= stop) load(from + step);
      uint32_t mask = 0, packed = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t m = (fabsf(v[j].x) >= Lf ? 1u : 0u) | (fabsf(v[j].y) >= Lf ? 2u : 0u) | (fabsf(v[j].z) >= Lf ? 4u : 0u) |
                           (fabsf(v[j].w) >= Lf ? 8u : 0u);
        mask |= m << (4 * j);
        packed |= __popc(m) << (8 * j);
      }
      if (__any_sync(kFull, mask)) {
        uint32_t incl = packed;                   // at most 128 in a byte
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t o = __shfl_up_sync(kFull, incl, d);
          if (lane >= (uint32_t)d) incl += o;
        }
        const uint32_t tot = __shfl_sync(kFull, incl, 31), excl = incl - packed;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t at = listed + ((excl >> (8 * j)) & 0xFFu);
          listed += (tot >> (8 * j)) & 0xFFu;
          const float e[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if ((mask >> (4 * j + q)) & 1u) {
              if (at < cap) {
                my_idx[at] = from + j * 128u + lane * 4u + q;
                my_val[at] = e[q];
              }
              ++at;
            }
        }
      }
    };
    if ((reinterpret_cast<uintptr_t>(x) & 15u) == 0) {
      if (from + 512u <= stop) load(from);
      for (; from + 512u <= stop; from += step) {
        take();
        if (DEALT && lane == 0) sh.list_end[turn][warp] = listed;
        ++turn;
      }
    }
    // what is left: the end of a run, the last tile, or all if the vector does not begin on a 16-byte boundary
    for (; from < stop; from += step) {
      const uint32_t end = DEALT ? min(from + 512u, stop) : stop;
      for (uint32_t at0 = from; at0 < end; at0 += 128) {
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t i = at0 + j * 32u + lane;
          v[j] = i < end ? __ldg(x + i) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t i = at0 + j * 32u + lane;
          const bool in = i < end && key_of(v[j]) >= L;
          const uint32_t m = __ballot_sync(kFull, in), at = listed + __popc(m & lt);
          if (in && at < cap) {
            my_idx[at] = i;
            my_val[at] = v[j];
          }
          listed += __popc(m);
        }
      }
      if (!DEALT) break;
      if (lane == 0) sh.list_end[turn][warp] = listed;
      ++turn;
    }
    if (DEALT && lane == 0)
      for (; turn < turns; ++turn) sh.list_end[turn][warp] = listed;
  }
  __syncwarp();
  const bool again = listed > cap;               // this warp's list is too short
  bool everything = false;                       // fewer than k elements are at least L
  // visits this warp's elements of a turn in index order, 32 at a time: fn(valid, index, value)
  auto each_of = [&](uint32_t turn, uint2 on_list, auto fn) {
    if (everything || again) {
      uint32_t lo = DEALT ? min(n, ((turn << lw) + g) << 9) : i0;
      const uint32_t hi = DEALT ? min(n, lo + 512u) : i1;
      for (; lo < hi; lo += 256u) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = lo + j * 32u + lane < hi ? __ldg(x + lo + j * 32u + lane) : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (lo + j * 32u < hi)
            fn(lo + j * 32u + lane < hi && (everything || key_of(v[j]) >= L), lo + j * 32u + lane, v[j]);
      }
    } else {
      for (uint32_t p = on_list.x + lane; p - lane < on_list.y; p += 32) {
        const bool valid = p < on_list.y;
        fn(valid, valid ? my_idx[p] : 0u, valid ? my_val[p] : 0.f);
      }
    }
  };
  // all turns, in any order
  auto each = [&](auto fn) {
    if (everything || again) {
      for (uint32_t t = 0; t < turns; ++t) each_of(t, make_uint2(0, 0), fn);
    } else {
      for (uint32_t p = lane; p - lane < listed; p += 32) {
        const bool valid = p < listed;
        fn(valid, valid ? my_idx[p] : 0u, valid ? my_val[p] : 0.f);
      }
    }
  };
  // counted from the list, where the lanes are full: counting while listing is an atomic per one or two elements
  each([&](bool valid, uint32_t, float v) {
    hist_add(sh.hist, !valid ? 0u : FINE ? bin_of(key_of(v), L) : key_of(v) >> 20, valid, (int)lane);
  });
  __syncthreads();
  cl.barrier_wait();
  // This CTA's counts to the first CTA's sums; once all are there it picks, and tells every CTA what it found.  (Every
  // CTA picking for itself would save a barrier, but 16 of them reading one CTA's shared memory took 12,000 cycles.)
  auto pick = [&](uint32_t* sum, auto bins, uint32_t k_left, uint32_t& bin, uint32_t& need) -> uint2 {
    constexpr int B = decltype(bins)::value;
    uint32_t* const to = cl.map_shared_rank(sum, 0);
    for (uint32_t b = tid; b < (uint32_t)B; b += kTopkThreads) {
      const uint32_t c = sh.hist[b];
      if (c) {
        atomicAdd(to + b, c);
        sh.hist[b] = 0;
      }
    }
    cl.sync();
    if (cta == 0) {
      uint32_t fb, fn;
      const uint32_t total = topk_pick<B, kTopkThreads>(sum, k_left, fb, fn, sh);
      if (tid < C) cl.map_shared_rank(&sh, tid)->told = make_uint4(fb, fn, total, sh.res[2]);
    }
    cl.sync();
    const uint4 t = sh.told;
    bin = t.x;
    need = t.y;
    return make_uint2(t.z, t.w);
  };
  using Bins1 = std::integral_constant<int, kBins1>;
  using Bins2 = std::integral_constant<int, kBins2>;
  uint32_t bin, need;
  const uint2 found = pick(sh.sum1, Bins1(), k, bin, need);
  everything = found.x < k;              // the same in the whole cluster
  uint32_t T, r;
  if (everything && L == 1u) {           // all that is not zero is taken, and as many zeros as are missing
    T = 0;
    r = k - found.x;
  } else if (FINE && !everything && found.y <= kTopkShort) {
    // The elements of the k-th's bin go to the first CTA, which compares each with all the others.
    uint32_t* const mine = sh.hist;
    each([&](bool valid, uint32_t, float v) {
      const uint32_t key = key_of(v);
      if (valid && bin_of(key, L) == bin) mine[atomicAdd(&sh.short_cnt, 1u)] = key;
    });
    __syncthreads();
    TopkShared* const head = cl.map_shared_rank(&sh, 0);
    const uint32_t count = sh.short_cnt;
    if (tid == 0) sh.short_at = atomicAdd(&head->short_all, count);
    __syncthreads();
    for (uint32_t q = tid; q < count; q += kTopkThreads) head->sum1[sh.short_at + q] = mine[q];
    cl.sync();
    if (cta == 0) {
      for (uint32_t q = tid; q < found.y; q += kTopkThreads) {
        const uint32_t key = sh.sum1[q];
        uint32_t above = 0, same = 0;
#pragma unroll 4
        for (uint32_t o = 0; o < found.y; ++o) {
          const uint32_t other = sh.sum1[o];
          above += other > key ? 1u : 0u;
          same += other == key ? 1u : 0u;
        }
        if (above < need && need <= above + same) {   // (the same for all that are equal)
          sh.res[0] = key;
          sh.res[1] = need - above;
        }
      }
      __syncthreads();
      if (tid < C) cl.map_shared_rank(&sh, tid)->told = make_uint4(sh.res[0], sh.res[1], 0, 0);
    }
    cl.sync();
    T = sh.told.x;
    r = sh.told.y;
  } else {
    // three radix levels (11 + 10 + 10 key bits)
    if (FINE || everything) {
      each([&](bool valid, uint32_t, float v) { hist_add(sh.hist, key_of(v) >> 20, valid, (int)lane); });
      __syncthreads();
      pick(sh.again1, Bins1(), k, bin, need);
    }
    uint32_t prefix = bin;
#pragma unroll 1
    for (int level = 2; level <= 3; ++level) {
      const int shift = level == 2 ? 10 : 0;
      each([&](bool valid, uint32_t, float v) {
        const uint32_t key = key_of(v);
        if (valid && (key >> (shift + 10)) == prefix) atomicAdd(sh.hist + ((key >> shift) & 1023u), 1u);
      });
      __syncthreads();
      pick(level == 2 ? sh.sum2 : sh.sum3, Bins2(), need, bin, need);
      prefix = (prefix << 10) | bin;
    }
    T = prefix;
    r = need;
  }

  // How many of either kind each warp has in each turn, and the turns, CTAs and warps before it.  Lane t looks after turn t.
  uint2 on_list = make_uint2(0, listed);
  if (DEALT && lane < turns) on_list = make_uint2(lane ? sh.list_end[lane - 1u][warp] : 0u, sh.list_end[lane][warp]);
  auto of_turn = [&](uint2 v, uint32_t t) { return make_uint2(__shfl_sync(kFull, v.x, t), __shfl_sync(kFull, v.y, t)); };
  uint2 mine = make_uint2(0, 0);
  for (uint32_t t = 0; t < turns; ++t) {
    uint32_t gt = 0, eq = 0;
    each_of(t, of_turn(on_list, t), [&](bool valid, uint32_t, float v) {
      const uint32_t key = key_of(v);
      gt += __popc(__ballot_sync(kFull, valid && key > T));
      eq += __popc(__ballot_sync(kFull, valid && key == T));
    });
    if (lane == t) mine = make_uint2(gt, eq);
  }
  if (lane < turns) sh.warp_tot[lane][warp] = mine;
  __syncthreads();
  if (!DEALT) {
    const uint2 q = lane < kTopkWarps ? sh.warp_tot[0][lane] : make_uint2(0, 0);
    const uint2 all = make_uint2(__reduce_add_sync(kFull, q.x), __reduce_add_sync(kFull, q.y));
    if (tid < C) cl.map_shared_rank(&sh, tid)->cta_tot[0][cta] = all;
    cl.sync();                    // (nobody looks into another CTA's memory after this)
    const uint2 o = lane < cta ? sh.cta_tot[0][lane] : make_uint2(0, 0);
    mine = make_uint2(__reduce_add_sync(kFull, o.x + (lane < warp ? q.x : 0u)), __reduce_add_sync(kFull, o.y + (lane < warp ? q.y : 0u)));
  } else {                        // a warp per turn
    uint2 before = make_uint2(0, 0);   // lane w: what the warps before w have of it
    if (warp < turns) {
      const uint2 q = lane < kTopkWarps ? sh.warp_tot[warp][lane] : make_uint2(0, 0);
      before = make_uint2(warp_incl(q.x, lane) - q.x, warp_incl(q.y, lane) - q.y);
      const uint2 all = of_turn(make_uint2(before.x + q.x, before.y + q.y), 31);
      if (lane < C) cl.map_shared_rank(&sh, lane)->cta_tot[warp][cta] = all;
    }
    cl.sync();
    if (warp < turns) {
      uint2 o = make_uint2(0, 0);      // of the turns before, and of the CTAs before in this turn
      for (uint32_t t = 0; t <= warp; ++t)
        if (lane < (t < warp ? C : cta)) {
          o.x += sh.cta_tot[t][lane].x;
          o.y += sh.cta_tot[t][lane].y;
        }
      sh.warp_tot[warp][lane] = make_uint2(before.x + __reduce_add_sync(kFull, o.x), before.y + __reduce_add_sync(kFull, o.y));
    }
    __syncthreads();
    if (lane < turns) mine = sh.warp_tot[lane][warp];
  }
  for (uint32_t t = 0; t < turns; ++t) {
    uint2 at = of_turn(mine, t);
    each_of(t, of_turn(on_list, t), [&](bool valid, uint32_t i, float v) {
      const uint32_t key = key_of(v);
      const uint32_t mg = __ballot_sync(kFull, valid && key > T), me = __ballot_sync(kFull, valid && key == T);
      const uint32_t eq_rank = at.y + __popc(me & lt);
      if (valid && (key > T || (key == T && eq_rank < r))) {
        const uint32_t pos = at.x + __popc(mg & lt) + min(eq_rank, r);
        if (pos < k) {
          out_idx[pos] = i;
          out_val[pos] = v;
        } else {
          atomicMin(&g_topk_status, kStatusRank);
        }
      }
      at.x += __popc(mg);
      at.y += __popc(me);
    });
  }
}

template <bool FINE>
__global__ void __launch_bounds__(topk_threads(FINE), 1) k_topk(const float* __restrict__ x, uint32_t n, uint32_t k,
                                                         uint32_t* __restrict__ out_idx, float* __restrict__ out_val,
                                                         uint32_t cap) {
  constexpr int kTopkThreads = topk_threads(FINE);
  constexpr uint32_t kTopkWarps = kTopkThreads / 32;
  extern __shared__ __align__(16) unsigned char topk_dyn[];
  __shared__ TopkShared sh;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t C = gridDim.x, cta = blockIdx.x, tid = threadIdx.x;

  for (uint32_t b = tid; b < (uint32_t)kBins1; b += kTopkThreads) {
    sh.hist[b] = 0;
    if (cta == 0) sh.sum1[b] = sh.again1[b] = 0;
  }
  if (cta == 0)
    for (uint32_t b = tid; b < (uint32_t)kBins2; b += kTopkThreads) sh.sum2[b] = sh.sum3[b] = 0;
  if (tid == 0) {
    sh.short_cnt = sh.short_all = sh.together = 0;
    if (cta == 0) g_topk_status = 0;
  }
  __syncthreads();
  cl.barrier_arrive();            // the first CTA's sums are clear (waited for before anything is added to them)

  // sample -> bound
  uint32_t L = 0;
  {
    const uint32_t s = min(n, kTopkSample);
    uint32_t key = 0;
    for (uint32_t q = tid; q < s; q += kTopkThreads) {
      key = key_of(__ldg(x + (uint32_t)((uint64_t)q * n / s)));
      atomicAdd(sh.hist + (key >> 20), 1u);
    }
    __syncthreads();
    // Of k in n, k s / n are expected in the sample; four standard deviations and a few more, so that at least k
    // elements lie above the bound all but surely.  A sample of everything needs no margin.
    uint32_t want = k;
    if (s < n) {
      const float mean = (float)k * ((float)s / (float)n);
      want = (uint32_t)(mean + 4.f * sqrtf(mean)) + 8u;
    }
    uint32_t bin, need, found = s;
    if (topk_pick<kBins1, kTopkThreads>(sh.hist, want, bin, need, sh) >= want) {
      L = bin << 20;
      found = want - need + sh.res[2];
    }
    L = max(L, 1u);               // (zeros need no list: they are what is left if it is too short)
    // A warp has 32 neighbours of the sample.  If one has many more than its share of those that are at least L (half as many
    // again and 8, five standard deviations where they lie at random), large elements lie together in the vector.
    if (!FINE && __popc(__ballot_sync(kFull, key >= L)) >= 8u + found * 3u / 64u) sh.together = 1;
    for (uint32_t b = tid; b < (uint32_t)kBins1; b += kTopkThreads) sh.hist[b] = 0;
    __syncthreads();
  }
  const uint32_t tiles = C * kTopkWarps * 512u;   // elements of a tile for every warp
  if (!FINE && sh.together && n >= tiles && n <= tiles * kTopkTurns)
    topk_rest<FINE, !FINE>(x, n, k, out_idx, out_val, cap, L, sh, topk_dyn);
  else
    topk_rest<FINE, false>(x, n, k, out_idx, out_val, cap, L, sh, topk_dyn);
}

}  // namespace dgs
