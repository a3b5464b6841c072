// Device code of the DGS push / apply / pull loop for sm_100a.
//
// Selection scheme (used for the worker's top-k of the velocity, Algorithm 3, and
// for the server's top-k of the model difference, Algorithm 2 / Eq. 6a):
//
//   stream pass   one read of the input by all SMs.  Every element whose magnitude
//                 key is at least a per-layer lower bound L becomes a "candidate".
//                 A warp handles one tile of 512 elements at a time and appends the
//                 tile's candidates, in index order, as one "run" to its CTA's region
//                 of the candidate buffer.  Everything below L is final at once (the
//                 push writes t*(1/m) there).
//   finalize      one small kernel (a few dozen co-resident CTAs with a barrier of
//                 their own) over the candidates only: the histogram that the stream
//                 pass has counted gives the bin of the k-th largest, a list of that
//                 bin's candidates the exact k-th largest key T and the number r of
//                 entries equal to T that still fit; ranks by ballot write the packet
//                 in index order.
//
// L is a guess carried over from an earlier selection of the same kind on that layer
// (the host picks the most recent one made in a comparable state).  The guess is
// checked exactly (a layer needs at least k candidates).  With nothing to carry
// over, a histogram pass over the entire input comes first and gives a bound that
// cannot fail; when a guess fails, finalize redoes both passes itself.  The result
// never depends on the guess.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace dgs {

constexpr int kWarpTile = 512;      // elements per tile (one warp, 4 x float4 per lane)
constexpr int kVecIters = 4;
constexpr int kThreads = 256;       // threads per CTA in every kernel here
constexpr int kWarps = kThreads / 32;
constexpr int kBins1 = 2048;        // bins of a layer's histogram, see bin_of
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kSpecSlack = 64; // a carried bound aims at max(1.5 k, k + 64) candidates next time
constexpr int kMaxGrid = 512;       // upper bound on the grid of a stream pass (= parts of the candidate buffer)
constexpr int kMaxFoldGrid = 320;   // upper bound on the grid of a pull's pass (every warp of it is a part)
constexpr int kFoldWarps = 10;      // most warps of a CTA of a pull's pass
constexpr int kMaxParts = (kMaxFoldGrid * kFoldWarps + 255) / 256 * 256;   // upper bound on the parts of the candidate buffer (a multiple of kThreads)
constexpr uint32_t kFoldSlack = 64; // part_cap is at least that much longer than a CTA's share (its tables round to groups and words)
constexpr int kMaxWorkers = 320;    // upper bound on the grid of finalize
constexpr uint32_t kSpinLimit = 1u << 22;  // bounded waits: give up and report after this many polls
constexpr int kStatusTimeout = -4;  // = DGS_ETIMEOUT
constexpr int kNumStats = 8;        // words of Workspace::stats (every owner of a Workspace provides that many)

enum Mode : int { kPushSam = 0, kPushResidual = 1, kPull = 2 };

struct Tile {          // a run of <= kWarpTile elements inside one layer
  uint32_t start;
  uint16_t len;
  uint16_t seg;
};

struct SegDesc {
  uint32_t tile_begin, tile_end;  // tiles of this layer
  uint32_t k[2];                  // [0] push, [1] pull
  uint32_t pkt_off[2];            // exclusive prefix of k over layers
  uint32_t list_off, list_cap;    // the layer's place in Workspace::list
};

struct SegSel {        // per layer, finalize
  uint32_t prefix;     // radix levels over all candidates: key bits fixed so far
  uint32_t krem;       //   entries still to take at or below the fixed prefix
};

struct LayerPick {     // finalize: what a CTA knows of a layer that its candidates lie in
  uint32_t L;          // bound of the stream pass
  uint32_t bin, krem, pop;   // bin of the k-th largest, entries needed of it, entries in it (= on the layer's list)
  uint32_t T, r;       // k-th largest key; entries with key == T that are taken (lowest indices)
  uint32_t pkt_off, list_off;
  uint32_t start_gt, start_eq, start_warp;   // a layer that begins in this CTA: what that warp had counted before it
};

// word indices in Workspace::sync
// (the barrier's count and the flags of layers whose guesses failed: two pairs, which the selections on a scratch set take in
// turn, see SelArgs::pair)
enum SyncWord : int { kBarCount = 0, kFail = 2, kParts = 4, kPlanParts = 5, kNumSyncWords = 8 };

struct Workspace {
  const Tile* tiles;
  const SegDesc* segs;
  uint32_t num_tiles, num_segs;
  uint32_t n, n_pad;      // elements, and elements a state vector is padded to
  uint32_t num_blocks;    // blocks of kWarpTile elements (the last one may be partial)
  const uint32_t* blk_seg;   // [num_blocks] layer of the first element of each block
  // candidates: part p (CTA p of the grid that ran a push's stream pass, warp p of a pull's) owns the slots
  // starting at the first element of its first block (of its first tile, where a selection has started over)
  uint32_t* cand_idx;     // [n]
  float* cand_val;        // [n]
  uint32_t* part_cands;   // [kMaxParts] candidates written by each part
  uint32_t* part_slot0;   // [kMaxParts] first slot of each part
  // Pull: where the CTAs of the NEXT pass over a difference vector on this scratch set begin (blocks), planned
  // beside finalize from what this pass cost each CTA; plan[G] == num_blocks and sync[kPlanParts] == G mark it valid.
  uint32_t* plan;         // [kMaxFoldGrid + 1], or null
  uint32_t* cta_cost;     // [kMaxFoldGrid] cost of each CTA's share in the last pass
  uint32_t part_cap;      // most blocks a CTA of the pass can take
  const uint32_t* seg_off;   // [S+1] first element of each layer, and n
  uint2* cta_tot;         // [kMaxWorkers] finalize: last layer of each CTA's candidates; how many of them in it lie above the k-th's bin
  uint32_t* cta_eq;       // [kMaxWorkers] ... and equal T, where the lists were too short (then the count above is exact)
  LayerPick* tab;         // [S + kMaxWorkers] picks of CTAs with too many layers for shared memory
  uint2* list;            // candidates in the k-th's bin: (key, flat number), every layer at its own place
  uint32_t* list_cnt;     // [S]
  uint32_t* hist1;        // [S][kBins1]
  SegSel* sel;            // [S]
  uint32_t* L_safe;       // [S] bound from the whole-input histogram (two-pass route)
  uint32_t* L_wide;       // [S] from the same histogram: the bound that admits about max(1.5 k, k+64) entries
  uint32_t* sync;         // [kNumSyncWords]
  int* status;            // sticky device status word
  // [kNumStats] counters: [0] single-pass selections, [1] two-pass selections, [2] candidates seen,
  // [3] chunks of difference vectors covered by the pulls' stream passes, [4] those of them read
  unsigned long long* stats;
};

struct SelArgs {
  const float* grad;      // push: f32[n]
  float** u_cur_slot;     // push: device slot holding the worker's velocity pointer
  float** u_spare_slot;   // push: device slot holding the spare buffer pointer
  float* D;               // pull: D_w
  float* theta_local;     // pull: theta_w or null
  uint32_t* blk_max;      // pull: per block of kWarpTile elements, an upper bound on the keys of D_w in it (or null)
  const uint32_t* L_in;   // [S] lower bounds guessed for this selection (single-pass route)
  uint32_t* L_next;       // [S] receives the bounds this selection suggests for a later, similar one (not L_in)
  uint32_t* slack;        // [S] eighths of k that the bounds of selections of this kind aim beyond the usual number
  uint32_t* pkt_idx;
  float* pkt_val;
  uint32_t pkt_count;
  float m, lr, inv_m;
  int force_two_pass;
  int speculate;          // 0: never carry a bound (L_next is left alone)
  uint32_t workers;       // CTAs of finalize that process the candidates
  uint32_t advisers;      // further ones that check the guesses and suggest the next bounds
  uint32_t seq;           // selections of this kind launched before
  uint32_t pair;          // which of the two pairs of sync words this selection uses: 0 or 1, the one before it used the other
  uint32_t fold_grid;     // pull: CTAs of the pass before this finalize (0: it was not k_fold, nothing to plan)
  uint32_t phantom_workers;  // testing only: CTAs the finalize barrier waits for beyond those launched (0 in normal use)
  uint32_t spin_limit;    // polls after which a bounded wait gives up (0: kSpinLimit)
  int packet_format;      // 0: packets carry float32 values; 1: bfloat16; 2: binary16 (see round16)
};

__device__ __forceinline__ uint32_t key_of(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
// A packet value in a 16-bit floating-point format, as the float32 number with that value (round to
// nearest, ties to even).  fmt 1: bfloat16 (8 exponent bits, 7 fraction bits).  fmt 2: IEEE binary16
// (5 exponent bits, 10 fraction bits, gradual underflow); a magnitude that would round beyond the largest
// finite binary16 number is sent as that number, 65504.  fmt 0: the value itself.  Inputs are finite.
__device__ __forceinline__ float round16(float x, int fmt) {
  if (fmt == 0) return x;
  const uint32_t b = __float_as_uint(x);
  uint32_t m = b & 0x7FFFFFFFu;
  if (fmt == 1) {
    m = (m + 0x7FFFu + ((m >> 16) & 1u)) & 0xFFFF0000u;
    if (m >= 0x7F800000u) m = 0x7F7F0000u;
  } else if (m >= 0x477FF000u) {          // 65520 and above
    m = 0x477FE000u;                      // 65504
  } else if (m >= 0x38800000u) {          // 2^-14 and above: 13 fraction bits go
    m = (m + 0xFFFu + ((m >> 13) & 1u)) & 0xFFFFE000u;
  } else {
    // steps of 2^-24 below 2^-14: the multiple nearest to |x| (scaling by powers of two is exact)
    const float scaled = __fmul_rn(__uint_as_float(m), 16777216.0f);
    const int whole = (int)scaled;        // truncation; scaled < 1024
    const float frac = __fsub_rn(scaled, (float)whole);
    const int up = (frac > 0.5f || (frac == 0.5f && (whole & 1))) ? 1 : 0;
    m = __float_as_uint(__fmul_rn((float)(whole + up), 1.0f / 16777216.0f));
  }
  return __uint_as_float(m | (b & 0x80000000u));
}
// candidates a carried bound should admit for a selection of k entries
__device__ __forceinline__ uint32_t spec_want(uint32_t k) { return max(k + k / 2, k + kSpecSlack); }
// A bound inside a bin of the first-level histogram (key bits 30..20 = bin): `need` of the bin's `pop`
// entries are wanted, counted from the largest down; the bin's keys are taken as evenly spread over
// [lo, hi), lo being the bin's lower edge or the bound that was in force if that cut the bin.  A quarter
// more than needed is admitted.  Only advice for a later selection: results never depend on it.
__device__ __forceinline__ uint32_t bound_inside_bin(uint32_t bin, uint32_t need, uint32_t pop, uint32_t floor_key) {
  const uint32_t hi = (bin + 1u) << 20;
  uint32_t lo = bin << 20;
  if (floor_key > lo && floor_key < hi) lo = floor_key;
  const uint32_t width = hi - lo;
  const float f = fminf(1.f, 1.25f * (float)need / (float)max(pop, 1u) + 0.02f);
  const uint32_t take = (uint32_t)ceilf(f * (float)width);
  return hi - min(width, take);
}
// Histogram bin of a candidate of a layer with bound L (key >= L).  The bins start at the bound and widen with the distance
// from it: 2^8 keys up to a distance of 2^15 (a 256th of an octave), from there on a 128th of the distance's power of two.
// What was never sent piles up right below the k-th: after 8000 events on 25.6 M elements a bin of 2^14 keys held 1500 to
// 7700 of 47,000 candidates, and the finalize took 50 us instead of 25.  At any scale the k-th's bin now holds about a
// percent of the candidates between the bound and the k-th.  A bound near zero says nothing about where the candidates
// are: then the bins are the top 11 key bits.
constexpr uint32_t kBinLinear = 1u << 15, kBinOff = (127u + 15u) << 7;
__device__ __forceinline__ bool coarse_bins(uint32_t L) { return L < (1u << 25); }
__device__ __forceinline__ uint32_t bin_of(uint32_t key, uint32_t L) {
  if (coarse_bins(L)) return key >> 20;
  return min((uint32_t)kBins1 - 1u, (__float_as_uint(__uint2float_rz(key - L + kBinLinear)) >> 16) - kBinOff);
}
// lowest key of a bin, and how many low bits its keys differ in (the last one is open-ended: all keys)
__device__ __forceinline__ uint32_t bin_edge(uint32_t bin, uint32_t L) {
  if (coarse_bins(L)) return bin << 20;
  return L + ((uint32_t)__uint_as_float((bin + kBinOff) << 16) - kBinLinear);
}
__device__ __forceinline__ int bin_bits(uint32_t bin, uint32_t L) { return coarse_bins(L) ? 20 : 8 + (int)(bin >> 7); }
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}
__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) {
  return *reinterpret_cast<const volatile uint32_t*>(p);
}
__device__ __forceinline__ uint32_t part_first_tile(uint32_t part, uint32_t parts, uint32_t num_tiles) {
  return (uint32_t)((uint64_t)part * num_tiles / parts);
}

// ---- the value an element contributes to the selection ------------------------
// push (Algorithm 3):  t = fl(fl(m*u) + fl(eta*g));  Algorithm 1:  t = fl(u + fl(eta*g));  pull:  D.
template <int MODE>
__device__ __forceinline__ float combine(float u, float g, float m, float lr) {
  if (MODE == kPushSam) return __fadd_rn(__fmul_rn(m, u), __fmul_rn(lr, g));
  if (MODE == kPushResidual) return __fadd_rn(u, __fmul_rn(lr, g));
  return u;
}
// what a push stores for an element that is certainly not sent
template <int MODE>
__device__ __forceinline__ float unsent(float t, float inv_m) {
  return MODE == kPushSam ? __fmul_rn(t, inv_m) : t;
}

template <int MODE>
__device__ __forceinline__ void load_tile_vec(const float* __restrict__ a, const float* __restrict__ g,
                                              uint32_t start, int lane, float m, float lr,
                                              float (&x)[4 * kVecIters]) {
  const float4* pa = reinterpret_cast<const float4*>(a + start) + lane;
  float4 va[kVecIters];
#pragma unroll
  for (int j = 0; j < kVecIters; ++j) va[j] = __ldcs(pa + j * 32);
  if (MODE != kPull) {
    const float4* pg = reinterpret_cast<const float4*>(g + start) + lane;
    float4 vg[kVecIters];
#pragma unroll
    for (int j = 0; j < kVecIters; ++j) vg[j] = __ldcs(pg + j * 32);
#pragma unroll
    for (int j = 0; j < kVecIters; ++j) {
      x[4 * j + 0] = combine<MODE>(va[j].x, vg[j].x, m, lr);
      x[4 * j + 1] = combine<MODE>(va[j].y, vg[j].y, m, lr);
      x[4 * j + 2] = combine<MODE>(va[j].z, vg[j].z, m, lr);
      x[4 * j + 3] = combine<MODE>(va[j].w, vg[j].w, m, lr);
    }
  } else {
#pragma unroll
    for (int j = 0; j < kVecIters; ++j) {
      x[4 * j + 0] = va[j].x;
      x[4 * j + 1] = va[j].y;
      x[4 * j + 2] = va[j].z;
      x[4 * j + 3] = va[j].w;
    }
  }
}

// ---- stream pass ----------------------------------------------------------------
// Candidates are appended in INDEX ORDER: a CTA owns a contiguous range of tiles and a region
// of the candidate buffer; it takes its tiles in rounds of kWarps consecutive tiles (one per
// warp).  In a round every warp first counts the candidates of its tile, the counts are
// exchanged through shared memory, and each warp then writes its candidates behind those of the
// warps holding earlier tiles.  Read part after part, the candidate buffer therefore lists all
// candidates of the vector in ascending index order, which is what lets the finalize kernel
// number the selected ones with a plain prefix sum.
struct StreamShared {
  uint32_t hist[kBins1];      // candidates of the layer being processed, by bin_of
  uint32_t wcnt[2][kWarps];   // candidates per warp of the current round (two rounds alternate)
};

__device__ __forceinline__ void flush_hist(uint32_t* s_hist, uint32_t* g_hist) {
  for (int b = threadIdx.x; b < kBins1; b += kThreads) {
    const uint32_t v = s_hist[b];
    if (v) {
      atomicAdd(g_hist + b, v);
      s_hist[b] = 0;
    }
  }
}

// One more candidate in a bin of layer `seg`: in shared memory for the CTA's main layer, else straight in global memory.
__device__ __forceinline__ void count_bin(const Workspace& ws, uint32_t* s_hist, uint32_t main_seg, uint32_t seg, uint32_t bin) {
  if (seg == main_seg) atomicAdd(s_hist + bin, 1u); else atomicAdd(ws.hist1 + (size_t)seg * kBins1 + bin, 1u);
}

// candidates of warps 0 .. warp-1 in this round, and of all warps
__device__ __forceinline__ uint32_t round_offset(const uint32_t* wcnt, int warp, uint32_t& total) {
  uint32_t before = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = wcnt[w];
    if (w < warp) before += c;
    tot += c;
  }
  total = tot;
  return before;
}

// A full tile held in registers: x[16] are this lane's values (4 float4 at elements
// j*128 + lane*4 + c of the tile).  Returns the candidate mask; writes the new velocity (push).
template <int MODE>
__device__ __forceinline__ uint32_t tile_mask_regs(const SelArgs& a, uint32_t tile_start,
                                                   const float (&x)[4 * kVecIters], uint32_t L, int lane,
                                                   float* __restrict__ out) {
  uint32_t mask = 0;
#pragma unroll
  for (int e = 0; e < 4 * kVecIters; ++e)
    if (key_of(x[e]) >= L) mask |= 1u << e;
  if (MODE != kPull) {
    float4* po = reinterpret_cast<float4*>(out + tile_start) + lane;
#pragma unroll
    for (int j = 0; j < kVecIters; ++j) {
      float4 o;
      o.x = (mask >> (j * 4 + 0)) & 1 ? x[4 * j + 0] : unsent<MODE>(x[4 * j + 0], a.inv_m);
      o.y = (mask >> (j * 4 + 1)) & 1 ? x[4 * j + 1] : unsent<MODE>(x[4 * j + 1], a.inv_m);
      o.z = (mask >> (j * 4 + 2)) & 1 ? x[4 * j + 2] : unsent<MODE>(x[4 * j + 2], a.inv_m);
      o.w = (mask >> (j * 4 + 3)) & 1 ? x[4 * j + 3] : unsent<MODE>(x[4 * j + 3], a.inv_m);
      __stcs(po + j * 32, o);
    }
  }
  return mask;
}

// Writes the candidates of a full tile (mask from tile_mask_*) from slot `base` on, in index
// order, and histograms them.  The cost is proportional to the candidates: one
// packed warp scan gives every lane the rank of its candidates (lane l holds elements
// j*128 + l*4 + c, order is j-major, so the four per-j counts travel as four bytes of one
// word), and a lane that has candidates walks its set bits.  value(off) returns element `off`; count(off, key)
// adds a candidate to the histogram of its layer.
template <typename ValueFn, typename CountFn>
__device__ __forceinline__ void tile_emit(const Workspace& ws, uint32_t tile_start, uint32_t mask, uint32_t base, int lane,
                                          ValueFn value, CountFn count) {
  if (!__any_sync(kFull, mask != 0)) return;
  // per-j candidate counts of this lane, one per byte
  uint32_t t = mask - ((mask >> 1) & 0x5555u);
  t = (t & 0x3333u) + ((t >> 2) & 0x3333u);                       // nibble j = count of nibble j of mask
  const uint32_t packed = (t & 0xFu) | ((t & 0xF0u) << 4) | ((t & 0xF00u) << 8) | ((t & 0xF000u) << 12);
  uint32_t incl = packed;                                          // byte j: inclusive prefix over lanes (<= 128)
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  const uint32_t tot = __shfl_sync(kFull, incl, 31);
  const uint32_t t0 = tot & 0xFFu, t1 = (tot >> 8) & 0xFFu, t2 = (tot >> 16) & 0xFFu;
  if (mask) {
    const uint32_t excl = incl - packed;                           // byte j: candidates of lower lanes at step j
    uint32_t m = mask;
    while (m) {
      const int e = __ffs(m) - 1;
      m &= m - 1;
      const int j = e >> 2, c = e & 3;
      const uint32_t before_j = j == 0 ? 0u : (j == 1 ? t0 : (j == 2 ? t0 + t1 : t0 + t1 + t2));
      const uint32_t in_lane = __popc((mask >> (4 * j)) & ((1u << c) - 1u));
      const uint32_t pos = base + before_j + ((excl >> (8 * j)) & 0xFFu) + in_lane;
      const uint32_t off = j * 128 + lane * 4 + c;
      const float v = value(off);
      ws.cand_idx[pos] = tile_start + off;
      ws.cand_val[pos] = v;
      count(off, key_of(v));
    }
  }
}

// A ragged tile (first or last of a layer, fewer than kWarpTile elements or not 16-byte
// aligned): one element per lane and step, straight from global memory, at most 16 steps, the
// loads of eight steps in flight together.  Returns the candidate flags (one bit per step) and
// leaves the values of this lane's elements in x[step]; writes the new velocity (push).
constexpr int kRaggedSteps = kWarpTile / 32;
template <int MODE>
__device__ __forceinline__ uint32_t ragged_mask(const SelArgs& a, const Tile tile, uint32_t L, int lane,
                                                const float* __restrict__ in, float* __restrict__ out,
                                                float (&x)[kRaggedSteps]) {
  uint32_t flags = 0;
#pragma unroll
  for (int s0 = 0; s0 < kRaggedSteps; s0 += 8) {
    if (s0 * 32 < (int)tile.len) {   // warp-uniform
      float vu[8], vg[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t off = (s0 + j) * 32 + lane;
        vu[j] = 0.f;
        vg[j] = 0.f;
        if (off < tile.len) {
          vu[j] = in[tile.start + off];
          if (MODE != kPull) vg[j] = a.grad[tile.start + off];
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t off = (s0 + j) * 32 + lane;
        x[s0 + j] = 0.f;
        if (off < tile.len) {
          const float v = combine<MODE>(vu[j], vg[j], a.m, a.lr);
          const bool cand = key_of(v) >= L;
          if (MODE != kPull) out[tile.start + off] = cand ? v : unsent<MODE>(v, a.inv_m);
          if (cand) flags |= 1u << (s0 + j);
          x[s0 + j] = v;
        }
      }
    }
  }
  return flags;
}
// Writes its candidates from slot `base` on, in index order.
__device__ __forceinline__ void ragged_emit(const Workspace& ws, StreamShared& sh, const Tile tile, uint32_t flags, uint32_t L,
                                            uint32_t base, int lane, uint32_t lt, const float (&x)[kRaggedSteps]) {
  if (!__any_sync(kFull, flags != 0)) return;
#pragma unroll
  for (int st = 0; st < kRaggedSteps; ++st) {
    if (st * 32 < (int)tile.len) {   // warp-uniform
      const bool cand = (flags >> st) & 1u;
      const uint32_t b = __ballot_sync(kFull, cand);
      if (cand) {
        const uint32_t pos = base + __popc(b & lt);
        ws.cand_idx[pos] = tile.start + st * 32 + lane;
        ws.cand_val[pos] = x[st];
        atomicAdd(sh.hist + bin_of(key_of(x[st]), L), 1u);
      }
      base += __popc(b);
    }
  }
}

// CTA `cta` of `G` handles a contiguous range of tiles, kWarps consecutive tiles per round,
// layer by layer, so that the CTA's shared histogram always belongs to one layer; it is added
// to the global one when the CTA leaves the layer.  Loads go straight from global memory to
// registers (used where only a few CTAs run the pass).
template <int MODE>
__device__ void stream_tiles(const Workspace& ws, const SelArgs& a, const uint32_t* Larr,
                             const float* __restrict__ in, float* __restrict__ out, uint32_t cta, uint32_t G,
                             StreamShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t t0 = part_first_tile(cta, G, ws.num_tiles), t1 = part_first_tile(cta + 1, G, ws.num_tiles);
  const uint32_t lt = lanemask_lt();
  for (int b = threadIdx.x; b < kBins1; b += kThreads) sh.hist[b] = 0;
  if (cta == 0 && threadIdx.x == 0) ws.sync[kParts] = G;
  __syncthreads();
  if (t0 >= t1) {
    if (threadIdx.x == 0) {
      ws.part_cands[cta] = 0;
      ws.part_slot0[cta] = 0;
    }
    return;
  }
  const uint32_t slot0 = ws.tiles[t0].start;  // first slot of this CTA's region
  const uint32_t seg_first = ws.tiles[t0].seg, seg_last = ws.tiles[t1 - 1].seg;
  uint32_t cur = 0;      // candidates appended so far (the same in every thread)
  uint32_t round = 0;
  for (uint32_t s = seg_first; s <= seg_last; ++s) {
    const uint32_t a0 = max(t0, ws.segs[s].tile_begin), a1 = min(t1, ws.segs[s].tile_end);
    const uint32_t L = Larr[s];
    for (uint32_t tb = a0; tb < a1; tb += kWarps, ++round) {
      const uint32_t t = tb + warp;
      Tile tile;
      tile.start = 0; tile.len = 0; tile.seg = 0;
      float x[4 * kVecIters];
      uint32_t mask = 0;
      if (t < a1) {
        tile = ws.tiles[t];
        if (tile.len == kWarpTile) {
          load_tile_vec<MODE>(in, a.grad, tile.start, lane, a.m, a.lr, x);
          mask = tile_mask_regs<MODE>(a, tile.start, x, L, lane, out);
        } else {
          mask = ragged_mask<MODE>(a, tile, L, lane, in, out, x);
        }
      }
      const uint32_t count = __reduce_add_sync(kFull, (uint32_t)__popc(mask));
      if (lane == 0) sh.wcnt[round & 1][warp] = count;
      __syncthreads();
      uint32_t total;
      const uint32_t base = slot0 + cur + round_offset(sh.wcnt[round & 1], warp, total);
      cur += total;
      if (t < a1) {
        if (tile.len == kWarpTile) {
          tile_emit(ws, tile.start, mask, base, lane, [&](uint32_t off) {
            // element off = j*128 + lane*4 + c is register 4*j + c of this lane
            const int e = (int)(((off >> 7) << 2) | (off & 3u));
            float v = x[0];
#pragma unroll
            for (int q = 1; q < 4 * kVecIters; ++q)
              if (q == e) v = x[q];
            return v;
          }, [&](uint32_t, uint32_t key) { atomicAdd(sh.hist + bin_of(key, L), 1u); });
        } else {
          ragged_emit(ws, sh, tile, mask, L, base, lane, lt, x);
        }
      }
    }
    __syncthreads();
    flush_hist(sh.hist, ws.hist1 + (size_t)s * kBins1);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    ws.part_cands[cta] = cur;
    ws.part_slot0[cta] = slot0;
  }
}

// Step one for a tile of a push staged in shared memory (su: the tile of the state vector, sg: the tile of the
// gradient): candidate mask, new velocity.
template <int MODE>
__device__ __forceinline__ uint32_t tile_mask_smem(const SelArgs& a, uint32_t tile_start, const float* su,
                                                   const float* sg, uint32_t L, int lane, float* __restrict__ out) {
  const float Lf = __uint_as_float(L);   // |x| >= Lf  <=>  key(x) >= L for finite x (no flush-to-zero)
  const float4* pu = reinterpret_cast<const float4*>(su) + lane;
  const float4* pg = reinterpret_cast<const float4*>(sg) + lane;
  uint32_t mask = 0;
#pragma unroll
  for (int j = 0; j < kVecIters; ++j) {
    float4 x = pu[j * 32];
    const float4 g = pg[j * 32];
    x.x = combine<MODE>(x.x, g.x, a.m, a.lr);
    x.y = combine<MODE>(x.y, g.y, a.m, a.lr);
    x.z = combine<MODE>(x.z, g.z, a.m, a.lr);
    x.w = combine<MODE>(x.w, g.w, a.m, a.lr);
    const bool c0 = fabsf(x.x) >= Lf, c1 = fabsf(x.y) >= Lf, c2 = fabsf(x.z) >= Lf, c3 = fabsf(x.w) >= Lf;
    mask |= ((c0 ? 1u : 0u) | (c1 ? 2u : 0u) | (c2 ? 4u : 0u) | (c3 ? 8u : 0u)) << (4 * j);
    float4 o;
    o.x = c0 ? x.x : unsent<MODE>(x.x, a.inv_m);
    o.y = c1 ? x.y : unsent<MODE>(x.y, a.inv_m);
    o.z = c2 ? x.z : unsent<MODE>(x.z, a.inv_m);
    o.w = c3 ? x.w : unsent<MODE>(x.w, a.inv_m);
    __stcs(reinterpret_cast<float4*>(out + tile_start) + lane + j * 32, o);
  }
  return mask;
}

// ---- the same pass with TMA-staged tiles --------------------------------------------
// Blocks of kWarpTile elements are brought into a ring of shared-memory stages by bulk asynchronous copies
// (cp.async.bulk, completion counted on an mbarrier per stage), one per warp of each
// input per stage, so that several stages are in flight while the warps work on one: the
// bytes in flight no longer depend on how many warps are waiting at a load.  One round of the
// ordered append = one stage; the barrier between counting and writing is also the one after
// which the stage of the round before is free, so a ring of kStages stages keeps kStages - 1
// of them in flight.
constexpr int kStageFloats = kWarps * kWarpTile;           // per input array: one block per warp and stage
// The ring: three stages (96 KB, two CTAs per SM, 128 KB of the SM's shared memory in flight); two where the pass is short.
template <int STAGES>
struct StreamRing {
  static constexpr int kStages = STAGES;
  static constexpr int kStageBytes = 2 * kStageFloats * 4;                // 16 KB per input
  static constexpr int kBytes = kStages * kStageBytes;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// bounded wait: false if the copies did not land within the poll limit
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
  for (; limit; --limit)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
// global -> shared bulk copy; src and dst 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

// The layers that elements [base, base + len) lie in, `seg` the first of them: calls fn(layer, lo, hi, its bound) for each in
// turn, elements base + lo .. base + hi - 1 being that layer's.  By a warp; 32 layers are looked up in one trip.
template <typename Fn>
__device__ __forceinline__ void each_layer(const Workspace& ws, const uint32_t* Larr, uint32_t seg, uint32_t base, uint32_t len,
                                           Fn fn) {
  uint32_t lo = 0;
  for (uint32_t s0 = seg;; s0 += 32) {
    const uint32_t s = min(s0 + (threadIdx.x & 31u), ws.num_segs - 1u);
    const uint32_t end = min(__ldg(ws.seg_off + s + 1) - base, len), L = Larr[s];
#pragma unroll 1
    for (uint32_t j = 0; j < 32; ++j) {
      const uint32_t hi = __shfl_sync(kFull, end, j);
      fn(s0 + j, lo, hi, __shfl_sync(kFull, L, j));
      if (hi == len) return;
      lo = hi;
    }
  }
}
// A block that lies in several layers, or the vector's last, shorter one (a warp; element st * 32 + lane of the block is bit
// st of the lane): every element is compared with the bound of its own layer.  su, sg: the block of the state vector and of
// the gradient, in shared or global memory; seg: layer of its first element.  Returns the candidates, writes the new velocity.
template <int MODE>
__device__ __noinline__ uint32_t mixed_mask(const Workspace& ws, const SelArgs& a, const uint32_t* Larr, const float* su,
                                            const float* sg, float* out, uint32_t base, uint32_t len, uint32_t seg) {
  const uint32_t lane = threadIdx.x & 31u;
  float x[kRaggedSteps];
#pragma unroll
  for (int st = 0; st < kRaggedSteps; ++st) {
    const uint32_t off = st * 32u + lane;
    x[st] = off < len ? combine<MODE>(su[off], sg[off], a.m, a.lr) : 0.f;
  }
  uint32_t mask = 0;
  each_layer(ws, Larr, seg, base, len, [&](uint32_t, uint32_t lo, uint32_t hi, uint32_t L) {
    const float Lf = __uint_as_float(L);   // |x| >= Lf  <=>  key(x) >= L for finite x (no flush-to-zero)
#pragma unroll
    for (int st = 0; st < kRaggedSteps; ++st) {
      const uint32_t off = st * 32u + lane;
      if (off >= lo && off < hi && fabsf(x[st]) >= Lf) mask |= 1u << st;
    }
  });
#pragma unroll
  for (int st = 0; st < kRaggedSteps; ++st) {
    const uint32_t off = st * 32u + lane;
    if (off < len) out[base + off] = (mask >> st) & 1u ? x[st] : unsent<MODE>(x[st], a.inv_m);
  }
  return mask;
}
// Writes its candidates from slot `pos` on, in index order; those of layer main_seg are counted in `hist`.
template <int MODE>
__device__ __noinline__ void mixed_emit(const Workspace& ws, const SelArgs& a, const uint32_t* Larr, uint32_t mask, const float* su,
                                        const float* sg, uint32_t base, uint32_t len, uint32_t seg, uint32_t pos, uint32_t main_seg,
                                        uint32_t* hist) {
  const uint32_t lane = threadIdx.x & 31u, lt = lanemask_lt();
  each_layer(ws, Larr, seg, base, len, [&](uint32_t s, uint32_t lo, uint32_t hi, uint32_t L) {
#pragma unroll 2
    for (uint32_t st = lo / 32u; st * 32u < hi; ++st) {
      const uint32_t off = st * 32u + lane;
      const bool cand = ((mask >> st) & 1u) && off >= lo && off < hi;
      const uint32_t b = __ballot_sync(kFull, cand);
      if (cand) {
        const uint32_t to = pos + __popc(b & lt);
        const float v = combine<MODE>(su[off], sg[off], a.m, a.lr);
        ws.cand_idx[to] = base + off;
        ws.cand_val[to] = v;
        count_bin(ws, hist, main_seg, s, bin_of(key_of(v), L));
      }
      pos += __popc(b);
    }
  });
}

// The pass runs over the blocks of the flat vector, kWarps of them a round, and takes no notice of where layers begin: a
// block inside one layer is compared with that layer's bound, one that lies in several element by element, and the ring
// never runs empty in between.  The candidates of the layer in the middle of the CTA's share are counted in shared memory,
// those of others straight in global memory.  (A layer at a time, the ring restarted and the histogram flushed for each and
// one warp at work on its ragged ends, 11.7 M elements in 62 layers took 54 us, and the CTAs with the small layers 58 us where
// the others took 24; now 37 us.)
// If a copy does not land in time the status word says so and *s_dead is set: the CTA's counts are then not complete, and a late
// copy may still write to the ring.  `phantom` is for tests: arrivals that the last CTA's copies wait for and that never come.
template <int MODE, typename R>
__device__ void stream_blocks_tma(const Workspace& ws, const SelArgs& a, const uint32_t* Larr, const float* __restrict__ in,
                                  float* __restrict__ out, uint32_t cta, uint32_t G, StreamShared& sh, float* ring, uint64_t* full,
                                  int* s_dead, uint32_t phantom, uint32_t spin_limit) {
  static_assert(MODE != kPull, "a pull's pass is k_fold");
  static_assert(R::kStages >= 2, "the ring needs a stage in flight besides the one being read");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t NB = ws.num_blocks, S = ws.num_segs, n = ws.n, whole_blocks = n / kWarpTile;
  const uint32_t t0 = part_first_tile(cta, G, NB), t1 = part_first_tile(cta + 1, G, NB);
  const uint32_t f1 = min(t1, whole_blocks);    // blocks [t0, f1) come through the ring; the vector's last one may be shorter
  const uint32_t rounds = (t1 - t0 + kWarps - 1) / kWarps;
  auto issue = [&](uint32_t r) {                // thread 0 only; round r has a whole block
    const uint32_t st = r % R::kStages, first = t0 + r * kWarps;
    const uint32_t bytes = min((uint32_t)kWarps, f1 - first) * kWarpTile * 4;
    const size_t elem = (size_t)first * kWarpTile;
    float* dst = ring + (size_t)st * (R::kStageBytes / 4);
    mbar_expect_tx(full + st, bytes * 2);
    bulk_load(dst, in + elem, bytes, full + st);
    bulk_load(dst + kStageFloats, a.grad + elem, bytes, full + st);
  };
  auto fetched = [&](uint32_t r) { return t0 + r * kWarps < f1; };   // (the shorter block may be alone in its round)
  if (threadIdx.x == 0) {
    *s_dead = 0;
    if (cta == 0) ws.sync[kParts] = G;
    for (int st = 0; st < R::kStages; ++st) mbar_init(full + st, 1u + (cta + 1 == G ? phantom : 0u));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (uint32_t r = 0; r < (uint32_t)R::kStages - 1 && r < rounds && fetched(r); ++r) issue(r);
  }
  for (int b = threadIdx.x; b < kBins1; b += kThreads) sh.hist[b] = 0;
  const uint32_t slot0 = t0 * kWarpTile;        // first slot of this CTA's region
  const uint32_t main_seg = S == 1 || t0 >= t1 ? 0u : __ldg(ws.blk_seg + t0 + (t1 - t0) / 2);
  // layer of the first element of this warp's block
  uint32_t seg = S == 1 || t0 + warp >= t1 ? 0u : __ldg(ws.blk_seg + t0 + warp);
  uint32_t seg_end = S == 1 ? n : __ldg(ws.seg_off + seg + 1), L = Larr[seg];
  __syncthreads();
  uint32_t cur = 0;   // candidates appended so far (same in every thread)
  for (uint32_t r = 0; r < rounds; ++r) {
    const uint32_t st = r % R::kStages, blk = t0 + r * kWarps + warp, base = blk * kWarpTile;
    if (blk < t1 && base >= seg_end) {
      seg = __ldg(ws.blk_seg + blk);
      seg_end = __ldg(ws.seg_off + seg + 1);
      L = Larr[seg];
    }
    const bool landed = !fetched(r) || mbar_wait(full + st, (r / R::kStages) & 1u, spin_limit);
    if (!landed) *s_dead = 1;
    const float* const su = ring + (size_t)st * (R::kStageBytes / 4) + warp * kWarpTile;
    const bool plain = blk < f1 && base + kWarpTile <= seg_end;
    uint32_t mask = 0;
    if (blk < t1 && landed) {
      if (plain) {
        mask = tile_mask_smem<MODE>(a, base, su, su + kStageFloats, L, lane, out);
      } else {                                  // (the shorter block straight from global memory)
        mask = mixed_mask<MODE>(ws, a, Larr, blk < f1 ? su : in + base, blk < f1 ? su + kStageFloats : a.grad + base, out, base,
                                min((uint32_t)kWarpTile, n - base), seg);
      }
    }
    const uint32_t count = __reduce_add_sync(kFull, (uint32_t)__popc(mask));
    if (lane == 0) sh.wcnt[r & 1][warp] = count;
    __syncthreads();   // the counts of this round are known, and every warp has left the stage of the round before
    if (*s_dead) break;
    const uint32_t ahead = r + R::kStages - 1;
    if (threadIdx.x == 0 && ahead < rounds && fetched(ahead)) issue(ahead);   // into the stage of the round before
    uint32_t total;
    const uint32_t pos = slot0 + cur + round_offset(sh.wcnt[r & 1], warp, total);
    cur += total;
    if (count == 0) continue;
    if (plain) {
      tile_emit(ws, base, mask, pos, lane, [&](uint32_t off) { return combine<MODE>(su[off], su[kStageFloats + off], a.m, a.lr); },
                [&](uint32_t, uint32_t key) { count_bin(ws, sh.hist, main_seg, seg, bin_of(key, L)); });
    } else {
      mixed_emit<MODE>(ws, a, Larr, mask, blk < f1 ? su : in + base, blk < f1 ? su + kStageFloats : a.grad + base, base,
                       min((uint32_t)kWarpTile, n - base), seg, pos, main_seg, sh.hist);
    }
  }
  __syncthreads();
  if (*s_dead) {
    // a copy did not land in time: report, give the copies still in flight one more bounded wait, leave
    if (threadIdx.x == 0) {
      atomicMin(ws.status, kStatusTimeout);
      for (int st = 0; st < R::kStages; ++st) {
        mbar_wait(full + st, 0, spin_limit);
        mbar_wait(full + st, 1, spin_limit);
      }
    }
    __syncthreads();
  } else {
    flush_hist(sh.hist, ws.hist1 + (size_t)main_seg * kBins1);
  }
  if (threadIdx.x == 0) {
    ws.part_cands[cta] = cur;
    ws.part_slot0[cta] = slot0;
  }
}

// ---- histogram of ALL elements (top 11 key bits), for the bound that cannot fail ----
// Adds one warp-wide batch of bins to the shared histogram.  Lanes holding the same
// bin as lane 0's are counted with one ballot (values cluster in few bins: zeros in a
// sparse difference vector, the bulk of a bell-shaped gradient); the rest use atomics.
__device__ __forceinline__ void hist_add(uint32_t* s_hist, uint32_t bin, bool valid, int lane) {
  const uint32_t lead = __shfl_sync(kFull, bin, 0);
  const bool same = valid && bin == lead;
  const uint32_t b = __ballot_sync(kFull, same);
  if (lane == 0 && b) atomicAdd(s_hist + lead, (uint32_t)__popc(b));
  if (valid && !same) atomicAdd(s_hist + bin, 1u);
}

template <int MODE>
__device__ void hist_all_tiles(const Workspace& ws, const SelArgs& a, const float* __restrict__ in,
                               uint32_t cta, uint32_t G, uint32_t* s_hist) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t t0 = part_first_tile(cta, G, ws.num_tiles), t1 = part_first_tile(cta + 1, G, ws.num_tiles);
  for (int b = threadIdx.x; b < kBins1; b += kThreads) s_hist[b] = 0;
  __syncthreads();
  if (t0 >= t1) return;
  const uint32_t seg_first = ws.tiles[t0].seg, seg_last = ws.tiles[t1 - 1].seg;
  for (uint32_t s = seg_first; s <= seg_last; ++s) {
    const uint32_t a0 = max(t0, ws.segs[s].tile_begin), a1 = min(t1, ws.segs[s].tile_end);
    for (uint32_t t = a0 + warp; t < a1; t += kWarps) {
      const Tile tile = ws.tiles[t];
      if (tile.len == kWarpTile) {
        float x[4 * kVecIters];
        load_tile_vec<MODE>(in, a.grad, tile.start, lane, a.m, a.lr, x);
#pragma unroll
        for (int e = 0; e < 4 * kVecIters; ++e) hist_add(s_hist, key_of(x[e]) >> 20, true, lane);
      } else {
        for (uint32_t base = 0; base < tile.len; base += 32) {
          const uint32_t off = base + lane;
          const bool valid = off < tile.len;
          float x = 0.f;
          if (valid) {
            const uint32_t i = tile.start + off;
            x = combine<MODE>(in[i], MODE != kPull ? a.grad[i] : 0.f, a.m, a.lr);
          }
          hist_add(s_hist, key_of(x) >> 20, valid, lane);
        }
      }
    }
    __syncthreads();
    flush_hist(s_hist, ws.hist1 + (size_t)s * kBins1);
    __syncthreads();
  }
}

// ---- block-wide helpers (kThreads threads) -----------------------------------------
// exclusive scan of one 64-bit value per thread; `total` is the block sum
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long v, unsigned long long* s_warp,
                                                              unsigned long long& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long inc = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long o = __shfl_up_sync(kFull, inc, d);
    if (lane >= d) inc += o;
  }
  __syncthreads();  // s_warp may still be read from a previous call
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  unsigned long long base = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const unsigned long long x = s_warp[w];
    if (w < warp) base += x;
    tot += x;
  }
  total = tot;
  return base + inc - v;
}

// From a histogram of B bins finds, counting from the top bin down, the bin that
// holds the k-th entry.  Returns total count; bin/krem are valid when total >= k:
// krem = k minus the entries in bins above `bin` (1 <= krem <= hist[bin]).
template <int B>
__device__ uint32_t block_pick(const uint32_t* hist, uint32_t k, uint32_t& bin, uint32_t& krem,
                               unsigned long long* s_warp, uint32_t* s_res) {
  constexpr int PER = B / kThreads;
  uint32_t loc[PER];
  uint32_t sum = 0;
  // thread 0 owns the top PER bins, thread 1 the next PER, ...
  const int top = B - 1 - threadIdx.x * PER;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    loc[j] = __ldcg(hist + top - j);
    sum += loc[j];
  }
  unsigned long long total;
  const uint32_t above = (uint32_t)block_excl_scan(sum, s_warp, total);
  if (above < k && k <= above + sum) {
    uint32_t acc = above;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (acc < k && k <= acc + loc[j]) {
        s_res[0] = (uint32_t)(top - j);
        s_res[1] = k - acc;
        s_res[2] = loc[j];
      }
      acc += loc[j];
    }
  }
  __syncthreads();
  bin = s_res[0];
  krem = s_res[1];
  __syncthreads();
  return (uint32_t)total;
}

// Flat numbering of the candidates over the parts: pre[p] = candidates of the parts before p (pre[parts] = all of
// them), in shared memory; ends with a barrier.
template <int MAXPARTS>
__device__ __forceinline__ void number_parts(const Workspace& ws, uint32_t parts, uint32_t* pre, unsigned long long* s_warp) {
  constexpr int PER = MAXPARTS / kThreads;
  static_assert(MAXPARTS % kThreads == 0, "the same number of parts for every thread");
  uint32_t v[PER], sum = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) v[j] = j * kThreads + threadIdx.x < parts ? __ldcg(ws.part_cands + j * kThreads + threadIdx.x) : 0u;
#pragma unroll
  for (int j = 0; j < PER; ++j) pre[j * kThreads + threadIdx.x] = v[j];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    v[j] = pre[threadIdx.x * PER + j];
    sum += v[j];
  }
  unsigned long long total;
  uint32_t at = (uint32_t)block_excl_scan(sum, s_warp, total);
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    pre[threadIdx.x * PER + j] = at;
    at += v[j];
  }
  if (threadIdx.x == 0) pre[parts] = (uint32_t)total;   // (the owner of that place writes the same)
  __syncthreads();
}

// From the histogram of a whole layer (top 11 key bits; cleared here): L_safe = lower edge of the bin holding the k-th
// largest key, L_wide = a bound that admits about max(1.5 k, k+64) entries.  By one CTA.
static __device__ void pick_lower(const Workspace& ws, uint32_t s, uint32_t k, unsigned long long* s_warp, uint32_t* s_res) {
  uint32_t bin, krem, wbin = 0, wrem = 0;
  uint32_t* const h = ws.hist1 + (size_t)s * kBins1;
  const uint32_t want = spec_want(k), total = block_pick<kBins1>(h, k, bin, krem, s_warp, s_res);
  if (total >= want) block_pick<kBins1>(h, want, wbin, wrem, s_warp, s_res);
  if (threadIdx.x == 0) {
    ws.L_safe[s] = bin << 20;
    // 0 (everything) when the layer has fewer than `want` entries
    ws.L_wide[s] = total >= want ? bound_inside_bin(wbin, wrem, __ldcg(h + wbin), 0u) : 0u;
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kBins1; b += kThreads) h[b] = 0;
}

// Barrier among the CTAs of finalize (all resident: cooperative launch).  One arrival
// counter that only grows: the i-th barrier of a launch is passed when the counter has
// reached i*W (it is cleared by the pass before finalize, or, where both are one kernel, by the selection before).
// Bounded: returns false, with the status word set, if the others do not arrive.
static __device__ bool worker_barrier(uint32_t* count, uint32_t W, int* status, int* s_ok, uint32_t& target,
                               uint32_t limit = kSpinLimit) {
  target += W;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    atomicAdd(count, 1u);
    uint32_t spins = 0;
    while ((int32_t)(ld_volatile(count) - target) < 0) {
      if (++spins > limit) {
        ok = 0;
        atomicMin(status, kStatusTimeout);
        break;
      }
    }
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// ---- finalize -------------------------------------------------------------------
// The candidates are numbered flat over the parts: part p holds part_cands[p] of them in consecutive slots from
// part_slot0[p] on.  Parts follow one another in index order and every part lists its candidates in index order, so
// the flat numbering is the index order of all candidates.  Every warp owns a run of consecutive flat candidates, 32
// of them at a time, kept in registers when they are few:
//   pick    every CTA finds, in the histograms of the layers its candidates lie in, the bin of the k-th largest
//   list    the candidates of that bin, and where they stand, go to a short list of the layer.  The bins are fine
//           (see bin_of), so the list is about a percent of the candidates.  Candidates above the bin are counted per warp
//   -- the only barrier among the CTAs --
//   exact   a radix selection over the list (a warp per layer) gives the k-th largest key T and the tie quota r.
//           With the counts above the bin and the places on the list every warp knows how many selected entries
//           stand before its candidates
//   emit    ranks by ballot  ->  packet in index order, state updates
// A few more CTAs check the guesses and work out the next bounds meanwhile, so that this is not on the way.
// What bounds it is the chain of trips to L2, and the fetching of instructions that run once (39 % of a warp's time in a
// form that kept four candidates a lane in unrolled code for any number of layers), not bytes.  So there are few
// phases, a variant for one layer and one for several, little unrolling, and the rare paths stay out of line.
// Measured between events (about 6 us of that is the events'), against three radix levels over global histograms with
// three barriers (one layer) or eight (several): 25 K of 47 K candidates, one layer: 23-26 us for 33-35; 120 K of 200 K,
// 62 layers: 40-42 us for 56-57; 148 layers: 50-57 us for 73-78; 670 K of 1 M, one layer: 63 us for 93.
constexpr int kSegCap = 1024;   // layers whose offsets fit in shared memory; more are looked up in global memory
// candidates a lane keeps in registers between the phases, and loads at a time
__host__ __device__ constexpr int finalize_keep(bool many) { return many ? 4 : 2; }
constexpr int kTouch = 40;      // layers of a CTA whose picks fit in shared memory; more are kept in global memory

constexpr int kListSmem = kThreads;    // entries of the list that are ranked in shared memory (one layer)
template <int MAXPARTS>
struct __align__(16) FinalizeShared {
  StreamShared stream;                 // redo of the passes (guess failed); its histogram also serves the warps' radix steps
  int ok;                              // (behind warp_scan instead, finalize spills up to a third more: alone, 25.6 M elements: 122.2 us, 123.6)
  unsigned long long warp_scan[kWarps];
  uint32_t res[3];
  uint32_t range[3];                   // layers of the candidate before this CTA's, of its first and of its last one
  uint32_t gt[kWarps], eq[kWarps];     // what each warp has counted
  LayerPick tab[kTouch];
  uint32_t pre[MAXPARTS + 1];          // exclusive prefix of part_cands
};
static_assert(kWarps * 128 <= kBins1, "a radix step of every warp fits the histogram's place");
static_assert(2 * kListSmem <= kBins1, "and so does the list");
// offsets of the layers in dynamic shared memory
__host__ __device__ inline uint32_t finalize_dyn_bytes(uint32_t S) {
  return S <= (uint32_t)kSegCap ? 4u * (S + 1u) : 0u;
}

// layer in [lo, hi] that holds element i: last s with off[s] <= i
__device__ __forceinline__ uint32_t seg_of(const uint32_t* off, uint32_t lo, uint32_t hi, uint32_t i) {
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}
// last part in [lo, hi] with pre[part] <= p
__device__ __forceinline__ uint32_t part_of(const uint32_t* pre, uint32_t lo, uint32_t hi, uint32_t p) {
#pragma unroll 1
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= p) lo = mid; else hi = mid - 1;
  }
  return lo;
}
// the same over all parts, found by a whole warp, 32 probes at a time (p the same in every lane)
__device__ __forceinline__ uint32_t warp_part_of(const uint32_t* pre, uint32_t parts, uint32_t p, int lane) {
  uint32_t lo = 0, span = parts;                 // the answer lies in [lo, lo + span)
#pragma unroll 1
  while (span > 1) {
    const uint32_t step = (span + 31u) / 32u, at = lo + lane * step;
    const uint32_t c = __popc(__ballot_sync(kFull, lane * step < span && pre[at] <= p));   // >= 1: pre[lo] <= p
    span = min(step, span - (c - 1u) * step);
    lo += (c - 1u) * step;
  }
  return lo;
}

// From a layer's histogram, counting from the top bin down, the bin that holds the k-th entry; by one warp.
struct BinPick { uint32_t bin, rem, pop; };   // rem: entries needed of the bin; pop: entries in it
// lane `lane` of the warp holds bins kBins1 - 64 (lane + 1) .. kBins1 - 1 - 64 lane: how many entries
__device__ __forceinline__ uint32_t lane_bins(const uint32_t* h, int lane) {
  const uint4* q = reinterpret_cast<const uint4*>(h + kBins1 - 64 * (lane + 1));
  uint32_t sum = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint4 x = __ldcg(q + j);
    sum += x.x + x.y + x.z + x.w;
  }
  return sum;
}
__device__ __forceinline__ uint32_t warp_incl(uint32_t v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, v, d);
    if (lane >= d) v += o;
  }
  return v;
}
// incl: inclusive prefix over the lanes of lane_bins; k <= its total
__device__ __forceinline__ BinPick warp_pick(const uint32_t* h, uint32_t incl, uint32_t own, uint32_t k, int lane) {
  const uint32_t src = __ffs(__ballot_sync(kFull, incl >= k)) - 1u;
  const uint32_t above = __shfl_sync(kFull, incl - own, src);
  const uint32_t top = kBins1 - 1u - 64u * src - 2u * lane;     // this lane: bins top, top - 1
  const uint2 x = __ldcg(reinterpret_cast<const uint2*>(h + top - 1u));
  const uint32_t in2 = above + warp_incl(x.x + x.y, lane);
  const uint32_t who = __ffs(__ballot_sync(kFull, in2 >= k)) - 1u;
  const uint32_t before = in2 - x.x - x.y;
  const bool high = before + x.y >= k;
  BinPick r;
  r.bin = __shfl_sync(kFull, high ? top : top - 1u, who);
  r.rem = __shfl_sync(kFull, high ? k - before : k - before - x.y, who);
  r.pop = __shfl_sync(kFull, high ? x.y : x.x, who);
  return r;
}

// Bound suggested for a later selection on layer s, by one warp: the one above which about `want` entries lie.
__device__ __forceinline__ uint32_t next_bound(const Workspace& ws, uint32_t s, const uint32_t* h, uint32_t L, uint32_t total,
                                               uint32_t want, uint32_t incl, uint32_t own, bool whole, int lane) {
  uint32_t key;
  if (total >= want) {
    const uint32_t roomy = want + want / 16;          // a little beyond, if there are that many
    key = max(L, bin_edge(warp_pick(h, incl, own, roomy <= total ? roomy : want, lane).bin, L));
  } else if (whole) {
    key = __ldcg(ws.L_wide + s);                      // known from the histogram of the whole input
  } else if (coarse_bins(L)) {
    key = 0;
  } else {
    // Fewer candidates than wished for (but at least k) and nothing known below the bound: lower it by as much as would
    // hold the missing ones at the density seen right above it -- what was never sent piles up below the k-th, so half
    // an octave down may hold a hundred times the wished-for number -- and by half an octave only where too few keys
    // lie above the bound to tell.
    uint32_t pop = 0, more = 0;
#pragma unroll
    for (int j = 0; j < 24; ++j) {       // an eighth of an octave: 640 bins; a quarter: 768
      const uint32_t v = __ldcg(h + j * 32 + lane);
      if (j < 20) pop += v;
      more += v;
    }
    pop = __reduce_add_sync(kFull, pop);
    uint32_t width = (1u << 20) - kBinLinear;
    if (pop < 64u) {
      pop = __reduce_add_sync(kFull, more);
      width = (1u << 21) - kBinLinear;
    }
    const float step = 1.5f * (float)(want + want / 16 - total) / (float)max(pop, 1u) * (float)width;
    const uint32_t down = pop >= 64u && step < (float)(4u << 20) ? (uint32_t)step + 1u : 4u << 20;
    key = L > down ? L - down : 0u;
  }
  // A bound of zero makes every element of the layer a candidate (zeros included).  That is fine for a
  // layer not much larger than the wished-for number of candidates, and for one that is small beside the
  // whole vector: a layer without enough candidates costs the next selection a histogram and a second pass
  // over all layers (148 layers of 124 M elements: 570 us a pull when every other one failed on layers of 768
  // to 3072 elements, 78 us without).  For a large one, no bound at all is the better advice: the next
  // selection finds nothing, notices, and takes its bound from a histogram.
  const uint32_t layer_cap = (ws.segs[s].tile_end - ws.segs[s].tile_begin) * (uint32_t)kWarpTile;
  const bool flood = key == 0 && layer_cap / 8 > want && layer_cap > max(8192u, ws.n / 1024u);
  return flood ? 0xFFFFFFFFu : key;
}

// The k-th largest of the `pop` keys of a list, all of them in [base, base + 2^bits), by one warp; hist: 128 words of
// shared memory of its own.  Returns T and, in r, how many of the keys equal to T are among the k.
static __device__ __noinline__ uint32_t warp_radix(const uint2* list, uint32_t pop, uint32_t k, uint32_t base, int bits, uint32_t* hist,
                                               int lane, uint32_t& r) {
  if (pop <= 32u) {                              // ranks by comparing with every other key
    const uint32_t key = (uint32_t)lane < pop ? __ldcg(&list[lane].x) : 0u;
    uint32_t above = 0, same = 0;
    for (uint32_t q = 0; q < pop; ++q) {
      const uint32_t o = __shfl_sync(kFull, key, q);
      above += o > key ? 1u : 0u;
      same += o == key ? 1u : 0u;
    }
    const uint32_t who = __ffs(__ballot_sync(kFull, (uint32_t)lane < pop && above < k && k <= above + same)) - 1u;
    r = __shfl_sync(kFull, k - above, who);
    return __shfl_sync(kFull, key, who);
  }
  constexpr int kKeep = 8;
  uint32_t prefix = 0, keep[kKeep];
  auto load = [&](uint32_t q0) {
#pragma unroll
    for (int u = 0; u < kKeep; ++u) {
      const uint32_t q = q0 + u * 32u + lane;
      keep[u] = q < pop ? __ldcg(&list[q].x) - base : kFull;
    }
  };
  if (pop <= 32u * kKeep) load(0);
#pragma unroll 1
  for (int shift = (bits - 1) / 7 * 7; shift >= 0; shift -= 7) {
    *reinterpret_cast<uint4*>(hist + lane * 4) = make_uint4(0, 0, 0, 0);
    __syncwarp();
    for (uint32_t q0 = 0; q0 < pop; q0 += 32u * kKeep) {
      if (pop > 32u * kKeep) load(q0);
#pragma unroll
      for (int u = 0; u < kKeep; ++u)
        if (q0 + u * 32u + lane < pop && (uint32_t)((uint64_t)keep[u] >> (shift + 7)) == prefix)
          atomicAdd(hist + ((keep[u] >> shift) & 127u), 1u);
    }
    __syncwarp();
    const uint4 x = *reinterpret_cast<const uint4*>(hist + 124 - lane * 4);   // lane's four bins, .w the highest
    const uint32_t sum = x.x + x.y + x.z + x.w, incl = warp_incl(sum, lane);
    const uint32_t who = __ffs(__ballot_sync(kFull, incl >= k)) - 1u;
    uint32_t left = k - (incl - sum), bin = 127u - lane * 4u;
    if (left > x.w) {
      left -= x.w; --bin;
      if (left > x.z) {
        left -= x.z; --bin;
        if (left > x.y) { left -= x.y; --bin; }
      }
    }
    prefix = (prefix << 7) | __shfl_sync(kFull, bin, who);
    k = __shfl_sync(kFull, left, who);
    __syncwarp();
  }
  r = k;
  return base + prefix;
}

// Where the CTAs of the next pass over a difference vector on this scratch set begin: ranges of blocks that cost
// about the same, judged by what this pass cost each CTA.  What has to be read and folded in clusters in the
// tensors with the largest updates, and those are the same for every worker; with equal ranges a few CTAs do most
// of the work.  Done by a CTA of its own beside the finalize, so that it adds nothing to the chain.
template <int MAXPARTS>
__device__ void plan_parts(const Workspace& ws, uint32_t G, FinalizeShared<MAXPARTS>& sh) {
  static_assert(MAXPARTS >= 512 + kMaxFoldGrid, "two tables in the place of the parts");
  uint32_t* const before = sh.pre;             // [G] cost of the CTAs before this one
  uint32_t* const first = sh.pre + 512;        // [G + 1] where they began
  uint32_t* const cost = sh.stream.hist;       // [G]
  uint32_t* const next = sh.stream.hist + kMaxFoldGrid;   // [G + 1]
  const bool had = ld_volatile(ws.sync + kPlanParts) == G && __ldcg(ws.plan + G) == ws.num_blocks;
  for (uint32_t p = threadIdx.x; p < G; p += kThreads) {
    cost[p] = __ldcg(ws.cta_cost + p);
    first[p] = had ? __ldcg(ws.plan + p) : part_first_tile(p, G, ws.num_blocks);
  }
  if (threadIdx.x == 0) first[G] = ws.num_blocks;
  __syncthreads();
  const uint32_t per = (G + kThreads - 1) / kThreads, p0 = min(G, threadIdx.x * per), p1 = min(G, p0 + per);
  uint32_t sum = 0;
  for (uint32_t p = p0; p < p1; ++p) sum += cost[p];
  unsigned long long total;
  block_excl_scan(sum, sh.warp_scan, total);
  // In 1/2^shift-ths, every block gets an amount on top that keeps a share of nothing but skipped blocks within
  // part_cap: with c the mean cost of a CTA it is 5/4 c / part_cap, which adds at most 5/32 to c (part_cap holds
  // eight even shares), so that a share ends after at most (37/32) / (5/4) part_cap blocks.
  const uint32_t shift = total < (1ull << 20) ? 10u : 0u;   // sums stay below 2^32: a block costs at most 255
  const float floor_cost = 1.25f * (float)((total << shift) / G + 1) / (float)(ws.part_cap - kFoldSlack);
  sum = 0;
  for (uint32_t p = p0; p < p1; ++p) {
    cost[p] = (cost[p] << shift) + (uint32_t)(floor_cost * (float)(first[p + 1] - first[p])) + 1u;
    sum += cost[p];
  }
  uint32_t at = (uint32_t)block_excl_scan(sum, sh.warp_scan, total);
  for (uint32_t p = p0; p < p1; ++p) {
    before[p] = at;
    at += cost[p];
  }
  __syncthreads();
  for (uint32_t j = threadIdx.x; j <= G; j += kThreads) {
    uint32_t g = j == 0 ? 0u : ws.num_blocks;
    if (j > 0 && j < G) {
      const unsigned long long target = total * j / G;
      uint32_t lo = 0, hi = G - 1;             // last CTA whose predecessors cost no more than the target
      while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (before[mid] <= target) lo = mid; else hi = mid - 1;
      }
      const unsigned long long into = target - before[lo], c = cost[lo];
      g = first[lo] + (uint32_t)((unsigned long long)(first[lo + 1] - first[lo]) * min(into, c) / c);
    }
    next[j] = g;
  }
  __syncthreads();
  int ok = 1;                                  // a CTA cannot take more blocks than its tables hold
  for (uint32_t j = threadIdx.x; j < G; j += kThreads)
    if (next[j + 1] < next[j] || next[j + 1] - next[j] + kFoldSlack > ws.part_cap) ok = 0;
  ok = __syncthreads_and(ok);
  for (uint32_t j = threadIdx.x; j < G; j += kThreads) ws.plan[j] = next[j];
  if (threadIdx.x == 0) {
    ws.plan[G] = ok ? ws.num_blocks : 0u;
    ws.sync[kPlanParts] = G;
  }
}

// The guess was too high for some layer: take the bound that cannot fail from a histogram of the whole input and repeat
// the stream pass, with the few CTAs this kernel has.  False: a barrier gave up.
template <int MODE>
__device__ __noinline__ bool redo_passes(const Workspace& ws, const SelArgs& a, const float* in, float* out, StreamShared& st,
                                         unsigned long long* s_warp, uint32_t* s_res, int* s_ok, uint32_t Wb, uint32_t spin_limit,
                                         uint32_t& bar_target) {
  const uint32_t cta = blockIdx.x, G = a.workers + a.advisers, S = ws.num_segs;
  auto barrier = [&]() { return worker_barrier(ws.sync + kBarCount + a.pair, Wb, ws.status, s_ok, bar_target, spin_limit); };
  for (size_t w = (size_t)cta * kThreads + threadIdx.x; w < (size_t)S * kBins1; w += (size_t)G * kThreads) ws.hist1[w] = 0;
  for (uint32_t s = cta * kThreads + threadIdx.x; s < S; s += G * kThreads) ws.list_cnt[s] = 0;
  if (cta == 0 && threadIdx.x == 0) ws.sync[kFail + a.pair] = 0;
  if (!barrier()) return false;
  hist_all_tiles<MODE>(ws, a, in, cta, G, st.hist);
  if (!barrier()) return false;
  for (uint32_t s = cta; s < S; s += G) {
    pick_lower(ws, s, ws.segs[s].k[MODE == kPull ? 1 : 0], s_warp, s_res);
    __syncthreads();
  }
  if (!barrier()) return false;
  stream_tiles<MODE>(ws, a, ws.L_safe, in, out, cta, G, st);
  return barrier();
}

// The k-th largest of the `pop` keys of a list, all of them in [base, base + 2^bits), by the whole CTA; hist: 256 words.
static __device__ __noinline__ uint32_t block_radix(const uint2* list, uint32_t pop, uint32_t k, uint32_t base, int bits, uint32_t* hist,
                                             uint32_t* s_res, uint32_t& r) {
  const int lane = threadIdx.x & 31;
  uint32_t prefix = 0;
#pragma unroll 1
  for (int shift = (bits - 1) / 8 * 8; shift >= 0; shift -= 8) {
    hist[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll 4
    for (uint32_t q = threadIdx.x; q < pop; q += kThreads) {
      const uint32_t key = __ldcg(&list[q].x) - base;
      if ((uint32_t)((uint64_t)key >> (shift + 8)) == prefix) atomicAdd(hist + ((key >> shift) & 255u), 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) {              // lane's eight bins, the highest first
      uint32_t sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += hist[255 - lane * 8 - j];
      uint32_t before = warp_incl(sum, lane) - sum;
      for (int j = 0; j < 8; ++j) {
        const uint32_t c = hist[255 - lane * 8 - j];
        if (before < k && k <= before + c) {
          s_res[0] = 255u - lane * 8u - j;
          s_res[1] = k - before;
        }
        before += c;
      }
    }
    __syncthreads();
    prefix = (prefix << 8) | s_res[0];
    k = s_res[1];
  }
  r = k;
  return base + prefix;
}

// 64 registers a thread: beside other kernels whatever the small ones hold is taken from the passes.  Runs without a join,
// us an event with 64 / 72 / 80 / 96 / 128: 62 layers of 11.7 M elements, 32 workers: 94 / 94 / 98 / 107 / 114; one layer of
// 25.6 M: 59.9 / 59.5 / 60.0 / 60.4 / 62.6.  Alone, 96 are 1 to 3 % faster.  (Shared memory is not what binds here: with
// eight warps a CTA in the pull's pass, 13.3 KB for a pull instead of 20.5 KB, with the parts numbered in groups of four, changed
// none of these by more than 0.5 %; with the parts of ten it is 23.5 KB.)
// BIG: for more candidates than the registers hold, where the kernel has the GPU to itself.  Such candidates are read again
// in every phase, and a phase is a chain of trips to memory: four of them a lane are on their way instead of two, and a run
// of candidates in one part needs neither a search nor a trip for its place.  Finalize of a pull, us, before / with BIG:
// 2^24 elements, 10 %: 128 / 95, 50 %: 878 / 497; 2^27, 10 %: 1447 / 815.  Beside other kernels its registers cost more
// than it gains (62 layers of 8.4 M elements, 1 %, runs of 32 events: 65 us an event without, 79 with).
// PASSED: in one kernel with the pass before it, all of whose CTAs come here; `bar_target`: their number.  in, out: the state
// vector that the pass has read, and for a push the one that it has written.
template <int MODE, bool MANY, bool BIG, int MAXPARTS, bool PASSED>
__device__ __forceinline__ void finalize(const Workspace& ws, const SelArgs& a, const float* in, float* out,
                                         FinalizeShared<MAXPARTS>& sh, unsigned char* fin_dyn, uint32_t bar_target) {
  constexpr int PM = MODE == kPull ? 1 : 0, kKeep = BIG ? 4 : finalize_keep(MANY);
  // CTAs [0, W) process the candidates, [W, W + A) look after the layers' bounds, and after k_fold one more plans the
  // next pass (it takes no part in the selection)
  const uint32_t cta = blockIdx.x, W = a.workers, A = a.advisers, S = ws.num_segs;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t gthread = cta * kThreads + threadIdx.x, nthreads = (W + A) * kThreads, lt = lanemask_lt(), le = lt | (1u << lane);
  // the barrier counts W + A arrivals; a test can make it wait for CTAs that do not exist, with a short limit,
  // to see the bounded wait give up (every CTA then leaves with DGS_ETIMEOUT in the status word)
  const uint32_t Wb = W + A + a.phantom_workers, spin_limit = a.spin_limit ? a.spin_limit : kSpinLimit;
  if (PASSED) {
    if (cta >= W + A + (MODE == kPull ? 1u : 0u)) {      // nothing to do here: the others only wait for its pass
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(ws.sync + kBarCount + a.pair, 1u);
      }
      return;
    }
    const uint32_t all = bar_target + (MODE == kPull ? a.phantom_workers : 0u);   // (a push: a CTA of its pass does not come)
    bar_target = 0;
    if (!worker_barrier(ws.sync + kBarCount + a.pair, all, ws.status, &sh.ok, bar_target, spin_limit)) return;
  }
  if constexpr (MODE == kPull) {
    if (cta == W + A) {
      plan_parts(ws, a.fold_grid, sh);
      return;
    }
  }
  auto barrier = [&]() { return worker_barrier(ws.sync + kBarCount + a.pair, Wb, ws.status, &sh.ok, bar_target, spin_limit); };

  const uint32_t* seg_off = ws.seg_off;
  if (MANY && S <= (uint32_t)kSegCap) {
    uint32_t* const sm = reinterpret_cast<uint32_t*>(fin_dyn);
    for (uint32_t s = threadIdx.x; s <= S; s += kThreads) sm[s] = ws.seg_off[s];
    seg_off = sm;
  }

  uint32_t parts = 0, clo = 0, chi = 0, wlo = 0, whi = 0;   // flat candidates of this CTA, of this warp
  uint32_t part0 = 0, part1 = 0;         // parts that this warp's candidates lie in
  bool kept = false;                     // this warp's candidates stay in registers
  float raw[kKeep];
  uint32_t idx[kKeep];
  auto slot_of = [&](uint32_t p, uint32_t lo, uint32_t hi) {
    const uint32_t part = part_of(sh.pre, lo, hi, p);
    return __ldcg(ws.part_slot0 + part) + (p - sh.pre[part]);
  };
  uint32_t run_part = 0, run_slot = 0;   // BIG: part of the last load's first candidate, its first slot - pre
  auto load = [&](uint32_t base) {       // candidates base + 32 u + lane of this warp's run (beyond its end: the last one)
    uint32_t slot[kKeep];
    bool one_part = false;
    if (BIG) {
      if (base == wlo || sh.pre[run_part + 1] <= base) {
        run_part = base == wlo ? part0 : part_of(sh.pre, run_part + 1, part1, base);
        run_slot = __ldcg(ws.part_slot0 + run_part) - sh.pre[run_part];
      }
      one_part = sh.pre[run_part + 1] >= min(base + 32u * kKeep, whi);   // no search, and no trip for the slots
    }
#pragma unroll
    for (int u = 0; u < kKeep; ++u)
      if (base + u * 32u < whi) {
        const uint32_t p = min(base + u * 32u + lane, whi - 1u);
        slot[u] = one_part ? run_slot + p : slot_of(p, part0, part1);
      }
#pragma unroll
    for (int u = 0; u < kKeep; ++u)
      if (base + u * 32u < whi) {
        raw[u] = __ldcg(ws.cand_val + slot[u]);
        idx[u] = __ldcg(ws.cand_idx + slot[u]);
      }
  };

  uint32_t s_lo = 0, s_last = 0;         // layers of this CTA's first and last candidate
  bool goes_on = false;                  // layer s_lo began before this CTA's first candidate
  LayerPick* tab = sh.tab;               // [s - s_lo]
  uint32_t near_t = 0, near_b = 1, near_e = 0;   // layer (counted from s_lo) that this lane looked at last
  auto row_of = [&](uint32_t i) -> LayerPick* {
    if (MANY && (i < near_b || i >= near_e)) {
      const uint32_t s = seg_of(seg_off, s_lo, s_last, i);
      near_t = s - s_lo;
      near_b = seg_off[s];
      near_e = seg_off[s + 1];
    }
    return tab + near_t;
  };
  // Visits this warp's candidates in flat order and counts them: classify(u, row, valid, equal) says whether a candidate
  // counts as above, and may set `equal`.  Notes where in the count the layers begin; batch(first flat number) is called
  // after each batch of candidates.  Then the counts of the CTA's last layer are published.
  auto count = [&](auto classify, auto batch) {
    uint32_t gt = 0, eq = 0, prev_t = kFull;     // the same in every lane; layer of the candidate before
    if (MANY && wlo < whi) {
      if (wlo > clo) {
        row_of(__ldcg(ws.cand_idx + slot_of(wlo - 1u, 0, parts - 1u)));
        prev_t = near_t;
      } else if (goes_on) {
        prev_t = 0;
      }
    }
#pragma unroll 1
    for (uint32_t base = wlo; base < whi; base += 32u * kKeep) {
      if (!kept) load(base);
#pragma unroll
      for (int u = 0; u < kKeep; ++u)
        if (base + u * 32u < whi) {
          const bool valid = base + u * 32u + lane < whi;
          LayerPick* const t = row_of(idx[u]);
          bool equal = false;
          const bool above = classify(u, t, valid, equal);
          const uint32_t mg = __ballot_sync(kFull, above), me = __ballot_sync(kFull, equal);
          if (MANY) {
            uint32_t before = __shfl_up_sync(kFull, near_t, 1);
            if (lane == 0) before = prev_t;
            if (valid && before != near_t) {
              t->start_gt = gt + __popc(mg & lt);
              t->start_eq = eq + __popc(me & lt);
              t->start_warp = warp;
            }
            prev_t = __shfl_sync(kFull, near_t, 31);
          }
          gt += __popc(mg);
          eq += __popc(me);
        }
      batch(base);
    }
    if (lane == 0) {
      sh.gt[warp] = gt;
      sh.eq[warp] = eq;
    }
    __syncthreads();
    if (threadIdx.x == 0 && cta < W) {
      uint32_t g = 0, e = 0;
      for (int w = 0; w < kWarps; ++w) {
        g += sh.gt[w];
        e += sh.eq[w];
      }
      if (clo < chi && !(goes_on && s_lo == s_last) && MANY) {
        const LayerPick& t = tab[s_last - s_lo];
        for (uint32_t w = 0; w < t.start_warp; ++w) {
          g -= sh.gt[w];
          e -= sh.eq[w];
        }
        g -= t.start_gt;
        e -= t.start_eq;
      }
      ws.cta_tot[cta] = make_uint2(clo < chi ? s_last : kFull, g);
      ws.cta_eq[cta] = e;
    }
  };

  bool redo = false;
  uint32_t flags = 0;
#pragma unroll 1
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (redo) {
      if (!redo_passes<MODE>(ws, a, in, out, sh.stream, sh.warp_scan, sh.res, &sh.ok, Wb, spin_limit, bar_target)) return;
    }
    const uint32_t* const L_used = redo ? ws.L_safe : a.L_in;
    if (cta >= W) {
      // checks the guesses (a layer needs at least k candidates) and suggests the next bounds
      uint32_t seen = 0;
      for (uint32_t s = (cta - W) * kWarps + warp; s < S; s += A * kWarps) {
        const uint32_t* const h = ws.hist1 + (size_t)s * kBins1;
        const uint32_t k = ws.segs[s].k[PM], L = __ldcg(L_used + s);
        const uint32_t sum = lane_bins(h, lane), incl = warp_incl(sum, lane), total = __shfl_sync(kFull, incl, 31);
        uint32_t flag = 1u;
        // A layer whose guesses fail gets more room: half of k on a failure, an eighth back every 32 selections.
        // (8 workers, 148 layers of 124 M elements: 5 % of the pulls started over, at 1.2 ms each, for layers that had
        // found 85 to 98 % of k.)
        uint32_t slack = a.speculate ? __ldcg(a.slack + s) : 0u;
        if (total >= k) {
          flag = warp_pick(h, incl, sum, k, lane).pop > ws.segs[s].list_cap ? 2u : 0u;
          if (a.speculate) {
            const uint32_t want = (uint32_t)min((uint64_t)spec_want(k) + (uint64_t)k * slack / 8u, (uint64_t)0xFFFFFFFFu);
            const uint32_t key = next_bound(ws, s, h, L, total, want, incl, sum, redo || a.force_two_pass, lane);
            if (lane == 0) {
              a.L_next[s] = key;
              if (slack && (a.seq & 31u) == 0) a.slack[s] = slack - 1u;
            }
          }
        } else if (a.speculate && lane == 0) {
          a.slack[s] = min(slack + 4u, 16u);       // (selections in flight beside this one may write it too: it is advice)
        }
        if (flag && lane == 0) atomicOr(ws.sync + kFail + a.pair, flag);
        seen += total;
      }
      if (lane == 0 && seen) atomicAdd(ws.stats + 2, (unsigned long long)seen);
      clo = chi = wlo = whi = 0;
    } else {
      // flat numbering of the candidates (the stream pass is complete: an earlier kernel, or the barrier above)
      parts = ld_volatile(ws.sync + kParts);
      number_parts<MAXPARTS>(ws, parts, sh.pre, sh.warp_scan);
      const uint32_t C = sh.pre[parts];
      const uint32_t per_warp = (uint32_t)(((uint64_t)C + W * kWarps * 32u - 1u) / (W * kWarps * 32u)) * 32u;
      clo = (uint32_t)min((uint64_t)C, (uint64_t)cta * kWarps * per_warp);
      chi = (uint32_t)min((uint64_t)C, (uint64_t)(cta + 1) * kWarps * per_warp);
      wlo = (uint32_t)min((uint64_t)chi, (uint64_t)clo + warp * per_warp);
      whi = (uint32_t)min((uint64_t)chi, (uint64_t)wlo + per_warp);
      kept = !BIG && per_warp <= 32u * kKeep;
      if (wlo < whi) {
        part0 = warp_part_of(sh.pre, parts, wlo, lane);
        part1 = warp_part_of(sh.pre, parts, whi - 1u, lane);
        if (kept) load(wlo);
      }
      s_lo = s_last = 0;
      near_t = 0;
      near_b = 1;
      near_e = 0;
      goes_on = clo > 0;
      if (MANY) {
        if (threadIdx.x < 3 && clo < chi) {
          const uint32_t p = threadIdx.x == 0 ? (clo > 0 ? clo - 1u : clo) : threadIdx.x == 1 ? clo : chi - 1u;
          sh.range[threadIdx.x] = seg_of(seg_off, 0, S - 1u, __ldcg(ws.cand_idx + slot_of(p, 0, parts - 1u)));
        }
        __syncthreads();
        if (clo < chi) {
          s_lo = sh.range[1];
          s_last = sh.range[2];
          goes_on = clo > 0 && sh.range[0] == s_lo;
        }
      }
    }
    const uint32_t touched = clo < chi ? s_last - s_lo + 1u : 0u;
    tab = touched <= (uint32_t)kTouch ? sh.tab : ws.tab + s_lo + cta;   // (two CTAs share at most a layer: their rows differ)
    if (!MANY ? touched != 0 : touched == 1) {
      uint32_t bin, krem;
      const uint32_t k = ws.segs[s_lo].k[PM];
      const uint32_t total = block_pick<kBins1>(ws.hist1 + (size_t)s_lo * kBins1, k, bin, krem, sh.warp_scan, sh.res);
      if (threadIdx.x == 0) {
        LayerPick& t = tab[0];
        const uint32_t pop = sh.res[2];
        t.L = __ldcg(L_used + s_lo);
        t.bin = total < k ? kFull : bin;
        t.krem = krem;
        t.pop = pop > ws.segs[s_lo].list_cap ? 0u : pop;
        t.pkt_off = ws.segs[s_lo].pkt_off[PM];
        t.list_off = ws.segs[s_lo].list_off;
      }
    } else if (MANY) {
#pragma unroll 1
      for (uint32_t t0 = warp; t0 < touched; t0 += kWarps) {
        const uint32_t s = s_lo + t0, k = ws.segs[s].k[PM], L = __ldcg(L_used + s);
        const uint32_t list_cap = ws.segs[s].list_cap, list_off = ws.segs[s].list_off, pkt_off = ws.segs[s].pkt_off[PM];
        const uint32_t* const h = ws.hist1 + (size_t)s * kBins1;
        const uint32_t sum = lane_bins(h, lane), incl = warp_incl(sum, lane);
        BinPick b = {kFull, 0, 0};
        if (__shfl_sync(kFull, incl, 31) >= k) b = warp_pick(h, incl, sum, k, lane);
        if (lane == 0) {
          LayerPick& t = tab[t0];
          t.L = L;
          t.bin = b.bin;
          t.krem = b.rem;
          t.pop = b.pop > list_cap ? 0u : b.pop;
          t.pkt_off = pkt_off;
          t.list_off = list_off;
        }
      }
    }
    __syncthreads();
    // Candidates above the k-th's bin are counted, those in it go to the layer's list.  (There are `pop` of them, the list's
    // place holds that many.  Only where an earlier barrier gave up, and left its counts behind, does the list begin later:
    // the bound keeps it in its place.)
    uint32_t hits = 0;
    count([&](int u, const LayerPick* t, bool valid, bool&) {
      const uint32_t b = bin_of(key_of(raw[u]), t->L), bin = t->bin;
      if (valid && b == bin && t->pop) hits |= 1u << u;
      return valid && bin != kFull && b > bin;
    }, [&](uint32_t base) {
      if (!MANY) {                       // one layer: a place for all hits of the warp at once
        uint32_t n = 0, at = 0;
#pragma unroll
        for (int u = 0; u < kKeep; ++u) n += __popc(__ballot_sync(kFull, (hits >> u) & 1u));
        if (n) {
          if (lane == 0) at = atomicAdd(ws.list_cnt, n);
          at = __shfl_sync(kFull, at, 0);
          uint2* const list = ws.list + sh.tab[0].list_off;
#pragma unroll
          for (int u = 0; u < kKeep; ++u) {
            const uint32_t m = __ballot_sync(kFull, (hits >> u) & 1u), to = at + __popc(m & lt);
            if (((hits >> u) & 1u) && to < sh.tab[0].pop) list[to] = make_uint2(key_of(raw[u]), base + u * 32u + lane);
            at += __popc(m);
          }
          hits = 0;
        }
      }
      if (MANY) {
        uint32_t todo;
        while ((todo = __ballot_sync(kFull, hits != 0)) != 0) {   // rarely more than one layer
          uint32_t i = idx[0];
#pragma unroll
          for (int u = 1; u < kKeep; ++u)
            if (hits && u == __ffs(hits) - 1) i = idx[u];
          const LayerPick* const t = row_of(__shfl_sync(kFull, i, __ffs(todo) - 1));   // the layer of the first hit: for all lanes
          uint32_t n = 0, at = 0, mine = 0;
#pragma unroll
          for (int u = 0; u < kKeep; ++u) {
            const bool in = ((hits >> u) & 1u) && idx[u] >= near_b && idx[u] < near_e;
            mine |= in ? 1u << u : 0u;
            n += __popc(__ballot_sync(kFull, in));
          }
          if (lane == 0) at = atomicAdd(ws.list_cnt + s_lo + near_t, n);
          at = __shfl_sync(kFull, at, 0);
          uint2* const list = ws.list + t->list_off;
#pragma unroll
          for (int u = 0; u < kKeep; ++u) {
            const uint32_t m = __ballot_sync(kFull, (mine >> u) & 1u), to = at + __popc(m & lt);
            if (((mine >> u) & 1u) && to < t->pop) list[to] = make_uint2(key_of(raw[u]), base + u * 32u + lane);
            at += __popc(m);
          }
          hits &= ~mine;
        }
      }
      __syncwarp();
    });
    if (!barrier()) return;
    flags = ld_volatile(ws.sync + kFail + a.pair);
    if (!(flags & 1u) || redo) break;
    if (!barrier()) return;              // everyone has seen the flags
    redo = true;
  }
  const uint32_t touched = clo < chi ? s_last - s_lo + 1u : 0u;
  // what the next selection expects to find cleared
  {
    uint4* const h4 = reinterpret_cast<uint4*>(ws.hist1);
    for (size_t w = gthread; w < (size_t)S * (kBins1 / 4); w += nthreads) h4[w] = make_uint4(0, 0, 0, 0);
  }
  if (cta >= W) {
    for (uint32_t s = (cta - W) * kThreads + threadIdx.x; s < S; s += A * kThreads) ws.list_cnt[s] = 0;
  }
  uint2* const s_list = reinterpret_cast<uint2*>(sh.stream.hist);   // the list, where it is ranked in shared memory
  const bool ranked = !MANY && touched && !(flags & 2u) && tab[0].pop <= (uint32_t)kListSmem;
  if (ranked) {
    // a thread per entry compares it with every other one
    const uint32_t pop = tab[0].pop, k = tab[0].krem;
    uint2 mine = make_uint2(0, 0);
    if (threadIdx.x < pop) {
      mine = __ldcg(ws.list + tab[0].list_off + threadIdx.x);
      s_list[threadIdx.x] = mine;
    }
    __syncthreads();
    if (threadIdx.x < pop) {
      uint32_t above = 0, same = 0;
#pragma unroll 4
      for (uint32_t q = 0; q < pop; ++q) {
        const uint32_t o = s_list[q].x;
        above += o > mine.x ? 1u : 0u;
        same += o == mine.x ? 1u : 0u;
      }
      if (above < k && k <= above + same) {   // (the same for all that are equal)
        tab[0].T = mine.x;
        tab[0].r = k - above;
      }
    }
    __syncthreads();
  } else if (!(flags & 2u)) {
    auto exact = [&](uint32_t t, auto radix) {
      const uint32_t L = tab[t].L, bin = tab[t].bin;
      const bool open = bin == (uint32_t)kBins1 - 1u;    // (the last bin is open-ended)
      return radix(ws.list + tab[t].list_off, tab[t].pop, tab[t].krem, open ? 0u : bin_edge(bin, L), open ? 31 : bin_bits(bin, L));
    };
    uint32_t r;
    if (MANY) {
#pragma unroll 1
      for (uint32_t t = warp; t < touched; t += kWarps) {
        const uint32_t T = exact(t, [&](const uint2* list, uint32_t pop, uint32_t k, uint32_t base, int bits) {
          return warp_radix(list, pop, k, base, bits, sh.stream.hist + warp * 128, lane, r);
        });
        if (lane == 0) {
          tab[t].T = T;
          tab[t].r = r;
        }
      }
    } else if (touched) {
      const uint32_t T = exact(0, [&](const uint2* list, uint32_t pop, uint32_t k, uint32_t base, int bits) {
        return block_radix(list, pop, k, base, bits, sh.stream.hist, sh.res, r);
      });
      if (threadIdx.x == 0) {
        tab[0].T = T;
        tab[0].r = r;
      }
    }
    __syncthreads();
  } else {
    // Some bin holds more candidates than its list (many equal values, or a bound far below the k-th): three radix
    // levels (11 + 10 + 10 key bits) over all candidates, counted in global memory, the picks spread over the CTAs.
    // A CTA counts the layer of its middle candidate in shared memory, others straight in global memory.  (All of them in
    // global memory, where the keys crowd into a few dozen bins: 2^24 elements, 20 %: 1326 us instead of 323.)
    uint32_t* const s_hist = sh.stream.hist;
    uint32_t main_t = 0;
    if (MANY && clo < chi) {
      row_of(__ldcg(ws.cand_idx + slot_of(clo + (chi - clo) / 2u, 0, parts - 1u)));
      main_t = near_t;
    }
    for (uint32_t b = threadIdx.x; b < (uint32_t)kBins1; b += kThreads) s_hist[b] = 0;
    if (!barrier()) return;              // the histograms are clear
#pragma unroll 1
    for (int level = 1; level <= 3; ++level) {
      const int sft = level == 1 ? 20 : level == 2 ? 10 : 0;
#pragma unroll 1
      for (uint32_t base = wlo; base < whi; base += 32u * kKeep) {
        if (!kept) load(base);
#pragma unroll
        for (int u = 0; u < kKeep; ++u)
          if (base + u * 32u < whi) {
            const uint32_t key = key_of(raw[u]);
            row_of(idx[u]);
            const uint32_t s = s_lo + near_t;
            const bool mine = base + u * 32u + lane < whi && (level == 1 || (key >> (sft + 10)) == __ldcg(&ws.sel[s].prefix));
            const uint32_t bin = level == 1 ? key >> 20 : (key >> sft) & 1023u, at = s * (uint32_t)kBins1 + bin;
            auto add = [&](uint32_t n) {
              if (!MANY || near_t == main_t) atomicAdd(s_hist + bin, n); else atomicAdd(ws.hist1 + at, n);
            };
            // lanes with the first one's bin are counted together: ties crowd into few bins
            const uint32_t m = __ballot_sync(kFull, mine);
            if (m) {
              const uint32_t lead = __shfl_sync(kFull, at, __ffs(m) - 1), same = __ballot_sync(kFull, mine && at == lead);
              if (lane == __ffs(m) - 1) add(__popc(same));
              if (mine && at != lead) add(1u);
            }
          }
      }
      __syncthreads();
      if (clo < chi)
        for (uint32_t b = threadIdx.x; b < (uint32_t)kBins1; b += kThreads)
          if (s_hist[b]) {
            atomicAdd(ws.hist1 + (size_t)(s_lo + main_t) * kBins1 + b, s_hist[b]);
            s_hist[b] = 0;
          }
      if (!barrier()) return;
      for (uint32_t s = cta; s < S; s += W + A) {
        uint32_t bin, krem;
        uint32_t* const h = ws.hist1 + (size_t)s * kBins1;
        const uint32_t k = level == 1 ? ws.segs[s].k[PM] : __ldcg(&ws.sel[s].krem);
        const uint32_t old = level == 1 ? 0u : __ldcg(&ws.sel[s].prefix);
        block_pick<kBins1>(h, k, bin, krem, sh.warp_scan, sh.res);
        if (threadIdx.x == 0) {
          ws.sel[s].prefix = level == 1 ? bin : (old << 10) | bin;
          ws.sel[s].krem = krem;
        }
        __syncthreads();
        for (int b = threadIdx.x; b < kBins1; b += kThreads) h[b] = 0;
      }
      if (!barrier()) return;
    }
    for (uint32_t t = threadIdx.x; t < touched; t += kThreads) {
      tab[t].T = __ldcg(&ws.sel[s_lo + t].prefix);
      tab[t].r = __ldcg(&ws.sel[s_lo + t].krem);
    }
    __syncthreads();
    count([&](int u, const LayerPick* t, bool valid, bool& equal) {
      const uint32_t key = key_of(raw[u]), T = t->T;
      equal = valid && key == T;
      return valid && key > T;
    }, [](uint32_t) {});
    if (!barrier()) return;
  }

  // ---- emit: packet in index order, and the state updates that depend on selection ----
  if (wlo < whi) {
    // selected entries of the first candidate's layer that stand before it
    uint32_t run_gt = 0, run_eq = 0;
    if (!kept) load(wlo);
    const LayerPick* const t0 = row_of(__shfl_sync(kFull, idx[0], 0));
    uint32_t carry_t = near_t;
    const bool before = goes_on && carry_t == 0;         // it began before this CTA
    if (!(flags & 2u)) {
      const uint32_t T = t0->T, pop = t0->pop;
      const uint2* const list = ws.list + t0->list_off;
#pragma unroll 1
      for (uint32_t q = lane; q < pop; q += 32) {
        const uint2 e = ranked ? s_list[q] : __ldcg(list + q);
        if (e.y < wlo) {
          run_gt += e.x > T ? 1u : 0u;
          run_eq += e.x == T ? 1u : 0u;
        }
      }
    }
    if (before)
#pragma unroll 4
      for (uint32_t c = lane; c < cta; c += 32) {
        const uint2 q = __ldcg(ws.cta_tot + c);
        const uint32_t e = __ldcg(ws.cta_eq + c);
        if (q.x == s_lo) {
          run_gt += q.y;
          run_eq += e;
        }
      }
    if (lane < kWarps && lane < warp) {
      run_gt += sh.gt[lane];
      run_eq += sh.eq[lane];
    }
    if (MANY && !before && lane <= (int)t0->start_warp) {   // the layer began in this CTA: without what was counted before it
      if (lane < (int)t0->start_warp) {
        run_gt -= sh.gt[lane];
        run_eq -= sh.eq[lane];
      } else {
        run_gt -= t0->start_gt;
        run_eq -= t0->start_eq;
      }
    }
    run_gt = __reduce_add_sync(kFull, run_gt);
    run_eq = __reduce_add_sync(kFull, run_eq);
#pragma unroll 1
    for (uint32_t base = wlo; base < whi; base += 32u * kKeep) {
      if (!kept && base != wlo) load(base);
      uint32_t pos[kKeep];               // place in the packet, kFull: not selected
#pragma unroll
      for (int u = 0; u < kKeep; ++u) {
        pos[u] = kFull;
        if (base + u * 32u < whi) {
          const bool valid = base + u * 32u + lane < whi;
          const LayerPick* const t = row_of(idx[u]);
          const uint32_t key = key_of(raw[u]), T = t->T;
          const bool above = valid && key > T, equal = valid && key == T;
          const uint32_t mg = __ballot_sync(kFull, above), me = __ballot_sync(kFull, equal);
          uint32_t in_layer = kFull, heads = 0;              // lanes of this lane's layer, counted from its first one
          if (MANY) {
            uint32_t prev = __shfl_up_sync(kFull, near_t, 1);
            if (lane == 0) prev = carry_t;
            heads = __ballot_sync(kFull, prev != near_t);
            carry_t = __shfl_sync(kFull, near_t, 31);
            if (heads & le) in_layer = kFull << (31 - __clz(heads & le));
          }
          const bool first = (heads & le) != 0;              // the layer begins among these 32
          const uint32_t gt_rank = (first ? 0u : run_gt) + __popc(mg & lt & in_layer);
          const uint32_t eq_rank = (first ? 0u : run_eq) + __popc(me & lt & in_layer);
          const uint32_t r = t->r;
          if (above || (equal && eq_rank < r)) pos[u] = t->pkt_off + gt_rank + min(eq_rank, r);
          const uint32_t tail = heads ? kFull << (31 - __clz(heads)) : kFull;
          run_gt = (heads ? 0u : run_gt) + __popc(mg & tail);
          run_eq = (heads ? 0u : run_eq) + __popc(me & tail);
        }
      }
      float local[kKeep];
      if (MODE == kPull && a.theta_local != nullptr) {
#pragma unroll
        for (int u = 0; u < kKeep; ++u) local[u] = pos[u] != kFull ? __ldcg(a.theta_local + idx[u]) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kKeep; ++u) {
        if (pos[u] != kFull) {
          const float q = round16(raw[u], a.packet_format);  // what the packet carries (the value itself with float32 packets)
          if (pos[u] < a.pkt_count) {
            a.pkt_idx[pos[u]] = idx[u];
            a.pkt_val[pos[u]] = q;
          } else {
            atomicMin(ws.status, -1000 - MODE);
          }
          // Algorithm 1: the sent part leaves v (what a rounded packet did not carry stays: val - q, else zero).
          // Algorithm 3 keeps the sent entry's velocity t (already stored): no residual exists to take val - q.
          if (MODE == kPushResidual) out[idx[u]] = __fsub_rn(raw[u], q);
          if (MODE == kPull) {
            a.D[idx[u]] = __fsub_rn(raw[u], q);              // Eq. 6b: v_k <- v_k + G; the rounding remainder stays
            if (a.theta_local) a.theta_local[idx[u]] = __fadd_rn(local[u], q);  // Eq. 5
          }
        } else if (MODE == kPushSam && base + u * 32u + lane < whi) {
          out[idx[u]] = __fmul_rn(raw[u], a.inv_m);          // Eq. 12, lower branch
        }
      }
    }
  }
  if (cta == W && threadIdx.x == 0) {
    if (MODE != kPull) {  // the spare buffer now holds the worker's velocity
      float* cur = *a.u_cur_slot;
      *a.u_cur_slot = *a.u_spare_slot;
      *a.u_spare_slot = cur;
    }
    atomicAdd(ws.stats + ((redo || a.force_two_pass) ? 1 : 0), 1ull);
  }
}

template <int MODE, bool MANY, bool BIG>
__global__ void __maxnreg__(BIG ? 96 : 64) k_finalize(const __grid_constant__ Workspace ws, const __grid_constant__ SelArgs a) {
  constexpr int kPartCap = MODE == kPull ? kMaxParts : kMaxGrid;   // parts that the pass before, or a redo, can leave
  __shared__ FinalizeShared<kPartCap> sh;
  extern __shared__ __align__(16) unsigned char fin_dyn[];   // finalize_dyn_bytes(S) bytes
  // pointers are read once, before anything may exchange them
  const float* const in = MODE == kPull ? a.D : *a.u_cur_slot;
  float* const out = MODE == kPull ? nullptr : *a.u_spare_slot;
  finalize<MODE, MANY, BIG, kPartCap, false>(ws, a, in, out, sh, fin_dyn, 0u);
}

// ---- the two passes as kernels of their own, for a selection with nothing to go by -------
template <int MODE>
__global__ void __launch_bounds__(kThreads, 4) k_hist_all(Workspace ws, SelArgs a) {
  __shared__ uint32_t s_hist[kBins1];
  const float* in = MODE == kPull ? a.D : *a.u_cur_slot;
  hist_all_tiles<MODE>(ws, a, in, blockIdx.x, gridDim.x, s_hist);
}

// one CTA per layer (strided)
template <int MODE>
__global__ void __launch_bounds__(kThreads) k_pick_lower(Workspace ws) {
  __shared__ unsigned long long s_warp[kWarps];
  __shared__ uint32_t s_res[3];
  for (uint32_t s = blockIdx.x; s < ws.num_segs; s += gridDim.x) {
    pick_lower(ws, s, ws.segs[s].k[MODE == kPull ? 1 : 0], s_warp, s_res);
    __syncthreads();
  }
}

using PushRing = StreamRing<3>;
// ---- stand-alone stream pass with the carried bound -------------------------------
template <int MODE>
__global__ void __maxnreg__(64) k_stream(const __grid_constant__ Workspace ws, const __grid_constant__ SelArgs a) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];   // the ring of stages
  __shared__ StreamShared sh;
  __shared__ __align__(8) uint64_t full[PushRing::kStages];
  __shared__ int s_dead;
  const float* in = *a.u_cur_slot;
  float* out = *a.u_spare_slot;
  if (blockIdx.x == 0 && threadIdx.x < 2) ws.sync[kBarCount + threadIdx.x] = ws.sync[kFail + threadIdx.x] = 0;   // for the finalize that follows
  stream_blocks_tma<MODE, PushRing>(ws, a, a.L_in, in, out, blockIdx.x, gridDim.x, sh, reinterpret_cast<float*>(dyn_smem), full,
                                    &s_dead, 0u, kSpinLimit);
}

// ---- server apply ---------------------------------------------------------------
// Algorithm 2 lowers theta and every D_q by the decoded packet.  D_q is read only by worker
// q's pull, so the library keeps D_q lazily: an apply lowers theta at once and files the
// packet in a ring of recent packets; a pull of worker q first folds into D_q, in arrival
// order, the packets filed since D_q was last brought up to date.  Every D_q[i] sees the
// same subtractions in the same order as with an eager update, so the result is the same
// bit for bit, and each packet is folded into D_q while the entries it touches are hot
// instead of being scattered into all N vectors at once.
struct PacketLog {
  uint2* ent;         // [ring][stride]: (index, bits of the value), each packet sorted by index
  uint32_t stride;    // entries between slots
  uint32_t ring;      // slots
  // pos[b][slot]: position of the first entry of the packet in `slot` whose index is >= b * kWarpTile, for every
  // block b of the vector and a little beyond (those hold the packet's size).  Block-major: a worker that catches up
  // reads a block's positions in all packets as one or two lines, where packet-major rows cost it a line per packet
  // (and, with a row per page, an address translation per packet).
  uint32_t* pos;      // [pos_rows][ring]
  uint32_t pos_rows;  // number of blocks + 1
  // sum[r][b]: entries in block b of all packets filed so far, when r packets had been (r counted modulo ring + 1; the
  // sums wrap): what a worker finds in a block is the difference of two rows
  uint32_t* sum;      // [ring + 1][sum_stride]
  uint32_t sum_stride;
};

// D -= packets of the log in slots first, first + 1, ... (count of them, in that order), and (SCAN) in the same trip
// the stream pass of the pull: candidates of D, block bounds, histogram.
// A warp owns a block of kWarpTile elements at a time and needs nothing from the other warps.  While it works on one
// block, the values of the next one and its entries in the packets are on their way to shared memory (asynchronous
// copies); lane p has looked up where that block begins and ends in packet p, and the entries lie in packet order.
// 32 of them at a time are subtracted; where several of the 32 hit one element the lane order is the packet order.
// Every D[i] sees the same subtractions in the same order as if the packets had been applied one by one, with one trip
// to memory instead of one per packet.  Only 128-byte lines that hold an entry are written back.
// Blocks are skipped when no packet has an entry in them and (SCAN) their bound lies below L.  The blocks of a CTA
// that are left are dealt out to its warps in runs of about equal cost; a warp is a part of the candidate
// buffer, so the candidates are in index order without any barrier between the warps.
// What bounds it is the warps' instructions: about 300 for a block without entries, 600 with 20 of them, one after the other,
// at half of the issue rate with 16 warps on an SM.  (More blocks of a warp on their way do not help: three or four instead
// of two: 2^26 elements without entries 74 and 84 us for 75.)  So the grid is two CTAs per SM, with ten warps each where
// the pull has the GPU to itself.  Eight / ten / twelve warps, alone: 2^26 elements without entries 73 / 67 / 67 us; 11.7 M in 62
// layers with 3.7 M entries 75 / 60 / 66; 124 M in 148 layers, 8 packets 122 / 111 / 106; 25.6 M 22.3 / 20.7 / 20.3.  Measured alone, in place of a catch-up by ranges of the log followed by the pull's own
// pass over D: 11.7 M elements in 62 layers, 3.7 M entries of 32 packets: 92 us for 272 + 62; 25.6 M elements, 0.8 M
// entries: 46 us for 78 + 28; 124 M elements, 4.0 M entries: 220 us for 434 + 211.
// The grid is the same whether a CTA has kFoldWarps warps or fewer, and so is the plan for it: a pull that has
// the GPU to itself takes the full number, one that shares it with the push passes of later events four (a round
// of 32 arrivals on 124 M elements: 11.6 ms with four warps, 11.7 ms with eight and 12.7 ms with two, whose buffers and threads
// slow the pushes down; one arrival at a time on 25.6 M elements with 8 workers: 127 us with ten, 129 us with eight).
constexpr int kFoldWarpsBeside = 4;
struct FoldStage {                  // one block of one warp
  float tile[kWarpTile];
  uint2 runs[32];                   // the packets with entries in the block, in order, see BlockRuns
  uint2 ent[1];                     // [ahead] entries that are fetched while the block before is worked on
};
struct FoldRange {                  // what a pass folds in
  uint32_t first, count;            // packets: first slot of the log, number
  uint32_t row0, row1;              // rows of running sums before and after them
  uint32_t ahead;                   // entries of a block that are fetched ahead
};
struct FoldShared {
  uint32_t hist[kBins1];            // SCAN: candidates of the CTA's main layer, by bin_of
  uint32_t warp_sum[kFoldWarps];
  uint32_t start[kFoldWarps + 1];   // first block of each warp's run (counted from the CTA's first)
  uint32_t read;
};
__host__ __device__ inline uint32_t fold_stage_bytes(uint32_t ahead) { return kWarpTile * 4u + 32u * 8u + ahead * 8u; }
// dynamic shared memory: two blocks per warp, then per block of the CTA's share one byte (its cost, 0 = skipped) and a bit
__host__ __device__ inline uint32_t fold_dyn_bytes(uint32_t warps, uint32_t ahead, uint32_t part_cap) {   // part_cap: a multiple of 128
  return warps * 2u * fold_stage_bytes(ahead) + part_cap + part_cap / 8u;
}
// cost of a block with that many entries, in units of about 16 entries
__device__ __forceinline__ uint32_t block_cost(uint32_t entries) { return min(255u, 4u + entries / 16u); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
// A block in shared memory is read 16 consecutive elements per lane (so that lane order is element order) and filled
// 16 bytes per lane in memory order; with the 16-byte pieces placed like this neither has bank conflicts.
__device__ __forceinline__ uint32_t tile_place(uint32_t off) {   // where element `off` of the block is
  return off ^ ((off >> 3) & 12u);
}

// The part of one block in up to 32 packets, lane p holding packet p's.  runs[r] = (d, slot) for the r-th packet with
// entries here: the block's entry number e, if it is that packet's, is entry d + e of that slot of the log.
struct BlockRuns {
  uint32_t excl, len;       // this lane's packet: entries of the earlier packets, own entries
  uint32_t total;           // entries of all packets
};
__device__ __forceinline__ BlockRuns block_runs(uint32_t lo, uint32_t hi, uint32_t slot, uint2* runs, int lane, uint32_t lt) {
  BlockRuns r;
  r.len = hi - lo;
  uint32_t incl = r.len;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  r.excl = incl - r.len;
  r.total = __shfl_sync(kFull, incl, 31);
  const uint32_t some = __ballot_sync(kFull, r.len != 0);   // (every lane has read the list before this one by now)
  if (r.len) runs[__popc(some & lt)] = make_uint2(lo - r.excl, slot);
  __syncwarp();
  return r;
}
// where in the log the block's entry e + lane is (e a multiple of 32, e + lane < total)
__device__ __forceinline__ const uint2* entry_at(const PacketLog& lg, const BlockRuns& r, uint32_t e, const uint2* runs, int lane,
                                                 uint32_t le) {
  const uint32_t rel = r.excl - e;
  const uint32_t heads = __reduce_or_sync(kFull, r.len != 0 && rel < 32u ? 1u << rel : 0u);   // entries that open a packet
  const uint32_t before = __popc(__ballot_sync(kFull, r.len != 0 && r.excl < e));
  const uint2 run = runs[max(before + __popc(heads & le), 1u) - 1u];
  return lg.ent + ((uint64_t)run.y * lg.stride + (run.x + e + lane));
}
__device__ __forceinline__ uint2 load_entry(const PacketLog& lg, const BlockRuns& r, uint32_t e, const uint2* runs, int lane, uint32_t le) {
  const uint2* const at = entry_at(lg, r, e, runs, lane, le);
  return e + lane < r.total ? __ldcg(at) : make_uint2(kFull, 0u);
}
// the block's entries e0 .. end - 1 (end <= total), on their way to shared memory; e0 a multiple of 32
__device__ __forceinline__ void fetch_entries(const PacketLog& lg, const BlockRuns& r, uint32_t e0, uint32_t end, const uint2* runs,
                                              uint2* ent, int lane, uint32_t le) {
#pragma unroll 1
  for (uint32_t e = e0; e < end; e += 32) {
    const uint2* const at = entry_at(lg, r, e, runs, lane, le);
    if (e + lane < end) cp_async8(ent + (e - e0) + lane, at);
  }
}
// Subtracts up to 32 entries (`has`: this lane has one) from the block.  Lane order is packet order, and inside one packet
// the indices ascend: 32 entries fall into ascending runs, in each of which every element occurs once, and the runs go
// one after the other, 36 cycles a step.  (Finding the lanes that share an element instead -- with the match instruction,
// with a ballot per bit of the offsets, or with a tag byte per element -- costs more than the steps it saves: a round of
// 32 arrivals on 11.7 M elements takes 3.19 ms by runs, 3.25 ms with ballots above 5 runs, 4.29 ms with tags.)
// Returns this lane's line that was changed.
__device__ __forceinline__ uint32_t subtract_group(float* tile, uint2 q, bool has, uint32_t base, uint32_t n, int lane, uint32_t le) {
  const uint32_t off = has && q.x < n ? q.x - base : kFull;
  const bool valid = off < (uint32_t)kWarpTile;
  const uint32_t prev = __shfl_up_sync(kFull, off, 1);
  const uint32_t opened = __ballot_sync(kFull, lane != 0 && off <= prev && has);   // lanes that open a run, but the first
  const uint32_t turn = __popc(opened & le), most = __popc(opened);
  float* const at = tile + tile_place(off & (uint32_t)(kWarpTile - 1));
  for (uint32_t k = 0;; ++k) {
    if (valid && turn == k) *at = __fsub_rn(*at, __uint_as_float(q.y));
    __syncwarp();
    if (k == most) break;
  }
  return valid ? 1u << (off >> 5) : 0u;
}

// What of a block was not fetched ahead: entries of the first 32 packets beyond the first `ahead` (a multiple of 32),
// and the packets after the first 32 (a worker that has been away for long).  128 entries are on their way while 128 are
// subtracted (a block with 1500 entries is a warp's whole share: with 32 on their way it took 50,000 cycles).
static __device__ __noinline__ uint32_t fold_rest(const PacketLog& lg, uint32_t first, uint32_t count, uint32_t ahead, uint32_t blk, uint32_t n,
                                           FoldStage* st) {
  constexpr int kDeep = 4;
  const int lane = threadIdx.x & 31;
  const uint32_t lt = lanemask_lt(), le = lt | (1u << lane);
  uint32_t dirty = 0;
#pragma unroll 1
  for (uint32_t p0 = 0; p0 < count; p0 += 32) {
    const uint32_t p = p0 + lane, slot = (first + p) % lg.ring;
    uint32_t l = 0, h = 0;
    if (p < count) {
      l = __ldcg(lg.pos + (uint64_t)blk * lg.ring + slot);
      h = __ldcg(lg.pos + (uint64_t)(blk + 1) * lg.ring + slot);
    }
    const BlockRuns r = block_runs(l, h, slot, st->runs, lane, lt);
    uint2 q[kDeep], next[kDeep];
    auto load = [&](uint32_t e) {
#pragma unroll
      for (int u = 0; u < kDeep; ++u)
        if (e + 32u * u < r.total) next[u] = load_entry(lg, r, e + 32u * u, st->runs, lane, le);
    };
    uint32_t e = p0 ? 0u : ahead;
    load(e);
#pragma unroll 1
    for (; e < r.total; e += 32u * kDeep) {
#pragma unroll
      for (int u = 0; u < kDeep; ++u) q[u] = next[u];
      load(e + 32u * kDeep);
#pragma unroll
      for (int u = 0; u < kDeep; ++u)
        if (e + 32u * u < r.total)
          dirty |= subtract_group(st->tile, q[u], e + 32u * u + lane < r.total, blk * kWarpTile, n, lane, le);
    }
    __syncwarp();
  }
  return dirty;
}

// exclusive prefix over the lanes of counts up to 31, and their sum
__device__ __forceinline__ uint32_t lane_offsets(uint32_t count, uint32_t lt, uint32_t& total) {
  uint32_t m = __ballot_sync(kFull, count & 1u), ex = __popc(m & lt);
  total = __popc(m);
  if (!__any_sync(kFull, count > 1)) return ex;    // as it mostly is
#pragma unroll
  for (int b = 1; b < 5; ++b) {
    m = __ballot_sync(kFull, (count >> b) & 1u);
    ex += __popc(m & lt) << b;
    total += __popc(m) << b;
  }
  return ex;
}

// A block in shared memory that is not a full one inside one layer (layer `seg` is its first): every element is compared
// with the bound of its own layer, a layer at a time.  Appends the candidates from slot `at` on, returns how many; top: this
// lane's largest key.  A layer with few entries to send has a bound that admits most of it, so there may be 16 a lane.
// (One element after the other, each with a look at its layer's bound: 15,000 to 21,000 cycles a block, and the warp
// with three of them kept a pass of 45,000 cycles waiting for another 45,000.  11.7 M elements in 62 layers, alone: 49 us, now
// 42, with 0.5 M entries to fold in, 86 us, now 74, with 3.7 M.)
template <bool SCAN>
__device__ __noinline__ uint32_t scan_mixed(const Workspace& ws, const SelArgs& a, const float* t, uint32_t base, uint32_t seg,
                                            uint32_t at, uint32_t main_seg, uint32_t* hist, uint32_t& top) {
  const uint32_t lane = threadIdx.x & 31u, sw = (lane >> 1) & 3u;
  const uint32_t len = min((uint32_t)kWarpTile, ws.n - base);
  const uint32_t len_here = min(16u, max(len, lane * 16u) - lane * 16u);   // of this lane's 16 elements, those in the vector
  uint32_t key[16], best = 0;
#pragma unroll
  for (int j = 0; j < kVecIters; ++j) {
    const uint4 q = *reinterpret_cast<const uint4*>(t + (lane * 4u + ((uint32_t)j ^ sw)) * 4u);
    key[4 * j] = q.x;
    key[4 * j + 1] = q.y;
    key[4 * j + 2] = q.z;
    key[4 * j + 3] = q.w;
  }
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    key[e] &= 0x7FFFFFFFu;
    if ((uint32_t)e < len_here) best = max(best, key[e]);
  }
  top = best;
  if (!SCAN) return 0;
  uint32_t mask = 0;
  // of this lane's 16 elements, those that lie in [lo, hi)
  auto part = [&](uint32_t lo, uint32_t hi) {
    const uint32_t first = min(16u, max(lo, lane * 16u) - lane * 16u), end = min(16u, max(hi, lane * 16u) - lane * 16u);
    return (1u << end) - (1u << first);
  };
  each_layer(ws, a.L_in, seg, base, len, [&](uint32_t, uint32_t lo, uint32_t hi, uint32_t L) {
    const uint32_t here = part(lo, hi);
    if (here) {
      uint32_t m = 0;
#pragma unroll
      for (int e = 0; e < 16; ++e) m |= key[e] >= L ? 1u << e : 0u;
      mask |= m & here;
    }
    __syncwarp();
  });
  uint32_t total;
  uint32_t pos = at + lane_offsets(__popc(mask), lanemask_lt(), total);
  if (total)
    each_layer(ws, a.L_in, seg, base, len, [&](uint32_t s, uint32_t lo, uint32_t hi, uint32_t L) {
      for (uint32_t m = mask & part(lo, hi); m; m &= m - 1) {
        const uint32_t off = lane * 16u + __ffs(m) - 1u;
        const float v = t[tile_place(off)];
        ws.cand_idx[pos] = base + off;
        ws.cand_val[pos] = v;
        ++pos;
        count_bin(ws, hist, main_seg, s, bin_of(key_of(v), L));
      }
      __syncwarp();
    });
  return total;
}

// 72 registers a thread: with 64 the loop over the blocks spills a few (a round of 32 arrivals on 124 M elements: 14.1 ms
// against 11.9), with 80 and 96 fewer warps of other kernels fit beside it (12.4 ms, 12.4 ms).
// ONE: in one kernel with finalize.
template <bool SCAN, bool ONE>
__device__ __forceinline__ void fold_blocks(const Workspace& ws, const SelArgs& a, const PacketLog& lg, const FoldRange& f,
                                            FoldShared& sh, unsigned char* fold_dyn) {
  const uint32_t first = f.first, count = f.count, row0 = f.row0, row1 = f.row1, ahead = f.ahead;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tid = threadIdx.x, nt = blockDim.x, nw = nt / 32u, cta = blockIdx.x, G = gridDim.x;
  const uint32_t lt = lanemask_lt(), le = lt | (1u << lane);
  const uint32_t NB = ws.num_blocks, S = ws.num_segs, n = ws.n;
  float* const D = a.D;
  const uint32_t stage_bytes = fold_stage_bytes(ahead);
  unsigned char* const stages = fold_dyn + warp * 2u * stage_bytes;
  uint8_t* const cost = fold_dyn + nw * 2u * stage_bytes;                        // [part_cap]
  uint32_t* const live = reinterpret_cast<uint32_t*>(cost + ws.part_cap);        // [part_cap / 32]

  // this CTA's blocks [b0, b1)
  uint32_t b0 = part_first_tile(cta, G, NB), b1 = part_first_tile(cta + 1, G, NB);
  if (SCAN && ws.plan != nullptr) {            // (one trip)
    const uint32_t of = ld_volatile(ws.sync + kPlanParts), end = __ldcg(ws.plan + G);
    const uint32_t p0 = __ldcg(ws.plan + cta), p1 = __ldcg(ws.plan + cta + 1);
    if (of == G && end == NB) {
      b0 = p0;
      b1 = p1;
    }
  }
  const uint32_t mine = b0 < b1 ? b1 - b0 : 0u, words = (mine + 31u) / 32u;   // words of `live`

  if (SCAN)
    for (uint32_t b = tid; b < (uint32_t)kBins1; b += nt) sh.hist[b] = 0;
  if (tid <= nw) sh.start[tid] = kFull;
  if (tid == 0) {
    sh.read = 0;
    if (SCAN && cta == 0) {
      ws.sync[kParts] = G * nw;
      // for the next selection, and for the finalize that follows
      ws.sync[kBarCount + (a.pair ^ 1u)] = ws.sync[kFail + (a.pair ^ 1u)] = 0;
      if (!ONE) ws.sync[kBarCount + a.pair] = ws.sync[kFail + a.pair] = 0;
    }
  }

  // A block is skipped if no packet has an entry in it and its bound lies below L.
  uint32_t read = 0;
  for (uint32_t w = warp; w < words; w += nw) {
    const uint32_t b = b0 + w * 32u + lane;
    uint32_t entries = 0;
    bool on = false;
    if (b < b1) {
      if (count) entries = __ldcg(lg.sum + (uint64_t)row1 * lg.sum_stride + b) - __ldcg(lg.sum + (uint64_t)row0 * lg.sum_stride + b);
      if (SCAN) {
        const uint32_t bound = __ldcg(a.blk_max + b);
        uint32_t s = S == 1 ? 0u : __ldg(ws.blk_seg + b);
        uint32_t L = a.L_in[s];
        // The lowest bound of the layers that have a part of the block.  A block in five or more is always read: it holds three of
        // them whole, and of every layer something is sent.
        if (S > 1) {
          const uint64_t end = (uint64_t)(b + 1) * kWarpTile;
          for (int j = 0; j < 4 && L && s + 1 < S && __ldg(ws.seg_off + s + 1) < end; ++j) L = j < 3 ? min(L, a.L_in[++s]) : 0u;
        }
        on = bound >= L;
      }
      on = on || entries != 0;
    }
    cost[w * 32u + lane] = on ? (uint8_t)block_cost(entries) : (uint8_t)0;
    const uint32_t word = __ballot_sync(kFull, on);
    if (lane == 0) {
      live[w] = word;
      read += (word & 0xFFu ? 1u : 0u) + (word & 0xFF00u ? 1u : 0u) + (word & 0xFF0000u ? 1u : 0u) + (word & 0xFF000000u ? 1u : 0u);
    }
  }
  if (SCAN && read) atomicAdd(&sh.read, read);
  __syncthreads();
  // Runs of about equal cost for the warps: warp w begins at the block where the cost so far passes w parts of nw.  A
  // thread adds up `per` consecutive blocks, four at a time.
  uint32_t all;
  {
    const uint32_t quads = words * 8u, per = (quads + nt - 1) / nt, q0 = min(quads, tid * per), q1 = min(quads, q0 + per);
    const uint32_t* const c4 = reinterpret_cast<const uint32_t*>(cost);
    uint32_t sum = 0;
    for (uint32_t q = q0; q < q1; ++q) sum = __dp4a(c4[q], 0x01010101u, sum);
    uint32_t at = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(kFull, at, d);
      if (lane >= d) at += o;
    }
    if (lane == 31) sh.warp_sum[warp] = at;
    __syncthreads();
    at -= sum;
    all = 0;
    for (uint32_t w = 0; w < nw; ++w) {
      if (w == (uint32_t)warp) at += all;
      all += sh.warp_sum[w];                     // (a share has fewer than 2^20 blocks, and a block costs at most 255)
    }
    // first warp whose run begins in this thread's blocks or later: the smallest k with k all / nw >= at
    uint32_t k = sum ? (at * nw + all - 1) / all : nw;     // (below 2^32: nw <= 10, and a block costs at most 255)
    while (k > 0 && sum && (k - 1) * all / nw >= at) --k;
    while (k < nw && k * all / nw < at) ++k;
    if (sum && k < nw && k * all / nw < at + sum) {
      for (uint32_t b = q0 * 4u; b < q1 * 4u; ++b) {
        const uint32_t c = cost[b];
        if (c == 0) continue;
        at += c;
        for (; k < nw && k * all / nw < at; ++k) sh.start[k] = b;
      }
    }
    if (tid == 0) sh.start[nw] = words * 32u;
  }
  __syncthreads();
  // this warp's blocks: the live ones in [run0, run1)
  const uint32_t run0 = sh.start[warp];
  uint32_t run1 = kFull;
  for (uint32_t w = nw; w > (uint32_t)warp; --w)
    if (sh.start[w] != kFull) run1 = sh.start[w];   // (two warps may start at one block: the later one takes it)
  // the layer whose candidates are counted in shared memory; those of others are counted in global memory
  const uint32_t main_seg = S == 1 || b0 >= b1 ? 0u : __ldg(ws.blk_seg + b0 + (b1 - b0) / 2);

  uint32_t walk_word = run0 == kFull ? 0u : run0 / 32u, walk_bits = run0 < run1 ? live[walk_word] & (kFull << (run0 & 31u)) : 0u;
  const uint32_t last_word = run0 < run1 ? (run1 - 1u) / 32u : walk_word;
  auto next_block = [&]() -> uint32_t {        // kFull after the last one
    while (walk_bits == 0) {
      if (walk_word >= last_word) return kFull;
      walk_bits = live[++walk_word];
    }
    const uint32_t b = walk_word * 32u + __ffs(walk_bits) - 1u;
    walk_bits &= walk_bits - 1u;
    return b < run1 ? b0 + b : kFull;
  };
  const uint32_t my_slot = (first + lane) % lg.ring;             // of the first 32 packets
  const uint32_t fill = (lane ^ ((lane >> 3) & 3)) * 4;          // where lane's 16 bytes of a 512-byte piece go
  uint32_t lo = 0, hi = 0;                     // where block blk1 lies in this lane's packet
  auto load_pos = [&](uint32_t b) {
    if (b != kFull && (uint32_t)lane < count) {
      const uint32_t* const pos = lg.pos + (uint64_t)b * lg.ring + my_slot;
      lo = __ldcg(pos);
      hi = __ldcg(pos + lg.ring);
    }
  };
  uint32_t blk = kFull, blk1 = next_block();   // the block in hand, the one that is on its way
  const uint32_t first_blk = blk1;
  load_pos(blk1);
  const uint32_t slot0 = first_blk == kFull ? 0u : first_blk * kWarpTile;   // first slot of this part
  uint32_t cands = 0;
  uint32_t seg = 0, seg_end = 0, L = 0;        // layer of the block in hand (blocks come in ascending order)
  if (first_blk != kFull) {
    seg = S == 1 ? 0u : __ldg(ws.blk_seg + first_blk);
    seg_end = S == 1 ? n : __ldg(ws.seg_off + seg + 1);
    if (SCAN) L = a.L_in[seg];
  }
  const int sw = (lane >> 1) & 3;
  uint32_t total = 0, total1 = 0, phase = 0;   // entries of the first 32 packets in blk, in blk1; stage of blk
  while (blk != kFull || blk1 != kFull) {
    const uint32_t blk2 = blk1 == kFull ? kFull : next_block();
    if (blk1 != kFull) {
      FoldStage* const st = reinterpret_cast<FoldStage*>(stages + (phase ^ stage_bytes));
      const float* const src = D + (size_t)blk1 * kWarpTile + lane * 4;
      const uint32_t len = blk1 + 1 < NB ? (uint32_t)kWarpTile : ws.n_pad - blk1 * kWarpTile;
#pragma unroll
      for (int j = 0; j < kVecIters; ++j)
        if ((uint32_t)(j * 128 + lane * 4) < len) cp_async16(st->tile + j * 128 + fill, src + j * 128);
      if (count) {
        const BlockRuns r = block_runs(lo, hi, my_slot, st->runs, lane, lt);
        total1 = r.total;
        fetch_entries(lg, r, 0, min(r.total, ahead), st->runs, st->ent, lane, le);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    load_pos(blk2);
    if (blk != kFull) {
    const uint32_t base = blk * kWarpTile;
    FoldStage* const st = reinterpret_cast<FoldStage*>(stages + phase);
    float* const t = st->tile;
    while (base >= seg_end) {
      ++seg;
      seg_end = __ldg(ws.seg_off + seg + 1);
      if (SCAN) L = a.L_in[seg];
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    // fold
    if (count) {
      uint32_t dirty = 0;
      const uint32_t ready = min(total, ahead);
#pragma unroll 1
      for (uint32_t e = 0; e < ready; e += 32)
        dirty |= subtract_group(t, st->ent[e + lane], e + lane < ready, base, n, lane, le);   // (ent is a multiple of 32 long)
      if (total > ahead || count > 32u) dirty |= fold_rest(lg, first, count, ahead, blk, n, st);
      dirty = __reduce_or_sync(kFull, dirty);
      if (dirty) {     // changed lines back to memory
        float* const dst = D + (size_t)base + lane * 4;
#pragma unroll
        for (int j = 0; j < kVecIters; ++j)
          if ((dirty >> (j * 4 + (lane >> 3))) & 1u)
            __stcg(reinterpret_cast<float4*>(dst + j * 128), *reinterpret_cast<const float4*>(t + j * 128 + fill));
      }
    }
    // scan: bound and candidates
    uint32_t top;
    if (blk + 1 < NB && base + kWarpTile <= seg_end) {   // a full block inside one layer
      float4 v[kVecIters];
#pragma unroll
      for (int j = 0; j < kVecIters; ++j) v[j] = *reinterpret_cast<const float4*>(t + (lane * 4 + (j ^ sw)) * 4);
      float m = 0.f;
#pragma unroll
      for (int j = 0; j < kVecIters; ++j)
        m = fmaxf(fmaxf(m, fmaxf(fabsf(v[j].x), fabsf(v[j].y))), fmaxf(fabsf(v[j].z), fabsf(v[j].w)));
      const uint32_t own = __float_as_uint(m);
      top = __reduce_max_sync(kFull, own);
      if (SCAN && top >= L) {
        const float Lf = __uint_as_float(L);   // |x| >= Lf  <=>  key(x) >= L for finite x (no flush-to-zero)
        uint32_t mask = 0;
        if (own >= L) {
#pragma unroll
          for (int j = 0; j < kVecIters; ++j)
            mask |= ((fabsf(v[j].x) >= Lf ? 1u : 0u) | (fabsf(v[j].y) >= Lf ? 2u : 0u) | (fabsf(v[j].z) >= Lf ? 4u : 0u) |
                     (fabsf(v[j].w) >= Lf ? 8u : 0u)) << (4 * j);
        }
        __syncwarp();
        uint32_t found;
        uint32_t pos = slot0 + cands + lane_offsets(__popc(mask), lt, found);
        cands += found;
        while (mask) {
          const uint32_t off = lane * 16 + __ffs(mask) - 1;
          mask &= mask - 1;
          const float c = t[tile_place(off)];
          ws.cand_idx[pos] = base + off;
          ws.cand_val[pos] = c;
          ++pos;
          count_bin(ws, sh.hist, main_seg, seg, bin_of(key_of(c), L));
        }
      }
    } else {
      cands += scan_mixed<SCAN>(ws, a, t, base, seg, slot0 + cands, main_seg, sh.hist, top);
      top = __reduce_max_sync(kFull, top);
    }
    if (lane == 0) a.blk_max[blk] = top;     // the block's bound is exact again (entries sent later only lower it)
    __syncwarp();   // the block's stage is free
    }
    phase ^= stage_bytes;
    blk = blk1;
    blk1 = blk2;
    total = total1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (SCAN) {
    if (lane == 0) {
      ws.part_cands[cta * nw + warp] = cands;
      ws.part_slot0[cta * nw + warp] = slot0;
    }
    __syncthreads();
    for (uint32_t b = tid; b < (uint32_t)kBins1; b += nt)
      if (sh.hist[b]) atomicAdd(ws.hist1 + (size_t)main_seg * kBins1 + b, sh.hist[b]);
    if (tid == 0) {
      if (ws.cta_cost != nullptr) ws.cta_cost[cta] = all;
      atomicAdd(ws.stats + 3, (unsigned long long)((mine + 7u) / 8u));
      atomicAdd(ws.stats + 4, (unsigned long long)sh.read);
    }
  }
}
template <bool SCAN>
__global__ void __maxnreg__(72) k_fold(const __grid_constant__ Workspace ws, const __grid_constant__ SelArgs a,
                                       const __grid_constant__ PacketLog lg, const __grid_constant__ FoldRange f) {
  __shared__ FoldShared sh;
  extern __shared__ __align__(16) unsigned char fold_dyn[];
  fold_blocks<SCAN, false>(ws, a, lg, f, sh, fold_dyn);
}

}  // namespace dgs
