// Host side of the C ABI declared in include/dgs.h: argument checks, the layout of
// the caller's arena, and the kernel launches of one push / apply / pull event.
//
// Work runs on streams of the library's own so that consecutive events overlap: an event's push, apply and pull
// follow one another on one stream, and events take kStreams streams in turn.  A push touches only the worker's
// velocity, the gradient and its scratch; a pull touches one difference vector.  The small, latency-bound kernels
// thus share the GPU with the bandwidth-bound passes of other events.  An event that starts while nothing else is
// in flight always takes the first stream, and streams are created when they are first taken: a caller that joins
// after every event uses one.  (Eleven streams per context -- four for pushes, one for applies, six for pulls --
// cost every event a hop from stream to stream between its steps, and every stream that is alive costs the others:
// with three contexts alive, one event of 25.6 M elements took 185 us where it took 158 us with one.)
// Order is kept by a small dependency tracker: every launch names the buffers it reads and writes, and waits
// (cudaStreamWaitEvent) for the last writer of what it reads and for the last writer and the readers of what it
// writes.  Per buffer the order of operations is therefore the order of the calls, which keeps the results
// bit-identical to a serial run.
#include "dgs.h"

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "dgs_apply.cuh"
#include "dgs_arrivals.h"
#include "dgs_kernels.cuh"
#include "dgs_one.cuh"
#include "dgs_topk.cuh"

using namespace dgs;

namespace {

constexpr uint64_t kAlign = 256;
constexpr uint32_t kMagic = 0x44475331u;  // "DGS1"
constexpr int kPushSlots = 8;  // push packet slots, used in turn (a slot is refilled once its apply has read it)
constexpr int kPullSlots = 8;             // pull packet slots
constexpr int kVarSlots = 4;              // packet slots of the pull without secondary compression
constexpr int kStreams = 8;               // most events in flight at a time
constexpr int kSets = kStreams;           // scratch sets and spare velocity buffers: one of each per stream
// Events in flight at a time: the push of an event runs beside the pulls of the ones before it, those of the same worker
// included, so even a few workers fill all of the streams.  Microseconds an event in runs of 256 without a join, 2 / 4 / 8
// streams: 2 workers, 8.4 M elements: 53 / 39 / 36; 4 workers, 25.6 M: 82 / 65 / 57; 32 workers: 87 / 66 / 60.  A single
// worker's events have one push and one pull at a time to overlap: 236 with two streams, 236 to 245 with more, 267 with one.
int streams_for(const dgs_config* c) {
  if (c->flags & DGS_SINGLE_STREAM) return 1;   // kernels run one after the other, in call order
  return c->num_workers == 1 ? 2 : kStreams;
}
constexpr int kCaller = kStreams;         // the caller's stream, where the tracker names streams by number
constexpr int kQueuesWanted = 12;         // hardware queues for the streams of one context, the caller's and a few more
constexpr int kLogRingMax = 128;            // most packets the apply log keeps
constexpr int kLogSlack = 32;               // slots of the log beyond one per worker
constexpr uint64_t kListCap = 4096;         // most entries of a layer's list of candidates in the k-th's bin
constexpr uint64_t kOneMaxN = 3ull << 19;   // longest vector whose selections are one kernel each
// ... beside other events: with more layers a CTA has more bounds to pick for, and finalize has fewer CTAs in that kernel.  Rounds of 12
// and 16 arrivals, us, two kernels a selection / one: one layer: 0.5 M elements 313 / 235, 1.05 M 250 / 180, 1.5 M 262 / 200; 2 layers:
// 1.05 M 212 / 206, 1.2 M 215 / 222; 8: 0.7 M 279 / 191, 1.05 M 216 / 218, 1.2 M 219 / 232; 20: 0.7 M 241 / 228, 0.9 M 225 / 231; 60: 0.5 M
// 317 / 255, 0.7 M 249 / 249, 0.88 M 251 / 266; 200: 0.25 M 307 / 280, 0.5 M 314 / 316, 0.7 M 330 / 356; 1000: 0.25 M 675 / 712, at 2 % 815 /
// 932.  Dense selections differ less: 1.5 M elements in one layer, 20 %: 1090 / 1075; 0.5 M in 60, 20 %: 645 / 648.
constexpr uint64_t one_max_beside(uint32_t layers) {
  constexpr uint64_t least = 1ull << 19, most = 1ull << 20;
  if (layers == 1) return kOneMaxN;
  return layers > 512 ? 0 : layers < 64 ? most - ((uint64_t)layers << 13) : least;
}
static_assert(one_max_beside(63) >= one_max_beside(64) && one_max_beside(2) < kOneMaxN, "fewer elements for more layers");
constexpr uint32_t kOneGridBeside = 64;     // most CTAs of that kernel beside other events

inline uint64_t align_up(uint64_t x, uint64_t a) { return (x + a - 1) / a * a; }

// Scratch of the selections on one stream
struct ScratchLayout {
  uint64_t cand_idx, cand_val, part_cands, part_slot0, plan, cta_cost, cta_tot, cta_eq, tab, list;
  uint64_t hist1, list_cnt, sel, L_safe, L_wide, sync;
  uint64_t zero_begin, zero_end;  // [hist1, end of sync): cleared at init
};

struct Layout {
  uint64_t n_pad = 0;  // elements per state vector, padded to 256 bytes
  uint32_t num_tiles = 0;
  uint64_t K[2] = {0, 0};
  // byte offsets into the arena
  uint64_t theta, u, D, theta_local, grad_stage;
  uint64_t pkt_idx[kPushSlots + kPullSlots], pkt_val[kPushSlots + kPullSlots];  // push slots, then pull slots
  uint64_t var_idx[kVarSlots], var_val[kVarSlots], var_count[kVarSlots], L_one;
  uint64_t tiles, segs, seg_off, blk_seg;
  ScratchLayout sc[kSets];
  uint64_t L_next, slack, u_slots, status, stats;
  uint64_t log_ent, log_pos, log_sum;   // ring of applied packets not yet folded into every D_q
  uint64_t blk_max;      // [N][blk_stride]: per block of kWarpTile elements, an upper bound on the keys of D_q in it
  uint64_t blk_stride = 0;
  uint32_t log_ring = 0, log_stride = 0, pos_rows = 0, sum_stride = 0;
  uint32_t num_blocks = 0;
  uint64_t total = 0;
};

int check_config(const dgs_config* c) {
  if (!c || !c->segments) return DGS_EINVAL;
  if (c->n == 0 || c->n >= (1ull << 32)) return DGS_EINVAL;
  if (c->num_workers == 0 || c->num_workers > 65535) return DGS_EINVAL;
  if (c->num_segments == 0 || c->num_segments >= 65536) return DGS_EINVAL;
  if (c->pull_all_capacity > c->n) return DGS_EINVAL;
  if ((c->flags & DGS_PACKET_BF16) && (c->flags & DGS_PACKET_FP16)) return DGS_EINVAL;
  if (!std::isfinite(c->lr)) return DGS_EINVAL;
  if (!(c->momentum > 0.0f) || !(c->momentum <= 1.0f)) return DGS_EINVAL;
  uint64_t pos = 0;
  for (uint32_t s = 0; s < c->num_segments; ++s) {
    const dgs_segment& g = c->segments[s];
    if (g.offset != pos || g.len == 0) return DGS_EINVAL;
    if (g.k_push == 0 || g.k_push > g.len || g.k_pull == 0 || g.k_pull > g.len) return DGS_EINVAL;
    pos += g.len;
  }
  if (pos != c->n) return DGS_EINVAL;
  return DGS_OK;
}

// Tiles: every layer is cut at the global multiples of kWarpTile, so that all full
// tiles start 2 KB-aligned and only the first and last tile of a layer can be ragged.
void build_tiles(const dgs_config* c, std::vector<Tile>* tiles, std::vector<SegDesc>* segs) {
  uint32_t koff[2] = {0, 0}, list_off = 0;
  for (uint32_t s = 0; s < c->num_segments; ++s) {
    const dgs_segment& g = c->segments[s];
    SegDesc d;
    d.tile_begin = (uint32_t)tiles->size();
    uint64_t pos = g.offset, end = g.offset + g.len;
    uint32_t count = 0;
    while (pos < end) {
      const uint64_t next = std::min<uint64_t>(end, (pos / kWarpTile + 1) * kWarpTile);
      Tile t;
      t.start = (uint32_t)pos;
      t.len = (uint16_t)(next - pos);
      t.seg = (uint16_t)s;
      tiles->push_back(t);
      ++count;
      pos = next;
    }
    d.tile_end = d.tile_begin + count;
    d.k[0] = g.k_push;
    d.k[1] = g.k_pull;
    d.pkt_off[0] = koff[0];
    d.pkt_off[1] = koff[1];
    d.list_off = list_off;
    d.list_cap = (uint32_t)std::min<uint64_t>(g.len, kListCap);
    list_off += d.list_cap;
    koff[0] += g.k_push;
    koff[1] += g.k_pull;
    segs->push_back(d);
  }
}

uint32_t count_tiles(const dgs_config* c) {
  uint64_t tiles = 0;
  for (uint32_t s = 0; s < c->num_segments; ++s) {
    const dgs_segment& g = c->segments[s];
    const uint64_t first = g.offset / kWarpTile, last = (g.offset + g.len - 1) / kWarpTile;
    tiles += last - first + 1;
  }
  return (uint32_t)tiles;
}

void make_layout(const dgs_config* c, Layout* L) {
  const uint64_t N = c->num_workers, S = c->num_segments;
  L->n_pad = align_up(c->n, kAlign / 4);
  L->num_tiles = count_tiles(c);
  L->num_blocks = (uint32_t)((c->n + kWarpTile - 1) / kWarpTile);
  L->K[0] = L->K[1] = 0;
  uint64_t list_entries = 0;
  for (uint32_t s = 0; s < S; ++s) {
    L->K[0] += c->segments[s].k_push;
    L->K[1] += c->segments[s].k_pull;
    list_entries += std::min<uint64_t>(c->segments[s].len, kListCap);
  }
  uint64_t off = 0;
  auto take = [&](uint64_t bytes) {
    const uint64_t at = off;
    off = align_up(off + bytes, kAlign);
    return at;
  };
  const uint64_t vec = L->n_pad * 4;
  L->theta = take(vec);
  L->u = take(vec * (N + streams_for(c)));  // N velocities and the spares that pushes write into
  L->D = take(vec * N);
  L->theta_local = (c->flags & DGS_KEEP_LOCAL_MODEL) ? take(vec * N) : 0;
  L->grad_stage = (c->flags & DGS_HOST_IO) ? take(vec) : 0;
  for (int p = 0; p < kPushSlots + kPullSlots; ++p) {
    const uint64_t K = L->K[p < kPushSlots ? 0 : 1];
    L->pkt_idx[p] = take(K * 4);
    L->pkt_val[p] = take(K * 4);
  }
  for (int p = 0; p < kVarSlots; ++p) {
    L->var_idx[p] = c->pull_all_capacity ? take((uint64_t)c->pull_all_capacity * 4) : 0;
    L->var_val[p] = c->pull_all_capacity ? take((uint64_t)c->pull_all_capacity * 4) : 0;
    L->var_count[p] = c->pull_all_capacity ? take(4) : 0;
  }
  L->L_one = take(S * 4);
  L->tiles = take((uint64_t)L->num_tiles * sizeof(Tile));
  L->segs = take(S * sizeof(SegDesc));
  L->seg_off = take((S + 1) * 4);
  L->blk_seg = take((uint64_t)L->num_blocks * 4);
  for (int k = 0; k < streams_for(c); ++k) {
    ScratchLayout& sc = L->sc[k];
    sc.cand_idx = take(vec);
    sc.cand_val = take(vec);
    sc.part_cands = take((uint64_t)kMaxParts * 4);
    sc.part_slot0 = take((uint64_t)kMaxParts * 4);
    sc.plan = take((uint64_t)(kMaxFoldGrid + 1) * 4);
    sc.cta_cost = take((uint64_t)kMaxFoldGrid * 4);
    sc.cta_tot = take((uint64_t)kMaxWorkers * sizeof(uint2));
    sc.cta_eq = take((uint64_t)kMaxWorkers * 4);
    sc.tab = take((S + kMaxWorkers) * sizeof(LayerPick));
    sc.list = take(list_entries * sizeof(uint2));
    sc.hist1 = take(S * kBins1 * 4);
    sc.zero_begin = sc.hist1;
    sc.list_cnt = take(S * 4);
    sc.sel = take(S * sizeof(SegSel));
    sc.L_safe = take(S * 4);
    sc.L_wide = take(S * 4);
    sc.sync = take(kNumSyncWords * 4);
    sc.zero_end = off;
  }
  // A slot of the log is reused `ring` packets later, and the apply that refills it waits for every catch-up that
  // still reads the old packet.  A worker that comes back after N events reads the N newest packets, so ring - N
  // is how many events the server side of an event may lag behind the pushes before the pushes stall.
  // (with irregular arrivals a worker is often away for more than N events -- one gap in eight is longer than 2 N when
  // every event's worker is drawn at random -- and a worker about to fall off the ring is caught up on the apply
  // stream, in the way of every later event: four rounds of room where that many packets fit the cap)
  L->log_ring = (uint32_t)std::min<uint64_t>(kLogRingMax, std::max<uint64_t>(std::max<uint64_t>(N + kLogSlack, 4 * N), 16));
  L->log_stride = (uint32_t)align_up(L->K[0], 64);
  L->log_ent = take((uint64_t)L->log_ring * L->log_stride * sizeof(uint2));
  L->pos_rows = L->num_blocks + 1;
  L->log_pos = take((uint64_t)L->log_ring * L->pos_rows * 4);
  L->sum_stride = (uint32_t)align_up(L->pos_rows, 64);
  L->log_sum = take((uint64_t)(L->log_ring + 1) * L->sum_stride * 4);
  L->blk_stride = align_up((c->n + kWarpTile - 1) / kWarpTile, 64);
  L->blk_max = take(N * L->blk_stride * 4);
  L->L_next = take(4 * N * S * 4);
  L->slack = take(2 * S * 4);
  L->u_slots = take((N + kSets) * sizeof(float*));
  L->status = take(4);
  L->stats = take((uint64_t)kNumStats * 8);
  L->total = off;
}

}  // namespace

struct dgs_ctx {
  uint32_t magic;
  dgs_config cfg;
  std::vector<dgs_segment> segments;
  Layout lay;
  char* base;
  cudaStream_t user;       // the caller's stream: entry point of dependencies, target of dgs_flush
  cudaStream_t st[kStreams + 1];   // null until first taken; [kCaller]: the caller's
  int streams;             // how many of them may be taken (1 under DGS_SINGLE_STREAM)
  int next_stream;         // the one that the next event takes ...
  bool idle;               // ... unless nothing has been enqueued since everything was last joined: then the first one
  bool dirty[kStreams + 1];    // stream has work that the caller's stream has not been made to wait for
  std::vector<int> worker_stream;   // per worker: stream of its last push if its pull is still to come, else -1
  int slot_stream[kPushSlots];      // per push packet slot: stream of its push
  cudaEvent_t ev_in;       // "everything the caller had enqueued when the call was made"
  bool forked[kStreams + 1];  // stream already waits for ev_in of the current call
  cudaEvent_t ev_tail[kStreams];  // for dgs_flush
  // dependency tracker
  struct Dep {
    cudaEvent_t ev = nullptr;
    int stream = -1;
    uint64_t seq = 0;  // position of the task in the order of all tasks (0: none)
  };
  struct Res {
    Dep last_write;
    std::vector<Dep> reads;  // readers since the last write
  };
  std::vector<Res> res;
  // one "done" event per task, reused in turn; a ring per stream, so that an event is only ever
  // re-recorded later on the same stream and waiting for a reused one still covers the older task
  std::vector<cudaEvent_t> ev_ring[kStreams + 1];
  size_t ev_next[kStreams + 1];
  uint64_t task_seq;                               // tasks filed so far
  uint64_t waited_seq[kStreams + 1][kStreams + 1];   // [waiting stream][stream]: newest task already waited for
  uint64_t push_count, pull_count, event_count, var_count;
  // Lazy difference vectors: packet number p (counted from 0) of the library's own pushes sits in slot
  // p % ring of the log from its apply on; applied[q] packets have been folded into D_q so far.
  PacketLog log;
  uint64_t log_head;              // packets filed so far
  std::vector<uint64_t> applied;  // per worker
  Workspace ws[kSets];
  float inv_m;
  int sms;               // SMs of the device
  int stream_grid[3];    // CTAs of the stand-alone stream pass, per mode
  int fold_grid;         // CTAs of k_fold
  uint32_t fold_ahead;   // entries of a block it fetches ahead
  // No pull has been enqueued since the caller's stream was last made to wait for everything (dgs_flush, or a call
  // that waits): the event in hand starts on an idle GPU.
  bool idle_gpu;
  Arrivals arrivals;
  int hist_grid[3];      // CTAs of the whole-input histogram pass, per mode
  int one_max[3];        // most CTAs of pass and finalize in one kernel, per mode
  uint32_t pair[kSets];  // pair of sync words that the last selection on each scratch set has used
  int finalize_max[3];   // most CTAs of the cooperative finalize kernel that can be resident at once, per mode
  uint64_t whole_layers;  // elements of layers that may be candidates as a whole (several layers)
  uint64_t kind_seq[2];  // selections of each kind launched so far
  // Carried bounds: row (kind, worker) of L_next holds the bounds suggested by that worker's
  // latest selection of that kind ([0] push, [1] pull).  There are two copies of a row, written in turn
  // (row_copy: the latest): the worker's next selection need not wait until nobody reads the bounds of its
  // last one.  With one copy, and one stream less than workers that arrive in turn, every selection read
  // the row of the worker that came next, and no two events overlapped (8 workers, 2^20 elements: 34 us an event
  // with 7 streams, 17 us with 6 or 8).  row_age says in which state it was
  // made: pushes the worker had done before (push), packets accumulated in D_w since its
  // previous pull (pull).  Thresholds grow with that age, so a row made at an age no larger
  // than the current one is a safe-side guess; the most recent such row is used.
  std::vector<uint8_t> row_valid[2], row_copy[2];
  std::vector<uint64_t> row_time[2], row_age[2];
  std::vector<uint64_t> pushes;  // pushes done per worker
  std::vector<int64_t> prev;
  uint64_t timestamp;
  uint64_t launches;
  int last_cuda;
  bool broken;
  // optional per-kernel timing (CUDA events on the launching stream)
  bool timing;
  std::vector<cudaEvent_t> ev_pool;   // pairs: [2i] start, [2i+1] stop
  std::vector<int> ev_kernel;         // kernel id of each recorded pair
  std::vector<int> ev_stream;         // index of the library stream it ran on
  double time_ms[DGS_NUM_KERNELS];
  uint64_t time_count[DGS_NUM_KERNELS];

  template <typename T>
  T* at(uint64_t off) const { return reinterpret_cast<T*>(base + off); }
  float* u_buf(uint32_t q) const { return at<float>(lay.u) + (uint64_t)q * lay.n_pad; }
  float* D_buf(uint32_t q) const { return at<float>(lay.D) + (uint64_t)q * lay.n_pad; }
  float* theta_local_buf(uint32_t q) const { return at<float>(lay.theta_local) + (uint64_t)q * lay.n_pad; }
  uint32_t* blk_max(uint32_t q) const { return at<uint32_t>(lay.blk_max) + (uint64_t)q * lay.blk_stride; }
  float** u_slot(uint32_t q) const { return at<float*>(lay.u_slots) + q; }
  uint32_t* L_next(int pm, int copy, uint32_t w) const {
    return at<uint32_t>(lay.L_next) + ((uint64_t)(2 * pm + copy) * cfg.num_workers + w) * cfg.num_segments;
  }
};

namespace {

// resources of the dependency tracker
struct ResIds {
  uint32_t N;
  uint32_t U(uint32_t w) const { return w; }
  uint32_t D(uint32_t q) const { return N + q; }
  uint32_t TL(uint32_t q) const { return 2 * N + q; }
  uint32_t ROW(int kind, int copy, uint32_t w) const { return 3 * N + (uint32_t)(2 * kind + copy) * N + w; }
  uint32_t THETA() const { return 7 * N; }
  uint32_t SPARE(int j) const { return THETA() + 1 + j; }
  uint32_t SCR(int set) const { return SPARE(kSets) + set; }
  uint32_t PKT(int slot) const { return SCR(kSets) + slot; }   // push slots, then pull slots
  uint32_t VPKT(int slot) const { return PKT(kPushSlots + kPullSlots) + (uint32_t)slot; }
  uint32_t STAGE() const { return VPKT(kVarSlots); }
  uint32_t LOG(uint32_t slot) const { return STAGE() + 1 + slot; }
  uint32_t count() const { return LOG(kLogRingMax); }
};

#define DGS_CUDA(ctx, call)                 \
  do {                                      \
    cudaError_t e_ = (call);                \
    if (e_ != cudaSuccess) {                \
      (ctx)->last_cuda = (int)e_;           \
      (ctx)->broken = true;                 \
      return DGS_ECUDA;                     \
    }                                       \
  } while (0)

inline int live(dgs_ctx* c) {
  if (!c || c->magic != kMagic) return DGS_ESTATE;
  if (c->broken) return DGS_ESTATE;
  return DGS_OK;
}

constexpr int kEventRing = 256;       // "done" events per stream, used in turn
constexpr size_t kMaxTimedLaunches = 1 << 16;
constexpr uint64_t kFinalizeMin = 32;  // fewest CTAs of the finalize kernel

// Records an event before and after one launch when timing is on.
struct TimedLaunch {
  dgs_ctx* c;
  cudaStream_t st;
  cudaEvent_t stop = nullptr;
  TimedLaunch(dgs_ctx* ctx, cudaStream_t stream, int kernel_id) : c(ctx), st(stream) {
    if (!c->timing || c->ev_kernel.size() >= kMaxTimedLaunches) return;
    const size_t i = c->ev_kernel.size();
    while (c->ev_pool.size() < 2 * (i + 1)) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return;
      c->ev_pool.push_back(e);
    }
    if (cudaEventRecord(c->ev_pool[2 * i], st) != cudaSuccess) return;
    stop = c->ev_pool[2 * i + 1];
    c->ev_kernel.push_back(kernel_id);
    int which = -1;
    for (int j = 0; j < kStreams; ++j)
      if (c->st[j] == st) which = j;
    c->ev_stream.push_back(which);
  }
  ~TimedLaunch() {
    if (stop) cudaEventRecord(stop, st);
  }
};

// Makes an internal stream wait for everything the caller had enqueued on its stream when the
// current API call began (ev_in is recorded once per call by begin_call).
int begin_call(dgs_ctx* c) {
  DGS_CUDA(c, cudaEventRecord(c->ev_in, c->user));
  for (int i = 0; i < kStreams; ++i) c->forked[i] = false;
  return DGS_OK;
}
int stream_ready(dgs_ctx* c, int which) {
  if (!c->ev_ring[which].empty()) return DGS_OK;
  if (which != kCaller) {
    DGS_CUDA(c, cudaStreamCreateWithFlags(&c->st[which], cudaStreamNonBlocking));
    DGS_CUDA(c, cudaEventCreateWithFlags(&c->ev_tail[which], cudaEventDisableTiming));
  }
  for (int i = 0; i < kEventRing; ++i) {
    cudaEvent_t e;
    DGS_CUDA(c, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    c->ev_ring[which].push_back(e);
  }
  return DGS_OK;
}
// The stream of the next event, and taking it.
int peek_stream(const dgs_ctx* c) { return c->idle ? 0 : c->next_stream; }
int take_stream(dgs_ctx* c) {
  const int s = peek_stream(c);
  c->idle = false;
  c->next_stream = (s + 1) % c->streams;
  return s;
}
int fork_from_user(dgs_ctx* c, int which) {
  const int rc = stream_ready(c, which);
  if (rc != DGS_OK) return rc;
  if (c->forked[which]) return DGS_OK;
  DGS_CUDA(c, cudaStreamWaitEvent(c->st[which], c->ev_in, 0));
  c->forked[which] = true;
  c->waited_seq[which][kCaller] = c->task_seq;   // (ev_in was recorded after the tasks on the caller's stream)
  return DGS_OK;
}

// Everything that was in flight is complete, or the caller's stream waits for it.
void joined(dgs_ctx* c) {
  c->arrivals.joined();
  c->idle = c->idle_gpu = true;
}
// Whether the event in hand has the GPU to itself.  The one that opens a round of several does not: the others are enqueued
// right behind it, and a finalize sized for an idle GPU, whose CTAs must all be resident, waits for room beside their passes and
// keeps them waiting.  What follows a join is taken to be as many events as between the last two.  (Rounds of 8 arrivals on
// 124 M elements in 148 layers, us, every event after a join taken for alone / this: 3022 / 2877; of 32 on 11.7 M in 62 layers
// 2870 / 2789; of 8 on 8.4 M in 2000 layers 1280 / 1115; one arrival at a time the same.)
bool has_gpu(const dgs_ctx* c) { return c->idle_gpu && c->arrivals.lone(); }

// Waits (on the host) for all internal streams ...
int sync_library(dgs_ctx* c) {
  for (int i = 0; i < kStreams; ++i) {
    if (c->st[i] && c->dirty[i]) DGS_CUDA(c, cudaStreamSynchronize(c->st[i]));
    c->dirty[i] = false;                     // nothing that the caller's stream would have to wait for
  }
  joined(c);
  return DGS_OK;
}
// ... and the caller's stream (which has been made to wait for those that are not dirty).
int sync_all(dgs_ctx* c) {
  const int rc = sync_library(c);
  if (rc != DGS_OK) return rc;
  DGS_CUDA(c, cudaStreamSynchronize(c->user));
  return DGS_OK;
}

// A task = the launches of one step on one stream.  task_begin makes the stream wait for
// whatever the task depends on; task_end records the task's completion and files it with
// the buffers it touched.
struct Task {
  int stream;
  std::vector<uint32_t> reads, writes;
};
int task_begin(dgs_ctx* c, const Task& t) {
  const int ready = stream_ready(c, t.stream);
  if (ready != DGS_OK) return ready;
  // Tasks of one stream complete in order, so per stream only the newest task that this one depends
  // on matters, and only if the stream has not already waited for that task or a newer one.
  dgs_ctx::Dep need[kStreams + 1];
  auto want = [&](const dgs_ctx::Dep& d) {
    if (!d.ev || d.stream == t.stream) return;   // same stream: already ordered
    if (d.seq > need[d.stream].seq) need[d.stream] = d;
  };
  for (uint32_t r : t.reads) want(c->res[r].last_write);
  for (uint32_t w : t.writes) {
    const dgs_ctx::Res& x = c->res[w];
    want(x.last_write);
    for (const dgs_ctx::Dep& rd : x.reads) want(rd);
  }
  for (int s = 0; s <= kCaller; ++s) {
    if (!need[s].ev || need[s].seq <= c->waited_seq[t.stream][s]) continue;
    DGS_CUDA(c, cudaStreamWaitEvent(c->st[t.stream], need[s].ev, 0));
    c->waited_seq[t.stream][s] = need[s].seq;
  }
  return DGS_OK;
}
int task_end(dgs_ctx* c, const Task& t) {
  c->dirty[t.stream] = true;
  dgs_ctx::Dep d;
  d.ev = c->ev_ring[t.stream][c->ev_next[t.stream]];
  d.stream = t.stream;
  d.seq = ++c->task_seq;
  c->ev_next[t.stream] = (c->ev_next[t.stream] + 1) % c->ev_ring[t.stream].size();
  DGS_CUDA(c, cudaEventRecord(d.ev, c->st[t.stream]));
  for (uint32_t r : t.reads) c->res[r].reads.push_back(d);
  for (uint32_t w : t.writes) {
    dgs_ctx::Res& x = c->res[w];
    x.last_write = d;
    x.reads.clear();
  }
  return DGS_OK;
}

// Dependencies of folding the filed packets that D_q has not seen yet into it.
void catch_up_deps(const dgs_ctx* c, uint32_t q, Task* t) {
  const ResIds R{c->cfg.num_workers};
  for (uint64_t p = c->applied[q]; p < c->log_head; ++p) t->reads.push_back(R.LOG((uint32_t)(p % c->log.ring)));
  t->writes.push_back(R.D(q));
}
// The filed packets that D_q has not seen yet.
FoldRange fold_range(const dgs_ctx* c, uint32_t q) {
  const uint32_t ring = c->log.ring;
  FoldRange f;
  f.first = (uint32_t)(c->applied[q] % ring);
  f.count = (uint32_t)(c->log_head - c->applied[q]);   // <= ring
  f.row0 = (uint32_t)(c->applied[q] % (ring + 1));
  f.row1 = (uint32_t)(c->log_head % (ring + 1));
  f.ahead = c->fold_ahead;
  return f;
}
// Warps of a CTA of the pass: ten where the pull has the GPU to itself, as with a single worker, whose pulls follow one another;
// eight where one other pull may be in flight (a worker has one at a time), four beside more.  us, 16 arrivals, eight / ten: 1
// worker, 8.4 M elements 3045 / 2976, 62 layers of 11.7 M 4774 / 4700; 2 workers 615 / 640, 1518 / 1536; but rounds of 2 workers on
// 19 M 173 / 174, on 50 M, where the passes are long beside everything else, 361 / 348.  us an event in runs of
// 256, eight / four: 2 workers, 8.4 M: 36 / 40, 62 layers of 11.7 M: 95 / 101; 3 workers, 25.6 M: 66 / 63; 8 workers: 61 / 57, 62
// layers of 11.7 M: 83 / 78.  (Vectors of 500 M elements with many entries, where an SM has room for one CTA of ten warps or two of
// eight: pass of a pull alone 1308 / 1342.)
// The pull that opens a round (idle) takes ten as well where it is a long one of a long vector, us a round, four / ten: 25.6 M
// elements, 32 workers 2072 / 2057, 16: 1026 / 1028, 8: 531 / 536; 124 M, 32 workers 11,130 / 11,060; but 8.4 M, 32 workers 1038 / 1059, 4:
// 166 / 178; 62 layers of 11.7 M, 32 workers 2779 / 2791.
constexpr uint32_t fold_warps(uint32_t workers, uint64_t n, bool idle, bool alone) {
  if (alone || workers == 1 || (workers == 2 && n >= 1ull << 25) || (idle && workers >= 16 && n >= 1ull << 24)) return kFoldWarps;
  return workers == 2 ? kWarps : kFoldWarpsBeside;
}
static_assert(fold_warps(32, 1000, true, true) == 10 && fold_warps(1, 1000, false, false) == 10, "alone");
static_assert(fold_warps(2, 1ull << 24, true, false) == 8 && fold_warps(2, 1ull << 25, false, false) == 10 && fold_warps(3, 1ull << 25, true, false) == 4, "a few in flight");
static_assert(fold_warps(16, 1ull << 24, true, false) == 10 && fold_warps(16, 1ull << 24, false, false) == 4, "");

// The launch itself, on a stream that task_begin has prepared with those dependencies; with SCAN the stream pass of a pull
// in the same trip over D_q.
template <bool SCAN>
int fold_launch(dgs_ctx* c, const Workspace& ws, const SelArgs& a, uint32_t q, cudaStream_t st) {
  TimedLaunch tl(c, st, SCAN ? DGS_KERNEL_STREAM_PULL : DGS_KERNEL_CATCH_UP);
  const uint32_t warps = fold_warps(c->cfg.num_workers, c->cfg.n, c->idle_gpu, has_gpu(c));
  k_fold<SCAN><<<c->fold_grid, warps * 32, fold_dyn_bytes(warps, c->fold_ahead, ws.part_cap), st>>>(ws, a, c->log, fold_range(c, q));
  DGS_CUDA(c, cudaGetLastError());
  c->launches += 1;
  c->applied[q] = c->log_head;
  return DGS_OK;
}
// Both, as a task of its own.
int catch_up_now(dgs_ctx* c, uint32_t q, int stream) {
  if (c->applied[q] == c->log_head) return DGS_OK;
  Task t;
  t.stream = stream;
  catch_up_deps(c, q, &t);
  int rc = task_begin(c, t);
  if (rc != DGS_OK) return rc;
  SelArgs a;
  std::memset(&a, 0, sizeof(a));
  a.D = c->D_buf(q);
  a.blk_max = c->blk_max(q);
  rc = fold_launch<false>(c, c->ws[0], a, q, c->st[stream]);   // (tables only: a fold without a scan writes no scratch)
  if (rc != DGS_OK) return rc;
  return task_end(c, t);
}

// Row of carried bounds for a selection of this kind at this age: the most recent row made at
// an age <= `age`, but preferably not one written by the selections that the other streams of
// this kind are still working on (waiting for those would chain the streams together; the row
// before them was written on this selection's own stream).  -1 if there is none.
int pick_row(const dgs_ctx* c, int kind, uint64_t age) {
  int best = -1, best_old = -1;
  const uint64_t in_flight = (uint64_t)c->streams - 1;
  const uint64_t newest = c->kind_seq[kind];
  for (uint32_t q = 0; q < c->cfg.num_workers; ++q) {
    if (!c->row_valid[kind][q] || c->row_age[kind][q] > age) continue;
    const uint64_t t = c->row_time[kind][q];
    if (best < 0 || t < c->row_time[kind][best]) best = (int)q;   // else the oldest: the likeliest to be complete
    if (t + in_flight <= newest && (best_old < 0 || t > c->row_time[kind][best_old])) best_old = (int)q;
  }
  return best_old >= 0 ? best_old : best;
}

inline int packet_format_of(const dgs_ctx* c) {
  return (c->cfg.flags & DGS_PACKET_BF16) ? 1 : (c->cfg.flags & DGS_PACKET_FP16) ? 2 : 0;
}

template <int MODE>
const void* finalize_kernel(const dgs_ctx* c, bool big) {
  if (c->cfg.num_segments > 1) return big ? (const void*)k_finalize<MODE, true, true> : (const void*)k_finalize<MODE, true, false>;
  return big ? (const void*)k_finalize<MODE, false, true> : (const void*)k_finalize<MODE, false, false>;
}

uint32_t one_bytes(const dgs_ctx* c, int mode) {
  return one_dyn_bytes(mode, c->cfg.num_segments, c->fold_ahead, c->ws[0].part_cap);
}

// CTAs of finalize beside other kernels, of the `want` that keep the candidates in registers.  What its CTAs hold is taken from the
// passes, which have the bytes to move, and with many events side by side a selection that takes longer only waits for its turn
// later: an eighth, but not fewer than 48, and not fewer than 96 with four to seven.  Where an event waits for the one before it,
// all.  us, all (one per SM at most) / 96 / 48, 62 layers of 11.7 M: 32 arrivals in turn of 1 worker 6090 / - / 9724, 2: 2637 / - / 2940,
// 4: 2447 / 2346 / 2343, 6: 2485 / 2355 / 2330, 8: 2524 / - / 2286, 32: 3045 / - / 2786; rounds of 4: 356 / 365 / 407, 6: 510 / 494 / 525,
// 8: 680 / - / 649; workers drawn at random, rounds of 8: 1184 / 1253 / 1668, 32: 4970 / 4955 / 5535.  60 layers of 25 M, 1 %, rounds of 4:
// 604 / 618 / 683, 6: 913 / 899 / 929, 8: 1210 / - / 1217, 16: 2500 / - / 2380; at random, 0.3 %, 8: 1520 / 1686 / 2071, 32: 6395 / 6540 / 7455.
// One layer of 25 M, 0.1 %, at random, 8: 1190 / 1202 / 1381, 32: 4786 / 4831 / 5395.
constexpr uint64_t finalize_beside(uint32_t abreast, uint64_t want) {
  const uint64_t few = abreast >= 8 ? 48 : 96, less = want / 8 > few ? want / 8 : few;
  return abreast < 4 || want < less ? want : less;
}
static_assert(finalize_beside(1, 204) == 204, "a chain of events");
static_assert(finalize_beside(4, 204) == 96 && finalize_beside(4, 60) == 60, "");
static_assert(finalize_beside(8, 204) == 48 && finalize_beside(8, 800) == 100 && finalize_beside(8, 33) == 33, "");

template <int MODE>
int launch_select(dgs_ctx* c, const SelArgs& a_in, uint32_t worker, uint64_t age, int stream_id, Task& task) {
  constexpr int KIND = MODE == kPull ? 1 : 0;
  const ResIds R{c->cfg.num_workers};
  cudaStream_t st = c->st[stream_id];
  Workspace& ws = c->ws[stream_id];
  SelArgs a = a_in;
  a.speculate = (c->cfg.flags & DGS_NO_SPECULATION) ? 0 : 1;
  int row = a.speculate ? pick_row(c, KIND, age) : -1;
  // A worker that comes straight back (no other worker's packet since its last pull) selects from what that pull
  // left plus its own packet, and no other pull's bound says anything about that: 44 % of such guesses admitted
  // fewer than k candidates (four workers drawn at random), each then starting over inside finalize.  The
  // histogram route costs less than that on average.  (With one worker every pull is like the one before it.)
  if (KIND == 1 && age < 2 && c->cfg.num_workers > 1) row = -1;
  const bool single_pass = row >= 0, alone = has_gpu(c);
  const int next_copy = c->row_copy[KIND][worker] ^ 1;
  a.L_next = c->L_next(KIND, next_copy, worker);
  a.slack = c->at<uint32_t>(c->lay.slack) + (uint64_t)KIND * c->cfg.num_segments;
  a.force_two_pass = single_pass ? 0 : 1;
  // CTAs of finalize: as many as keep the candidates in the threads' registers, but not fewer than 32, since every step of a
  // warp is a chain, and no more than two per SM.  There are 2 to 4 times as many candidates as entries; where the kernel has
  // the GPU to itself it is sized for 3 (one arrival at a time on 25.6 M elements: 128.5 us sized for 1.75, 123 for 3; on 11.7 M
  // in 62 layers its two finalize kernels take 28 and 31 us instead of 34 and 36), and where it opens a round whose events wait for one
  // another (workers drawn at random, rounds of 4, us, without / with: 17 M elements 646 / 609, 60 layers of 25 M 1034 / 969; of 16: 2005 /
  // 1961, 3198 / 3116).  A warp per two layers for the advice.
  const uint32_t advisers = std::min<uint32_t>(32u, (c->cfg.num_segments + 2 * kWarps - 1) / (2 * kWarps));
  const uint64_t keep = finalize_keep(c->cfg.num_segments > 1);
  // Layers that are small enough to be candidates as a whole (see next_bound) often are: 60 layers of 2^20 elements, alone, 18.3
  // and 20.8 us without them, 16.5 and 18.2 with.
  const bool opens_chain = !alone && c->idle_gpu && c->arrivals.chained();
  const uint64_t cands = alone || opens_chain ? std::max<uint64_t>(3ull * a.pkt_count + 64ull * c->cfg.num_segments, c->whole_layers)
                                  : (uint64_t)a.pkt_count + a.pkt_count / 4 * 3 + 64ull * c->cfg.num_segments;
  uint64_t want = std::max<uint64_t>(kFinalizeMin, (cands + kThreads * keep - 1) / (kThreads * keep));
  if (!alone) want = finalize_beside(c->streams > 1 ? c->arrivals.abreast() : 1, want);
  // Two CTAs an SM where it has the GPU to itself, as where it opens a chain of events of a single worker.  (Selections from 2^26
  // elements, 10 %, by one worker, two between joins: the first on one CTA an SM 733 us, on two 530; but rounds of 4 at random,
  // 8.4 M elements, 2 %: 506 / 560.)
  const bool wide = alone || (opens_chain && c->cfg.num_workers == 1);
  const uint64_t most = (uint64_t)(std::min(c->finalize_max[MODE], wide ? 2 * c->sms : c->sms) - (int)advisers);
  const int fin_grid = (int)std::min(most, want);
  // More candidates than the registers of all CTAs hold: k_finalize<.., BIG>, but beside other kernels only for one layer
  // and fifty times as many (runs of 32 events on 8.4 M elements, us an event without / with: one layer, 10 %, 20 times as
  // many: 153 / 156; 50 %, 97 times: 823 / 733; 60 layers, 50 %: 750 / 818), or where it opens a chain of events (rounds of 2 and 4 at
  // random, 8.4 M elements, 10 %: 1027 / 930, 1360 / 1281).
  const uint64_t held = (wide ? (uint64_t)fin_grid : most) * kThreads * keep;
  const bool big = wide ? cands > held : c->cfg.num_segments == 1 && cands > (opens_chain ? held : 50 * held);
  a.workers = (uint32_t)fin_grid;
  a.advisers = advisers;
  a.fold_grid = MODE == kPull ? (uint32_t)c->fold_grid : 0u;   // one CTA more plans the next pull's pass
  // Short vectors: pass and finalize in one kernel.  Beside other events the host is what such vectors wait for, 3 us a launch
  // (see one_max_beside; 2^21 elements: 20 us an event with two kernels a selection, 27 with one).  Alone it is the GPU, and only a
  // pull of one layer gains: its pass takes little longer with half of the CTAs (2^20 elements: pull 22.3 / 19.6 us, push 19.6 /
  // 20.2; in 60 layers 40 / 42 and 31 / 34; select from 1.5 M elements, 0.1 to 3 %: 34-41 / 32-37, 5 %: 46 / 46).  While launches are
  // timed each kernel stays on its own.
  const uint32_t others = advisers + (MODE == kPull ? 1u : 0u);
  uint32_t one_grid = std::min<uint32_t>(alone ? kOneMaxGrid : kOneGridBeside, (c->lay.num_blocks + kWarps - 1) / kWarps);
  one_grid = std::min<uint32_t>(std::max<uint32_t>(one_grid, (uint32_t)kFinalizeMin + others), (uint32_t)c->one_max[MODE]);
  const uint64_t one_max_n = !alone ? one_max_beside(c->cfg.num_segments) : MODE == kPull && c->cfg.num_segments == 1 ? kOneMaxN : 0;
  const bool one = c->cfg.n <= one_max_n && !big && !c->timing &&
                   one_grid > others && (c->lay.num_blocks + one_grid - 1) / one_grid + kFoldSlack <= ws.part_cap;
  if (one) {
    a.workers = std::min<uint32_t>(a.workers, one_grid - others);
    if (MODE == kPull) a.fold_grid = one_grid;
  }
  a.pair = c->pair[stream_id] ^= 1u;
  a.packet_format = packet_format_of(c);
  if (c->cfg.flags & DGS_TEST_STALLED_BARRIER) {
    a.phantom_workers = 1;
    a.spin_limit = 4096;
  }
  a.seq = (uint32_t)c->kind_seq[KIND];
  a.L_in = single_pass ? c->L_next(KIND, c->row_copy[KIND][row], (uint32_t)row) : ws.L_safe;
  task.stream = stream_id;
  if (single_pass) task.reads.push_back(R.ROW(KIND, c->row_copy[KIND][row], (uint32_t)row));
  if (a.speculate) task.writes.push_back(R.ROW(KIND, next_copy, worker));
  task.writes.push_back(R.SCR(stream_id));
  int rc = task_begin(c, task);
  if (rc != DGS_OK) return rc;
  if (!single_pass) {
    // nothing to go by: histogram of the whole input first, its bounds cannot fail
    if (MODE == kPull && c->applied[worker] < c->log_head) {
      rc = fold_launch<false>(c, ws, a, worker, st);
      if (rc != DGS_OK) return rc;
    }
    TimedLaunch t(c, st, MODE == kPull ? DGS_KERNEL_TWO_PASS_PULL : DGS_KERNEL_TWO_PASS_PUSH);
    k_hist_all<MODE><<<c->hist_grid[MODE], kThreads, 0, st>>>(ws, a);
    DGS_CUDA(c, cudaGetLastError());
    const int pick_grid = (int)std::min<uint32_t>(c->cfg.num_segments, 1024u);
    k_pick_lower<MODE><<<pick_grid, kThreads, 0, st>>>(ws);
    DGS_CUDA(c, cudaGetLastError());
    c->launches += 2;
  }
  if (one) {
    FoldRange f = MODE == kPull ? fold_range(c, worker) : FoldRange{};
    void* args[] = {(void*)&ws, (void*)&a, (void*)&c->log, (void*)&f};
    DGS_CUDA(c, cudaLaunchCooperativeKernel(one_kernel(MODE, c->cfg.num_segments > 1), dim3(one_grid), dim3(kThreads), args,
                                            one_bytes(c, MODE), st));
    c->launches += 1;
    if (MODE == kPull) c->applied[worker] = c->log_head;
  } else if constexpr (MODE == kPull) {
    rc = fold_launch<true>(c, ws, a, worker, st);
    if (rc != DGS_OK) return rc;
  } else {
    TimedLaunch t(c, st, DGS_KERNEL_STREAM_PUSH);
    k_stream<MODE><<<c->stream_grid[MODE], kThreads, PushRing::kBytes, st>>>(ws, a);
    DGS_CUDA(c, cudaGetLastError());
    c->launches += 1;
  }
  if (!one) {
    // cooperative launch: the CTAs synchronise among themselves, so all must be resident
    TimedLaunch t(c, st, MODE == kPull ? DGS_KERNEL_FINALIZE_PULL : DGS_KERNEL_FINALIZE_PUSH);
    void* args[] = {(void*)&ws, (void*)&a};
    DGS_CUDA(c, cudaLaunchCooperativeKernel(finalize_kernel<MODE>(c, big), dim3(fin_grid + advisers + (MODE == kPull ? 1 : 0)),
                                            dim3(kThreads), args, finalize_dyn_bytes(c->cfg.num_segments), st));
    c->launches += 1;
  }
  rc = task_end(c, task);
  if (rc != DGS_OK) return rc;
  c->kind_seq[KIND] += 1;
  if (a.speculate) {
    c->row_valid[KIND][worker] = 1;
    c->row_copy[KIND][worker] = (uint8_t)next_copy;
    c->row_time[KIND][worker] = c->kind_seq[KIND];
    c->row_age[KIND][worker] = age;
  }
  return DGS_OK;
}

// Grid of k_fold and the room for its tables and buffers.
constexpr int kFoldMaxDyn = 208 * 1024;   // beside its static shared memory
int fold_setup(dgs_ctx* c, int sms) {
  c->fold_grid = (int)std::min<uint32_t>((c->lay.num_blocks + 7) / 8, (uint32_t)std::min(2 * sms, kMaxFoldGrid));
  // A quarter more than the mean number of entries of a block, for a worker that has missed a packet per worker.
  const uint64_t mean = std::min<uint64_t>(c->cfg.num_workers, 32) * c->lay.K[0] * kWarpTile / c->cfg.n;
  c->fold_ahead = (uint32_t)std::min<uint64_t>(192, std::max<uint64_t>(64, align_up(mean + mean / 4, 64)));
  // Eight even shares: where most of the vector is cold, the shares of the CTAs that have only cold blocks grow
  // (a share never gets longer than an even one without a plan).
  const uint32_t even = (c->lay.num_blocks + c->fold_grid - 1) / c->fold_grid + kFoldSlack;
  const uint32_t cap = (uint32_t)align_up(std::max<uint32_t>(even, std::min<uint32_t>(32768u, 8 * even)), 128);
  for (int k = 0; k < kSets; ++k) c->ws[k].part_cap = cap;
  DGS_CUDA(c, cudaFuncSetAttribute(k_fold<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldMaxDyn));
  DGS_CUDA(c, cudaFuncSetAttribute(k_fold<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldMaxDyn));
  if (fold_dyn_bytes(kFoldWarps, c->fold_ahead, cap) > (uint32_t)kFoldMaxDyn) return DGS_EINVAL;   // (n < 2^32 keeps an even share well below)
  return DGS_OK;
}

template <int MODE>
int occupancy_grids(dgs_ctx* c, int sms) {
  int occ = 0;
  if constexpr (MODE != kPull) {
    DGS_CUDA(c, cudaFuncSetAttribute(k_stream<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, PushRing::kBytes));
    DGS_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_stream<MODE>, kThreads, PushRing::kBytes));
    if (occ < 1) occ = 1;
    c->stream_grid[MODE] = std::min(sms * occ, kMaxGrid);
  }
  DGS_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_hist_all<MODE>, kThreads, 0));
  if (occ < 1) occ = 1;
  c->hist_grid[MODE] = std::min(sms * occ, kMaxGrid);
  c->finalize_max[MODE] = kMaxWorkers;
  for (const bool big : {false, true}) {
    DGS_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, finalize_kernel<MODE>(c, big), kThreads,
                                                              finalize_dyn_bytes(c->cfg.num_segments)));
    if (occ < 1) {
      c->last_cuda = (int)cudaErrorCooperativeLaunchTooLarge;
      c->broken = true;
      return DGS_ECUDA;
    }
    c->finalize_max[MODE] = std::min(c->finalize_max[MODE], sms * occ);
  }
  if (MODE == kPull) c->finalize_max[MODE] -= 1;   // the CTA that plans the next pass
  c->one_max[MODE] = 0;
  if (c->cfg.n <= one_max_beside(c->cfg.num_segments) && one_bytes(c, MODE) <= (uint32_t)kFoldMaxDyn) {
    const void* const f = one_kernel(MODE, c->cfg.num_segments > 1);
    DGS_CUDA(c, cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldMaxDyn));
    DGS_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, kThreads, one_bytes(c, MODE)));
    c->one_max[MODE] = std::min(kOneMaxGrid, sms * occ);
  }
  return DGS_OK;
}

void destroy_ctx(dgs_ctx* c) {
  for (int i = 0; i < kStreams; ++i) {
    if (c->st[i]) cudaStreamDestroy(c->st[i]);
    if (c->ev_tail[i]) cudaEventDestroy(c->ev_tail[i]);
  }
  if (c->ev_in) cudaEventDestroy(c->ev_in);
  for (int i = 0; i <= kCaller; ++i)
    for (cudaEvent_t e : c->ev_ring[i]) cudaEventDestroy(e);
  for (cudaEvent_t e : c->ev_pool) cudaEventDestroy(e);
  c->magic = 0;
  delete c;
}

}  // namespace

extern "C" {

const char* dgs_error_string(int err) {
  switch (err) {
    case DGS_OK: return "ok";
    case DGS_EINVAL: return "invalid argument";
    case DGS_ENOMEM: return "arena too small";
    case DGS_ECUDA: return "CUDA runtime error";
    case DGS_ETIMEOUT: return "bounded device wait expired";
    case DGS_ESTATE: return "context freed or unusable";
    case DGS_ELIMIT: return "size beyond the fixed capacity of the static scratch";
  }
  return "unknown error";
}

int dgs_arena_bytes(const dgs_config* cfg, uint64_t* out_bytes) {
  if (!out_bytes) return DGS_EINVAL;
  const int rc = check_config(cfg);
  if (rc != DGS_OK) return rc;
  Layout L;
  make_layout(cfg, &L);
  *out_bytes = L.total;
  return DGS_OK;
}

int dgs_init(const dgs_config* cfg, dgs_ctx** out) {
  if (!out) return DGS_EINVAL;
  *out = nullptr;
  int rc = check_config(cfg);
  if (rc != DGS_OK) return rc;
  if (!cfg->theta0 || !cfg->arena) return DGS_EINVAL;
  if ((reinterpret_cast<uintptr_t>(cfg->arena) % kAlign) != 0) return DGS_EINVAL;
  dgs_ctx* c = new (std::nothrow) dgs_ctx();
  if (!c) return DGS_ENOMEM;
  c->magic = kMagic;
  c->cfg = *cfg;
  c->segments.assign(cfg->segments, cfg->segments + cfg->num_segments);
  c->cfg.segments = c->segments.data();
  make_layout(&c->cfg, &c->lay);
  c->whole_layers = 0;
  for (const dgs_segment& g : c->segments)
    if (cfg->num_segments > 1 && g.len <= std::max<uint64_t>(8192, cfg->n / 1024)) c->whole_layers += g.len;
  for (int i = 0; i < kStreams; ++i) {
    c->st[i] = nullptr;
    c->ev_tail[i] = nullptr;
    c->forked[i] = c->dirty[i] = false;
  }
  c->streams = streams_for(cfg);
  c->next_stream = 0;
  c->idle = true;
  c->worker_stream.assign(cfg->num_workers, -1);
  for (int i = 0; i < kPushSlots; ++i) c->slot_stream[i] = 0;
  c->ev_in = nullptr;
  c->task_seq = 0;
  for (int i = 0; i <= kCaller; ++i) {
    c->ev_next[i] = 0;
    for (int j = 0; j <= kCaller; ++j) c->waited_seq[i][j] = 0;
  }
  c->forked[kCaller] = c->dirty[kCaller] = false;
  c->pull_count = c->event_count = c->var_count = 0;
  c->log_head = 0;
  c->applied.assign(cfg->num_workers, 0);
  c->kind_seq[0] = c->kind_seq[1] = 0;
  c->res.assign(ResIds{cfg->num_workers}.count(), dgs_ctx::Res());
  if (c->lay.total > cfg->arena_bytes) {
    delete c;
    return DGS_ENOMEM;
  }
  c->base = static_cast<char*>(cfg->arena);
  c->user = c->st[kCaller] = static_cast<cudaStream_t>(cfg->stream);
  c->push_count = 0;
  for (uint32_t& p : c->pair) p = 0;
  c->inv_m = 1.0f / cfg->momentum;  // one IEEE division; the kernels multiply by this constant
  c->timestamp = 0;
  c->launches = 0;
  c->last_cuda = 0;
  c->broken = false;
  c->idle_gpu = true;
  c->arrivals = Arrivals(cfg->num_workers);
  c->timing = false;
  for (int i = 0; i < DGS_NUM_KERNELS; ++i) {
    c->time_ms[i] = 0.0;
    c->time_count[i] = 0;
  }
  for (int k = 0; k < 2; ++k) {
    c->row_valid[k].assign(cfg->num_workers, 0);
    c->row_copy[k].assign(cfg->num_workers, 0);
    c->row_time[k].assign(cfg->num_workers, 0);
    c->row_age[k].assign(cfg->num_workers, 0);
  }
  c->pushes.assign(cfg->num_workers, 0);
  c->prev.assign(cfg->num_workers, -1);

  auto fail = [&](int code) {
    destroy_ctx(c);
    return code;
  };
#define INIT_CUDA(call)                         \
  do {                                          \
    cudaError_t e_ = (call);                    \
    if (e_ != cudaSuccess) return fail(DGS_ECUDA); \
  } while (0)

  int dev = 0, sms = 0, coop = 0;
  INIT_CUDA(cudaGetDevice(&dev));
  INIT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  INIT_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return fail(DGS_ECUDA);
  c->sms = sms;
  if (fold_setup(c, sms) != DGS_OK || occupancy_grids<kPushSam>(c, sms) != DGS_OK || occupancy_grids<kPushResidual>(c, sms) != DGS_OK ||
      occupancy_grids<kPull>(c, sms) != DGS_OK)
    return fail(DGS_ECUDA);
  INIT_CUDA(cudaEventCreateWithFlags(&c->ev_in, cudaEventDisableTiming));
  if (stream_ready(c, 0) != DGS_OK) return fail(DGS_ECUDA);

  const Layout& L = c->lay;
  const uint64_t N = cfg->num_workers, vec = L.n_pad * 4;
  std::vector<Tile> tiles;
  std::vector<SegDesc> segs;
  tiles.reserve(L.num_tiles);
  build_tiles(&c->cfg, &tiles, &segs);
  if (tiles.size() != L.num_tiles) return fail(DGS_EINVAL);
  cudaStream_t st = c->user;
  // state: u = 0, D = 0 (initialisation lines of Algorithm 3 and Algorithm 2), theta = theta_0
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.u), 0, vec * (N + c->streams), st));
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.D), 0, vec * N, st));
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.theta), 0, vec, st));
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.theta), cfg->theta0, cfg->n * 4, cudaMemcpyDeviceToDevice, st));
  if (cfg->flags & DGS_KEEP_LOCAL_MODEL) {
    INIT_CUDA(cudaMemsetAsync(c->at<char>(L.theta_local), 0, vec * N, st));
    for (uint32_t q = 0; q < N; ++q)
      INIT_CUDA(cudaMemcpyAsync(c->theta_local_buf(q), cfg->theta0, cfg->n * 4, cudaMemcpyDeviceToDevice, st));
  }
  // scratch that kernels expect to find cleared, and the static tables
  for (int k = 0; k < c->streams; ++k) {
    const ScratchLayout& sc = L.sc[k];
    INIT_CUDA(cudaMemsetAsync(c->at<char>(sc.zero_begin), 0, sc.zero_end - sc.zero_begin, st));
    INIT_CUDA(cudaMemsetAsync(c->at<char>(sc.part_cands), 0, (uint64_t)kMaxParts * 4, st));
    INIT_CUDA(cudaMemsetAsync(c->at<char>(sc.part_slot0), 0, (uint64_t)kMaxParts * 4, st));
    INIT_CUDA(cudaMemsetAsync(c->at<char>(sc.plan), 0, (uint64_t)(kMaxFoldGrid + 1) * 4, st));   // no plan yet
  }
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.log_sum), 0, (uint64_t)L.sum_stride * 4, st));   // no packet filed
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.blk_max), 0, N * L.blk_stride * 4, st));   // D = 0
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.L_next), 0xFF, 4 * N * cfg->num_segments * 4, st));
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.slack), 0, 2ull * cfg->num_segments * 4, st));
  INIT_CUDA(cudaMemsetAsync(c->at<char>(L.status), 0, L.total - L.status, st));
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.tiles), tiles.data(), tiles.size() * sizeof(Tile), cudaMemcpyHostToDevice, st));
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.segs), segs.data(), segs.size() * sizeof(SegDesc), cudaMemcpyHostToDevice, st));
  std::vector<uint32_t> seg_off(cfg->num_segments + 1);
  for (uint32_t q = 0; q < cfg->num_segments; ++q) {
    seg_off[q] = (uint32_t)cfg->segments[q].offset;
  }
  seg_off[cfg->num_segments] = (uint32_t)cfg->n;  // n < 2^32
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.seg_off), seg_off.data(), seg_off.size() * 4, cudaMemcpyHostToDevice, st));
  std::vector<uint32_t> blk_seg(L.num_blocks);
  for (uint32_t b = 0, q = 0; b < L.num_blocks; ++b) {
    while (segs.size() > q + 1 && (uint64_t)seg_off[q + 1] <= (uint64_t)b * kWarpTile) ++q;
    blk_seg[b] = q;
  }
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.blk_seg), blk_seg.data(), blk_seg.size() * 4, cudaMemcpyHostToDevice, st));
  std::vector<uint32_t> ones(cfg->num_segments, 1u);   // the bound that admits every nonzero value
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.L_one), ones.data(), ones.size() * 4, cudaMemcpyHostToDevice, st));
  std::vector<float*> slots(N + c->streams);
  for (uint32_t q = 0; q < N + c->streams; ++q) slots[q] = c->u_buf(q);
  INIT_CUDA(cudaMemcpyAsync(c->at<char>(L.u_slots), slots.data(), slots.size() * sizeof(float*), cudaMemcpyHostToDevice, st));
  // the host vectors above go out of scope, and the library's own streams start from a ready arena
  INIT_CUDA(cudaStreamSynchronize(st));
#undef INIT_CUDA

  for (int k = 0; k < c->streams; ++k) {
    Workspace& w = c->ws[k];
    const ScratchLayout& sc = L.sc[k];
    w.tiles = c->at<Tile>(L.tiles);
    w.segs = c->at<SegDesc>(L.segs);
    w.num_tiles = L.num_tiles;
    w.num_segs = cfg->num_segments;
    w.seg_off = c->at<uint32_t>(L.seg_off);
    w.cand_idx = c->at<uint32_t>(sc.cand_idx);
    w.cand_val = c->at<float>(sc.cand_val);
    w.part_cands = c->at<uint32_t>(sc.part_cands);
    w.part_slot0 = c->at<uint32_t>(sc.part_slot0);
    w.plan = c->at<uint32_t>(sc.plan);
    w.cta_cost = c->at<uint32_t>(sc.cta_cost);
    w.n = (uint32_t)cfg->n;
    w.n_pad = (uint32_t)std::min<uint64_t>(L.n_pad, 0xFFFFFFFFull);
    w.num_blocks = L.num_blocks;
    w.blk_seg = c->at<uint32_t>(L.blk_seg);
    w.cta_tot = c->at<uint2>(sc.cta_tot);
    w.cta_eq = c->at<uint32_t>(sc.cta_eq);
    w.tab = c->at<LayerPick>(sc.tab);
    w.list = c->at<uint2>(sc.list);
    w.list_cnt = c->at<uint32_t>(sc.list_cnt);
    w.hist1 = c->at<uint32_t>(sc.hist1);
    w.sel = c->at<SegSel>(sc.sel);
    w.L_safe = c->at<uint32_t>(sc.L_safe);
    w.L_wide = c->at<uint32_t>(sc.L_wide);
    w.sync = c->at<uint32_t>(sc.sync);
    w.status = c->at<int>(L.status);
    w.stats = c->at<unsigned long long>(L.stats);
  }
  c->log.ent = c->at<uint2>(L.log_ent);
  c->log.stride = L.log_stride;
  c->log.ring = L.log_ring;
  c->log.pos = c->at<uint32_t>(L.log_pos);
  c->log.pos_rows = L.pos_rows;
  c->log.sum = c->at<uint32_t>(L.log_sum);
  c->log.sum_stride = L.sum_stride;
  *out = c;
  return DGS_OK;
}

namespace {

int push_impl(dgs_ctx* c, uint32_t worker, const float* grad, dgs_packet* out, int stream_id, bool grad_is_stage) {
  const Layout& L = c->lay;
  const ResIds R{c->cfg.num_workers};
  const int slot = (int)(c->push_count % kPushSlots);
  int rc = fork_from_user(c, stream_id);  // the gradient may have been produced on the caller's stream
  if (rc != DGS_OK) return rc;
  SelArgs a;
  std::memset(&a, 0, sizeof(a));
  a.grad = grad;
  a.u_cur_slot = c->u_slot(worker);
  a.u_spare_slot = c->u_slot(c->cfg.num_workers + stream_id);
  a.pkt_idx = c->at<uint32_t>(L.pkt_idx[slot]);
  a.pkt_val = c->at<float>(L.pkt_val[slot]);
  a.pkt_count = (uint32_t)L.K[0];
  a.m = c->cfg.momentum;
  a.lr = c->cfg.lr;
  a.inv_m = c->inv_m;
  c->arrivals.arrived(worker);
  Task task;
  task.writes = {R.U(worker), R.SPARE(stream_id), R.PKT(slot)};
  if (grad_is_stage) task.reads.push_back(R.STAGE());
  const uint64_t age = c->pushes[worker];
  rc = (c->cfg.flags & DGS_RESIDUAL_MODE)
           ? launch_select<kPushResidual>(c, a, worker, age, stream_id, task)
           : launch_select<kPushSam>(c, a, worker, age, stream_id, task);
  if (rc != DGS_OK) return rc;
  c->pushes[worker] += 1;
  c->push_count += 1;
  c->worker_stream[worker] = stream_id;
  c->slot_stream[slot] = stream_id;
  if (out) {
    out->idx = a.pkt_idx;
    out->val = a.pkt_val;
    out->count = a.pkt_count;
  }
  return DGS_OK;
}

int apply_impl(dgs_ctx* c, uint32_t worker, const dgs_packet* pkt) {
  (void)worker;
  const ResIds R{c->cfg.num_workers};
  const uint32_t N = c->cfg.num_workers;
  // whose packet is it?  one of the push slots: the tracker knows its writer; anything else: the caller's stream
  int slot = -1;
  for (int i = 0; i < kPushSlots; ++i)
    if (pkt->idx == c->at<uint32_t>(c->lay.pkt_idx[i])) slot = i;
  const bool own = slot >= 0 && pkt->val == c->at<float>(c->lay.pkt_val[slot]) && pkt->count == c->lay.K[0];
  const int stream_id = own ? c->slot_stream[slot] : peek_stream(c);   // after its push; else where a pull comes next
  const uint32_t gx = (pkt->count + kThreads - 1) / kThreads;
  int rc = DGS_OK;
  // theta and the D_q that are caught up may be what the caller's stream is still reading (nothing to do inside an event)
  if (pkt->count > 0) rc = fork_from_user(c, stream_id);
  if (rc != DGS_OK) return rc;
  if (pkt->count == 0) {
    // nothing to subtract
  } else if (pkt->count <= c->log.stride) {
    // theta now, the D_q lazily.  Any packet that fits a slot of the log is filed, a caller's own as well (16 of them
    // and 16 pulls on 25.6 M elements: 1136 us with a scatter into theta and all 16 D_q each, which also kept every
    // event from overlapping the next, 392 us filed).
    // Its slot of the log still holds the packet filed `ring` applies ago; whoever has not folded that
    // one in yet does so first.
    const uint32_t lslot = (uint32_t)(c->log_head % c->log.ring);
    if (c->log_head >= c->log.ring) {
      const uint64_t oldest = c->log_head - c->log.ring;
      for (uint32_t q = 0; q < N; ++q)
        if (c->applied[q] <= oldest) {
          rc = catch_up_now(c, q, stream_id);
          if (rc != DGS_OK) return rc;
        }
    }
    Task t;
    t.stream = stream_id;
    if (slot >= 0) t.reads.push_back(R.PKT(slot));
    t.writes = {R.THETA(), R.LOG(lslot)};
    rc = task_begin(c, t);
    if (rc != DGS_OK) return rc;
    {
      TimedLaunch tl(c, c->st[stream_id], DGS_KERNEL_SCATTER);
      const uint32_t pos_ctas = (c->log.pos_rows + kThreads - 1) / kThreads;
      k_apply_log<<<gx + pos_ctas, kThreads, 0, c->st[stream_id]>>>(pkt->idx, pkt->val, pkt->count, c->at<float>(c->lay.theta),
                                                                    c->cfg.n, c->ws[0].status, c->log, lslot,
                                                                    (uint32_t)(c->log_head % (c->log.ring + 1)), gx);
      DGS_CUDA(c, cudaGetLastError());
      c->launches += 1;
    }
    rc = task_end(c, t);
    if (rc != DGS_OK) return rc;
    c->log_head += 1;
  } else {
    // A packet too long for the log: bring every D_q up to date, then subtract from theta and all of them at once.
    for (uint32_t q = 0; q < N; ++q) {
      rc = catch_up_now(c, q, stream_id);
      if (rc != DGS_OK) return rc;
    }
    Task t;
    t.stream = stream_id;
    if (slot >= 0) t.reads.push_back(R.PKT(slot));
    t.writes.push_back(R.THETA());
    for (uint32_t q = 0; q < N; ++q) t.writes.push_back(R.D(q));
    rc = task_begin(c, t);
    if (rc != DGS_OK) return rc;
    {
      TimedLaunch tl(c, c->st[stream_id], DGS_KERNEL_SCATTER);
      k_scatter_sub<<<dim3(gx, N + 1), kThreads, 0, c->st[stream_id]>>>(
          pkt->idx, pkt->val, pkt->count, c->at<float>(c->lay.theta), c->at<float>(c->lay.D), c->lay.n_pad, N,
          c->cfg.n, c->ws[0].status, c->blk_max(0), c->lay.blk_stride);
      DGS_CUDA(c, cudaGetLastError());
      c->launches += 1;
    }
    rc = task_end(c, t);
    if (rc != DGS_OK) return rc;
  }
  c->timestamp += 1;  // t counts updates made to the server parameters
  return DGS_OK;
}

int pull_impl(dgs_ctx* c, uint32_t worker, dgs_packet* out) {
  const Layout& L = c->lay;
  const ResIds R{c->cfg.num_workers};
  const int slot = kPushSlots + (int)(c->pull_count % kPullSlots);
  if (c->worker_stream[worker] < 0) c->arrivals.arrived(worker);
  const int stream_id = c->worker_stream[worker] >= 0 ? c->worker_stream[worker] : take_stream(c);
  int rc = fork_from_user(c, stream_id);  // the caller may still be reading an older pull packet on its stream
  if (rc != DGS_OK) return rc;
  SelArgs a;
  std::memset(&a, 0, sizeof(a));
  a.D = c->D_buf(worker);
  a.blk_max = c->blk_max(worker);
  a.theta_local = (c->cfg.flags & DGS_KEEP_LOCAL_MODEL) ? c->theta_local_buf(worker) : nullptr;
  a.pkt_idx = c->at<uint32_t>(L.pkt_idx[slot]);
  a.pkt_val = c->at<float>(L.pkt_val[slot]);
  a.pkt_count = (uint32_t)L.K[1];
  a.m = c->cfg.momentum;
  a.lr = c->cfg.lr;
  a.inv_m = c->inv_m;
  Task task;
  task.writes = {R.PKT(slot)};
  catch_up_deps(c, worker, &task);  // D_worker is brought up to date first, on the same stream
  if (a.theta_local) task.writes.push_back(R.TL(worker));
  // packets that entered D_worker since its previous pull
  const uint64_t age = c->timestamp - (c->prev[worker] < 0 ? 0 : (uint64_t)c->prev[worker]);
  rc = launch_select<kPull>(c, a, worker, age, stream_id, task);
  if (rc != DGS_OK) return rc;
  c->prev[worker] = (int64_t)c->timestamp;
  c->pull_count += 1;
  c->worker_stream[worker] = -1;
  c->idle_gpu = false;
  if (out) {
    out->idx = a.pkt_idx;
    out->val = a.pkt_val;
    out->count = a.pkt_count;
  }
  return DGS_OK;
}

// Pull without secondary compression: catch-up, the pull's stream pass with the bound 1 (every nonzero entry
// becomes a candidate, in index order), then the copy into the packet.  Shares the pulls' streams and scratch sets.
int pull_all_impl(dgs_ctx* c, uint32_t worker, dgs_var_packet* out) {
  const Layout& L = c->lay;
  const ResIds R{c->cfg.num_workers};
  const int vslot = (int)(c->var_count % kVarSlots);
  if (c->worker_stream[worker] < 0) c->arrivals.arrived(worker);
  const int stream_id = c->worker_stream[worker] >= 0 ? c->worker_stream[worker] : take_stream(c);
  int rc = fork_from_user(c, stream_id);  // the caller may still be reading an older packet on its stream
  if (rc != DGS_OK) return rc;
  cudaStream_t st = c->st[stream_id];
  Workspace& ws = c->ws[stream_id];
  SelArgs a;
  std::memset(&a, 0, sizeof(a));
  a.D = c->D_buf(worker);
  a.blk_max = c->blk_max(worker);
  a.theta_local = (c->cfg.flags & DGS_KEEP_LOCAL_MODEL) ? c->theta_local_buf(worker) : nullptr;
  a.L_in = c->at<uint32_t>(L.L_one);
  a.m = c->cfg.momentum;
  a.lr = c->cfg.lr;
  a.inv_m = c->inv_m;
  Task task;
  task.stream = stream_id;
  task.writes = {R.VPKT(vslot), R.SCR(stream_id)};
  catch_up_deps(c, worker, &task);  // D_worker is brought up to date first, on the same stream
  if (a.theta_local) task.writes.push_back(R.TL(worker));
  rc = task_begin(c, task);
  if (rc != DGS_OK) return rc;
  rc = fold_launch<true>(c, ws, a, worker, st);
  if (rc != DGS_OK) return rc;
  uint32_t* vi = c->at<uint32_t>(L.var_idx[vslot]);
  float* vv = c->at<float>(L.var_val[vslot]);
  uint32_t* vc = c->at<uint32_t>(L.var_count[vslot]);
  {
    TimedLaunch t(c, st, DGS_KERNEL_FINALIZE_PULL);
    k_emit_all<<<2 * c->sms, kThreads, 0, st>>>(ws, a.D, a.theta_local, a.blk_max, vi, vv, vc, c->cfg.pull_all_capacity,
                                                packet_format_of(c));
    DGS_CUDA(c, cudaGetLastError());
    c->launches += 1;
  }
  rc = task_end(c, task);
  if (rc != DGS_OK) return rc;
  c->prev[worker] = (int64_t)c->timestamp;
  c->pull_count += 1;
  c->worker_stream[worker] = -1;
  c->var_count += 1;
  c->idle_gpu = false;
  if (out) {
    out->idx = vi;
    out->val = vv;
    out->count = vc;
    out->capacity = c->cfg.pull_all_capacity;
  }
  return DGS_OK;
}

}  // namespace

int dgs_worker_pull_all(dgs_ctx* c, uint32_t worker, dgs_var_packet* out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (worker >= c->cfg.num_workers || c->cfg.pull_all_capacity == 0) return DGS_EINVAL;
  rc = begin_call(c);
  if (rc != DGS_OK) return rc;
  return pull_all_impl(c, worker, out);
}

int dgs_worker_push(dgs_ctx* c, uint32_t worker, const float* grad, dgs_packet* out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (worker >= c->cfg.num_workers || !grad) return DGS_EINVAL;
  if ((reinterpret_cast<uintptr_t>(grad) % 16) != 0) return DGS_EINVAL;
  rc = begin_call(c);
  if (rc != DGS_OK) return rc;
  return push_impl(c, worker, grad, out, take_stream(c), false);
}

int dgs_server_apply(dgs_ctx* c, uint32_t worker, const dgs_packet* pkt) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (worker >= c->cfg.num_workers || !pkt) return DGS_EINVAL;
  if (pkt->count > 0 && (!pkt->idx || !pkt->val)) return DGS_EINVAL;
  rc = begin_call(c);
  if (rc != DGS_OK) return rc;
  return apply_impl(c, worker, pkt);
}

int dgs_worker_pull(dgs_ctx* c, uint32_t worker, dgs_packet* out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (worker >= c->cfg.num_workers) return DGS_EINVAL;
  rc = begin_call(c);
  if (rc != DGS_OK) return rc;
  return pull_impl(c, worker, out);
}

int dgs_event(dgs_ctx* c, uint32_t worker, const float* grad, dgs_packet* push_out, dgs_packet* pull_out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (worker >= c->cfg.num_workers || !grad) return DGS_EINVAL;
  if ((reinterpret_cast<uintptr_t>(grad) % 16) != 0) return DGS_EINVAL;
  rc = begin_call(c);
  if (rc != DGS_OK) return rc;
  dgs_packet p, g;
  rc = push_impl(c, worker, grad, &p, take_stream(c), false);
  if (rc != DGS_OK) return rc;
  rc = apply_impl(c, worker, &p);
  if (rc != DGS_OK) return rc;
  rc = pull_impl(c, worker, &g);
  if (rc != DGS_OK) return rc;
  if (push_out) *push_out = p;
  if (pull_out) *pull_out = g;
  return DGS_OK;
}

int dgs_flush(dgs_ctx* c) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  for (int i = 0; i < kStreams; ++i) {
    if (!c->dirty[i]) continue;              // joined by an earlier call
    DGS_CUDA(c, cudaEventRecord(c->ev_tail[i], c->st[i]));
    DGS_CUDA(c, cudaStreamWaitEvent(c->user, c->ev_tail[i], 0));
    c->dirty[i] = false;
    c->waited_seq[kCaller][i] = c->task_seq;
  }
  joined(c);
  return DGS_OK;
}

int dgs_event_host(dgs_ctx* c, uint32_t worker, const float* grad_host, uint32_t* out_idx, float* out_val) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!(c->cfg.flags & DGS_HOST_IO) || !grad_host || worker >= c->cfg.num_workers) return DGS_EINVAL;
  rc = begin_call(c);
  if (rc != DGS_OK) return rc;
  const ResIds R{c->cfg.num_workers};
  float* stage = c->at<float>(c->lay.grad_stage);
  const int stream_id = take_stream(c);
  {
    // host -> staging buffer, on the stream of the push that will read it
    Task t;
    t.stream = stream_id;
    t.writes.push_back(R.STAGE());
    rc = fork_from_user(c, t.stream);
    if (rc != DGS_OK) return rc;
    rc = task_begin(c, t);
    if (rc != DGS_OK) return rc;
    DGS_CUDA(c, cudaMemcpyAsync(stage, grad_host, c->cfg.n * 4, cudaMemcpyHostToDevice, c->st[t.stream]));
    rc = task_end(c, t);
    if (rc != DGS_OK) return rc;
  }
  dgs_packet p, g;
  rc = push_impl(c, worker, stage, &p, stream_id, true);
  if (rc != DGS_OK) return rc;
  rc = apply_impl(c, worker, &p);
  if (rc != DGS_OK) return rc;
  rc = pull_impl(c, worker, &g);
  if (rc != DGS_OK) return rc;
  cudaStream_t ps = c->st[stream_id];
  if (out_idx) DGS_CUDA(c, cudaMemcpyAsync(out_idx, g.idx, (uint64_t)g.count * 4, cudaMemcpyDeviceToHost, ps));
  if (out_val) DGS_CUDA(c, cudaMemcpyAsync(out_val, g.val, (uint64_t)g.count * 4, cudaMemcpyDeviceToHost, ps));
  // Push, apply and pull follow one another on this stream; what earlier calls have enqueued is complete as well when
  // this one returns.
  return sync_library(c);
}

int dgs_state_ptr(dgs_ctx* c, int which, uint32_t worker, const float** out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!out) return DGS_EINVAL;
  if (which != DGS_THETA && worker >= c->cfg.num_workers) return DGS_EINVAL;
  switch (which) {
    case DGS_THETA: *out = c->at<float>(c->lay.theta); break;
    case DGS_D:
      rc = begin_call(c);
      if (rc == DGS_OK) rc = fork_from_user(c, 0);   // the caller's stream may still be reading the vector as it is
      if (rc == DGS_OK) rc = catch_up_now(c, worker, 0);
      if (rc != DGS_OK) return rc;
      *out = c->D_buf(worker);
      break;
    case DGS_THETA_LOCAL:
      if (!(c->cfg.flags & DGS_KEEP_LOCAL_MODEL)) return DGS_EINVAL;
      *out = c->theta_local_buf(worker);
      break;
    case DGS_U: {
      float* p = nullptr;
      rc = sync_all(c);
      if (rc != DGS_OK) return rc;
      DGS_CUDA(c, cudaMemcpy(&p, c->u_slot(worker), sizeof(p), cudaMemcpyDeviceToHost));
      *out = p;
      return DGS_OK;
    }
    default: return DGS_EINVAL;
  }
  return sync_all(c);
}

int dgs_state_load(dgs_ctx* c, int which, uint32_t worker, const float* src) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!src) return DGS_EINVAL;
  if (which != DGS_THETA && worker >= c->cfg.num_workers) return DGS_EINVAL;
  const ResIds R{c->cfg.num_workers};
  Task t;
  t.stream = kCaller;          // src may be given back to a stream-ordered allocator right after the call
  const float* dst = nullptr;
  switch (which) {
    case DGS_THETA:
      dst = c->at<float>(c->lay.theta);
      t.writes.push_back(R.THETA());
      break;
    case DGS_D:
      dst = c->D_buf(worker);
      t.writes.push_back(R.D(worker));
      break;
    case DGS_THETA_LOCAL:
      if (!(c->cfg.flags & DGS_KEEP_LOCAL_MODEL)) return DGS_EINVAL;
      dst = c->theta_local_buf(worker);
      t.writes.push_back(R.TL(worker));
      break;
    case DGS_U:                // the buffer is known on the device only: waits for all work in flight
      rc = dgs_state_ptr(c, which, worker, &dst);
      if (rc != DGS_OK) return rc;
      t.writes.push_back(R.U(worker));
      break;
    default: return DGS_EINVAL;
  }
  // A vector of the library's own (the model into a worker's copy, say): events in flight may still be writing it.
  const char* const s = reinterpret_cast<const char*>(src);
  if (s >= c->base && s < c->base + c->lay.total) {
    rc = dgs_flush(c);
    if (rc != DGS_OK) return rc;
  }
  rc = task_begin(c, t);
  if (rc != DGS_OK) return rc;
  DGS_CUDA(c, cudaMemcpyAsync(const_cast<float*>(dst), src, c->cfg.n * 4, cudaMemcpyDeviceToDevice, c->user));
  if (which == DGS_D) {
    // Nothing is known about the new contents: every block may hold anything.  Packets filed so far belong to the old.
    DGS_CUDA(c, cudaMemsetAsync(c->blk_max(worker), 0xFF, c->lay.blk_stride * 4, c->user));
    c->applied[worker] = c->log_head;
  }
  return task_end(c, t);
}

int dgs_status(dgs_ctx* c, int* device_status) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!device_status) return DGS_EINVAL;
  rc = sync_all(c);
  if (rc != DGS_OK) return rc;
  DGS_CUDA(c, cudaMemcpy(device_status, c->ws[0].status, 4, cudaMemcpyDeviceToHost));
  return DGS_OK;
}

int dgs_stats(dgs_ctx* c, uint64_t out[4]) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!out) return DGS_EINVAL;
  unsigned long long s[4] = {0, 0, 0, 0};
  rc = sync_all(c);
  if (rc != DGS_OK) return rc;
  DGS_CUDA(c, cudaMemcpy(s, c->ws[0].stats, sizeof(s), cudaMemcpyDeviceToHost));
  out[0] = s[0];
  out[1] = s[1];
  out[2] = c->timestamp;
  out[3] = s[2];
  return DGS_OK;
}

int dgs_pull_read_stats(dgs_ctx* c, uint64_t out[2]) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!out) return DGS_EINVAL;
  unsigned long long s[2] = {0, 0};
  rc = sync_all(c);
  if (rc != DGS_OK) return rc;
  DGS_CUDA(c, cudaMemcpy(s, c->ws[0].stats + 3, sizeof(s), cudaMemcpyDeviceToHost));
  out[0] = s[0];
  out[1] = s[1];
  return DGS_OK;
}

int dgs_prev(dgs_ctx* c, uint32_t worker, int64_t* out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!out || worker >= c->cfg.num_workers) return DGS_EINVAL;
  *out = c->prev[worker];
  return DGS_OK;
}

int dgs_launch_count(dgs_ctx* c, uint64_t* out) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!out) return DGS_EINVAL;
  *out = c->launches;
  return DGS_OK;
}

int dgs_timing_enable(dgs_ctx* c, int on) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  c->timing = on != 0;
  return DGS_OK;
}

int dgs_timing_read(dgs_ctx* c, double ms[DGS_NUM_KERNELS], uint64_t count[DGS_NUM_KERNELS]) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!ms || !count) return DGS_EINVAL;
  rc = sync_all(c);
  if (rc != DGS_OK) return rc;
  for (size_t i = 0; i < c->ev_kernel.size(); ++i) {
    float t = 0.f;
    DGS_CUDA(c, cudaEventElapsedTime(&t, c->ev_pool[2 * i], c->ev_pool[2 * i + 1]));
    c->time_ms[c->ev_kernel[i]] += t;
    c->time_count[c->ev_kernel[i]] += 1;
  }
  c->ev_kernel.clear();
  c->ev_stream.clear();
  for (int i = 0; i < DGS_NUM_KERNELS; ++i) {
    ms[i] = c->time_ms[i];
    count[i] = c->time_count[i];
    c->time_ms[i] = 0.0;
    c->time_count[i] = 0;
  }
  return DGS_OK;
}

int dgs_timing_trace(dgs_ctx* c, uint32_t cap, float* start_ms, float* stop_ms, int32_t* kernel, int32_t* stream,
                     uint32_t* count) {
  int rc = live(c);
  if (rc != DGS_OK) return rc;
  if (!start_ms || !stop_ms || !kernel || !stream || !count) return DGS_EINVAL;
  rc = sync_all(c);
  if (rc != DGS_OK) return rc;
  const size_t m = std::min<size_t>(cap, c->ev_kernel.size());
  for (size_t i = 0; i < m; ++i) {
    DGS_CUDA(c, cudaEventElapsedTime(start_ms + i, c->ev_pool[0], c->ev_pool[2 * i]));
    DGS_CUDA(c, cudaEventElapsedTime(stop_ms + i, c->ev_pool[0], c->ev_pool[2 * i + 1]));
    kernel[i] = c->ev_kernel[i];
    stream[i] = c->ev_stream[i];
  }
  *count = (uint32_t)m;
  c->ev_kernel.clear();
  c->ev_stream.clear();
  return DGS_OK;
}

int dgs_hardware_queues(int* needed, int* configured) {
  if (needed) *needed = kQueuesWanted;
  if (configured) {
    int v = 8;   // the driver's default
    if (const char* e = std::getenv("CUDA_DEVICE_MAX_CONNECTIONS")) {
      char* endp = nullptr;
      const long x = std::strtol(e, &endp, 10);
      if (endp != e && x >= 1 && x <= 32) v = (int)x;
    }
    *configured = v;
  }
  return DGS_OK;
}

int dgs_last_cuda_error(dgs_ctx* c) {
  if (!c || c->magic != kMagic) return 0;
  return c->last_cuda;
}

int dgs_free(dgs_ctx* c) {
  if (!c || c->magic != kMagic) return DGS_ESTATE;
  for (int i = 0; i < kStreams; ++i)
    if (c->st[i]) cudaStreamSynchronize(c->st[i]);
  cudaStreamSynchronize(c->user);
  destroy_ctx(c);
  return DGS_OK;
}

}  // extern "C"

// ---- top-k + encode without any scratch in global memory (dgs_topk_encode_static) --------
namespace {

struct TopkDevice {
  bool ready = false;
  uint32_t max_cluster[2] = {0, 0};   // CTAs of the largest cluster the device takes, for either variant of k_topk
};
constexpr int kMaxDevices = 64;
TopkDevice g_topk_dev[kMaxDevices];
std::mutex g_topk_mu;

struct TopkLaunch {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  TopkLaunch(bool fine, uint32_t cluster, uint32_t cap, cudaStream_t st) {
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(topk_threads(fine));
    cfg.dynamicSmemBytes = (size_t)topk_threads(fine) / 32 * cap * 8;
    cfg.stream = st;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = cluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
  }
};

template <bool FINE>
bool topk_max_cluster(uint32_t* most) {
  if (cudaFuncSetAttribute(k_topk<FINE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           topk_threads(FINE) / 32 * (int)topk_cap(FINE) * 8) != cudaSuccess ||
      cudaFuncSetAttribute(k_topk<FINE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return false;
  for (uint32_t c = kTopkMaxCluster; c >= 1; c /= 2) {
    const TopkLaunch l(FINE, c, topk_cap(FINE), nullptr);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_topk<FINE>, &l.cfg) == cudaSuccess && clusters > 0) {
      *most = c;
      return true;
    }
    cudaGetLastError();
  }
  return false;
}

// Once per device, with that device current.
int topk_setup(int dev, const TopkDevice** out) {
  std::lock_guard<std::mutex> lock(g_topk_mu);
  TopkDevice& d = g_topk_dev[dev];
  if (!d.ready) {
    if (!topk_max_cluster<false>(&d.max_cluster[0]) || !topk_max_cluster<true>(&d.max_cluster[1])) return DGS_ECUDA;
    d.ready = true;
  }
  *out = &d;
  return DGS_OK;
}

}  // namespace

extern "C" int dgs_topk_encode_static(const float* x, uint32_t n, uint32_t k, uint32_t* out_idx, float* out_val,
                                      void* stream) {
  if (!x || !out_idx || !out_val || n == 0 || k == 0 || k > n) return DGS_EINVAL;
  if (n > DGS_STATIC_MAX_N) return DGS_ELIMIT;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DGS_ECUDA;
  const TopkDevice* d = nullptr;
  const int rc = topk_setup(dev, &d);
  if (rc != DGS_OK) return rc;
  const bool fine = n <= kTopkFine;
  // An element a thread, up to the largest cluster: the barriers of 16 CTAs cost no more than those of 2 (16384
  // elements: 12.3 us with 16, 13.0 with 4, 14.3 with 1; 262144: 14.3, 21.7, 45).
  const uint32_t warps = (uint32_t)topk_threads(fine) / 32;
  uint32_t cluster = 1;
  while (cluster < d->max_cluster[fine] && cluster * warps * 32 < n) cluster *= 2;
  // the lists hold all elements of a warp where that fits (shared out as in k_topk)
  const uint32_t W = cluster * warps, unit = n >= W * 512u ? 512u : 32u, slice = ((n + unit - 1) / unit + W - 1) / W * unit;
  const uint32_t cap = std::min(topk_cap(fine), slice);
  const TopkLaunch l(fine, cluster, cap, static_cast<cudaStream_t>(stream));
  const cudaError_t e = fine ? cudaLaunchKernelEx(&l.cfg, k_topk<true>, x, n, k, out_idx, out_val, cap)
                             : cudaLaunchKernelEx(&l.cfg, k_topk<false>, x, n, k, out_idx, out_val, cap);
  return e == cudaSuccess ? DGS_OK : DGS_ECUDA;
}

extern "C" int dgs_topk_encode_static_status(void* stream, int* device_status) {
  if (!device_status) return DGS_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int word = 0;
  if (cudaMemcpyFromSymbolAsync(&word, g_topk_status, sizeof(word), 0, cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return DGS_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return DGS_ECUDA;
  *device_status = word;
  return DGS_OK;
}
