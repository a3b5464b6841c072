// Selections as one kernel, see dgs_one.cuh.  (In the module of the others they cost the rounds on long vectors, which never run
// them, nothing: 8 arrivals on 124 M elements in 148 layers 2880 us apart, 2883 together, 32 on 25.6 M 2070 and 2069.)
#include "dgs_one.cuh"

namespace dgs {
namespace {

template <int MODE>
using OneShared = FinalizeShared<MODE == kPull ? kOneParts : 256>;

template <int MODE, bool MANY>
__global__ void __maxnreg__(80) k_one_push(const __grid_constant__ Workspace ws, const __grid_constant__ SelArgs a) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  __shared__ StreamShared sh;
  __shared__ __align__(8) uint64_t full[OnePushRing::kStages];
  __shared__ int s_dead;
  const float* in = *a.u_cur_slot;
  float* out = *a.u_spare_slot;
  if (blockIdx.x == 0 && threadIdx.x == 0) ws.sync[kBarCount + (a.pair ^ 1u)] = ws.sync[kFail + (a.pair ^ 1u)] = 0;   // for the next selection
  stream_blocks_tma<MODE, OnePushRing>(ws, a, a.L_in, in, out, blockIdx.x, gridDim.x, sh, reinterpret_cast<float*>(dyn_smem), full,
                                       &s_dead, a.phantom_workers, a.spin_limit ? a.spin_limit : kSpinLimit);
  __syncthreads();
  if (s_dead) return;   // finalize's tables would lie where a late copy may land; the others give up at the barrier
  finalize<MODE, MANY, false, 256, true>(ws, a, in, out, *reinterpret_cast<OneShared<MODE>*>(dyn_smem),
                                         dyn_smem + sizeof(OneShared<MODE>), gridDim.x);
}
template <bool MANY>
__global__ void __maxnreg__(80) k_one_pull(const __grid_constant__ Workspace ws, const __grid_constant__ SelArgs a,
                                           const __grid_constant__ PacketLog lg, const __grid_constant__ FoldRange f) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  __shared__ FoldShared sh;
  fold_blocks<true, true>(ws, a, lg, f, sh, dyn_smem);
  __syncthreads();
  finalize<kPull, MANY, false, kOneParts, true>(ws, a, a.D, nullptr, *reinterpret_cast<OneShared<kPull>*>(dyn_smem),
                                                dyn_smem + sizeof(OneShared<kPull>), gridDim.x);
}

}  // namespace

const void* one_kernel(int mode, bool many) {
  switch (mode) {
    case kPushSam: return many ? (const void*)k_one_push<kPushSam, true> : (const void*)k_one_push<kPushSam, false>;
    case kPushResidual: return many ? (const void*)k_one_push<kPushResidual, true> : (const void*)k_one_push<kPushResidual, false>;
    default: return many ? (const void*)k_one_pull<true> : (const void*)k_one_pull<false>;
  }
}

uint32_t one_dyn_bytes(int mode, uint32_t num_segs, uint32_t ahead, uint32_t part_cap) {
  const uint32_t pass = mode == kPull ? fold_dyn_bytes(kWarps, ahead, part_cap) : (uint32_t)OnePushRing::kBytes;
  const uint32_t fin = (uint32_t)(mode == kPull ? sizeof(OneShared<kPull>) : sizeof(OneShared<kPushSam>)) + finalize_dyn_bytes(num_segs);
  return pass > fin ? pass : fin;
}

}  // namespace dgs
