// A selection as one kernel: the pass over the vector and finalize, with a barrier among all CTAs in between in the place of
// the end of a kernel and the start of another (all resident: cooperative launch).  For short vectors, where launches are what a
// selection costs: the host needs 3 us for one, and the GPU leaves 2.4 us between two kernels on a stream where a barrier takes
// 1.3 us.
#pragma once
#include "dgs_kernels.cuh"

namespace dgs {

constexpr int kOneMaxGrid = 148;                                      // upper bound on the grid
constexpr int kOneParts = (kOneMaxGrid * kWarps + 255) / 256 * 256;   // ... and on the parts of a pull's candidates
// Two stages: the next copy is asked for when a round's counts are known and overlaps the writing of its candidates.  A third one
// gains nothing where a CTA has few rounds and takes 32 KB from the passes beside it: rounds of 12 or 16 arrivals, us, two / three:
// 0.5 M elements, 0.2 % 235 / 233, 20 % 506 / 570; 1.5 M, 0.2 % 200 / 199, 1 % 300 / 333.
using OnePushRing = StreamRing<2>;

// The kernel for a mode, and its dynamic shared memory: the pass's and then finalize's, in one place.  ahead, part_cap: of the
// pull's pass.
const void* one_kernel(int mode, bool many);
uint32_t one_dyn_bytes(int mode, uint32_t num_segs, uint32_t ahead, uint32_t part_cap);

}  // namespace dgs
