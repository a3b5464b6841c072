// Who arrived when: for rules that depend on how many events the GPU works on side by side.  Plain C++, host side.
#pragma once
#include <algorithm>
#include <cstdint>
#include <vector>

namespace dgs {

// An arrival is an event of a worker (its push, or its pull where nothing was pushed); a join makes the caller's stream, or the
// host, wait for all events before it.
class Arrivals {
 public:
  explicit Arrivals(uint32_t workers = 0) : window_(std::min<uint32_t>(32, std::max<uint32_t>(8, 2 * workers))), last_(workers, 0) {}
  void arrived(uint32_t worker) {
    count_ += 1;
    // An event waits for the one before it of the same worker, if that may still be in flight.
    const uint64_t gap = last_[worker] > joined_at_ ? count_ - last_[worker] : 8;
    if (gap < 8) near8_ = count_ + window_;
    if (gap < 4) near4_ = count_ + window_;
    last_[worker] = count_;
  }
  void joined() {
    if (count_ > joined_at_) batch_ = count_ - joined_at_;
    joined_at_ = count_;
  }
  // Between the last two joins that had any there was one arrival.
  bool lone() const { return batch_ == 1; }
  // Lately an event had to wait for one of the three before it.
  bool chained() const { return count_ < near4_; }
  // How many events run side by side: 8 (or more), 4 to 7 (reported as 4), or fewer (1).  That many have to come between two joins,
  // and lately, for as long as every worker takes to come twice, none may have waited for one so few arrivals before it.
  uint32_t abreast() const {
    const uint64_t batch = std::max(batch_, count_ - joined_at_);
    return batch >= 8 && count_ >= near8_ ? 8 : batch >= 5 && !chained() ? 4 : 1;
  }

 private:
  uint64_t count_ = 0, joined_at_ = 0;   // arrivals so far, and at the last join
  uint64_t batch_ = 1;                   // arrivals between the last two joins that had any
  uint64_t near4_ = 0, near8_ = 0;       // until so many arrivals, one of the last few is taken to be in an event's way
  uint32_t window_;
  std::vector<uint64_t> last_;           // number of each worker's latest arrival, counted from 1 (0: none)
};

}  // namespace dgs
