// Which of the server's streams a request goes to (plain C++: also tested on
// the host).
//
// Each lane has three streams: copies in, kernels, copies out.  Queue q: 0 ..
// lanes - 1 the kernel streams, then the copy-in, then the copy-out streams.
// A staged request uses all three of its lane, and whatever follows on any of
// them waits for its copies, its kernel or both: its bytes count on all three.
// A direct request is one kernel on one queue.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace pm {

class ServeQueues {
 public:
  void reset(int lanes) {
    lanes_ = lanes;
    beyond_ = 0;
    load_.assign((size_t)3 * lanes, 0);
  }
  int lanes() const { return lanes_; }
  int queues() const { return 3 * lanes_; }
  uint64_t load(int q) const { return load_[q]; }
  // the queues that may hold requests: past the lanes only while a direct
  // request is on one of them (24 empty queues looked at on every pass cost
  // the server thread 1 % of a request's 4.4 us)
  int occupied() const { return beyond_ ? queues() : lanes_; }

  // The queue of a request that moves `weight` bytes, charged with them (a
  // staged request's queue is the kernel stream of its lane).
  int admit(bool direct, uint64_t weight) {
    const int q = direct ? pick_direct(weight) : pick_lane();
    add(q, direct, (int64_t)weight);
    return q;
  }
  // the request has left the queue
  void release(int q, bool direct, uint64_t weight) { add(q, direct, -(int64_t)weight); }

 private:
  static constexpr uint64_t kLarge = 1u << 20;

  void add(int q, bool direct, int64_t w) {
    load_[q] += (uint64_t)w;
    if (q >= lanes_) beyond_ += w < 0 ? -1 : 1;
    if (!direct) {
      load_[lanes_ + q] += (uint64_t)w;
      load_[2 * lanes_ + q] += (uint64_t)w;
    }
  }
  // The lane with the least work on its busiest stream: a small request does
  // not queue behind a large one while another lane is idle.
  int pick_lane() const {
    auto busiest = [&](int l) { return std::max({load_[l], load_[lanes_ + l], load_[2 * lanes_ + l]}); };
    int best = 0;
    for (int l = 1; l < lanes_; ++l)
      if (busiest(l) < busiest(best)) best = l;
    return best;
  }
  // A kernel stream; a direct request of a MB or more finds another queue
  // when every lane is busy, one of half a MB when every lane has 2 MB ahead.
  // Its kernel spends most of its time waiting for the host link, so three
  // times as many of them in flight keep the link busier (200 requests of 2^12
  // .. 2^14, up to 8 primes, 8 lanes: 1.23 ms on the kernel streams alone).
  // The link moves a MB in about the 4.4 us that the server thread needs per
  // request: below that the thread is the bound, unless a backlog shows that
  // larger requests hold the link, and launches on more streams cost it more.
  // The other queues for half a MB always / from 2 MB ahead / never: that list
  // 1.080 / 1.089 / 1.100 ms, 1000 requests of 2^10 .. 2^12 4.57 / 4.46 / 4.47,
  // 300 of 2^12 1.475 / 1.424 / 1.393.
  int pick_direct(uint64_t weight) const {
    int best = 0;
    for (int l = 1; l < lanes_; ++l)
      if (load_[l] < load_[best]) best = l;
    const uint64_t ahead = load_[best];
    if ((weight >= kLarge && ahead > 0) || (weight >= kLarge / 2 && ahead >= 2 * kLarge))
      for (int l = lanes_; l < queues(); ++l)
        if (load_[l] < load_[best]) best = l;
    return best;
  }

  int lanes_ = 0;
  int beyond_ = 0;              // direct requests on queues past the lanes
  std::vector<uint64_t> load_;  // bytes of the requests in flight on each queue
};

}  // namespace pm
