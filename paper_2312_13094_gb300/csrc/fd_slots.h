// Fixed scratch slots shared by concurrent calls (fd_update.cu).
#pragma once

#include <atomic>

namespace fd {

// Slot of one call: taken from N flags on construction (index N: none was free),
// given back when the call leaves.  Work of the call that may still be queued (an
// error between a launch and the wait behind it) would go on using the slot's
// memory, so unless the call has noted its wait with idle(), the slot waits
// itself, by `wait`, before it gives the slot back.
template <int N, class Wait>
class ScratchSlot {
 public:
  ScratchSlot(std::atomic<bool> (&taken)[N], Wait wait) : taken_(taken), wait_(wait) {
    while (i_ < N && taken_[i_].exchange(true)) ++i_;
  }
  ~ScratchSlot() {
    if (i_ >= N) return;
    if (!idle_) wait_();
    taken_[i_] = false;
  }
  ScratchSlot(const ScratchSlot&) = delete;
  ScratchSlot& operator=(const ScratchSlot&) = delete;
  int index() const { return i_; }
  void idle() { idle_ = true; }

 private:
  std::atomic<bool> (&taken_)[N];
  Wait wait_;
  int i_ = 0;
  bool idle_ = false;
};

}  // namespace fd
