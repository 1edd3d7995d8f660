// Set-up that holds for one device of the process: function attributes (limits of
// dynamic shared memory), context limits.
#pragma once

#include <mutex>
#include <vector>

namespace cello {

// Runs a set-up once for each device, with that device current; threads that come
// meanwhile wait for it.
class OncePerDevice {
 public:
  template <typename F>
  void run(int device, F set_up) {
    if (device < 0) return;
    const std::lock_guard<std::mutex> lock(mutex_);
    if (device >= (int)done_.size()) done_.resize((size_t)device + 1, false);
    if (done_[(size_t)device]) return;
    set_up();
    done_[(size_t)device] = true;
  }

 private:
  std::mutex mutex_;
  std::vector<bool> done_;
};

}  // namespace cello
