// What a launch asks the device about a kernel once and keeps: plain host code, for
// the library and for host tests.
#pragma once

#include <cstddef>
#include <mutex>

namespace jet {

// Answers by (device, kernel, shared memory). The kernel is its address: kernels of
// the same signature are different kernels. At most kEntries answers are kept, the
// oldest making room; any thread may ask.
class PairCache {
 public:
  static constexpr int kEntries = 64;

  // the kept answer, or ask()'s; an answer below 1 is a failure and is not kept
  template <typename Ask>
  int get(int device, const void* kernel, size_t smem, Ask ask) {
    {
      std::lock_guard<std::mutex> lock(mu_);
      for (int i = 0; i < held_; ++i) {
        const Entry& e = entries_[i];
        if (e.kernel == kernel && e.smem == smem && e.device == device) return e.answer;
      }
    }
    const int answer = ask();
    if (answer < 1) return answer;
    std::lock_guard<std::mutex> lock(mu_);
    entries_[next_] = Entry{device, kernel, smem, answer};
    next_ = (next_ + 1) % kEntries;
    if (held_ < kEntries) ++held_;
    return answer;
  }

 private:
  struct Entry {
    int device;
    const void* kernel;
    size_t smem;
    int answer;
  };
  std::mutex mu_;
  Entry entries_[kEntries] = {};
  int held_ = 0, next_ = 0;
};

}  // namespace jet
