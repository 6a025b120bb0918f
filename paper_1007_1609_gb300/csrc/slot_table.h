// slot_table.h -- what the device answered about a launch shape, kept for the
// process: by key (device and shape), for any number of threads.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>

namespace cbdg {

template <typename Key>
class SlotTable {
 public:
  // The number kept under key, or ask()'s answer: at least 0 (0: the shape does not
  // fit, which stays so and is kept), or negative for a query that failed, which is
  // not kept and asked again by the next call.
  template <typename Ask>
  int get(const Key &key, Ask ask) {
    std::lock_guard<std::mutex> lock(mutex_);
    const auto it = known_.find(key);
    if (it != known_.end()) return it->second;
    const int n = ask();
    if (n < 0) return n;
    if (known_.size() >= kMost) known_.clear();  // (keys hold sizes that callers choose)
    return known_[key] = n;
  }
  std::size_t size() const { return known_.size(); }
  static constexpr std::size_t kMost = 4096;

 private:
  std::mutex mutex_;
  std::map<Key, int> known_;
};

}  // namespace cbdg
