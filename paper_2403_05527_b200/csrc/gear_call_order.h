// Which of the library's calls lie behind one another on a stream: a decode call may request its first copies before its
// kernel waits for the kernel in front only if that kernel cannot be the one that last wrote the cache.  Host only.
#pragma once
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <unordered_map>

namespace gear {

// A number is drawn from one counter when a call begins, and another one when a write has been queued.  A call that began
// after a write was numbered, and whose kernels have been queued since, lies behind the write on their common stream, whatever
// other threads do between drawing a number and launching; a call that failed is never reported as queued and counts for
// nothing.
class CallOrder {
 public:
  struct Key {                 // a place where kernels line up
    uint64_t stream;           // the handle
    uint64_t capture;          // id of the capture that the stream is in, 0 if none: captured kernels line up in the graph alone
    int device;                // the default stream has one handle on every device
    bool ordered;              // false: the handle does not name one line of kernels, nothing is known about it
    bool operator==(const Key& o) const {
      return stream == o.stream && capture == o.capture && device == o.device && ordered == o.ordered;
    }
  };
  struct Write {               // the last call that wrote something
    Key key = {0, 0, 0, false};
    uint64_t number = 0;       // 0: there was none
  };

  uint64_t begin() { return counter_.fetch_add(1) + 1; }
  void queued(const Key& key, uint64_t begun) {
    if (!key.ordered) return;
    std::lock_guard<std::mutex> lock(mutex_);
    if (last_.size() >= kMost && last_.find(key) == last_.end()) last_.clear();   // forgetting only makes calls wait
    uint64_t& last = last_[key];
    if (begun > last) last = begun;
  }
  Write written(const Key& key) { return {key, begin()}; }
  // Whether another call lies between write `w` and what is queued with `key` next.  A write that a graph holds may be repeated
  // by it at any time: only calls of the same capture are known to lie behind it.
  bool another_since(const Key& key, const Write& w) {
    if (!key.ordered || w.number == 0 || !w.key.ordered || w.key.stream != key.stream || w.key.device != key.device ||
        (w.key.capture != 0 && w.key.capture != key.capture))
      return false;
    std::lock_guard<std::mutex> lock(mutex_);
    const auto it = last_.find(key);
    return it != last_.end() && it->second > w.number;
  }

 private:
  static constexpr size_t kMost = 1024;
  struct Hash {
    size_t operator()(const Key& k) const { return (size_t)((k.stream ^ (k.capture << 20) ^ (uint64_t)k.device) * 0x9E3779B97F4A7C15ull >> 7); }
  };
  std::atomic<uint64_t> counter_{0};
  std::mutex mutex_;
  std::unordered_map<Key, uint64_t, Hash> last_;    // number of the latest call whose kernels have been queued there
};

}  // namespace gear
