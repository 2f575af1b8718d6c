// Remembered tile choices (host code, see best_tile): a training loop repeats a handful of shapes, and the estimate walks every
// tile of every schedule.  The newest kEntries shapes are kept, whatever came before them; a shape's choice belongs to
// a device, because how many clusters are resident at once differs between GPUs with the same number of SMs.
#pragma once
#include <algorithm>
#include <mutex>

namespace nvfp4 {

class TileMemo {
 public:
  static constexpr int kEntries = 256, kKey = 8;  // M, N, K of up to two problems, output types, device
  bool find(const int (&key)[kKey], int* tile) {
    std::lock_guard<std::mutex> lock(mu_);
    for (int i = 0; i < n_; ++i)
      if (std::equal(key, key + kKey, entries_[i].key)) {
        *tile = entries_[i].tile;
        return true;
      }
    return false;
  }
  void put(const int (&key)[kKey], int tile) {
    std::lock_guard<std::mutex> lock(mu_);
    Entry& e = entries_[next_];
    std::copy(key, key + kKey, e.key);
    e.tile = tile;
    next_ = (next_ + 1) % kEntries;
    n_ = std::max(n_, next_ == 0 ? kEntries : next_);
  }

 private:
  struct Entry {
    int key[kKey], tile;
  };
  std::mutex mu_;
  Entry entries_[kEntries];
  int n_ = 0, next_ = 0;
};

}  // namespace nvfp4
