// A few words of pinned host memory that the results of a call are copied to, kept between
// calls (a few per process: one for each call under way).  Host code only; the memory comes
// from the functions given, so it can be tested without a GPU.
#pragma once
#include <cstddef>
#include <mutex>
#include <vector>

namespace dem {

class PinnedWords {
 public:
  using Alloc = void *(*)(size_t);
  using Free = void (*)(void *);
  PinnedWords(Alloc alloc, Free release) : alloc_(alloc), free_fn_(release) {}

  double *take() {
    {
      std::lock_guard<std::mutex> l(mu_);
      if (!free_.empty()) {
        double *p = free_.back();
        free_.pop_back();
        return p;
      }
    }
    return static_cast<double *>(alloc_(kBytes));
  }
  void give(double *p) {
    {
      std::lock_guard<std::mutex> l(mu_);
      if (free_.size() < kKept) {
        free_.push_back(p);
        return;
      }
    }
    free_fn_(p);
  }

  static constexpr size_t kBytes = 128, kKept = 16;

 private:
  std::mutex mu_;
  std::vector<double *> free_;
  Alloc alloc_;
  Free free_fn_;
};

// The words of one call.  They go back to the pool at its end unless a copy into them may
// still be under way: one that was issued and not seen to complete, whatever the reason (a
// timeout, an error of the wait or of the copy itself).  Such words are not used again.
class PinnedLease {
 public:
  explicit PinnedLease(PinnedWords &pool) : pool_(pool), p_(pool.take()) {}
  ~PinnedLease() {
    if (p_ && !in_flight_) pool_.give(p_);
  }
  PinnedLease(const PinnedLease &) = delete;
  PinnedLease &operator=(const PinnedLease &) = delete;

  double *words() const { return p_; }
  // copy() issues a copy into the words, wait() sees the work before it done; true: both did
  template <class Copy, class Wait>
  bool fetch(Copy &&copy, Wait &&wait) {
    in_flight_ = true;
    if (!copy() || !wait()) return false;
    in_flight_ = false;
    return true;
  }

 private:
  PinnedWords &pool_;
  double *p_;
  bool in_flight_ = false;
};

}  // namespace dem
