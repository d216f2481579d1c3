// launch_sample.h -- which launches of a filter are timed, and what their times say about all of
// them.  Long launches are all timed.  Of short ones, whose work shrinks as columns reach their
// degrees, the fourth of every eight stands for the eight (the first would be the longest of them),
// the last of these for the one to three after it too; the first of all stands in where a filter has
// fewer than four.
#pragma once

#include <cstddef>
#include <vector>

namespace chase {

class LaunchSample {
 public:
  // Whether the next launch is to be timed; times are added in the order of the launches timed.
  bool next(bool few_us) {
    if (!few_us) {
      kind_.push_back(kLong);
      return true;
    }
    const size_t i = few_all_++;
    if (i != 0 && i % 8 != 3) return false;
    kind_.push_back(i == 0 ? kSpare : kFew);
    return true;
  }
  // The time of all launches from those of the timed ones, of which the first `n` are known.
  double total(const double* t, size_t n) const {
    double s = 0.0, last = 0.0;
    size_t left = few_all_;  // short launches that no sample stands for yet
    for (size_t i = 0; i < n && i < kind_.size(); ++i) {
      if (kind_[i] == kLong) {
        s += t[i];
      } else {
        last = t[i];
        if (kind_[i] == kSpare) continue;
        const size_t m = left < 8 ? left : 8;
        s += last * (double)m;
        left -= m;
      }
    }
    return s + last * (double)left;
  }
  void clear() {
    kind_.clear();
    few_all_ = 0;
  }

 private:
  enum : char { kLong, kSpare, kFew };
  std::vector<char> kind_;
  size_t few_all_ = 0;
};

}  // namespace chase
