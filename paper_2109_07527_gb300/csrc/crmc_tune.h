// crmc_tune.h -- the choice among launch forms by timing the sweeps that a
// program runs anyway (host code; no CUDA types).
#pragma once

#include <algorithm>
#include <cstddef>
#include <limits>
#include <vector>

namespace crmc {

// Each sweep runs the current candidate and records its time, in rounds over
// the candidates.  A sweep may be disturbed (a context kept 256 threads where
// 512 ran 12 % faster, when single times decided), so a form is chosen by the
// shortest of COUNTED times.  Those are taken after the first
// round, which only drops the forms that are far off -- all but the fastest
// third -- so that the choice takes no more sweeps than two rounds over all
// forms would.  settling: a box that starts without its ions grows for a dozen
// sweeps, and times of different sweeps then compare states, not forms; the
// first COUNTED rounds are not counted and drop nothing (the global schedule,
// which has a third of the forms).
class FormTuner {
 public:
  static constexpr int COUNTED = 3;
  bool on = true;

  void restart() {
    on = true;
    cand_.clear();
  }
  bool begun() const { return !cand_.empty(); }
  void begin(const std::vector<int> &candidates, bool settling) {
    cand_ = candidates;
    settling_ = settling;
    round_ = 0;
    clear();
    on = !cand_.empty();
  }
  int current() const { return cand_[at_]; }
  // the current candidate's time; true when the choice is made, which is then
  // the current one
  bool record(float ms) {
    ms_[at_] = std::min(ms_[at_], ms);
    if (++at_ < cand_.size()) return false;
    const int first = settling_ ? COUNTED : 1;  // the first counted round
    if (++round_ == first + COUNTED) {
      keep(1);
      on = false;
    } else if (round_ == first) {
      if (!settling_) keep(std::max<size_t>(2, (cand_.size() + 2) / 3));
      clear();
    }
    at_ = 0;
    return !on;
  }

 private:
  std::vector<int> cand_;
  std::vector<float> ms_;  // shortest time of each candidate since clear()
  size_t at_ = 0;
  int round_ = 0;
  bool settling_ = false;

  void clear() {
    ms_.assign(cand_.size(), std::numeric_limits<float>::infinity());
    at_ = 0;
  }
  void keep(size_t n) {  // the n fastest, in their order
    std::vector<float> t = ms_;
    std::sort(t.begin(), t.end());
    const float worst = t[std::min(n, t.size()) - 1];
    std::vector<int> kept;
    for (size_t i = 0; i < cand_.size() && kept.size() < n; ++i)
      if (ms_[i] <= worst) kept.push_back(cand_[i]);
    cand_ = kept;
    at_ = 0;
  }
};

}  // namespace crmc
