// crmc_tune.h -- the choice among launch forms by timing sweeps that a program
// runs anyway (host code; no CUDA types).
#pragma once

#include <algorithm>
#include <cstddef>
#include <limits>
#include <vector>

namespace crmc {

// n forms are tried in the first n sweeps, one each; the fastest third of them,
// four at most, is compared on three later sweeps, each run in every one of these
// forms from the same state (all give the same one).  The time of a sweep varies by 15 %
// with where its domains lie on dense particles, more than the best forms
// differ: times of different sweeps chose at random among them (two
// nanoparticles: 1.82 to 1.98 ms per four cycles), and one disturbed sweep could
// decide.  A form's score adds its times over the fastest form's on each of the
// three sweeps, without the worst of them, so that no single run decides.  The
// comparison ends with sweep 2 n, when a box has moved away from its start.
// settling (the global schedule, which has a third of the forms): a box that
// starts without its ions grows for a dozen sweeps; a second round over the
// forms replaces the first, and the comparison ends with sweep 3 n.
class FormTuner {
 public:
  static constexpr int FINAL_SWEEPS = 3;
  static constexpr size_t MOST = 4;  // forms in the comparison
  bool on = true;

  void restart() {
    on = true;
    cand_.clear();
  }
  bool begun() const { return !cand_.empty(); }
  void begin(const std::vector<int> &candidates, bool settling) {
    cand_ = candidates;
    ms_.assign(cand_.size(), 0.0f);
    ratio_.assign(cand_.size(), {});
    const int n = (int)cand_.size(), rounds = settling ? 2 : 1;
    sweep_ = 0;
    trials_ = rounds * n;
    finals_ = std::max(trials_, (rounds + 1) * n - FINAL_SWEEPS);
    on = n > 0;
  }
  // the forms that the coming sweep is to be timed in (0: none)
  int forms() const { return sweep_ < trials_ ? 1 : sweep_ < finals_ ? 0 : (int)cand_.size(); }
  int form(int i) const { return cand_[place(i)]; }
  void time(int i, float ms) { ms_[place(i)] = ms; }
  // a sweep was run; the form to run from here on
  int pass() {
    ++sweep_;
    if (sweep_ < trials_) return cand_[best(ms_, (size_t)std::min(sweep_, (int)cand_.size()))];
    if (sweep_ == trials_) keep_third();
    if (sweep_ <= finals_) return cand_[best(ms_, cand_.size())];
    const float fastest = *std::min_element(ms_.begin(), ms_.end());
    std::vector<float> score(cand_.size());
    for (size_t i = 0; i < cand_.size(); ++i) {
      ratio_[i].push_back(ms_[i] / fastest);
      for (float r : ratio_[i]) score[i] += r;
      if (ratio_[i].size() > 1) score[i] -= *std::max_element(ratio_[i].begin(), ratio_[i].end());
    }
    on = sweep_ < finals_ + FINAL_SWEEPS && cand_.size() > 1;
    return cand_[best(score, score.size())];
  }

 private:
  std::vector<int> cand_;
  std::vector<float> ms_;                  // each form's last time
  std::vector<std::vector<float>> ratio_;  // over the fastest form's, on the sweeps of the comparison
  int sweep_ = 0, trials_ = 0, finals_ = 0;

  size_t place(int i) const { return sweep_ < trials_ ? (size_t)sweep_ % cand_.size() : (size_t)i; }
  static size_t best(const std::vector<float> &x, size_t n) {
    return (size_t)(std::min_element(x.begin(), x.begin() + (std::ptrdiff_t)n) - x.begin());
  }
  void keep_third() {
    std::vector<float> t = ms_;
    std::sort(t.begin(), t.end());
    const size_t n = std::min(t.size(), std::min(std::max<size_t>(2, (t.size() + 2) / 3), MOST));
    size_t k = 0;
    for (size_t i = 0; i < cand_.size() && k < n; ++i)
      if (ms_[i] <= t[n - 1]) {
        cand_[k] = cand_[i];
        ms_[k++] = ms_[i];
      }
    cand_.resize(k);
    ms_.resize(k);
    ratio_.resize(k);
  }
};

}  // namespace crmc
