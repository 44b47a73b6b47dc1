// pt_tuner.h — which configuration the FP32 ensemble engine runs a round in (host logic only).
//
// A configuration changes how a round's correction sweeps are cut into tiles and branches, so only they are
// timed, and only rounds in which every member takes the same number of them are compared: the members a
// round runs, its FP64 phases and a member's spent budget differ from round to round. A step runs the
// configurations not timed yet, one a round, until a round does other work than the ones timed so far (members
// have stopped), and goes on with the fastest; the next step takes up the rest. A step whose first round
// differs (other members start) begins a new comparison, and after four times as many timed rounds as there are
// configurations the fastest of the comparison at hand stays.
#pragma once

#include <vector>

namespace pt {

struct MixConfig {
  int zchunk, groups;   // depth of a correction tile, member groups (parallel branches)
};
constexpr MixConfig kMixConfigs[] = {{64, 1}, {32, 1}, {64, 4}, {32, 4}, {32, 8}, {64, 8}, {64, 16}};
constexpr int kMixConfigCount = (int)(sizeof kMixConfigs / sizeof kMixConfigs[0]);

class MixTuner {
 public:
  void reserve(int members) { like_.reserve(members); }
  void begin_step() {
    timing_ = !done_;
    first_ = true;
  }
  bool timing() const { return timing_; }                  // the next round is to be timed
  int config() const { return timing_ ? next() : best(); }
  int best() const {                                       // the fastest timed, the first if none is
    int b = 0;
    for (int k = 0; k < kMixConfigCount; ++k)
      if (ms_[k] > 0.f && (!(ms_[b] > 0.f) || ms_[k] < ms_[b])) b = k;
    return b;
  }
  // A timed round in config() took `ms` for its correction sweeps; sweeps: how many each member ran.
  void timed_round(const std::vector<int>& sweeps, float ms) {
    const int k = next();                                  // = config()
    bool any = false;
    for (int s : sweeps) any = any || s > 0;
    if (any && sweeps != like_ && first_) {
      like_ = sweeps;
      for (int c = 0; c < kMixConfigCount; ++c)
        if (c != k) ms_[c] = 0.f;
    }
    first_ = false;
    if (!any || sweeps != like_) {
      timing_ = false;
      return;
    }
    ms_[k] = ms > 0.f ? ms : 1e-6f;
    done_ = ++rounds_ >= 4 * kMixConfigCount || next() == kMixConfigCount;
    timing_ = !done_;
  }

 private:
  int next() const {                                       // the first configuration not timed
    int k = 0;
    while (k < kMixConfigCount && ms_[k] > 0.f) ++k;
    return k;
  }
  std::vector<int> like_;
  float ms_[kMixConfigCount] = {};
  int rounds_ = 0;
  bool done_ = false, timing_ = false, first_ = false;
};

}  // namespace pt
