// When an engine's delivery mode may change, and the tuner's last question
// (host-only; no CUDA dependency).
#pragma once

#include <cstdint>

namespace dbn {

// Steps from iteration g to the next one before which the mode may change: a
// window of wmask + 1 steps starts there, and no earlier spike waits for the
// end of its bin of bin_lead + 1 steps.
inline int64_t steps_to_switch(unsigned long long g, int32_t wmask, int32_t bin_lead) {
  int64_t k = 0;  // (at most a window's steps times a bin's)
  while (((g + (unsigned long long)k) & (unsigned long long)wmask) != 0ull ||
         (g + (unsigned long long)k) % (unsigned long long)(bin_lead + 1) != 0ull)
    ++k;
  return k;
}

// Whether the mode that the rule chose stays after the tuner's turns: it does
// unless the best per-step shape was faster by a tenth than each of three
// timed turns (the first one pays for the graph's upload).  The verdict to
// leave stands until the mode has been changed, at the next step where it may
// be: turns end off a bin's edge for most bin lengths.
class RuleVerdict {
 public:
  void open() { state_ = kTiming, slow_ = 0; }
  bool is_open() const { return state_ != kClosed; }
  bool leaving() const { return state_ == kLeaving; }
  // a timed turn of the rule's mode against the best per-step shape's
  void turn(double ms, double best_ms) {
    if (!(ms > 1.1 * best_ms)) state_ = kClosed;
    else if (++slow_ == 3) state_ = kLeaving;
  }
  void left() { state_ = kClosed; }

 private:
  enum { kClosed, kTiming, kLeaving } state_ = kClosed;
  int slow_ = 0;  // turns in which the rule was the slower one
};

}  // namespace dbn
