// Epochs of the barriers between the blocks of the small-lattice kernels
// (small.cuh), over the launches of one engine.  Host only.
//
// A block waits until the words in its inbox carry the epoch it waits for; a
// barrier's flags may be ahead of it (the even-odd form has two barriers in a
// row), so they are compared by signed difference, which holds for words less
// than 2^31 epochs old.  A group of blocks may go unused for as long as the
// engine lives (the number of groups follows the load), so the inboxes are
// cleared and the epochs start anew long before that: every 2^22 epochs, 1024
// launches (a clearing takes a few microseconds).
#pragma once

namespace swc {

struct BarrierEpochs {
  static constexpr unsigned kLaunch = 1u << 12;   // epochs set aside for a launch
  static constexpr unsigned kRestart = 1u << 22;
  unsigned at = 0;  // every epoch of the launches since the last clearing is at most this
  // Before a launch: whether the inboxes have to be cleared first.
  bool restart() {
    if (at < kRestart) return false;
    at = 0;
    return true;
  }
  // The launch's epochs are above the returned one (which no word exceeds).
  unsigned take() {
    const unsigned base = at;
    at += kLaunch;
    return base;
  }
};

}  // namespace swc
