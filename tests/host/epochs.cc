// Host check of the barrier epochs of the small-lattice kernels (csrc/epochs.h):
// over more launches than 2^32 epochs make, the word an inbox may hold -- zero
// since the last clearing, or any epoch of a launch since -- is behind every
// epoch of the next launch by signed difference, the kernels' comparison, and
// equal to none.  Prints the launches checked and the clearings.
#include <cstdio>
#include <initializer_list>

#include "../../paper_1312_3265_gb300/csrc/epochs.h"

int main() {
  swc::BarrierEpochs e;
  const long long launches = 3LL << 20;
  long long clearings = 0;
  unsigned newest = 0;  // the newest word; the oldest a group may hold is 0
  for (long long i = 0; i < launches; ++i) {
    if (e.restart()) {
      newest = 0;
      ++clearings;
    }
    const unsigned base = e.take(), first = base + 1, last = base + swc::BarrierEpochs::kLaunch - 1;
    for (unsigned word : {0u, newest})
      for (unsigned epoch : {first, last})
        if ((int)(word - epoch) >= 0) {
          std::printf("launch %lld: word %u passes epoch %u\n", i, word, epoch);
          return 1;
        }
    newest = last;
  }
  std::printf("%lld %lld\n", launches, clearings);
  return 0;
}
