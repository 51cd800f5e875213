// The host's knowledge of the counts (csrc/counts_state.h) against a device that is only modelled:
// its counts are zero or not.  Every sequence of up to six calls: passes that run, are cut short
// after their advance, or are recorded into a graph (whole or cut short), replays of that graph.
// Prints "dirty N": passes that started from counts that were not zero; "clears N": clears that
// passes ran in a sequence of steps alone.
#include <cstdio>
#include <vector>

#include "counts_state.h"

namespace {

enum Op { kStep, kCut, kCapture, kCaptureCut, kReplay, kGrid, kOps };

struct Model {
  pdfx::CountsState host;
  bool zero = false;            // the device's counts
  bool graph = false, graph_clears = false;
  long dirty = 0, clears = 0;

  void pass(bool clear, bool whole) {
    if (clear) { zero = true; ++clears; }
    if (!zero) ++dirty;
    zero = whole;               // the last kernel clears them
  }
  void run(int op) {
    switch (op) {
      case kStep:
      case kCut: {
        const bool clear = host.begin(false);
        pass(clear, op == kStep);
        if (op == kStep) host.end(true);
        break;
      }
      case kCapture:
      case kCaptureCut: {
        const bool clear = host.begin(true);
        if (op == kCapture) {
          host.end(true);
          graph = true;
          graph_clears = clear;
        }
        break;
      }
      case kReplay:
        if (graph) pass(graph_clears, true);
        break;
      case kGrid:
        host = pdfx::CountsState{};
        zero = graph = false;
        break;
    }
  }
};

}  // namespace

int main() {
  long dirty = 0;
  for (int n = 1; n <= 6; ++n) {
    std::vector<int> op(n, 0);
    for (;;) {
      Model m;
      for (int o : op) m.run(o);
      dirty += m.dirty;
      int k = 0;
      while (k < n && ++op[k] == kOps) op[k++] = 0;
      if (k == n) break;
    }
  }
  Model steps;
  for (int k = 0; k < 6; ++k) steps.run(kStep);
  std::printf("dirty %ld\nclears %ld\n", dirty, steps.clears);
}
