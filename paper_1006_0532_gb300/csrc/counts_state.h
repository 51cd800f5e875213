// What the host knows of the counts per element and the brute-force list's length.
#pragma once

namespace pdfx {

// Both start a step at zero, left so by the statistics pass before it (its last kernel clears
// them), so that a step needs no memsets.  Whether they are zero where the stream stands is known
// on the host: not before the first pass, and not after one that was cut short.  What a capture
// records has not run, so it changes nothing of this; and its graph may be replayed after
// anything, so a captured pass clears for itself.  (The library's own graph of a re-order cycle
// holds no clears: its launch goes through begin() and end() like a pass, and what its capture does
// to this state is undone.)
struct CountsState {
  bool zero = false;

  // Before a pass (an advance or a count).  capturing: the stream only records.  True: clear first.
  bool begin(bool capturing) {
    const bool clear = !zero || capturing;
    kept_ = capturing && zero;
    recorded_ = capturing;
    zero = false;
    return clear;
  }
  // After the pass's last kernel was launched (ok) or the launches failed.
  void end(bool ok) { zero = recorded_ ? kept_ : ok; }

 private:
  bool kept_ = false, recorded_ = false;
};

}  // namespace pdfx
