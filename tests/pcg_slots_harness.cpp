// Every interleaving of a few blocks that run the one-launch solve's passes over the sum slots
// (csrc/eulerian_ops.h: pcg_sum_slot): publish the pass's sums, arrive, and once all have arrived
// read every block's sums, one at a time.  Prints "library N", the number of schedules' states
// in which a block reads a sum of another pass, and "shared N", the same with one set per sum
// that all passes share, which the search has to find wrong.
#include <cstdio>
#include <set>
#include <vector>

#include "eulerian_ops.h"

namespace {

constexpr int kBlocks = 3, kComponents = 2, kPasses = 6;   // a block holds one item of each component

size_t shared_slot(int, int which, int C, int per, int c, int item) {
  return (static_cast<size_t>(which) * C + c) * static_cast<size_t>(per) + item;
}

struct Step {
  enum { kPublish, kArrive, kRead } what;
  int pass, which, c, item;
};

// The steps of block b, in order; a read of pass p needs kBlocks (p + 1) arrivals.
std::vector<Step> program(int b) {
  std::vector<Step> v;
  for (int n = 0; n < kPasses; ++n) {
    const int sums = n % 2 + 1;
    for (int w = 0; w < sums; ++w)
      for (int c = 0; c < kComponents; ++c) v.push_back({Step::kPublish, n, w, c, b});
    v.push_back({Step::kArrive, n, 0, 0, 0});
    for (int w = 0; w < sums; ++w)
      for (int c = 0; c < kComponents; ++c) v.push_back({Step::kRead, n, w, c, (b + 1) % kBlocks});
  }
  return v;
}

template <typename Slot>
long wrong_reads(Slot slot) {
  std::vector<Step> prog[kBlocks];
  for (int b = 0; b < kBlocks; ++b) prog[b] = program(b);
  // a state: each block's place, and the pass whose sum each slot holds
  struct State {
    std::vector<int> at, mem;
    bool operator<(const State& o) const { return at != o.at ? at < o.at : mem < o.mem; }
  };
  std::set<State> seen;
  std::vector<State> todo{{std::vector<int>(kBlocks, 0),
                           std::vector<int>(pdfx::eops::kPcgSumSets * kComponents * kBlocks, -1)}};
  long wrong = 0;
  while (!todo.empty()) {
    const State s = todo.back();
    todo.pop_back();
    if (!seen.insert(s).second) continue;
    int arrived = 0;
    for (int b = 0; b < kBlocks; ++b)
      for (int k = 0; k < s.at[b]; ++k) arrived += prog[b][k].what == Step::kArrive;
    for (int b = 0; b < kBlocks; ++b) {
      if (s.at[b] == static_cast<int>(prog[b].size())) continue;
      const Step& q = prog[b][s.at[b]];
      if (q.what == Step::kRead && arrived < kBlocks * (q.pass + 1)) continue;
      State t = s;
      ++t.at[b];
      if (q.what != Step::kArrive) {
        int& m = t.mem.at(slot(q.pass % 2, q.which, kComponents, kBlocks, q.c, q.item));
        if (q.what == Step::kPublish) m = q.pass;
        else wrong += m != q.pass;
      }
      todo.push_back(t);
    }
  }
  return wrong;
}

}  // namespace

int main() {
  std::printf("library %ld\n", wrong_reads(pdfx::eops::pcg_sum_slot));
  std::printf("shared %ld\n", wrong_reads(shared_slot));
  // distinct places for everything a pass and the next one hold
  std::set<size_t> places;
  size_t n = 0;
  for (int which = 0; which < 3; ++which)
    for (int c = 0; c < 9; ++c)
      for (int item = 0; item < 256; ++item, ++n)
        places.insert(pdfx::eops::pcg_sum_slot(which > 0, which > 0 ? which - 1 : 0, 9, 256, c, item));
  std::printf("places %d\n", places.size() == n && *places.rbegin() == pdfx::eops::kPcgSumSets * 9 * 256 - 1);
}
