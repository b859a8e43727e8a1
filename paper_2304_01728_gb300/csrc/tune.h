// Choice between the forms of a product from timings (solve.cu, pick_variant).
#pragma once
#include <algorithm>
#include <vector>

namespace dpgmg {

constexpr int TUNE_REPS = 5;     // launches of each form per timing, the forms in turn
constexpr int TUNE_ROUNDS = 3;   // timings beside other work after which a choice is settled all the same

// What the timings of one product have shown.  A form's time is its smallest:
// other work on the GPU only ever adds to a launch, and a sum of a few would let
// one disturbed launch decide (forms differ by up to five times, and a choice is
// kept for the life of the process).  A timing during which no other setup or
// solve of the process ran settles the choice; one that had company is kept as a
// candidate, and the next systems of that shape time again, up to TUNE_ROUNDS.
struct TuneRecord {
  std::vector<float> ms;   // smallest time of each form
  int rounds = 0;
  bool settled = false;
  void add(const std::vector<std::vector<float>>& t, bool alone) {   // t[form][repetition]
    if (ms.size() != t.size()) {
      ms.assign(t.size(), 0.f);
      rounds = 0;
    }
    for (size_t v = 0; v < t.size(); ++v) {
      const float m = *std::min_element(t[v].begin(), t[v].end());
      ms[v] = rounds ? std::min(ms[v], m) : m;
    }
    settled = alone || ++rounds >= TUNE_ROUNDS;
  }
  // the first form unless another is at least 5% faster, then the fastest
  size_t best() const {
    size_t b = 0;
    for (size_t v = 1; v < ms.size(); ++v)
      if (ms[v] < (b == 0 ? 0.95f : 1.0f) * ms[b]) b = v;
    return b;
  }
};

}  // namespace dpgmg
