// Independent pieces of work shared out over a bounded number of streams.
#pragma once
#include <algorithm>
#include <vector>

namespace rslb {

// The chain of each item: loads in the order of launch, heaviest first; an item
// joins the chain with the least load so far (of equals the first), so up to `most`
// items have a chain each and more share them evenly.
inline std::vector<int> assign_chains(const std::vector<double>& load, int most) {
  std::vector<double> sum(std::min<size_t>(load.size(), most), 0.0);
  std::vector<int> chain;
  for (double x : load) {
    const size_t c = std::min_element(sum.begin(), sum.end()) - sum.begin();
    sum[c] += x;
    chain.push_back((int)c);
  }
  return chain;
}

}  // namespace rslb
