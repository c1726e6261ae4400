// opm::schedule_lpt against the plain statement of its rule (two stable sorts and
// a search for the least loaded list): the same order and offsets, also for costs
// beyond its counting sort's buckets and for no units at all.
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>

#include "opm_sched.h"

int main() {
  std::mt19937 rng(7);
  for (int trial = 0; trial < 300; ++trial) {
    const int n = trial == 0 ? 0 : (int)(rng() % 3000), L = 1 + (int)(rng() % 700);
    const int longest = trial % 4 == 0 ? 20000 : trial % 4 == 1 ? 4100 : trial % 4 == 2 ? 3 : 300;
    std::vector<opm::WorkUnit> u(n);
    for (int i = 0; i < n; ++i) u[i] = opm::WorkUnit{i, 0, 0, 0, (int)(rng() % longest), 0, 0, 0};
    std::vector<opm::WorkUnit> want = u;
    std::stable_sort(want.begin(), want.end(), [](const opm::WorkUnit& a, const opm::WorkUnit& b) {
      return opm::unit_cost(a) > opm::unit_cost(b);
    });
    std::vector<long long> load(L, 0);
    for (auto& w : want) {
      w.list = (int)(std::min_element(load.begin(), load.end()) - load.begin());
      load[w.list] += opm::unit_cost(w);
    }
    std::stable_sort(want.begin(), want.end(),
                     [](const opm::WorkUnit& a, const opm::WorkUnit& b) { return a.list < b.list; });
    std::vector<int> off(L + 1);
    opm::schedule_lpt(u.data(), n, L, off.data());
    bool ok = off[0] == 0 && off[L] == n;
    for (int i = 0; i < n && ok; ++i)
      ok = u[i].item == want[i].item && u[i].list == want[i].list && off[u[i].list] <= i && i < off[u[i].list + 1];
    if (!ok) {
      std::printf("trial %d failed: n=%d L=%d\nFAIL\n", trial, n, L);
      return 1;
    }
  }
  std::printf("OK\n");
  return 0;
}
