// CPU check of choose_tiles (worklist.h): over lattice sizes, storage widths and
// mixes, the chosen heights are admissible, the split is one build_worklist takes
// and covers every plane once, small lattices are spread over the SMs (at least
// half of them from 16^3 up) and large ones keep the tallest tiles on every SM.
// Prints "OK <n>" or "FAIL <case>: <reason>".
#include <algorithm>
#include <cstdio>
#include <vector>

#include "worklist.h"

using namespace clg;

static int fails = 0, done = 0;

static void check(const std::vector<int>& Ns, int vx, const PlaneCost& cost, bool up_only, int nsm) {
  std::vector<LatTiles> lats;
  std::vector<std::vector<int>> cand;
  long long tallest = 0;
  int small = 1 << 30;
  for (int N : Ns) {
    std::vector<int> c;
    for (int by = std::min(N, 512 / (N / vx)); by >= 1; --by)
      if (N % by == 0) c.push_back(by);
    lats.push_back({N, 0, 512 * vx});
    cand.push_back(c);
    tallest += (long long)(N / c[0]) * N;
    small = std::min(small, N);
  }
  const int grid = choose_tiles(lats, cand, nsm, up_only, cost);
  const char* why = nullptr;
  std::vector<Seg> segs;
  std::vector<int> first, sb, se;
  if (grid < 1 || grid > nsm) why = "CTA count";
  for (size_t l = 0; l < lats.size() && !why; ++l)
    if (std::find(cand[l].begin(), cand[l].end(), lats[l].BY) == cand[l].end()) why = "height not admissible";
  if (!why && !build_worklist(lats, grid, up_only, segs, first, sb, se)) why = "split refused";
  if (!why) {
    std::vector<std::vector<int>> cover(lats.size());
    for (size_t l = 0; l < lats.size(); ++l) cover[l].assign((size_t)(lats[l].N / lats[l].BY) * lats[l].N, 0);
    for (const Seg& s : segs)
      for (int z = s.z0; z < s.z0 + s.nz; ++z) cover[s.lat][(size_t)s.ytile * lats[s.lat].N + z] += 1;
    for (auto& v : cover)
      for (int n : v)
        if (n != 1) why = "a plane covered other than once";
  }
  if (!why && small >= 16 && 2 * grid < nsm && lats.size() == 1) why = "SMs left idle";
  if (!why && tallest >= (long long)kFewPlanes * nsm) {
    if (grid != nsm) why = "large lattices: not every SM";
    for (size_t l = 0; l < lats.size(); ++l)
      if (lats[l].BY != cand[l][0]) why = "large lattices: not the tallest tiles";
  }
  ++done;
  if (why) {
    ++fails;
    std::printf("FAIL N %d (%zu lattices) vx %d up %d nsm %d: %s\n", Ns[0], Ns.size(), vx, up_only, nsm, why);
  }
}

int main() {
  const PlaneCost costs[] = {{1.0, 0.0002}, {1.2, 0.009}, {1.2, 0.0045}, {1.0, 0.002}, {1.2, 0.072}};
  for (int nsm : {152, 148, 60})
    for (const PlaneCost& c : costs)
      for (int up = 0; up < 2; ++up)
        for (int vx : {1, 2, 4}) {
          for (int N : {8, 16, 24, 32, 48, 64, 72, 96, 128, 144, 192, 216, 256, 288, 384, 432, 512})
            if (N / vx <= 512) check({N}, vx, c, up != 0, nsm);
          check({16, 32}, vx, c, up != 0, nsm);
          check({32, 32, 32, 64, 8}, vx, c, up != 0, nsm);
          check(std::vector<int>(512, 8), vx, c, up != 0, nsm);
          check({128, 96, 64, 32, 128, 96, 64, 32}, vx, c, up != 0, nsm);
        }
  if (!fails) std::printf("OK %d\n", done);
  return fails != 0;
}
