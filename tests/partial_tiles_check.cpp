// CPU check of the work list of single lattices whose tiles have sites for only part of a
// CTA (csrc/worklist.h): every plane task once, at most one CTA per slot, segments within
// bounds, for every lattice size and tile height.  Prints "OK <splits>" or "FAIL ...".
#include <cstdio>
#include <map>
#include <vector>

#include "worklist.h"

using namespace clg;

int main() {
  int n = 0;
  for (int N = 8; N <= 512; N += 8)
    for (int BY = 1; BY <= N; ++BY)
      for (int min_sites : {512, 1024, 2048})
        for (int grid : {1, 37, 100, 152}) {
          if (N % BY || BY * N > min_sites || BY > 32) continue;
          for (bool up : {false, true}) {
            std::vector<Seg> segs;
            std::vector<int> cta, sb, se;
            if (!build_worklist({{N, BY, min_sites}}, grid, up, segs, cta, sb, se)) continue;  // too many segments a CTA
            std::vector<int> cover((size_t)(N / BY) * N, 0);
            std::map<int, int> owner;
            bool ok = (int)cta.size() == grid + 1 && cta[grid] == (int)segs.size();
            for (int c = 0; c < grid && ok; ++c)
              for (int i = cta[c]; i < cta[c + 1] && ok; ++i) {
                const Seg& s = segs[i];
                ok = s.ytile >= 0 && s.ytile < N / BY && s.nz >= 1 && s.z0 >= 0 && s.z0 + s.nz <= N &&
                     (s.dir == 1 || (s.dir == -1 && !up)) && s.slot >= sb[0] && s.slot < se[0] &&
                     owner.emplace(s.slot, c).first->second == c;
                for (int z = s.z0; ok && z < s.z0 + s.nz; ++z) ++cover[(size_t)s.ytile * N + z];
              }
            for (int v : cover) ok = ok && v == 1;
            if (!ok) {
              std::printf("FAIL N %d BY %d min %d grid %d up %d\n", N, BY, min_sites, grid, (int)up);
              return 1;
            }
            ++n;
          }
        }
  std::printf("OK %d\n", n);
  return 0;
}
