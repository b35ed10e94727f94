// CPU check of the work split (csrc/worklist.h) that the block-aligned form is there and is what
// its name says, also for tiles that fill only part of a CTA: the sizes that gained by it get it, the
// interior tiles of a block march the same planes in the same direction, and no split is
// refused at the heights and CTA counts that choose_tiles returns.  Prints "OK <n>" or "FAIL ...".
#include <algorithm>
#include <cstdio>
#include <vector>

#include "worklist.h"

using namespace clg;

static int fails = 0, splits = 0, aligned = 0;

static bool admissible(int N) {
  int m = N;
  while (m % 2 == 0) m /= 2;
  while (m % 3 == 0) m /= 3;
  return m == 1;
}

static void check(int N, int vx, const PlaneCost& cost, bool up, int nsm, bool must) {
  std::vector<int> cand;
  for (int by = std::min(N, 512 / (N / vx)); by >= 1; --by)
    if (N % by == 0) cand.push_back(by);
  std::vector<LatTiles> lats = {{N, 0, 512 * vx}};
  const int grid = choose_tiles(lats, {cand}, nsm, up, cost);
  std::vector<Seg> segs;
  std::vector<int> first, sb, se;
  if (!build_worklist(lats, grid, up, segs, first, sb, se)) {
    ++fails;
    std::printf("FAIL N %d vx %d up %d nsm %d: split of height %d on %d CTAs refused\n", N, vx, up, nsm, lats[0].BY, grid);
    return;
  }
  ++splits;
  AlignedPlan A;
  std::vector<Seg> as;
  std::vector<int> af;
  if (!aligned_split(lats[0], grid, up, as, af)) {
    if (must) {
      ++fails;
      std::printf("FAIL N %d vx %d up %d nsm %d: no aligned split of height %d on %d CTAs\n", N, vx, up, nsm, lats[0].BY, grid);
    }
    return;
  }
  ++aligned;
  aligned_plan(lats[0], grid, A);
  const int YT = N / lats[0].BY;
  auto seg_of = [&](int cta) { return segs[first[cta]]; };
  for (int blk = 0; blk < A.nb; ++blk)
    for (int yt = 1; yt + 1 < YT; ++yt) {
      const Seg s = seg_of(blk * YT + yt), t = seg_of(blk * YT + 1);
      if (s.ytile != yt || s.z0 != blk * A.Zb || s.nz != A.Zb || s.dir != t.dir || (up && s.dir != 1) ||
          first[blk * YT + yt + 1] - first[blk * YT + yt] != 1) {
        ++fails;
        std::printf("FAIL N %d vx %d up %d nsm %d: block %d tile %d marches %d planes from %d\n", N, vx, up, nsm, blk, yt, s.nz, s.z0);
        return;
      }
    }
}

int main() {
  const PlaneCost fp32 = {1.0, 0.0002}, u1 = {1.0, 0.002}, fp64 = {1.2, 0.009};
  for (int N : {288, 384, 432})  // two fields FP32, where the tile fills 56 to 84 % of a CTA
    check(N, 4, fp32, false, 152, true);
  for (int N : {144, 216}) check(N, 2, u1, true, 152, true);
  for (int N : {256, 512}) check(N, 4, fp32, false, 152, true);
  for (int nsm : {132, 148, 152, 160})
    for (int N = 8; N <= 512; N += 8) {
      if (!admissible(N)) continue;
      for (int vx : {1, 2, 4}) {
        if (N / vx > 512) continue;
        check(N, vx, vx == 1 ? fp64 : fp32, false, nsm, false);
        check(N, vx, u1, true, nsm, false);
      }
    }
  if (splits < 400 || aligned < 100) {
    ++fails;
    std::printf("FAIL only %d splits, %d of them aligned\n", splits, aligned);
  }
  if (!fails) std::printf("OK %d splits, %d aligned\n", splits, aligned);
  return fails != 0;
}
