// Host-side check of granted_tile (mbar.cuh): what a CTA makes of an answer to
// its request for another tile that comes in time, late, or not at all.  Prints
// "cases N bad B".
#include <cstdio>

#include "../paper_2504_19410_gb300/csrc/mbar.cuh"

int main() {
  int cases = 0, bad = 0;
  // arrives: the wait at which the answer is there (3: neither); tile: what it grants (-1: nothing)
  for (int arrives = 1; arrives <= 3; ++arrives)
    for (int tile : {-1, 0, 7}) {
      int waits = 0, reads = 0, lates = 0;
      const int next = fsa::granted_tile([&] { return ++waits >= arrives; },
                                         [&] {
                                           ++reads;
                                           return tile;
                                         },
                                         [&] { ++lates; });
      const int want = arrives <= 2 ? tile : -1;
      ++cases;
      if (next != want || waits != (arrives == 1 ? 1 : 2) || reads != (arrives <= 2) || lates != (arrives > 1)) ++bad;
    }
  std::printf("cases %d bad %d\n", cases, bad);
  return bad != 0;
}
