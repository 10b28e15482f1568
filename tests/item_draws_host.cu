// Host simulation of the blocks of one launch that draw their items from a
// counter (Draws): blocks run in a random order, and some give up at either of
// an item's two barriers.  Every item is taken at most once (exactly once when
// no block gives up), and the counter is zero again at the end.
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2604_02624_gb300/csrc/dos_pass_bulk.cuh"

using dos::Draws;

struct Block {
  Draws d;
  unsigned it;
  bool live;
};

static bool launch(unsigned blocks, unsigned items, double fail, unsigned* work, std::mt19937& rng) {
  std::vector<Block> b;
  std::vector<int> taken(items, 0);
  for (unsigned i = 0; i < blocks; ++i) {
    b.push_back({{work, blocks, items, 0u}, i, true});
    b[i].d.ahead();
  }
  std::uniform_real_distribution<double> u(0.0, 1.0);
  unsigned live = blocks;
  bool any = false;
  while (live) {
    Block& x = b[rng() % blocks];
    if (!x.live) continue;
    const unsigned next = x.d.item();
    if (u(rng) < fail) {  // at the first barrier: the published item is the latest number's
      x.d.drain(next);
      x.live = false, --live, any = true;
      continue;
    }
    if (next < items) x.d.ahead();
    if (u(rng) < fail) {  // at the second: another number has been drawn
      x.d.drain(next < items ? x.d.item() : next);
      x.live = false, --live, any = true;
      continue;
    }
    if (++taken[x.it] > 1) return false;
    x.it = next;
    if (next >= items) x.live = false, --live;
  }
  if (!any)
    for (int t : taken)
      if (t != 1) return false;
  return *work == 0u;
}

int main() {
  std::mt19937 rng(1);
  unsigned work = 0;
  int bad = 0;
  for (int rep = 0; rep < 3000; ++rep) {
    const unsigned items = 1 + rng() % 300;
    const unsigned blocks = 1 + rng() % items;
    const double fails[4] = {0.0, 0.01, 0.2, 1.0};
    if (!launch(blocks, items, fails[rep % 4], &work, rng)) ++bad, work = 0;
  }
  std::printf(bad ? "%d bad\n" : "OK\n", bad);
  return bad != 0;
}
