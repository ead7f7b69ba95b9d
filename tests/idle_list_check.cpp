// IdleList against a plain account of what is alive: objects taken, given back and
// destroyed by owners in a random order.  None is given to another owner or lost:
// each is idle in the list, in use, or was handed out for destruction once, to a
// caller of its own owner.  Prints the number of violations.
#include <cstdio>
#include <map>
#include <random>
#include <set>
#include <vector>

#include "idle_list.h"

struct Key {
  int ctx, shape;
  bool operator==(const Key& k) const { return ctx == k.ctx && shape == k.shape; }
};

int main() {
  long bad = 0;
  for (int seed = 0; seed < 200; ++seed) {
    std::mt19937 rng(seed);
    flame::IdleList<Key, int, 8> list;
    std::map<int, Key> alive;  // object -> its key
    std::set<int> idle;
    std::vector<int> used;
    int next = 0;
    for (int step = 0; step < 400; ++step) {
      if (rng() % 2) {
        const Key k{(int)(rng() % (1 + seed % 3)), (int)(rng() % 5)};
        int o = -1;
        if (list.take(k, &o)) {
          if (!idle.erase(o) || !(alive.at(o) == k)) ++bad;
        } else {
          for (int i : idle)
            if (alive.at(i) == k) ++bad;  // there was one
          o = next++;
          alive[o] = k;
        }
        used.push_back(o);
      } else if (!used.empty()) {
        const int i = (int)(rng() % used.size()), o = used[i], ctx = alive.at(o).ctx;
        used.erase(used.begin() + i);
        idle.insert(o);
        int drop = -1;
        if (list.give(alive.at(o), o, &drop)) {
          if (!idle.erase(drop) || alive.at(drop).ctx != ctx) ++bad;
          alive.erase(drop);
        }
      }
      if (list.size() > 8 || list.size() != (int)idle.size() || alive.size() != idle.size() + used.size()) ++bad;
    }
  }
  std::printf("bad %ld\n", bad);
  return bad != 0;
}
