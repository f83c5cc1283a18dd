// EdgeSet against std::unordered_set on a random sequence of insertions,
// removals and look-ups with many collisions; exit code 0 when all agree.
#include <random>
#include <unordered_set>

#include "edge_set.h"

int main() {
  std::mt19937_64 r(1);
  sr::EdgeSet a;
  std::unordered_set<uint64_t> b;
  for (int i = 0; i < 400000; ++i) {
    const uint64_t k = ((r() % 300) << 32) | (r() % 20);
    switch (r() % 3) {
      case 0:
        if (a.insert(k) != b.insert(k).second) return 1;
        break;
      case 1:
        if (a.erase(k) != (b.erase(k) > 0)) return 2;
        break;
      default:
        if (a.contains(k) != (b.count(k) > 0)) return 3;
    }
    if (a.size() != b.size()) return 4;
    if (i == 200000) a.reserve(50000);
  }
  for (uint64_t k : b)
    if (!a.contains(k)) return 5;
  return 0;
}
