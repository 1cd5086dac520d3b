// Replays calls through the library's PartialSets: input lines "workspace layout"
// (decimal), output lines "set fresh".
#include <cstdio>

#include "sdv_sets.h"

int main() {
  static sdv::PartialSets sets;
  unsigned long long ws, layout;
  while (std::scanf("%llu %llu", &ws, &layout) == 2) {
    bool fresh = false;
    const int set = sets.next(reinterpret_cast<const void*>((uintptr_t)ws), layout, &fresh);
    std::printf("%d %d\n", set, (int)fresh);
  }
  return 0;
}
