// Test probe: reads lines "<items> <partners> <sms>", prints pick_split and pick_split_small of each.
#include <cstdio>

#include "tc_setup.hpp"

int main() {
  int items = 0, partners = 0, sms = 0;
  while (std::scanf("%d %d %d", &items, &partners, &sms) == 3)
    std::printf("%d %d\n", tc::pick_split(items, partners, sms), tc::pick_split_small(items, partners, sms));
  return 0;
}
