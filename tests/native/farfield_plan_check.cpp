// Workspace plans of the far-field sums: prints one line per (lattice, SM count)
// with the largest number of bytes by which the launches for any smaller count
// of directions would pass a region of the plan they run in, and the whole
// workspace (0: none does), and by which the partial sums pass 64 MB.
#include <algorithm>
#include <cstdio>

#include "farfield_plan.h"

using namespace dda;

int main() {
  const int lat[][3] = {{1, 1, 1},    {4, 40, 40},    {40, 40, 40},  {48, 48, 48},    {64, 64, 64},
                        {6, 70, 70},  {145, 30, 17},  {128, 128, 128}, {256, 256, 256}, {536, 536, 536},
                        {300, 1, 300}};
  const int sms[] = {1, 76, 148, 152, 160};
  const int cap = 8192;
  for (const auto& l : lat)
    for (int sm : sms) {
      const int nr = l[1] * l[2];
      const FarfieldPlan p = farfield_plan(cap, l[0], l[1], l[2], nr, sm);
      long long over = 0;
      for (int nd = 1; nd <= cap; ++nd) {
        const size_t tab = ff_tab_bytes(nd, l[0], l[1], l[2]), pack = ff_pack_bytes(nd, l[0]),
                     part = ff_part_bytes(nd, p.groups);
        over = std::max({over, (long long)tab - (long long)p.tab, (long long)pack - (long long)p.pack,
                         (long long)part - (long long)p.part,
                         (long long)(p.tab + p.pack + part) - (long long)p.bytes()});
      }
      const long long big = std::max(0LL, (long long)ff_part_bytes(cap, p.groups) - (64LL << 20));
      const int ok = p.groups >= 1 && p.groups <= ff_units(ff_shape(l[0]), nr) && p.tab % 256 == 0 && p.pack % 256 == 0;
      std::printf("%dx%dx%d %d %lld %lld %d\n", l[0], l[1], l[2], sm, std::max(0LL, over), big, ok);
    }
  return 0;
}
