// steps_to_switch against a search by its definition, and the verdict of the
// tuner's last turns played through the bookkeeping of one long step call.
#include "turns.h"

#include <cstdio>
#include <initializer_list>

using namespace dbn;

static int fail(const char* what, long long a, long long b, long long c) {
  std::printf("%s: %lld %lld %lld\n", what, a, b, c);
  return 1;
}

int main() {
  for (int W : {1, 2, 4, 8})
    for (int lead : {0, 1, 2, 4, 6, 9, 19, 49, 99, 250})
      for (unsigned long long g = 0; g < 4000; ++g) {
        const int64_t k = steps_to_switch(g, W - 1, lead);
        for (int64_t j = 0; j <= k; ++j) {
          const unsigned long long at = g + (unsigned long long)j;
          const bool may = at % (unsigned)W == 0 && at % (unsigned)(lead + 1) == 0;
          if (may != (j == k)) return fail("steps_to_switch", W, lead, (long long)g);
        }
      }
  // a rule that loses every turn is left, at a step where it may be, whatever
  // the bin's length; one that wins a turn stays
  for (int W : {1, 4, 8})
    for (int lead : {0, 2, 6, 9, 19, 99})
      for (int wins : {0, 1, 2, 3}) {  // the turn that it wins
        RuleVerdict v;
        if (v.is_open()) return fail("closed at first", W, lead, wins);
        v.open();
        unsigned long long g = 40ull * (unsigned)W * (unsigned)(lead + 1);
        int turns = 0;
        bool changed = false;
        while (v.is_open() && g < 100000ull) {
          if (v.leaving()) {
            const int64_t k = steps_to_switch(g, W - 1, lead);
            g += (unsigned long long)k;
            if (k > 0) continue;
            changed = true;
            v.left();
          } else if (g % (unsigned)W != 0) {
            ++g;
          } else {
            ++turns;
            v.turn(turns == wins ? 1.05 : 1.2, 1.0);
            g += 64;
          }
        }
        if (v.is_open() || changed != (wins == 0) || turns != (wins == 0 ? 3 : wins))
          return fail("verdict", W, lead, wins);
        if (changed && steps_to_switch(g, W - 1, lead) != 0) return fail("left off the edge", W, lead, (long long)g);
      }
  std::printf("ok\n");
  return 0;
}
