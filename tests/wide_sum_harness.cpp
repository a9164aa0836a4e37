// Host harness for the limb sums and the fast conversion of the dataflow
// iterations' totals (cgp_fixed.h): reads lines "E lo hi" of up to 32 integers
// (hex halves; E the exponent of the group) ended by an empty group marker
// "S", and prints for every group the limb sum's halves, the fast conversion's
// bits and the general one's.  Exit status 3: a block's word did not give its sum
// or exponent back; 4: its tag did not tell the reduction from another.
#include <cstdio>
#include <vector>

#include "cgp_fixed.h"

using namespace cgp::fx;

int main() {
  char tag[8];
  int E = 1;
  unsigned s[kLimbs] = {0, 0, 0, 0, 0};
  unsigned long long lo, hi;
  while (std::scanf("%7s", tag) == 1) {
    if (tag[0] == 'E') {
      if (std::scanf("%d", &E) != 1) return 1;
      for (unsigned& v : s) v = 0;
    } else if (tag[0] == 'X') {
      if (std::scanf("%llx %llx", &lo, &hi) != 2) return 1;
      const I128 x = ((I128)(long long)hi << 64) | (I128)lo;
      for (int i = 0; i < kLimbs; ++i) s[i] += limb(x, i);   // 32 limbs of 27 bits: no carry out of 32 bits
    } else {
      const I128 v = limbs_value(s);
      if (v < ((I128)1 << 115) && v >= -((I128)1 << 115)) {   // a block's partial through its word
        uint64_t wl, wh;
        for (int red : {0, 1, 2046, 2047, 2048, 1 << 30}) {
          pack_word(v, E, red, wl, wh);
          if (word_sum(wl, wh) != v >> kWordShift || word_exponent(wh) != E) return 3;
          if (!word_current(wh, red) || word_current(wh, red + 2) || word_current(0, red)) return 4;
        }
      }
      std::printf("%016llx %016llx %016llx %016llx\n", (unsigned long long)v, (unsigned long long)(v >> 64),
                  (unsigned long long)dbits(to_double_normal(v, E)), (unsigned long long)dbits(to_double(v, E)));
    }
  }
  return 0;
}
