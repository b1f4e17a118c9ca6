// Host check of pol_plan.h: for every number of chunks, unit count and tuning value, the segments cover the
// chunks once, none is empty and none is longer than allowed.
#include <cstdio>
#include <initializer_list>

#include "pol_plan.h"

int main() {
  long checked = 0, bad = 0;
  for (int sms : {132, 148, 152, 160})
    for (int seg_chunks : {1, 3, 8, 31, 32})
      for (int base_units : {1, 2, 8, 16, 24, 32, 48, 64, 72, 96, 128, 151, 152, 256, 304, 1536})
        for (int total = 1; total <= 8192; total += total < 1024 ? 1 : 37) {
          const int n = gwi::pol_segments(total, base_units, seg_chunks, sms), len = gwi::pol_seg_len(total, n);
          const bool ok = n >= 1 && len >= 1 && len <= seg_chunks && (long)(n - 1) * len < total && (long)n * len >= total;
          ++checked;
          if (!ok && bad++ < 10)
            std::printf("total %d base_units %d seg_chunks %d sms %d: %d segments of %d\n", total, base_units, seg_chunks, sms, n, len);
        }
  std::printf("%ld plans, %ld with an empty or overlong segment\n", checked, bad);
  return bad != 0;
}
