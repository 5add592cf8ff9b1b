// Host check of the tensor-core Gram's split (csrc/internal.h): with a buffer of any size a CTA never
// gets more chunks than its 64-bit sums have room for; where the buffer is too small for that there is
// no split.  Prints "ok".
#include "internal.h"

#include <cstdio>

int main() {
  using namespace pbs;
  const int sides[] = {4, 6, 30, 34, 208, 1024, 4096, 16384};
  for (int n : sides)
    for (int m : sides)
      for (int want : {1, 7, 304, 608, 5000})
        for (long fit : {-3L, 0L, 1L, 2L, 15L, 16L, 511L, 100000L}) {
          const int np = gram_tc_npart(n, m, want, fit);
          const long chunks = gram_tc_chunks(n, m), most = fit < want ? fit : want;
          const bool enough = most >= 1 && (chunks + most - 1) / most <= kGramTcRoom;
          if (chunks * 256 < (long)n * m || np != (enough ? most : 0)) {
            std::printf("%d x %d, %d wanted, %ld fit: %d\n", n, m, want, fit, np);
            return 1;
          }
        }
  std::puts("ok");
}
