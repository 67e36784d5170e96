// Host check of the column solve's scratch: for every size that the
// allocation-free entry point accepts (n_cols * (nlev + 1) up to its limit), the
// whole groups of columns that the solve addresses fit the static array.  The
// spare columns of a group count most just above a multiple of it and where the
// form changes, so every n_cols is tried.
#include <cstdio>

#include "internal.h"

int main() {
  const size_t limit = 1047232;
  size_t sizes = 0;
  for (int nlev = 2; nlev <= 256; ++nlev)
    for (size_t n = 1; n * (nlev + 1) <= limit; ++n, ++sizes)
      if (icon::scratch_points((int)n, nlev) > limit || icon::scratch_points((int)n, nlev) < n * nlev) {
        std::printf("n_cols %zu nlev %d\n", n, nlev);
        return 1;
      }
  std::printf("ok %zu\n", sizes);
  return 0;
}
