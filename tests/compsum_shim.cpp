// C entry points over compsum.h for test_compsum_host.py.
#include "compsum.h"

extern "C" double shim_compsum(const float* p, int n) {
  rpt::CompSum s;
  for (int k = 0; k < n; ++k) s.add(p[k]);
  return s.value();
}

// The same numbers dealt to `parts` sums, which are then added up pair by pair.
extern "C" double shim_compsum_parts(const float* p, int n, int parts) {
  rpt::CompSum s[64];
  for (int k = 0; k < n; ++k) s[k % parts].add(p[k]);
  for (int d = 1; d < parts; d *= 2)
    for (int i = 0; i + d < parts; i += 2 * d) s[i].add(s[i + d]);
  return s[0].value();
}
