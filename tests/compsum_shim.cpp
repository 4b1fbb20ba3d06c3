// C entry points over compsum.h for test_compsum_host.py.
#include "compsum.h"

extern "C" double shim_compsum(const float* p, int n) {
  rpt::CompSum s;
  for (int k = 0; k < n; ++k) s.add(p[k]);
  return s.value();
}
