// C entry point over layout.h's choice of the row pass, for test_pass_rule_host.py.
#include "layout.h"

extern "C" int shim_private_sums_pay(int accs, int exact, int value_format, long long cols_per_cta, long long width,
                                     int ring_cols) {
  return rpt::layout::private_sums_pay(accs, exact != 0, value_format, cols_per_cta, width, ring_cols) ? 1 : 0;
}
