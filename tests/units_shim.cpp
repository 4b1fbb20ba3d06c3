// C entry points over layout.h's item classes and units, for test_units_host.py.
#include "layout.h"

using namespace rpt::layout;

extern "C" {

// Items of a scenario with bundle offsets off [nb + 1]: q, cnt [items]; returns their number.
int shim_items(const int* off, int nb, int* cls3, int* q, int* cnt) {
  std::vector<int4> rec(nb + 1);
  for (int k = 0; k <= nb; ++k) rec[k] = int4{off[k], 0, 0, 0};
  const ItemClasses c = item_classes(rec.data(), nb);
  cls3[0] = c.n32;
  cls3[1] = c.n16;
  cls3[2] = c.n8;
  for (int it = 0; it < c.items(); ++it) item_range(c, it, &q[it], &cnt[it]);
  return c.items();
}

// Units of N scenarios whose offsets follow each other in off (scenario s: nb[s] + 1
// of them); ubeg has room for cap entries; returns the number of units.
int shim_units(const int* off, const int* nb, int N, long long parts, int col_bytes, int* ubeg, int cap, int* uoff,
               int* widest) {
  RowLists R;
  R.rec_base.assign(N + 1, 0);
  R.nrows.assign(nb, nb + N);
  for (int s = 0; s < N; ++s) R.rec_base[s + 1] = R.rec_base[s] + nb[s] + 1;
  R.rec.resize(R.rec_base[N]);
  for (int k = 0; k < R.rec_base[N]; ++k) R.rec[k] = int4{off[k], 0, 0, 0};
  std::vector<ItemClasses> cls;
  std::vector<int> u, o;
  cut_units(R, N, parts, col_bytes, &cls, &u, &o, widest);
  if ((int)u.size() > cap) return -1;
  std::copy(u.begin(), u.end(), ubeg);
  std::copy(o.begin(), o.end(), uoff);
  return (int)u.size();
}
}
