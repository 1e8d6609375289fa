// df_packed_host.cpp -- host build of the packed double-float operations of
// df.cuh beside the scalar ones (test_df_packed_host.py).
#include "df.cuh"
using namespace ens::df;
extern "C" void packed_ops(int n, const double* a, const double* b, float* out) {
  // out [n][6][4]: add, add_terms, mul of (a, b): the halves of the packed pair (a, b) op (b, a), then the scalar pairs
  for (int i = 0; i < n; ++i) {
    const DF x = from_double(a[i]), y = from_double(b[i]);
    const DF2 p = pack(x, y), q = pack(y, x);
    const DF2 r[3] = {add(p, q), add_terms(p, q), mul(p, q)};
    const DF s[3][2] = {{add(x, y), add(y, x)}, {add_terms(x, y), add_terms(y, x)}, {mul(x, y), mul(y, x)}};
    for (int k = 0; k < 3; ++k) {
      DF u, v;
      unpack(r[k], &u, &v);
      float* o = out + (i * 6 + 2 * k) * 4;
      o[0] = u.hi, o[1] = u.lo, o[2] = v.hi, o[3] = v.lo;
      o[4] = s[k][0].hi, o[5] = s[k][0].lo, o[6] = s[k][1].hi, o[7] = s[k][1].lo;
    }
  }
}
