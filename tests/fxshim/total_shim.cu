// Host-side shim over the totals of the tensor-core Gram products (fx.cuh), for
// the CPU tests.  Test infrastructure only.
#include "fx.cuh"

using namespace eo::fx;

static i128 mk(const long long* w) { return (i128)(((u128)(unsigned long long)w[1] << 64) | (unsigned long long)w[0]); }
static void put(i128 w, long long* o) {
  o[0] = (long long)(unsigned long long)(u128)w;
  o[1] = (long long)(w >> 64);
}

extern "C" {

// Sum of 2^spare totals w 2^s the way the kernel adds its parts.
void tots_sum(int spare, const long long* w, const int* s, long long* out, int* s_out) {
  i128 v[16];
  int e[16], top = -(1 << 30);
  for (int i = 0; i < 1 << spare; ++i) {
    v[i] = mk(w + 2 * i);
    e[i] = s[i];
    make_room(v[i], e[i], spare);
    top = e[i] > top ? e[i] : top;
  }
  i128 sum = 0;
  for (int i = 0; i < 1 << spare; ++i) sum += w_shift(v[i], top - e[i]);
  put(sum, out);
  *s_out = top;
}
}

extern "C" {

// m terms w + lo 2^-20, added; shifted down by sh; narrowed with room for 2^spare.
void tots_total(int m, const long long* w, const unsigned* lo, int sh, int spare, long long* out, int* s_out) {
  Total t{0, 0u};
  for (int i = 0; i < m; ++i) total_add(t, mk(w + 2 * i), lo[i]);
  total_shift(t, sh);
  int s = 0;
  put(total_narrow(t.hi, t.lo, spare, s), out);
  *s_out = s;
}
}
