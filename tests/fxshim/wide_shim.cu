// Host-side shim over the wide floating-point arithmetic (wide.cuh) of the
// k-by-k steps, for the CPU tests.  Test infrastructure only.
#include "wide.cuh"

using namespace eo::fx;

namespace {
wide get(const unsigned long long* w) { return wide{((u128)w[0] << 64) | w[1], (int)(long long)w[2], (int)w[3]}; }
void put(wide a, unsigned long long* w) {
  w[0] = (unsigned long long)(a.m >> 64);
  w[1] = (unsigned long long)a.m;
  w[2] = (unsigned long long)(long long)a.e;
  w[3] = (unsigned long long)a.s;
}
}  // namespace

extern "C" {
// op: 0 add, 1 sub, 2 mul, 3 dot2 (a b + c d), 4 recip, 5 rsqrt, 6 sqrt
void wides_op(int op, const unsigned long long* a, const unsigned long long* b, const unsigned long long* c,
              const unsigned long long* d, unsigned long long* r) {
  const wide x = get(a), y = get(b);
  switch (op) {
    case 0: put(wide_add(x, y), r); break;
    case 1: put(wide_sub(x, y), r); break;
    case 2: put(wide_mul(x, y), r); break;
    case 3: put(wide_dot2(x, y, get(c), get(d)), r); break;
    case 4: put(wide_recip(x), r); break;
    case 5: put(wide_rsqrt(x), r); break;
    default: put(wide_sqrt(x), r); break;
  }
}
void wides_from(double hi, double lo, unsigned long long* r) { put(wide_from(hi, lo), r); }
void wides_to(const unsigned long long* a, double* hi, double* lo) { wide_to_dd(get(a), *hi, *lo); }
}
