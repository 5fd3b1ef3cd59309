// Host-side shim over the FP32 rounding of exact sums (fx.cuh), for the CPU
// tests.  Test infrastructure only.
#include "fx.cuh"

using namespace eo::fx;

extern "C" float flt_w_to_float(long long lo, long long hi, int S) {
  return w_to_float((i128)(((u128)(unsigned long long)hi << 64) | (unsigned long long)lo), S);
}
