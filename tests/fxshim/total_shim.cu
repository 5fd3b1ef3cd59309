// Host-side shim over the scale of the tensor-core Gram products' totals
// (fx.cuh), for the CPU tests.  Test infrastructure only.
#include "fx.cuh"

extern "C" int tots_fold_bits(unsigned rows) { return eo::fx::fold_bits(rows); }
