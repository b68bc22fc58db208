// Host build of the backward recurrence (csrc/hankel.cuh) for test_recurrence_start_cpu.py:
// one lane, its start from a table.
#include <cmath>

static inline unsigned __activemask() { return 1u; }
static inline int __reduce_max_sync(unsigned, int v) { return v; }

#include "../paper_2203_13283_gb300/csrc/hankel.cuh"

// out: J0, J1, Y0, Y1 at x, the recurrence started where the table says
extern "C" void recurrence_from(double x, int tabulated, double* out) {
  const wcs::Bessel01 b = wcs::bessel01_miller_real<true>(x, tabulated);
  out[0] = b.J0;
  out[1] = b.J1;
  out[2] = b.Y0;
  out[3] = b.Y1;
}

extern "C" int recurrence_start(double x) { return wcs::miller_start(x); }
