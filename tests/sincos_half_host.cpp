// sincos2pi_half (csrc/sincos_fx.cuh) beside sincos2pi_fx, for the host test
#include "sincos_fx.cuh"

extern "C" void sincos_halves(long n, const double* x, double* both, double* halves) {
  for (long i = 0; i < n; ++i) {
    ens::sincos2pi_fx(x[i], both + 2 * i, both + 2 * i + 1);
    bool s0, s1;
    const double p = ens::sincos2pi_half<true>(x[i], &s0), q = ens::sincos2pi_half<false>(x[i], &s1);
    halves[2 * i + (s0 ? 0 : 1)] = p;
    halves[2 * i + (s1 ? 0 : 1)] = q;
  }
}
