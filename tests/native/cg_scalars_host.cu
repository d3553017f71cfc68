// Host entry points over the CG scalars' integer arithmetic (csrc/pcg_scalar.cuh), for the CPU
// tests: the same functions the CG kernels run on the device, compiled for the host.
#include "pcg_scalar.cuh"

extern "C" {
// One step of the recurrence from gamma_old, den_old and this iteration's gamma and delta.
void sch_step(double gamma_old, double den_old, double gamma, double delta, double* alpha, double* beta) {
  ccm::CgState st{ccm::cg_inverse(ccm::sc_of_double(gamma_old)), ccm::sc_of_double(den_old)};
  ccm::cg_scalars(ccm::sc_of_double(gamma), ccm::sc_of_double(delta), st, *alpha, *beta);
}

// The value of digit sums S[0..4] in the window of bottom 2^lo, rounded to FP64.
double sch_digits(const long long* S, int lo) { return ccm::sc_double(ccm::sc_of_digits(S, lo)); }
}
