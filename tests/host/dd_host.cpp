// The double-double fraction and its 128-bit fixed point, on the host.
#include "emri_common.cuh"

extern "C" void frac_fx128(double hi, double lo, unsigned long long* out) {
  emri::dd_to_fx128(emri::dd_frac(emri::dd{hi, lo}), out[0], out[1]);
}
