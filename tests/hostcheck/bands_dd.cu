// Host entry to the digit form's rounding (signed160_to_dd in bigfloat.cuh):
// six two's complement words of V and the scale s give the dd nearest to
// V 2^s, as the recombination kernel calls it.  Built as a shared library for
// the CPU test.
#include <cstdint>

#include "bigfloat.cuh"

extern "C" void bands_to_dd(const uint32_t *z, int s, double *out) {
    uint32_t w[6];
    for (int t = 0; t < 6; ++t) w[t] = z[t];
    mpdd::bigf::signed160_to_dd(w, s, out[0], out[1]);
}
