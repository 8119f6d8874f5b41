// band.cuh -- the binary32 band around the cutoff in which the pair test is
// decided exactly in binary64 (host code; its users are in kernels.cuh).
#pragma once
#include <cmath>

namespace mtpt {

struct PairBand {
    float lo;       // binary32 d2 below this: certainly a neighbour
    float hi;       // binary32 d2 above this: certainly not a neighbour
    float reach2;   // hi (1 + 2^-16)
};

// The band of half-width eta psi2 around psi2, rounded outwards.  Neither bound has
// a sign bit or is a NaN, whatever the parameters: the searches compare them with
// squared distances by their bits.  In boxes so sparse, or so far from the origin,
// that the half-width passes psi2 (cells some 1e5 psi wide), lo is +0 and every
// candidate below hi gets the exact test.
inline PairBand pair_band(double psi2, double eta) {
    PairBand b;
    const float lo = float(psi2 * (1.0 - eta));
    const double hi = psi2 * (1.0 + eta);       // (0 times infinity where psi2 underflows)
    b.lo = lo > 0.0f ? std::nextafter(lo, 0.0f) : 0.0f;
    b.hi = std::isnan(hi) ? INFINITY : std::nextafter(float(hi), INFINITY);
    b.reach2 = std::nextafter(float(double(b.hi) * (1.0 + std::ldexp(1.0, -16))), INFINITY);
    return b;
}

}  // namespace mtpt
