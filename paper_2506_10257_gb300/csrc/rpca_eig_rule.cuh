// rpca_eig_rule.cuh -- when an eigen-step may stop (included inside namespace
// rpca by rpca_jacobi.cuh; plain C++ too, for tests without a GPU).
//
// A step forms Wbar = f(diag(d) + E), f(sigma^2) = min(1, tau / sigma), to first
// order in E.  What that neglects of a pair (p, q), in the entries of f:
//   both sigma above tau: f is smooth there, 3/8 E^2 / (d_p d_q) at most;
//   one above, one not: f has a kink at tau^2, where its slope jumps by
//     1 / (2 tau^2), and the divided difference over the gap d_p - d_q is off by
//     E^2 / (2 tau^2 gap) at most, which no bound on E alone limits;
//   neither: f is constant, unless the pairs together lift an eigenvalue above
//     tau^2, by w = sum of min(|E|, E^2 / gap) over the row at most: w / (2 tau^2).
//     Likewise pairs of two above tau may push the lower one below.
// The limits below keep the first under FP32's rounding (2^-24 = 6e-8) and what the
// kink adds under 5e-7, half of what the FP32 partial sums of the Gram leave unknown
// of an eigenvalue anyway.  A bound on |E| alone let 1e-4 pass beside tau; holding the
// kinks to 8e-8 as well changed no error of L or S and took up to twice as many
// further rounds (300 x 300 x 97: 280 -> 298 us a step; with these limits 277).
#pragma once
#ifdef __CUDACC__
#define RPCA_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#define RPCA_HD static inline
#endif

constexpr float kEigMaxOff = 4e-4f;   // largest |E_pq| relative to the divisor that its case above names
constexpr float kEigMaxOm = 2.4e-4f;  // largest |Omega_pq| (its square is neglected)
constexpr float kEigEps = 1e-6f;      // crossing of tau^2 that matters, relative to it; smaller |E| never does

// Whether E_pq = e >= 0 is too large in a pair that Wbar depends on: hi >= lo the
// singular values, kept how many of them are above tau (1 or 2).
RPCA_HD bool eig_pair_off(float e, float om, float hi, float lo, int kept) {
  if (om > kEigMaxOm) return true;
  if (kept == 2) return e > kEigMaxOff * hi * lo;
  return e > kEigEps * hi * hi && e * e > kEigEps * hi * hi * ((hi - lo) * (hi + lo));
}

// What an off-diagonal entry e >= 0 shifts either of two eigenvalues `gap` apart by, at most.
RPCA_HD float eig_shift(float e, float gap) { return e * e < gap * e ? e * e / gap : e; }

// What a pair of the same side of tau may shift an eigenvalue by.
RPCA_HD float eig_pair_shift(float e, float om, float hi, float lo) {
  if (om > kEigMaxOm) return e + om * om * hi * hi;
  return eig_shift(e, (hi - lo) * (hi + lo));
}

// ... without a division, no less.
RPCA_HD float eig_pair_most(float e, float om, float hi) { return om > kEigMaxOm ? e + om * om * hi * hi : e; }

// Whether a row's shifts, summed, may carry its eigenvalue s^2 across tau^2.
RPCA_HD bool eig_row_off(bool kept, float s, float shift, float tau) {
  if (!(shift > kEigEps * tau * tau)) return false;
  return kept ? s * s - shift < tau * tau : s * s + shift > tau * tau;
}
