// character.h -- characters of one-dimensional irreps as pairs of doubles; host code.
#pragma once
#include <cmath>
#include <cstdint>

// (c, s) = exp(2 pi i num / denom) within 1.1e-16 per part.  cos and sin of the double nearest to
// 2 pi num / denom carry the rounding of that angle: 1.9e-16 at 2 pi / 3, as much as a whole row's
// sum, and coset arithmetic multiplies a term by two characters.  The angle is taken to the first
// octant in integers; there its rounding, a_lo, enters in first order.
inline void ed_character(int64_t num, int64_t denom, double *c, double *s) {
  const int64_t q = (num % denom + denom) % denom, oct = 8 * q / denom;
  int64_t rem = 8 * q - oct * denom;             // of an octant, in parts of denom
  if (oct & 1) rem = denom - rem;                // from the octant's other end
  const double p_hi = 0.78539816339744828, p_lo = 3.0616169978683830e-17;   // pi / 4
  const double r = (double)rem, d = (double)denom, m = p_hi * r, a = m / d;
  const double a_lo = (std::fma(-a, d, m) + std::fma(p_hi, r, -m) + p_lo * r) / d;
  const double ca = std::cos(a), sa = std::sin(a);
  const double x = std::fma(-a_lo, sa, ca), y = std::fma(a_lo, ca, sa);
  const bool swap = ((oct + 1) & 2) != 0;        // octants 1, 2, 5, 6: nearest to the imaginary axis
  const double u = swap ? y : x, v = swap ? x : y;
  *c = oct >= 2 && oct < 6 ? -u : u;
  *s = oct >= 4 ? -v : v;
}
