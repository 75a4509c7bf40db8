// pa_regions.h -- host arithmetic of the image metrics' regions (plain C++, no
// device code, so that it can be compiled and checked by itself).
#pragma once

#include <algorithm>

#include "pa_hodmas.h"

namespace pa {

// At least the members of a region whose pixels lie in a box of width x rows
// pixels of dx x dz: that box, or for a round region (`inside`: its box lies
// within the image) its area in pixels and half a boundary pixel at each end of
// every column: with f the chord over a column, unimodal, the sum of f over the
// columns differs from its integral by its maximum at most, and the rows in a
// chord from its length by one.
inline long long most_members(int shape, double a, double b, int width, int rows, bool inside,
                              double dx, double dz) {
  const long long box = (long long)width * rows;
  if (shape == PA_REGION_RECT || !inside) return box;
  const bool hole = shape == PA_REGION_ANNULUS;
  const double out = hole ? b : a, in = hole ? std::min(a, b) : 0.0;
  const double n = 3.1416 * out * out / (dx * dz) - 3.1415 * in * in / (dx * dz) +
                   2.0 * (out + in) / dz + 2.0 * width + 16.0;
  return n < (double)box ? (long long)n : box;
}

}  // namespace pa
