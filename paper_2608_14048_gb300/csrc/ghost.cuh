// Ghost cells of a block in one pass (Sec. 2.3): the cells of the padded array
// outside the interior, linearly numbered, and the interior cell each one
// copies.  Filling axis after axis (x, then y from the x-filled rows, then z)
// gives every ghost the interior value that the three axis maps lead to, so the
// composite map fills edges and corners in the same launch, with no order
// between the cells: sources are never ghosts.
//
// One launch instead of three: a shell 2g + 1 cells thick is bound by latency
// and by the launches themselves.  us a fill, three launches -> one: 32^3 16.5
// -> 4.0 (a step, with the CFL minimum in its pass, 67.7 -> 47.3), 512 uneven
// boxes 603 -> 365.
#pragma once
#include "runtime.hpp"

namespace aeth {

// Ghost cell number el of layout L (z layers, then y rows, then x columns).
// Indices run from -g to n + g; index n (face n's place) counts as ghost.
__device__ __forceinline__ void ghost_cell(const Layout& L, unsigned el, int* c) {
  const unsigned g = L.g, T = 2 * g + 1;
  const unsigned X = L.n[0] + T, Y = L.n[1] + T;
  // layer t of an axis of n cells: -g .. -1, n .. n + g
  auto layer = [&](unsigned t, int n) { return t < g ? (int)t - (int)g : n + (int)(t - g); };
  const unsigned nz = T * X * Y;
  if (el < nz) {
    const unsigned r = el / X;
    c[0] = (int)(el - r * X) - (int)g;
    c[1] = (int)(r % Y) - (int)g;
    c[2] = layer(r / Y, L.n[2]);
    return;
  }
  el -= nz;
  const unsigned ny = (unsigned)L.n[2] * T * X;
  if (el < ny) {
    const unsigned r = el / X;
    c[0] = (int)(el - r * X) - (int)g;
    c[1] = layer(r % T, L.n[1]);
    c[2] = (int)(r / T);
    return;
  }
  el -= ny;
  const unsigned r = el / T;
  c[0] = layer(el - r * T, L.n[0]);
  c[1] = (int)(r % (unsigned)L.n[1]);
  c[2] = (int)(r / (unsigned)L.n[1]);
}

// Axis e of the map of an unlinked side: the interior cell that cell index p
// copies; up: an outflow side's upper ghosts, where the face arrays of that
// axis copy face n, one above the cell.
__device__ __forceinline__ int ghost_axis(const Layout& L, int e, int p, bool& up) {
  const int n = L.n[e];
  up = false;
  if (p >= 0 && p < n) return p;
  if (L.bc[e] == AETH_BC_PERIODIC) return ((p % n) + n) % n;
  up = p >= n;
  return p < 0 ? 0 : n - 1;
}

}  // namespace aeth
