// Constants of a level's cells and the cell lists of the operator applies (order 2).
#pragma once
#include "cell.cuh"
#include "level.h"

namespace als {

template <typename T>
struct CellConst {
  T s[3];
  T wdet, inv_m0, inv_m1, gamma;
};

template <typename T>
inline CellConst<T> cell_const(const Geom& g, double gamma) {
  CellConst<T> c;
  double vol = 1.0;
  double wdet = 1.0;
  for (int k = 0; k < 3; ++k) {
    c.s[k] = (T)(k < g.dim ? 2.0 / g.h[k] : 0.0);
    if (k < g.dim) { vol *= g.h[k]; wdet *= 0.5 * g.h[k]; }
  }
  c.wdet = (T)wdet;
  c.inv_m0 = (T)(1.0 / vol);
  c.inv_m1 = (T)(3.0 / vol);
  c.gamma = (T)gamma;
  return c;
}

// cells of one colour: index t -> (step i + bx, step j + by, step k + bz);
// step 2 selects one parity class, step 1 (bits 0) all cells
struct Colour {
  int b[3];      // parity bits
  int m[3];      // cells of this colour per axis
  int step;
  long long count;
};

inline Colour all_cells(const Geom& g) {
  Colour c{};
  c.step = 1;
  c.count = g.ncells;
  for (int k = 0; k < 3; ++k) { c.b[k] = 0; c.m[k] = g.n[k]; }
  return c;
}

inline Colour make_colour(const Geom& g, int colour) {
  Colour c{};
  c.step = 2;
  c.count = 1;
  for (int k = 0; k < 3; ++k) {
    c.b[k] = (k < g.dim) ? (colour >> k) & 1 : 0;
    c.m[k] = (k < g.dim) ? (g.n[k] - c.b[k] + 1) / 2 : 1;
    c.count *= c.m[k];
  }
  return c;
}

// 32-bit arithmetic: cell counts stay below 2^31 (checked when a context is created)
__device__ __forceinline__ bool colour_cell(const Colour& col, long long t, int& cx, int& cy, int& cz) {
  if (t >= col.count) return false;
  const unsigned tu = (unsigned)t, m0 = (unsigned)col.m[0], m1 = (unsigned)col.m[1];
  const unsigned r = tu / m0;
  const int i = (int)(tu - r * m0);
  const unsigned k = r / m1;
  const int j = (int)(r - k * m1);
  cx = col.step * i + col.b[0];
  cy = col.step * j + col.b[1];
  cz = col.step * k + col.b[2];
  return true;
}

}  // namespace als
