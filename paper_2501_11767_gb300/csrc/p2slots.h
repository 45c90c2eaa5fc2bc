// Node types, stencil slots and grid-transfer weights of the P2 lattice
// (device side; see p2stencil.h for the layout).
#pragma once

#include "p2stencil.h"

namespace chnss {

// node type of lattice parity: 0 vertex, 1 horizontal, 2 vertical, 3 diagonal edge midpoint
__host__ __device__ constexpr int type_of(int pi, int pj) { return (pi & 1) + 2 * (pj & 1); }

// couplings of the four node types, in CSR (ascending lattice) order
__host__ __device__ constexpr int slot_base(int ty) { return ty == 0 ? 0 : 10 + 9 * ty; }
__host__ __device__ constexpr int slot_count(int ty) { return ty == 0 ? 19 : 9; }
struct SlotTable {
  signed char di[kP2Slots], dj[kP2Slots];
};
__host__ __device__ constexpr SlotTable slot_table() {
  return {{-2, -1, 0, -2, -1, 0, 1, -2, -1, 0, 1, 2, -1, 0, 1, 2, 0, 1, 2,   // vertex
           -1, -1, 0, -1, 0, 1, 0, 1, 1,                                     // horizontal edge
           -2, -1, 0, -1, 0, 1, 0, 1, 2,                                     // vertical edge
           -1, 0, 1, -1, 0, 1, -1, 0, 1},                                    // diagonal edge
          {-2, -2, -2, -1, -1, -1, -1, 0, 0, 0, 0, 0, 1, 1, 1, 1, 2, 2, 2,
           -2, -1, -1, 0, 0, 0, 1, 1, 2,
           -1, -1, -1, 0, 0, 0, 1, 1, 1,
           -1, -1, -1, 0, 0, 0, 1, 1, 1}};
}

// prescribed velocity at lattice point (I, J) of an m x m lattice (or outside it)
__device__ __forceinline__ bool prescribed(int I, int J, int m, int open) {
  return I <= 0 || J <= 0 || I >= m - 1 || (open ? J >= m : J >= m - 1);
}

// Weight at fine lattice point (I, J) of the quadratic function of coarse
// lattice node (ci, cj) (fine lattice twice as dense; I, J, ci, cj >= 0): an
// exact dyadic number, 0 outside the function's support.
__host__ __device__ constexpr double p2_weight(int I, int J, int ci, int cj) {
  const int i = I / 4, j = J / 4;
  const double xi = I / 4.0 - i, eta = J / 4.0 - j;
  const bool lower = xi >= eta;
  const double l0 = lower ? 1 - xi : 1 - eta, l1 = lower ? xi - eta : xi, l2 = lower ? eta : eta - xi;
  const int x1 = i + 1, y1 = lower ? j : j + 1, x2 = lower ? i + 1 : i, y2 = j + 1;
  if (ci == 2 * i && cj == 2 * j) return l0 * (2 * l0 - 1);
  if (ci == 2 * x1 && cj == 2 * y1) return l1 * (2 * l1 - 1);
  if (ci == 2 * x2 && cj == 2 * y2) return l2 * (2 * l2 - 1);
  if (ci == x1 + x2 && cj == y1 + y2) return 4 * l1 * l2;
  if (ci == i + x2 && cj == j + y2) return 4 * l0 * l2;
  if (ci == i + x1 && cj == j + y1) return 4 * l0 * l1;
  return 0.0;
}

// Restriction to a coarse node of each type: fine offsets from twice its
// lattice point, ascending.  Prolongation to the fine nodes of each class
// (I mod 4) + 4 (J mod 4): coarse offsets from (2 (I / 4), 2 (J / 4)), ascending.
struct P2Transfers {
  int rn[4] = {}, pn[16] = {};
  signed char ri[4][25] = {}, rj[4][25] = {}, pi[16][6] = {}, pj[16][6] = {};
  float rw[4][25] = {}, pw[16][6] = {};
};
__host__ __device__ constexpr P2Transfers p2_transfers() {
  P2Transfers t;
  for (int ty = 0; ty < 4; ++ty) {
    const int ci = 4 + (ty & 1), cj = 4 + (ty >> 1);
    for (int dj = -3; dj <= 3; ++dj)
      for (int di = -3; di <= 3; ++di) {
        const double w = p2_weight(2 * ci + di, 2 * cj + dj, ci, cj);
        if (w == 0.0) continue;
        const int k = t.rn[ty]++;
        t.ri[ty][k] = (signed char)di;
        t.rj[ty][k] = (signed char)dj;
        t.rw[ty][k] = (float)w;
      }
  }
  for (int c = 0; c < 16; ++c)
    for (int dj = 0; dj <= 2; ++dj)
      for (int di = 0; di <= 2; ++di) {
        const double w = p2_weight(4 + (c & 3), 4 + (c >> 2), 2 + di, 2 + dj);
        if (w == 0.0) continue;
        const int k = t.pn[c]++;
        t.pi[c][k] = (signed char)di;
        t.pj[c][k] = (signed char)dj;
        t.pw[c][k] = (float)w;
      }
  return t;
}

}  // namespace chnss
