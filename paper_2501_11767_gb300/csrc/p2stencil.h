// The P2 velocity operator of the structured meshes as a stencil over cells.
//
// Node types on the once-refined lattice, per cell (i, j), 0 <= i, j <= n:
// vertices (2i, 2j) with 19 couplings, and the midpoints of horizontal
// (2i + 1, 2j), vertical (2i, 2j + 1) and diagonal (2i + 1, 2j + 1) edges with
// 9 each; kDI / kDJ list them in CSR order (46 slots a cell).  Every 2x2 block
// is s I + eta K_ab: mass and convection act on both components alike, so its
// off-diagonal entries come from the symmetric gradient alone and are the
// same for every node of a type (twice over: the open top's nodes see only
// the elements below them).  A level therefore stores the two diagonal values
// of each block, at slot * ld + cell, and a table of the off-diagonal ones;
// columns follow from the cell.  Rows and columns of nodes with prescribed
// velocity are the identity's and need no values.  A fine sweep moves 92
// bytes of matrix per node in FP32 where the 2x2-block SELL moves 230.
#pragma once

#include "kernels.h"

namespace chnss {

constexpr int kP2Slots = 46;
constexpr int kP2TopSlots = 28;                  // vertex and horizontal slots of the open top's rows

// off-diagonal entries (0,1) and (1,0) by slot; rows on an open top from kP2Slots on
struct P2Table {
  double c[2 * (kP2Slots + kP2TopSlots)];
  // device copies: rounded to FP32, rounded to BF16 (as FP32)
  const float *d32 = nullptr, *d16 = nullptr;
  bool ok = false;                               // every row of the level matches it
  bool seen[kP2Slots + kP2TopSlots] = {};        // the level couples two free nodes by the slot (else: zeros)
  // o's entries hold for this level as well: equal wherever it has the coupling
  bool holds(const P2Table &o) const {
    for (int k = 0; k < kP2Slots + kP2TopSlots; ++k)
      if (seen[k] && !(o.seen[k] && o.c[2 * k] == c[2 * k] && o.c[2 * k + 1] == c[2 * k + 1])) return false;
    return true;
  }
};

inline long p2_ld(int n) { return ((long)(n + 1) * (n + 1) + 31) / 32 * 32; }
inline long p2_values_count(int n) { return 2 * kP2Slots * p2_ld(n); }   // scalars

// Whether a level of table t takes the stencil for values of value_size
// bytes: in FP32 and BF16 (384^2: fine level 31.0 -> 18.0 us a sweep, 192^2
// level 12.1 -> 10.9, coarser ones 6.1 -> 4.4-5.1).  FP64 sweeps stay on the
// 2x2-block SELL: they keep the FP64 pipe 73 % (256^2) and 64 % (128^2) busy at
// 40 and 24 % of HBM, so saved bytes buy little, and the stencil's fewer,
// longer threads keep it less busy (FP64 steps with the stencil from 241^2 on
// against SELL: 512^2 137 and 131 ms, 768^2 287 and 267, 1024^2 497 and 460; a
// sweep of 128^2 18.7 and 16.5 us).
bool p2_applies(const P2Table &t, size_t value_size);
// Table of the level's constant blocks A (CSR order, 4 values each) and
// whether all its rows match it (synchronises s); device copies from keep.
P2Table p2_table(Arena &keep, const Level &L, int open_top, const double *A, cudaStream_t s);
// Diagonal values of A in stencil order
template <typename VT>
void p2_values(const Level &L, int open_top, const double *A, VT *out, cudaStream_t s);

// How a Chebyshev sweep (SPMV_CHEB) takes its previous iterates:
//   P2_PLAIN  u from u, w from args.w (or none)
//   P2_FIRST  u = *scale dinv b, formed on the fly; no w
//   P2_SECOND u from u, w = *scale dinv b, formed on the fly
enum P2Start { P2_PLAIN = 0, P2_FIRST = 1, P2_SECOND = 2 };

// Same row sums, in the same order, as spmv_sell_bsr2 on the level's pattern.
template <typename VT>
void p2_spmv(const Level &L, int open_top, const P2Table &tab, const VT *val, const float *u, float *out, SpmvMode mode,
             const SpmvArgs &a, P2Start start, const double *scale, cudaStream_t s);

// b = R r onto the mesh of nc cells a side; x += P xc from it: quadratic
// interpolation between the nodes without prescribed velocity of both meshes
// and its transpose (vectors aligned to a node)
template <typename T>
void p2_restrict(int nc, int open_top, const T *r, T *b, cudaStream_t s);
template <typename T>
void p2_prolong_add(int nc, int open_top, const T *xc, T *x, cudaStream_t s);

}  // namespace chnss
