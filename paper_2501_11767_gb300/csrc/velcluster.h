// The coarse end of a velocity V-cycle on a structured mesh in one launch of
// a thread-block cluster (see k_vel_cluster).
#pragma once

#include "p2stencil.h"

namespace chnss {

constexpr int kVlcMaxLevels = 6;
constexpr int kVlcCtas = 8;
constexpr int kVlcMaxPhases = 96;

// Offsets into shared memory count nodes (pairs).
struct VlcLevel {
  int n = 0, w = 0;                // cells and lattice nodes per side
  unsigned inv_w = 0, inv_w1 = 0;  // 2^32 / w and 2^32 / (n + 1), rounded up
  long ld = 0;                     // cell stride of the values in global memory
  const void *val = nullptr, *dinv = nullptr;
  const double *coef = nullptr;
  int ncoef = 0;
  int lb[kVlcCtas + 1] = {};       // first lattice line of each block (levels spread over the cluster)
  int cells = 0, vec = 0;          // cell stride of the values, nodes of a vector
  int val_off = 0, dinv_off = 0, x_off = 0, t_off = 0, b_off = 0;
};
// One phase of the cycle: INIT level: out = coef_0 dinv b; SWEEP level: from
// u to out; RESTRICT, PROLONG: between level and level + 1 (u: the residual);
// DENSE: coarsest level; BROADCAST: nodes [u, u + out) of block 0 to all.
enum VlcOp { VLC_INIT = 0, VLC_SWEEP, VLC_RESTRICT, VLC_PROLONG, VLC_DENSE, VLC_BROADCAST };
enum VlcWhere { VLC_HERE = 0, VLC_HALO, VLC_HALO_ABOVE, VLC_GATHER, VLC_RESULT };
enum VlcSync { VLC_NONE = 0, VLC_BLOCK, VLC_CLUSTER };
struct VlcPhase {
  signed char op = 0, level = 0, where = 0, sync = 0;
  signed char alone = 0;           // block 0 only
  signed char coef = 0, has_w = 0; // SWEEP: first of the three coefficients (0: residual)
  int u = 0, out = 0;
};
constexpr int kVlcRest = 25;       // entries of a restriction row (padded with zero weights)
struct alignas(16) VlcDesc {
  int nlev = 0, na = 0;            // levels; the first na are spread over the cluster, the rest one block's
  int nphase = 0, open = 0;
  int pre_steps = 0, post_steps = 0;   // Chebyshev steps of the first level, from zero and after the correction
  int nc = 0, share = 0;           // dense coarsest level: rows, whether every block takes some
  const double *cinv = nullptr;
  int cinv_off = 0, cinv_rows = 0; // its interior part in shared memory (offset in doubles)
  int r_off = 0;                   // residual of the last spread level, gathered by block 0
  const void *b = nullptr;         // global: right-hand side and result of the first level
  void *x = nullptr;
  VlcLevel lv[kVlcMaxLevels];
  VlcPhase ph[kVlcMaxPhases];
  // transfers between level and level + 1: offsets and weights by node type / class
  int ro[kVlcMaxLevels][4][kVlcRest] = {}, po[kVlcMaxLevels][16][6] = {};
  float rw[4][kVlcRest] = {}, pw[16][6] = {};
};
struct VlcPlan {
  VlcDesc *desc = nullptr;
  int first = -1, ctas = 1, bf16 = 0, open = 0;
  size_t smem = 0;
  float tab[2 * (kP2Slots + kP2TopSlots)] = {};   // off-diagonal entries, rounded to the values' precision
};

// Plan for the coarse end of an FP32 hierarchy (values FP32, or BF16 in val16)
// whose levels are in stencil order; first = -1 if no level fits or the
// device has no place for its cluster.
VlcPlan vlc_plan(Arena &ar, const std::vector<const Level *> &lev, int open_top, const std::vector<P2Table> &tab,
                 const std::vector<float *> &val, const std::vector<__nv_bfloat16 *> &val16,
                 const std::vector<float *> &dinv, const std::vector<double *> &coef, const std::vector<float *> &b,
                 const std::vector<float *> &x, int degree, bool coarse_iter, int nc, const double *cinv);
void vlc_apply(const VlcPlan &p, cudaStream_t s);

}  // namespace chnss
