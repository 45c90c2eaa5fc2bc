// The coarse end of a scalar V-cycle on a structured mesh in one launch of a
// thread-block cluster (see k_p1_cluster).
#pragma once

#include "kernels.h"

namespace chnss {

constexpr int kMgcMaxLevels = 8;
constexpr int kMgcMaxCtas = 16;

template <typename T>
struct MgcLevel {
  int n = 0, w = 0;                // cells and nodes per side
  const T *val = nullptr;          // stencil layout (Sell::stencil), 7 entries a row
  const T *dinv = nullptr;
  const double *coef = nullptr;
  int lb[kMgcMaxCtas + 1] = {};    // first line of each block (levels spread over the cluster)
  int vs = 0, vec = 0;             // rows of the value storage, entries of a vector
  int val_off = 0, dinv_off = 0, x_off = 0, t_off = 0, b_off = 0;   // shared memory, in T; vectors vec apart
};
template <typename T>
struct MgcDesc {
  int nlev = 0, na = 0;            // levels; the first na are spread over the cluster, the rest one block's
  int degree = 2, nc = 0, coarse_degree = 0;
  const double *cinv = nullptr;
  int r_off = 0, r_vec = 0;        // residual of the last spread level, gathered by block 0
  MultiPtr<T> b, x;                // global: right-hand sides and results of the first level
  MgcLevel<T> lv[kMgcMaxLevels];
};
// What the launch needs beside the device copy of the descriptor.
template <typename T>
struct MgcPlan {
  MgcDesc<T> *desc = nullptr;
  int first = -1;                  // first level of the hierarchy it handles
  int nr = 1, ctas = 1;
  size_t smem = 0;
};

// Plan for the coarse end of a hierarchy of stencil levels `pats` (finest
// first, P1 transfers between them) and nr vectors; first = -1 if none fits
// or the device has no place for its cluster.
// The arrays are those of MGHier / MGBatch.
template <typename T>
MgcPlan<T> mgc_plan(Arena &ar, int nr, const std::vector<const Pattern *> &pats, const std::vector<const Transfer *> &trs,
                    const std::vector<T *> &val, const std::vector<T *> &dinv, const std::vector<double *> &coef,
                    const std::vector<MultiPtr<T>> &b, const std::vector<MultiPtr<T>> &x, int degree, bool coarse_iter,
                    int nc, const double *cinv);
template <typename T>
void mgc_apply(const MgcPlan<T> &p, cudaStream_t s);

}  // namespace chnss
