// One-launch coarse end of the scalar V-cycles (see mgcluster.h).
#include <cooperative_groups.h>

#include "cluster.h"
#include "mgcluster.h"

namespace cg = cooperative_groups;

namespace chnss {
namespace {

constexpr int kSerialCells = 16;   // levels of at most this size are one block's
constexpr size_t kSmemLimit = 227 * 1024 - 1024;

template <typename T> constexpr int mgc_threads() { return sizeof(T) == 4 ? 1024 : 512; }

// owned lines [lb, le) of a level; entry (J, I) of a vector at base + J w + I
struct Own {
  int lb, le, base;
};
template <typename T>
__device__ __forceinline__ Own own_lines(const MgcDesc<T> &d, int l, int me) {
  const MgcLevel<T> &q = d.lv[l];
  Own o;
  o.lb = l < d.na ? q.lb[me] : 0;
  o.le = l < d.na ? q.lb[me + 1] : q.w;
  o.base = 1 - (o.lb - 1) * q.w;
  return o;
}

// value v of owned row lr of the vector at `off` is also the halo of the
// block below / above
template <typename T>
__device__ __forceinline__ void push(const MgcLevel<T> &q, const Own &o, T *sm, int off, int lr, T v) {
  cg::cluster_group cl = cg::this_cluster();
  const int me = (int)cl.block_rank();
  if (lr < q.w && me > 0) {
    const int below = o.lb - q.lb[me - 1];
    *cl.map_shared_rank(sm + off + 1 + (below + 1) * q.w + lr, me - 1) = v;
  }
  const int last = (o.le - o.lb - 1) * q.w;
  if (lr >= last && me + 1 < (int)cl.num_blocks()) *cl.map_shared_rank(sm + off + 1 + (lr - last), me + 1) = v;
}

// One sweep of the owned rows; cf null: b - A u, else a Chebyshev step.
// where: 0 nothing more, 1 halo push, 2 gather in block 0's residual,
// 3 result to global memory.
template <typename T, int NR>
__device__ __forceinline__ void sweep(const MgcDesc<T> &d, T *sm, int l, int u_off, int out_off, const double *cf,
                                      bool has_w, int where) {
  cg::cluster_group cl = cg::this_cluster();
  const MgcLevel<T> &q = d.lv[l];
  const Own o = own_lines(d, l, (int)cl.block_rank());
  const int rows = (o.le - o.lb) * q.w, w = q.w;
  T c0 = 0, c1 = 0, c2 = 0;
  if (cf) {
    c0 = (T)cf[0];
    c1 = (T)cf[1];
    c2 = (T)cf[2];
  }
  for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) {
    T v[7];
#pragma unroll
    for (int j = 0; j < 7; ++j) v[j] = sm[q.val_off + j * q.vs + lr];
    const int e = 1 + w + lr;
    const T di = sm[q.dinv_off + e];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const T *u = sm + u_off + k * q.vec + e;
      const T ui = u[0];
      T acc = v[0] * u[-w - 1];
      acc = fma_of(v[1], u[-w], acc);
      acc = fma_of(v[2], u[-1], acc);
      acc = fma_of(v[3], ui, acc);
      acc = fma_of(v[4], u[1], acc);
      acc = fma_of(v[5], u[w], acc);
      acc = fma_of(v[6], u[w + 1], acc);
      const T bi = sm[q.b_off + k * q.vec + e];
      T *out = sm + out_off + k * q.vec + e;
      const T r = !cf ? bi - acc : cheb_step<T>(c0, c1, c2, ui, di, bi, acc, has_w, has_w ? *out : (T)0);
      *out = r;
      if (where == 1) push<T>(q, o, sm, out_off + k * q.vec, lr, r);
      else if (where == 2) *cl.map_shared_rank(sm + d.r_off + k * d.r_vec + 1 + w + o.lb * w + lr, 0) = r;
      else if (where == 3) d.x.p[k][o.lb * w + lr] = r;
    }
  }
}

// A V-cycle's levels from at most 128 (FP32) or 64 (FP64) cells a side down,
// for NR vectors.  As launches these sweeps take a few microseconds each
// whatever their size: 10 a level, and 37 us (FP32) or 59 us (FP64) for the
// one-block kernel that swept the levels of 32^2 and less from L2.  Here the
// lattice lines of a level are spread over the cluster's blocks, the matrix,
// the Jacobi diagonal and all vectors stay in shared memory for the whole
// cycle, and a sweep ends with its first and last line pushed into the
// neighbours' halo lines and one cluster barrier.  Level l + 1's block owns
// line J where level l's owns line 2 J, so the transfers need one halo line.
// Levels of 16^2 and less are block 0's alone (block barriers; the residual
// comes, and the correction goes back, through distributed shared memory).
// Every row is computed by the expressions, and in the order, of the
// per-sweep kernels, so the result is theirs bit for bit.  Bound by barriers
// and shared-memory latency.  FP64 stops at 64 cells a side: above, the sweeps
// need the FP64 pipes of more multiprocessors than a cluster has.
// 128^2 FP64 adjoint step 70.6 -> 55.8 ms, 100^2 mixed step with inner solves
// 34.8 -> 26.1 ms, 1024^2 mixed step 298.8 -> 288.7 ms.
//
// Shared-memory vectors hold the owned lines between two halo lines (zero
// outside the mesh) and one entry of padding at both ends, so that every
// stencil neighbour can be read; absent couplings have zero values.
template <typename T, int NR>
__global__ void __launch_bounds__(mgc_threads<T>()) k_p1_cluster(const MgcDesc<T> *__restrict__ dp) {
  extern __shared__ __align__(16) unsigned char raw[];
  T *sm = reinterpret_cast<T *>(raw);
  __shared__ __align__(16) unsigned char fixed[sizeof(MgcDesc<T>)];
  MgcDesc<T> &d = *reinterpret_cast<MgcDesc<T> *>(fixed);
  cg::cluster_group cl = cg::this_cluster();
  const int me = (int)cl.block_rank(), ctas = (int)cl.num_blocks(), tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < (int)(sizeof(d) / 4); i += nt) reinterpret_cast<int *>(&d)[i] = reinterpret_cast<const int *>(dp)[i];
  __syncthreads();

  auto own = [&](int l) { return own_lines(d, l, me); };
  // load: values of the owned rows, Jacobi data with the halo, zeroed vectors
  for (int l = 0; l < d.nlev; ++l) {
    if (l >= d.na && me != 0) break;
    const MgcLevel<T> &q = d.lv[l];
    const Own o = own(l);
    const int rows = (o.le - o.lb) * q.w, r0 = o.lb * q.w, N = q.w * q.w;
    if (q.val)
      for (int lr = tid; lr < rows; lr += nt) {
        const int row = r0 + lr;
        const T *vp = q.val + (long)(row >> 5) * (7 * 32) + (row & 31);
#pragma unroll
        for (int j = 0; j < 7; ++j) sm[q.val_off + j * q.vs + lr] = vp[j * 32];
      }
    for (int e = tid; e < q.vec; e += nt) {
      const int row = e - 1 + (o.lb - 1) * q.w;
      const bool in = e >= 1 && row >= 0 && row < N && row < (o.le + 1) * q.w;
      sm[q.dinv_off + e] = in && q.dinv ? q.dinv[row] : (T)0;
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        sm[q.x_off + k * q.vec + e] = 0;
        sm[q.t_off + k * q.vec + e] = 0;
        sm[q.b_off + k * q.vec + e] = l == 0 && in ? d.b.p[k][row] : (T)0;
      }
    }
  }
  if (me == 0 && d.r_vec > 0)
    for (int e = tid; e < NR * d.r_vec; e += nt) sm[d.r_off + e] = 0;
  if (me != 0 && d.na < d.nlev)   // the correction of the first one-block level arrives here
    for (int e = tid; e < NR * d.lv[d.na].vec; e += nt) sm[d.lv[d.na].x_off + e] = 0;
  cl.sync();

  auto sync = [&](bool spread) {
    if (spread) cl.sync();
    else __syncthreads();
  };
  // Chebyshev steps from zero; returns whether the last iterate is in x
  auto from_zero = [&](int l, int deg) {
    const MgcLevel<T> &q = d.lv[l];
    const bool spread = l < d.na;
    const Own o = own(l);
    int cur = (deg - 1) % 2 == 0 ? q.x_off : q.t_off, oth = cur == q.x_off ? q.t_off : q.x_off;
    const T c = (T)*q.coef;
    const int e0 = 1 + (o.lb == 0 ? q.w : 0), e1 = 1 + ((o.le == q.w ? o.le : o.le + 1) - o.lb + 1) * q.w;
    for (int e = e0 + tid; e < e1; e += nt)
#pragma unroll
      for (int k = 0; k < NR; ++k)
        sm[cur + k * q.vec + e] = c * sm[q.dinv_off + e] * sm[q.b_off + k * q.vec + e];
    __syncthreads();
    for (int s = 1; s < deg; ++s) {
      sweep<T, NR>(d, sm, l, cur, oth, q.coef + 4 + 3 * (s - 1), s > 1, spread ? 1 : 0);
      sync(spread);
      const int t = cur;
      cur = oth;
      oth = t;
    }
  };
  // b of level l + 1 (lines [lb, le) of it) from the residual at r: entry (J, I) of level l at r_base + J w + I
  auto restrict_to = [&](int l, int r_off, int r_vec, int r_base, bool spread) {
    const MgcLevel<T> &q = d.lv[l + 1];
    const Own o = own(l + 1);
    const int w = d.lv[l].w, wc = q.w, rows = (o.le - o.lb) * wc;
    for (int lr = tid; lr < rows; lr += nt) {
      const int J = o.lb + lr / wc, I = lr % wc;
      const bool left = I > 0, right = I + 1 < wc;
      const int c = r_base + 2 * J * w + 2 * I;
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        const T *r = sm + r_off + k * r_vec + c;
        T acc = 0;
        if (left) acc += (T)0.5 * r[-w - 1];
        acc += (T)0.5 * r[-w];
        if (left) acc += (T)0.5 * r[-1];
        acc += (T)1 * r[0];
        if (right) acc += (T)0.5 * r[1];
        acc += (T)0.5 * r[w];
        if (right) acc += (T)0.5 * r[w + 1];
        sm[q.b_off + k * q.vec + 1 + wc + lr] = acc;
        if (spread) push<T>(q, o, sm, q.b_off + k * q.vec, lr, acc);
      }
    }
  };
  // x of level l (owned and halo lines) += P x of level l + 1
  auto prolong = [&](int l) {
    const MgcLevel<T> &q = d.lv[l], &qc = d.lv[l + 1];
    const Own o = own(l), oc = own(l + 1);
    const int w = q.w, wc = qc.w;
    const int J0 = o.lb > 0 ? o.lb - 1 : 0, J1 = o.le < w ? o.le + 1 : w;
    for (int t = tid; t < (J1 - J0) * w; t += nt) {
      const int J = J0 + t / w, I = t % w;
      const int ca = oc.base + (J / 2) * wc + I / 2;
      const int cb = ca + (J & 1) * wc + (I & 1);
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        const T *xc = sm + qc.x_off + k * qc.vec;
        T acc = 0;
        if (ca == cb) {
          acc += (T)1 * xc[ca];
        } else {
          acc += (T)0.5 * xc[ca];
          acc += (T)0.5 * xc[cb];
        }
        T &xi = sm[q.x_off + k * q.vec + o.base + J * w + I];
        xi = xi + acc;
      }
    }
    __syncthreads();
  };
  auto post = [&](int l) {   // degree sweeps from x, ending in x (even degree)
    const MgcLevel<T> &q = d.lv[l];
    const bool spread = l < d.na;
    int cur = q.x_off, oth = q.t_off;
    for (int s = 0; s < d.degree; ++s) {
      const bool last = s + 1 == d.degree;
      sweep<T, NR>(d, sm, l, cur, oth, s == 0 ? q.coef + 1 : q.coef + 4 + 3 * (s - 1), s > 0, last && l == 0 ? 3 : spread ? 1 : 0);
      if (!(last && l == 0)) sync(spread);
      const int t = cur;
      cur = oth;
      oth = t;
    }
  };

  const int L = d.nlev - 1;
  // down, levels spread over the cluster
  for (int l = 0; l < d.na; ++l) {
    const MgcLevel<T> &q = d.lv[l];
    const Own o = own(l);
    from_zero(l, l == L ? d.coarse_degree : d.degree);
    if (l == L) break;
    const bool next = l + 1 < d.na;
    sweep<T, NR>(d, sm, l, q.x_off, q.t_off, nullptr, false, next ? 1 : 2);
    cl.sync();
    if (next) {
      restrict_to(l, q.t_off, q.vec, o.base, true);
      cl.sync();
    }
  }
  if (d.na == L && d.na > 0) {
    // the spread levels end in a dense coarsest one (9^2 to 25^2): its rows
    // are spread too (FP64 sums: 676 rows take one multiprocessor 120 us)
    const MgcLevel<T> &q = d.lv[L];
    const int at = 1 + q.w;
    if (me == 0) {
      restrict_to(L - 1, d.r_off, d.r_vec, 1 + d.lv[L - 1].w, false);
      __syncthreads();
      for (int t = tid; t < (ctas - 1) * NR * q.vec; t += nt) {
        const int e = q.b_off + t % (NR * q.vec);
        *cl.map_shared_rank(sm + e, 1 + t / (NR * q.vec)) = sm[e];
      }
    }
    cl.sync();
    for (int t = tid; t < NR * ((d.nc - me + ctas - 1) / ctas); t += nt) {
      const int k = t % NR, r = me + ctas * (t / NR);
      const T *b = sm + q.b_off + k * q.vec + at;
      const double *row = d.cinv + (long)r * d.nc;
      double s = 0.0;
#pragma unroll 8
      for (int c = 0; c < d.nc; ++c) s = fma(row[c], (double)b[c], s);
      for (int z = 0; z < ctas; ++z) *cl.map_shared_rank(sm + q.x_off + k * q.vec + at + r, z) = (T)s;
    }
  } else if (me == 0 && d.na < d.nlev) {   // one-block levels
    for (int l = d.na; l <= L; ++l) {
      const MgcLevel<T> &q = d.lv[l];
      if (l > 0) {
        if (l == d.na) restrict_to(l - 1, d.r_off, d.r_vec, 1 + d.lv[l - 1].w, false);
        else restrict_to(l - 1, d.lv[l - 1].t_off, d.lv[l - 1].vec, 1 + d.lv[l - 1].w, false);
        __syncthreads();
      }
      if (l < L) {
        from_zero(l, d.degree);
        sweep<T, NR>(d, sm, l, q.x_off, q.t_off, nullptr, false, 0);
        __syncthreads();
      } else if (d.coarse_degree > 0) {
        from_zero(l, d.coarse_degree);
      } else {
        for (int t = tid; t < NR * d.nc; t += nt) {
          const int k = t / d.nc, r = t % d.nc;
          const T *b = sm + q.b_off + k * q.vec + 1 + q.w;
          const double *row = d.cinv + (long)r * d.nc;
          double s = 0.0;
#pragma unroll 8
          for (int c = 0; c < d.nc; ++c) s = fma(row[c], (double)b[c], s);
          sm[q.x_off + k * q.vec + 1 + q.w + r] = (T)s;
        }
        __syncthreads();
      }
    }
    for (int l = L - 1; l >= d.na; --l) {
      prolong(l);
      post(l);
    }
    if (d.na > 0) {   // the correction to every block
      const MgcLevel<T> &q = d.lv[d.na];
      for (int t = tid; t < (ctas - 1) * NR * q.vec; t += nt) {
        const int e = q.x_off + t % (NR * q.vec);
        *cl.map_shared_rank(sm + e, 1 + t / (NR * q.vec)) = sm[e];
      }
    }
  }
  if (d.na > 0 && d.na < d.nlev) cl.sync();
  // up
  for (int l = (d.na < d.nlev ? d.na : L) - 1; l >= 0; --l) {
    prolong(l);
    post(l);
  }
}

template <typename T>
bool runs(int nr, int ctas, size_t smem) {
  constexpr size_t most = kSmemLimit - sizeof(MgcDesc<T>);
  switch (nr) {
    case 1: return cluster_runs<k_p1_cluster<T, 1>>(ctas, mgc_threads<T>(), smem, most);
    case 2: return cluster_runs<k_p1_cluster<T, 2>>(ctas, mgc_threads<T>(), smem, most);
    case 3: return cluster_runs<k_p1_cluster<T, 3>>(ctas, mgc_threads<T>(), smem, most);
    default: return false;
  }
}

}  // namespace

template <typename T>
MgcPlan<T> mgc_plan(Arena &ar, int nr, const std::vector<const Pattern *> &pats, const std::vector<const Transfer *> &trs,
                    const std::vector<T *> &val, const std::vector<T *> &dinv, const std::vector<double *> &coef,
                    const std::vector<MultiPtr<T>> &b, const std::vector<MultiPtr<T>> &x, int degree, bool coarse_iter,
                    int nc, const double *cinv) {
  MgcPlan<T> plan;
  const int nl = (int)pats.size();
  const int largest = sizeof(T) == 4 ? 128 : 64;
  auto cells = [&](int l) {
    int n = 0;
    while ((long)(n + 1) * (n + 1) < pats[l]->nrows) ++n;
    return n;
  };
  if (degree % 2 != 0) return plan;
  for (int first = 0; first < nl - 1; ++first) {
    if (cells(first) > largest) continue;
    MgcDesc<T> d;
    d.nlev = nl - first;
    if (d.nlev > kMgcMaxLevels) continue;
    d.degree = degree;
    d.nc = nc;
    d.cinv = cinv;
    d.coarse_degree = coarse_iter ? kCoarseDegree : 0;
    bool ok = true;
    for (int l = first; l < nl; ++l) {
      MgcLevel<T> &q = d.lv[l - first];
      q.n = cells(l);
      q.w = q.n + 1;
      ok = ok && pats[l]->sell.stencil && (l == nl - 1 || trs[l]->p1_cells == cells(l + 1));
      const bool bare = l == nl - 1 && !coarse_iter;     // dense coarsest level: no sweeps
      q.val = bare ? nullptr : val[l];
      q.dinv = bare ? nullptr : dinv[l];
      q.coef = bare ? nullptr : coef[l];
      // a dense coarsest level is one block's whatever its size
      if (q.n > kSerialCells && !bare && d.na == l - first) d.na = l - first + 1;
    }
    if (!ok) return plan;
    plan.ctas = d.na == 0 ? 1 : kMgcMaxCtas;
    if (d.na > 0) {   // lines by the coarsest spread level, doubled towards the finer ones
      const int lc = d.na - 1;
      for (int k = 0; k <= plan.ctas; ++k) {
        d.lv[lc].lb[k] = k * d.lv[lc].w / plan.ctas;
        for (int l = lc - 1; l >= 0; --l) d.lv[l].lb[k] = k == plan.ctas ? d.lv[l].w : 2 * d.lv[l + 1].lb[k];
      }
    }
    int off = 0;
    auto take = [&](int count) {
      const int o = off;
      off += (count + 3) / 4 * 4;
      return o;
    };
    for (int l = 0; l < d.nlev; ++l) {
      MgcLevel<T> &q = d.lv[l];
      int lines = q.w;
      if (l < d.na) {
        lines = 0;
        for (int k = 0; k < plan.ctas; ++k) {
          const int own = q.lb[k + 1] - q.lb[k];
          if (own < 1) ok = false;
          lines = std::max(lines, own);
        }
      }
      q.vs = lines * q.w;
      q.vec = (lines + 2) * q.w + 2;
      q.val_off = take(q.val ? 7 * q.vs : 0);
      q.dinv_off = take(q.vec);
      q.x_off = take(nr * q.vec);
      q.t_off = take(nr * q.vec);
      q.b_off = take(nr * q.vec);
    }
    if (d.na > 0 && d.na < d.nlev) {
      const int w = d.lv[d.na - 1].w;
      d.r_vec = (w + 2) * w + 2;
      d.r_off = take(nr * d.r_vec);
    }
    const size_t bytes = (size_t)off * sizeof(T);
    if (!ok || bytes > kSmemLimit - sizeof(MgcDesc<T>) || !runs<T>(nr, plan.ctas, bytes)) continue;
    for (int k = 0; k < nr; ++k) {
      d.b.p[k] = b[first].p[k];
      d.x.p[k] = x[first].p[k];
    }
    plan.first = first;
    plan.nr = nr;
    plan.smem = bytes;
    plan.desc = ar.alloc<MgcDesc<T>>(1);
    CHNSS_CK(cudaMemcpy(plan.desc, &d, sizeof(d), cudaMemcpyHostToDevice));
    return plan;
  }
  return plan;
}

template <typename T>
void mgc_apply(const MgcPlan<T> &p, cudaStream_t s) {
  const MgcDesc<T> *d = p.desc;
  switch (p.nr) {
    case 1:
      launch_cluster(k_p1_cluster<T, 1>, p.ctas, 1, mgc_threads<T>(), p.smem, s, d);
      break;
    case 2:
      launch_cluster(k_p1_cluster<T, 2>, p.ctas, 1, mgc_threads<T>(), p.smem, s, d);
      break;
    case 3:
      launch_cluster(k_p1_cluster<T, 3>, p.ctas, 1, mgc_threads<T>(), p.smem, s, d);
      break;
    default: throw Error{CHNSS_ERR_ARG, "coarse-level cluster: 1 to 3 vectors"};
  }
  CHNSS_LAUNCH_CK();
}

template MgcPlan<float> mgc_plan<float>(Arena &, int, const std::vector<const Pattern *> &,
                                        const std::vector<const Transfer *> &, const std::vector<float *> &,
                                        const std::vector<float *> &, const std::vector<double *> &,
                                        const std::vector<MultiPtr<float>> &, const std::vector<MultiPtr<float>> &, int,
                                        bool, int, const double *);
template MgcPlan<double> mgc_plan<double>(Arena &, int, const std::vector<const Pattern *> &,
                                          const std::vector<const Transfer *> &, const std::vector<double *> &,
                                          const std::vector<double *> &, const std::vector<double *> &,
                                          const std::vector<MultiPtr<double>> &, const std::vector<MultiPtr<double>> &,
                                          int, bool, int, const double *);
template void mgc_apply<float>(const MgcPlan<float> &, cudaStream_t);
template void mgc_apply<double>(const MgcPlan<double> &, cudaStream_t);

}  // namespace chnss
