// One-launch coarse end of the velocity V-cycles (see velcluster.h).
#include <cooperative_groups.h>
#include <cuda_pipeline.h>

#include "cluster.h"
#include "p2slots.h"
#include "velcluster.h"

namespace cg = cooperative_groups;

namespace chnss {
namespace {

constexpr size_t kSmemLimit = 226 * 1024;
// halo lines stored below and above: a coarse line takes residuals from three
// lines below; two lines of an iterate are exchanged both ways
constexpr int kBelow = 3, kAbove = 3, kHalo = 2;
constexpr int kSums = 8;   // partial sums of a row, as the sweeps of levels of this size have
constexpr int kCoefs = 4 + 3 * (kMaxSmoothDegree - 1);

// cells a side of the levels a cluster takes: one block's up to kSerial,
// spread over the cluster from 16 to kLargest (at least four lines a block)
constexpr int kSerial = 15, kLargest = 32;
constexpr int kThreads = 512, kRoles = 2;   // vertices / edge midpoints of a cell
static_assert(kVlcMaxLevels * kCoefs <= kThreads, "one pass loads the coefficients");

__device__ __forceinline__ float2 pair_at(const __nv_bfloat16 *p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
}
// t / w for t w < 2^32, inv = 2^32 / w rounded up
__device__ __forceinline__ int div_by(int t, unsigned inv) { return (int)__umulhi((unsigned)t, inv); }

struct Fixed {   // static shared memory
  VlcDesc d;
  float coef[kVlcMaxLevels][kCoefs];
};

// The FP32 velocity V-cycle's levels from at most 32 cells a side down.  As launches these levels take 10 sweeps and transfers of 4 to 8
// us each whatever their size.  Here the lattice lines of a level are spread
// over the cluster's blocks, matrix and vectors stay in shared memory for the
// whole cycle, and a sweep ends with its outer two lines pushed into the
// neighbours' halos and one cluster barrier; smaller levels are block 0's
// alone.  Level l + 1's block owns line J where level l's owns line 2 J.  The
// cycle is a list of phases run by one loop, so that its code stays in the
// instruction caches.  Two threads sweep a cell, one its vertex and one its
// edge midpoints: the chains of instructions are what a sweep of so few nodes
// takes (a node a thread: 4600 to 6000 clocks a sweep, of which 200 the
// barrier), and a cell's 19 neighbours and 46 blocks are independent.  Nodes
// with prescribed velocity hold zeros in shared memory; on the first level
// their decoupled rows (the identity) are run through the cycle's recurrence
// one by one at the end.  Rows are summed by the expressions, and in the
// order, of the per-sweep kernels: results are the same bit for bit.
// 384^2 (levels 24 to 3): 58 us a cycle, 38 us less of an Oseen iteration than
// as launches; 384^2 Oseen solve 36.8 -> 34.8 ms, 512^2 step 62.4 -> 60.3 ms.
// FP64 hierarchies stay on launches: a quarter of a multiprocessor issues one
// FP64 warp instruction in 64 clocks, and a sweep of 4^2 took 22000.
struct Coef {
  float c[2 * (kP2Slots + kP2TopSlots)];   // off-diagonal entries by slot
};

template <typename VT, bool OPEN>
__global__ void __launch_bounds__(kThreads) k_vel_cluster(const VlcDesc *__restrict__ dp,
                                                          const __grid_constant__ Coef tab) {
  using P = float2;
  extern __shared__ __align__(16) unsigned char raw[];
  P *sm = reinterpret_cast<P *>(raw);
  __shared__ __align__(16) unsigned char fixed[sizeof(Fixed)];
  Fixed &f = *reinterpret_cast<Fixed *>(fixed);
  const VlcDesc &d = f.d;
  cg::cluster_group cl = cg::this_cluster();
  const int me = (int)cl.block_rank(), ctas = (int)cl.num_blocks(), tid = threadIdx.x;
  constexpr int nt = kThreads, open = OPEN ? 1 : 0;
  const int lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < (int)(sizeof(VlcDesc) / 16); i += nt)
    reinterpret_cast<int4 *>(&f.d)[i] = reinterpret_cast<const int4 *>(dp)[i];
  __syncthreads();

  if (tid < kVlcMaxLevels * kCoefs && tid / kCoefs < d.nlev && tid % kCoefs < d.lv[tid / kCoefs].ncoef)
    f.coef[tid / kCoefs][tid % kCoefs] = (float)d.lv[tid / kCoefs].coef[tid % kCoefs];
  // matrix values (asynchronous copies), Jacobi data, zeroed vectors, tables
  for (int l = 0; l < d.nlev; ++l) {
    const VlcLevel &q = d.lv[l];
    const bool mine = l < d.na || me == 0;
    const int lb = l < d.na ? q.lb[me] : 0, le = l < d.na ? q.lb[me + 1] : q.w;
    if (q.val && mine) {
      const int c0 = (lb / 2) * (q.n + 1), nc = ((le + 1) / 2) * (q.n + 1) - c0;
      for (int k = warp; k < kP2Slots; k += nt / 32)
        for (int c = lane; c < nc; c += 32) {
          const VT *src = static_cast<const VT *>(q.val) + 2 * (k * q.ld + c0 + c);
          P *dst = sm + q.val_off + k * q.cells + c;
          if constexpr (std::is_same<VT, float>::value) __pipeline_memcpy_async(dst, src, sizeof(P));
          else *dst = pair_at(src);
        }
    }
    for (int e = tid; e < q.vec; e += nt) {
      const int line = div_by(e, q.inv_w), J = lb - kBelow + line, I = e - line * q.w, row = J * q.w + I;
      const bool in = mine && J < le + kHalo && !prescribed(I, J, q.w, open);
      const bool ld = in && q.dinv != nullptr, lbv = in && l == 0;
      __pipeline_memcpy_async(sm + q.dinv_off + e, ld ? static_cast<const P *>(q.dinv) + row : static_cast<const P *>(d.b),
                              sizeof(P), ld ? 0 : sizeof(P));
      __pipeline_memcpy_async(sm + q.b_off + e, lbv ? static_cast<const P *>(d.b) + row : static_cast<const P *>(d.b),
                              sizeof(P), lbv ? 0 : sizeof(P));
      sm[q.x_off + e] = sm[q.t_off + e] = make_float2(0, 0);
    }
  }
  if (me == 0 && d.na > 0 && d.na < d.nlev) {
    const int w = d.lv[d.na - 1].w;
    for (int e = tid; e < (w + kBelow + kAbove) * w; e += nt) sm[d.r_off + e] = make_float2(0, 0);
  }
  // dense inverse on the coarsest level: interior rows me, me + step, ... with their interior columns
  const int wi = d.lv[d.nlev - 1].w - 2, ni = 2 * wi * (wi + open), step = d.share ? ctas : 1;
  const unsigned inv_wi = 0xffffffffu / wi + 1;
  auto interior = [&](int t) {   // dof of interior dof t of the coarsest level
    const int nd = t >> 1, j = div_by(nd, inv_wi);
    return 2 * ((1 + j) * (wi + 2) + 1 + nd - j * wi) + (t & 1);
  };
  double *ci = reinterpret_cast<double *>(raw) + d.cinv_off, *cb = ci + d.cinv_rows * ni;
  if (d.nc > 0 && (me == 0 || d.share))
    for (int t = me + step * warp; t < ni; t += step * (nt / 32)) {
      const double *row = d.cinv + (long)interior(t) * d.nc;
      for (int c = lane; c < ni; c += 32)
        __pipeline_memcpy_async(ci + (t / step) * ni + c, row + interior(c), sizeof(double));
    }
  __pipeline_commit();
  __pipeline_wait_prior(0);
  cl.sync();

  for (int p = 0; p < d.nphase; ++p) {
    const VlcPhase ph = d.ph[p];
    if (ph.alone && me != 0) {
      if (ph.sync == VLC_CLUSTER) cl.sync();
      continue;
    }
    const int l = ph.level;
    const VlcLevel &q = d.lv[l];
    const int w = q.w, lb = l < d.na ? q.lb[me] : 0, le = l < d.na ? q.lb[me + 1] : w;
    const int base = (kBelow - lb) * w;   // node (J, I) of a vector at base + J w + I
    // owned node (J, I) of the vector at `off` of level h is also a neighbour's halo
    auto push = [&](const VlcLevel &h, int hb, int he, int off, int J, int I, P v, bool up_only) {
      if (!up_only && J < hb + kHalo && me > 0)
        *cl.map_shared_rank(sm + off + (kBelow + J - h.lb[me - 1]) * h.w + I, me - 1) = v;
      if (J >= he - (up_only ? kBelow : kHalo) && me + 1 < ctas)
        *cl.map_shared_rank(sm + off + (kBelow + J - he) * h.w + I, me + 1) = v;
    };
    if (ph.op == VLC_SWEEP) {
      const int w1 = q.n + 1, nc = ((le - lb + 1) / 2) * w1;
      const float *cf = f.coef[l] + ph.coef;
      const float c0 = cf[0], c1 = cf[1], c2 = cf[2];
      constexpr SlotTable st = slot_table();
      const int role = tid / (nt / kRoles);   // the same for a warp
      for (int c = tid % (nt / kRoles); c < nc; c += nt / kRoles) {
        const int cj = div_by(c, q.inv_w1), i0 = 2 * (c - cj * w1), j0 = lb + 2 * cj;
        const int e0 = base + j0 * w + i0;
        const P *v = sm + q.val_off + c, *u = sm + ph.u + e0;
        P x[19];
#pragma unroll
        for (int k = 0; k < 19; ++k) x[k] = u[st.dj[k] * w + st.di[k]];
        auto row = [&](auto tyc) {
          constexpr int ty = decltype(tyc)::value, oi = ty & 1, oj = ty >> 1, s0k = slot_base(ty), cnt = slot_count(ty);
          const int I = i0 + oi, J = j0 + oj;
          if (J >= le || prescribed(I, J, w, open)) return;
          const int e = e0 + oj * w + oi;
          const int top = OPEN && ty < 2 && J == w - 1 ? kP2Slots : 0;
          const P b = sm[q.b_off + e], di = sm[q.dinv_off + e];
          P &out = sm[ph.out + e];
          const P wv = out;
          P ui = b;
          float p0[kSums], p1[kSums];
#pragma unroll
          for (int k = 0; k < kSums; ++k) p0[k] = p1[k] = 0;
#pragma unroll
          for (int k = 0; k < cnt; ++k) {
            constexpr SlotTable sk = slot_table();
            int xi = 0;
#pragma unroll
            for (int h = 0; h < 19; ++h)
              if (sk.di[h] == oi + sk.di[s0k + k] && sk.dj[h] == oj + sk.dj[s0k + k]) xi = h;
            const P a = v[(s0k + k) * q.cells], xk = x[xi];
            if (sk.di[s0k + k] == 0 && sk.dj[s0k + k] == 0) ui = xk;
            p0[k % kSums] = fma_of(tab.c[2 * (top + s0k + k)], xk.y, fma_of(a.x, xk.x, p0[k % kSums]));
            p1[k % kSums] = fma_of(a.y, xk.y, fma_of(tab.c[2 * (top + s0k + k) + 1], xk.x, p1[k % kSums]));
          }
          float s0 = p0[0], s1 = p1[0];
#pragma unroll
          for (int k = 1; k < kSums; ++k) {
            s0 += p0[k];
            s1 += p1[k];
          }
          P r;
          if (ph.coef == 0) {
            r = make_float2(b.x - s0, b.y - s1);
          } else {
            r = make_float2(cheb_step<float>(c0, c1, c2, ui.x, di.x, b.x, s0, ph.has_w, wv.x),
                      cheb_step<float>(c0, c1, c2, ui.y, di.y, b.y, s1, ph.has_w, wv.y));
          }
          out = r;
          if (ph.where == VLC_HALO || ph.where == VLC_HALO_ABOVE)
            push(q, lb, le, ph.out, J, I, r, ph.where == VLC_HALO_ABOVE);
          else if (ph.where == VLC_GATHER)
            *cl.map_shared_rank(sm + d.r_off + (kBelow + J) * w + I, 0) = r;
          else if (ph.where == VLC_RESULT)
            static_cast<P *>(d.x)[J * w + I] = r;
        };
        if (role == 0) {
          row(std::integral_constant<int, 0>());
        } else {
          row(std::integral_constant<int, 1>());
          row(std::integral_constant<int, 2>());
          row(std::integral_constant<int, 3>());
        }
      }
    } else if (ph.op == VLC_INIT) {   // owned and halo lines; zero elsewhere
      const float c = f.coef[l][0];
      for (int e = tid; e < q.vec; e += nt) {
        const P di = sm[q.dinv_off + e], b = sm[q.b_off + e];
        sm[ph.out + e] = make_float2(c * di.x * b.x, c * di.y * b.y);
      }
    } else if (ph.op == VLC_RESTRICT) {
      const VlcLevel &h = d.lv[l + 1];
      const bool spread = l + 1 < d.na;
      const int hb = spread ? h.lb[me] : 0, he = spread ? h.lb[me + 1] : h.w;
      const int rbase = spread ? base : kBelow * w;   // block 0 gathers whole levels
      for (int t = tid; t < (he - hb) * h.w; t += nt) {
        const int line = div_by(t, h.inv_w), J = hb + line, I = t - line * h.w;
        if (prescribed(I, J, h.w, open)) continue;
        const int ty = type_of(I, J), cnt = ty == 0 ? 25 : 10;   // multiples of five, zero weights at the end
        const P *r = sm + ph.u + rbase + 2 * J * w + 2 * I;
        const int *o = d.ro[l][ty];
        const float *rw = d.rw[ty];
        float a0 = 0, a1 = 0;
#pragma unroll 1
        for (int k0 = 0; k0 < cnt; k0 += 5) {
#pragma unroll
          for (int k = 0; k < 5; ++k) {
            const P v = r[o[k0 + k]];
            a0 = fma_of(rw[k0 + k], v.x, a0);
            a1 = fma_of(rw[k0 + k], v.y, a1);
          }
        }
        sm[h.b_off + (kBelow + J - hb) * h.w + I] = make_float2(a0, a1);
        if (spread) push(h, hb, he, h.b_off, J, I, make_float2(a0, a1), false);
      }
    } else if (ph.op == VLC_PROLONG) {
      const VlcLevel &h = d.lv[l + 1];
      const int hb = l + 1 < d.na ? h.lb[me] : 0;
      for (int t = tid; t < (le - lb) * w; t += nt) {
        const int line = div_by(t, q.inv_w), J = lb + line, I = t - line * w;
        if (prescribed(I, J, w, open)) continue;
        const int c = (I & 3) + 4 * (J & 3);
        const P *xc = sm + h.x_off + (kBelow - hb + 2 * (J >> 2)) * h.w + 2 * (I >> 2);
        const int *o = d.po[l][c];
        const float *pw = d.pw[c];
        float a0 = 0, a1 = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const P v = xc[o[k]];
          a0 = fma_of(pw[k], v.x, a0);
          a1 = fma_of(pw[k], v.y, a1);
        }
        P &x = sm[q.x_off + base + J * w + I];
        x = make_float2(x.x + a0, x.y + a1);
        if (ph.where == VLC_HALO) push(q, lb, le, q.x_off, J, I, x, false);
      }
    } else if (ph.op == VLC_DENSE) {
      for (int t = tid; t < ni; t += nt) {
        const int j = interior(t);
        cb[t] = (double)reinterpret_cast<const float *>(sm + q.b_off + kBelow * w)[j];
      }
      __syncthreads();
      for (int t = me + step * tid; t < ni; t += step * nt) {
        const double *row = ci + (t / step) * ni;
        double s = 0.0;
#pragma unroll 6
        for (int c = 0; c < ni; ++c) s = fma(row[c], cb[c], s);
        const int j = interior(t);
        reinterpret_cast<float *>(cl.map_shared_rank(sm + q.x_off + kBelow * w + (j >> 1), 0))[j & 1] = (float)s;
      }
    } else {   // VLC_BROADCAST
      for (int e = tid; e < ph.out; e += nt) {
        const P v = sm[ph.u + e];
        for (int z = 1; z < ctas; ++z) *cl.map_shared_rank(sm + ph.u + e, z) = v;
      }
    }
    if (ph.sync == VLC_CLUSTER) cl.sync();
    else if (ph.sync == VLC_BLOCK) __syncthreads();
  }
  // prescribed nodes of the first level: u <- the cycle on the identity row
  {
    const VlcLevel &q = d.lv[0];
    const int lb = d.na > 0 ? q.lb[me] : 0, le = d.na > 0 ? q.lb[me + 1] : q.w;
    const float *cf = f.coef[0];
    for (int t = tid; t < (le - lb) * q.w; t += nt) {
      const int line = div_by(t, q.inv_w), J = lb + line, I = t - line * q.w;
      if (!prescribed(I, J, q.w, open)) continue;
      const int row = J * q.w + I;
      const P b = static_cast<const P *>(d.b)[row], di = static_cast<const P *>(q.dinv)[row];
      P u = make_float2(cf[0] * di.x * b.x, cf[0] * di.y * b.y), w = make_float2(0, 0);
      for (int s = 1; s < d.pre_steps + d.post_steps; ++s) {
        const bool post = s >= d.pre_steps;
        const int k = post ? s - d.pre_steps : s;                 // step of its half
        const float *c = cf + (k == 0 ? 1 : 4 + 3 * (k - 1));
        const bool has_w = post ? k > 0 : k > 1;
        const P v = make_float2(cheb_step<float>(c[0], c[1], c[2], u.x, di.x, b.x, u.x, has_w, w.x),
                          cheb_step<float>(c[0], c[1], c[2], u.y, di.y, b.y, u.y, has_w, w.y));
        w = u;
        u = v;
      }
      static_cast<P *>(d.x)[row] = u;
    }
  }
}

// the descriptor's layout and phases from level `first` on; false if it does not fit
bool layout(int first, const std::vector<const Level *> &lev, int open, int degree, bool coarse_iter, VlcDesc &d,
            int &ctas, size_t &smem) {
  const int nl = (int)lev.size(), L = nl - 1 - first;
  d = VlcDesc();
  d.nlev = nl - first;
  d.open = open;
  const int coarse_degree = coarse_iter ? kCoarseDegree : 0;
  if (d.nlev < (coarse_iter ? 1 : 2) || d.nlev > kVlcMaxLevels || degree % 2 != 0 || degree > kMaxSmoothDegree) return false;
  for (int l = 0; l <= L; ++l) {
    VlcLevel &q = d.lv[l];
    q.n = lev[first + l]->n;
    q.w = 2 * q.n + 1;
    q.inv_w = 0xffffffffu / q.w + 1;
    q.inv_w1 = 0xffffffffu / (q.n + 1) + 1;
    q.ld = p2_ld(q.n);
    const bool bare = l == L && !coarse_iter;
    if (q.n > kLargest) return false;
    if (!bare && q.n > kSerial) d.na = l + 1;
  }
  ctas = d.na == 0 ? 1 : kVlcCtas;
  if (d.na > 0) {   // even line counts by the coarsest spread level, doubled towards the finer ones
    const int lc = d.na - 1;
    for (int k = 0; k <= ctas; ++k) {
      d.lv[lc].lb[k] = k == ctas ? d.lv[lc].w : k * d.lv[lc].w / ctas / 2 * 2;
      for (int l = lc - 1; l >= 0; --l) d.lv[l].lb[k] = k == ctas ? d.lv[l].w : 2 * d.lv[l + 1].lb[k];
    }
  }
  int off = 0;
  auto take = [&](int count) {
    const int o = off;
    off += (count + 1) / 2 * 2;
    return o;
  };
  for (int l = 0; l <= L; ++l) {
    VlcLevel &q = d.lv[l];
    int lines = q.w;
    if (l < d.na) {
      lines = 0;
      for (int k = 0; k < ctas; ++k) {
        const int own = q.lb[k + 1] - q.lb[k];
        if (own < 4) return false;
        lines = std::max(lines, own);
      }
    }
    q.cells = (lines + 1) / 2 * (q.n + 1);
    q.vec = (lines + kBelow + kAbove) * q.w;
    q.val_off = take(l == L && !coarse_iter ? 0 : kP2Slots * q.cells);
    q.dinv_off = take(q.vec);
    q.x_off = take(q.vec);
    q.t_off = take(q.vec);
    q.b_off = take(q.vec);
  }
  if (d.na > 0 && d.na <= L) {
    const int w = d.lv[d.na - 1].w;
    d.r_off = take((w + kBelow + kAbove) * w);
  }
  size_t bytes = (size_t)off * sizeof(float2);
  if (!coarse_iter) {
    const int wi = d.lv[L].w - 2, ni = 2 * wi * (wi + open);
    d.share = ctas > 1 && ni > 64;
    const int rows = d.share ? (ni + ctas - 1) / ctas : ni;
    bytes = (bytes + 15) / 16 * 16;
    d.cinv_off = (int)(bytes / 8);
    d.cinv_rows = rows;
    bytes += (size_t)(rows + 1) * ni * 8;
  }
  smem = bytes;
  // phases
  bool ok = true;
  auto add = [&](VlcPhase p, bool alone, int sync) {
    p.alone = alone;
    p.sync = (signed char)sync;
    if (d.nphase >= kVlcMaxPhases) ok = false;
    else d.ph[d.nphase++] = p;
  };
  auto from_zero = [&](int l, int deg) {   // ends in x
    const VlcLevel &q = d.lv[l];
    const bool spread = l < d.na;
    int cur = (deg - 1) % 2 == 0 ? q.x_off : q.t_off, oth = cur == q.x_off ? q.t_off : q.x_off;
    VlcPhase p;
    p.level = (signed char)l;
    p.op = VLC_INIT;
    p.out = cur;
    add(p, !spread, VLC_BLOCK);
    for (int s = 1; s < deg; ++s) {
      const bool result = d.nlev == 1 && s + 1 == deg;   // the coarsest level alone
      p.op = VLC_SWEEP;
      p.u = cur;
      p.out = oth;
      p.coef = (signed char)(4 + 3 * (s - 1));
      p.has_w = s > 1;
      p.where = result ? VLC_RESULT : spread ? VLC_HALO : VLC_HERE;
      add(p, !spread, result ? VLC_NONE : spread ? VLC_CLUSTER : VLC_BLOCK);
      std::swap(cur, oth);
    }
  };
  for (int l = 0; l <= L; ++l) {
    const VlcLevel &q = d.lv[l];
    const bool spread = l < d.na;
    VlcPhase p;
    p.level = (signed char)l;
    if (l == L) {
      if (coarse_iter) {
        from_zero(l, coarse_degree);
      } else {
        if (d.share) {
          VlcPhase bc;
          bc.op = VLC_BROADCAST;
          bc.u = q.b_off;
          bc.out = q.vec;
          add(bc, true, VLC_CLUSTER);
        }
        p.op = VLC_DENSE;
        add(p, !d.share, d.share ? VLC_CLUSTER : VLC_BLOCK);
      }
      break;
    }
    from_zero(l, degree);
    p.op = VLC_SWEEP;   // residual into t
    p.u = q.x_off;
    p.out = q.t_off;
    p.where = !spread ? VLC_HERE : l + 1 < d.na ? VLC_HALO_ABOVE : VLC_GATHER;
    add(p, !spread, spread ? VLC_CLUSTER : VLC_BLOCK);
    VlcPhase r;
    r.op = VLC_RESTRICT;
    r.level = (signed char)l;
    r.u = spread && l + 1 >= d.na ? d.r_off : q.t_off;
    add(r, l + 1 >= d.na, l + 1 < d.na ? VLC_CLUSTER : VLC_BLOCK);
  }
  for (int l = L - 1; l >= 0; --l) {
    const VlcLevel &q = d.lv[l];
    const bool spread = l < d.na;
    if (spread && l + 1 == d.na) {   // block 0's correction to every block
      VlcPhase bc;
      bc.op = VLC_BROADCAST;
      bc.u = d.lv[l + 1].x_off;
      bc.out = d.lv[l + 1].vec;
      add(bc, true, VLC_CLUSTER);
    }
    VlcPhase p;
    p.level = (signed char)l;
    p.op = VLC_PROLONG;
    p.where = spread ? VLC_HALO : VLC_HERE;
    add(p, !spread, spread ? VLC_CLUSTER : VLC_BLOCK);
    int cur = q.x_off, oth = q.t_off;
    for (int s = 0; s < degree; ++s) {
      const bool result = l == 0 && s + 1 == degree;
      p.op = VLC_SWEEP;
      p.u = cur;
      p.out = oth;
      p.coef = (signed char)(s == 0 ? 1 : 4 + 3 * (s - 1));
      p.has_w = s > 0;
      p.where = result ? VLC_RESULT : spread ? VLC_HALO : VLC_HERE;
      add(p, !spread, result ? VLC_NONE : spread ? VLC_CLUSTER : VLC_BLOCK);
      std::swap(cur, oth);
    }
  }
  d.pre_steps = d.nlev == 1 ? coarse_degree : degree;
  d.post_steps = d.nlev == 1 ? 0 : degree;
  return ok && smem + sizeof(Fixed) <= kSmemLimit;
}

// the transfer tables of every level pair
void transfer_tables(VlcDesc &d) {
  constexpr P2Transfers t = p2_transfers();
  for (int ty = 0; ty < 4; ++ty)
    for (int k = 0; k < t.rn[ty]; ++k) {
      d.rw[ty][k] = t.rw[ty][k];
      for (int l = 0; l + 1 < d.nlev; ++l) d.ro[l][ty][k] = t.rj[ty][k] * d.lv[l].w + t.ri[ty][k];
    }
  for (int c = 0; c < 16; ++c)
    for (int k = 0; k < t.pn[c]; ++k) {
      d.pw[c][k] = t.pw[c][k];
      for (int l = 0; l + 1 < d.nlev; ++l) d.po[l][c][k] = t.pj[c][k] * d.lv[l + 1].w + t.pi[c][k];
    }
}

bool runs(bool bf16, bool open, int ctas, size_t smem) {
  constexpr size_t most = kSmemLimit - sizeof(Fixed);
  if (bf16)
    return open ? cluster_runs<k_vel_cluster<__nv_bfloat16, true>>(ctas, kThreads, smem, most)
                : cluster_runs<k_vel_cluster<__nv_bfloat16, false>>(ctas, kThreads, smem, most);
  return open ? cluster_runs<k_vel_cluster<float, true>>(ctas, kThreads, smem, most)
              : cluster_runs<k_vel_cluster<float, false>>(ctas, kThreads, smem, most);
}

}  // namespace

VlcPlan vlc_plan(Arena &ar, const std::vector<const Level *> &lev, int open_top, const std::vector<P2Table> &tab,
                 const std::vector<float *> &val, const std::vector<__nv_bfloat16 *> &val16,
                 const std::vector<float *> &dinv, const std::vector<double *> &coef, const std::vector<float *> &b,
                 const std::vector<float *> &x, int degree, bool coarse_iter, int nc, const double *cinv) {
  VlcPlan plan;
  VlcDesc d;
  int first = 0;
  for (;; ++first) {
    if (first == (int)lev.size()) return plan;
    bool ok = layout(first, lev, open_top, degree, coarse_iter, d, plan.ctas, plan.smem);
    // one table for all of them
    for (size_t l = first; ok && l + (coarse_iter ? 0 : 1) < lev.size(); ++l) ok = tab[l].ok && tab[l].holds(tab[first]);
    if (ok && runs(val[first] == nullptr, open_top != 0, plan.ctas, plan.smem)) break;
  }
  transfer_tables(d);
  plan.bf16 = val[first] == nullptr;
  d.nc = coarse_iter ? 0 : nc;
  d.cinv = cinv;
  d.b = b[first];
  d.x = x[first];
  plan.open = open_top;
  for (int k = 0; k < 2 * (kP2Slots + kP2TopSlots); ++k)
    plan.tab[k] = plan.bf16 ? __bfloat162float(__double2bfloat16(tab[first].c[k])) : (float)tab[first].c[k];
  for (int l = 0; l < d.nlev; ++l) {
    VlcLevel &q = d.lv[l];
    if (l == d.nlev - 1 && !coarse_iter) break;
    q.val = plan.bf16 ? (const void *)val16[first + l] : (const void *)val[first + l];
    q.dinv = dinv[first + l];
    q.coef = coef[first + l];
    q.ncoef = 4 + 3 * ((l == d.nlev - 1 ? kCoarseDegree : degree) - 1);
  }
  plan.first = first;
  plan.desc = ar.alloc<VlcDesc>(1);
  CHNSS_CK(cudaMemcpy(plan.desc, &d, sizeof(d), cudaMemcpyHostToDevice));
  return plan;
}

namespace {
template <typename VT, bool OPEN>
void launch(const VlcPlan &p, cudaStream_t s) {
  Coef tab;
  for (int k = 0; k < 2 * (kP2Slots + kP2TopSlots); ++k) tab.c[k] = p.tab[k];
  launch_cluster(k_vel_cluster<VT, OPEN>, p.ctas, 1, kThreads, p.smem, s, (const VlcDesc *)p.desc, tab);
  CHNSS_LAUNCH_CK();
}
}  // namespace

void vlc_apply(const VlcPlan &p, cudaStream_t s) {
  if (p.bf16) {
    if (p.open) launch<__nv_bfloat16, true>(p, s);
    else launch<__nv_bfloat16, false>(p, s);
  } else if (p.open) {
    launch<float, true>(p, s);
  } else {
    launch<float, false>(p, s);
  }
}

}  // namespace chnss
